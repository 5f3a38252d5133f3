// Discrete adjoint of one free-surface LBM step (SRT, EQ refilling, no
// surface tension, walls and periodic faces), for gradients of a misfit of
// the surface elevation with respect to the viscosity, the gravity and the
// initial state.
//
// The forward step t -> t+1 (the library's own kernels) is replayed from a
// tape: for every step of a segment the stored PDFs F (post-collision, time
// level t), the cell flags, the interface mass M and the fill level Phi.
// The cell types and every conversion decision are taken from the tape
// (types at t and at t+1 tell which cells filled, emptied, were created or
// turned from liquid into interface), so the step is a smooth function of
// (F, M, Phi) and of the parameters, and its vector-Jacobian product is
// written out here by hand:
//
//   fin_i(x) = F_i(x - c_i)                       fluid source (streaming)
//            = F_i'(x)                            wall (halfway bounce-back)
//            = feq_i(rho_G, u*) + feq_i'(rho_G, u*) - F_i'(x)
//                                                 gas (Eq. nm-fslbm-boundary-condition),
//              u* = sum c F(x) / sum F(x) - g/2
//   m_new(x) = M(x) + sum_i d_i(x)                interface (Eq. nm-fslbm-mass-flux,
//              d_i = F_i'(y) - F_i(x), y = x + c_i liquid;
//              d_i = (Phi_x + Phi_y)/2 * br_i, y interface, br from Thuerey's table
//   rho = sum fin, u = sum c fin / rho + g/2, F = rho g
//   fn_i(x) = fin_i - omega (fin_i - feq_i(rho, u)) + (1 - omega/2) G_i(u, F)
//                                                 (Eqs. nm-lbm-collision, nm-lbm-force-guo)
//   interface at t+1: M1 = base + excess share, Phi1 = M1 / rho;
//     base = m_new (stayed interface), rho (liquid turned interface), 0 (new)
//   filled cell: m_ex = m_new - rho; emptied cell: m_ex = m_new (Eq. nm-fslbm-excess-mass),
//     shared evenly over its interface neighbours at t+1 (counted per direction)
//   new cell: fn(x) = feq(mean rho_y, mean u_y) over its valid neighbours y,
//     rho_y, u_y the moments of F(t+1)(y) (Sec. 3.1, EQ); its rho = sum fn(x)
//
// Every kernel is a gather (one thread per cell, no atomics on the adjoint
// fields) over the cells whose result a later kernel reads: the fields of
// other cells keep whatever they held.  The parameter gradients are summed in
// FP64, per block first and then with one atomic per block: one atomic per
// thread put 130,000 additions to the same four addresses in the way of each
// step (k_adj_collide has the figures).
#pragma once
// Included by fsl_api.cu after fsl_kernels.cuh.

namespace fsl {

// the tape entry of one time level
struct AdjLevel {
  const void* F;          // stored PDFs (storage type of the path), q planes
  const uint8_t* flags;   // cell flags (with the Thuerey classes of the level)
  const double* M;        // interface mass
  const double* Phi;      // fill level
};

// adjoint fields (arithmetic type R) and accumulators
template <class R>
struct AdjFields {
  R* lF;     // q planes: adjoint of F at t+1 (fluid cells)
  R* lF0;    // q planes: adjoint of F at t; the two swap roles every step
  R* lfin;   // q planes: adjoint of the pulled values fin at t (fluid cells)
  R* lM;     // cells: adjoint of M at t+1 (swaps with lM0)
  R* lM0;
  R* lP;     // cells: adjoint of Phi at t+1 (swaps with lP0)
  R* lP0;
  R* lm1;    // cells: adjoint of the mass at t+1 of interface-at-t+1 cells
  R* lrhoP;  // cells: adjoint of rho through Phi1 = M1 / rho (and the base m = rho)
  R* lmnew;  // cells: adjoint of m_new (interface-at-t cells)
  R* lbar;   // 4 per cell: (rho_bar, u_bar) adjoint of a new cell / |V|
  R* lg;     // 3 per cell: adjoint of u* of the gas boundary condition (interface at t)
  double* acc;  // [0] dJ/domega, [1..3] dJ/dg_a
};

constexpr int kAdjThreads = 128;

// v summed over the block's threads and added to *out by one atomic; every
// thread of the block calls it (it synchronises the block)
__device__ __forceinline__ void adj_block_add(double v, double* out) {
  __shared__ double part[kAdjThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = part[0];
    for (int w = 1; w < kAdjThreads / 32; ++w) s += part[w];
    if (s != 0.0) atomicAdd(out, s);
  }
  __syncthreads();
}

template <int Q, class ST>
__device__ __forceinline__ typename ST::R adj_ld(const void* F, long long plane, int i, int c) {
  using T = typename ST::T;
  return (typename ST::R)ST::ldf(reinterpret_cast<const T*>(F) + i * plane + c, wgt<Q>(i));
}

// Thuerey class of an interface cell from the flag byte of its level: 0
// standard, 1 no liquid neighbour (NF), 2 no gas neighbour (NE)
__device__ __forceinline__ int adj_class(uint8_t fl) {
  return (fl & F_NF) ? 1 : (fl & F_NE) ? 2 : 0;
}

// coefficients of f_in and f_out in the bracket of an interface pair
// (classes of the cell and of its neighbour); simple = plain f_in - f_out
__device__ __forceinline__ void adj_bracket(int cx, int cy, bool simple, int& a_in, int& a_out) {
  a_in = 1;
  a_out = -1;
  if (simple) return;
  if (cx == 0) {
    if (cy == 1) a_out = 0;
    else if (cy == 2) a_in = 0;
  } else if (cx == 1) {
    if (cy != 1) a_in = 0;
  } else {
    if (cy != 2) a_out = 0;
  }
}

template <int Q, class R>
__device__ __forceinline__ R adj_feq(int i, R rho, R ux, R uy, R uz) {
  const R cu = dot3r<R>(dir_c(i, 0), dir_c(i, 1), dir_c(i, 2), ux, uy, uz);
  const R usq = ux * ux + uy * uy + uz * uz;
  return (R)wgt<Q>(i) * rho * ((R)1 + (R)3 * cu + (R)4.5 * cu * cu - (R)1.5 * usq);
}

// density and momentum of q values, summed in direction order
template <int Q, class R>
__device__ __forceinline__ void adj_moments(const R* f, R& rho, R* j) {
  rho = f[0];
  j[0] = j[1] = j[2] = (R)0;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    rho += f[i];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (dir_c(i, a) == 1) j[a] += f[i];
      if (dir_c(i, a) == -1) j[a] -= f[i];
    }
  }
}

// The pulled values at t of a fluid cell, a bit mask of the directions whose
// source is gas, and the stored velocity u* of the cell (0 unless a source is
// gas).  A liquid cell with no wall or obstacle in its stencil pulls from
// fluid cells only (closed interface layer): no flag is read for it.
template <int Q, class ST>
__device__ __forceinline__ unsigned adj_fin(const Geom& g, const Phys& p, const AdjLevel& L, int c,
                                            uint8_t fl, const Nbr& nb, typename ST::R* fin,
                                            typename ST::R* us) {
  using R = typename ST::R;
  const long long P = g.plane;
  us[0] = us[1] = us[2] = (R)0;
  if ((fl & F_TYPE) == T_LIQ && !(fl & F_NEAR_OBST)) {
#pragma unroll
    for (int i = 0; i < Q; ++i)
      fin[i] = adj_ld<Q, ST>(L.F, P, i, nb.in(-dir_c(i, 0), -dir_c(i, 1), -dir_c(i, 2)));
    return 0u;
  }
  R own[Q];
  unsigned gas = 0u;
#pragma unroll
  for (int i = 0; i < Q; ++i) own[i] = adj_ld<Q, ST>(L.F, P, i, c);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int n = nb.at(-dir_c(i, 0), -dir_c(i, 1), -dir_c(i, 2));
    const int ns = n >= 0 ? n : c;
    const int t = n >= 0 ? (L.flags[ns] & F_TYPE) : T_OBST;
    const R v = adj_ld<Q, ST>(L.F, P, i, ns);
    fin[i] = is_fluid(t) ? v : own[opp(i)];
    if (t == T_GAS) gas |= 1u << i;
  }
  if (gas) {
    R r, j[3];
    adj_moments<Q, R>(own, r, j);
#pragma unroll
    for (int a = 0; a < 3; ++a) us[a] = j[a] / r - (R)0.5 * (R)p.g[a];
    const R rhoG = (R)(3.0 * p.p_v);
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if ((gas >> i) & 1u)
        fin[i] = adj_feq<Q, R>(i, rhoG, us[0], us[1], us[2]) +
                 adj_feq<Q, R>(opp(i), rhoG, us[0], us[1], us[2]) - fin[i];
  }
  return gas;
}

// B1: cells that are interface at t+1: adjoint of their mass and of the
// density that divides it; new cells (gas at t) also the adjoint of the means
// that their equilibrium was built from.  dj is d J / d (column height) at
// t+1, which spreads over the fill levels at x = 0 (the column height is
// their sum over y averaged over z).
template <int Q, class ST>
__global__ void __launch_bounds__(kAdjThreads)
    k_adj_interface(Geom g, Phys p, AdjLevel L0, AdjLevel L1, AdjFields<typename ST::R> A,
                    double dj) {
  using R = typename ST::R;
  const long long P = g.plane;
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  double dg[3] = {0.0, 0.0, 0.0};
  int x = 0, y = 0, z = 0;
  const int c = k < g.cells ? (int)k : 0;
  cell_xyz(g, c, x, y, z);
  const bool on = k < g.cells && x < g.nx && (L1.flags[c] & F_TYPE) == T_IF;
  if (!__syncthreads_or(on)) return;
  if (on) {
    Nbr nb;
    nb.setup(g, x, y, z);
    const uint8_t f0 = L0.flags[c];
    const bool born = (f0 & F_TYPE) == T_GAS;
    R rho, f[Q], tmp[3];
    if (born) {  // new cell: density of its refilled PDFs
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = adj_ld<Q, ST>(L1.F, P, i, c);
    } else {
      adj_fin<Q, ST>(g, p, L0, c, f0, nb, f, tmp);
    }
    rho = f[0];
#pragma unroll
    for (int i = 1; i < Q; ++i) rho += f[i];
    R lP = A.lP[c];
    if (x == 0) lP += (R)(dj / (double)g.nz);
    const R rp = -lP * (R)L1.Phi[c] / rho;
    A.lm1[c] = A.lM[c] + lP / rho;
    A.lrhoP[c] = rp;
    if (born) {
      int cnt = 0;
      R rsum = 0, us[3] = {0, 0, 0};
      // rolled: rare cells, and the body holds q loads
#pragma unroll 1
      for (int d = 1; d < Q; ++d) {
        const int n = nb.at(rc(d, 0), rc(d, 1), rc(d, 2));
        if (n < 0) continue;
        const int tn0 = L0.flags[n] & F_TYPE, tn1 = L1.flags[n] & F_TYPE;
        if (!is_fluid(tn1) || (tn0 == T_GAS)) continue;  // valid: fluid at t+1, not new
        R v[Q], r, j[3];
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = adj_ld<Q, ST>(L1.F, P, i, n);
        adj_moments<Q, R>(v, r, j);
        rsum += r;
#pragma unroll
        for (int a = 0; a < 3; ++a) us[a] += j[a] / r - (R)0.5 * (R)p.g[a];
        ++cnt;
      }
      R out[4] = {0, 0, 0, 0};
      if (cnt > 0) {
        const R rb = rsum / (R)cnt;
        const R ub[3] = {us[0] / (R)cnt, us[1] / (R)cnt, us[2] / (R)cnt};
        const R usq = ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2];
        R lrb = 0, lub[3] = {0, 0, 0};
#pragma unroll 1
        for (int i = 0; i < Q; ++i) {
          // fn_i = feq_i(rb, ub); rho of the cell = sum fn
          const R lf = A.lF[i * P + c] + rp;
          const R cu = (R)rc(i, 0) * ub[0] + (R)rc(i, 1) * ub[1] + (R)rc(i, 2) * ub[2];
          const R w = (R)rw<Q>(i);
          lrb += lf * w * ((R)1 + (R)3 * cu + (R)4.5 * cu * cu - (R)1.5 * usq);
#pragma unroll
          for (int a = 0; a < 3; ++a)
            lub[a] += lf * w * rb * ((R)3 * (R)rc(i, a) + (R)9 * cu * (R)rc(i, a) - (R)3 * ub[a]);
        }
        // u_y = j_y / rho_y - g/2 for every y: d ub / d g = -1/2
#pragma unroll
        for (int a = 0; a < 3; ++a) dg[a] = -0.5 * (double)lub[a];
        out[0] = lrb / (R)cnt;
#pragma unroll
        for (int a = 0; a < 3; ++a) out[1 + a] = lub[a] / (R)cnt;
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) A.lbar[4 * (long long)c + a] = out[a];
    }
  }
  for (int a = 0; a < 3; ++a) adj_block_add(dg[a], &A.acc[1 + a]);
}

// The collision's part of B2 in FP32: one operation after the other in the
// order of the formulas (out: the sums Lr, Lu, LF, dJ/domega).
template <int Q>
__device__ __forceinline__ void adj_collide_sums(const float* lfn, const float* fin, float rho,
                                                 const float* u, const float* F, float om,
                                                 float pre, float& Lr, float* Lu, float* LF,
                                                 double& dom) {
  using R = float;
  const R usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const R w = (R)wgt<Q>(i);
    const R cu = dot3r<R>(dir_c(i, 0), dir_c(i, 1), dir_c(i, 2), u[0], u[1], u[2]);
    const R cF = dot3r<R>(dir_c(i, 0), dir_c(i, 1), dir_c(i, 2), F[0], F[1], F[2]);
    const R feq = w * rho * ((R)1 + (R)3 * cu + (R)4.5 * cu * cu - (R)1.5 * usq);
    const R G = w * ((R)3 * (((R)dir_c(i, 0) - u[0]) * F[0] + ((R)dir_c(i, 1) - u[1]) * F[1] +
                             ((R)dir_c(i, 2) - u[2]) * F[2]) +
                     (R)9 * cu * cF);
    // fn = fin - om (fin - feq) + pre G
    Lr += lfn[i] * (om * feq / rho);  // d feq / d rho at fixed u
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const R ci = (R)dir_c(i, a);
      Lu[a] += lfn[i] * (om * w * rho * ((R)3 * ci + (R)9 * cu * ci - (R)3 * u[a]) +
                         pre * w * ((R)-3 * F[a] + (R)9 * ci * cF));
      LF[a] += lfn[i] * pre * w * ((R)3 * (ci - u[a]) + (R)9 * cu * ci);
    }
    dom += (double)(lfn[i] * (feq - fin[i] - (R)0.5 * G));
  }
}
// The same sums in FP64, regrouped for the two FP64 lanes of an SM: with
// wl = w_i lfn_i the terms of Lu and LF that do not depend on c_i need only
// S0 = sum wl, and those along c_i only sum wl c_i (3 + 9 cu) and
// sum wl c_i cF; about 25 fused operations per direction in place of 90.
template <int Q>
__device__ __forceinline__ void adj_collide_sums(const double* lfn, const double* fin, double rho,
                                                 const double* u, const double* F, double om,
                                                 double pre, double& Lr, double* Lu, double* LF,
                                                 double& dom) {
  const double usq = fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0]));
  const double uF = fma(u[2], F[2], fma(u[1], F[1], u[0] * F[0]));
  double S0 = 0.0, E = 0.0, Sc[3] = {0.0, 0.0, 0.0}, SF[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double wl = wgt<Q>(i) * lfn[i];
    const double cu = dot3r<double>(dir_c(i, 0), dir_c(i, 1), dir_c(i, 2), u[0], u[1], u[2]);
    const double cF = dot3r<double>(dir_c(i, 0), dir_c(i, 1), dir_c(i, 2), F[0], F[1], F[2]);
    S0 += wl;
    if (i == 0) {
      const double e = fma(-1.5, usq, 1.0);
      E = fma(wl, e, E);
      dom = fma(lfn[i], fma(wgt<Q>(i) * 1.5, uF, fma(wgt<Q>(i) * rho, e, -fin[i])), dom);
      continue;
    }
    const double t = fma(9.0, cu, 3.0);            // 3 + 9 cu
    const double e = fma(cu, fma(4.5, cu, 3.0), fma(-1.5, usq, 1.0));
    E = fma(wl, e, E);
    const double s = wl * t, v = wl * cF;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (dir_c(i, a) == 1) { Sc[a] += s; SF[a] += v; }
      if (dir_c(i, a) == -1) { Sc[a] -= s; SF[a] -= v; }
    }
    // G / w = 3 (cF - u.F) + 9 cu cF
    const double G = fma(t, cF, -3.0 * uF);
    dom = fma(lfn[i], fma(wgt<Q>(i), fma(rho, e, -0.5 * G), -fin[i]), dom);
  }
  Lr = om * E;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Lu[a] = fma(om * rho, fma(-3.0 * u[a], S0, Sc[a]), pre * fma(-3.0 * F[a], S0, 9.0 * SF[a]));
    LF[a] = pre * fma(-3.0 * u[a], S0, Sc[a]);
  }
}

// B2: every fluid cell at t: adjoint of m_new and of the collision density
// (including the excess mass of converted cells, gathered from receivers),
// then of the collision and of the gas boundary condition.
// What bounded it: the q-long arrays of a cell lived in local memory (loops
// over directions that were not unrolled), 57 divisions per cell, and one
// FP64 atomic per thread and parameter.  128x64x4 D3Q19 FP64 wave: 397 us and
// 7 us for the separate mass kernel before, 70 us now; the FP64 sums (16,000
// fluid cells of about 700 FP64 operations on two lanes per SM) are what is
// left.
template <int Q, class ST>
__global__ void __launch_bounds__(kAdjThreads)
    k_adj_collide(Geom g, Phys p, AdjLevel L0, AdjLevel L1, AdjFields<typename ST::R> A) {
  using R = typename ST::R;
  const long long P = g.plane;
  const R om = (R)p.omega, pre = (R)1 - (R)0.5 * om;
  const R gv[3] = {(R)p.g[0], (R)p.g[1], (R)p.g[2]};
  double dom = 0.0, dg[3] = {0.0, 0.0, 0.0};
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int x = 0, y = 0, z = 0;
  const int c = k < g.cells ? (int)k : 0;
  cell_xyz(g, c, x, y, z);
  const uint8_t f0 = L0.flags[c];
  const bool on = k < g.cells && x < g.nx && is_fluid(f0 & F_TYPE);
  if (!__syncthreads_or(on)) return;
  if (on) {
    Nbr nb;
    nb.setup(g, x, y, z);
    const int t0 = f0 & F_TYPE, t1 = L1.flags[c] & F_TYPE;
    // adjoint of the post-collision values fn(x) = F(t+1)(x)
    R lfn[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) lfn[i] = is_fluid(t1) ? A.lF[i * P + c] : (R)0;
    R lr = 0;
    if (t1 == T_IF) {
      const R m1 = A.lm1[c];
      lr = A.lrhoP[c];
      if (t0 == T_IF) A.lmnew[c] = m1;  // M1 = m_new + share
      else lr += m1;                    // liquid turned interface: M1 = rho + share
    } else if (t0 == T_IF) {
      // converted: excess mass to the interface neighbours at t+1
      int nr = 0;
      R s = 0;
#pragma unroll 1
      for (int d = 1; d < Q; ++d) {
        const int n = nb.at(rc(d, 0), rc(d, 1), rc(d, 2));
        if (n >= 0 && (L1.flags[n] & F_TYPE) == T_IF) {
          ++nr;
          s += A.lm1[n];
        }
      }
      const R lex = nr > 0 ? s / (R)nr : (R)0;  // no receiver: lost mass, no later effect
      A.lmnew[c] = lex;                         // m_ex = m_new - rho or m_new
      if (t1 == T_LIQ) lr = -lex;
    }
    if (t0 == T_IF && is_fluid(t1)) {
      // this cell's F(t+1) also fed the equilibrium of new neighbours (gas at
      // t, so only an interface cell has any)
      unsigned born = 0u;
#pragma unroll
      for (int d = 1; d < Q; ++d) {
        const int n = nb.at(dir_c(d, 0), dir_c(d, 1), dir_c(d, 2));
        const int ns = n >= 0 ? n : c;
        if (n >= 0 && (L0.flags[ns] & F_TYPE) == T_GAS && (L1.flags[ns] & F_TYPE) == T_IF)
          born |= 1u << d;
      }
      if (born) {
        R v1[Q], r1, j1[3];
#pragma unroll
        for (int i = 0; i < Q; ++i) v1[i] = adj_ld<Q, ST>(L1.F, P, i, c);
        adj_moments<Q, R>(v1, r1, j1);
#pragma unroll 1
        for (; born; born &= born - 1) {
          const int d = __ffs(born) - 1;
          const R* lb = A.lbar + 4 * (long long)nb.at(rc(d, 0), rc(d, 1), rc(d, 2));
          const R b0 = lb[0], b[3] = {lb[1], lb[2], lb[3]};
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            R v = b0;
#pragma unroll
            for (int a = 0; a < 3; ++a) v += b[a] * ((R)dir_c(i, a) - j1[a] / r1) / r1;
            lfn[i] += v;
          }
        }
      }
    }
    R fin[Q], us[3];
    const unsigned gas = adj_fin<Q, ST>(g, p, L0, c, f0, nb, fin, us);
    R rho, j[3];
    adj_moments<Q, R>(fin, rho, j);
    const R u[3] = {j[0] / rho + (R)0.5 * gv[0], j[1] / rho + (R)0.5 * gv[1], j[2] / rho + (R)0.5 * gv[2]};
    const R F[3] = {rho * gv[0], rho * gv[1], rho * gv[2]};
    R Lr = 0, Lu[3] = {0, 0, 0}, LF[3] = {0, 0, 0};
    adj_collide_sums<Q>(lfn, fin, rho, u, F, om, pre, Lr, Lu, LF, dom);
    // F = rho g: through rho and through g
#pragma unroll
    for (int a = 0; a < 3; ++a) Lr += LF[a] * gv[a];
#pragma unroll
    for (int a = 0; a < 3; ++a) dg[a] += (double)((R)0.5 * Lu[a] + LF[a] * rho);
    Lr += lr;
    // d u_a / d fin_i = (c_ia - j_a / rho) / rho: three values per axis
    R q[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int m = 0; m < 3; ++m) q[a][m] = (R)(m - 1) - j[a] / rho;
    R lgs[3] = {0, 0, 0};
    const R rhoG = (R)(3.0 * p.p_v);
    const R ir = (R)1 / rho;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      R v = ((R)1 - om) * lfn[i] + Lr;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const R t = Lu[a] * q[a][dir_c(i, a) + 1];
        if constexpr (sizeof(R) == 8) v = fma(t, ir, v);
        else v += t / rho;
      }
      A.lfin[i * P + c] = v;
      // gas sources: feq_i + feq_i' at (rho_G, u*)
      if ((gas >> i) & 1u) {
        const R w = (R)wgt<Q>(i);
        const R cu = dot3r<R>(dir_c(i, 0), dir_c(i, 1), dir_c(i, 2), us[0], us[1], us[2]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
          lgs[a] += v * (R)2 * w * rhoG * ((R)9 * cu * (R)dir_c(i, a) - (R)3 * us[a]);
      }
    }
    if (t0 == T_IF) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        A.lg[3 * (long long)c + a] = lgs[a];
        dg[a] += -0.5 * (double)lgs[a];  // u* = j*/rho* - g/2
      }
    }
  }
  adj_block_add(dom, &A.acc[0]);
  for (int a = 0; a < 3; ++a) adj_block_add(dg[a], &A.acc[1 + a]);
}

// B3: adjoint of the state at t (F, M, Phi) by gathering every use of it
template <int Q, class ST>
__global__ void __launch_bounds__(kAdjThreads)
    k_adj_state(Geom g, Phys p, AdjLevel L0, AdjFields<typename ST::R> A) {
  using R = typename ST::R;
  const long long P = g.plane;
  const bool simple = (p.options & 1u) != 0;
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= g.cells) return;
  const int c = (int)k;
  int x, y, z;
  cell_xyz(g, c, x, y, z);
  const uint8_t f0 = L0.flags[c];
  const int t0 = f0 & F_TYPE;
  if (x >= g.nx || !is_fluid(t0)) return;
  Nbr nb;
  nb.setup(g, x, y, z);
  const bool iface = t0 == T_IF;
  if (!iface) {
    // liquid: streaming and bounce-back, and the fluxes of interface neighbours
#pragma unroll
    for (int kd = 0; kd < Q; ++kd) {
      const int n = nb.at(dir_c(kd, 0), dir_c(kd, 1), dir_c(kd, 2));
      const int ns = n >= 0 ? n : c;
      const int tn = n >= 0 ? (L0.flags[ns] & F_TYPE) : T_OBST;
      const bool wall = tn == T_OBST;
      R v = A.lfin[(wall ? opp(kd) : kd) * P + (wall ? c : ns)];
      if (kd > 0 && tn == T_IF) v += A.lmnew[ns];  // d_k'(n) = F_k(x) - F_k'(n)
      A.lF0[kd * P + c] = v;
    }
    A.lM0[c] = (R)0;
    A.lP0[c] = (R)0;
    return;
  }
  const int cls = adj_class(f0);
  const R phx = (R)L0.Phi[c];
  const R lmx = A.lmnew[c];
  // stored moments of the cell (gas boundary condition)
  R own[Q], rs, js[3];
#pragma unroll
  for (int i = 0; i < Q; ++i) own[i] = adj_ld<Q, ST>(L0.F, P, i, c);
  adj_moments<Q, R>(own, rs, js);
  const R lg[3] = {A.lg[3 * (long long)c], A.lg[3 * (long long)c + 1], A.lg[3 * (long long)c + 2]};
  R q[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int m = 0; m < 3; ++m) q[a][m] = (R)(m - 1) - js[a] / rs;
  R lphi = 0;
#pragma unroll
  for (int kd = 0; kd < Q; ++kd) {
    const int ko = opp(kd);
    // the cell in direction c_k: consumer of F_k(x) by streaming, and the
    // partner of the interface pair (x, x + c_k)
    const int n = nb.at(dir_c(kd, 0), dir_c(kd, 1), dir_c(kd, 2));
    const int ns = n >= 0 ? n : c;
    const uint8_t fn = L0.flags[ns];
    const int tn = n >= 0 ? (fn & F_TYPE) : T_OBST;
    // streaming; bounce-back into direction k'; gas: - F_k(x) in fin_k'
    const bool fluid = is_fluid(tn);
    const R in = A.lfin[(fluid ? kd : ko) * P + (fluid ? ns : c)];
    R v = tn == T_GAS ? (R)0 - in : in;
#pragma unroll
    for (int a = 0; a < 3; ++a) v += lg[a] * q[a][dir_c(kd, a) + 1] / rs;
    if (kd > 0 && fluid) {
      // pair (x, n): own flux d_k(x) has f_out = F_k(x); n's flux d_k'(n)
      // has f_in = F_k(x)
      if (tn == T_LIQ) {
        v -= lmx;
      } else {
        const R phn = (R)L0.Phi[ns];
        const R lmn = A.lmnew[ns];
        const int cn = adj_class(fn);
        int a_in, a_out;
        adj_bracket(cls, cn, simple, a_in, a_out);
        const R half = (R)0.5 * (phx + phn);
        v += half * (R)a_out * lmx;
        // fill-level weights of both fluxes of the pair
        const R fin_x = adj_ld<Q, ST>(L0.F, P, ko, ns), fout_x = own[kd];
        const R br_x = (R)a_in * fin_x + (R)a_out * fout_x;
        int b_in, b_out;
        adj_bracket(cn, cls, simple, b_in, b_out);
        const R br_n = (R)b_in * fout_x + (R)b_out * fin_x;  // n's f_in = F_k(x), f_out = F_k'(n)
        lphi += (R)0.5 * br_x * lmx + (R)0.5 * br_n * lmn;
        v += half * (R)b_in * lmn;
      }
    }
    A.lF0[kd * P + c] = v;
  }
  A.lM0[c] = lmx;
  A.lP0[c] = lphi;
}

// The current state into a tape level: PDFs in 16-byte words, mass and fill
// level, flags.  One launch in place of four device copies per replayed step.
static __global__ void __launch_bounds__(256)
    k_adj_record(Dev d, int cur, long long f16, long long cells, uint4* F, uint8_t* flags, double* M,
                 double* Phi) {
  const long long t = blockIdx.x * 256ll + threadIdx.x, stride = gridDim.x * 256ll;
  const uint4* src = reinterpret_cast<const uint4*>(d.pdf[cur]);
  for (long long k = t; k < f16; k += stride) F[k] = src[k];
  for (long long k = t; k < cells; k += stride) {
    M[k] = d.mass[k];
    Phi[k] = d.phi[k];
    flags[k] = d.flags[k];
  }
}

// the initial state's adjoint: F = feq(rho0, 0), M = phi0 rho0 (interface) or
// rho0 (liquid), Phi = phi0; per cell d J / d rho0 and d J / d phi0 (dense
// x-fastest layout), and the hydrostatic rho0 = 1 + 3 g_a (x_a + 1/2 - h_ref)
// added to d J / d g_a
template <int Q, class ST>
__global__ void __launch_bounds__(kAdjThreads)
    k_adj_init(Geom g, Phys p, AdjLevel L0, AdjFields<typename ST::R> A, double h_ref,
               double* drho0, double* dphi0) {
  double dga = 0.0;
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int x = 0, y = 0, z = 0;
  const int c = k < g.cells ? (int)k : 0;
  cell_xyz(g, c, x, y, z);
  if (k < g.cells && x < g.nx) {
    const long long u = x + (long long)g.nx * (y + (long long)g.ny * z);
    const int t0 = L0.flags[c] & F_TYPE;
    double dr = 0.0, dp = 0.0;
    if (is_fluid(t0)) {
#pragma unroll
      for (int i = 0; i < Q; ++i) dr += (double)A.lF[i * g.plane + c] * wgt<Q>(i);
      if (t0 == T_IF) {
        dr += (double)A.lM[c] * L0.Phi[c];
        // rho0 of the cell: M0 / Phi0 when Phi0 > 0, else from the PDFs
        double r0 = 0.0;
#pragma unroll
        for (int i = 0; i < Q; ++i) r0 += (double)adj_ld<Q, ST>(L0.F, g.plane, i, c);
        dp = (double)A.lM[c] * r0 + (double)A.lP[c];
      } else {
        dr += (double)A.lM[c];
      }
      if (p.gaxis >= 0 && !isnan(h_ref)) {
        const int pa = p.gaxis == 0 ? x : p.gaxis == 1 ? y : z;
        dga += dr * 3.0 * (((double)pa + 0.5) - h_ref);
      }
    }
    drho0[u] = dr;
    dphi0[u] = dp;
  }
  if (p.gaxis >= 0) adj_block_add(dga, &A.acc[1 + p.gaxis]);
}

}  // namespace fsl
