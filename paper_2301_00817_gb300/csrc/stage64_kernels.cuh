// stage64_kernels.cuh -- kernel templates of the per-pass residual (node,
// viscosity, interface flux, update).  Instantiated for double by stage64.cu
// (the FP64 form) and for Dual by adjoint.cu (exact Jacobian-vector products
// used to check the hand-written adjoint).
#pragma once

#include "lesjet_dev.cuh"
#include "lesjet_host.h"

namespace lesjet {

template <typename R>
inline Consts<R> make_consts(const les_params& p) {
  Consts<R> K;
  K.gamma = (R)p.gamma;
  K.gm1 = (R)(p.gamma - 1.0);
  K.k2 = (R)p.k2;
  K.k4 = (R)p.k4;
  K.mu_scale = (R)(p.Re > 0.0 ? p.Mj / p.Re : 0.0);
  K.S_suth = (R)(110.4 / p.T_ref);
  K.axis = p.axis;
  K.cs2 = (R)(p.sgs_model == LES_SGS_VREMAN ? 2.5 * p.Cs * p.Cs : p.Cs * p.Cs);
  K.inv_gm1_pr = (R)(1.0 / ((p.gamma - 1.0) * p.Pr));
  K.inv_gm1_prs = (R)(1.0 / ((p.gamma - 1.0) * p.Pr_sgs));
  K.sgs = p.sgs_model;
  return K;
}

inline int blocks_for(long long count, int threads, long long cap = 0) {
  if (cap <= 0) cap = 64LL * sm_count();
  long long b = (count + threads - 1) / threads;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

constexpr int kFluxThreads = 128;  // k_flux3's block

template <typename R>
__device__ __forceinline__ R dot3(const R& a0, const R& a1, const R& a2, const R& b0, const R& b1,
                                  const R& b2) {
  return dev_fma(a2, b2, dev_fma(a1, b1, dev_mul(a0, b0)));
}

// ------------------------------------------------------------------ k_node
// Primitive recovery (System I energy), spectral radii lambda_d = |U_d| +
// a |grad d| and lbar_xi = lambda_xi + sqrt(lambda_xi lambda_eta) +
// sqrt(lambda_xi lambda_zeta) (= lambda_xi [1 + (lambda_eta/lambda_xi)^0.5 +
// (lambda_zeta/lambda_xi)^0.5]), cyclic for eta and zeta.  |grad d| is read
// from gn ([3][N], taken once at set-up) when given, else evaluated from M.
// Bound by the FP64 pipe: the kinetic energy is taken from the momenta and the
// mixed radii from the three roots (192 x 96 x 128: 326 -> 298 us).
template <typename R, typename TQ, typename TM, bool WITH_DT>
__global__ void __launch_bounds__(256) k_node(Grid g, Consts<R> K, const TQ* __restrict__ Q,
                                              const TM* __restrict__ M,
                                              const double* __restrict__ gn, R* __restrict__ node,
                                              double* __restrict__ partials,
                                              DevScalars* __restrict__ sc,
                                              double* __restrict__ dtl = nullptr,
                                              double cfl = 0.0) {
  begin_dependent();
  const long long N = g.N;
  double local_min = 1.0e300;
  int bad = 0;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const R rho = (R)Q[n];
    const R inv_rho = R(1) / rho;
    const R u = (R)Q[N + n] * inv_rho;
    const R v = (R)Q[2 * N + n] * inv_rho;
    const R w = (R)Q[3 * N + n] * inv_rho;
    const R ke = dot3((R)Q[N + n], (R)Q[2 * N + n], (R)Q[3 * N + n], u, v, w);
    const R p = K.gm1 * dev_fma(R(-0.5), ke, (R)Q[4 * N + n]);
    const R T = K.gamma * p * inv_rho;
    const R a = dev_sqrt(T);
    // the radii's node: itself, or for an axis node (J^-1 = 0 on ring j = 0,
    // Reading A27) its inward neighbour (i, 1, k), whose radii it takes
    long long nr = n;
    R ur = u, vr = v, wr = w, ar = a;
    if (K.axis && (R)M[9 * N + n] == R(0) && (n / g.n[2]) % g.n[1] == 0) {
      nr = n + g.stride[1];
      const R rho1 = (R)Q[nr];
      const R ir1 = R(1) / rho1;
      ur = (R)Q[N + nr] * ir1;
      vr = (R)Q[2 * N + nr] * ir1;
      wr = (R)Q[3 * N + nr] * ir1;
      const R k1 = dot3((R)Q[N + nr], (R)Q[2 * N + nr], (R)Q[3 * N + nr], ur, vr, wr);
      const R p1 = K.gm1 * dev_fma(R(-0.5), k1, (R)Q[4 * N + nr]);
      ar = dev_sqrt(K.gamma * p1 * ir1);
    }
    R lam[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const R mx = (R)M[(3 * d) * N + nr], my = (R)M[(3 * d + 1) * N + nr],
              mz = (R)M[(3 * d + 2) * N + nr];
      const R gd = gn ? (R)gn[d * N + nr] : dev_sqrt(mx * mx + my * my + mz * mz);
      lam[d] = dev_abs(mx * ur + my * vr + mz * wr) + ar * gd;
    }
    // lbar_d = r_d (r_0 + r_1 + r_2), r_d = sqrt(lambda_d)
    const R r0 = dev_sqrt(lam[0]), r1 = dev_sqrt(lam[1]), r2 = dev_sqrt(lam[2]);
    const R rs = r0 + r1 + r2;
    node[n] = u;
    node[N + n] = v;
    node[2 * N + n] = w;
    node[3 * N + n] = p;
    node[4 * N + n] = T;
    node[5 * N + n] = r0 * rs;
    node[6 * N + n] = r1 * rs;
    node[7 * N + n] = r2 * rs;
    if (WITH_DT) {
      const double inv = 1.0 / ((double)lam[0] + (double)lam[1] + (double)lam[2]);
      if ((g.glo | g.ghi) == 0 || owned_plane(g, (int)(n / g.stride[0]))) {  // a slab's ghost planes are its neighbour's
        if (!(rho > R(0)) || !(p > R(0)) || !(inv > 0.0) || !(inv < 1.0e300)) bad = 1;
        local_min = inv < local_min ? inv : local_min;
      }
      if (dtl) dtl[n] = cfl * inv;  // local step of Eq. localdt
    }
  }
  if (WITH_DT) {
    fill_partials(partials);
    __shared__ double smin[32];
    __shared__ int sbad;
    if (threadIdx.x == 0) sbad = 0;
    for (int off = 16; off > 0; off >>= 1)
      local_min = fmin(local_min, __shfl_xor_sync(0xffffffffu, local_min, off));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) smin[threadIdx.x >> 5] = local_min;
    if (bad) atomicOr(&sbad, 1);
    __syncthreads();
    if (threadIdx.x < 32) {
      double m = threadIdx.x < (blockDim.x >> 5) ? smin[threadIdx.x] : 1.0e300;
      for (int off = 16; off > 0; off >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, off));
      if (threadIdx.x == 0) {
        partials[blockIdx.x] = m;
        if (sbad) atomicOr(&sc->status, 1);
      }
    }
  }
}

// -------------------------------------------------------------------- k_mu
// Twice the node-centred computational derivative (central; one-sided second
// order at non-periodic faces).
template <typename R>
__device__ __forceinline__ R node_diff(const Grid& g, const R* __restrict__ f, long long n,
                                       const int c[3], int d) {
  const long long s = g.stride[d];
  const int nd = g.n[d];
  if (g.per[d]) {
    const long long np = (c[d] == nd - 1) ? n - (long long)(nd - 1) * s : n + s;
    const long long nm = (c[d] == 0) ? n + (long long)(nd - 1) * s : n - s;
    return f[np] - f[nm];
  }
  if (c[d] == 0) return R(-3) * f[n] + R(4) * f[n + s] - f[n + 2 * s];
  if (c[d] == nd - 1) return R(3) * f[n] - R(4) * f[n - s] + f[n - 2 * s];
  return f[n + s] - f[n - s];
}

// mu_eff = (Mj/Re) T^1.5 (1+S)/(T+S) + mu_sgs; kappa_eff = mu_lam/((g-1)Pr)
// + mu_sgs/((g-1)Pr_sgs).  Smagorinsky: rho (Cs Delta)^2 |S|; Vreman:
// rho c sqrt(B_beta/alpha:alpha) (0 when alpha:alpha = 0, B_beta >= 0);
// dynamic: C_ds rho Delta^2 |S| with the dynamic Pr_sgs and the Yoshizawa
// sigma_ll = 2 C_I rho Delta^2 |S|^2 as a third field (coefficients dyn[6..8]
// from the dynamic procedure); Delta = (J^-1)^(1/3), Delta^2 from del2 (set-up).
// The gradient is kept at twice its value and the strain at four times, whose
// powers of two leave with one constant (FP64-pipe bound: 158 operations per
// node with Smagorinsky before, when it also took the cube root, 82 now; 192 x
// 96 x 128 593 -> 448 us).
template <typename R, typename TQ, typename TM>
__global__ void __launch_bounds__(256) k_mu(Grid g, Consts<R> K, const TQ* __restrict__ Q,
                                            const TM* __restrict__ M,
                                            const R* __restrict__ node, R* __restrict__ mk,
                                            const double* __restrict__ del2,
                                            const double* __restrict__ dyn = nullptr) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const R T = node[4 * N + n];
    const R mu_l = K.mu_scale * T * dev_sqrt(T) * (R(1) + K.S_suth) / (T + K.S_suth);
    R mu_s = R(0);
    R kap_s = R(0);
    bool kap_set = false;
    if (K.sgs != LES_SGS_NONE) {
      int c[3];
      decompose(g, n, c);
      R gr[3][3];  // 2 d u_i / d x_x
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        R dd[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) dd[d] = node_diff(g, node + q * N, n, c, d);
#pragma unroll
        for (int x = 0; x < 3; ++x)
          gr[q][x] = (R)M[x * N + n] * dd[0] + (R)M[(3 + x) * N + n] * dd[1] +
                     (R)M[(6 + x) * N + n] * dd[2];
      }
      const R rd2 = (R)Q[n] * (R)del2[n];  // rho Delta^2
      if (K.sgs == LES_SGS_SMAGORINSKY || K.sgs == LES_SGS_DYNAMIC) {
        // |S|^2 = 2 S:S = 2 sum_i g_ii^2 + sum_{i<j} (g_ij + g_ji)^2 of the
        // gradient g = gr/2
        const R d = gr[0][0] * gr[0][0] + gr[1][1] * gr[1][1] + gr[2][2] * gr[2][2];
        const R s01 = gr[0][1] + gr[1][0], s02 = gr[0][2] + gr[2][0], s12 = gr[1][2] + gr[2][1];
        const R o = s01 * s01 + s02 * s02 + s12 * s12;
        const R smag2 = R(0.25) * (R(2) * d + o);  // |S|^2
        const R smag = dev_sqrt(smag2);
        if (K.sgs == LES_SGS_SMAGORINSKY) {
          mu_s = rd2 * K.cs2 * smag;
        } else {
          mu_s = R(dyn[6]) * rd2 * smag;
          kap_s = mu_s / (K.gm1 * R(dyn[8]));
          kap_set = true;
          mk[2 * N + n] = R(2) * R(dyn[7]) * rd2 * smag2;
        }
      } else {
        // alpha_ij = d u_j / d x_i = gr[j][i]; beta_ij = Delta^2 alpha_mi alpha_mj:
        // sqrt(B_beta/alpha:alpha) = Delta^2 sqrt(B_gg/alpha:alpha) with gg =
        // alpha_mi alpha_mj, here 4x (B_gg 16x, alpha:alpha 4x)
        R b[3][3], aa = R(0);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = i; j < 3; ++j)
            b[i][j] = gr[i][0] * gr[j][0] + gr[i][1] * gr[j][1] + gr[i][2] * gr[j][2];
        aa = b[0][0] + b[1][1] + b[2][2];
        R B = b[0][0] * b[1][1] - b[0][1] * b[0][1] + b[0][0] * b[2][2] - b[0][2] * b[0][2] +
              b[1][1] * b[2][2] - b[1][2] * b[1][2];
        B = B > R(0) ? B : R(0);
        mu_s = (aa == R(0)) ? R(0) : rd2 * K.cs2 * R(0.5) * dev_sqrt(B / aa);
      }
    }
    mk[n] = mu_l + mu_s;
    mk[N + n] = mu_l * K.inv_gm1_pr + (kap_set ? kap_s : mu_s * K.inv_gm1_prs);
  }
}

// ----------------------------------------------------------------- k_flux3
// Pressure sensor |p+ - 2p + p-| / (p+ + 2p + p-) from the three pressures
// around a node; a face node of a non-periodic direction takes its inward
// neighbour's value.  The second difference is that of the two first ones,
// which are exact where the pressures are close, and the sum is it plus 4 p.
template <typename R>
__device__ __forceinline__ R sensor3(R pm, R p0, R pp) {
  const R s = (pp - p0) - (p0 - pm);
  return dev_abs(s) / dev_fma(R(4), p0, s);
}

template <int D, typename R>
__device__ __forceinline__ R sensor(const Grid& g, const R* __restrict__ P, long long x, int cx) {
  const long long s = g.stride[D];
  const int nd = g.n[D];
  long long xc = x;
  int cc = cx;
  if (!g.per[D]) {
    if (cx == 0) { xc = x + s; cc = 1; }
    else if (cx == nd - 1) { xc = x - s; cc = nd - 2; }
  }
  const long long xp = (cc == nd - 1) ? xc - (long long)(nd - 1) * s : xc + s;
  const long long xm = (cc == 0) ? xc + (long long)(nd - 1) * s : xc - s;
  return sensor3(P[xm], P[xc], P[xp]);
}

// What an interface flux along D reads at one of its two nodes.
template <typename R>
struct FluxNode {
  R W[5], p;         // rho, rho u, rho v, rho w, e + p; p
  R u, v, w, T;
  R m[9], J;         // metrics and J^-1
  R lb, mu, ka, sg;  // lbar_D, mu_eff, kappa_eff, sigma_ll (dynamic model)
  // per node, shared by its two interfaces along D:
  R F[5];            // J^-1 times the inviscid flux (Eq. hat-flux-G, xi_t = 0)
  R t1[4], t2[4];    // phi(+t) - phi(-t) of u, v, w, T along T1, T2
};

template <typename R, typename TQ, typename TM>
struct FluxIO {
  const TQ* Q;
  const TM* M;
  const R* node;
  const R* mk;
  R* F;
};

template <typename R, typename TQ, typename TM>
__device__ __forceinline__ void flux_W(const FluxIO<R, TQ, TM>& io, long long N, long long n,
                                       R W[5], R& p) {
  p = io.node[3 * N + n];
#pragma unroll
  for (int q = 0; q < 4; ++q) W[q] = (R)io.Q[q * N + n];
  W[4] = (R)io.Q[4 * N + n] + p;
}

// The node's data but W and p, without the part its interfaces share.
template <int D, typename R, typename TQ, typename TM>
__device__ __forceinline__ void flux_load(const FluxIO<R, TQ, TM>& io, long long N, bool dyn,
                                          long long n, FluxNode<R>& x) {
  x.u = io.node[n];
  x.v = io.node[N + n];
  x.w = io.node[2 * N + n];
  x.T = io.node[4 * N + n];
  x.lb = io.node[(5 + D) * N + n];
#pragma unroll
  for (int t = 0; t < 9; ++t) x.m[t] = (R)io.M[t * N + n];
  x.J = (R)io.M[9 * N + n];
  x.mu = io.mk[n];
  x.ka = io.mk[N + n];
  if (dyn) x.sg = io.mk[2 * N + n];
}

// The shared part: node flux and tangential differences (c: the node's
// coordinates along T1 and T2, inside their faces).
template <int D, typename R, typename TQ, typename TM>
__device__ __forceinline__ void flux_shared(const Grid& g, const FluxIO<R, TQ, TM>& io,
                                            long long n, const int c[3], FluxNode<R>& x) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  const long long N = g.N;
  const long long p1 = step(g, n, c, T1, 1), m1 = step(g, n, c, T1, -1);
  const long long p2 = step(g, n, c, T2, 1), m2 = step(g, n, c, T2, -1);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const R* phi = io.node + (q == 3 ? 4 : q) * N;
    x.t1[q] = phi[p1] - phi[m1];
    x.t2[q] = phi[p2] - phi[m2];
  }
  const R mx = x.m[3 * D], my = x.m[3 * D + 1], mz = x.m[3 * D + 2];
  const R Jt = dev_mul(x.J, dot3(mx, my, mz, x.u, x.v, x.w)), Jp = dev_mul(x.J, x.p);
  x.F[0] = dev_mul(x.W[0], Jt);
  // (the pressure part, the larger one outside the jet, in the fma: two
  // roundings of it instead of three)
  x.F[1] = dev_fma(Jp, mx, dev_mul(x.W[1], Jt));
  x.F[2] = dev_fma(Jp, my, dev_mul(x.W[2], Jt));
  x.F[3] = dev_fma(Jp, mz, dev_mul(x.W[3], Jt));
  x.F[4] = dev_mul(x.W[4], Jt);
}

// Exactly twice the flux through the interface (a, b = a + e_D): centred
// inviscid flux minus J^-1 times the Turkel-Vatsa dissipation minus the
// viscous + SGS flux.  The interface means are left as sums of the two
// nodes' values and their powers of two are folded into a few factors
// (exact in binary floating point); k_update halves J once per node.
template <int D, typename R>
__device__ __forceinline__ void flux_iface(const Consts<R>& K, const FluxNode<R>& a,
                                           const FluxNode<R>& b, const R Wm[5], const R Wp[5],
                                           R nua, R nub, R F[5]) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  // Turkel-Vatsa dissipation (Eqs. dissip_term, eps_2/4_dissip, W_dissip).
  // With D1 = W_b - W_a and E = W_{b+1} - W_{a-1}, the third difference is
  // E - 3 D1, so eps2 D1 - eps4 D3 = (eps2 + 3 eps4) D1 - eps4 E: two
  // differences and two multiply-adds per component.  At a face the missing
  // outside difference is minus the first inside one, i.e. the caller's
  // W_{a-1} = W_b or W_{b+1} = W_a.
  const R k2h = R(0.5) * K.k2, k4h = R(0.5) * K.k4, nu = dev_max(nua, nub);
  const R eps2 = dev_mul(k2h, nu);                          // half of eps^(2)
  const R eps4 = dev_max(R(0), dev_fma(-k2h, nu, k4h));     // half of eps^(4)
  const R sJ = a.J + b.J;                                   // 2 J^-1 at the interface
  const R lJ = dev_mul(a.lb + b.lb, sJ);                    // 4 lambda J^-1
  const R d1 = dev_mul(lJ, dev_fma(R(3), eps4, eps2)), d3 = dev_mul(lJ, eps4);
  // The momentum fluxes carry the pressure, whose magnitude sets the rounding
  // of the whole residual: their dissipation is collected first and meets it
  // in one rounding (three operations more than the chain of two; error of the
  // residual against the plain form in 64 bits 4.5e-14 -> 3.4e-14).  Mass and
  // energy take the small terms one by one on either node's flux before the
  // sum, at half its magnitude.
  R Fb[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    if (q >= 1 && q <= 3) {
      F[q] = (a.F[q] + b.F[q]) - dev_fma(-d3, Wp[q] - Wm[q], dev_mul(d1, b.W[q] - a.W[q]));
    } else {
      F[q] = dev_fma(-d1, b.W[q] - a.W[q], a.F[q]);
      Fb[q] = dev_fma(d3, Wp[q] - Wm[q], b.F[q]);
    }
  }

  // viscous + SGS flux with compact interface gradients (Eqs.
  // hat-flux-Ev/Fv/Gv, tau_mod, q_mod with Fourier's sign): the normal
  // differences, and 4x the tangential derivatives (the mean of the two
  // nodes' central differences)
  const R dn[4] = {b.u - a.u, b.v - a.v, b.w - a.w, b.T - a.T};
  R s1[4], s2[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    s1[q] = a.t1[q] + b.t1[q];
    s2[q] = a.t2[q] + b.t2[q];
  }
  // interface metrics at 2x their mean
  R mh[9];
  if (K.axis) {
    // a grid with an axis (Reading A27): the J^-1-weighted mean
    // (J^-1_a m_a + J^-1_b m_b)/(J^-1_a + J^-1_b), kept at 2x like the
    // plain sum; an axis node's stored metric is J^-1 m already
    const R wa = (a.J == R(0)) ? R(1) : a.J, wb = (b.J == R(0)) ? R(1) : b.J;
    const R r2 = R(2) / sJ;
#pragma unroll
    for (int t = 0; t < 9; ++t) mh[t] = dev_mul(dev_fma(wa, a.m[t], dev_mul(wb, b.m[t])), r2);
  } else {
#pragma unroll
    for (int t = 0; t < 9; ++t) mh[t] = a.m[t] + b.m[t];
  }
  // The flux needs only m.tau and m.q (m = the interface metric of
  // direction D), which follow from the contractions g_t = m . m_t and
  // c_t = sum_j m_j dphi_j,t and the divergence without forming the
  // gradient tensor:
  //   m.tau_i / mu = sum_t g_t dphi_i,t + sum_t m_t,i c_t - 2/3 m_i div,
  //   m.grad T     = sum_t g_t dphi_T,t,
  // where the normal part of div is c_D itself.  With 2x metrics, 1x normal
  // and 4x tangential differences every sum is 16x its value (g_D and c_D
  // take the missing factor 4).
  const R* m = mh + 3 * D;
  const R* m1 = mh + 3 * T1;
  const R* m2 = mh + 3 * T2;
  const R gD = dev_mul(R(4), dot3(m[0], m[1], m[2], m[0], m[1], m[2]));
  const R g1 = dot3(m[0], m[1], m[2], m1[0], m1[1], m1[2]);
  const R g2 = dot3(m[0], m[1], m[2], m2[0], m2[1], m2[2]);
  const R cD = dev_mul(R(4), dot3(m[0], m[1], m[2], dn[0], dn[1], dn[2]));
  const R c1 = dot3(m[0], m[1], m[2], s1[0], s1[1], s1[2]);
  const R c2 = dot3(m[0], m[1], m[2], s2[0], s2[1], s2[2]);
  R div = cD;  // 8 div
#pragma unroll
  for (int i = 0; i < 3; ++i) div = dev_fma(m2[i], s2[i], dev_fma(m1[i], s1[i], div));
  const R eD = dev_fma(R(-2.0 / 3.0), div, cD);
  R sv[3];  // 16 m.tau_i / mu
#pragma unroll
  for (int i = 0; i < 3; ++i)
    sv[i] = dev_fma(m2[i], c2, dev_fma(m1[i], c1, dev_fma(m[i], eD,
                    dot3(gD, g1, g2, dn[i], s1[i], s2[i]))));
  const R aT = dot3(gD, g1, g2, dn[3], s1[3], s2[3]);  // 16 m.grad T
  const R uf[3] = {a.u + b.u, a.v + b.v, a.w + b.w};  // 2 u at the interface
  // 2 J^-1 m.tau_i = sJ (2 mu) sv_i / 32; 2 J^-1 m.(tau u_f + kappa grad T) =
  // sJ (2 mu) (2 u_f . sv) / 64 + sJ (2 kappa) aT / 32
  const R sJ32 = dev_mul(sJ, R(1.0 / 32.0));
  const R cm = dev_mul(sJ32, a.mu + b.mu), ck = dev_mul(sJ32, a.ka + b.ka);
#pragma unroll
  for (int i = 0; i < 3; ++i) F[1 + i] = dev_fma(-cm, sv[i], F[1 + i]);
  F[4] = dev_fma(dev_mul(R(-0.5), cm), dot3(uf[0], uf[1], uf[2], sv[0], sv[1], sv[2]), F[4]);
  Fb[4] = dev_fma(-ck, aT, Fb[4]);
  if (K.sgs == LES_SGS_DYNAMIC) {
    // the modelled isotropic SGS stress sigma_ll/3 (Eq. yoshizawa) at the
    // interface mean, subtracted from the normal stresses: m.tau_i gains
    // -m_i sigma/3 and u_f.(m.tau) gains -(u_f . m) sigma/3
    const R e = dev_mul(dev_mul(sJ, a.sg + b.sg), R(1.0 / 12.0));
#pragma unroll
    for (int i = 0; i < 3; ++i) F[1 + i] = dev_fma(e, m[i], F[1 + i]);
    F[4] = dev_fma(dev_mul(R(0.5), e), dot3(uf[0], uf[1], uf[2], m[0], m[1], m[2]), F[4]);
  }
#pragma unroll
  for (int q = 0; q < 5; q += 4) F[q] = F[q] + Fb[q];
}

// Interfaces along xi (D = 0) or eta (D = 1): a thread walks a chunk of len
// interfaces along D and keeps node b's data as the next interface's node
// a, so the node flux, the tangential differences and the sensor are
// evaluated once per node (plus one per chunk).
template <int D, typename R, typename TQ, typename TM>
__device__ __forceinline__ void flux_chain(const Grid& g, const Consts<R>& K,
                                           const FluxIO<R, TQ, TM>& io, long long id, int len) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  const long long N = g.N;
  const int nif = g.per[D] ? g.n[D] : g.n[D] - 1;  // interfaces of a line
  const int nch = (nif + len - 1) / len;
  // consecutive threads take consecutive k
  int c[3];
  const long long r = id / g.n[2];
  c[2] = (int)(id - r * g.n[2]);
  if (D == 0) {
    c[0] = (int)(r / g.n[1]);
    c[1] = (int)(r - (long long)c[0] * g.n[1]);
  } else {
    c[0] = (int)(r / nch);
    c[1] = (int)(r - (long long)c[0] * nch);
  }
  if (c[0] >= (D == 0 ? nch : g.n[0])) return;
  c[D] *= len;
  if (!g.per[T1] && (c[T1] == 0 || c[T1] == g.n[T1] - 1)) return;
  if (!g.per[T2] && (c[T2] == 0 || c[T2] == g.n[T2] - 1)) return;
  const int end = c[D] + len < nif ? c[D] + len : nif;
  const bool dyn = K.sgs == LES_SGS_DYNAMIC;
  R* F = io.F + 5 * N * D;

  long long na = idx3(g, c[0], c[1], c[2]);
  FluxNode<R> a, b;
  R Wm[5], pm = R(0);
  const long long nm = step(g, na, c, D, -1);
  bool has_m = nm >= 0;
  if (has_m) flux_W(io, N, nm, Wm, pm);
  flux_W(io, N, na, a.W, a.p);
  flux_load<D>(io, N, dyn, na, a);
  flux_shared<D>(g, io, na, c, a);
  long long nb = step(g, na, c, D, 1);
  flux_W(io, N, nb, b.W, b.p);
  R nua = R(0);
  if (has_m) nua = sensor3(pm, a.p, b.p);
  for (int x = c[D]; x < end; ++x) {
    c[D] = x;
    const long long np = step(g, na, c, D, 2);
    const bool has_p = np >= 0;
    R Wp[5], pp = R(0);
    if (has_p) flux_W(io, N, np, Wp, pp);
    flux_load<D>(io, N, dyn, nb, b);
    flux_shared<D>(g, io, nb, c, b);
    R nub = nua;
    if (has_p) {
      nub = sensor3(a.p, b.p, pp);
    } else {
#pragma unroll
      for (int q = 0; q < 5; ++q) Wp[q] = a.W[q];
    }
    if (!has_m) {
      nua = nub;
#pragma unroll
      for (int q = 0; q < 5; ++q) Wm[q] = b.W[q];
    }
    R Fq[5];
    flux_iface<D>(K, a, b, Wm, Wp, nua, nub, Fq);
#pragma unroll
    for (int q = 0; q < 5; ++q) F[q * N + na] = Fq[q];
#pragma unroll
    for (int q = 0; q < 5; ++q) Wm[q] = a.W[q];
    has_m = true;
    a = b;
    nua = nub;
    na = nb;
    nb = np;
#pragma unroll
    for (int q = 0; q < 5; ++q) b.W[q] = Wp[q];
    b.p = pp;
  }
}

// Interfaces along zeta: one per thread over a block's run of consecutive
// nodes, which share each node's part through shared memory; only the last
// node of the run (and a wrap that leaves it) evaluates its neighbour's.
template <typename R, typename TQ, typename TM>
__device__ __forceinline__ void flux_zeta(const Grid& g, const Consts<R>& K,
                                          const FluxIO<R, TQ, TM>& io, long long n0,
                                          R (*sh)[kFluxThreads]) {
  const long long N = g.N, n = n0 + threadIdx.x;
  const R* P = io.node + 3 * N;
  const bool dyn = K.sgs == LES_SGS_DYNAMIC;
  int c[3] = {0, 0, 0};
  bool in = n < N;
  if (in) {
    decompose(g, n, c);
    in = (g.per[0] || (c[0] > 0 && c[0] < g.n[0] - 1)) &&
         (g.per[1] || (c[1] > 0 && c[1] < g.n[1] - 1));
  }
  FluxNode<R> a, b;
  R nua = R(0);
  if (in) {
    flux_W(io, N, n, a.W, a.p);
    flux_load<2>(io, N, dyn, n, a);
    flux_shared<2>(g, io, n, c, a);
    nua = sensor<2>(g, P, n, c[2]);
#pragma unroll
    for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = a.F[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sh[5 + q][threadIdx.x] = a.t1[q];
      sh[9 + q][threadIdx.x] = a.t2[q];
    }
    sh[13][threadIdx.x] = nua;
  }
  __syncthreads();
  if (!in) return;
  const long long nb = step(g, n, c, 2, 1);
  if (nb < 0) return;
  flux_W(io, N, nb, b.W, b.p);
  flux_load<2>(io, N, dyn, nb, b);
  R nub;
  if (nb >= n0 && nb < n0 + kFluxThreads) {
    const int s = (int)(nb - n0);
#pragma unroll
    for (int q = 0; q < 5; ++q) b.F[q] = sh[q][s];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      b.t1[q] = sh[5 + q][s];
      b.t2[q] = sh[9 + q][s];
    }
    nub = sh[13][s];
  } else {
    flux_shared<2>(g, io, nb, c, b);
    nub = sensor<2>(g, P, nb, coord_step(g, c, 2, 1));
  }
  R Wm[5], Wp[5], unused;
  const long long nm = step(g, n, c, 2, -1), np = step(g, n, c, 2, 2);
  flux_W(io, N, nm >= 0 ? nm : nb, Wm, unused);  // at a face W_{a-1} = W_b
  flux_W(io, N, np >= 0 ? np : n, Wp, unused);   // and W_{b+1} = W_a
  R Fq[5];
  flux_iface<2>(K, a, b, Wm, Wp, nua, nub, Fq);
#pragma unroll
  for (int q = 0; q < 5; ++q) io.F[(10 + q) * N + n] = Fq[q];
}

// The interface fluxes of the three directions in one launch (2x their
// value, F[D][5][N] at the interface's node a): blocks [0, b0) take xi and the
// next b1 eta in chunks of len interfaces, the rest zeta.  Bound by
// the FP64 pipe, which issues one warp instruction per 64 cycles and
// scheduler, so the shape is chosen for the fewest FP64 operations: 160 per
// interface with chunks of 16 (162 with 8, 165 with 4, 172 with 2, 185 without;
// 218 with the sensor pass's share before the node part was shared and the
// dissipation and viscous sums regrouped); 85 to 88 % of the pipe's rate.
// Comparisons and absolute values are done on the integer pipe (dev_max,
// dev_abs).  Against one launch per direction with a sensor pass ahead of
// them: the 192 x 96 x 128 step 18.3 -> 13.0 ms, the 48 x 24 x 32 step (three
// launches fewer per residual) 0.50 -> 0.26 ms.
template <typename R, typename TQ, typename TM>
__global__ void __launch_bounds__(kFluxThreads, sizeof(R) == 8 ? 2 : 1)
    k_flux3(Grid g, Consts<R> K, FluxIO<R, TQ, TM> io, unsigned b0, unsigned b1, int len) {
  begin_dependent();
  __shared__ R sh[14][kFluxThreads];
  const unsigned b = blockIdx.x;
  if (b < b0) {
    flux_chain<0>(g, K, io, (long long)b * kFluxThreads + threadIdx.x, len);
  } else if (b < b0 + b1) {
    flux_chain<1>(g, K, io, (long long)(b - b0) * kFluxThreads + threadIdx.x, len);
  } else {
    flux_zeta(g, K, io, (long long)(b - b0 - b1) * kFluxThreads, sh);
  }
}

// Blocks of k_flux3 for chunks of at most len interfaces.
struct FluxPlan {
  unsigned b2, b0, b1;
  int len;
};
inline FluxPlan flux_plan(const Grid& g) {
  // A chunk repeats one node's part, 39 FP64 operations beside the 159 of each
  // interface.  The chunks' blocks come first and zeta's, one interface per
  // thread, fill the end, so a chunk may last half of an SM's share (waves of
  // the two resident blocks of one interface per thread).  Against a dozen
  // waves of chunks behind zeta's blocks: 48 x 24 x 32 (waves 2) 280 -> 269 us a
  // step, residual on 73 x 53 x 45 (13) 290 -> 263 us, adjoint window on 64 x 40 x
  // 48 (9) 28.7 -> 27.4 ms; 8 instead of 4 at 13 waves 272 us, 4 instead of 2 at
  // 2 waves 324; 16 instead of 8 on 192 x 96 x 128 (181) 12.80 -> 12.62 ms.
  const long long waves = 3 * g.N / ((long long)kFluxThreads * 2 * sm_count());
  const int len =
      waves >= 64 ? 16 : (waves >= 16 ? 8 : (waves >= 4 ? 4 : (waves >= 2 ? 2 : 1)));
  auto blocks = [](long long t) { return (unsigned)((t + kFluxThreads - 1) / kFluxThreads); };
  auto chunks = [&](int d) { return ((g.per[d] ? g.n[d] : g.n[d] - 1) + len - 1) / len; };
  FluxPlan f;
  f.len = len;
  f.b2 = blocks(g.N);
  f.b0 = blocks((long long)chunks(0) * g.n[1] * g.n[2]);
  f.b1 = blocks((long long)g.n[0] * chunks(1) * g.n[2]);
  return f;
}

// ---------------------------------------------------------------- k_update
template <typename R, typename TM, typename TO, int MODE>
__global__ void __launch_bounds__(256) k_update(Grid g, const R* __restrict__ F,
                                                const double* __restrict__ Q0,
                                                const TM* __restrict__ M,
                                                const DevScalars* __restrict__ sc, double alpha,
                                                TO* __restrict__ out,
                                                const double* __restrict__ dtl = nullptr,
                                                const double* __restrict__ jh = nullptr) {
  begin_dependent();
  const long long N = g.N;
  const R* F0 = F;
  const R* F1 = F + 5 * N;
  const R* F2 = F + 10 * N;
  const double adt = (MODE == 0) ? 0.0 : alpha * sc->dt;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    if (!is_interior(g, c)) {
      if (MODE == 0) {
#pragma unroll
        for (int q = 0; q < 5; ++q) out[q * N + n] = (TO)0;
      } else if (MODE == 1) {
#pragma unroll
        for (int q = 0; q < 5; ++q) out[q * N + n] = (TO)Q0[q * N + n];
      }
      continue;
    }
    const long long m0 = step(g, n, c, 0, -1);
    const long long m1 = step(g, n, c, 1, -1);
    const long long m2 = step(g, n, c, 2, -1);
    // J once per node, halved: k_flux3 writes 2x the interface fluxes (jh
    // holds the same quotient, taken at set-up)
    const double Jn = (MODE == 0) ? 0.0 : (jh ? jh[n] : 0.5 / (double)M[9 * N + n]);
    const double a = (MODE == 0) ? 0.0 : (dtl ? alpha * dtl[n] : adt);
    const double aJ = a * Jn;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const R r = ((F0[q * N + n] - F0[q * N + m0]) + (F1[q * N + n] - F1[q * N + m1])) +
                  (F2[q * N + n] - F2[q * N + m2]);
      if (MODE == 0) {
        out[q * N + n] = (TO)(R(0.5) * r);
      } else {
        out[q * N + n] = (TO)(Q0[q * N + n] - aJ * (double)r);
      }
    }
  }
}

}  // namespace lesjet
