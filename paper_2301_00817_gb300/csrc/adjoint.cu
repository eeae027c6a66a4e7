// adjoint.cu -- discrete adjoint (vector-Jacobian products) of the FP64 time
// step, and the tangent (Jacobian-vector product) of the residual used to
// check it.
//
// Residual adjoint: for every interface I = (a, b) the flux F_I enters RHS_a
// with + and RHS_b with -, so its cotangent is lamR_a - lamR_b.  k_adj_flux3
// recomputes what it needs of the interface's forward intermediates and runs
// its dissipation and viscous flux in reverse into a record of that
// interface (what it owes the nodes it read); k_adj_sensor_terms gathers the
// sensors' cotangents; k_adj_node then sums, per node and in a fixed order,
// the records of the interfaces that read it, adds the centred flux's part
// (a node quantity: the cotangents of a node's two interfaces telescope) and
// reverses the node quantities (radii, primitive recovery) into cotangents of
// Q.  No atomics: the result is bitwise reproducible.
//
// Non-differentiable points follow the forward kernels' branch choices:
// |x| has derivative -1 for x < 0 and +1 otherwise, max(a, b) passes the
// cotangent to the operand the comparison selected.  (The boundary formulas
// select by a Mach number that they round in their own way: within an ulp or two
// of 1, 0 or -1 they may differentiate the branch beside the forward's.)
//
// Step adjoint (Eq. localdt with a fixed time step): with stage states S_l,
// Q^(l) = Q^(0) - alpha_l dt J RHS(Q^(l-1)) on interior nodes and Q^(l) =
// Q^(0) on boundary nodes, the reverse sweep accumulates lamQ0 += lamS_l and
// lamS_{l-1} = RHS^T(-alpha_l dt J lamS_l); the frozen viscosity mu(T(Q^n))
// collects its cotangent over the five stages and is reversed once.  The
// boundary conditions are reversed surface-only: the inner ring is linear,
// far-field and exit formulas use local 5x5 Jacobians from dual numbers, and
// the entrance plane turns its cotangent into the forcing-amplitude gradient.
#include <cuda_runtime.h>

#include "dual.cuh"
#include "lesjet_dev.cuh"
#include "lesjet_host.h"
#include "stage64_kernels.cuh"

namespace lesjet {

// Per-interface record (each [N] doubles, indexed by the interface's node a,
// one record array per direction): the cotangents it owes the nodes it read.
// The conserved state's are products that k_adj_node forms: the dissipation
// owes W_a d1 l, W_b -d1 l, W_{b+1} d3 l and W_{a-1} -d3 l, with l = (lamR_a -
// lamR_b)/2, so the two coefficients and l are kept.
enum {
  RUA = 0,    // u, v, w at a (3), then at b
  RUB = 3,
  RT = 6,     // T at b; minus it at a
  RG1 = 7,    // tangential difference cotangents (T1, then T2): +g at a+t and
  RG2 = 11,   //   b+t, -g at a-t and b-t, for u, v, w, T (4 each)
  RNUA = 15,  // sensor of direction D at a, at b
  RNUB = 16,
  RLB = 17,   // lbar (a and b each)
  RMU = 18,   // mu_eff and kappa_eff (a and b each)
  RKA = 19,
  RD1 = 20,   // d1 and d3
  RD3 = 21,
  RL = 22,    // l (5)
  NREC = kAdjRecords
};

// face-shifted centre triple of the pressure sensor of node x along D
template <int D>
__device__ __forceinline__ void sensor_triple(const Grid& g, long long x, int cx, long long& xm,
                                              long long& xc, long long& xp) {
  const long long s = g.stride[D];
  const int nd = g.n[D];
  xc = x;
  int cc = cx;
  if (!g.per[D]) {
    if (cx == 0) {
      xc = x + s;
      cc = 1;
    } else if (cx == nd - 1) {
      xc = x - s;
      cc = nd - 2;
    }
  }
  xp = (cc == nd - 1) ? xc - (long long)(nd - 1) * s : xc + s;
  xm = (cc == 0) ? xc + (long long)(nd - 1) * s : xc - s;
}

__device__ __forceinline__ void sensor_triple_at(const Grid& g, int D, long long x, int cx,
                                                 long long& xm, long long& xc, long long& xp) {
  if (D == 0) sensor_triple<0>(g, x, cx, xm, xc, xp);
  else if (D == 1) sensor_triple<1>(g, x, cx, xm, xc, xp);
  else sensor_triple<2>(g, x, cx, xm, xc, xp);
}

__device__ __forceinline__ double sgn_abs(double x) { return x < 0.0 ? -1.0 : 1.0; }

// ------------------------------------------------------------- interface
struct AdjIO {
  FluxIO<double, double, double> f;  // the stage input's state, metrics, node quantities, viscosity
  const double* lamR;                // [5][N], 0 on the open faces
  double* rec;                       // [3][NREC][N]
};

// Reverse of flux_iface for the cotangent l of the doubled flux (half the
// flux's own), without the centred part: the dissipation and the viscous
// flux, in flux_iface's terms and scaling.
template <int D>
__device__ __forceinline__ void adj_iface(const Consts<double>& K, const FluxNode<double>& a,
                                          const FluxNode<double>& b, const double Wm[5],
                                          const double Wp[5], double nua, double nub,
                                          const double l[5], double out[NREC]) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  // ---- dissipation: -d1 D1 + d3 E, d1 = lJ (eps2 + 3 eps4), d3 = lJ eps4
  const double k2h = 0.5 * K.k2, k4h = 0.5 * K.k4;
  const double nu = dev_max(nua, nub);
  // dev_max(nua, nub) = nua > nub ? nua : nub, and max(0, x) keeps x for x >= 0
  const bool pick_b = !(nua > nub);
  const double eps2 = k2h * nu, e4 = fma(-k2h, nu, k4h);
  const bool e4on = !(0.0 > e4);
  const double eps4 = e4on ? e4 : 0.0;
  const double sJ = a.J + b.J, lJ = (a.lb + b.lb) * sJ, e23 = eps2 + 3.0 * eps4;
  double ld1 = 0.0, ld3 = 0.0;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    ld1 = fma(-l[q], b.W[q] - a.W[q], ld1);
    ld3 = fma(l[q], Wp[q] - Wm[q], ld3);
  }
  out[RD1] = lJ * e23;
  out[RD3] = lJ * eps4;
  out[RLB] = sJ * (ld1 * e23 + ld3 * eps4);
  const double leps4 = 3.0 * ld1 + ld3;
  const double lnu = (k2h * lJ) * (e4on ? ld1 - leps4 : ld1);
  out[RNUA] = pick_b ? 0.0 : lnu;
  out[RNUB] = pick_b ? lnu : 0.0;

  // ---- viscous flux, forward
  const double dn[4] = {b.u - a.u, b.v - a.v, b.w - a.w, b.T - a.T};
  double s1[4], s2[4], mh[9];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    s1[q] = a.t1[q] + b.t1[q];
    s2[q] = a.t2[q] + b.t2[q];
  }
#pragma unroll
  for (int t = 0; t < 9; ++t) mh[t] = a.m[t] + b.m[t];
  const double* m = mh + 3 * D;
  const double* m1 = mh + 3 * T1;
  const double* m2 = mh + 3 * T2;
  const double gD = 4.0 * dot3(m[0], m[1], m[2], m[0], m[1], m[2]);
  const double g1 = dot3(m[0], m[1], m[2], m1[0], m1[1], m1[2]);
  const double g2 = dot3(m[0], m[1], m[2], m2[0], m2[1], m2[2]);
  const double cD = 4.0 * dot3(m[0], m[1], m[2], dn[0], dn[1], dn[2]);
  const double c1 = dot3(m[0], m[1], m[2], s1[0], s1[1], s1[2]);
  const double c2 = dot3(m[0], m[1], m[2], s2[0], s2[1], s2[2]);
  double div = cD;
#pragma unroll
  for (int i = 0; i < 3; ++i) div = fma(m2[i], s2[i], fma(m1[i], s1[i], div));
  const double eD = fma(-2.0 / 3.0, div, cD);
  double sv[3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
    sv[i] = fma(m2[i], c2, fma(m1[i], c1, fma(m[i], eD, dot3(gD, g1, g2, dn[i], s1[i], s2[i]))));
  const double aT = dot3(gD, g1, g2, dn[3], s1[3], s2[3]);
  const double sJ32 = sJ * (1.0 / 32.0);
  const double cm = sJ32 * (a.mu + b.mu), ck = sJ32 * (a.ka + b.ka);

  // ---- reverse: F_i -= cm sv_i, F_4 -= cm/2 (u_a + u_b) . sv + ck aT
  const double h4 = 0.5 * l[4];
  const double rr[3] = {fma(h4, a.u + b.u, l[1]), fma(h4, a.v + b.v, l[2]), fma(h4, a.w + b.w, l[3])};
  out[RMU] = -sJ32 * dot3(rr[0], rr[1], rr[2], sv[0], sv[1], sv[2]);
  out[RKA] = -sJ32 * (l[4] * aT);
  const double kf = -cm * h4;  // times sv: the interface velocity's
  const double ls[3] = {-cm * rr[0], -cm * rr[1], -cm * rr[2]};  // sv's
  const double lT = -ck * l[4];                                  // aT's
  // sv_i = gD dn_i + g1 s1_i + g2 s2_i + m_i eD + m1_i c1 + m2_i c2
  const double leD = dot3(ls[0], ls[1], ls[2], m[0], m[1], m[2]);
  const double lc1 = dot3(ls[0], ls[1], ls[2], m1[0], m1[1], m1[2]);
  const double lc2 = dot3(ls[0], ls[1], ls[2], m2[0], m2[1], m2[2]);
  // eD = cD - 2/3 div and div = cD + ..., cD = 4 m . dn
  const double l43 = (4.0 / 3.0) * leD, l23 = (-2.0 / 3.0) * leD;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double ldn = fma(m[i], l43, gD * ls[i]);
    out[RUA + i] = fma(kf, sv[i], -ldn);
    out[RUB + i] = fma(kf, sv[i], ldn);
    out[RG1 + i] = fma(m1[i], l23, fma(m[i], lc1, g1 * ls[i]));
    out[RG2 + i] = fma(m2[i], l23, fma(m[i], lc2, g2 * ls[i]));
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) out[RL + q] = l[q];
  out[RT] = gD * lT;
  out[RG1 + 3] = g1 * lT;
  out[RG2 + 3] = g2 * lT;
}

template <int D>
__device__ __forceinline__ void adj_put(const AdjIO& io, long long N, long long n,
                                        const double out[NREC]) {
  double* R = io.rec + (long long)D * NREC * N + n;
#pragma unroll
  for (int r = 0; r < NREC; ++r) R[r * N] = out[r];
}

template <int D>
__device__ __forceinline__ void adj_empty(const AdjIO& io, long long N, long long n) {
  double* R = io.rec + (long long)D * NREC * N + n;
#pragma unroll 1
  for (int r = 0; r < NREC; ++r) R[r * N] = 0.0;
}

// Tangential differences only (the centred flux is reversed per node).
template <int D>
__device__ __forceinline__ void adj_shared(const Grid& g, const double* node, long long n,
                                           const int c[3], FluxNode<double>& x) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  const long long N = g.N;
  const long long p1 = step(g, n, c, T1, 1), m1 = step(g, n, c, T1, -1);
  const long long p2 = step(g, n, c, T2, 1), m2 = step(g, n, c, T2, -1);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double* phi = node + (q == 3 ? 4 : q) * N;
    x.t1[q] = phi[p1] - phi[m1];
    x.t2[q] = phi[p2] - phi[m2];
  }
}

// Records of the interfaces along xi or eta: chunks of len interfaces per
// thread, as flux_chain walks them.  An interface without a cotangent (a
// window's cotangent spreads from one ring) gets an empty record.
template <int D>
__device__ __forceinline__ void adj_chain(const Grid& g, const Consts<double>& K, const AdjIO& io,
                                          long long id, int len) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  const long long N = g.N;
  const int nd = g.n[D];  // entries of a line (the last one empty on an open line)
  const int nch = (nd + len - 1) / len;
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
  const int end = c[D] + len < nd ? c[D] + len : nd;
  long long na = idx3(g, c[0], c[1], c[2]);
  if ((!g.per[T1] && (c[T1] == 0 || c[T1] == g.n[T1] - 1)) ||
      (!g.per[T2] && (c[T2] == 0 || c[T2] == g.n[T2] - 1))) {
    for (int x = c[D]; x < end; ++x, na += g.stride[D]) adj_empty<D>(io, N, na);
    return;
  }
  FluxNode<double> a, b;
  double Wm[5], pm = 0.0, la[5];
  const long long nm = step(g, na, c, D, -1);
  bool has_m = nm >= 0;
  if (has_m) flux_W(io.f, N, nm, Wm, pm);
  flux_W(io.f, N, na, a.W, a.p);
  flux_load<D>(io.f, N, false, na, a);
  adj_shared<D>(g, io.f.node, na, c, a);
#pragma unroll
  for (int q = 0; q < 5; ++q) la[q] = io.lamR[q * N + na];
  long long nb = step(g, na, c, D, 1);
  double nua = 0.0;
  if (nb >= 0) {
    flux_W(io.f, N, nb, b.W, b.p);
    if (has_m) nua = sensor3(pm, a.p, b.p);
  }
  for (int x = c[D]; x < end; ++x) {
    if (nb < 0) {  // past the last interface of an open line
      adj_empty<D>(io, N, na);
      return;
    }
    c[D] = x;
    const long long np = step(g, na, c, D, 2);
    const bool has_p = np >= 0;
    double Wp[5], pp = 0.0, l[5], lb[5];
    if (has_p) flux_W(io.f, N, np, Wp, pp);
    flux_load<D>(io.f, N, false, nb, b);
    adj_shared<D>(g, io.f.node, nb, c, b);
    double nub = nua;
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
    bool any = false;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      lb[q] = io.lamR[q * N + nb];
      l[q] = 0.5 * (la[q] - lb[q]);
      any = any || l[q] != 0.0;
      la[q] = lb[q];
    }
    if (any) {
      double out[NREC];
      adj_iface<D>(K, a, b, Wm, Wp, nua, nub, l, out);
      adj_put<D>(io, N, na, out);
    } else {
      adj_empty<D>(io, N, na);
    }
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

// Records of the zeta interfaces, one per thread; a block's run of nodes
// shares their tangential differences and sensors, as flux_zeta.
__device__ __forceinline__ void adj_zeta(const Grid& g, const Consts<double>& K, const AdjIO& io,
                                         long long n0, double (*sh)[kFluxThreads]) {
  const long long N = g.N, n = n0 + threadIdx.x;
  const double* P = io.f.node + 3 * N;
  int c[3] = {0, 0, 0};
  bool in = n < N;
  if (in) {
    decompose(g, n, c);
    in = (g.per[0] || (c[0] > 0 && c[0] < g.n[0] - 1)) &&
         (g.per[1] || (c[1] > 0 && c[1] < g.n[1] - 1));
    if (!in) adj_empty<2>(io, N, n);
  }
  FluxNode<double> a, b;
  double nua = 0.0;
  if (in) {
    flux_W(io.f, N, n, a.W, a.p);
    flux_load<2>(io.f, N, false, n, a);
    adj_shared<2>(g, io.f.node, n, c, a);
    nua = sensor<2>(g, P, n, c[2]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sh[q][threadIdx.x] = a.t1[q];
      sh[4 + q][threadIdx.x] = a.t2[q];
    }
    sh[8][threadIdx.x] = nua;
  }
  __syncthreads();
  if (!in) return;
  const long long nb = step(g, n, c, 2, 1);
  double l[5];
  bool any = false;
  if (nb >= 0) {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      l[q] = 0.5 * (io.lamR[q * N + n] - io.lamR[q * N + nb]);
      any = any || l[q] != 0.0;
    }
  }
  if (!any) {
    adj_empty<2>(io, N, n);
    return;
  }
  flux_W(io.f, N, nb, b.W, b.p);
  flux_load<2>(io.f, N, false, nb, b);
  double nub;
  if (nb >= n0 && nb < n0 + kFluxThreads) {
    const int s = (int)(nb - n0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      b.t1[q] = sh[q][s];
      b.t2[q] = sh[4 + q][s];
    }
    nub = sh[8][s];
  } else {
    adj_shared<2>(g, io.f.node, nb, c, b);
    nub = sensor<2>(g, P, nb, coord_step(g, c, 2, 1));
  }
  double Wm[5], Wp[5], unused;
  const long long nm = step(g, n, c, 2, -1), np = step(g, n, c, 2, 2);
  flux_W(io.f, N, nm >= 0 ? nm : nb, Wm, unused);
  flux_W(io.f, N, np >= 0 ? np : n, Wp, unused);
  double out[NREC];
  adj_iface<2>(K, a, b, Wm, Wp, nua, nub, l, out);
  adj_put<2>(io, N, n, out);
}

// The three directions' records in one launch, split as k_flux3's.  Bound by
// the FP64 pipe like the forward kernel: 206 operations per interface with
// chunks of 16 (209 with 4, 222 without; 429 when the gradient tensor was formed,
// the stress reversed term by term and the centred flux reversed twice per node).
__global__ void __launch_bounds__(kFluxThreads, 2)
    k_adj_flux3(Grid g, Consts<double> K, AdjIO io, unsigned b0, unsigned b1, int len) {
  begin_dependent();
  __shared__ double sh[9][kFluxThreads];
  const unsigned b = blockIdx.x;
  if (b < b0)
    adj_chain<0>(g, K, io, (long long)b * kFluxThreads + threadIdx.x, len);
  else if (b < b0 + b1)
    adj_chain<1>(g, K, io, (long long)(b - b0) * kFluxThreads + threadIdx.x, len);
  else
    adj_zeta(g, K, io, (long long)(b - b0 - b1) * kFluxThreads, sh);
}

// Sensor cotangents to the pressures of the (face-shifted) centre triple:
// per node x and direction d the two terms it owes (ls + lden to its outer
// pair, -2 ls + 2 lden to its centre) into ST[2 d], ST[2 d + 1]; k_adj_node
// gathers, in a fixed order, the terms of the nodes whose triple holds a
// node (x within two nodes along d).
__global__ void __launch_bounds__(256) k_adj_sensor_terms(Grid g, const double* __restrict__ node,
                                                          const double* __restrict__ rec,
                                                          double* __restrict__ ST) {
  begin_dependent();
  const long long N = g.N;
  const double* P = node + 3 * N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double* R = rec + (long long)d * NREC * N;
      const long long mB = step(g, n, c, d, -1);
      const double ln = R[RNUA * N + n] + (mB >= 0 ? R[RNUB * N + mB] : 0.0);
      double outer = 0.0, centre = 0.0;
      if (ln != 0.0) {
        long long xm, xc, xp;
        sensor_triple_at(g, d, n, c[d], xm, xc, xp);
        // nu = |s| / den, rounded as sensor3 does (the sign of s decides the
        // branch where the pressure is uniform to rounding)
        const double p0 = P[xc];
        const double s = (P[xp] - p0) - (p0 - P[xm]), den = fma(4.0, p0, s);
        const double iden = 1.0 / den;
        const double ls = ln * sgn_abs(s) * iden;
        const double lden = -ln * fabs(s) * iden * iden;
        outer = ls + lden;
        centre = -2.0 * ls + 2.0 * lden;
      }
      ST[(2 * d) * N + n] = outer;
      ST[(2 * d + 1) * N + n] = centre;
    }
  }
}

// Per node, in a fixed order: what the interface records owe it, the centred
// flux's part, the sensors' part, then the node quantities back to Q: radii
// lbar(lambda_d), lambda_d = |m_d.u| + sqrt(T)|grad d|, u = Q1/rho, p =
// (g-1)(Q4 - rho|u|^2/2), T = g p/rho.  mu/kappa cotangents are added to
// lamMK.  |grad d| comes from gn ([3][N], set-up).
// A node reads about 240 values (its interfaces' records within two nodes
// along each direction), few of them twice by one thread, and does 373 FP64
// operations, whose pipe bounds it; gathering straight into
// the node's reverse saves the 18 accumulator fields of a pass of their own.
__global__ void __launch_bounds__(128, 3)
    k_adj_node(Grid g, Consts<double> K, const double* __restrict__ Q,
               const double* __restrict__ M, const double* __restrict__ gn,
               const double* __restrict__ node, const double* __restrict__ rec,
               const double* __restrict__ ST,
               double* __restrict__ lamQ, double* __restrict__ lamMK) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    const double u = node[n], v = node[N + n], w = node[2 * N + n], p = node[3 * N + n],
                 T = node[4 * N + n];
    const double Jv = M[9 * N + n];
    double lW[5] = {0.0, 0.0, 0.0, 0.0, 0.0};   // the cotangents of W
    double lv[4] = {0.0, 0.0, 0.0, 0.0};        // u, v, w, T
    double lp = 0.0, lmu = 0.0, lka = 0.0, llb[3], th[3];
#pragma unroll
    for (int D = 0; D < 3; ++D) {
      const double* R = rec + (long long)D * NREC * N;
      const long long m1 = step(g, n, c, D, -1), p1 = step(g, n, c, D, 1);
      const long long m2 = step(g, n, c, D, -2), p2 = step(g, n, c, D, 2);
      // interfaces (m2, m1), (m1, n), (n, p1), (p1, p2), by their node a
      double kB = 0.0, kA = 0.0, kP = 0.0, kM = 0.0;
      if (m1 >= 0) kB = R[RD1 * N + m1];
      if (p1 >= 0) kA = R[RD1 * N + n];
      if (m2 >= 0) kP = R[RD3 * N + m2];
      else if (m1 >= 0) kB += R[RD3 * N + m1];  // its W_{a-1} was W_b, this node
      if (p2 >= 0) kM = R[RD3 * N + p1];
      else if (p1 >= 0) kA += R[RD3 * N + n];   // its W_{b+1} was W_a, this node
      const double mx = M[(3 * D) * N + n], my = M[(3 * D + 1) * N + n], mz = M[(3 * D + 2) * N + n];
      th[D] = dot3(mx, my, mz, u, v, w);
      const double Jt = Jv * th[D];
      double lJt = 0.0, lF[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const double* L = R + (RL + q) * N;
        const double eA = L[n], eB = m1 >= 0 ? L[m1] : 0.0;
        const double eP = m2 >= 0 ? L[m2] : 0.0, eM = p1 >= 0 ? L[p1] : 0.0;
        lW[q] = fma(kP, eP, fma(Jt - kB, eB, fma(Jt + kA, eA, fma(-kM, eM, lW[q]))));
        lF[q] = eB + eA;  // the cotangent of the node's flux along D
        const double W = Q[q * N + n] + (q == 4 ? p : 0.0);
        lJt = fma(W, lF[q], lJt);
      }
      // node flux: W Jt (+ Jp m in the momentum), Jt = J^-1 m . u, Jp = J^-1 p
      const double lth = Jv * lJt;
      lp = fma(Jv, dot3(mx, my, mz, lF[1], lF[2], lF[3]), lp);
      lv[0] = fma(mx, lth, lv[0]);
      lv[1] = fma(my, lth, lv[1]);
      lv[2] = fma(mz, lth, lv[2]);
      // as a, as b
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        lv[k] += R[(RUA + k) * N + n];
        if (m1 >= 0) lv[k] += R[(RUB + k) * N + m1];
      }
      lv[3] -= R[RT * N + n];
      if (m1 >= 0) lv[3] += R[RT * N + m1];
      llb[D] = R[RLB * N + n];
      lmu += R[RMU * N + n];
      lka += R[RKA * N + n];
      if (m1 >= 0) {
        llb[D] += R[RLB * N + m1];
        lmu += R[RMU * N + m1];
        lka += R[RKA * N + m1];
      }
      // as a tangential neighbour (a + t, b + t, a - t, b - t) of the
      // interfaces at n - e_t, n - e_t - e_D, n + e_t, n + e_t - e_D
#pragma unroll
      for (int s = 1; s <= 2; ++s) {
        const int t = (D + s) % 3;
        const double* G = R + (s == 1 ? RG1 : RG2) * N;
        const long long tm = step(g, n, c, t, -1), tp = step(g, n, c, t, 1);
        const long long dB = m1 - n;  // to the interface's node a when n + t is its b
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (tm >= 0) lv[k] += G[k * N + tm];
          if (tp >= 0) lv[k] -= G[k * N + tp];
          if (m1 >= 0) {
            if (tm >= 0) lv[k] += G[k * N + tm + dB];
            if (tp >= 0) lv[k] -= G[k * N + tp + dB];
          }
        }
      }
      // the sensors along D whose triple holds this node
#pragma unroll
      for (int off = -2; off <= 2; ++off) {
        const long long x = off == 0 ? n : (off == -2 ? m2 : (off == -1 ? m1 : (off == 1 ? p1 : p2)));
        if (x < 0) continue;
        const int cx = off == 0 ? c[D] : coord_step(g, c, D, off);
        if ((off == -2 || off == 2) && (g.per[D] || (cx != 0 && cx != g.n[D] - 1))) continue;
        long long xm, xc, xp;
        sensor_triple_at(g, D, x, cx, xm, xc, xp);
        if (xp == n) lp += ST[(2 * D) * N + x];
        if (xc == n) lp += ST[(2 * D + 1) * N + x];
        if (xm == n) lp += ST[(2 * D) * N + x];
      }
    }
    lp += lW[4];  // W4 = Q4 + p
    double lT = lv[3];
    // lbar -> lambda
    if (llb[0] != 0.0 || llb[1] != 0.0 || llb[2] != 0.0) {
      const double ra = rsqrt(T), a = T * ra;
      double l[3], gm[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        gm[d] = gn[d * N + n];
        l[d] = fma(a, gm[d], fabs(th[d]));
      }
      // d sqrt(l_a l_b)/d l_a = l_b/(2 sqrt(l_a l_b)): one reciprocal root per pair
      const double h01 = 0.5 * (llb[0] + llb[1]) * rsqrt(l[0] * l[1]);
      const double h02 = 0.5 * (llb[0] + llb[2]) * rsqrt(l[0] * l[2]);
      const double h12 = 0.5 * (llb[1] + llb[2]) * rsqrt(l[1] * l[2]);
      double ll[3];
      ll[0] = llb[0] + h01 * l[1] + h02 * l[2];
      ll[1] = llb[1] + h01 * l[0] + h12 * l[2];
      ll[2] = llb[2] + h02 * l[0] + h12 * l[1];
      double la = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double lth = ll[d] * sgn_abs(th[d]);
        lv[0] = fma(M[(3 * d) * N + n], lth, lv[0]);
        lv[1] = fma(M[(3 * d + 1) * N + n], lth, lv[1]);
        lv[2] = fma(M[(3 * d + 2) * N + n], lth, lv[2]);
        la = fma(ll[d], gm[d], la);
      }
      lT = fma(0.5 * la, ra, lT);
    }
    const double rho = Q[n], ir = 1.0 / rho;
    // T = gamma p / rho
    const double gT = K.gamma * ir * lT;
    lp += gT;
    double lrho = -(p * ir) * gT;
    // p = (gamma-1)(Q4 - rho |u|^2 / 2)
    const double lQ4 = K.gm1 * lp;
    lrho = fma(-0.5 * lQ4, dot3(u, v, w, u, v, w), lrho);
    const double rl = rho * lQ4;
    const double lu = fma(-rl, u, lv[0]), lvv = fma(-rl, v, lv[1]), lw = fma(-rl, w, lv[2]);
    // u = Q1 / rho
    lrho = fma(-ir, dot3(u, v, w, lu, lvv, lw), lrho);
    lamQ[n] = lW[0] + lrho;
    lamQ[N + n] = fma(ir, lu, lW[1]);
    lamQ[2 * N + n] = fma(ir, lvv, lW[2]);
    lamQ[3 * N + n] = fma(ir, lw, lW[3]);
    lamQ[4 * N + n] = lW[4] + lQ4;
    if (lamMK) {
      lamMK[n] += lmu;
      lamMK[N + n] += lka;
    }
  }
}

// Sutherland viscosity (no SGS model): mu = s T^1.5 (1+S)/(T+S), kappa =
// mu/((g-1)Pr), T = g p/rho of Q^n; adds the Q cotangent to lamQ.
__global__ void k_adj_mu(Grid g, Consts<double> K, const double* __restrict__ Q,
                         const double* __restrict__ lamMK, double* __restrict__ lamQ) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const double lmu = lamMK[n] + lamMK[N + n] * K.inv_gm1_pr;
    if (lmu == 0.0) continue;
    const double rho = Q[n], ir = 1.0 / rho;
    const double u = Q[N + n] * ir, v = Q[2 * N + n] * ir, w = Q[3 * N + n] * ir;
    const double p = K.gm1 * (Q[4 * N + n] - 0.5 * rho * (u * u + v * v + w * w));
    const double T = K.gamma * p * ir;
    const double S = K.S_suth;
    const double sq = sqrt(T);
    // d/dT [T^1.5 / (T+S)] = (1.5 sqrt(T)(T+S) - T^1.5)/(T+S)^2
    const double dmu = K.mu_scale * (1.0 + S) * (1.5 * sq * (T + S) - T * sq) / ((T + S) * (T + S));
    const double lT = dmu * lmu;
    const double lp = K.gamma * ir * lT;
    double lrho = -K.gamma * p * ir * ir * lT;
    lrho += -0.5 * K.gm1 * (u * u + v * v + w * w) * lp;
    const double lu = -K.gm1 * rho * u * lp, lv = -K.gm1 * rho * v * lp, lw = -K.gm1 * rho * w * lp;
    lrho += -ir * (u * lu + v * lv + w * lw);
    lamQ[n] += lrho;
    lamQ[N + n] += ir * lu;
    lamQ[2 * N + n] += ir * lv;
    lamQ[3 * N + n] += ir * lw;
    lamQ[4 * N + n] += K.gm1 * lp;
  }
}

// ------------------------------------------------------------ RK helpers
// lamR = -alpha dt J lamS on interior nodes, 0 on boundary nodes; lamQ0 += lamS
// (jh: J/2 of set-up)
__global__ void k_adj_stage_prep(Grid g, const double* __restrict__ jh, double coef,
                                 const double* __restrict__ lamS, double* __restrict__ lamR,
                                 double* __restrict__ lamQ0) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    const bool in = is_interior(g, c);
    const double cJ = in ? -2.0 * coef * jh[n] : 0.0;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const double ls = lamS[q * N + n];
      lamQ0[q * N + n] += ls;
      lamR[q * N + n] = in ? cJ * ls : 0.0;
    }
  }
}

// out = lam, 0 on the faces of non-periodic directions (where the residual is 0)
__global__ void k_mask_faces(Grid g, const double* __restrict__ lam, double* __restrict__ out) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    bool in = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) in = in && (g.per[d] || (c[d] > 0 && c[d] < g.n[d] - 1));
#pragma unroll
    for (int q = 0; q < 5; ++q) out[q * N + n] = in ? lam[q * N + n] : 0.0;
  }
}

__global__ void k_axpy(long long count, double a, const double* __restrict__ x, double* __restrict__ y) {
  begin_dependent();
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < count;
       n += (long long)gridDim.x * blockDim.x)
    y[n] += a * x[n];
}

// ------------------------------------------------------- boundary reverse
// x^(2/(gamma-1)), by multiplication where the exponent is an integer up to 8,
// as the forward boundary conditions take it: two powers of dual numbers were
// the longest chain of the far-field kernel (adjoint window on 64 x 40 x 48
// 28.67 -> 28.49 ms together with J/2 of set-up in k_adj_stage_prep).
template <typename T>
__device__ T pow_entropy_of(const T& x, double e) {
  const double n = rint(e);
  if (fabs(e - n) < 1e-12 && n >= 1.0 && n <= 8.0) {
    T r = x;
    for (int i = 1; i < (int)n; ++i) r = r * x;
    return r;
  }
  return pow(x, e);
}

template <typename T>
__device__ void farfield_formula(const T qe[5], double nx, double ny, double nz, double gamma,
                                 T qf[5]) {
  const double gm1 = gamma - 1.0;
  const T rho = qe[0];
  const T u = qe[1] / rho, v = qe[2] / rho, w = qe[3] / rho;
  const T p = gm1 * (qe[4] - 0.5 * rho * (u * u + v * v + w * w));
  const T ae = sqrt(gamma * p / rho);
  const T qne = u * nx + v * ny + w * nz;
  const T Rp = qne + 2.0 * ae / gm1;
  const double Rm = 0.0 - 2.0 * 1.0 / gm1;
  const T qnf = 0.5 * (Rp + Rm);
  const T af = 0.25 * gm1 * (Rp - Rm);
  const T Mn = qne / ae;
  T rf, uf, vf, wf, pf;
  if (Mn >= 1.0) {
    for (int q = 0; q < 5; ++q) qf[q] = qe[q];
    return;
  } else if (Mn >= 0.0) {
    const T dq = qnf - qne;
    rf = rho * pow_entropy_of(af / ae, 2.0 / gm1);
    uf = u + dq * nx;
    vf = v + dq * ny;
    wf = w + dq * nz;
    pf = rf * af * af / gamma;
  } else if (Mn > -1.0) {
    rf = pow_entropy_of(af, 2.0 / gm1);
    uf = qnf * nx;
    vf = qnf * ny;
    wf = qnf * nz;
    pf = rf * af * af / gamma;
  } else {
    rf = T(1.0);
    uf = T(0.0);
    vf = T(0.0);
    wf = T(0.0);
    pf = T(1.0 / gamma);
  }
  qf[0] = rf;
  qf[1] = rf * uf;
  qf[2] = rf * vf;
  qf[3] = rf * wf;
  qf[4] = pf / gm1 + 0.5 * rf * (uf * uf + vf * vf + wf * wf);
}

template <typename T>
__device__ void exit_formula(const T qe[5], double ex, double ey, double ez, double gamma, T qo[5]) {
  const double gm1 = gamma - 1.0;
  const double inv = 1.0 / ::sqrt(ex * ex + ey * ey + ez * ez);
  const T rho = qe[0];
  const T u = qe[1] / rho, v = qe[2] / rho, w = qe[3] / rho;
  const T p = gm1 * (qe[4] - 0.5 * rho * (u * u + v * v + w * w));
  const T ae = sqrt(gamma * p / rho);
  const T qn = (u * ex + v * ey + w * ez) * inv;
  if (qn / ae >= 1.0) {
    for (int q = 0; q < 5; ++q) qo[q] = qe[q];
    return;
  }
  const T eint = p / (gm1 * rho);
  const T rf = (1.0 / gamma) / (gm1 * eint);
  qo[0] = rf;
  qo[1] = rf * u;
  qo[2] = rf * v;
  qo[3] = rf * w;
  qo[4] = rf * (eint + 0.5 * (u * u + v * v + w * w));
}

// Component i of J^T lam for a 5 -> 5 map evaluated by forward-mode dual
// numbers.
template <int KIND>
__device__ double local_vjp(int i, const double qe[5], double a0, double a1, double a2,
                            double gamma, const double lam[5]) {
  Dual x[5], y[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) x[q] = Dual(qe[q], q == i ? 1.0 : 0.0);
  if (KIND == 0)
    farfield_formula<Dual>(x, a0, a1, a2, gamma, y);
  else
    exit_formula<Dual>(x, a0, a1, a2, gamma, y);
  double s = 0.0;
#pragma unroll
  for (int q = 0; q < 5; ++q) s += y[q].d * lam[q];
  return s;
}

// lamS = lamNext on interior nodes, 0 on boundary nodes (their stage values
// are overwritten by the boundary conditions)
__global__ void k_adjbc_init(Grid g, const double* __restrict__ lamNext, double* __restrict__ lamS) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    const bool in = is_interior(g, c);
#pragma unroll
    for (int q = 0; q < 5; ++q) lamS[q * N + n] = in ? lamNext[q * N + n] : 0.0;
  }
}

// exit: the plane i = ni-1 copies / extrapolates the post-phase-1 column
// i = ni-2 (taken from Qnext).  Interior rows go straight into lamS; the two
// face rows (j = 0, nj-1) go to E for the ring / far-field reverse.  Block row
// y takes component y of every node: a node's five derivatives are
// independent, each a chain of a few hundred dependent FP64 operations, and
// a face has too few nodes to fill the SMs with all five in one thread
// (the far field's launch took 191 us whatever its size, most of it two pows).
__global__ void __launch_bounds__(64) k_adjbc_exit(Grid g, double gamma,
                                                   const double* __restrict__ M,
                                                   const double* __restrict__ Qnext,
                                                   const double* __restrict__ lamNext,
                                                   double* __restrict__ lamS,
                                                   double* __restrict__ E) {
  begin_dependent();
  const int ni = g.n[0], nj = g.n[1], nk = g.n[2], i5 = blockIdx.y;
  const long long plane = (long long)nj * nk, N = g.N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < plane;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e / nk);
    const long long nx_ = (long long)(ni - 1) * plane + e, ne = nx_ - plane;
    double qe[5], lam[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      qe[q] = Qnext[q * N + ne];
      lam[q] = lamNext[q * N + nx_];
    }
    const double out = local_vjp<1>(i5, qe, M[nx_], M[N + nx_], M[2 * N + nx_], gamma, lam);
    if (j == 0 || j == nj - 1)
      E[i5 * plane + e] = out;
    else
      lamS[i5 * N + ne] += out;
  }
}

// far field: node (i, nj-1, k) from (i, nj-2, k) of the stage-5 state
__global__ void __launch_bounds__(64) k_adjbc_farfield(Grid g, double gamma,
                                                       const double* __restrict__ M,
                                                       const double* __restrict__ S5,
                                                       const double* __restrict__ lamNext,
                                                       const double* __restrict__ E,
                                                       double* __restrict__ lamS) {
  begin_dependent();
  const int ni = g.n[0], nj = g.n[1], nk = g.n[2], i5 = blockIdx.y;
  const long long count = (long long)(ni - 2) * nk, N = g.N, plane = (long long)nj * nk;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = 1 + (int)(e / nk), k = (int)(e % nk);
    const long long nf = idx3(g, i, nj - 1, k), ne = idx3(g, i, nj - 2, k);
    const double ex = M[3 * N + nf], ey = M[4 * N + nf], ez = M[5 * N + nf];
    const double inv = 1.0 / sqrt(ex * ex + ey * ey + ez * ez);
    double qe[5], lam[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      qe[q] = S5[q * N + ne];
      lam[q] = lamNext[q * N + nf] + (i == ni - 2 ? E[q * plane + (long long)(nj - 1) * nk + k] : 0.0);
    }
    lamS[i5 * N + ne] += local_vjp<0>(i5, qe, ex * inv, ey * inv, ez * inv, gamma, lam);
  }
}

// inner ring: Q(i,0,k) = mean_k S5(i,1,k), one block per axial station
__global__ void k_adjbc_ring(Grid g, const double* __restrict__ lamNext, const double* __restrict__ E,
                             double* __restrict__ lamS) {
  begin_dependent();
  const int i = 1 + blockIdx.x;
  const int ni = g.n[0], nk = g.n[2];
  const long long N = g.N;
  __shared__ double red[5][32];
  double s[5] = {0, 0, 0, 0, 0};
  const long long base0 = idx3(g, i, 0, 0), base1 = idx3(g, i, 1, 0);
  for (int k = threadIdx.x; k < nk; k += blockDim.x)
    for (int q = 0; q < 5; ++q)
      s[q] += lamNext[q * N + base0 + k] + (i == ni - 2 ? E[q * (long long)g.n[1] * nk + k] : 0.0);
  for (int q = 0; q < 5; ++q)
    for (int off = 16; off > 0; off >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
  if ((threadIdx.x & 31) == 0)
    for (int q = 0; q < 5; ++q) red[q][threadIdx.x >> 5] = s[q];
  __syncthreads();
  if (threadIdx.x < 32) {
    for (int q = 0; q < 5; ++q) {
      double v = threadIdx.x < (blockDim.x >> 5) ? red[q][threadIdx.x] : 0.0;
      for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if (threadIdx.x == 0) red[q][0] = v / (double)nk;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nk; k += blockDim.x)
    for (int q = 0; q < 5; ++q) lamS[q * N + base1 + k] += red[q][0];
}

// entrance: Q = (1, u, 0, 0, p/(g-1) + u^2/2), u = profile + sum a_mf g(r)
// cos(m theta - 2 pi St_f Mj t): grad_mf += sum over the plane of
// (lam1 + u lam4) g(r) cos(...); one partial per block and mode.
struct AdjInflow {
  double Mj, r_jet, theta_m, width, t;
  double St[4], amp[16];
};

__global__ void __launch_bounds__(64) k_adjbc_inflow(Grid g, AdjInflow b,
                                                     const double* __restrict__ rth,
                                                     const double* __restrict__ lamNext,
                                                     double* __restrict__ partials) {
  begin_dependent();
  const long long plane = (long long)g.n[1] * g.n[2], N = g.N;
  const double two_pi = 6.283185307179586476925286766559;
  // cos(m theta - phi_f) = cos(m theta) cos(phi_f) + sin(m theta) sin(phi_f), as
  // the forward entrance forms it; lane f of the warp takes phase f mod 4
  double sf[4], cf[4];
  {
    const int f = threadIdx.x & 3;
    double s, c;
    sincos(two_pi * (f == 0 ? b.St[0] : (f == 1 ? b.St[1] : (f == 2 ? b.St[2] : b.St[3]))) * b.Mj * b.t,
           &s, &c);
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      sf[l] = __shfl_sync(0xffffffffu, s, l);
      cf[l] = __shfl_sync(0xffffffffu, c, l);
    }
  }
  double acc[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) acc[m] = 0.0;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < plane;
       n += (long long)gridDim.x * blockDim.x) {
    const double r = rth[n], th = rth[plane + n];
    double u = 0.5 * b.Mj * (1.0 + tanh((b.r_jet - r) / (2.0 * b.theta_m)));
    const double x = (r - b.r_jet) / b.width;
    const double gr = exp(-(x * x));
    double s1, c1;
    sincos(th, &s1, &c1);
    double cm[4] = {1.0, c1, 0.0, 0.0}, sm[4] = {0.0, s1, 0.0, 0.0};
#pragma unroll
    for (int m = 2; m < 4; ++m) {
      cm[m] = cm[m - 1] * c1 - sm[m - 1] * s1;
      sm[m] = sm[m - 1] * c1 + cm[m - 1] * s1;
    }
    double cs[16], f = 0.0;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      cs[m] = cm[m >> 2] * cf[m & 3] + sm[m >> 2] * sf[m & 3];
      f += b.amp[m] * cs[m];
    }
    u += gr * f;
    const double lu = gr * (lamNext[N + n] + u * lamNext[4 * N + n]);
#pragma unroll
    for (int m = 0; m < 16; ++m) acc[m] += lu * cs[m];
  }
  __shared__ double red[16][2];
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    double v = acc[m];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[m][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 16) partials[blockIdx.x * 16 + threadIdx.x] = red[threadIdx.x][0] + red[threadIdx.x][1];
}

// out[m] += sum of the block partials of item m = this block's, in a fixed
// order (a warp per item; lanes take the blocks in turn)
__global__ void k_sum_partials(const double* __restrict__ partials, int nb, int items,
                               double* __restrict__ out) {
  begin_dependent();
  const int m = blockIdx.x, lane = threadIdx.x;
  double s = 0.0;
  for (int b = lane; b < nb; b += 32) s += partials[b * items + m];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) out[m] += s;
}

// ------------------------------------------------------------ functional
// J_f contribution of one state: dt sum_{i,k} (p(i, j5, k) - 1/gamma)^2 dA,
// dA = J^-1 |grad eta| (eta-face area); and its Q cotangent.
template <typename TM>
__global__ void k_functional(Grid g, double gamma, int j5, double dt, const TM* __restrict__ M,
                             const double* __restrict__ Q, double* __restrict__ lam,
                             double* __restrict__ partials) {
  begin_dependent();
  const int ni = g.n[0], nk = g.n[2];
  const long long count = (long long)ni * nk, N = g.N;
  const double gm1 = gamma - 1.0;
  double acc = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / nk), k = (int)(e % nk);
    const long long n = idx3(g, i, j5, k);
    const double ex = (double)M[3 * N + n], ey = (double)M[4 * N + n], ez = (double)M[5 * N + n];
    const double dA = (double)M[9 * N + n] * sqrt(ex * ex + ey * ey + ez * ez);
    const double rho = Q[n], u = Q[N + n] / rho, v = Q[2 * N + n] / rho, w = Q[3 * N + n] / rho;
    const double p = gm1 * (Q[4 * N + n] - 0.5 * rho * (u * u + v * v + w * w));
    const double dp = p - 1.0 / gamma;
    acc += dt * dp * dp * dA;
    if (lam) {
      const double lp = 2.0 * dt * dp * dA;
      lam[n] += lp * gm1 * 0.5 * (u * u + v * v + w * w);
      lam[N + n] += -lp * gm1 * u;
      lam[2 * N + n] += -lp * gm1 * v;
      lam[3 * N + n] += -lp * gm1 * w;
      lam[4 * N + n] += lp * gm1;
    }
  }
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    partials[blockIdx.x] = s;
  }
}

__global__ void k_pack_dual(long long count, const double* __restrict__ v,
                            const double* __restrict__ d, Dual* __restrict__ out) {
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < count;
       n += (long long)gridDim.x * blockDim.x)
    out[n] = Dual(v[n], d ? d[n] : 0.0);
}

__global__ void k_unpack_dual(long long count, const Dual* __restrict__ in, double* __restrict__ v,
                              double* __restrict__ d) {
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < count;
       n += (long long)gridDim.x * blockDim.x) {
    if (v) v[n] = in[n].v;
    d[n] = in[n].d;
  }
}

// ------------------------------------------------------------- launchers
constexpr int kAdjBlocks = kRedBlocks;  // fixed reduction grid (deterministic sums)

static int nb_for(long long count) {
  long long b = (count + 255) / 256;
  const long long cap = 32LL * sm_count();
  if (b > cap) b = cap;
  return (int)(b < 1 ? 1 : b);
}

void launch_rhs_vjp(const Grid& g, const les_params& p, const double* Q, const double* M,
                    const double* gn, const double* node, const double* mk, const double* lamR,
                    double* acc, double* lamQ, double* lamMK, const Launch& L) {
  const Consts<double> K = make_consts<double>(p);
  // acc holds the sensor terms, then the three directions' records
  double* ST = acc;
  double* rec = acc + (size_t)kAdjSensorTerms * g.N;
  // chunk lengths as the forward's; a line has an entry for every node
  const FluxPlan f = flux_plan(g);
  auto blocks = [](long long t) { return (unsigned)((t + kFluxThreads - 1) / kFluxThreads); };
  auto chunks = [&](int d) { return (g.n[d] + f.len - 1) / f.len; };
  const unsigned b0 = blocks((long long)chunks(0) * g.n[1] * g.n[2]);
  const unsigned b1 = blocks((long long)g.n[0] * chunks(1) * g.n[2]);
  const AdjIO io{FluxIO<double, double, double>{Q, M, node, mk, nullptr}, lamR, rec};
  launch_dependent(k_adj_flux3, f.b2 + b0 + b1, kFluxThreads, 0, L, g, K, io, b0, b1, f.len);
  launch_dependent(k_adj_sensor_terms, nb_for(g.N), 256, 0, L, g, node, rec, ST);
  launch_dependent(k_adj_node, blocks_for(g.N, 128), 128, 0, L, g, K, Q, M, gn, node, rec, ST, lamQ,
                   lamMK);
  *L.counter += 3;
}

void launch_mask_faces(const Grid& g, const double* lam, double* out, const Launch& L) {
  launch_dependent(k_mask_faces, nb_for(g.N), 256, 0, L, g, lam, out);
  ++*L.counter;
}

void launch_rhs_jvp(const Grid& g, const les_params& p, const Dual* Q, const double* M,
                    const Dual* mk, Dual* node, Dual* flux, Dual* R, const Launch& L) {
  const Consts<Dual> K = make_consts<Dual>(p);
  const int nb = nb_for(g.N);
  launch_dependent(k_node<Dual, Dual, double, false>, nb, 256, 0, L, g, K, Q, M, nullptr, node,
                   nullptr, nullptr, nullptr, 0.0);
  const FluxPlan f = flux_plan(g);
  launch_dependent(k_flux3<Dual, Dual, double>, f.b2 + f.b0 + f.b1, kFluxThreads, 0, L, g, K,
                   FluxIO<Dual, Dual, double>{Q, M, node, mk, flux}, f.b0, f.b1, f.len);
  launch_dependent(k_update<Dual, double, Dual, 0>, nb, 256, 0, L, g, flux, nullptr, M, nullptr,
                   0.0, R, nullptr, nullptr);
  *L.counter += 3;
}

void launch_pack_dual(long long count, const double* v, const double* d, Dual* out, const Launch& L) {
  k_pack_dual<<<nb_for(count), 256, 0, L.s>>>(count, v, d, out);
  ++*L.counter;
}

void launch_unpack_dual(long long count, const Dual* in, double* v, double* d, const Launch& L) {
  k_unpack_dual<<<nb_for(count), 256, 0, L.s>>>(count, in, v, d);
  ++*L.counter;
}

void launch_mu_vjp(const Grid& g, const les_params& p, const double* Q, const double* lamMK,
                   double* lamQ, const Launch& L) {
  launch_dependent(k_adj_mu, nb_for(g.N), 256, 0, L, g, make_consts<double>(p), Q, lamMK, lamQ);
  ++*L.counter;
}

void launch_stage_prep(const Grid& g, const double* jh, double coef, const double* lamS,
                       double* lamR, double* lamQ0, const Launch& L) {
  launch_dependent(k_adj_stage_prep, nb_for(g.N), 256, 0, L, g, jh, coef, lamS, lamR, lamQ0);
  ++*L.counter;
}

void launch_axpy(long long count, double a, const double* x, double* y, const Launch& L) {
  launch_dependent(k_axpy, nb_for(count), 256, 0, L, count, a, x, y);
  ++*L.counter;
}

void launch_bc_vjp(const Grid& g, const les_params& p, const double* M, const double* rth,
                   const double* S5, const double* Qnext, const double* lamNext, double t_next,
                   double* lamS, double* E, double* partials, double* grad, const Launch& L) {
  const long long plane = (long long)g.n[1] * g.n[2];
  launch_dependent(k_adjbc_init, nb_for(g.N), 256, 0, L, g, lamNext, lamS);
  auto nb64 = [](long long count) {
    const long long b = (count + 63) / 64;
    return (unsigned)(b < kAdjBlocks ? b : kAdjBlocks);
  };
  launch_dependent(k_adjbc_exit, dim3(nb64(plane), 5), 64, 0, L, g, p.gamma, M, Qnext, lamNext,
                   lamS, E);
  launch_dependent(k_adjbc_farfield, dim3(nb64((long long)(g.n[0] - 2) * g.n[2]), 5), 64, 0, L, g,
                   p.gamma, M, S5, lamNext, E, lamS);
  launch_dependent(k_adjbc_ring, g.n[0] - 2, 256, 0, L, g, lamNext, E, lamS);
  AdjInflow in;
  in.Mj = p.Mj;
  in.r_jet = p.r_jet;
  in.theta_m = p.theta_m;
  in.width = p.force_width;
  in.t = t_next;
  for (int i = 0; i < 4; ++i) in.St[i] = p.St[i];
  for (int i = 0; i < 16; ++i) in.amp[i] = p.amp[i];
  const unsigned nbi = nb64(plane);
  launch_dependent(k_adjbc_inflow, nbi, 64, 0, L, g, in, rth, lamNext, partials);
  launch_dependent(k_sum_partials, 16, 32, 0, L, partials, (int)nbi, 16, grad);
  *L.counter += 6;
}

void launch_functional(const Grid& g, const les_params& p, int j5, double dt, const double* M,
                       const double* Q, double* lam, double* partials, double* Jout,
                       const Launch& L) {
  const long long count = (long long)g.n[0] * g.n[2];
  const int nb = nb_for(count) < kAdjBlocks ? nb_for(count) : kAdjBlocks;
  launch_dependent(k_functional<double>, nb, 256, 0, L, g, p.gamma, j5, dt, M, Q, lam, partials);
  launch_dependent(k_sum_partials, 1, 32, 0, L, partials, nb, 1, Jout);
  *L.counter += 2;
}

void launch_functional(const Grid& g, const les_params& p, int j5, double dt, const float* M,
                       const double* Q, double* partials, double* Jout, const Launch& L) {
  const long long count = (long long)g.n[0] * g.n[2];
  const int nb = nb_for(count) < kAdjBlocks ? nb_for(count) : kAdjBlocks;
  launch_dependent(k_functional<float>, nb, 256, 0, L, g, p.gamma, j5, dt, M, Q, nullptr, partials);
  launch_dependent(k_sum_partials, 1, 32, 0, L, partials, nb, 1, Jout);
  *L.counter += 2;
}

}  // namespace lesjet
