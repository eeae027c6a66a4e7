// dynamic.cu -- the dynamic Smagorinsky procedure (Sec. "Dynamic Smagorinsky
// Model", Eqs. yoshizawa, av_ci, av_cd, av_Pr_sgs), for the FP64 form and,
// with FP32 node fields, products, filter and per-node terms (the sums
// still in FP64, fixed order), for the mixed forms.
//
// Once per viscosity evaluation, from the node primitives of the state:
//   k_dyn_products  per node: the 25 fields the test filter acts on (rho,
//                   rho u_i, rho T, rho u_i u_j, rho|S| S_ij, rho|S| S_mm,
//                   rho|S|^2, rho u_j T, rho|S| dT/dx_j);
//   k_dyn_filter3   the test filter (a tensor product of 3-point filters,
//                   applied along zeta, eta, xi in that order) in one pass
//                   over the FP32 fields; k_dyn_filter1, one direction per
//                   pass, for the FP64 fields;
//   k_dyn_favre     the Favre-filtered velocity and temperature per node;
//   k_dyn_sums      per interior node: the strain of the Favre-filtered
//                   velocity, the Leonard-type terms, and the six
//                   J^-1-weighted sums of the numerators and denominators;
//                   fixed-grid block partials (deterministic);
//   k_dyn_final     one block: fixed-order totals and the coefficients
//                   C_ds, C_I (clipped at 0) and Pr_sgs (the configured
//                   value when the dynamic one is not positive).
// The viscosity pass (k_mu) then forms mu_sgs = C_ds rho Delta^2 |S|, the
// dynamic kappa_sgs and the Yoshizawa sigma_ll = 2 C_I rho Delta^2 |S|^2.
// Test filter: the (1/4, 1/2, 1/4) trapezoidal filter along each direction
// (width 2 Delta), identity along a non-periodic direction at its faces.
#include <type_traits>

#include "stage64_kernels.cuh"

namespace lesjet {

namespace {

constexpr int kDynFields = 25;
constexpr int kDynSums = 7;  // six weighted sums and the sum of the weights

// The neighbours that a node's central differences read, found once per node
// for all fields (mode 0; at an open face the two of the one-sided
// difference: mode 1 at the low face, n + s and n + 2 s, mode 2 at the high
// one, n - 2 s and n - s).
// (The mixed forms' fields, FP32, have fewer than 2^31 points.)
template <typename R>
struct Stencil {
  using I = typename std::conditional<sizeof(R) == 4, int, long long>::type;
  I p[3], m[3];
  int mode[3];
};

template <typename R>
__device__ __forceinline__ Stencil<R> stencil_of(const Grid& g, long long node, const int c[3]) {
  using I = typename Stencil<R>::I;
  Stencil<R> t;
  const I n = (I)node;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const I s = (I)g.stride[d];
    const int last = g.n[d] - 1;
    t.mode[d] = 0;
    t.p[d] = c[d] == last ? n - last * s : n + s;
    t.m[d] = c[d] == 0 ? n + last * s : n - s;
    if (!g.per[d] && c[d] == 0) {
      t.m[d] = n + 2 * s;
      t.mode[d] = 1;
    } else if (!g.per[d] && c[d] == last) {
      t.p[d] = n - 2 * s;
      t.mode[d] = 2;
    }
  }
  return t;
}

// Cartesian gradient of a node field; mh: half the node's metrics (the
// differences are twice the derivatives).  INTERIOR: mode 0 in every direction.
template <bool INTERIOR, typename R>
__device__ __forceinline__ void grad_of(const R* __restrict__ f, long long n, const Stencil<R>& t,
                                        const R mh[9], R out[3]) {
  R dd[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const R fp = f[t.p[d]], fm = f[t.m[d]];
    dd[d] = fp - fm;
    if (!INTERIOR) {
      if (t.mode[d] == 1) dd[d] = R(-3) * f[n] + R(4) * fp - fm;
      if (t.mode[d] == 2) dd[d] = R(3) * f[n] - R(4) * fm + fp;
    }
  }
#pragma unroll
  for (int x = 0; x < 3; ++x) out[x] = mh[x] * dd[0] + mh[3 + x] * dd[1] + mh[6 + x] * dd[2];
}

// S_ij from a velocity gradient gr[i][x] = d u_i/d x_x; returns |S|.
template <typename R>
__device__ __forceinline__ R strain(const R gr[3][3], R S[3][3]) {
  R ss = R(0);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      S[i][j] = R(0.5) * (gr[i][j] + gr[j][i]);
      ss += S[i][j] * S[i][j];
    }
  return dev_sqrt(R(2) * ss);
}

// Component k of a symmetric tensor: (0,0) (1,1) (2,2) (0,1) (0,2) (1,2).
// (Functions, so that the unrolled loops index registers: a table in constant
// memory had put the tensors into local memory.)
__device__ constexpr int i6(int k) { return k < 3 ? k : (k == 5 ? 1 : 0); }
__device__ constexpr int j6(int k) { return k < 3 ? k : (k == 3 ? 1 : 2); }

// u, v, w, T of the mixed forms' float state (node fields 0, 1, 2 and 4; the
// procedure reads no other).
__global__ void __launch_bounds__(256) k_dyn_node(long long N, float gamma, float gm1,
                                                  const float* __restrict__ Q,
                                                  float* __restrict__ node) {
  begin_dependent();
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const float rho = Q[n], ir = 1.f / rho;
    const float u = Q[N + n] * ir, v = Q[2 * N + n] * ir, w = Q[3 * N + n] * ir;
    const float p = gm1 * (Q[4 * N + n] - 0.5f * rho * (u * u + v * v + w * w));
    node[n] = u;
    node[N + n] = v;
    node[2 * N + n] = w;
    node[4 * N + n] = gamma * p * ir;
  }
}

// Register bounds (here and on k_dyn_sums): left free, the compiler gave
// these kernels 230-254 registers, one 256-thread block per SM for a
// latency-bound pass; the FP32 forms run at 64 (the sums spill 276 bytes there
// and 108 at 80, but the fourth block per SM is worth more: two mixed steps on
// 192 x 96 x 128 2.61 and 2.59 ms; five blocks 2.71).
template <typename R, typename TQ, typename TM>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 2) k_dyn_products(Grid g, const TQ* __restrict__ Q,
                                                      const TM* __restrict__ M,
                                                      const R* __restrict__ node,
                                                      R* __restrict__ D) {
  begin_dependent();
  const long long N = g.N;
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    const R rho = (R)Q[n];
    const R vel[3] = {node[n], node[N + n], node[2 * N + n]};
    const R T = node[4 * N + n];
    const Stencil<R> st = stencil_of<R>(g, n, c);
    R mh[9], gr[3][3], S[3][3], dT[3];
#pragma unroll
    for (int t = 0; t < 9; ++t) mh[t] = R(0.5) * (R)M[t * N + n];
#pragma unroll
    for (int q = 0; q < 3; ++q) grad_of<false>(node + q * N, n, st, mh, gr[q]);
    grad_of<false>(node + 4 * N, n, st, mh, dT);
    const R Sm = strain(gr, S);
    D[n] = rho;
#pragma unroll
    for (int i = 0; i < 3; ++i) D[(1 + i) * N + n] = rho * vel[i];
    D[4 * N + n] = rho * T;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int i = i6(k), j = j6(k);
      D[(5 + k) * N + n] = rho * vel[i] * vel[j];
      D[(11 + k) * N + n] = rho * Sm * S[i][j];
    }
    D[17 * N + n] = rho * Sm * (S[0][0] + S[1][1] + S[2][2]);
    D[18 * N + n] = rho * Sm * Sm;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      D[(19 + j) * N + n] = rho * vel[j] * T;
      D[(22 + j) * N + n] = rho * Sm * dT[j];
    }
  }
}

// One pass of the test filter along direction D for `count` fields:
// dst = (src_{-1} + 2 src_0 + src_{+1})/4 along D (periodic wrap), the
// identity at the faces of a non-periodic D.
template <int D, typename R>
__global__ void __launch_bounds__(256) k_dyn_filter1(Grid g, const R* __restrict__ src,
                                                     int count, R* __restrict__ dst) {
  begin_dependent();
  const long long N = g.N;
  const long long s = g.stride[D];
  const int nd = g.n[D];
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    const bool face = !g.per[D] && (c[D] == 0 || c[D] == nd - 1);
    if (face) {
      for (int q = 0; q < count; ++q) dst[q * N + n] = src[q * N + n];
      continue;
    }
    const long long np = (c[D] == nd - 1) ? n - (long long)(nd - 1) * s : n + s;
    const long long nm = (c[D] == 0) ? n + (long long)(nd - 1) * s : n - s;
#pragma unroll 5
    for (int q = 0; q < count; ++q)
      dst[q * N + n] = R(0.25) * src[q * N + nm] + R(0.5) * src[q * N + n] + R(0.25) * src[q * N + np];
  }
}

// The test filter's three directions in one kernel (blockIdx.z: field, then
// axial chunk).  A thread owns kF3R rows of one column and marches along xi
// over planes i0 - 1 .. i1: it reads the plane's kF3R + 2 rows at its column
// and the two beside it (the next plane's while it works on this one), filters
// along zeta, then eta, and keeps the last two planes' values in registers to
// filter along xi.  Each output takes the same operations in the same order
// as three one-direction passes would (zeta, eta, xi; identity at the faces of
// a non-periodic direction).  Bound by those loads, most of them L1 hits: one
// field per block, no shared memory and no barriers, and four rows per thread,
// whose 18 loads give four outputs (12 gave two).
constexpr int kF3J = 2, kF3K = 32, kF3R = 4;  // 64 threads: 8 rows x 32 columns

template <typename R>
__global__ void __launch_bounds__(kF3J * kF3K) k_dyn_filter3(Grid g, const R* __restrict__ src,
                                                             int fields, R* __restrict__ dst) {
  begin_dependent();
  const long long N = g.N;
  const int ni = g.n[0], nj = g.n[1], nk = g.n[2];
  const int tx = threadIdx.x % kF3K, ty = threadIdx.x / kF3K;
  const int k = blockIdx.x * kF3K + tx, j0 = (blockIdx.y * kF3J + ty) * kF3R;
  const int f = blockIdx.z % fields, ch = blockIdx.z / fields, nch = gridDim.z / fields;
  const int i0 = (int)((long long)ch * ni / nch), i1 = (int)((long long)(ch + 1) * ni / nch);
  if (k >= nk || j0 >= nj) return;
  src += (long long)f * N;
  dst += (long long)f * N;
  // a missing neighbour (an open face's) is the node itself, and not used
  const bool kface = !g.per[2] && (k == 0 || k == nk - 1);
  const int km = kface ? k : (k == 0 ? nk - 1 : k - 1), kp = kface ? k : (k == nk - 1 ? 0 : k + 1);
  int row[kF3R + 2];  // offsets of rows j0 - 1 .. j0 + kF3R within a plane
  bool jface[kF3R];
#pragma unroll
  for (int q = 0; q < kF3R + 2; ++q) {
    int j = j0 - 1 + q;
    if (j < 0) j = g.per[1] ? nj - 1 : 0;
    if (j >= nj) j = g.per[1] ? j % nj : nj - 1;
    row[q] = j * nk;
  }
#pragma unroll
  for (int q = 0; q < kF3R; ++q) jface[q] = !g.per[1] && (j0 + q == 0 || j0 + q == nj - 1);
  R s[kF3R + 2][3];  // the raw values of the plane to come
  auto fetch = [&](int x) {
    const int ig = (x >= 0 && x < ni) ? x : (g.per[0] ? (x < 0 ? ni - 1 : 0) : -1);
    if (ig < 0) return;  // outside an open xi: read by no output
    const R* S = src + (long long)ig * g.stride[0];
#pragma unroll
    for (int q = 0; q < kF3R + 2; ++q) {
      s[q][0] = S[row[q] + km];
      s[q][1] = S[row[q] + k];
      s[q][2] = S[row[q] + kp];
    }
  };
#pragma unroll
  for (int q = 0; q < kF3R + 2; ++q) s[q][0] = s[q][1] = s[q][2] = R(0);
  fetch(i0 - 1);
  R em[kF3R], ec[kF3R];  // 2-D-filtered values of planes x - 2, x - 1
#pragma unroll
  for (int q = 0; q < kF3R; ++q) em[q] = ec[q] = R(0);
  for (int x = i0 - 1; x <= i1; ++x) {
    R z[kF3R + 2], e[kF3R];
#pragma unroll
    for (int q = 0; q < kF3R + 2; ++q)
      z[q] = kface ? s[q][1] : R(0.25) * s[q][0] + R(0.5) * s[q][1] + R(0.25) * s[q][2];
    if (x < i1) fetch(x + 1);
#pragma unroll
    for (int q = 0; q < kF3R; ++q)
      e[q] = jface[q] ? z[q + 1] : R(0.25) * z[q] + R(0.5) * z[q + 1] + R(0.25) * z[q + 2];
    // plane x - 1 has both xi neighbours now
    const int xo = x - 1;
    if (xo >= i0) {
      const bool face = !g.per[0] && (xo == 0 || xo == ni - 1);
      const long long o = (long long)xo * g.stride[0] + (long long)j0 * nk + k;
#pragma unroll
      for (int q = 0; q < kF3R; ++q)
        if (j0 + q < nj)
          dst[o + q * nk] = face ? ec[q] : R(0.25) * em[q] + R(0.5) * ec[q] + R(0.25) * e[q];
    }
#pragma unroll
    for (int q = 0; q < kF3R; ++q) {
      em[q] = ec[q];
      ec[q] = e[q];
    }
  }
}

// Favre-filtered velocity and temperature u^_i = (rho u_i)^/rho^,
// T^ = (rho T)^/rho^ at every node, from the filtered fields F.
template <typename R>
__global__ void __launch_bounds__(256) k_dyn_favre(long long N, const R* __restrict__ F,
                                                   R* __restrict__ H) {
  begin_dependent();
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    const R ir = R(1) / F[n];
#pragma unroll
    for (int q = 0; q < 4; ++q) H[q * N + n] = F[(1 + q) * N + n] * ir;
  }
}

// Per interior node the six terms (numerators and denominators of the
// three coefficients), in R; their J^-1-weighted sums in FP64.
template <typename R, typename TM>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 1) k_dyn_sums(Grid g, const TM* __restrict__ M,
                                                  const R* __restrict__ node,
                                                  const R* __restrict__ Fh,
                                                  const R* __restrict__ H,
                                                  double* __restrict__ partials) {
  begin_dependent();
  const long long N = g.N;
  double acc[kDynSums] = {0, 0, 0, 0, 0, 0, 0};
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
       n += (long long)gridDim.x * blockDim.x) {
    int c[3];
    decompose(g, n, c);
    if (!is_interior(g, c)) continue;
    const double wgt = widen(M[9 * N + n]);
    const R Delta = cbrt((R)M[9 * N + n]);
    const R D2 = Delta * Delta, Dh2 = R(4) * D2;
    const Stencil<R> st = stencil_of<R>(g, n, c);
    R mm[9], gr[3][3], S[3][3], dT[3], grh[3][3], Sh[3][3], dTh[3];
#pragma unroll
    for (int t = 0; t < 9; ++t) mm[t] = R(0.5) * (R)M[t * N + n];
#pragma unroll
    for (int q = 0; q < 3; ++q) grad_of<true>(node + q * N, n, st, mm, gr[q]);
    grad_of<true>(node + 4 * N, n, st, mm, dT);
    strain(gr, S);
#pragma unroll
    for (int q = 0; q < 3; ++q) grad_of<true>(H + q * N, n, st, mm, grh[q]);
    grad_of<true>(H + 3 * N, n, st, mm, dTh);
    const R Shm = strain(grh, Sh);
    // the filtered fields at this node (Fh holds all 25)
    R fh[kDynFields];
#pragma unroll
    for (int q = 5; q < kDynFields; ++q) fh[q] = Fh[q * N + n];
    const R rh = Fh[n], irh = R(1) / rh;  // one division per node
    const R mh[3] = {Fh[N + n], Fh[2 * N + n], Fh[3 * N + n]};
    R L[3][3], Fs[3][3];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int i = i6(k), j = j6(k);
      L[i][j] = L[j][i] = fh[5 + k] - mh[i] * mh[j] * irh;
      Fs[i][j] = Fs[j][i] = fh[11 + k];
    }
    const R trS = S[0][0] + S[1][1] + S[2][2];
    const R trSh = Sh[0][0] + Sh[1][1] + Sh[2][2];
    R LS = R(0), FS = R(0), ShS = R(0);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        LS += L[i][j] * S[i][j];
        FS += Fs[i][j] * S[i][j];
        ShS += Sh[i][j] * S[i][j];
      }
    const R Lkk = L[0][0] + L[1][1] + L[2][2];
    const R tr3 = trS * R(1.0 / 3.0);
    const R numC = LS - Lkk * tr3;
    const R denC = R(2) * D2 * (FS - fh[17] * tr3) -
                   R(2) * Dh2 * (rh * Shm * ShS - rh * Shm * trSh * tr3);
    const R denI = R(2) * Dh2 * rh * Shm * Shm - R(2) * D2 * fh[18];
    R numP = R(0), denP = R(0);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const R K = fh[19 + j] - mh[j] * Fh[4 * N + n] * irh;
      numP += D2 * fh[22 + j] * dT[j] - Dh2 * rh * Shm * dTh[j] * dT[j];
      denP += K * dT[j];
    }
    acc[0] += wgt * widen(numC);
    acc[1] += wgt * widen(denC);
    acc[2] += wgt * widen(Lkk);
    acc[3] += wgt * widen(denI);
    acc[4] += wgt * widen(numP);
    acc[5] += wgt * widen(denP);
    acc[6] += wgt;
  }
  __shared__ double red[kDynSums][32];
#pragma unroll
  for (int q = 0; q < kDynSums; ++q)
    for (int off = 16; off > 0; off >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < kDynSums; ++q) red[q][threadIdx.x >> 5] = acc[q];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int q = 0; q < kDynSums; ++q) {
      double v = threadIdx.x < (blockDim.x >> 5) ? red[q][threadIdx.x] : 0.0;
      for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if (threadIdx.x == 0) partials[q * kRedBlocks + blockIdx.x] = v;
    }
  }
}

// One block of kDynSums warps: warp q totals partial array q in a fixed order.
__global__ void k_dyn_final(const double* __restrict__ partials, double pr_default,
                            DevScalars* __restrict__ sc) {
  begin_dependent();
  __shared__ double tot[kDynSums];
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < kDynSums) {
    double v = 0.0;
#pragma unroll 19
    for (int b = lane; b < kRedBlocks; b += 32) v += partials[q * kRedBlocks + b];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) tot[q] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double* out = sc->dyn;
    for (int k = 0; k < 6; ++k) out[k] = tot[k] / tot[6];
    double Cd = out[1] != 0.0 ? out[0] / out[1] : 0.0;
    if (!(Cd > 0.0)) Cd = 0.0;
    double CI = out[3] != 0.0 ? out[2] / out[3] : 0.0;
    if (!(CI > 0.0)) CI = 0.0;
    double Pr = out[5] != 0.0 ? Cd * out[4] / out[5] : 0.0;
    if (!(Pr > 0.0) || !(Pr < 1e300)) Pr = pr_default;
    out[6] = Cd;
    out[7] = CI;
    out[8] = Pr;
  }
}

}  // namespace

template <typename R, typename TQ, typename TM>
static void dynamic_t(const Grid& g, const les_params& p, const TQ* Q, const TM* M, const R* node,
                      R* scratch, double* partials, DevScalars* sc, const Launch& L) {
  const int th = 256, nb = blocks_for(g.N, th);
  R* D = scratch;                                 // products, then the eta pass
  R* T = scratch + (long long)kDynFields * g.N;  // zeta pass, then the filtered fields
  launch_dependent(k_dyn_products<R, TQ, TM>, nb, th, 0, L, g, Q, M, node, D);
  if constexpr (sizeof(R) == 4) {
    // FP32 fields: the test filter in one pass (k_dyn_filter3), with enough
    // axial chunks for some sixty CTAs per SM (each reads two planes more
    // than it writes)
    const long long tk = (g.n[2] + kF3K - 1) / kF3K,
                    tj = (g.n[1] + kF3J * kF3R - 1) / (kF3J * kF3R), tiles = tk * tj * kDynFields;
    const long long want = 64LL * sm_count();
    const long long most = g.n[0] / 12 > 1 ? g.n[0] / 12 : 1;
    long long nch = (want + tiles - 1) / tiles;
    nch = nch < 1 ? 1 : (nch > most ? most : nch);
    launch_dependent(k_dyn_filter3<R>, dim3((unsigned)tk, (unsigned)tj,
                     (unsigned)(nch * kDynFields)), kF3J * kF3K, 0, L, g, D, kDynFields, T);
    *L.counter += 1;
  } else {
    // FP64 fields: three one-direction passes (the one-pass kernel is bound
    // by its FP64 work and latency there: 1.24 against 0.86 ms on 1.97M points)
    launch_dependent(k_dyn_filter1<2, R>, nb, th, 0, L, g, D, kDynFields, T);
    launch_dependent(k_dyn_filter1<1, R>, nb, th, 0, L, g, T, kDynFields, D);
    launch_dependent(k_dyn_filter1<0, R>, nb, th, 0, L, g, D, kDynFields, T);
    *L.counter += 3;
  }
  launch_dependent(k_dyn_favre<R>, nb, th, 0, L, g.N, T, D);  // D is free again: u^, v^, w^, T^
  launch_dependent(k_dyn_sums<R, TM>, kRedBlocks, kRedThreads, 0, L, g, M, node, T, D, partials);
  launch_dependent(k_dyn_final, 1, 32 * kDynSums, 0, L, partials, p.Pr_sgs, sc);
  *L.counter += 4;
}

void launch_dynamic64(const Grid& g, const les_params& p, const StageIO64& io, double* scratch,
                      const Launch& L) {
  dynamic_t<double, double, double>(g, p, io.Qin, io.M, io.node, scratch, io.partials, io.sc, L);
}

void launch_dynamic32(const Grid& g, const les_params& p, const float* Q, const float* M,
                      float* node, float* scratch, double* partials, DevScalars* sc,
                      const Launch& L) {
  const int th = 256, nb = blocks_for(g.N, th);
  launch_dependent(k_dyn_node, nb, th, 0, L, g.N, (float)p.gamma, (float)(p.gamma - 1.0), Q, node);
  ++*L.counter;
  dynamic_t<float, float, float>(g, p, Q, M, node, scratch, partials, sc, L);
}

}  // namespace lesjet
