// lesjet_dev.cuh -- device-side types and helpers shared by the CUDA
// translation units of liblesjet (sm_103a).  Nothing here is shared with the
// CPU oracle.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lesjet.h"

namespace lesjet {

// Structured grid, k fastest: node n = (i*nj + j)*nk + k.
struct Grid {
  int n[3];
  int per[3];
  long long N;
  long long stride[3];  // {nj*nk, nk, 1}
  // ghost planes at the low / high xi end of an axial slab (0 at a physical
  // face): those planes belong to the neighbouring slab, which refreshes
  // them between the stages; this grid updates, reduces and sums only its
  // own planes [glo, n[0] - ghi)
  int glo = 0, ghi = 0;
};

// Own planes of a slab (every plane of an undivided grid).
__host__ __device__ inline bool owned_plane(const Grid& g, int i) {
  return i >= g.glo && i < g.n[0] - g.ghi;
}

// Scheme constants in the compute precision R.
template <typename R>
struct Consts {
  R gamma, gm1;      // gamma, gamma - 1
  R k2, k4;          // dissipation constants
  R mu_scale;        // M_j / Re (0 when inviscid)
  R S_suth;          // 110.4 K / T_ref
  R cs2;             // Cs^2 (Smagorinsky) or 2.5 Cs^2 (Vreman)
  R inv_gm1_pr;      // 1/((gamma-1) Pr)
  R inv_gm1_prs;     // 1/((gamma-1) Pr_sgs)
  int sgs;           // LES_SGS_*
  int axis;          // 1: ring j = 0 on the axis (J^-1 = 0 there), Reading A27
};

// Device-resident scalars of a context (inside the workspace).
struct DevScalars {
  double t;          // simulation time (t^{n+1} once a step's dt is known)
  double dt;         // current step
  int status;        // LES_OK or LES_ERR_NONFINITE (sticky)
  int steps;
  unsigned int ticket;  // blocks of a reduction that have finished (its last
                        // block finalises and resets it to 0)
  int pad_;
  double totals[5];
  double dyn[9];     // dynamic SGS procedure: 6 averaged terms, C_ds, C_I, Pr_sgs
};

// Reductions run on a fixed grid (whatever the GPU's SM count), so their
// block partials and summation order, hence their bits, never change.
constexpr int kRedBlocks = 1216;
constexpr int kRedThreads = 256;
constexpr int kMaxPartials = kRedBlocks;
// Blocks of a reduction over n items: at most kRedBlocks, and none without an
// item (on 48 x 24 x 32 most of the 1216 blocks had only queued for the
// ticket or written an empty partial).  It depends on the grid alone.
inline int red_blocks(long long n) {
  const long long b = (n + kRedThreads - 1) / kRedThreads;
  return b < kRedBlocks ? (int)(b < 1 ? 1 : b) : kRedBlocks;
}
// The partials that a smaller reduction grid leaves unwritten, as the
// minimum's neutral element (by block 0).
__device__ __forceinline__ void fill_partials(double* __restrict__ partials) {
  if (blockIdx.x == 0)
    for (int b = gridDim.x + threadIdx.x; b < kRedBlocks; b += blockDim.x) partials[b] = 1.0e300;
}

// Multiprocessor count of the current device (cached per device), for
// sizing grid-stride launches in whole waves.
inline int sm_count() {
  static int cache[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  if (cache[dev] == 0) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      sms = 152;
    cache[dev] = sms;
  }
  return cache[dev];
}

__host__ __device__ inline long long idx3(const Grid& g, int i, int j, int k) {
  return ((long long)i * g.n[1] + j) * g.n[2] + k;
}

__device__ __forceinline__ void decompose(const Grid& g, long long n, int c[3]) {
  if (g.N <= 0x7fffffffLL) {  // every index fits 32 bits: the cheaper division
    const unsigned u = (unsigned)n, nk = (unsigned)g.n[2], nj = (unsigned)g.n[1];
    const unsigned r = u / nk;
    c[2] = (int)(u - r * nk);
    c[0] = (int)(r / nj);
    c[1] = (int)(r - (unsigned)c[0] * nj);
    return;
  }
  long long r = n / g.n[2];
  c[2] = (int)(n - r * g.n[2]);
  c[0] = (int)(r / g.n[1]);
  c[1] = (int)(r - (long long)c[0] * g.n[1]);
}

// Node 'off' steps from node n (coordinates c) along direction d; -1 when it
// falls outside a non-periodic direction.  Periodic directions wrap.
__device__ __forceinline__ long long step(const Grid& g, long long n, const int c[3],
                                          int d, int off) {
  int nd = g.n[d];
  int v = c[d] + off;
  if (g.per[d]) {
    if (v >= nd) v -= nd;
    else if (v < 0) v += nd;
  } else if (v < 0 || v >= nd) {
    return -1;
  }
  return n + (long long)(v - c[d]) * g.stride[d];
}

// Coordinate along d of the node step(g, n, c, d, off) returned (valid only
// when that node exists): c[d] + off, wrapped like step().
__device__ __forceinline__ int coord_step(const Grid& g, const int c[3], int d, int off) {
  int v = c[d] + off;
  if (v >= g.n[d]) v -= g.n[d];
  else if (v < 0) v += g.n[d];
  return v;
}

// A node the stages update: inside every non-periodic face, and along xi
// inside the slab's own planes (a ghost plane is refreshed by the exchange).
__device__ __forceinline__ bool is_interior(const Grid& g, const int c[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (!g.per[d] && (c[d] == 0 || c[d] == g.n[d] - 1)) return false;
  return c[0] >= g.glo && c[0] < g.n[0] - g.ghi;
}

template <typename T>
__device__ __forceinline__ T dev_sqrt(T x);
template <>
__device__ __forceinline__ double dev_sqrt<double>(double x) { return sqrt(x); }
template <>
__device__ __forceinline__ float dev_sqrt<float>(float x) { return sqrtf(x); }

template <typename T>
__device__ __forceinline__ T dev_abs(T x) { return x < T(0) ? -x : x; }
template <>
__device__ __forceinline__ double dev_abs<double>(double x) { return fabs(x); }  // no FP64 compare
template <>
__device__ __forceinline__ float dev_abs<float>(float x) { return fabsf(x); }  // a source modifier

// a > b ? a : b
template <typename T>
__device__ __forceinline__ T dev_max(T a, T b) { return a > b ? a : b; }
// For floats one instruction, which gives NaN if either operand is one (the
// comparison would select b and could hide a NaN in a).
template <>
__device__ __forceinline__ float dev_max<float>(float a, float b) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}
// For doubles the comparison runs on the integer pipe (an FP64 compare takes
// a slot of the FP64 pipe, which bounds these kernels): the bit patterns of
// two doubles order like their values, in reverse when both are negative.
// A NaN on either side selects b, as the comparison would.
template <>
__device__ __forceinline__ double dev_max<double>(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  const bool gt = (x & y) < 0 ? x < y : x > y;
  const unsigned inf = 0x7ff00000u;
  const bool ordered = ((unsigned)__double2hiint(a) & 0x7fffffffu) <= inf &&
                       ((unsigned)__double2hiint(b) & 0x7fffffffu) <= inf;
  return gt && ordered ? a : b;
}

// (double)x on the integer pipe (exact; infinities and NaN take the conversion,
// subnormals that of their integer: a float conversion would flush them in the
// translation units built so, and not in the others).
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), mag = b & 0x7fffffffu;
  const int sign = (int)(b & 0x80000000u);
  if (mag - 0x00800000u < 0x7f000000u)
    return __hiloint2double(sign | (int)((mag >> 3) + 0x38000000u), (int)(b << 29));
  if (mag == 0u) return __hiloint2double(sign, 0);
  if (mag > 0x007fffffu) return (double)x;
  const double m = (double)(int)mag * 0x1p-149;
  return __hiloint2double(sign | __double2hiint(m), __double2loint(m));
}
__device__ __forceinline__ double widen(double x) { return x; }

// a*b + c in one rounding, and a*b in a rounding of its own: with these the
// rounding of an expression does not depend on which products the compiler
// contracts, so that a dual-number run rounds as the double run does.
__device__ __forceinline__ double dev_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double dev_mul(double a, double b) { return __dmul_rn(a, b); }

// First statement of every kernel that launch_dependent starts: nothing runs on
// before the kernel ahead of it has finished and its writes are visible.  (In
// a launch without the attribute it returns at once.)
__device__ __forceinline__ void begin_dependent() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ----------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64 multiplies with the round multipliers, word swap, xor with the
// key; the key advances by the two Weyl increments between rounds.
__device__ inline void philox4x32_10(uint32_t x[4], uint32_t k0, uint32_t k1) {
  const uint32_t A = 0xD2511F53u, B = 0xCD9E8D57u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    uint32_t hiA = __umulhi(A, x[0]), loA = A * x[0];
    uint32_t hiB = __umulhi(B, x[2]), loB = B * x[2];
    uint32_t y0 = hiB ^ x[1] ^ k0;
    uint32_t y2 = hiA ^ x[3] ^ k1;
    x[0] = y0;
    x[1] = loB;
    x[2] = y2;
    x[3] = loA;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

}  // namespace lesjet

// Host-side launch helpers implemented in the .cu files.
namespace lesjet {

struct Launch {
  cudaStream_t s;
  unsigned long long* counter;
};

// A launch whose blocks may take their places, and fetch their code and
// arguments, while the kernel ahead of it in the stream drains; they wait for
// its end in begin_dependent.  For the FP64 and adjoint paths, 18 launches and
// more a step in series: the gap between two was a tenth of the 48 x 24 x 32
// step (323 -> 285 us; the adjoint window on 64 x 40 x 48 30.8 -> 29.5 ms).
// Letting the next kernel start before the last block of this one (an early
// trigger) was slower everywhere, its waiting blocks taking SM places.  The
// mixed step's graph, whose edges are cheap, gains nothing: its prestep, axis
// viscosity and stage kernels are launched plainly, while its boundary
// conditions and dynamic procedure are launched so, as in the FP64 form (the
// captured graph holds programmatic edges there).  Every kernel that is launched
// so begins with begin_dependent, so the end of one implies that of all before it.
template <typename... P, typename... A>
inline void launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                             const Launch& L, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = L.s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// On a grid with an axis (Reading A27) an axis node's SGS viscosity is the
// azimuthal mean of ring 1's at its plane, summed in increasing k; its
// laminar part is its own.  One block per plane i, after k_mu (or the mixed
// prestep) has written mk for every node: ring 1's SGS part is mk minus its
// laminar part.  T(n) gives a node's temperature.
template <typename R>
__device__ __forceinline__ R mu_laminar(const Consts<R>& K, R T) {
  return K.mu_scale * T * dev_sqrt(T) * (R(1) + K.S_suth) / (T + K.S_suth);
}

template <typename R, class TempOf>
__global__ void k_mu_axis(Grid g, Consts<R> K, TempOf T, R* __restrict__ mk) {
  begin_dependent();
  extern __shared__ __align__(16) unsigned char smu_raw[];
  R* smu = reinterpret_cast<R*>(smu_raw);
  const int nk = g.n[2];
  const long long N = g.N;
  const long long base0 = (long long)blockIdx.x * g.stride[0];  // (i, 0, 0)
  const long long base1 = base0 + g.stride[1];                  // (i, 1, 0)
  for (int k = threadIdx.x; k < nk; k += blockDim.x)
    smu[k] = mk[base1 + k] - mu_laminar(K, T(base1 + k));
  __syncthreads();
  __shared__ R mean;
  if (threadIdx.x == 0) {
    R s = R(0);
    for (int k = 0; k < nk; ++k) s += smu[k];
    mean = s / R(nk);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    const long long n = base0 + k;
    const R ml = mu_laminar(K, T(n));
    mk[n] = ml + mean;
    mk[N + n] = ml * K.inv_gm1_pr + mean * K.inv_gm1_prs;
  }
}

// Temperature of a node from a node array (FP64 form: node[4 N + n]).
template <typename R>
struct TempFromNode {
  const R* node;
  long long N;
  __device__ R operator()(long long n) const { return node[4 * N + n]; }
};

// Temperature of a node recovered from the conserved state (System I
// energy), as the mixed prestep does.
template <typename R, typename TQ>
struct TempFromState {
  const TQ* Q;
  long long N;
  R gamma, gm1;
  __device__ R operator()(long long n) const {
    const R rho = (R)Q[n];
    const R ir = R(1) / rho;
    const R u = (R)Q[N + n] * ir, v = (R)Q[2 * N + n] * ir, w = (R)Q[3 * N + n] * ir;
    const R p = gm1 * ((R)Q[4 * N + n] - R(0.5) * rho * (u * u + v * v + w * w));
    return gamma * p * ir;
  }
};


}  // namespace lesjet
