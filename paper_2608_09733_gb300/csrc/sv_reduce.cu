// sv_reduce.cu -- read-only expectation reductions for sm_103a.
//
// <Z_q> for every qubit in one pass (Sec. 5.3 probabilities p_b = x_b^2 + y_b^2,
// Sec. 4.4 Pauli path): <Z_q> = T - 2 S_q with T = sum_b p_b and S_q the sum
// over the amplitudes whose bit q is set.  A warp owns a chunk of 32 x 32
// 16-byte vectors; inside a chunk the low index bits are the vector element,
// the lane and the iteration, so S_q for those bits is accumulated with
// compile-time-known adds and a warp butterfly; bits above the chunk are the
// same for the whole chunk.
//
// General Pauli terms (Sec. 4.4): <psi|P|psi> = i^{nY} sum_b (-1)^{popc(b&z)}
// conj(psi_{b^x}) psi_b.  For x != 0 the sum is taken over half the indices
// (bit h = top bit of x clear) and doubled: the partner's term is the complex
// conjugate of this one, so <P> = 2 Re[i^{nY} sum_half ...].  Terms that share
// an x mask share one pass.
//
// Precision (complex64): each thread sums p in float over a short run (64
// amplitudes); the warp adds its 32 runs in float (a chunk of 2048
// amplitudes: relative error below 70 float roundings, 4e-6, of the chunk's
// sum) and the chunk sums go into double, as do the block and grid
// reductions.  (Warp sums in double took most of the kernel's time: the FP64
// pipe of this part runs a warp-wide add in about 16 cycles.)  complex128
// accumulates in double throughout.
// The grid writes one partial per block and a second kernel adds them in a
// fixed order, so results are identical run to run.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <utility>
#include <vector>

#include "sv_internal.h"

namespace sv {

namespace {

constexpr int kRedThreads = 256;
constexpr int kRedWarps = kRedThreads / 32;
constexpr int kJ = 32;          // vectors per lane per chunk
constexpr int kMaxTermsPerPass = 16;
constexpr int kMaxTermSlots = 128;  // terms whose partials one finish launch adds up

int red_grid() { return device_sm_count() * 4; }

template <typename R>
struct Acc;  // accumulation type for short runs
template <>
struct Acc<float> {
  using T = float;
};
template <>
struct Acc<double> {
  using T = double;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of W values over the warp's lanes: each step hands half of the values
// to the partner lane, so W sums take W + log2(32 / W) - 1 adds a lane instead
// of 5 W (an FP64 add occupies the SM's FP64 pipe for about 16 cycles).  The
// lane ends with the sum of value lane / (32 / W), added as the tree that
// warp_sum adds.
template <int W, int O = 16, typename T>
__device__ __forceinline__ T warp_fold(T (&a)[W], int lane) {
  if constexpr (W == 1) {
    T v = a[0];
#pragma unroll
    for (int o = O; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  } else {
    T b[W / 2];
    const bool hi = lane & O;
#pragma unroll
    for (int k = 0; k < W / 2; k++) {
      const T keep = hi ? a[k + W / 2] : a[k], send = hi ? a[k] : a[k + W / 2];
      b[k] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
    return warp_fold<W / 2, O / 2>(b, lane);
  }
}

// ------------------------------------------------------------ <Z_q> for all q
//
// grid.y is the state of a batch (one for a single read-out): state b starts
// at state + (b << n), its partial rows at (b * gridDim.x) rows.

// A = amplitudes per 16-byte vector (2 for complex64, 1 for complex128).
// Chunk = 32 lanes x kJ vectors x A amplitudes; chunk bits C = log2(1024 A).
template <typename R>
__global__ void __launch_bounds__(kRedThreads) k_expect_z_all(const Cx<R>* __restrict__ state, int n,
                                                            double* __restrict__ partials) {
  constexpr int A = 16 / sizeof(Cx<R>);
  constexpr int EB = (A == 2) ? 1 : 0;  // index bits taken by the vector element
  constexpr int C = EB + 5 + 5;         // chunk bits
  using T = typename Acc<R>::T;
  __shared__ double red[kRedWarps][SV_MAX_QUBITS + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, block_warps = blockDim.x >> 5;
  const uint64_t nchunks = 1ull << (n - C);
  const uint64_t gwarp = (uint64_t)blockIdx.x * block_warps + warp;
  const uint64_t nwarps = (uint64_t)gridDim.x * block_warps;
  state += (uint64_t)blockIdx.y << n;
  double accq0 = 0.0, accq1 = 0.0, acct = 0.0;  // qubits lane and lane + 32; total
  for (uint64_t ch = gwarp; ch < nchunks; ch += nwarps) {
    const uint4* src = reinterpret_cast<const uint4*>(state + (ch << C));
    // the lane's sums: total, element 1, iteration bits 0..4 set, lane bits
    // 0..4 set (the total where the bit is set)
    T v[16];
#pragma unroll
    for (int k = 0; k < 16; k++) v[k] = 0;
    if constexpr (A == 2) {
#pragma unroll
      for (int j = 0; j < kJ; j++) {
        uint4 w = __ldg(src + j * 32 + lane);
        float2 a = *reinterpret_cast<float2*>(&w.x), b = *reinterpret_cast<float2*>(&w.z);
        T p0 = fmaf(a.x, a.x, a.y * a.y), p1 = fmaf(b.x, b.x, b.y * b.y);
        v[1] += p1;
        const T p = p0 + p1;
        v[0] += p;
#pragma unroll
        for (int b2 = 0; b2 < 5; b2++)
          if ((j >> b2) & 1) v[2 + b2] += p;
      }
    } else {
      // pairwise over the iteration bits: 62 adds for the total and the five
      // bit sums of 32 values, against 112 added one by one (FP64 pipe bound)
      T p[kJ];
#pragma unroll
      for (int j = 0; j < kJ; j++) {
        uint4 w = __ldg(src + j * 32 + lane);
        double2 a = *reinterpret_cast<double2*>(&w);
        p[j] = fma(a.x, a.x, a.y * a.y);
      }
#pragma unroll
      for (int b2 = 0; b2 < 5; b2++) {
#pragma unroll
        for (int j = 0; j < (kJ >> (b2 + 1)); j++) {
          v[2 + b2] += p[2 * j + 1];
          p[j] = p[2 * j] + p[2 * j + 1];
        }
      }
      v[0] = p[0];
    }
#pragma unroll
    for (int b = 0; b < 5; b++) v[7 + b] = ((lane >> b) & 1) ? v[0] : T(0);
    // the sum of value k sits in lanes 2 k and 2 k + 1 (in the run's
    // precision), then into double
    const double sum = (double)warp_fold(v, lane);
    const double t = __shfl_sync(0xffffffffu, sum, 0);
    // lane q picks S_q for its qubits q = lane and lane + 32: bits inside the
    // chunk from the lane holding their sum, bits above it from the chunk index
    const int k = (EB && lane == 0) ? 1 : lane < EB + 5 ? 7 + lane - EB : 2 + lane - EB - 5;
    const double in_chunk = __shfl_sync(0xffffffffu, sum, lane < C ? 2 * k : 0);
    if (lane < C)
      accq0 += in_chunk;
    else if (lane < n)
      accq0 += ((ch >> (lane - C)) & 1ull) ? t : 0.0;
    if (lane + 32 < n) accq1 += ((ch >> (lane + 32 - C)) & 1ull) ? t : 0.0;
    acct += t;
  }
  if (lane < n) red[warp][lane] = accq0;
  if (lane + 32 < n) red[warp][lane + 32] = accq1;
  if (lane == 0) red[warp][n] = acct;
  __syncthreads();
  for (int q = threadIdx.x; q <= n; q += blockDim.x) {
    double s = 0.0;
    for (int w = 0; w < block_warps; w++) s += red[w][q];
    partials[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (n + 1) + q] = s;
  }
}

// States below one warp chunk (2^n <= 1024 amplitudes): one block a state,
// amplitude a = thread + 256 i, so bits 0..4 are the lane, 5..7 the warp, 8
// and 9 the iteration.
template <typename R>
__global__ void __launch_bounds__(256) k_expect_z_small(const Cx<R>* __restrict__ state, int n,
                                                        double* __restrict__ partials) {
  __shared__ double red[8][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  state += (uint64_t)blockIdx.x << n;
  double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};  // total, lane bits 0..4, iteration bits 0..1
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const uint32_t a = threadIdx.x + 256u * i;
    if (a >> n) continue;
    const Cx<R> x = state[a];
    const double p = (double)x.re * x.re + (double)x.im * x.im;
    v[0] += p;
    if (i & 1) v[6] += p;
    if (i & 2) v[7] += p;
  }
#pragma unroll
  for (int b = 0; b < 5; b++) v[1 + b] = ((lane >> b) & 1) ? v[0] : 0.0;
  const double sum = warp_fold(v, lane);  // value k in lanes 4 k ..
  if ((lane & 3) == 0) red[warp][lane >> 2] = sum;
  __syncthreads();
  if (threadIdx.x <= n) {
    const int q = threadIdx.x;
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; w++) {
      const int k = q == n ? 0 : q < 5 ? 1 + q : q < 8 ? 0 : 6 + q - 8;
      const bool in = q == n || q < 5 || q >= 8 || ((w >> (q - 5)) & 1);
      if (in) s += red[w][k];
    }
    partials[(size_t)blockIdx.x * (n + 1) + q] = s;
  }
}

// Adds a state's partial rows (one block a state): warp w takes rows w,
// w + 32, ..., a lane the columns lane and lane + 32; the warps' sums are
// added in warp order.  (One thread per column walking all 608 rows of a
// 26-qubit state took 81 us; this takes 17.)
__global__ void __launch_bounds__(1024) k_finish_z_all(const double* __restrict__ partials, int nblocks, int n,
                                                       double* __restrict__ out) {
  __shared__ double s[32][SV_MAX_QUBITS + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  partials += (size_t)blockIdx.x * nblocks * (n + 1);
  out += (size_t)blockIdx.x * (n + 1);
  double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
  for (int b = warp; b < nblocks; b += nwarps) {
    const double* row = partials + (size_t)b * (n + 1);
    if (lane <= n) a0 += row[lane];
    if (lane + 32 <= n) a1 += row[lane + 32];
  }
  if (lane <= n) s[warp][lane] = a0;
  if (lane + 32 <= n) s[warp][lane + 32] = a1;
  __syncthreads();
  if (warp == 0) {
    double c0 = 0.0, c1 = 0.0;
#pragma unroll 8
    for (int w = 0; w < nwarps; w++) {
      if (lane <= n) c0 += s[w][lane];
      if (lane + 32 <= n) c1 += s[w][lane + 32];
    }
    const double T = __shfl_sync(0xffffffffu, n < 32 ? c0 : c1, n & 31);
    const double z0 = lane < n ? T - 2.0 * c0 : 0.0, z1 = lane + 32 < n ? T - 2.0 * c1 : 0.0;
    if (lane < n) out[lane] = z0;
    if (lane + 32 < n) out[lane + 32] = z1;
    const double sum = warp_sum(z0 + z1);
    if (lane == 0) out[n] = sum;
  }
}

// ------------------------------------------------------------ Pauli terms
//
// Terms that share an X mask share a pass of up to 16; grid.y runs over the
// passes of one launch, so a Hamiltonian of many masks is a few launches and
// the blocks of one pass fill in behind the blocks of the last.  Each term
// adds one real number per amplitude: the real part of conj(c) a when its
// count of Y letters is even, else (IMAG) the imaginary part, with the sign
// flipped by an XOR; terms of one mask and different kinds take a pass each,
// so that a pass forms one part.  NT is the accumulators a thread holds: a pass of one term (X on
// one site) pays for one, not for 16.  24 qubits complex64, 24 X terms and 24
// ZZ terms: 0.46 ms of kernels (14.8 us a one-term pass, 9.1 TB/s with L2's
// share; 62 us for 16 signed terms, ALU bound), where 16 accumulators for every
// pass and a one-warp finish took 7.2 + 2.4 ms.  complex128 is bound by the
// FP64 pipe: 5.6 us a one-term pass at 21 qubits (95 before).
// The order of a thread's single-precision runs (64 elements a grid stride
// apart) is fixed, whatever NT is.

template <int NT>
struct TermPass {
  uint64_t x;
  uint64_t z[NT];
  int32_t h;      // top bit of x
  int32_t slot;   // first partial row
  int32_t nt;     // terms (<= NT)
};
template <int NT>
constexpr int kPassesPerLaunch = 3840 / (int)sizeof(TermPass<NT>);
template <int NT>
struct TermPasses {
  TermPass<NT> p[kPassesPerLaunch<NT>];
};

__device__ __forceinline__ float flip_sign(float v, uint32_t sign) {
  return __uint_as_float(__float_as_uint(v) ^ sign);
}
__device__ __forceinline__ double flip_sign(double v, uint32_t sign) {
  return __hiloint2double(__double2hiint(v) ^ (int)sign, __double2loint(v));
}

template <typename R, int NT, bool PAIRED, bool IMAG>
__global__ void __launch_bounds__(kRedThreads) k_expect_terms(const Cx<R>* __restrict__ state, int n,
                                                            const __grid_constant__ TermPasses<NT> passes,
                                                            double* __restrict__ partials) {
  using T = typename Acc<R>::T;
  const TermPass<NT>& tp = passes.p[blockIdx.y];
  // signs of all terms at an index: with four terms and more the XOR of one
  // 32-bit word per index byte (term j's parity at bit 31 - j), built here;
  // fewer terms take a popcount each (its rate is a quarter of an XOR's)
  constexpr bool kTable = NT >= 4;
  constexpr int kBytes = (SV_MAX_QUBITS + 7) / 8;
  __shared__ uint32_t sgn[kTable ? kBytes : 1][256];
  __shared__ double red[kRedWarps][NT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t x = tp.x, low = PAIRED ? (1ull << tp.h) - 1ull : 0ull;
  if constexpr (kTable) {
    for (int e = threadIdx.x; e < kBytes * 256; e += blockDim.x) {
      uint32_t m = 0;
#pragma unroll
      for (int j = 0; j < NT; j++)
        m |= (uint32_t)(__popc((uint32_t)(tp.z[j] >> (8 * (e >> 8))) & (uint32_t)(e & 255)) & 1) << (31 - j);
      sgn[e >> 8][e & 255] = m;
    }
    __syncthreads();
  }
  const uint64_t count = PAIRED ? (1ull << (n - 1)) : (1ull << n);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  double acc[NT];
#pragma unroll
  for (int j = 0; j < NT; j++) acc[j] = 0.0;
  constexpr int U = sizeof(R) == 4 ? 8 : 4;  // elements in flight per thread
  static_assert(64 % U == 0, "whole groups in a run");
  T run[NT] = {};
  auto index_of = [&](uint64_t i) { return PAIRED ? i + (i & ~low) : i; };  // a zero inserted at bit h
  auto add = [&](const Cx<R>& a, const Cx<R>& c, uint64_t b) {
    uint32_t m = 0;
    if constexpr (kTable) {
      m = sgn[0][b & 255] ^ sgn[1][(b >> 8) & 255] ^ sgn[2][(b >> 16) & 255];
      if (n > 24) m ^= sgn[3][(b >> 24) & 255] ^ sgn[4][(b >> 32) & 255];
    } else {
#pragma unroll
      for (int j = 0; j < NT; j++) {
        const uint32_t w = ((uint32_t)b & (uint32_t)tp.z[j]) ^ ((uint32_t)(b >> 32) & (uint32_t)(tp.z[j] >> 32));
        m |= (uint32_t)__popc(w) << (31 - j) & (0x80000000u >> j);
      }
    }
    if constexpr (PAIRED && NT == 1 && sizeof(R) == 8) {  // FP64 pipe bound: the sign rides on a, two FMAs
      const T p = flip_sign(IMAG ? a.im : a.re, m & 0x80000000u);
      const T q = flip_sign(IMAG ? a.re : a.im, (m & 0x80000000u) ^ (IMAG ? 0x80000000u : 0u));
      run[0] = fma(c.re, p, fma(c.im, q, run[0]));
    } else {
      T v;
      if constexpr (PAIRED)  // conj(c) * a
        v = IMAG ? (T)c.re * (T)a.im - (T)c.im * (T)a.re : (T)c.re * (T)a.re + (T)c.im * (T)a.im;
      else
        v = (T)a.re * (T)a.re + (T)a.im * (T)a.im;
#pragma unroll
      for (int j = 0; j < NT; j++) run[j] += flip_sign(v, (m << j) & 0x80000000u);
    }
  };
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  while (i < count) {
#pragma unroll
    for (int j = 0; j < NT; j++) run[j] = 0;
    // a short run in the run precision, then fold into double
    for (int r = 0; r < 64 && i < count;) {
      if (i + (U - 1) * stride < count) {
        Cx<R> a[U], c[U];
#pragma unroll
        for (int k = 0; k < U; k++) {
          const uint64_t b = index_of(i + k * stride);
          a[k] = state[b];
          if constexpr (PAIRED) c[k] = state[b ^ x];
        }
#pragma unroll
        for (int k = 0; k < U; k++) add(a[k], PAIRED ? c[k] : a[k], index_of(i + k * stride));
        r += U;
        i += U * stride;
      } else {
        const uint64_t b = index_of(i);
        const Cx<R> a = state[b];
        add(a, PAIRED ? state[b ^ x] : a, b);
        r++;
        i += stride;
      }
    }
#pragma unroll
    for (int j = 0; j < NT; j++) acc[j] += (double)run[j];
  }
  const double s = warp_fold(acc, lane);
  if (lane % (32 / NT) == 0) red[warp][lane / (32 / NT)] = s;
  __syncthreads();
  if ((int)threadIdx.x < tp.nt) {
    double a = 0.0;
    for (int w = 0; w < kRedWarps; w++) a += red[w][threadIdx.x];
    partials[(size_t)(tp.slot + threadIdx.x) * gridDim.x + blockIdx.x] = a;
  }
}

struct TermOut {
  uint16_t dst[kMaxTermSlots];  // output index of each slot's term
  uint8_t how[kMaxTermSlots];   // bits 0..1: Y letters mod 4; bit 2: paired
};

// One block per term adds its partials; Re[i^{nY} (a + i b)], of which the
// pass kernel kept a (nY even) or b (odd).
__global__ void __launch_bounds__(128) k_finish_terms(const double* __restrict__ partials, int nblocks,
                                                      const __grid_constant__ TermOut to, double* __restrict__ out) {
  __shared__ double red[4];
  const int j = blockIdx.x;
  double a = 0.0;
  for (int k = threadIdx.x; k < nblocks; k += blockDim.x) a += partials[(size_t)j * nblocks + k];
  a = warp_sum(a);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    a = (red[0] + red[1]) + (red[2] + red[3]);
    const int ny = to.how[j] & 3;
    const double re = ny == 1 || ny == 2 ? -a : a;
    out[to.dst[j]] = (to.how[j] & 4) ? 2.0 * re : re;
  }
}

}  // namespace

// Sized for the largest state whatever n is, so the per-stream scratch never
// regrows: regrowing frees the old buffer, and cudaFree synchronizes the whole
// device (it would wait for a resident serving kernel).
size_t expect_z_all_scratch_doubles(int n) {
  (void)n;
  return (size_t)red_grid() * (SV_MAX_QUBITS + 1);
}
size_t expect_terms_scratch_doubles(int n, int n_terms) {
  (void)n;
  (void)n_terms;
  return (size_t)red_grid() * kMaxTermSlots;
}

// Blocks of a state's read-out: a warp a chunk; blocks of one warp until the
// grid holds a block an SM over the whole batch (a small state spreads over the
// SMs), then of up to eight.  More than 4096 chunks take up to four blocks an
// SM: the finish adds a row a block, which is most of the time of a small state
// (complex64, us, four blocks an SM against one: 18 qubits 12.5 and 12.5, 20
// qubits 19.7 and 14.5, 23 qubits 24.8 and 18.7, 24 qubits 41 and 46, 26 qubits
// 95 and 137).
static int z_all_blocks(int n, int chunk_bits, int batch, int* warps) {
  if (n < chunk_bits) return 1;
  const uint64_t chunks = 1ull << (n - chunk_bits);
  const uint64_t blocks = chunks * batch <= 4096 ? device_sm_count() : red_grid();
  const uint64_t most = (blocks + batch - 1) / batch;
  const uint64_t g = chunks < most ? chunks : most;
  *warps = 1;
  while (*warps < kRedWarps && chunks > g * *warps) *warps *= 2;
  return (int)g;
}
constexpr int z_chunk_bits(size_t amp_bytes) { return amp_bytes == 8 ? 11 : 10; }

size_t expect_z_batch_scratch_doubles(int n, int batch, size_t amp_bytes) {
  int warps = 0;
  return (size_t)batch * z_all_blocks(n, z_chunk_bits(amp_bytes), batch, &warps) * (n + 1);
}

template <typename R>
cudaError_t launch_expect_z_batch(const Cx<R>* states, int n, int batch, double* scratch, size_t scratch_doubles,
                                  double* out, cudaStream_t stream) {
  constexpr int C = z_chunk_bits(sizeof(Cx<R>));
  int warps = 0;
  const int grid = z_all_blocks(n, C, batch, &warps);
  if ((size_t)batch * grid * (n + 1) > scratch_doubles) return cudaErrorInvalidValue;
  if (n < C)
    k_expect_z_small<R><<<batch, kRedThreads, 0, stream>>>(states, n, scratch);
  else
    k_expect_z_all<R><<<dim3((unsigned)grid, (unsigned)batch), 32 * warps, 0, stream>>>(states, n, scratch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_finish_z_all<<<batch, grid >= 32 ? 1024 : 32 * grid, 0, stream>>>(scratch, grid, n, out);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_expect_z_all(const Cx<R>* state, int n, double* scratch, size_t scratch_doubles, double* out,
                                cudaStream_t stream) {
  return launch_expect_z_batch<R>(state, n, 1, scratch, scratch_doubles, out, stream);
}

namespace {

// The passes of one accumulator count, launched in groups of what fits the
// kernel's parameters.
template <typename R, int NT, bool PAIRED, bool IMAG>
cudaError_t launch_term_passes(const Cx<R>* state, int n, const std::vector<TermPass<kMaxTermsPerPass>>& list,
                               int grid, double* scratch, cudaStream_t stream) {
  TermPasses<NT> tp;
  for (size_t at = 0; at < list.size();) {
    int k = 0;
    for (; at < list.size() && k < kPassesPerLaunch<NT>; at++, k++) {
      const TermPass<kMaxTermsPerPass>& p = list[at];
      TermPass<NT>& d = tp.p[k];
      d.x = p.x;
      d.h = p.h;
      d.slot = p.slot;
      d.nt = p.nt;
      for (int j = 0; j < NT; j++) d.z[j] = j < p.nt ? p.z[j] : 0ull;
    }
    k_expect_terms<R, NT, PAIRED, IMAG><<<dim3((unsigned)grid, (unsigned)k), kRedThreads, 0, stream>>>(state, n, tp, scratch);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename R, bool PAIRED, bool IMAG>
cudaError_t launch_terms_by_count(const Cx<R>* state, int n, const std::vector<TermPass<kMaxTermsPerPass>>& list,
                                  int grid, double* scratch, cudaStream_t stream) {
  std::vector<TermPass<kMaxTermsPerPass>> by[5];  // 1, 2, 3..4, 5..8, 9..16 terms
  for (const TermPass<kMaxTermsPerPass>& p : list) by[p.nt <= 1 ? 0 : p.nt <= 2 ? 1 : p.nt <= 4 ? 2 : p.nt <= 8 ? 3 : 4].push_back(p);
  cudaError_t e = launch_term_passes<R, 1, PAIRED, IMAG>(state, n, by[0], grid, scratch, stream);
  if (e == cudaSuccess) e = launch_term_passes<R, 2, PAIRED, IMAG>(state, n, by[1], grid, scratch, stream);
  if (e == cudaSuccess) e = launch_term_passes<R, 4, PAIRED, IMAG>(state, n, by[2], grid, scratch, stream);
  if (e == cudaSuccess) e = launch_term_passes<R, 8, PAIRED, IMAG>(state, n, by[3], grid, scratch, stream);
  if (e == cudaSuccess) e = launch_term_passes<R, 16, PAIRED, IMAG>(state, n, by[4], grid, scratch, stream);
  return e;
}

int term_grid(uint64_t count) {
  const uint64_t g = (count + kRedThreads - 1) / kRedThreads;
  return (int)(g < (uint64_t)red_grid() ? g : (uint64_t)red_grid());
}

}  // namespace

template <typename R>
cudaError_t launch_expect_terms(const Cx<R>* state, int n, const sv_pauli_term* terms, int n_terms, double* scratch,
                                size_t scratch_doubles, double* out, cudaStream_t stream) {
  if ((size_t)red_grid() * kMaxTermSlots > scratch_doubles) return cudaErrorInvalidValue;
  const int grid_z = term_grid(1ull << n), grid_x = term_grid(1ull << (n - 1));
  std::vector<TermPass<kMaxTermsPerPass>> lists[3];  // no X mask; real part; imaginary part
  TermOut to[3] = {};
  int slots[3] = {0, 0, 0};
  // runs what has been collected of one kind and writes its terms' values
  auto flush = [&](int kind) -> cudaError_t {
    if (!slots[kind]) return cudaSuccess;
    const int grid = kind ? grid_x : grid_z;
    cudaError_t e = kind == 0   ? launch_terms_by_count<R, false, false>(state, n, lists[0], grid, scratch, stream)
                    : kind == 1 ? launch_terms_by_count<R, true, false>(state, n, lists[1], grid, scratch, stream)
                                : launch_terms_by_count<R, true, true>(state, n, lists[2], grid, scratch, stream);
    if (e != cudaSuccess) return e;
    k_finish_terms<<<slots[kind], 128, 0, stream>>>(scratch, grid, to[kind], out);
    lists[kind].clear();
    slots[kind] = 0;
    return cudaGetLastError();
  };
  // terms by kind and X mask, in the order of each mask's first term
  std::map<std::pair<uint64_t, int>, int> first;
  std::vector<std::vector<int>> groups;
  auto kind_of = [&](int t) {
    const uint64_t x = terms[t].x_mask;
    return !x ? 0 : 1 + (__builtin_popcountll(x & terms[t].z_mask) & 1);
  };
  for (int t = 0; t < n_terms; t++) {
    const auto at = first.emplace(std::make_pair(terms[t].x_mask, kind_of(t)), (int)groups.size());
    if (at.second) groups.emplace_back();
    groups[at.first->second].push_back(t);
  }
  for (const std::vector<int>& g : groups) {
    const uint64_t x = terms[g[0]].x_mask;
    const int kind = kind_of(g[0]);
    for (size_t k = 0; k < g.size();) {
      const int nt = (int)std::min<size_t>(kMaxTermsPerPass, g.size() - k);
      if (slots[kind] + nt > kMaxTermSlots) {
        const cudaError_t e = flush(kind);
        if (e != cudaSuccess) return e;
      }
      TermPass<kMaxTermsPerPass> p{};
      p.x = x;
      p.h = x ? 63 - __builtin_clzll(x) : 0;
      p.slot = slots[kind];
      p.nt = nt;
      for (int j = 0; j < nt; j++, k++) {
        const uint64_t z = terms[g[k]].z_mask;
        p.z[j] = z;
        to[kind].dst[p.slot + j] = (uint16_t)g[k];
        to[kind].how[p.slot + j] = (uint8_t)((__builtin_popcountll(x & z) & 3) | (kind ? 4 : 0));
      }
      slots[kind] += nt;
      lists[kind].push_back(p);
    }
  }
  for (int kind = 0; kind < 3; kind++) {
    const cudaError_t e = flush(kind);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template cudaError_t launch_expect_z_all<float>(const Cx<float>*, int, double*, size_t, double*, cudaStream_t);
template cudaError_t launch_expect_z_all<double>(const Cx<double>*, int, double*, size_t, double*, cudaStream_t);
template cudaError_t launch_expect_z_batch<float>(const Cx<float>*, int, int, double*, size_t, double*, cudaStream_t);
template cudaError_t launch_expect_z_batch<double>(const Cx<double>*, int, int, double*, size_t, double*,
                                                   cudaStream_t);
template cudaError_t launch_expect_terms<float>(const Cx<float>*, int, const sv_pauli_term*, int, double*, size_t,
                                                double*, cudaStream_t);
template cudaError_t launch_expect_terms<double>(const Cx<double>*, int, const sv_pauli_term*, int, double*, size_t,
                                                 double*, cudaStream_t);

}  // namespace sv
