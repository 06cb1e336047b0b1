// sv_sample.cu -- measurement: the probability vector and finite-shot draws
// (Sec. 5.3: p_i = x_i^2 + y_i^2 for psi_i = x_i + i y_i, normalised on the
// device; a finite-shot run draws basis indices from it).
//
// Draws use exact integer arithmetic so that they do not depend on the order
// of any floating-point sum (a blocked GPU sum and a sequential one agree bit
// for bit):
//   q_i = floor(p_i 2^61), p_i = x_i^2 + y_i^2 in double with each product
//         and the sum rounded once (no fused multiply-add),
//   Q   = sum_i q_i,
//   t_k = floor(floor(u_k 2^53) Q / 2^53) for the caller's uniform u_k,
//   index_k = the smallest i with q_0 + ... + q_i > t_k.
// The state is cut into chunks of 128 amplitudes (more on states above 30
// qubits, so that the table stays at 64 MB): one pass sums q per chunk, a scan
// turns the sums into their prefix in place, and a shot finds its chunk by
// binary search over the prefix and its index by a warp scan inside it.
//
// complex64 forms p_i in integers: this part runs one FP64 warp instruction in
// about 16 cycles, and the two conversions, two products, sum, scaling and
// integer conversion of q_i bound every kernel here (28 qubits, 2^20 shots:
// 3.5 ms of chunk sums and 21.4 ms of draws, which also walked 1024
// amplitudes a shot).  The squares of two 24-bit mantissas and their sum are a
// few dozen integer instructions with the same bits: 0.50 ms of sums (HBM alone
// 0.32) and 0.52 ms of draws, both bound by the integer pipe.
#include <cuda_runtime.h>

#include <cstring>
#include <vector>

#include "sv_internal.h"

namespace sv {
namespace {

constexpr int kChunkLog = 7;      // amplitudes per chunk: 128 = 32 lanes x 4
constexpr int kTableLogMax = 23;  // chunks of a state at most
int chunk_log_for(int n) {
  const int cl = n < kChunkLog ? n : kChunkLog;
  return n - cl > kTableLogMax ? n - kTableLogMax : cl;
}

__device__ __forceinline__ uint32_t magnitude(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t mantissa(uint32_t mag) { return (mag & 0x7fffffu) | 0x800000u; }

// p = x^2 + y^2 from the magnitudes' bits bh >= bl, bh a normal number, bl a
// normal number or 0: rounded once to 53 bits, as m * 2^(e - 52) with m in
// [2^52, 2^53].  With both squares shifted up by 15 the larger one holds 61
// to 63 bits; the smaller one, shifted down by the difference of the
// exponents, loses only bits below the rounding position, and whether it lost
// any is kept in bit 0.
__device__ __forceinline__ uint64_t square_sum(uint32_t bh, uint32_t bl, int& e) {
  const int eh = (int)(bh >> 23), el = (int)(bl >> 23);
  const uint32_t mh = mantissa(bh), ml = bl ? mantissa(bl) : 0u;
  const uint64_t a = (uint64_t)(mh << 8) * (mh << 7), b = (uint64_t)(ml << 8) * (ml << 7);  // squares << 15
  const int d = min(2 * (eh - el), 63);
  const uint64_t low = b >> d;
  uint64_t s = a + low;
  s |= (low << d) != b ? 1ull : 0ull;
  const int lz = __clz((int)(s >> 32));  // 0..2
  e = 2 * eh - 252 - lz;                 // s << lz has bit 63 set: p = (s << lz) * 2^(e - 63)
  s <<= lz;
  const uint64_t m = s >> 11;
  return m + (((uint32_t)s & 0x7ffu) + ((uint32_t)m & 1u) > 0x400u ? 1ull : 0ull);
}

// The same in FP64, and q from it.  Not inlined: a predicated-off FP64
// instruction still takes its slot in the FP64 pipe (inlined, the rare cases
// below cost the common one five such slots an amplitude).
__device__ __noinline__ double p_fp64(float re, float im) {
  const double x = (double)re, y = (double)im;
  return __dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y));
}
__device__ __forceinline__ uint64_t q_of_p(double p) {
  return __double2ull_rz(__dmul_rn(p, 2305843009213693952.0));  // p * 2^61, exact scaling
}
__device__ __noinline__ uint64_t q_fp64(float re, float im) { return q_of_p(p_fp64(re, im)); }

// p_i as a double.  FP64 for infinities, NaN and subnormal parts (of which
// the larger magnitude is 0 only when p is).
__device__ __forceinline__ double p_of(const Cx<float>& a) {
  const uint32_t x = magnitude(a.re), y = magnitude(a.im);
  const uint32_t bh = max(x, y), bl = min(x, y);
  if (bh >= 0x7f800000u || bl - 1u < 0x7fffffu || bh - 1u < 0x7fffffu) return p_fp64(a.re, a.im);
  int e;
  const uint64_t m = square_sum(bh, bl, e);  // a carry into 2^53 steps the exponent field
  return bh ? __longlong_as_double((long long)(((uint64_t)(1022 + e) << 52) + m)) : 0.0;
}
__device__ __forceinline__ double p_of(const Cx<double>& a) {
  return __dadd_rn(__dmul_rn(a.re, a.re), __dmul_rn(a.im, a.im));
}

// q_i.  Magnitudes below 2^-12 (p < 2^-23, q < 2^38; a deep circuit's state of
// 24 qubits and more) skip the rounding: RN53(p) 2^61 passes the next whole
// number only when the 15 bits below it are all ones, so otherwise q is the
// plain shift of the sum.  (A subnormal or zero part may take the implicit
// bit: its square is below 2^-250 either way.)
__device__ __forceinline__ uint64_t q_of(const Cx<double>& a) { return q_of_p(p_of(a)); }
__device__ __forceinline__ uint64_t q_of(const Cx<float>& a) {
  const uint32_t x = magnitude(a.re), y = magnitude(a.im);
  const uint32_t bh = max(x, y), bl = min(x, y);
  if (bh < (115u << 23)) {
    const int eh = (int)(bh >> 23), el = (int)(bl >> 23);
    const uint32_t mh = mantissa(bh) << 7, ml = mantissa(bl) << 7;
    const uint64_t s = (uint64_t)mh * mh + (((uint64_t)ml * ml) >> min(2 * (eh - el), 63));  // < 2^63
    const uint64_t t = s >> (min(253 - 2 * eh, 63) - 15);  // s * 2^(2 eh - 314) in units of 2^-61, and 15 bits more
    if ((t & 0x7fffu) != 0x7fffu) return t >> 15;
  }
  // |x| >= 2: q may pass 2^64 (saturates); infinities, NaN, subnormal parts
  if (bh >= 0x40000000u || bl - 1u < 0x7fffffu || bh - 1u < 0x7fffffu) return q_fp64(a.re, a.im);
  int e;
  const uint64_t m = square_sum(bh, bl, e);  // p < 8: q < 2^64
  const int up = e + 9;                      // q = floor(m * 2^(e - 52 + 61))
  return !bh ? 0ull : up >= 0 ? m << min(up, 63) : m >> min(-up, 63);
}

// Amplitudes i and i + 1 in one 16-byte load (complex64; i even).
__device__ __forceinline__ void load2(const Cx<float>* a, Cx<float>& u, Cx<float>& v) {
  const float4 w = __ldg(reinterpret_cast<const float4*>(a));
  u = {w.x, w.y};
  v = {w.z, w.w};
}
__device__ __forceinline__ void load2(const Cx<double>* a, Cx<double>& u, Cx<double>& v) {
  const double2 p = __ldg(reinterpret_cast<const double2*>(a)), q = __ldg(reinterpret_cast<const double2*>(a) + 1);
  u = {p.x, p.y};
  v = {q.x, q.y};
}

// Sum of q over a lane's segment of 2^seg_log consecutive amplitudes.
template <typename R>
__device__ __forceinline__ uint64_t segment_sum(const Cx<R>* a, int seg_log) {
  if (seg_log == 0) return q_of(a[0]);
  uint64_t s = 0;
#pragma unroll 2
  for (int i = 0; i < (1 << seg_log); i += 2) {
    Cx<R> u, v;
    load2(a + i, u, v);
    s += q_of(u) + q_of(v);
  }
  return s;
}

__device__ __forceinline__ uint64_t warp_sum(uint64_t s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
__device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// q sums per chunk, a warp per chunk; a block takes `per` consecutive chunks
// and leaves their total for the scan.
template <typename R>
__global__ void __launch_bounds__(256) k_chunk_sums(const Cx<R>* __restrict__ psi, uint64_t nchunks, int chunk_log,
                                                    uint64_t per, uint64_t* __restrict__ sums,
                                                    uint64_t* __restrict__ totals) {
  __shared__ uint64_t part[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int seg_log = chunk_log - 5;
  const uint64_t b = blockIdx.x * per, e = b + per < nchunks ? b + per : nchunks;
  uint64_t total = 0;
  if (chunk_log == kChunkLog) {  // the usual width, unrolled: the next chunk's loads overlap this one's sums
#pragma unroll 2
    for (uint64_t c = b + warp; c < e; c += 8) {
      const Cx<R>* a = psi + (c << kChunkLog) + 4 * lane;
      Cx<R> v[4];
      load2(a, v[0], v[1]);
      load2(a + 2, v[2], v[3]);
      const uint64_t s = warp_sum((q_of(v[0]) + q_of(v[1])) + (q_of(v[2]) + q_of(v[3])));
      if (lane == 0) sums[c] = s;
      total += s;
    }
  } else {
    for (uint64_t c = b + warp; c < e; c += 8) {
      const uint64_t s = warp_sum(segment_sum(psi + (c << chunk_log) + ((uint64_t)lane << seg_log), seg_log));
      if (lane == 0) sums[c] = s;
      total += s;
    }
  }
  if (lane == 0) part[warp] = total;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t s = 0;
    for (int w = 0; w < 8; w++) s += part[w];
    totals[blockIdx.x] = s;
  }
}

// Exclusive prefix of the chunk sums, in place; pre[n] = Q.  Block b adds the
// totals of the blocks before it, then scans its own `per` chunks, 1024 at a
// time.  (One CTA scanning all sums took 0.44 ms at 28 qubits.)
__global__ void __launch_bounds__(256) k_scan_chunks(uint64_t* __restrict__ pre, uint64_t n, uint64_t per,
                                                     const uint64_t* __restrict__ totals) {
  __shared__ uint64_t part[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t s = 0;
  for (unsigned i = threadIdx.x; i < blockIdx.x; i += 256) s += totals[i];
  s = warp_sum(s);
  if (lane == 0) part[warp] = s;
  __syncthreads();
  uint64_t run = 0;  // the prefix of the tile's first chunk
  for (int w = 0; w < 8; w++) run += part[w];
  const uint64_t b = blockIdx.x * per, e = b + per < n ? b + per : n;
  for (uint64_t t = b; t < e; t += 1024) {
    const uint64_t i0 = t + 4 * threadIdx.x;
    uint64_t v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      v[k] = i0 + k < e ? pre[i0 + k] : 0;
      sum += v[k];
    }
    uint64_t inc = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    __syncthreads();  // part[] is free
    if (lane == 31) part[warp] = inc;
    __syncthreads();
    uint64_t at = run + inc - sum;
    for (int w = 0; w < 8; w++) {
      if (w < warp) at += part[w];
      run += part[w];
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (i0 + k < e) pre[i0 + k] = at;
      at += v[k];
    }
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) pre[n] = run;
}

// A warp takes `group` shots (1..32): lane k finds the chunk of shot k by
// binary search, then the warp walks the shots' chunks together.  A search
// step is a dependent read of the prefix table; done by one lane a shot, 32
// of them overlap.
template <typename R>
__global__ void __launch_bounds__(256) k_draw(const Cx<R>* __restrict__ psi, const uint64_t* __restrict__ pre,
                                              uint64_t nchunks, int chunk_log, const double* __restrict__ u,
                                              uint64_t nshots, int group, uint64_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  const int seg_log = chunk_log - 5;
  const uint64_t Q = pre[nchunks];
  for (uint64_t k0 = (blockIdx.x * (uint64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)) * group; k0 < nshots;
       k0 += warps * group) {
    const int shots = nshots - k0 < (uint64_t)group ? (int)(nshots - k0) : group;
    uint64_t chunk = 0, left = 0;
    if (lane < shots) {
      const uint64_t m = __double2ull_rz(__dmul_rn(u[k0 + lane], 9007199254740992.0));  // floor(u 2^53)
      const uint64_t lo = m * Q, hi = __umul64hi(m, Q);
      const uint64_t t = (hi << 11) | (lo >> 53);  // floor(m Q / 2^53) < Q
      // the chunk c with pre[c] <= t < pre[c + 1]
      uint64_t a = 0, b = nchunks - 1;
      while (a < b) {
        const uint64_t mid = (a + b + 1) >> 1;
        if (pre[mid] <= t)
          a = mid;
        else
          b = mid - 1;
      }
      chunk = a;
      left = t - pre[a];
    }
    for (int k = 0; k < shots; k++) {
      const uint64_t c = __shfl_sync(0xffffffffu, chunk, k), r = __shfl_sync(0xffffffffu, left, k);
      // lane segments of 2^(chunk_log - 5) amplitudes, scanned across the warp
      const uint64_t at = (c << chunk_log) + ((uint64_t)lane << seg_log);
      const Cx<R>* base = psi + at;
      const uint64_t s = segment_sum(base, seg_log);
      uint64_t inc = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      uint64_t run = inc - s;
      if (run <= r && r < inc) {  // this lane's segment holds the index
        int i = 0;
        for (; i < (1 << seg_log) - 1; i++) {
          run += q_of(base[i]);
          if (run > r) break;
        }
        out[k0 + k] = at + (uint64_t)i;
      }
    }
  }
}

// p_i of two amplitudes per thread and step, times *scale when SCALED (a
// template: a multiply predicated off still takes its slot in the FP64 pipe,
// which bounds complex128: 25 qubits raw 271 us with it, 211 without).
template <typename R, bool SCALED>
__global__ void __launch_bounds__(256) k_probs(const Cx<R>* __restrict__ psi, uint64_t pairs,
                                               const double* __restrict__ scale, double* __restrict__ p) {
  const double f = SCALED ? *scale : 1.0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < pairs; i += stride) {
    Cx<R> u, v;
    load2(psi + 2 * i, u, v);
    double2 w = make_double2(p_of(u), p_of(v));
    if constexpr (SCALED) w = make_double2(w.x * f, w.y * f);
    *reinterpret_cast<double2*>(p + 2 * i) = w;
  }
}

// Partial sums of p in double, one per block.
template <typename R>
__global__ void __launch_bounds__(256) k_psum(const Cx<R>* __restrict__ psi, uint64_t pairs,
                                              double* __restrict__ part) {
  __shared__ double red[8];
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  double s = 0.0;
#pragma unroll 4
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < pairs; i += stride) {
    Cx<R> u, v;
    load2(psi + 2 * i, u, v);
    s += p_of(u) + p_of(v);
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; w++) t += red[w];
    part[blockIdx.x] = t;
  }
}

// The factor that normalises: 1 / (sum of the partials), or 1 when the sum is
// not positive.
__global__ void __launch_bounds__(1024) k_psum_final(const double* __restrict__ part, int n,
                                                     double* __restrict__ scale) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[w];
    *scale = t > 0.0 ? 1.0 / t : 1.0;
  }
}

unsigned grid_for(uint64_t work_items, int per_block) {
  uint64_t g = (work_items + per_block - 1) / per_block;
  const uint64_t cap = (uint64_t)device_sm_count() * 8;
  if (g > cap) g = cap;
  return (unsigned)(g ? g : 1);
}

// Normalised: one pass sums p over the state, a second writes p times the
// factor (24 bytes an amplitude; writing p, summing it and scaling it in place
// moved 40).  26 qubits, complex64: 0.19 + 0.21 ms (FP64 adds and integer
// pipe; HBM alone 0.08 + 0.16), 1.02 ms before.
template <typename R>
void probabilities(const Cx<R>* psi, int n, double* p, bool normalise, cudaStream_t s) {
  const uint64_t pairs = 1ull << (n - 1);
  double* scale = nullptr;
  if (normalise) {
    const unsigned grid = grid_for(pairs, 256);
    double* part = (double*)scratch_buffer(s, "prob_partials", sizeof(double) * ((size_t)device_sm_count() * 8 + 1));
    scale = part + grid;
    k_psum<R><<<grid, 256, 0, s>>>(psi, pairs, part);
    k_psum_final<<<1, 1024, 0, s>>>(part, (int)grid, scale);
  }
  if (scale)
    k_probs<R, true><<<grid_for(pairs, 256), 256, 0, s>>>(psi, pairs, scale, p);
  else
    k_probs<R, false><<<grid_for(pairs, 256), 256, 0, s>>>(psi, pairs, scale, p);
  cuda_check(cudaGetLastError(), "probabilities");
}

template <typename R>
void sample(const Cx<R>* psi, int n, const double* u_host, size_t nshots, uint64_t* out, bool out_on_device,
            cudaStream_t s) {
  const int cl = chunk_log_for(n);
  if (cl < 5) fail(SV_ERR_UNSUPPORTED, "sampling needs n_qubits >= 5 (32-amplitude lane segments)");
  const uint64_t nch = 1ull << (n - cl);
  const unsigned grid = grid_for(nch, 8);
  const uint64_t per = (nch + grid - 1) / grid;  // chunks of a block
  uint64_t* pre = (uint64_t*)scratch_buffer(s, "sample_sums", sizeof(uint64_t) * (nch + 1 + grid));
  uint64_t* totals = pre + nch + 1;
  double* du = (double*)scratch_buffer(s, "sample_u", sizeof(double) * nshots);
  uint64_t* dout = out_on_device ? out : (uint64_t*)scratch_buffer(s, "sample_out", sizeof(uint64_t) * nshots);
  k_chunk_sums<R><<<grid, 256, 0, s>>>(psi, nch, cl, per, pre, totals);
  k_scan_chunks<<<grid, 256, 0, s>>>(pre, nch, per, totals);
  cuda_check(cudaMemcpyAsync(du, u_host, sizeof(double) * nshots, cudaMemcpyHostToDevice, s), "uniforms upload");
  // shots per warp: enough warps to fill the chip first, then up to 32
  const uint64_t fill = (uint64_t)device_sm_count() * 64;
  int group = 1;
  while (group < 32 && nshots > fill * group) group *= 2;
  const uint64_t shot_groups = (nshots + group - 1) / group;
  k_draw<R><<<grid_for(shot_groups, 8), 256, 0, s>>>(psi, pre, nch, cl, du, nshots, group, dout);
  cuda_check(cudaGetLastError(), "draw");
  uint64_t Q = 0;
  cuda_check(cudaMemcpyAsync(&Q, pre + nch, sizeof(Q), cudaMemcpyDeviceToHost, s), "total read");
  cuda_check(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  if (Q == 0) fail(SV_ERR_INVALID, "the state has no probability mass above 2^-61");  // nothing was drawn
  if (!out_on_device) {
    cuda_check(cudaMemcpyAsync(out, dout, sizeof(uint64_t) * nshots, cudaMemcpyDeviceToHost, s), "result read");
    cuda_check(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  }
}

}  // namespace
}  // namespace sv

using namespace sv;

extern "C" sv_status sv_probabilities(const void* state, int n_qubits, sv_dtype dtype, double* out, int normalise,
                                      void* stream) {
  return guarded([&] {
    if (dtype != SV_C64 && dtype != SV_C128) fail(SV_ERR_INVALID, "unknown dtype");
    if (n_qubits < 1 || n_qubits > SV_MAX_QUBITS) fail(SV_ERR_INVALID, "n_qubits must be in 1..34");
    const size_t amp = dtype == SV_C64 ? 8 : 16;
    check_device_buffer(state, amp << n_qubits, "state");
    check_device_buffer(out, sizeof(double) << n_qubits, "out");
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == SV_C64)
      probabilities<float>((const Cx<float>*)state, n_qubits, out, normalise != 0, s);
    else
      probabilities<double>((const Cx<double>*)state, n_qubits, out, normalise != 0, s);
  });
}

extern "C" sv_status sv_sample(const void* state, int n_qubits, sv_dtype dtype, const double* uniforms,
                               size_t n_shots, uint64_t* out, int out_on_device, void* stream) {
  return guarded([&] {
    if (dtype != SV_C64 && dtype != SV_C128) fail(SV_ERR_INVALID, "unknown dtype");
    if (n_qubits < 5 || n_qubits > SV_MAX_QUBITS) fail(SV_ERR_INVALID, "n_qubits must be in 5..34");
    if (n_shots == 0) return;
    if (!uniforms || !out) fail(SV_ERR_INVALID, "uniforms or out is NULL");
    int bad = 0;  // no early exit, so that the check runs as vector code
    for (size_t k = 0; k < n_shots; k++) bad |= !(uniforms[k] >= 0.0) | !(uniforms[k] < 1.0);
    if (bad) fail(SV_ERR_INVALID, "uniforms must lie in [0, 1)");
    const size_t amp = dtype == SV_C64 ? 8 : 16;
    check_device_buffer(state, amp << n_qubits, "state");
    if (out_on_device) check_device_buffer(out, sizeof(uint64_t) * n_shots, "out");
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == SV_C64)
      sample<float>((const Cx<float>*)state, n_qubits, uniforms, n_shots, out, out_on_device != 0, s);
    else
      sample<double>((const Cx<double>*)state, n_qubits, uniforms, n_shots, out, out_on_device != 0, s);
  });
}
