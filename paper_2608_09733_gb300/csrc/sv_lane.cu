// sv_lane.cu -- the pass kernel of small states for sm_103a: a tile of up to
// 2^14 amplitudes spread over the shared memories of a thread-block cluster,
// one amplitude per lane.
//
// The pass kernels of sv_sweep.cu give a tile to one CTA and 16 or 32
// amplitudes to a thread, which is what a state of many tiles wants.  A state
// of one or a few tiles then runs on one or a few SMs, each thread working
// through its amplitudes one after the other: 12 qubits in complex128 took
// 690 us for 350 gates on two SMs.  What bounds it is the serial chain -- a
// warp's FP64 instruction occupies its scheduler's FP64 pipe for about 73
// cycles whatever the warp holds, so 16 amplitudes a thread put 16 of them in
// a row -- and that the other SMs hold nothing.
//
// Here the five register qubits of a phase (the program format of sv_program,
// rq = 5) sit in the lane index instead: a gate's partner amplitude comes by a
// warp shuffle, a warp holds one group of 32 amplitudes (A groups, for the
// larger tiles, to share the decoding of the ops), and the groups spread over
// up to 16 SMs.  A phase reads its amplitudes from the cluster's shared memory
// (wherever their home slice is), applies its ops and writes them back to the
// same places; one cluster barrier a phase.  Every CTA of a cluster meets
// every barrier: which phases and ops run depends on the program and the tile
// only, and a skipped op skips no barrier.  The program is staged into shared
// memory and each op's descriptor is loaded one op ahead.
//
// Measured (us a circuit, one CTA a tile -> here): 12 qubits complex128, ten
// RY/RZ/CNOT layers 690 -> 162; 14 qubits, 20 layers of U3 and CZ 811 -> 542;
// complex64, U3 and CNOT ladder of depth 22 on 15 qubits 465 -> 303; 200 one-
// and 100 two-qubit random matrices on 13 qubits 476 -> 77 (joined matrices,
// two passes).  A pass of the 12-qubit ansatz (36 us, 16 SMs of two warps a
// scheduler) issues an instruction of each warp every 11 cycles (4.8 of them
// wait for shared-memory round trips of shuffles and operands, 2.9 for fixed
// latencies), its FP64 pipe 44 % busy: the serial chain still bounds it.
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>

#include "sv_internal.h"
#include "sv_pass_ops.cuh"
#include "sv_stage.cuh"

namespace sv {
namespace {

constexpr int kLaneWarps = 8;       // warps of a CTA at most
constexpr int kLaneClusterLog = 4;  // CTAs of a cluster at most: 16

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ Cx<float> ld_peer(uint32_t a, float) {
  Cx<float> v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.re), "=f"(v.im) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ Cx<double> ld_peer(uint32_t a, double) {
  Cx<double> v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.re), "=d"(v.im) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer(uint32_t a, const Cx<float>& v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.re), "f"(v.im) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, const Cx<double>& v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.re), "d"(v.im) : "memory");
}
__device__ __forceinline__ void tile_sync(int log_c) {
  if (log_c == 0) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
}

// Slot of local amplitude l: the index of its 16-byte (complex128) or 8-byte
// slot within a wavefront is XORed with every higher group of as many bits, so
// lanes that differ in any run of consecutive local bits reach different banks.
template <typename R>
__device__ __forceinline__ uint32_t lane_slot(uint32_t l) {
  if constexpr (sizeof(R) == 4)
    return l ^ (((l >> 4) ^ (l >> 8) ^ (l >> 12)) & 15u);
  else
    return l ^ (((l >> 3) ^ (l >> 6) ^ (l >> 9) ^ (l >> 12)) & 7u);
}

template <typename R>
__device__ __forceinline__ Cx<R> shfl_partner(const Cx<R>& v, int mask) {
  return Cx<R>{__shfl_xor_sync(0xffffffffu, v.re, mask), __shfl_xor_sync(0xffffffffu, v.im, mask)};
}
template <typename R>
__device__ __forceinline__ R negate_if(R x, bool neg) {
  return neg ? -x : x;
}

// An op's descriptor in registers (the words of DevOp), loaded one op ahead:
// the fields of an op read one by one from shared memory cost more than its
// arithmetic on one amplitude.
struct OpWords {
  uint4 a, b, c, d;
  __device__ __forceinline__ void load(const DevOp& op) {
    const uint4* p = reinterpret_cast<const uint4*>(&op);
    a = p[0];
    b = p[1];
    c = p[2];
    d = p[3];
  }
  __device__ __forceinline__ uint32_t k() const { return (a.x >> 8) & 255u; }
  __device__ __forceinline__ uint32_t pos(int i) const { return (a.x >> (16 + 8 * i)) & 255u; }  // i < 2
  __device__ __forceinline__ uint32_t gq(int i) const { return (a.w >> (8 * i)) & 255u; }         // i < 4
  __device__ __forceinline__ uint32_t rs(int i) const {  // i < 5
    return (i < 3 ? b.x >> (8 + 8 * i) : b.y >> (8 * (i - 3))) & 255u;
  }
  __device__ __forceinline__ uint32_t lmask() const { return b.z; }
  __device__ __forceinline__ uint32_t lval() const { return b.w; }
  __device__ __forceinline__ uint32_t tmask() const { return c.x; }
  __device__ __forceinline__ uint32_t tval() const { return c.y; }
  __device__ __forceinline__ uint64_t xmask() const { return c.z | ((uint64_t)c.w << 32); }
  __device__ __forceinline__ uint64_t xval() const { return d.x | ((uint64_t)d.y << 32); }
  __device__ __forceinline__ uint32_t coef() const { return d.z; }
  __device__ __forceinline__ uint32_t code() const { return d.w; }
};
static_assert(offsetof(DevOp, k) == 1 && offsetof(DevOp, pos) == 2 && offsetof(DevOp, gq) == 12 &&
                  offsetof(DevOp, rs) == 17 && offsetof(DevOp, lmask) == 24 && offsetof(DevOp, lval) == 28 &&
                  offsetof(DevOp, tmask) == 32 && offsetof(DevOp, tval) == 36 &&
                  offsetof(DevOp, xmask) == 40 && offsetof(DevOp, xval) == 48 && offsetof(DevOp, coef) == 56 &&
                  offsetof(DevOp, pad) == 60,
              "OpWords reads DevOp by word");

// A dense matrix of three to five qubits, all on the lane's bits: the 2^k
// amplitudes of a group sit in one warp.  Row r (the lane's) times the group, by
// columns r ^ d in Gray-code order of d, so that each step's partner is one
// shuffle away and the lanes' coefficients M[r][r ^ d] lie in different banks.
// (Read one by one from the cluster's shared memory, 2^k round trips an
// amplitude, 100 gates as five-qubit blocks on 16 qubits took 1012 us in
// complex64, where the one-CTA pass takes 392.)
template <typename R, int A>
__device__ __forceinline__ void lane_dense(Cx<R> (&v)[A], const OpWords& op, const Cx<R>* cf, const uint32_t (&tb)[A],
                                           uint32_t tm, uint32_t tv, bool lane_on, uint32_t lane) {
  const int k = (int)op.k();
  uint32_t r = 0, slots = 0;  // slots: five bits a matrix bit
#pragma unroll
  for (int i = 0; i < 5; i++) {
    if (i >= k) continue;
    r |= ((lane >> op.rs(i)) & 1u) << i;
    slots |= op.rs(i) << (5 * i);
  }
  const Cx<R>* row = cf + (r << k);
  Cx<R> acc[A];
  const Cx<R> c0 = row[r];
#pragma unroll
  for (int a = 0; a < A; a++) acc[a] = cmul(c0, v[a]);
  uint32_t d = 0;
  int mask = 0;
  for (uint32_t step = 1; step < (1u << k); step++) {
    const int bit = __ffs((int)step) - 1;
    d ^= 1u << bit;
    mask ^= 1 << ((slots >> (5 * bit)) & 31u);
    const Cx<R> c = row[r ^ d];
#pragma unroll
    for (int a = 0; a < A; a++) acc[a] = cfma(c, shfl_partner(v[a], mask), acc[a]);
  }
#pragma unroll
  for (int a = 0; a < A; a++)
    if (lane_on && (tb[a] & tm) == tv) v[a] = acc[a];
}

// One register-phase op on the thread's A amplitudes: amplitude a is register
// combination `lane` of the group whose other local bits are tb[a].
template <typename R, int A>
__device__ __forceinline__ void lane_op(Cx<R> (&v)[A], const OpWords& op, const Cx<R>* pool, const uint32_t (&tb)[A],
                                        uint64_t base, uint32_t lane) {
  const uint32_t code = op.code();
  const uint32_t kind = code & 15u, fl = (code >> 4) & 7u;
  if ((fl & OPF_XCOND) && (base & op.xmask()) != op.xval()) return;  // same for the whole tile
  const Cx<R>* cf = pool + (code >> 17);
  const uint32_t rm = (code >> 7) & 31u, rv = (code >> 12) & 31u;
  const uint32_t tm = (fl & OPF_TCOND) ? op.tmask() : 0u, tv = (fl & OPF_TCOND) ? op.tval() : 0u;
  const bool lane_on = (lane & rm) == rv;  // controls on register slots (ops that have them)
  const uint32_t s0 = op.rs(0), s1 = op.rs(1);
  switch (kind) {
    case OPK_SIGN: {
      const bool neg = (op.coef() >> lane) & 1u;
#pragma unroll
      for (int a = 0; a < A; a++)
        if (neg && (tb[a] & tm) == tv) v[a] = {-v[a].re, -v[a].im};
      break;
    }
    case OPK_KROT: {
      Cx<R> c[5];
#pragma unroll
      for (int s = 0; s < 5; s++) c[s] = cf[s];
#pragma unroll
      for (int s = 0; s < 5; s++) {
        if (!((rm >> s) & 1u)) continue;
        const bool up = (lane >> s) & 1u;
        if constexpr (sizeof(R) == 4) {  // (tan(alpha/2), sin(alpha)): cos = 1 - sin tan(alpha/2)
          const R cs = fma(-c[s].im, c[s].re, R(1)), sn = negate_if(c[s].im, !up);
#pragma unroll
          for (int a = 0; a < A; a++) {
            const Cx<R> p = shfl_partner(v[a], 1 << s);
            v[a] = {fma(cs, v[a].re, sn * p.re), fma(cs, v[a].im, sn * p.im)};
          }
        } else {
          // clear: (a - t b, b + t a), own + (+-t) partner; set: (t a - b,
          // a + t b), t own +- partner
          const bool cot = (rv >> s) & 1u;
          const R t = c[s].re, st = negate_if(t, !up && !cot);
#pragma unroll
          for (int a = 0; a < A; a++) {
            const Cx<R> p = shfl_partner(v[a], 1 << s);
            const Cx<R> x = cot ? v[a] : p;
            const Cx<R> y = cot ? Cx<R>{negate_if(p.re, !up), negate_if(p.im, !up)} : v[a];
            v[a] = {fma(st, x.re, y.re), fma(st, x.im, y.im)};
          }
        }
      }
      break;
    }
    case OPK_PHASE: {
      const uint32_t k = op.k();
      uint32_t var[A];
#pragma unroll
      for (int a = 0; a < A; a++) var[a] = 0;
#pragma unroll
      for (int i = 0; i < 3; i++) {
        if (i >= k) continue;
        const uint32_t c = op.gq(i);
        const uint32_t x = (uint32_t)(base >> (c & 63u));
#pragma unroll
        for (int a = 0; a < A; a++) var[a] |= ((c < 64 ? tb[a] >> (c & 31u) : x) & 1u) << i;
      }
#pragma unroll
      for (int a = 0; a < A; a++) v[a] = cmul(cf[var[a] * (uint32_t)table_stride<R>(5) + lane], v[a]);
      break;
    }
    case OPK_KRON:
      for (int s = 0; s < 5; s++) {
        if (!((rm >> s) & 1u)) continue;
        const bool up = (lane >> s) & 1u;
        const Cx<R> own = cf[4 * s + (up ? 3 : 0)], oth = cf[4 * s + (up ? 2 : 1)];
#pragma unroll
        for (int a = 0; a < A; a++) {
          const Cx<R> p = shfl_partner(v[a], 1 << s);
          v[a] = cfma(oth, p, cmul(own, v[a]));
        }
      }
      break;
    case OPK_DENSE:
    case OPK_REAL:
      if (op.k() == 2) {
        const uint32_t r = ((lane >> s0) & 1u) | (((lane >> s1) & 1u) << 1);
        const Cx<R> u0 = cf[r * 4 + r], u1 = cf[r * 4 + (r ^ 1u)], u2 = cf[r * 4 + (r ^ 2u)],
                    u3 = cf[r * 4 + (r ^ 3u)];
#pragma unroll
        for (int a = 0; a < A; a++) {
          if ((tb[a] & tm) != tv) continue;
          const Cx<R> p1 = shfl_partner(v[a], 1 << s0), p2 = shfl_partner(v[a], 1 << s1),
                      p3 = shfl_partner(v[a], (1 << s0) | (1 << s1));
          Cx<R> o = cmul(u0, v[a]);
          o = cfma(u1, p1, o);
          o = cfma(u2, p2, o);
          o = cfma(u3, p3, o);
          if (lane_on) v[a] = o;
        }
      } else if (op.k() == 1) {
        const bool up = (lane >> s0) & 1u;
        const Cx<R> own = cf[up ? 3 : 0], oth = cf[up ? 2 : 1];
        const bool real = kind == OPK_REAL;
#pragma unroll
        for (int a = 0; a < A; a++) {
          if ((tb[a] & tm) != tv) continue;  // the same for the warp
          const Cx<R> p = shfl_partner(v[a], 1 << s0);
          Cx<R> o;
          if (real)
            o = {fma(own.re, v[a].re, oth.re * p.re), fma(own.re, v[a].im, oth.re * p.im)};
          else
            o = cfma(oth, p, cmul(own, v[a]));
          if (lane_on) v[a] = o;
        }
      } else {
        lane_dense<R, A>(v, op, cf, tb, tm, tv, lane_on, lane);
      }
      break;
    case OPK_ANTIDIAG: {
      const bool up = (lane >> s0) & 1u;
      if (fl & OPF_FLIP) {
#pragma unroll
        for (int a = 0; a < A; a++) {
          const bool on = (tb[a] & tm) == tv && lane_on;
          const Cx<R> p = shfl_partner(v[a], 1 << s0);
          v[a] = on ? p : v[a];
        }
      } else {
        const Cx<R> c = cf[up ? 1 : 0];
#pragma unroll
        for (int a = 0; a < A; a++) {
          if ((tb[a] & tm) != tv) continue;
          const Cx<R> p = cmul(c, shfl_partner(v[a], 1 << s0));
          if (lane_on) v[a] = p;
        }
      }
      break;
    }
    case OPK_PERM: {
      uint32_t from = op.lval();
#pragma unroll
      for (int q = 0; q < 5; q++) from ^= (lane >> q) & 1u ? (op.lmask() >> (5 * q)) & 31u : 0u;
      uint32_t src[A];
#pragma unroll
      for (int a = 0; a < A; a++) src[a] = from;
      const uint32_t k = op.k();
#pragma unroll
      for (int i = 0; i < 4; i++) {
        if (i >= k) continue;
        const uint32_t c = op.gq(i), v_i = op.rs(i);
        const uint32_t x = (uint32_t)(base >> (c & 63u));
#pragma unroll
        for (int a = 0; a < A; a++) src[a] ^= (c < 64 ? tb[a] >> (c & 31u) : x) & 1u ? v_i : 0u;
      }
#pragma unroll
      for (int a = 0; a < A; a++)
        v[a] = Cx<R>{__shfl_sync(0xffffffffu, v[a].re, src[a]), __shfl_sync(0xffffffffu, v[a].im, src[a])};
      break;
    }
    case OPK_SWAP: {
      const bool differ = ((lane >> s0) ^ (lane >> s1)) & 1u;
#pragma unroll
      for (int a = 0; a < A; a++) {
        if ((tb[a] & tm) != tv) continue;
        const Cx<R> p = shfl_partner(v[a], (1 << s0) | (1 << s1));
        if (lane_on && differ) v[a] = p;
      }
      break;
    }
    default: {  // OPK_DIAG, at most two matrix bits
      const uint32_t k = op.k();
#pragma unroll
      for (int a = 0; a < A; a++) {
        uint32_t d = 0;
#pragma unroll
        for (int i = 0; i < 2; i++) {
          if (i >= k) continue;
          const uint32_t b = op.rs(i) != 0xFF    ? lane >> op.rs(i)
                             : op.pos(i) != 0xFF ? tb[a] >> op.pos(i)
                                                 : (uint32_t)(base >> op.gq(i));
          d |= (b & 1u) << i;
        }
        if ((tb[a] & tm) != tv) continue;
        const Cx<R> o = cmul(cf[d], v[a]);
        if (lane_on) v[a] = o;
      }
    }
  }
}

// Local amplitude l under a shared-memory op: a diagonal of three to five
// qubits (dense blocks are register ops here).
template <typename R>
__device__ __forceinline__ Cx<R> wide_diagonal(const DevOp& op, const Cx<R>* cf, uint32_t l, uint64_t base,
                                               const Cx<R>& own) {
  if ((l & op.lmask) != op.lval) return own;
  uint32_t row = 0;  // the op's bits of l (bits outside the tile: fixed)
  for (int i = 0; i < op.k; i++)
    row |= (op.pos[i] != 0xFF ? (l >> op.pos[i]) & 1u : (uint32_t)(base >> op.gq[i]) & 1u) << i;
  return cmul(cf[row], own);
}

// One pass: cluster t of 2^log_c CTAs takes tile t.  A warp holds A groups of
// 32 amplitudes; warps x CTAs x A = 2^(m - 5).
template <typename R, int A>
__global__ void __launch_bounds__(32 * kLaneWarps)
    k_lane_pass(Cx<R>* __restrict__ state, const __grid_constant__ SweepProgram<R> param, int log_c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const ProgramHeader& h = param.h;
  const int log_s = h.m - log_c;  // this CTA's home slice holds 2^log_s amplitudes
  const uint32_t slice = 1u << log_s;
  Cx<R>* home = reinterpret_cast<Cx<R>*>(smem_raw);
  const SweepProgram<R>& P = stage_program<false>(param, home + slice);
  const Cx<R>* coef = P.coef;
  const uint32_t rank = log_c ? cluster_rank() : 0u;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const uint32_t first_group = (rank * warps + warp) * A;
  uint64_t base = blockIdx.x >> log_c;
  for (int i = 0; i < h.m; i++) base = ins0_64(base, h.tq[i]);
  const bool whole = h.m == h.n;
  auto global = [&](uint32_t i) {  // the state's index of the slice's amplitude i
    const uint32_t l = (rank << log_s) | i;
    return whole ? (uint64_t)l : base | tile_offset(l, h);
  };
  for (uint32_t i = threadIdx.x; i < slice; i += blockDim.x) home[lane_slot<R>((rank << log_s) | i) & (slice - 1u)] = state[global(i)];
  tile_sync(log_c);
  const uint32_t home_addr = smem_addr(home);
  auto addr_of = [&](uint32_t l) {
    const uint32_t at = home_addr + (lane_slot<R>(l) & (slice - 1u)) * (uint32_t)sizeof(Cx<R>);
    return log_c ? peer_addr(at, l >> log_s) : at;
  };
  for (int p = 0; p < h.nphases; p++) {
    const Phase& ph = P.ph[p];
    Cx<R> v[A];
    uint32_t at[A];
    if (ph.kind == PH_REG) {
      OpWords op;
      op.load(P.ops[ph.first]);
      // the lane's bits go to the register positions, the group's to the
      // others; the low bits of the group's index (its place among the warp's
      // A) to the first two of those
      uint32_t ll = 0, tb[A];
      tb[0] = first_group;
#pragma unroll
      for (int i = 0; i < 5; i++) {
        const int q = ph.rp[i];
        ll |= ((lane >> i) & 1u) << q;
        tb[0] = ins0(tb[0], q);
      }
#pragma unroll
      for (int a = 1; a < A; a++) tb[a] = tb[0] | ((a & 1u) << ph.tpos[0]) | ((a >> 1) << ph.tpos[1]);
#pragma unroll
      for (int a = 0; a < A; a++) {
        at[a] = addr_of(tb[a] | ll);
        v[a] = ld_peer(at[a], R(0));
      }
      const int last = ph.first + ph.nops;
      for (int o = ph.first; o < last; o++) {
        OpWords next;
        next.load(P.ops[o + 1 < last ? o + 1 : o]);
        lane_op<R, A>(v, op, coef, tb, base, lane);
        op = next;
      }
    } else {
      const DevOp& op = P.ops[ph.first];
      if ((base & op.xmask) != op.xval) continue;  // the whole cluster skips it
      const Cx<R>* cf = coef + op.coef;
#pragma unroll
      for (int a = 0; a < A; a++) {
        const uint32_t l = (first_group + a) * 32u + lane;
        at[a] = addr_of(l);
        v[a] = wide_diagonal<R>(op, cf, l, base, ld_peer(at[a], R(0)));
      }
    }
#pragma unroll
    for (int a = 0; a < A; a++) st_peer(at[a], v[a]);
    tile_sync(log_c);
  }
  for (uint32_t i = threadIdx.x; i < slice; i += blockDim.x) state[global(i)] = home[lane_slot<R>((rank << log_s) | i) & (slice - 1u)];
}

// How a tile of 2^m amplitudes is spread: CTAs (a power of two), warps per CTA
// and groups per warp, with CTAs x warps x groups = 2^(m - 5).
struct LaneShape {
  int log_c, warps, groups;
};
template <typename R>
LaneShape lane_shape(int m) {
  LaneShape s;
  const int v = m - 5;  // log2 of the tile's groups
  int lc = v - 3 > 0 ? v - 3 : 0;  // eight warps a CTA before the next CTA
  if (sizeof(R) == 8 && lc < (v + 1) / 2) lc = (v + 1) / 2;  // fewer: every scheduler has its own FP64 pipe
  if (lc > kLaneClusterLog) lc = kLaneClusterLog;
  int lg = v - lc - 3 > 0 ? v - lc - 3 : 0, lw = v - lc - lg;
  s.log_c = lc;
  s.warps = 1 << lw;
  s.groups = 1 << lg;
  return s;
}

template <typename R>
size_t lane_smem(int m, int log_c, int ncoef) {
  return (sizeof(Cx<R>) << (m - log_c)) + staged_bytes<R>(ncoef);
}

template <typename R, int A>
cudaError_t launch_lane(Cx<R>* state, const SweepProgram<R>& prog, const LaneShape& s, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(1ull << (prog.h.n - prog.h.m + s.log_c)));
  cfg.blockDim = dim3(32u * s.warps);
  cfg.dynamicSmemBytes = lane_smem<R>(prog.h.m, s.log_c, prog.h.ncoef);
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1u << s.log_c;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_lane_pass<R, A>, state, prog, s.log_c);
}

template <typename R, int A>
bool allow_clusters() {
  return cudaFuncSetAttribute(k_lane_pass<R, A>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
}

// Whether the device takes a cluster of 16 of these CTAs.
bool probe_clusters() {
  if (!(allow_clusters<float, 1>() && allow_clusters<float, 2>() && allow_clusters<float, 4>() &&
        allow_clusters<double, 1>() && allow_clusters<double, 2>() && allow_clusters<double, 4>())) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << kLaneClusterLog);
  cfg.blockDim = dim3(32u * kLaneWarps);
  cfg.dynamicSmemBytes = 48 * 1024;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1u << kLaneClusterLog;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_lane_pass<double, 4>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= 1;
}

}  // namespace

bool lane_pass_available() {
  static std::atomic<int> known[64];  // per device: 0 not asked, 1 yes, 2 no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return false;
  }
  int k = known[dev].load();
  if (!k) known[dev] = k = probe_clusters() ? 1 : 2;
  return k == 1 && !session_live(dev);
}

template <typename R>
cudaError_t launch_lane_pass(Cx<R>* state, const SweepProgram<R>& prog, cudaStream_t stream) {
  const LaneShape s = lane_shape<R>(prog.h.m);
  switch (s.groups) {
    case 1: return launch_lane<R, 1>(state, prog, s, stream);
    case 2: return launch_lane<R, 2>(state, prog, s, stream);
    case 4: return launch_lane<R, 4>(state, prog, s, stream);
    default: return cudaErrorInvalidConfiguration;
  }
}
template cudaError_t launch_lane_pass<float>(Cx<float>*, const SweepProgram<float>&, cudaStream_t);
template cudaError_t launch_lane_pass<double>(Cx<double>*, const SweepProgram<double>&, cudaStream_t);

}  // namespace sv
