// Device-side building blocks of the lossy data-parallel step (sm_100a).
//
// Work decomposition of the register kernels: the bucket is walked in "chunks" of 256 contiguous elements (one warp, 8 elements =
// 16 or 32 bytes per lane; the fused step: 64, 128 or 256) that never straddle a packet, so the delivery masks of a chunk are
// warp-uniform. Chunk q belongs to packet k_begin + q / chunks_per_packet. Warps take chunks grid-stride, so at any moment the
// grid streams one contiguous window of every buffer.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lossy_divide.h"

namespace lossy {

constexpr int kMaxW = 64;
#ifndef LOSSY_THREADS
#define LOSSY_THREADS 256
#endif
#ifndef LOSSY_MIN_BLOCKS
#define LOSSY_MIN_BLOCKS 1
#endif
constexpr int kThreads = LOSSY_THREADS;
constexpr int kWarps = kThreads / 32;
constexpr int kChunk = 256;  // elements per warp-chunk

enum Phase : int { AGG = 1, STEP = 2, BCAST = 4, DRIFT = 8 };
// bits of Params::flags that the kernels look at (the values of the public flags of the same meaning)
constexpr uint32_t kSelfLossless = 1u, kZeroSkip = 2u, kSkipOwner = 8u;

struct Params {
  const void* grads[kMaxW];
  void* replicas[kMaxW];
  float* master;
  float* m;
  float* v;
  float* ghat;            // AGG: optional output; STEP without AGG: input
  float* ghat_prev;       // non-NULL: Algorithm 1's gradient half (last surviving aggregate, in/out)
  uint8_t* count;         // optional output (AGG)
  uint64_t* recv_bits;    // optional output (AGG)
  uint64_t* stale_bits;   // optional output (BCAST)
  const uint8_t* count_in;  // STEP without AGG and ZERO_SKIP: received counts
  double* partials;       // DRIFT: [gridDim.x][kMaxW] per-block squared sums
  // Drift finalisation inside the last block to finish (no second launch): `ticket` counts finished blocks
  // over all launches of one call; NULL = a separate finalize kernel follows.
  uint32_t* ticket;
  uint32_t total_rows;    // partial rows (= blocks) of the whole call
  float* norms;           // [W] or NULL
  double* sumsq;          // [W], added to, or NULL
  const uint64_t* reliable;  // [2][K] (row 0 gradient links, row 1 broadcast links): set bits are never lost; or NULL
  const uint64_t* burst_in;  // bursty loss: link states after the previous step, [2][K] (row 0 gradient links, row 1 broadcast links)
  uint64_t* burst_out;       // link states after this step, same layout (a different buffer)
  uint64_t n;
  uint64_t packet_base;
  uint64_t step_key;      // hash key of (seed, step), derived on the host
  uint32_t k_begin;       // first packet a register launch covers (a pipeline's launch may have those before it)
  uint32_t num_chunks;    // chunks of that launch, counted from packet k_begin
  uint32_t partials_row0; // first row of `partials` this launch writes
  uint32_t chunks_per_packet;
  uint32_t pps;           // packets per shard (of the whole bucket)
  uint64_t cpp_magic, pps_magic;   // of the two above, for divide_by
  uint32_t k0;            // bucket packet index of this context's packet 0 (a context may cover a packet range)
  uint32_t P;
  uint32_t W;
  uint32_t Tg, Tp;        // drop iff hash < T
  uint32_t Tenter, Tstay; // bursty loss: a good link turns bad iff hash < Tenter, a bad one stays bad iff hash < Tstay
  uint32_t K;             // packets in the bucket
  uint32_t flags;
  float lr, b1, b2, omb1, omb2, ibc1, ibc2, eps;
  float neg_zero;         // -0 (optimizer_n)
  // Owner-elided replicas (kSkipOwner): replica i stores this context's elements WITHOUT the packets worker i
  // owns, so everything behind worker i's shard sits rep_skip[i] elements lower in its array. All zero otherwise.
  uint64_t rep_skip[kMaxW];
#ifdef LOSSY_DEVCHECK
  // Debug build: where a failed index check is recorded (4 words: site, element offset low and high, length; the first failure
  // wins) and the element count the checks hold a range against (n, or less when the self-test shrinks it).
  uint32_t* check;
  uint64_t check_n;
#endif
  // A call whose short last packet has a launch of its own beside the launch of the complete ones (open_gate): the context's
  // gate word, and this call's number. Else NULL and 0.
  uint32_t* gate;
  uint32_t gate_id;
};

// Programmatic dependent launch: most kernels are launched with leave to begin before the kernel ahead of them in the stream
// has ended (launch_after in lossy_api.cu). Such a kernel sets up its barriers, then waits here until that kernel is
// complete and its writes are visible, and in turn lets the kernel behind it be set up. Every thread calls this before
// it touches global memory. What is saved is the launch, the blocks' start and the barriers: 2 to 4 us per kernel.
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// The launch of a short last packet (lossy_kernel, TAIL) runs beside the launch of the complete packets, on what the kernels
// ahead of both have written. Those writes are visible to a grid that has waited, and that is the complete packets' one: it
// says so in a word of the context, with a release, and the short packet's threads read the word with an acquire before
// anything else. That it may begin at all says nothing about memory. A thread that does not find this call's number there
// waits like any other kernel (for the complete packets' launch to end), so nothing spins and no launch depends on another one
// running. The word is cleared by the short packet's launch, for a graph replays a call's number.
// open_gate: the store warp, which has nothing to do at first, behind wait_for_previous. By the first thread, in front of the
// block's barrier, the release delayed block 0, and the branch in every kernel cost buckets without a short packet up to 4 %
// (W = 2, P = 128, n = 8 M: 61.0 -> 63.5 us, this 61.6; W = 16, P = 256, p = 0.3, 201 M: 2663 -> 2723, 2649).
__device__ __forceinline__ void open_gate(const Params& P, int lane) {
  const uint32_t id = (blockIdx.x | (uint32_t)lane) == 0u ? P.gate_id : 0u;   // (0: a call with one launch)
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p st.release.gpu.u32 [%0], %1;\n\t}" ::"l"(P.gate), "r"(id) : "memory");
}
__device__ __forceinline__ void begin_beside_previous(const Params& P) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  uint32_t open;
  asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(open) : "l"(P.gate) : "memory");
  if (open != P.gate_id) asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void end_after_previous(const Params& P) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.gate = 0u;   // (a block that has not looked yet will wait)
}

// Owner-elided replicas: rep_skip[i] = elements of worker i's shard inside the context's packet range
// [k0, k0 + K) of a bucket cut into shards of pps packets (the last packet may be short: n elements in all).
__host__ inline void fill_rep_skip(Params& P, bool elide) {
  if (!elide) return;          // (zero already)
  for (uint32_t i = 0; i < P.W; ++i) {
    const uint64_t s0 = (uint64_t)i * P.pps, s1 = s0 + P.pps;          // shard i in bucket packets
    const uint64_t c0 = P.k0, c1 = (uint64_t)P.k0 + P.K;                // this context in bucket packets
    const uint64_t lo = s0 > c0 ? s0 : c0, hi = s1 < c1 ? s1 : c1;
    if (lo >= hi) continue;
    const uint64_t e0 = (lo - c0) * P.P, e1 = (hi - c0) * P.P;
    P.rep_skip[i] = (e1 < P.n ? e1 : P.n) - (e0 < P.n ? e0 : P.n);
  }
}
// Index of bucket element e, which lies in a packet owned by worker j, inside replica i's array (i != j when
// the replicas are owner-elided; with full replicas every rep_skip is 0 and the index is e).
__device__ __forceinline__ uint64_t rep_index(const Params& P, uint32_t i, uint32_t j, uint64_t e) {
  return e - (j > i ? P.rep_skip[i] : 0ull);
}
// Debug build (compiled with -DLOSSY_DEVCHECK, a library of its own): before a kernel of the step path touches
// memory for a chunk or tile it checks the element range and the packet index against the context's sizes, and
// every replica's range (through the owner-elided index map) against that replica's length. A range that fails
// is recorded in Params::check and not touched: the register kernel skips the chunk, a pipeline raises its abort
// flag and every role leaves through the bounded-wait exit. Nothing traps or asserts. In the normal build all of
// this compiles to nothing.
#ifdef LOSSY_DEVCHECK
constexpr bool kDevCheck = true;
#else
constexpr bool kDevCheck = false;
#endif
enum CheckSite : uint32_t { kSiteRegister = 1, kSiteFusedPacked = 2, kSiteFused = 3, kSitePhase = 4, kSiteGather = 5, kSiteReplica = 16 };
#ifdef LOSSY_DEVCHECK
__device__ __forceinline__ void check_record(const Params& P, uint32_t site, uint64_t e0, uint64_t len) {
  if (atomicCAS(&P.check[0], 0u, site) == 0u) {
    P.check[1] = (uint32_t)e0;
    P.check[2] = (uint32_t)(e0 >> 32);
    P.check[3] = (uint32_t)len;
  }
}
// elements [e0, e0 + len) of packet k: inside the slab, and k a packet of it
__device__ __forceinline__ bool span_ok(const Params& P, uint32_t k, uint64_t e0, uint64_t len, uint32_t site) {
  if (!P.check) return true;      // a caller without a context (the no-allocation entry point) has nowhere to record
  if (k < P.K && (len == 0 || (len <= P.check_n && e0 <= P.check_n - len))) return true;   // an empty range touches nothing
  check_record(P, site, e0, len);
  return false;
}
// the same elements inside replica i's array (owner j; the owner has no copy when the replicas are owner-elided)
__device__ __forceinline__ bool rep_span_ok(const Params& P, uint32_t i, uint32_t j, uint64_t e0, uint64_t len, uint32_t site) {
  if (!P.check || len == 0 || ((P.flags & kSkipOwner) && i == j)) return true;
  const uint64_t limit = P.check_n - (P.rep_skip[i] < P.check_n ? P.rep_skip[i] : P.check_n);
  const uint64_t at = e0 - (j > i ? P.rep_skip[i] : 0ull);
  if (at <= e0 && len <= limit && at <= limit - len) return true;
  check_record(P, site | kSiteReplica, at, len);
  return false;
}
// every replica's range of a tile or chunk, the workers dealt over the lanes; warp-uniform result
__device__ __forceinline__ bool tile_ok(const Params& P, uint32_t k, uint32_t j, uint64_t e0, uint64_t len, uint32_t site, int lane) {
  bool ok = span_ok(P, k, e0, len, site);
  for (uint32_t i = (uint32_t)lane; i < P.W; i += 32u) ok = rep_span_ok(P, i, j, e0, len, site) && ok;
  return __all_sync(0xFFFFFFFFu, ok);
}
#else
__device__ __forceinline__ bool span_ok(const Params&, uint32_t, uint64_t, uint64_t, uint32_t) { return true; }
__device__ __forceinline__ bool rep_span_ok(const Params&, uint32_t, uint32_t, uint64_t, uint64_t, uint32_t) { return true; }
__device__ __forceinline__ bool tile_ok(const Params&, uint32_t, uint32_t, uint64_t, uint64_t, uint32_t, int) { return true; }
#endif

// The replica that does not exist for a packet of owner j (as a bit), or 0 with full replicas.
__device__ __forceinline__ uint64_t own_bit(const Params& P, uint32_t j) {
  return (P.flags & kSkipOwner) ? 1ull << j : 0ull;
}

// ---- delivery-indicator hash (Section 3: s, r ~ Bernoulli(1-p)) -------------
// 64-bit finalizer of the splitmix64 generator; the constants of the keyed
// rounds are this library's own choice and are part of its documented contract.
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z ^= z >> 30; z *= 0xBF58476D1CE4E5B9ULL;
  z ^= z >> 27; z *= 0x94D049BB133111EBULL;
  z ^= z >> 31;
  return z;
}
__host__ __device__ __forceinline__ uint64_t step_key_of(uint64_t seed, uint64_t step) {
  return mix64(mix64(seed ^ 0x6A09E667F3BCC908ULL) + step * 0x9E3779B97F4A7C15ULL);
}
__host__ __device__ __forceinline__ uint64_t packet_key_of(uint64_t step_key, uint64_t packet) {
  return mix64(step_key ^ (packet * 0xD6E8FEB86659FD93ULL));
}
__host__ __device__ __forceinline__ uint32_t pair_hash(uint64_t packet_key, uint32_t src, uint32_t dst) {
  const uint64_t pair = ((uint64_t)src << 32) | (uint64_t)dst;
  return (uint32_t)(mix64(packet_key + pair * 0xC2B2AE3D27D4EB4FULL) >> 32);
}

// ---- streaming 128-bit memory operations ------------------------------------
// Everything on this path is touched exactly once per step, so loads and stores
// carry the evict-first ("streaming") cache operator.
__device__ __forceinline__ uint4 ld_stream(const void* p) {
  return __ldcs(reinterpret_cast<const uint4*>(p));
}
__device__ __forceinline__ void st_stream(void* p, uint4 v) {
  __stcs(reinterpret_cast<uint4*>(p), v);
}
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// ---- element-type adapters ----------------------------------------------------
struct F32 { using raw = float; static constexpr int kVecs = 2; };       // 8 elements = 2 x 16 B
struct BF16 { using raw = uint16_t; static constexpr int kVecs = 1; };   // 8 elements = 1 x 16 B

template <class T> struct Vec8 { uint4 q[T::kVecs]; };

template <class T>
__device__ __forceinline__ Vec8<T> load8(const void* base, uint64_t e) {
  Vec8<T> r;
  const typename T::raw* p = reinterpret_cast<const typename T::raw*>(base) + e;
#pragma unroll
  for (int i = 0; i < T::kVecs; ++i) r.q[i] = ld_stream(reinterpret_cast<const uint4*>(p) + i);
  return r;
}
// Ragged tail of the bucket: the last vector may hold fewer than 8 elements.
template <class T>
__device__ __forceinline__ Vec8<T> load8_tail(const void* base, uint64_t e, int nvalid) {
  Vec8<T> r;
  typename T::raw tmp[8];
  const typename T::raw* p = reinterpret_cast<const typename T::raw*>(base) + e;
#pragma unroll
  for (int i = 0; i < 8; ++i) tmp[i] = i < nvalid ? p[i] : (typename T::raw)0;
  if constexpr (T::kVecs == 2) {
    r.q[0] = make_uint4(__float_as_uint(tmp[0]), __float_as_uint(tmp[1]), __float_as_uint(tmp[2]), __float_as_uint(tmp[3]));
    r.q[1] = make_uint4(__float_as_uint(tmp[4]), __float_as_uint(tmp[5]), __float_as_uint(tmp[6]), __float_as_uint(tmp[7]));
  } else {
    r.q[0] = make_uint4((uint32_t)tmp[0] | ((uint32_t)tmp[1] << 16), (uint32_t)tmp[2] | ((uint32_t)tmp[3] << 16),
                        (uint32_t)tmp[4] | ((uint32_t)tmp[5] << 16), (uint32_t)tmp[6] | ((uint32_t)tmp[7] << 16));
  }
  return r;
}
// Accesses of a lane with nvalid of its eight elements. `tail`: the bucket's end may fall into this lane or another one of its warp (best
// the same for the whole warp), whose elements are then taken one by one. Where it does not, a lane behind a short packet's end skips the access
// (the four single phases, W = 38, P = 128, 33 M: 3138 -> 2452 us; W = 6, P = 736, 20 M: 322 -> 302); where it does, such a lane runs along
// beside that one: a third way through every access made broadcasts of buckets that end inside eight elements a third longer (W = 60,
// 75 k: 6.8 -> 9.0 us).
template <class T>
__device__ __forceinline__ void store8(void* base, uint64_t e, const Vec8<T>& v, int nvalid, bool tail) {
  typename T::raw* p = reinterpret_cast<typename T::raw*>(base) + e;
  if (nvalid == 8) {
#pragma unroll
    for (int i = 0; i < T::kVecs; ++i) st_stream(reinterpret_cast<uint4*>(p) + i, v.q[i]);
  } else if (tail) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&v.q[0]);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i < nvalid) {
        if constexpr (T::kVecs == 2) p[i] = __uint_as_float(w[i]);
        else p[i] = (uint16_t)(w[i >> 1] >> ((i & 1) * 16));
      }
    }
  }
}
template <class T>
__device__ __forceinline__ Vec8<T> load8_any(const void* base, uint64_t e, int nvalid, bool tail) {
  if (nvalid == 8) return load8<T>(base, e);
  if (tail) return load8_tail<T>(base, e, nvalid);
  Vec8<T> r;
#pragma unroll
  for (int i = 0; i < T::kVecs; ++i) r.q[i] = make_uint4(0u, 0u, 0u, 0u);
  return r;
}

// widen 8 elements to fp32 (bf16 -> fp32 is a 16-bit shift, exact)
template <class T>
__device__ __forceinline__ void widen(const Vec8<T>& v, float (&f)[8]) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(&v.q[0]);
  if constexpr (T::kVecs == 2) {
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = __uint_as_float(w[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
}
// f += the two elements of a word, f - the two elements, and the elements - f, for bf16 elements: the sum of an fp32 and a
// widened bf16 value is one instruction of sm_100 (exact widening, one rounding), so nothing is unpacked first.
__device__ __forceinline__ void add_pair_bf16(uint32_t w, float& a, float& b) {
  asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}" : "+f"(a), "+f"(b) : "r"(w));
}
__device__ __forceinline__ float2 pair_minus_bf16(uint32_t w, float a, float b) {
  float2 d;
  asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tsub.rn.f32.bf16 %0, lo, %3;\n\tsub.rn.f32.bf16 %1, hi, %4;\n\t}" : "=f"(d.x), "=f"(d.y) : "r"(w), "f"(a), "f"(b));
  return d;
}
// acc += the 8 elements of v
template <class T>
__device__ __forceinline__ void add8(const Vec8<T>& v, float (&acc)[8]) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(&v.q[0]);
#pragma unroll
  for (int x = 0; x < 8; x += 2) {
    if constexpr (T::kVecs == 2) {
      const float2 s = __fadd2_rn(make_float2(acc[x], acc[x + 1]), make_float2(__uint_as_float(w[x]), __uint_as_float(w[x + 1])));
      acc[x] = s.x;
      acc[x + 1] = s.y;
    } else {
      add_pair_bf16(w[x / 2], acc[x], acc[x + 1]);
    }
  }
}
// d = the 8 elements of v minus x
template <class T>
__device__ __forceinline__ void minus8(const Vec8<T>& v, const float (&x)[8], float (&d)[8]) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(&v.q[0]);
#pragma unroll
  for (int y = 0; y < 8; y += 2) {
    const float2 s = T::kVecs == 2 ? __fadd2_rn(make_float2(__uint_as_float(w[y]), __uint_as_float(w[(y + 1) % (4 * T::kVecs)])), make_float2(-x[y], -x[y + 1]))
                                   : pair_minus_bf16(w[y / 2], x[y], x[y + 1]);
    d[y] = s.x;
    d[y + 1] = s.y;
  }
}
// narrow 8 fp32 values to the wire type (bf16: IEEE round-to-nearest-even)
template <class T>
__device__ __forceinline__ Vec8<T> narrow(const float (&f)[8]) {
  Vec8<T> r;
  uint32_t* w = reinterpret_cast<uint32_t*>(&r.q[0]);
  if constexpr (T::kVecs == 2) {
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = __float_as_uint(f[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<uint32_t*>(&h);
    }
  }
  return r;
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = __fadd_rn(x, __shfl_xor_sync(0xFFFFFFFFu, x, o));
  return x;
}

__device__ __forceinline__ double warp_sum64(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
  return x;
}

// Warp totals of N (2, 4 or 8) per-lane values at once. Each exchange (lane distance 16, 8, ...) halves the
// values a lane carries: the lanes whose bit is set keep the upper half and hand over the lower half. The
// one value left is then summed over the remaining lane bits, so every lane ends with the warp total of
// value number lane / (32 / N), in N + 1 (N = 8), N + 2 (N = 4) or N + 3 (N = 2) shuffles instead of 5 N.
template <int N>
__device__ __forceinline__ float warp_sum_multi(float (&v)[N], int lane) {
  static_assert(N == 2 || N == 4 || N == 8, "2, 4 or 8 values");
  constexpr unsigned kFull = 0xFFFFFFFFu;
  int o = 16;
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int x = 0; x < h; ++x) {
      const float keep = up ? v[x + h] : v[x];
      const float give = up ? v[x] : v[x + h];
      v[x] = __fadd_rn(keep, __shfl_xor_sync(kFull, give, o));
    }
    o >>= 1;
  }
#pragma unroll
  for (int r = 32 / N / 2; r >= 1; r >>= 1) v[0] = __fadd_rn(v[0], __shfl_xor_sync(kFull, v[0], r));
  return v[0];
}

// The same totals added in fp64: lanes exchange fp32 values once and widen both sides of the first addition, so only
// the lanes' own sums are fp32.
template <int N>
__device__ __forceinline__ double warp_sum_multi64(const float (&v)[N], int lane) {
  static_assert(N == 2 || N == 4 || N == 8, "2, 4 or 8 values");
  constexpr unsigned kFull = 0xFFFFFFFFu;
  double w[N / 2];
  const bool up16 = (lane & 16) != 0;
#pragma unroll
  for (int x = 0; x < N / 2; ++x) {
    const float keep = up16 ? v[x + N / 2] : v[x];
    const float give = up16 ? v[x] : v[x + N / 2];
    w[x] = (double)keep + (double)__shfl_xor_sync(kFull, give, 16);
  }
  int o = 8;
#pragma unroll
  for (int h = N / 4; h >= 1; h >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int x = 0; x < h; ++x) {
      const double keep = up ? w[x + h] : w[x];
      const double give = up ? w[x] : w[x + h];
      w[x] = keep + __shfl_xor_sync(kFull, give, o);
    }
    o >>= 1;
  }
#pragma unroll
  for (int r = 32 / N / 2; r >= 1; r >>= 1) w[0] += __shfl_xor_sync(kFull, w[0], r);
  return w[0];
}

}  // namespace lossy
