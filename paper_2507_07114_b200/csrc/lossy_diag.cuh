// What an experiment reads out between steps: the squared norm of every gradient piece and the pairwise drift of the
// replicas. Read-only kernels; the floor of both is one read of their input at the memory rate.
#pragma once
#include <type_traits>

#include "lossy_device.cuh"

namespace lossy {

// ---- squared norm of every (worker, packet) gradient piece: out[i * K + k] ----------------------------------
// One warp per piece (blockIdx.y = the worker), each lane's vectors summed in ascending order, then a shuffle tree.
// A warp that waits for one 16-byte load per lane at a time has too few bytes in flight, so kSqLoads vectors are
// requested before the first is used: of one piece when it is longer than kChunk elements (MANY = false), else of
// kSqLoads pieces, one vector each, whose totals come from one multi-value reduction. W = 16 bf16 pieces of 2048
// elements, 537 MB: 87 us (floor 82 us); W = 32, P = 128, 31 MB: 31 -> 17 us. The grid is one or two
// times what is resident (eight blocks per SM; four with fp32 pieces longer than a chunk) and no block more.
struct SqnormArgs {
  const void* grads[kMaxW];
  float* out;
  uint64_t n;
  uint32_t W, P, K;
};
constexpr int kSqLoads = 4;
template <class GT, bool MANY>
static __global__ void __launch_bounds__(256) packet_sqnorms_kernel(const __grid_constant__ SqnormArgs A) {
  const int lane = threadIdx.x & 31;
  const uint32_t i = blockIdx.y;
  wait_for_previous();
  const void* grads = A.grads[i];
  const uint32_t warps = gridDim.x * (blockDim.x >> 5), warp0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  auto add = [](float s, const Vec8<GT>& raw, int nvalid) {
    float f[8];
    widen<GT>(raw, f);
#pragma unroll
    for (int x = 0; x < 8; ++x) s = __fadd_rn(s, x < nvalid ? __fmul_rn(f[x], f[x]) : 0.0f);
    return s;
  };
  if constexpr (MANY) {
    const uint32_t tasks = A.K / kSqLoads + (A.K % kSqLoads != 0);
    for (uint32_t t = warp0; t < tasks; t += warps) {   // (tasks < 2^30: no wrap)
      Vec8<GT> raw[kSqLoads];
      int nvalid[kSqLoads];
#pragma unroll
      for (int u = 0; u < kSqLoads; ++u) {
        const uint64_t k = (uint64_t)t * kSqLoads + u;
        const uint64_t e0 = k * A.P, e1 = e0 + A.P < A.n ? e0 + A.P : A.n, e = e0 + (uint64_t)lane * 8;
        nvalid[u] = e >= e1 ? 0 : e1 - e >= 8 ? 8 : (int)(e1 - e);
        raw[u] = load8_any<GT>(grads, e, nvalid[u], nvalid[u] > 0);
      }
      float s[kSqLoads];
#pragma unroll
      for (int u = 0; u < kSqLoads; ++u) s[u] = add(0.0f, raw[u], nvalid[u]);
      const float tot = warp_sum_multi<kSqLoads>(s, lane);
      const uint64_t k = (uint64_t)t * kSqLoads + ((uint32_t)lane >> 3);
      if ((lane & 7) == 0 && k < A.K) A.out[(size_t)i * A.K + k] = tot;
    }
  } else {
    for (uint32_t k = warp0; k < A.K; k = A.K - k > warps ? k + warps : A.K) {   // (k + warps may pass 2^32)
      const uint64_t e0 = (uint64_t)k * A.P;
      const uint64_t e1 = e0 + A.P < A.n ? e0 + A.P : A.n;
      float s = 0.0f;
      for (uint64_t eb = e0 + (uint64_t)lane * 8; eb < e1; eb += kSqLoads * kChunk) {
        Vec8<GT> raw[kSqLoads];
        int nvalid[kSqLoads];
#pragma unroll
        for (int u = 0; u < kSqLoads; ++u) {
          const uint64_t e = eb + (uint64_t)u * kChunk;
          nvalid[u] = e >= e1 ? 0 : e1 - e >= 8 ? 8 : (int)(e1 - e);
          raw[u] = load8_any<GT>(grads, e, nvalid[u], nvalid[u] > 0);
        }
#pragma unroll
        for (int u = 0; u < kSqLoads; ++u) s = add(s, raw[u], nvalid[u]);
      }
      s = warp_sum(s);
      if (lane == 0) A.out[(size_t)i * A.K + k] = s;
    }
  }
}

// ---- pairwise drift, the theorem's own quantity: d2[i*W + k] += sum_e (replica_i[e] - replica_k[e])^2 -------
// The W(W-1)/2 differences per element are the cost, not the W reads, unless most of them are known to be zero: after
// a broadcast every replica that took it holds the same bits. So a warp takes a chunk of 256 elements, compares every
// replica's piece with one reference piece bit by bit (a copy of what most replicas hold, found by trying) and is left
// with the pieces that differ. Pairs of equal pieces add exactly zero; a differing piece has ONE difference to all the
// pieces equal to the reference; pairs of differing pieces are computed one by one. With nothing equal this is the
// full set of pairs, each difference taken directly (never through inner products, whose cancellation would cost the
// small distances their digits).
// A piece counts as equal only where the reference is finite, so infinities and NaN give what their differences give.
// Differing pieces are kept in shared memory, kPairSlots at a time (fetching them again cost an L2 round trip per row
// of pairs). The pieces behind the slots meet all slots at once, so one fetch serves kPairSlots pairs, whose totals
// come from one multi-value reduction.
// Sums: fp32 over a lane's eight elements, two multiply-add chains of four, fp64 from there on: over the warp, in a table of
// pairs per warp in shared memory, and with fp64 atomics into d2 at the end (their order is not fixed: results agree to ~1e-15
// relative). With the warp's tree in fp32 as well a pair of bf16 copies that differ by N(0, 3e-4) came out 8.5e-9 low, as it
// is 4e-10 (fp32 copies: 6e-10 high); differences from 1.2e18 on overflowed where they now do from 6.5e18 on.
// Measured on B200, W = 16 bf16 replicas of 16 M elements (floor of one read: 79 us), by the share of packets a
// replica missed: 5 % 97 us, 15 % 129 us, 35 % 197 us; 4 x 4 blocks of replicas
// with every pair computed and fp64 sums per lane took 2512 us whatever the data. Bound by its issue slots and the latency
// of the steps per differing piece, not by memory, once pieces differ.
// How many pieces differ is the same for a whole packet and differs from packet to packet, and with it a chunk's work, so a
// block's chunks are every gridDim.x-th one and its warps take them as they come free, by a counter in shared memory (dealt
// out in advance, grid-stride, the three times above were 119, 161 and 263 us; W = 64, 4 M, 15 %: 242 and 469 us). Runs of four
// chunks per turn, with the lanes' sums kept over a run, unbalance the warps again (216 us for 161). Where there are fewer chunks than warps, 2^lgsplit warps share a chunk: each
// finds the differing pieces and computes every 2^lgsplit-th row of pairs (60 k elements, W = 64, fp32, all copies distinct: 246 ->
// 126 us; W = 16, 35 % of the packets late: 27 -> 23 us).
// (a kernel's arguments cost the host about 1 ns per byte: rep_skip only where it is read)
template <bool ELIDE> struct PairwiseArgs {
  const void* replicas[kMaxW];
  double* d2;
  uint64_t n;
  uint32_t W;
  // The elements fall into segments of seg_len (the last may be shorter): with owner-elided replicas the shards, whose
  // owner holds no copy; else one segment. Segment s starts at element s * seg_len - seg_off.
  uint64_t seg_len, seg_off;
  uint32_t seg0, segs;          // first segment of this context, and how many
  uint32_t chunks_per_seg;
  uint32_t lgsplit;             // sets kernel: log2 of the warps that share a chunk's pairs
  uint64_t rep_skip[ELIDE ? kMaxW : 1];   // as in Params
};
// Both kernels, block 0, warp 0: the last elements behind a multiple of eight, each pair's differences one by one.
template <class RT, bool ELIDE>
__device__ __forceinline__ void pairwise_tail(const PairwiseArgs<ELIDE>& A, int lane, uint32_t warp) {
  if (blockIdx.x != 0 || warp != 0 || (A.n & 7u) == 0) return;
  const uint32_t W = A.W, j = ELIDE ? A.seg0 + A.segs - 1u : ~0u;   // the owner of the last packet
  auto value = [&](uint32_t i, uint64_t e) {
    const typename RT::raw* p = reinterpret_cast<const typename RT::raw*>(A.replicas[i]);
    const uint64_t at = ELIDE && j > i ? e - A.rep_skip[i] : e;
    if constexpr (RT::kVecs == 2) return (float)p[at];
    else return __uint_as_float((uint32_t)p[at] << 16);
  };
  for (uint32_t q = lane; q < W * W; q += 32) {
    const uint32_t i = q / W, k = q - i * W;
    if (i > k || i == j || k == j) continue;
    double t = 0.0;
    for (uint64_t e = A.n & ~7ull; e < A.n; ++e) {
      const float d = __fsub_rn(value(i, e), value(k, e));
      t += (double)__fmul_rn(d, d);
    }
    if (t == 0.0) continue;
    atomicAdd(&A.d2[q], t);                               // (i == k: x - x, the NaN of an infinity or NaN)
    if (i != k) atomicAdd(&A.d2[(size_t)k * W + i], t);
  }
}

// Two to eight replicas (NW: room for four or eight): every pair directly. Nothing is compared and the time does not depend on
// how many copies differ: a lane loads its eight elements of every replica and keeps an fp64 sum per pair, with no
// shuffles until the end. W = 4, 16 M fp32 elements: 49 us (floor 40), where sets of differing copies take 60 to 213 and
// 4 x 4 blocks of replicas took 130; W = 8, 250 k: 10 us (10 to 18, 12). Bound by memory up to four replicas, by registers and
// arithmetic with eight (16 M bf16: 154 us whatever the data, the sets 54 to 138 up to 35 % late).
template <class RT, bool ELIDE, int NW>
static __global__ void __launch_bounds__(128) drift_pairwise_few_kernel(const __grid_constant__ PairwiseArgs<ELIDE> A) {
  constexpr unsigned kFull = 0xFFFFFFFFu;
  constexpr int kPairs = NW * (NW - 1) / 2;
  __shared__ double sh[4][kPairs];
  const int lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5, W = A.W;
  double acc[kPairs];
#pragma unroll
  for (int x = 0; x < kPairs; ++x) acc[x] = 0.0;
  uint32_t bad = 0;                                       // replicas seen to hold an infinity or NaN: x - x is NaN
  wait_for_previous();
  const uint64_t total = (uint64_t)A.segs * A.chunks_per_seg;
  for (uint64_t q = (uint64_t)blockIdx.x * 4u + warp; q < total; q += (uint64_t)gridDim.x * 4u) {
    const uint32_t seg = ELIDE ? (uint32_t)q / A.chunks_per_seg : 0u, j = A.seg0 + seg;
    const uint64_t c = (uint32_t)q - seg * A.chunks_per_seg;
    const uint64_t b0 = (uint64_t)j * A.seg_len, b1 = b0 + A.seg_len;
    const uint64_t lo = b0 > A.seg_off ? b0 - A.seg_off : 0ull;
    const uint64_t hi = b1 - A.seg_off < A.n ? b1 - A.seg_off : A.n;
    const uint64_t e = lo + c * kChunk + (uint64_t)lane * 8;
    if (e + 8 > hi) continue;
    float2 f[NW][4];
    bool held[NW];
    {
      Vec8<RT> v[NW];
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        held[i] = (uint32_t)i < W && !(ELIDE && j == (uint32_t)i);   // (the owner of a packet holds no copy of it)
        if (held[i]) {
          const uint64_t at = ELIDE && j > (uint32_t)i ? e - A.rep_skip[i] : e;
          const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const typename RT::raw*>(A.replicas[i]) + at);
#pragma unroll
          for (int x = 0; x < RT::kVecs; ++x) v[i].q[x] = __ldcs(p + x);
        }
      }
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        if (!held[i]) continue;
        float g[8];
        widen<RT>(v[i], g);
        bool odd = false;
#pragma unroll
        for (int x = 0; x < 4; ++x) f[i][x] = make_float2(g[2 * x], g[2 * x + 1]);
#pragma unroll
        for (int x = 0; x < 8; ++x) odd |= (__float_as_uint(g[x]) & 0x7F800000u) == 0x7F800000u;
        if (odd) bad |= 1u << i;
      }
    }
    int at = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i)
#pragma unroll
      for (int k = i + 1; k < NW; ++k, ++at)
        if (held[i] && held[k]) {
          float2 t = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const float2 d = __fadd2_rn(f[i][x], make_float2(-f[k][x].x, -f[k][x].y));
            t = __ffma2_rn(d, d, t);
          }
          acc[at] += (double)__fadd_rn(t.x, t.y);
        }
  }
#pragma unroll
  for (int x = 0; x < kPairs; ++x) {
    double t = acc[x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    if (lane == 0) sh[warp][x] = t;
  }
  pairwise_tail<RT, ELIDE>(A, lane, warp);
  bad = __reduce_or_sync(kFull, bad);
  __syncthreads();
  for (uint32_t q = threadIdx.x; q < W * W; q += blockDim.x) {
    const uint32_t i = q / W, k = q - i * W, lo = i < k ? i : k, hi = i < k ? k : i;
    if (lo == hi) continue;
    const uint32_t at = lo * (2u * NW - lo - 1u) / 2u + hi - lo - 1u;
    const double t = (sh[0][at] + sh[1][at]) + (sh[2][at] + sh[3][at]);
    if (t != 0.0) atomicAdd(&A.d2[q], t);
  }
  if (lane < NW && ((bad >> lane) & 1u)) atomicAdd(&A.d2[(size_t)lane * W + lane], __longlong_as_double(0x7FF8000000000000ll));
}

constexpr int kPairSlots = 8;
// Warps per block, one block per SM, and bytes of pieces in flight per lane. As many warps as 72 registers allow; with more
// than 32 replicas the tables of pairs leave room for 11 or fewer in any case, which keep more loads in flight each. SMALL:
// for buckets without work for that many warps, whose time is the latency of one chunk (60 k elements, W = 32, fp32, 35 % late:
// 47 -> 26 us, 15 %: 21 -> 13 us).
template <class M, bool SMALL> struct PairShape {
  static constexpr int kMaxWarps = SMALL ? 8 : sizeof(M) == 4 ? 28 : 16, kBytes = SMALL ? 256 : sizeof(M) == 4 ? 64 : 128;
};
__host__ __device__ inline uint32_t pair_table(uint32_t W) { return W * (W - 1u) / 2u; }   // doubles per warp
// shared memory of one warp: the table of pairs, the slots, the slots' replica numbers
__host__ __device__ inline uint32_t pair_warp_bytes(uint32_t W, uint32_t elem_bytes) {
  return (pair_table(W) * 8u + 15u) / 16u * 16u + kPairSlots * kChunk * elem_bytes + kPairSlots * 4u;
}

// M: the type of a set of replicas (32 bits where W <= 32)
template <class RT, bool ELIDE, class M, bool SMALL>
static __global__ void __launch_bounds__(PairShape<M, SMALL>::kMaxWarps * 32, 1) drift_pairwise_kernel(const __grid_constant__ PairwiseArgs<ELIDE> A) {
  extern __shared__ __align__(16) unsigned char pair_smem[];
  __shared__ uint32_t taken;                              // tasks of this block that its warps have taken
  constexpr unsigned kFull = 0xFFFFFFFFu;
  constexpr uint32_t kRB = sizeof(typename RT::raw);
  constexpr int kW = RT::kVecs * 4;                       // 32-bit words of a lane's 8 elements
  constexpr int kLoads = PairShape<M, SMALL>::kBytes / (RT::kVecs * 16);   // pieces in flight per lane
  const int lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t W = A.W, nt = pair_table(W), wb = pair_warp_bytes(W, kRB);
  double* tab = reinterpret_cast<double*>(pair_smem + (size_t)warp * wb);
  unsigned char* slots = pair_smem + (size_t)warp * wb + (nt * 8u + 15u) / 16u * 16u;
  volatile uint32_t* slot_id = reinterpret_cast<volatile uint32_t*>(slots + kPairSlots * kChunk * kRB);
  for (uint32_t q = lane; q < nt; q += 32) tab[q] = 0.0;
  if (threadIdx.x == 0) taken = 0;
  wait_for_previous();
  __syncthreads();
  // (debug build: one warp of a block far ahead of the others, so that it takes more than one of the tasks they share)
  if constexpr (kDevCheck) {
    if (A.lgsplit && warp) __nanosleep(1000000u);
  }
  M bad_diag = 0;                                         // replicas seen to hold an infinity or NaN: x - x is NaN
  const M everyone = W == sizeof(M) * 8 ? ~(M)0 : ((M)1 << W) - 1;
  auto first_of = [](M x) { return (uint32_t)(sizeof(M) == 8 ? __ffsll((long long)x) : __ffs((int)x)) - 1u; };
  auto size_of = [](M x) { return sizeof(M) == 8 ? __popcll(x) : __popc((uint32_t)x); };
  auto pair_at = [&](uint32_t a, uint32_t b) {
    const uint32_t lo = a < b ? a : b, hi = a < b ? b : a;
    return lo * (2u * W - lo - 1u) / 2u + hi - lo - 1u;
  };
  auto nonfinite = [&](const Vec8<RT>& v) {
    float f[8];
    widen<RT>(v, f);
    bool bad = false;
#pragma unroll
    for (int x = 0; x < 8; ++x) bad |= (__float_as_uint(f[x]) & 0x7F800000u) == 0x7F800000u;
    return bad;
  };
  auto put = [&](uint32_t slot, const Vec8<RT>& v) {      // a lane reads back what it wrote itself
#pragma unroll
    for (int x = 0; x < RT::kVecs; ++x) *reinterpret_cast<uint4*>(slots + (slot * RT::kVecs + x) * 512u + lane * 16) = v.q[x];
  };
  auto get = [&](uint32_t slot) {
    Vec8<RT> v;
#pragma unroll
    for (int x = 0; x < RT::kVecs; ++x) v.q[x] = *reinterpret_cast<const uint4*>(slots + (slot * RT::kVecs + x) * 512u + lane * 16);
    return v;
  };

  const uint64_t total = ((uint64_t)A.segs * A.chunks_per_seg) << A.lgsplit;
  const uint32_t others = (1u << A.lgsplit) - 1u;         // warps a chunk is shared with
  uint32_t guess = 0;                                     // the reference of the chunk before (a shared chunk: 0)
  for (;;) {
    uint32_t next = 0;
    if (lane == 0) next = atomicAdd(&taken, 1u);
    const uint64_t task = (uint64_t)__shfl_sync(kFull, next, 0) * gridDim.x + blockIdx.x;
    if (task >= total) break;
    const uint64_t q = task >> A.lgsplit;
    // Rows of pairs are dealt out: this warp takes those met at turn 0. The warps that share a chunk meet the same rows only
    // if they choose the same reference, so the search for it starts from replica 0 and not from the warp's last one: a
    // warp may have taken a task before, of another chunk, and its siblings none.
    uint32_t turn = (uint32_t)task & others;
    auto mine = [&]() { const bool m = turn == 0u; turn = (turn - 1u) & others; return m; };
    const uint32_t seg = ELIDE ? (uint32_t)q / A.chunks_per_seg : 0u, j = A.seg0 + seg;
    const uint64_t c = (uint32_t)q - seg * A.chunks_per_seg;
    const uint64_t b0 = (uint64_t)j * A.seg_len, b1 = b0 + A.seg_len;
    const uint64_t lo = b0 > A.seg_off ? b0 - A.seg_off : 0ull;
    const uint64_t hi = b1 - A.seg_off < A.n ? b1 - A.seg_off : A.n;
    // Lanes with eight elements; the others read what lane 0 reads and add nothing. Elements behind the last multiple of
    // eight are taken at the end: with tests of the count in every load, 64-bit sets and a vote per piece a chunk of
    // W = 16 took 1520 warp instructions, without them 1080.
    const uint64_t e_warp = lo + c * kChunk;
    if (e_warp + 8 > hi) continue;
    const bool live = e_warp + (uint64_t)lane * 8 + 8 <= hi;
    const uint64_t e = e_warp + (live ? (uint64_t)lane * 8 : 0ull);
    M present = everyone;
    if constexpr (ELIDE) present &= ~((M)1 << j);          // the owner of a packet holds no copy of it
    if (!present) continue;
    // (plain cached loads: a second reference, or a piece behind the slots, is fetched again)
    auto fetch = [&](uint32_t i) {
      const uint64_t at = ELIDE && j > i ? e - A.rep_skip[i] : e;
      Vec8<RT> v;
      const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const typename RT::raw*>(A.replicas[i]) + at);
#pragma unroll
      for (int x = 0; x < RT::kVecs; ++x) v.q[x] = __ldg(p + x);
      return v;
    };
    // ---- the reference, and the pieces that differ from it: the first kPairSlots of them into the slots ----
    Vec8<RT> ref;
    uint32_t r = (present >> guess) & 1 ? guess : first_of(present);
    M differ = 0;
    bool ref_finite = true;
    int best = -1;
    uint32_t best_r = r;
    M left = present;                               // references not yet known to be worse
    for (int tries = 0;; ++tries) {
      ref = fetch(r);
      ref_finite = !nonfinite(ref);
      differ = 0;
      uint32_t m = 0;
      for (uint32_t i0 = 0; i0 < W; i0 += kLoads) {
        const uint32_t here = (uint32_t)(present >> i0) & ((1u << kLoads) - 1u);
        Vec8<RT> v[kLoads];
#pragma unroll
        for (int u = 0; u < kLoads; ++u)
          if ((here >> u) & 1u) v[u] = fetch(i0 + u);
        uint32_t off = ref_finite ? 0u : here;             // bit u: this lane's part of piece u differs from the reference
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
          const uint32_t *a = reinterpret_cast<const uint32_t*>(&v[u].q[0]), *b = reinterpret_cast<const uint32_t*>(&ref.q[0]);
          uint32_t x = 0;
#pragma unroll
          for (int y = 0; y < kW; ++y) x |= a[y] ^ b[y];
          if (x) off |= 1u << u;
        }
        off = __reduce_or_sync(kFull, off) & here;
        if (r - i0 < (uint32_t)kLoads) off &= ~(1u << (r - i0));
        if (!off) continue;
        differ |= (M)off << i0;
#pragma unroll
        for (int u = 0; u < kLoads; ++u)
          if (((off >> u) & 1u) && m < (uint32_t)kPairSlots) {
            put(m, v[u]);
            if (lane == 0) slot_id[m] = i0 + u;
            ++m;
          }
      }
      const int equal = size_of(present & ~differ);
      if (r == best_r && tries > 0) break;                 // the best of those tried, once more
      if (equal > best) { best = equal; best_r = r; }
      if (2 * best >= size_of(present)) break;            // a majority: no other reference can be much better
      left &= differ;                                      // pieces equal to this one would do as badly
      if (left && tries < 3) r = first_of(left);
      else if (r == best_r) break;
      else r = best_r;
    }
    guess = A.lgsplit ? 0u : r;                            // (shared: see mine)
    if (!__all_sync(kFull, ref_finite)) bad_diag |= (M)1 << r;
    const M fresh = present & ~differ;              // pieces equal to the reference, itself among them
    // ---- the differing pieces, kPairSlots rows at a time, against everything behind them ----
    for (M rest = differ; rest;) {
      uint32_t rows = 0;
      const bool filled = rest == differ;                  // the first rows are in the slots already
      while (rest && rows < (uint32_t)kPairSlots) {
        const uint32_t i = first_of(rest);
        rest &= rest - 1;
        if (!filled) {
          put(rows, fetch(i));
          if (lane == 0) slot_id[rows] = i;
        }
        ++rows;
      }
      __syncwarp();
      // Totals of the squared distances of `partner` to the first N slots: slot u's in the 32 / N lanes of segment u. Slots
      // behind the last row hold what an earlier chunk left there; their totals are not used. (With a test per slot
      // the N chains ran one after the other.)
      auto against = [&](const Vec8<RT>& partner, auto count) {
        constexpr int N = decltype(count)::value;
        float f[8];
        widen<RT>(partner, f);
        float s[N];
#pragma unroll
        for (int u = 0; u < N; ++u) {
          float g[8];
          minus8<RT>(get(u), f, g);
          float2 t = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const float2 d = make_float2(g[2 * x], g[2 * x + 1]);
            t = __ffma2_rn(d, d, t);
          }
          s[u] = live ? __fadd_rn(t.x, t.y) : 0.0f;
        }
        return warp_sum_multi64<N>(s, lane);
      };
      using Two = std::integral_constant<int, 2>;
      using Four = std::integral_constant<int, 4>;
      using Eight = std::integral_constant<int, 8>;
      // one distance for all the pieces equal to the reference
      auto to_fresh = [&](auto count) {
        constexpr int N = decltype(count)::value, kSeg = 32 / N;
        const double tot = against(ref, count);
        const uint32_t odd = __ballot_sync(kFull, !(tot < __longlong_as_double(0x7FF0000000000000ll)));
#pragma unroll
        for (int u0 = 0; u0 < N; u0 += 4) {
          constexpr int B = N < 4 ? N : 4;
          double sum[B * sizeof(M) / 4];                   // (all read before the first is written: no two are the same entry)
          uint32_t at[B * sizeof(M) / 4];
#pragma unroll
          for (int u = 0; u < B; ++u) {
            if ((uint32_t)(u0 + u) >= rows) break;
            const uint32_t i = slot_id[u0 + u];
            const double t = __shfl_sync(kFull, tot, (u0 + u) * kSeg);
#pragma unroll
            for (int h = 0; h < (int)sizeof(M) / 4; ++h) {
              at[B * h + u] = pair_at(i, (uint32_t)lane + 32u * h);
              if ((fresh >> (lane + 32 * h)) & 1) sum[B * h + u] = tab[at[B * h + u]] + t;
            }
          }
#pragma unroll
          for (int u = 0; u < B; ++u) {
            if ((uint32_t)(u0 + u) >= rows) break;
#pragma unroll
            for (int h = 0; h < (int)sizeof(M) / 4; ++h)
              if ((fresh >> (lane + 32 * h)) & 1) tab[at[B * h + u]] = sum[B * h + u];
          }
        }
        if (odd)
          for (uint32_t u = 0; u < rows; ++u)
            if (((odd >> (u * kSeg)) & 1u) && __any_sync(kFull, nonfinite(get(u)))) bad_diag |= (M)1 << slot_id[u];
        __syncwarp();
      };
      auto add_pairs = [&](uint32_t b, const Vec8<RT>& partner, uint32_t used, auto count) {
        constexpr int N = decltype(count)::value, kSeg = 32 / N;
        const double tot = against(partner, count);
        const uint32_t u = (uint32_t)lane / kSeg;
        if ((lane & (kSeg - 1)) == 0 && u < used) tab[pair_at(slot_id[u], b)] += tot;
        __syncwarp();
      };
      if (!mine()) {}
      else if (rows > 4) to_fresh(Eight{});
      else if (rows > 2) to_fresh(Four{});
      else to_fresh(Two{});
      for (uint32_t u = 1; u < rows; ++u) {
        if (!mine()) continue;
        if (u > 4) add_pairs(slot_id[u], get(u), u, Eight{});
        else if (u > 2) add_pairs(slot_id[u], get(u), u, Four{});
        else add_pairs(slot_id[u], get(u), u, Two{});
      }
      for (M todo = rest; todo;) {
        const uint32_t b = first_of(todo);
        todo &= todo - 1;
        if (!mine()) continue;
        add_pairs(b, fetch(b), rows, Eight{});             // (there are pieces behind the slots only when these are full)
      }
    }
  }

  pairwise_tail<RT, ELIDE>(A, lane, warp);
  __syncthreads();
  // (both halves of the matrix row by row: neighbouring threads add to neighbouring entries, four to a 32-byte sector)
  for (uint32_t q = threadIdx.x; q < W * W; q += blockDim.x) {
    const uint32_t i = q / W, k = q - i * W;
    if (i == k) continue;
    const uint32_t at = pair_at(i, k);
    double t = 0.0;
    for (uint32_t w = 0; w < nwarps; ++w) t += reinterpret_cast<const double*>(pair_smem + (size_t)w * wb)[at];
    if (t != 0.0) atomicAdd(&A.d2[q], t);
  }
  // (uniform over the warp: a repeated NaN is a NaN)
  while (bad_diag) {
    const uint32_t i = first_of(bad_diag);
    bad_diag &= bad_diag - 1;
    atomicAdd(&A.d2[(size_t)i * W + i], __longlong_as_double(0x7FF8000000000000ll));
  }
}

}  // namespace lossy
