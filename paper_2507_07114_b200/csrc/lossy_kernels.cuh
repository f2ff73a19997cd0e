// The arithmetic of the lossy data-parallel step, its delivery draws, the end of every kernel with drift norms, and the single
// phases (AGG, STEP, BCAST, DRIFT) on registers alone: one template, specialised by the phase. The fused step: lossy_register.cuh.
#pragma once
#include "lossy_device.cuh"

namespace lossy {

// acc / count as the IEEE fp32 quotient. A power-of-two count is an exact scaling, so the multiplication by
// its reciprocal gives the same correctly rounded value as the division (also in the subnormal range) at a
// tenth of the instructions; count 0 leaves the zeros in place.
// CORRECTED: other counts take a * RN(1 / c), corrected once by its own remainder, which an FMA gives exactly (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", 1990). For every count up to 64 and every
// mantissa that is the correctly rounded quotient (all enumerated in tests/test_gpu_count_quotient.py) while quotient and
// remainder stay in the normal range; sums under 2^-119, infinities and NaN take the division. (A sum that starts at +0 is
// never -0.) The register kernel is bound by its issue slots: W = 8, P = 304, n = 1 M, SGD: 25.1 -> 21.8 us; the
// pipelines' compute warps are not, and lost up to 2 % with it.
template <int N, bool CORRECTED = false>
__device__ __forceinline__ void divide_by_count(float (&a)[N], uint32_t cnt) {
  if (cnt <= 1) return;
  const float fc = (float)cnt;
  if ((cnt & (cnt - 1)) == 0) {
    const float inv = __uint_as_float((127u - (uint32_t)(__ffs(cnt) - 1)) << 23);   // 2^-log2(cnt)
#pragma unroll
    for (int x = 0; x < N; ++x) a[x] = __fmul_rn(a[x], inv);
    return;
  }
  if constexpr (CORRECTED) {
    uint32_t most = 0, least = ~0u;    // of the bits without the sign, doubled: 2^-119 is 8 << 24, infinity 255 << 24; zero counts as large
#pragma unroll
    for (int x = 0; x < N; ++x) {
      const uint32_t u = __float_as_uint(a[x]) << 1;
      most = max(most, u);
      least = min(least, u - 1u);
    }
    if (most < 0xFF000000u && least >= 0x08000000u - 1u) {
      const float inv = __frcp_rn(fc);
      const float2 fc2 = make_float2(fc, fc), inv2 = make_float2(inv, inv);
#pragma unroll
      for (int x = 0; x < N; x += 2) {
        const float2 s = make_float2(a[x], a[x + 1]), q = __fmul2_rn(s, inv2);
        const float2 r = __ffma2_rn(make_float2(-q.x, -q.y), fc2, s);
        const float2 d = __ffma2_rn(r, inv2, q);
        a[x] = d.x;
        a[x + 1] = d.y;
      }
      return;
    }
  }
#pragma unroll
  for (int x = 0; x < N; ++x) a[x] = __fdiv_rn(a[x], fc);
}

// One optimizer update of N elements, every operation rounded on its own
// (Section 3 step (3); Adam as bias-corrected Kingma-Ba with host-side corrections). PAIRED: two elements per instruction
// (packed fp32 pairs of sm_100) but for the square root and the division: the same values. Fewer instructions are less
// power, and the large steps run at the power limit (W = 8, P = 736, 135 M elements: 1245 -> 1191 us).
// The assembler joins a packed product and the packed addition behind it into one multiply-add, whatever rounding either
// asks for (-fmad=false holds for scalars). A product that is added to something is therefore a multiply-add already, with
// P.neg_zero: x + (-0) is x for every x, and the assembler cannot know that the parameter is -0. (The packed sums of squares of the
// pairwise drift and of the gather pipeline's drift norms are multiply-adds.)
template <int OPT, int N, bool PAIRED = true>
__device__ __forceinline__ void optimizer_n(const Params& P, const float (&g)[N], float (&th)[N], float (&m)[N],
                                            float (&v)[N]) {
  constexpr int kStep = PAIRED ? 2 : 1;
  static_assert(N % kStep == 0, "pairs");
  auto all = [](float x) { return make_float2(x, x); };
  auto at = [](const float (&a)[N], int x) { return make_float2(a[x], a[PAIRED ? x + 1 : x]); };
  auto put = [](float (&a)[N], int x, float2 y) { a[x] = y.x; if constexpr (PAIRED) a[x + 1] = y.y; };
  auto mul = [](float2 a, float2 b) { if constexpr (PAIRED) return __fmul2_rn(a, b); else return make_float2(__fmul_rn(a.x, b.x), 0.0f); };
  auto mul_then_add = [&](float2 a, float2 b) { if constexpr (PAIRED) return __ffma2_rn(a, b, all(P.neg_zero)); else return make_float2(__fmul_rn(a.x, b.x), 0.0f); };
  auto add = [](float2 a, float2 b) { if constexpr (PAIRED) return __fadd2_rn(a, b); else return make_float2(__fadd_rn(a.x, b.x), 0.0f); };
  auto neg = [](float2 a) { return make_float2(-a.x, -a.y); };
  auto root = [](float2 a) { return make_float2(__fsqrt_rn(a.x), PAIRED ? __fsqrt_rn(a.y) : 0.0f); };
  auto div = [](float2 a, float2 b) { return make_float2(__fdiv_rn(a.x, b.x), PAIRED ? __fdiv_rn(a.y, b.y) : 0.0f); };
#pragma unroll
  for (int x = 0; x < N; x += kStep) {
    const float2 gx = at(g, x);
    if constexpr (OPT == 0) {
      put(th, x, add(at(th, x), neg(mul_then_add(all(P.lr), gx))));
    } else {
      const float2 mn = add(mul_then_add(all(P.b1), at(m, x)), mul_then_add(all(P.omb1), gx));
      const float2 vn = add(mul_then_add(all(P.b2), at(v, x)), mul_then_add(mul(all(P.omb2), gx), gx));
      const float2 den = add(root(mul(vn, all(P.ibc2))), all(P.eps));
      put(th, x, add(at(th, x), neg(div(mul(all(P.lr), mul(mn, all(P.ibc1))), den))));
      put(m, x, mn);
      put(v, x, vn);
    }
  }
}
template <int OPT>
__device__ __forceinline__ void optimizer8(const Params& P, const float (&g)[8], float (&th)[8], float (&m)[8],
                                           float (&v)[8]) {
  optimizer_n<OPT, 8>(P, g, th, m, v);
}

// The end of a kernel with drift norms. The `nwarps` warps that call this have left their sums of squares in shared
// memory, `rows` rows of kMaxW; the first of them adds the rows up and stores the block's row of `partials`, and the block
// that draws the last ticket sums the rows of each replica in a fixed order (lane l takes rows l, l + 32, ..., then a shuffle
// tree), so the result does not depend on which block happens to be last. Nothing here waits on another block.
// This is the tail of every step, a chain of latencies (2 us), so only one warp fences, behind nothing but its own stores,
// the warp that drains the bulk stores is not waited for, and a lane's rows are requested together, two replicas and ten rows at a
// time: with one replica and five rows 64 replicas' sums over 296 blocks were sixteen round trips to L2 one after the other, now four
// (W = 64, P = 4096, 3 M: 154 -> 148 us; W = 47, P = 1464, 2.2 M: 156 -> 149; W = 24, P = 512, 6 M: 126 -> 121).
constexpr int kFinishRows = 10;
__device__ __forceinline__ void drift_finish(const Params& P, const double* sums, int rows, uint32_t row, int warp, int nwarps, int lane) {
  __shared__ uint32_t is_last;
  auto sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nwarps * 32) : "memory"); };
  sync();
  if (warp == 0) {
    double t0[4] = {}, t1[4] = {};
    for (int w = 0; w < rows; w += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (w + u < rows) {
          t0[u] += sums[(w + u) * kMaxW + lane];
          t1[u] += sums[(w + u) * kMaxW + lane + 32];
        }
    double* out = P.partials + (size_t)row * kMaxW;
    out[lane] = (t0[0] + t0[1]) + (t0[2] + t0[3]);
    out[lane + 32] = (t1[0] + t1[1]) + (t1[2] + t1[3]);
    __syncwarp();
    if (P.ticket && lane == 0) {
      // the warp's row is visible device-wide before its ticket is, and every row before what follows the last one
      uint32_t prev;
      asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(prev) : "l"(P.ticket) : "memory");
      is_last = prev + 1u == P.total_rows ? 1u : 0u;
    }
  }
  if (!P.ticket) return;
  sync();
  if (!is_last) return;
  // two replicas per warp at a time, so that a lane's requests are 16 bytes
  for (uint32_t i = 2u * warp; i < P.W; i += 2u * nwarps) {
    double t0 = 0.0, t1 = 0.0;
    for (uint32_t b0 = lane; b0 < P.total_rows; b0 += 32 * kFinishRows) {
      double2 x[kFinishRows];
#pragma unroll
      for (int u = 0; u < kFinishRows; ++u)
        x[u] = b0 + 32u * u < P.total_rows ? __ldcg(reinterpret_cast<const double2*>(&P.partials[(size_t)(b0 + 32u * u) * kMaxW + i])) : make_double2(0.0, 0.0);
#pragma unroll
      for (int u = 0; u < kFinishRows; ++u) {
        t0 += x[u].x;
        t1 += x[u].y;
      }
    }
    t0 = warp_sum64(t0);
    t1 = warp_sum64(t1);
    if (lane < 2 && i + lane < P.W) {
      const double t = lane ? t1 : t0;
      if (P.sumsq) P.sumsq[i + lane] += t;
      if (P.norms) P.norms[i + lane] = (float)sqrt(t);
    }
  }
  if (warp == 0 && lane == 0) *P.ticket = 0u;  // ready for the next call on this context
}

// Delivery indicators of packet k (owner j), evaluated one worker per lane and gathered by ballot:
// recv bit i = gradient piece of worker i reached the owner; stale bit i = replica i missed the broadcast.
// Independent loss: one threshold compare per link. Bursty loss (P.burst_in set): each link is a two-state
// chain on the same hash value, bad_t = bad_{t-1} ? (u < Tstay) : (u < Tenter), lost iff bad; the new states
// come back in gbad / pbad for the one caller that stores them.
// LINKS says what is known of that: nothing (the words are loaded here where they are needed), or that the loss is bursty and gin and
// pin are the words, or that it is independent.
enum Links : int { kLinksLook = 0, kLinksGiven = 1, kLinksNone = 2 };
template <int PH, int LINKS = kLinksLook>
__device__ __forceinline__ void packet_masks(const Params& P, uint32_t k, uint32_t j, int lane, uint64_t& recv,
                                             uint64_t& stale, uint64_t& gbad, uint64_t& pbad, uint64_t gin_given = 0, uint64_t pin_given = 0) {
  const uint32_t W = P.W;
  const uint64_t pkey = packet_key_of(P.step_key, P.packet_base + k);
  const uint32_t i0 = lane, i1 = lane + 32;
  const bool bursty = LINKS == kLinksGiven || (LINKS == kLinksLook && P.burst_in != nullptr);
  gbad = 0;
  pbad = 0;
  if constexpr (PH & AGG) {
    // Algorithm 1's gradient half: the reduce is reliable and ONE draw (the owner's own link of the
    // hash) keeps or drops the packet's whole aggregate; otherwise one draw per contributing worker.
    const bool alg1 = P.ghat_prev != nullptr;
    const uint32_t src0 = alg1 ? j : i0, src1 = alg1 ? j : i1;
    const uint64_t gin = LINKS == kLinksGiven ? gin_given : bursty ? P.burst_in[k] : 0ull;
    const uint32_t u0 = pair_hash(pkey, src0, j);
    const bool was0 = (gin >> (alg1 ? 0u : i0)) & 1ull;
    bool lost0 = bursty ? (was0 ? u0 < P.Tstay : u0 < P.Tenter) : u0 < P.Tg;
    if (!alg1 && (P.flags & 1u) && i0 == j) lost0 = false;
    uint32_t lo = __ballot_sync(0xFFFFFFFFu, i0 < W && !lost0), hi = 0;
    uint32_t blo = __ballot_sync(0xFFFFFFFFu, i0 < W && lost0), bhi = 0;
    if (W > 32) {
      const uint32_t u1 = pair_hash(pkey, src1, j);
      const bool was1 = (gin >> (alg1 ? 0u : i1)) & 1ull;
      bool lost1 = bursty ? (was1 ? u1 < P.Tstay : u1 < P.Tenter) : u1 < P.Tg;
      if (!alg1 && (P.flags & 1u) && i1 == j) lost1 = false;
      hi = __ballot_sync(0xFFFFFFFFu, i1 < W && !lost1);
      bhi = __ballot_sync(0xFFFFFFFFu, i1 < W && lost1);
    }
    recv = ((uint64_t)hi << 32) | lo;
    gbad = alg1 ? (uint64_t)(blo & 1u) : (((uint64_t)bhi << 32) | blo);
    if (P.reliable) {   // transmissions on the reliable channel always arrive
      const uint64_t all = W == 64 ? ~0ull : ((1ull << W) - 1ull);
      const uint64_t rel = P.reliable[k];
      if (alg1) { if (rel & 1ull) recv = all; }
      else recv |= rel & all;
    }
  }
  if constexpr (PH & BCAST) {
    const uint64_t pin = LINKS == kLinksGiven ? pin_given : bursty ? P.burst_in[(size_t)P.K + k] : 0ull;
    const uint32_t u0 = pair_hash(pkey, j, i0);
    const bool was0 = (pin >> i0) & 1ull;
    const bool d0 = i0 < W && i0 != j && (bursty ? (was0 ? u0 < P.Tstay : u0 < P.Tenter) : u0 < P.Tp);
    uint32_t lo = __ballot_sync(0xFFFFFFFFu, d0), hi = 0;
    if (W > 32) {
      const uint32_t u1 = pair_hash(pkey, j, i1);
      const bool was1 = (pin >> i1) & 1ull;
      const bool d1 = i1 < W && i1 != j && (bursty ? (was1 ? u1 < P.Tstay : u1 < P.Tenter) : u1 < P.Tp);
      hi = __ballot_sync(0xFFFFFFFFu, d1);
    }
    stale = ((uint64_t)hi << 32) | lo;
    pbad = stale;
    if (P.reliable) stale &= ~P.reliable[(size_t)P.K + k];
  }
}

// The same draws for several packets per ballot (W <= 32, not Algorithm 1's aggregate): the warp's lanes
// are split into 32 / Wp segments of Wp lanes (Wp = W rounded up to a power of two); a lane evaluates
// link `i` of the packet `k` (owner `j`) of its segment. One warp evaluating one packet at a time is a
// chain of dependent instructions (the hash) that bounds a producer warp when tiles carry few bytes.
struct BatchDraws {
  uint32_t recv_ok;     // bit = gradient piece delivered
  uint32_t grad_lost;   // bit = gradient link in its lossy state (before the reliable channel)
  uint32_t bcast_lost;  // bit = replica missed the broadcast (before the reliable channel)
};
template <int PH, int LINKS = kLinksLook>
__device__ __forceinline__ BatchDraws batch_draws(const Params& P, uint32_t k, uint32_t j, uint32_t i, bool valid, uint64_t gin = 0, uint64_t pin = 0) {
  const uint64_t pkey = packet_key_of(P.step_key, P.packet_base + k);
  const bool bursty = LINKS == kLinksGiven || (LINKS == kLinksLook && P.burst_in != nullptr);
  BatchDraws d = {0u, 0u, 0u};
  if constexpr (PH & AGG) {
    const bool was = bursty && (((LINKS == kLinksGiven ? gin : P.burst_in[k]) >> i) & 1ull);
    const uint32_t u = pair_hash(pkey, i, j);
    bool lost = bursty ? (was ? u < P.Tstay : u < P.Tenter) : u < P.Tg;
    if ((P.flags & 1u) && i == j) lost = false;
    d.recv_ok = __ballot_sync(0xFFFFFFFFu, valid && !lost);
    d.grad_lost = __ballot_sync(0xFFFFFFFFu, valid && lost);
  }
  if constexpr (PH & BCAST) {
    const bool was = bursty && (((LINKS == kLinksGiven ? pin : P.burst_in[(size_t)P.K + k]) >> i) & 1ull);
    const uint32_t u = pair_hash(pkey, j, i);
    const bool lost = i != j && (bursty ? (was ? u < P.Tstay : u < P.Tenter) : u < P.Tp);
    d.bcast_lost = __ballot_sync(0xFFFFFFFFu, valid && lost);
  }
  return d;
}
// masks of the packet `k` whose segment starts at lane `src` (segment mask `wmask`), as packet_masks returns them
template <int PH>
__device__ __forceinline__ void batch_masks(const Params& P, const BatchDraws& d, uint32_t k, int src, uint32_t wmask,
                                            uint64_t& recv, uint64_t& stale, uint64_t& gbad, uint64_t& pbad) {
  recv = stale = gbad = pbad = 0;
  if constexpr (PH & AGG) {
    recv = (d.recv_ok >> src) & wmask;
    gbad = (d.grad_lost >> src) & wmask;
    if (P.reliable) recv |= P.reliable[k] & ((1ull << P.W) - 1ull);   // W <= 32 here
  }
  if constexpr (PH & BCAST) {
    stale = (d.bcast_lost >> src) & wmask;
    pbad = stale;
    if (P.reliable) stale &= ~P.reliable[(size_t)P.K + k];
  }
}

// ELIDE = owner-elided replicas: a build of its own, so that the index arithmetic of that layout costs the
// default layout nothing (this kernel is bound by its issue slots, not by memory).
// TAIL = the launch of a call's short last packet, behind the launch that has the complete ones. It shares nothing but the
// ticket counter with that launch, whose blocks let it begin once they have passed their own wait. So it need not wait
// for that launch to begin (how it knows that the kernels ahead of both are done: open_gate), only to
// end (what follows waits for this launch alone). A build of its own: with the wait behind the loop of every build the single phases
// ran 5-28 % slower where packets leave lanes idle (W = 3, P = 128, n = 65 M, step: 518 -> 661 us).
template <int PH, class GT, class RT, int OPT, bool ELIDE = false, bool TAIL = false>
__global__ void __launch_bounds__(kThreads, LOSSY_MIN_BLOCKS) lossy_kernel(const __grid_constant__ Params P) {
  auto rep_at = [&](uint32_t i, uint32_t j, uint64_t e) { return ELIDE ? rep_index(P, i, j, e) : e; };
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const uint32_t W = P.W;
  if constexpr (TAIL) begin_beside_previous(P);
  else wait_for_previous();

  double dacc0 = 0.0, dacc1 = 0.0;   // drift sums: lane l holds replicas l and l + 32

  const uint32_t warps_in_grid = gridDim.x * kWarps;
  for (uint32_t q = blockIdx.x * kWarps + warp; q < P.num_chunks; q += warps_in_grid) {
    const uint32_t kq = q / P.chunks_per_packet;
    const uint32_t c = q - kq * P.chunks_per_packet;
    const uint32_t k = P.k_begin + kq;
    const uint32_t j = (P.k0 + k) / P.pps;  // owner W_j of packet k
    const uint32_t in_pkt = c * kChunk + lane * 8;
    const uint64_t e = (uint64_t)k * P.P + in_pkt;
    int nvalid = 0;
    if (in_pkt < P.P && e < P.n) nvalid = (P.n - e >= 8) ? 8 : (int)(P.n - e);
    const bool tail = __any_sync(0xFFFFFFFFu, (nvalid & 7) != 0);   // the bucket ends inside a lane of this chunk
    if constexpr (kDevCheck) {   // debug build: the chunk's range, in the slab and in every replica
      const uint64_t c0 = (uint64_t)k * P.P + (uint64_t)c * kChunk;
      const uint64_t in_packet = P.P - c * kChunk < (uint32_t)kChunk ? P.P - c * kChunk : (uint32_t)kChunk;   // a chunk ends with its packet
      const uint64_t cl = c0 < P.n ? (P.n - c0 < in_packet ? P.n - c0 : in_packet) : 0;
      if (!tile_ok(P, k, j, c0, cl, kSiteRegister, lane)) continue;
    }

    // ---- delivery indicators of this packet (warp-uniform) -------------------
    uint64_t recv = 0, stale = 0, gbad = 0, pbad = 0;
    packet_masks<PH>(P, k, j, lane, recv, stale, gbad, pbad);
    uint32_t cnt = __popcll(recv);
    if (c == 0 && lane == 0) {
      if constexpr (PH & AGG) {
        if (P.count) P.count[k] = (uint8_t)cnt;
        if (P.recv_bits) P.recv_bits[k] = recv;
      }
      if constexpr (PH & BCAST) {
        if (P.stale_bits) P.stale_bits[k] = stale;
      }
      if (P.burst_out) {   // the first chunk of a packet stores its links' new states
        if constexpr (PH & AGG) P.burst_out[k] = gbad;
        if constexpr (PH & BCAST) P.burst_out[(size_t)P.K + k] = pbad;
      }
    }
    // Lanes past a short packet or past the bucket end keep nvalid == 0: they stay in the
    // warp for the shuffles below and every load/store helper skips them.

    // ---- optimizer state: issue these loads before the gradient loop ---------
    Vec8<F32> rth, rm, rv;
    if constexpr (PH & (STEP | BCAST | DRIFT)) rth = load8_any<F32>(P.master, e, nvalid, tail);
    if constexpr ((PH & STEP) && OPT == 1) {
      rm = load8_any<F32>(P.m, e, nvalid, tail);
      rv = load8_any<F32>(P.v, e, nvalid, tail);
    }

    // ---- (2) unbiased aggregate: masked sum in ascending worker order / count --
    float g[8];
    if constexpr (PH & AGG) {
#pragma unroll
      for (int x = 0; x < 8; ++x) g[x] = 0.0f;
      for (uint32_t g0 = 0; g0 < W; g0 += 8) {
        const uint32_t bits = (uint32_t)(recv >> g0) & 0xFFu;
        if (bits == 0) continue;
        Vec8<GT> raw[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if ((bits >> u) & 1u) raw[u] = load8_any<GT>(P.grads[g0 + u], e, nvalid, tail);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if ((bits >> u) & 1u) add8<GT>(raw[u], g);
      }
      divide_by_count<8, true>(g, cnt);
      if (P.ghat_prev) {
        // Algorithm 1: a dropped packet falls back to the saved aggregate, a surviving one is saved
        if (cnt == 0) {
          const Vec8<F32> pv = load8_any<F32>(P.ghat_prev, e, nvalid, tail);
          widen<F32>(pv, g);
        } else {
          store8<F32>(P.ghat_prev, e, narrow<F32>(g), nvalid, tail);
        }
      }
      if (P.ghat) {
        Vec8<F32> o = narrow<F32>(g);
        store8<F32>(P.ghat, e, o, nvalid, tail);
      }
    } else if constexpr (PH & STEP) {
      Vec8<F32> r = load8_any<F32>(P.ghat, e, nvalid, tail);
      widen<F32>(r, g);
      cnt = (P.flags & 2u) ? (uint32_t)P.count_in[k] : 1u;
    }

    // ---- (3) the owner's update ------------------------------------------------
    float th[8];
    if constexpr (PH & (STEP | BCAST | DRIFT)) widen<F32>(rth, th);
    if constexpr (PH & STEP) {
      if (!((P.flags & 2u) && cnt == 0)) {
        float m[8], v[8];
        if constexpr (OPT == 1) {
          widen<F32>(rm, m);
          widen<F32>(rv, v);
        }
        optimizer8<OPT>(P, g, th, m, v);
        store8<F32>(P.master, e, narrow<F32>(th), nvalid, tail);
        if constexpr (OPT == 1) {
          store8<F32>(P.m, e, narrow<F32>(m), nvalid, tail);
          store8<F32>(P.v, e, narrow<F32>(v), nvalid, tail);
        }
      }
    }

    // ---- (4) broadcast with stale retention, and the drift of every copy -------
    if constexpr (PH & (BCAST | DRIFT)) {
      const Vec8<RT> wire = narrow<RT>(th);
      float xw[8];
      widen<RT>(wire, xw);
      const uint64_t own = ELIDE ? 1ull << j : 0ull;   // owner-elided replicas: worker j holds no copy of this packet
      if constexpr (PH & BCAST) {
        const uint64_t keep = stale | own;
        for (uint32_t i = 0; i < W; ++i)
          if (!((keep >> i) & 1ull)) store8<RT>(P.replicas[i], rep_at(i, j, e), wire, nvalid, tail);
      }
      if constexpr (PH & DRIFT) {
        uint64_t todo = (W == 64 ? ~0ull : ((1ull << W) - 1ull)) & ~own;
        while (todo) {
          // up to four copies are fetched before the first is used
          int ids[4];
          Vec8<RT> old[4];
          int nb = 0;
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            ids[b] = -1;
            if (todo) {
              ids[b] = __ffsll((long long)todo) - 1;
              todo &= todo - 1;
              nb = b + 1;
              old[b] = load8_any<RT>(P.replicas[ids[b]], rep_at((uint32_t)ids[b], j, e), nvalid, tail);
            }
          }
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            if (b < nb) {
              float diff[8], s = 0.0f;
              minus8<RT>(old[b], xw, diff);
#pragma unroll
              for (int x = 0; x < 8; ++x) {
                const float d = x < nvalid ? diff[x] : 0.0f;
                s = __fadd_rn(s, __fmul_rn(d, d));
              }
              const float tot = warp_sum(s);
              if ((ids[b] & 31) == lane) {
                if (ids[b] < 32) dacc0 += (double)tot; else dacc1 += (double)tot;
              }
            }
          }
        }
      }
    }
  }

  // ---- per-block drift partials, fixed order ------------------------------------
  if constexpr (PH & DRIFT) {
    __shared__ double dsum[kWarps * kMaxW];   // per warp and replica
    dsum[warp * kMaxW + lane] = dacc0;
    dsum[warp * kMaxW + lane + 32] = dacc1;
    drift_finish(P, dsum, kWarps, P.partials_row0 + blockIdx.x, warp, kWarps, lane);
  }
  if constexpr (TAIL) end_after_previous(P);
}

// Sum the per-block partials of replica blockIdx.x in a fixed order (lane l takes rows l, l+32, ...,
// then a shuffle tree); add to sumsq, write the norm. One warp per replica.
static __global__ void drift_finalize_kernel(const double* __restrict__ partials, uint32_t nblocks, uint32_t W,
                                      float* norms, double* sumsq) {
  const uint32_t i = blockIdx.x;
  wait_for_previous();
  if (i >= W) return;
  double t = 0.0;
  for (uint32_t b = threadIdx.x; b < nblocks; b += 32) t += partials[(size_t)b * kMaxW + i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
  if (threadIdx.x == 0) {
    if (sumsq) sumsq[i] += t;
    if (norms) norms[i] = (float)sqrt(t);
  }
}

// Closed-loop stand-in for the local gradient computation (Section 3 step (1)): worker i's gradient of
// 1/2 sum a (theta - x*)^2 at ITS OWN replica plus its noise, g_i = cast(a * (replica_i - x*) + noise_i),
// each operation rounded on its own. One lane per 8 elements, workers four at a time.
struct ClosedLoopArgs {
  const void* noise[kMaxW];
  const void* replicas[kMaxW];
  void* grads[kMaxW];
  const float* curv;
  const float* target;
  uint64_t n;
  uint32_t W;
};

template <class GT, class RT>
static __global__ void __launch_bounds__(256) closed_loop_grads_kernel(const __grid_constant__ ClosedLoopArgs A) {
  const uint64_t nvec = (A.n + 7) / 8;
  wait_for_previous();
  for (uint64_t vi = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; vi < nvec; vi += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e = vi * 8;
    const int nvalid = A.n - e >= 8 ? 8 : (int)(A.n - e);
    float a[8], xs[8];
    widen<F32>(load8_any<F32>(A.curv, e, nvalid, true), a);
    widen<F32>(load8_any<F32>(A.target, e, nvalid, true), xs);
    for (uint32_t i0 = 0; i0 < A.W; i0 += 4) {
      Vec8<RT> rep[4];
      Vec8<GT> nz[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < A.W) {
          rep[u] = load8_any<RT>(A.replicas[i0 + u], e, nvalid, true);
          nz[u] = load8_any<GT>(A.noise[i0 + u], e, nvalid, true);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < A.W) {
          float g[8];
          minus8<RT>(rep[u], xs, g);
#pragma unroll
          for (int x = 0; x < 8; ++x) g[x] = __fmul_rn(a[x], g[x]);
          add8<GT>(nz[u], g);
          store8<GT>(A.grads[i0 + u], e, narrow<GT>(g), nvalid, true);
        }
    }
  }
}

// Delivery indicators on a dense grid of tuples (host/device agreement check).
static __global__ void mask_grid_kernel(uint64_t seed, uint64_t step, const uint32_t* src, const uint32_t* dst,
                                 const uint64_t* packet, uint64_t count, uint32_t T, uint8_t* out) {
  const uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= count) return;
  const uint64_t pkey = packet_key_of(step_key_of(seed, step), packet[q]);
  out[q] = pair_hash(pkey, src[q], dst[q]) >= T ? 1 : 0;
}

}  // namespace lossy
