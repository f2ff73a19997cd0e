// The fused step from registers alone: every phase on a lane's EPL elements, no shared-memory pipeline.
#pragma once
#include <type_traits>

#include "lossy_kernels.cuh"

namespace lossy {

// EPL consecutive elements of one lane as 32-bit words
template <class T, int EPL> struct LaneVec { uint32_t w[EPL * sizeof(typename T::raw) / 4]; };

// Loads and stores of a whole lane under a predicate: a branch per worker costs more instructions than the access (a piece that is
// not taken is zero, and adding +0 to a sum that began at +0 changes no bit of it).
template <class T, int EPL>
__device__ __forceinline__ LaneVec<T, EPL> lane_load(const void* base, uint64_t e, bool take = true) {
  LaneVec<T, EPL> r;
  constexpr int kWords = sizeof(r.w) / 4;
  const typename T::raw* p = reinterpret_cast<const typename T::raw*>(base) + e;
#pragma unroll
  for (int i = 0; i < kWords; ++i) r.w[i] = 0u;
  if constexpr (kWords == 1) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.global.cs.u32 %0, [%1];\n\t}" : "+r"(r.w[0]) : "l"(p), "r"((uint32_t)take));
  } else if constexpr (kWords == 2) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.global.cs.v2.u32 {%0, %1}, [%2];\n\t}" : "+r"(r.w[0]), "+r"(r.w[1]) : "l"(p), "r"((uint32_t)take));
  } else {
#pragma unroll
    for (int i = 0; i < kWords; i += 4)
      asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                   : "+r"(r.w[i]), "+r"(r.w[i + 1]), "+r"(r.w[i + 2]), "+r"(r.w[i + 3]) : "l"(reinterpret_cast<const uint32_t*>(p) + i), "r"((uint32_t)take));
  }
  return r;
}
template <class T, int EPL>
__device__ __forceinline__ void lane_store(void* base, uint64_t e, const LaneVec<T, EPL>& r, bool take = true) {
  constexpr int kWords = sizeof(r.w) / 4;
  typename T::raw* p = reinterpret_cast<typename T::raw*>(base) + e;
  if constexpr (kWords == 1) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.cs.u32 [%0], %1;\n\t}" ::"l"(p), "r"(r.w[0]), "r"((uint32_t)take) : "memory");
  } else if constexpr (kWords == 2) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.global.cs.v2.u32 [%0], {%1, %2};\n\t}" ::"l"(p), "r"(r.w[0]), "r"(r.w[1]), "r"((uint32_t)take) : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < kWords; i += 4)
      asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p st.global.cs.v4.u32 [%0], {%1, %2, %3, %4};\n\t}"
                   ::"l"(reinterpret_cast<uint32_t*>(p) + i), "r"(r.w[i]), "r"(r.w[i + 1]), "r"(r.w[i + 2]), "r"(r.w[i + 3]), "r"((uint32_t)take) : "memory");
  }
}
template <class T>
__device__ __forceinline__ float load_one(const void* base, uint64_t e) {
  const typename T::raw x = reinterpret_cast<const typename T::raw*>(base)[e];
  if constexpr (T::kVecs == 2) return x;
  else return __uint_as_float((uint32_t)x << 16);
}
template <class T, int EPL>
__device__ __forceinline__ void lane_widen(const LaneVec<T, EPL>& r, float (&f)[EPL]) {
#pragma unroll
  for (int x = 0; x < EPL; ++x) {
    if constexpr (T::kVecs == 2) f[x] = __uint_as_float(r.w[x]);
    else f[x] = __uint_as_float(x & 1 ? r.w[x / 2] & 0xFFFF0000u : r.w[x / 2] << 16);
  }
}
template <class T, int EPL>
__device__ __forceinline__ LaneVec<T, EPL> lane_narrow(const float (&f)[EPL]) {
  LaneVec<T, EPL> r;
#pragma unroll
  for (int i = 0; i < (int)(sizeof(r.w) / 4); ++i) {
    if constexpr (T::kVecs == 2) {
      r.w[i] = __float_as_uint(f[i]);
    } else {
      __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      r.w[i] = *reinterpret_cast<uint32_t*>(&h);
    }
  }
  return r;
}
template <class T, int EPL>
__device__ __forceinline__ typename T::raw lane_element(const LaneVec<T, EPL>& r, int x) {
  if constexpr (T::kVecs == 2) return __uint_as_float(r.w[x]);
  else return (uint16_t)(r.w[x / 2] >> ((x & 1) * 16));
}
template <class T, int EPL>
__device__ __forceinline__ void lane_add(const LaneVec<T, EPL>& r, float (&acc)[EPL]) {
#pragma unroll
  for (int x = 0; x < EPL; x += 2) {
    if constexpr (T::kVecs == 2) {
      const float2 s = __fadd2_rn(make_float2(acc[x], acc[x + 1]), make_float2(__uint_as_float(r.w[x]), __uint_as_float(r.w[x + 1])));
      acc[x] = s.x;
      acc[x + 1] = s.y;
    } else {
      add_pair_bf16(r.w[x / 2], acc[x], acc[x + 1]);
    }
  }
}
// the squares of the elements minus x, summed one by one
template <class T, int EPL>
__device__ __forceinline__ float lane_squares(const LaneVec<T, EPL>& r, const float (&x)[EPL]) {
  float s = 0.0f;
#pragma unroll
  for (int y = 0; y < EPL; y += 2) {
    const float2 d = T::kVecs == 2 ? make_float2(__fsub_rn(__uint_as_float(r.w[y % (EPL * T::kVecs / 2)]), x[y]), __fsub_rn(__uint_as_float(r.w[(y + 1) % (EPL * T::kVecs / 2)]), x[y + 1]))
                                   : pair_minus_bf16(r.w[y / 2], x[y], x[y + 1]);
    s = __fadd_rn(s, __fmul_rn(d.x, d.x));
    s = __fadd_rn(s, __fmul_rn(d.y, d.y));
  }
  return s;
}

// The fused step of a small bucket is a chain of latencies: launch, draws, one round trip to memory, the update, the end of the
// drift norms. A pipeline adds its own filling and draining. Here a warp takes a chunk of 32 lanes' elements from the draws to
// the stores, one block per SM has as many warps as its share of the chunks needs, and everything that can be requested together is:
// state before the draws, stale copies before the gradients, all of up to 16 gradient pieces before the first sum. With 8 elements
// per lane, as this kernel's predecessor had, 300 thousand elements gave an SM eight warps; with 2 or 4 they give it 32 or 16, each
// with the same chain. What is left is instructions in a row (W = 8, P = 256, 0.45 M elements: 795 warp instructions per chunk, the block's
// end included, one of a warp's every 17 cycles, the issue slots used to a third), hence the predicated accesses, divisions by
// multiplication and both directions' draws at once for W <= 16.
// Steps of 2000 random buckets (us in a graph, mean of the pipelines' or the predecessor's time over this kernel's, by tiles of
// 2048 elements per SM): W = 2-4: 1.44 under one, 1.6 at two to four, 1.4 to eight, 1.1 to 16; W = 5-8: 1.42, 1.4, 1.13, 1.04; W = 9-16:
// 1.57, 1.46, 1.27, 1.1; W = 17-32: 1.6, 1.34, 1.15, 1.06; W = 33-64: 1.75, 1.4, 1.22, 1.08.
// A few thousand elements: 1.4 to 2.1 by workers. (Buckets of tens of rounds that only LOSSY_REGISTER_PATH brings here, W = 5-21, p near 0:
// 0.93-1.0 of the predecessor, whose eight elements per lane the octs have: 1.01-1.05, but 0.65-0.95 where packets leave chunks part empty.)
//
// The builds: two elements per lane, four, four with room for four workers and no more, four with room for more stale copies, and
// eight. Warps a block may have, gradient pieces, replica stores and stale copies a lane has in flight. (Five of the 144 spill: up to four
// workers with Adam, fp32 replicas and drift norms, 16 or 20 bytes at 64 registers, and eight elements with bf16 and Adam, 4 bytes.) Pairs are
// ahead of quads where they take no more rounds of the chip (W = 33-64, 0.3 tiles per SM: 0.83 of their time; W = 5-8, 1 tile: 1.2). Eight stale copies
// instead of four: 1.04-1.09 from two stale replicas per packet on, 0.9-0.98 below.
enum StepForm : int { kStepPairs = 0, kStepQuads = 1, kStepFew = 2, kStepStale = 3, kStepOcts = 4 };
template <class GT, class RT, int FORM> struct StepShape {
  static constexpr int kEpl = FORM == kStepPairs ? 2 : FORM == kStepOcts ? 8 : 4;
  static constexpr int kMaxWarps = FORM == kStepPairs || FORM == kStepFew ? 32 : FORM == kStepOcts ? (GT::kVecs == 1 ? 16 : 12) : GT::kVecs == 1 ? 24 : 20;
  static constexpr int kGrads = FORM == kStepFew ? 4 : FORM == kStepPairs && GT::kVecs == 1 ? 16 : 8;
  static constexpr int kStores = FORM == kStepFew ? 4 : 8;
  static constexpr int kStale = FORM == kStepFew ? 2 : (FORM == kStepPairs || FORM == kStepStale) && RT::kVecs == 1 ? 8 : 4;
};
constexpr uint32_t kStepFewWorkers = 4;

template <int N, int M>
__device__ __forceinline__ double totals_of(const float (&sq)[M], int lane, int& seg) {
  float first[N];
#pragma unroll
  for (int b = 0; b < N; ++b) first[b] = sq[b];
  seg = 32 / N;
  return warp_sum_multi64<N>(first, lane);
}

// TAIL = the launch of a call's short last packet, behind the launch that has the complete ones. It shares nothing but the
// ticket counter with that launch, whose blocks let it begin once they have passed their own wait. So it need not wait
// for that launch to begin (how it knows that the kernels ahead of both are done: open_gate), only to
// end (what follows waits for this launch alone).
template <class GT, class RT, int OPT, bool DRIFTK, bool ELIDE, bool TAIL, int FORM>
__global__ void __launch_bounds__(StepShape<GT, RT, FORM>::kMaxWarps * 32, 1) lossy_step_kernel(const __grid_constant__ Params P) {
  using Shape = StepShape<GT, RT, FORM>;
  constexpr int EPL = Shape::kEpl;
  constexpr uint32_t kSpan = 32 * EPL;       // elements of a warp's chunk
  constexpr int kG = Shape::kGrads, kB = Shape::kStale, kS = Shape::kStores;
  auto rep_at = [&](uint32_t i, uint32_t j, uint64_t e) { return ELIDE ? rep_index(P, i, j, e) : e; };
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const uint32_t nwarps = blockDim.x >> 5, W = P.W;
  const uint64_t all_workers = ~0ull >> (64u - W);
  __shared__ double dsum[DRIFTK ? Shape::kMaxWarps * kMaxW : 1];   // drift sums per warp and replica; a warp writes its own row alone
  if constexpr (DRIFTK) {
    dsum[warp * kMaxW + lane] = 0.0;
    dsum[warp * kMaxW + lane + 32] = 0.0;
  }
  if constexpr (TAIL) begin_beside_previous(P);
  else wait_for_previous();
  __syncwarp();

  const uint32_t rest = (uint32_t)(P.n % EPL);   // elements behind the last whole lane: a task of their own, behind the chunks
  const uint32_t tasks = P.num_chunks + (rest ? 1u : 0u);
  for (uint32_t q = warp * gridDim.x + blockIdx.x; q < tasks; q += gridDim.x * nwarps) {
    const bool end = q == P.num_chunks;
    const uint32_t kq = end ? P.K - 1u - P.k_begin : divide_by(q, P.chunks_per_packet, P.cpp_magic);
    const uint32_t c = end ? 1u : q - kq * P.chunks_per_packet;
    const uint32_t k = P.k_begin + kq;
    const uint32_t in_pkt = c * kSpan + lane * EPL;
    const uint64_t e = end ? P.n - rest : (uint64_t)k * P.P + in_pkt;
    const uint32_t j = divide_by(P.k0 + k, P.pps, P.pps_magic);  // owner W_j of packet k
    if constexpr (kDevCheck) {   // debug build: the chunk's range, in the slab and in every replica
      const uint64_t c0 = end ? e : (uint64_t)k * P.P + (uint64_t)c * kSpan;
      const uint64_t in_packet = end ? rest : P.P - c * kSpan < kSpan ? P.P - c * kSpan : kSpan;   // a chunk ends with its packet
      const uint64_t cl = c0 < P.n ? (P.n - c0 < in_packet ? P.n - c0 : in_packet) : 0;
      if (!tile_ok(P, k, j, c0, cl, kSiteRegister, lane)) continue;
    }
    // Lanes behind a packet's end hold nothing and skip every load, sum and store; they stay for the shuffles.
    const bool live = !end && in_pkt < P.P && e + EPL <= P.n;
    // optimizer state first: it does not depend on the draws
    LaneVec<F32, EPL> rth, rm, rv;
    if (live) {
      rth = lane_load<F32, EPL>(P.master, e);
      if constexpr (OPT == 1) {
        rm = lane_load<F32, EPL>(P.m, e);
        rv = lane_load<F32, EPL>(P.v, e);
      }
    }

    // ---- delivery indicators of this packet (warp-uniform) -------------------
    uint64_t recv = 0, stale = 0, gbad = 0, pbad = 0;
    if (W <= 16 && !P.ghat_prev) {
      // both directions at once: the lower half of the lanes draws the gradient links, the upper half the broadcast links
      const uint32_t i = (uint32_t)lane & 15u;
      const bool down = lane >= 16;
      const uint32_t u = pair_hash(packet_key_of(P.step_key, P.packet_base + k), down ? j : i, down ? i : j);
      bool lost = u < (down ? P.Tp : P.Tg);
      if (P.burst_in) {
        const uint64_t before = P.burst_in[(down ? (size_t)P.K : 0) + k];
        lost = u < ((before >> i) & 1ull ? P.Tstay : P.Tenter);
      }
      lost = lost && i < W && !(i == j && (down || (P.flags & kSelfLossless)));
      const uint32_t b = __ballot_sync(0xFFFFFFFFu, lost);
      gbad = b & 0xFFFFu;
      pbad = b >> 16;
      recv = ~gbad & all_workers;
      stale = pbad;
      if (P.reliable) {
        recv |= P.reliable[k] & all_workers;
        stale &= ~P.reliable[(size_t)P.K + k];
      }
    } else {
      packet_masks<AGG | BCAST>(P, k, j, lane, recv, stale, gbad, pbad);
    }
    const uint32_t cnt = __popcll(recv);
    const uint64_t take = all_workers & ~(ELIDE ? stale | 1ull << j : stale);   // owner-elided replicas: worker j holds no copy of this packet
    if (end) {
      // a lane per worker (and one 32 on): every lane comes by the same sums and the same update
      const uint32_t i0 = lane, i1 = lane + 32;
      float own0[EPL], own1[EPL], old0[EPL], old1[EPL], g[EPL], th[EPL], m[EPL], v[EPL];
      auto bit = [](uint64_t set, uint32_t i) { return ((set >> i) & 1ull) != 0; };
#pragma unroll
      for (int x = 0; x < EPL; ++x) {
        const bool in = (uint32_t)x < rest;
        own0[x] = in && bit(recv, i0) ? load_one<GT>(P.grads[i0], e + x) : 0.0f;
        own1[x] = in && bit(recv, i1) ? load_one<GT>(P.grads[i1], e + x) : 0.0f;
        old0[x] = DRIFTK && in && bit(stale, i0) ? load_one<RT>(P.replicas[i0], rep_at(i0, j, e + x)) : 0.0f;
        old1[x] = DRIFTK && in && bit(stale, i1) ? load_one<RT>(P.replicas[i1], rep_at(i1, j, e + x)) : 0.0f;
        th[x] = in ? P.master[e + x] : 0.0f;
        m[x] = OPT == 1 && in ? P.m[e + x] : 0.0f;
        v[x] = OPT == 1 && in ? P.v[e + x] : 0.0f;
        g[x] = 0.0f;
      }
      for (uint32_t i = 0; i < W; ++i)
#pragma unroll
        for (int x = 0; x < EPL; ++x) g[x] = __fadd_rn(g[x], __shfl_sync(0xFFFFFFFFu, i < 32 ? own0[x] : own1[x], (int)(i & 31u)));
      divide_by_count<EPL>(g, cnt);
#pragma unroll
      for (int x = 0; x < EPL; ++x) {
        if (P.ghat_prev && (uint32_t)x < rest) {
          if (cnt == 0) g[x] = P.ghat_prev[e + x];
          else if (lane == 0) P.ghat_prev[e + x] = g[x];
        }
        if (P.ghat && (uint32_t)x < rest && lane == 0) P.ghat[e + x] = g[x];
      }
      if (!((P.flags & kZeroSkip) && cnt == 0)) {
        optimizer_n<OPT, EPL>(P, g, th, m, v);
        if (lane == 0)
#pragma unroll
          for (int x = 0; x < EPL; ++x)
            if ((uint32_t)x < rest) {
              P.master[e + x] = th[x];
              if constexpr (OPT == 1) {
                P.m[e + x] = m[x];
                P.v[e + x] = v[x];
              }
            }
      }
      const LaneVec<RT, EPL> wire = lane_narrow<RT, EPL>(th);
      float xw[EPL], sq0 = 0.0f, sq1 = 0.0f;
      lane_widen<RT, EPL>(wire, xw);
#pragma unroll
      for (int x = 0; x < EPL; ++x) {
        if ((uint32_t)x >= rest) continue;
        const typename RT::raw out = lane_element<RT, EPL>(wire, x);
        if (bit(take, i0)) reinterpret_cast<typename RT::raw*>(P.replicas[i0])[rep_at(i0, j, e + x)] = out;
        if (bit(take, i1)) reinterpret_cast<typename RT::raw*>(P.replicas[i1])[rep_at(i1, j, e + x)] = out;
        const float d0 = bit(stale, i0) ? __fsub_rn(old0[x], xw[x]) : 0.0f, d1 = bit(stale, i1) ? __fsub_rn(old1[x], xw[x]) : 0.0f;
        sq0 = __fadd_rn(sq0, __fmul_rn(d0, d0));
        sq1 = __fadd_rn(sq1, __fmul_rn(d1, d1));
      }
      if constexpr (DRIFTK) {
        dsum[warp * kMaxW + lane] += (double)sq0;
        dsum[warp * kMaxW + lane + 32] += (double)sq1;
      }
      continue;
    }
    if (c == 0 && lane == 0) {
      if (P.count) P.count[k] = (uint8_t)cnt;
      if (P.recv_bits) P.recv_bits[k] = recv;
      if (P.stale_bits) P.stale_bits[k] = stale;
      if (P.burst_out) {   // the first chunk of a packet stores its links' new states
        P.burst_out[k] = gbad;
        P.burst_out[(size_t)P.K + k] = pbad;
      }
    }

    // ---- old copies of the replicas that miss the broadcast: the first kB requested now, the rest started toward L2 ------
    uint64_t todo = DRIFTK ? stale : 0ull;
    uint64_t batch = 0;                        // the copies in `old`, in ascending order
    int nb = 0;
    LaneVec<RT, EPL> old[kB];
    auto request = [&]() {
      batch = todo;
      nb = 0;
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        if (todo) {
          const uint32_t i = (uint32_t)__ffsll((long long)todo) - 1u;
          todo &= todo - 1;
          nb = b + 1;
          if (live) old[b] = lane_load<RT, EPL>(P.replicas[i], rep_at(i, j, e));
        }
      }
      batch ^= todo;
    };
    if constexpr (DRIFTK) {
      request();
      if (live)
        for (uint64_t sm = todo; sm; sm &= sm - 1) {
          const uint32_t i = (uint32_t)__ffsll((long long)sm) - 1u;
          prefetch_l2(reinterpret_cast<const typename RT::raw*>(P.replicas[i]) + rep_at(i, j, e));
        }
    }

    // ---- (2) unbiased aggregate: masked sum in ascending worker order / count --
    LaneVec<RT, EPL> wire = {};
    if (live) {
      float g[EPL], th[EPL];
#pragma unroll
      for (int x = 0; x < EPL; ++x) g[x] = 0.0f;
      for (uint32_t g0 = 0; g0 < (FORM == kStepFew ? 1u : W); g0 += kG) {
        const uint32_t bits = (uint32_t)(recv >> g0) & ((1u << kG) - 1u);
        LaneVec<GT, EPL> raw[kG];
#pragma unroll
        for (int u = 0; u < kG; ++u) raw[u] = lane_load<GT, EPL>(P.grads[g0 + u], e, bits & (1u << u));
#pragma unroll
        for (int u = 0; u < kG; ++u) lane_add<GT, EPL>(raw[u], g);
      }
      divide_by_count<EPL, true>(g, cnt);
      if (P.ghat_prev) {
        // Algorithm 1: a dropped packet falls back to the saved aggregate, a surviving one is saved
        if (cnt == 0) lane_widen<F32, EPL>(lane_load<F32, EPL>(P.ghat_prev, e), g);
        else lane_store<F32, EPL>(P.ghat_prev, e, lane_narrow<F32, EPL>(g));
      }
      if (P.ghat) lane_store<F32, EPL>(P.ghat, e, lane_narrow<F32, EPL>(g));

      // ---- (3) the owner's update ------------------------------------------------
      lane_widen<F32, EPL>(rth, th);
      if (!((P.flags & kZeroSkip) && cnt == 0)) {
        float m[EPL], v[EPL];
        if constexpr (OPT == 1) {
          lane_widen<F32, EPL>(rm, m);
          lane_widen<F32, EPL>(rv, v);
        }
        optimizer_n<OPT, EPL>(P, g, th, m, v);
        lane_store<F32, EPL>(P.master, e, lane_narrow<F32, EPL>(th));
        if constexpr (OPT == 1) {
          lane_store<F32, EPL>(P.m, e, lane_narrow<F32, EPL>(m));
          lane_store<F32, EPL>(P.v, e, lane_narrow<F32, EPL>(v));
        }
      }

      // ---- (4) broadcast with stale retention --------------------------------------
      wire = lane_narrow<RT, EPL>(th);
      for (uint32_t i0 = 0; i0 < (FORM == kStepFew ? 1u : W); i0 += kS) {
        const uint32_t bits = (uint32_t)(take >> i0);
#pragma unroll
        for (int u = 0; u < kS; ++u) lane_store<RT, EPL>(P.replicas[i0 + u], rep_at(i0 + u, j, e), wire, bits & (1u << u));
      }
    }

    // ---- the drift of the copies that differ ------------------------------------------
    // A lane's squares are added in fp32, everything else in fp64, as the pairwise drift's are: bf16 copies
    // N(0, 3e-4) apart come out 3e-10 low, with a tree of 256 squares in fp32 8.8e-9, and the pipelines' 128 squares, whose
    // small buckets this kernel takes, 6.0e-9.
    if constexpr (DRIFTK) {
      float xw[EPL];
      lane_widen<RT, EPL>(wire, xw);
      while (nb) {
        float sq[kB];
#pragma unroll
        for (int b = 0; b < kB; ++b) sq[b] = b < nb && live ? lane_squares<RT, EPL>(old[b], xw) : 0.0f;
        double tot;
        int seg = 32;                      // lanes of a segment, whose first lane adds the segment's copy's total
        if (kB == 8 && nb > 4) {
          tot = totals_of<kB>(sq, lane, seg);
        } else if (kB >= 4 && nb > 2) {
          tot = totals_of<kB < 4 ? kB : 4>(sq, lane, seg);
        } else if (nb == 2) {
          tot = totals_of<2>(sq, lane, seg);
        } else {
          tot = warp_sum64((double)sq[0]);
        }
        const int to = lane / seg;
        if (lane % seg == 0 && to < nb) {
          for (int b = 0; b < to; ++b) batch &= batch - 1;
          dsum[warp * kMaxW + __ffsll((long long)batch) - 1] += tot;
        }
        __syncwarp();                      // (another lane may add to this copy's sum next time)
        request();
      }
    }
  }
  if constexpr (DRIFTK) drift_finish(P, dsum, (int)nwarps, P.partials_row0 + blockIdx.x, warp, (int)nwarps, lane);
  if constexpr (TAIL) end_after_previous(P);
}

}  // namespace lossy
