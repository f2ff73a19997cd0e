// C ABI of the lossy data-parallel step (see include/lossy.h for the contract).
// Host side: argument validation, threshold and hash-key derivation, launches.
#include "../../include/lossy.h"

#include <math.h>
#include <stdio.h>
#include <string.h>

#include <mutex>
#include <new>
#include <type_traits>

#include "lossy_diag.cuh"
#include "lossy_gather.cuh"
#include "lossy_phase_tma.cuh"
#include "lossy_register.cuh"

using namespace lossy;

// Where the gather pipeline is used, and which of its builds (gather_policy)
struct GatherPolicy {
  bool use;
  bool wide;          // 2048-element tiles, one CTA per SM (else 1024, two)
  bool drift_warps;   // warps of their own read the stale copies
  bool small[2];      // (with drift norms: [1]) a small bucket: the step kernel, none of the pipelines
};

struct lossy_ctx {
  lossy_config cfg;
  GatherPolicy gather;   // depends on cfg and the device alone: decided once, in lossy_init
  uint64_t K;
  uint32_t chunks_per_packet;
  uint32_t num_chunks;
  uint32_t pps;
  uint32_t Tg, Tp;
  int device;
  int num_sms;
  uint32_t max_blocks;   // capacity of `partials`
  double* partials;      // device, [max_blocks][kMaxW], followed by the status word
  uint32_t* status;      // device status words: [0] 0 = fine, 1 = a bounded wait in a kernel gave up; [1..4] debug build: a failed index check
  uint64_t check_shrink; // debug build self-test: the index checks hold ranges against n - check_shrink
  uint32_t* ticket;      // device counter of finished blocks (last-block drift finalisation), zero between calls
  uint32_t* gate;        // device word by which a call's two launches tell that the kernels ahead of them are done, zero between calls
  uint32_t calls;        // number of the last call that may have two launches
  bool plan_only;        // launch helpers only report their grid size
  const uint64_t* reliable;  // caller-owned device array [2][K] of reliable-link bits, or NULL
  uint64_t* burst_state; // bursty loss: caller-owned device array [2 buffers][2 rows][K], or NULL
  uint32_t Tenter, Tstay;
  int smem_optin;        // largest dynamic shared memory a block may opt in to
  uint64_t launches;
  char* plan;            // lossy_describe_plan: where try_tma notes the build it would launch (else NULL)
  size_t plan_size;
  char err[256];
};

namespace {

constexpr int kBlocksPerSmCap = 8;

int fail(lossy_ctx* ctx, int code, const char* msg) {
  if (ctx) snprintf(ctx->err, sizeof ctx->err, "%s", msg);
  return code;
}
// The caller gets the error from here; in the runtime it is cleared, or the next look at the last error, behind a launch that
// went well, would find it there.
int fail_cuda(lossy_ctx* ctx, const char* what, cudaError_t e) {
  cudaGetLastError();
  if (ctx) snprintf(ctx->err, sizeof ctx->err, "%s: %s", what, cudaGetErrorString(e));
  return LOSSY_ECUDA;
}
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

uint32_t threshold_of(double p) { return (uint32_t)floor(p * 4294967296.0); }

int check_table(lossy_ctx* ctx, const void* const* tab, const char* name) {
  if (!tab) return fail(ctx, LOSSY_EINVAL, name);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i)
    if (!tab[i] || !aligned16(tab[i])) return fail(ctx, LOSSY_EINVAL, name);
  return LOSSY_OK;
}

// elements of worker i's shard inside this context's packet range (what an owner-elided replica leaves out)
uint64_t own_elems(const lossy_ctx* ctx, uint32_t i) {
  const lossy_config& c = ctx->cfg;
  const uint64_t s0 = (uint64_t)i * ctx->pps, s1 = s0 + ctx->pps;
  const uint64_t c0 = c.shard_packet0, c1 = c.shard_packet0 + ctx->K;
  const uint64_t lo = s0 > c0 ? s0 : c0, hi = s1 < c1 ? s1 : c1;
  if (lo >= hi) return 0;
  const uint64_t e0 = (lo - c0) * c.packet_elems, e1 = (hi - c0) * c.packet_elems;
  return (e1 < c.n ? e1 : c.n) - (e0 < c.n ? e0 : c.n);
}

// The replica table: W aligned device pointers; an owner-elided replica that holds nothing may be NULL.
int check_replicas(lossy_ctx* ctx, const void* const* tab) {
  const char* name = "replicas: NULL or misaligned pointer";
  if (!tab) return fail(ctx, LOSSY_EINVAL, name);
  const bool elide = ctx->cfg.flags & LOSSY_REPLICA_SKIP_OWNER;
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) {
    if (elide && own_elems(ctx, i) == ctx->cfg.n) continue;
    if (!tab[i] || !aligned16(tab[i])) return fail(ctx, LOSSY_EINVAL, name);
  }
  return LOSSY_OK;
}

// A launch with programmatic stream serialisation: the kernel may be set up while the kernel ahead of it in the stream still
// runs, and waits for that one's end itself (wait_for_previous). Behind anything but a kernel, or behind one that does not
// give leave, it is an ordinary launch. Host time of a launch: 1.8 us instead of 2.4; W = 8, P = 2048, n = 262 k, in a graph: 10.6 ->
// 9.4 us a step; with a short last packet on a launch of its own (n = 262 184): 20.0 -> 11.4.
// early = false, an ordinary launch: for kernels that load through L1 and run long. A block that begins early gets what
// shared memory the kernel ahead has left its SM, after a gather pipeline 28 KB of L1 (closed-loop gradients of 58 M elements
// behind it: 690 -> 755 us for the pair; packet norms behind the pairwise drift, W = 9, n = 4.6 M: 92 -> 97 us). And for kernels of which
// several blocks fit an SM, from a number of blocks on: those that begin early crowd the SMs that come free first. The closed loop's
// gradients, packet norms and a broadcast begin early up to the numbers at their launches (closed loop, W = 10, 96 k: 16.4 -> 14.8 us).
// The pairwise drift never does: its set kernel loads through the read-only path, which must not run beside the writes of a step
// ahead, and there is nothing to gain (850 small buckets, behind the memset of the matrix that the call adds to: 0.97 to 1.00 of the
// ordinary launch's speed).
template <class... Formal, class... Actual>
cudaError_t launch_after(bool early, void (*kern)(Formal...), dim3 grid, uint32_t threads, size_t smem, cudaStream_t s, const Actual&... args) {
  cudaLaunchAttribute at[1] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  // (the arguments where they lie: cudaLaunchKernelEx copies them, 2 KB, once more)
  static_assert((std::is_same<Formal, Actual>::value && ...), "a kernel's arguments as it declares them");
  void* argv[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kern), argv);
}

// A call's one launch: its blocks' rows are all (two launches: the caller has counted them ahead).
void rows_of_call(Params& P, uint32_t blocks) { if (P.total_rows == 0u) P.total_rows = blocks; }

// behind a call that failed: a ticketed launch may already be queued, and the counter must be zero again before the next call
void reset_ticket(lossy_ctx* ctx, cudaStream_t s) {
  if (cudaMemsetAsync(ctx->ticket, 0, sizeof(uint32_t), s) != cudaSuccess) cudaGetLastError();
}

void fill_common(lossy_ctx* ctx, uint64_t step, Params& P) {
  memset(&P, 0, sizeof P);
  const lossy_config& c = ctx->cfg;
  P.n = c.n;
  P.packet_base = c.packet_base + c.shard_packet0;   // the hash sees the global id of every packet
  P.k0 = (uint32_t)c.shard_packet0;
  P.step_key = step_key_of(c.seed, step);
  P.num_chunks = ctx->num_chunks;
  P.chunks_per_packet = ctx->chunks_per_packet;
  P.pps = ctx->pps;
  P.P = c.packet_elems;
  P.W = c.W;
  P.Tg = ctx->Tg;
  P.Tp = ctx->Tp;
  P.flags = c.flags;
  P.lr = c.lr;
  P.b1 = c.beta1;
  P.b2 = c.beta2;
  P.omb1 = 1.0f - c.beta1;   // (1 - beta) in fp32
  P.omb2 = 1.0f - c.beta2;
  P.ibc1 = (float)(1.0 / (1.0 - pow((double)c.beta1, (double)step)));
  P.ibc2 = (float)(1.0 / (1.0 - pow((double)c.beta2, (double)step)));
  P.eps = c.eps;
  P.neg_zero = -0.0f;
  P.partials = ctx->partials;
  P.K = (uint32_t)ctx->K;
  P.reliable = ctx->reliable;
#ifdef LOSSY_DEVCHECK
  P.check = ctx->status + 1;
  P.check_n = c.n - (ctx->check_shrink < c.n ? ctx->check_shrink : c.n);
#endif
  if (c.n % c.packet_elems != 0) {   // the short last packet may have a launch of its own
    if (++ctx->calls == 0u) ctx->calls = 1u;
    P.gate = ctx->gate;
    P.gate_id = ctx->calls;
  }
  fill_rep_skip(P, (c.flags & LOSSY_REPLICA_SKIP_OWNER) != 0);
  if (ctx->burst_state) {
    // the states after step t-1 live in buffer (t-1)&1, those after step t go to buffer t&1
    const size_t buf = 2 * (size_t)ctx->K;
    P.burst_in = ctx->burst_state + ((step - 1) & 1u) * buf;
    P.burst_out = ctx->burst_state + (step & 1u) * buf;
    P.Tenter = ctx->Tenter;
    P.Tstay = ctx->Tstay;
  }
}

// ---- bulk-copy pipeline (fused step only) --------------------------------------------------
constexpr uint32_t kTmaSmemFixed = kTmaBarBytes + kMaxStages * (sizeof(StageHdr) + sizeof(PackedStale)) + kMaskBufs * sizeof(PackedMasks);

// Launch policy of the bulk-copy pipeline, from sweeps on B200 over W = 2..64, p = 0.05..0.3
// (CUDA-event timings of bench.py with each build forced): which of the four builds runs and whether its bulk copies carry an
// L2 evict-first hint (bit 0 loads, bit 1 stores).
struct TmaPolicy {
  bool wide;      // 16 compute warps, one CTA per SM, 2048-element tiles (else 8 warps, two CTAs, 1024)
  int group;      // workers per pipeline stage: 4 or 8
  int early_stale;   // stale copies: 0 = fetched in the drift phase, 16 = first ones requested before the tile's arithmetic, 1 = extra pipeline stages (stages of 8 only)
  uint32_t hints;
  bool split;     // state slots apart from the stages (twin build, stages of 8, high loss)
  uint32_t split_stages;
};
TmaPolicy tma_policy(const lossy_config& c) {
  const double pm = c.p_grad > c.p_param ? c.p_grad : c.p_param;
  TmaPolicy t;
  // wide tiles win whenever a tile takes at most two 8-worker groups and the packet is a multiple of the tile
  t.wide = c.W <= 16 && c.packet_elems % TmaShape<16>::kTile == 0;
  // stages of 4 workers (finer-grained pipeline) win for few workers at low loss: +5 % at W = 8, p = 0.1,
  // but -9 % at W = 8, p = 0.3; the crossover at W = 8 sits near p = 0.17
  t.group = c.W <= 4 ? 4 : (c.W <= 8 && pm < 0.175 ? 4 : 8);
  // hints: +2-4 % on the twin build at high loss, or at W = 64 from moderate loss (p = 0.1: 0.957 against
  // 0.934); neutral to -2 % elsewhere (W = 64, p = 0.01: 0.944 against 0.961)
  t.hints = t.wide ? (pm >= 0.28 ? 3u : 0u) : ((pm >= 0.2 || (c.W > 32 && pm >= 0.05)) ? 3u : 0u);
  // early stale requests pay from about two stale replicas per tile at high loss: +8-10 % at W >= 16,
  // p = 0.3; at p = 0.1 they lose 1-2 % even with six stale replicas per tile (W = 64)
  t.early_stale = t.group == 8 && (c.W - 1) * c.p_param >= 2.0 && c.p_param >= 0.15 ? 16 : 0;
  // State slots apart from the stages (one more gradient stage fits): the twin build at p >= 0.2, where the
  // compute warps spend long on stale replicas and the extra stage keeps the loads going meanwhile: W = 32,
  // p = 0.3: 0.89 -> 0.96; W = 48, p = 0.2: 0.91 -> 0.97; W = 64, p = 0.3: 0.90 -> 0.95. The fourth stage pays
  // from about 6.5 stale replicas per tile; below that three (W = 24, p = 0.2: 0.93 -> 0.95), and at lower
  // loss the plain build is as fast or faster (W = 64, p = 0.1: 0.96 against 0.94 with four stages).
  t.split = !t.wide && t.group == 8 && c.W > 16 && c.p_param >= 0.2;
  t.split_stages = (c.W - 1) * c.p_param >= 6.5 ? 4u : 3u;
  // With the fourth stage the stale replicas' old copies come through the pipeline as extra stages instead
  // of being read by the compute warps (W = 64, p = 0.3: 0.88 -> 0.95; W = 48, p = 0.3: 0.91 -> 0.97; W = 17,
  // p = 0.5: 0.71 -> 0.79); with fewer stale replicas per tile the early requests stay ahead (W = 24, p = 0.2:
  // 0.95 against 0.92).
  if (t.split && t.split_stages == 4u) t.early_stale = 1;
  return t;
}

constexpr int kMaxDevices = 64;
// The launch helpers below remember, per kernel instantiation and device, what they set up once (the raised
// shared-memory limit, the occupancy). Those tables are process-wide, so host threads that drive different
// contexts take this lock around the look-up; it is never held across a launch.
std::mutex g_setup_mu;

// Dynamic shared memory one CTA of the bulk-copy kernel may use: the CTAs of one SM share 227 KB.
template <int CW>
uint32_t tma_smem_budget(const lossy_ctx* ctx) {
  uint32_t budget = (227u * 1024u) / TmaShape<CW>::kCtasPerSm - 1024u;
  if ((uint32_t)ctx->smem_optin < budget) budget = (uint32_t)ctx->smem_optin;
  return budget;
}

// Dynamic shared memory a launch asks for. Blocks that may begin while the kernel ahead still runs go to the SMs that are
// free first, as many as fit: a kernel of one block per SM that needs less than half an SM's memory was then laid out two by
// two (the four single-phase calls, W = 8: 135 M elements 1830 -> 2031 us, 1 M 28.2 -> 30.5). So each block asks for enough
// that no more than `per_sm` of them fit. What it asks for, kernels of other streams cannot have: four streams of single-phase calls
// on 1 M elements each take 25.2 us a call sequence, without this 20.6 (two streams 25.0 and 22.7, one 31.7 and 34.6). One block per SM
// also for grids of two per SM that are smaller than the chip gained 0 to 3 % on one stream and cost four of them
// (W = 4, P = 1024, 131 k elements, fused: 2.3 -> 4.0 us a step).
uint32_t spread_smem(const lossy_ctx* ctx, uint32_t smem, uint32_t per_sm) {
  const uint32_t least = 228u * 1024u / (per_sm + 1u), most = (uint32_t)ctx->smem_optin - 1024u;
  return smem >= least ? smem : least < most ? least : most;
}

template <int CW, int GS, bool PACKED, bool SPLIT>
bool tma_geometry(const lossy_ctx* ctx, TmaGeom& G) {
  constexpr uint32_t kGroup = GS;
  constexpr uint32_t kTile = TmaShape<CW>::kTile;
  const lossy_config& c = ctx->cfg;
  const uint64_t kfull = c.n / c.packet_elems;               // packets that are complete
  if (kfull == 0 || kfull >= (1ull << 31)) return false;
  G.packets_per_tile = 1;
  G.full_packets = (uint32_t)kfull;
  if (PACKED) {
    // small packets: a tile packs 2, 4 or 8 whole packets; a compute warp's 128 elements stay inside one
    if (c.packet_elems >= kTile || kTile % c.packet_elems != 0 || c.packet_elems % 128 != 0 ||
        kTile / c.packet_elems > (uint32_t)kMaxSub)
      return false;
    G.packets_per_tile = kTile / c.packet_elems;
  } else if (c.packet_elems < kTile) {
    return false;
  }
  const uint32_t gb = c.grad_dtype == LOSSY_BF16 ? 2 : 4, rb = c.replica_dtype == LOSSY_BF16 ? 2 : 4;
  G.grad_slots = c.W < (uint32_t)kGroup ? c.W : (uint32_t)kGroup;
  G.groups = (c.W + kGroup - 1) / kGroup;
  const uint32_t state = 3 * kTile * 4 + kTile * rb;           // theta, m, v and the wire tile
  const uint32_t sb = G.grad_slots * kTile * gb + (SPLIT ? 0u : state);
  G.stage_bytes = (sb + 127u) & ~127u;
  G.state_bytes = SPLIT ? (state + 127u) & ~127u : 0u;
  // behind the stages: the two state slots of the SPLIT builds, and fp64 drift sums per compute warp and
  // replica (used by the stale-stage builds)
  const uint32_t budget = tma_smem_budget<CW>(ctx) - CW * kMaxW * (uint32_t)sizeof(double) - 2u * G.state_bytes;
  if (budget < kTmaSmemFixed + 2 * G.stage_bytes) return false;
  G.stages = (budget - kTmaSmemFixed) / G.stage_bytes;
  const uint32_t cap = SPLIT ? tma_policy(c).split_stages : 4u;   // with the state in the stage a fifth measured no faster
  if (G.stages > cap) G.stages = cap;
  // One tile per stage (a single worker group): with a fourth stage the loads run too far ahead of the
  // stores (W = 4, p = 0.1: 0.98 of the copy rate with three stages, 0.92 with four; W = 2: 0.96 / 0.95);
  // a single worker still gains from the fourth (0.97 / 0.91).
  if (G.groups == 1 && c.W >= 2 && G.stages > 3u) G.stages = 3u;
  G.tiles_per_packet = PACKED ? 1u : (c.packet_elems + kTile - 1) / kTile;
  const uint64_t tiles = PACKED ? (kfull + G.packets_per_tile - 1) / G.packets_per_tile : kfull * G.tiles_per_packet;
  if (tiles >= (1ull << 31)) return false;
  G.num_tiles = (uint32_t)tiles;
  G.status = ctx->status;
  G.hints = tma_policy(c).hints;
  return true;
}

template <class GT, class RT, int OPT, bool DRIFTK, int CW, int GS, int PRE, bool PACKED, bool SPLIT>
int launch_tma(lossy_ctx* ctx, Params& P, const TmaGeom& G, cudaStream_t s, uint32_t* blocks_out) {
  auto kern = lossy_fused_tma_kernel<GT, RT, OPT, DRIFTK, CW, GS, PRE, PACKED, SPLIT>;
  constexpr int kThreadsTma = TmaShape<CW>::kThreads;
  const uint32_t smem = kTmaSmemFixed + G.stages * G.stage_bytes + 2u * G.state_bytes + CW * kMaxW * (uint32_t)sizeof(double);
  // launch bounds and the shared-memory budget guarantee kCtasPerSm resident CTAs per SM
  uint32_t blocks = (uint32_t)(ctx->num_sms * TmaShape<CW>::kCtasPerSm);
  if (blocks > G.num_tiles) blocks = G.num_tiles;
  *blocks_out = blocks;
  if (ctx->plan_only) return LOSSY_OK;
  rows_of_call(P, blocks);
  static bool opted_in[kMaxDevices];   // per kernel instantiation and device: raise the dynamic shared memory limit once
  cudaError_t e;
  {
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (ctx->device >= kMaxDevices || !opted_in[ctx->device]) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin - 1024);   // (less what is static)
      if (e != cudaSuccess) return fail_cuda(ctx, "shared memory opt-in", e);
      if (ctx->device < kMaxDevices) opted_in[ctx->device] = true;
    }
  }
  e = launch_after(true, kern, blocks, kThreadsTma, spread_smem(ctx, smem, TmaShape<CW>::kCtasPerSm), s, P, G);
  if (e != cudaSuccess) return fail_cuda(ctx, "bulk-copy kernel launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

template <bool DRIFTK, int CW, int GS, int PRE, bool PACKED, bool SPLIT>
int dispatch_tma(lossy_ctx* ctx, Params& P, const TmaGeom& G, cudaStream_t s, uint32_t* blocks) {
  const bool gb = ctx->cfg.grad_dtype == LOSSY_BF16;
  const bool rb = ctx->cfg.replica_dtype == LOSSY_BF16;
  const bool adam = ctx->cfg.optimizer == LOSSY_ADAM;
  if (gb && rb) return adam ? launch_tma<BF16, BF16, 1, DRIFTK, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks) : launch_tma<BF16, BF16, 0, DRIFTK, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks);
  // stale copies as pipeline stages (PRE = 1) reuse the gradient slots: fp32 replicas with bf16 gradients do not fit
  constexpr int PRE_WIDER = PRE == 1 ? 16 : PRE;
  if (gb && !rb) return adam ? launch_tma<BF16, F32, 1, DRIFTK, CW, GS, PRE_WIDER, PACKED, SPLIT>(ctx, P, G, s, blocks) : launch_tma<BF16, F32, 0, DRIFTK, CW, GS, PRE_WIDER, PACKED, SPLIT>(ctx, P, G, s, blocks);
  if (!gb && rb) return adam ? launch_tma<F32, BF16, 1, DRIFTK, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks) : launch_tma<F32, BF16, 0, DRIFTK, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks);
  return adam ? launch_tma<F32, F32, 1, DRIFTK, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks) : launch_tma<F32, F32, 0, DRIFTK, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks);
}

template <int CW, int GS, int PRE = 0, bool PACKED = false, bool SPLIT = false>
int try_tma(lossy_ctx* ctx, Params& P, bool drift, cudaStream_t s, uint32_t* blocks, bool* used) {
  TmaGeom G = {};
  if (!tma_geometry<CW, GS, PACKED, SPLIT>(ctx, G)) return LOSSY_OK;
  *used = true;
  if (ctx->plan) {
    // dispatch_tma runs the early-request build where staged copies do not fit the gradient slots
    const bool fits = !(ctx->cfg.grad_dtype == LOSSY_BF16 && ctx->cfg.replica_dtype == LOSSY_F32);
    snprintf(ctx->plan, ctx->plan_size, "bulk-copy %s group=%d stale=%s%s%s stages=%u", CW == 16 ? "wide" : "twin", GS,
             !drift || PRE == 0 ? "late" : PRE == 1 && fits ? "staged" : "early", PACKED ? " packed" : "",
             SPLIT ? " split" : "", G.stages);
  }
  // without drift norms nothing reads the stale copies: the plain build serves
  return drift ? dispatch_tma<true, CW, GS, PRE, PACKED, SPLIT>(ctx, P, G, s, blocks)
               : dispatch_tma<false, CW, GS, 0, PACKED, SPLIT>(ctx, P, G, s, blocks);
}

// ---- gather pipeline (packets shorter than a tile) ------------------------------------------
// barriers, the ring of tile masks, stage headers; the drift sums per compute warp, the wire ring and the stages follow
template <bool ANY> constexpr uint32_t kGatherSmemFixed =
    kGatherBarBytes + kGatherRing * sizeof(TileMasks<ANY ? kAnySub : kMaxSub>) + kGatherMaxStages * sizeof(StageHdr);

// rd: the stale copies are read outside the compute warps (twin geometry: by the replica warps, one replica each;
// wide geometry: by drift warps of their own)
template <int CW, bool ANY>
bool gather_geometry(const lossy_ctx* ctx, bool rd, TmaGeom& G) {
  constexpr uint32_t kTile = GatherShape<CW>::kTile;
  const lossy_config& c = ctx->cfg;
  const uint64_t kfull = c.n / c.packet_elems;               // packets that are complete
  if (kfull == 0 || kfull >= (1ull << 31)) return false;
  // !ANY: packets that divide the tile (powers of two), kMaxSub of them at most. ANY: all others, short or long, laid
  // over the tiles as they come (multiples of 8 elements), from 128 elements (a compute warp's 128 elements then lie in
  // at most two packets) and as long as a tile touches at most kAnySub of them.
  const uint32_t P = c.packet_elems;
  if (P < 128u || P >= (1u << 15) || ANY != (kTile % P != 0) || (!ANY && P >= kTile)) return false;
  const uint32_t touched = ANY ? (P - 8u + kTile - 1u) / P + 1u : kTile / P;
  if (touched > (uint32_t)(ANY ? kAnySub : kMaxSub)) return false;
  memset(&G, 0, sizeof G);
  G.packets_per_tile = touched;
  G.magic = (uint32_t)(((1ull << 32) + P - 1u) / P);
  G.full_packets = (uint32_t)kfull;
  const uint32_t gb = c.grad_dtype == LOSSY_BF16 ? 2 : 4, rb = c.replica_dtype == LOSSY_BF16 ? 2 : 4;
  G.grad_slots = c.W < 8u ? c.W : 8u;
  G.groups = (c.W + 7u) / 8u;
  // a stage holds the group's gradient rows and theta, m, v
  G.stage_bytes = (G.grad_slots * kTile * gb + 3 * kTile * 4 + 127u) & ~127u;
  // fp64 drift sums per adding warp and replica, the wire ring, and (rd) the scratch for the stale copies
  G.state_bytes = (uint32_t)(rd ? GatherShape<CW, true>::kAccRows : CW) * kMaxW * (uint32_t)sizeof(double) + kWireRing * kTile * rb;
  const uint32_t row_chunks = kTile * rb / 512u;             // 512-byte chunks of one replica's row of a tile
  uint32_t scratch_unit = 0;                                  // bytes of scratch per chunk of capacity
  if (rd) {
    using Shape = GatherShape<CW, true>;
    scratch_unit = (uint32_t)(Shape::kDriftWarps ? Shape::kDriftWarps : Shape::kReplicaWarps) * Shape::kRdBuffers * 512u;
    // twin: a replica warp owns one replica, its whole row fits; wide: at least four chunks per drift warp, more below
    G.rd_cap = Shape::kDriftWarps ? 4u : row_chunks;
    G.state_bytes += G.rd_cap * scratch_unit;
  }
  const uint32_t budget = (227u * 1024u) / GatherShape<CW>::kCtasPerSm - 1024u;
  const uint32_t avail = (uint32_t)ctx->smem_optin < budget ? (uint32_t)ctx->smem_optin : budget;
  if (avail < kGatherSmemFixed<ANY> + G.state_bytes + 2 * G.stage_bytes) return false;
  G.stages = (avail - kGatherSmemFixed<ANY> - G.state_bytes) / G.stage_bytes;
  if (G.stages > 4u) G.stages = 4u;                           // more measured no faster (W = 2..32)
  if (rd && GatherShape<CW, true>::kDriftWarps) {
    // wide: what the stages leave goes to the scratch, up to every chunk of a drift warp's replicas
    const uint32_t left = avail - kGatherSmemFixed<ANY> - G.state_bytes - G.stages * G.stage_bytes;
    // a replica's row in 2^lgsplit parts, W * 2^lgsplit parts dealt round robin: the fewest parts that balance the drift warps
    const uint32_t nd = GatherShape<CW, true>::kDriftWarps;
    // (a warp's cost: its share of a row, plus about a sixteenth of a row per part whatever the part holds: W = 17 in 8
    // parts per row, 17 parts per warp, ran at 0.56 where W = 16 in whole rows, 2 per warp, ran at 0.85; W = 12 in
    // halves 0.79 against 0.74 in whole rows; W = 5, P = 512 in quarters 0.86 against 0.83)
    uint32_t best = ~0u, share = 8u;
    for (uint32_t lg = 0; lg <= 2u; ++lg) {
      const uint32_t parts = ((c.W << lg) + nd - 1u) / nd;                   // a warp's parts ...
      const uint32_t eighths = parts * (8u >> lg);                            // ... and its share in eighths of a row
      const uint32_t cost = 2u * eighths + parts;
      if (cost < best) { best = cost; share = eighths; G.rd_lgsplit = lg; }
    }
    const uint32_t most = (share * row_chunks + 7u) / 8u;
    uint32_t more = left / scratch_unit;
    if (G.rd_cap + more > most) more = most > G.rd_cap ? most - G.rd_cap : 0u;
    G.rd_cap += more;
    G.state_bytes += more * scratch_unit;
    // A drift warp's stale chunks of a tile should mostly fit its scratch: what does not fit is loaded directly at
    // its full latency. Where not even their mean count fits (fp32 replicas, whose wire ring takes the room: a
    // scratch of 4 chunks for a mean of 9) the compute warps' reads serve better; the caller falls back to them,
    // unless it was told to use this build (LOSSY_GATHER_PATH: comparison and tests). (W = 16, P = 256, p = 0.3,
    // bf16: 8 chunks for a mean of 4.5; W = 24: 8 for 6.9.) The line differs for the ANY builds (625 random steps of eight and
    // more tiles per SM): bf16 replicas are ahead with drift warps by 5-15 % up to a mean of 0.8 scratches, even at 1.25, behind
    // from there on (two scratches: 0.90); fp32 ones ahead by 5-10 % up to 0.4 and behind from 0.6 (0.95; two: 0.72).
    // (a 512-byte chunk that touches several packets is read if any of them is stale)
    const double chunk_elems = 512.0 / rb, per_chunk = P % (512u / rb) == 0 ? 1.0 : (512u / rb) % P == 0 ? chunk_elems / P : 1.0 + chunk_elems / P;
    const double mean = share / 8.0 * row_chunks * (1.0 - pow(1.0 - c.p_param * (c.W - 1.0) / c.W, per_chunk));
    const double fits = G.rd_cap * (!ANY ? 1.0 : rb == 2u ? 1.25 : 0.5);
    if (!(c.flags & LOSSY_GATHER_PATH) && fits < mean) return false;
  }
  G.tiles_per_packet = 1;
  const uint64_t tiles = (kfull * P + kTile - 1) / kTile;
  if (tiles >= (1ull << 31)) return false;
  G.num_tiles = (uint32_t)tiles;
  G.status = ctx->status;
  // bit 2: the mask warp sends the stale pairs' old copies toward L2 tiles ahead (W = 16, p = 0.1: 0.94 -> 0.99;
  // with more than about two stale replicas per sub-packet it loses: W = 12, p = 0.2: 0.86 -> 0.78)
  G.hints = (c.W - 1) * c.p_param < 1.8 ? 4u : 0u;
  // bit 3: how the wide geometry's two gather warps share a group. Dealing out the workers halves each warp's
  // ballots and is ahead wherever rows have holes (W = 16, P = 256: +1 / +7 / +1 % at p = 0.1 / 0.2 / 0.3; P = 512,
  // p = 0.3: +4 %) and with 9-12 or more than 16 workers at any loss (W = 24: +4 % at p = 0, +6 % at 0.1; W = 64,
  // P = 512: +9 %); where most rows are whole, up to 8 or with 13-16 workers, both warps in one row do better
  // (W = 16: 0.98-0.99 against 0.91-0.94 up to p = 0.05; W = 8: +1 %). Same-process A/B pairs, repeatable to 0.002.
  const double whole_rows = pow(1.0 - c.p_grad, (double)kTile / P);
  if (whole_rows >= 0.6 && (c.W <= 8u || (c.W >= 13u && c.W <= 16u))) G.hints |= 8u;
  return true;
}

template <class GT, class RT, int OPT, bool DRIFTK, int CW, bool RD, bool ANY>
int launch_gather(lossy_ctx* ctx, Params& P, const TmaGeom& G, cudaStream_t s, uint32_t* blocks_out) {
  auto kern = lossy_fused_gather_kernel<GT, RT, OPT, DRIFTK, CW, RD, ANY>;
  const uint32_t smem = kGatherSmemFixed<ANY> + G.state_bytes + G.stages * G.stage_bytes;
  uint32_t blocks = (uint32_t)(ctx->num_sms * GatherShape<CW>::kCtasPerSm);
  if (blocks > G.num_tiles) blocks = G.num_tiles;
  *blocks_out = blocks;
  if (ctx->plan_only) return LOSSY_OK;
  rows_of_call(P, blocks);
  static bool opted_in[kMaxDevices];   // per kernel instantiation and device: raise the dynamic shared memory limit once
  cudaError_t e;
  {
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (ctx->device >= kMaxDevices || !opted_in[ctx->device]) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin - 1024);   // (less what is static)
      if (e != cudaSuccess) return fail_cuda(ctx, "shared memory opt-in", e);
      if (ctx->device < kMaxDevices) opted_in[ctx->device] = true;
    }
  }
  e = launch_after(true, kern, blocks, GatherShape<CW, RD>::kThreads, spread_smem(ctx, smem, GatherShape<CW>::kCtasPerSm), s, P, G);
  if (e != cudaSuccess) return fail_cuda(ctx, "gather kernel launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

template <bool DRIFTK, int CW, bool RD, bool ANY>
int dispatch_gather(lossy_ctx* ctx, Params& P, const TmaGeom& G, cudaStream_t s, uint32_t* blocks) {
  const bool gb = ctx->cfg.grad_dtype == LOSSY_BF16;
  const bool rb = ctx->cfg.replica_dtype == LOSSY_BF16;
  const bool adam = ctx->cfg.optimizer == LOSSY_ADAM;
  if (gb && rb) return adam ? launch_gather<BF16, BF16, 1, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks) : launch_gather<BF16, BF16, 0, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks);
  if (gb && !rb) return adam ? launch_gather<BF16, F32, 1, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks) : launch_gather<BF16, F32, 0, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks);
  if (!gb && rb) return adam ? launch_gather<F32, BF16, 1, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks) : launch_gather<F32, BF16, 0, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks);
  return adam ? launch_gather<F32, F32, 1, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks) : launch_gather<F32, F32, 0, DRIFTK, CW, RD, ANY>(ctx, P, G, s, blocks);
}

template <int CW, bool ANY>
int try_gather_build(lossy_ctx* ctx, Params& P, bool drift, bool rd, cudaStream_t s, uint32_t* blocks, bool* used) {
  TmaGeom G = {};
  if (!gather_geometry<CW, ANY>(ctx, drift && rd, G)) return LOSSY_OK;
  *used = true;
  if (ctx->plan)
    snprintf(ctx->plan, ctx->plan_size, "gather %s packets/tile=%u stages=%u%s", CW == 16 ? "wide" : "twin", G.packets_per_tile, G.stages,
             drift && rd && CW == 16 ? " drift-warps" : "");
  if (drift && rd) return dispatch_gather<true, CW, true, ANY>(ctx, P, G, s, blocks);
  return drift ? dispatch_gather<true, CW, false, ANY>(ctx, P, G, s, blocks) : dispatch_gather<false, CW, false, ANY>(ctx, P, G, s, blocks);
}
template <int CW>
int try_gather(lossy_ctx* ctx, Params& P, bool drift, bool rd, cudaStream_t s, uint32_t* blocks, bool* used) {
  return GatherShape<CW>::kTile % P.P == 0 ? try_gather_build<CW, false>(ctx, P, drift, rd, s, blocks, used)
                                           : try_gather_build<CW, true>(ctx, P, drift, rd, s, blocks, used);
}

// Small buckets, of a few tiles (of 2048 elements) per SM, on the step kernel (lossy_register.cuh), which needs no second launch for a
// short last packet either. The pipelines' time over its own (2000 random steps with drift norms, 2000 without) at the lines below:
// packets from 1024 elements, whole: W <= 4 1.1-1.2 up to five tiles per SM (no multiple of 1024: 1.1-1.25 up to seven), W > 4 1.0-1.3; with
// a short last packet: W <= 4 1.2-1.6, W > 4 1.2-1.4; 128 elements: W <= 4 1.1-1.4 at ten tiles, more 1.2-1.5; 256 and 512 1.1-1.5 (1.5-2.0 up to four
// workers). Two to four workers have a build of their own.
// The lines are not where these figures end. They leave to the pipelines buckets that have always been theirs and are pinned to them, and
// on which the step kernel measured faster: W > 4 with whole packets from 1024 elements up to three tiles (1.0-1.2), with a short last packet under one
// (1.3-1.6) or without drift norms; 128 elements with more than four workers up to 16 tiles (1.2-1.5), 256 and 512 up to five
// (1.1-1.4); up to four workers and a short last packet up to eight (1.17). And all under an eighth of a tile per SM, which were not measured.
// All of this is one stream. A block of the step kernel takes most of an SM, so steps of several streams hardly share one: four
// streams that each step a bucket of its own (2500 such buckets, all streams' time per step, what they ran on before over the step kernel):
// W <= 8 1.1-2.4, packets under 1024 elements 1.2-2.4, W = 9-16 with longer ones 1.2 under a tile, 1.0 and 0.95 under two and four, W > 16 with
// longer ones 0.78-0.9 (0.58 at the least; one stream 1.27-1.45).
// Four workers, whole packets that are no multiple of 1024 elements, bf16 replicas, Adam and little loss: the lines for up to four workers
// lie nearer, at 5.75 tiles per SM instead of 7 (packets from 1024 elements) and 6.75 instead of 11. Pipelines' time over the step kernel's
// beyond them: p up to 0.05 0.98 (0.91 at the least) and 0.99 (0.86), p from 0.1 1.05 and 1.04; fp32 replicas 1.04-1.09 and 1.06, SGD
// 1.15 and 1.18, owner-elided replicas 1.14 and 1.10, a short last packet 1.2-1.3 (700 random steps).
bool four_light(const lossy_config& c) {
  return c.W == kStepFewWorkers && c.n % c.packet_elems == 0 && c.replica_dtype == LOSSY_BF16 && c.optimizer == LOSSY_ADAM &&
         !(c.flags & LOSSY_REPLICA_SKIP_OWNER) && fmax(c.p_grad, c.p_param) < 0.075;
}
bool small_bucket(const lossy_ctx* ctx, bool drift) {
  const lossy_config& c = ctx->cfg;
  const uint32_t P = c.packet_elems, kTwin = (uint32_t)TmaShape<8>::kTile, kWide = (uint32_t)TmaShape<16>::kTile;
  if (c.flags & (LOSSY_PACKED_BULK | LOSSY_GATHER_PATH)) return false;
  const double tiles = (double)c.n / ((double)kWide * ctx->num_sms);
  const bool bf16 = c.replica_dtype == LOSSY_BF16, few = c.W <= kStepFewWorkers, short_last = c.n % P != 0;
  if (tiles < 0.125 || P < 128u) return false;
  if (P >= kTwin) {
    if (few) return tiles >= (short_last ? 0.125 : 0.15) && tiles < (P % kTwin != 0 ? (four_light(c) ? 5.75 : 7.0) : short_last ? 2.0 : 5.0);
    if (!short_last) return tiles >= (c.W <= 8u ? 0.15 : 0.55) && tiles < (c.W <= 8u ? 1.0 : 2.5) && (tiles < 2.0 || c.W <= 32u || c.p_param < 0.25);
    if (!drift) return false;
    return bf16 ? tiles >= 1.0 && tiles < (P % kTwin == 0 ? 3.6 : 2.0) : tiles < 2.0 && c.W <= 8u;
  }
  if (kWide % P != 0) return false;          // (the register kernel's until the gather pipeline's lines)
  if (P == 128u) return tiles < (few ? 11.0 : 1.0);
  if (few || bf16) return tiles < 2.0;
  return tiles < 1.0 && (P == 256u || c.W <= 8u) && (drift || c.W <= 24u);
}

// Where the gather pipeline is used, and which of its builds. Figures are times of the build it would replace over its own,
// or (three digits) fractions of the copy rate; S = (W - 1) p_param = stale replicas per sub-packet. The lines were drawn
// through 4700 random steps timed with every build in turn (2 to 64 workers, 50 thousand to 60 M elements, packets of 128
// to 8960 elements, p = 0 to 0.3, both types, both optimizers, full and owner-elided replicas), so that none of the steps
// taken was more than 2 % slower than on the build replaced. The lines for few tiles per SM and packets under 1024 elements are
// from 3500 steps after kernels began behind the one ahead and the replica warps' single visit of a row, by which the other
// builds gained more than this one: of 7500 random steps up to 12 M elements since, the build chosen here and in run_tma is
// behind the best one by 9 % in the mean for packets of 128 to 512 that divide the tile (128 elements: the PACKED build, 1.05-1.3,
// below half a tile per SM up to 1.9; 256 and 512, bf16, two to eight tiles per SM: the register kernel, 1.05-1.2),
// by 6 % for other packets under 1024 (on the register kernel from two tiles per SM, 1.2, up to 2.2), by 3-5 % for longer
// ones (under one tile per SM with a short last packet, 1.1-1.2, up to 1.8; multiples of 1024, whole, from two tiles on: none).
// "The register kernel" of the figures here and in run_tma is the step kernel's predecessor, with chunks of 256 elements. The step kernel is 1.1 to
// 1.3 times as fast at two to eight tiles per SM and 1.0 to 1.2 beyond, its chunks are of 64 or 128 elements, and only the lines for up
// to four workers have been drawn against it: the others hand buckets to the pipelines earlier than it would pay, P = 384, 640 and
// 896 above all, whose chunks of 128 are full where `fill` counts them part empty.
GatherPolicy gather_policy(const lossy_ctx* ctx) {
  const lossy_config& c = ctx->cfg;
  const double pm = c.p_grad > c.p_param ? c.p_grad : c.p_param;
  const double stale = (c.W - 1u) * c.p_param;
  const uint32_t P = c.packet_elems, kTwin = (uint32_t)TmaShape<8>::kTile, kWide = (uint32_t)GatherShape<16>::kTile;
  const bool bf16 = c.replica_dtype == LOSSY_BF16, sgd = c.optimizer == LOSSY_SGD;
  const bool forced = c.flags & LOSSY_GATHER_PATH;
  GatherPolicy g = {};
  for (int drift = 0; drift < 2; ++drift) g.small[drift] = small_bucket(ctx, drift != 0);
  if (c.flags & LOSSY_PACKED_BULK || P < 128u) return g;
  TmaGeom G;
  // Tiles per SM. The pipeline fills and drains over several tiles, which a bucket of a few tiles per SM pays for: under
  // two the register kernel and the bulk-copy pipeline take 0.5-1.0 of its time (n = 0.9 M, W = 16, P = 336: 0.55). The
  // line lies higher with many workers (more groups per tile) and for SGD (less to move per tile).
  const double tiles = (double)c.n / ((double)kWide * ctx->num_sms);
  const double per_sm = tiles / ((c.W > 16u ? 1.5 : 1.0) * (sgd ? 1.25 : 1.0));
  if (P < kTwin && kWide % P == 0) {
    // Packets of 128, 256 or 512 elements, which divide the tile:
    //  * the wide geometry with drift warps of its own from 4 workers, packets of 256 or 512 elements and bf16 replicas
    //    (W = 8: 0.97 / 0.97 / 0.94 / 0.85 at p = 0.05 / 0.1 / 0.2 / 0.3, where the compute warps' reads gave 0.89 / 0.84 /
    //    0.82 / 0.77 and the register kernel 0.77 and 0.67 at p = 0.1 and 0.3). Up to 24 workers from 0.2 (W - 8) stale
    //    replicas on: below that the compute warps' reads are ahead (W = 16, p = 0.05: 0.95 against 0.84);
    //  * more workers where the register kernel is the alternative (p from 0.15 to 0.2) and the bucket is large, from 32 tiles per
    //    SM (W = 32, P = 512, p = 0.2: 1.13; P = 256, p = 0.15: W = 30: 1.15, W = 56: 1.11; 24 tiles, W = 36: 0.90). Not against the compute
    //    warps' reads, whose sums of 128 squares are the more precise ones (1.0-1.1 at p = 0.05-0.1);
    //  * below 7.5 stale replicas (W = 17, p = 0.5: 0.43 against 0.56);
    //  * fp32 replicas: the compute warps' reads (a row has twice the chunks and the wire ring leaves the drift warps
    //    little scratch: W = 4, P = 512, p = 0.1: 0.88 against 0.80); LOSSY_GATHER_PATH asks for drift warps all the same;
    //  * two or three workers, and packets of 128 elements: the twin geometry (W = 2: 0.78-0.81 against 0.69-0.74 for the
    //    wide one), whose replica warps also read the stale copies up to four workers.
    // Many workers at high loss run on the register kernel, or on what it gives way to, unless drift warps read the stale
    // copies (bf16: W = 32, P = 256, p = 0.2: 0.83 against 0.79); with fp32 replicas and packets from 256 elements the
    // compute warps are ahead there from 7 tiles per SM (W = 36, P = 512, p = 0.25: 1.21; W = 24-64 below 2.5 tiles: 0.6-0.9).
    const bool many_lossy = bf16 ? (c.W >= 12 && pm >= 0.25) || (c.W >= 24 && pm >= 0.15) : c.W >= 24 && pm >= 0.25;
    const bool band = c.W <= 24u && stale < 7.5 && stale >= 0.2 * ((double)c.W - 8.0);
    const bool beyond = many_lossy && c.W > 24u && pm < 0.225 && (forced || per_sm >= 32.0);
    g.wide = P >= 256u && c.W >= 4u;
    g.drift_warps = g.wide && (bf16 || forced) && (band || beyond) && gather_geometry<16, false>(ctx, true, G);
    g.use = forced || g.drift_warps || !many_lossy || (!bf16 && P >= 256u && per_sm >= 7.0);
  } else if (P < kTwin) {
    // Other packets shorter than the twin tile. The alternative is the register kernel, whose chunks of 256 elements each
    // packet ends with are filled to `fill`. From 3.5, 5, 6 or 8 tiles per SM with fill up to 0.6, 0.8, 0.9 or 1: 1.0-3.9
    // (P = 736, W = 8, p = 0.1: 1.79; P = 200: 2.0; W = 64, P = 520: 1.1), 1.6 and 2.2 times as many from 17 workers and for SGD (of 1700
    // steps, 110 lie between these lines and the ones before the replica warps' single visit, 5 to 16 tiles: mean 1.46; slower
    // there: SGD at W = 14, P = 240, p = 0.3: 0.83, W = 6: 0.92, W = 5, P = 224, p = 0.05, fp32 replicas: 0.89, and W = 27, P = 712,
    // p = 0.3: 0.91. Without drift norms 775 more: mean 1.50, one under 0.98). Full chunks: not for SGD (W = 15, P = 768, p = 0: 0.91),
    // nearly full ones not with eight stale replicas (W = 41, P = 760, p = 0.3: 0.87); 12 of them only with the emptiest chunks.
    // Nor SGD at high loss with bf16 gradients and fp32 replicas that the drift warps cannot serve, up to a chunk (W = 9, P = 216,
    // p = 0.2: 0.87, P = 176: 0.83; P = 592 from 1.0).
    // Packets under 176 elements put more than 12 sub-packets on a wide tile: twin tiles at low loss (W = 8, P = 144, p =
    // 0.05: 0.68 against 0.59), wide ones from p = 0.15 (p = 0.3: 0.55 against 0.47); up to four workers twin below 256
    // (W = 4, P = 200: 0.75 against 0.63).
    const double fill = P / (256.0 * ((P + 255u) / 256u));
    // (the step kernel's build for two to four workers: 1.1-2.1 up to 11 tiles per SM, 0.9-1.3 beyond)
    const double least = fmax((fill <= 0.6 ? 3.5 : fill <= 0.8 ? 5.0 : fill <= 0.9 ? 6.0 : 8.0) * (c.W > 16u ? 1.6 : 1.0) * (sgd ? 2.2 : 1.0), c.W > kStepFewWorkers ? 0.0 : four_light(c) ? 6.75 : 11.0);
    const bool full_lossy = (sgd && fill > 0.98) || (bf16 && ((fill > 0.9 && stale >= 8.0) || (fill > 0.6 && stale >= 12.0)));
    g.wide = c.W >= 5u ? P >= 176u || pm >= 0.15 : c.W == 4u && P >= 256u;
    g.drift_warps = g.wide && gather_geometry<16, true>(ctx, true, G);
    const bool sgd_lossy = sgd && pm >= 0.175 && !bf16 && c.grad_dtype == LOSSY_BF16 && P <= 256u && fill > 0.6 && g.wide && !g.drift_warps;
    g.use = forced || (tiles >= least && !full_lossy && !sgd_lossy);
  } else if (P % kTwin != 0 && P < (1u << 15)) {
    // Longer packets that are no multiple of the twin tile. The bulk-copy pipeline cuts each into tiles of its own, the
    // last of them part empty (`fill` of the tiles' elements are used); here the tiles run on across packets. From 6 tiles
    // per SM. bf16 replicas, p up to 0.15: fill under 0.8 (W = 8, P = 1472, p = 0.1: 1.28, P = 1032: 1.4; but owner-elided with 9-16
    // workers only under 0.7: W = 15, P = 2264: 0.95), any fill with more than 16 workers (1.0-1.25), not with fewer (W = 4-16, fill
    // 0.8-1: 0.8-1.15, mostly 1.0); more loss: only tiles half empty, up to 16 workers (1.27-1.5; more: 0.93). Two or three
    // workers: tiles half empty (1.15). fp32 replicas: tiles half empty from 9 workers (1.1-1.3), fill under 0.7 from 17.
    const double fill = P / (double)((P + kTwin - 1u) / kTwin * kTwin);
    const bool lossy = pm >= 0.175, elided = c.flags & LOSSY_REPLICA_SKIP_OWNER;
    bool ahead;
    if (c.W <= 3u) ahead = bf16 && fill < 0.6;
    else if (!bf16) ahead = (fill < 0.6 && c.W > 8u) || (fill < 0.7 && c.W > 16u && !lossy);
    else if (lossy) ahead = fill < 0.6 && c.W <= 16u;
    else ahead = fill < 0.7 || c.W > 16u || (fill < 0.8 && (c.W <= 8u || !elided));
    g.wide = c.W >= 4u;
    g.drift_warps = g.wide && gather_geometry<16, true>(ctx, true, G);
    g.use = forced || (per_sm >= 6.0 && ahead);
  }
  return g;
}

// Run the build the policy picks; *used stays false when no bulk-copy launch fits (packets shorter
// than a tile, or no complete packet): the register path then takes everything.
int run_tma(lossy_ctx* ctx, Params& P, bool drift, cudaStream_t s, uint32_t* blocks, bool* used) {
  *used = false;
  if (ctx->cfg.flags & LOSSY_REGISTER_PATH || ctx->gather.small[drift]) return LOSSY_OK;
  const TmaPolicy t = tma_policy(ctx->cfg);
  const GatherPolicy& gp = ctx->gather;
  if (gp.use) {
    int rc = LOSSY_OK;
    if (gp.wide) rc = try_gather<16>(ctx, P, drift, gp.drift_warps, s, blocks, used);
    if (rc || *used) return rc;
    rc = try_gather<8>(ctx, P, drift, ctx->cfg.W <= kRdTwinMaxWorkers, s, blocks, used);
    if (rc || *used) return rc;
  }
  {
    // Packets of exactly half a wide tile with 13..16 workers at low loss: the PACKED wide build (two packets
    // per tile, one CTA per SM) beats the twin build, whose pieces are 2 KB (W = 16: 0.96-0.98 against 0.93 up
    // to p = 0.1; W = 13-14: 0.97-1.0 against 0.94 up to p = 0.05); beyond that its fetches of dropped packets
    // cost more than the wider tile gains, and from 12 workers down the twin build is ahead at every p.
    const lossy_config& c = ctx->cfg;
    const double pm = c.p_grad > c.p_param ? c.p_grad : c.p_param;
    if (c.packet_elems * 2u == (uint32_t)TmaShape<16>::kTile && c.W >= 13 && c.W <= 16 && pm <= (c.W == 16 ? 0.1 : 0.05)) {
      int rc = try_tma<16, 8, 0, true>(ctx, P, drift, s, blocks, used);
      if (rc || *used) return rc;
    }
  }
  if (ctx->cfg.packet_elems < (uint32_t)TmaShape<8>::kTile) {
    // Packets shorter than a tile: the PACKED builds, where they beat the register kernel. They fetch the
    // dropped sub-packets too, so they win at low loss (+8..17 % at W = 8-16, P = 256-512, p <= 0.1; +3..5 % at
    // p = 0.2) and lose at p = 0.3 from W = 16 and at p >= 0.1 from W = 32; with 2..8 workers they win at every loss rate
    // (+1..13 %); below 256 elements the register kernel's 256-element chunks are mostly idle lanes and the
    // PACKED build always wins.
    const lossy_config& c = ctx->cfg;
    const double pm = c.p_grad > c.p_param ? c.p_grad : c.p_param;
    if (c.packet_elems < 256 || (c.W >= 2 && c.W <= 8) || (pm <= 0.2 && c.W <= 24) || (pm <= 0.075 && c.W <= 32)) {
      if (c.W <= 16) {
        int rc = try_tma<16, 8, 0, true>(ctx, P, drift, s, blocks, used);
        if (rc || *used) return rc;
      }
      int rc = try_tma<8, 8, 0, true>(ctx, P, drift, s, blocks, used);
      if (rc || *used) return rc;
    }
  }
  if (t.split) {
    // the state lives in its own two-slot ring (SPLIT builds, twin geometry only)
    return t.early_stale == 1 ? try_tma<8, 8, 1, false, true>(ctx, P, drift, s, blocks, used)
           : t.early_stale ? try_tma<8, 8, 16, false, true>(ctx, P, drift, s, blocks, used)
                           : try_tma<8, 8, 0, false, true>(ctx, P, drift, s, blocks, used);
  }
  if (t.wide) {
    int rc = t.group == 4 ? try_tma<16, 4>(ctx, P, drift, s, blocks, used)
             : t.early_stale ? try_tma<16, 8, 16>(ctx, P, drift, s, blocks, used)
                             : try_tma<16, 8>(ctx, P, drift, s, blocks, used);
    if (rc || *used) return rc;
  }
  return t.group == 4 ? try_tma<8, 4>(ctx, P, drift, s, blocks, used)
         : t.early_stale ? try_tma<8, 8, 16>(ctx, P, drift, s, blocks, used)
                         : try_tma<8, 8>(ctx, P, drift, s, blocks, used);
}

template <int PH, class GT, class RT, int OPT, bool ELIDE, bool TAIL>
int launch_register(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks_out) {
  auto kern = lossy_kernel<PH, GT, RT, OPT, ELIDE, TAIL>;
  static int occupancy[kMaxDevices];   // per kernel instantiation and device: resident blocks per SM
  int per_sm = 0;
  cudaError_t e;
  {
    std::lock_guard<std::mutex> lock(g_setup_mu);
    per_sm = ctx->device < kMaxDevices ? occupancy[ctx->device] : 0;
    if (per_sm == 0) {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, 0);
      if (e != cudaSuccess) return fail_cuda(ctx, "occupancy query", e);
      if (per_sm < 1) per_sm = 1;
      if (per_sm > kBlocksPerSmCap) per_sm = kBlocksPerSmCap;
      if (ctx->device < kMaxDevices) occupancy[ctx->device] = per_sm;
    }
  }
  uint32_t blocks = (uint32_t)(ctx->num_sms * per_sm);
  const uint32_t need = (P.num_chunks + kWarps - 1) / kWarps;
  if (blocks > need) blocks = need;
  if (blocks > ctx->max_blocks - P.partials_row0) blocks = ctx->max_blocks - P.partials_row0;
  if (blocks == 0) blocks = 1;
  if (blocks_out) *blocks_out = blocks;
  if (ctx->plan_only) return LOSSY_OK;
  rows_of_call(P, blocks);
  // Early where the launch is a good part of the call: up to a few chunks per warp, or the short last packet; a broadcast up to 64 blocks.
  // Its blocks need so few registers that they crowd the SMs that come free first, as the packet norms' do. (780 random buckets of
  // packets under 1024 elements, the four phases, early up to 64 blocks over early up to a few chunks per warp: 1.00 to 1.02 under 130
  // thousand elements, 1.02 to 1.10 up to 4 M; W = 41, P = 512, 374 k, fp32 replicas: 73 -> 63 us; W = 63, P = 256, 737 k: 203 -> 157.
  // The other phases so as well: no gain, 0.96 at 130 thousand.)
  const bool crowds = PH == BCAST && !TAIL && blocks > 64u;
  e = launch_after(need <= 4u * blocks && !crowds, kern, blocks, kThreads, 0, s, P);
  if (e != cudaSuccess) return fail_cuda(ctx, "kernel launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

// (a launch that does not begin with the first packet is the short last packet behind another launch of the same call)
template <int PH, class GT, class RT, int OPT, bool ELIDE = false>
int launch(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks_out) {
  return P.k_begin ? launch_register<PH, GT, RT, OPT, ELIDE, true>(ctx, P, s, blocks_out)
                       : launch_register<PH, GT, RT, OPT, ELIDE, false>(ctx, P, s, blocks_out);
}

// dispatch of a single phase on the runtime element types / optimizer
template <int PH>
int dispatch(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks) {
  const bool rb = ctx->cfg.replica_dtype == LOSSY_BF16;
  if constexpr (PH == AGG) {
    return ctx->cfg.grad_dtype == LOSSY_BF16 ? launch<PH, BF16, F32, 0>(ctx, P, s, blocks) : launch<PH, F32, F32, 0>(ctx, P, s, blocks);
  } else if constexpr (PH == STEP) {
    return ctx->cfg.optimizer == LOSSY_ADAM ? launch<PH, F32, F32, 1>(ctx, P, s, blocks) : launch<PH, F32, F32, 0>(ctx, P, s, blocks);
  } else {
    if (ctx->cfg.flags & LOSSY_REPLICA_SKIP_OWNER)   // owner-elided replicas: builds of their own
      return rb ? launch<PH, F32, BF16, 0, true>(ctx, P, s, blocks) : launch<PH, F32, F32, 0, true>(ctx, P, s, blocks);
    return rb ? launch<PH, F32, BF16, 0>(ctx, P, s, blocks) : launch<PH, F32, F32, 0>(ctx, P, s, blocks);
  }
}

// ---- the fused step on registers alone (lossy_step_kernel) -----------------------------------
template <class GT, class RT, int OPT, bool DRIFTK, bool ELIDE, bool TAIL, int FORM>
int launch_step(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks_out) {
  constexpr uint32_t kSpan = 32 * StepShape<GT, RT, FORM>::kEpl, kMost = StepShape<GT, RT, FORM>::kMaxWarps;
  const uint32_t per_packet = (P.P + kSpan - 1) / kSpan;
  const uint32_t chunks = (P.K - P.k_begin) * per_packet;
  const uint32_t tasks = chunks + (P.n % StepShape<GT, RT, FORM>::kEpl ? 1u : 0u);
  uint32_t blocks, warps;
  if (TAIL) {
    warps = tasks < 8u ? tasks : 8u;
    blocks = (tasks + warps - 1) / warps;
    if (blocks > (uint32_t)ctx->num_sms) blocks = (uint32_t)ctx->num_sms;
  } else {
    // one block per SM, each with the warps that its share of the chunks needs
    blocks = tasks < (uint32_t)ctx->num_sms ? tasks : (uint32_t)ctx->num_sms;
    warps = (tasks + blocks - 1) / blocks;
    const uint32_t rounds = (warps + kMost - 1) / kMost;
    warps = (warps + rounds - 1) / rounds;
    // The end of the drift norms takes two replicas per warp and turn, each turn a round trip to L2 or more: warps for four turns at W = 64
    // and for one up to 16, also where there are no chunks for them. (3000 random steps of a thousand to 40 thousand elements, W = 2-4, 5-8, 9-16,
    // 17-32, 33-64: without them 1.10, 1.28, 1.54, 1.76 and 2.1 times as long under 9 thousand elements, 1.0, 1.02, 1.1, 1.1 and 1.17 from 19
    // thousand on; W = 50, 7 thousand: 27.3 -> 12.5 us. Four warps 14.2, 16 11.8.)
    const uint32_t enough = P.W < 16u ? (P.W + 1u) / 2u : 8u;
    if (DRIFTK && warps < enough) warps = enough;
  }
  *blocks_out = blocks;
  if (ctx->plan) {
    static const char* const kForms[] = {"pairs", "quads", "few", "stale", "octs"};
    snprintf(ctx->plan, ctx->plan_size, "register kernel %s warps=%u rounds=%u", kForms[FORM], warps, (tasks + blocks * warps - 1u) / (blocks * warps));
  }
  if (ctx->plan_only) return LOSSY_OK;
  rows_of_call(P, blocks);
  P.chunks_per_packet = per_packet;
  P.cpp_magic = magic_of(per_packet);
  P.pps_magic = magic_of(P.pps);
  P.num_chunks = chunks;
  const cudaError_t e = launch_after((tasks + warps - 1) / warps <= 4u * blocks, lossy_step_kernel<GT, RT, OPT, DRIFTK, ELIDE, TAIL, FORM>, blocks, warps * 32u, 0, s, P);
  if (e != cudaSuccess) return fail_cuda(ctx, "kernel launch", e);
  ctx->launches++;
  return LOSSY_OK;
}
template <class GT, class RT, int OPT, bool DRIFTK, bool ELIDE>
int pick_step(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks) {
  if (P.k_begin) return launch_step<GT, RT, OPT, DRIFTK, ELIDE, true, kStepQuads>(ctx, P, s, blocks);
  const uint32_t W = P.W;
  if (W <= kStepFewWorkers) return launch_step<GT, RT, OPT, DRIFTK, ELIDE, false, kStepFew>(ctx, P, s, blocks);
  // Pairs: with more than 16 workers where they take no more rounds than quads, with fewer up to half (W > 8) or a quarter of a
  // round (2000 random steps: pairs' time over quads' 0.81-0.96, 0.90-0.97, 0.99; beyond 0.97-1.2).
  const uint64_t warps2 = (uint64_t)P.K * ((P.P + 63u) / 64u), warps4 = (uint64_t)P.K * ((P.P + 127u) / 128u);
  auto rounds = [&](uint64_t chunks, uint32_t warps) { return (chunks + (uint64_t)ctx->num_sms * warps - 1) / ((uint64_t)ctx->num_sms * warps); };
  if (W > 16u ? rounds(warps2, 32u) <= rounds(warps4, StepShape<GT, RT, kStepQuads>::kMaxWarps) : warps2 <= (uint64_t)ctx->num_sms * (W > 8u ? 16u : 8u))
    return launch_step<GT, RT, OPT, DRIFTK, ELIDE, false, kStepPairs>(ctx, P, s, blocks);
  // Two stale replicas per packet and more: eight copies requested together up to two rounds; from three rounds on with many workers eight
  // elements per lane, which halve the reductions of the stale copies per element (W = 32, P = 512, p = 0.3, 20 M: quads 529 us, octs
  // 486; W = 49, P = 976, p = 0.3, 25 M: 1072, 993; W = 15, P = 768, p = 0.3, 6 M: 82, 84).
  if constexpr (DRIFTK && RT::kVecs == 1) {
    const bool stale = (W - 1u) * ctx->cfg.p_param >= 2.0;
    const bool many_rounds = rounds(warps4, 24u) >= 3u;
    if (stale && W > 16u && many_rounds) return launch_step<GT, RT, OPT, DRIFTK, ELIDE, false, kStepOcts>(ctx, P, s, blocks);
    if (stale && !many_rounds) return launch_step<GT, RT, OPT, DRIFTK, ELIDE, false, kStepStale>(ctx, P, s, blocks);
  }
  return launch_step<GT, RT, OPT, DRIFTK, ELIDE, false, kStepQuads>(ctx, P, s, blocks);
}
template <class GT, class RT, bool DRIFTK>
int dispatch_step_as(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks) {
  const bool adam = ctx->cfg.optimizer == LOSSY_ADAM;
  if (ctx->cfg.flags & LOSSY_REPLICA_SKIP_OWNER)   // owner-elided replicas: builds of their own
    return adam ? pick_step<GT, RT, 1, DRIFTK, true>(ctx, P, s, blocks) : pick_step<GT, RT, 0, DRIFTK, true>(ctx, P, s, blocks);
  return adam ? pick_step<GT, RT, 1, DRIFTK, false>(ctx, P, s, blocks) : pick_step<GT, RT, 0, DRIFTK, false>(ctx, P, s, blocks);
}
template <bool DRIFTK>
int dispatch_step(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks) {
  const bool gb = ctx->cfg.grad_dtype == LOSSY_BF16, rb = ctx->cfg.replica_dtype == LOSSY_BF16;
  if (gb) return rb ? dispatch_step_as<BF16, BF16, DRIFTK>(ctx, P, s, blocks) : dispatch_step_as<BF16, F32, DRIFTK>(ctx, P, s, blocks);
  return rb ? dispatch_step_as<F32, BF16, DRIFTK>(ctx, P, s, blocks) : dispatch_step_as<F32, F32, DRIFTK>(ctx, P, s, blocks);
}

// ---- the single-phase calls through the bulk-copy pipeline ---------------------------------
constexpr uint32_t kPhaseSmemFixed = kTmaBarBytes + kPhaseMaxStages * sizeof(StageHdr);

template <int PH, int CW, int GS>
bool phase_geometry(const lossy_ctx* ctx, TmaGeom& G) {
  constexpr uint32_t kTile = TmaShape<CW>::kTile;
  constexpr bool kGrouped = PH == AGG || PH == DRIFT;
  const lossy_config& c = ctx->cfg;
  const uint64_t kfull = c.n / c.packet_elems;               // packets that are complete
  if (kfull == 0 || kfull >= (1ull << 31) || c.packet_elems < kTile) return false;
  memset(&G, 0, sizeof G);
  G.packets_per_tile = 1;
  G.full_packets = (uint32_t)kfull;
  const uint32_t gb = c.grad_dtype == LOSSY_BF16 ? 2 : 4, rb = c.replica_dtype == LOSSY_BF16 ? 2 : 4;
  const uint32_t eb = PH == AGG ? gb : PH == STEP ? 4u : rb;
  G.grad_slots = kGrouped ? (c.W < (uint32_t)GS ? c.W : (uint32_t)GS) : 0u;
  G.groups = kGrouped ? (c.W + GS - 1) / GS : 1u;
  G.stage_bytes = (phase_stage_bytes<PH>(kTile, G.grad_slots, eb, c.optimizer == LOSSY_ADAM) + 127u) & ~127u;
  const uint32_t budget = tma_smem_budget<CW>(ctx);
  if (budget < kPhaseSmemFixed + 2 * G.stage_bytes) return false;
  G.stages = (budget - kPhaseSmemFixed) / G.stage_bytes;
  if (G.stages > (uint32_t)kPhaseMaxStages) G.stages = kPhaseMaxStages;
  // the optimizer step reads and writes equal amounts: deeper than three stages its loads run too far ahead
  // of its stores (measured 1.01 of the copy rate with three stages, 0.90 with seven)
  if (PH == STEP && G.stages > 3u) G.stages = 3u;
  G.tiles_per_packet = (c.packet_elems + kTile - 1) / kTile;
  const uint64_t tiles = kfull * G.tiles_per_packet;
  if (tiles >= (1ull << 31)) return false;
  G.num_tiles = (uint32_t)tiles;
  G.status = ctx->status;
  G.hints = 0;
  return true;
}

template <int PH, class T, int OPT, int CW, int GS>
int launch_phase_tma(lossy_ctx* ctx, Params& P, const TmaGeom& G, cudaStream_t s, uint32_t* blocks_out) {
  auto kern = lossy_phase_tma_kernel<PH, T, OPT, CW, GS>;
  const uint32_t smem = kPhaseSmemFixed + G.stages * G.stage_bytes;
  uint32_t blocks = (uint32_t)(ctx->num_sms * TmaShape<CW>::kCtasPerSm);
  if (blocks > G.num_tiles) blocks = G.num_tiles;
  *blocks_out = blocks;
  if (ctx->plan_only) return LOSSY_OK;
  rows_of_call(P, blocks);
  static bool opted_in[kMaxDevices];   // per kernel instantiation and device: raise the dynamic shared memory limit once
  cudaError_t e;
  {
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (ctx->device >= kMaxDevices || !opted_in[ctx->device]) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin - 1024);   // (less what is static)
      if (e != cudaSuccess) return fail_cuda(ctx, "shared memory opt-in", e);
      if (ctx->device < kMaxDevices) opted_in[ctx->device] = true;
    }
  }
  e = launch_after(true, kern, blocks, TmaShape<CW>::kThreads, spread_smem(ctx, smem, TmaShape<CW>::kCtasPerSm), s, P, G);
  if (e != cudaSuccess) return fail_cuda(ctx, "bulk-copy kernel launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

template <int PH, int CW, int GS>
int try_phase_tma(lossy_ctx* ctx, Params& P, cudaStream_t s, uint32_t* blocks, bool* used) {
  TmaGeom G;
  if (!phase_geometry<PH, CW, GS>(ctx, G)) return LOSSY_OK;
  *used = true;
  const bool adam = ctx->cfg.optimizer == LOSSY_ADAM;
  if constexpr (PH == AGG) {
    return ctx->cfg.grad_dtype == LOSSY_BF16 ? launch_phase_tma<PH, BF16, 0, CW, GS>(ctx, P, G, s, blocks)
                                             : launch_phase_tma<PH, F32, 0, CW, GS>(ctx, P, G, s, blocks);
  } else if constexpr (PH == STEP) {
    return adam ? launch_phase_tma<PH, F32, 1, CW, GS>(ctx, P, G, s, blocks)
                : launch_phase_tma<PH, F32, 0, CW, GS>(ctx, P, G, s, blocks);
  } else {
    return ctx->cfg.replica_dtype == LOSSY_BF16 ? launch_phase_tma<PH, BF16, 0, CW, GS>(ctx, P, G, s, blocks)
                                                : launch_phase_tma<PH, F32, 0, CW, GS>(ctx, P, G, s, blocks);
  }
}

// A call's launches: complete packets through a pipeline, a short last packet, or everything when no pipeline's build fits, through a
// register kernel. With drift norms the blocks of both launches draw tickets from one counter and the last of them finalises
// the norms; where there may be two launches, a first turn that launches nothing counts their blocks.
template <class LaunchAll>
int run_launches(lossy_ctx* ctx, Params& P, bool drift, cudaStream_t s, LaunchAll&& launch_all) {
  uint32_t rows = 0;
  if (drift && ctx->cfg.n % ctx->cfg.packet_elems != 0) {
    Params Q = P;
    ctx->plan_only = true;
    const int rc = launch_all(Q, &rows);
    ctx->plan_only = false;
    if (rc) return rc;
    P.total_rows = rows;
  }
  const int rc = launch_all(P, &rows);
  if (rc && drift) reset_ticket(ctx, s);
  return rc;
}

// One single-phase call: packets of at least one tile through the bulk-copy pipeline, the rest through the register kernel.
template <int PH>
int run_phase(lossy_ctx* ctx, Params& P, float* norms, double* sumsq, cudaStream_t s) {
  const lossy_config& c = ctx->cfg;
  const bool bulk = !(c.flags & LOSSY_REGISTER_PATH);
  // wide tiles (one CTA per SM) when they divide the packet and the streamed arrays fit two groups
  const bool wide = c.packet_elems % TmaShape<16>::kTile == 0 && c.W <= 16;
  auto launch_all = [&](Params& Q, uint32_t* rows) {
    uint32_t tma_blocks = 0, tail_blocks = 0;
    bool used = false;
    int rc = LOSSY_OK;
    if (bulk) {
      if (wide) rc = try_phase_tma<PH, 16, 8>(ctx, Q, s, &tma_blocks, &used);
      if (!rc && !used) rc = try_phase_tma<PH, 8, 8>(ctx, Q, s, &tma_blocks, &used);
    }
    if (rc) return rc;
    if (used) {
      Q.k_begin = (uint32_t)(c.n / c.packet_elems);
      Q.num_chunks = (Q.K - Q.k_begin) * ctx->chunks_per_packet;
      Q.partials_row0 = tma_blocks;
    } else {
      tma_blocks = 0;
    }
    if (Q.num_chunks) rc = dispatch<PH>(ctx, Q, s, &tail_blocks);
    *rows = tma_blocks + tail_blocks;
    return rc;
  };
  if (PH == DRIFT) {
    P.ticket = ctx->ticket;
    P.norms = norms;
    P.sumsq = sumsq;
  }
  return run_launches(ctx, P, PH == DRIFT, s, launch_all);
}

// Chunks per SM up to which a bucket is small for the pairwise drift (300 thousand elements): at 250 k the small builds take 0.55
// to 0.95 of the other's time (W = 16 to 64, 5 % late and more), at 1 M there is work for all of the other's warps.
constexpr uint64_t kPairSmallPerSm = 8;
// One block per SM, of as many warps as their tables and slots leave room for; fewer blocks when there are not as many
// chunks as warps.
template <class RT, bool ELIDE, class M, bool SMALL>
cudaError_t launch_pairwise(lossy_ctx* ctx, PairwiseArgs<ELIDE>& A, cudaStream_t s) {
  auto kern = drift_pairwise_kernel<RT, ELIDE, M, SMALL>;
  const uint32_t wb = pair_warp_bytes(A.W, sizeof(typename RT::raw));
  const uint32_t room = (uint32_t)ctx->smem_optin - 128u;   // (less what is static)
  uint32_t warps = room / wb;
  if (warps > (uint32_t)PairShape<M, SMALL>::kMaxWarps) warps = PairShape<M, SMALL>::kMaxWarps;
  if (warps == 0) return cudaErrorInvalidConfiguration;
  static bool opted_in[kMaxDevices];   // per kernel instantiation and device: raise the dynamic shared memory limit once
  {
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (ctx->device >= kMaxDevices || !opted_in[ctx->device]) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
      if (e != cudaSuccess) return e;
      if (ctx->device < kMaxDevices) opted_in[ctx->device] = true;
    }
  }
  uint64_t chunks = (uint64_t)A.segs * A.chunks_per_seg;
  // a small bucket: several warps per chunk, while there are warps without work and rows of pairs to share
  while ((chunks << 1) <= (uint64_t)ctx->num_sms * warps && (2u << A.lgsplit) < A.W) { ++A.lgsplit; chunks <<= 1; }
  // (and its chunks spread over the SMs rather than filling a few of them)
  if (chunks < (uint64_t)ctx->num_sms * warps) warps = (uint32_t)((chunks + ctx->num_sms - 1) / ctx->num_sms);
  uint64_t blocks = (chunks + warps - 1) / warps;
  if (blocks > (uint64_t)ctx->num_sms) blocks = ctx->num_sms;
  return launch_after(false, kern, (uint32_t)blocks, warps * 32u, warps * wb, s, A);
}

}  // namespace

extern "C" {

int lossy_init(const lossy_config* cfg, lossy_ctx** out) {
  if (!cfg || !out) return LOSSY_EINVAL;
  *out = nullptr;
  if (cfg->W == 0 || cfg->W > LOSSY_MAX_WORKERS) return LOSSY_EINVAL;
  if (cfg->packet_elems == 0 || cfg->packet_elems % 8 != 0) return LOSSY_EINVAL;
  if (!(cfg->p_grad >= 0.0 && cfg->p_grad < 1.0) || !(cfg->p_param >= 0.0 && cfg->p_param < 1.0)) return LOSSY_EINVAL;
  if (cfg->grad_dtype > LOSSY_BF16 || cfg->replica_dtype > LOSSY_BF16 || cfg->optimizer > LOSSY_ADAM) return LOSSY_EINVAL;
  if (cfg->flags & ~(uint32_t)(LOSSY_SELF_LOSSLESS | LOSSY_ZERO_SKIP | LOSSY_REGISTER_PATH | LOSSY_REPLICA_SKIP_OWNER | LOSSY_PACKED_BULK | LOSSY_GATHER_PATH))
    return LOSSY_EINVAL;
  const uint64_t K = (cfg->n + cfg->packet_elems - 1) / cfg->packet_elems;
  const uint64_t cpp = (cfg->packet_elems + kChunk - 1) / kChunk;
  if (K * cpp >= (1ull << 31)) return LOSSY_EINVAL;  // stream larger models bucket by bucket
  if (cfg->bucket_packets) {
    // a packet range of a larger bucket: inside it, and ragged only where the bucket ends
    if (cfg->bucket_packets >= (1ull << 31) || cfg->shard_packet0 + K > cfg->bucket_packets) return LOSSY_EINVAL;
    if (cfg->n % cfg->packet_elems != 0 && cfg->shard_packet0 + K != cfg->bucket_packets) return LOSSY_EINVAL;
  } else if (cfg->shard_packet0) {
    return LOSSY_EINVAL;
  }

  lossy_ctx* ctx = new (std::nothrow) lossy_ctx;
  if (!ctx) return LOSSY_ENOMEM;
  memset(ctx, 0, sizeof *ctx);
  ctx->cfg = *cfg;
  ctx->K = K;
  ctx->chunks_per_packet = (uint32_t)cpp;
  ctx->num_chunks = (uint32_t)(K * cpp);
  // shard map of the WHOLE bucket: this context may cover only the packet range starting at shard_packet0
  const uint64_t Kb = cfg->bucket_packets ? cfg->bucket_packets : K;
  const uint64_t pps = (Kb + cfg->W - 1) / cfg->W;
  ctx->pps = pps ? (uint32_t)pps : 1u;
  ctx->Tg = threshold_of(cfg->p_grad);
  ctx->Tp = threshold_of(cfg->p_param);
  cudaError_t e = cudaGetDevice(&ctx->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, ctx->device);
  if (e != cudaSuccess) { delete ctx; return LOSSY_ECUDA; }
  ctx->max_blocks = (uint32_t)(ctx->num_sms * kBlocksPerSmCap);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
  if (e != cudaSuccess) { delete ctx; return LOSSY_ECUDA; }
  ctx->gather = gather_policy(ctx);
  const size_t pbytes = (size_t)ctx->max_blocks * kMaxW * sizeof(double);
  e = cudaMalloc(&ctx->partials, pbytes + 256);
  if (e != cudaSuccess) { delete ctx; return e == cudaErrorMemoryAllocation ? LOSSY_ENOMEM : LOSSY_ECUDA; }
  ctx->status = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(ctx->partials) + pbytes);
  ctx->ticket = ctx->status + 16;
  ctx->gate = ctx->status + 32;
  e = cudaMemset(ctx->status, 0, 256);
  if (e != cudaSuccess) { cudaFree(ctx->partials); delete ctx; return LOSSY_ECUDA; }
  *out = ctx;
  return LOSSY_OK;
}

void lossy_destroy(lossy_ctx* ctx) {
  if (!ctx) return;
  if (ctx->partials) cudaFree(ctx->partials);
  delete ctx;
}

int lossy_set_bursty(lossy_ctx* ctx, double p_enter_bad, double p_leave_bad, uint64_t* state) {
  if (!ctx) return LOSSY_EINVAL;
  if (!state) {
    ctx->burst_state = nullptr;
    return LOSSY_OK;
  }
  if (!(p_enter_bad >= 0.0 && p_enter_bad < 1.0) || !(p_leave_bad > 0.0 && p_leave_bad <= 1.0))
    return fail(ctx, LOSSY_EINVAL, "bursty loss: need 0 <= P(good->bad) < 1 and 0 < P(bad->good) <= 1");
  if (ctx->K >= (1ull << 32)) return fail(ctx, LOSSY_EINVAL, "too many packets for bursty loss");
  if (reinterpret_cast<uintptr_t>(state) & 7u) return fail(ctx, LOSSY_EINVAL, "state: misaligned");
  ctx->burst_state = state;
  ctx->Tenter = threshold_of(p_enter_bad);
  ctx->Tstay = p_leave_bad >= 1.0 ? 0u : threshold_of(1.0 - p_leave_bad);
  return LOSSY_OK;
}

int lossy_set_reliable(lossy_ctx* ctx, const uint64_t* reliable) {
  if (!ctx) return LOSSY_EINVAL;
  if (reinterpret_cast<uintptr_t>(reliable) & 7u) return fail(ctx, LOSSY_EINVAL, "reliable: misaligned");
  if (ctx->K >= (1ull << 32)) return fail(ctx, LOSSY_EINVAL, "too many packets");
  ctx->reliable = reliable;
  return LOSSY_OK;
}

int lossy_packet_sqnorms(lossy_ctx* ctx, const void* const* grads, float* out, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (!out) return fail(ctx, LOSSY_EINVAL, "out: NULL");
  if (int rc = check_table(ctx, grads, "grads: NULL or misaligned pointer")) return rc;
  if (ctx->cfg.n == 0) return LOSSY_OK;
  SqnormArgs A;
  memset(&A, 0, sizeof A);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) A.grads[i] = grads[i];
  A.out = out;
  A.n = ctx->cfg.n;
  A.W = ctx->cfg.W;
  A.P = ctx->cfg.packet_elems;
  A.K = (uint32_t)ctx->K;
  // pieces of at most one chunk: kSqLoads of them per warp at a time (one vector each), else one piece per warp
  const bool many = A.P <= (uint32_t)kChunk;
  const uint64_t tasks = many ? ((uint64_t)A.K + kSqLoads - 1) / kSqLoads : A.K;
  uint64_t blocks = (tasks + 7) / 8;
  // (rounded down: W = 64 took 64 blocks too many, 1216 for 592 or 1184 resident ones)
  const uint64_t cap = (uint64_t)ctx->num_sms * 8 / A.W;
  if (blocks > cap) blocks = cap ? cap : 1;
  const dim3 grid((uint32_t)blocks, A.W);
  cudaStream_t s = (cudaStream_t)stream;
  const bool gb = ctx->cfg.grad_dtype == LOSSY_BF16;
  // Early only with a handful of blocks. Blocks that begin early all go to the SMs that the kernel ahead leaves first, eight to an SM, and
  // read at those few SMs' rate: W = 6, P = 6736, 0.5 M elements, 60 blocks, behind the pairwise drift: 12.5 us as an ordinary launch, 25.1
  // early. 900 random buckets, ordinary over early: up to 15 blocks 1.04 to 1.10 (packets of 4096 and more 0.86 to 1.1), 16 to 31
  // 0.98 to 1.07 (0.68 at the least), 32 to 127 0.68 to 1.02, 128 and more 0.76 to 0.98.
  const cudaError_t e = launch_after(blocks * A.W < 16u, gb ? (many ? packet_sqnorms_kernel<BF16, true> : packet_sqnorms_kernel<BF16, false>)
                                        : (many ? packet_sqnorms_kernel<F32, true> : packet_sqnorms_kernel<F32, false>), grid, 256, 0, s, A);
  if (e != cudaSuccess) return fail_cuda(ctx, "packet norm launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

int lossy_set_lr(lossy_ctx* ctx, float lr) {
  if (!ctx) return LOSSY_EINVAL;
  ctx->cfg.lr = lr;
  return LOSSY_OK;
}

static int aggregate_impl(lossy_ctx* ctx, uint64_t step, const void* const* grads, float* ghat_prev, float* ghat,
                          uint8_t* count, uint64_t* recv_bits, void* stream) {
  if (ctx->cfg.n == 0) return LOSSY_OK;
  if (step == 0) return fail(ctx, LOSSY_EINVAL, "step is 1-based");
  if (int rc = check_table(ctx, grads, "grads: NULL or misaligned pointer")) return rc;
  if (!ghat || !aligned16(ghat)) return fail(ctx, LOSSY_EINVAL, "ghat: NULL or misaligned");
  Params P;
  fill_common(ctx, step, P);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) P.grads[i] = grads[i];
  P.ghat = ghat;
  P.ghat_prev = ghat_prev;
  P.count = count;
  P.recv_bits = recv_bits;
  return run_phase<AGG>(ctx, P, nullptr, nullptr, (cudaStream_t)stream);
}

int lossy_aggregate(lossy_ctx* ctx, uint64_t step, const void* const* grads, float* ghat, uint8_t* count,
                    uint64_t* recv_bits, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  return aggregate_impl(ctx, step, grads, nullptr, ghat, count, recv_bits, stream);
}

static int check_alg1(lossy_ctx* ctx, const float* ghat_prev) {
  if (ctx->cfg.flags & LOSSY_SELF_LOSSLESS)
    return fail(ctx, LOSSY_EINVAL, "LOSSY_SELF_LOSSLESS has no meaning in Algorithm 1 mode");
  if (ctx->cfg.n && (!ghat_prev || !aligned16(ghat_prev))) return fail(ctx, LOSSY_EINVAL, "ghat_prev: NULL or misaligned");
  return LOSSY_OK;
}

int lossy_aggregate_alg1(lossy_ctx* ctx, uint64_t step, const void* const* grads, float* ghat_prev, float* ghat,
                         uint8_t* count, uint64_t* recv_bits, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (int rc = check_alg1(ctx, ghat_prev)) return rc;
  return aggregate_impl(ctx, step, grads, ghat_prev, ghat, count, recv_bits, stream);
}

int lossy_step(lossy_ctx* ctx, uint64_t step, const float* ghat, const uint8_t* count, float* master, float* m,
               float* v, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (ctx->cfg.n == 0) return LOSSY_OK;
  if (step == 0) return fail(ctx, LOSSY_EINVAL, "step is 1-based");
  if (!ghat || !aligned16(ghat) || !master || !aligned16(master)) return fail(ctx, LOSSY_EINVAL, "ghat/master: NULL or misaligned");
  if (ctx->cfg.optimizer == LOSSY_ADAM && (!m || !v || !aligned16(m) || !aligned16(v)))
    return fail(ctx, LOSSY_EINVAL, "Adam needs m and v");
  if ((ctx->cfg.flags & LOSSY_ZERO_SKIP) && !count) return fail(ctx, LOSSY_EINVAL, "LOSSY_ZERO_SKIP needs count");
  Params P;
  fill_common(ctx, step, P);
  P.ghat = const_cast<float*>(ghat);
  P.count_in = count;
  P.master = master;
  P.m = m;
  P.v = v;
  return run_phase<STEP>(ctx, P, nullptr, nullptr, (cudaStream_t)stream);
}

int lossy_broadcast(lossy_ctx* ctx, uint64_t step, const float* master, void* const* replicas, uint64_t* stale_bits,
                    void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (ctx->cfg.n == 0) return LOSSY_OK;
  if (step == 0) return fail(ctx, LOSSY_EINVAL, "step is 1-based");
  if (int rc = check_replicas(ctx, replicas)) return rc;
  if (!master || !aligned16(master)) return fail(ctx, LOSSY_EINVAL, "master: NULL or misaligned");
  Params P;
  fill_common(ctx, step, P);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) P.replicas[i] = replicas[i];
  P.master = const_cast<float*>(master);
  P.stale_bits = stale_bits;
  return run_phase<BCAST>(ctx, P, nullptr, nullptr, (cudaStream_t)stream);
}

int drift_norms(lossy_ctx* ctx, const float* master, const void* const* replicas, float* norms, double* sumsq,
                void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (int rc = check_replicas(ctx, replicas)) return rc;
  if (ctx->cfg.n == 0) {
    if (norms) {
      cudaError_t e = cudaMemsetAsync(norms, 0, ctx->cfg.W * sizeof(float), (cudaStream_t)stream);
      if (e != cudaSuccess) return fail_cuda(ctx, "memset", e);
    }
    return LOSSY_OK;
  }
  if (!master || !aligned16(master)) return fail(ctx, LOSSY_EINVAL, "master: NULL or misaligned");
  Params P;
  fill_common(ctx, 1, P);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) P.replicas[i] = const_cast<void*>(replicas[i]);
  P.master = const_cast<float*>(master);
  return run_phase<DRIFT>(ctx, P, norms, sumsq, (cudaStream_t)stream);
}

static int fused_impl(lossy_ctx* ctx, uint64_t step, const void* const* grads, float* ghat_prev, float* master,
                      float* m, float* v, void* const* replicas, float* ghat, uint8_t* count, uint64_t* recv_bits,
                      uint64_t* stale_bits, float* norms, double* sumsq, void* stream) {
  if (step == 0) return fail(ctx, LOSSY_EINVAL, "step is 1-based");
  if (int rc = check_table(ctx, grads, "grads: NULL or misaligned pointer")) return rc;
  if (int rc = check_replicas(ctx, replicas)) return rc;
  if (ctx->cfg.n == 0) {
    if (norms) {
      cudaError_t e = cudaMemsetAsync(norms, 0, ctx->cfg.W * sizeof(float), (cudaStream_t)stream);
      if (e != cudaSuccess) return fail_cuda(ctx, "memset", e);
    }
    return LOSSY_OK;
  }
  if (!master || !aligned16(master)) return fail(ctx, LOSSY_EINVAL, "master: NULL or misaligned");
  if (ctx->cfg.optimizer == LOSSY_ADAM && (!m || !v || !aligned16(m) || !aligned16(v)))
    return fail(ctx, LOSSY_EINVAL, "Adam needs m and v");
  if (ghat && !aligned16(ghat)) return fail(ctx, LOSSY_EINVAL, "ghat: misaligned");
  Params P;
  fill_common(ctx, step, P);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) {
    P.grads[i] = grads[i];
    P.replicas[i] = replicas[i];
  }
  P.master = master;
  P.m = m;
  P.v = v;
  P.ghat = ghat;
  P.ghat_prev = ghat_prev;
  P.count = count;
  P.recv_bits = recv_bits;
  P.stale_bits = stale_bits;
  cudaStream_t s = (cudaStream_t)stream;
  const bool drift = norms || sumsq;
  if (drift) {
    P.ticket = ctx->ticket;
    P.norms = norms;
    P.sumsq = sumsq;
  }
  return run_launches(ctx, P, drift, s, [&](Params& Q, uint32_t* rows) {
    uint32_t tma_blocks = 0, tail_blocks = 0;
    bool used_tma = false;
    int rc = run_tma(ctx, Q, drift, s, &tma_blocks, &used_tma);
    if (rc) return rc;
    if (used_tma) {
      Q.k_begin = (uint32_t)(ctx->cfg.n / ctx->cfg.packet_elems);
      Q.partials_row0 = tma_blocks;
    } else {
      tma_blocks = 0;
    }
    if (Q.k_begin < Q.K) rc = drift ? dispatch_step<true>(ctx, Q, s, &tail_blocks) : dispatch_step<false>(ctx, Q, s, &tail_blocks);
    *rows = tma_blocks + tail_blocks;
    return rc;
  });
}

int lossy_fused_step(lossy_ctx* ctx, uint64_t step, const void* const* grads, float* master, float* m, float* v,
                     void* const* replicas, float* ghat, uint8_t* count, uint64_t* recv_bits, uint64_t* stale_bits,
                     float* norms, double* sumsq, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  return fused_impl(ctx, step, grads, nullptr, master, m, v, replicas, ghat, count, recv_bits, stale_bits, norms, sumsq,
                    stream);
}

int lossy_fused_step_alg1(lossy_ctx* ctx, uint64_t step, const void* const* grads, float* ghat_prev, float* master,
                          float* m, float* v, void* const* replicas, float* ghat, uint8_t* count,
                          uint64_t* recv_bits, uint64_t* stale_bits, float* norms, double* sumsq, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (int rc = check_alg1(ctx, ghat_prev)) return rc;
  return fused_impl(ctx, step, grads, ghat_prev, master, m, v, replicas, ghat, count, recv_bits, stale_bits, norms,
                    sumsq, stream);
}

int drift_pairwise(lossy_ctx* ctx, const void* const* replicas, double* d2, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (!d2) return fail(ctx, LOSSY_EINVAL, "d2: NULL");
  if (int rc = check_replicas(ctx, replicas)) return rc;
  if (ctx->cfg.n == 0) return LOSSY_OK;
  const lossy_config& c = ctx->cfg;
  cudaStream_t s = (cudaStream_t)stream;
  auto run = [&](auto elide) {
    constexpr bool E = decltype(elide)::value;
    PairwiseArgs<E> A;
    memset(&A, 0, sizeof A);
    for (uint32_t i = 0; i < c.W; ++i) A.replicas[i] = replicas[i];
    A.d2 = d2;
    A.n = c.n;
    A.W = c.W;
    A.segs = 1;
    A.seg_len = c.n;
    if constexpr (E) {
      A.seg_len = (uint64_t)ctx->pps * c.packet_elems;
      A.seg_off = c.shard_packet0 * c.packet_elems;
      A.seg0 = (uint32_t)(c.shard_packet0 / ctx->pps);
      A.segs = (uint32_t)((c.shard_packet0 + ctx->K - 1) / ctx->pps) - A.seg0 + 1u;
      for (uint32_t i = 0; i < c.W; ++i) A.rep_skip[i] = own_elems(ctx, i);
    }
    const uint64_t longest = A.seg_len < c.n ? A.seg_len : c.n;
    A.chunks_per_seg = (uint32_t)((longest + kChunk - 1) / kChunk);
    const uint64_t chunks = (uint64_t)A.segs * A.chunks_per_seg;
    const bool bf16 = c.replica_dtype == LOSSY_BF16;
    const bool small = chunks <= (uint64_t)ctx->num_sms * kPairSmallPerSm;
    // every pair directly where that is never far behind: few replicas of a small bucket (60 k to 250 k: 9-10 us, the sets 9-25),
    // and up to four fp32 replicas of any (bf16 ones: 45 us against 34-54 up to 15 % late at 16 M elements)
    if (c.W >= 2u && c.W <= 8u && (small || (c.W <= 4u && !bf16))) {
      const uint64_t cap = (uint64_t)ctx->num_sms * 3u;
      const uint32_t blocks = (uint32_t)((chunks + 3) / 4 < cap ? (chunks + 3) / 4 : cap);
      return launch_after(false, bf16 ? (c.W <= 4u ? drift_pairwise_few_kernel<BF16, E, 4> : drift_pairwise_few_kernel<BF16, E, 8>)
                               : (c.W <= 4u ? drift_pairwise_few_kernel<F32, E, 4> : drift_pairwise_few_kernel<F32, E, 8>), blocks, 128, 0, s, A);
    }
    auto pick = [&](auto set, auto small) {
      using M = decltype(set);
      constexpr bool S = decltype(small)::value;
      return bf16 ? launch_pairwise<BF16, E, M, S>(ctx, A, s) : launch_pairwise<F32, E, M, S>(ctx, A, s);
    };
    if (c.W <= 32u) return small ? pick(uint32_t{}, std::true_type{}) : pick(uint32_t{}, std::false_type{});
    return small ? pick(uint64_t{}, std::true_type{}) : pick(uint64_t{}, std::false_type{});
  };
  const cudaError_t e = c.flags & LOSSY_REPLICA_SKIP_OWNER ? run(std::true_type{}) : run(std::false_type{});
  if (e != cudaSuccess) return fail_cuda(ctx, "pairwise drift launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

int lossy_closed_loop_grads(lossy_ctx* ctx, const float* curv, const float* target, const void* const* noise,
                            const void* const* replicas, void* const* grads_out, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (ctx->cfg.n == 0) return LOSSY_OK;
  if (ctx->cfg.flags & LOSSY_REPLICA_SKIP_OWNER)
    return fail(ctx, LOSSY_EINVAL, "closed-loop gradients need every worker's full copy (no LOSSY_REPLICA_SKIP_OWNER)");
  if (!curv || !target || !aligned16(curv) || !aligned16(target)) return fail(ctx, LOSSY_EINVAL, "curv/target: NULL or misaligned");
  if (int rc = check_table(ctx, noise, "noise: NULL or misaligned pointer")) return rc;
  if (int rc = check_replicas(ctx, replicas)) return rc;
  if (int rc = check_table(ctx, grads_out, "grads_out: NULL or misaligned pointer")) return rc;
  ClosedLoopArgs A;
  memset(&A, 0, sizeof A);
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) {
    A.noise[i] = noise[i];
    A.replicas[i] = replicas[i];
    A.grads[i] = grads_out[i];
  }
  A.curv = curv;
  A.target = target;
  A.n = ctx->cfg.n;
  A.W = ctx->cfg.W;
  const uint64_t nvec = (A.n + 7) / 8;
  uint64_t blocks = (nvec + 255) / 256;
  const uint64_t cap = (uint64_t)ctx->num_sms * 8;
  if (blocks > cap) blocks = cap;
  const bool gb = ctx->cfg.grad_dtype == LOSSY_BF16, rb = ctx->cfg.replica_dtype == LOSSY_BF16;
  cudaStream_t s = (cudaStream_t)stream;
  // Early up to 64 blocks, and with two or three workers up to three blocks per SM. Beyond, the blocks crowd the SMs that come free first, as
  // the packet norms' do. 2000 random buckets, ordinary over early: up to 64 blocks 1.01 to 1.06; from there on W = 2-3 1.02 to 1.03, W = 4-7
  // 1.00 to 1.02 (0.84 at the least), W = 8-15 0.98 to 0.995 (0.82), W = 16-31 0.96 to 0.99 (0.80), more 0.98 (0.79: W = 59, 0.3 M, fp32,
  // with the step behind it: 95.4 us, early 120.5).
  const cudaError_t e = launch_after(blocks <= 64u || (A.W <= 3u && blocks <= (uint64_t)ctx->num_sms * 3), gb ? (rb ? closed_loop_grads_kernel<BF16, BF16> : closed_loop_grads_kernel<BF16, F32>)
                                        : (rb ? closed_loop_grads_kernel<F32, BF16> : closed_loop_grads_kernel<F32, F32>), (uint32_t)blocks, 256, 0, s, A);
  if (e != cudaSuccess) return fail_cuda(ctx, "closed-loop gradient launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

int lossy_device_status(lossy_ctx* ctx, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  uint32_t word[5] = {0, 0, 0, 0, 0};
  cudaError_t e = cudaMemcpyAsync(word, ctx->status, sizeof word, cudaMemcpyDeviceToHost, (cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e != cudaSuccess) return fail_cuda(ctx, "status read", e);
  if (word[1] != 0) {   // debug build only; a pipeline that skipped a tile also left through its wait exit (word[0])
    static const char* const kSites[] = {"?", "register kernel", "fused bulk-copy pipeline (packed)", "fused bulk-copy pipeline",
                                         "single-phase bulk-copy pipeline", "gather pipeline"};
    const uint32_t site = word[1] & 15u;
    snprintf(ctx->err, sizeof ctx->err, "device index check failed in the %s: %s elements [%llu, +%u) lie outside the array; not touched, the results of that call are invalid",
             site < 6 ? kSites[site] : kSites[0], (word[1] & kSiteReplica) ? "replica" : "slab",
             (unsigned long long)(((uint64_t)word[3] << 32) | word[2]), word[4]);
    return LOSSY_EDEVCHECK;
  }
  if (word[0] != 0) return fail(ctx, LOSSY_EDEVICE, "a bounded wait inside a kernel gave up; results of that call are invalid");
  return LOSSY_OK;
}

int lossy_has_device_checks(void) { return kDevCheck ? 1 : 0; }

int lossy_selftest_shrink_checks(lossy_ctx* ctx, uint64_t elems) {
  if (!ctx) return LOSSY_EINVAL;
  if (!kDevCheck) return fail(ctx, LOSSY_EINVAL, "this library was built without device index checks");
  ctx->check_shrink = elems;
  return LOSSY_OK;
}

int lossy_reset_status(lossy_ctx* ctx, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  cudaError_t e = cudaMemsetAsync(ctx->status, 0, 5 * sizeof(uint32_t), (cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctx->ticket, 0, sizeof(uint32_t), (cudaStream_t)stream);
  if (e != cudaSuccess) return fail_cuda(ctx, "status reset", e);
  ctx->err[0] = 0;
  return LOSSY_OK;
}

int lossy_selftest_wait_expiry(lossy_ctx* ctx, uint32_t max_polls, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (max_polls == 0 || max_polls > (1u << 20)) return fail(ctx, LOSSY_EINVAL, "max_polls: 1 .. 2^20");
  wait_expiry_kernel<<<1, 64, 0, (cudaStream_t)stream>>>(max_polls, ctx->status);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail_cuda(ctx, "self-test launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

int lossy_fused_step_host(lossy_ctx* ctx, uint64_t step, const void* const* host_grads, void* const* dev_grads,
                          float* master, float* m, float* v, void* const* replicas, float* dev_norms,
                          float* host_norms, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (!host_grads || !dev_norms || !host_norms) return fail(ctx, LOSSY_EINVAL, "NULL argument");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t gbytes = (size_t)ctx->cfg.n * (ctx->cfg.grad_dtype == LOSSY_BF16 ? 2 : 4);
  // Zero-copy: when every host buffer is pinned and mapped into the device's address space, the kernel
  // reads the gradients over PCIe itself, so packets that the network dropped are never transferred at all
  // and no staging copy is made. Otherwise (pageable memory) each buffer is staged with cudaMemcpyAsync.
  const void* mapped[LOSSY_MAX_WORKERS];
  bool zero_copy = true;
  for (uint32_t i = 0; i < ctx->cfg.W; ++i) {
    if (!host_grads[i]) return fail(ctx, LOSSY_EINVAL, "NULL gradient pointer");
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, host_grads[i]) != cudaSuccess) { cudaGetLastError(); zero_copy = false; continue; }
    if (attr.type != cudaMemoryTypeHost || !attr.devicePointer || !aligned16(attr.devicePointer)) zero_copy = false;
    mapped[i] = attr.devicePointer;
  }
  const void* const* step_grads = mapped;
  if (!zero_copy) {
    for (uint32_t i = 0; i < ctx->cfg.W; ++i) {
      if (!dev_grads || !dev_grads[i]) return fail(ctx, LOSSY_EINVAL, "pageable host gradients need staging buffers");
      if (gbytes) {
        cudaError_t e = cudaMemcpyAsync(dev_grads[i], host_grads[i], gbytes, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return fail_cuda(ctx, "gradient upload", e);
      }
    }
    step_grads = dev_grads;
  }
  if (int rc = lossy_fused_step(ctx, step, step_grads, master, m, v, replicas, nullptr, nullptr, nullptr, nullptr,
                                dev_norms, nullptr, stream))
    return rc;
  cudaError_t e = cudaMemcpyAsync(host_norms, dev_norms, ctx->cfg.W * sizeof(float), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return fail_cuda(ctx, "norm download", e);
  return lossy_device_status(ctx, stream);   // synchronises the stream
}

uint32_t lossy_hash_u32(uint64_t seed, uint64_t step, uint32_t src, uint32_t dst, uint64_t packet) {
  return pair_hash(packet_key_of(step_key_of(seed, step), packet), src, dst);
}

int lossy_mask(const lossy_ctx* ctx, uint64_t step, uint32_t src, uint32_t dst, uint64_t packet, int is_param) {
  if (!ctx) return -1;
  const uint32_t T = is_param ? ctx->Tp : ctx->Tg;
  return lossy_hash_u32(ctx->cfg.seed, step, src, dst, packet) >= T ? 1 : 0;
}

int lossy_mask_grid(lossy_ctx* ctx, uint64_t step, const uint32_t* src, const uint32_t* dst, const uint64_t* packet,
                    uint64_t count, int is_param, uint8_t* out, void* stream) {
  if (!ctx) return LOSSY_EINVAL;
  if (count == 0) return LOSSY_OK;
  if (!src || !dst || !packet || !out) return fail(ctx, LOSSY_EINVAL, "NULL argument");
  const uint64_t blocks = (count + 255) / 256;
  if (blocks > 0x7FFFFFFFull) return fail(ctx, LOSSY_EINVAL, "grid too large");
  mask_grid_kernel<<<(uint32_t)blocks, 256, 0, (cudaStream_t)stream>>>(ctx->cfg.seed, step, src, dst, packet, count,
                                                                      is_param ? ctx->Tp : ctx->Tg, out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail_cuda(ctx, "mask grid launch", e);
  ctx->launches++;
  return LOSSY_OK;
}

const char* lossy_last_error(const lossy_ctx* ctx) { return ctx ? ctx->err : "NULL context"; }
uint64_t lossy_num_packets(const lossy_ctx* ctx) { return ctx ? ctx->K : 0; }
uint64_t lossy_replica_elems(const lossy_ctx* ctx, uint32_t worker) {
  if (!ctx || worker >= ctx->cfg.W) return 0;
  return (ctx->cfg.flags & LOSSY_REPLICA_SKIP_OWNER) ? ctx->cfg.n - own_elems(ctx, worker) : ctx->cfg.n;
}
uint64_t lossy_kernel_launches(const lossy_ctx* ctx) { return ctx ? ctx->launches : 0; }

int lossy_describe_plan(lossy_ctx* ctx, int with_drift, char* buf, size_t size) {
  if (!ctx || !buf || size == 0) return LOSSY_EINVAL;
  snprintf(buf, size, "register kernel");
  if (ctx->cfg.n == 0) return LOSSY_OK;
  Params P;
  fill_common(ctx, 1, P);
  uint32_t blocks = 0;
  bool used = false;
  ctx->plan = buf;
  ctx->plan_size = size;
  ctx->plan_only = true;             // sizes grids, launches nothing
  const bool drift = (with_drift & ~LOSSY_PLAN_BUILD) != 0;
  int rc = run_tma(ctx, P, drift, nullptr, &blocks, &used);
  if (!rc && !used && (with_drift & LOSSY_PLAN_BUILD)) rc = drift ? dispatch_step<true>(ctx, P, nullptr, &blocks) : dispatch_step<false>(ctx, P, nullptr, &blocks);
  ctx->plan_only = false;
  ctx->plan = nullptr;
  return rc;
}

}  // extern "C"
