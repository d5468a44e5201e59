// engine.cuh -- batched execution of requests (f12int_submit / f12int_poll).
//
// Included by f12int.cu after the kernels and the context definition.
//
// A request asks for the blocks of some classes over one quartet list of one
// basis.  A worker thread merges the pending requests -- of any bases and any
// mix of (la, lb, lc, ld) -- into a batch, writes the batch's lists to pinned
// staging memory, copies them to fixed device buffers and replays one
// captured CUDA graph: one for bases inside the factor's grid of auxiliary
// functions, one for those that go family by family (a batch holds requests of
// one sort).  A graph holds, for every class, the Hermite rows of the general
// quartets (behind the four passes over the work items in the second graph),
// one contraction launch per tier (threads and shared memory of a block) and
// one per key of the thin kernel, all persistent (grid-stride over counts read
// from device memory), so the same graph serves every batch.  The six class
// pipelines are parallel branches of the graph, each with its own buffers, and
// the contraction launches of a class go over four streams.  A batch whose rows
// exceed a class's buffer is replayed in passes; a single quartet that does is
// launched by itself.  Two staging buffers let the host build batch
// k+1 while batch k runs.  The method is that of f12int_compute_class; only
// the scheduling differs.

namespace {

// Default work of one contraction task of a batch, in flops, and the unit of
// the schedules that f12int_batch_autotune tries.
constexpr double kTaskFlops = 5e7;

// contraction tiers: threads and shared memory of a block
constexpr int kTiers = 6;                // per precision
constexpr int kTierThreads[kTiers] = {32, 64, 96, 192, 256, 256};
constexpr size_t kTierCap[kTiers] = {14 * 1024, 28 * 1024, 42 * 1024, 54 * 1024, 72 * 1024, 200 * 1024};
constexpr int kLaunches = 2 * kTiers;     // FP64 tiers, then FP32 tiers (mixed requests)
constexpr int kThinSlot = kLaunches;      // then the thin contraction (total order <= 3, I5 <= 2), one
constexpr int kSlots = kLaunches + kThinKeys;   // launch per (la, lb, lc, ld)

struct EngineReq {
  uint64_t ticket = 0;
  int basis = 0;
  const f12int_ctx::BasisData *B = nullptr;   // stable: the deque never moves its elements
  uint32_t mask = 0;
  bool grid = false;                  // every class from the auxiliary grid
  int precision = 0;                  // 1: contraction in FP32 below the FP32 bound
  double thresh = 0.0;
  double *out = nullptr;
  std::vector<int32_t> q;
  std::vector<int64_t> off;       // [nclass][n]
  int64_t quartets[7] = {0};      // quartets per class (before screening)
  int64_t items[7] = {0};         // work items per class (before screening)
  int64_t tasks[7] = {0};         // contraction tasks per class (before screening)
};

using f12engine::TicketState;

// Contraction plan of a quartet in a batch: ket ranges (the fewest that fit,
// more while a task would exceed `target` flops), the tier that holds them,
// and the work of one task.
struct BatchPlan {
  int tier, nsplit;
  bool swap;        // listed as (cd|ab), the bra inner
  double work;
};

static bool batch_plan(int la, int lb, int lc, int ld, int cls, int64_t npab, int64_t npcd, double target,
                       BatchPlan *bp, bool fp32 = false) {
  const int key = (la << 6) | (lb << 4) | (lc << 2) | ld;
  bp->swap = false;
  if (thin_quartet(key, cls)) {   // one warp, FP64 (mixed requests too)
    bp->tier = kThinSlot + thin_slot(key, cls == 5);
    bp->nsplit = 1;
    bp->work = (double)(npab * npcd);
    return true;
  }
  bp->swap = bra_inner(la, lb, lc, ld, cls, npab, npcd);
  const ContractShape s = contract_shape(la, lb, lc, ld, cls, bp->swap);
  const int64_t nprimq = npab * npcd, nin = bp->swap ? npab : npcd;
  const size_t esz = fp32 ? 4 : 8;
  const ContractPlan pl = contract_plan(s, nprimq, nin, esz, 0.5 * target);
  if (pl.smem == 0) return false;
  const size_t least = contract_smem(s, 1, pl.nsplit, esz, 0);
  for (int t = 0; t < kTiers; ++t)
    if (kTierCap[t] >= least && (kTierThreads[t] >= pl.nthr || t == kTiers - 1)) {
      bp->tier = t + (fp32 ? kTiers : 0);
      bp->nsplit = pl.nsplit;
      bp->work = (double)nprimq * task_fmas(s, nin, (s.ncd() + pl.nsplit - 1) / pl.nsplit);
      return true;
    }
  return false;
}

// Per-class lists of a batch; the same layout on the device and in each
// pinned staging buffer.
struct ClassLists {
  int32_t *quartets = nullptr;    // [qcap][4]
  int64_t *pq_off = nullptr;      // [qcap + 1]
  int64_t *row_off = nullptr;     // [qcap + 1] first double of a general quartet's Hermite rows
  int64_t *offsets = nullptr;     // [qcap]
  int32_t *qslot = nullptr;       // [qcap]
  CTask *tasks = nullptr;         // [tcap], tier after tier
  int64_t *counts = nullptr;      // n, npq, npq before the thin quartets, then (begin, end) of the tasks of each tier
  PairView *views = nullptr;      // [scap]
  double **outs = nullptr;        // [scap]
};
constexpr int kCounts = 3 + 2 * kSlots;
constexpr int kTaskCounts = 3;           // first of the tiers' (begin, end)

struct Engine {
  // limits
  int64_t qcap = (int64_t)1 << 19;   // quartets per class per batch
  int64_t icap = 0;                   // work items per class per batch (0: from free HBM)
  int64_t tcap = 0;                   // contraction tasks per class per batch
  int64_t scap = 4096;                // requests per batch
  int64_t zcap = 0;                   // zero-filled blocks per batch
  bool ready = false;
  // device buffers
  ClassLists dev[7];
  double **zero_dst = nullptr;
  int64_t *zero_len = nullptr, *zero_count = nullptr;
  int *keys[7] = {nullptr};             // per class: item keys, key order, histogram, partials
  unsigned *order[7] = {nullptr}, *hist[7] = {nullptr};
  double *part[7] = {nullptr};
  double *rows[2][7] = {};              // Hermite rows: per class by graph (the grid graph's are all of part)
  bool rows_own = false;                // rows[0] are buffers of their own (else the ends of part)
  int64_t rcap[2] = {0, 0};             // doubles of them
  unsigned *status = nullptr;
  size_t bytes = 0;
  // staging (pinned), two buffers
  ClassLists stage[2][7];
  double **zstage_dst[2] = {nullptr, nullptr};
  int64_t *zstage_len[2] = {nullptr, nullptr}, *zstage_count[2] = {nullptr, nullptr};
  unsigned *stage_status[2] = {nullptr, nullptr};
  cudaEvent_t ev[2] = {nullptr, nullptr};
  std::vector<uint64_t> inflight[2];
  // graph
  cudaStream_t stream = nullptr;
  cudaStream_t branch[7] = {nullptr};   // capture streams of the class branches
  cudaStream_t sub[7][3] = {};          // and of their parallel parts
  // one graph for batches evaluated from the auxiliary grid, one for batches
  // evaluated family by family; a batch is all of one kind
  cudaGraphExec_t exec[2] = {nullptr, nullptr};
  bool graph_dirty[2] = {true, true};
  int items_blocks = 0, quad_blocks = 0, classify_blocks = 0, grid_blocks = 0, tier_blocks[kLaunches] = {0};
  int thin_blocks = 0;           // persistent thin contraction launches
  double fp32_below = 1e-5;           // mixed requests: FP32 below this screening estimate
  // per-class schedule (f12int_batch_autotune): work target of a contraction
  // task and the divisor of the auxiliary-stage grid
  double task_target[7] = {kTaskFlops, kTaskFlops, kTaskFlops, kTaskFlops, kTaskFlops, kTaskFlops, kTaskFlops};
  int items_div[7] = {1, 1, 1, 1, 1, 1, 1};
  // queue
  std::thread worker;
  std::mutex mu;
  std::condition_variable cv;
  bool stop = false;
  std::deque<EngineReq *> pending;
  std::unordered_map<uint64_t, TicketState> tickets;
  uint64_t next_ticket = 1;
  int cur = 0;
  int64_t batches = 0, requests_done = 0;
};

template <class T>
static int engine_alloc(f12int_ctx *ctx, Engine &E, T **p, size_t n) {
  int rc = dalloc(ctx, p, sizeof(T) * std::max<size_t>(n, 1));
  if (rc == F12INT_OK) E.bytes += sizeof(T) * std::max<size_t>(n, 1);
  return rc;
}

template <class T>
static int stage_alloc(T **p, size_t n) {
  const cudaError_t e = cudaHostAlloc((void **)p, sizeof(T) * std::max<size_t>(n, 1), cudaHostAllocDefault);
  if (e == cudaSuccess) return F12INT_OK;
  cuda_fail(e);
  return F12INT_ENOMEM;
}

static int lists_alloc_dev(f12int_ctx *ctx, Engine &E, ClassLists &L) {
  int rc = engine_alloc(ctx, E, &L.quartets, 4 * (size_t)E.qcap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.pq_off, (size_t)E.qcap + 1);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.row_off, (size_t)E.qcap + 1);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.offsets, (size_t)E.qcap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.qslot, (size_t)E.qcap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.tasks, (size_t)E.tcap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.counts, (size_t)kCounts);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.views, (size_t)E.scap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &L.outs, (size_t)E.scap);
  return rc;
}

static int lists_alloc_host(Engine &E, ClassLists &L) {
  int rc = stage_alloc(&L.quartets, 4 * (size_t)E.qcap);
  if (rc == F12INT_OK) rc = stage_alloc(&L.pq_off, (size_t)E.qcap + 1);
  if (rc == F12INT_OK) rc = stage_alloc(&L.row_off, (size_t)E.qcap + 1);
  if (rc == F12INT_OK) rc = stage_alloc(&L.offsets, (size_t)E.qcap);
  if (rc == F12INT_OK) rc = stage_alloc(&L.qslot, (size_t)E.qcap);
  if (rc == F12INT_OK) rc = stage_alloc(&L.tasks, (size_t)E.tcap);
  if (rc == F12INT_OK) rc = stage_alloc(&L.counts, (size_t)kCounts);
  if (rc == F12INT_OK) rc = stage_alloc(&L.views, (size_t)E.scap);
  if (rc == F12INT_OK) rc = stage_alloc(&L.outs, (size_t)E.scap);
  return rc;
}

static void lists_free(ClassLists &L, bool host) {
  void *ps[] = {L.quartets, L.pq_off, L.row_off, L.offsets, L.qslot, L.tasks, L.counts, L.views, L.outs};
  for (void *p : ps)
    if (p) host ? cudaFreeHost(p) : cudaFree(p);
  L = ClassLists{};
}

// Zero-fill the blocks of screened-out quartets.
__global__ void k_zero_blocks(double *const *dst, const int64_t *len, const int64_t *count) {
  const int64_t n = *count;
  for (int64_t b = blockIdx.x; b < n; b += gridDim.x) {
    double *d = dst[b];
    for (int64_t i = threadIdx.x; i < len[b]; i += blockDim.x) d[i] = 0.0;
  }
}

// Capture the launch sequence of one batch (every class, every tier).
static int engine_capture(f12int_ctx *ctx, Engine &E, bool grid) {
  if (E.exec[grid]) {
    cudaGraphExecDestroy(E.exec[grid]);
    E.exec[grid] = nullptr;
  }
  for (int t = 0; t < kTiers; ++t)
    if (kTierCap[t] > 48 * 1024) {
      CK(cudaFuncSetAttribute(k_contract<true, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
      CK(cudaFuncSetAttribute(k_contract<true, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    }
  cudaStream_t cs = nullptr;
  CK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  cudaEvent_t fork = nullptr, join[7] = {nullptr}, mid[2][7] = {}, done[3][7] = {};
  CK(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
  for (int c = 1; c <= 6; ++c) {
    CK(cudaEventCreateWithFlags(&join[c], cudaEventDisableTiming));
    for (cudaEvent_t *e : {&mid[0][c], &mid[1][c], &done[0][c], &done[1][c], &done[2][c]})
      CK(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
  }
  const PairView none{};
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    k_zero_blocks<<<4 * kSMs, 128, 0, cs>>>(E.zero_dst, E.zero_len, E.zero_count);
    cudaEventRecord(fork, cs);
    for (int cls = 1; cls <= 6; ++cls) {
      cudaStream_t bs = E.branch[cls];
      cudaStreamWaitEvent(bs, fork, 0);
      const int kcls = cls == 5 ? 3 : cls;
      // (a class without a grid has no quartets in a grid batch)
      const GridView G = grid ? class_view(ctx, cls) : GridView{nullptr, nullptr, nullptr};
      if (grid && !G.direct()) {
        cudaEventRecord(join[cls], bs);
        cudaStreamWaitEvent(cs, join[cls], 0);
        continue;
      }
      const int nf = G.direct() ? 1 : ctx->tables.nfam[kcls];
      if (nf <= 0) {   // a class the factor leaves out
        cudaEventRecord(join[cls], bs);
        cudaStreamWaitEvent(cs, join[cls], 0);
        continue;
      }
      const ClassLists &L = E.dev[cls];
      QuartetView QV{L.quartets, L.pq_off, 0, L.counts, L.qslot, L.views, L.outs};
      const RowView rows{E.rows[grid][cls], L.row_off, 0, 0};
      // parallel parts of the class: the branch itself and E.sub
      cudaStream_t part[4] = {bs, E.sub[cls][0], E.sub[cls][1], E.sub[cls][2]};
      auto spread = [&](cudaEvent_t ev) {
        cudaEventRecord(ev, bs);
        for (int i = 1; i < 4; ++i) cudaStreamWaitEvent(part[i], ev, 0);
      };
      auto thin = [&](int first, int count) {   // one persistent launch per thin (la, lb, lc, ld) of the class kind
        int i = 0;
        for (int k = 0; k < 256; ++k) {
          const int slot = thin_quartet(k, cls) ? thin_slot(k, cls == 5) : -1;
          if (slot < 0) continue;
          thin_kernel(k, cls == 5)<<<E.thin_blocks, 32 * kThinWarps, 0, part[first + i++ % count]>>>(
              none, QV, nf, 0, G, L.tasks, 0, L.counts + kTaskCounts + 2 * (kThinSlot + slot), E.keys[cls],
              E.part[cls], nullptr, L.offsets, nullptr);
        }
      };
      if (G.direct()) {
        // the thin contraction needs no rows and runs beside them
        spread(mid[0][cls]);
        thin(2, 2);
        k_hermite_rows<true, true><<<E.grid_blocks, BLOCK_AUX, 0, bs>>>(G, none, QV, cls, 1, 0, -1, E.keys[cls],
                                                                        nullptr, rows, nullptr);
      } else {
        cudaMemsetAsync(E.hist[cls], 0, sizeof(unsigned) * kNKeys, bs);
        k_items_classify<true><<<E.classify_blocks, BLOCK_AUX, 0, bs>>>(ctx->tables, none, QV, cls, 0, 0,
                                                                        E.keys[cls], E.hist[cls]);
        k_items_scan<<<1, 1024, 0, bs>>>(E.hist[cls], kNKeys);
        k_items_scatter<<<E.classify_blocks, BLOCK_AUX, 0, bs>>>(QV, nf, 0, E.keys[cls], E.hist[cls], 0,
                                                                 E.order[cls]);
        k_items_eval<true><<<std::max(1, E.items_blocks / E.items_div[cls]), BLOCK_AUX, 0, bs>>>(
            ctx->tables, none, QV, cls, 0, 0, E.order[cls], E.keys[cls], E.part[cls], E.status, nullptr);
        if (ctx->cls_quad[cls])   // families evaluated by quadrature (b < 0, alpha0 < -1)
          k_items_eval<true, true><<<E.quad_blocks, BLOCK_AUX, 0, bs>>>(ctx->tables, none, QV, cls, 0, 0,
                                                                         E.order[cls], E.keys[cls], E.part[cls],
                                                                         E.status, nullptr);
        spread(mid[0][cls]);
        thin(2, 2);
        k_hermite_rows<true, false><<<E.grid_blocks, BLOCK_AUX, 0, bs>>>(G, none, QV, cls, nf, 0, -1, E.keys[cls],
                                                                         E.part[cls], rows, nullptr);
      }
      cudaEventRecord(mid[1][cls], bs);
      cudaStreamWaitEvent(part[1], mid[1][cls], 0);
      for (int t = 0; t < kLaunches; ++t) {
        const int tt = t % kTiers;
        const auto kern = t < kTiers ? k_contract<true, double> : k_contract<true, float>;
        kern<<<E.tier_blocks[t], kTierThreads[tt], kTierCap[tt], part[t & 1]>>>(
            none, QV, cls, nf, 0, L.tasks, 0, L.counts + kTaskCounts + 2 * t, E.keys[cls], rows, nullptr, L.offsets,
            -1, -1, nullptr);
      }
      for (int i = 1; i < 4; ++i) {
        cudaEventRecord(done[i - 1][cls], part[i]);
        cudaStreamWaitEvent(bs, done[i - 1][cls], 0);
      }
      cudaEventRecord(join[cls], bs);
      cudaStreamWaitEvent(cs, join[cls], 0);
    }
    e = cudaStreamEndCapture(cs, &g);
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&E.exec[grid], g, 0);
  if (g) cudaGraphDestroy(g);
  cudaStreamDestroy(cs);
  cudaEventDestroy(fork);
  for (int c = 1; c <= 6; ++c)
    for (cudaEvent_t e : {join[c], mid[0][c], mid[1][c], done[0][c], done[1][c], done[2][c]}) cudaEventDestroy(e);
  if (e != cudaSuccess) return cuda_fail(e);
  E.graph_dirty[grid] = false;
  return F12INT_OK;
}

// Hermite rows of the family path's batches (a batch with more of them runs in
// several passes): 64 MB a class where that is little of the memory left, else
// the ends of the item buffers.  Allocated with the other buffers, under the
// context's lock: the worker allocates nothing, and a request that was
// admitted is not refused later for want of memory.
static void engine_family_rows(f12int_ctx *ctx, Engine &E) {
  const int64_t least = f12engine::rows_least(E.icap);
  size_t left = 0, total = 0;
  if (cudaMemGetInfo(&left, &total) != cudaSuccess) left = 0;
  if (ctx->budget) left = std::min(left, ctx->budget > ctx->used ? ctx->budget - ctx->used : (size_t)0);
  const int64_t want = std::min({(int64_t)8 << 20, E.icap * kPartPitch + least, (int64_t)(left / (16 * 6 * sizeof(double)))});
  int rc = want > least ? F12INT_OK : F12INT_ENOMEM;
  for (int c = 1; c <= 6 && rc == F12INT_OK; ++c) rc = engine_alloc(ctx, E, &E.rows[0][c], (size_t)want);
  E.rows_own = rc == F12INT_OK;
  E.rcap[0] = E.rows_own ? want : least;
  if (E.rows_own) return;
  for (int c = 1; c <= 6; ++c) {
    if (E.rows[0][c]) {
      dfree(ctx, E.rows[0][c], sizeof(double) * (size_t)want);
      E.bytes -= sizeof(double) * (size_t)want;
    }
    E.rows[0][c] = E.part[c] + E.icap * kPartPitch;
  }
}

// Buffers, streams and launch shapes; called once, at the first submit.
static int engine_init(f12int_ctx *ctx, Engine &E) {
  if (E.icap == 0) {
    // admission by free device memory: the six classes' item buffers take at
    // most a quarter of what is free (and of what the budget leaves)
    size_t free_b = 0, total_b = 0;
    CK(cudaMemGetInfo(&free_b, &total_b));
    if (ctx->budget) free_b = std::min(free_b, ctx->budget > ctx->used ? ctx->budget - ctx->used : (size_t)0);
    const size_t per_item = sizeof(int) + sizeof(unsigned) + sizeof(double) * kPartPitch;
    const int64_t fit = (int64_t)(free_b / 4 / (6 * per_item));
    E.icap = std::min<int64_t>((int64_t)1 << 26, fit);
    if (E.icap < ((int64_t)1 << 16)) return F12INT_ENOMEM;
  }
  E.tcap = 4 * E.qcap;
  E.zcap = 6 * E.qcap;
  int rc = F12INT_OK;
  for (int c = 1; c <= 6 && rc == F12INT_OK; ++c) rc = lists_alloc_dev(ctx, E, E.dev[c]);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.zero_dst, (size_t)E.zcap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.zero_len, (size_t)E.zcap);
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.zero_count, 1);
  for (int c = 1; c <= 6 && rc == F12INT_OK; ++c) {
    rc = engine_alloc(ctx, E, &E.keys[c], (size_t)E.icap);
    if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.order[c], (size_t)E.icap);
    // the items' partial rows and, past them, the Hermite rows that any request
    // needs; a batch on the grid has no items, and takes all of it for its rows
    E.rcap[1] = E.icap * kPartPitch + f12engine::rows_least(E.icap);
    if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.part[c], (size_t)E.rcap[1]);
    E.rows[1][c] = E.part[c];
    if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.hist[c], (size_t)kNKeys);
    if (rc == F12INT_OK && cudaStreamCreateWithFlags(&E.branch[c], cudaStreamNonBlocking) != cudaSuccess)
      rc = F12INT_ECUDA;
    for (cudaStream_t &t : E.sub[c])
      if (rc == F12INT_OK && cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking) != cudaSuccess) rc = F12INT_ECUDA;
  }
  if (rc == F12INT_OK) rc = engine_alloc(ctx, E, &E.status, 1);
  for (int b = 0; b < 2 && rc == F12INT_OK; ++b) {
    for (int c = 1; c <= 6 && rc == F12INT_OK; ++c) rc = lists_alloc_host(E, E.stage[b][c]);
    if (rc == F12INT_OK) rc = stage_alloc(&E.zstage_dst[b], (size_t)E.zcap);
    if (rc == F12INT_OK) rc = stage_alloc(&E.zstage_len[b], (size_t)E.zcap);
    if (rc == F12INT_OK) rc = stage_alloc(&E.zstage_count[b], 1);
    if (rc == F12INT_OK) rc = stage_alloc(&E.stage_status[b], 1);
    if (rc == F12INT_OK && cudaEventCreateWithFlags(&E.ev[b], cudaEventDisableTiming) != cudaSuccess)
      rc = F12INT_ECUDA;
  }
  if (rc == F12INT_OK && cudaStreamCreateWithFlags(&E.stream, cudaStreamNonBlocking) != cudaSuccess)
    rc = F12INT_ECUDA;
  if (rc == F12INT_OK && clear(E.status, sizeof(unsigned), E.stream) != cudaSuccess) rc = F12INT_ECUDA;
  if (rc != F12INT_OK) return rc;
  engine_family_rows(ctx, E);
  // persistent launch shapes: resident blocks per SM from registers and shared memory
  int nsm = 0;
  CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  int per = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_items_eval<true>, BLOCK_AUX, 0));
  E.items_blocks = nsm * std::max(per, 1);
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_items_eval<true, true>, BLOCK_AUX, 0));
  E.quad_blocks = nsm * std::max(per, 1);
  E.classify_blocks = nsm * 8;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_hermite_rows<true, true>, BLOCK_AUX, 0));
  E.grid_blocks = nsm * std::max(per, 1);
  for (int t = 0; t < kTiers; ++t) {
    if (kTierCap[t] > 48 * 1024) {
      CK(cudaFuncSetAttribute(k_contract<true, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
      CK(cudaFuncSetAttribute(k_contract<true, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    }
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_contract<true, double>, kTierThreads[t], kTierCap[t]));
    E.tier_blocks[t] = nsm * std::max(per, 1);
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_contract<true, float>, kTierThreads[t], kTierCap[t]));
    E.tier_blocks[kTiers + t] = nsm * std::max(per, 1);
  }
  E.thin_blocks = nsm * 4;   // 16 warps per SM: the thin launches of a batch are mostly small
  E.ready = true;
  return F12INT_OK;
}

// Mark the requests of the batch in staging buffer b done (the batch's event
// has completed).  Caller holds E.mu.
static void engine_finish_batch(Engine &E, int b) {
  const int rc = *E.stage_status[b] ? F12INT_EDEVICE : F12INT_OK;
  for (uint64_t t : E.inflight[b]) {
    auto it = E.tickets.find(t);
    if (it != E.tickets.end()) {
      it->second.done = true;
      it->second.rc = rc;
      it->second.batch = -1;
    }
    ++E.requests_done;
  }
  E.inflight[b].clear();
}

// One general quartet whose Hermite rows exceed the class's buffer, alone in
// the lists: a few of its bra primitive pairs at a time, by plain launches.
static int engine_large(f12int_ctx *ctx, Engine &E, int cls, bool grid, int64_t npab, int64_t npq, int64_t rows_q,
                        int tier) {
  const ClassLists &L = E.dev[cls];
  cudaStream_t st = E.stream;
  const PairView none{};
  QuartetView QV{L.quartets, L.pq_off, 0, L.counts, L.qslot, L.views, L.outs};
  const GridView G = grid ? class_view(ctx, cls) : GridView{nullptr, nullptr, nullptr};
  const int nf = G.direct() ? 1 : ctx->tables.nfam[cls == 5 ? 3 : cls];
  if (!G.direct()) {
    CK(cudaMemsetAsync(E.hist[cls], 0, sizeof(unsigned) * kNKeys, st));
    k_items_classify<true><<<E.classify_blocks, BLOCK_AUX, 0, st>>>(ctx->tables, none, QV, cls, 0, 0, E.keys[cls],
                                                                    E.hist[cls]);
    k_items_scan<<<1, 1024, 0, st>>>(E.hist[cls], kNKeys);
    k_items_scatter<<<E.classify_blocks, BLOCK_AUX, 0, st>>>(QV, nf, 0, E.keys[cls], E.hist[cls], 0, E.order[cls]);
    k_items_eval<true><<<E.items_blocks, BLOCK_AUX, 0, st>>>(ctx->tables, none, QV, cls, 0, 0, E.order[cls],
                                                             E.keys[cls], E.part[cls], E.status, nullptr);
    if (ctx->cls_quad[cls])
      k_items_eval<true, true><<<E.quad_blocks, BLOCK_AUX, 0, st>>>(ctx->tables, none, QV, cls, 0, 0, E.order[cls],
                                                                     E.keys[cls], E.part[cls], E.status, nullptr);
  }
  const int64_t npcd = npq / npab, per = rows_q / npab, step = E.rcap[grid] / per;
  if (step < 1) return F12INT_ENOMEM;
  for (int64_t i0 = 0; i0 < npab; i0 += step) {
    const int64_t i1 = std::min(npab, i0 + step), a = i0 * npcd, n = (i1 - i0) * npcd;
    const RowView rows{E.rows[grid][cls], L.row_off, i0 * per, 0};
    const unsigned nb = (unsigned)((n + BLOCK_AUX - 1) / BLOCK_AUX);
    if (G.direct())
      k_hermite_rows<true, true><<<nb, BLOCK_AUX, 0, st>>>(G, none, QV, cls, 1, a, n, E.keys[cls], nullptr, rows,
                                                           nullptr);
    else
      k_hermite_rows<true, false><<<nb, BLOCK_AUX, 0, st>>>(G, none, QV, cls, nf, a, n, E.keys[cls] + a * nf,
                                                            E.part[cls] + a * nf * kPartPitch, rows, nullptr);
    const auto kern = tier < kTiers ? k_contract<true, double> : k_contract<true, float>;
    kern<<<E.tier_blocks[tier], kTierThreads[tier % kTiers], kTierCap[tier % kTiers], st>>>(
        none, QV, cls, nf, G.direct() ? a : 0, L.tasks, 0, L.counts + kTaskCounts + 2 * tier, E.keys[cls], rows,
        nullptr, L.offsets, (int)i0, (int)i1, nullptr);
  }
  CK(cudaGetLastError());
  return F12INT_OK;
}

// Build the lists of one batch in staging buffer b and launch it: one replay of
// the graph, or several where the Hermite rows of the batch exceed a class's
// buffer.
static int engine_launch(f12int_ctx *ctx, Engine &E, const std::vector<EngineReq *> &batch, int b, bool grid) {
  struct Item {
    int32_t q[4];
    int32_t req;
    int64_t off;
    int64_t npab, npcd, rows;
    int tier, nsplit;
    bool swap;
    double work;      // per task
  };
  int64_t nzero = 0;
  std::vector<Item> all[7];
  for (int cls = 1; cls <= 6; ++cls) {
    std::vector<Item> &items = all[cls];
    // gather the class's quartets of every request
    double total = 0.0;
    for (size_t r = 0; r < batch.size(); ++r) {
      const EngineReq &R = *batch[r];
      if (!(R.mask & (1u << (cls - 1)))) continue;
      int row = 0;
      for (int c = 1; c < cls; ++c) row += (R.mask >> (c - 1)) & 1;
      const f12int_ctx::BasisData &B = *R.B;
      const int nq = (int)(R.q.size() / 4);
      const bool mixed = R.precision == 1;
      for (int i = 0; i < nq; ++i) {
        const int32_t *s = &R.q[4 * (size_t)i];
        const int64_t off = R.off[(size_t)row * nq + i];
        const int la = B.l[s[0]], lb = B.l[s[1]], lc = B.l[s[2]], ld = B.l[s[3]];
        const double est =
            (R.thresh > 0.0 || mixed) ? screen_estimate(ctx, B, cls, s[0], s[1], s[2], s[3]) : 0.0;
        if (R.thresh > 0.0 && est < R.thresh) {
          E.zstage_dst[b][nzero] = R.out + off;
          E.zstage_len[b][nzero] = (int64_t)ncart(la) * ncart(lb) * ncart(lc) * ncart(ld);
          ++nzero;
          continue;
        }
        Item it{};
        for (int k = 0; k < 4; ++k) it.q[k] = s[k];
        it.req = (int32_t)r;
        it.off = off;
        it.npab = (int64_t)B.nprim[s[0]] * B.nprim[s[1]];
        it.npcd = (int64_t)B.nprim[s[2]] * B.nprim[s[3]];
        it.tier = mixed && est < E.fp32_below ? 1 : 0;   // (the tier proper below)
        if (!thin_quartet((la << 6) | (lb << 4) | (lc << 2) | ld, cls)) {
          it.swap = bra_inner(la, lb, lc, ld, cls, it.npab, it.npcd);
          const ContractShape sh = contract_shape(la, lb, lc, ld, cls, it.swap);
          it.rows = it.npab * it.npcd * row_pitch(sh.L());
          total += (double)(it.npab * it.npcd) * task_fmas(sh, it.swap ? it.npab : it.npcd, sh.ncd());
        }
        items.push_back(it);
      }
    }
    // about a dozen tasks per SM where the batch has the work for it, within
    // the task capacity (a block's result does not depend on the cut)
    auto plan = [&](double target) {
      int64_t nt = 0;
      for (Item &it : items) {
        const f12int_ctx::BasisData &B = *batch[(size_t)it.req]->B;
        BatchPlan bp{};
        const bool fp32 = it.tier >= kTiers ? it.tier < 2 * kTiers : false;
        batch_plan(B.l[it.q[0]], B.l[it.q[1]], B.l[it.q[2]], B.l[it.q[3]], cls, it.npab, it.npcd, target, &bp,
                   fp32);   // checked at submit
        it.tier = bp.tier;
        it.nsplit = bp.nsplit;
        it.work = bp.work;
        nt += bp.nsplit;
      }
      return nt;
    };
    for (Item &it : items) it.tier = it.tier ? kTiers : 0;
    if (plan(std::min(E.task_target[cls], std::max(1e5, 2.0 * total / (kSMs * 12)))) > E.tcap)
      plan(std::max(E.task_target[cls], kTaskFlops / 8));
    // working order: by tier, then decreasing work per task (the longest
    // tasks start first)
    std::stable_sort(items.begin(), items.end(), [](const Item &x, const Item &y) {
      if (x.tier != y.tier) return x.tier < y.tier;
      return x.work > y.work;
    });
  }
  size_t at[7] = {0};
  bool first = true;
  for (;;) {
    // a pass: of every class the next quartets whose rows fit
    bool more = false;
    int large = 0;   // class of a quartet larger than the buffer, alone in its pass
    for (int cls = 1; cls <= 6 && !large; ++cls)
      if (at[cls] < all[cls].size() && all[cls][at[cls]].rows > E.rcap[grid]) large = cls;
    Item big{};
    if (large) big = all[large][at[large]];
    for (int cls = 1; cls <= 6; ++cls) {
      ClassLists &S = E.stage[b][cls];
      const std::vector<Item> &items = all[cls];
      const size_t i0 = at[cls];
      size_t i1 = i0;
      int64_t rows = 0;
      if (large) {
        if (cls == large) i1 = i0 + 1;
      } else {
        while (i1 < items.size() && rows + items[i1].rows <= E.rcap[grid]) rows += items[i1++].rows;
      }
      at[cls] = i1;
      more = more || i1 < items.size();
      const int64_t n = (int64_t)(i1 - i0);
      int64_t npq = 0, npq_gen = 0, nt = 0, row = 0, i = 0;
      for (int t = 0; t < kSlots; ++t) {
        if (t == kThinSlot) npq_gen = npq;
        S.counts[kTaskCounts + 2 * t] = nt;
        for (; i < n && items[i0 + (size_t)i].tier == t; ++i) {
          const Item &it = items[i0 + (size_t)i];
          for (int k = 0; k < 4; ++k) S.quartets[4 * i + k] = it.q[it.swap ? k ^ 2 : k];
          S.offsets[i] = it.off;
          S.qslot[i] = it.req;
          S.pq_off[i] = npq;
          S.row_off[i] = row;
          npq += it.npab * it.npcd;
          row += it.rows;
          const int16_t mark = (int16_t)(it.swap ? -it.nsplit : it.nsplit);
          for (int sp = 0; sp < it.nsplit; ++sp) S.tasks[nt++] = CTask{(int32_t)i, (int16_t)sp, mark};
        }
        S.counts[kTaskCounts + 1 + 2 * t] = nt;
      }
      S.pq_off[n] = npq;
      S.row_off[n] = row;
      S.counts[0] = n;
      S.counts[1] = npq;
      S.counts[2] = npq_gen;
      for (size_t r = 0; r < batch.size(); ++r) {
        if (!(batch[r]->mask & (1u << (cls - 1)))) continue;
        S.views[r] = pair_view(ctx, *batch[r]->B, cls, batch[r]->B->prim_screen);
        S.outs[r] = batch[r]->out;
      }
      // copy what this pass uses
      const ClassLists &D = E.dev[cls];
      cudaStream_t st = E.stream;
      const size_t ns = batch.size();
      CK(cudaMemcpyAsync(D.counts, S.counts, sizeof(int64_t) * kCounts, cudaMemcpyHostToDevice, st));
      if (n > 0) {
        CK(cudaMemcpyAsync(D.quartets, S.quartets, sizeof(int32_t) * 4 * n, cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.pq_off, S.pq_off, sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.row_off, S.row_off, sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.offsets, S.offsets, sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.qslot, S.qslot, sizeof(int32_t) * n, cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.tasks, S.tasks, sizeof(CTask) * nt, cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.views, S.views, sizeof(PairView) * ns, cudaMemcpyHostToDevice, st));
        CK(cudaMemcpyAsync(D.outs, S.outs, sizeof(double *) * ns, cudaMemcpyHostToDevice, st));
      }
    }
    *E.zstage_count[b] = first ? nzero : 0;
    cudaStream_t st = E.stream;
    CK(cudaMemcpyAsync(E.zero_count, E.zstage_count[b], sizeof(int64_t), cudaMemcpyHostToDevice, st));
    if (first && nzero > 0) {
      CK(cudaMemcpyAsync(E.zero_dst, E.zstage_dst[b], sizeof(double *) * nzero, cudaMemcpyHostToDevice, st));
      CK(cudaMemcpyAsync(E.zero_len, E.zstage_len[b], sizeof(int64_t) * nzero, cudaMemcpyHostToDevice, st));
    }
    if (large) {
      const int rc = engine_large(ctx, E, large, grid, big.swap ? big.npcd : big.npab, big.npab * big.npcd, big.rows, big.tier);
      if (rc != F12INT_OK) return rc;
      if (first && nzero > 0) k_zero_blocks<<<4 * kSMs, 128, 0, st>>>(E.zero_dst, E.zero_len, E.zero_count);
    } else {
      CK(cudaGraphLaunch(E.exec[grid], st));
    }
    first = false;
    if (!more) break;
    CK(cudaStreamSynchronize(st));   // the next pass's lists take the staging buffer
  }
  cudaStream_t st = E.stream;
  CK(cudaMemcpyAsync(E.stage_status[b], E.status, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
  CK(cudaMemsetAsync(E.status, 0, sizeof(unsigned), st));
  CK(cudaEventRecord(E.ev[b], st));
  return F12INT_OK;
}

static void engine_worker(f12int_ctx *ctx, Engine *Ep) {
  Engine &E = *Ep;
  cudaSetDevice(ctx->device);
  std::unique_lock<std::mutex> lk(E.mu);
  for (;;) {
    E.cv.wait(lk, [&] { return E.stop || !E.pending.empty(); });
    if (E.pending.empty()) break;   // stop requested and nothing left
    const int b = E.cur;
    E.cur ^= 1;
    // staging buffer b is free once the batch that used it has finished
    if (!E.inflight[b].empty()) {
      lk.unlock();
      cudaEventSynchronize(E.ev[b]);
      lk.lock();
      engine_finish_batch(E, b);
    }
    // admission: take requests while every class fits the batch limits
    std::vector<EngineReq *> batch;
    int64_t nq[7] = {0}, ni[7] = {0}, nt[7] = {0};
    while (!E.pending.empty() && (int64_t)batch.size() < E.scap) {
      EngineReq *R = E.pending.front();
      bool fits = true;
      for (int c = 1; c <= 6; ++c)
        if (nq[c] + R->quartets[c] > E.qcap || ni[c] + R->items[c] > E.icap || nt[c] + R->tasks[c] > E.tcap)
          fits = false;
      if (!batch.empty() && (!fits || R->grid != batch.front()->grid)) break;
      for (int c = 1; c <= 6; ++c) {
        nq[c] += R->quartets[c];
        ni[c] += R->items[c];
        nt[c] += R->tasks[c];
      }
      batch.push_back(R);
      E.pending.pop_front();
    }
    int rc = F12INT_OK;
    const bool grid = batch.front()->grid;
    if (E.graph_dirty[grid]) rc = engine_capture(ctx, E, grid);
    for (EngineReq *R : batch) E.tickets[R->ticket].batch = b;
    lk.unlock();
    if (rc == F12INT_OK) rc = engine_launch(ctx, E, batch, b, grid);
    lk.lock();
    for (EngineReq *R : batch) {
      if (rc == F12INT_OK) {
        E.inflight[b].push_back(R->ticket);
      } else {
        TicketState &T = E.tickets[R->ticket];
        T.done = true;
        T.rc = rc;
        T.batch = -1;
      }
      delete R;
    }
    ++E.batches;
  }
}

}  // namespace

static void engine_shutdown(f12int_ctx *ctx) {
  Engine *E = ctx->engine;
  if (!E) return;
  {
    std::lock_guard<std::mutex> lk(E->mu);
    E->stop = true;
  }
  E->cv.notify_all();
  if (E->worker.joinable()) E->worker.join();
  if (E->stream) cudaStreamSynchronize(E->stream);
  for (int c = 1; c <= 6; ++c) lists_free(E->dev[c], false);
  for (int b = 0; b < 2; ++b) {
    for (int c = 1; c <= 6; ++c) lists_free(E->stage[b][c], true);
    cudaFreeHost(E->zstage_dst[b]);
    cudaFreeHost(E->zstage_len[b]);
    cudaFreeHost(E->zstage_count[b]);
    cudaFreeHost(E->stage_status[b]);
    if (E->ev[b]) cudaEventDestroy(E->ev[b]);
  }
  void *ds[] = {E->zero_dst, E->zero_len, E->zero_count, E->status};
  for (void *p : ds)
    if (p) cudaFree(p);
  for (int c = 1; c <= 6; ++c) {
    void *cs[] = {E->keys[c], E->order[c], E->part[c], E->hist[c], E->rows_own ? E->rows[0][c] : nullptr};
    for (void *p : cs)
      if (p) cudaFree(p);
    if (E->branch[c]) cudaStreamDestroy(E->branch[c]);
    for (cudaStream_t t : E->sub[c])
      if (t) cudaStreamDestroy(t);
  }
  ctx->used -= std::min(ctx->used, E->bytes);
  for (cudaGraphExec_t x : E->exec)
    if (x) cudaGraphExecDestroy(x);
  if (E->stream) cudaStreamDestroy(E->stream);
  for (EngineReq *R : E->pending) delete R;
  delete E;
  ctx->engine = nullptr;
}

// No request queued or running.
static bool engine_idle(f12int_ctx *ctx) {
  Engine *E = ctx->engine;
  if (!E) return true;
  std::lock_guard<std::mutex> lk(E->mu);
  return E->pending.empty() &&
         f12engine::tickets_idle(E->tickets, E->inflight, [&](int b) { return cudaEventQuery(E->ev[b]) == cudaSuccess; });
}

// The captured graph holds the factor's tables by value.
static void engine_factor_changed(f12int_ctx *ctx) {
  if (ctx->engine) {
    std::lock_guard<std::mutex> lk(ctx->engine->mu);
    ctx->engine->graph_dirty[0] = ctx->engine->graph_dirty[1] = true;
  }
}

extern "C" {

int f12int_batch_limits(f12int_ctx *ctx, int64_t max_quartets, int64_t max_items) {
  if (!ctx || max_quartets < 1 || max_items < 1 || max_quartets > ((int64_t)1 << 30)) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (ctx->engine && ctx->engine->ready) return F12INT_EINVAL;   // fixed once the engine runs
  if (!ctx->engine) ctx->engine = new (std::nothrow) Engine();
  if (!ctx->engine) return F12INT_ENOMEM;
  ctx->engine->qcap = max_quartets;
  ctx->engine->icap = max_items;
  return F12INT_OK;
}

// Device memory the one-time primitive bounds of (basis, class) take at most:
// the per-primitive basis's pair data (E and F tables of every primitive
// pair), the diagonal blocks of every primitive pair and the work items of
// one call over them (the buffers of ensure_prim_bounds).
static size_t prim_bounds_bytes(const f12int_ctx *ctx, const f12int_ctx::BasisData &B, int cls) {
  std::vector<int> lp;
  for (int s = 0; s < B.nshell; ++s)
    for (int k = 0; k < B.nprim[s]; ++k) lp.push_back(B.l[s]);
  const size_t np = lp.size();
  size_t pair_data = 0, diag = 0;
  for (size_t a = 0; a < np; ++a)
    for (size_t b = 0; b <= a; ++b) {
      const size_t la = (size_t)lp[a], lb = (size_t)lp[b];
      pair_data += 2 * (6 * (la + 1) * (lb + 1) * (la + lb + 1) + 16) * sizeof(double);
      const size_t nab = (size_t)ncart((int)la) * ncart((int)lb);
      diag += nab * nab * sizeof(double) + 3 * sizeof(int64_t) + 4 * sizeof(int32_t);
    }
  const size_t npairs = np * (np + 1) / 2;
  const size_t nf = (size_t)std::max(1, ctx->tables.nfam[cls == 5 ? 3 : cls]);
  const size_t items = npairs * nf * (sizeof(int) + sizeof(unsigned) + sizeof(double) * kPartPitch);
  return pair_data + diag + items;
}

int f12int_submit(f12int_ctx *ctx, int basis_id, const f12int_request *req, uint64_t *ticket) {
  if (!ctx || !req || !ticket) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size() || !ctx->factor_ready) return F12INT_ENOTREADY;
  if (req->n_quartets < 0 || (req->n_quartets > 0 && (!req->quartets || !req->offsets || !req->out_dev)))
    return F12INT_EINVAL;
  if (req->class_mask == 0 || (req->class_mask >> 6) != 0) return F12INT_EINVAL;
  for (int c = 1; c <= 6; ++c)
    if (((req->class_mask >> (c - 1)) & 1) && !ctx->cls_ok[c]) return F12INT_EDOMAIN;
  if (req->precision != 0 && req->precision != 1) return F12INT_EINVAL;
  if (!(req->schwarz_thresh >= 0.0)) return F12INT_EINVAL;
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  const int64_t n = req->n_quartets;
  int nclass = 0;
  for (int c = 1; c <= 6; ++c) nclass += (req->class_mask >> (c - 1)) & 1;
  EngineReq *R = new (std::nothrow) EngineReq();
  if (!R) return F12INT_ENOMEM;
  R->basis = basis_id;
  R->B = &B;
  R->mask = req->class_mask;
  R->precision = req->precision;
  R->thresh = req->schwarz_thresh;
  R->out = req->out_dev;
  R->q.assign(req->quartets, req->quartets + 4 * n);
  R->off.assign(req->offsets, req->offsets + (size_t)nclass * n);
  R->grid = true;
  int64_t npq = 0;
  for (int64_t i = 0; i < n; ++i) {
    const int32_t *s = &R->q[4 * (size_t)i];
    for (int k = 0; k < 4; ++k)
      if (s[k] < 0 || s[k] >= B.nshell) {
        delete R;
        return F12INT_EINVAL;
      }
    npq += (int64_t)B.nprim[s[0]] * B.nprim[s[1]] * B.nprim[s[2]] * B.nprim[s[3]];
  }
  // one-time per (basis, class) work: primitive and shell-pair bounds
  for (int c = 1; c <= 6; ++c) {
    if (!((R->mask >> (c - 1)) & 1)) continue;
    for (int64_t i = 0; i < n; ++i) {
      const int32_t *s = &R->q[4 * (size_t)i];
      BatchPlan bp{};
      if (!batch_plan(B.l[s[0]], B.l[s[1]], B.l[s[2]], B.l[s[3]], c, (int64_t)B.nprim[s[0]] * B.nprim[s[1]],
                      (int64_t)B.nprim[s[2]] * B.nprim[s[3]], kTaskFlops / 8, &bp)) {
        delete R;
        return F12INT_EINVAL;
      }
      R->tasks[c] += bp.nsplit;
    }
    // admission by free device memory: the one-time bounds allocate, so a
    // request whose bounds would not fit in what is free now (or in the
    // context's budget) is refused before anything is allocated
    if (B.prim_screen && !B.d_qprim[c]) {
      size_t free_b = 0, total_b = 0;
      const size_t need = prim_bounds_bytes(ctx, B, c);
      if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess &&
          (need > free_b || (ctx->budget && ctx->used + need > ctx->budget))) {
        delete R;
        return F12INT_ENOMEM;
      }
    }
    int rc = ensure_prim_bounds(ctx, basis_id, c);
    if (rc == F12INT_OK && (R->thresh > 0.0 || R->precision == 1)) rc = ensure_pair_bounds(ctx, basis_id, c);
    if (rc != F12INT_OK) {
      delete R;
      return rc;
    }
    if (R->grid && !grid_view(ctx, B, c).direct()) R->grid = false;
    R->quartets[c] = n;
    R->items[c] = npq * ctx->tables.nfam[c == 5 ? 3 : c];
  }
  Engine *E = nullptr;
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (!ctx->engine) ctx->engine = new (std::nothrow) Engine();
    E = ctx->engine;
    if (!E) {
      delete R;
      return F12INT_ENOMEM;
    }
    if (!E->ready) {
      CK(cudaSetDevice(ctx->device));
      int rc = engine_init(ctx, *E);
      if (rc != F12INT_OK) {
        delete R;
        return rc;
      }
      E->worker = std::thread(engine_worker, ctx, E);
    }
  }
  for (int c = 1; c <= 6; ++c)
    if (R->quartets[c] > E->qcap || R->items[c] > E->icap || R->tasks[c] > 4 * E->qcap) {
      delete R;
      return F12INT_ENOMEM;   // larger than one batch: not admitted
    }
  {
    std::lock_guard<std::mutex> lk(E->mu);
    R->ticket = E->next_ticket++;
    *ticket = R->ticket;
    E->tickets[R->ticket] = TicketState{};
    E->pending.push_back(R);
  }
  E->cv.notify_one();
  return F12INT_OK;
}

int f12int_poll(f12int_ctx *ctx, uint64_t ticket, int64_t timeout_us, int *done) {
  if (!ctx || !done || timeout_us < 0) return F12INT_EINVAL;
  Engine *E = ctx->engine;
  if (!E) return F12INT_EINVAL;
  *done = 0;
  const auto deadline = std::chrono::steady_clock::now() + std::chrono::microseconds(timeout_us);
  for (;;) {
    {
      std::lock_guard<std::mutex> lk(E->mu);
      auto it = E->tickets.find(ticket);
      if (it == E->tickets.end()) return F12INT_EINVAL;
      if (!it->second.done && it->second.batch >= 0) {
        const int b = it->second.batch;
        bool mine = false;
        for (uint64_t t : E->inflight[b]) mine |= (t == ticket);
        if (mine && cudaEventQuery(E->ev[b]) == cudaSuccess) engine_finish_batch(*E, b);
      }
      if (it->second.done) {
        const int rc = it->second.rc;
        E->tickets.erase(it);
        *done = 1;
        return rc;
      }
    }
    if (std::chrono::steady_clock::now() >= deadline) return timeout_us > 0 ? F12INT_ETIMEOUT : F12INT_OK;
    std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
}

int f12int_batch_autotune(f12int_ctx *ctx, int basis_id, const int32_t *quartets, int64_t n, uint32_t class_mask,
                          double *report) {
  if (!ctx || !quartets || n <= 0 || class_mask == 0 || (class_mask >> 6) != 0) return F12INT_EINVAL;
  if (basis_id < 0 || basis_id >= (int)ctx->bases.size() || !ctx->factor_ready) return F12INT_ENOTREADY;
  if (!engine_idle(ctx)) return F12INT_EINVAL;
  const f12int_ctx::BasisData &B = ctx->bases[basis_id];
  std::vector<int64_t> off((size_t)n);
  int64_t tot = 0;
  for (int64_t i = 0; i < n; ++i) {
    const int32_t *s = quartets + 4 * i;
    for (int k = 0; k < 4; ++k)
      if (s[k] < 0 || s[k] >= B.nshell) return F12INT_EINVAL;
    off[i] = tot;
    tot += (int64_t)ncart(B.l[s[0]]) * ncart(B.l[s[1]]) * ncart(B.l[s[2]]) * ncart(B.l[s[3]]);
  }
  {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (!ctx->engine) ctx->engine = new (std::nothrow) Engine();
    if (!ctx->engine) return F12INT_ENOMEM;
  }
  double *out = nullptr;
  int rc = dalloc(ctx, &out, sizeof(double) * (size_t)tot);
  if (rc != F12INT_OK) return rc;
  const double targets[4] = {kTaskFlops / 8, kTaskFlops * 0.3, kTaskFlops, kTaskFlops * 4};
  const int divs[2] = {1, 2};
  // one request of class c, alone in its batch; seconds from submit to done
  auto run = [&](int c, double *sec) -> int {
    f12int_request rq{n, quartets, 1u << (c - 1), 0, 0.0, out, off.data()};
    uint64_t t = 0;
    const auto t0 = std::chrono::steady_clock::now();
    int r = f12int_submit(ctx, basis_id, &rq, &t);
    int done = 0;
    // wait until the request is done (a 100 ms wait that runs out returns
    // F12INT_ETIMEOUT with done = 0: keep waiting)
    while ((r == F12INT_OK || r == F12INT_ETIMEOUT) && !done) r = f12int_poll(ctx, t, 100000, &done);
    *sec = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return r;
  };
  for (int c = 1; c <= 6 && rc == F12INT_OK; ++c) {
    if (!((class_mask >> (c - 1)) & 1)) continue;
    double best = 1e300, bt = kTaskFlops;
    int bd = 1;
    for (double tg : targets)
      for (int dv : divs) {
        {
          std::lock_guard<std::mutex> lk(ctx->engine->mu);
          ctx->engine->task_target[c] = tg;
          ctx->engine->items_div[c] = dv;
          ctx->engine->graph_dirty[0] = ctx->engine->graph_dirty[1] = true;
        }
        double t1 = 0.0, t2 = 0.0;
        rc = run(c, &t1);   // first run after a change includes the graph capture
        if (rc == F12INT_OK) rc = run(c, &t2);
        if (rc != F12INT_OK) break;
        if (t2 < best) {
          best = t2;
          bt = tg;
          bd = dv;
        }
      }
    if (rc != F12INT_OK) break;
    {
      std::lock_guard<std::mutex> lk(ctx->engine->mu);
      ctx->engine->task_target[c] = bt;
      ctx->engine->items_div[c] = bd;
      ctx->engine->graph_dirty[0] = ctx->engine->graph_dirty[1] = true;
    }
    if (report) {
      report[3 * (c - 1)] = bt;
      report[3 * (c - 1) + 1] = bd;
      report[3 * (c - 1) + 2] = best;
    }
  }
  // the sample's output may be freed only once no batch writes it any more
  // (an error above can leave one in flight): bounded wait, else keep it
  bool idle = engine_idle(ctx);
  for (int k = 0; k < 6000 && !idle; ++k) {
    std::this_thread::sleep_for(std::chrono::milliseconds(10));
    idle = engine_idle(ctx);
  }
  if (idle) dfree(ctx, out, sizeof(double) * (size_t)tot);
  return idle ? rc : F12INT_ETIMEOUT;
}

int f12int_set_fp32_below(f12int_ctx *ctx, double bound) {
  if (!ctx || !(bound >= 0.0)) return F12INT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (!ctx->engine) ctx->engine = new (std::nothrow) Engine();
  if (!ctx->engine) return F12INT_ENOMEM;
  std::lock_guard<std::mutex> lk2(ctx->engine->mu);
  ctx->engine->fp32_below = bound;
  return F12INT_OK;
}

int f12int_batch_stats(f12int_ctx *ctx, int64_t *stats) {
  if (!ctx || !stats) return F12INT_EINVAL;
  Engine *E = ctx->engine;
  if (!E) {
    stats[0] = stats[1] = stats[2] = 0;
    return F12INT_OK;
  }
  std::lock_guard<std::mutex> lk(E->mu);
  stats[0] = E->batches;
  stats[1] = E->requests_done;
  stats[2] = (int64_t)E->pending.size();
  return F12INT_OK;
}

}  // extern "C"
