// hot.cu -- host runtime and C ABI (include/hot.h) of the GSW hologram engine.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <iterator>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/hot.h"
#include "gsw_kernels.cuh"
#include "batch_kernels.cuh"
#include "tc.h"
#include "tile.h"

static_assert(hot::kLossTraps * hot::kLossThreads >= HOT_MAX_TRAPS, "traps per thread of the loss kernel");

namespace {

thread_local char g_err[512] = "";

int fail(int code, const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return code;
}

#define HOT_CUDA(call)                                                                  \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess)                                                              \
      return fail(e_ == cudaErrorMemoryAllocation ? HOT_ENOMEM : HOT_ECUDA, "%s: %s (%s:%d)", \
                  #call, cudaGetErrorString(e_), __FILE__, __LINE__);                   \
  } while (0)

thread_local int g_refuse = 0;  // hot_test_refuse_alloc

template <typename T>
int dalloc(T **p, size_t count) {
  *p = nullptr;
  if (count == 0) return HOT_OK;
  if (g_refuse && --g_refuse == 0) return fail(HOT_ENOMEM, "cudaMalloc(%zu B): refused", count * sizeof(T));
  cudaError_t e = cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T));
  if (e != cudaSuccess) {
    *p = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? HOT_ENOMEM : HOT_ECUDA, "cudaMalloc(%zu B): %s",
                count * sizeof(T), cudaGetErrorString(e));
  }
  return HOT_OK;
}

template <typename T>
void dfree(T *&p);

// A device copy of v; nothing allocated on failure.
template <typename T>
int upload(T **p, const std::vector<T> &v) {
  const int rc = dalloc(p, v.size());
  if (rc != HOT_OK) return rc;
  const cudaError_t e = cudaMemcpy(*p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) return HOT_OK;
  dfree(*p);
  return fail(HOT_ECUDA, "copying a schedule: %s", cudaGetErrorString(e));
}

template <typename T>
void dfree(T *&p) {
  if (p) cudaFree(p);
  p = nullptr;
}

}  // namespace

struct hot_ctx {
  int W = 0, H = 0;
  int H_total = 0, y_off = 0;  // row band: rows y_off .. y_off+H-1 of a W x H_total hologram
  double pitch = 0, lam = 0, focal = 0;
  cudaStream_t st = nullptr;
  int dev = 0;
  int precision = HOT_PREC_ACCURATE;
  // work schedule of the step kernels (see hot::SubTile)
  int grid = 0, n_sub = 0;
  hot::SubTile *sub = nullptr;  // [n_sub]
  int *first = nullptr;         // [grid + 1]
  // tiling (hot_set_tiling): rows per sub-tile (pixels per thread), resident blocks per SM
  // (0: as many as fit), traps per staged chunk
  int tile_rows = hot::kRowsMax, tile_bps = 0, tile_chunk = hot::kChunk;
  int sched_bps = 0, sched_bps_max = 0;  // resident blocks per SM in the schedule; occupancy limit
  int tile_merge = 1;  // hot_set_block_merge: schedule blocks per launched block of the GSW step (1, 2, 4)
  int groups = 1;      // schedule blocks per launched block of the direct GSW step (1 or 4)
  // register-tiled kernels (tile_kernels.cuh): the separable mode, and the accurate and fast modes
  // unless hot_set_once turned them to the direct step kernels; their own schedule
  bool once_req = true;
  bool once = false;  // in effect: the state keeps unit phasors (accurate and fast, M <= hot::kOnceMaxM)
  hot::SubTile *tsub = nullptr;  // [teams][tstride] (hot::TileArgs)
  int tgrid = 0, tteam = 1, tpairs = 3, tstride = 1;
  // the unit phasors u_j = S_j/|S_j| of phi, written by the last step of a hot_gsw whose state
  // keeps them (once); valid while phi is the phases that step wrote.  The next hot_gsw's first
  // forward field then reads them (gsw_from_u) and so adds the terms an uninterrupted run adds.
  float2 *ubuf = nullptr;  // [N]
  bool u_valid = false, gsw_from_u = false;
  int shard_k = -1;                      // last launch of a sharded sequence (hot_sharded_*)
  // state
  float *phi = nullptr;  // [N]
  int M = 0;
  unsigned char *io = nullptr;  // one allocation: abc, w, Vsum (in this order: see IoBytes)
  double *abc = nullptr;                                       // [M][3]
  float *Xt = nullptr, *Yt = nullptr, *Xr = nullptr, *Yr = nullptr;  // tables
  float *Y4t = nullptr, *Y4r = nullptr;  // [4][M][ldy4] shifted row tables (hot::StepArgs::Y4)
  int ldy4 = 0;
  float2 *Xc = nullptr, *Yc = nullptr;                               // complex tables (tensor mode)
  float2 *Xb = nullptr, *Yb = nullptr;  // [M][W], [2][M][ldy4]: complex tables (separable batches)
  float2 *Xq = nullptr;   // the tile kernels' tables (hot::TileArgs)
  float4 *Yq = nullptr;
  int Mp = 0, ldp = 0;
  bool unbuilt = false;  // some of the tables were allocated since launch_build_tables last ran
  float *w = nullptr;                                          // [2][M] weights (home: w[0])
  unsigned long long *acc = nullptr;                           // [3][copies][2][M] fixed-point field sums
  long long *Vsum = nullptr;                                   // [2][M] sums of the last forward
  float *metrics = nullptr;                                    // [2], and the words of sync behind them
  int fx_shift = 0;                                            // fixed-point scale 2^fx_shift
  unsigned char *u8 = nullptr;                                 // [N] staging for host output
  bool have_fields = false;
  long long launches = 0;
  // instrumentation
  struct Rec {
    int kind;
    cudaEvent_t a, b;
  };
  bool profiling = false;
  std::vector<Rec> recs;
  std::vector<cudaEvent_t> spare;
  // CUDA graphs of whole hot_gsw(iters) launch sequences, keyed by (iters, precision)
  struct Graph {
    int iters, precision;
    bool from_u;  // the first forward field reads ubuf
    long long kernels;
    cudaGraphExec_t exec;
  };
  bool use_graphs = true;
  cudaStream_t cap = nullptr;  // capture stream (capture is not allowed on the legacy stream)
  // persistent form (one cooperative launch per hot_gsw): grid barrier state [count, gen, err]
  bool persistent = false;
  // convergence trace (hot_set_trace): e, u of the field read by each iteration of hot_gsw
  bool tracing = false;
  float *trace = nullptr;  // [trace_cap][2]
  int trace_cap = 0, trace_iters = -1;
  double wait_limit_s = 2.0;
  unsigned int *sync = nullptr;  // (behind metrics: one copy reads both)
  std::vector<Graph> graphs;
  // HOT_PREC_TENSOR: operands and launch shapes of the tensor-core iteration (built on first use)
  hot_tc::Plan *tc = nullptr;
  float2 *G = nullptr;  // [M] coefficients of hot_intensity_loss and hot_superposition (allocated on first use)
  // Pinned staging of the small transfers: what the calls send (abc and weights, coefficients), whose
  // last copy ev_in ends, then what they read back.  A copy from pageable memory stops the host for
  // the stream's work and a round trip, as a synchronisation before the buffer's release does.
  unsigned char *pin = nullptr;
  cudaEvent_t ev_in = nullptr;
};

constexpr size_t kStatusBytes = 20;  // two metrics, three words of sync

// Layout of hot_ctx::io and of the pinned staging for M traps, in bytes.
struct IoBytes {
  size_t abc, w, Vsum, end;  // io: abc [M][3] double, w [2][M] float, Vsum [2][M] int64
  size_t back;               // pin: [0, back) sent (as io's abc and w); from back on: w, Vsum, 2 metrics, 3 words
  explicit IoBytes(size_t M) : abc(0), w(24 * M), Vsum(32 * M), end(48 * M), back(32 * M) {}
  size_t read() const { return end - w; }                 // bytes of w and Vsum
  size_t pinned() const { return back + read() + 32; }
};

namespace {

bool finite_pos(double v) { return std::isfinite(v) && v > 0; }

// Modes whose kernels evaluate no pair exponential: HOT_PREC_SEPARABLE, and HOT_PREC_TENSOR for
// every launch outside the GSW loop (forward field and adjoint of given phases, superposition).
bool separable_kernels(const hot_ctx *c) {
  return c->precision == HOT_PREC_SEPARABLE || c->precision == HOT_PREC_TENSOR;
}
// The register-tiled kernels (otherwise the direct step kernels, on request: hot_set_once).
bool tile_kernels(const hot_ctx *c) { return separable_kernels(c) || c->once_req; }

// Copies of each fixed-point accumulator buffer (StepArgs::copies).  With few traps all blocks
// add into the same 2M addresses at nearly the same moment; 8 copies (block b adds into copy
// b % 8) spread those atomics.  The tile kernels read the copies; the direct kernels,
// whose registers are fully used, and the tensor-core kernels keep one.  Storage is sized for the
// largest count.
int acc_copies(const hot_ctx *c) {
  return (c->precision != HOT_PREC_TENSOR && tile_kernels(c) && c->M <= 512) ? 8 : 1;
}

size_t acc_elems(int M) { return 6 * (size_t)M * (M <= 512 ? 8 : 1); }

// Pixels of the whole hologram (all row bands): the normalisation 1/N of Eq. 1.
double n_total(const hot_ctx *c) { return (double)c->W * (double)c->H_total; }

// Fixed-point scale of the field sums: |sum| <= N (whole hologram), kept below 2^61.
int fixed_point_shift(long long n) {
  int bits = 0;
  while ((1LL << bits) < n) bits++;
  return 61 - bits;
}

void drop_graphs(hot_ctx *c) {
  for (auto &g : c->graphs) cudaGraphExecDestroy(g.exec);
  c->graphs.clear();
}

void free_traps(hot_ctx *c) {
  drop_graphs(c);
  hot_tc::plan_destroy(c->tc);
  c->tc = nullptr;
  dfree(c->io);
  c->abc = nullptr;
  c->w = nullptr;
  c->Vsum = nullptr;
  if (c->pin) cudaFreeHost(c->pin);
  c->pin = nullptr;
  dfree(c->Xt);
  dfree(c->Yt);
  dfree(c->Xr);
  dfree(c->Yr);
  dfree(c->Y4t);
  dfree(c->Y4r);
  dfree(c->Xc);
  dfree(c->Yc);
  dfree(c->Xb);
  dfree(c->Yb);
  dfree(c->Xq);
  dfree(c->Yq);
  dfree(c->acc);
  dfree(c->G);
  c->M = 0;
  c->have_fields = false;
  c->u_valid = false;
}

int check_launch(hot_ctx *c, const char *what) {
  c->launches++;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(HOT_ECUDA, "launch of %s: %s", what, cudaGetErrorString(e));
  return HOT_OK;
}

cudaEvent_t take_event(hot_ctx *c) {
  if (!c->spare.empty()) {
    cudaEvent_t e = c->spare.back();
    c->spare.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
  return e;
}

void clear_records(hot_ctx *c) {
  for (auto &r : c->recs) {
    c->spare.push_back(r.a);
    c->spare.push_back(r.b);
  }
  c->recs.clear();
}

// Brackets one kernel launch with events when profiling is on.
struct Probe {
  hot_ctx *c;
  int kind;
  cudaEvent_t a = nullptr, b = nullptr;
  Probe(hot_ctx *ctx, int k) : c(ctx), kind(k) {
    if (!c->profiling) return;
    a = take_event(c);
    b = take_event(c);
    if (a && b) cudaEventRecord(a, c->st);
  }
  ~Probe() {
    if (!a || !b) return;
    cudaEventRecord(b, c->st);
    c->recs.push_back({kind, a, b});
  }
};

// Launches kernel<<<grid, block, smem, c->st>>>(args...); with pdl, as a programmatic
// dependent of the previous kernel in the stream (its prologue may overlap that kernel).
template <typename... KArgs, typename... Args>
void launch(hot_ctx *c, void (*kernel)(KArgs...), int grid, int block, int smem, bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Launch k of a hot_gsw sequence (k = 0: forward field of the starting phases; k >= 1:
// iteration k).  Accumulators rotate over three buffers, weights over two.
hot::StepArgs make_step_args(const hot_ctx *c, int k, const float *phi, const float2 *G, float *grad) {
  const bool fast = c->precision == HOT_PREC_FAST;
  hot::StepArgs a = {};
  a.W = c->W;
  a.H = c->H;
  a.M = c->M;
  a.chunk = c->tile_chunk;
  a.sub = c->sub;
  a.first = c->first;
  a.X = fast ? c->Xr : c->Xt;
  a.Y = fast ? c->Yr : c->Yt;
  a.Y4 = fast ? c->Y4r : c->Y4t;
  a.ldy4 = c->ldy4;
  a.phi = c->phi;
  const size_t M2 = 2 * (size_t)c->M * acc_copies(c);
  a.copies = acc_copies(c);
  a.acc_in = c->acc + M2 * ((k + 2) % 3);
  a.acc_out = c->acc + M2 * (k % 3);
  a.acc_clear = c->acc + M2 * ((k + 1) % 3);
  a.w_in = c->w + (size_t)c->M * ((k + 1) & 1);
  a.w_out = c->w + (size_t)c->M * (k & 1);
  a.fx_scale = ldexpf(1.0f, c->fx_shift);
  a.inv_fx_n = (float)(1.0 / (n_total(c) * ldexp(1.0, c->fx_shift)));
  a.angle_units = fast ? 1.0f : 0.15915494309189535f;
  a.angle_eta = fast ? hot::kFastEta : 0.0f;
  if (phi) a.phi = const_cast<float *>(phi);  // read only: forward field or adjoint of given phases
  a.G = G;
  a.grad = grad;
  a.inv_n = (float)(1.0 / (n_total(c)));
  a.trace = (c->tracing && c->trace && k >= 1 && k <= c->trace_cap) ? c->trace + 2 * (k - 1) : nullptr;
  a.once_flags = 0;
  return a;
}

template <bool FAST, bool BACK, bool FWD, bool ADJ = false>
int launch_direct(hot_ctx *c, bool pdl, int k, const float *phi = nullptr, const float2 *G = nullptr,
                float *grad = nullptr) {
  const hot::StepArgs a = make_step_args(c, k, phi, G, grad);
  const int smem = hot::step_smem_bytes(c->M, BACK);
  Probe p(c, BACK && FWD ? HOT_KERNEL_STEP : FWD ? HOT_KERNEL_FORWARD : HOT_KERNEL_OTHER);
  if (BACK && FWD && !ADJ && c->groups == 4)  // the GSW step, merged: one block per SM
    launch(c, hot::gsw_step_kernel<FAST, true, true, false, 4>, c->grid / 4, hot::kThreads * 4, smem * 4, pdl, a);
  else if (BACK && FWD && !ADJ && c->groups == 2)  // two blocks per SM, two schedule blocks each
    launch(c, hot::gsw_step_kernel<FAST, true, true, false, 2>, c->grid / 2, hot::kThreads * 2, smem * 2, pdl, a);
  else
    launch(c, hot::gsw_step_kernel<FAST, BACK, FWD, ADJ>, c->grid, hot::kThreads, smem, pdl, a);
  return check_launch(c, "gsw_step_kernel");
}

// Parameters of a tile-kernel launch: launch k of a sequence (make_step_args).
hot::TileArgs make_tile_args(const hot_ctx *c, int k, const float *phi, const float2 *G, float *grad) {
  hot::TileArgs t = {};
  t.s = make_step_args(c, k, phi, G, grad);
  t.s.sub = c->tsub;
  t.stride = c->tstride;
  t.X = c->Xq;
  t.Y = c->Yq;
  t.Mp = c->Mp;
  t.ldp = c->ldp;
  t.team = c->tteam;
  t.pairs = c->tpairs;
  return t;
}

// last: the last launch of a call (with unit phasors as the state, phases are written only then).
template <bool BACK, bool FWD, bool ADJ = false>
int launch_tile(hot_ctx *c, bool pdl, int k, const float *phi = nullptr, const float2 *G = nullptr,
                float *grad = nullptr, bool last = true) {
  hot::TileArgs t = make_tile_args(c, k, phi, G, grad);
  if (c->once && FWD) {
    t.s.u = c->ubuf;
    t.s.once_flags = BACK ? hot::kOnceState | (last ? hot::kOnceLast : 0) : !phi && c->gsw_from_u ? hot::kOnceReadU : 0;
  }
  Probe p(c, BACK && FWD ? HOT_KERNEL_STEP : FWD ? HOT_KERNEL_FORWARD : HOT_KERNEL_OTHER);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c->tgrid);
  cfg.blockDim = dim3(hot::kThreads);
  cfg.stream = c->st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  hot_tile::launch(BACK, FWD, ADJ, cfg, t);
  return check_launch(c, "gsw_tile_kernel");
}

// The kernel of the context's mode: register-tiled, or the direct step kernels.
template <bool BACK, bool FWD, bool ADJ = false>
int launch_mode(hot_ctx *c, bool pdl, int k, const float *phi = nullptr, const float2 *G = nullptr,
                float *grad = nullptr, bool last = true) {
  if (tile_kernels(c)) return launch_tile<BACK, FWD, ADJ>(c, pdl, k, phi, G, grad, last);
  if (c->precision == HOT_PREC_FAST) return launch_direct<true, BACK, FWD, ADJ>(c, pdl, k, phi, G, grad);
  return launch_direct<false, BACK, FWD, ADJ>(c, pdl, k, phi, G, grad);
}

// Raises the dynamic shared-memory limit of every step-kernel variant to what M needs.
int set_step_smem(int M) {
  const int back = hot::step_smem_bytes(M, true), fwd = hot::step_smem_bytes(M, false);
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, true, true, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, true, true, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, true, true, false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, true, true, false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_persistent_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_persistent_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, back));
  return HOT_OK;
}

// The W/32 x H row segments dealt out to G blocks in equal contiguous runs (to within one
// segment), each run cut evenly into sub-tiles of at most `rows` rows; block b walks sub-tiles
// first[b] .. first[b + 1] - 1.  (The tile kernels: strips of kTileCols columns, H in row pairs.)
void cut_schedule(int W, int H, int G, int rows, std::vector<hot::SubTile> &sub, std::vector<int> &first,
                  int strip_cols = hot::kTileW) {
  const int strips = (W + strip_cols - 1) / strip_cols;
  const long long U = (long long)strips * H;
  sub.clear();
  first.assign(G + 1, 0);
  for (int b = 0; b < G; b++) {
    first[b] = (int)sub.size();
    long long s = U * b / G;
    const long long s1 = U * (b + 1) / G;
    while (s < s1) {
      const int strip = (int)(s / H), row = (int)(s % H);
      const long long run_end = std::min<long long>(s1, (long long)(strip + 1) * H);
      const int L = (int)(run_end - s);
      const int nsub = (L + rows - 1) / rows;
      for (int i = 0; i < nsub; i++) {
        const int r0 = row + (int)((long long)L * i / nsub), r1 = row + (int)((long long)L * (i + 1) / nsub);
        sub.push_back({strip * strip_cols, r0, r1 - r0, 0});
      }
      s = run_end;
    }
  }
  first[G] = (int)sub.size();
}

// Warps that share a tile of the tile kernels (hot::TileArgs::team): the cheapest by a model of a
// team's time, in units of one warp step over two traps on one row pair.  A step costs its row pairs
// + 4 (ring, column phasors, lane sums), a tile 2 per row pair + 6 (exchange of the partial
// superpositions, phasors).  Measured us per iteration with 1 / 2 / 4 / 8 warps (the model's
// choice in brackets): 256^2, M = 16 7.9 / 5.9 / 4.9 / [4.9]; 768^2, M = 8 8.3 / [8.5] / 9.4 / 12.3;
// 801 x 603, M = 37 25 / 17.3 / [15.5] / 17.4; 768^2, M = 100 56 / 39 / [32] / 35; 512^2, M = 100
// 40 / 24 / 17.4 / [15.9]; 1920 x 1152, M = 100 [103] / 98 / 101 / 107.  Up to 1024
// traps at most 128 are added in a row (FP32 rounding of S_j), above that an eighth of them.
int tile_team(int M, long long row_pairs, int sms) {
  int best = hot::kWarps;
  double best_cost = 1e300;
  for (int team = hot::kWarps; team >= 1 && M <= 128 * team; team /= 2) {
    const long long teams = 2LL * sms * (hot::kWarps / team);
    const double run = (double)((row_pairs + teams - 1) / teams), n = std::ceil(run / hot::kTilePairs);
    const double rp = std::ceil(run / n), steps = std::ceil((M + 1) / 2 / (double)team);
    const double cost = n * (steps * (rp + 4) + 2 * rp + 6);
    if (cost < best_cost) {
      best = team;
      best_cost = cost;
    }
  }
  return best;
}

// A hologram's tiles (hot::TileArgs): one wave of blocks, the strips' row pairs dealt out to the
// teams in equal runs, cut into tiles of at most hot::kTilePairs pairs.
struct TileCut {
  int grid = 0, team = 1, pairs = 3, stride = 1;
  std::vector<hot::SubTile> tiles;  // team i's are [i stride], ...; the first one's pad says how many
};

int cut_tiles(int W, int H, int M, int sms, TileCut &cut) {
  const int P = (H + 1) / 2;
  const long long U = (long long)((W + hot::kTileCols - 1) / hot::kTileCols) * P;
  cut.team = tile_team(M, U, sms);
  const int teams = hot::kWarps / cut.team;
  std::vector<hot::SubTile> sub;
  std::vector<int> first;
  int per_sm = 0;
  // two blocks per SM, or the one that fits beside very many traps' coefficients
  for (int want = 2; want >= 1; want--) {
    cut.grid = (int)std::min<long long>((long long)sms * want, (U + teams - 1) / teams);
    cut_schedule(W, P, cut.grid * teams, hot::kTilePairs, sub, first, hot::kTileCols);
    cut.pairs = 3;
    for (const hot::SubTile &t : sub) cut.pairs = std::max(cut.pairs, t.rows);
    HOT_CUDA(hot_tile::occupancy(M, cut.team, cut.pairs, &per_sm));
    if (per_sm >= want) break;
  }
  if (per_sm < 1) return fail(HOT_ECUDA, "no tile kernel for %d traps", M);
  const int n = cut.grid * teams;
  cut.stride = 1;
  for (int i = 0; i < n; i++) cut.stride = std::max(cut.stride, first[i + 1] - first[i]);
  cut.tiles.assign((size_t)n * cut.stride, hot::SubTile{0, 0, 0, 0});
  for (int i = 0; i < n; i++)
    for (int j = first[i]; j < first[i + 1]; j++) {
      hot::SubTile &t = cut.tiles[(size_t)i * cut.stride + j - first[i]] = sub[j];
      t.y0 *= 2;
      t.pad = first[i + 1] - j;
    }
  return HOT_OK;
}

// One wave of persistent blocks (SMs x resident blocks per SM: as many as fit, at most
// tile_bps); the W/32 x H row segments are dealt out in equal contiguous runs, cut into
// sub-tiles of <= tile_rows rows.  Also the tile kernels' schedule.  On failure the schedule stays as
// it was.
int build_schedule(hot_ctx *c) {
  int rc = set_step_smem(c->M);
  if (rc != HOT_OK) return rc;
  int sms = 0, per_sm = 0;
  HOT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->dev));
  // the per-iteration and the persistent kernels share the schedule (so that they compute the
  // same bits): as many blocks per SM as both can keep resident
  int per_sm_p = 0;
  {
    const int smem = hot::step_smem_bytes(c->M, true);
    HOT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hot::gsw_step_kernel<true, true, true>,
                                                           hot::kThreads, smem));
    HOT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_p, hot::gsw_persistent_kernel<true>,
                                                           hot::kThreads, smem));
    int per_sm_a = 0;
    HOT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_a, hot::gsw_persistent_kernel<false>,
                                                           hot::kThreads, smem));
    per_sm_p = std::min(per_sm_p, per_sm_a);
  }
  per_sm = std::min(per_sm, per_sm_p);
  if (per_sm < 1) per_sm = 1;
  const int bps_max = per_sm;
  if (c->tile_bps > 0 && c->tile_bps < per_sm) per_sm = c->tile_bps;
  // Merged (hot_set_block_merge), with four schedule blocks per SM the direct modes' GSW step
  // runs one block per SM holding four of them (see gsw_step_kernel), if such a block fits.
  int groups = 1;
  if (c->tile_merge > 1 && !separable_kernels(c) && per_sm == hot::kMaxGroups) {
    int per_sm_g = 0;
    const int smem = c->tile_merge * hot::step_smem_bytes(c->M, true);
    if (c->tile_merge == 4)
      HOT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_g, hot::gsw_step_kernel<true, true, true, false, 4>,
                                                             hot::kThreads * 4, smem));
    else
      HOT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_g, hot::gsw_step_kernel<true, true, true, false, 2>,
                                                             hot::kThreads * 2, smem));
    if (per_sm_g * c->tile_merge >= per_sm) groups = c->tile_merge;
  }
  const int strips = (c->W + hot::kTileW - 1) / hot::kTileW;
  const long long U = (long long)strips * c->H;
  int G = (int)std::min<long long>((long long)sms * per_sm, U);
  // whole merged blocks; rounded the same way unmerged, so that merging never changes the schedule
  // (and with it the bits of the results)
  if (!separable_kernels(c) && per_sm == hot::kMaxGroups) G = (G + hot::kMaxGroups - 1) / hot::kMaxGroups * hot::kMaxGroups;
  std::vector<hot::SubTile> sub;
  std::vector<int> first;
  cut_schedule(c->W, c->H, G, c->tile_rows, sub, first);
  const bool tile = tile_kernels(c), once = tile && !separable_kernels(c) && c->M <= hot::kOnceMaxM;
  TileCut cut;
  if (tile) rc = cut_tiles(c->W, c->H, c->M, sms, cut);
  HOT_CUDA(cudaStreamSynchronize(c->st));
  hot::SubTile *nsub = nullptr, *ntsub = nullptr;
  int *nfirst = nullptr;
  if (rc == HOT_OK) rc = upload(&nsub, sub);
  if (rc == HOT_OK) rc = upload(&nfirst, first);
  if (rc == HOT_OK && tile) rc = upload(&ntsub, cut.tiles);
  if (rc == HOT_OK && once && !c->ubuf) rc = dalloc(&c->ubuf, (size_t)c->W * c->H);
  if (rc != HOT_OK) {
    dfree(nsub);
    dfree(nfirst);
    dfree(ntsub);
    return rc;
  }
  drop_graphs(c);  // graphs hold the old schedule
  dfree(c->sub);
  dfree(c->first);
  dfree(c->tsub);
  c->sub = nsub;
  c->first = nfirst;
  c->tsub = ntsub;
  c->sched_bps_max = bps_max;
  c->sched_bps = per_sm;
  c->groups = groups;
  c->grid = G;
  c->n_sub = (int)sub.size();
  c->once = once;
  c->tgrid = tile ? cut.grid : 0;
  c->tteam = cut.team;
  c->tpairs = cut.pairs;
  c->tstride = cut.stride;
  return HOT_OK;
}

// One step-kernel launch (launch k of the sequence): weight update + back-projection and/or
// forward field.  last: the last launch of a call (with unit phasors as the state the phases are written only
// then; every other kernel writes them at each launch).
int launch_step(hot_ctx *c, bool back, bool fwd, bool pdl, int k, bool last = true) {
  if (back && fwd) return launch_mode<true, true>(c, pdl, k, nullptr, nullptr, nullptr, last);
  if (back) return launch_mode<true, false>(c, pdl, k);
  return launch_mode<false, true>(c, pdl, k);
}

// After the last launch (k = iters): Eq. 4 metrics, field sums, weights home, accumulators cleared.
// V: NULL, or the caller's device buffer for the fields (hot_field).
int launch_finalize(hot_ctx *c, bool pdl, int iters, float *V = nullptr) {
  hot::FinalizeArgs f = {};  // done = NULL: no completion stamp
  const size_t M2 = 2 * (size_t)c->M * acc_copies(c);
  f.M = c->M;
  f.copies = acc_copies(c);
  f.acc = c->acc + M2 * (iters % 3);
  f.acc_all = c->acc;
  f.w_src = c->w + (size_t)c->M * (iters & 1);
  f.w_dst = c->w;
  f.Vsum = c->Vsum;
  f.metrics = c->metrics;
  f.inv_V = 1.0 / (n_total(c) * ldexp(1.0, c->fx_shift));
  f.inv_fx_n = (float)f.inv_V;
  f.V = reinterpret_cast<float2 *>(V);
  Probe p(c, HOT_KERNEL_FINISH);
  launch(c, hot::gsw_finalize_kernel, 1, hot::kFinalizeThreads, 0, pdl, f);
  return check_launch(c, "gsw_finalize_kernel");
}

// The launch sequence of hot_gsw(iters) on c->st.
// Inside the sequence every kernel is a programmatic dependent of the one before it (except
// when profiling, where events separate the launches); the first one waits normally for
// whatever preceded hot_gsw in the stream (trap tables, phases).
// Phase tables of the context's traps (Eq. 2 split into column and row parts): the tile kernels',
// and those of the direct kernels and of the tensor mode where they are allocated.
int launch_build_tables(hot_ctx *c) {
  Probe p(c, HOT_KERNEL_OTHER);
  const hot::TileTables t = {c->W, c->H, c->H_total, c->y_off, c->M, c->Mp, c->ldp, c->abc, c->Xq, c->Yq, c->Xc, c->Yc};
  hot::tile_tables_kernel<<<dim3((c->W + (c->H + 1) / 2 + 127) / 128, c->M), 128, 0, c->st>>>(t);
  int rc = check_launch(c, "tile_tables_kernel");
  if (rc == HOT_OK && c->Y4r) {
    const long long total = (long long)c->M * (c->W + c->H);
    const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
    hot::build_tables_kernel<<<blocks, 256, 0, c->st>>>(c->W, c->H, c->H_total, c->y_off, c->M, c->abc, c->Xt, c->Yt,
                                                        c->Xr, c->Yr, c->Y4t, c->Y4r, c->ldy4);
    rc = check_launch(c, "build_tables_kernel");
  }
  if (rc == HOT_OK && c->Yb) {
    const long long total = (long long)c->M * (c->W + c->H);
    const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
    hot::batch_tables_kernel<<<blocks, 256, 0, c->st>>>(c->W, c->H, c->M, c->abc, c->Xb, c->Yb, c->ldy4);
    rc = check_launch(c, "batch_tables_kernel");
  }
  if (rc == HOT_OK && c->tc) {  // the tensor-core operands derive from the tables
    cudaError_t e = hot_tc::plan_refresh(c->tc, c->st);
    if (e != cudaSuccess) rc = fail(HOT_ECUDA, "rebuilding the tensor-core operands: %s", cudaGetErrorString(e));
    c->launches++;
  }
  if (rc == HOT_OK) c->unbuilt = false;
  return rc;
}

// Row stride of the shifted row tables: rows y0 .. y0 + 15 of copy (4 - y0 % 4) % 4 (of copy y0 % 2 of
// Yb) start 16-byte aligned.
int shifted_rows(const hot_ctx *c) { return (c->H + 18 + 3) & ~3; }

// Allocates the direct kernels' tables for M traps, once (c->unbuilt: to be built).
int alloc_direct_tables(hot_ctx *c, int M) {
  if (c->Y4r) return HOT_OK;
  c->ldy4 = shifted_rows(c);
  const size_t n4 = 4 * (size_t)M * c->ldy4;
  int rc = dalloc(&c->Xt, (size_t)M * c->W);
  if (rc == HOT_OK) rc = dalloc(&c->Xr, (size_t)M * c->W);
  if (rc == HOT_OK) rc = dalloc(&c->Yt, (size_t)M * c->H);
  if (rc == HOT_OK) rc = dalloc(&c->Yr, (size_t)M * c->H);
  if (rc == HOT_OK) rc = dalloc(&c->Y4t, n4);
  if (rc == HOT_OK) rc = dalloc(&c->Y4r, n4);
  if (rc == HOT_OK && (cudaMemsetAsync(c->Y4t, 0, sizeof(float) * n4, c->st) != cudaSuccess ||
                       cudaMemsetAsync(c->Y4r, 0, sizeof(float) * n4, c->st) != cudaSuccess))
    rc = fail(HOT_ECUDA, "clearing the shifted row tables failed");
  if (rc != HOT_OK) {
    dfree(c->Xt);
    dfree(c->Xr);
    dfree(c->Yt);
    dfree(c->Yr);
    dfree(c->Y4t);
    dfree(c->Y4r);
    return rc;
  }
  c->unbuilt = true;
  return HOT_OK;
}

// The same for the complex tables of a separable batch's member.
int alloc_batch_tables(hot_ctx *c) {
  if (c->Yb) return HOT_OK;
  c->ldy4 = shifted_rows(c);
  const size_t n2 = 2 * (size_t)c->M * c->ldy4;
  int rc = dalloc(&c->Xb, (size_t)c->M * c->W);
  if (rc == HOT_OK) rc = dalloc(&c->Yb, n2);
  if (rc == HOT_OK && cudaMemsetAsync(c->Yb, 0, sizeof(float2) * n2, c->st) != cudaSuccess)
    rc = fail(HOT_ECUDA, "clearing the shifted complex row table failed");
  if (rc != HOT_OK) {
    dfree(c->Xb);
    dfree(c->Yb);
    return rc;
  }
  c->unbuilt = true;
  return HOT_OK;
}

// Allocates the tables that only the direct kernels or only the tensor mode read, once the context
// is in such a mode.
int alloc_mode_tables(hot_ctx *c, int M) {
  int rc = HOT_OK;
  if (!tile_kernels(c)) rc = alloc_direct_tables(c, M);
  if (rc == HOT_OK && c->precision == HOT_PREC_TENSOR && !c->Yc) {
    rc = dalloc(&c->Xc, (size_t)M * c->W);
    if (rc == HOT_OK) rc = dalloc(&c->Yc, (size_t)M * c->H);
    if (rc != HOT_OK) {
      dfree(c->Xc);
      return rc;
    }
    c->unbuilt = true;
  }
  return rc;
}

// Brings the context into a mode: its tables, its schedule (resched).  On failure the context stays in the
// mode it was in; tables that it has by then are kept.
int enter_mode(hot_ctx *c, int precision, bool once_req, bool resched) {
  const int precision0 = c->precision;
  const bool once_req0 = c->once_req;
  c->precision = precision;
  c->once_req = once_req;
  int rc = HOT_OK;
  if (c->M) {
    rc = alloc_mode_tables(c, c->M);
    if (rc == HOT_OK && c->unbuilt) rc = launch_build_tables(c);
    if (rc == HOT_OK && resched) rc = build_schedule(c);
  }
  if (rc != HOT_OK) {
    c->precision = precision0;
    c->once_req = once_req0;
    return rc;
  }
  c->u_valid = false;
  return HOT_OK;
}

// The tensor-core plan of the context's traps (HOT_PREC_TENSOR), built on first use.
int ensure_tc_plan(hot_ctx *c) {
  if (c->tc) return HOT_OK;
  const char *what = "";
  cudaError_t e = hot_tc::plan_create(&c->tc, c->W, c->H, c->M, c->Xc, c->Yc, c->st, &what);
  if (e != cudaSuccess)
    return fail(e == cudaErrorMemoryAllocation ? HOT_ENOMEM : HOT_ECUDA, "%s: %s", what, cudaGetErrorString(e));
  c->launches++;
  return HOT_OK;
}

hot_tc::Step tc_step(hot_ctx *c, int k) {
  const hot::StepArgs a = make_step_args(c, k, nullptr, nullptr, nullptr);
  hot_tc::Step s;
  s.M = c->M;
  s.acc_in = a.acc_in;
  s.acc_out = a.acc_out;
  s.acc_clear = a.acc_clear;
  s.w_in = a.w_in;
  s.w_out = a.w_out;
  s.phi = c->phi;
  s.trace = a.trace;
  s.fx_scale = a.fx_scale;
  s.inv_fx_n = a.inv_fx_n;
  s.err = reinterpret_cast<int *>(c->sync + 2);
  s.limit_ns = (long long)(c->wait_limit_s * 1e9);
  return s;
}

// Launch k of the tensor-core sequence: k = 0 the forward field of the phases, k >= 1 iteration k.
int launch_tc(hot_ctx *c, bool pdl, int k) {
  Probe p(c, k ? HOT_KERNEL_STEP : HOT_KERNEL_FORWARD);
  int kernels = 0;
  const bool chain = !c->profiling;
  const cudaError_t e = k ? hot_tc::launch_iteration(c->tc, tc_step(c, k), c->st, pdl, chain, &kernels)
                          : hot_tc::launch_forward(c->tc, tc_step(c, k), c->st, pdl, chain, &kernels);
  c->launches += kernels;
  if (e != cudaSuccess) return fail(HOT_ECUDA, "tensor-core launch %d: %s", k, cudaGetErrorString(e));
  return HOT_OK;
}

// The whole sequence of enqueue_gsw's step launches as one cooperative launch (all blocks
// resident; the grid is one wave by construction of the schedule).
int launch_persistent(hot_ctx *c, int iters) {
  const hot::GridSync sync = {c->sync, reinterpret_cast<int *>(c->sync + 2), (long long)(c->wait_limit_s * 1e9)};
  float *const trace = c->tracing ? c->trace : nullptr;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(hot::kThreads);
  cfg.stream = c->st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  HOT_CUDA(cudaMemsetAsync(c->sync, 0, sizeof(unsigned int), c->st));  // arrival count
  Probe probe(c, HOT_KERNEL_STEP);
  if (tile_kernels(c)) {
    hot::TilePersistArgs p = {};
    for (int j = 0; j < 6; j++) {
      p.step[j] = make_tile_args(c, j, nullptr, nullptr, nullptr);
      if (c->once) p.step[j].s.u = c->ubuf;
      p.step[j].s.once_flags = (c->once ? hot::kOnceState : 0) | (c->gsw_from_u ? hot::kOnceReadU : 0);
    }
    p.iters = iters;
    p.sync = sync;
    p.trace = trace;
    cfg.gridDim = dim3(c->tgrid);
    hot_tile::launch_persistent(cfg, p);
    return check_launch(c, "gsw_tile_persistent_kernel");
  }
  hot::PersistArgs p = {};
  for (int j = 0; j < 6; j++) p.step[j] = make_step_args(c, j, nullptr, nullptr, nullptr);
  p.iters = iters;
  p.trace = trace;
  p.sync = sync;
  cfg.gridDim = dim3(c->grid);
  cfg.dynamicSmemBytes = hot::step_smem_bytes(c->M, true);
  if (c->precision == HOT_PREC_FAST)
    cudaLaunchKernelEx(&cfg, hot::gsw_persistent_kernel<true>, p);
  else
    cudaLaunchKernelEx(&cfg, hot::gsw_persistent_kernel<false>, p);
  return check_launch(c, "gsw_persistent_kernel");
}

// After a bounded wait ran out: the accumulators and the barrier are reset; the phases are undefined.
int wait_ran_out(hot_ctx *c, const char *who) {
  HOT_CUDA(cudaMemsetAsync(c->sync, 0, 3 * sizeof(unsigned int), c->st));
  if (c->M) HOT_CUDA(cudaMemsetAsync(c->acc, 0, sizeof(unsigned long long) * acc_elems(c->M), c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  c->have_fields = false;
  c->u_valid = false;
  return fail(HOT_ETIMEOUT, "%s: a bounded device-side wait ran out (limit %.3g s)", who, c->wait_limit_s);
}

// Reads the barrier's error flag (synchronises): HOT_ETIMEOUT after a wait ran out.
int check_wait_error(hot_ctx *c, const char *who) {
  unsigned int st[3] = {0, 0, 0};  // [2]: error flag of the bounded waits
  HOT_CUDA(cudaMemcpyAsync(st, c->sync, sizeof st, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  return st[2] ? wait_ran_out(c, who) : HOT_OK;
}

// What read_back leaves in the pinned staging.
const float *read_w(const hot_ctx *c) { return reinterpret_cast<const float *>(c->pin + IoBytes(c->M).back); }
const long long *read_sums(const hot_ctx *c) {
  const IoBytes b(c->M);
  return reinterpret_cast<const long long *>(c->pin + b.back + b.Vsum - b.w);
}
const float *read_metrics(const hot_ctx *c) {
  const IoBytes b(c->M);
  return reinterpret_cast<const float *>(c->pin + b.back + b.read());
}

// Brings the metrics with the barrier's words behind them, and weights and field sums (fields), to the
// pinned staging with one synchronisation; HOT_ETIMEOUT after a bounded wait ran out.  The error flag is
// always looked at: which launches with bounded waits ran since the last look is not known here (replays
// of a captured call, batches on a stream of their own).
int read_back(hot_ctx *c, const char *who, bool fields) {
  const IoBytes b(c->M);
  unsigned char *const back = c->pin + b.back;
  if (fields) HOT_CUDA(cudaMemcpyAsync(back, c->io + b.w, b.read(), cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaMemcpyAsync(back + b.read(), c->metrics, kStatusBytes, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  return reinterpret_cast<const unsigned int *>(back + b.read())[4] ? wait_ran_out(c, who) : HOT_OK;
}

// Waits until the last copy out of the pinned staging is done, so that it can be filled again.  A
// stream under capture is refused: a replay would send what the staging holds by then.
int staging_free(hot_ctx *c, const char *who) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  HOT_CUDA(cudaStreamIsCapturing(c->st, &st));
  if (st != cudaStreamCaptureStatusNone) return fail(HOT_ECUDA, "%s: the stream is being captured", who);
  HOT_CUDA(cudaEventSynchronize(c->ev_in));
  return HOT_OK;
}

// e and u to the caller's non-NULL outputs (synchronises); nothing when both are NULL.
int return_metrics(hot_ctx *c, const char *who, double *eff_out, double *unif_out) {
  if (!eff_out && !unif_out) return HOT_OK;
  const int rc = read_back(c, who, false);
  if (rc != HOT_OK) return rc;
  if (eff_out) *eff_out = read_metrics(c)[0];
  if (unif_out) *unif_out = read_metrics(c)[1];
  return HOT_OK;
}

// Queues the copy of the first `bytes` of the staging, from byte `from`, to dst.
int send_staged(hot_ctx *c, void *dst, size_t from, size_t bytes) {
  HOT_CUDA(cudaMemcpyAsync(dst, c->pin + from, bytes, cudaMemcpyHostToDevice, c->st));
  HOT_CUDA(cudaEventRecord(c->ev_in, c->st));
  return HOT_OK;
}

int enqueue_gsw(hot_ctx *c, int iters) {
  if (c->persistent) {
    int rc = launch_persistent(c, iters);
    if (rc == HOT_OK) rc = launch_finalize(c, false, iters);
    return rc;
  }
  const bool pdl = !c->profiling;
  if (c->precision == HOT_PREC_TENSOR) {
    int rc = launch_tc(c, false, 0);
    for (int k = 1; k <= iters && rc == HOT_OK; k++) rc = launch_tc(c, pdl, k);
    if (rc == HOT_OK) rc = launch_finalize(c, pdl, iters);
    return rc;
  }
  int rc = launch_step(c, false, true, false, 0);       // V^1 = F(phi^0)
  for (int k = 1; k <= iters && rc == HOT_OK; k++)      // w^k, c^k from V^k; phi^k; V^{k+1} = F(phi^k)
    rc = launch_step(c, true, true, pdl, k, k == iters);
  if (rc == HOT_OK) rc = launch_finalize(c, pdl, iters);  // e, u of V^{iters+1}
  return rc;
}

// Replays (capturing on first use) the graph of enqueue_gsw(iters).
int launch_gsw_graph(hot_ctx *c, int iters) {
  for (auto &g : c->graphs)
    if (g.iters == iters && g.precision == c->precision && g.from_u == c->gsw_from_u) {
      HOT_CUDA(cudaGraphLaunch(g.exec, c->st));
      c->launches += g.kernels;
      return HOT_OK;
    }
  if (!c->cap) HOT_CUDA(cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking));
  if (c->graphs.size() >= 8) {
    cudaGraphExecDestroy(c->graphs.front().exec);
    c->graphs.erase(c->graphs.begin());
  }
  cudaStream_t user = c->st;
  const long long before = c->launches;
  HOT_CUDA(cudaStreamBeginCapture(c->cap, cudaStreamCaptureModeThreadLocal));
  c->st = c->cap;
  int rc = enqueue_gsw(c, iters);
  c->st = user;
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(c->cap, &graph);
  const long long kernels = c->launches - before;
  c->launches = before;
  if (rc != HOT_OK) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return fail(HOT_ECUDA, "hot_gsw: graph capture: %s", cudaGetErrorString(e));
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return fail(HOT_ECUDA, "hot_gsw: graph instantiation: %s", cudaGetErrorString(e));
  c->graphs.push_back({iters, c->precision, c->gsw_from_u, kernels, exec});
  HOT_CUDA(cudaGraphLaunch(exec, c->st));
  c->launches += kernels;
  return HOT_OK;
}

}  // namespace

extern "C" {

const char *hot_last_error(void) { return g_err; }

// Test seam, not part of the interface: the calling thread's nth device allocation from now on is refused
// with HOT_ENOMEM, once (0: none).
void hot_test_refuse_alloc(int nth) { g_refuse = nth; }

int hot_create(hot_ctx **out, int width, int height, double pitch_m, double wavelength_m,
               double focal_m, void *cuda_stream) {
  g_err[0] = 0;
  if (!out) return fail(HOT_EINVAL, "hot_create: out is NULL");
  *out = nullptr;
  if (width < 1 || height < 1 || (long long)width * height >= (1LL << 31))
    return fail(HOT_EINVAL, "hot_create: invalid size %d x %d", width, height);
  if (!finite_pos(pitch_m) || !finite_pos(wavelength_m) || !finite_pos(focal_m))
    return fail(HOT_EINVAL, "hot_create: pitch, wavelength and focal length must be finite and > 0");
  hot_ctx *c = new (std::nothrow) hot_ctx;
  if (!c) return fail(HOT_ENOMEM, "hot_create: out of host memory");
  c->W = width;
  c->H = height;
  c->pitch = pitch_m;
  c->lam = wavelength_m;
  c->focal = focal_m;
  c->st = static_cast<cudaStream_t>(cuda_stream);
  c->H_total = height;
  c->fx_shift = fixed_point_shift((long long)width * height);
  int rc = HOT_OK;
  cudaError_t e = cudaGetDevice(&c->dev);
  if (e != cudaSuccess) rc = fail(HOT_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  const size_t N = (size_t)width * height;
  if (rc == HOT_OK) rc = dalloc(&c->phi, N);
  if (rc == HOT_OK) rc = dalloc(&c->metrics, kStatusBytes / sizeof(float));
  if (rc == HOT_OK) c->sync = reinterpret_cast<unsigned int *>(c->metrics + 2);
  if (rc == HOT_OK && cudaMemsetAsync(c->sync, 0, 3 * sizeof(unsigned int), c->st) != cudaSuccess)
    rc = fail(HOT_ECUDA, "hot_create: clearing the barrier state failed");
  if (rc == HOT_OK) {
    e = cudaMemsetAsync(c->phi, 0, N * sizeof(float), c->st);
    if (e != cudaSuccess) rc = fail(HOT_ECUDA, "hot_create: %s", cudaGetErrorString(e));
  }
  if (rc != HOT_OK) {
    hot_destroy(c);
    return rc;
  }
  *out = c;
  return HOT_OK;
}

void hot_destroy(hot_ctx *c) {
  if (!c) return;
  if (c->phi || c->M) cudaStreamSynchronize(c->st);
  drop_graphs(c);
  if (c->cap) cudaStreamDestroy(c->cap);
  clear_records(c);
  for (cudaEvent_t e : c->spare) cudaEventDestroy(e);
  c->spare.clear();
  free_traps(c);
  dfree(c->phi);
  dfree(c->sub);
  dfree(c->first);
  dfree(c->tsub);
  dfree(c->ubuf);
  dfree(c->metrics);
  dfree(c->u8);
  dfree(c->trace);
  if (c->ev_in) cudaEventDestroy(c->ev_in);
  delete c;
}

int hot_set_traps(hot_ctx *c, int M, const double *xyz_m, const double *w0) {
  if (!c) return fail(HOT_EINVAL, "hot_set_traps: NULL context");
  if (M < 1 || M > HOT_MAX_TRAPS) return fail(HOT_EINVAL, "hot_set_traps: M = %d not in [1, %d]", M, HOT_MAX_TRAPS);
  if (!xyz_m) return fail(HOT_EINVAL, "hot_set_traps: xyz is NULL");
  for (int i = 0; i < 3 * M; i++)
    if (!std::isfinite(xyz_m[i])) return fail(HOT_EINVAL, "hot_set_traps: coordinate %d not finite", i);
  if (w0)
    for (int m = 0; m < M; m++)
      if (!finite_pos(w0[m])) return fail(HOT_EINVAL, "hot_set_traps: weight %d not finite and > 0", m);
  int rc = HOT_OK;
  if (M != c->M) {
    cudaStreamSynchronize(c->st);
    free_traps(c);
    c->M = M;
    rc = build_schedule(c);
    c->M = 0;
    if (rc != HOT_OK) return rc;
    const IoBytes io((size_t)M);
    rc = dalloc(&c->io, io.end);
    if (rc == HOT_OK) {
      c->abc = reinterpret_cast<double *>(c->io + io.abc);
      c->w = reinterpret_cast<float *>(c->io + io.w);
      c->Vsum = reinterpret_cast<long long *>(c->io + io.Vsum);
      if (cudaHostAlloc(reinterpret_cast<void **>(&c->pin), io.pinned(), cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        c->pin = nullptr;
        rc = fail(HOT_ENOMEM, "hot_set_traps: no pinned memory");
      }
    }
    if (rc == HOT_OK && !c->ev_in && cudaEventCreateWithFlags(&c->ev_in, cudaEventDisableTiming) != cudaSuccess) {
      c->ev_in = nullptr;
      rc = fail(HOT_ECUDA, "hot_set_traps: cudaEventCreate failed");
    }
    if (rc == HOT_OK) rc = alloc_mode_tables(c, M);
    // the tile kernels' tables, zero past the image: whole strips, whole trap pairs, row pairs read
    // kTilePairs at a time
    const size_t nx = (size_t)((c->W + hot::kTileCols - 1) / hot::kTileCols) * hot::kTileCols;
    c->Mp = (M + 1) & ~1;
    c->ldp = (c->H + 1) / 2 + hot::kTilePairs;
    if (rc == HOT_OK) rc = dalloc(&c->Xq, c->Mp * nx);
    if (rc == HOT_OK) rc = dalloc(&c->Yq, (size_t)c->Mp * c->ldp);
    if (rc == HOT_OK && (cudaMemsetAsync(c->Xq, 0, sizeof(float2) * c->Mp * nx, c->st) != cudaSuccess ||
                         cudaMemsetAsync(c->Yq, 0, sizeof(float4) * (size_t)c->Mp * c->ldp, c->st) != cudaSuccess))
      rc = fail(HOT_ECUDA, "hot_set_traps: clearing the tile kernels' tables failed");
    if (rc == HOT_OK) rc = dalloc(&c->acc, acc_elems(M));
    if (rc == HOT_OK && cudaMemsetAsync(c->acc, 0, sizeof(unsigned long long) * acc_elems(M), c->st) != cudaSuccess)
      rc = fail(HOT_ECUDA, "hot_set_traps: clearing the field accumulators failed");
    if (rc != HOT_OK) {
      free_traps(c);
      return rc;
    }
    c->M = M;
  }
  rc = staging_free(c, "hot_set_traps");
  if (rc != HOT_OK) return rc;
  // Eq. 2 in turns per pixel index: a = x p/(lambda f), b = y p/(lambda f), c = z p^2/(2 lambda f^2)
  double *const abc = reinterpret_cast<double *>(c->pin);
  float *const wh = reinterpret_cast<float *>(c->pin + IoBytes(M).w);
  const double lin = c->pitch / (c->lam * c->focal);
  const double quad = c->pitch * c->pitch / (2.0 * c->lam * c->focal * c->focal);
  for (int m = 0; m < M; m++) {
    abc[3 * m] = xyz_m[3 * m] * lin;
    abc[3 * m + 1] = xyz_m[3 * m + 1] * lin;
    abc[3 * m + 2] = xyz_m[3 * m + 2] * quad;
    wh[m] = w0 ? (float)w0[m] : 1.0f;
  }
  rc = send_staged(c, c->io, 0, IoBytes(M).w + sizeof(float) * M);
  if (rc != HOT_OK) return rc;
  c->have_fields = false;
  c->u_valid = false;
  return launch_build_tables(c);
}

int hot_set_weights(hot_ctx *c, const double *w) {
  if (!c || !w) return fail(HOT_EINVAL, "hot_set_weights: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_set_weights: no traps set");
  for (int m = 0; m < c->M; m++)
    if (!finite_pos(w[m])) return fail(HOT_EINVAL, "hot_set_weights: weight %d not finite and > 0", m);
  const int rc = staging_free(c, "hot_set_weights");
  if (rc != HOT_OK) return rc;
  const size_t at = IoBytes(c->M).w;
  float *const wf = reinterpret_cast<float *>(c->pin + at);
  for (int m = 0; m < c->M; m++) wf[m] = (float)w[m];
  return send_staged(c, c->w, at, sizeof(float) * c->M);
}

int hot_set_phase(hot_ctx *c, const float *phi, int on_device) {
  if (!c || !phi) return fail(HOT_EINVAL, "hot_set_phase: NULL argument");
  const size_t bytes = sizeof(float) * (size_t)c->W * c->H;
  if (on_device) {
    HOT_CUDA(cudaMemcpyAsync(c->phi, phi, bytes, cudaMemcpyDeviceToDevice, c->st));
  } else {
    HOT_CUDA(cudaMemcpyAsync(c->phi, phi, bytes, cudaMemcpyHostToDevice, c->st));
    HOT_CUDA(cudaStreamSynchronize(c->st));
  }
  c->have_fields = false;
  c->u_valid = false;
  return HOT_OK;
}

int hot_set_precision(hot_ctx *c, int precision) {
  if (!c) return fail(HOT_EINVAL, "hot_set_precision: NULL context");
  if (precision != HOT_PREC_ACCURATE && precision != HOT_PREC_FAST && precision != HOT_PREC_SEPARABLE &&
      precision != HOT_PREC_TENSOR)
    return fail(HOT_EINVAL, "hot_set_precision: unknown mode %d", precision);
  const bool was_sep = separable_kernels(c);
  const bool resched = was_sep != (precision == HOT_PREC_SEPARABLE || precision == HOT_PREC_TENSOR);
  const bool copies_change = (precision == HOT_PREC_TENSOR) != (c->precision == HOT_PREC_TENSOR);
  if (resched || copies_change) HOT_CUDA(cudaStreamSynchronize(c->st));
  return enter_mode(c, precision, c->once_req, resched);  // (the kernels' occupancies differ)
}

int hot_gsw(hot_ctx *c, int iters, double *eff_out, double *unif_out) {
  if (!c) return fail(HOT_EINVAL, "hot_gsw: NULL context");
  if (iters < 0) return fail(HOT_EINVAL, "hot_gsw: iters = %d < 0", iters);
  if (!c->M) return fail(HOT_ESTATE, "hot_gsw: no traps set");
  if (c->precision == HOT_PREC_TENSOR) {
    if (c->persistent) return fail(HOT_EINVAL, "hot_gsw: the persistent form has no tensor-core variant");
    const int rc = ensure_tc_plan(c);
    if (rc != HOT_OK) return rc;
  }
  if (c->tracing) {
    if (iters > c->trace_cap) {  // the launches' trace slots change: recapture the graphs
      HOT_CUDA(cudaStreamSynchronize(c->st));
      drop_graphs(c);
      dfree(c->trace);
      c->trace_cap = 0;
      const int cap = std::max(iters, 64);
      const int rc = dalloc(&c->trace, 2 * (size_t)cap);
      if (rc != HOT_OK) return rc;
      c->trace_cap = cap;
    }
    c->trace_iters = iters;
  }
  const bool had_u = c->u_valid;
  c->gsw_from_u = c->u_valid && c->once;
  c->u_valid = false;
  const int rc = (c->use_graphs && !c->profiling && !c->persistent) ? launch_gsw_graph(c, iters) : enqueue_gsw(c, iters);
  c->gsw_from_u = false;
  if (rc != HOT_OK) return rc;
  // where the state keeps unit phasors, the last step left u_j of the phases it wrote in ubuf
  c->u_valid = iters > 0 ? c->once : had_u;
  c->have_fields = true;
  return return_metrics(c, "hot_gsw", eff_out, unif_out);
}

int hot_phase_out(hot_ctx *c, void *dst, int fmt, int on_device) {
  if (!c || !dst) return fail(HOT_EINVAL, "hot_phase_out: NULL argument");
  if (fmt != HOT_FMT_F32 && fmt != HOT_FMT_U8) return fail(HOT_EINVAL, "hot_phase_out: unknown format %d", fmt);
  const size_t N = (size_t)c->W * c->H;
  if (fmt == HOT_FMT_F32) {
    HOT_CUDA(cudaMemcpyAsync(dst, c->phi, N * sizeof(float),
                             on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c->st));
  } else {
    unsigned char *g = static_cast<unsigned char *>(dst);
    if (!on_device) {
      if (!c->u8) {
        int rc = dalloc(&c->u8, N);
        if (rc != HOT_OK) return rc;
      }
      g = c->u8;
    }
    const int blocks = (int)(((long long)N + 255) / 256 < 8192 ? ((long long)N + 255) / 256 : 8192);
    int rc;
    {
      Probe p(c, HOT_KERNEL_OTHER);
      hot::quantize_kernel<<<blocks, 256, 0, c->st>>>(c->phi, g, (long long)N);
      rc = check_launch(c, "quantize_kernel");
    }
    if (rc != HOT_OK) return rc;
    if (!on_device) HOT_CUDA(cudaMemcpyAsync(dst, c->u8, N, cudaMemcpyDeviceToHost, c->st));
  }
  if (!on_device) HOT_CUDA(cudaStreamSynchronize(c->st));
  return HOT_OK;
}

int hot_get_fields(hot_ctx *c, double *V, double *w) {
  if (!c) return fail(HOT_EINVAL, "hot_get_fields: NULL context");
  if (!c->M) return fail(HOT_ESTATE, "hot_get_fields: no traps set");
  if (V && !c->have_fields) return fail(HOT_ESTATE, "hot_get_fields: no forward evaluation since the last change");
  const int rc = read_back(c, "hot_get_fields", V || w);
  if (rc != HOT_OK) return rc;
  const long long *const vs = read_sums(c);
  const float *const wf = read_w(c);
  const double inv = 1.0 / (n_total(c) * ldexp(1.0, c->fx_shift));
  for (int m = 0; V && m < c->M; m++) {  // fixed-point sums -> V_m
    V[2 * m] = (double)vs[m] * inv;
    V[2 * m + 1] = (double)vs[c->M + m] * inv;
  }
  for (int m = 0; w && m < c->M; m++) w[m] = wf[m];
  return HOT_OK;
}

int hot_field(hot_ctx *c, const float *phi, float *V) {
  if (!c || !phi || !V) return fail(HOT_EINVAL, "hot_field: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_field: no traps set");
  // the finalize kernel (w stays in w[0]; accumulators cleared) follows as a programmatic dependent
  int rc = launch_mode<false, true>(c, false, 0, phi);
  if (rc == HOT_OK) rc = launch_finalize(c, !c->profiling, 0, V);
  if (rc == HOT_OK) c->have_fields = true;
  return rc;
}

int hot_superposition(hot_ctx *c, const double *coef) {
  if (!c || !coef) return fail(HOT_EINVAL, "hot_superposition: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_superposition: no traps set");
  for (int i = 0; i < 2 * c->M; i++)
    if (!std::isfinite(coef[i])) return fail(HOT_EINVAL, "hot_superposition: coefficient %d not finite", i / 2);
  int rc = c->G ? HOT_OK : dalloc(&c->G, c->M);
  if (rc == HOT_OK) rc = staging_free(c, "hot_superposition");
  if (rc != HOT_OK) return rc;
  float *const cf = reinterpret_cast<float *>(c->pin);
  for (int i = 0; i < 2 * c->M; i++) cf[i] = (float)coef[i];
  rc = send_staged(c, c->G, 0, 2 * sizeof(float) * c->M);
  if (rc == HOT_OK) rc = launch_mode<true, false>(c, false, 0, nullptr, c->G);
  c->have_fields = false;
  c->u_valid = false;
  return rc;
}

int hot_field_adjoint(hot_ctx *c, const float *phi, const float *G, float *grad) {
  if (!c || !phi || !G || !grad) return fail(HOT_EINVAL, "hot_field_adjoint: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_field_adjoint: no traps set");
  const float2 *g = reinterpret_cast<const float2 *>(G);
  return launch_mode<true, false, true>(c, false, 0, phi, g, grad);
}

int hot_intensity_loss(hot_ctx *c, const float *phi, double beta, float *loss, float *grad) {
  if (!c || !phi || !loss) return fail(HOT_EINVAL, "hot_intensity_loss: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_intensity_loss: no traps set");
  if (!std::isfinite(beta)) return fail(HOT_EINVAL, "hot_intensity_loss: beta not finite");
  if (!c->G) {
    const int rc = dalloc(&c->G, c->M);
    if (rc != HOT_OK) return rc;
  }
  int rc = launch_mode<false, true>(c, false, 0, phi);  // sums of V = F(phi) in accumulator 0
  if (rc != HOT_OK) return rc;
  hot::LossArgs a = {};
  a.M = c->M;
  a.copies = acc_copies(c);
  a.acc = c->acc;
  a.acc_all = c->acc;
  a.Vsum = c->Vsum;
  a.metrics = c->metrics;
  a.inv_fx_n = 1.0 / (n_total(c) * ldexp(1.0, c->fx_shift));
  a.beta = beta;
  a.G = c->G;
  a.loss = loss;
  {
    Probe p(c, HOT_KERNEL_FINISH);
    launch(c, hot::intensity_loss_kernel, 1, hot::kLossThreads, 0, !c->profiling, a);
  }
  rc = check_launch(c, "intensity_loss_kernel");
  if (rc != HOT_OK) return rc;
  c->have_fields = true;
  if (!grad) return HOT_OK;
  return launch_mode<true, false, true>(c, !c->profiling, 0, phi, c->G, grad);
}

int hot_set_band(hot_ctx *c, int total_height, int y0) {
  if (!c) return fail(HOT_EINVAL, "hot_set_band: NULL context");
  if (total_height < c->H || y0 < 0 || y0 > total_height - c->H || (long long)c->W * total_height >= (1LL << 31))
    return fail(HOT_EINVAL, "hot_set_band: rows %d .. %d not inside a hologram of %d rows", y0, y0 + c->H - 1,
                total_height);
  HOT_CUDA(cudaStreamSynchronize(c->st));
  drop_graphs(c);
  c->H_total = total_height;
  c->y_off = y0;
  c->fx_shift = fixed_point_shift((long long)c->W * total_height);
  c->have_fields = false;
  c->u_valid = false;
  c->shard_k = -1;
  return c->M ? launch_build_tables(c) : HOT_OK;
}

int hot_sharded_begin(hot_ctx *c) {
  if (!c) return fail(HOT_EINVAL, "hot_sharded_begin: NULL context");
  if (!c->M) return fail(HOT_ESTATE, "hot_sharded_begin: no traps set");
  c->shard_k = -1;
  c->have_fields = false;
  c->u_valid = false;
  int rc = HOT_OK;
  if (c->precision == HOT_PREC_TENSOR) {
    rc = ensure_tc_plan(c);
    if (rc == HOT_OK) rc = launch_tc(c, false, 0);
  } else {
    rc = launch_step(c, false, true, false, 0);
  }
  if (rc == HOT_OK) c->shard_k = 0;
  return rc;
}

int hot_sharded_step(hot_ctx *c, int k) {
  if (!c) return fail(HOT_EINVAL, "hot_sharded_step: NULL context");
  if (c->shard_k < 0 || k != c->shard_k + 1)
    return fail(HOT_ESTATE, "hot_sharded_step: launch %d does not follow launch %d", k, c->shard_k);
  const int rc = c->precision == HOT_PREC_TENSOR ? launch_tc(c, false, k) : launch_step(c, true, true, false, k);
  if (rc == HOT_OK) c->shard_k = k;
  return rc;
}

int hot_sharded_sums(hot_ctx *c, int k, void **sums_dev, int *count) {
  if (!c || !sums_dev || !count) return fail(HOT_EINVAL, "hot_sharded_sums: NULL argument");
  if (c->shard_k < 0 || k != c->shard_k)
    return fail(HOT_ESTATE, "hot_sharded_sums: launch %d is not the last one (%d)", k, c->shard_k);
  const size_t n = 2 * (size_t)c->M * acc_copies(c);
  *sums_dev = c->acc + n * (k % 3);
  *count = (int)n;
  return HOT_OK;
}

int hot_sharded_end(hot_ctx *c, int iters, double *eff_out, double *unif_out) {
  if (!c) return fail(HOT_EINVAL, "hot_sharded_end: NULL context");
  if (c->shard_k < 0 || iters != c->shard_k)
    return fail(HOT_ESTATE, "hot_sharded_end: iters = %d, last launch %d", iters, c->shard_k);
  const int rc = launch_finalize(c, false, iters);
  c->shard_k = -1;
  if (rc != HOT_OK) return rc;
  c->have_fields = true;
  return return_metrics(c, "hot_sharded_end", eff_out, unif_out);
}

int hot_get_metrics(hot_ctx *c, double *eff_out, double *unif_out) {
  if (!c) return fail(HOT_EINVAL, "hot_get_metrics: NULL context");
  if (!c->M || !c->have_fields) return fail(HOT_ESTATE, "hot_get_metrics: no forward evaluation since the last change");
  const int rc = read_back(c, "hot_get_metrics", false);
  if (rc != HOT_OK) return rc;
  if (eff_out) *eff_out = read_metrics(c)[0];
  if (unif_out) *unif_out = read_metrics(c)[1];
  return HOT_OK;
}

int hot_sync(hot_ctx *c) {
  if (!c) return fail(HOT_EINVAL, "hot_sync: NULL context");
  HOT_CUDA(cudaStreamSynchronize(c->st));
  return check_wait_error(c, "hot_sync");
}

int hot_set_trace(hot_ctx *c, int enable) {
  if (!c) return fail(HOT_EINVAL, "hot_set_trace: NULL context");
  if ((enable != 0) != c->tracing) {
    HOT_CUDA(cudaStreamSynchronize(c->st));
    drop_graphs(c);  // the captured launches carry (or not) trace slots
  }
  c->tracing = enable != 0;
  c->trace_iters = -1;
  return HOT_OK;
}

int hot_get_trace(hot_ctx *c, double *eff, double *unif, int n) {
  if (!c || !eff || !unif) return fail(HOT_EINVAL, "hot_get_trace: NULL argument");
  if (!c->tracing || c->trace_iters < 0 || !c->have_fields)
    return fail(HOT_ESTATE, "hot_get_trace: no traced hot_gsw since tracing was enabled");
  const int K = c->trace_iters;
  if (n != K + 1) return fail(HOT_EINVAL, "hot_get_trace: n = %d, the last call has %d values", n, K + 1);
  const int rc = check_wait_error(c, "hot_get_trace");
  if (rc != HOT_OK) return rc;
  std::vector<float> t(2 * (size_t)K + 2);
  if (K) HOT_CUDA(cudaMemcpyAsync(t.data(), c->trace, sizeof(float) * 2 * K, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaMemcpyAsync(t.data() + 2 * K, c->metrics, sizeof(float) * 2, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  for (int k = 0; k <= K; k++) {
    eff[k] = t[2 * k];
    unif[k] = t[2 * k + 1];
  }
  return HOT_OK;
}

int hot_get_state(hot_ctx *c, float *phi, float *w) {
  if (!c || !phi || !w) return fail(HOT_EINVAL, "hot_get_state: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_get_state: no traps set");
  const int rc = check_wait_error(c, "hot_get_state");
  if (rc != HOT_OK) return rc;
  HOT_CUDA(cudaMemcpyAsync(phi, c->phi, sizeof(float) * (size_t)c->W * c->H, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaMemcpyAsync(w, c->w, sizeof(float) * c->M, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  return HOT_OK;
}

int hot_set_state(hot_ctx *c, const float *phi, const float *w) {
  if (!c || !phi || !w) return fail(HOT_EINVAL, "hot_set_state: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_set_state: no traps set");
  for (int m = 0; m < c->M; m++)
    if (!(std::isfinite(w[m]) && w[m] > 0.f)) return fail(HOT_EINVAL, "hot_set_state: weight %d not finite and > 0", m);
  HOT_CUDA(cudaMemcpyAsync(c->phi, phi, sizeof(float) * (size_t)c->W * c->H, cudaMemcpyHostToDevice, c->st));
  HOT_CUDA(cudaMemcpyAsync(c->w, w, sizeof(float) * c->M, cudaMemcpyHostToDevice, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  c->have_fields = false;
  c->u_valid = false;
  return HOT_OK;
}

int hot_get_phasors(hot_ctx *c, float *u) {
  if (!c || !u) return fail(HOT_EINVAL, "hot_get_phasors: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_get_phasors: no traps set");
  if (!c->u_valid)
    return fail(HOT_ESTATE, "hot_get_phasors: no unit phasors of the current phases (hot_gsw leaves them in the accurate and fast modes with up to 128 traps)");
  const int rc = check_wait_error(c, "hot_get_phasors");
  if (rc != HOT_OK) return rc;
  HOT_CUDA(cudaMemcpyAsync(u, c->ubuf, sizeof(float2) * (size_t)c->W * c->H, cudaMemcpyDeviceToHost, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  return HOT_OK;
}

int hot_set_phasors(hot_ctx *c, const float *u) {
  if (!c || !u) return fail(HOT_EINVAL, "hot_set_phasors: NULL argument");
  if (!c->M) return fail(HOT_ESTATE, "hot_set_phasors: no traps set");
  if (!c->once) return fail(HOT_ESTATE, "hot_set_phasors: unit phasors are not in effect (hot_set_once)");
  const size_t n = 2 * (size_t)c->W * c->H;
  for (size_t i = 0; i < n; i++)
    if (!std::isfinite(u[i]) || std::fabs(u[i]) > 2.f)
      return fail(HOT_EINVAL, "hot_set_phasors: value %zu is not a unit phasor component", i);
  HOT_CUDA(cudaMemcpyAsync(c->ubuf, u, sizeof(float) * n, cudaMemcpyHostToDevice, c->st));
  HOT_CUDA(cudaStreamSynchronize(c->st));
  c->u_valid = true;
  return HOT_OK;
}

int hot_use_persistent(hot_ctx *c, int enable) {
  if (!c) return fail(HOT_EINVAL, "hot_use_persistent: NULL context");
  c->persistent = enable != 0;
  return HOT_OK;
}

int hot_set_wait_limit(hot_ctx *c, double seconds) {
  if (!c) return fail(HOT_EINVAL, "hot_set_wait_limit: NULL context");
  if (!(seconds >= 0.0) || seconds > 60.0) return fail(HOT_EINVAL, "hot_set_wait_limit: %g s not in [0, 60]", seconds);
  if (seconds != c->wait_limit_s) drop_graphs(c);  // the tensor-core launches carry the limit
  c->wait_limit_s = seconds;
  return HOT_OK;
}

long long hot_kernel_launches(const hot_ctx *c) { return c ? c->launches : 0; }

int hot_use_graphs(hot_ctx *c, int enable) {
  if (!c) return fail(HOT_EINVAL, "hot_use_graphs: NULL context");
  c->use_graphs = enable != 0;
  return HOT_OK;
}

int hot_profile(hot_ctx *c, int enable) {
  if (!c) return fail(HOT_EINVAL, "hot_profile: NULL context");
  if (!enable && c->profiling) {
    HOT_CUDA(cudaStreamSynchronize(c->st));
    clear_records(c);
  }
  c->profiling = enable != 0;
  return HOT_OK;
}

int hot_profile_read(hot_ctx *c, double *ms, long long *launches) {
  if (!c) return fail(HOT_EINVAL, "hot_profile_read: NULL context");
  HOT_CUDA(cudaStreamSynchronize(c->st));
  double t[HOT_KERNEL_KINDS] = {0, 0, 0, 0};
  long long n[HOT_KERNEL_KINDS] = {0, 0, 0, 0};
  for (auto &r : c->recs) {
    float x = 0.f;
    cudaError_t e = cudaEventElapsedTime(&x, r.a, r.b);
    if (e != cudaSuccess) {
      clear_records(c);
      return fail(HOT_ECUDA, "hot_profile_read: %s", cudaGetErrorString(e));
    }
    t[r.kind] += x;
    n[r.kind] += 1;
  }
  clear_records(c);
  for (int k = 0; k < HOT_KERNEL_KINDS; k++) {
    if (ms) ms[k] = t[k];
    if (launches) launches[k] = n[k];
  }
  return HOT_OK;
}

}  // extern "C"


// ---------------------------------------------------------------------------------------------
// Batches of holograms (hot_batch_*).
struct hot_batch {
  int count = 0, precision = HOT_PREC_ACCURATE, dev = 0;
  std::vector<hot_ctx *> ctx;
  cudaStream_t st = nullptr, cap = nullptr;
  cudaEvent_t ev = nullptr;  // the members' streams' work that a run starts after (batch_after_members)
  int sms = 0, per_sm_max = 1;
  // tiling (hot_batch_set_tiling) and group threshold in pixel-trap pairs per iteration
  int rows = hot::kRowsMax, bps = 0, chunk = hot::kChunk;
  double group_pairs = 67108864.0;
  struct Group {
    std::vector<int> members;         // context indices (<= kBatchMax); SubTile::pad indexes this list
    int grid = 0, n_sub = 0;
    hot::SubTile *sub = nullptr;
    int *first = nullptr;
    std::vector<int> owner;                  // block that writes each hologram's weights
    std::vector<hot::StepArgs> holo[6];      // parameters for launch k (k % 6; k = 0 uses set 0)
    bool alone = false;                      // one hologram on hot_gsw's own step ...
    hot::TileArgs own[6];                    // ... whose parameters these are
    hot::FinalizeArgs *fin[6] = {};          // finalize descriptors for iters % 6
  };
  std::vector<Group> groups;
  unsigned long long *stamps = nullptr;  // [count + 1]: completion of hologram h; [count]: start
  bool ran = false;
  // HOT_PREC_TENSOR: each member runs its own hot_gsw launch sequence; the members are dealt out
  // to up to kTensorChains streams (largest work first, each to the least loaded chain) whose
  // launches overlap, forked from and joined to the batch's stream inside its graph
  std::vector<std::vector<int>> chains;
  std::vector<cudaStream_t> chain_st;
  std::vector<cudaEvent_t> chain_ev;  // [0]: fork; [1 + i]: end of chain i

  struct Graph {
    int iters;
    std::vector<double> limits;  // HOT_PREC_TENSOR: the members' wait limits, which the launches carry
    cudaGraphExec_t exec;
  };
  std::vector<Graph> graphs;
};

namespace {

std::vector<double> batch_limits(const hot_batch *b) {
  std::vector<double> v;
  if (b->precision == HOT_PREC_TENSOR)
    for (const hot_ctx *c : b->ctx) v.push_back(c->wait_limit_s);
  return v;
}

int batch_mode(const hot_batch *b) {
  return b->precision == HOT_PREC_SEPARABLE ? hot::kModeSeparable
                                            : b->precision == HOT_PREC_FAST ? hot::kModeFast : hot::kModeAccurate;
}

// Dynamic shared memory of the batch kernels: the separable one stages `chunk` complex traps.
int batch_smem(const hot_batch *b) {
  return b->precision == HOT_PREC_SEPARABLE ? hot::sep_smem_bytes(b->chunk) : hot::step_smem_bytes(0, true);
}

template <int MODE>
int batch_set_smem() {
  const int bytes = MODE == hot::kModeSeparable ? hot::sep_smem_bytes(hot::kChunk) : hot::step_smem_bytes(0, true);
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_batch_kernel<MODE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  HOT_CUDA(cudaFuncSetAttribute(hot::gsw_batch_kernel<MODE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  return HOT_OK;
}

// Resident blocks per SM of the batch's fused kernel at its current staging chunk.
int batch_occupancy(hot_batch *b) {
  int per_sm = 0;
  const int smem = batch_smem(b);
  cudaError_t e;
  switch (batch_mode(b)) {
    case hot::kModeSeparable:
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hot::gsw_batch_kernel<hot::kModeSeparable, true>,
                                                        hot::kThreads, smem);
      break;
    case hot::kModeFast:
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hot::gsw_batch_kernel<hot::kModeFast, true>,
                                                        hot::kThreads, smem);
      break;
    default:
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hot::gsw_batch_kernel<hot::kModeAccurate, true>,
                                                        hot::kThreads, smem);
  }
  if (e != cudaSuccess) return fail(HOT_ECUDA, "batch occupancy query: %s", cudaGetErrorString(e));
  b->per_sm_max = per_sm < 1 ? 1 : per_sm;
  return HOT_OK;
}

void batch_drop_graphs(hot_batch *b) {
  for (auto &g : b->graphs) cudaGraphExecDestroy(g.exec);
  b->graphs.clear();
}

void group_free(hot_batch::Group &g) {
  dfree(g.sub);
  dfree(g.first);
  for (auto &p : g.fin) dfree(p);
}

void batch_free(hot_batch *b) {
  batch_drop_graphs(b);
  for (auto &g : b->groups) group_free(g);
  b->groups.clear();
  dfree(b->stamps);
  if (b->cap) cudaStreamDestroy(b->cap);
  b->cap = nullptr;
  if (b->ev) cudaEventDestroy(b->ev);
  b->ev = nullptr;
  for (cudaStream_t s : b->chain_st) cudaStreamDestroy(s);
  for (cudaEvent_t e : b->chain_ev) cudaEventDestroy(e);
  b->chain_st.clear();
  b->chain_ev.clear();
}

// Copies of the accumulators of a batch's member: as acc_copies, but the batched kernel of the accurate
// and fast modes keeps one.
int batch_copies(const hot_batch *b, const hot_ctx *c) { return b->precision == HOT_PREC_SEPARABLE && c->M <= 512 ? 8 : 1; }

// Batched-kernel parameters of context c for launch k of a sequence (buffers rotate as in hot_gsw).
hot::StepArgs batch_args(const hot_batch *b, const hot_ctx *c, int k) {
  hot::StepArgs a = {};
  const bool fast = b->precision == HOT_PREC_FAST;
  const size_t M2 = 2 * (size_t)c->M * batch_copies(b, c);
  a.W = c->W;
  a.H = c->H;
  a.M = c->M;
  a.chunk = b->chunk;
  a.copies = batch_copies(b, c);
  a.X = fast ? c->Xr : c->Xt;
  a.Y = fast ? c->Yr : c->Yt;
  a.Y4 = fast ? c->Y4r : c->Y4t;
  a.ldy4 = c->ldy4;
  a.Xc = c->Xb;
  a.Yc = c->Yb;
  a.phi = c->phi;
  a.acc_in = c->acc + M2 * ((k + 2) % 3);
  a.acc_out = c->acc + M2 * (k % 3);
  a.acc_clear = c->acc + M2 * ((k + 1) % 3);
  a.w_in = c->w + (size_t)c->M * ((k + 1) & 1);
  a.w_out = c->w + (size_t)c->M * (k & 1);
  a.fx_scale = ldexpf(1.0f, c->fx_shift);
  a.inv_fx_n = (float)(1.0 / (n_total(c) * ldexp(1.0, c->fx_shift)));
  a.angle_units = fast ? 1.0f : 0.15915494309189535f;
  a.angle_eta = fast ? hot::kFastEta : 0.0f;
  a.inv_n = (float)(1.0 / (n_total(c)));
  return a;
}

double pairs_of(const hot_ctx *c) { return n_total(c) * (double)c->M; }

// One group's work schedule: the row segments of its holograms in order, each weighted by its
// trap count, dealt out to one wave of G blocks in equal shares (a segment goes to the block
// that holds the midpoint of its weight interval); each block's run of rows in a strip is cut
// into equal sub-tiles of <= rows rows.
// A group of one hologram runs hot_gsw's own step on its own cut where one group per hologram was
// asked for (group_pairs <= 1) with the default tiling, and hot_gsw runs the tile kernels.
int build_group(hot_batch *b, hot_batch::Group &g) {
  const int count = (int)g.members.size();
  const int per_sm = b->bps > 0 ? std::min(b->bps, b->per_sm_max) : b->per_sm_max;
  long double T = 0;
  long long segments = 0;
  for (int h : g.members) {
    const hot_ctx *c = b->ctx[h];
    const long long seg = (long long)((c->W + hot::kTileW - 1) / hot::kTileW) * c->H;
    segments += seg;
    T += (long double)seg * c->M;
  }
  g.alone = count == 1 && b->group_pairs <= 1.0 && b->rows == hot::kRowsMax && per_sm == b->per_sm_max &&
            b->chunk == hot::kChunk && tile_kernels(b->ctx[g.members[0]]);
  TileCut cut;
  if (g.alone) {
    const hot_ctx *c = b->ctx[g.members[0]];
    const int rc = cut_tiles(c->W, c->H, c->M, b->sms, cut);
    if (rc != HOT_OK) return rc;
  }
  const int G = (int)std::min<long long>((long long)b->sms * per_sm, segments);
  std::vector<hot::SubTile> sub;
  std::vector<int> first(G + 1, 0), owner(count, -1);
  long double w0 = 0;
  int cur_b = 0;
  for (int i = 0; i < count; i++) {
    const hot_ctx *c = b->ctx[g.members[i]];
    const int strips = (c->W + hot::kTileW - 1) / hot::kTileW;
    for (int s = 0; s < strips; s++) {
      auto block_of = [&](int row) {
        const long double mid = w0 + ((long double)row + 0.5L) * c->M;
        const int bb = (int)(mid * G / T);
        return bb < 0 ? 0 : (bb >= G ? G - 1 : bb);
      };
      int r = 0;
      while (r < c->H) {  // the run of rows of this strip that goes to block bb, cut evenly
        const int bb = block_of(r);
        int r1 = r + 1;
        while (r1 < c->H && block_of(r1) == bb) r1++;
        while (cur_b < bb) first[++cur_b] = (int)sub.size();
        if (owner[i] < 0) owner[i] = bb;
        const int L = r1 - r, nsub = (L + b->rows - 1) / b->rows;
        for (int q = 0; q < nsub; q++) {
          const int q0 = r + (int)((long long)L * q / nsub), q1 = r + (int)((long long)L * (q + 1) / nsub);
          sub.push_back({s * hot::kTileW, q0, q1 - q0, i});
        }
        r = r1;
      }
      w0 += (long double)c->H * c->M;
    }
  }
  while (cur_b < G) first[++cur_b] = (int)sub.size();
  if (g.alone) sub = cut.tiles;
  g.grid = g.alone ? cut.grid : G;
  g.n_sub = (int)sub.size();
  g.owner = owner;
  for (int k = 0; k < 6; k++) {
    g.holo[k].resize(count);
    for (int i = 0; i < count; i++) g.holo[k][i] = batch_args(b, b->ctx[g.members[i]], k == 0 ? 6 : k);
  }
  int rc = dalloc(&g.sub, sub.size());
  if (rc == HOT_OK) rc = dalloc(&g.first, first.size());
  for (int k = 0; g.alone && k < 6; k++) {
    hot::TileArgs &t = g.own[k];
    t = make_tile_args(b->ctx[g.members[0]], k == 0 ? 6 : k, nullptr, nullptr, nullptr);
    t.s.sub = g.sub;
    t.s.trace = nullptr;
    t.team = cut.team;
    t.pairs = cut.pairs;
    t.stride = cut.stride;
  }
  for (int r6 = 0; rc == HOT_OK && r6 < 6; r6++) {  // finalize after `iters` iterations, iters % 6 == r6
    rc = dalloc(&g.fin[r6], (size_t)count);
    std::vector<hot::FinalizeArgs> fs(count);
    for (int i = 0; i < count; i++) {
      const hot_ctx *c = b->ctx[g.members[i]];
      hot::FinalizeArgs &f = fs[i];
      f.M = c->M;
      f.copies = g.alone ? acc_copies(c) : batch_copies(b, c);
      f.acc = c->acc + 2 * (size_t)c->M * f.copies * (r6 % 3);  // the last launch accumulated into acc[iters % 3]
      f.acc_all = c->acc;
      f.w_src = c->w + (size_t)c->M * (r6 & 1);       // and left the weights in w[iters & 1]
      f.w_dst = c->w;
      f.Vsum = c->Vsum;
      f.metrics = c->metrics;
      f.inv_fx_n = (float)(1.0 / (n_total(c) * ldexp(1.0, c->fx_shift)));
      f.done = b->stamps + g.members[i];
    }
    if (rc == HOT_OK && cudaMemcpy(g.fin[r6], fs.data(), sizeof(hot::FinalizeArgs) * count, cudaMemcpyHostToDevice) != cudaSuccess)
      rc = fail(HOT_ECUDA, "batch schedule: copy of descriptors failed");
  }
  if (rc == HOT_OK) {
    cudaError_t e = cudaMemcpy(g.sub, sub.data(), sizeof(hot::SubTile) * sub.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(g.first, first.data(), sizeof(int) * first.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) rc = fail(HOT_ECUDA, "batch schedule: %s", cudaGetErrorString(e));
  }
  return rc;
}

// The tables that the batched kernel reads, where the member does not have them yet.
int batch_tables(const hot_batch *b, hot_ctx *c) {
  const int rc = b->precision == HOT_PREC_SEPARABLE ? alloc_batch_tables(c) : alloc_direct_tables(c, c->M);
  if (rc != HOT_OK || !c->unbuilt) return rc;
  return launch_build_tables(c);  // (on the member's stream, behind which a run starts)
}

// Orders the holograms by pairs per iteration (smallest first, stable), cuts them into
// groups of >= group_pairs (a short last group joins the one before) and builds each group.
int batch_schedule(hot_batch *b) {
  HOT_CUDA(cudaStreamSynchronize(b->st));
  batch_drop_graphs(b);
  int rc0 = batch_occupancy(b);
  for (size_t h = 0; h < b->ctx.size() && rc0 == HOT_OK; h++) rc0 = batch_tables(b, b->ctx[h]);
  if (rc0 != HOT_OK) return rc0;
  for (auto &g : b->groups) group_free(g);
  b->groups.clear();
  b->ran = false;
  std::vector<int> order(b->count);
  for (int h = 0; h < b->count; h++) order[h] = h;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return pairs_of(b->ctx[x]) < pairs_of(b->ctx[y]); });
  std::vector<std::vector<int>> parts;
  double sum = 0;
  for (int h : order) {
    if (parts.empty() || sum >= b->group_pairs || (int)parts.back().size() == hot::kBatchMax) {
      parts.emplace_back();
      sum = 0;
    }
    parts.back().push_back(h);
    sum += pairs_of(b->ctx[h]);
  }
  if (parts.size() > 1 && sum < b->group_pairs && parts.back().size() + parts[parts.size() - 2].size() <= hot::kBatchMax) {
    auto last = parts.back();
    parts.pop_back();
    parts.back().insert(parts.back().end(), last.begin(), last.end());
  }
  b->groups.resize(parts.size());
  for (size_t i = 0; i < parts.size(); i++) {
    b->groups[i].members = parts[i];
    const int rc = build_group(b, b->groups[i]);
    if (rc != HOT_OK) {
      for (auto &g : b->groups) group_free(g);
      b->groups.clear();
      return rc;
    }
  }
  return HOT_OK;
}

template <int MODE, bool BACK>
int batch_launch(hot_batch *b, const hot_batch::Group &g, int k) {
  hot::BatchArgs a = {};
  const int count = (int)g.members.size();
  for (int i = 0; i < count; i++) {
    a.holo[i] = g.holo[k % 6][i];
    a.owner[i] = g.owner[i];
  }
  a.sub = g.sub;
  a.first = g.first;
  a.count = count;
  hot_ctx tmp;  // launch() needs a context only for the stream
  tmp.st = b->st;
  launch(&tmp, hot::gsw_batch_kernel<MODE, BACK>, g.grid, hot::kThreads, batch_smem(b), true, a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(HOT_ECUDA, "launch of gsw_batch_kernel: %s", cudaGetErrorString(e));
  return HOT_OK;
}

// Launch k of a group of one hologram on hot_gsw's own step.
template <bool BACK>
int batch_launch_own(hot_batch *b, const hot_batch::Group &g, int k) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.grid);
  cfg.blockDim = dim3(hot::kThreads);
  cfg.stream = b->st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  hot_tile::launch(BACK, true, false, cfg, g.own[k % 6]);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(HOT_ECUDA, "launch of gsw_tile_kernel: %s", cudaGetErrorString(e));
  return HOT_OK;
}

// Launch k of a group: BACK an iteration, otherwise the forward field of the starting phases (k = 0).
template <bool BACK>
int batch_launch_mode(hot_batch *b, const hot_batch::Group &g, int k) {
  if (g.alone) return batch_launch_own<BACK>(b, g, k);
  switch (batch_mode(b)) {
    case hot::kModeSeparable: return batch_launch<hot::kModeSeparable, BACK>(b, g, k);
    case hot::kModeFast: return batch_launch<hot::kModeFast, BACK>(b, g, k);
    default: return batch_launch<hot::kModeAccurate, BACK>(b, g, k);
  }
}

constexpr int kTensorChains = 8;

// Tensor-mode batch set-up: every member's tensor-core operands, and its chain (largest work
// N M first, each to the chain with the least work so far).
int batch_setup_tensor(hot_batch *b) {
  for (hot_ctx *c : b->ctx) {
    const int rc = ensure_tc_plan(c);
    if (rc != HOT_OK) return rc;
    HOT_CUDA(cudaStreamSynchronize(c->st));
  }
  const int n = std::min(b->count, kTensorChains);
  std::vector<int> order(b->count);
  for (int h = 0; h < b->count; h++) order[h] = h;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return pairs_of(b->ctx[x]) > pairs_of(b->ctx[y]); });
  std::vector<double> load(n, 0.0);
  b->chains.assign(n, {});
  for (int h : order) {
    const int i = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    b->chains[i].push_back(h);
    load[i] += pairs_of(b->ctx[h]);
  }
  b->chain_st.assign(n, nullptr);
  b->chain_ev.assign(n + 1, nullptr);
  for (int i = 0; i < n; i++) HOT_CUDA(cudaStreamCreateWithFlags(&b->chain_st[i], cudaStreamNonBlocking));
  for (int i = 0; i <= n; i++) HOT_CUDA(cudaEventCreateWithFlags(&b->chain_ev[i], cudaEventDisableTiming));
  return HOT_OK;
}

// Tensor-mode batch: a start stamp, then every chain on its own stream (forked from the batch's
// stream by an event), each member's hot_gsw sequence followed by its completion stamp, and the
// chains joined back.  Each member computes exactly what hot_gsw(iters) computes for it.
int batch_enqueue_tensor(hot_batch *b, int iters) {
  hot::stamp_kernel<<<1, 1, 0, b->st>>>(b->stamps + b->count);
  HOT_CUDA(cudaGetLastError());
  HOT_CUDA(cudaEventRecord(b->chain_ev[0], b->st));
  for (size_t i = 0; i < b->chains.size(); i++) {
    cudaStream_t s = b->chain_st[i];
    HOT_CUDA(cudaStreamWaitEvent(s, b->chain_ev[0], 0));
    for (int h : b->chains[i]) {
      hot_ctx *c = b->ctx[h];
      cudaStream_t own = c->st;
      c->st = s;
      const int rc = enqueue_gsw(c, iters);
      c->st = own;
      if (rc != HOT_OK) return rc;
      hot::stamp_kernel<<<1, 1, 0, s>>>(b->stamps + h);
      HOT_CUDA(cudaGetLastError());
    }
    HOT_CUDA(cudaEventRecord(b->chain_ev[1 + i], s));
    HOT_CUDA(cudaStreamWaitEvent(b->st, b->chain_ev[1 + i], 0));
  }
  return HOT_OK;
}

// A start stamp, then the groups in order: forward field of the starting phases (k = 0),
// iterations 1..iters, and the per-hologram finalize with its completion stamp.
int batch_enqueue(hot_batch *b, int iters) {
  if (b->precision == HOT_PREC_TENSOR) return batch_enqueue_tensor(b, iters);
  hot::stamp_kernel<<<1, 1, 0, b->st>>>(b->stamps + b->count);
  cudaError_t e0 = cudaGetLastError();
  if (e0 != cudaSuccess) return fail(HOT_ECUDA, "launch of stamp_kernel: %s", cudaGetErrorString(e0));
  for (size_t gi = 0; gi < b->groups.size(); gi++) {
    const hot_batch::Group &g = b->groups[gi];
    int rc = batch_launch_mode<false>(b, g, 0);
    for (int k = 1; k <= iters && rc == HOT_OK; k++) rc = batch_launch_mode<true>(b, g, k);
    if (rc != HOT_OK) return rc;
    hot_ctx tmp;
    tmp.st = b->st;
    launch(&tmp, hot::gsw_finalize_batch_kernel, (int)g.members.size(), hot::kFinalizeThreads, 0, true,
           (const hot::FinalizeArgs *)g.fin[iters % 6]);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(HOT_ECUDA, "launch of gsw_finalize_batch_kernel: %s", cudaGetErrorString(e));
  }
  return HOT_OK;
}

// Orders the batch's stream behind what the members queued on other streams: traps, weights, phases
// and superpositions are queued (their calls return before the work is done).  A member's stream
// under capture is left to its owner; a batch's stream under capture can only wait on the host.
int batch_after_members(hot_batch *b) {
  std::vector<cudaStream_t> seen = {b->st};
  cudaStreamCaptureStatus mine = cudaStreamCaptureStatusNone;
  for (const hot_ctx *c : b->ctx) {
    if (std::find(seen.begin(), seen.end(), c->st) != seen.end()) continue;
    if (seen.size() == 1) HOT_CUDA(cudaStreamIsCapturing(b->st, &mine));
    seen.push_back(c->st);
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaStreamCaptureStatus theirs = cudaStreamCaptureStatusNone;
    if (mine == cudaStreamCaptureStatusNone) {
      const cudaError_t e = cudaStreamIsCapturing(c->st, &theirs);
      if (e == cudaErrorStreamCaptureImplicit) cudaGetLastError();  // the legacy stream, beside another's capture
      else HOT_CUDA(e);
      if (e != cudaSuccess || theirs != cudaStreamCaptureStatusNone) continue;
      if (!b->ev) HOT_CUDA(cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming));
      HOT_CUDA(cudaEventRecord(b->ev, c->st));
      HOT_CUDA(cudaStreamWaitEvent(b->st, b->ev, 0));
    } else if (c->st) {
      HOT_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
      cudaError_t e = cudaStreamIsCapturing(c->st, &theirs);
      if (e == cudaSuccess && theirs == cudaStreamCaptureStatusNone) e = cudaStreamSynchronize(c->st);
      cudaThreadExchangeStreamCaptureMode(&mode);
      if (e != cudaSuccess) return fail(HOT_ECUDA, "hot_batch_gsw: waiting for a member's stream: %s", cudaGetErrorString(e));
    }
  }
  return HOT_OK;
}

int check_tiling(const char *who, int rows, int bps, int chunk) {
  if (rows < 0 || rows > hot::kRowsMax) return fail(HOT_EINVAL, "%s: rows = %d not in [1, %d] (0: default)", who, rows, hot::kRowsMax);
  if (bps < 0 || bps > 32) return fail(HOT_EINVAL, "%s: blocks_per_sm = %d not in [1, 32] (0: default)", who, bps);
  if (chunk < 0 || chunk > hot::kChunk) return fail(HOT_EINVAL, "%s: chunk = %d not in [1, %d] (0: default)", who, chunk, hot::kChunk);
  return HOT_OK;
}

struct Tiling {
  int rows, bps, chunk, merge;
  bool operator==(const Tiling &o) const {
    return rows == o.rows && bps == o.bps && chunk == o.chunk && merge == o.merge;
  }
};

// The kernels are launch-bounded to at most 4 resident blocks per SM; a candidate above what
// the current staging chunk leaves room for is clamped to it by the schedule.
constexpr int kMaxBlocksPerSm = 4;

// Coordinate search: each parameter in turn takes the fastest of its candidates with the
// others fixed; a candidate replaces the incumbent only if it is more than 1 % faster; at
// most two passes.  apply(t) installs a tiling, time(&us) measures it.  Leaves `best` applied.
// With merge, the blocks-per-SM candidates include max_bps blocks merged four and two to a
// launched block (Tiling::merge: schedule blocks per launched block).
template <typename Apply, typename Time>
int tune_tiling(int max_bps, Tiling &best, double &best_us, Apply apply, Time time, bool merge = false) {
  static const int rows_c[] = {14, 12, 10, 8, 6, 4, 2};
  static const int chunk_c[] = {128, 96, 64, 32};
  int rc = apply(best);
  if (rc == HOT_OK) rc = time(&best_us);
  for (int pass = 0; rc == HOT_OK && pass < 2; pass++) {
    bool changed = false;
    for (int dim = 0; rc == HOT_OK && dim < 3; dim++) {
      std::vector<int> cand;  // blocks per SM; -4 and -2: max_bps blocks merged 4 or 2 to a block
      if (dim == 0) cand.assign(std::begin(rows_c), std::end(rows_c));
      if (dim == 1) {
        if (merge) {
          cand.push_back(-4);
          cand.push_back(-2);
        }
        for (int v = max_bps; v >= 1; v--) cand.push_back(v);
      }
      if (dim == 2) cand.assign(std::begin(chunk_c), std::end(chunk_c));
      for (int v : cand) {
        Tiling t = best;
        if (dim == 1) {
          t.bps = v < 0 ? max_bps : v;
          t.merge = v < 0 ? -v : 1;
        } else {
          (dim == 0 ? t.rows : t.chunk) = v;
        }
        if (t == best) continue;
        double us = 0;
        rc = apply(t);
        if (rc == HOT_OK) rc = time(&us);
        if (rc != HOT_OK) break;
        if (us < 0.99 * best_us) {
          best = t;
          best_us = us;
          changed = true;
        }
      }
    }
    if (!changed) break;
  }
  const int rc2 = apply(best);
  return rc != HOT_OK ? rc : rc2;
}

// Device copies of phases and weights that an autotuner restores before every timed run.
struct Saved {
  float *phi = nullptr, *w = nullptr;
  ~Saved() {
    dfree(phi);
    dfree(w);
  }
};

int save_state(hot_ctx *c, Saved &s, cudaStream_t st) {
  const size_t N = (size_t)c->W * c->H;
  int rc = dalloc(&s.phi, N);
  if (rc == HOT_OK) rc = dalloc(&s.w, (size_t)c->M);
  if (rc != HOT_OK) return rc;
  HOT_CUDA(cudaMemcpyAsync(s.phi, c->phi, N * sizeof(float), cudaMemcpyDeviceToDevice, st));
  HOT_CUDA(cudaMemcpyAsync(s.w, c->w, c->M * sizeof(float), cudaMemcpyDeviceToDevice, st));
  return HOT_OK;
}

int restore_state(hot_ctx *c, const Saved &s, cudaStream_t st) {
  c->u_valid = false;
  HOT_CUDA(cudaMemcpyAsync(c->phi, s.phi, (size_t)c->W * c->H * sizeof(float), cudaMemcpyDeviceToDevice, st));
  HOT_CUDA(cudaMemcpyAsync(c->w, s.w, c->M * sizeof(float), cudaMemcpyDeviceToDevice, st));
  return HOT_OK;
}

// Best of three timed runs after one untimed run (graph capture, warm-up), in microseconds
// per iteration; restore() is queued before each run, outside the timed events.
template <typename Restore, typename Run>
int time_runs(cudaStream_t st, int iters, double *us, Restore restore, Run run) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  HOT_CUDA(cudaEventCreate(&e0));
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return fail(HOT_ECUDA, "autotune: cudaEventCreate failed");
  }
  double best = 1e300;
  int rc = HOT_OK;
  for (int r = 0; rc == HOT_OK && r < 4; r++) {
    rc = restore();
    if (rc == HOT_OK && cudaEventRecord(e0, st) != cudaSuccess) rc = fail(HOT_ECUDA, "autotune: event record failed");
    if (rc == HOT_OK) rc = run();
    if (rc == HOT_OK && cudaEventRecord(e1, st) != cudaSuccess) rc = fail(HOT_ECUDA, "autotune: event record failed");
    float ms = 0.f;
    if (rc == HOT_OK) {
      cudaError_t e = cudaEventSynchronize(e1);
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e != cudaSuccess) rc = fail(HOT_ECUDA, "autotune: %s", cudaGetErrorString(e));
    }
    if (rc == HOT_OK && r > 0) best = std::min(best, (double)ms);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc == HOT_OK) *us = best * 1000.0 / iters;
  return rc;
}

}  // namespace

extern "C" {

int hot_set_tiling(hot_ctx *c, int rows, int blocks_per_sm, int chunk) {
  if (!c) return fail(HOT_EINVAL, "hot_set_tiling: NULL context");
  int rc = check_tiling("hot_set_tiling", rows, blocks_per_sm, chunk);
  if (rc != HOT_OK) return rc;
  HOT_CUDA(cudaStreamSynchronize(c->st));
  const int rows0 = c->tile_rows, bps0 = c->tile_bps, chunk0 = c->tile_chunk;
  c->tile_rows = rows ? rows : hot::kRowsMax;
  c->tile_bps = blocks_per_sm;
  c->tile_chunk = chunk ? chunk : hot::kChunk;
  rc = c->M ? build_schedule(c) : HOT_OK;
  if (rc != HOT_OK) {
    c->tile_rows = rows0;
    c->tile_bps = bps0;
    c->tile_chunk = chunk0;
  }
  return rc;
}

int hot_get_tiling(const hot_ctx *c, int *rows, int *blocks_per_sm, int *chunk) {
  if (!c) return fail(HOT_EINVAL, "hot_get_tiling: NULL context");
  if (rows) *rows = c->tile_rows;
  if (blocks_per_sm) *blocks_per_sm = c->sched_bps;
  if (chunk) *chunk = c->tile_chunk;
  return HOT_OK;
}

int hot_set_block_merge(hot_ctx *c, int merge) {
  if (!c) return fail(HOT_EINVAL, "hot_set_block_merge: NULL context");
  if (merge != 1 && merge != 2 && merge != 4) return fail(HOT_EINVAL, "hot_set_block_merge: merge = %d is not 1, 2 or 4", merge);
  HOT_CUDA(cudaStreamSynchronize(c->st));
  const int merge0 = c->tile_merge;
  c->tile_merge = merge;
  const int rc = c->M ? build_schedule(c) : HOT_OK;
  if (rc != HOT_OK) c->tile_merge = merge0;
  return rc;
}

int hot_get_block_merge(const hot_ctx *c, int *requested, int *in_effect) {
  if (!c) return fail(HOT_EINVAL, "hot_get_block_merge: NULL context");
  if (requested) *requested = c->tile_merge;
  if (in_effect) *in_effect = c->groups;
  return HOT_OK;
}

int hot_set_once(hot_ctx *c, int on) {
  if (!c) return fail(HOT_EINVAL, "hot_set_once: NULL context");
  if (on != 0 && on != 1) return fail(HOT_EINVAL, "hot_set_once: on = %d is not 0 or 1", on);
  HOT_CUDA(cudaStreamSynchronize(c->st));
  return enter_mode(c, c->precision, on != 0, true);
}

int hot_get_once(const hot_ctx *c, int *requested, int *in_effect) {
  if (!c) return fail(HOT_EINVAL, "hot_get_once: NULL context");
  if (requested) *requested = c->once_req ? 1 : 0;
  if (in_effect) *in_effect = c->once ? 1 : 0;
  return HOT_OK;
}

int hot_autotune(hot_ctx *c, int iters, int *rows, int *blocks_per_sm, int *chunk, double *us_per_iter) {
  if (!c) return fail(HOT_EINVAL, "hot_autotune: NULL context");
  if (!c->M) return fail(HOT_ESTATE, "hot_autotune: no traps set");
  if (iters < 1) return fail(HOT_EINVAL, "hot_autotune: iters = %d < 1", iters);
  if (c->precision == HOT_PREC_TENSOR)
    return fail(HOT_EINVAL, "hot_autotune: HOT_PREC_TENSOR has no tiling parameters (its tiles are fixed)");
  Saved saved;
  int rc = save_state(c, saved, c->st);
  if (rc != HOT_OK) return rc;
  const bool profiling = c->profiling;
  c->profiling = false;
  auto timed_gsw = [&](double *us) {
    return time_runs(c->st, iters, us, [&]() { return restore_state(c, saved, c->st); },
                     [&]() { return hot_gsw(c, iters, nullptr, nullptr); });
  };
  // The tile kernels, where they apply, against the best tiling of the direct kernels; the
  // separable mode has no others.
  const bool once_req = c->once_req, tile = tile_kernels(c);
  Tiling best = {c->tile_rows, c->sched_bps, c->tile_chunk, c->tile_merge};
  double best_us = 0, tile_us = 0;
  if (tile) rc = timed_gsw(&tile_us);
  if (separable_kernels(c)) {
    best_us = tile_us;
  } else {
    if (rc == HOT_OK && tile) rc = hot_set_once(c, 0);
    if (rc == HOT_OK) rc = tune_tiling(
        kMaxBlocksPerSm, best, best_us,
        [&](const Tiling &t) {
          c->tile_merge = t.merge;  // applied by the schedule that hot_set_tiling rebuilds
          return hot_set_tiling(c, t.rows, t.bps, t.chunk);
        },
        timed_gsw, true);
    if (rc == HOT_OK && tile && tile_us < best_us) {
      rc = hot_set_once(c, 1);
      best_us = tile_us;
    } else if (rc != HOT_OK && c->once_req != once_req) {
      hot_set_once(c, once_req ? 1 : 0);  // back to the kernels it had; the first error is reported
    }
  }
  c->profiling = profiling;
  const int rc2 = restore_state(c, saved, c->st);
  cudaStreamSynchronize(c->st);
  c->have_fields = false;
  c->u_valid = false;
  if (rc != HOT_OK) return rc;
  if (rc2 != HOT_OK) return rc2;
  if (rows) *rows = best.rows;
  if (blocks_per_sm) *blocks_per_sm = best.bps;
  if (chunk) *chunk = best.chunk;
  if (us_per_iter) *us_per_iter = best_us;
  return HOT_OK;
}

int hot_batch_create(hot_batch **out, int count, hot_ctx *const *ctxs, void *cuda_stream) {
  if (!out) return fail(HOT_EINVAL, "hot_batch_create: out is NULL");
  *out = nullptr;
  if (count < 1 || !ctxs) return fail(HOT_EINVAL, "hot_batch_create: no contexts");
  for (int i = 0; i < count; i++) {
    if (!ctxs[i]) return fail(HOT_EINVAL, "hot_batch_create: context %d is NULL", i);
    if (!ctxs[i]->M) return fail(HOT_ESTATE, "hot_batch_create: context %d has no traps", i);
    if (ctxs[i]->precision != ctxs[0]->precision)
      return fail(HOT_EINVAL, "hot_batch_create: contexts differ in precision mode");
    if (ctxs[i]->H_total != ctxs[i]->H)
      return fail(HOT_EINVAL, "hot_batch_create: context %d is a row band (its sums need an exchange)", i);
    if (ctxs[i]->dev != ctxs[0]->dev) return fail(HOT_EINVAL, "hot_batch_create: contexts on different devices");
    for (int j = 0; j < i; j++)
      if (ctxs[j] == ctxs[i]) return fail(HOT_EINVAL, "hot_batch_create: context %d given twice", i);
  }
  hot_batch *b = new (std::nothrow) hot_batch;
  if (!b) return fail(HOT_ENOMEM, "hot_batch_create: out of host memory");
  b->count = count;
  b->ctx.assign(ctxs, ctxs + count);
  b->st = static_cast<cudaStream_t>(cuda_stream);
  b->precision = ctxs[0]->precision;
  b->dev = ctxs[0]->dev;
  const bool tensor = b->precision == HOT_PREC_TENSOR;
  int rc = tensor                                 ? HOT_OK
           : batch_mode(b) == hot::kModeSeparable ? batch_set_smem<hot::kModeSeparable>()
           : batch_mode(b) == hot::kModeFast      ? batch_set_smem<hot::kModeFast>()
                                                  : batch_set_smem<hot::kModeAccurate>();
  if (rc == HOT_OK && cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->dev) != cudaSuccess)
    rc = fail(HOT_ECUDA, "hot_batch_create: device query failed");
  if (rc == HOT_OK) rc = dalloc(&b->stamps, (size_t)count + 1);
  if (rc == HOT_OK) rc = tensor ? batch_setup_tensor(b) : batch_schedule(b);
  if (rc != HOT_OK) {
    batch_free(b);
    delete b;
    return rc;
  }
  *out = b;
  return HOT_OK;
}

int hot_batch_set_tiling(hot_batch *b, int rows, int blocks_per_sm, int chunk, double group_pairs) {
  if (!b) return fail(HOT_EINVAL, "hot_batch_set_tiling: NULL batch");
  if (b->precision == HOT_PREC_TENSOR) return fail(HOT_EINVAL, "hot_batch_set_tiling: a HOT_PREC_TENSOR batch has no tiling");
  int rc = check_tiling("hot_batch_set_tiling", rows, blocks_per_sm, chunk);
  if (rc != HOT_OK) return rc;
  if (!(group_pairs >= 0) || !std::isfinite(group_pairs))
    return fail(HOT_EINVAL, "hot_batch_set_tiling: group_pairs must be finite and >= 0");
  b->rows = rows ? rows : hot::kRowsMax;
  b->bps = blocks_per_sm;
  b->chunk = chunk ? chunk : hot::kChunk;
  b->group_pairs = group_pairs > 0 ? group_pairs : 67108864.0;
  return batch_schedule(b);
}

int hot_batch_get_tiling(const hot_batch *b, int *rows, int *blocks_per_sm, int *chunk, double *group_pairs,
                         int *groups) {
  if (!b) return fail(HOT_EINVAL, "hot_batch_get_tiling: NULL batch");
  if (rows) *rows = b->rows;
  if (blocks_per_sm) *blocks_per_sm = b->bps > 0 ? std::min(b->bps, b->per_sm_max) : b->per_sm_max;
  if (chunk) *chunk = b->chunk;
  if (group_pairs) *group_pairs = b->group_pairs;
  if (groups) *groups = (int)(b->precision == HOT_PREC_TENSOR ? b->chains.size() : b->groups.size());
  return HOT_OK;
}

int hot_batch_gsw(hot_batch *b, int iters) {
  if (!b) return fail(HOT_EINVAL, "hot_batch_gsw: NULL batch");
  if (iters < 0) return fail(HOT_EINVAL, "hot_batch_gsw: iters = %d < 0", iters);
  const std::vector<double> limits = batch_limits(b);
  for (auto &g : b->graphs)
    if (g.iters == iters && g.limits == limits) {
      const int rc = batch_after_members(b);
      if (rc != HOT_OK) return rc;
      HOT_CUDA(cudaGraphLaunch(g.exec, b->st));
      for (auto *c : b->ctx) {
        c->have_fields = true;
        c->u_valid = false;  // the batch kernels wrote the phases
      }
      b->ran = true;
      return HOT_OK;
    }
  if (!b->cap) HOT_CUDA(cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking));
  if (b->graphs.size() >= 8) {
    cudaGraphExecDestroy(b->graphs.front().exec);
    b->graphs.erase(b->graphs.begin());
  }
  cudaStream_t user = b->st;
  HOT_CUDA(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal));
  b->st = b->cap;
  int rc = batch_enqueue(b, iters);
  b->st = user;
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(b->cap, &graph);
  if (rc != HOT_OK) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return fail(HOT_ECUDA, "hot_batch_gsw: graph capture: %s", cudaGetErrorString(e));
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return fail(HOT_ECUDA, "hot_batch_gsw: graph instantiation: %s", cudaGetErrorString(e));
  b->graphs.push_back({iters, limits, exec});
  rc = batch_after_members(b);
  if (rc != HOT_OK) return rc;
  HOT_CUDA(cudaGraphLaunch(exec, b->st));
  for (auto *c : b->ctx) {
    c->have_fields = true;
    c->u_valid = false;  // the batch kernels wrote the phases
  }
  b->ran = true;
  return HOT_OK;
}

int hot_batch_autotune(hot_batch *b, int iters, int *rows, int *blocks_per_sm, int *chunk, double *us_per_iter) {
  if (!b) return fail(HOT_EINVAL, "hot_batch_autotune: NULL batch");
  if (b->precision == HOT_PREC_TENSOR) return fail(HOT_EINVAL, "hot_batch_autotune: a HOT_PREC_TENSOR batch has no tiling");
  if (iters < 1) return fail(HOT_EINVAL, "hot_batch_autotune: iters = %d < 1", iters);
  std::vector<Saved> saved(b->count);
  int rc = batch_after_members(b);
  for (int h = 0; rc == HOT_OK && h < b->count; h++) rc = save_state(b->ctx[h], saved[h], b->st);
  if (rc != HOT_OK) return rc;
  auto restore = [&]() {
    for (int h = 0; h < b->count; h++) {
      const int r = restore_state(b->ctx[h], saved[h], b->st);
      if (r != HOT_OK) return r;
    }
    return (int)HOT_OK;
  };
  Tiling best = {b->rows, b->bps > 0 ? std::min(b->bps, b->per_sm_max) : b->per_sm_max, b->chunk, 1};
  double best_us = 0;
  const double gp = b->group_pairs;
  rc = tune_tiling(
      kMaxBlocksPerSm, best, best_us, [&](const Tiling &t) { return hot_batch_set_tiling(b, t.rows, t.bps, t.chunk, gp); },
      [&](double *us) { return time_runs(b->st, iters, us, restore, [&]() { return hot_batch_gsw(b, iters); }); });
  const int rc2 = restore();
  cudaStreamSynchronize(b->st);
  for (auto *c : b->ctx) {
    c->have_fields = false;
    c->u_valid = false;
  }
  b->ran = false;
  if (rc != HOT_OK) return rc;
  if (rc2 != HOT_OK) return rc2;
  if (rows) *rows = best.rows;
  if (blocks_per_sm) *blocks_per_sm = best.bps;
  if (chunk) *chunk = best.chunk;
  if (us_per_iter) *us_per_iter = best_us;
  return HOT_OK;
}

int hot_batch_latency(hot_batch *b, double *ms, int count) {
  if (!b || !ms) return fail(HOT_EINVAL, "hot_batch_latency: NULL argument");
  if (count != b->count) return fail(HOT_EINVAL, "hot_batch_latency: count = %d, the batch has %d", count, b->count);
  if (!b->ran) return fail(HOT_ESTATE, "hot_batch_latency: no hot_batch_gsw since the batch was (re)scheduled");
  std::vector<unsigned long long> t(count + 1);
  HOT_CUDA(cudaMemcpyAsync(t.data(), b->stamps, sizeof(unsigned long long) * (count + 1), cudaMemcpyDeviceToHost, b->st));
  HOT_CUDA(cudaStreamSynchronize(b->st));
  for (int h = 0; h < count; h++) ms[h] = (double)(long long)(t[h] - t[count]) * 1e-6;
  return HOT_OK;
}

void hot_batch_destroy(hot_batch *b) {
  if (!b) return;
  cudaStreamSynchronize(b->st);
  batch_free(b);
  delete b;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// SFU throughput probe (hot_sfu_rate).
namespace {

template <int OP>
__global__ void __launch_bounds__(1024) sfu_rate_kernel(float *out, long long *cycles, int iters, float step) {
  float acc[8], x[8];
#pragma unroll
  for (int i = 0; i < 8; i++) {
    x[i] = 0.37f * i + 1e-3f * (threadIdx.x & 63) - 3.0f;
    acc[i] = 0.f;
  }
  __syncthreads();
  const long long t0 = clock64();
  for (int it = 0; it < iters; it++) {
#pragma unroll
    for (int i = 0; i < 8; i++) {
      if (OP != 3) x[i] += step;  // a new argument every iteration
      if (OP == 0) {
        acc[i] = fmaf(hot::sin_approx(x[i]), hot::cos_approx(x[i]), acc[i]);
      } else if (OP == 1) {
        acc[i] += hot::sin_approx(x[i]);
      } else if (OP == 2) {
        float y;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x[i] * 0.001f));
        acc[i] += y;
      } else {
        acc[i] = fmaf(acc[i], 0.999f, x[i]);  // FP32 FMA pipe: 8 independent chains
      }
    }
  }
  __syncthreads();
  const long long t1 = clock64();
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 8; i++) s += acc[i];
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
  if (threadIdx.x == 0) cycles[blockIdx.x] = t1 - t0;
}

}  // namespace

extern "C" int hot_tc_shape(int width, int height, int M, int sms, int *shape) {
  if (width < 1 || height < 1 || M < 1 || sms < 1 || !shape)
    return fail(HOT_EINVAL, "hot_tc_shape: invalid argument");
  const hot_tc::Shape sh = hot_tc::shape_for(width, height, M, sms);
  const int v[9] = {sh.bn_back, sh.bn_fwd, sh.fwd_splits, sh.fwd_cps, sh.Kb, sh.Kf, sh.rows_h, sh.rows_b, sh.rows_f};
  for (int i = 0; i < 9; i++) shape[i] = v[i];
  return HOT_OK;
}

extern "C" int hot_tc_gemm(int rows, int cols, int K, const float *A, const float *B, float *C, int tile_n,
                           int operands, void *cuda_stream) {
  if (rows < 1 || cols < 1 || K < 1) return fail(HOT_EINVAL, "hot_tc_gemm: sizes %d x %d x %d", rows, cols, K);
  if (!A || !B || !C) return fail(HOT_EINVAL, "hot_tc_gemm: NULL argument");
  if (tile_n != 32 && tile_n != 64 && tile_n != 128 && tile_n != 256)
    return fail(HOT_EINVAL, "hot_tc_gemm: tile_n = %d not 32, 64, 128 or 256", tile_n);
  if (operands != HOT_TC_TF32 && operands != HOT_TC_FP16)
    return fail(HOT_EINVAL, "hot_tc_gemm: operands = %d not HOT_TC_TF32 or HOT_TC_FP16", operands);
  if ((long long)rows * K >= (1LL << 31) || (long long)cols * K >= (1LL << 31) || (long long)rows * cols >= (1LL << 31))
    return fail(HOT_EINVAL, "hot_tc_gemm: operands of 2^31 elements or more");
  int timed_out = 0;
  const char *what = "";
  const cudaError_t e = hot_tc::gemm(rows, cols, K, A, B, C, tile_n, operands == HOT_TC_FP16 ? 1 : 0,
                                     static_cast<cudaStream_t>(cuda_stream), &timed_out, &what);
  if (e != cudaSuccess)
    return fail(e == cudaErrorMemoryAllocation ? HOT_ENOMEM : HOT_ECUDA, "hot_tc_gemm: %s: %s", what,
                cudaGetErrorString(e));
  if (timed_out) return fail(HOT_ETIMEOUT, "hot_tc_gemm: a bounded device-side wait ran out");
  return HOT_OK;
}

extern "C" int hot_sfu_rate(int op, double *per_clk_per_sm, int *sms) {
  if (!per_clk_per_sm || op < 0 || op > 3) return fail(HOT_EINVAL, "hot_sfu_rate: invalid argument");
  int dev = 0, n = 0;
  HOT_CUDA(cudaGetDevice(&dev));
  HOT_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
  const int threads = 1024, iters = 2048;
  float *out = nullptr;
  long long *cyc = nullptr;
  int rc = dalloc(&out, (size_t)n * threads);
  if (rc == HOT_OK) rc = dalloc(&cyc, (size_t)n);
  std::vector<long long> h(n);
  for (int rep = 0; rc == HOT_OK && rep < 2; rep++) {  // the first run warms up
    if (op == 0) sfu_rate_kernel<0><<<n, threads>>>(out, cyc, iters, 1e-4f);
    else if (op == 1) sfu_rate_kernel<1><<<n, threads>>>(out, cyc, iters, 1e-4f);
    else if (op == 2) sfu_rate_kernel<2><<<n, threads>>>(out, cyc, iters, 1e-4f);
    else sfu_rate_kernel<3><<<n, threads>>>(out, cyc, iters, 1e-4f);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(h.data(), cyc, sizeof(long long) * n, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) rc = fail(HOT_ECUDA, "hot_sfu_rate: %s", cudaGetErrorString(e));
  }
  dfree(out);
  dfree(cyc);
  if (rc != HOT_OK) return rc;
  double mean = 0.0;
  for (long long v : h) mean += (double)v;
  mean /= n;
  const double results = (op == 0 ? 2.0 : 1.0) * threads * (double)iters * 8;  // per block (= per SM)
  *per_clk_per_sm = results / mean;
  if (sms) *sms = n;
  return HOT_OK;
}

// ---------------------------------------------------------------------------------------------
// Allocation-free trap-field evaluation (hot_field_noalloc): all working memory is carved out
// of one file-scope device array, whose device address is looked up once per device.
namespace {

__device__ __align__(256) unsigned char g_noalloc_scratch[HOT_NOALLOC_SCRATCH_BYTES];

constexpr int kNoallocMaxDevices = 64;

// What the first call on a device sets up: the scratch array's device address, the
// step kernels' shared-memory limit and the resident blocks per SM of the work schedule.
struct NoallocDevice {
  unsigned char *base;  // NULL until set up
  int sms, per_sm;
};
std::mutex g_noalloc_mutex;
NoallocDevice g_noalloc_dev[kNoallocMaxDevices];

// Set-up of device dev (the current device), once: the device address of the scratch array
// (in host code its name is a host-side stand-in, not a device address), the dynamic
// shared-memory limit of the forward-field kernels and the occupancy that sizes the grid
// (the same per-SM block count a context's schedule uses; it does not depend on M).
int noalloc_device(int dev, NoallocDevice *out) {
  if (dev < 0 || dev >= kNoallocMaxDevices) return fail(HOT_EINVAL, "hot_field_noalloc: device %d beyond %d", dev, kNoallocMaxDevices);
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  NoallocDevice &d = g_noalloc_dev[dev];
  if (!d.base) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail(HOT_ECUDA, "hot_field_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
    const int fwd = hot::step_smem_bytes(1, false), step = hot::step_smem_bytes(1, true);
    HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd));
    HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd));
    HOT_CUDA(cudaFuncSetAttribute(hot::gsw_step_kernel<true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, step));
    int sms = 0, per_sm = 0;
    HOT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    HOT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hot::gsw_step_kernel<true, true, true>, hot::kThreads, step));
    d.sms = sms;
    d.per_sm = per_sm < 1 ? 1 : per_sm;
    d.base = static_cast<unsigned char *>(p);
  }
  *out = d;
  return HOT_OK;
}

// Number of sub-tiles block b of G receives: its run of the U = strips x H row segments,
// cut at strip ends and into pieces of at most kRowsMax rows (the rule of build_schedule).
__host__ __device__ int noalloc_block_subtiles(long long U, int G, int H, int b, hot::SubTile *out) {
  long long s = U * b / G;
  const long long s1 = U * (b + 1) / G;
  int n = 0;
  while (s < s1) {
    const int strip = (int)(s / H), row = (int)(s % H);
    const long long run_end = (s1 < (long long)(strip + 1) * H) ? s1 : (long long)(strip + 1) * H;
    const int L = (int)(run_end - s);
    const int nsub = (L + hot::kRowsMax - 1) / hot::kRowsMax;
    for (int i = 0; out && i < nsub; i++) {
      const int r0 = row + (int)((long long)L * i / nsub), r1 = row + (int)((long long)L * (i + 1) / nsub);
      out[n + i] = {strip * hot::kTileW, r0, r1 - r0, 0};
    }
    n += nsub;
    s = run_end;
  }
  return n;
}

// Writes the schedule (sub-tiles and per-block first index) for G blocks.
__global__ void noalloc_schedule_kernel(long long U, int G, int H, hot::SubTile *sub, int *first) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b > G) return;
  int f = 0;
  for (int q = 0; q < b; q++) f += noalloc_block_subtiles(U, G, H, q, nullptr);
  first[b] = f;
  if (b < G) noalloc_block_subtiles(U, G, H, b, sub + f);
}

// a_m, b_m, c_m of Eq. 2 in turns per pixel index, from device trap coordinates.
__global__ void noalloc_abc_kernel(int M, const double *xyz, double lin, double quad, double *abc) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < M) {
    abc[3 * m] = xyz[3 * m] * lin;
    abc[3 * m + 1] = xyz[3 * m + 1] * lin;
    abc[3 * m + 2] = xyz[3 * m + 2] * quad;
  }
}

// Fixed-point field sums and metrics of the step kernel -> the caller's double outputs.
__global__ void noalloc_out_kernel(int M, const long long *Vsum, float, int width, int height, int fx_shift,
                                   const float *metrics, double *V, double *eu) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  const double inv = 1.0 / ((double)width * (double)height * ldexp(1.0, fx_shift));
  if (m < M) {
    V[2 * m] = (double)Vsum[m] * inv;
    V[2 * m + 1] = (double)Vsum[M + m] * inv;
  }
  if (eu && m == 0) {
    eu[0] = metrics[0];
    eu[1] = metrics[1];
  }
}

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

}  // namespace

extern "C" int hot_field_noalloc(int width, int height, double pitch_m, double wavelength_m, double focal_m,
                                 int M, const double *xyz_m, const float *phi, int precision, double *V,
                                 double *eu, void *cuda_stream) {
  if (width < 1 || height < 1 || (long long)width * height >= (1LL << 31))
    return fail(HOT_EINVAL, "hot_field_noalloc: invalid size %d x %d", width, height);
  if (!finite_pos(pitch_m) || !finite_pos(wavelength_m) || !finite_pos(focal_m))
    return fail(HOT_EINVAL, "hot_field_noalloc: pitch, wavelength and focal length must be finite and > 0");
  if (M < 1 || M > HOT_MAX_TRAPS) return fail(HOT_EINVAL, "hot_field_noalloc: M = %d not in [1, %d]", M, HOT_MAX_TRAPS);
  if (!xyz_m || !phi || !V) return fail(HOT_EINVAL, "hot_field_noalloc: NULL input or output");
  if (precision != HOT_PREC_ACCURATE && precision != HOT_PREC_FAST)
    return fail(HOT_EINVAL, "hot_field_noalloc: unknown precision %d", precision);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const bool fast = precision == HOT_PREC_FAST;
  int dev = 0;
  HOT_CUDA(cudaGetDevice(&dev));
  NoallocDevice d = {};
  int rc = noalloc_device(dev, &d);
  if (rc != HOT_OK) return rc;

  // Work schedule: identical to a context's (one wave of step-kernel blocks).
  const int strips = (width + hot::kTileW - 1) / hot::kTileW;
  const long long U = (long long)strips * height;
  const int G = (int)std::min<long long>((long long)d.sms * d.per_sm, U);
  int n_sub = 0;
  for (int b = 0; b < G; b++) n_sub += noalloc_block_subtiles(U, G, height, b, nullptr);

  // Carve the scratch array.
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t o = off; off += align256(bytes); return o; };
  const size_t o_abc = take(sizeof(double) * 3 * M);
  const size_t o_xt = take(sizeof(float) * (size_t)M * width), o_xr = take(sizeof(float) * (size_t)M * width);
  const size_t o_yt = take(sizeof(float) * (size_t)M * height), o_yr = take(sizeof(float) * (size_t)M * height);
  const size_t o_sub = take(sizeof(hot::SubTile) * n_sub), o_first = take(sizeof(int) * (G + 1));
  const size_t o_acc = take(sizeof(unsigned long long) * 6 * M), o_vsum = take(sizeof(long long) * 2 * M);
  const size_t o_met = take(sizeof(float) * 2);
  if (off > HOT_NOALLOC_SCRATCH_BYTES)
    return fail(HOT_EINVAL, "hot_field_noalloc: %d x %d pixels and %d traps need %zu bytes of scratch, the limit is %u",
                width, height, M, off, (unsigned)HOT_NOALLOC_SCRATCH_BYTES);
  unsigned char *const base = d.base;
  double *abc = reinterpret_cast<double *>(base + o_abc);
  float *Xt = reinterpret_cast<float *>(base + o_xt), *Xr = reinterpret_cast<float *>(base + o_xr);
  float *Yt = reinterpret_cast<float *>(base + o_yt), *Yr = reinterpret_cast<float *>(base + o_yr);
  hot::SubTile *d_sub = reinterpret_cast<hot::SubTile *>(base + o_sub);
  int *d_first = reinterpret_cast<int *>(base + o_first);
  unsigned long long *acc = reinterpret_cast<unsigned long long *>(base + o_acc);
  long long *Vsum = reinterpret_cast<long long *>(base + o_vsum);
  float *metrics = reinterpret_cast<float *>(base + o_met);

  // The schedule is written on the device; the accumulators start at zero (the array keeps
  // whatever the previous call left).
  noalloc_schedule_kernel<<<(G + 1 + 255) / 256, 256, 0, st>>>(U, G, height, d_sub, d_first);
  HOT_CUDA(cudaGetLastError());
  HOT_CUDA(cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 6 * M, st));

  const double lin = pitch_m / (wavelength_m * focal_m);
  const double quad = pitch_m * pitch_m / (2.0 * wavelength_m * focal_m * focal_m);
  noalloc_abc_kernel<<<(M + 255) / 256, 256, 0, st>>>(M, xyz_m, lin, quad, abc);
  HOT_CUDA(cudaGetLastError());
  const long long total = (long long)M * (width + height);
  const int tb = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  hot::build_tables_kernel<<<tb, 256, 0, st>>>(width, height, height, 0, M, abc, Xt, Yt, Xr, Yr);
  HOT_CUDA(cudaGetLastError());

  int bits = 0;
  while ((1LL << bits) < (long long)width * height) bits++;
  const int fx_shift = 61 - bits;
  hot::StepArgs a = {};  // the forward-only kernel reads no weights, coefficients or separable tables
  a.W = width;
  a.H = height;
  a.M = M;
  a.chunk = hot::kChunk;
  a.copies = 1;
  a.sub = d_sub;
  a.first = d_first;
  a.X = fast ? Xr : Xt;
  a.Y = fast ? Yr : Yt;
  a.phi = const_cast<float *>(phi);  // the forward-only kernel reads the phases and writes none
  a.acc_in = acc + 4 * (size_t)M;
  a.acc_out = acc;
  a.acc_clear = acc + 2 * (size_t)M;
  a.fx_scale = ldexpf(1.0f, fx_shift);
  a.inv_fx_n = (float)(1.0 / ((double)width * (double)height * ldexp(1.0, fx_shift)));
  a.angle_units = fast ? 1.0f : 0.15915494309189535f;
  a.angle_eta = fast ? hot::kFastEta : 0.0f;
  const int smem = hot::step_smem_bytes(M, false);
  if (fast) hot::gsw_step_kernel<true, false, true><<<G, hot::kThreads, smem, st>>>(a);
  else hot::gsw_step_kernel<false, false, true><<<G, hot::kThreads, smem, st>>>(a);
  HOT_CUDA(cudaGetLastError());
  hot::FinalizeArgs f = {};  // no weights to move (w_src = w_dst = NULL), no completion stamp
  f.M = M;
  f.copies = 1;
  f.acc = acc;
  f.acc_all = acc;
  f.Vsum = Vsum;
  f.metrics = metrics;
  f.inv_fx_n = a.inv_fx_n;
  hot::gsw_finalize_kernel<<<1, hot::kFinalizeThreads, 0, st>>>(f);
  HOT_CUDA(cudaGetLastError());
  noalloc_out_kernel<<<(M + 255) / 256, 256, 0, st>>>(M, Vsum, a.inv_fx_n, width, height, fx_shift, metrics, V, eu);
  HOT_CUDA(cudaGetLastError());
  return HOT_OK;
}
