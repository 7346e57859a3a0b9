// tc.cu -- host side of the separable GSW iteration on the tensor cores (see tc_kernels.cuh).
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "tc.h"
#include "tc_kernels.cuh"

namespace hot_tc {

// Operand type of the GSW iteration's GEMMs: FP16 halves (kind::f16, twice the TF32 rate; the
// operands are unit phasors and coefficients normalised to max |c_m| = 1).
constexpr int kPlanOp = tc::kOpF16;
constexpr int kSliceK = tc::slice_k<kPlanOp>();
constexpr size_t kElem = tc::Op<kPlanOp>::kBytes;

struct Plan {
  int W = 0, H = 0, M = 0;
  // K of the back GEMM (2M) and of the forward GEMM (2W), padded to a K slice: each component has
  // half of it, in rows of ldb, ldu elements (whole slices)
  int Kb = 0, Kf = 0, ldb = 0, ldu = 0;
  int rows_h = 0;                   // H padded to the tile height (rows of P and U)
  int bn_back = 64, bn_fwd = 64;    // tile widths of the back and forward GEMMs
  int rows_b = 0, rows_f = 0;       // 2W and 2M padded to the tile width: B has half as many rows per component
  int fwd_splits = 1, fwd_cps = 1;  // K splits of the forward GEMM, units (half slices) per split
  int sms = 0;
  // operands by component and part: back and forward B (constant), P, U
  __half *bb[2][2] = {}, *bf[2][2] = {}, *p[2][2] = {}, *u[2][2] = {};
  float2 *YT = nullptr;
  const float2 *Xc = nullptr, *Yc = nullptr;  // the context's complex tables [M][W], [M][H]
  tc::Maps back{}, fwd{};
};

namespace {

int round_up(int x, int m) { return (x + m - 1) / m * m; }

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// A row-major operand matrix [rows][inner] of OP elements (inner a multiple of one K slice, base
// 16-byte aligned) read in boxes of one 128-byte K slice x box_rows with 128-byte swizzle; rows
// is a multiple of box_rows: no box leaves the matrix but the last of a K range that starts inside
// a slice, whose second half is filled and not used.
template <int OP>
cudaError_t encode(CUtensorMap *map, const void *base, int inner, int rows, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)inner * tc::Op<OP>::kBytes};
  const cuuint32_t box[2] = {(cuuint32_t)tc::slice_k<OP>(), (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUtensorMapDataType dt = OP == tc::kOpF16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  const CUresult r = fn(map, dt, 2, const_cast<void *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, int block, int smem, cudaStream_t st, bool pdl,
                   Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int BN, int EPI, int OP = kPlanOp>
cudaError_t set_smem() {
  return cudaFuncSetAttribute(tc::tc_gemm_kernel<BN, EPI, OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              tc::Cfg<BN>::kSmem);
}

template <typename T>
cudaError_t alloc(T **p, size_t count) {
  return cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T));
}
cudaError_t alloc_bytes(void **p, size_t bytes) { return cudaMalloc(p, bytes); }

template <int BN, int EPI, int OP = kPlanOp>
cudaError_t launch_gemm(const tc::Maps &maps, const tc::GemmArgs &g, dim3 grid, cudaStream_t st, bool pdl) {
  return launch(tc::tc_gemm_kernel<BN, EPI, OP>, grid, tc::Cfg<BN>::kThreads, tc::Cfg<BN>::kSmem, st, pdl, maps, g);
}

template <int EPI>
cudaError_t launch_gemm_bn(int bn, const tc::Maps &maps, const tc::GemmArgs &g, dim3 grid, cudaStream_t st, bool pdl) {
  return bn == 256 ? launch_gemm<256, EPI>(maps, g, grid, st, pdl)
         : bn == 128 ? launch_gemm<128, EPI>(maps, g, grid, st, pdl)
         : bn == 64  ? launch_gemm<64, EPI>(maps, g, grid, st, pdl)
                     : launch_gemm<32, EPI>(maps, g, grid, st, pdl);
}

// CTAs share K in `splits` ranges of `cps` units each (>= 1, the last not empty) when the tiles alone
// leave SMs idle.
void split_range(int tiles, int units, int sms, int *cps, int *splits) {
  const int want = std::max(1, std::min(units, sms / std::max(tiles, 1)));
  *cps = (units + want - 1) / want;
  *splits = (units + *cps - 1) / *cps;
}

// Tile width of a GEMM with `rows` x `cols` outputs and `units` half slices of K: the one with the least
// estimated time, waves of CTAs (one per SM) x (units of a CTA x time of a unit + time of the rest).
// Times in 10 ns, fitted to both GEMMs at 16 sizes and every width (512 .. 1920 columns, 8 .. 1500 traps):
// a unit of 12 MMAs takes 0.7 us up to 128 columns (issuing both components' MMAs turn about, or waiting
// without the timer, changed nothing) and 0.95 us at 256 (the MMAs' own rate);
// the rest (launch, pipeline fill, epilogue) grows with the width, more so where the epilogue forms
// phases.  Against the widest tiles that still occupied 4 of 5 SMs, an iteration of 1281 x 515 with
// 1500 traps goes from 166 to 87 us, 512^2 with 400 from 33.6 to 26.0, 1000 x 700 with 300 from 38.7 to
// 29.4; 1920 x 1152 with 1000 keeps its 256.
// Widths that add more than 12.5% of padding to what 32 columns need are not taken.
int pick_width(int rows, int cols, int units, int sms, bool forward) {
  struct Width {
    int bn, unit, back, fwd;
  };
  static constexpr Width kWidths[] = {{256, 95, 950, 630}, {128, 70, 580, 440}, {64, 74, 380, 340}, {32, 73, 290, 290}};
  int best = 32;
  long long least = -1;
  for (const Width &w : kWidths) {
    if (8 * round_up(cols, w.bn) > 9 * round_up(cols, 32)) continue;
    const int tiles = ((rows + tc::kBM - 1) / tc::kBM) * ((cols + w.bn - 1) / w.bn);
    int cps = units, splits = 1;
    if (forward) split_range(tiles, units, sms, &cps, &splits);
    const long long waves = ((long long)tiles * splits + sms - 1) / sms;
    const long long cost = waves * ((long long)cps * w.unit + (forward ? w.fwd : w.back));
    if (least < 0 || cost < least) {
      least = cost;
      best = w.bn;
    }
  }
  return best;
}

}  // namespace

Shape shape_for(int W, int H, int M, int sms) {
  Shape sh;
  sh.Kb = round_up(2 * M, kSliceK);
  sh.Kf = round_up(2 * W, kSliceK);
  sh.rows_h = round_up(H, tc::kBM);
  sh.bn_back = pick_width(H, 2 * W, sh.Kb / kSliceK, sms, false);
  sh.bn_fwd = pick_width(H, 2 * M, sh.Kf / kSliceK, sms, true);
  sh.rows_b = round_up(2 * W, sh.bn_back);
  sh.rows_f = round_up(2 * M, sh.bn_fwd);
  // forward GEMM: the K range split over CTAs so that the tiles fill the SMs about once
  split_range((sh.rows_h / tc::kBM) * (sh.rows_f / sh.bn_fwd), sh.Kf / kSliceK, sms, &sh.fwd_cps, &sh.fwd_splits);
  return sh;
}

void plan_destroy(Plan *p) {
  if (!p) return;
  for (auto *set : {&p->bb, &p->bf, &p->p, &p->u})
    for (auto &c : *set)
      for (__half *b : c)
        if (b) cudaFree(b);
  if (p->YT) cudaFree(p->YT);
  delete p;
}

cudaError_t plan_refresh(Plan *p, cudaStream_t st) {
  tc::TableArgs t = {};
  t.W = p->W;
  t.H = p->H;
  t.M = p->M;
  t.Kp = p->Kb / 2;
  t.ldb = p->ldb;
  t.ldu = p->ldu;
  t.rows_b = p->rows_b / 2;
  t.rows_f = p->rows_f / 2;
  t.Xc = p->Xc;
  t.Yc = p->Yc;
  for (int k = 0; k < 4; k++) {
    t.b[k >> 1][k & 1] = p->bb[k >> 1][k & 1];
    t.f[k >> 1][k & 1] = p->bf[k >> 1][k & 1];
  }
  t.YT = p->YT;
  const long long total =
      (long long)t.rows_b * (t.ldb / 2) + (long long)t.rows_f * (t.ldu / 2) + (long long)p->H * (t.Kp / 2);
  const int blocks = (int)std::min<long long>((total + 255) / 256, 8LL * p->sms);
  return launch(tc::tc_tables_kernel, dim3(blocks), 256, 0, st, false, t);
}

cudaError_t plan_create(Plan **out, int W, int H, int M, const float2 *Xc, const float2 *Yc, cudaStream_t st,
                        const char **what) {
  *out = nullptr;
  Plan *p = new Plan;
  p->W = W;
  p->H = H;
  p->M = M;
  p->Xc = Xc;
  p->Yc = Yc;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, dev);
  const Shape sh = shape_for(W, H, M, p->sms);
  p->Kb = sh.Kb;
  p->Kf = sh.Kf;
  p->rows_h = sh.rows_h;
  p->bn_back = sh.bn_back;
  p->bn_fwd = sh.bn_fwd;
  p->rows_b = sh.rows_b;
  p->rows_f = sh.rows_f;
  p->fwd_cps = sh.fwd_cps;
  p->fwd_splits = sh.fwd_splits;
  *what = "allocating the tensor-core operands";
  p->ldb = round_up(p->Kb / 2, kSliceK);
  p->ldu = round_up(p->Kf / 2, kSliceK);
  const size_t nb = (size_t)(p->rows_b / 2) * p->ldb, nf = (size_t)(p->rows_f / 2) * p->ldu;
  const size_t np = (size_t)p->rows_h * p->ldb, nu = (size_t)p->rows_h * p->ldu;
  for (int k = 0; k < 4; k++) {
    const int c = k >> 1, part = k & 1;
    if (e == cudaSuccess) e = alloc(&p->bb[c][part], nb);
    if (e == cudaSuccess) e = alloc(&p->bf[c][part], nf);
    if (e == cudaSuccess) e = alloc(&p->p[c][part], np);
    if (e == cudaSuccess) e = alloc(&p->u[c][part], nu);
    // padding rows and columns of P and U stay zero (the kernels write only the image)
    if (e == cudaSuccess) e = cudaMemsetAsync(p->p[c][part], 0, np * kElem, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(p->u[c][part], 0, nu * kElem, st);
  }
  if (e == cudaSuccess) e = alloc(&p->YT, (size_t)H * (p->Kb / 2));
  if (e == cudaSuccess) {
    *what = "building the tensor-core operand tables";
    e = plan_refresh(p, st);
  }
  if (e == cudaSuccess) {
    *what = "encoding the tensor maps";
    for (int k = 0; k < 4; k++) {
      const int c = k >> 1, part = k & 1;
      if (e == cudaSuccess) e = encode<kPlanOp>(&p->back.a[c][part], p->p[c][part], p->ldb, p->rows_h, tc::kBM);
      if (e == cudaSuccess) e = encode<kPlanOp>(&p->back.b[c][part], p->bb[c][part], p->ldb, p->rows_b / 2, p->bn_back / 2);
      if (e == cudaSuccess) e = encode<kPlanOp>(&p->fwd.a[c][part], p->u[c][part], p->ldu, p->rows_h, tc::kBM);
      if (e == cudaSuccess) e = encode<kPlanOp>(&p->fwd.b[c][part], p->bf[c][part], p->ldu, p->rows_f / 2, p->bn_fwd / 2);
    }
  }
  if (e == cudaSuccess) {
    *what = "setting the tensor-core kernels' shared memory";
    e = set_smem<32, tc::kEpiBack>();
    if (e == cudaSuccess) e = set_smem<64, tc::kEpiBack>();
    if (e == cudaSuccess) e = set_smem<128, tc::kEpiBack>();
    if (e == cudaSuccess) e = set_smem<256, tc::kEpiBack>();
    if (e == cudaSuccess) e = set_smem<32, tc::kEpiFwd>();
    if (e == cudaSuccess) e = set_smem<64, tc::kEpiFwd>();
    if (e == cudaSuccess) e = set_smem<128, tc::kEpiFwd>();
    if (e == cudaSuccess) e = set_smem<256, tc::kEpiFwd>();
  }
  if (e != cudaSuccess) {
    cudaStreamSynchronize(st);
    plan_destroy(p);
    return e;
  }
  *out = p;
  return cudaSuccess;
}

namespace {

// The forward GEMM of a step: T = U X^H, weighted and added into s.acc_out.
cudaError_t forward_gemm(Plan *p, const Step &s, cudaStream_t st, bool chain, int *kernels) {
  tc::GemmArgs g = {};
  g.rows = p->H;
  g.cols = 2 * p->M;
  g.k_chunks = p->Kf / kSliceK;
  g.chunks_per_split = p->fwd_cps;
  g.limit_ns = s.limit_ns;
  g.err = s.err;
  g.W = p->W;
  g.H = p->H;
  g.M = p->M;
  g.Kp = p->Kb / 2;
  g.YT = p->YT;
  g.acc_out = s.acc_out;
  g.fx_scale = s.fx_scale;
  const dim3 grid(p->rows_f / p->bn_fwd, p->rows_h / tc::kBM, p->fwd_splits);
  const cudaError_t e = launch_gemm_bn<tc::kEpiFwd>(p->bn_fwd, p->fwd, g, grid, st, chain);
  if (e == cudaSuccess) ++*kernels;
  return e;
}

}  // namespace

cudaError_t launch_forward(Plan *p, const Step &s, cudaStream_t st, bool pdl, bool chain, int *kernels) {
  *kernels = 0;
  const long long N = (long long)p->W * p->H;
  const int blocks = (int)std::min<long long>((N + 511) / 512, 8LL * p->sms);
  tc::PhaseArgs a = {};
  a.W = p->W;
  a.H = p->H;
  a.ldu = p->ldu;
  a.phi = s.phi;
  for (int k = 0; k < 4; k++) a.u[k >> 1][k & 1] = p->u[k >> 1][k & 1];
  a.acc_clear = s.acc_clear;
  a.n_clear = 2 * s.M;
  const cudaError_t e = launch(tc::tc_phase_kernel, dim3(blocks), 256, 0, st, pdl, a);
  if (e != cudaSuccess) return e;
  ++*kernels;
  return forward_gemm(p, s, st, chain, kernels);
}

cudaError_t launch_iteration(Plan *p, const Step &s, cudaStream_t st, bool pdl, bool chain, int *kernels) {
  *kernels = 0;
  tc::PrepArgs pa = {};
  pa.H = p->H;
  pa.M = p->M;
  pa.Kp = p->Kb / 2;
  pa.ldb = p->ldb;
  pa.acc_in = s.acc_in;
  pa.acc_clear = s.acc_clear;
  pa.w_in = s.w_in;
  pa.w_out = s.w_out;
  pa.YT = p->YT;
  for (int k = 0; k < 4; k++) pa.p[k >> 1][k & 1] = p->p[k >> 1][k & 1];
  pa.inv_fx_n = s.inv_fx_n;
  pa.trace = s.trace;
  // blocks take even shares of the rows (each block also forms all M coefficients)
  const long long pairs = (long long)p->H * (pa.Kp / 2);
  const int prep_blocks =
      (int)std::max<long long>(1, std::min<long long>({(pairs + 255) / 256, 2LL * p->sms, (long long)p->H}));
  cudaError_t e = launch(tc::tc_prep_kernel, dim3(prep_blocks), tc::kPrepThreads, (int)(sizeof(float2) * p->M), st, pdl, pa);
  if (e != cudaSuccess) return e;
  ++*kernels;
  tc::GemmArgs g = {};
  g.rows = p->H;
  g.cols = 2 * p->W;
  g.k_chunks = p->Kb / kSliceK;
  g.chunks_per_split = g.k_chunks;
  g.limit_ns = s.limit_ns;
  g.err = s.err;
  g.W = p->W;
  g.H = p->H;
  g.ldu = p->ldu;
  g.phi = s.phi;
  for (int k = 0; k < 4; k++) g.u[k >> 1][k & 1] = p->u[k >> 1][k & 1];
  const dim3 grid_b(p->rows_b / p->bn_back, p->rows_h / tc::kBM, 1);
  e = launch_gemm_bn<tc::kEpiBack>(p->bn_back, p->back, g, grid_b, st, chain);
  if (e != cudaSuccess) return e;
  ++*kernels;
  return forward_gemm(p, s, st, chain, kernels);
}

namespace {

template <int OP>
cudaError_t gemm_op(int rows, int cols, int K, const float *A, const float *B, float *C, int tile_n, cudaStream_t st,
                    int *timed_out, const char **what) {
  *timed_out = 0;
  constexpr int sk = tc::slice_k<OP>();
  const int Kp = round_up(K, sk), ra = round_up(rows, tc::kBM), rb = round_up(cols, tile_n);
  void *buf[4] = {nullptr, nullptr, nullptr, nullptr};
  int *err = nullptr;
  *what = "allocating the GEMM operands";
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 4 && e == cudaSuccess; i++)
    e = alloc_bytes(&buf[i], (size_t)(i < 2 ? ra : rb) * Kp * tc::Op<OP>::kBytes);
  if (e == cudaSuccess) e = alloc(&err, 1);
  if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), st);
  if (e == cudaSuccess) {
    *what = "splitting the GEMM operands";
    const long long ta = (long long)ra * Kp, tb = (long long)rb * Kp;
    e = launch(tc::tc_split_kernel<OP>, dim3((int)std::min<long long>((ta + 255) / 256, 4096)), 256, 0, st, false, A,
               rows, K, Kp, ta, buf[0], buf[1]);
    if (e == cudaSuccess)
      e = launch(tc::tc_split_kernel<OP>, dim3((int)std::min<long long>((tb + 255) / 256, 4096)), 256, 0, st, false, B,
                 cols, K, Kp, tb, buf[2], buf[3]);
  }
  tc::Maps maps{};
  if (e == cudaSuccess) {
    *what = "encoding the GEMM tensor maps";
    for (int part = 0; part < 2; part++) {
      if (e == cudaSuccess) e = encode<OP>(&maps.a[0][part], buf[part], Kp, ra, tc::kBM);
      if (e == cudaSuccess) e = encode<OP>(&maps.b[0][part], buf[2 + part], Kp, rb, tile_n / 2);
      maps.b[1][part] = maps.b[0][part];
    }
  }
  if (e == cudaSuccess) {
    *what = "running the GEMM";
    tc::GemmArgs g = {};
    g.rows = rows;
    g.cols = cols;
    g.k_chunks = Kp / sk;
    g.chunks_per_split = g.k_chunks;
    g.limit_ns = 2000000000LL;
    g.err = err;
    g.C = C;
    const dim3 grid(rb / tile_n, ra / tc::kBM, 1);
    if (tile_n == 32) {
      e = set_smem<32, tc::kEpiPlain, OP>();
      if (e == cudaSuccess) e = launch_gemm<32, tc::kEpiPlain, OP>(maps, g, grid, st, false);
    } else if (tile_n == 256) {
      e = set_smem<256, tc::kEpiPlain, OP>();
      if (e == cudaSuccess) e = launch_gemm<256, tc::kEpiPlain, OP>(maps, g, grid, st, false);
    } else if (tile_n == 128) {
      e = set_smem<128, tc::kEpiPlain, OP>();
      if (e == cudaSuccess) e = launch_gemm<128, tc::kEpiPlain, OP>(maps, g, grid, st, false);
    } else {
      e = set_smem<64, tc::kEpiPlain, OP>();
      if (e == cudaSuccess) e = launch_gemm<64, tc::kEpiPlain, OP>(maps, g, grid, st, false);
    }
  }
  int flag = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&flag, err, sizeof flag, cudaMemcpyDeviceToHost, st);
  cudaError_t e2 = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = e2;
  *timed_out = flag;
  for (void *b : buf)
    if (b) cudaFree(b);
  if (err) cudaFree(err);
  return e;
}

}  // namespace

cudaError_t gemm(int rows, int cols, int K, const float *A, const float *B, float *C, int tile_n, int operands,
                 cudaStream_t st, int *timed_out, const char **what) {
  return operands == 1 ? gemm_op<tc::kOpF16>(rows, cols, K, A, B, C, tile_n, st, timed_out, what)
                       : gemm_op<tc::kOpTF32>(rows, cols, K, A, B, C, tile_n, st, timed_out, what);
}

}  // namespace hot_tc
