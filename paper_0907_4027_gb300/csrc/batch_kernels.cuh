// batch_kernels.cuh -- the batched GSW step (hot_batch_*): one launch per iteration over the sub-tiles of
// several holograms, with the direct evaluation of every pair's exponential in the accurate and fast
// modes (process_subtile) and the separable step below.
//
// A batch goes on from the phases and weights that its last call left, and with many traps on few
// pixels the iteration amplifies rounding: 512^2 px with 1442 traps, two evaluations whose sums differ by
// 1e-7 are 6e-7 apart in the fields after 5 iterations, 1e-5 after 50, 1e-4 after 125 and up to 9e-4 after 200,
// each of them as far from the 64-bit iteration.  So the batches keep these kernels, their schedule and
// their tables (FP64 cos and sin), and with them the bits of every earlier sequence of calls; the
// register-tiled step (tile_kernels.cuh), which takes 14.8 instead of 34.4 ms for 5 iterations of 8
// holograms of 512^2 to 1920 x 1152 px with up to 2000 traps, is what the members of a batch of one-hologram groups
// run on request (hot_batch_set_tiling, group_pairs <= 1).
#pragma once
#include "gsw_kernels.cuh"

namespace hot {

// Separable step.  Eq. 2 is a sum of a column part and a row part, so every pair's
// exponential factorises: e^{i Delta_j^m} = Xc_m(ix) Yc_m(iy), with both factors tabulated once
// per trap (FP64 cos/sin of the reduced turns, stored as FP32 complex).  Per pair the
// back-projection then takes one complex multiply-add,
//   S_j += Yc_m(iy) [c_m Xc_m(ix)]           (the bracket once per trap and lane),
// and the forward field another,
//   V_m += conj(Xc_m(ix)) sum_iy u_j conj(Yc_m(iy))   with u_j = e^{i phi_j},
// i.e. 8 FP32 FMA per pixel-trap update and no per-pair transcendental function (one sincos
// per pixel and iteration gives u_j from the stored phase).  The coefficients are kept
// complex, c_m = w_m V_m/|V_m| (Sec. 3).
// The work decomposition, staging, reductions and fixed-point sums are the direct kernel's.
constexpr int kSepUsFloats = kRowsMax * kTileW * 2;

__host__ __device__ constexpr int sep_smem_bytes(int chunk) {
  return chunk * (kTileW + kYStride) * 8 + 2 * chunk * 8 + kWarps * kHalfRows * kTileW * 8 + kSepUsFloats * 4;
}

struct SepSmem {
  float2 *Xs, *Ys, *Cs, *Sp, *Us, *C0;
  __device__ __forceinline__ SepSmem(unsigned char *raw, int chunk) {
    Xs = reinterpret_cast<float2 *>(raw);  // [chunk][kTileW]
    Ys = Xs + chunk * kTileW;              // [chunk][kYStride]
    Cs = Ys + chunk * kYStride;            // [chunk]
    Sp = Cs + chunk;                       // [kWarps][kHalfRows][kTileW]
    Us = Sp + kWarps * kHalfRows * kTileW; // [kRowsMax][kTileW] unit phasors of the sub-tile
    C0 = Us + kRowsMax * kTileW;           // [chunk] coefficients of the first chunk (prologue)
  }
};

// Sec. 3 coefficient of trap m in complex form: w_m' V_m/|V_m| with w_m' = w_m <|V|>/|V_m|
// (R4: |V_m| = 0 keeps w_m and takes the unit field 1).
__device__ __forceinline__ float2 complex_coefficient(const StepArgs &a, int m, float mean) {
  return update_from<true>(field_from_sums<true>(a, m), __ldcg(a.w_in + m), mean, 1.f);
}

template <bool BACK>
__device__ __forceinline__ void stage_sep(const StepArgs &a, int m0, int n, const SubTile &st, const SepSmem &sm,
                                          bool xy = true, float mean = 0.f, bool coef = true) {
  if (xy) {
    if ((a.W & 1) == 0 && st.x0 + kTileW <= a.W) {
      // thread t copies columns 2 (t % 16), +1 of traps t / 16, t / 16 + 16, ... (16 bytes:
      // rows start 16-byte aligned for even W)
      const int q = gthread() % (kTileW / 2), kx = gthread() / (kTileW / 2);
      const float2 *src = a.Xc + (size_t)(m0 + kx) * a.W + st.x0 + 2 * q;
      const size_t sx = (size_t)(kThreads / (kTileW / 2)) * a.W;
      for (int k = kx; k < n; k += kThreads / (kTileW / 2), src += sx) cp_async16(sm.Xs + k * kTileW + 2 * q, src);
    } else {
      // thread t copies column t % 32 of traps t / 32, t / 32 + 8, ...: fixed column, pointers
      // advanced by whole trap strides
      const int col = gthread() % kTileW, kx = gthread() / kTileW;
      const bool okx = st.x0 + col < a.W;
      const float2 *src = a.Xc + (okx ? (size_t)(m0 + kx) * a.W + st.x0 + col : 0);
      const size_t sx = okx ? (size_t)(kThreads / kTileW) * a.W : 0;
      for (int k = kx; k < n; k += kThreads / kTileW, src += sx) cp_async8(sm.Xs + k * kTileW + col, src, okx);
    }
    // rows y0 .. y0 + 15 of copy y0 % 2 (16-byte aligned): thread t copies rows 2 (t % 8), +1 of
    // traps t / 8, t / 8 + 32, ...
    const int s = st.y0 & 1, q = gthread() % (kYStride / 2), ky = gthread() / (kYStride / 2);
    const float2 *srcy = a.Yc + ((size_t)s * a.M + m0 + ky) * a.ldy4 + st.y0 + s + 2 * q;
    const size_t sy = (size_t)(kThreads / (kYStride / 2)) * a.ldy4;
    for (int k = ky; k < n; k += kThreads / (kYStride / 2), srcy += sy) cp_async16(sm.Ys + k * kYStride + 2 * q, srcy);
  }
  if (BACK && coef)
    for (int i = gthread(); i < n; i += kThreads)
      sm.Cs[i] = complex_coefficient(a, m0 + i, mean);
  cp_async_wait_all();
}

// S_r += Yc_m(r) (c_m Xc_m(lane)) for traps [lo, hi) of the staged chunk (coefficients C).
template <int R>
__device__ __forceinline__ void back_traps_sep(const SepSmem &sm, const float2 *C, int lo, int hi, int lane,
                                               float2 (&S)[kRowsMax]) {
  for (int k = lo; k < hi; k++) {
    const float2 x = sm.Xs[k * kTileW + lane], c = C[k];
    const float2 b = make_float2(c.x * x.x - c.y * x.y, c.x * x.y + c.y * x.x);
    const float4 *yq = reinterpret_cast<const float4 *>(sm.Ys + k * kYStride);
#pragma unroll
    for (int q = 0; q < (R + 1) / 2; q++) {
      const float4 y2 = yq[q];
      const float2 yy[2] = {make_float2(y2.x, y2.y), make_float2(y2.z, y2.w)};
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const int r = 2 * q + j;
        if (r < R) {
          S[r].x = fmaf(yy[j].x, b.x, fmaf(-yy[j].y, b.y, S[r].x));
          S[r].y = fmaf(yy[j].x, b.y, fmaf(yy[j].y, b.x, S[r].y));
        }
      }
    }
  }
}

// Forward field of traps [lo, hi): conj(Xc_m(lane)) sum_r u_r conj(Yc_m(r)), summed over the
// warp 8 traps at a time and added in fixed point (as forward_traps).  u is zero outside the
// image, so no mask is needed.
template <int R>
__device__ __forceinline__ void forward_traps_sep(const SepSmem &sm, int lo, int hi, int lane,
                                                  const float2 (&u)[kRowsMax], const StepArgs &a, int m0) {
  for (int g = lo; g < hi; g += kGroup) {
    float2 acc[kGroup];
#pragma unroll
    for (int i = 0; i < kGroup; i++) {
      acc[i] = make_float2(0.f, 0.f);
      const int k = g + i;
      if (k < hi) {
        const float4 *yq = reinterpret_cast<const float4 *>(sm.Ys + k * kYStride);
        float2 t = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < (R + 1) / 2; q++) {
          const float4 y2 = yq[q];
          const float2 yy[2] = {make_float2(y2.x, y2.y), make_float2(y2.z, y2.w)};
#pragma unroll
          for (int j = 0; j < 2; j++) {
            const int r = 2 * q + j;
            if (r < R) {
              t.x = fmaf(u[r].x, yy[j].x, fmaf(u[r].y, yy[j].y, t.x));
              t.y = fmaf(u[r].y, yy[j].x, fmaf(-u[r].x, yy[j].y, t.y));
            }
          }
        }
        const float2 x = sm.Xs[k * kTileW + lane];
        acc[i] = make_float2(t.x * x.x + t.y * x.y, t.y * x.x - t.x * x.y);
      }
    }
    const float2 v = warp_reduce8(acc, lane);
    const int k = g + ((lane >> 2) & 7);
    if ((lane & 3) == 0 && k < hi) {
      unsigned long long *acc = block_acc(a);
      atomicAdd(acc + m0 + k, (unsigned long long)__float2ll_rn(v.x * a.fx_scale));
      atomicAdd(acc + a.M + m0 + k, (unsigned long long)__float2ll_rn(v.y * a.fx_scale));
    }
  }
}

template <bool BACK>
__device__ __forceinline__ void process_subtile_sep(const StepArgs &a, const SubTile st, float mean, bool &prestaged,
                                                    const SepSmem &sm, const float2 *C0 = nullptr) {
  const int lane = threadIdx.x & 31, warp = gthread() >> 5;
  const int mc = a.M < a.chunk ? a.M : a.chunk;
  const int nchunks = (a.M + mc - 1) / mc;
  const int ix = st.x0 + lane;
  const bool col_ok = ix < a.W;

  if (BACK) {
    float2 S[kRowsMax];
#pragma unroll
    for (int r = 0; r < kRowsMax; r++) S[r] = make_float2(0.f, 0.f);
    for (int ch = 0; ch < nchunks; ch++) {
      const int m0 = ch * mc, n = min(mc, a.M - m0);
      const bool pre = C0 && ch == 0;
      group_sync();  // earlier readers of the tables are done
      stage_sep<true>(a, m0, n, st, sm, !prestaged, mean, !pre);
      prestaged = false;
      group_sync();
      int lo, hi;
      warp_traps(n, warp, lo, hi);
      const float2 *C = pre ? C0 : sm.Cs;
      HOT_WITH_ROWS(st.rows, (back_traps_sep<R>(sm, C, lo, hi, lane, S)));
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
      if (h * kHalfRows >= st.rows) break;
      group_sync();  // Sp and the phasor rows are free
#pragma unroll
      for (int i = 0; i < kHalfRows; i++)
        if (h * kHalfRows + i < st.rows) sm.Sp[(warp * kHalfRows + i) * kTileW + lane] = S[h * kHalfRows + i];
      group_sync();
      if (warp < kHalfRows && h * kHalfRows + warp < st.rows) {
        const int r = h * kHalfRows + warp;
        float2 s = sm.Sp[warp * kTileW + lane];
#pragma unroll
        for (int w = 1; w < kWarps; w++) {
          const float2 q = sm.Sp[(w * kHalfRows + warp) * kTileW + lane];
          s.x += q.x;
          s.y += q.y;
        }
        const size_t j = (size_t)(st.y0 + r) * a.W + ix;
        const float ph = atan2f(s.y, s.x);
        if (col_ok) a.phi[j] = ph;
        // u = e^{i phi} of the stored phase (so that a resumed run is identical)
        float2 u = make_float2(0.f, 0.f);
        if (col_ok) sincosf(ph, &u.y, &u.x);
        sm.Us[r * kTileW + lane] = u;
      }
    }
  } else {
    group_sync();  // earlier readers of the phasors and of the tables are done
    for (int r = warp; r < st.rows; r += kWarps) {
      float2 u = make_float2(0.f, 0.f);
      if (col_ok) sincosf(a.phi[(size_t)(st.y0 + r) * a.W + ix], &u.y, &u.x);
      sm.Us[r * kTileW + lane] = u;
    }
  }

  group_sync();  // the phasors are complete
  float2 u[kRowsMax];
#pragma unroll
  for (int r = 0; r < kRowsMax; r++) u[r] = r < st.rows ? sm.Us[r * kTileW + lane] : make_float2(0.f, 0.f);
  for (int ch = 0; ch < nchunks; ch++) {
    const int m0 = ch * mc, n = min(mc, a.M - m0);
    if (!BACK || nchunks > 1) {  // with one chunk the back-projection's tables are still staged
      if (ch) group_sync();
      stage_sep<false>(a, m0, n, st, sm);
      group_sync();
    }
    int lo, hi;
    warp_traps(n, warp, lo, hi);
    HOT_WITH_ROWS(st.rows, (forward_traps_sep<R>(sm, lo, hi, lane, u, a, m0)));
  }
}

// Batched launch: the sub-tiles of up to kBatchMax holograms (SubTile::pad = hologram index)
// in one grid.  The holograms' parameters travel in the launch itself (a __grid_constant__
// argument read through the constant cache, as the single-hologram kernel reads its own).
// Every block that meets a hologram computes its <|V|> and coefficients itself; the weights
// of hologram h are written by block owner[h].
constexpr int kBatchMax = 22;  // keeps the launch argument under 4 KB

struct BatchArgs {
  StepArgs holo[kBatchMax];
  int owner[kBatchMax];
  const SubTile *sub;
  const int *first;  // [gridDim.x + 1]
  int count;
};
static_assert(sizeof(BatchArgs) <= 4096, "launch argument above 4 KB");

// MODE: kModeAccurate, kModeFast or kModeSeparable (the separable kernel's staging capacity is
// the batch's chunk, the same for all holograms of a launch).
template <int MODE, bool BACK>
__global__ void __launch_bounds__(kThreads, MODE == kModeSeparable ? 2 : 4)
    gsw_batch_kernel(const __grid_constant__ BatchArgs b) {
  constexpr bool FAST = MODE == kModeFast, SEP = MODE == kModeSeparable;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int t_begin = b.first[blockIdx.x], t_end = b.first[blockIdx.x + 1];
  const int cap = b.holo[0].chunk;
  float2 *const C0 = SEP ? SepSmem(smem_raw, cap).C0 : StepSmem(smem_raw).C0;

  allow_dependents();
  bool prestaged = false;
  if (BACK && t_begin < t_end) {
    const SubTile st0 = b.sub[t_begin];
    const StepArgs &a0 = b.holo[st0.pad];
    const int mc0 = a0.M < a0.chunk ? a0.M : a0.chunk;
    if constexpr (SEP) {
      stage_sep<false>(a0, 0, mc0, st0, SepSmem(smem_raw, cap));
    } else {
      const StepSmem sm(smem_raw);
      stage_tables<false>(a0, 0, mc0, st0, sm.Xs, sm.Ys, sm.Cs);
    }
    prestaged = true;
  }
  grid_dependency_wait();
  for (int h = 0; h < b.count; h++) {  // clear the buffers the next launch accumulates into, for every hologram
    unsigned long long *clr = b.holo[h].acc_clear;
    const int n2 = 2 * b.holo[h].M * b.holo[h].copies;
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < n2; i += gridDim.x * kThreads) clr[i] = 0ull;
  }
  int cur = -1;
  LateWeight lw;  // the owner block writes all weights of a hologram, after its sub-tiles
  for (int t = t_begin; t < t_end; t++) {
    const SubTile st = b.sub[t];
    const StepArgs &a = b.holo[st.pad];
    if (BACK && st.pad != cur) {
      if (cur >= 0) write_weights<SEP>(b.holo[cur], lw, 1);
      const int mc = a.M < a.chunk ? a.M : a.chunk;
      gsw_prologue<SEP>(a, mc, C0, b.owner[st.pad] == (int)blockIdx.x ? 0 : a.M, 1, lw);
    }
    cur = st.pad;
    if constexpr (SEP)
      process_subtile_sep<BACK>(a, st, 1.f, prestaged, SepSmem(smem_raw, cap), BACK ? C0 : nullptr);
    else
      process_subtile<FAST, BACK, true, false>(a, st, 1.f, prestaged, StepSmem(smem_raw), BACK ? C0 : nullptr);
  }
  if (BACK && cur >= 0) write_weights<SEP>(b.holo[cur], lw, 1);
}

// Column and row phasors of a separable batch's member: Xc [M][W], Yc [2][M][ldy4] (StepArgs), whose
// entries outside the shifted rows stay as they are (zero from allocation).
static __global__ void batch_tables_kernel(int W, int H, int M, const double *abc, float2 *Xc, float2 *Yc, int ldy4) {
  const long long total = (long long)M * (W + H);
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(idx / (W + H)), i = (int)(idx % (W + H));
    const double am = abc[3 * m], bm = abc[3 * m + 1], cm = abc[3 * m + 2];
    double t;
    if (i < W) {
      const double q = (double)(i - W / 2);
      t = fma(cm * q, q, am * q);
    } else {
      const double q = (double)((i - W) - H / 2);
      t = fma(cm * q, q, bm * q);
    }
    t -= rint(t);  // [-1/2, 1/2] turns
    double sn, cs;
    sincospi(2.0 * t, &sn, &cs);
    const float2 e = make_float2((float)cs, (float)sn);
    if (i < W)
      Xc[(size_t)m * W + i] = e;
    else
      for (int sh = 0; sh < 2; sh++) Yc[((size_t)sh * M + m) * ldy4 + (i - W) + sh] = e;
  }
}

}  // namespace hot
