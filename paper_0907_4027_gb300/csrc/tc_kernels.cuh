// tc_kernels.cuh -- the separable GSW iteration on the tensor cores (tcgen05, sm_103a).
//
// Eq. 2 is separable: e^{i Delta_j^m} = X_m(ix) Y_m(iy) with X_m(ix) = e^{i 2pi [a_m ix' + c_m ix'^2]}
// and Y_m(iy) = e^{i 2pi [b_m iy' + c_m iy'^2]}.  Both steps of a GSW iteration are then complex
// matrix products over the pixel grid:
//   back-projection (Sec. 4)  S[iy][ix] = sum_m (c_m Y_m(iy)) X_m(ix)        = P . X     (H x M by M x W)
//   forward field   (Eq. 1)   T[iy][m]  = sum_ix u[iy][ix] conj(X_m(ix))     = U . X^H   (H x W by W x M)
//                             N V_m     = sum_iy conj(Y_m(iy)) T[iy][m]
// with u = e^{i phi}.  Real and imaginary parts are separate matrices.  A tile's right-hand operand
// is the stack [X_r; X_i] of BN/2 traps or columns, and each K slice of it meets first A_r, then A_i
// (A = P or U): the two accumulators A_r [X_r | X_i] and A_i [X_r | X_i] hold the four real products,
// which the drain adds with the signs of X (back) or conj(X) (forward).  (What bounds the GEMMs is
// the operand traffic from L2: against the 2x2 real embedding [[xr, -xi], [xi, xr]] of B this moves
// 64 instead of 96 KB per 12 MMAs of a 128 x 256 tile; with the epilogues below, an iteration of 1920 x 1152
// with 1000 traps went from 119.8 to 99.6 us, 1024^2 with 256 from 41.9 to 27.7, 512^2 with 100 from 17.5 to
// 15.2, 256^2 with 16 from 12.7 to 11.3.  What bounds the widest tiles now is the MMAs' own rate: leaving out
// the loads or the drain changes nothing, one MMA in three less saves its 128 cycles and a little more.)
// The GEMMs run on tcgen05.mma with FP32 accumulators in tensor
// memory.  A 16-bit or TF32 tensor-core operand keeps 11 significant bits, so every operand is
// split x = hi + lo and a product takes three MMAs, a_hi b_hi + a_hi b_lo + a_lo b_hi (the omitted
// a_lo b_lo is ~2^-22 relative): the products keep about FP32 accuracy.  The GSW iteration uses
// two FP16 parts (kind::f16: twice the TF32 rate, half the bytes; its operands are unit phasors and
// coefficients scaled to <= 1, where FP16 keeps its 11 bits); the GEMM also runs two TF32 parts
// (kind::tf32, the FP32 exponent range).
//
// A CTA computes one 128 x BN tile of a GEMM over a range of K, warp-specialised: one thread of
// warp 0 issues TMA loads of K slices (one 128-byte row per matrix row, 128-byte swizzle) of A and
// of B (both parts, hi and lo) into two rings of shared-memory stages; one thread of warp 1 issues the 12 MMAs of
// a slice into one of 2-4 tensor-memory accumulators and returns the stage to the loader with
// tcgen05.commit; the drain warps (TMEM lane quadrant = warp % 4, i.e. 32 rows each, and a group
// of <= 128 columns) add every slice's accumulator into FP32 registers while the MMAs of the next
// slices run in the other accumulators.  The tensor core's own accumulation into TMEM is not
// round-to-nearest (measured: a magnitude bias growing with the MMAs accumulated, ~1e-4 relative on
// small |V_m| after 190), so each accumulator holds the 12 MMAs of one slice only and the K sum
// runs in the registers (round-to-nearest, fixed order).  Then the epilogue:
//   back:    phi = arg S (atan2f), u = e^{i phi}, written as phases and as the split U operand;
//   forward: the tile's rows weighted by conj(Y_m(iy)) and summed, added into the 64-bit
//            fixed-point field accumulators (integer atomics: exact and order-independent, so
//            the K range may be split over CTAs);
//   plain:   C = A B^T (the GEMM alone, for tests).
// Every wait on an mbarrier is bounded by %globaltimer; when one runs out the CTA sets the error
// flag, stops issuing, waits (bounded by kDrainNs at least, whatever the caller's limit) for the copies
// and the MMAs it has in flight, frees its tensor memory and returns.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace tc {

constexpr int kBM = 128;         // rows of a tile: the 128 lanes of tensor memory
constexpr int kSliceBytes = 128; // one K slice per stage: one 128-byte swizzle row of every operand row
constexpr int kMmaKBytes = 32;   // K of one MMA: 8 TF32 or 16 FP16 elements
constexpr long long kDrainNs = 1000000000;  // what a CTA that gives up grants its copies and MMAs at least

// Operand types.  TF32: FP32 storage, kind::tf32 (the MMA reads the top 19 bits).  FP16: halves,
// kind::f16 at twice the TF32 rate; its 11-bit significand equals TF32's, so the split keeps the
// same precision for operands of magnitude ~1 (the GSW operands are unit phasors and normalised
// coefficients), while subnormals limit it below ~2^-2 (the low part) and ~2^-14 (the high part).
constexpr int kOpTF32 = 0, kOpF16 = 1;
template <int OP>
struct Op;
template <>
struct Op<kOpTF32> {
  using T = float;
  static constexpr int kBytes = 4;
  static constexpr uint32_t kFmt = 2;  // instruction-descriptor operand format TF32
};
template <>
struct Op<kOpF16> {
  using T = __half;
  static constexpr int kBytes = 2;
  static constexpr uint32_t kFmt = 0;  // F16
};
template <int OP>
__host__ __device__ constexpr int slice_k() {  // K elements per slice: 32 (TF32) or 64 (FP16)
  return kSliceBytes / Op<OP>::kBytes;
}

constexpr int kEpiPlain = 0, kEpiBack = 1, kEpiFwd = 2;

// Tile width BN (32, 64, 128 or 256 columns): shared-memory stages as fit in 224 KB; the accumulator
// is drained by 4 warps per column group (a thread keeps its row's columns of the group in registers).
// The groups are many for the epilogues' sake, which are chains of latencies: one group of 32, 64 or 128
// columns and two of 256 took 12.0, 16.1, 22.3, 32.8 and 101 us per iteration at 256^2 / 16, 512^2 / 100,
// 768^2 / 100, 1024^2 / 256 and 1920 x 1152 / 1000 traps, these take 11.3, 15.2, 19.6, 27.7 and 99.6; groups
// of 8 columns for BN = 32 (15.6, 20.2) were slower again.
template <int BN>
struct Cfg {
  static_assert(BN == 32 || BN == 64 || BN == 128 || BN == 256, "tile width");
  // stages of the rings of A and of B: with two stages of A the loads of a step had only the step
  // before it to arrive in
  static constexpr int kStagesA = BN >= 128 ? 3 : 4, kStagesB = BN == 256 ? 2 : BN == 128 ? 3 : 4;
  static constexpr int kABytes = kBM * kSliceBytes;  // 16 KB: one part (hi or lo) of a slice
  static constexpr int kBBytes = BN * kSliceBytes;
  static constexpr int kRingBytes = 2 * (kStagesA * kABytes + kStagesB * kBBytes);
  // the row table under a forward tile, fetched before the K loop, where it fits beside the rings (with it
  // 12.2, 16.3, 21.7 us at 256^2 / 16, 512^2 / 100, 768^2 / 100 against 12.9, 17.4, 22.3)
  static constexpr int kYBytes = BN <= 64 ? kBM * (BN / 2) * 8 : 0;
  static constexpr int kSmem = kRingBytes + kYBytes + 1024;  // + slack to align the rings to 1 KB
  static constexpr int kGroups = BN >= 64 ? 4 : 2;        // column groups of the drain
  static constexpr int kCols = BN / kGroups;                  // columns per drain warp
  static constexpr int kEpiWarps = 4 * kGroups;               // one per TMEM lane quadrant and group
  static constexpr int kThreads = 32 * (2 + kEpiWarps);       // warp 0: TMA, warp 1: MMA, then drain
  static constexpr int kBufs = BN == 256 ? 2 : 4;             // accumulators in the 512 TMEM columns
  static constexpr int kTmemCols = kBufs * BN;                // a power of two >= 32
};
// The operand maps of one GEMM (2-D, box of one 128-byte K slice x rows, 128-byte swizzle), by
// component (real, imaginary; plain GEMM: a[0], and b[0] = b[1]) and part (hi, lo).  B's boxes have
// BN / 2 rows, one component.
struct Maps {
  CUtensorMap a[2][2], b[2][2];
};

struct GemmArgs {
  int rows, cols;        // GEMM M and N: outputs outside are not written
  int k_chunks;          // K in units: slices (plain), half slices of one component (back, forward)
  int chunks_per_split;  // units per CTA: CTA z takes units z*cps .. min(k_chunks, (z+1)*cps)-1
  long long limit_ns;    // bound of every wait
  int *err;              // set to 1 when a wait runs out
  // plain
  float *C;              // [rows][cols]
  // back: S -> phi, U
  int W, H, ldu;         // pixels; row stride of U (elements)
  float *phi;            // [H][W]
  __half *u[2][2];       // [..][ldu] cos phi, sin phi (component), hi and lo (part)
  // forward: T -> fixed-point field sums
  int M;
  int Kp;                        // row stride of YT
  const float2 *YT;              // [H][Kp] Y_m(iy)
  unsigned long long *acc_out;   // [2][M] Re, Im (zero before the first split adds)
  float fx_scale;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for the completion of the phase of parity `parity`; false after limit_ns.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = timer_ns();
  for (;;) {
    for (int i = 0; i < 32; i++)
      if (mbar_try_wait(bar, parity)) return true;
    if ((long long)(timer_ns() - t0) > limit_ns) return false;
  }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major operand tile written by TMA with 128-byte
// swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart (stride byte offset), start address
// in 16-byte units; bits 46-47 = 1 (tcgen05 descriptor), bits 61-63 = 2 (128-byte swizzle).
// The leading byte offset is unused for a swizzled K-major tile whose K fits in one row.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor of kind::tf32 / kind::f16: FP32 accumulator (bits 4-5 = 1), A and B
// format at bits 7-9 and 10-12 (TF32 = 2, F16 = 0), both K-major (bits 15, 16 = 0), N >> 3 at
// bit 17, M >> 4 at bit 24.
template <int OP>
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
  return (1u << 4) | (Op<OP>::kFmt << 7) | (Op<OP>::kFmt << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

template <int OP>
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  if (OP == kOpF16)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The barrier receives one arrival when every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 32 consecutive accumulator columns of this warp's 32 lanes (thread t: lane 32w + t); the wait
// sits in the same statement, so the registers are complete when the statement ends.
__device__ __forceinline__ void tmem_load32(uint32_t taddr, float *v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_load16(uint32_t taddr, float *v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_load8(uint32_t taddr, float *v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

// acc[0 .. N-1] += sign (+-1: exact) times N accumulator columns from taddr (N = 8, 16 or a multiple of 32).
template <int N>
__device__ __forceinline__ void drain_columns(uint32_t taddr, float *acc, float sign) {
  constexpr int STEP = N < 16 ? 8 : N < 32 ? 16 : 32;
#pragma unroll
  for (int c = 0; c < N; c += STEP) {
    float v[STEP];
    if constexpr (STEP == 8)
      tmem_load8(taddr + (uint32_t)c, v);
    else if constexpr (STEP == 32)
      tmem_load32(taddr + (uint32_t)c, v);
    else
      tmem_load16(taddr + (uint32_t)c, v);
#pragma unroll
    for (int j = 0; j < STEP; j++) acc[c + j] = fmaf(sign, v[j], acc[c + j]);
  }
}

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// x ~ hi + lo, both exactly representable in the operand type (returned as floats).  TF32: hi is
// x with the 13 low mantissa bits cleared, lo the exact FP32 rest (the MMA reads its TF32 part).
// FP16: hi = x rounded to half, lo = the rest rounded to half.
template <int OP>
__device__ __forceinline__ float2 split2(float x) {
  if (OP == kOpF16) {
    const float hi = __half2float(__float2half_rn(x));
    return make_float2(hi, __half2float(__float2half_rn(x - hi)));
  }
  const float hi = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
  return make_float2(hi, x - hi);
}

// Element i of an operand array (a value split2 produced, so the conversion is exact).
template <int OP>
__device__ __forceinline__ void store1(void *base, size_t i, float v) {
  if (OP == kOpF16)
    static_cast<__half *>(base)[i] = __float2half_rn(v);
  else
    static_cast<float *>(base)[i] = v;
}
// u = e^{i phi} of a phase in any range: reduced to [-pi, pi] (Cody-Waite with 2 pi split in
// two floats; a no-op for the back-projection's own phases in (-pi, pi]), then the SFU's
// sin/cos approximations (|error| ~ 4e-7 on that interval).  The forward operand of the phases
// a call starts from and of the phases an iteration writes come from this one function, so a
// resumed run repeats the bits of an uninterrupted one.
__device__ __forceinline__ void unit_phasor(float ph, float &sn, float &cs) {
  const float k = rintf(ph * 0.15915494309189535f);
  const float x = fmaf(-k, -1.74845553e-07f, fmaf(-k, 6.28318548e+00f, ph));
  __sincosf(x, &sn, &cs);
}

// Two values' hi (x) and lo (y) FP16 parts, packed.
__device__ __forceinline__ uint2 split_pair(float a, float b) {
  const __half2 hi = __floats2half2_rn(a, b);
  const float2 h = __half22float2(hi);
  const __half2 lo = __floats2half2_rn(a - h.x, b - h.y);
  return make_uint2(*reinterpret_cast<const uint32_t *>(&hi), *reinterpret_cast<const uint32_t *>(&lo));
}

// Complex values (re[0], im[0]), (re[1], im[1]) into the split component arrays at elements i, i + 1 (i even).
__device__ __forceinline__ void store_pair(__half *const (&dst)[2][2], size_t i, float2 re, float2 im) {
  const uint2 r = split_pair(re.x, re.y), m = split_pair(im.x, im.y);
  *reinterpret_cast<uint32_t *>(dst[0][0] + i) = r.x;
  *reinterpret_cast<uint32_t *>(dst[0][1] + i) = r.y;
  *reinterpret_cast<uint32_t *>(dst[1][0] + i) = m.x;
  *reinterpret_cast<uint32_t *>(dst[1][1] + i) = m.y;
}

// N accumulator columns n0 .. of one row of the plain GEMM: C.
template <int N>
__device__ __forceinline__ void epilogue_plain(const GemmArgs &a, const float *v, int row, int n0) {
  if (row < a.rows)
#pragma unroll
    for (int c = 0; c < N; c++)
      if (n0 + c < a.cols) a.C[(size_t)row * a.cols + n0 + c] = v[c];
}

// The back and forward epilogues start from the tile in shared memory (the rings are free by then),
// real and imaginary halves of BN / 2 columns in rows of kStage floats: a drain thread holds one row,
// and its registers can only be walked by straight-line code (64 pixels of atan2, sin and cos: 100 KB
// of instructions run once, 1.2 warps of the drain waiting for the instruction cache at any time), while the
// epilogues want short loops and neighbouring columns in neighbouring lanes (measured together with the operands above).
template <int BN>
constexpr int kStage = BN + 4;  // floats: 16-byte stores of eight rows fall on different banks
template <int BN>
__device__ __forceinline__ void stage_tile(float *tile, const float *acc, int q, int g) {
  constexpr int HALF = Cfg<BN>::kCols / 2;
  float *row = tile + (q * 32 + (threadIdx.x & 31)) * kStage<BN> + g * HALF;
#pragma unroll
  for (int c = 0; c < HALF; c += 4) {
    *reinterpret_cast<float4 *>(row + c) = make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
    *reinterpret_cast<float4 *>(row + BN / 2 + c) =
        make_float4(acc[HALF + c], acc[HALF + c + 1], acc[HALF + c + 2], acc[HALF + c + 3]);
  }
  asm volatile("bar.sync 1, %0;" ::"n"(32 * Cfg<BN>::kEpiWarps) : "memory");  // the drain warps only
}

// Back-projection: S of the tile's pixels -> phi = arg S (Sec. 4; atan2(0, 0) = 0) and u = e^{i phi},
// split: two neighbouring pixels per thread and step.
template <int BN>
__device__ __forceinline__ void epilogue_back(const GemmArgs &a, const float *tile, int m0, int x0) {
  constexpr int PAIRS = BN / 4;  // pixel pairs of a row
  const bool two = (a.W & 1) == 0;  // rows start 8-byte aligned
#pragma unroll 1
  for (int i = threadIdx.x - 64; i < kBM * PAIRS; i += 32 * Cfg<BN>::kEpiWarps) {
    const int r = i / PAIRS, p = 2 * (i % PAIRS), iy = m0 + r, ix = x0 + p;
    if (iy >= a.H || ix >= a.W) continue;
    const float2 re = *reinterpret_cast<const float2 *>(tile + r * kStage<BN> + p);
    const float2 im = *reinterpret_cast<const float2 *>(tile + r * kStage<BN> + BN / 2 + p);
    float2 ph, cs, sn;
    ph.x = atan2f(im.x, re.x);
    ph.y = atan2f(im.y, re.y);
    unit_phasor(ph.x, sn.x, cs.x);
    unit_phasor(ph.y, sn.y, cs.y);
    float *out = a.phi + (size_t)iy * a.W + ix;
    if (ix + 1 >= a.W) {  // an odd row's last pixel: the padding of U stays zero
      out[0] = ph.x;
      cs.y = sn.y = 0.f;
    } else if (two) {
      *reinterpret_cast<float2 *>(out) = ph;
    } else {
      out[0] = ph.x;
      out[1] = ph.y;
    }
    store_pair(a.u, (size_t)iy * a.ldu + ix, cs, sn);
  }
}

// The rows of YT under a forward tile into shared memory [kBM][BN / 2], by the drain warps (16-byte pieces:
// t0 and Kp are even); rows and traps beyond the image are not fetched and not read.
template <int BN>
__device__ __forceinline__ void fetch_rows(const GemmArgs &a, unsigned char *y, int m0, int t0) {
  constexpr int PIECES = BN / 4;
  for (int i = threadIdx.x - 64; i < kBM * PIECES; i += 32 * Cfg<BN>::kEpiWarps) {
    const int r = i / PIECES, m = t0 + 2 * (i % PIECES);
    if (m0 + r < a.H && m < a.Kp)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(y) + 16 * i),
                   "l"(a.YT + (size_t)(m0 + r) * a.Kp + m)
                   : "memory");
  }
}

// Forward: the tile's T[row][m] times conj(Y_m(row)), summed over its rows -- a thread takes one trap
// and every PARTS-th row, in four partial sums -- and added into the fixed-point sums, one atomic
// per trap and component.  The partial sums meet in red.
template <int BN>
__device__ __forceinline__ void epilogue_fwd(const GemmArgs &a, const float *tile, float4 *red, const float2 *ys, int m0, int t0) {
  constexpr int TRAPS = BN / 2, THREADS = 32 * Cfg<BN>::kEpiWarps, PARTS = THREADS / TRAPS;
  const int t = threadIdx.x - 64, j = t % TRAPS, part = t / TRAPS, m = t0 + j;
  const int rows = min(kBM, a.H - m0);
  float2 v[4];
#pragma unroll
  for (int k = 0; k < 4; k++) v[k] = make_float2(0.f, 0.f);
  if (m < a.M) {
    const float *z = tile + j;
    const float2 *y = a.YT + (size_t)m0 * a.Kp + m;
#pragma unroll 4
    for (int r = part; r < kBM; r += 4 * PARTS)
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int rr = r + k * PARTS;
        if (rr < rows) {
          const float2 yy = Cfg<BN>::kYBytes ? ys[rr * TRAPS + j] : __ldg(y + (size_t)rr * a.Kp);
          const float tr = z[rr * kStage<BN>], ti = z[rr * kStage<BN> + BN / 2];
          v[k].x = fmaf(tr, yy.x, fmaf(ti, yy.y, v[k].x));
          v[k].y = fmaf(ti, yy.x, fmaf(-tr, yy.y, v[k].y));
        }
      }
  }
  const float2 s = make_float2((v[0].x + v[1].x) + (v[2].x + v[3].x), (v[0].y + v[1].y) + (v[2].y + v[3].y));
  float2 *const sums = reinterpret_cast<float2 *>(red);
  sums[t] = s;
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (part == 0 && m < a.M) {
    float2 w = s;
#pragma unroll
    for (int k = 1; k < PARTS; k++) {
      w.x += sums[t + k * TRAPS].x;
      w.y += sums[t + k * TRAPS].y;
    }
    // |w| <= N, so w * 2^fx_shift rounds to an integer below 2^61
    atomicAdd(a.acc_out + m, (unsigned long long)__float2ll_rn(w.x * a.fx_scale));
    atomicAdd(a.acc_out + a.M + m, (unsigned long long)__float2ll_rn(w.y * a.fx_scale));
  }
}

// One 128 x BN output tile over a K range: TMA loader (warp 0, one lane), MMA issuer (warp 1,
// one lane), accumulator drain and epilogue (the other warps).  grid = (N tiles, M tiles, K splits).
// A step is one slice of one component of A against the slice of B: NA steps per slice of B.
template <int BN, int EPI, int OP>
__global__ void __launch_bounds__(Cfg<BN>::kThreads, 1) tc_gemm_kernel(const __grid_constant__ Maps maps,
                                                                       const __grid_constant__ GemmArgs a) {
  using C = Cfg<BN>;
  constexpr int NA = EPI == kEpiPlain ? 1 : 2, SA = C::kStagesA, SB = C::kStagesB;
  constexpr int kSteps = kSliceBytes / kMmaKBytes;  // MMA steps along K per slice
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_a[SA], empty_a[SA], full_b[SB], empty_b[SB], tfull[C::kBufs], tempty[C::kBufs];
  __shared__ uint32_t tmem_slot;
  __shared__ int issued_a, issued_b, consumed_a, consumed_b, failed;
  // the rings start on a 1 KB boundary of the shared window (the 128-byte swizzle pattern repeats
  // every 8 rows of 128 bytes and the descriptors assume aligned tiles)
  unsigned char *ring_a = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char *ring_b = ring_a + SA * 2 * C::kABytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * kBM;
  const int kc0 = blockIdx.z * a.chunks_per_split;
  const int nk = min(a.k_chunks - kc0, a.chunks_per_split);  // >= 1 (the host sizes the splits)
  const int nb = NA == 1 ? nk : (nk + 1) / 2;                // slices of B; the last one may be half
  const int steps = NA * nb;
  if (threadIdx.x == 0) {
    for (int s = 0; s < SA; s++) {
      mbar_init(&full_a[s], 1);
      mbar_init(&empty_a[s], 1);
    }
    for (int s = 0; s < SB; s++) {
      mbar_init(&full_b[s], 1);
      mbar_init(&empty_b[s], 1);
    }
    for (int b = 0; b < C::kBufs; b++) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], C::kEpiWarps);
    }
    issued_a = issued_b = consumed_a = consumed_b = failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1 && lane < 8 && (NA == 2 || (lane & 6) != 2)) {  // the operand maps (plain: no second component of A)
    const CUtensorMap *map = lane < 4 ? &maps.a[lane >> 1][lane & 1] : &maps.b[(lane - 4) >> 1][lane & 1];
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
  }
  if (warp == 0) {  // the whole warp allocates kBufs FP32 accumulators of BN columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(C::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  grid_wait();  // the A operand is the previous kernel's output
  grid_release();

  if (warp == 0) {
    if (lane == 0) {
      const int kx0 = kc0 * (NA == 1 ? slice_k<OP>() : slice_k<OP>() / 2);
      const int nrow = n0 / NA, nhalf = NA == 1 ? BN / 2 : 0;  // B rows of the tile's two halves
      for (int j = 0; j < steps; j++) {
        const int i = j / NA, c = j % NA;
        const int kx = kx0 + i * slice_k<OP>();
        if (c == 0) {
          const int s = i % SB;
          if (i >= SB && !mbar_wait(&empty_b[s], ((uint32_t)(i / SB) & 1u) ^ 1u, a.limit_ns)) {
            failed = 1;
            break;
          }
          if (*(volatile int *)&failed) break;
          unsigned char *st = ring_b + s * 2 * C::kBBytes;
          mbar_expect_tx(&full_b[s], 2 * C::kBBytes);
          tma_load_2d(st, &maps.b[0][0], kx, nrow, &full_b[s]);
          tma_load_2d(st + C::kBBytes / 2, &maps.b[1][0], kx, nrow + nhalf, &full_b[s]);
          tma_load_2d(st + C::kBBytes, &maps.b[0][1], kx, nrow, &full_b[s]);
          tma_load_2d(st + C::kBBytes + C::kBBytes / 2, &maps.b[1][1], kx, nrow + nhalf, &full_b[s]);
          *(volatile int *)&issued_b = i + 1;
        }
        const int s = j % SA;
        if (j >= SA && !mbar_wait(&empty_a[s], ((uint32_t)(j / SA) & 1u) ^ 1u, a.limit_ns)) {
          failed = 1;
          break;
        }
        if (*(volatile int *)&failed) break;
        unsigned char *st = ring_a + s * 2 * C::kABytes;
        mbar_expect_tx(&full_a[s], 2 * C::kABytes);
        tma_load_2d(st, &maps.a[c][0], kx, m0, &full_a[s]);
        tma_load_2d(st + C::kABytes, &maps.a[c][1], kx, m0, &full_a[s]);
        *(volatile int *)&issued_a = j + 1;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc<OP>(kBM, BN);
      for (int j = 0; j < steps; j++) {
        const int b = j % C::kBufs, i = j / NA;
        // accumulator b is free once the drain warps have emptied its previous slice
        if (j >= C::kBufs && !mbar_wait(&tempty[b], (uint32_t)(j / C::kBufs - 1) & 1u, a.limit_ns)) {
          failed = 1;
          break;
        }
        const int sa = j % SA, sb = i % SB;
        if (*(volatile int *)&failed || !mbar_wait(&full_b[sb], (uint32_t)(i / SB) & 1u, a.limit_ns)) {
          failed = 1;
          break;
        }
        *(volatile int *)&consumed_b = i + 1;
        if (!mbar_wait(&full_a[sa], (uint32_t)(j / SA) & 1u, a.limit_ns)) {
          failed = 1;
          break;
        }
        *(volatile int *)&consumed_a = j + 1;
        tc_fence_after();
        const uint32_t pa = smem_u32(ring_a + sa * 2 * C::kABytes), pb = smem_u32(ring_b + sb * 2 * C::kBBytes);
        const uint32_t d = tmem + (uint32_t)(b * BN);
        const int n = NA == 2 && (nk & 1) && i == nb - 1 ? kSteps / 2 : kSteps;
#pragma unroll
        for (int kk = 0; kk < kSteps; kk++) {
          if (kk < n) {
            const uint32_t off = kk * kMmaKBytes;  // 32 bytes per MMA step along K
            const uint64_t ahi = smem_desc(pa + off), alo = smem_desc(pa + C::kABytes + off);
            const uint64_t bhi = smem_desc(pb + off), blo = smem_desc(pb + C::kBBytes + off);
            mma<OP>(d, ahi, bhi, idesc, kk != 0);
            mma<OP>(d, ahi, blo, idesc, 1u);
            mma<OP>(d, alo, bhi, idesc, 1u);
          }
        }
        mma_commit(&empty_a[sa]);  // the stages return to the loader when these MMAs have read them
        if (j % NA == NA - 1) mma_commit(&empty_b[sb]);
        mma_commit(&tfull[b]);     // and the accumulator goes to the epilogue warps
      }
    }
    __syncwarp();
  } else {
    // drain: step j's partial product (accumulator j % kBufs) added into registers in step order.  A
    // warp's group g holds HALF real (acc[0 ..]) and HALF imaginary parts (acc[HALF ..]) of the tile's
    // traps or pixels g HALF ..; plain: columns g HALF .. of both halves of the tile.
    constexpr int COLS = C::kCols, HALF = COLS / 2;
    const int q = warp & 3;          // TMEM lane quadrant of this warp: rows 32q .. 32q+31
    const int g = (warp - 2) >> 2;   // its column group
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(g * HALF);
    float acc[COLS];
#pragma unroll
    for (int c = 0; c < COLS; c++) acc[c] = 0.f;
    bool ok = true;
    if constexpr (EPI == kEpiFwd && C::kYBytes > 0) fetch_rows<BN>(a, ring_a + C::kRingBytes, m0, n0 / 2);
    for (int j = 0; j < steps; j++) {
      const int b = j % C::kBufs;
      ok = mbar_wait(&tfull[b], (uint32_t)(j / C::kBufs) & 1u, a.limit_ns);
      ok = __all_sync(0xffffffffu, ok) && !*(volatile int *)&failed;
      if (!ok) break;
      tc_fence_after();
      // the halves of the accumulator: A_c X_r, A_c X_i.  Re: A_r X_r, then -A_i X_i (conj(X): +); Im:
      // A_r X_i (conj(X): -), then A_i X_r
      const bool im = NA == 2 && (j & 1);
      const uint32_t x = tq + (uint32_t)(b * BN);
      drain_columns<HALF>(x + (im ? BN / 2 : 0), acc, im && EPI == kEpiBack ? -1.f : 1.f);
      drain_columns<HALF>(x + (im ? 0 : BN / 2), acc + HALF, !im && EPI == kEpiFwd ? -1.f : 1.f);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[b]);
    }
    if (!ok && lane == 0) {
      failed = 1;
      atomicExch(a.err, 1);
    }
    if constexpr (EPI == kEpiPlain) {
      const int row = m0 + q * 32 + lane;
      if (ok) {
        epilogue_plain<HALF>(a, acc, row, n0 + g * HALF);
        epilogue_plain<HALF>(a, acc + HALF, row, n0 + BN / 2 + g * HALF);
      }
    } else {
      // The rings are free once the last step was drained: every MMA that read them has completed.
      // After a failure copies may still be in flight: nothing is staged, and an incomplete tile
      // adds and writes nothing (the drain warps agree at a barrier).
      constexpr int THREADS = 32 * C::kEpiWarps;
      static_assert(kBM * kStage<BN> * 4 + THREADS * 8 <= C::kRingBytes, "the staged tile fits the rings");
      if constexpr (EPI == kEpiFwd && C::kYBytes > 0) asm volatile("cp.async.wait_all;" ::: "memory");
      asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
      if (!*(volatile int *)&failed) {
        float *const tile = reinterpret_cast<float *>(ring_a);
        stage_tile<BN>(tile, acc, q, g);
        if constexpr (EPI == kEpiBack)
          epilogue_back<BN>(a, tile, m0, n0 / 2);
        else
          epilogue_fwd<BN>(a, tile, reinterpret_cast<float4 *>(tile + kBM * kStage<BN>),
                           reinterpret_cast<const float2 *>(ring_a + C::kRingBytes), m0, n0 / 2);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && failed) {
    atomicExch(a.err, 1);
    // Copies that no MMA waited for, and the MMAs issued (steps 0 .. consumed_a - 1), may still be at work
    // in this CTA's shared and tensor memory: wait (bounded) for the copies and for the last commits, which
    // complete after the MMAs before them, and so for their arrivals too, before the CTA exits.
    const long long limit = a.limit_ns > kDrainNs ? a.limit_ns : kDrainNs;
    for (int j = consumed_a; j < issued_a; j++) mbar_wait(&full_a[j % SA], (uint32_t)(j / SA) & 1u, limit);
    for (int i = consumed_b; i < issued_b; i++) mbar_wait(&full_b[i % SB], (uint32_t)(i / SB) & 1u, limit);
    if (consumed_a > 0) {
      const int j = consumed_a - 1, i = consumed_a / NA - 1;  // the last steps that committed each barrier
      mbar_wait(&empty_a[j % SA], (uint32_t)(j / SA) & 1u, limit);
      if (i >= 0) mbar_wait(&empty_b[i % SB], (uint32_t)(i / SB) & 1u, limit);
      mbar_wait(&tfull[j % C::kBufs], (uint32_t)(j / C::kBufs) & 1u, limit);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------
// Operand preparation

// Constant right-hand operands from the complex column tables Xc[m][ix] (once per trap set), by
// component and part:
//   back    b[n = ix][k = m]  (W x ldb, rows padded to rows_b),
//   forward f[n = m][k = ix]  (M x ldu, rows padded to rows_f),
// and the row table transposed, YT[iy][m] = Y_m(iy) (m < Kp, zero beyond M).  Padding is zero.
struct TableArgs {
  int W, H, M, Kp, ldb, ldu, rows_b, rows_f;
  const float2 *Xc, *Yc;
  __half *b[2][2], *f[2][2];
  float2 *YT;
};

// One thread per two elements along K.
static __global__ void tc_tables_kernel(TableArgs a) {
  const long long nb = (long long)a.rows_b * (a.ldb / 2), nf = (long long)a.rows_f * (a.ldu / 2);
  const long long ny = (long long)a.H * (a.Kp / 2);
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nb + nf + ny; i += stride) {
    const long long j = i < nb ? i : i < nb + nf ? i - nb : i - nb - nf;
    const int half = i < nb ? a.ldb / 2 : i < nb + nf ? a.ldu / 2 : a.Kp / 2;
    const int n = (int)(j / half), k = 2 * (int)(j % half);
    float2 e[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      e[h] = make_float2(0.f, 0.f);
      if (i < nb) {
        if (n < a.W && k + h < a.M) e[h] = a.Xc[(size_t)(k + h) * a.W + n];
      } else if (i < nb + nf) {
        if (n < a.M && k + h < a.W) e[h] = a.Xc[(size_t)n * a.W + k + h];
      } else if (k + h < a.M) {
        e[h] = a.Yc[(size_t)(k + h) * a.H + n];
      }
    }
    if (i < nb)
      store_pair(a.b, (size_t)n * a.ldb + k, make_float2(e[0].x, e[1].x), make_float2(e[0].y, e[1].y));
    else if (i < nb + nf)
      store_pair(a.f, (size_t)n * a.ldu + k, make_float2(e[0].x, e[1].x), make_float2(e[0].y, e[1].y));
    else
      *reinterpret_cast<float4 *>(a.YT + (size_t)n * a.Kp + k) = make_float4(e[0].x, e[0].y, e[1].x, e[1].y);
  }
}

// The forward operand of given phases: u = e^{i phi} (unit_phasor), split; and one accumulator
// buffer cleared for the launch after next.
struct PhaseArgs {
  int W, H, ldu;
  const float *phi;
  __half *u[2][2];
  unsigned long long *acc_clear;
  int n_clear;
};
static __global__ void tc_phase_kernel(PhaseArgs a) {
  grid_wait();
  const int half = (a.W + 1) / 2;
  const long long n = (long long)a.H * half, stride = (long long)gridDim.x * blockDim.x;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n; j += stride) {
    const int iy = n <= 0x7fffffffll ? (int)((unsigned)j / (unsigned)half) : (int)(j / half);
    const int ix = 2 * (int)(j - (long long)iy * half);
    const float *ph = a.phi + (size_t)iy * a.W + ix;
    float2 sn, cs;
    unit_phasor(ph[0], sn.x, cs.x);
    sn.y = cs.y = 0.f;
    if (ix + 1 < a.W) unit_phasor(ph[1], sn.y, cs.y);
    store_pair(a.u, (size_t)iy * a.ldu + ix, cs, sn);
  }
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.n_clear; i += stride) a.acc_clear[i] = 0ull;
  grid_release();
}

struct PrepArgs {
  int H, M, Kp, ldb;                 // Kp: M padded (row stride of YT); ldb: row stride of P
  const unsigned long long *acc_in;  // [2][M] sums of the previous forward
  unsigned long long *acc_clear;     // [2][M] cleared here
  const float *w_in;
  float *w_out;                      // written by block 0
  const float2 *YT;                  // [H][Kp]
  __half *p[2][2];                   // [..][ldb] by component and part
  float inv_fx_n;
  float *trace;                      // NULL, or e, u of the fields read (block 0)
};

struct ffp {
  float hi, lo;
};
__device__ __forceinline__ ffp ffp_add(ffp a, ffp b) {  // TwoSum (Knuth) + renormalisation
  const float s = a.hi + b.hi;
  const float bb = s - a.hi;
  const float err = (a.hi - (s - bb)) + (b.hi - bb);
  const float e = err + (a.lo + b.lo);
  const float hi = s + e;
  return {hi, e - (hi - s)};
}

constexpr int kPrepThreads = 256;
constexpr int kPrepWeights = 4;   // weights a thread of tc_prep_kernel fetches before the wait
constexpr int kPrepPrefetch = 8;  // pairs of row-table elements a thread of tc_prep_kernel fetches before the wait

// Sec. 3 weight update and the back-projection operand of one iteration: every block reads the
// field sums, forms V_m and the coefficients c_m = w_m' V_m/|V_m| with w_m' = w_m <|V|>/|V_m|
// (|V_m| < 1e-30: c_m = w_m, w kept) in shared memory, up to a common factor -- so <|V|>, a block-wide
// sum, is not waited for unless a field vanishes -- then writes its share of P[iy][m] = c_m Y_m(iy),
// split.  Block 0 then writes the new weights (and the trace), <|V|> from a float-float sum in one
// fixed order; the blocks clear the next buffer.
// The row table is constant during hot_gsw, and the weights are the previous iteration's, which ended
// before the kernel ahead of this one could start: a thread's first elements of both are fetched before
// the wait for that kernel (the table comes from HBM: the GEMMs' operands have pushed it out of L2;
// the weights ahead of the wait save 0.2 us of 12 at 256^2, 1.5 of 100 at 1920 x 1152 with 1000 traps).
static __global__ void __launch_bounds__(kPrepThreads) tc_prep_kernel(PrepArgs a) {
  extern __shared__ float2 cs[];  // [M]
  __shared__ ffp part[2][kPrepThreads / 32];
  __shared__ float ext[2][kPrepThreads / 32];
  __shared__ float cmx[kPrepThreads / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // this block's rows of P: an even share of the H rows, all Kp (padded) traps of each, two at a time
  const int half = a.Kp / 2;
  const float4 *const YT = reinterpret_cast<const float4 *>(a.YT);
  const int r0 = (int)((long long)a.H * blockIdx.x / gridDim.x);
  const int r1 = (int)((long long)a.H * (blockIdx.x + 1) / gridDim.x);
  const int n = (r1 - r0) * half;
  float4 ypre[kPrepPrefetch];
#pragma unroll
  for (int j = 0; j < kPrepPrefetch; j++) {
    const int i = t + j * kPrepThreads;
    ypre[j] = i < n ? __ldg(YT + (size_t)r0 * half + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float wpre[kPrepWeights];
#pragma unroll
  for (int j = 0; j < kPrepWeights; j++) wpre[j] = t + j * kPrepThreads < a.M ? __ldcg(a.w_in + t + j * kPrepThreads) : 0.f;
  grid_wait();
  ffp s = {0.f, 0.f}, si = {0.f, 0.f};
  float mx = -1.f, mn = 3.0e38f;
#pragma unroll 4
  for (int m = t; m < a.M; m += kPrepThreads) {
    const float vr = (float)(long long)__ldcg(a.acc_in + m) * a.inv_fx_n;
    const float vi = (float)(long long)__ldcg(a.acc_in + a.M + m) * a.inv_fx_n;
    cs[m] = make_float2(vr, vi);
    const float I = vr * vr + vi * vi;
    s = ffp_add(s, {sqrtf(I), 0.f});
    si = ffp_add(si, {I, 0.f});
    mx = fmaxf(mx, I);
    mn = fminf(mn, I);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    s = ffp_add(s, {__shfl_down_sync(0xffffffffu, s.hi, o), __shfl_down_sync(0xffffffffu, s.lo, o)});
    si = ffp_add(si, {__shfl_down_sync(0xffffffffu, si.hi, o), __shfl_down_sync(0xffffffffu, si.lo, o)});
    mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    mn = fminf(mn, __shfl_down_sync(0xffffffffu, mn, o));
  }
  if (lane == 0) {
    part[0][warp] = s;
    part[1][warp] = si;
    ext[0][warp] = mx;
    ext[1][warp] = mn;
  }
  // the coefficients over <|V|> (arg S does not depend on a common factor)
  float cmax = 0.f;  // largest magnitude: they are scaled by its inverse below
  bool zero = false;
  auto coefficient = [&](int m, float w) {
    const float2 v = cs[m];
    const float am = sqrtf(v.x * v.x + v.y * v.y), wn = w / am;
    if (am >= 1e-30f) {
      cs[m] = make_float2(wn * (v.x / am), wn * (v.y / am));
      cmax = fmaxf(cmax, wn);
    } else {
      zero = true;
    }
  };
#pragma unroll
  for (int j = 0; j < kPrepWeights; j++)
    if (t + j * kPrepThreads < a.M) coefficient(t + j * kPrepThreads, wpre[j]);
  for (int m = t + kPrepWeights * kPrepThreads; m < a.M; m += kPrepThreads) coefficient(m, __ldcg(a.w_in + m));
#pragma unroll
  for (int o = 16; o; o >>= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
  if (lane == 0) cmx[warp] = cmax;
  const long long stride = (long long)gridDim.x * kPrepThreads;
  for (long long i = blockIdx.x * (long long)kPrepThreads + t; i < 2LL * a.M; i += stride) a.acc_clear[i] = 0ull;
  const bool any_zero = __syncthreads_or(zero);
  // A factor common to all coefficients leaves arg S unchanged (Sec. 4; the weights' scale is
  // free): P is formed from c_m / max |c| so that its magnitudes stay near 1 whatever the
  // weights' scale (the FP16 operands lose precision below ~0.25).
  float top = cmx[0];
  for (int i = 1; i < kPrepThreads / 32; i++) top = fmaxf(top, cmx[i]);
  auto mean_field = [&] {
    ffp q = part[0][0];
    for (int i = 1; i < kPrepThreads / 32; i++) q = ffp_add(q, part[0][i]);
    return (q.hi + q.lo) / (float)a.M;
  };
  if (any_zero) {  // vanishing fields: c_m = w_m / <|V|> in this scale (w_m where every field vanishes)
    const float mean = mean_field(), inv = mean > 0.f ? 1.f / mean : 1.f;
    float zmax = 0.f;
    for (int m = 0; m < a.M; m++) {  // (every thread: the largest of them)
      const float vr = (float)(long long)__ldcg(a.acc_in + m) * a.inv_fx_n;
      const float vi = (float)(long long)__ldcg(a.acc_in + a.M + m) * a.inv_fx_n;
      if (sqrtf(vr * vr + vi * vi) >= 1e-30f) continue;
      const float w = __ldcg(a.w_in + m) * inv;
      zmax = fmaxf(zmax, w);
      if (m % kPrepThreads == t) cs[m] = make_float2(w, 0.f);
    }
    top = fmaxf(top, zmax);
    __syncthreads();
  }
  const float scale = top > 0.f ? 1.f / top : 1.f;
  // pair i of the block's rows is P[r0 + i / half][m = 2 (i % half), + 1], pair i of the row table
  auto put = [&](int i, float4 y) {
    const int m = 2 * (i % half);
    float2 c[2];
#pragma unroll
    for (int h = 0; h < 2; h++)
      c[h] = m + h < a.M ? make_float2(cs[m + h].x * scale, cs[m + h].y * scale) : make_float2(0.f, 0.f);
    store_pair(a.p, (size_t)(r0 + i / half) * a.ldb + m,
               make_float2(c[0].x * y.x - c[0].y * y.y, c[1].x * y.z - c[1].y * y.w),
               make_float2(c[0].x * y.y + c[0].y * y.x, c[1].x * y.w + c[1].y * y.z));
  };
#pragma unroll
  for (int j = 0; j < kPrepPrefetch; j++)
    if (t + j * kPrepThreads < n) put(t + j * kPrepThreads, ypre[j]);
  for (int i = t + kPrepPrefetch * kPrepThreads; i < n; i += kPrepThreads) put(i, __ldg(YT + (size_t)r0 * half + i));
  grid_release();
  if (blockIdx.x) return;
  // Block 0: the weights w_m' = w_m <|V|>/|V_m| (Sec. 3), and e, u (Eq. 4) of the fields read
  const float mean = mean_field();
  for (int m = t; m < a.M; m += kPrepThreads) {
    const float w = __ldcg(a.w_in + m);
    const float vr = (float)(long long)__ldcg(a.acc_in + m) * a.inv_fx_n;
    const float vi = (float)(long long)__ldcg(a.acc_in + a.M + m) * a.inv_fx_n;
    const float am = sqrtf(vr * vr + vi * vi);
    a.w_out[m] = am < 1e-30f ? w : w * mean / am;
  }
  if (a.trace && t == 0) {
    ffp e = part[1][0];
    float hi = ext[0][0], lo = ext[1][0];
    for (int i = 1; i < kPrepThreads / 32; i++) {
      e = ffp_add(e, part[1][i]);
      hi = fmaxf(hi, ext[0][i]);
      lo = fminf(lo, ext[1][i]);
    }
    a.trace[0] = e.hi + e.lo;
    a.trace[1] = (hi + lo > 0.f) ? 1.f - (hi - lo) / (hi + lo) : 0.f;
  }
}

// Operands of the plain GEMM entry point: src [rows][K] -> hi, lo [rows_pad][K_pad], zero padded.
template <int OP>
__global__ void tc_split_kernel(const float *src, int rows, int K, int K_pad, long long total, void *hi, void *lo) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / K_pad), k = (int)(i % K_pad);
    const float x = (r < rows && k < K) ? src[(size_t)r * K + k] : 0.f;
    const float2 h = split2<OP>(x);
    store1<OP>(hi, i, h.x);
    store1<OP>(lo, i, h.y);
  }
}

}  // namespace tc
