// tile_kernels.cuh -- the register-tiled step kernel of the accurate, fast and separable modes.
//
// Eq. 2 is a sum of a column part and a row part, so a pair's exponential is the product of two
// tabulated unit phasors, e^{i Delta_j^m} = X_m(ix) Y_m(iy) (cos and sin of the exactly reduced
// turns, rounded to FP32 once per trap set).  Both sums of an iteration are then complex
// multiply-adds,
//   S_j = sum_m (c_m X_m(ix)) Y_m(iy)                            (back-projection, Sec. 3-4)
//   N V_m = sum_ix conj(X_m(ix)) sum_iy u_j conj(Y_m(iy))        (forward field, Eq. 1),
// 8 FP32 FMA per pixel-trap pair and iteration and no transcendental function per pair.
//
// What bounds it: the FP32 pipe behind its register ports.  A packed multiply-add (fma.rn.f32x2)
// on three different register pairs takes 3 cycles (two words per bank and cycle), so a step over
// two traps cannot go below 12 cycles per 32 pairs; scalar multiply-adds came out the same.  A thread
// keeps 16 rows x 2 columns of pixels in registers, packed over row pairs, and walks the traps: one
// broadcast 16-byte load per row pair and two 8-byte column loads per trap for 64 multiply-adds.
// Alone (no exchange, no field sums) the two loops take 6.9 + 7.0 cycles per 32 pairs, 5.8 + 6.4
// without the table ring.  Taller tiles (32 rows, one block per SM) run 5 % faster at 1920 x 1152
// but 5-15 % slower at 512^2.
//
// Work split: a warp's tile is 64 columns x up to 16 rows.  A team of `team` warps (1, 2, 4 or 8 of
// the block's 8) shares a tile and splits the traps; its partial superpositions meet in shared
// memory, in warp order.  Each warp streams its own traps' table rows through a private ring in
// shared memory (cp.async), so no barrier stands in the trap loops.
#pragma once
#include "gsw_kernels.cuh"
#include "turns.cuh"

namespace hot {

constexpr int kTileCols = 64;     // columns of a warp's tile: two per lane, 32 apart
constexpr int kTilePairs = 8;     // row pairs of a tile at most
constexpr int kRing = 3;          // stages of a warp's table ring, two traps each
constexpr int kStageX = kTileCols * 8, kStageY = kTilePairs * 16;  // bytes of a trap in a stage
constexpr int kStageBytes = 2 * (kStageX + kStageY);
constexpr int kSumGroup = 8;      // traps whose field sums a warp reduces together
constexpr int kSumStride = 36;    // ... and the stride of their lane sums: eight lanes' columns of four traps
                                  // fall on different banks (33: 858 us per iteration at 1920 x 1152,
                                  // M = 1000 in groups of 4; 36: 840)

struct TileArgs {
  StepArgs s;        // sub: tiles (rows = row pairs, y0 even)
  const float2 *X;   // [strips][Mp][kTileCols] column phasors of the 64-column strips, zero from W on
  const float4 *Y;   // [Mp][ldp] row phasors by row pair: (re, re, im, im), zero from H on
  int Mp, ldp;       // Mp: M rounded up to a whole number of trap pairs (the added trap: zeros)
  int team;          // warps that share a tile
  int stride;        // team i's tiles are sub[i stride], ...; the first one's pad says how many
  int pairs;         // row pairs of the tallest tile, at least 3 (shared memory is sized by it)
};


constexpr int kSumBytes = kSumGroup * kSumStride * 8;  // lane sums of kSumGroup traps
constexpr int kOwnMax = 32;  // traps a block keeps for its weight updates (more are read again)

__host__ __device__ constexpr int tile_smem_bytes(int M, int team, int pairs) {
  return (M + 1) / 2 * 16 + kWarps * (kRing * kStageBytes + pairs * 1024) + (team > 1 ? kWarps / team * kSumBytes : 0);
}

// What the weight update at a launch's end keeps from its start (static shared memory: no register
// holds an address across the trap loops, where they are short).
struct OwnWeights {
  ff part[kThreads];    // the threads' shares of sum |V_m|
  float2 own[kOwnMax];  // weight and |V_m| of the block's own traps
};
__device__ __forceinline__ OwnWeights &own_weights() {
  __shared__ OwnWeights w;
  return w;
}

struct TileSmem {
  float2 *C;            // [Mp] coefficients (0 for the added trap)
  unsigned char *ring;  // this warp's stages
  float4 *S;            // [team][2 pairs][32] the team's partial superpositions (rows 2p, 2p+1: re, re, im, im);
                        // the first part then takes the tile's unit phasors
  float2 *sums;         // [kSumGroup][kSumStride] lane sums of the warp's current traps: in its part of S, or apart
                        // where the phasors are
  int team, g;          // warps of the team, this warp's place in it
  int part_stride;      // float4 from one warp's part of S to the next
  __device__ __forceinline__ TileSmem(unsigned char *raw, int M, int team_, int pairs)
      : team(team_), part_stride(pairs * 64) {
    const int warp = threadIdx.x >> 5;
    g = warp & (team - 1);
    C = reinterpret_cast<float2 *>(raw);
    raw += (M + 1) / 2 * 16;
    ring = raw + warp * kRing * kStageBytes;
    raw += kWarps * kRing * kStageBytes;
    S = reinterpret_cast<float4 *>(raw) + (warp - g) * part_stride;
    sums = reinterpret_cast<float2 *>(g == 0 && team > 1 ? raw + kWarps * pairs * 1024 + warp / team * kSumBytes
                                                         : raw + warp * pairs * 1024);
  }
  // Barrier of the team (ids 2 .. 9).
  __device__ __forceinline__ void sync() const {
    if (team == 1)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(2 + (int)(threadIdx.x >> 5) / team), "r"(32 * team) : "memory");
  }
};

// The trap pairs [lo, hi) of warp g of a team (teams of 8: the pairs of warps that share an SM
// sub-partition get equal shares to within one, see warp_traps).
__device__ __forceinline__ void team_traps(int M, int team, int g, int &lo, int &hi) {
  const int n = (M + 1) / 2;
  if (team == kWarps) {
    warp_traps(n, g, lo, hi);
  } else {
    lo = g * n / team;
    hi = (g + 1) * n / team;
  }
}

// A warp's stream of table rows: for each of its tiles, `passes` times its trap pairs lo .. lo + T - 1,
// one stage per pair, kRing - 1 stages ahead of the consumer.
struct TileStream {
  const TileArgs &a;
  unsigned int ring;             // shared address of the warp's stages
  int lo, T, passes, tile, end;  // of the producer
  int k, pass, fill;
  const float2 *x;
  const float4 *y;
  __device__ __forceinline__ TileStream(const TileArgs &args, const TileSmem &sm, int passes_, int t_begin, int t_end)
      : a(args), ring((unsigned)__cvta_generic_to_shared(sm.ring)), passes(passes_), tile(t_begin), end(t_end), k(0),
        pass(0), fill(0), x(nullptr), y(nullptr) {
    int hi;
    team_traps(a.s.M, sm.team, sm.g, lo, hi);
    T = hi - lo;
    if (T == 0) tile = end;
    seek();
    for (int i = 0; i < kRing - 1; i++) issue();
  }
  __device__ __forceinline__ void seek() {
    if (tile >= end) return;
    const SubTile st = a.s.sub[tile];
    const int lane = threadIdx.x & 31;
    x = a.X + ((size_t)(st.x0 / kTileCols) * a.Mp + 2 * lo) * kTileCols + 2 * lane;
    y = a.Y + (size_t)(2 * lo + ((lane >> 3) & 1)) * a.ldp + (st.y0 >> 1) + (lane & 7);
  }
  // Starts the copies of the next pair's 2 x 64 column and 2 x 8 row-pair phasors (always one group).
  __device__ __forceinline__ void issue() {
    if (tile < end) {
      const int lane = threadIdx.x & 31;
      const unsigned st = ring + fill + 16 * lane;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(st), "l"(x) : "memory");
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(st + kStageX), "l"(x + kTileCols) : "memory");
      if (lane < 2 * kTilePairs)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(st + 2 * kStageX), "l"(y) : "memory");
      x += 2 * kTileCols;
      y += 2 * a.ldp;
      if (++k == T) {
        k = 0;
        if (++pass == passes) {
          pass = 0;
          tile++;
        }
        seek();
      }
    }
    cp_async_commit();
    fill = fill == (kRing - 1) * kStageBytes ? 0 : fill + kStageBytes;
  }
  // The next pair's stage (byte offset in the ring); frees the one before it.
  __device__ __forceinline__ int next() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 2) : "memory");
    __syncwarp();
    issue();
    return fill;  // kRing - 1 stages ahead of the stage to read: the one after the stage just filled
  }
};

// Sec. 3 coefficients of all traps from the previous launch's sums, without the common factor
// <|V|> (arg S_j does not depend on it), into C, and the threads' shares of sum |V_m| into part;
// explicit coefficients a.G instead when given.  trace: NULL, or where block 0 writes e and u
// (Eq. 4) of the fields read.  The block synchronises afterwards.
// own, stride: the traps whose weights the block writes (own + stride k, tile_weights).
__device__ __forceinline__ void tile_prologue(const StepArgs &a, const TileSmem &sm, int own, int stride, float *trace) {
  const int t = threadIdx.x;
  if (t == 0 && (a.M & 1)) sm.C[a.M] = make_float2(0.f, 0.f);
  if (a.G) {
    for (int m = t; m < a.M; m += kThreads) sm.C[m] = a.G[m];
    return;
  }
  ff s = {0.f, 0.f}, si = {0.f, 0.f};
  float mx = -1.f, mn = 3.0e38f;
  const bool tr = trace && blockIdx.x == 0;
  for (int m = t; m < a.M; m += kThreads) {
    const float2 v = field_from_sums<true>(a, m);
    const float w = __ldcg(a.w_in + m), I = abs2(v), am = sqrtf(I);
    const float r = 1.f / am;  // (w / |V|) (V / |V|): no |V|^2 in the denominator, which could underflow
    sm.C[m] = am < 1e-30f ? make_float2(w, 0.f) : make_float2((w * r) * (v.x * r), (w * r) * (v.y * r));
    s = ff_add(s, {am, 0.f});
    const int k = (m - own) / stride;
    if (m >= own && k * stride == m - own && k < kOwnMax) own_weights().own[k] = make_float2(w, am);
    if (tr) {
      si = ff_add(si, {I, 0.f});
      mx = fmaxf(mx, I);
      mn = fminf(mn, I);
    }
  }
  own_weights().part[t] = s;
  if (!tr) return;
  __shared__ ff tpart[kWarps];
  __shared__ float ext[2][kWarps];
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    si = ff_add(si, {__shfl_down_sync(0xffffffffu, si.hi, o), __shfl_down_sync(0xffffffffu, si.lo, o)});
    mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    mn = fminf(mn, __shfl_down_sync(0xffffffffu, mn, o));
  }
  if ((t & 31) == 0) {
    tpart[t >> 5] = si;
    ext[0][t >> 5] = mx;
    ext[1][t >> 5] = mn;
  }
  __syncthreads();
  if (t == 0) {
    ff e = tpart[0];
    float hi = ext[0][0], lo = ext[1][0];
    for (int i = 1; i < kWarps; i++) {
      e = ff_add(e, tpart[i]);
      hi = fmaxf(hi, ext[0][i]);
      lo = fminf(lo, ext[1][i]);
    }
    trace[0] = e.hi + e.lo;
    trace[1] = (hi + lo > 0.f) ? 1.f - (hi - lo) / (hi + lo) : 0.f;
  }
}

// Blocks that own weights (own < M; a block-uniform condition), after the block's work: <|V|> from
// the prologue's shares in one fixed order, and w_m <- w_m <|V|>/|V_m| of traps own + stride t, ...
// (the sums they come from are cleared by the next launch only).
__device__ __forceinline__ void tile_weights(const StepArgs &a, const TileSmem &sm, int own, int stride) {
  if (own >= a.M) return;
  __shared__ ff wpart[kWarps];
  const int t = threadIdx.x;
  ff s = own_weights().part[t];
#pragma unroll
  for (int o = 16; o; o >>= 1)
    s = ff_add(s, {__shfl_down_sync(0xffffffffu, s.hi, o), __shfl_down_sync(0xffffffffu, s.lo, o)});
  if ((t & 31) == 0) wpart[t >> 5] = s;
  __syncthreads();
  ff q = wpart[0];
#pragma unroll
  for (int i = 1; i < kWarps; i++) q = ff_add(q, wpart[i]);
  const float mean = (q.hi + q.lo) / (float)a.M;
  for (int k = t; own + stride * k < a.M; k += kThreads) {
    const int m = own + stride * k;
    const float2 wv = k < kOwnMax ? own_weights().own[k] : make_float2(__ldcg(a.w_in + m), sqrtf(abs2(field_from_sums<true>(a, m))));
    a.w_out[m] = wv.y < 1e-30f ? wv.x : wv.x * mean / wv.y;  // (Sec. 3; a vanishing field keeps its weight)
  }
}

// S_{r, c} += (c_m X_m(c)) Y_m(r) of a stage's two traps on the lane's RP row pairs x 2 columns.
template <int RP>
__device__ __forceinline__ void tile_back(const unsigned char *st, float4 c2, int lane, unsigned long long (&Sr)[RP][2],
                                          unsigned long long (&Si)[RP][2]) {
  const float2 *X = reinterpret_cast<const float2 *>(st) + lane;
  const ulonglong2 *Y = reinterpret_cast<const ulonglong2 *>(st + 2 * kStageX);
  unsigned long long rr[2][2], ii[2][2], ni[2][2];
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const float2 c = k ? make_float2(c2.z, c2.w) : make_float2(c2.x, c2.y);
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const float2 x = X[k * kTileCols + 32 * q];
      const float br = fmaf(c.x, x.x, -__fmul_rn(c.y, x.y)), bi = fmaf(c.x, x.y, __fmul_rn(c.y, x.x));
      rr[k][q] = pack2(br, br);
      ii[k][q] = pack2(bi, bi);
      ni[k][q] = pack2(-bi, -bi);
    }
  }
#pragma unroll
  for (int p = 0; p < RP; p++) {
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const ulonglong2 y = Y[k * kTilePairs + p];  // (re of the two rows), (im of the two rows)
#pragma unroll
      for (int q = 0; q < 2; q++) {
        Sr[p][q] = fma2(y.x, rr[k][q], Sr[p][q]);
        Si[p][q] = fma2(y.x, ii[k][q], Si[p][q]);
      }
#pragma unroll
      for (int q = 0; q < 2; q++) {
        Sr[p][q] = fma2(y.y, ni[k][q], Sr[p][q]);
        Si[p][q] = fma2(y.y, rr[k][q], Si[p][q]);
      }
    }
  }
}

// sum over the lane's pixels of u_{r, c} conj(X_m(c) Y_m(r)) of a stage's two traps.
template <int RP>
__device__ __forceinline__ void tile_forward(const unsigned char *st, int lane, const unsigned long long (&ur)[RP][2],
                                             const unsigned long long (&ui)[RP][2], float2 (&v)[2]) {
  const float2 *X = reinterpret_cast<const float2 *>(st) + lane;
  const ulonglong2 *Y = reinterpret_cast<const ulonglong2 *>(st + 2 * kStageX);
  unsigned long long t[2][2], A[2][2], B[2][2];
#pragma unroll
  for (int p = 0; p < RP; p++) {
    const ulonglong2 y0 = Y[p], y1 = Y[kTilePairs + p];
#pragma unroll
    for (int q = 0; q < 2; q++) {
      if (p == 0) {
        t[0][q] = mul2(ur[0][q], y0.x);
        t[1][q] = mul2(ur[0][q], y1.x);
        B[0][q] = mul2(ur[0][q], y0.y);
        B[1][q] = mul2(ur[0][q], y1.y);
        A[0][q] = mul2(ui[0][q], y0.x);
        A[1][q] = mul2(ui[0][q], y1.x);
        t[0][q] = fma2(ui[0][q], y0.y, t[0][q]);
        t[1][q] = fma2(ui[0][q], y1.y, t[1][q]);
        continue;
      }
      t[0][q] = fma2(ur[p][q], y0.x, t[0][q]);
      t[1][q] = fma2(ur[p][q], y1.x, t[1][q]);
      B[0][q] = fma2(ur[p][q], y0.y, B[0][q]);
      B[1][q] = fma2(ur[p][q], y1.y, B[1][q]);
      A[0][q] = fma2(ui[p][q], y0.x, A[0][q]);
      A[1][q] = fma2(ui[p][q], y1.x, A[1][q]);
      t[0][q] = fma2(ui[p][q], y0.y, t[0][q]);
      t[1][q] = fma2(ui[p][q], y1.y, t[1][q]);
    }
  }
#pragma unroll
  for (int k = 0; k < 2; k++) {
    v[k] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const float2 x = X[k * kTileCols + 32 * q], t2 = unpack2(t[k][q]), d2 = unpack2(fma2(B[k][q], pack2(-1.f, -1.f), A[k][q]));
      const float tr = t2.x + t2.y, ti = d2.x + d2.y;
      v[k].x = fmaf(ti, x.y, fmaf(tr, x.x, v[k].x));
      v[k].y = fmaf(-tr, x.y, fmaf(ti, x.x, v[k].y));
    }
  }
}

// The value of one pixel from its superposition: the phase (written), and its unit phasor for the
// forward field; or the gradient of the adjoint.
template <bool FWD, bool ADJ>
__device__ __forceinline__ float2 tile_pixel(const StepArgs &a, int flags, float2 s, int row, int col) {
  const bool in = row < a.H && col < a.W;
  const size_t j = (size_t)row * a.W + col;
  float2 u = make_float2(0.f, 0.f);
  if (ADJ) {
    if (in) {
      float sp, cp;
      sincosf(a.phi[j], &sp, &cp);
      a.grad[j] = fmaf(cp, s.y, -__fmul_rn(sp, s.x)) * a.inv_n;  // Im[(cos - i sin)(S.x + i S.y)] / N
    }
    return u;
  }
  if (flags & kOnceState) {
    u = unit_of(s);
    if ((flags & kOnceLast) && in) {
      a.phi[j] = atan2f(s.y, s.x);
      if (a.u) a.u[j] = u;
    }
    return u;
  }
  const float ph = atan2f(s.y, s.x);
  if (in) a.phi[j] = ph;
  if (FWD) sincosf(ph, &u.y, &u.x);  // of the stored phase, so that a resumed run is identical
  return u;
}

// The unit phasor of a given pixel phase (0 outside the image).
__device__ __forceinline__ float2 tile_given(const StepArgs &a, int flags, int row, int col) {
  float2 u = make_float2(0.f, 0.f);
  if (row < a.H && col < a.W) {
    const size_t j = (size_t)row * a.W + col;
    if (flags & kOnceReadU)
      u = a.u[j];
    else
      sincosf(a.phi[j], &u.y, &u.x);
  }
  return u;
}

// Forward field of a tile: the team's phasors (in sm.S) against the warp's traps, the sums added in
// fixed point.  P, Q: registers for the phasors' real and imaginary parts.
template <int RP>
__device__ __forceinline__ void tile_fields(const StepArgs &a, const TileSmem &sm, TileStream &in,
                                            unsigned long long (&P)[RP][2], unsigned long long (&Q)[RP][2]) {
  const int lane = threadIdx.x & 31, lo = 2 * in.lo, T = in.T;
#pragma unroll
  for (int p = 0; p < RP; p++)
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const ulonglong2 u = reinterpret_cast<const ulonglong2 *>(sm.S)[(2 * p + q) * 32 + lane];
      P[p][q] = u.x;
      Q[p][q] = u.y;
    }
  if (sm.team == 1) __syncwarp();  // (the phasors lie in the scratch)
  float2 *const vb = sm.sums;
  unsigned long long *const out = block_acc(a);
  for (int k = 0; k < 2 * T; k += 2) {
    float2 v2[2];
    tile_forward<RP>(sm.ring + in.next(), lane, P, Q, v2);
    const int j = k & (kSumGroup - 1);
    vb[j * kSumStride + lane] = v2[0];
    vb[(j + 1) * kSumStride + lane] = v2[1];
    if (j + 2 == kSumGroup || k + 2 == 2 * T) {  // the group's totals: lane l sums trap l / 4
      __syncwarp();
      const int tr = lane >> 2, sub = lane & 3;
      float2 v8[8];
#pragma unroll
      for (int i = 0; i < 8; i++) v8[i] = vb[tr * kSumStride + sub + 4 * i];
#pragma unroll
      for (int w = 4; w; w >>= 1)
#pragma unroll
        for (int i = 0; i < w; i++) {
          v8[i].x += v8[i + w].x;
          v8[i].y += v8[i + w].y;
        }
      float2 v = v8[0];
#pragma unroll
      for (int o = 2; o; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      }
      // |v| <= 1024 pixels, so v * 2^fx_shift is an exact integer far below 2^63
      const int m = lo + k - j + tr;
      if (tr < j + 2 && m < a.M && sub < 2)
        atomicAdd(out + (sub ? a.M : 0) + m, (unsigned long long)__float2ll_rn((sub ? v.y : v.x) * a.fx_scale));
    }
  }
}

// One tile of RP row pairs: back-projection and/or forward field.
template <int RP, bool BACK, bool FWD, bool ADJ>
__device__ __forceinline__ void tile_one(const StepArgs &a, const TileSmem &sm, TileStream &in, const SubTile st,
                                         int flags) {
  const int lane = threadIdx.x & 31;
  unsigned long long P[RP][2], Q[RP][2];  // (re, re), (im, im) of the row pairs: S, then u
  if (BACK) {
#pragma unroll
    for (int p = 0; p < RP; p++)
#pragma unroll
      for (int q = 0; q < 2; q++) P[p][q] = Q[p][q] = 0ull;
    const float4 *C = reinterpret_cast<const float4 *>(sm.C) + in.lo;
    for (int k = 0; k < in.T; k++) {
      const unsigned char *const stage = sm.ring + in.next();
      tile_back<RP>(stage, C[k], lane, P, Q);
    }
    sm.sync();  // the phasors and lane sums of the tile before are read
    ulonglong2 *const mine = reinterpret_cast<ulonglong2 *>(sm.S + sm.g * sm.part_stride);
#pragma unroll
    for (int p = 0; p < RP; p++)
#pragma unroll
      for (int q = 0; q < 2; q++) mine[(2 * p + q) * 32 + lane] = make_ulonglong2(P[p][q], Q[p][q]);
  }
  sm.sync();  // the team's superpositions are written (FWD alone: the phasors and lane sums of the tile before read)
#pragma unroll 1
  for (int i = sm.g; i < 2 * RP; i += sm.team) {
    const int row = st.y0 + (i & ~1), col = st.x0 + 32 * (i & 1) + lane;
    float2 u0, u1;
    if (BACK) {
      float4 s = sm.S[i * 32 + lane];
      for (int w = 1; w < sm.team; w++) {
        const float4 q = sm.S[w * sm.part_stride + i * 32 + lane];
        s.x += q.x;
        s.y += q.y;
        s.z += q.z;
        s.w += q.w;
      }
      u0 = tile_pixel<FWD, ADJ>(a, flags, make_float2(s.x, s.z), row, col);
      u1 = tile_pixel<FWD, ADJ>(a, flags, make_float2(s.y, s.w), row + 1, col);
    } else {
      u0 = tile_given(a, flags, row, col);
      u1 = tile_given(a, flags, row + 1, col);
    }
    if (FWD) sm.S[i * 32 + lane] = make_float4(u0.x, u1.x, u0.y, u1.y);
  }
  sm.sync();  // the phasors are complete; the superpositions are read
  if constexpr (FWD) tile_fields<RP>(a, sm, in, P, Q);
}

template <bool BACK, bool FWD, bool ADJ>
__device__ __forceinline__ void tile_run(const StepArgs &a, const TileSmem &sm, TileStream &in, int t_begin, int t_end,
                                         int flags) {
  for (int t = t_begin; t < t_end; t++) {
    const SubTile st = a.sub[t];
    switch (st.rows) {
      case 1: tile_one<1, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      case 2: tile_one<2, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      case 3: tile_one<3, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      case 4: tile_one<4, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      case 5: tile_one<5, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      case 6: tile_one<6, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      case 7: tile_one<7, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
      default: tile_one<8, BACK, FWD, ADJ>(a, sm, in, st, flags); break;
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}
static_assert(kTilePairs == 8, "tile_run covers 1..8 row pairs");

// One launch: weight update, back-projection and forward field (BACK, FWD), the field of given
// phases (FWD), a superposition (BACK), or the adjoint (BACK, ADJ).
template <bool BACK, bool FWD, bool ADJ>
__global__ void __launch_bounds__(kThreads, 2) gsw_tile_kernel(const __grid_constant__ TileArgs t) {
  static_assert(!ADJ || (BACK && !FWD), "the adjoint is a back-projection without forward field");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const StepArgs &a = t.s;
  const TileSmem sm(smem_raw, a.M, t.team, t.pairs);
  const int t_begin = (blockIdx.x * (kWarps / t.team) + (threadIdx.x >> 5) / t.team) * t.stride;
  const int t_end = t_begin + a.sub[t_begin].pad;
  allow_dependents();
  TileStream in(t, sm, (BACK ? 1 : 0) + (FWD ? 1 : 0), t_begin, t_end);  // the tables are constant during a sequence
  grid_dependency_wait();
  if (FWD)
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < 2 * a.M * a.copies; i += gridDim.x * kThreads) a.acc_clear[i] = 0ull;
  if (BACK) {
    tile_prologue(a, sm, blockIdx.x, gridDim.x, a.trace);
    __syncthreads();
  }
  tile_run<BACK, FWD, ADJ>(a, sm, in, t_begin, t_end, a.once_flags);
  if (BACK && FWD && !a.G) tile_weights(a, sm, blockIdx.x, gridDim.x);
}

// Persistent form: all launches of a call in one cooperative launch (see gsw_persistent_kernel),
// launch k with step[k % 6].
struct TilePersistArgs {
  TileArgs step[6];
  int iters;
  GridSync sync;
  float *trace;  // NULL, or [iters][2]
};

static __global__ void __launch_bounds__(kThreads, 2) gsw_tile_persistent_kernel(const __grid_constant__ TilePersistArgs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TileArgs &t0 = p.step[0];
  const TileSmem sm(smem_raw, t0.s.M, t0.team, t0.pairs);
  const int t_begin = (blockIdx.x * (kWarps / t0.team) + (threadIdx.x >> 5) / t0.team) * t0.stride;
  const int t_end = t_begin + t0.s.sub[t_begin].pad;
  unsigned int epoch = 0u;
  for (int k = 0; k <= p.iters; k++) {
    const TileArgs &t = p.step[k % 6];
    const StepArgs &a = t.s;
    TileStream in(t, sm, k ? 2 : 1, t_begin, t_end);
    const bool go = k == 0 || grid_sync(p.sync, epoch);
    if (!go) {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      return;
    }
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < 2 * a.M * a.copies; i += gridDim.x * kThreads) a.acc_clear[i] = 0ull;
    if (k == 0) {
      tile_run<false, true, false>(a, sm, in, t_begin, t_end, a.once_flags & ~kOnceLast);
    } else {
      tile_prologue(a, sm, blockIdx.x, gridDim.x, p.trace ? p.trace + 2 * (k - 1) : nullptr);
      __syncthreads();
      tile_run<true, true, false>(a, sm, in, t_begin, t_end, (a.once_flags & ~(kOnceReadU | kOnceLast)) | (k == p.iters ? kOnceLast : 0));
      tile_weights(a, sm, blockIdx.x, gridDim.x);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Tables of the column and row phasors (once per trap set), from the phases of turns.cuh.

struct TileTables {
  int W, H, H_total, y_off;  // a row band: rows y_off .. of a hologram of H_total rows
  int M, Mp, ldp;
  const double *abc;  // [M][3] turns per pixel index (see the file header of gsw_kernels.cuh)
  float2 *X;          // TileArgs::X, Y
  float4 *Y;
  float2 *Xc, *Yc;    // NULL, or [M][W], [M][H] (tensor mode)
};

// One thread per column and row pair of a trap (blockIdx.y); what lies outside the image stays zero.
static __global__ void __launch_bounds__(128) tile_tables_kernel(TileTables t) {
  const int m = blockIdx.y, j = blockIdx.x * 128 + threadIdx.x, P = (t.H + 1) / 2;
  if (j >= t.W + P) return;
  const bool col = j < t.W;
  const TrapTurns k = trap_turns(t.abc[3 * m + (col ? 0 : 1)], t.abc[3 * m + 2]);
  if (col) {
    const float2 e = cis_turns(phase_at(k, j - t.W / 2));
    t.X[((size_t)(j / kTileCols) * t.Mp + m) * kTileCols + j % kTileCols] = e;
    if (t.Xc) t.Xc[(size_t)m * t.W + j] = e;
    return;
  }
  const int p = j - t.W, q = 2 * p + t.y_off - t.H_total / 2;
  const bool two = 2 * p + 1 < t.H;
  const float2 e = cis_turns(phase_at(k, q)), f = two ? cis_turns(phase_at(k, q + 1)) : make_float2(0.f, 0.f);
  t.Y[(size_t)m * t.ldp + p] = make_float4(e.x, f.x, e.y, f.y);
  if (t.Yc) {
    t.Yc[(size_t)m * t.H + 2 * p] = e;
    if (two) t.Yc[(size_t)m * t.H + 2 * p + 1] = f;
  }
}

}  // namespace hot
