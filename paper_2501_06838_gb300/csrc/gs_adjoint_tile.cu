// Tile adjoint of the scale-aware 2D Gaussian render (GSASR, arXiv 2501.06838,
// Eq. 4 with the Algorithm-1 window; differentiable render, Sec. 3.1 "Fast
// Rasterization" and Sec. 3.2 "Rendering"), one lane per Gaussian.
//
// The exponent of a record is the completed square (log2 units, HR pixels)
//   e = -d^2 + g Y^2 + l,   d = sA X - sK Y,   X = x - cx, Y = y - cy,
// and the render adds c_k 2^e to channel k (c the record colour alpha * rgb).
// For every (tile, Gaussian) pair of the forward's per-tile lists this kernel
// adds the Gaussian's record-space moments over the tile's pixels,
//   Sd = sum Gw d, SY = sum Gw Y, Sdd = sum Gw d^2, SdY = sum Gw d Y,
//   SYY = sum Gw Y^2, C_k = sum g_k 2^e,   Gw = (sum_k g_k c_k) 2^e,
// (g = dL/dI) to the Gaussian's accumulator with two 16-byte atomics (eight
// 4-byte ones took 1.5% longer on four dense crops, 0.3% at 5760 x 3240). The
// moments are taken in the exponent's own coordinates (d, Y), not in (X, Y):
// for |rho| -> 1 the X moments enter the chain rule with coefficients of
// order 1/(1 - rho^2)^2 that cancel to order 1/(1 - rho^2), which float32
// moments cannot resolve; in (d, Y) no such cancellation occurs.
//
// Layout: one warp per tile, walking the tile's list in chunks of 32 entries;
// lane l owns the chunk's l-th Gaussian. The warp first stages the tile's
// upstream gradient in shared memory, two columns per entry:
//   sgA[r][j] = (g_r(2j), g_r(2j + 1), g_g(2j), g_g(2j + 1)),  sgB[r][j] = (g_b(2j), g_b(2j + 1)).
// All lanes then walk the tile's pixels in the same order (row by row, two
// columns at a time), so every shared-memory read is a broadcast, and each
// lane evaluates its own Gaussian there in packed FP32x2 arithmetic:
//   d = Xs - sK Y (one fused step), e = R - d^2, w = 2^e   (Xs = sA X per
//   column, R = g Y^2 + l per row),
//   G = g . c, C_k += g_k w, Gw = G w, per row A0 += Gw, A1 += Gw d, A2 += Gw d^2,
// and after each row folds (A0, A1, A2) into the moments with that row's Y:
//   SY += Y A0, SYY += Y^2 A0, Sd += A1, SdY += Y A1, Sdd += A2.
// Per pixel that is 13 FP32 lane-operations (two pixels per packed
// instruction) and one MUFU.EX2; no cross-lane reduction. Window masks are in
// the operands (Xs = 1e18 outside the window's columns, so that d stays finite
// and every product with w = +0 is 0; R = -inf outside its rows); rows that no
// lane's window reaches are skipped.
#include <algorithm>

#include "gs_internal.cuh"

namespace gs {

namespace {

constexpr int kBwdParts = 64;    // parts of a tile's list at most
constexpr float kInfG = __builtin_huge_valf();
constexpr float kFarG = 1e18f;   // masked column: d^2 = 1e36 (finite), e = -1e36, w = +0

__device__ __forceinline__ float2 p2(float a, float b) { return make_float2(a, b); }

// Stages the upstream gradient of the E x E pixel block at image column ox,
// image row oy (0 outside the output) into sgA/sgB, E * E / 2 entries each.
template <int E>
__device__ __forceinline__ void stage_grad(const Ws& w, const ImageDesc* D, int ox, int oy,
                                           float4* sgA, float2* sgB) {
  constexpr int CP = E / 2;
  const int H = D->out_h, W = D->out_w;
  const int64_t plane = (int64_t)H * W;
  const float* go = w.direct ? w.grad_out0 : D->grad_out;
  float* fa = reinterpret_cast<float*>(sgA);
  float* fb = reinterpret_cast<float*>(sgB);
  for (int idx = threadIdx.x; idx < E * E; idx += 32) {
    const int r = idx / E, x = idx - r * E;
    const int gx = ox + x, gy = oy - D->row0 + r;
    const bool in = gx < W && gy < H;
    const int64_t o = in ? (int64_t)gy * W + gx : 0;   // always a valid address
    const float vr = __ldg(go + o), vg = __ldg(go + plane + o), vb = __ldg(go + 2 * plane + o);
    const int e = r * CP + (x >> 1), hb = x & 1;
    fa[4 * e + hb] = in ? vr : 0.0f;
    fa[4 * e + 2 + hb] = in ? vg : 0.0f;
    fb[2 * e + hb] = in ? vb : 0.0f;
  }
  __syncwarp();
}

// One chunk of the E x E block at (ox, oy): lane l adds Gaussian gid's
// moments over the block (valid false: an empty lane). A Gaussian whose
// window misses the block adds nothing.
template <int E>
__device__ __forceinline__ void bwd_chunk(const Ws& w, uint32_t gid, bool valid, int ox, int oy,
                                          const float4* sgA, const float2* sgB) {
  constexpr int CP = E / 2;                 // column pairs per block row
  constexpr int SEG = E < 16 ? E : 16;      // columns per register table
  constexpr int SP = SEG / 2;               // column pairs per table
  float4 f[kRecordF4];
  if (valid) {
    const float4* rec = w.records + (int64_t)gid * kRecordF4;
#pragma unroll
    for (int q = 0; q < kRecordF4; ++q) f[q] = rec[q];
  }
  // the Gaussian's record in tile-local coordinates
  float cxl = 0.f, cyl = 0.f, sA = 0.f, sK = 0.f, gy2 = 0.f, l = 0.f, cr = 0.f, cg = 0.f, cb = 0.f;
  int lx0 = 1, lx1 = 0, ly0 = E, ly1 = -1;
  if (valid) {
    cxl = __fadd_rn(__fsub_rn(f[0].x, (float)ox), f[0].y);
    cyl = __fadd_rn(__fsub_rn(f[0].z, (float)oy), f[0].w);
    sA = f[1].x; sK = f[1].y; gy2 = f[1].z; l = f[1].w;
    cr = f[2].x; cg = f[2].y; cb = f[2].z;
    lx0 = max(__float_as_int(f[3].x) - ox, 0);
    lx1 = min(__float_as_int(f[3].y) - ox, E - 1);
    ly0 = max(__float_as_int(f[3].z) - oy, 0);
    ly1 = min(__float_as_int(f[3].w) - oy, E - 1);
    if (lx0 > lx1 || ly0 > ly1) { ly0 = E; ly1 = -1; }
  }
  // rows some lane's window reaches
  const int rlo = __reduce_min_sync(0xffffffffu, ly0);
  const int rhi = __reduce_max_sync(0xffffffffu, ly1);

  const float2 cr2 = p2(cr, cr), cg2 = p2(cg, cg), cb2 = p2(cb, cb), nsK2 = p2(-sK, -sK);
  float2 Cr = p2(0.f, 0.f), Cg = Cr, Cb = Cr;
  float Sd = 0.f, SY = 0.f, Sdd = 0.f, SdY = 0.f, SYY = 0.f;
#pragma unroll
  for (int seg = 0; seg < E / SEG; ++seg) {
    // per column pair: Xs = sA X (kFarG outside the window)
    float2 Xs2[SP];
#pragma unroll
    for (int j = 0; j < SP; ++j) {
      const int c0 = seg * SEG + 2 * j, c1 = c0 + 1;
      const float a = __fsub_rn((float)c0, cxl), b = __fsub_rn((float)c1, cxl);
      Xs2[j] = p2((c0 >= lx0 && c0 <= lx1) ? sA * a : kFarG,
                  (c1 >= lx0 && c1 <= lx1) ? sA * b : kFarG);
    }
    for (int r = rlo; r <= rhi; ++r) {
      const float Y = __fsub_rn((float)r, cyl);
      const float R = (r >= ly0 && r <= ly1) ? fmaf(gy2 * Y, Y, l) : -kInfG;
      const float2 Y2 = p2(Y, Y), R2 = p2(R, R);
      const float4* ga = sgA + r * CP + seg * SP;
      const float2* gb = sgB + r * CP + seg * SP;
      float2 A0, A1, A2;
#pragma unroll
      for (int j = 0; j < SP; ++j) {
        const float4 q = ga[j];
        const float2 gbj = gb[j];
        const float2 gr2 = p2(q.x, q.y), gg2 = p2(q.z, q.w);
        const float2 d = __ffma2_rn(nsK2, Y2, Xs2[j]);   // one rounding: d cancels for |rho| -> 1
        const float2 e = __ffma2_rn(p2(-d.x, -d.y), d, R2);
        const float2 wv = p2(ex2_approx(e.x), ex2_approx(e.y));
        const float2 G = __ffma2_rn(gbj, cb2, __ffma2_rn(gg2, cg2, __fmul2_rn(gr2, cr2)));
        Cr = __ffma2_rn(gr2, wv, Cr);
        Cg = __ffma2_rn(gg2, wv, Cg);
        Cb = __ffma2_rn(gbj, wv, Cb);
        const float2 Gw = __fmul2_rn(G, wv);
        const float2 Gwd = __fmul2_rn(Gw, d);
        if (j == 0) {
          A0 = Gw;
          A1 = Gwd;
          A2 = __fmul2_rn(Gwd, d);
        } else {
          A0 = __fadd2_rn(A0, Gw);
          A1 = __fadd2_rn(A1, Gwd);
          A2 = __ffma2_rn(Gwd, d, A2);
        }
      }
      const float a0 = A0.x + A0.y, a1 = A1.x + A1.y, a2 = A2.x + A2.y;
      const float ty = Y * a0;
      SY += ty;
      SYY = fmaf(ty, Y, SYY);
      Sd += a1;
      SdY = fmaf(Y, a1, SdY);
      Sdd += a2;
    }
  }
  if (valid) {   // two 16-byte reductions; rows of 12 floats are 16-byte aligned
    float4* acc = reinterpret_cast<float4*>(w.grec + (int64_t)gid * 12);
    atomicAdd(acc, make_float4(Sd, SY, Sdd, SdY));
    atomicAdd(acc + 1, make_float4(SYY, Cr.x + Cr.y, Cg.x + Cg.y, Cb.x + Cb.y));
  }
}

// The entries [lo, hi), relative to its start, of a tile's list that one unit
// of work covers: all of it, or part `part` of w.bwd_parts in whole chunks of
// 32 entries (SPLIT). False: none.
template <bool SPLIT>
__device__ __forceinline__ bool list_part(const Ws& w, uint2 range, int part, int& lo, int& hi) {
  const int n = (int)range.y - (int)range.x;
  lo = 0;
  hi = n;
  if (SPLIT) {
    const int chunks = (n + 31) >> 5;
    lo = 32 * (int)((int64_t)chunks * part / w.bwd_parts);
    hi = min(n, 32 * (int)((int64_t)chunks * (part + 1) / w.bwd_parts));
  }
  return lo < hi;
}

// The adjoint of tile t by one warp, over one part of the tile's list.
template <int TILE, bool SPLIT>
__device__ __forceinline__ void bwd_one_tile(const Ws& w, const uint32_t* vals, int t, int part,
                                             float4* sgA, float2* sgB) {
  const uint2 range = w.ranges[t];
  int lo, n;
  if (!list_part<SPLIT>(w, range, part, lo, n)) return;   // no entry (uniform)
  const int lane = threadIdx.x;
  // tile origin (image rows: a band's output holds rows row0 ..)
  const int im = image_of_tile(w.images, w.n_images, t);
  const ImageDesc* D = &w.images[im];
  const int lt = t - D->t_base;
  const int tyi = lt / D->tiles_x;
  const int ox = (lt - tyi * D->tiles_x) * TILE;
  const int oy = tyi * TILE + D->row0;
  stage_grad<TILE>(w, D, ox, oy, sgA, sgB);
  for (int base = lo; base < n; base += 32) {
    const int i = base + lane;
    const uint32_t gid = i < n ? __ldg(vals + range.x + i) : 0xffffffffu;
    bwd_chunk<TILE>(w, gid, gid < (uint32_t)w.n, ox, oy, sgA, sgB);   // the list holds Gaussian ids
  }
}

// The adjoint over blocks of 8 columns x kBh rows of 16 x 16 tiles, for small
// windows: a CTA of kBwWarps warps takes a tile (or one part of its list). It
// stages the tile's upstream gradient and, 32 kBwWarps list entries at a time,
// the entries' records in shared memory, lists the (entry, block) items whose
// window meets the block (block by block, entries in list order) and walks the
// items in chunks of 32, one per lane: each lane evaluates its own Gaussian
// over its own block, so chunks are full across blocks, and a chunk waits on
// shared memory only. Lanes of a chunk are in at most 16 / kBh * 2 blocks, so
// a step's gradient loads touch that many addresses; rows of blocks are padded
// apart to keep those in different banks. Each item ends in two 16-byte
// reductions to its Gaussian's accumulator.
//
// What bounds it: the FP32 pipe (58% busy in the profile; FFMA2s with three
// operands take 2.3 to 2.9 cycles, so 70% to 80% of what it can do), then the
// pixels of blocks outside the windows. Against one warp per quadrant, which
// filtered the tile's list and fetched each chunk's records from L2 by itself
// and ran its last chunk 40% empty: 53.8 -> 43.8 us on 65,536 Gaussians at
// 1024 x 1024, 86 -> 76 us on 220,052 at 1002 x 751, 55.7 -> 48.0 us on 100,000
// at absolute centres. Blocks of 4 rows evaluate fewer pixels but fold twice as
// often: 44.8, 73.7 and 48.6 us. Two warps per CTA: 49.3, 84.4 and 55.9 us;
// eight: 59.9, 81.0 and 52.2 us.
constexpr int kBh = 8;
constexpr int kBwWarps = 4;
constexpr int kBlocksX = 2, kBlocksY = 16 / kBh, kBlocks = kBlocksX * kBlocksY;
constexpr int kBwPad = kBh == 8 ? 2 : 1;   // entries between two rows of blocks

struct BlockSmem {
  float4 gA[128 + kBwPad * kBlocksY];   // gradient, as stage_grad's sgA / sgB, padded
  float2 gB[128 + kBwPad * kBlocksY];
  float4 rec[kRecordF4][32 * kBwWarps];
  uint16_t item[kBlocks * 32 * kBwWarps];   // entry | block << 8
  int cnt[kBwWarps][kBlocks];
  uint32_t gid[32 * kBwWarps];
};

// One chunk of items: the lane's Gaussian (entry e of the staged records) over
// the lane's block q, as bwd_chunk does over a whole tile.
__device__ __forceinline__ void bwd_block(const Ws& w, const BlockSmem& S, int e, int q, bool valid,
                                          int tox, int toy) {
  const int bx = 8 * (q % kBlocksX), by = kBh * (q / kBlocksX);
  const int ox = tox + bx, oy = toy + by;
  float cxl = 0.f, cyl = 0.f, sA = 0.f, sK = 0.f, gy2 = 0.f, l = 0.f, cr = 0.f, cg = 0.f, cb = 0.f;
  int lx0 = 1, lx1 = 0, ly0 = kBh, ly1 = -1;
  if (valid) {
    const float4 f0 = S.rec[0][e], f1 = S.rec[1][e], f2 = S.rec[2][e], f3 = S.rec[3][e];
    cxl = __fadd_rn(__fsub_rn(f0.x, (float)ox), f0.y);
    cyl = __fadd_rn(__fsub_rn(f0.z, (float)oy), f0.w);
    sA = f1.x; sK = f1.y; gy2 = f1.z; l = f1.w;
    cr = f2.x; cg = f2.y; cb = f2.z;
    lx0 = __float_as_int(f3.x) - ox;
    lx1 = __float_as_int(f3.y) - ox;
    ly0 = max(__float_as_int(f3.z) - oy, 0);
    ly1 = min(__float_as_int(f3.w) - oy, kBh - 1);
  }
  // rows some lane's window reaches
  const int rlo = __reduce_min_sync(0xffffffffu, ly0);
  const int rhi = __reduce_max_sync(0xffffffffu, ly1);
  const float2 cr2 = p2(cr, cr), cg2 = p2(cg, cg), cb2 = p2(cb, cb), nsK2 = p2(-sK, -sK);
  float2 Cr = p2(0.f, 0.f), Cg = Cr, Cb = Cr;
  float Sd = 0.f, SY = 0.f, Sdd = 0.f, SdY = 0.f, SYY = 0.f;
  float2 Xs2[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c0 = 2 * j, c1 = c0 + 1;
    const float a = __fsub_rn((float)c0, cxl), b = __fsub_rn((float)c1, cxl);
    Xs2[j] = p2((c0 >= lx0 && c0 <= lx1) ? sA * a : kFarG, (c1 >= lx0 && c1 <= lx1) ? sA * b : kFarG);
  }
  const int at = by * 8 + bx / 2 + kBwPad * (q / kBlocksX);
  const float4* ga = S.gA + at;
  const float2* gb = S.gB + at;
  for (int r = rlo; r <= rhi; ++r) {
    const float Y = __fsub_rn((float)r, cyl);
    const float R = (r >= ly0 && r <= ly1) ? fmaf(gy2 * Y, Y, l) : -kInfG;
    const float2 Y2 = p2(Y, Y), R2 = p2(R, R);
    float2 A0, A1, A2;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 v = ga[r * 8 + j];
      const float2 gbj = gb[r * 8 + j];
      const float2 gr2 = p2(v.x, v.y), gg2 = p2(v.z, v.w);
      const float2 d = __ffma2_rn(nsK2, Y2, Xs2[j]);   // one rounding: d cancels for |rho| -> 1
      const float2 ex = __ffma2_rn(p2(-d.x, -d.y), d, R2);
      const float2 wv = p2(ex2_approx(ex.x), ex2_approx(ex.y));
      const float2 G = __ffma2_rn(gbj, cb2, __ffma2_rn(gg2, cg2, __fmul2_rn(gr2, cr2)));
      Cr = __ffma2_rn(gr2, wv, Cr);
      Cg = __ffma2_rn(gg2, wv, Cg);
      Cb = __ffma2_rn(gbj, wv, Cb);
      const float2 Gw = __fmul2_rn(G, wv);
      const float2 Gwd = __fmul2_rn(Gw, d);
      if (j == 0) {
        A0 = Gw;
        A1 = Gwd;
        A2 = __fmul2_rn(Gwd, d);
      } else {
        A0 = __fadd2_rn(A0, Gw);
        A1 = __fadd2_rn(A1, Gwd);
        A2 = __ffma2_rn(Gwd, d, A2);
      }
    }
    const float a0 = A0.x + A0.y, a1 = A1.x + A1.y, a2 = A2.x + A2.y;
    const float ty = Y * a0;
    SY += ty;
    SYY = fmaf(ty, Y, SYY);
    Sd += a1;
    SdY = fmaf(Y, a1, SdY);
    Sdd += a2;
  }
  if (valid) {   // two 16-byte reductions; rows of 12 floats are 16-byte aligned
    float4* acc = reinterpret_cast<float4*>(w.grec + (int64_t)S.gid[e] * 12);
    atomicAdd(acc, make_float4(Sd, SY, Sdd, SdY));
    atomicAdd(acc + 1, make_float4(SYY, Cr.x + Cr.y, Cg.x + Cg.y, Cb.x + Cb.y));
  }
}

template <bool SPLIT>
__global__ void __launch_bounds__(32 * kBwWarps) k_raster_bwd_quad(Ws w, const uint32_t* vals) {
  griddep_enter(w);
  constexpr int NT = 32 * kBwWarps;
  __shared__ BlockSmem S;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = SPLIT ? (int)(blockIdx.x / (uint32_t)w.bwd_parts) : (int)blockIdx.x;
  const uint2 range = w.ranges[t];
  int lo, hi;
  if (!list_part<SPLIT>(w, range, SPLIT ? (int)blockIdx.x - t * w.bwd_parts : 0, lo, hi)) return;
  const int im = image_of_tile(w.images, w.n_images, t);
  const ImageDesc* D = &w.images[im];
  const int lt = t - D->t_base;
  const int tyi = lt / D->tiles_x;
  const int ox = (lt - tyi * D->tiles_x) * 16;
  const int oy = tyi * 16 + D->row0;
  {
    const int H = D->out_h, W = D->out_w;
    const int64_t plane = (int64_t)H * W;
    const float* go = w.direct ? w.grad_out0 : D->grad_out;
    float* fa = reinterpret_cast<float*>(S.gA);
    float* fb = reinterpret_cast<float*>(S.gB);
#pragma unroll
    for (int idx = threadIdx.x; idx < 256; idx += NT) {
      const int r = idx >> 4, x = idx & 15;
      const int gx = ox + x, gy = oy - D->row0 + r;
      const bool in = gx < W && gy < H;
      const int64_t o = in ? (int64_t)gy * W + gx : 0;   // always a valid address
      const float vr = __ldg(go + o), vg = __ldg(go + plane + o), vb = __ldg(go + 2 * plane + o);
      const int e = r * 8 + (x >> 1) + kBwPad * (r / kBh), hb = x & 1;
      fa[4 * e + hb] = in ? vr : 0.0f;
      fa[4 * e + 2 + hb] = in ? vg : 0.0f;
      fb[2 * e + hb] = in ? vb : 0.0f;
    }
  }
  for (int base = lo; base < hi; base += NT) {
    // this thread's entry: its record, and the blocks its window meets
    const int i = base + (int)threadIdx.x;
    const uint32_t gid = i < hi ? __ldg(vals + range.x + i) : 0xffffffffu;
    uint32_t meets = 0u;
    if (gid < (uint32_t)w.n) {   // the list holds Gaussian ids
      const float4* rec = w.records + (int64_t)gid * kRecordF4;
      const float4 f0 = rec[0], f1 = rec[1], f2 = rec[2], f3 = rec[3];
      S.rec[0][threadIdx.x] = f0;
      S.rec[1][threadIdx.x] = f1;
      S.rec[2][threadIdx.x] = f2;
      S.rec[3][threadIdx.x] = f3;
      S.gid[threadIdx.x] = gid;
      const int x0 = __float_as_int(f3.x) - ox, x1 = __float_as_int(f3.y) - ox;
      const int y0 = __float_as_int(f3.z) - oy, y1 = __float_as_int(f3.w) - oy;
#pragma unroll
      for (int q = 0; q < kBlocks; ++q) {
        const int bx = 8 * (q % kBlocksX), by = kBh * (q / kBlocksX);
        if (x0 <= bx + 7 && x1 >= bx && y0 <= by + kBh - 1 && y1 >= by) meets |= 1u << q;
      }
    }
    uint32_t bal[kBlocks];
#pragma unroll
    for (int q = 0; q < kBlocks; ++q) {
      bal[q] = __ballot_sync(0xffffffffu, (meets >> q) & 1u);
      if (lane == 0) S.cnt[warp][q] = __popc(bal[q]);
    }
    __syncthreads();
    int items = 0;
#pragma unroll
    for (int q = 0; q < kBlocks; ++q) {
#pragma unroll
      for (int k = 0; k < kBwWarps; ++k) {
        if (k == warp && ((meets >> q) & 1u))
          S.item[items + __popc(bal[q] & ((1u << lane) - 1u))] = (uint16_t)(threadIdx.x | (q << 8));
        items += S.cnt[k][q];
      }
    }
    __syncthreads();
    for (int c = 32 * warp; c < items; c += NT) {
      const bool valid = c + lane < items;
      const int it = valid ? S.item[c + lane] : 0;
      bwd_block(w, S, it & 0xff, it >> 8, valid, ox, oy);
    }
    if (base + NT < hi) __syncthreads();   // every warp is done with the records and the items
  }
}

// Persistent: at most as many one-warp CTAs as are resident at once. CTA b
// takes tile b first; when there are more tiles than CTAs, each then takes
// the next tile from the workspace counter (reset by the forward's setup and
// by the chain rule after each adjoint) until the tiles run out, so that no
// partial last wave idles SMs. The counter is asked only after a tile is done,
// which spreads the (same-address) atomics over the launch. Registers capped
// at 64 for 32 resident CTAs per SM (no spills, but for 8 bytes in tile 16's form
// over parts of lists).
template <int TILE, bool SPLIT>
__global__ void __launch_bounds__(32, 32) k_raster_bwd_tile(Ws w, const uint32_t* vals) {
  griddep_enter(w);
  __shared__ float4 sgA[TILE * TILE / 2];
  __shared__ float2 sgB[TILE * TILE / 2];
  const uint32_t parts = SPLIT ? (uint32_t)w.bwd_parts : 1u, units = (uint32_t)w.tiles * parts;
  const bool more = gridDim.x < units;   // uniform over the grid
  uint32_t cur = blockIdx.x;
  while (cur < units) {
    const uint32_t t = cur / parts;
    bwd_one_tile<TILE, SPLIT>(w, vals, (int)t, (int)(cur - t * parts), sgA, sgB);
    if (!more) break;
    uint32_t nx = 0;
    if (threadIdx.x == 0) nx = gridDim.x + atomicAdd(&w.hdr->bwd_counter, 1u);
    cur = __shfl_sync(0xffffffffu, nx, 0);
    __syncwarp();   // every lane is done with the staged gradient before the next tile's
  }
}

}  // namespace

namespace {

// Parts each tile's list is cut into. Where the tiles fill at most half of the
// CTAs that are resident at once (`full`), one CTA per tile leaves the chip idle
// while the longest lists are walked: every list is then cut into parts (whole
// chunks of 32 entries, at most kBwdParts) that fill the chip twice over.
// Measured, 4 images of 48 x 48 LR pixels with 16 Gaussians each (250 tiles,
// lists of 4,000 to 10,000): 656 -> 86 us (parts that fill the chip once: 106).
// A part stages the tile's gradient again and leaves a chunk short, so a fuller
// chip keeps whole lists: 16 crops with short lists took 38.7 us in parts
// against 37.1. And a part costs a CTA whether or not it has a chunk, so a list
// is cut into no more than one part per `entries` of the lists' mean length,
// which the pair capacity bounds (sized by a count, it is the mean), or into as
// many as make `spare` CTAs in all: those are next to free, and shorten what one
// long list among short ones takes. Adjoint, us, whole lists / cut so / a chip's
// worth of parts. Tile 16 (16 entries, 512 CTAs), 256 tiles, lists of 16 9.7 / 10.4
// / 16.3, 62 19.2 / 12.7 / 18.7, 125 33.5 / 16.4 / 21.7; 1,024 tiles, 16 12.1 / 12.1
// / 21.2, 64 27.6 / 25.3 / 26.5; 2,025 tiles, 16 15.6 / 15.6 / 24.7. Quadrants (16,
// 512), 256 tiles, 63 9.4 / 9.4 / 10.3. Tile 8 (24, 2,048), 1,024 tiles, 7 10.0 / 9.8
// / 14.1, 44 10.6 / 10.5 / 16.1, 176 23.9 / 21 / 22.7. Tile 32 (6, 512), 400 tiles, 8
// 23.0 / 23.0 / 41.0, 49 56.5 / 48 / 48.9. With half the Gaussians in a 25th of the
// tiles: tile 16, 64 tiles, mean 14 26.1 / 9.6 / 10.4, 256 tiles, 62 132 / 41 / 19;
// quadrants, 256 tiles, 62 27.8 / 12.7 / 10.7. Over 449 such scenes and reference
// grids, forward and adjoint together, at most 10% slower than whole lists
// anywhere, where a chip's worth took up to 33% more.
int32_t list_parts(const Ws& w, int64_t full, int64_t entries, int64_t spare) {
  const int64_t tiles = w.tiles;
  if (2 * tiles > full) return 1;
  const int64_t fill = std::min<int64_t>(kBwdParts, (2 * full + tiles - 1) / tiles);
  const int64_t mean = w.capacity / tiles;
  const int64_t worth = std::max((mean + entries / 2) / entries, spare / tiles);
  return (int32_t)std::max<int64_t>(1, std::min(fill, worth));
}

using BwdKernel = void (*)(Ws, const uint32_t*);

// The tile adjoint's kernels over whole lists and over parts.
BwdKernel tile_kernel(int tile, bool split) {
  switch (tile) {
    case 8: return split ? k_raster_bwd_tile<8, true> : k_raster_bwd_tile<8, false>;
    case 32: return split ? k_raster_bwd_tile<32, true> : k_raster_bwd_tile<32, false>;
    default: return split ? k_raster_bwd_tile<16, true> : k_raster_bwd_tile<16, false>;
  }
}

}  // namespace

int32_t raster_bwd_parts(const Ws& w, bool quadrants) {
  if (quadrants)
    return list_parts(w, resident_grid((const void*)k_raster_bwd_quad<false>, 32 * kBwWarps, INT32_MAX),
                      16, 512);
  return list_parts(w, resident_grid((const void*)tile_kernel(w.tile, false), 32, INT32_MAX),
                    w.tile == 8 ? 24 : w.tile == 32 ? 6 : 16, w.tile == 8 ? 2048 : 512);
}

cudaError_t launch_raster_bwd_tile(const Ws& ws, const uint32_t* lists, bool quadrants,
                                   cudaStream_t s) {
  if (ws.tiles == 0) return cudaSuccess;
  LaunchScope ls(kKRasterBwd, s);
  Ws w = ws;
  w.bwd_parts = raster_bwd_parts(w, quadrants);
  const bool split = w.bwd_parts > 1;
  const int64_t units = (int64_t)w.tiles * w.bwd_parts;
  if (quadrants)   // tile 16 (the caller checks): a CTA per tile, or per part of a tile's list
    return launch_chain(split ? k_raster_bwd_quad<true> : k_raster_bwd_quad<false>,
                        dim3((unsigned)units), dim3(32 * kBwWarps), 0, s, w, lists);
  // a persistent launch of one-warp CTAs
  const BwdKernel kernel = tile_kernel(w.tile, split);
  return launch_chain(kernel, dim3((unsigned)resident_grid((const void*)kernel, 32, units)), dim3(32),
                      0, s, w, lists);
}

}  // namespace gs
