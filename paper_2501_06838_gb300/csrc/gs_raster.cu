// Tile rasterizer of the scale-aware 2D Gaussian splatting render (GSASR,
// arXiv 2501.06838, Eq. 4 with the Algorithm-1 window): the forward. (The
// adjoint, one lane per Gaussian over a tile's pixels, is gs_adjoint_tile.cu.)
//
// Tile 16, one warp per tile: k_raster_fwd16 (the tile in four strips, below);
// one warp per pair of tiles: k_raster_fwd_pair; several warps per tile:
// k_raster_fwd_team. The rest of this comment is the layout of tiles 8 and 32,
// k_raster_fwd:
// one CTA of NT = TILE*TILE/BY threads renders one TILE x TILE tile of HR
// pixels; thread t owns column t % TILE and the BY consecutive rows
// [(t / TILE) * BY, + BY). The tile's Gaussians (a contiguous run of the sorted
// pair list) go through shared memory in batches of NT * PF, double buffered:
//   copy:    each thread cp.async-copies the 64-byte records of its Gaussians
//            of the NEXT batch into a raw buffer while the CTA computes this
//            batch (their ids are loaded one batch earlier still);
//   stage 1: one thread per Gaussian moves its centre into tile-local
//            coordinates (cx - x_tile: small numbers, so X = x - cx keeps full
//            float32 precision even at x ~ 5760) and clips its window;
//   stage 2: per (Gaussian, pair of tile rows) the row terms of the exponent
//              e = -(sA X - sK Y)^2 + g Y^2 + l        (log2 units)
//            as one float4 (-K(r), -K(r+1), R(r), R(r+1)), with K = sK*Y and
//            R = g*Y^2 + l (R = -inf outside the window rows);
//   compute: per Gaussian each thread forms Xs = sA*(col - cxl) (+inf outside
//            the window columns) and, for each of its row pairs, in packed
//            FP32x2 arithmetic (one instruction for both rows),
//              d = Xs - K, e = R - d*d, w = 2^e (MUFU.EX2, one per pixel),
//              out += c*w  (three FFMA2 for the three channels),
//            i.e. per pixel 2.5 FP32 instructions + 1 MUFU. The next
//            Gaussian's shared-memory operands load while the current one
//            is computed.
// The window masks are folded into the exponent: -inf rows and +inf columns
// both give e = -inf and w = +0, so masked pairs cost no branch. The completed
// square has no cancellation for any |rho| < 1 (the Y term is the marginal).
#include <type_traits>

#include "gs_internal.cuh"

namespace gs {

namespace {

constexpr float kInf = __builtin_huge_valf();

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <int TILE>
__device__ __forceinline__ void tile_origin(const Ws& w, int t, const ImageDesc*& D, int& ox,
                                            int& oy, int& tx, int& ty) {
  const int im = image_of_tile(w.images, w.n_images, t);
  D = &w.images[im];
  const int lt = t - D->t_base;
  ty = lt / D->tiles_x;
  tx = lt - ty * D->tiles_x;
  ox = tx * TILE;
  oy = ty * TILE + D->row0;   // image rows (the output holds rows row0 ..)
}

// Copy the records of batch entries t, t + NT, ... (ids in gid[]) to raw.
template <int NT, int PF>
__device__ __forceinline__ void issue_records(const Ws& w, const uint32_t (&gid)[PF], int nb,
                                              float4* raw) {
#pragma unroll
  for (int j = 0; j < PF; ++j) {
    const int i = j * NT + threadIdx.x;
    if (i < nb) {
      const float4* rec = w.records + (int64_t)gid[j] * kRecordF4;
#pragma unroll
      for (int q = 0; q < kRecordF4; ++q) cp_async16(raw + i * kRecordF4 + q, rec + q);
    }
  }
  cp_async_commit();
}

template <int NT, int PF>
__device__ __forceinline__ void load_ids(const uint32_t* vals, int bs, int nb, uint32_t (&gid)[PF]) {
#pragma unroll
  for (int j = 0; j < PF; ++j) {
    const int i = j * NT + threadIdx.x;
    gid[j] = i < nb ? __ldg(vals + bs + i) : 0u;
  }
}

// A tile's list is summed in segments of kSeg entries, one after the other:
// out = ((S0 + S1) + S2) + .... One warp writes each segment's sums onto the
// output as it ends; a team of warps sums them side by side and adds them in
// the same order (k_raster_fwd_team): the same bits in every layout of tile 16.
// (Tiles 8 and 32 sum a tile's whole list in one run, k_raster_fwd.)
constexpr int kSeg = 512;

// Where a tile's Gaussian ids come from, one batch at a time (ids ascending,
// so both sources give a tile the same Gaussians in the same order and the
// forward the same bits).
//
// SortedSource: the tile's run [start, end) of the radix-sorted pair list.
template <int NT, int PF>
struct SortedSource {
  const uint32_t* vals;
  int pos, end;
  __device__ __forceinline__ int next(uint32_t (&gid)[PF]) {
    const int nb = max(0, min(NT * PF, end - pos));
    load_ids<NT, PF>(vals, pos, nb, gid);
    pos += nb;
    return nb;
  }
};

// GridSource (grid-implicit binning): with centres mu = p + o on the reference
// grid, a Gaussian of LR cell (i, j) has its window within
// [s j - DL, s j + DR] x [s i - DT, s i + DB], the per-image reach measured by
// the footprint pass. So the tile's candidates are the Gaussians of a box of
// LR cells: rows i0..i1, each a contiguous run of gids. Every candidate's
// window is tested against the tile (the same test that puts a pair into the
// sorted list); the survivors go through a shared-memory queue in gid order.
// All warps run the enumeration (the same loads and ballots); warp 0 writes.
//
// Candidates: the 32 lanes' current candidates of such a box, 32 apart in the
// box's row-major order. Moving on is an add and, at a row's end, a wrap; the
// window test is two packed 16-bit comparisons. (With a division per candidate
// and four unpacked comparisons, half the instructions more, the pair forward
// took 1007 instead of 945 us on 518,400 Gaussians at 5760 x 3240, where 7
// candidates are tested per pair kept.)
struct Candidates {
  const uint2* win;      // (x0, y0) and (x1, y1) of every window, 16 bits each
  int64_t rb0, rstride;  // gid of the first candidate of row r: rb0 + r * rstride
  int L, total, cur;     // candidates per row, in all, next to test
  uint32_t gid, wrap;    // this lane's candidate; from a row's end to the next row's start
  int col;               // its position in its row
  int step;              // advance_flat: 32 candidates on, modulo whole rows
  uint32_t jump;         // ... and in gids
  uint32_t lo, hi;       // the region: (X0, Y0) and (X1, Y1), output rows
  // to candidate `from` (lane 0's)
  __device__ __forceinline__ void seek(int from) {
    const int c = from + (int)(threadIdx.x & 31);
    const int r = L > 0 ? c / L : 0;
    col = c - r * L;
    gid = (uint32_t)(rb0 + (int64_t)r * rstride + col);
    cur = from;
  }
  __device__ __forceinline__ void start(int X0, int X1, int Y0, int Y1) {
    wrap = (uint32_t)(rstride - L);
    const int rows = L > 0 ? 32 / L : 0;
    step = 32 - rows * L;
    jump = 32u + (uint32_t)rows * wrap;
    lo = (uint32_t)(X0 & 0xffff) | ((uint32_t)Y0 << 16);
    hi = (uint32_t)(X1 & 0xffff) | ((uint32_t)Y1 << 16);
    seek(0);
  }
  // the window of this lane's k-th candidate from cur on, g (none: one that meets nothing)
  __device__ __forceinline__ uint2 load(int k, uint32_t g) const {
    return cur + 32 * k + (int)(threadIdx.x & 31) < total ? win[g]
                                                          : make_uint2(0x7fff7fffu, 0x80008000u);
  }
  __device__ __forceinline__ void advance() {
    col += 32;
    gid += 32u;
    if (L >= 32) {
      if (col >= L) { col -= L; gid += wrap; }
    } else if (L > 0) {
      while (col >= L) { col -= L; gid += wrap; }
    }
  }
  // the same without a branch, for tile 32: its tiles are few and their boxes, at a
  // large scale, rows of a few cells that the loop above wraps one at a time (us:
  // 5 images of 121 x 119 LR pixels at scale 18 392 -> 379, 178 x 203 at 23 301 ->
  // 290; in the pair forward 913 -> 936 at 5760 x 3240, in tile 16's 48.6 -> 50)
  __device__ __forceinline__ void advance_flat() {
    col += step;
    gid += jump;
    if (col >= L) { col -= L; gid += wrap; }
  }
  // the window meets the region: x0 <= X1, y0 <= Y1, x1 >= X0, y1 >= Y0
  __device__ __forceinline__ bool meets(uint2 v) const {
    return __vmaxs2(v.x, hi) == hi && __vmins2(v.y, lo) == lo;
  }
};

template <int NT, int PF>
struct GridSource {
  static constexpr int BATCH = NT * PF;
  static constexpr int KR = 4;                          // candidates per lane per round
  static constexpr int QCAP = BATCH + 32 * KR <= 256 ? 256 : 512;
  uint32_t* q;           // shared [QCAP]
  Candidates cand;
  int head, tail;        // queue positions (monotonic)

  __device__ __forceinline__ void sync() {
    if (NT == 32) __syncwarp(); else __syncthreads();
  }
  __device__ __forceinline__ int next(uint32_t (&gid)[PF]) {
    const int lane = threadIdx.x & 31;
    while (tail - head < BATCH && cand.cur < cand.total) {   // uniform over the CTA
      // KR independent window loads per lane, then the ballots in candidate order
      uint32_t g[KR];
      uint2 v[KR];
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        g[k] = cand.gid;
        if constexpr (NT == 64 && PF == 1) cand.advance_flat(); else cand.advance();
      }
#pragma unroll
      for (int k = 0; k < KR; ++k) v[k] = cand.load(k, g[k]);
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        const bool hit = cand.meets(v[k]);
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        if ((NT == 32 || threadIdx.x < 32) && hit)
          q[(tail + __popc(bal & ((1u << lane) - 1u))) & (QCAP - 1)] = g[k];
        tail += __popc(bal);
      }
      cand.cur += 32 * KR;
    }
    sync();
    const int nb = min(BATCH, tail - head);
#pragma unroll
    for (int j = 0; j < PF; ++j) {
      const int i = j * NT + (NT == 32 ? lane : (int)threadIdx.x);
      gid[j] = i < nb ? q[(head + i) & (QCAP - 1)] : 0u;
    }
    head += nb;
    return nb;
  }
};

// A source's next batch as a call of its own, for the grid forward of tile 32 with
// 64 Gaussians a round: inlined there, the candidate walk took the registers (168)
// that overlap the operand loads with the arithmetic. Us, before that walk /
// inlined / as a call: 5 images of 69 x 16 LR pixels, 4 Gaussians each,
// whole-image windows at scale 7 853 / 957 / 843; 16 x 275, ratio window at 1.9
// 461 / 540 / 445; 256 x 256, 1 each, at 4 87 / 93 / 87. Tile 8 and rounds of 128
// keep it inline (as a call 49 -> 54, 55 -> 82; 478 -> 531).
template <class Source, int PF>
__device__ __noinline__ int next_apart(Source& src, uint32_t (&gid)[PF]) {
  return src.next(gid);
}

// The candidate box of the pixel region [X0, X1] x [Y0, Y1] in grid mode (see
// GridSource). A Gaussian of column j meets it only if s j - DL < x0 <= X1 and
// s j + DR > x1 >= X0; the reach (DL, DR, DT, DB) carries a pixel of margin,
// far more than the float32 rounding of these quotients, so floor/ceil bound
// the cells exactly. Y0 and Y1 are image rows; the windows and the region they
// are tested against are output rows (from row0), which fit 16 bits.
__device__ __forceinline__ void candidate_box(const Ws& w, const ImageDesc* D, int X0, int X1,
                                              int Y0, int Y1, Candidates& c) {
  const int4 e = w.ext[D - w.images];   // HR px
  const float r = __frcp_rn(D->scale);
  const int j0 = max(0, (int)ceilf((float)(X0 - e.y) * r));
  const int j1 = e.x < kFarReach ? min(D->lr_w - 1, (int)floorf((float)(X1 + e.x) * r)) : D->lr_w - 1;
  const int i0 = max(0, (int)ceilf((float)(Y0 - e.w) * r));
  const int i1 = e.z < kFarReach ? min(D->lr_h - 1, (int)floorf((float)(Y1 + e.z) * r)) : D->lr_h - 1;
  c.win = reinterpret_cast<const uint2*>(w.win);
  c.rstride = (int64_t)D->lr_w * D->m;
  c.rb0 = D->g_base + ((int64_t)i0 * D->lr_w + j0) * D->m;
  c.L = (j1 - j0 + 1) * D->m;
  c.total = (j0 <= j1 && i0 <= i1) ? (i1 - i0 + 1) * c.L : 0;
  c.start(X0, X1, Y0 - D->row0, Y1 - D->row0);
}

template <int TILE, int NT, int PF>
__device__ __forceinline__ void grid_source_init(const Ws& w, const ImageDesc* D, int ox, int oy,
                                                 uint32_t* q, GridSource<NT, PF>& g) {
  g.q = q;
  candidate_box(w, D, ox, ox + TILE - 1, oy, oy + TILE - 1, g.cand);
  g.head = g.tail = 0;
}

// Stage 1 from the raw records:
//   gA = (cxl, sA, lx0, lx1)   gB = (cyl, sK, g, l)   gC = (r, g, b, ly0 | ly1 << 16)
template <int TILE, int NT>
__device__ __forceinline__ void stage_records(const float4* raw, int nb, int ox, int oy,
                                              float4* gA, float4* gB, float4* gC) {
  for (int i = threadIdx.x; i < nb; i += NT) {
    const float4 f0 = raw[i * kRecordF4], f1 = raw[i * kRecordF4 + 1];
    const float4 f2 = raw[i * kRecordF4 + 2], f3 = raw[i * kRecordF4 + 3];
    const float cxl = __fadd_rn(__fsub_rn(f0.x, (float)ox), f0.y);
    const float cyl = __fadd_rn(__fsub_rn(f0.z, (float)oy), f0.w);
    const int lx0 = max(__float_as_int(f3.x) - ox, 0), lx1 = min(__float_as_int(f3.y) - ox, TILE - 1);
    const int ly0 = max(__float_as_int(f3.z) - oy, 0), ly1 = min(__float_as_int(f3.w) - oy, TILE - 1);
    gA[i] = make_float4(cxl, f1.x, (float)lx0, (float)lx1);
    gB[i] = make_float4(cyl, f1.y, f1.z, f1.w);
    gC[i] = make_float4(f2.x, f2.y, f2.z, __int_as_float(ly0 | (ly1 << 16)));
  }
}

// Stage 2: row terms (-K(2p), -K(2p+1), R(2p), R(2p+1)) of every staged
// Gaussian and pair of tile rows; the packed window rows come from gC[i].w.
template <int TILE, int NT>
__device__ __forceinline__ void stage_rowpairs(int nb, const float4* gB, const float4* gC,
                                               float4* rq) {
  constexpr int HP = TILE / 2;
  for (int idx = threadIdx.x; idx < nb * HP; idx += NT) {
    const int i = idx / HP, p = idx - i * HP;
    const float4 b = gB[i];
    const int pk = __float_as_int(gC[i].w);
    const int ly0 = pk & 0xffff, ly1 = pk >> 16;
    const int r0 = 2 * p, r1 = 2 * p + 1;
    const float Y0 = (float)r0 - b.x, Y1 = (float)r1 - b.x;
    float R0 = fmaf(b.z * Y0, Y0, b.w), R1 = fmaf(b.z * Y1, Y1, b.w);
    if (r0 < ly0 || r0 > ly1) R0 = -kInf;
    if (r1 < ly0 || r1 > ly1) R1 = -kInf;
    rq[idx] = make_float4(-b.y * Y0, -b.y * Y1, R0, R1);
  }
}

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

// Shared-memory operands of one Gaussian for one thread: gA, gC and the row
// terms of its NQ = BY / 2 row pairs.
template <int NQ>
struct FwdOps {
  float4 a, c, q[NQ];
  __device__ __forceinline__ void load(const float4* gA, const float4* gC, const float4* rq,
                                       int i, int hp, int pair0) {
    a = gA[i];
    c = gC[i];
    const float4* rr = rq + i * hp + pair0;
#pragma unroll
    for (int j = 0; j < NQ; ++j) q[j] = rr[j];
  }
};

template <int NQ>
__device__ __forceinline__ void fwd_gaussian(float2 (&acc)[NQ][3], const FwdOps<NQ>& o, float fcol) {
  float Xs = o.a.y * (fcol - o.a.x);
  if (fcol < o.a.z || fcol > o.a.w) Xs = kInf;
  const float2 X2 = f2(Xs, Xs);
  const float2 c0 = f2(o.c.x, o.c.x), c1 = f2(o.c.y, o.c.y), c2 = f2(o.c.z, o.c.z);
#pragma unroll
  for (int j = 0; j < NQ; ++j) {
    const float2 d = __fadd2_rn(X2, f2(o.q[j].x, o.q[j].y));
    const float2 e = __ffma2_rn(f2(-d.x, -d.y), d, f2(o.q[j].z, o.q[j].w));
    const float2 wv = f2(ex2_approx(e.x), ex2_approx(e.y));
    acc[j][0] = __ffma2_rn(c0, wv, acc[j][0]);
    acc[j][1] = __ffma2_rn(c1, wv, acc[j][1]);
    acc[j][2] = __ffma2_rn(c2, wv, acc[j][2]);
  }
}

// ---------------------------------------------------------------------------
// Forward of a 16 x 16 tile by one warp, in four strips of 4 columns x 16 rows.
//
// Lane l works on strip l / 8 and owns that strip's four columns on the row
// pair l % 8 (8 pixels). The strips walk a staged batch independently: a
// 32-bit mask per strip says which of the batch's Gaussians have a window that
// meets the strip's columns, and in each step every strip takes its own next
// one, so a Gaussian costs the strips it touches and not the whole tile.
// Staging (one lane per Gaussian) leaves everything a step reads as three
// 16-byte loads: the strip's four column terms Xs = sA (x - cx) (+inf outside
// the window), the row pair's (-K, -K', R, R') (R = -inf outside the window)
// and the colour. The slots run backwards (the batch's first Gaussian in the
// last slot), so that "highest set bit first" is ascending id order and every
// pixel sums its Gaussians in the order, and with the arithmetic, of the other
// layouts: the same bits.
//
// What bounds it: a 16-byte shared load takes 2.5 cycles of the SM for 1 to 8
// distinct addresses (4.0 for 32), an FFMA2 2.3 of its scheduler, a MUFU 4.2;
// the former layout (lane: one column of eight rows) spent 6 such loads, 59
// scheduler cycles, on 8 pixels per lane whose arithmetic takes 47. Here the
// step's 3 loads take 36, and the step alone in a loop 64 cycles. Measured
// against it: 41.2 -> 34.4 us on 65,536 Gaussians at 1024 x 1024 (windows of
// 22 px on average: 0.68 of the tile's columns per Gaussian), 81.8 -> 53.5 us
// on 220,052 at 1002 x 751 (14 px), 4134 -> 3776 us on 518,400 at 720 x 720
// under the ratio window (144 px). Ids run along LR rows, so a batch's windows
// share rows and spread over the columns: strips of whole columns are evenly
// filled. Strips cut in halves of 8 rows (51 us at 1002 x 751 against 50) or
// tiles cut in quadrants (54) were not.
// ---------------------------------------------------------------------------
constexpr int kStripSlots = 33;   // 32 slots and, in front, one that adds nothing (odd: no bank conflicts)

// NQ: groups of four columns per strip and lane (1: the strips of one tile; 2:
// strips of 8 columns over a pair of tiles).
template <int NQ>
struct StripTables {
  float4 x[4 * NQ * kStripSlots];   // [strip][quad][slot] Xs of four columns
  float4 r[8 * kStripSlots];        // [row pair][slot] (-K(2p), -K(2p+1), R(2p), R(2p+1))
  float4 c[kStripSlots];            // [slot] colour
  // the front slots: Xs = 0, K = 0, R = -inf, colour 0
  __device__ __forceinline__ void clear_front(int lane) {
    if (lane < 4 * NQ) x[lane * kStripSlots] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < 8) r[lane * kStripSlots] = make_float4(0.f, 0.f, -kInf, -kInf);
    if (lane == 0) c[0] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// A lane's pixels: [row of its pair][column pair][channel].
template <int NQ>
using StripAcc = float2[2][2 * NQ][3];

// Operands of one step for one lane.
template <int NQ>
struct StripOps {
  float4 x[NQ], r, c;
};

template <int NQ>
__device__ __forceinline__ void strip_step(StripAcc<NQ>& acc, const StripOps<NQ>& o) {
  const float2 c0 = f2(o.c.x, o.c.x), c1 = f2(o.c.y, o.c.y), c2 = f2(o.c.z, o.c.z);
#pragma unroll
  for (int j = 0; j < 2; ++j) {     // the row of the pair
    const float2 nK = j ? f2(o.r.y, o.r.y) : f2(o.r.x, o.r.x);
    const float2 R = j ? f2(o.r.w, o.r.w) : f2(o.r.z, o.r.z);
#pragma unroll
    for (int h = 0; h < 2 * NQ; ++h) {   // the columns two by two
      const float4 xq = o.x[h / 2];
      const float2 d = __fadd2_rn((h & 1) ? f2(xq.z, xq.w) : f2(xq.x, xq.y), nK);
      const float2 e = __ffma2_rn(f2(-d.x, -d.y), d, R);
      const float2 wv = f2(ex2_approx(e.x), ex2_approx(e.y));
      acc[j][h][0] = __ffma2_rn(c0, wv, acc[j][h][0]);
      acc[j][h][1] = __ffma2_rn(c1, wv, acc[j][h][1]);
      acc[j][h][2] = __ffma2_rn(c2, wv, acc[j][h][2]);
    }
  }
}

// Bits lo .. hi of a 32-bit word, as far as they lie in it.
__device__ __forceinline__ uint32_t window_bits(int lo, int hi) {
  if (lo > 31 || hi < 0) return 0u;
  return (0xffffffffu >> (31 - min(hi, 31))) & (0xffffffffu << max(lo, 0));
}

// Stages slot `lane` of a table from the Gaussian's record (a lane without a
// Gaussian: live false) and returns the strips its window meets as four bits.
// Column terms are relative to the 16-column tile they belong to.
template <int NQ>
__device__ __forceinline__ uint32_t stage_strips(const float4* raw, int lane, bool live, int ox,
                                                 int oy, StripTables<NQ>& t) {
  if (!live) return 0u;
  const float4 f0 = raw[lane], f1 = raw[32 + lane], f2v = raw[64 + lane], f3 = raw[96 + lane];
  const float cyl = __fadd_rn(__fsub_rn(f0.z, (float)oy), f0.w);
  // the window's columns and rows in the region, a bit each: one test and one
  // select per value below
  const uint32_t cols = window_bits(__float_as_int(f3.x) - ox, __float_as_int(f3.y) - ox);
  const uint32_t rows = window_bits(__float_as_int(f3.z) - oy, __float_as_int(f3.w) - oy);
  // two values at a time: packed for a pair of tiles (927 -> 916 us at 5760 x
  // 3240, 779 -> 761 us on 16 uneven images), scalar for one (packed, teams took
  // 3.08 instead of 2.90 ms); the same roundings
  auto add = [](float2 a, float2 b) { return NQ == 2 ? __fadd2_rn(a, b) : f2(a.x + b.x, a.y + b.y); };
  auto mul = [](float2 a, float2 b) { return NQ == 2 ? __fmul2_rn(a, b) : f2(a.x * b.x, a.y * b.y); };
  auto fma = [](float2 a, float2 b, float2 c) {
    return NQ == 2 ? __ffma2_rn(a, b, c) : f2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
  };
  const float2 sA = f2(f1.x, f1.x), nsK = f2(-f1.y, -f1.y), g = f2(f1.z, f1.z), l = f2(f1.w, f1.w);
#pragma unroll
  for (int q = 0; q < 4 * NQ; ++q) {
    const int tx = 16 * (q / 4);   // the tile's first column
    const float cxl = __fadd_rn(__fsub_rn(f0.x, (float)(ox + tx)), f0.y);
    const float c0 = (float)(4 * q - tx);
    const float2 va = mul(sA, add(f2(c0, c0 + 1.0f), f2(-cxl, -cxl)));
    const float2 vb = mul(sA, add(f2(c0 + 2.0f, c0 + 3.0f), f2(-cxl, -cxl)));
    float v[4] = {va.x, va.y, vb.x, vb.y};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (!(cols & (1u << (4 * q + k)))) v[k] = kInf;
    t.x[q * kStripSlots + 1 + lane] = make_float4(v[0], v[1], v[2], v[3]);
  }
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const float2 Y = add(f2((float)(2 * p), (float)(2 * p + 1)), f2(-cyl, -cyl));
    const float2 nK = mul(nsK, Y);
    float2 R = fma(mul(g, Y), Y, l);
    if (!(rows & (1u << (2 * p)))) R.x = -kInf;
    if (!(rows & (2u << (2 * p)))) R.y = -kInf;
    t.r[p * kStripSlots + 1 + lane] = make_float4(nK.x, nK.y, R.x, R.y);
  }
  uint32_t hit = 0u;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (cols & (((1u << (4 * NQ)) - 1u) << (4 * NQ * q))) hit |= 1u << q;
  t.c[1 + lane] = f2v;
  return hit;
}

// One staged table: the strips' masks from the lanes' hits, then the walk.
// Returns nothing; every lane adds its strip's Gaussians to acc.
struct StripMasks {
  uint32_t m;   // this lane's strip's mask
  int steps;    // the largest number of Gaussians any strip has
};
__device__ __forceinline__ StripMasks strip_masks(uint32_t hit, int strip) {
  StripMasks s{0u, 0};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t bal = __ballot_sync(0xffffffffu, (hit >> q) & 1u);
    s.steps = max(s.steps, __popc(bal));
    if (strip == q) s.m = bal;
  }
  return s;
}

template <int NQ>
__device__ __forceinline__ void walk_strips(StripAcc<NQ>& acc, StripMasks s, int strip, int rp,
                                            const StripTables<NQ>& t) {
  const float4* tx = t.x + strip * NQ * kStripSlots;
  const float4* tr = t.r + rp * kStripSlots;
  uint32_t m = s.m;
  auto load = [&](StripOps<NQ>& o) {
    // highest set bit (none: -1, the front slot); the shift by -1 gives 0
    int b;
    uint32_t bit;
    asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(m));
    asm("shl.b32 %0, 1, %1;" : "=r"(bit) : "r"(b));
    m ^= bit;
#pragma unroll
    for (int h = 0; h < NQ; ++h) o.x[h] = tx[b + 1 + h * kStripSlots];
    o.r = tr[b + 1];
    o.c = t.c[b + 1];
  };
  // two operand sets: a step's loads overlap the step before it
  StripOps<NQ> A, B;
  load(A);
  for (int i = 0; i < s.steps; i += 2) {
    load(B);
    strip_step<NQ>(acc, A);
    load(A);
    strip_step<NQ>(acc, B);   // past the last step: the front slot, which adds nothing
  }
}

// Copies the records of a batch: entry j * 32 + k goes to raw[j], slot 31 - k.
template <int PF>
__device__ __forceinline__ void issue_slots(const Ws& w, const uint32_t (&ids)[PF], int n,
                                            float4 (&raw)[PF][4 * 32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < PF; ++j) {
    if (j * 32 + lane < n) {
      const float4* rec = w.records + (int64_t)ids[j] * kRecordF4;
#pragma unroll
      for (int q = 0; q < kRecordF4; ++q) cp_async16(&raw[j][q * 32 + 31 - lane], rec + q);
    }
  }
  cp_async_commit();
}

// The region's pixels through shared memory, for stores in whole rows: 128-byte
// lines of a row (NQ 2) or a row pair (NQ 1), their 16-byte pieces permuted by
// the row pair so that neither side has bank conflicts.
template <int NQ>
__device__ __forceinline__ void strips_to_rows(const StripAcc<NQ>& acc, float* buf, int lane) {
  const int strip = lane >> 3, rp = lane & 7;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int h = 0; h < NQ; ++h)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int line = NQ == 2 ? 2 * rp + j : rp, piece = NQ == 2 ? 2 * strip + h : 4 * j + strip;
        const float2 a = acc[j][2 * h][k], b = acc[j][2 * h + 1][k];
        *reinterpret_cast<float4*>(buf + k * 256 * NQ + line * 32 + 4 * (piece ^ rp)) =
            make_float4(a.x, a.y, b.x, b.y);
      }
}
// Column lane % (16 NQ) of row r of channel k.
template <int NQ>
__device__ __forceinline__ float row_value(const float* buf, int k, int r, int lane) {
  return buf[k * 256 * NQ + (NQ == 2 ? r : r >> 1) * 32 + 4 * ((lane >> 2) ^ (r >> 1)) + (lane & 3)];
}

// Writes the region's pixels: 16 NQ columns from ox, 16 rows from output row y0.
// A pair of tiles goes out in whole rows by way of the table's memory: stored by
// their lanes, 16 bytes or (rows not 16-byte aligned) 4 at a time, its pixels
// were parts of 32-byte sectors (16 images of odd widths, 630 MB, with all but
// the stores left out: 2 TB/s; in all 760 -> 702 us; 915 -> 912 us at 5760 x
// 3240). One tile's lanes store their own: a store has four whole strips in a
// row, and the way through shared memory took as long (1002 x 751: 50.6 us both,
// 16 crops 37.3 against 36.4).
template <int NQ>
__device__ __forceinline__ void store_strips(const ImageDesc* D, const StripAcc<NQ>& acc,
                                             StripTables<NQ>& t, int ox, int y0) {
  const int lane = threadIdx.x & 31, strip = lane >> 3, rp = lane & 7;
  const int H = D->out_h, W = D->out_w;
  float* out = D->out;
  const int64_t plane = (int64_t)H * W;
  // four columns per store where the output's rows are 16-byte aligned
  const bool vec = (W & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  if constexpr (NQ == 1) {
    const int x = ox + 4 * strip, y = y0 + 2 * rp;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (y + j >= H || x >= W) continue;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float* o = out + k * plane + (int64_t)(y + j) * W + x;
        const float2 a = acc[j][0][k], b = acc[j][1][k];
        if (vec) {
          *reinterpret_cast<float4*>(o) = make_float4(a.x, a.y, b.x, b.y);
        } else {
          o[0] = a.x;
          if (x + 1 < W) o[1] = a.y;
          if (x + 2 < W) o[2] = b.x;
          if (x + 3 < W) o[3] = b.y;
        }
      }
    }
  } else {
    float* buf = reinterpret_cast<float*>(&t);
    strips_to_rows<NQ>(acc, buf, lane);
    __syncwarp();
    if (vec) {
      const int piece = lane & 7, r0 = lane >> 3, x = ox + 4 * piece;
      const int rows = x < W ? H - y0 - r0 : 0;   // of this lane, from its first
      float* o = out + (int64_t)(y0 + r0) * W + x;
#pragma unroll
      for (int k = 0; k < 3; ++k, o += plane)
#pragma unroll
        for (int i = 0; i < 16; i += 4)
          if (i < rows)
            *reinterpret_cast<float4*>(o + (int64_t)i * W) = *reinterpret_cast<const float4*>(
                buf + k * 512 + (r0 + i) * 32 + 4 * (piece ^ ((r0 + i) >> 1)));
    } else {
      const int x = ox + lane;
      const int rows = x < W ? H - y0 : 0;
      float* o = out + (int64_t)y0 * W + x;
#pragma unroll
      for (int k = 0; k < 3; ++k, o += plane)
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (i < rows) o[(int64_t)i * W] = row_value<NQ>(buf, k, i, lane);
    }
  }
}

// A segment's end (rare: its code is kept small): puts the region's pixels onto
// the output and clears them. go / add, the same over a tile's lanes: whether
// the lane's tile is written, and whether onto what an earlier segment left.
template <int NQ>
__device__ __forceinline__ void fold_strips(const ImageDesc* D, StripAcc<NQ>& acc,
                                            StripTables<NQ>& t, int ox, int y0, bool go, bool add) {
  constexpr int C = 16 * NQ;
  static_assert(sizeof(t.x) + sizeof(t.r) >= 48 * C * sizeof(float), "the sums fit the table");
  const int lane = threadIdx.x & 31;
  float* buf = reinterpret_cast<float*>(&t);
  __syncwarp();
  if (go) {
    strips_to_rows<NQ>(acc, buf, lane);
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int h = 0; h < 2 * NQ; ++h) acc[j][h][0] = acc[j][h][1] = acc[j][h][2] = f2(0.0f, 0.0f);
  }
  __syncwarp();
  const int H = D->out_h, W = D->out_w;
  const int x = ox + lane % C;
  if (go && x < W) {
    float* o = D->out + (int64_t)y0 * W + x;
#pragma unroll 1
    for (int k = 0; k < 3; ++k, o += (int64_t)H * W) {
#pragma unroll 4
      for (int r = lane / C; r < 16; r += 32 / C) {
        if (y0 + r >= H) break;
        const float v = row_value<NQ>(buf, k, r, lane);
        o[(int64_t)r * W] = add ? o[(int64_t)r * W] + v : v;
      }
    }
  }
  __syncwarp();
  t.clear_front(lane);
  __syncwarp();
}

template <int PF, bool GRID>
__global__ void __launch_bounds__(32) k_raster_fwd16(Ws w, const uint32_t* vals) {
  griddep_release();
  griddep_wait();
  __shared__ __align__(16) float4 raw[PF][4 * 32];
  __shared__ StripTables<1> T[PF];
  __shared__ uint32_t qbuf[GRID ? GridSource<32, PF>::QCAP : 1];

  const int lane = threadIdx.x;
  const ImageDesc* D;
  int ox, oy, tx, ty;
  tile_origin<16>(w, blockIdx.x, D, ox, oy, tx, ty);
  const int strip = lane >> 3, rp = lane & 7;

  StripAcc<1> acc;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int h = 0; h < 2; ++h) acc[j][h][0] = acc[j][h][1] = acc[j][h][2] = f2(0.0f, 0.0f);
#pragma unroll
  for (int j = 0; j < PF; ++j) T[j].clear_front(lane);

  typename std::conditional<GRID, GridSource<32, PF>, SortedSource<32, PF>>::type src;
  // grid mode: the tile's slice [lbase, lbase + lcount) of the pair list, where
  // the forward leaves its Gaussian ids (ascending) for the adjoint
  int lbase = 0, lcount = 0;
  bool lok = false;
  if constexpr (GRID) {
    grid_source_init<16, 32, PF>(w, D, ox, oy, qbuf, src);
    {
      // the tile's pair count: the prefix, along its tile row, of the
      // footprint pass's per-row differences
      const uint32_t* row = w.tcount + (blockIdx.x - tx);
      uint32_t s = 0u;
      for (int x = lane; x <= tx; x += 32) s += row[x];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      lcount = (int)s;
    }
    if (lane == 0) {
      const unsigned long long b = atomicAdd(&w.hdr->list_cursor, (unsigned long long)lcount);
      const bool fits = b + (unsigned long long)lcount <= (unsigned long long)w.capacity;
      lbase = fits ? (int)b : -1;
      w.ranges[blockIdx.x] = fits ? make_uint2((uint32_t)b, (uint32_t)(b + lcount)) : make_uint2(0u, 0u);
      if (!fits && lcount > 0) atomicOr(&w.hdr->status, kStCapacity);
    }
    lbase = __shfl_sync(0xffffffffu, lbase, 0);
    lok = lbase >= 0;
  } else {
    const uint2 range = w.ranges[blockIdx.x];
    src.vals = vals;
    src.pos = (int)range.x;
    src.end = (int)range.y;
  }
  int total;   // the tile's Gaussians (grid mode: the footprint count)
  if constexpr (GRID) total = lcount; else total = src.end - src.pos;
  // the next batch's ids, appended in grid mode to the tile's slice of the list
  int got = 0;
  uint32_t gid[PF];
  auto take = [&]() -> int {
    if (got >= total) return 0;
    const int n = src.next(gid);
    if constexpr (GRID) {
      if (got + n > lcount) {   // the footprint count and the tile test disagree
        if (lane == 0) atomicOr(&w.hdr->status, kStInternal);
        lok = false;
      }
      if (lok) {
#pragma unroll
        for (int j = 0; j < PF; ++j) {
          const int i = j * 32 + lane;
          if (i < n) w.vals[0][lbase + got + i] = gid[j];
        }
      }
    }
    got += n;
    return n;
  };
  int nb = take(), nn = 0;   // entries of this batch and of the next
  if (nb > 0) {
    issue_slots<PF>(w, gid, nb, raw);
    nn = take();
  }
  int done = 0;   // entries summed
  while (nb > 0) {
    if (done > 0 && done % kSeg == 0)
      fold_strips<1>(D, acc, T[0], ox, oy - D->row0, true, done > kSeg);   // a segment ends
    cp_async_wait_all();
    __syncwarp();
    StripMasks ms[PF];
#pragma unroll
    for (int j = 0; j < PF; ++j)
      ms[j] = strip_masks(stage_strips<1>(raw[j], lane, j * 32 + 31 - lane < nb, ox, oy, T[j]), strip);
    __syncwarp();
    int n2 = 0;
    if (nn > 0) {
      issue_slots<PF>(w, gid, nn, raw);
      n2 = take();
    }
#pragma unroll
    for (int j = 0; j < PF; ++j) walk_strips<1>(acc, ms[j], strip, rp, T[j]);
    __syncwarp();
    done += nb;
    nb = nn;
    nn = n2;
  }
  if constexpr (GRID) {   // fewer found than counted: the list is incomplete
    if (got < total && lane == 0) atomicOr(&w.hdr->status, kStInternal);
  }

  if (done > kSeg)
    fold_strips<1>(D, acc, T[0], ox, oy - D->row0, true, true);
  else
    store_strips<1>(D, acc, T[0], ox, oy - D->row0);
}

// ---------------------------------------------------------------------------
// Forward of a 16 x 16 tile by a team of NW warps, for images of few tiles: the
// warps sum the segments of the tile's list side by side, each as
// k_raster_fwd16 does, and their sums are added in list order. In grid mode the
// team first builds the tile's list together (each warp a run of the
// candidates: count, prefix over the warps, write).
//
// What bounds it: the strips' arithmetic, once enough warps run. One warp per
// tile left 2,025 tiles with lists of 23,000 at 3 or 4 warps per scheduler (the
// fuller ones last: 3.73 ms; teams of four: 2.99) and 250 tiles with lists of
// 4,000 to 10,000 waiting for the longest (514 us; teams of eight: 108). The
// host's rule says where a team runs and what else was measured.
// ---------------------------------------------------------------------------
struct TeamWarp {
  float4 raw[1][4 * 32];
  StripTables<1> t;     // a segment's sums (768 floats) go to t.r once it is walked
  uint32_t q[256];      // fallback enumeration (a list that did not fit)
};
static_assert(GridSource<32, 1>::QCAP == 256, "TeamWarp::q");
static_assert(sizeof(StripTables<1>::r) >= 768 * sizeof(float), "segment sums");

// The tile's list from the workspace (this launch may have written it).
struct ListSource {
  const uint32_t* list;
  int pos, end;
  __device__ __forceinline__ int next(uint32_t (&gid)[1]) {
    const int nb = max(0, min(32, end - pos)), lane = threadIdx.x & 31;
    gid[0] = lane < nb ? __ldcg(list + pos + lane) : 0u;
    pos += nb;
    return nb;
  }
};

// Two CTAs of eight per SM are all that fit: with the 128 registers that this
// leaves instead of 86, 250 tiles with lists of 4,000 to 10,000 take 108 instead
// of 116 us and 64 to 225 tiles of k-sigma boxes 7% to 11% less. For four warps
// the compiler's own choice (96) is the best: 2.90 ms on the paper's 2,025
// tiles, 2.99 with five CTAs asked for, 3.10 with one.
template <int NW, bool GRID>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 2 : 0) k_raster_fwd_team(Ws w, const uint32_t* vals) {
  griddep_release();
  griddep_wait();
  constexpr int NT = NW * 32, PER = 768 / NT;
  extern __shared__ float4 team_smem[];
  TeamWarp* team = reinterpret_cast<TeamWarp*>(team_smem);
  __shared__ int s_base, s_cnt[NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  TeamWarp& M = team[warp];
  const ImageDesc* D;
  int ox, oy, tx, ty;
  tile_origin<16>(w, blockIdx.x, D, ox, oy, tx, ty);
  const int strip = lane >> 3, rp = lane & 7;

  int total;
  const uint32_t* list;
  bool listed = true;
  GridSource<32, 1> cells;
  if constexpr (GRID) {
    grid_source_init<16, 32, 1>(w, D, ox, oy, M.q, cells);
    // the tile's pair count: the prefix, along its tile row, of the footprint
    // pass's per-row differences
    const uint32_t* row = w.tcount + (blockIdx.x - tx);
    uint32_t s = 0u;
    for (int x = lane; x <= tx; x += 32) s += row[x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    total = (int)s;
    if (threadIdx.x == 0) {
      const unsigned long long b = atomicAdd(&w.hdr->list_cursor, (unsigned long long)total);
      const bool fits = b + (unsigned long long)total <= (unsigned long long)w.capacity;
      s_base = fits ? (int)b : -1;
      w.ranges[blockIdx.x] = fits ? make_uint2((uint32_t)b, (uint32_t)(b + total)) : make_uint2(0u, 0u);
      if (!fits && total > 0) atomicOr(&w.hdr->status, kStCapacity);
    }
    // this warp's run of candidates, counted
    Candidates c = cells.cand;
    const int run = ((c.total + NW * 128 - 1) / (NW * 128)) * 128;
    const int c0 = min(c.total, warp * run);
    c.total = min(c.total, c0 + run);
    int cnt = 0;
    for (c.seek(c0); c.cur < c.total; c.cur += 128) {
      uint2 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) { v[k] = c.load(k, c.gid); c.advance(); }
#pragma unroll
      for (int k = 0; k < 4; ++k) cnt += __popc(__ballot_sync(0xffffffffu, c.meets(v[k])));
    }
    if (lane == 0) s_cnt[warp] = cnt;
    __syncthreads();
    int at = 0, all = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
      if (k == warp) at = all;
      all += s_cnt[k];
    }
    if (all != total && threadIdx.x == 0) atomicOr(&w.hdr->status, kStInternal);
    listed = s_base >= 0;
    uint32_t* slice = w.vals[0] + (listed ? s_base : 0);
    list = slice;
    total = min(total, all);
    if (listed) {
      for (c.seek(c0); c.cur < c.total; c.cur += 128) {
        uint2 v[4];
        uint32_t g[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { g[k] = c.gid; v[k] = c.load(k, c.gid); c.advance(); }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bool hit = c.meets(v[k]);
          const unsigned bal = __ballot_sync(0xffffffffu, hit);
          const int i = at + __popc(bal & ((1u << lane) - 1u));
          if (hit && i < total) slice[i] = g[k];
          at += __popc(bal);
        }
      }
      __syncthreads();   // the list is complete (and visible to the team)
    }
  } else {
    const uint2 range = w.ranges[blockIdx.x];
    list = vals + range.x;
    total = (int)(range.y - range.x);
  }

  const int nseg = (total + kSeg - 1) / kSeg;
  float sum[PER];   // of the values threadIdx.x + i * NT, value = channel * 256 + row * 16 + column
#pragma unroll
  for (int i = 0; i < PER; ++i) sum[i] = 0.0f;
  int passed = 0;   // fallback: list entries enumerated so far
  for (int first = 0; first < nseg; first += NW) {   // uniform over the team
    const int seg = first + warp;
    if (seg < nseg) {
      StripAcc<1> acc;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[j][h][0] = acc[j][h][1] = acc[j][h][2] = f2(0.0f, 0.0f);
      M.t.clear_front(lane);
      const int lo = seg * kSeg, hi = min(total, lo + kSeg);
      ListSource src{list, lo, hi};
      uint32_t gid[1];
      // the next batch: from the list, or (a list that did not fit) enumerated
      // again, past the other warps' segments
      auto next = [&]() -> int {
        if (!GRID || listed) return src.next(gid);
        if (passed >= hi) return 0;
        int nb = cells.next(gid);
        __syncwarp();
        while (passed < lo && nb > 0) {
          passed += nb;
          nb = cells.next(gid);
          __syncwarp();
        }
        passed += nb;
        return nb;
      };
      int nb = next(), nn = 0;
      if (nb > 0) {
        issue_slots<1>(w, gid, nb, M.raw);
        nn = next();
      }
      while (nb > 0) {
        cp_async_wait_all();
        __syncwarp();
        const StripMasks ms =
            strip_masks(stage_strips<1>(M.raw[0], lane, 31 - lane < nb, ox, oy, M.t), strip);
        __syncwarp();
        int n2 = 0;
        if (nn > 0) {
          issue_slots<1>(w, gid, nn, M.raw);
          n2 = next();
        }
        walk_strips<1>(acc, ms, strip, rp, M.t);
        __syncwarp();
        nb = nn;
        nn = n2;
      }
      float* ps = reinterpret_cast<float*>(M.t.r);
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k)
          *reinterpret_cast<float4*>(ps + k * 256 + (2 * rp + j) * 16 + 4 * strip) =
              make_float4(acc[j][0][k].x, acc[j][0][k].y, acc[j][1][k].x, acc[j][1][k].y);
    }
    __syncthreads();
    const int n = min(NW, nseg - first);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      for (int k = 0; k < n; ++k) {
        const float v = reinterpret_cast<const float*>(team[k].t.r)[threadIdx.x + i * NT];
        sum[i] = first + k == 0 ? v : sum[i] + v;
      }
    }
    __syncthreads();
  }
  const int H = D->out_h, W = D->out_w;
  const int64_t plane = (int64_t)H * W;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int v = threadIdx.x + i * NT;
    const int x = ox + (v & 15), y = oy - D->row0 + ((v >> 4) & 15);
    if (x < W && y < H) D->out[(v >> 8) * plane + (int64_t)y * W + x] = sum[i];
  }
}

template <int TILE, int BY, int PF, bool GRID>
__global__ void __launch_bounds__(TILE * TILE / BY) k_raster_fwd(Ws w, const uint32_t* vals) {
  griddep_release();
  griddep_wait();
  constexpr int NT = TILE * TILE / BY, BATCH = NT * PF, NQ = BY / 2, HP = TILE / 2;
  __shared__ __align__(16) float4 raw[2][BATCH * kRecordF4];
  __shared__ float4 gA[BATCH], gB[BATCH], gC[BATCH];
  __shared__ float4 rq[BATCH * HP];
  __shared__ uint32_t qbuf[GRID ? GridSource<NT, PF>::QCAP : 1];

  const ImageDesc* D;
  int ox, oy, tx, ty;
  tile_origin<TILE>(w, blockIdx.x, D, ox, oy, tx, ty);
  const int col = threadIdx.x % TILE;
  const int row0 = (threadIdx.x / TILE) * BY;
  const int pair0 = row0 / 2;
  const float fcol = (float)col;

  float2 acc[NQ][3];
#pragma unroll
  for (int j = 0; j < NQ; ++j) acc[j][0] = acc[j][1] = acc[j][2] = f2(0.0f, 0.0f);

  typename std::conditional<GRID, GridSource<NT, PF>, SortedSource<NT, PF>>::type src;
  // grid mode: the tile's slice [lbase, lbase + lcount) of the pair list, where
  // the forward leaves its Gaussian ids (ascending) for the adjoint
  __shared__ int sl_base;
  int lbase = 0, lcount = 0;
  bool lok = false;
  if constexpr (GRID) {
    grid_source_init<TILE, NT, PF>(w, D, ox, oy, qbuf, src);
    {
      // the tile's pair count: the prefix, along its tile row, of the
      // footprint pass's per-row differences
      const int lane = threadIdx.x & 31;
      const uint32_t* row = w.tcount + (blockIdx.x - tx);
      uint32_t acc = 0u;
      for (int x = lane; x <= tx; x += 32) acc += row[x];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      lcount = (int)acc;
    }
    if (threadIdx.x == 0) {
      const unsigned long long b = atomicAdd(&w.hdr->list_cursor, (unsigned long long)lcount);
      const bool fits = b + (unsigned long long)lcount <= (unsigned long long)w.capacity;
      sl_base = fits ? (int)b : -1;
      w.ranges[blockIdx.x] = fits ? make_uint2((uint32_t)b, (uint32_t)(b + lcount)) : make_uint2(0u, 0u);
      if (!fits && lcount > 0) atomicOr(&w.hdr->status, kStCapacity);
    }
    __syncthreads();
    lbase = sl_base;
    lok = lbase >= 0;
  } else {
    const uint2 range = w.ranges[blockIdx.x];
    src.vals = vals;
    src.pos = (int)range.x;
    src.end = (int)range.y;
  }
  int total;   // the tile's Gaussians (grid mode: the footprint count)
  if constexpr (GRID) total = lcount; else total = src.end - src.pos;
  // the next batch's ids, appended in grid mode to the tile's slice of the list
  int got = 0;
  uint32_t gid[PF];
  auto take = [&]() -> int {
    if (got >= total) return 0;
    const int n = GRID && TILE == 32 && PF == 1 ? next_apart(src, gid) : src.next(gid);
    if constexpr (GRID) {
      if (got + n > lcount) {   // the footprint count and the tile test disagree
        if (threadIdx.x == 0) atomicOr(&w.hdr->status, kStInternal);
        lok = false;
      }
      if (lok) {
#pragma unroll
        for (int j = 0; j < PF; ++j) {
          const int i = j * NT + threadIdx.x;
          if (i < n) w.vals[0][lbase + got + i] = gid[j];
        }
      }
    }
    got += n;
    return n;
  };
  int nb = take(), nn = 0;   // entries of this batch and of the next
  if (nb > 0) {
    issue_records<NT, PF>(w, gid, nb, raw[0]);
    nn = take();
  }
  for (int b = 0; nb > 0; ++b) {
    cp_async_wait_all();
    __syncthreads();
    stage_records<TILE, NT>(raw[b & 1], nb, ox, oy, gA, gB, gC);
    __syncthreads();
    stage_rowpairs<TILE, NT>(nb, gB, gC, rq);
    __syncthreads();
    int n2 = 0;
    if (nn > 0) {
      issue_records<NT, PF>(w, gid, nn, raw[(b + 1) & 1]);
      n2 = take();
    }
    // Two operand sets in registers: Gaussian i + 1's loads overlap i's math.
    FwdOps<NQ> A, B;
    A.load(gA, gC, rq, 0, HP, pair0);
    for (int i = 0; i < nb; i += 2) {
      if (i + 1 < nb) B.load(gA, gC, rq, i + 1, HP, pair0);
      fwd_gaussian<NQ>(acc, A, fcol);
      if (i + 1 >= nb) break;
      if (i + 2 < nb) A.load(gA, gC, rq, i + 2, HP, pair0);
      fwd_gaussian<NQ>(acc, B, fcol);
    }
    __syncthreads();
    nb = nn;
    nn = n2;
  }
  if constexpr (GRID) {   // fewer found than counted: the list is incomplete
    if (got < total && threadIdx.x == 0) atomicOr(&w.hdr->status, kStInternal);
  }

  const int H = D->out_h, W = D->out_w;
  const int x = ox + col;
  if (x < W) {
    float* out = D->out;
    const int64_t plane = (int64_t)H * W;
#pragma unroll
    for (int k = 0; k < BY; ++k) {
      const int y = oy - D->row0 + row0 + k;   // output row
      if (y < H) {
        const int64_t o = (int64_t)y * W + x;
        const int j = k / 2;
        out[o] = (k & 1) ? acc[j][0].y : acc[j][0].x;
        out[plane + o] = (k & 1) ? acc[j][1].y : acc[j][1].x;
        out[2 * plane + o] = (k & 1) ? acc[j][2].y : acc[j][2].x;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Forward over a pair of horizontally adjacent 16 x 16 tiles (grid-implicit
// binning, tile 16): one warp renders a 32 x 16 region in four strips of 8
// columns (two per tile), each lane 8 columns of a row pair, so that a step's
// loads and mask work serve 16 pixels. The pair's candidates are enumerated and
// staged once; the two tiles' lists are left for the adjoint exactly as the
// single-tile forward leaves them (same Gaussians, ascending ids). Column
// terms are relative to their own tile and every pixel sums its Gaussians in
// the same order, so the image is bitwise the single-tile forward's.
//
// A step in a loop of its own takes 111 scheduler cycles for 16 pixels per
// lane, the single tile's 64 for 8: the arithmetic (94 at 2.3 cycles per FFMA2)
// bounds it. Against the former pair layout (each lane a column of both tiles,
// 7 shared loads per 16 pixels): 1168 -> 1007 us on 518,400 Gaussians at
// 5760 x 3240 (windows of 74 px on average), 857 -> 799 us on 16 uneven images,
// 87 -> 73 us at scale 24. Wider strips cost small windows more columns
// (1002 x 751 at scale 3.7, 14 px windows: 52 us by tiles, 70 by pairs) and pairs
// make half as many warps: the host's rule says where they pay. The register cap
// (128; spills, 8 bytes, with 64 Gaussians a round only) gives 16 CTAs per SM; 18
// CTAs (112, spills) were 2% faster on the uneven batch and 1% to 10% slower
// elsewhere.
// ---------------------------------------------------------------------------
template <int PF>
struct PairSource {
  static constexpr int NT = 32, BATCH = NT * PF, KR = 4;
  static constexpr int QCAP = BATCH + 32 * KR <= 256 ? 256 : 512;
  uint32_t* q;           // shared [QCAP] ids
  uint8_t* qf;           // shared [QCAP] hit flags: 1 tile A, 2 tile B
  Candidates cand;       // of the pair's region
  int head, tail, XM;    // tile A [X0, XM - 1], tile B [XM, X1]
  // the next batch: ids and flags of up to BATCH kept candidates, gid order, at
  // most room_a of them in tile A and room_b in tile B
  __device__ __forceinline__ int next(uint32_t (&gid)[PF], uint32_t (&fl)[PF], int room_a,
                                      int room_b) {
    const int lane = threadIdx.x & 31;
    while (tail - head < BATCH && cand.cur < cand.total) {
      uint32_t g[KR];
      uint2 v[KR];
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        g[k] = cand.gid;
        v[k] = cand.load(k, cand.gid);
        cand.advance();
      }
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        const bool hit = cand.meets(v[k]);
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        if (hit) {
          const int at = (tail + __popc(bal & ((1u << lane) - 1u))) & (QCAP - 1);
          q[at] = g[k];
          qf[at] = (uint8_t)(((short)(v[k].x & 0xffffu) < XM ? 1 : 0) |
                             ((short)(v[k].y & 0xffffu) >= XM ? 2 : 0));
        }
        tail += __popc(bal);
      }
      cand.cur += 32 * KR;
    }
    __syncwarp();
    int nb = min(BATCH, tail - head);
    const int n = nb;
#pragma unroll
    for (int j = 0; j < PF; ++j) {
      const int i = j * NT + lane;
      const int at = (head + i) & (QCAP - 1);
      gid[j] = i < n ? q[at] : 0u;
      fl[j] = i < n ? (uint32_t)qf[at] : 0u;
      if (min(room_a, room_b) < 32) {   // a segment may end inside: the batch ends with it
        const unsigned ba = __ballot_sync(0xffffffffu, fl[j] & 1u);
        const unsigned bb = __ballot_sync(0xffffffffu, fl[j] & 2u);
        if (__popc(ba) > room_a) nb = min(nb, j * NT + (int)__fns(ba, 0, room_a + 1));
        if (__popc(bb) > room_b) nb = min(nb, j * NT + (int)__fns(bb, 0, room_b + 1));
        room_a = max(0, room_a - __popc(ba));
        room_b = max(0, room_b - __popc(bb));
      } else {
        room_a -= 32;
        room_b -= 32;
      }
    }
    head += nb;
    __syncwarp();
    return nb;
  }
};

template <int PF>
__global__ void __launch_bounds__(32, 16) k_raster_fwd_pair(Ws w) {
  griddep_release();
  griddep_wait();
  using Src = PairSource<PF>;
  __shared__ __align__(16) float4 raw[PF][4 * 32];
  __shared__ StripTables<2> T[PF];
  __shared__ uint32_t qbuf[Src::QCAP];
  __shared__ uint8_t qflg[Src::QCAP];
  __shared__ int sbase;

  const int lane = threadIdx.x;
  // the pair: image, tile row, tile A's column (tile B = A + 1 when it exists)
  int im = 0;
  {
    int lo = 0, hi = w.n_images - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (w.images[mid].p_base <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    im = lo;
  }
  const ImageDesc* D = &w.images[im];
  const int pairs_x = (D->tiles_x + 1) >> 1;
  const int lp = blockIdx.x - D->p_base;
  const int ty = lp / pairs_x;
  const int txa = 2 * (lp - ty * pairs_x);
  const bool has_b = txa + 1 < D->tiles_x;
  const int ox = txa * 16, oy = ty * 16 + D->row0;   // image rows (a band's start at row0)
  const int ta = D->t_base + ty * D->tiles_x + txa;

  // pair counts of tiles A and B: prefixes, along their tile row, of the
  // footprint pass's per-row differences
  int na, nb_ = 0;
  {
    const uint32_t* row = w.tcount + D->t_base + (int64_t)ty * D->tiles_x;
    uint32_t s = 0u;
    for (int x = lane; x <= txa; x += 32) s += row[x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    na = (int)s;
    if (has_b) nb_ = na + (int)row[txa + 1];
  }
  // the two tiles' slices of the pair list: A at [base, base + na), B after it
  if (lane == 0) {
    const unsigned long long tot = (unsigned long long)(na + nb_);
    const unsigned long long b = atomicAdd(&w.hdr->list_cursor, tot);
    const bool fits = b + tot <= (unsigned long long)w.capacity;
    sbase = fits ? (int)b : -1;
    w.ranges[ta] = fits ? make_uint2((uint32_t)b, (uint32_t)(b + na)) : make_uint2(0u, 0u);
    if (has_b)
      w.ranges[ta + 1] = fits ? make_uint2((uint32_t)(b + na), (uint32_t)(b + na + nb_))
                              : make_uint2(0u, 0u);
    if (!fits && tot > 0) atomicOr(&w.hdr->status, kStCapacity);
  }
  __syncwarp();
  const int lbase = sbase;
  bool lok = lbase >= 0;
  int pos_a = 0, pos_b = 0;

  // candidate cells of the pair region (the per-image reach of the windows)
  Src src;
  src.q = qbuf;
  src.qf = qflg;
  src.XM = ox + 16;
  src.head = src.tail = 0;
  candidate_box(w, D, ox, ox + (has_b ? 31 : 15), oy, oy + 15, src.cand);
  // append a batch to the two tiles' lists (each in id order), checking the
  // footprint pass's counts against the tile tests
  auto keep = [&](const uint32_t (&ids)[PF], const uint32_t (&fl)[PF], int n) {
#pragma unroll
    for (int j = 0; j < PF; ++j) {
      const int i = j * 32 + lane;
      const bool fa = i < n && (fl[j] & 1u), fb = i < n && (fl[j] & 2u);
      const unsigned ba = __ballot_sync(0xffffffffu, fa), bb = __ballot_sync(0xffffffffu, fb);
      const unsigned lt = (1u << lane) - 1u;
      const int at = pos_a + __popc(ba & lt), bt = pos_b + __popc(bb & lt);
      if (lok && fa && at < na) w.vals[0][lbase + at] = ids[j];
      if (lok && fb && bt < nb_) w.vals[0][lbase + na + bt] = ids[j];
      pos_a += __popc(ba);
      pos_b += __popc(bb);
    }
    if (pos_a > na || pos_b > nb_) {
      if (lane == 0) atomicOr(&w.hdr->status, kStInternal);
      lok = false;
    }
  };

  const int strip = lane >> 3, rp = lane & 7;
  StripAcc<2> acc;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int h = 0; h < 4; ++h) acc[j][h][0] = acc[j][h][1] = acc[j][h][2] = f2(0.0f, 0.0f);
#pragma unroll
  for (int j = 0; j < PF; ++j) T[j].clear_front(lane);

  auto next = [&](uint32_t (&ids)[PF], uint32_t (&fl)[PF]) {
    return src.next(ids, fl, kSeg - (pos_a & (kSeg - 1)), kSeg - (pos_b & (kSeg - 1)));
  };
  uint32_t gid[PF], fl[PF];
  int nb0 = next(gid, fl);   // batch 0
  keep(gid, fl, nb0);
  int next_a = pos_a, next_b = pos_b;   // the two lists' entries up to and with batch b
  int nb1 = 0;
  if (nb0 > 0) {
    issue_slots<PF>(w, gid, nb0, raw);
    nb1 = next(gid, fl);      // batch 1
    keep(gid, fl, nb1);
  }
  int done_a = 0, done_b = 0;         // list entries of the two tiles summed so far
  int written_a = 0, written_b = 0;   // ... and already on the output
  while (nb0 > 0) {
    const bool end_a = done_a > written_a && (done_a & (kSeg - 1)) == 0;   // a segment ends
    const bool end_b = done_b > written_b && (done_b & (kSeg - 1)) == 0;
    if (end_a || end_b) {
      fold_strips<2>(D, acc, T[0], ox, oy - D->row0, strip < 2 ? end_a : end_b,
                     (strip < 2 ? written_a : written_b) > 0);
      if (end_a) written_a = done_a;
      if (end_b) written_b = done_b;
    }
    done_a = next_a;
    done_b = next_b;
    next_a = pos_a;
    next_b = pos_b;
    cp_async_wait_all();
    __syncwarp();
    StripMasks ms[PF];
#pragma unroll
    for (int j = 0; j < PF; ++j)
      ms[j] = strip_masks(stage_strips<2>(raw[j], lane, j * 32 + 31 - lane < nb0, ox, oy, T[j]), strip);
    __syncwarp();
    int nb2 = 0;
    if (nb1 > 0) {
      issue_slots<PF>(w, gid, nb1, raw);
      nb2 = next(gid, fl);    // batch b + 2
      keep(gid, fl, nb2);
    }
#pragma unroll
    for (int j = 0; j < PF; ++j) walk_strips<2>(acc, ms[j], strip, rp, T[j]);
    __syncwarp();
    nb0 = nb1;
    nb1 = nb2;
  }
  if (pos_a != na || pos_b != nb_) {   // fewer kept than counted: stale list entries
    if (lane == 0) atomicOr(&w.hdr->status, kStInternal);
  }

  if (written_a + written_b > 0)
    fold_strips<2>(D, acc, T[0], ox, oy - D->row0, true, (strip < 2 ? written_a : written_b) > 0);
  else
    store_strips<2>(D, acc, T[0], ox, oy - D->row0);
}

template <int TILE, int BY, int PF>
cudaError_t run(const Ws& w, const uint32_t* vals, cudaStream_t s) {
  constexpr int NT = TILE * TILE / BY;
  LaunchScope ls(kKRasterFwd, s);
  if (w.grid) return launch_chain(k_raster_fwd<TILE, BY, PF, true>, dim3(w.tiles), dim3(NT), 0, s, w, vals);
  return launch_chain(k_raster_fwd<TILE, BY, PF, false>, dim3(w.tiles), dim3(NT), 0, s, w, vals);
}

template <int PF>
cudaError_t run16(const Ws& w, const uint32_t* vals, cudaStream_t s) {
  LaunchScope ls(kKRasterFwd, s);
  if (w.grid) return launch_chain(k_raster_fwd16<PF, true>, dim3(w.tiles), dim3(32), 0, s, w, vals);
  return launch_chain(k_raster_fwd16<PF, false>, dim3(w.tiles), dim3(32), 0, s, w, vals);
}

template <int NW>
cudaError_t run_team(const Ws& w, const uint32_t* vals, cudaStream_t s) {
  constexpr size_t smem = NW * sizeof(TeamWarp);
  auto kernel = w.grid ? k_raster_fwd_team<NW, true> : k_raster_fwd_team<NW, false>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  LaunchScope ls(kKRasterFwd, s);
  return launch_chain(kernel, dim3(w.tiles), dim3(NW * 32), smem, s, w, vals);
}

// Launch configurations: tile edge -> rows per thread (threads = TILE^2 / BY);
// batch = Gaussians staged per round = threads * PF, PF in {1, 2} (the host
// accepts only these batches; 0 selects PF = 1). Tile 16 with 64 a round never
// measured faster than 32 (forward calls, us, 32 / 64: 65,536 Gaussians at 1024 x
// 1024 36 / 40, 220,052 at 1002 x 751 66 / 74, pairs at 5760 x 3240 1032 / 1230, the
// ratio window at 720 x 720 2,933 / 3,906, whose teams take 32 only): it costs a
// second table per warp. It stays for callers that name it, at 0.7 to 0.84 of what
// the layout before the strips took with it (53, 105, 1603, 4,633).
cudaError_t dispatch(const Ws& w, const uint32_t* vals, int batch, cudaStream_t s) {
  if (w.tiles == 0) return cudaSuccess;
  if (w.pair) {   // grid binning, tile 16: one warp per horizontal pair of tiles
    LaunchScope ls(kKRasterFwd, s);
    if (batch >= 64)
      return launch_chain(k_raster_fwd_pair<2>, dim3(w.n_pairs), dim3(32), 0, s, w);
    return launch_chain(k_raster_fwd_pair<1>, dim3(w.n_pairs), dim3(32), 0, s, w);
  }
  switch (w.tile) {
    case 8:   // 32 threads
      return batch >= 64 ? run<8, 2, 2>(w, vals, s) : run<8, 2, 1>(w, vals, s);
    case 32:  // 64 threads
      return batch >= 128 ? run<32, 16, 2>(w, vals, s) : run<32, 16, 1>(w, vals, s);
    default:  // 32 threads
      if (w.team) return w.team > 4 ? run_team<8>(w, vals, s) : run_team<4>(w, vals, s);
      return batch >= 64 ? run16<2>(w, vals, s) : run16<1>(w, vals, s);
  }
}

}  // namespace

cudaError_t launch_raster_fwd(const Ws& w, const uint32_t* vals, int batch, cudaStream_t s) {
  return dispatch(w, vals, batch, s);
}

}  // namespace gs
