// X-ray rasterizer of FaCT-GS (Sec. 3.2, 3.5; Eq. 3, Eq. 4), forward and backward, sm_103a,
// for a batch of up to 32 independent instances (own Gaussians, views and detector size) in
// one launch per pass; a single reconstruction is a batch of one.
//
// Pipeline of one call (all on `stream`, no host read-back); a block of the first kernels is 256
// consecutive Gaussians of one view:
//   preprocess   one thread per (instance, view, Gaussian): the view's camera frame, local-affine
//                (EWA) projection, integration factor mu, conic, 3-sigma box, and the box's
//                tiles that the cut ellipse actually meets (tight tile rule, a range of tiles
//                per tile row)
//   then the (view, tile) lists, by one of two routes with the same lists:
//   direct       (up to 1600 tiles per view, 2048 in small calls) preprocess also counts each
//                block's records per tile; key_scan turns the counts into each block's offset in
//                every list, the ranges and the pair total; emit writes each record to its place
//                in the lists
//   sorted       (more tiles) block sums and their scan, emit of (key, record) pairs in record
//                order, stable radix sort over the tile bits, ranges
//   raster_fwd   one CTA per (instance, view, tile), records on lanes
//   raster_bwd   one warp per (instance, view, tile), records on lanes; six moment sums of
//                g * exp(-q/2) per record, then one pair of float4 atomics (per-Gaussian backward,
//                Sec. 3.5)
//   chain        a thread per (Gaussian, 8 views): moments -> footprint gradients ->
//                d(mean, rho, scale, quaternion)
// The instance table travels by value as a __grid_constant__ kernel parameter, so a call does
// no host-to-device copy and can be captured in a CUDA graph.
#include <algorithm>
#include <cmath>

#include "gs_footprint.cuh"

namespace gs {
namespace {

using gsd::ex2;

constexpr int kThreads = 256;
constexpr int kMaxInst = GS_MAX_INSTANCES;
// widest digit of the tile-key sort: 10 tile bits (512^2 at tile 16) sort in two passes of 5
constexpr int kTileDigitBits = 8;

// The direct route keeps a counter per (block of 256 records, tile) and, in emit, a 32-bit lane
// mask per (warp, tile) in shared memory: 44 bytes a tile, 88 KB at 2048.  Its cost grows with the
// blocks times the tiles (10 bytes of counts and offsets each; two CTAs of emit per SM from 1764
// tiles on), the sort's with the pairs (about 60 bytes each) and its launches.  Forward, sorted
// against direct, us, from 4.6 pairs a record (scale 0.005) to 14 (0.02):
//   75 views, 50k or 200k: 1024 tiles 894 / 824 (50k, 0.006) to 4926 / 4331 (200k, 0.012), 1296:
//     2745 / 2676 to 3036 / 2655, 1600: 3006 / 3158 to 3563 / 3215, 1764: 3141 / 3659 to 3832 / 3652,
//     2025: 3359 / 3982 to 4269 / 4047
//   30 views, 20k: 2025 tiles 343 / 328, 522 / 493; 8 views, 5k: 124 / 101
//   40, 60 and 75 views of 20k at 2025 tiles (6, 10 and 12 million counters) 434 / 436, 630 / 650, 780 /
//     812; at 1600 tiles 373 / 348, 543 / 522, 668 / 650
//   one view of 500k (key_scan walks 244 blocks in a row): 1024 tiles 133 / 130, 1296: 132 / 135, 2025:
//     146 / 160
// So the lists are direct up to 1600 tiles a view, and up to 2048 while the counters (6 bytes each)
// take less than half of L2 and no view has more than 512 blocks.
constexpr int kDirectTiles = 1600, kDirectTilesSmall = 2048, kDirectViewBlocks = 512;
constexpr int64_t kDirectSmall = 8 << 20;

struct Inst {
  int n, nv, W, H, TW, TH, g_off, v_off;
  int bpv;  // blocks of 256 records per view
  int tp;   // tiles per view rounded up to 8: row pitch of the (block, tile) matrices
  long long item_off, key_off, img_off, blk_off;
  long long mat_off;  // first entry of the instance in the (block, tile) count matrix
};

// Pair keys are (global view << tbits) | tile, tbits the bits of the largest instance's tile
// count.  Pairs are emitted in view order, so the radix sort runs over the tile bits only: the
// sorted lists are grouped by tile, then view, then record, which keeps every (view, tile)
// list contiguous and in record order with fewer, narrower passes than a sort of the full key.
struct Batch {
  int count, T, lT;  // lT = log2 T
  float cut2, eps, znear;
  int tbits;
  Inst in[kMaxInst];
};

// The records of block blk: view v of instance I, Gaussians i0 .. i0 + 255 (below I.n).
struct BlockItems {
  int inst, v, i0;
};
__device__ __forceinline__ BlockItems block_items(const Batch& b, int64_t blk) {
  int k = 0;
  while (k + 1 < b.count && b.in[k + 1].blk_off <= blk) ++k;
  const uint32_t local = (uint32_t)(blk - b.in[k].blk_off), bpv = (uint32_t)b.in[k].bpv;
  const uint32_t v = local / bpv;
  return BlockItems{k, (int)v, (int)(local - v * bpv) * kThreads};
}
__device__ __forceinline__ int inst_of_key(const Batch& b, int64_t key) {
  int k = 0;
  while (k + 1 < b.count && b.in[k + 1].key_off <= key) ++k;
  return k;
}
__device__ __forceinline__ int inst_of_view(const Batch& b, int v) {
  int k = 0;
  while (k + 1 < b.count && b.in[k + 1].v_off <= v) ++k;
  return k;
}
__device__ __forceinline__ int inst_of_gaussian(const Batch& b, int g) {
  int k = 0;
  while (k + 1 < b.count && b.in[k + 1].g_off <= g) ++k;
  return k;
}

struct Layout {
  gs_status* st = nullptr;
  ViewFrame* frames = nullptr;
  // two float4 per record, one 32-byte sector: (px, py, A, e_cut), e_cut = -1/2 log2(e) * Q, and
  // -1/2 log2(e) * (a, 2b, c) with the widened cut: exponent = a'dx^2 + b'dx dy + c'dy^2
  float4* rec = nullptr;
  short4* rect = nullptr;   // clipped inclusive pixel box (x0, y0, x1, y1); x0 > x1 if culled
  uint32_t* tmask = nullptr;  // tight tile rule answers for the box's first 32 tiles
  uint32_t* counts = nullptr;
  uint32_t* block_sums = nullptr;
  uint32_t* block_offs = nullptr;
  uint32_t *keys = nullptr, *vals = nullptr, *keys_alt = nullptr, *vals_alt = nullptr;
  uint2* ranges = nullptr;
  uint32_t* hist = nullptr;
  float4* fpgrad = nullptr;  // 2 float4 per record: moment sums of the backward
  // direct route
  uint16_t* tcount = nullptr;     // records per (block, tile)
  uint32_t* toffset = nullptr;    // the block's offset inside the tile's list
  uint32_t* klocal = nullptr;     // a key's first pair, relative to its group of kScanKeys keys
  unsigned long long* gsum = nullptr;  // pairs of a group, then their exclusive sums
  uint32_t* ticket = nullptr;     // groups done
  long long* vkeys = nullptr;     // first key of every view, and the total (for gs_read_pairs)
  size_t bytes = 0;
};
constexpr int kScanKeys = 64, kScanSegs = 8;  // key_scan: keys and block segments per CTA

struct Plan {
  Batch b;
  int total_n = 0, total_v = 0;
  int64_t items = 0, n_keys = 0, cap = 0, mat = 0;
  int nblocks = 0, key_bits = 0, max_tp = 8;
  bool direct = false;
  SortPlan sort;
};

int make_plan(const gs_instance* inst, int n_inst, const gs_opts* o, int64_t cap, Plan& p) {
  if (!inst || n_inst < 1 || n_inst > kMaxInst || !o || cap < 0) return GS_ERR_ARG;
  if (o->tile != 8 && o->tile != 16 && o->tile != 32) return GS_ERR_ARG;
  if (!(o->cut > 0.f) || !(o->eps >= 0.f) || !(o->znear >= 0.f)) return GS_ERR_ARG;
  Batch& b = p.b;
  memset(&b, 0, sizeof(b));
  b.count = n_inst;
  b.T = o->tile;
  b.lT = o->tile == 8 ? 3 : o->tile == 16 ? 4 : 5;
  b.cut2 = o->cut * o->cut;
  b.eps = o->eps;
  b.znear = o->znear;
  int64_t items = 0, keys = 0, img = 0, gsum = 0, vsum = 0, blocks = 0, mat = 0, max_tiles = 1, max_bpv = 0;
  for (int k = 0; k < n_inst; ++k) {
    const gs_instance& s = inst[k];
    if (s.n < 0 || s.n_views < 1 || s.W < 1 || s.H < 1 || s.W > 32767 || s.H > 32767)
      return GS_ERR_ARG;
    Inst& d = b.in[k];
    d.n = s.n;
    d.nv = s.n_views;
    d.W = s.W;
    d.H = s.H;
    d.TW = (s.W + b.T - 1) / b.T;
    d.TH = (s.H + b.T - 1) / b.T;
    d.g_off = (int)gsum;
    d.v_off = (int)vsum;
    d.item_off = items;
    d.key_off = keys;
    d.img_off = img;
    d.bpv = (s.n + kThreads - 1) / kThreads;
    d.tp = (d.TW * d.TH + 7) / 8 * 8;
    max_bpv = std::max<int64_t>(max_bpv, d.bpv);
    d.blk_off = blocks;
    d.mat_off = mat;
    blocks += (int64_t)s.n_views * d.bpv;
    mat += (int64_t)s.n_views * d.bpv * d.tp;
    items += (int64_t)s.n * s.n_views;
    keys += (int64_t)s.n_views * d.TW * d.TH;
    max_tiles = std::max<int64_t>(max_tiles, (int64_t)d.TW * d.TH);
    img += ((int64_t)s.n_views * s.W * s.H + 63) / 64 * 64;  // blocks start 256-byte aligned
    gsum += s.n;
    vsum += s.n_views;
  }
  b.tbits = bits_for(max_tiles);
  if (items > ((int64_t)1 << 31) - kThreads || blocks > ((int64_t)1 << 31) - 1 || keys > ((int64_t)1 << 31) - 1 ||
      gsum > ((int64_t)1 << 31) - 1 ||
      (vsum << b.tbits) > ((int64_t)1 << 32))  // implied by the key bound (2^tbits < 2 tiles)
    return GS_ERR_ARG;
  p.total_n = (int)gsum;
  p.total_v = (int)vsum;
  p.items = items;
  p.n_keys = keys;
  p.cap = std::min<int64_t>(cap, ((int64_t)1 << 31) - 1);
  p.nblocks = (int)blocks;
  p.max_tp = (int)((max_tiles + 7) / 8 * 8);
  p.direct = max_tiles <= kDirectTiles || (max_tiles <= kDirectTilesSmall && mat <= kDirectSmall &&
                                           max_bpv <= kDirectViewBlocks);
  p.mat = p.direct ? mat : 0;
  p.key_bits = b.tbits;
  p.sort = make_sort_plan(p.key_bits, kTileDigitBits);
  return GS_OK;
}

Layout carve(void* ws, const Plan& p) {
  Carve c(ws);
  Layout L;
  L.st = c.take<gs_status>(1);
  L.frames = c.take<ViewFrame>(p.total_v);
  L.rec = c.take<float4>(2 * p.items);
  L.rect = c.take<short4>(p.items);
  L.tmask = c.take<uint32_t>(p.items);
  L.counts = c.take<uint32_t>(p.items);
  L.block_sums = c.take<uint32_t>(p.nblocks + 1);
  L.block_offs = c.take<uint32_t>(p.nblocks + 1);
  L.ranges = c.take<uint2>(p.n_keys);
  L.hist = c.take<uint32_t>(sort_hist_words(p.sort));
  L.fpgrad = c.take<float4>(2 * p.items);
  if (p.direct) {
    const int64_t groups = (p.n_keys + kScanKeys - 1) / kScanKeys;
    L.tcount = c.take<uint16_t>(p.mat);
    L.toffset = c.take<uint32_t>(p.mat);
    L.klocal = c.take<uint32_t>(p.n_keys);
    L.gsum = c.take<unsigned long long>(groups);
    L.ticket = c.take<uint32_t>(1);
    L.vkeys = c.take<long long>(p.total_v + 1);
    // the lists; 16 bytes per pair as on the other route, so that both hold the same capacity
    L.vals = c.take<uint32_t>(4 * p.cap);
  } else {
    L.keys = c.take<uint32_t>(p.cap);
    L.vals = c.take<uint32_t>(p.cap);
    L.keys_alt = c.take<uint32_t>(p.cap);
    L.vals_alt = c.take<uint32_t>(p.cap);
  }
  L.bytes = align_up(c.off, 256);
  return L;
}

// Every operation of the tile rule is one fixed instruction: preprocess counts the tiles and emit
// places them, so both must get the same answers.  The approximate reciprocals and roots are within
// two ulp; without subnormals, which only footprints beyond 10^15 pixels reach, each is one
// instruction.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// What the closed forms below (tiles of a row, rows of a column slab, columns of a row) need of a
// record's cut ellipse e = a x^2 + b x y + c y^2 > e_cut, so that each keeps every pixel of the box
// that the per-pixel FP32 test accepts.
// D = 4ac - b^2 is a small difference for thin ellipses: Kahan's difference of products gives it
// to two ulp of the stored conic, and every extent comes from D instead of from another difference.
// The per-pixel test itself is off by at most 15 u k |e_cut| inside the box (u = 2^-24, k = 4ac / D;
// at the tips a x^2, b x y / 2 and c y^2 all reach k e_cut), so the cut is widened by 32 u k, twice
// that, and by the 1e-3 that covers the closed forms' own rounding.  From k = 2^21 (an aspect ratio
// of 2900 at 45 degrees) the stored conic no longer fixes the ellipse, and beyond 2^22 pixels FP32
// no longer resolves them: there the whole box counts, by a cut of -infinity.
// (c - b^2 / (4a) and a fixed margin of 1e-3 lost in-cut pixels from aspect ratios of 300 on:
// 0.01 % of them at 1000, 4 % at 5000, sigma 60 pixels.)
__device__ __forceinline__ float conic_det(const float4 c) {
  const float bb = __fmul_rn(c.y, c.y), rest = __fmaf_rn(c.y, c.y, -bb);
  return __fsub_rn(__fmaf_rn(__fmul_rn(4.f, c.x), c.z, -bb), rest);
}
// The widened cut of a record centred at column px; preprocess keeps it in c.w.
__device__ __forceinline__ float wide_cut(float cut, float px, const float4 c) {
  constexpr float kFar = 4194304.f, kThin = 2097152.f;  // 2^22, 2^21
  const float iD = rcp_approx(conic_det(c));
  const float k = __fmaf_rn(__fmul_rn(c.y, c.y), iD, 1.f);
  const float cm = __fmul_rn(cut, __fmaf_rn(k, 1.f / 524288.f, 1.001f));
  const float ext2 = __fmul_rn(__fmul_rn(4.f * fminf(c.x, c.z), cm), iD);  // the longer half extent
  return k >= 1.f && k < kThin && fabsf(px) < kFar && ext2 < kFar * kFar ? cm : -INFINITY;
}

// Tight tile rule: a tile is listed for a record if its cut ellipse, widened as above, meets the
// rectangle of pixel centres the tile shares with the record's clipped box; a tile left out never
// held a contribution.  Per tile row the ellipse's section by the row's slab of pixel centres is
// convex, so the tiles it meets are those whose pixel columns meet its x extent [xa, xb]: the left
// (right) end lies at the ellipse's own leftmost (rightmost) point when that is inside the slab,
// else on the slab's nearer edge.  The ends become pixel columns through the centre's integer and
// fractional parts, where FP32 resolves far more than the margin.
struct Ell {
  float py, fx, ia, hb, kap, vr, cm;  // 1/a, -b/(2a), c - b^2/(4a), v of the rightmost point
  int ix;                             // centre column px = ix + fx
};
__device__ __forceinline__ Ell make_ell(const float4 g, const float4 c) {
  Ell E;
  const float D = conic_det(c);
  const float fl = floorf(g.x);
  E.ix = (int)fl;
  E.fx = __fsub_rn(g.x, fl);
  E.py = g.y;
  E.ia = rcp_approx(c.x);
  const float hb = __fmul_rn(-0.5f, c.y);
  E.hb = __fmul_rn(hb, E.ia);
  E.kap = __fmul_rn(__fmul_rn(0.25f, D), E.ia);
  E.cm = c.w;
  // the rightmost point: u = sqrt(4 c e / D), v = -b / (2c) u
  const float u2 = __fmul_rn(__fmul_rn(__fmul_rn(4.f, c.z), c.w), rcp_approx(D));
  E.vr = __fmul_rn(__fmul_rn(hb, rcp_approx(c.z)), sqrt_approx(fmaxf(u2, 0.f)));
  return E;
}
__device__ __forceinline__ float half_width(const Ell& E, float v) {
  const float d = __fmul_rn(__fmaf_rn(__fmul_rn(-E.kap, v), v, E.cm), E.ia);
  return sqrt_approx(fmaxf(d, 0.f));
}
// Tiles ta .. tb (none if ta > tb) of tile row ty for the clipped box (x0, y0)-(x1, y1).
__device__ __forceinline__ void row_tiles(const Ell& E, int lT, int ty, int x0, int y0, int x1,
                                          int y1, int& ta, int& tb) {
  const float v0 = __fsub_rn((float)max(ty << lT, y0), E.py);
  const float v1 = __fsub_rn((float)min((ty << lT) + (1 << lT) - 1, y1), E.py);
  const float vb = fminf(fmaxf(E.vr, v0), v1), va = fminf(fmaxf(-E.vr, v0), v1);
  const float xb = __fmaf_rn(E.hb, vb, half_width(E, vb));
  const float xa = __fmaf_rn(E.hb, va, -half_width(E, va));
  // first pixel column >= xa and last <= xb, from the centre's integer and fractional column
  const int ca = E.ix + (int)ceilf(__fadd_rn(xa, E.fx)), cb = E.ix + (int)floorf(__fadd_rn(xb, E.fx));
  const bool whole = E.cm == -INFINITY;
  const int fa = whole ? x0 : ca, fb = whole ? x1 : cb;
  // an extent between two neighbouring columns (fa = fb + 1) meets their tile if both are the
  // box's and in one tile; one left or right of the box meets none
  const bool none = fb < x0 || fa > x1;
  ta = none ? 1 : max(fa, x0) >> lT;
  tb = none ? 0 : min(fb, x1) >> lT;
}

// Preprocess keeps the answers for boxes of up to 32 tiles as a bit mask in the box's tile order;
// emit reads the mask, or evaluates the rows again for larger boxes.
constexpr int kMaskTiles = 32;
// Calls f(ty, ta, tb) for every tile row of a record's box with listed tiles ta .. tb.
template <typename F>
__device__ __forceinline__ void listed_rows(const short4 r, uint32_t tm, const float4* rec,
                                            size_t idx, int lT, F f) {
  const int tx0 = r.x >> lT, ty0 = r.y >> lT;
  const int ntx = (r.z >> lT) - tx0 + 1, nty = (r.w >> lT) - ty0 + 1;
  if (ntx * nty <= kMaskTiles) {
    const uint32_t row = 0xffffffffu >> (32 - ntx);
    for (int k = 0, sh = 0; k < nty; ++k, sh += ntx) {
      const uint32_t bits = (tm >> sh) & row;
      if (bits) {
        const int ta = tx0 + __ffs(bits) - 1;
        f(ty0 + k, ta, ta + __popc(bits) - 1);
      }
    }
  } else {
    const Ell E = make_ell(rec[2 * idx], rec[2 * idx + 1]);
    for (int ty = ty0; ty < ty0 + nty; ++ty) {
      int ta, tb;
      row_tiles(E, lT, ty, r.x, r.y, r.z, r.w, ta, tb);
      if (ta <= tb) f(ty, ta, tb);
    }
  }
}

// ------------------------------------------------------------------------------------------
// preprocess
// ------------------------------------------------------------------------------------------
template <bool DIRECT>
__global__ void __launch_bounds__(kThreads)
    k_preprocess(const __grid_constant__ Batch b, const float4* __restrict__ mean_rho,
                 const float4* __restrict__ scale, const float4* __restrict__ quat,
                 const gs_view* __restrict__ views, ViewFrame* __restrict__ frames,
                 float4* __restrict__ rec, short4* __restrict__ rect,
                 uint32_t* __restrict__ tmask, uint32_t* __restrict__ counts,
                 uint32_t* __restrict__ block_sums, uint16_t* __restrict__ tcount,
                 uint32_t* __restrict__ ticket, gs_status* st) {
  extern __shared__ __align__(16) uint32_t s_tiles[];  // DIRECT: records of the block per tile
  __shared__ uint32_t warp_sums[kThreads / 32];
  __shared__ ViewFrame f;
  const BlockItems bi = block_items(b, blockIdx.x);
  const Inst& I = b.in[bi.inst];
  const int i = bi.i0 + threadIdx.x;
  const bool in = i < I.n;
  const int gi = I.g_off + (in ? i : I.n - 1);
  // the parameters are requested before the view's frame is built, which takes one thread a
  // chain of divisions
  const float4 mr = mean_rho[gi], sc = scale[gi], qt = quat[gi];
  if (DIRECT)
    for (int t = threadIdx.x; t < I.tp / 4; t += kThreads)
      reinterpret_cast<uint4*>(s_tiles)[t] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x == 0) {
    ViewFrame fr;
    make_frame(views[I.v_off + bi.v], I.W, I.H, fr);
    f = fr;
    if (bi.i0 == 0) frames[I.v_off + bi.v] = fr;
    if (blockIdx.x == 0) {
      st->code = GS_OK;
      st->pairs = 0;
      if (DIRECT) *ticket = 0u;
    }
  }
  __syncthreads();
  uint32_t cnt = 0;
  if (in) {
    const size_t idx = (size_t)(I.item_off + (int64_t)bi.v * I.n + i);
    Fwd o;
    int x0, y0, x1, y1;
    const bool live = footprint(mr, sc, qt, f, I.W, I.H, b.cut2, b.eps, b.znear, o, x0, y0, x1, y1);
    if (live) {
      const float k = gsd::kNegHalfLog2e;
      const float4 gg = make_float4(o.px, o.py, o.A, k * o.Q);
      float4 cc = make_float4(k * o.ca, 2.f * k * o.cb, k * o.cc, 0.f);
      cc.w = wide_cut(gg.w, o.px, cc);
      const Ell E = make_ell(gg, cc);
      const int lT = b.lT, tx0 = x0 >> lT, ty0 = y0 >> lT;
      const int ntx = (x1 >> lT) - tx0 + 1, ty1 = y1 >> lT;
      uint32_t tm = 0u;
      int sh = 0;
      for (int ty = ty0; ty <= ty1; ++ty, sh += ntx) {
        int ta, tb;
        row_tiles(E, lT, ty, x0, y0, x1, y1, ta, tb);
        if (ta > tb) continue;
        cnt += (uint32_t)(tb - ta + 1);
        if (sh + ntx <= kMaskTiles) tm |= (0xffffffffu >> (31 - (tb - ta))) << (sh + ta - tx0);
        if (DIRECT)
          for (int t = ty * I.TW + ta; t <= ty * I.TW + tb; ++t) atomicAdd(&s_tiles[t], 1u);
      }
      tmask[idx] = tm;
      rec[2 * idx] = gg;
      rec[2 * idx + 1] = cc;
      rect[idx] = make_short4((short)x0, (short)y0, (short)x1, (short)y1);
    } else {
      rec[2 * idx] = rec[2 * idx + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
      rect[idx] = make_short4(1, 1, 0, 0);
    }
    counts[idx] = cnt;
  }
  if constexpr (DIRECT) {
    __syncthreads();
    // the row in 16-byte vectors (entries past the last tile are zero)
    uint4* row = reinterpret_cast<uint4*>(tcount + I.mat_off +
                                          ((int64_t)bi.v * I.bpv + bi.i0 / kThreads) * I.tp);
    for (int t = threadIdx.x; t < I.tp / 8; t += kThreads) {
      const uint4 x = reinterpret_cast<const uint4*>(s_tiles)[2 * t];
      const uint4 y = reinterpret_cast<const uint4*>(s_tiles)[2 * t + 1];
      row[t] = make_uint4(x.x | x.y << 16, x.z | x.w << 16, y.x | y.y << 16, y.z | y.w << 16);
    }
  } else {
    // culled pairs drop out of the warp's count via the ballot; the block sum feeds the scan
    const unsigned live_mask = __ballot_sync(0xffffffffu, cnt > 0);
    uint32_t s = live_mask ? gsd::warp_sum(cnt) : 0u;
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t bs = 0;
#pragma unroll
      for (int w = 0; w < kThreads / 32; ++w) bs += warp_sums[w];
      block_sums[blockIdx.x] = bs;
    }
  }
}

// ------------------------------------------------------------------------------------------
// direct route: counts per (block, tile) -> offsets -> lists
// ------------------------------------------------------------------------------------------
// A CTA owns kScanKeys consecutive keys, a thread one key and an eighth of its view's blocks: the
// column of counts is summed, then walked again to write each block's offset in the list (the
// second read hits L2).  ranges[key] gets (offset in the group, count), completed by emit.  The
// last CTA to finish turns the groups' sums into offsets and records the pair total and whether
// it fits.  Bound by memory: 2 + 2 + 4 bytes per (block, tile).
__global__ void __launch_bounds__(kScanKeys * kScanSegs, 4)
    k_key_scan(const __grid_constant__ Batch b, int64_t n_keys, const uint16_t* tcount,
               uint32_t* __restrict__ toffset, uint32_t* __restrict__ klocal,
               uint2* __restrict__ ranges, unsigned long long* __restrict__ gsum, uint32_t* ticket,
               long long* __restrict__ vkeys, int total_v, gs_status* st, int64_t cap,
               int64_t vals_off, int64_t ranges_off, int64_t vkeys_off) {
  gsd::pdl_begin();
  __shared__ uint32_t part[kScanSegs][kScanKeys];
  __shared__ unsigned long long wtot[kScanKeys * kScanSegs / 32];
  __shared__ bool last;
  const int t = threadIdx.x, lane = t & 31, kl = t % kScanKeys, seg = t / kScanKeys;
  const int64_t key = (int64_t)blockIdx.x * kScanKeys + kl;
  uint32_t sum = 0;
  int b0 = 0, b1 = 0, tp = 0;
  int64_t at = 0;
  if (key < n_keys) {
    const Inst& I = b.in[inst_of_key(b, key)];
    const int tiles = I.TW * I.TH;
    const int64_t lk = key - I.key_off;
    tp = I.tp;
    const int v = (int)(lk / tiles), tile = (int)(lk - (int64_t)v * tiles);
    const int per = (I.bpv + kScanSegs - 1) / kScanSegs;
    b0 = min(I.bpv, seg * per);
    b1 = min(I.bpv, b0 + per);
    at = I.mat_off + (int64_t)v * I.bpv * tp + tile;
    if (seg == 0 && tile == 0) vkeys[I.v_off + v] = key;
#pragma unroll 8
    for (int k = b0; k < b1; ++k) sum += tcount[at + (int64_t)k * tp];
  }
  if (blockIdx.x == 0 && t == 0) vkeys[total_v] = n_keys;
  part[seg][kl] = sum;
  __syncthreads();
  uint32_t run = 0, total = 0;
#pragma unroll
  for (int q = 0; q < kScanSegs; ++q) {
    const uint32_t x = part[q][kl];
    run += q < seg ? x : 0u;
    total += x;
  }
  const uint16_t* q = tcount + at + (int64_t)b0 * tp;
  uint32_t* o = toffset + at + (int64_t)b0 * tp;
  int left = b1 - b0;
  for (; left >= 8; left -= 8, q += 8 * tp, o += 8 * tp) {  // eight loads ahead of the stores
    uint32_t x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = q[j * tp];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      o[j * tp] = run;
      run += x[j];
    }
  }
  for (; left > 0; --left, q += tp, o += tp) {
    *o = run;
    run += *q;
  }
  if (seg == 0) {  // the first two warps hold the group's keys
    // (in 64 bits: 2^27 records that each cover 32 neighbouring tiles pass 2^32; where a 32-bit
    // place would wrap, the pair total is above any capacity and nothing is placed)
    unsigned long long incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) wtot[t >> 5] = incl;
    asm volatile("bar.sync 1, %0;" ::"n"(kScanKeys) : "memory");
    const uint32_t first = (uint32_t)(incl - total + (t >= 32 ? wtot[0] : 0ull));
    if (key < n_keys) {
      klocal[key] = first;
      ranges[key] = make_uint2(first, total);
    }
    if (t == 0) {
      unsigned long long g = 0;
      for (int w = 0; w < kScanKeys / 32; ++w) g += wtot[w];
      gsum[blockIdx.x] = g;
      __threadfence();
      last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // exclusive sums over the groups
  constexpr int NT = kScanKeys * kScanSegs;
  const int ng = (int)gridDim.x;
  unsigned long long base = 0;
  for (int g0 = 0; g0 < ng; g0 += NT) {
    const int g = g0 + t;
    const unsigned long long x = g < ng ? __ldcg(gsum + g) : 0ull;
    unsigned long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) wtot[t >> 5] = incl;
    __syncthreads();
    unsigned long long before = base, all = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
      before += w < (t >> 5) ? wtot[w] : 0ull;
      all += wtot[w];
    }
    if (g < ng) gsum[g] = before + incl - x;
    base += all;
    __syncthreads();
  }
  if (t == 0) {
    st->pairs = (int64_t)base;
    st->capacity = cap;
    if ((int64_t)base > cap) st->code = GS_ERR_CAPACITY;
    st->reserved[0] = -1;  // the keys are not stored: gs_read_pairs takes them from the ranges
    st->reserved[1] = vals_off;
    st->reserved[2] = n_keys;
    st->reserved[3] = ranges_off;
    st->reserved[4] = vkeys_off;
    st->reserved[5] = total_v;
    st->reserved[6] = b.tbits;
  }
}

// Writes every record to its place in the lists of its tiles.  A block's records keep their order
// inside a list: a record's place is the list's start, plus the block's offset in it, plus the
// records of the same tile in earlier warps and lanes of the block (a lane mask per (warp, tile)
// in shared memory; its set bits give the counts).  Blocks of one view run together, so the scattered 4-byte
// stores of a list's neighbourhood meet in L2.
__global__ void __launch_bounds__(kThreads)
    k_emit_direct(const __grid_constant__ Batch b, const uint32_t* __restrict__ counts,
                  const float4* __restrict__ rec,
                  const short4* __restrict__ rect, const uint32_t* __restrict__ tmask,
                  const uint32_t* __restrict__ toffset, const uint32_t* __restrict__ klocal,
                  const unsigned long long* __restrict__ gsum, uint2* __restrict__ ranges,
                  uint32_t* __restrict__ vals, const gs_status* st) {
  constexpr int NW = kThreads / 32;
  extern __shared__ __align__(16) uint32_t s_emit[];
  static_assert(NW == 8, "eight bytes of warp counts per tile");
  const BlockItems bi = block_items(b, blockIdx.x);
  const Inst& I = b.in[bi.inst];
  const int tiles = I.TW * I.TH, t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int i = bi.i0 + t;
  const size_t idx = (size_t)(I.item_off + (int64_t)bi.v * I.n + i);
  const uint32_t cnt = i < I.n ? counts[idx] : 0u;
  const short4 r = i < I.n ? rect[idx] : make_short4(0, 0, 0, 0);
  const uint32_t tm = i < I.n ? tmask[idx] : 0u;
  if (st->code != GS_OK) return;
  // [NW][tp] lane masks, [tp] first place of the block in the tile's list, [tp] eight bytes: records
  // of the tile in the warps before each
  const int tp = I.tp;
  uint32_t* lanes = s_emit;
  uint32_t* first = lanes + NW * tp;
  uint2* before = reinterpret_cast<uint2*>(first + tp);
  for (int k = t; k < NW * tp / 4; k += kThreads)
    reinterpret_cast<uint4*>(lanes)[k] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  const uint32_t bit = 1u << lane;
  uint32_t* mine = lanes + w * tp;
  if (cnt)
    listed_rows(r, tm, rec, idx, b.lT, [&](int ty, int ta, int tb) {
      uint32_t* q = mine + ty * I.TW;
      for (int k = ta; k <= tb; ++k) atomicOr(q + k, bit);
    });
  const int64_t key0 = I.key_off + (int64_t)bi.v * tiles;
  const uint32_t* row = toffset + I.mat_off + ((int64_t)bi.v * I.bpv + bi.i0 / kThreads) * tp;
  __syncthreads();
  for (int k = t; k < tiles; k += kThreads) {
    const uint32_t start = (uint32_t)gsum[(key0 + k) / kScanKeys] + klocal[key0 + k];
    first[k] = start + row[k];
    if (bi.i0 == 0) ranges[key0 + k] = make_uint2(start, start + ranges[key0 + k].y);
    uint32_t run = 0, lo = 0, hi = 0;  // at most 7 x 32 before the last warp: a byte
#pragma unroll
    for (int ww = 0; ww < 4; ++ww) {
      lo |= run << (8 * ww);
      run += __popc(lanes[ww * tp + k]);
    }
#pragma unroll
    for (int ww = 0; ww < 4; ++ww) {
      hi |= run << (8 * ww);
      run += __popc(lanes[(ww + 4) * tp + k]);
    }
    before[k] = make_uint2(lo, hi);
  }
  __syncthreads();
  const uint8_t* pre = reinterpret_cast<const uint8_t*>(before) + w;
  if (cnt)
    listed_rows(r, tm, rec, idx, b.lT, [&](int ty, int ta, int tb) {
      for (int k = ty * I.TW + ta; k <= ty * I.TW + tb; ++k)
        vals[first[k] + pre[8 * k] + __popc(mine[k] & (bit - 1u))] = (uint32_t)idx;
    });
}

// ------------------------------------------------------------------------------------------
// sorted route: emit in record order (same block decomposition as preprocess; in-block exclusive
// prefix by warp scans)
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads)
    k_emit(const __grid_constant__ Batch b, const uint32_t* __restrict__ counts,
           const float4* __restrict__ rec,
           const short4* __restrict__ rect, const uint32_t* __restrict__ tmask,
           const uint32_t* __restrict__ block_offs,
           uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
           gs_status* st, int64_t sorted_keys_off, int64_t sorted_vals_off) {
  __shared__ uint32_t warp_pre[kThreads / 32];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->reserved[0] = sorted_keys_off;
    st->reserved[1] = sorted_vals_off;
    st->reserved[2] = b.in[b.count - 1].key_off +
                      (int64_t)b.in[b.count - 1].nv * b.in[b.count - 1].TW * b.in[b.count - 1].TH;
  }
  const BlockItems bi = block_items(b, blockIdx.x);
  const Inst& I = b.in[bi.inst];
  const int i = bi.i0 + threadIdx.x;
  const size_t idx = (size_t)(I.item_off + (int64_t)bi.v * I.n + i);
  // every input of the thread is requested up front, with the status word, so that the
  // emission waits for one round trip instead of a chain of them
  const bool in = i < I.n;
  const uint32_t cnt = in ? counts[idx] : 0u;
  const short4 r = in ? rect[idx] : make_short4(0, 0, 0, 0);
  const uint32_t tm = in ? tmask[idx] : 0u;
  const uint32_t boff = block_offs[blockIdx.x];
  if (st->code != GS_OK) return;
  const uint32_t incl = gsd::warp_inclusive_scan(cnt);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 31) warp_pre[w] = incl;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t a = 0;
#pragma unroll
    for (int k = 0; k < kThreads / 32; ++k) {
      uint32_t x = warp_pre[k];
      warp_pre[k] = a;
      a += x;
    }
  }
  __syncthreads();
  const uint32_t wbase = boff + warp_pre[w];  // the warp's first pair
  const uint32_t wtotal = __shfl_sync(0xffffffffu, incl, 31);
  if (wtotal == 0) return;
  // this lane's record (meaningful where cnt > 0)
  const int lT = b.lT, TW = I.TW;
  const uint32_t kbase = (uint32_t)(I.v_off + bi.v) << b.tbits;
  const int tx0i = r.x >> lT, ty0i = r.y >> lT, ntx = (r.z >> lT) - tx0i + 1;
  const bool small = ntx * ((r.w >> lT) - ty0i + 1) <= kMaskTiles;
  // records with at most 32 box tiles: the warp writes its contiguous range of pairs
  // cooperatively, pair p going to lane p % 32, which finds the owning record by a binary
  // search over the lanes' inclusive counts and the tile as the owner's k-th listed tile
  const uint32_t excl = incl - cnt;
  for (uint32_t p0 = 0; p0 < wtotal; p0 += 32) {
    const uint32_t p = p0 + lane;
    int o = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const uint32_t ci = __shfl_sync(0xffffffffu, incl, o + step - 1);
      if (ci <= p) o += step;
    }
    const uint32_t oe = __shfl_sync(0xffffffffu, excl, o);
    const uint32_t otm = __shfl_sync(0xffffffffu, tm, o);
    const int ontx = __shfl_sync(0xffffffffu, ntx, o);
    const int otx0 = __shfl_sync(0xffffffffu, tx0i, o);
    const int oty0 = __shfl_sync(0xffffffffu, ty0i, o);
    const bool osmall = __shfl_sync(0xffffffffu, small ? 1 : 0, o) != 0;
    if (p < wtotal && osmall) {
      const int bit = (int)__fns(otm, 0, (int)(p - oe) + 1);
      const int ty = oty0 + bit / ontx, tx = otx0 + bit % ontx;
      keys[wbase + p] = kbase + (uint32_t)(ty * TW + tx);
      vals[wbase + p] = (uint32_t)(idx - lane + o);
    }
  }
  if (cnt == 0 || small) return;
  uint32_t off = wbase + excl;
  listed_rows(r, tm, rec, idx, lT, [&](int ty, int ta, int tb) {
    for (int tx = ta; tx <= tb; ++tx, ++off) {
      keys[off] = kbase + (uint32_t)(ty * TW + tx);
      vals[off] = (uint32_t)idx;
    }
  });
}

// [start, end) of every (view, tile) list.  The sorted keys are grouped by tile and then view,
// so each key's pairs are contiguous (though keys are not ascending); a boundary's key maps to
// its (instance, view, tile) slot.  Four keys per thread through one 16-byte load.
__device__ __forceinline__ uint32_t range_slot(const Batch& b, uint32_t key) {
  const int gv = (int)(key >> b.tbits);
  const Inst& I = b.in[inst_of_view(b, gv)];
  return (uint32_t)(I.key_off + (int64_t)(gv - I.v_off) * I.TW * I.TH +
                    (key & ((1u << b.tbits) - 1u)));
}
__global__ void __launch_bounds__(kThreads)
    k_tile_ranges(const __grid_constant__ Batch b, const uint32_t* __restrict__ keys,
                  uint2* __restrict__ ranges, const gs_status* st) {
  if (st->code != GS_OK) return;
  const int64_t n = st->pairs;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; 4 * q < n; q += stride) {
    const int64_t i0 = 4 * q;
    uint32_t k[4];
    if (i0 + 4 <= n) {
      const uint4 v = *reinterpret_cast<const uint4*>(keys + i0);
      k[0] = v.x, k[1] = v.y, k[2] = v.z, k[3] = v.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) k[j] = i0 + j < n ? keys[i0 + j] : 0u;
    }
    const uint32_t prev = i0 > 0 ? keys[i0 - 1] : 0u;
    const uint32_t next = i0 + 4 < n ? keys[i0 + 4] : 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t i = i0 + j;
      if (i < n) {
        const bool first = i == 0 || (j == 0 ? prev : k[j - 1]) != k[j];
        const bool last = i == n - 1 || (j == 3 ? next : k[j + 1]) != k[j];
        if (first) ranges[range_slot(b, k[j])].x = (uint32_t)i;
        if (last) ranges[range_slot(b, k[j])].y = (uint32_t)(i + 1);
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// raster forward (and the in-cut evaluation counter)
// ------------------------------------------------------------------------------------------
// Exponent of a footprint record at pixel offset (dx, dy), base 2 and pre-scaled by
// -1/2 log2(e): e = a' dx^2 + b' dx dy + c' dy^2, evaluated as ((a' dx + b' dy) dx + c' dy^2)
// with the row terms b' dy and c' dy^2 shared by every pixel of a row: per pixel
// fma(fma(a', dx, b' dy), dx, c' dy^2), two pixels at a time in packed FP32x2 (each component
// rounds like the scalar fmaf).  The forward, the evaluation counter and the backward all
// decide the cut e > e_cut with this exact sequence.
__device__ __forceinline__ float row_b(const float4 c, float dy) { return c.y * dy; }
__device__ __forceinline__ float row_c(const float4 c, float dy) { return (c.z * dy) * dy; }

// Rows [ylo, yhi] (tile-local, not clamped to it; ylo > yhi if none) that a record's widened cut
// ellipse reaches inside the column slab of pixel centres [x0, x1].  The ellipse's
// section by the slab is convex, so its rows form an interval: its top (bottom) is the ellipse's own
// top (bottom) point when that lies in the slab, else the boundary at the slab's nearer edge (the
// upper boundary is concave).  Widened by 1/100 pixel and 16 u of the ellipse's half height, for the
// rounding of rows far from the centre: a superset of the rows the per-pixel test accepts.
struct SlabExt {
  float D, c4, inv2c;   // 4ac - b^2, 4 c e (> 0), 1 / (2c) (< 0)
  float dxt;            // the ellipse's top point left or right of its centre
  float ylo, yhi;       // the centre's row in the tile, less and plus the rows' margin
};
__device__ __forceinline__ SlabExt make_slab(const float4 g, const float4 c, int ty0) {
  SlabExt X;
  X.D = conic_det(c);
  // the top point: its height is sqrt(a t), its column -b / (2a) times that
  const float t = 4.f * c.w * rcp_approx(X.D), at = c.x * t, r = rsqrt_approx(at);
  X.dxt = -0.5f * c.y * t * r;
  X.c4 = 4.f * c.z * c.w;
  X.inv2c = 0.5f * rcp_approx(c.z);
  const float my = c.w == -INFINITY ? 1e9f : fmaf(at * r, 1.f / 1048576.f, 0.01f);
  const float gy = g.y - (float)ty0;
  X.ylo = gy - my;
  X.yhi = gy + my;
  return X;
}
__device__ __forceinline__ void slab_rows(const float4 g, const float4 c, const SlabExt& X,
                                          float x0, float x1, int& ylo, int& yhi) {
  const float u0 = x0 - g.x, u1 = x1 - g.x;
  const float xu = fminf(fmaxf(X.dxt, u0), u1), xl = fminf(fmaxf(-X.dxt, u0), u1);
  const float Du = fmaxf(fmaf(-X.D * xu, xu, X.c4), 0.f);  // (b x)^2 - 4 c (a x^2 - e)
  const float Dl = fmaxf(fmaf(-X.D * xl, xl, X.c4), 0.f);
  ylo = (int)ceilf(fmaf(-c.y * xl + sqrt_approx(Dl), X.inv2c, X.ylo));
  yhi = (int)floorf(fmaf(-c.y * xu - sqrt_approx(Du), X.inv2c, X.yhi));
}

// Bit mask of the (4-row x BW-column) blocks of a (T x T) tile at (tx0, ty0) that a record's cut
// ellipse reaches, bit column * NBY + band: per column slab of its box the reached rows
// (slab_rows) make a run of bands.
template <int T, int BW>
__device__ __forceinline__ uint32_t block_mask(const float4 g, const float4 c, const short4 bx,
                                               int tx0, int ty0) {
  constexpr int LBW = BW == 16 ? 4 : 3, NBX = T / BW, NBY = T / 4;
  const SlabExt X = make_slab(g, c, ty0);
  const int bx0 = (bx.x - tx0) >> LBW, bx1 = (bx.z - tx0) >> LBW;
  const int ry0 = max(0, bx.y - ty0), ry1 = min(T - 1, bx.w - ty0);
  uint32_t mask = 0u;
#pragma unroll
  for (int k = 0; k < NBX; ++k) {
    const float x0 = (float)(tx0 + k * BW);
    int ylo, yhi;
    slab_rows(g, c, X, x0, x0 + (float)(BW - 1), ylo, yhi);
    ylo = max(ylo, ry0);
    yhi = min(yhi, ry1);
    if (k >= bx0 && k <= bx1 && ylo <= yhi)
      mask |= ((2u << (yhi >> 2)) - (1u << (ylo >> 2))) << (k * NBY);
  }
  return mask;
}

// Raster forward (and the in-cut evaluation counter) with records on lanes, LPB lanes per
// 4 x BW block of the (view, tile), 32 / LPB vertically adjacent blocks per warp.  Per batch of
// staged records each warp lists the records whose cut ellipse reaches each of its blocks (block
// masks); the LPB lanes of a block take its records one per lane, and every
// lane walks the block's pixels in the same unrolled order (pixel pairs in packed FP32x2
// arithmetic, the exponent and the cut exactly as the backward computes them) and adds A 2^e to
// its own accumulator of each pixel.  The accumulators live through all batches; at the end one
// butterfly reduce-scatter over the block's lanes sums them per pixel, lane l keeping NPR / LPB
// consecutive pairs.  A pixel's sum is thus taken in a fixed order: per lane in list order, then
// over the lanes.
// Bound by issue and latency (64 accumulators leave 16 warps per SM).  Fewer lanes per block make
// the reduction cheaper per pixel (with 32 lanes it is 12 % of the instructions at 75 x 512^2) and
// the tile's CTA smaller, so that more CTAs load and walk independently on an SM; but a warp
// walks as long as the longest of its blocks' lists.  75 x 1024^2, tile 32: 32 lanes 6.48 ms (one
// CTA of 16 warps per SM, idle while it loads), 16 lanes 5.14, 8 lanes 4.49, 4 lanes 4.70, with
// 4 records staged per thread and batch (3: 4.58, 6: 4.82; the rest of the SM's memory caches the
// gathers).  30 x 512^2, tile 8: 32 lanes 0.57, 16 lanes 0.48 ms.  Tiles of 16 keep 32 lanes: 16
// would take 1.00 -> 0.88 ms at 75 x 512^2, but in another order of the sums, and the L1 term of
// a reconstruction step turns last-bit differences into flipped signs of its gradient.
// Staging (two dependent gathers per record and its block mask) is about 30 % of the kernel:
// records as one 32-byte sector, two gathers in flight per thread, approximate roots in the mask and
// its bands set as runs of bits took tile 16 from 1.00 to 0.93 ms and tile 32 from 4.49 to 4.11.
template <int T>
struct FwdBlocks {
  static constexpr int BW = T >= 16 ? 16 : 8;  // block width; 4 rows
  static constexpr int NBX = T / BW, NBY = T / 4, NB = NBX * NBY;
  static constexpr int LPB = T == 32 ? 8 : T == 16 ? 32 : 16;  // lanes per block
  static constexpr int BPW = 32 / LPB;             // blocks per warp, one above the other
  static constexpr int NW = NB / BPW;
  static constexpr int NT = 32 * NW;
  static constexpr int SB = (T == 8 ? 8 : 4) * NT;  // records staged per batch
};

template <int T, bool COUNT>
__global__ void __launch_bounds__(FwdBlocks<T>::NT, 512 / FwdBlocks<T>::NT)
    k_raster_fwd(const __grid_constant__ Batch b, const uint2* __restrict__ ranges,
                 const uint32_t* __restrict__ vals, const float4* __restrict__ recs,
                 const short4* __restrict__ rect,
                 float* __restrict__ img, gs_status* st) {
  using S = FwdBlocks<T>;
  constexpr int BW = S::BW, HP = BW / 2;  // pixel pairs per row
  __shared__ float4 s_geo[S::SB];
  __shared__ float4 s_con[S::SB];
  __shared__ uint32_t s_mask[S::SB];
  __shared__ uint16_t s_list[S::NB][S::SB];
  __shared__ unsigned long long s_cnt;
  const int64_t key = blockIdx.x;
  const uint2 r = ranges[key];  // requested together with the status word, not after it
  if (st->code != GS_OK) return;
  const Inst& I = b.in[inst_of_key(b, key)];
  const int64_t lk = key - I.key_off;
  const int v = (int)(lk / (I.TW * I.TH)), tile = (int)(lk - (int64_t)v * I.TW * I.TH);
  const int W = I.W, H = I.H;
  const int tx0 = (tile % I.TW) * T, ty0 = (tile / I.TW) * T;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  constexpr int LPB = S::LPB, BPW = S::BPW;
  const int part = lane / LPB, lp = lane % LPB;
  const int bit0 = (w % S::NBX) * S::NBY + (w / S::NBX) * BPW;  // the warp's blocks: bits bit0 ..
  const int bxl = (w % S::NBX) * BW, byl = ((w / S::NBX) * BPW + part) * 4;
  const float fx0 = (float)(tx0 + bxl), fy0 = (float)(ty0 + byl);
  const unsigned lt = gsd::lanemask_lt();
  constexpr int NPR = 4 * HP;  // float2 accumulators per lane: pair ry * HP + p
  float2 acc[NPR];
#pragma unroll
  for (int i = 0; i < NPR; ++i) acc[i] = make_float2(0.f, 0.f);
  uint32_t cnt_eval = 0;
  if (COUNT && t == 0) s_cnt = 0ull;
  for (uint32_t base = r.x; base < r.y; base += S::SB) {
    const int m = (int)min((uint32_t)S::SB, r.y - base);
    __syncthreads();
    // two records per thread at a time, so that their gathers overlap
    for (int q = t; q < m; q += 2 * S::NT) {
      const bool two = q + S::NT < m;
      const uint32_t rec0 = vals[base + q], rec1 = two ? vals[base + q + S::NT] : rec0;
      const float4 g0 = recs[2 * (size_t)rec0], c0 = recs[2 * (size_t)rec0 + 1];
      const float4 g1 = recs[2 * (size_t)rec1], c1 = recs[2 * (size_t)rec1 + 1];
      const short4 b0 = rect[rec0], b1 = rect[rec1];
      s_geo[q] = g0;
      s_con[q] = c0;
      s_mask[q] = block_mask<T, BW>(g0, c0, b0, tx0, ty0);
      if (two) {
        s_geo[q + S::NT] = g1;
        s_con[q + S::NT] = c1;
        s_mask[q + S::NT] = block_mask<T, BW>(g1, c1, b1, tx0, ty0);
      }
    }
    __syncthreads();
    int cnts[BPW];
#pragma unroll
    for (int k = 0; k < BPW; ++k) cnts[k] = 0;
    for (int j0 = 0; j0 < m; j0 += 32) {
      const int jl = j0 + lane;
      const uint32_t mk = jl < m ? s_mask[jl] >> bit0 : 0u;
#pragma unroll
      for (int k = 0; k < BPW; ++k) {
        const bool hit = (mk >> k) & 1u;
        const unsigned bits = __ballot_sync(0xffffffffu, hit);
        if (hit) s_list[BPW * w + k][cnts[k] + __popc(bits & lt)] = (uint16_t)jl;
        cnts[k] += __popc(bits);
      }
    }
    __syncwarp();
    const uint16_t* list = s_list[BPW * w + part];
    int cnt = 0, most = 0;
#pragma unroll
    for (int k = 0; k < BPW; ++k) {
      cnt = part == k ? cnts[k] : cnt;
      most = max(most, cnts[k]);
    }
    for (int c0 = 0; c0 < most; c0 += LPB) {
      const int li = c0 + lp;
      const bool active = li < cnt;
      const int j = active ? list[li] : 0;
      const float4 g = s_geo[j];
      const float4 c = s_con[j];
      const float cut = active ? g.w : INFINITY;  // an idle lane never passes
      float2 dx[HP];
#pragma unroll
      for (int p = 0; p < HP; ++p)
        dx[p] = make_float2(fx0 + (float)(2 * p) - g.x, fx0 + (float)(2 * p + 1) - g.x);
      const float2 ca = make_float2(c.x, c.x);
#pragma unroll
      for (int ry = 0; ry < 4; ++ry) {
        const float dy = (fy0 + (float)ry) - g.y;
        const float B = row_b(c, dy), cdy2 = row_c(c, dy);
        const float2 B2 = make_float2(B, B), C2 = make_float2(cdy2, cdy2);
#pragma unroll
        for (int p = 0; p < HP; ++p) {
          const float2 e = __ffma2_rn(__ffma2_rn(ca, dx[p], B2), dx[p], C2);
          if (COUNT) {
            const int x = tx0 + bxl + 2 * p, y = ty0 + byl + ry;
            cnt_eval += (e.x > cut && x < W && y < H) ? 1u : 0u;
            cnt_eval += (e.y > cut && x + 1 < W && y < H) ? 1u : 0u;
          } else {
            // the cut as a predicate on the accumulating FMA (no select): each component rounds
            // like the packed FMA with a zero value would leave it, so sums are unchanged
            const float vx = ex2(e.x), vy = ex2(e.y);
            if (e.x > cut) acc[ry * HP + p].x = fmaf(g.z, vx, acc[ry * HP + p].x);
            if (e.y > cut) acc[ry * HP + p].y = fmaf(g.z, vy, acc[ry * HP + p].y);
          }
        }
      }
    }
    __syncwarp();
  }
  if constexpr (COUNT) {
    __syncthreads();
    const uint32_t ws = gsd::warp_sum(cnt_eval);
    if (lane == 0 && ws) atomicAdd(&s_cnt, (unsigned long long)ws);
    __syncthreads();
    if (t == 0 && s_cnt) atomicAdd((unsigned long long*)&st->evals, s_cnt);
  } else {
    // butterfly reduce-scatter of the block's 4 x BW pixel sums over its LPB lanes: at each stage a
    // lane keeps the half of its pairs on its side of the partner bit and adds the partner's copy of
    // that half; after log2 LPB stages lane l of them holds the sums of pairs l NPR / LPB and up
    constexpr int KEEP = NPR / LPB;
#pragma unroll
    for (int bit = LPB / 2, n = NPR / 2; bit >= 1; bit >>= 1, n >>= 1) {
      const bool up = (lane & bit) != 0;
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const float2 mine = up ? acc[i + n] : acc[i];
        const float2 send = up ? acc[i] : acc[i + n];
        float2 recv;
        recv.x = __shfl_xor_sync(0xffffffffu, send.x, bit);
        recv.y = __shfl_xor_sync(0xffffffffu, send.y, bit);
        acc[i] = __fadd2_rn(mine, recv);
      }
    }
    const int pi = lp * KEEP;  // first pair: row pi / HP, columns 2 (pi % HP) and up
    const int y = ty0 + byl + pi / HP, x = tx0 + bxl + 2 * (pi % HP);
    if (y >= H) return;
    float* row = img + I.img_off + ((int64_t)v * H + y) * W;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
      if (x + 2 * k < W) row[x + 2 * k] = acc[k].x;
      if (x + 2 * k + 1 < W) row[x + 2 * k + 1] = acc[k].y;
    }
  }
}

// ------------------------------------------------------------------------------------------
// raster backward, per Gaussian (Sec. 3.5), with records on lanes: one warp per (view, tile), or
// per part of its list.  A lane holds one record at a time, walks the 4 x 8 blocks of the tile that
// the record's cut ellipse reaches (closed-form test of the ellipse against the block's columns, a
// superset of the per-pixel test), one block per round, keeps the six moments of g exp(-q/2) in
// registers over all of them, adds them to the record's moments with two float4 atomics and takes
// the next record from a queue that the warp refills 32 records at a time.  So every lane has a
// block in every round but the list's last ones, nothing is summed through shared memory, and no
// warp waits for another.  A round is fully unrolled and the same for all lanes: dL/dI comes from
// shared memory at the lane's own block (blocks lie in different bank groups), the cut is decided
// exactly as in the forward (same offsets, same expression).
// Bound by instruction issue (71 %; FMA pipe 59 % of its cycles): per pixel pair two FMAs for the
// exponent, two ex2, the cut, one product and three moment sums, and as much again per block for the
// record's row coefficients, the centre shift and the queue.  Against warps that own 4 x 16 blocks,
// list their records per batch and meet in shared atomics: tile 16, 75 x 512^2, 1228 -> 1020 us;
// tile 32, 75 x 1024^2, 7.33 -> 5.80 ms; 41 x 389 x 517 parallel, 270 -> 238; 16 small
// reconstructions 391 -> 311.  4 x 16 blocks here: 1172 instead of 1132, 6.38 instead of 6.41 ms at
// the same stage.
// Blocks that start at the record's own box instead of the grid cost their gain in bank conflicts
// (1211).  24, 28, 32 warps per SM: 1051, 1043, 1079 (tile 32: 5.81, 5.88, 6.41 ms).  The last rows
// of the grid take the narrow records (below), which the tiles' warps leave out.
// ------------------------------------------------------------------------------------------
template <int T>
struct BwdBlocks {
  static constexpr int BW = 8;             // block of 4 rows x 8 columns
  static constexpr int NBX = T / BW, NBY = T / 4, NB = NBX * NBY;
  // dL/dI in shared memory, in float4: per block, per pair of mirrored columns (p, 7 - p), the
  // pair's four rows; one more float4 puts the blocks' equal places in different bank groups
  static constexpr int GS = 9;
  static constexpr int CW = T >= 16 ? 16 : 8;  // columns about whose centre narrow records sum
};
constexpr uint32_t kMinPart = 128;  // records of a list's part (64: one view of 1024^2, 20k, 29 instead of 25 us)

// Narrow records: the footprint may have a variance below kNarrowVar square pixels in some direction
// (the trace of the conic bounds its inverse), in a box of at most 32 x 32 pixels.  Moved from a
// block's centre to such a record's, second moments lose the digits that the centres' distance
// squared has over the variance (50 times the rounding at 0.16 and 16-column blocks), so the order
// of their sums shows in the gradients: they keep the one about 16-column runs, row by row (8 at
// tile 8), and one thread takes all pixels of a record.  Gradients then move by at most 5e-6 (2-norm) against
// warps that walk those blocks, instead of up to 2e-5.
template <int T>
__device__ __forceinline__ bool is_narrow(const float4 c, const short4 bx) {
  constexpr float kNarrowVar = T >= 16 ? 0.16f : 0.04f;
  return -(c.x + c.z) * kNarrowVar > 0.72134752f /* log2(e) / 2 */ &&
         bx.z - bx.x < 32 && bx.w - bx.y < 32;
}

// The moments of a narrow record, one thread for all its pixels: bands of four rows by runs of CW
// columns, about each run's centre, or about the record's own where its variance may lie below 0.005
// (the move would cost more than four digits there).
template <int T>
__device__ __forceinline__ void narrow_moments(const float4 g, const float4 c, const short4 bx,
                                               const float* __restrict__ dv, int W,
                                               float4* __restrict__ out) {
  constexpr int CW = BwdBlocks<T>::CW;
  const bool whole = c.w == -INFINITY;
  const float ia = 0.5f * rcp_approx(c.x);  // < 0
  const float D4 = whole ? 0.f : conic_det(c), a4 = 4.f * c.x * c.w;  // whole: rows without end
  const bool own = -(c.x + c.z) * 0.005f > 0.72134752f;
  float m0 = 0.f, mx = 0.f, my = 0.f, mxx = 0.f, mxy = 0.f, myy = 0.f;
  for (int by = bx.y & ~3; by <= bx.w; by += 4)
    for (int x0 = bx.x & ~(CW - 1); x0 <= bx.z; x0 += CW) {
      const float xc = own ? g.x : (float)x0 + 0.5f * (float)(CW - 1);
      float s0 = 0.f, sx = 0.f, sy = 0.f, sxx = 0.f, sxy = 0.f, syy = 0.f;
      for (int y = max(by, (int)bx.y); y <= min(by + 3, (int)bx.w); ++y) {
        const float dy = (float)y - g.y;
        const float B = row_b(c, dy), C = row_c(c, dy);
        // the row's section of the widened cut ellipse, to 1/50 pixel
        const float D = fmaf(-D4 * dy, dy, a4);  // (b y)^2 - 4 a (c y^2 - e)
        if (!(D >= 0.f)) continue;
        const float mid = g.x - B * ia, half = 0.02f - sqrt_approx(D) * ia;
        const int xa = max(x0, (int)ceilf(mid - half));
        const int xb = min(min(x0 + CW, W) - 1, (int)floorf(mid + half));
        float2 r0 = make_float2(0.f, 0.f), rx = r0, rxx = r0;  // even and odd columns
        const float* row = dv + (size_t)y * W;
        for (int x = xa & ~1; x <= xb; x += 4) {  // four pixels' loads at once
          float G[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float dx = (float)(x + k) - g.x;
            const float e = fmaf(fmaf(c.x, dx, B), dx, C);
            const bool in = x + k >= xa && x + k <= xb;
            G[k] = in && e > g.w ? __ldg(row + x + k) * ex2(e) : 0.f;
          }
#pragma unroll
          for (int k = 0; k < 4; k += 2) {
            const float X = (float)(x + k) - xc, X1 = (float)(x + k + 1) - xc;
            r0.x += G[k];
            r0.y += G[k + 1];
            rx.x = fmaf(G[k], X, rx.x);
            rx.y = fmaf(G[k + 1], X1, rx.y);
            rxx.x = fmaf(G[k], X * X, rxx.x);
            rxx.y = fmaf(G[k + 1], X1 * X1, rxx.y);
          }
        }
        const float r0s = r0.x + r0.y, rxs = rx.x + rx.y;
        s0 += r0s;
        sx += rxs;
        sxx += rxx.x + rxx.y;
        sy = fmaf(dy, r0s, sy);
        sxy = fmaf(dy, rxs, sxy);
        syy = fmaf(dy * dy, r0s, syy);
      }
      const float o = xc - g.x;  // to moments about the record's centre: dx = X + o
      m0 += s0;
      mx += fmaf(o, s0, sx);
      my += sy;
      mxx += fmaf(o, fmaf(2.f, sx, o * s0), sxx);
      mxy += fmaf(o, sy, sxy);
      myy += syy;
    }
  out[0] = make_float4(m0, mx, my, mxx);
  out[1] = make_float4(mxy, myy, 0.f, 0.f);
}

// The same out of line, for tiles of 16: inlined there, the rows of narrow records take longer (75 x
// 512^2, 50k Gaussians of half a pixel: raster_bwd 422 instead of 398 us); tiles of 8 and 32 are better
// off inlined (75 x 1024^2, 100k at 32: 3064 instead of 3110).
template <int T>
__device__ __noinline__ void narrow_moments_call(const float4 g, const float4 c, const short4 bx,
                                                 const float* __restrict__ dv, int W,
                                                 float4* __restrict__ out) {
  narrow_moments<T>(g, c, bx, dv, W, out);
}

template <int T>
__global__ void __launch_bounds__(32, T == 32 ? 24 : 28)
    k_raster_bwd(const __grid_constant__ Batch b, const uint2* __restrict__ ranges,
                 const uint32_t* __restrict__ vals, const float4* __restrict__ recs,
                 const short4* __restrict__ rect,
                 const float* __restrict__ dimg, float4* __restrict__ fpgrad,
                 const gs_status* st, int parts, int nblocks, int chunk) {
  using S = BwdBlocks<T>;  // blockIdx.y: the part of the list this warp takes
  __shared__ float4 s_g[(S::NB + 1) * S::GS];  // one block more, of zeros, for lanes without a record
  __shared__ float2 s_xy[S::NB + 1];           // a block's first pixel centre
  __shared__ float4 q_geo[32];  // the queue: records of a staged run that reach the tile
  __shared__ float4 q_con[32];
  __shared__ uint2 q_rm[32];    // record and block mask
  const int64_t key = blockIdx.x;
  const int lane = threadIdx.x;
  if (blockIdx.y >= parts) {  // the last rows of the grid: narrow records, 32 chunk of them a warp
    const int per = kThreads / 32 / chunk;  // warps per block of records
    if (st->code != GS_OK) return;
    const int64_t n = (int64_t)nblocks * per, step = (int64_t)(gridDim.y - parts) * gridDim.x;
    for (int64_t w = (int64_t)(blockIdx.y - parts) * gridDim.x + blockIdx.x; w < n; w += step) {
      const BlockItems bi = block_items(b, w / per);
      const Inst& I = b.in[bi.inst];
      const float* dv = dimg + I.img_off + (int64_t)bi.v * I.H * I.W;
      const int64_t item0 = I.item_off + (int64_t)bi.v * I.n;
      const int i0 = bi.i0 + (int)(w % per) * 32 * chunk + lane;
#pragma unroll 4
      for (int i = i0; i < min(I.n, i0 + 32 * chunk); i += 32) {
        const float4 c = recs[2 * (item0 + i) + 1];
        const short4 bx = rect[item0 + i];
        if (is_narrow<T>(c, bx)) {
          float4* out = fpgrad + 2 * (item0 + i);
          if constexpr (T == 16)
            narrow_moments_call<T>(recs[2 * (item0 + i)], c, bx, dv, I.W, out);
          else
            narrow_moments<T>(recs[2 * (item0 + i)], c, bx, dv, I.W, out);
        }
      }
    }
    return;
  }
  uint2 r = ranges[key];  // requested together with the status word, not after it
  if (st->code != GS_OK) return;
  if (parts > 1) {  // an equal part, in whole warps of records, none of less than kMinPart
    const uint32_t part = max(kMinPart, ((r.y - r.x + parts - 1) / parts + 31u) & ~31u);
    r.x = min(r.y, r.x + blockIdx.y * part);
    r.y = min(r.y, r.x + part);
  }
  if (r.x >= r.y) return;  // (>: lists of an instance without Gaussians, which no emit completes)
  const Inst& I = b.in[inst_of_key(b, key)];
  const int64_t lk = key - I.key_off;
  const int v = (int)(lk / (I.TW * I.TH)), tile = (int)(lk - (int64_t)v * I.TW * I.TH);
  const int W = I.W, H = I.H;
  const int tx0 = (tile % I.TW) * T, ty0 = (tile / I.TW) * T;
  const float* dv = dimg + I.img_off + (int64_t)v * H * W;
#pragma unroll
  for (int k = 0; k < T * T / 32; ++k) {
    const int q = lane + 32 * k, px = q % T, py = q / T, x = tx0 + px, y = ty0 + py;
    const int col = px & 7, pair = col < 4 ? col : 7 - col;
    reinterpret_cast<float*>(s_g)[((px >> 3) * S::NBY + (py >> 2)) * 4 * S::GS + pair * 8 +
                                  (py & 3) * 2 + (col >> 2)] =
        (x < W && y < H) ? dv[(size_t)y * W + x] : 0.f;
  }
  if (lane < S::GS) s_g[S::NB * S::GS + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (lane == 0) s_xy[S::NB] = make_float2((float)tx0, (float)ty0);
  if (lane < S::NB)
    s_xy[lane] = make_float2((float)(tx0 + (lane / S::NBY) * S::BW),
                             (float)(ty0 + (lane % S::NBY) * 4));
  const unsigned lt = gsd::lanemask_lt();
  uint32_t pos = r.x;    // next record of the list to stage
  // the next run's records are requested one run ahead, so that staging waits for one gather, not
  // two (75 x 512^2: 1059 -> 1032 us; at tile 32 the register costs more, 5.82 -> 5.94 ms)
  constexpr bool AHEAD = T < 32;
  uint32_t ahead = AHEAD && pos + lane < r.y ? vals[pos + lane] : 0u;
  int qh = 0, qn = 0;    // the queue's next and its end
  // the lane's record: the blocks still to walk, its coefficients and its six sums
  uint32_t rec = 0u, mask = 0u;
  float gx = 0.f, gy = 0.f, cut = INFINITY, c0 = 0.f, c1 = 0.f, c2 = 0.f;
  float m0 = 0.f, mx = 0.f, my = 0.f, mxx = 0.f, mxy = 0.f, myy = 0.f;
  for (;;) {
    bool need = mask == 0u;
    unsigned idle = __ballot_sync(0xffffffffu, need);
    if (idle) {
      // finished records leave, waiting ones come in
      if (need) {
        if ((__float_as_uint(m0) | __float_as_uint(mx) | __float_as_uint(my)) |
            (__float_as_uint(mxx) | __float_as_uint(mxy) | __float_as_uint(myy))) {
          atomicAdd(&fpgrad[2 * (size_t)rec], make_float4(m0, mx, my, mxx));
          atomicAdd(&fpgrad[2 * (size_t)rec + 1], make_float4(mxy, myy, 0.f, 0.f));
        }
        m0 = mx = my = mxx = mxy = myy = 0.f;
        cut = INFINITY;  // an idle lane never passes, whatever a thin ellipse's e rounds to
      }
      for (;;) {
        const int slot = qh + __popc(idle & lt);
        if (need && slot < qn) {
          const float4 g = q_geo[slot], c = q_con[slot];
          const uint2 rm = q_rm[slot];
          gx = g.x;
          gy = g.y;
          cut = g.w;
          c0 = c.x;
          c1 = c.y;
          c2 = c.z;
          rec = rm.x;
          mask = rm.y;
          need = false;
        }
        qh += __popc(idle);
        if (qh <= qn) {  // every lane has one
          idle = 0u;
          break;
        }
        qh = qn;
        idle = __ballot_sync(0xffffffffu, need);
        if (pos >= r.y) break;
        // the queue is empty: stage the next run of records
        const bool in = pos + lane < r.y;
        float4 g, c;
        uint32_t nrec = 0, nmask = 0;
        if (in) {
          nrec = AHEAD ? ahead : vals[pos + lane];
          g = recs[2 * (size_t)nrec];
          c = recs[2 * (size_t)nrec + 1];
          const short4 bx = rect[nrec];
          if (!is_narrow<T>(c, bx)) nmask = block_mask<T, S::BW>(g, c, bx, tx0, ty0);
        }
        pos += 32;
        if (AHEAD) ahead = pos + lane < r.y ? vals[pos + lane] : 0u;
        __syncwarp();  // the queue's last reads are done
        const unsigned keep = __ballot_sync(0xffffffffu, nmask != 0u);
        if (nmask) {
          const int q = __popc(keep & lt);
          q_geo[q] = g;
          q_con[q] = c;
          q_rm[q] = make_uint2(nrec, nmask);
        }
        qh = 0;
        qn = __popc(keep);
        __syncwarp();
      }
      if (idle == 0xffffffffu) break;
    }
    // ---- every lane walks the next block of its record
    const int blk = mask ? 31 - __clz(mask) : S::NB;
    mask &= ~(1u << (blk & 31));
    const float2 xy = s_xy[blk];
    const float4* gp = s_g + blk * S::GS;
    // pixel pairs of a row in packed FP32x2 arithmetic: each component rounds like the scalar
    // fmaf / add / mul, so e and the cut are exactly the forward's
    const float2 ca = make_float2(c0, c0);
    float2 B2[4], C2[4];
#pragma unroll
    for (int ry = 0; ry < 4; ++ry) {
      const float dy = (xy.y + (float)ry) - gy;
      const float B = c1 * dy, cdy2 = (c2 * dy) * dy;
      B2[ry] = make_float2(B, B);
      C2[ry] = make_float2(cdy2, cdy2);
    }
    // Moments about the block's centre.  Per pair of mirrored columns the four rows fold into
    // Q = sum G, D = 2 sum Y G and P0, the outer rows' part (sum Y^2 G = 2 P0 + Q / 4).  Along x the
    // outermost pair comes first and running sums give the weights: with n = 3 - p, |X| = n + 1/2
    // and X^2 = 2 (n (n + 1) / 2) + 1/4, where the sum of the running sums weighs pair p by n and
    // the sum of those by n (n + 1) / 2.  (No constants, so every step is one packed addition.)
    float2 a0, q0, q1, q2, d0, d1;
    float2 xp = make_float2(xy.x, xy.x + 7.f);
    const float2 ngx = make_float2(-gx, -gx), m1 = make_float2(-1.f, -1.f);
    const float2 step = make_float2(1.f, -1.f), three = make_float2(3.f, 3.f);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const float2 dx = __fadd2_rn(xp, ngx);
      xp = __fadd2_rn(xp, step);  // exact
      const float4 ga = gp[2 * p], gb = gp[2 * p + 1];  // rows 0, 1 and 2, 3
      float2 G[4];
#pragma unroll
      for (int ry = 0; ry < 4; ++ry) {
        const float2 e = __ffma2_rn(__ffma2_rn(ca, dx, B2[ry]), dx, C2[ry]);
        const float2 gg = ry == 0   ? make_float2(ga.x, ga.y)
                          : ry == 1 ? make_float2(ga.z, ga.w)
                          : ry == 2 ? make_float2(gb.x, gb.y)
                                    : make_float2(gb.z, gb.w);
        const float2 val = make_float2(ex2(e.x), ex2(e.y));
        G[ry] = __fmul2_rn(gg, make_float2(e.x > cut ? val.x : 0.f, e.y > cut ? val.y : 0.f));
      }
      const float2 P0 = __fadd2_rn(G[0], G[3]), P1 = __fadd2_rn(G[1], G[2]);
      const float2 M0 = __ffma2_rn(G[0], m1, G[3]), M1 = __ffma2_rn(G[1], m1, G[2]);
      const float2 D = __ffma2_rn(M0, three, M1), Q = __fadd2_rn(P0, P1);
      if (p == 0) {
        a0 = P0;
        q0 = q1 = q2 = Q;
        d0 = d1 = D;
      } else {
        a0 = __fadd2_rn(a0, P0);
        q0 = __fadd2_rn(q0, Q);
        d0 = __fadd2_rn(d0, D);
        if (p < 3) {
          q1 = __fadd2_rn(q1, q0);
          q2 = __fadd2_rn(q2, q1);
          d1 = __fadd2_rn(d1, d0);
        }
      }
    }
    const float t0 = q0.x + q0.y, tx = fmaf(0.5f, q0.y - q0.x, q1.y - q1.x);
    const float txx = fmaf(2.f, q2.x + q2.y, 0.25f * t0);
    const float ty = 0.5f * (d0.x + d0.y), txy = 0.5f * fmaf(0.5f, d0.y - d0.x, d1.y - d1.x);
    const float tyy = fmaf(2.f, a0.x + a0.y, 0.25f * t0);
    // to moments about the record's centre: dx = X + ox, dy = Y + oy
    const float ox = (xy.x + 3.5f) - gx, oy = (xy.y + 1.5f) - gy;
    const float ux = fmaf(ox, t0, tx);
    m0 += t0;
    mx += ux;
    my += fmaf(oy, t0, ty);
    mxx += fmaf(ox, tx + ux, txx);
    mxy += fmaf(ox, ty, fmaf(oy, ux, txy));
    myy += fmaf(oy, fmaf(2.f, ty, oy * t0), tyy);
  }
}

// ------------------------------------------------------------------------------------------
// chain: a thread per (Gaussian, chunk of up to kChainViews views), consecutive threads on
// consecutive Gaussians of one chunk, so that the moment loads of a warp are one contiguous
// run and the view frame is the same for all its lanes; each thread chains its views'
// moments to the Gaussian's parameters (the rotation's gradient stays a matrix until the last
// view), requests the next view's moments one view ahead, and adds its sums with float4
// atomics (the gradients are zeroed first unless accumulating).  Bound by FP32 issue.
// 75 x 512^2, 50k Gaussians: 107 -> 89 us; a third CTA per SM costs spills (112), one leaves
// latency open (137).  Small calls take fewer views per thread (one at 2000 Gaussians x 8 views,
// 17 -> 8 us): the chunks then fill the SMs.
// ------------------------------------------------------------------------------------------
constexpr int kChainViews = 8;

__global__ void __launch_bounds__(kThreads, 2)
    k_project_chain(const __grid_constant__ Batch b, const float4* __restrict__ mean_rho,
                    const float4* __restrict__ scale, const float4* __restrict__ quat,
                    int total_n, int vchunks, int cv, const ViewFrame* __restrict__ frames,
                    const float4* fpgrad, float4* __restrict__ g_mr,
                    float4* __restrict__ g_sc, float4* __restrict__ g_q,
                    const uint32_t* __restrict__ counts, float* __restrict__ stat,
                    int* __restrict__ vis) {
  gsd::pdl_begin();
  const int64_t tid = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (tid >= (int64_t)total_n * vchunks) return;
  const int gi = (int)(tid % total_n), ch = (int)(tid / total_n);
  const Inst& I = b.in[inst_of_gaussian(b, gi)];
  const int il = gi - I.g_off;
  const int v0 = ch * cv, v1 = min(v0 + cv, I.nv);
  if (v0 >= v1) return;
  const float4 mr = mean_rho[gi], sc = scale[gi], qt = quat[gi];
  float gp[3] = {0.f, 0.f, 0.f}, grho = 0.f, gsc[3] = {0.f, 0.f, 0.f};
  float gR[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  bool any = false;
  float qn[4] = {0.f, 0.f, 0.f, 0.f}, inv_norm = 0.f;
  // adaptive density control statistics: NDC detector-position gradient norms and the
  // number of views with a listed tile
  float st_acc = 0.f;
  int vis_acc = 0;
  size_t rec = (size_t)(I.item_off + (int64_t)v0 * I.n + il);
  float4 n0 = fpgrad[2 * rec], n1 = fpgrad[2 * rec + 1];  // the next view's moments, one ahead
  for (int v = v0; v < v1; ++v, rec += I.n) {
    if (stat && counts[rec] > 0u) ++vis_acc;
    const float4 m0 = n0, m1 = n1;
    if (v + 1 < v1) {
      n0 = fpgrad[2 * (rec + I.n)];
      n1 = fpgrad[2 * (rec + I.n) + 1];
    }
    if (m0.x == 0.f && m0.y == 0.f && m0.z == 0.f && m0.w == 0.f && m1.x == 0.f && m1.y == 0.f)
      continue;
    const ViewFrame f = frames[I.v_off + v];
    Fwd o;
    int x0, y0, x1, y1;
    if (!footprint(mr, sc, qt, f, I.W, I.H, b.cut2, b.eps, b.znear, o, x0, y0, x1, y1)) continue;
    chain_one(o, f, m0, m1, gp, grho, gsc, gR);
    any = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) qn[k] = o.qn[k];
    inv_norm = o.inv_norm;
    if (stat) {
      // dI/dpx = A e (ca dx + cb dy) summed against dL/dI: the moments' first-order terms
      const float dpx = o.A * (o.ca * m0.y + o.cb * m0.z);
      const float dpy = o.A * (o.cb * m0.y + o.cc * m0.z);
      const float nx = 0.5f * (float)I.W * dpx, ny = 0.5f * (float)I.H * dpy;
      st_acc += sqrtf(nx * nx + ny * ny);
    }
  }
  if (any) {
    float gq[4];
    gsd::rot_to_quat_grad(qn[0], qn[1], qn[2], qn[3], gR, gq);
    gsd::quat_normalize_grad(qn, inv_norm, gq);
    atomicAdd(&g_mr[gi], make_float4(gp[0], gp[1], gp[2], grho));
    atomicAdd(&g_sc[gi], make_float4(gsc[0], gsc[1], gsc[2], 0.f));
    atomicAdd(&g_q[gi], make_float4(gq[0], gq[1], gq[2], gq[3]));
  }
  if (stat) {
    if (st_acc != 0.f) atomicAdd(&stat[gi], st_acc);
    if (vis_acc) atomicAdd(&vis[gi], vis_acc);
  }
}

// Zeroes the backward's accumulators in one launch: the record moments and, unless the caller
// accumulates, the three gradient arrays.
__global__ void __launch_bounds__(kThreads)
    k_zero(float4* __restrict__ fp, int64_t n_fp, float4* __restrict__ g0, float4* __restrict__ g1,
           float4* __restrict__ g2, int64_t n_g) {
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  for (int64_t i = t; i < n_fp; i += stride) fp[i] = z;
  for (int64_t i = t; i < n_g; i += stride) g0[i] = g1[i] = g2[i] = z;
}

// ------------------------------------------------------------------------------------------
// Host orchestration
// ------------------------------------------------------------------------------------------
bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

int check_common(const float* mr, const float* sc, const float* qt, const Plan& p,
                 const gs_view* views, void* ws) {
  if (p.total_n > 0 && (!mr || !sc || !qt)) return GS_ERR_ARG;
  if (!views || !ws) return GS_ERR_ARG;
  if (!aligned16(mr) || !aligned16(sc) || !aligned16(qt) || !aligned16(ws)) return GS_ERR_ARG;
  return GS_OK;
}

int cap_from_ws(const gs_instance* inst, int n_inst, const gs_opts* o, size_t ws_bytes,
                int64_t& cap) {
  Plan p0;
  GS_TRY(make_plan(inst, n_inst, o, 0, p0));
  const size_t base = carve(nullptr, p0).bytes;
  if (ws_bytes < base) return GS_ERR_CAPACITY;
  // each unit of capacity costs 16 bytes (keys, vals and their alternates) plus alignment
  int64_t c = (int64_t)((ws_bytes - base) / 16);
  while (c > 0) {
    Plan p;
    GS_TRY(make_plan(inst, n_inst, o, c, p));
    if (carve(nullptr, p).bytes <= ws_bytes) break;
    c -= 64;
  }
  cap = std::max<int64_t>(c, 0);
  return GS_OK;
}

// Validates the table and the pointers (host only, before any launch), then plans the
// workspace's pair capacity from its size.
int prepare(const gs_instance* inst, int n_inst, const gs_opts* o, const float* mr,
            const float* sc, const float* qt, const gs_view* views, void* ws, size_t ws_bytes,
            Plan& p, Layout& L) {
  {
    Plan p0;
    GS_TRY(make_plan(inst, n_inst, o, 0, p0));
    GS_TRY(check_common(mr, sc, qt, p0, views, ws));
  }
  int64_t cap = 0;
  GS_TRY(cap_from_ws(inst, n_inst, o, ws_bytes, cap));
  GS_TRY(make_plan(inst, n_inst, o, cap, p));
  L = carve(ws, p);
  return GS_OK;
}

// Dynamic shared memory above 48 KB needs the kernel's limit raised (host-side state of the
// current device, set on every call that needs it).
size_t emit_smem(const Plan& p) { return (size_t)(3 + kThreads / 32) * p.max_tp * sizeof(uint32_t); }

int preprocess_and_scan(const Plan& p, const Layout& L, const float* mr, const float* sc,
                        const float* qt, const gs_view* views, cudaStream_t s, void* ws) {
  const size_t smem = p.direct ? (size_t)p.max_tp * sizeof(uint32_t) : 0;
  GS_TRY(launch("preprocess", p.direct ? k_preprocess<true> : k_preprocess<false>,
                dim3(p.nblocks), dim3(kThreads), smem, s, p.b, (const float4*)mr,
                (const float4*)sc, (const float4*)qt, views, L.frames, L.rec, L.rect,
                L.tmask, L.counts, L.block_sums, L.tcount, L.ticket, L.st));
  if (!p.direct) return scan_block_sums(L.block_sums, L.block_offs, p.nblocks, L.st, p.cap, s);
  auto off = [&](const void* q) { return (int64_t)((const char*)q - (const char*)ws); };
  return launch_after("key_scan", k_key_scan, dim3((unsigned)((p.n_keys + kScanKeys - 1) / kScanKeys)),
                dim3(kScanKeys * kScanSegs), 0, s, p.b, p.n_keys, (const uint16_t*)L.tcount,
                L.toffset, L.klocal, L.ranges, L.gsum, L.ticket, L.vkeys, p.total_v, L.st, p.cap,
                off(L.vals), off(L.ranges), off(L.vkeys));
}

// preprocess -> lists and ranges of every (view, tile), by the direct or the sorted route.  On
// return *svals points at the lists inside the workspace.
int bin_pairs(const Plan& p, const Layout& L, const float* mr, const float* sc, const float* qt,
              const gs_view* views, cudaStream_t s, void* ws, uint32_t** svals) {
  *svals = L.vals;
  if (p.total_n == 0) {
    GS_CUDA(cudaMemsetAsync(L.st, 0, sizeof(gs_status), s));
    GS_CUDA(cudaMemsetAsync(L.ranges, 0, (size_t)p.n_keys * sizeof(uint2), s));
    return GS_OK;
  }
  GS_TRY(preprocess_and_scan(p, L, mr, sc, qt, views, s, ws));
  if (p.direct) {
    const size_t smem = emit_smem(p);
    if (smem > 48 * 1024)
      GS_CUDA(cudaFuncSetAttribute(k_emit_direct, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)smem));
    return launch("emit", k_emit_direct, dim3(p.nblocks), dim3(kThreads), smem, s, p.b,
                  (const uint32_t*)L.counts, (const float4*)L.rec,
                  (const short4*)L.rect, (const uint32_t*)L.tmask, (const uint32_t*)L.toffset,
                  (const uint32_t*)L.klocal, (const unsigned long long*)L.gsum, L.ranges, L.vals,
                  (const gs_status*)L.st);
  }
  uint32_t* k = L.keys;
  uint32_t* v = L.vals;
  const bool odd = (p.sort.passes & 1) != 0;
  uint32_t* fk = odd ? L.keys_alt : L.keys;
  uint32_t* fv = odd ? L.vals_alt : L.vals;
  GS_TRY(launch("emit", k_emit, dim3(p.nblocks), dim3(kThreads), 0, s, p.b,
                (const uint32_t*)L.counts, (const float4*)L.rec,
                (const short4*)L.rect, (const uint32_t*)L.tmask, (const uint32_t*)L.block_offs,
                L.keys, L.vals, L.st, (int64_t)((char*)fk - (char*)ws),
                (int64_t)((char*)fv - (char*)ws)));
  GS_TRY(radix_sort(&k, &v, L.keys_alt, L.vals_alt, L.hist, p.sort, L.st, p.cap, s));
  GS_CUDA(cudaMemsetAsync(L.ranges, 0, (size_t)p.n_keys * sizeof(uint2), s));
  GS_TRY(launch("ranges", k_tile_ranges, dim3(4 * num_sms()), dim3(kThreads), 0, s, p.b,
                (const uint32_t*)k, L.ranges, (const gs_status*)L.st));
  *svals = v;
  return GS_OK;
}

// Where the lists of the last binning lie.
uint32_t* sorted_vals(const Plan& p, const Layout& L) {
  return !p.direct && (p.sort.passes & 1) ? L.vals_alt : L.vals;
}

template <int T>
int raster_fwd(const Plan& p, const Layout& L, const uint32_t* vals, float* img, bool count,
               cudaStream_t s) {
  dim3 grid((unsigned)p.n_keys), block(FwdBlocks<T>::NT);
  if (count)
    return launch("raster_count", k_raster_fwd<T, true>, grid, block, 0, s, p.b,
                  (const uint2*)L.ranges, vals, (const float4*)L.rec,
                  (const short4*)L.rect, img, L.st);
  return launch("raster_fwd", k_raster_fwd<T, false>, grid, block, 0, s, p.b,
                (const uint2*)L.ranges, vals, (const float4*)L.rec,
                (const short4*)L.rect, img, L.st);
}

template <int T>
int raster_bwd(const Plan& p, const Layout& L, const uint32_t* vals, const float* dimg,
               cudaStream_t s) {
  // few tiles: their lists are split over up to 16 warps (the records' sums meet in atomics anyway),
  // while the grid holds less than 64 warps per SM, two waves; a part that a short list does not
  // need leaves before it reads dL/dI.  raster_bwd, us, unsplit below 16 warps per SM (as before) and now,
  // against CTAs of a whole tile's warps: 8 views of 512^2, 2k large Gaussians, tile 16 257 -> 215 (184),
  // tile 32 356 -> 246 (204); 50k, tile 32 208 -> 139 (154); 20 views of 256^2, 20k, tile 32 222 -> 137
  // (178); 8 views of 64^2, 2k 10.8 -> 9.2 (15); short lists pay for the idle warps: one view of
  // 1024^2, 20k, tile 32 44 -> 50 (27), tile 16 24.3 -> 24.6 (22).  Two waves' worth of parts for more
  // tiles cost more than they bring (one view of 2048^2, 16,384 tiles: 63 -> 68).
  const int64_t slots = 64 * (int64_t)num_sms();
  const int parts = p.n_keys > slots ? 1 : (int)std::max<int64_t>(2, std::min<int64_t>(16, slots / p.n_keys));
  // warps for the narrow records: 32 records each while they are few, up to 256
  int chunk = 1;
  while (chunk < 8 && (int64_t)p.nblocks * (8 / chunk) > 16 * (int64_t)num_sms()) chunk *= 2;
  const int64_t rows = std::min<int64_t>(
      ((int64_t)p.nblocks * (8 / chunk) + p.n_keys - 1) / p.n_keys, 65535 - parts);
  return launch("raster_bwd", k_raster_bwd<T>, dim3((unsigned)p.n_keys, (unsigned)(parts + rows)),
                dim3(32), 0, s,
                p.b, (const uint2*)L.ranges, vals, (const float4*)L.rec,
                (const short4*)L.rect, dimg, L.fpgrad, (const gs_status*)L.st, parts, p.nblocks, chunk);
}

int dispatch_fwd(const Plan& p, const Layout& L, const uint32_t* vals, float* img, bool count,
                 cudaStream_t s) {
  switch (p.b.T) {
    case 8: return raster_fwd<8>(p, L, vals, img, count, s);
    case 16: return raster_fwd<16>(p, L, vals, img, count, s);
    default: return raster_fwd<32>(p, L, vals, img, count, s);
  }
}

gs_instance one(int n, int nv, int W, int H) {
  gs_instance i;
  memset(&i, 0, sizeof(i));
  i.n = n;
  i.n_views = nv;
  i.W = W;
  i.H = H;
  return i;
}

}  // namespace
}  // namespace gs

using namespace gs;

extern "C" {

size_t gs_project_batch_workspace_size(const gs_instance* inst, int n_inst, const gs_opts* opts,
                                       int64_t max_pairs) {
  Plan p;
  if (make_plan(inst, n_inst, opts, max_pairs, p) != GS_OK) return 0;
  return carve(nullptr, p).bytes;
}

int gs_project_batch_count_pairs(const float* d_mean_rho, const float* d_scale,
                                 const float* d_quat, const gs_view* d_views,
                                 const gs_instance* inst, int n_inst, const gs_opts* opts,
                                 void* d_ws, size_t ws_bytes, void* stream, int64_t* h_pairs) {
  if (!h_pairs) return GS_ERR_ARG;
  Plan p;
  Layout L;
  GS_TRY(prepare(inst, n_inst, opts, d_mean_rho, d_scale, d_quat, d_views, d_ws, ws_bytes, p,
                 L));
  cudaStream_t s = (cudaStream_t)stream;
  if (p.total_n == 0) {
    *h_pairs = 0;
    return GS_OK;
  }
  GS_TRY(preprocess_and_scan(p, L, d_mean_rho, d_scale, d_quat, d_views, s, d_ws));
  gs_status st;
  GS_TRY(gs_read_status(d_ws, stream, &st));
  *h_pairs = st.pairs;
  return GS_OK;
}

int gs_project_batch(const float* d_mean_rho, const float* d_scale, const float* d_quat,
                     const gs_view* d_views, const gs_instance* inst, int n_inst,
                     const gs_opts* opts, float* d_img, void* d_ws, size_t ws_bytes,
                     void* stream) {
  if (!d_img) return GS_ERR_ARG;
  Plan p;
  Layout L;
  GS_TRY(prepare(inst, n_inst, opts, d_mean_rho, d_scale, d_quat, d_views, d_ws, ws_bytes, p,
                 L));
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t* v;
  GS_TRY(bin_pairs(p, L, d_mean_rho, d_scale, d_quat, d_views, s, d_ws, &v));
  return dispatch_fwd(p, L, v, d_img, false, s);
}

int gs_project_batch_count_evals(const float* d_mean_rho, const float* d_scale,
                                 const float* d_quat, const gs_view* d_views,
                                 const gs_instance* inst, int n_inst, const gs_opts* opts,
                                 void* d_ws, size_t ws_bytes, void* stream) {
  Plan p;
  Layout L;
  GS_TRY(prepare(inst, n_inst, opts, d_mean_rho, d_scale, d_quat, d_views, d_ws, ws_bytes, p,
                 L));
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t* v;
  GS_TRY(bin_pairs(p, L, d_mean_rho, d_scale, d_quat, d_views, s, d_ws, &v));
  GS_CUDA(cudaMemsetAsync(&L.st->evals, 0, sizeof(int64_t), s));
  return dispatch_fwd(p, L, v, nullptr, true, s);
}

int gs_project_batch_backward_stats(const float* d_mean_rho, const float* d_scale,
                                    const float* d_quat, const gs_view* d_views,
                                    const gs_instance* inst, int n_inst, const gs_opts* opts,
                                    const float* d_dimg, float* d_g_mean_rho,
                                    float* d_g_scale, float* d_g_quat, float* d_grad_stat,
                                    int32_t* d_vis, int accumulate, int reuse, void* d_ws,
                                    size_t ws_bytes, void* stream) {
  if ((d_grad_stat == nullptr) != (d_vis == nullptr)) return GS_ERR_ARG;
  Plan p;
  Layout L;
  GS_TRY(prepare(inst, n_inst, opts, d_mean_rho, d_scale, d_quat, d_views, d_ws, ws_bytes, p,
                 L));
  if (!d_dimg || (p.total_n > 0 && (!d_g_mean_rho || !d_g_scale || !d_g_quat)))
    return GS_ERR_ARG;
  if (!aligned16(d_g_mean_rho) || !aligned16(d_g_scale) || !aligned16(d_g_quat))
    return GS_ERR_ARG;
  if (p.total_n == 0) return GS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  uint32_t* v;
  if (reuse)
    v = sorted_vals(p, L);
  else
    GS_TRY(bin_pairs(p, L, d_mean_rho, d_scale, d_quat, d_views, s, d_ws, &v));
  const int64_t n_fp = 2 * p.items, n_g = accumulate ? 0 : p.total_n;
  GS_TRY(launch("zero", k_zero,
                dim3((unsigned)std::min<int64_t>((std::max(n_fp, n_g) + kThreads - 1) / kThreads,
                                                 8 * (int64_t)num_sms())),
                dim3(kThreads), 0, s, L.fpgrad, n_fp, (float4*)d_g_mean_rho, (float4*)d_g_scale,
                (float4*)d_g_quat, n_g));
  switch (p.b.T) {
    case 8: GS_TRY(raster_bwd<8>(p, L, v, d_dimg, s)); break;
    case 16: GS_TRY(raster_bwd<16>(p, L, v, d_dimg, s)); break;
    default: GS_TRY(raster_bwd<32>(p, L, v, d_dimg, s)); break;
  }
  int max_nv = 1;
  for (int k = 0; k < p.b.count; ++k) max_nv = std::max(max_nv, p.b.in[k].nv);
  int cv = kChainViews;  // halved while the chunks make less than two CTAs per SM
  while (cv > 1 && (int64_t)p.total_n * ((max_nv + cv - 1) / cv) < 2 * (int64_t)num_sms() * kThreads)
    cv /= 2;
  const int vchunks = (max_nv + cv - 1) / cv;
  const int64_t threads = (int64_t)p.total_n * vchunks;
  const int blocks = (int)((threads + kThreads - 1) / kThreads);
  return launch_after("project_chain", k_project_chain, dim3(blocks), dim3(kThreads), 0, s, p.b,
                (const float4*)d_mean_rho, (const float4*)d_scale, (const float4*)d_quat,
                p.total_n, vchunks, cv, (const ViewFrame*)L.frames, (const float4*)L.fpgrad,
                (float4*)d_g_mean_rho, (float4*)d_g_scale, (float4*)d_g_quat,
                (const uint32_t*)L.counts, d_grad_stat, (int*)d_vis);
}

int gs_project_batch_backward(const float* d_mean_rho, const float* d_scale,
                              const float* d_quat, const gs_view* d_views,
                              const gs_instance* inst, int n_inst, const gs_opts* opts,
                              const float* d_dimg, float* d_g_mean_rho, float* d_g_scale,
                              float* d_g_quat, int accumulate, int reuse, void* d_ws,
                              size_t ws_bytes, void* stream) {
  return gs_project_batch_backward_stats(d_mean_rho, d_scale, d_quat, d_views, inst, n_inst,
                                         opts, d_dimg, d_g_mean_rho, d_g_scale, d_g_quat,
                                         nullptr, nullptr, accumulate, reuse, d_ws, ws_bytes,
                                         stream);
}

// ---- single instance = batch of one ------------------------------------------------------

size_t gs_project_workspace_size(int n, int n_views, int W, int H, const gs_opts* opts,
                                 int64_t max_pairs) {
  const gs_instance i = one(n, n_views, W, H);
  return gs_project_batch_workspace_size(&i, 1, opts, max_pairs);
}

int gs_project_count_pairs(const float* d_mean_rho, const float* d_scale, const float* d_quat,
                           int n, const gs_view* d_views, int n_views, int W, int H,
                           const gs_opts* opts, void* d_ws, size_t ws_bytes, void* stream,
                           int64_t* h_pairs) {
  const gs_instance i = one(n, n_views, W, H);
  return gs_project_batch_count_pairs(d_mean_rho, d_scale, d_quat, d_views, &i, 1, opts, d_ws,
                                      ws_bytes, stream, h_pairs);
}

int gs_project(const float* d_mean_rho, const float* d_scale, const float* d_quat, int n,
               const gs_view* d_views, int n_views, int W, int H, const gs_opts* opts,
               float* d_img, void* d_ws, size_t ws_bytes, void* stream) {
  const gs_instance i = one(n, n_views, W, H);
  return gs_project_batch(d_mean_rho, d_scale, d_quat, d_views, &i, 1, opts, d_img, d_ws,
                          ws_bytes, stream);
}

int gs_project_count_evals(const float* d_mean_rho, const float* d_scale, const float* d_quat,
                           int n, const gs_view* d_views, int n_views, int W, int H,
                           const gs_opts* opts, void* d_ws, size_t ws_bytes, void* stream) {
  const gs_instance i = one(n, n_views, W, H);
  return gs_project_batch_count_evals(d_mean_rho, d_scale, d_quat, d_views, &i, 1, opts, d_ws,
                                      ws_bytes, stream);
}

int gs_project_backward(const float* d_mean_rho, const float* d_scale, const float* d_quat,
                        int n, const gs_view* d_views, int n_views, int W, int H,
                        const gs_opts* opts, const float* d_dimg, float* d_g_mean_rho,
                        float* d_g_scale, float* d_g_quat, int accumulate, int reuse,
                        void* d_ws, size_t ws_bytes, void* stream) {
  const gs_instance i = one(n, n_views, W, H);
  return gs_project_batch_backward(d_mean_rho, d_scale, d_quat, d_views, &i, 1, opts, d_dimg,
                                   d_g_mean_rho, d_g_scale, d_g_quat, accumulate, reuse, d_ws,
                                   ws_bytes, stream);
}

int gs_project_backward_stats(const float* d_mean_rho, const float* d_scale,
                              const float* d_quat, int n, const gs_view* d_views, int n_views,
                              int W, int H, const gs_opts* opts, const float* d_dimg,
                              float* d_g_mean_rho, float* d_g_scale, float* d_g_quat,
                              float* d_grad_stat, int32_t* d_vis, int accumulate, int reuse,
                              void* d_ws, size_t ws_bytes, void* stream) {
  const gs_instance i = one(n, n_views, W, H);
  return gs_project_batch_backward_stats(d_mean_rho, d_scale, d_quat, d_views, &i, 1, opts,
                                         d_dimg, d_g_mean_rho, d_g_scale, d_g_quat,
                                         d_grad_stat, d_vis, accumulate, reuse, d_ws, ws_bytes,
                                         stream);
}

}  // extern "C"
