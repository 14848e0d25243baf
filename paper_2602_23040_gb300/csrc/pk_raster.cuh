// Shared pieces of the forward (a4) and backward (a5) compositing kernels:
// tile -> view lookup, batch staging of a tile's splats into shared memory,
// and the per-pixel alpha evaluation.  The evaluation is written with
// explicit round-to-nearest intrinsics so that both kernels take exactly
// the same skip / clamp decisions for the same (pixel, splat).
#pragma once

#include "pk_common.cuh"
#include "pk_f32x2.cuh"

namespace pk {

constexpr int kTileSide = 16;   // side of the pixel block of one compositing CTA
// Splats staged per batch: a template parameter of the compositing
// kernels (64, 128 or 256; pk_options.batch, chosen by pk_autotune).
constexpr int kBatchMax = 256;

// One CTA per 16 x 16 pixel block with kPx pixels per thread (2, 4 or 8).
// A warp covers a kBW x kBH block (8 x 8 for 2 pixels, 16 x 8 for 4, the
// whole 16 x 16 for 8) and skips as a whole every splat that misses its
// block; a lane holds one column of it, kPx pixels kRowStep rows apart.
// More pixels per lane spread the per-splat work of a warp (shared-memory
// loads, the block test, the gradient reduction) over more pixels, at the
// price of a coarser block test and more registers.
template <int kPx>
struct Geo {
  static_assert(kPx == 2 || kPx == 4 || kPx == 8, "2, 4 or 8 pixels per thread");
  static constexpr int kThreads = kTileSide * kTileSide / kPx;   // 128, 64 or 32
  static constexpr int kWarps = kThreads / 32;
  static constexpr int kBW = kPx == 2 ? 8 : 16;
  static constexpr int kBH = kPx == 8 ? 16 : 8;
  static constexpr int kRowStep = kBH / kPx;                      // 4, 2 or 2
  static constexpr int kBlocksX = kTileSide / kBW;                // warp blocks per row
  static_assert(kBW * kBH == 32 * kPx, "a warp's block holds its lanes' pixels");
};

// Pixels per thread: the forward keeps 2 (its per-splat work is small, and
// 8 x 8 blocks skip more), the backward 4 (its per-splat reduction of nine
// gradients is spread over twice the pixels); measured at the 52-view rig.
constexpr int kFwdPx = 2, kBwdPx = 4;

// Lane's column ox and first row oy in the tile; (bx, by) = its warp block's corner.
template <int kPx>
__device__ __forceinline__ void pixel_of(int tid, int &ox, int &oy, int &bx, int &by) {
  using G = Geo<kPx>;
  const int w = tid >> 5, l = tid & 31;
  bx = (w % G::kBlocksX) * G::kBW;
  by = (w / G::kBlocksX) * G::kBH;
  ox = bx + (l % G::kBW);
  oy = by + l / G::kBW;
}

// View that owns global tile t (binary search over tile offsets).
__device__ __forceinline__ int view_of_tile(const uint32_t *__restrict__ toff, int V, uint32_t t) {
  int lo = 0, hi = V - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(toff + mid) <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

struct Staged {
  float4 *a;     // m_x, m_y, A = k conic_a, B = 2 k conic_b      (k = -log2(e) / 2)
  float4 *b;     // C = k conic_c, -opacity, red, green
  float4 *c;     // blue, pair index (bits), pcut, -1 / opacity
  float4 *box;   // conservative pixel-centre box of the contributing ellipse
  float4 *q;     // conic_a, conic_b, conic_c, qlim = min(9, 2 ln(255 o)) for the block test
};

// 2^x on the MUFU unit (one instruction; relative error below 2^-22).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1 / x and sqrt(x) on the MUFU unit (one instruction each, relative error
// near 2^-22): used only for the culling box, whose margins are far wider.
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

// Stage one splat.  The exponent of the Gaussian is evaluated directly as
// power = k q = A dx^2 + B dx dy + C dy^2, so alpha = o 2^power; a pixel is
// skipped unless power >= pcut = max(9 k, -log2(255 o)), i.e. unless both
// q <= 9 and o e^{-q/2} >= 1/255 hold.  The box bounds every pixel where
// q <= min(9, 2 ln(255 o)), widened by a relative 1e-3 and 0.01 px so that
// rounding can never put a passing pixel outside; it only lets whole warps
// skip, the per-pixel test still decides.
__device__ __forceinline__ void stage_from(const float4 r0, const float4 r1, const float4 r2, uint32_t pid,
                                           const Staged &s, int j) {
  const float ca = r0.z, cb = r0.w, cc = r1.x, o = r1.y;
  s.a[j] = make_float4(r0.x, r0.y, __fmul_rn(kExpScale, ca), __fmul_rn(2.f * kExpScale, cb));
  s.b[j] = make_float4(__fmul_rn(kExpScale, cc), -o, r2.x, r2.y);
  const float pcut = fmaxf(9.f * kExpScale, -__log2f(255.f * o));
  s.c[j] = make_float4(r2.z, __uint_as_float(pid), pcut, __fdividef(-1.f, o));   // (read only where the splat blends: o >= 1/255)
  const float qlim = fminf(kQMax, 2.f * __logf(255.f * o));
  s.q[j] = make_float4(ca, cb, cc, qlim);
  const float detq = ca * cc - cb * cb;
  float4 box;
  if (!(qlim >= 0.f)) {
    box = make_float4(1.f, -1.f, 1.f, -1.f);    // can never pass the alpha test
  } else if (detq > 0.f && isfinite(detq)) {
    const float rd = qlim * rcp_approx(detq);
    const float hx = sqrt_approx(rd * cc) * 1.001f + 0.01f;
    const float hy = sqrt_approx(rd * ca) * 1.001f + 0.01f;
    box = make_float4(r0.x - hx, r0.x + hx, r0.y - hy, r0.y + hy);
  } else {
    box = make_float4(-INFINITY, INFINITY, -INFINITY, INFINITY);
  }
  s.box[j] = box;
}

// A list entry that names no pair of the plan (a list that pk_bin_and_sort
// did not write for this plan): staged as a splat that reaches no pixel.
constexpr uint32_t kNoPair = 0xffffffffu;   // never a pair index (pairs < 2^32 - 1)
__device__ __forceinline__ void stage_none(const Staged &s, int j) {
  s.a[j] = make_float4(0.f, 0.f, 0.f, 0.f);
  s.b[j] = make_float4(0.f, 0.f, 0.f, 0.f);
  s.c[j] = make_float4(0.f, __uint_as_float(kNoPair), INFINITY, 0.f);
  s.q[j] = make_float4(0.f, 0.f, 0.f, -1.f);
  s.box[j] = make_float4(1.f, -1.f, 1.f, -1.f);   // misses every block
}

__device__ __forceinline__ void stage_splat(const float *__restrict__ rec, uint32_t pid, uint32_t npairs,
                                            const Staged &s, int j, pk_device_status *status) {
  if (pid >= npairs) {
    stage_none(s, j);
    atomicOr(&status->flags, PK_DEV_BOUNDS);
    return;
  }
  const float4 *r = reinterpret_cast<const float4 *>(rec + (size_t)pid * kRec);
  stage_from(__ldg(r), __ldg(r + 1), __ldg(r + 2), pid, s, j);
}

// The exponent power = k q = A dx^2 + B dx dy + C dy^2 of a staged splat at
// two pixel centres of one column, two lanes at a time, from the per-splat
// terms zxdx = (A dx) dx and bdx = B dx of the column: power = (C dy + bdx)
// dy + zxdx, dy = py - m_y, each step rounded to nearest in this order,
// exactly the steps of splat_power below (the forward's scalar form), so the
// two kernels take identical skip and clamp decisions.  A pixel skips the
// splat unless power >= pcut; then alpha = min(0.99, o 2^power).
__device__ __forceinline__ f32x2 splat_power2(const float4 &a, const float4 &b, float bdx, float zxdx, f32x2 py,
                                              f32x2 &dy) {
  dy = sub2(py, dup2(a.y));
  return fma2(fma2(dup2(b.x), dy, dup2(bdx)), dy, dup2(zxdx));
}

// The same exponent at one pixel centre (the forward's scalar form): the
// steps and rounding of splat_power2, so the two kernels take identical
// skip and clamp decisions.
__device__ __forceinline__ float splat_power(const float4 &a, const float4 &b, float bdx, float zxdx, float py) {
  const float dy = __fsub_rn(py, a.y);
  return __fmaf_rn(__fmaf_rn(b.x, dy, bdx), dy, zxdx);
}

__device__ __forceinline__ bool box_misses(const float4 &box, float x0, float x1, float y0, float y1) {
  return box.x > x1 || box.y < x0 || box.z > y1 || box.w < y0;
}

// Can the staged splat pass both skip tests anywhere in the pixel-centre
// rectangle [x0, x1] x [y0, y1] of a warp's block?  First the box, then the
// least q over the rectangle (0 with the mean inside, else on an edge facing
// the mean, at the clamped 1-D minimiser) against qlim, with a relative
// 1e-3 + 1e-3 margin so rounding can only keep a splat, never drop one.
__device__ __forceinline__ bool block_may_hit(const float4 &box, const float4 &q, float mx, float my, float x0,
                                              float x1, float y0, float y1) {
  if (box_misses(box, x0, x1, y0, y1)) return false;
  const float a = q.x, b = q.y, c = q.z;
  if (!(a > 0.f) || !(c > 0.f)) return true;
  const bool inx = mx >= x0 && mx <= x1, iny = my >= y0 && my <= y1;
  if (inx && iny) return true;
  const float lx = x0 - mx, hx = x1 - mx, ly = y0 - my, hy = y1 - my;
  float best = INFINITY;
  if (!inx) {
    const float dx = mx < x0 ? lx : hx;
    const float dy = fminf(fmaxf(-__fdividef(b * dx, c), ly), hy);
    best = fminf(best, (a * dx + 2.f * b * dy) * dx + c * dy * dy);
  }
  if (!iny) {
    const float dy = my < y0 ? ly : hy;
    const float dx = fminf(fmaxf(-__fdividef(b * dy, a), lx), hx);
    best = fminf(best, (a * dx + 2.f * b * dy) * dx + c * dy * dy);
  }
  return best <= q.w * 1.001f + 1e-3f;
}

// ---------------------------------------------------------------------------
// Long lists.  One CTA walks its block's list in order, so a long list of a
// block that does not saturate (the rim of a dense cluster, a small view of
// many splats) is a serial chain of some 40 ns per entry on one CTA while the
// rest of the GPU has run dry: a 97 x 403 view of 34 K splats kept the
// forward and the backward for 1.5 and 2.0 ms, most of it one CTA.
//
// So once few CTAs are left of a pass of not too many work items, one that
// still has a long way to go in its list leaves the rest of it to kernels
// that spread one list over more of the GPU (k_raster_fwd_long, the backward's
// segments below).  While more of them run, lists are walked whole, which
// takes less work in all: the forward's other kernel spends about 2.4 times
// the instructions per entry, the backward's 1.4 times.  The lines lie at an
// eighth (forward) and a quarter (backward) of the resident CTAs: with the
// hand-over as soon as the tile queue is dry instead, 44 views of 195 x 195
// pixels on 253 K splats take 11.1 ms for 6.7 (whole lists: 9.2).
// And passes of more than kLongMostItems work items (1,000 per SM, 100 for each
// of the forward's resident CTAs at its usual batch) run without it: their
// tail is short, and the test in its loop costs the forward 2 % (52-view rig,
// 306 K items: 4.11 -> 4.20 ms; at 66 K items a 16-view step gains 13 %).  Nor
// do passes that count their evaluations.  The plan settles it (long_items),
// since its workspace holds the state.
constexpr int64_t kLongMostItems = int64_t(1000) * kSms;
__device__ __forceinline__ bool few_left(const RasterQueue *q, uint32_t few) {
  return gridDim.x - *reinterpret_cast<const volatile uint32_t *>(&q->exited) <= few;
}
// Entries walked and left: a hand-over costs about as much as 256; where there
// are many more work items than CTAs the last ones end at about the same
// time, and only a walk of 1,024 more is worth one.
__device__ __forceinline__ uint32_t long_least(uint32_t n_items) {
  return n_items <= 4u * gridDim.x ? 256u : 1024u;
}
// A launch that leaves most of the GPU idle from its start: lists of kTinyList
// entries and more go over before their first batch.
constexpr uint32_t kTinyList = 128;

// What the forward hands over: work item, entries walked (a multiple of every
// batch) and, per pixel (row-major in the block), colour sum and
// transmittance, and the last blended entry (bit 31: the pixel has stopped).
// w = kNoPair: a slot taken for a block that ended by itself.
struct LongItems {
  float4 *state;
  uint32_t *last, *w, *first;
  static size_t bytes(uint64_t slots) { return slots * (kSplitBlock * (sizeof(float4) + sizeof(uint32_t)) + 8); }
  static LongItems of(void *base, uint64_t slots) {
    LongItems l;
    l.state = static_cast<float4 *>(base);
    l.last = reinterpret_cast<uint32_t *>(l.state + slots * kSplitBlock);
    l.w = l.last + slots * kSplitBlock;
    l.first = l.w + slots;
    return l;
  }
};

// The backward's split lists: the rest of a long walk is cut into segments
// that other CTAs walk at the same time.  A segment's transmittance and
// colour behind follow from the later segments' products of (1 - alpha) and
// colour sums (compositing is associative), which a first pass over the
// segments takes.  (The forward keeps one rounding order whatever a list
// holds besides a pixel's contributors, so it does not cut its lists.)
// Segments of split_least entries at least (one batch; half a batch in a
// launch that leaves most of the GPU idle from its start), 64 of the first 128
// lists at most and 16 of the others, so that a pass's segments fill the GPU a
// few times over; all of about the same length, since the longest is the
// pass's time.
__device__ __forceinline__ uint32_t split_least(uint32_t few) { return gridDim.x <= few ? 64u : 128u; }
__device__ __forceinline__ uint32_t split_segments(uint32_t len, uint32_t least, uint32_t item) {
  return min(len / least, item < 128u ? 64u : 16u);
}

// A split list: work item w (tile and quadrant), its first unit (segment
// slot), segments of x entries (the last the rest of them), entries.
struct SplitItem {
  uint32_t w, unit0, nseg, x, len;
};

// Per unit and pixel of the block (row-major): tl = product of (1 - alpha)
// over the segment, ls = sum of alpha T dL/dC.rgb with T = 1 before it.  Per
// item and pixel: T and -dL/dC.(colour behind) at the end of its entries.
struct SplitBwd {
  float2 *state;
  float *tl, *ls;
  SplitItem *items;
  static size_t bytes(uint64_t items, uint64_t units) {
    return items * (sizeof(SplitItem) + kSplitBlock * sizeof(float2)) + units * kSplitBlock * 2 * sizeof(float);
  }
  static SplitBwd of(void *base, uint64_t items, uint64_t units) {
    SplitBwd s;
    s.state = static_cast<float2 *>(base);
    s.tl = reinterpret_cast<float *>(s.state + items * kSplitBlock);
    s.ls = s.tl + units * kSplitBlock;
    s.items = reinterpret_cast<SplitItem *>(s.ls + units * kSplitBlock);
    return s;
  }
};

// Enter the first `len` entries of a list as a split item; its index, or
// kNoPair when the slots are used up (the caller then walks on).  One thread.
__device__ __forceinline__ uint32_t split_enter(RasterQueue *q, SplitItem *items, uint32_t max_items, uint32_t units,
                                                uint32_t w, uint32_t len, uint32_t least) {
  const uint32_t i = atomicAdd(&q->items, 1u);
  if (i >= max_items) return kNoPair;
  const uint32_t n = split_segments(len, least, i), x = (len + n - 1u) / n, nseg = (len + x - 1u) / x;
  const uint32_t unit0 = atomicAdd(&q->units, nseg);
  const bool fits = unit0 < units && nseg <= units - unit0;
  items[i] = SplitItem{w, unit0, fits ? nseg : 0u, x, len};
  if (!fits) return kNoPair;
  atomicMax(&q->max_seg, nseg);
  return i;
}

// The next (item, segment) of queue k, segment `first` or later.  False when
// none is left.  One thread.
__device__ __forceinline__ bool split_next(RasterQueue *q, const SplitItem *items, uint32_t max_items, int k,
                                           uint32_t first, uint32_t &it, uint32_t &seg) {
  const uint32_t n = min(q->items, max_items), most = q->max_seg;
  if (n == 0 || most <= first) return false;
  const uint64_t total = (uint64_t)n * (most - first);
  for (;;) {
    const uint32_t v = atomicAdd(&q->seg_q[k], 1u);
    if (v >= total) return false;
    seg = first + v / n;
    it = v % n;
    if (seg < items[it].nseg) return true;
  }
}

// Bounds of a warp's pixel centres that satisfy `on` (any of the warp's
// pixels; the empty rectangle otherwise).
struct WarpRect {
  float x0, x1, y0, y1;
};
__device__ __forceinline__ WarpRect warp_rect(bool any, int x, int ylo, int yhi) {
  WarpRect r;
  r.x0 = (float)__reduce_min_sync(0xffffffffu, any ? x : 0x3fffffff) + 0.5f;
  r.x1 = (float)__reduce_max_sync(0xffffffffu, any ? x : -0x3fffffff) + 0.5f;
  r.y0 = (float)__reduce_min_sync(0xffffffffu, any ? ylo : 0x3fffffff) + 0.5f;
  r.y1 = (float)__reduce_max_sync(0xffffffffu, any ? yhi : -0x3fffffff) + 0.5f;
  return r;
}

}  // namespace pk
