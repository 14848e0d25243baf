// a4 -- front-to-back compositing (Supp. "Viewer": C = sum_i T_i a_i c_i,
// T_i = prod_{j<i} (1 - a_j)) over the depth-sorted list of each tile.
//
// One persistent launch covers the tiles of every view: each CTA takes the
// next tile from a device counter, stages the tile's splats batch by
// batch into shared memory and composites two pixels per thread.  Warps
// cover 8 x 8 pixel blocks and skip, as a whole, every splat whose
// contributing ellipse misses their block.  The CTA leaves a tile as soon
// as every pixel has stopped (transmittance cutoff) or the list ends.
#include "pk_raster.cuh"
#include "pk_tma.cuh"

using namespace pk;

namespace {

// kTma: the records of the next batch are fetched into shared memory by
// bulk copies (one 48-byte copy per splat, completed on an mbarrier) while
// the current batch is composited; the derived per-splat values are then
// computed from shared memory.  kPx: pixels per thread (Geo).
// At 2 pixels per thread the kernel is held to 48 registers (a few
// spilled) for 10 resident CTAs per SM instead of 9.
// kT: side of the tiles the lists were binned for (16 or 32); each CTA
// composites a 16 x 16 quadrant of one, walking the whole list of its tile
// (its warps' block tests skip what misses them), so a pixel still stops
// as soon as its own 16 x 16 block is done.
// With a target (not null) the epilogue also takes the L1 term of the
// objective: dL/dimage = sign(image - target) * scale and the sum of
// |image - target| (FP32 per thread, FP64 across warps) into loss_acc.
// kCount: count the (pixel, splat) evaluations into evals_out (a
// measurement; the variant without it carries no counter in its loop).
// kHand: once at most `few` CTAs are left, a block with a long way to go
// (long_least entries walked and left) goes on in k_raster_fwd_long.
// clr (may be null): clr_n4 float4 set to zero along the way, clr_per of
// them per work item -- the backward's gradient records, cleared by stores
// that ride along with the compositing instead of a pass of their own.
template <int kBatch, bool kTma, int kPx, int kT, bool kCount, bool kHand>
__global__ __launch_bounds__(Geo<kPx>::kThreads, (kPx == 2 ? 10 : 1)) void k_raster_fwd(
    const float *__restrict__ rec, const uint32_t *__restrict__ vals, const uint64_t *__restrict__ ranges,
    const DevView *__restrict__ views, const uint32_t *__restrict__ toff, int V, uint32_t n_items, float bg0,
    float bg1, float bg2, float *__restrict__ image, float *__restrict__ Tout, uint32_t *__restrict__ ncontrib,
    RasterQueue *rq, unsigned long long *evals_out, pk_device_status *status, const float *__restrict__ target,
    float *__restrict__ dimg, float scale, double *loss_acc, uint32_t first_polls, uint32_t npairs,
    float4 *__restrict__ clr, uint64_t clr_n4, uint64_t clr_per, LongItems longs, uint32_t long_items,
    uint32_t few) {
  using G = Geo<kPx>;
  constexpr uint32_t kQuads = (kT / kTileSide) * (kT / kTileSide);   // CTAs per list tile
  __shared__ float4 s_a[kBatch], s_b[kBatch], s_c[kBatch], s_box[kBatch], s_q[kBatch];
  __shared__ __align__(16) float4 s_raw[kTma ? 3 * kBatch : 1];
  __shared__ uint32_t s_pid[kTma ? kBatch : 1];
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_hand[2];   // long-list slot taken for this block's rest
  __shared__ int s_view;
  const int tid = threadIdx.x, lane = tid & 31;
  const Staged st{s_a, s_b, s_c, s_box, s_q};
  int ox, oy, bx, by;
  pixel_of<kPx>(tid, ox, oy, bx, by);
  uint32_t evals = 0;   // per thread: far below 2^32
  uint32_t phase = 0;
  bool timed_out = false;
  float lsum = 0.f;     // sum of |image - target| over this thread's pixels
  if (kTma) {
    if (tid == 0) {
      mbar_init(&s_bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
  }
  // bulk copies of the records of list entries [b, b + nb) into s_raw
  // (expect_tx is set by thread 0 before the block barrier that precedes this)
  auto fetch = [&](uint64_t b, int nb) {
    for (int j = tid; j < nb; j += G::kThreads) {
      const uint32_t pid = __ldg(vals + b + j);
      const bool named = pid < npairs;   // else record 0 is fetched in its place and not used
      s_pid[j] = named ? pid : kNoPair;
      tma_load_1d(&s_raw[3 * j], rec + (size_t)(named ? pid : 0u) * kRec, 3 * sizeof(float4), &s_bar);
    }
  };
  for (;;) {
    // work item: (list tile t, 16 x 16 quadrant q of it)
    if (tid == 0) {
      const uint32_t w = atomicAdd(&rq->tile, 1u);
      s_tile = w;
      s_view = w < n_items ? view_of_tile(toff, V, w / kQuads) : -1;
    }
    __syncthreads();
    const uint32_t w = s_tile;
    if (w >= n_items) break;
    if (clr) {   // this work item's share of the buffer to clear (every item takes one, so all of it is)
      const uint64_t c0 = (uint64_t)w * clr_per, c1 = min(clr_n4, c0 + clr_per);
      for (uint64_t i = c0 + tid; i < c1; i += G::kThreads) clr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const uint32_t t = w / kQuads, q = w - t * kQuads;
    const DevView &view = views[s_view];
    const int W = view.width, H = view.height;
    const uint32_t local = t - (uint32_t)view.tile_off;
    const int ty = (int)(local / (uint32_t)view.tiles_x), tx = (int)(local - (uint32_t)ty * view.tiles_x);
    const int X0 = tx * kT + (int)(q % (kT / kTileSide)) * kTileSide;
    const int Y0 = ty * kT + (int)(q / (kT / kTileSide)) * kTileSide;
    if (X0 >= W || Y0 >= H) {   // a quadrant past the view's edge
      __syncthreads();
      continue;
    }
    const int x = X0 + ox, y0 = Y0 + oy;
    const float px = (float)x + 0.5f, py0 = (float)y0 + 0.5f;
    // pixel-centre bounds of this warp's block
    const float wx0 = (float)(X0 + bx) + 0.5f, wx1 = wx0 + (float)(G::kBW - 1);
    const float wy0 = (float)(Y0 + by) + 0.5f, wy1 = wy0 + (float)(G::kBH - 1);
    const uint64_t s = __ldg(ranges + 2 * (size_t)t);
    uint64_t e = __ldg(ranges + 2 * (size_t)t + 1);
    uint32_t hand = kNoPair;   // long-list slot this block's rest went to
    if (kHand && gridDim.x <= 2u * few && e >= s + kTinyList) {
      if (tid == 0) {
        const uint32_t slot = atomicAdd(&rq->items, 1u);
        if (slot < long_items) {
          longs.w[slot] = w;
          longs.first[slot] = 0u;
        }
        s_hand[0] = slot;
      }
      __syncthreads();
      if (s_hand[0] < long_items) {
        hand = s_hand[0];
        e = s;   // no batch here
      }
    }
    float T[kPx], c0[kPx], c1[kPx], c2[kPx];
    uint32_t last[kPx];
    uint32_t live = 0;   // bit k: pixel k is inside the view and still compositing
#pragma unroll
    for (int k = 0; k < kPx; ++k) {
      T[k] = 1.f;
      c0[k] = c1[k] = c2[k] = 0.f;
      last[k] = 0;
      if (x < W && y0 + k * G::kRowStep < H) live |= 1u << k;
    }
    bool pending = false;   // a fetch is in flight (uniform over the block)
    if (kTma && s < e) {
      if (tid == 0) mbar_expect_tx(&s_bar, (uint32_t)min((uint64_t)kBatch, e - s) * 3u * sizeof(float4));
      __syncthreads();
      fetch(s, (int)min((uint64_t)kBatch, e - s));
      pending = true;
    }
    // plain loads: each thread's list entries of the next batch are read a
    // batch ahead, so staging waits for one load (the record) instead of two
    constexpr int kPer = (kBatch + G::kThreads - 1) / G::kThreads;
    uint32_t npid[kPer];
    if (!kTma) {
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int j = tid + u * G::kThreads;
        npid[u] = j < kBatch && s + j < e ? __ldg(vals + s + j) : 0u;
      }
    }
    for (uint64_t base = s; base < e; base += kBatch) {
      const int nb = (int)min((uint64_t)kBatch, e - base);
      // may this walk be handed over after this batch?  (every 256 entries)
      const uint32_t walked = (uint32_t)(base - s) + kBatch;
      const bool may_hand = kHand && (walked & 255u) == 0 && walked >= long_least(n_items) &&
                            (uint32_t)(e - s) >= walked + long_least(n_items);
      if (kTma) {
        if (!mbar_wait_bounded(&s_bar, phase, first_polls)) {
          timed_out = true;
          mbar_wait_bounded(&s_bar, phase);   // let this batch's copies land before leaving
        }
        phase ^= 1u;
        pending = false;
#pragma unroll
        for (int j = tid; j < kBatch; j += G::kThreads)
          if (j < nb) {
            if (s_pid[j] == kNoPair) {
              stage_none(st, j);
              atomicOr(&status->flags, PK_DEV_BOUNDS);
            } else {
              stage_from(s_raw[3 * j], s_raw[3 * j + 1], s_raw[3 * j + 2], s_pid[j], st, j);
            }
          }
        fence_proxy_async();   // these reads of s_raw before the next bulk writes into it
        const uint64_t nxt = base + kBatch;
        const int nbn = nxt < e ? (int)min((uint64_t)kBatch, e - nxt) : 0;
        if (tid == 0 && nbn > 0) mbar_expect_tx(&s_bar, (uint32_t)nbn * 3u * sizeof(float4));
        if (__syncthreads_or(timed_out)) {
          timed_out = true;
          break;
        }
        // a slot only for a batch that arrived: one taken before the barrier
        // above would go to the other kernel without its state
        if (may_hand && tid == 0) {
          const uint32_t slot = few_left(rq, few) ? atomicAdd(&rq->items, 1u) : kNoPair;
          if (slot < long_items) {
            longs.w[slot] = w;
            longs.first[slot] = walked;
          }
          s_hand[(walked >> 8) & 1u] = slot;
        }
        if (nbn > 0) {
          fetch(nxt, nbn);
          pending = true;
        }
      } else {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
          const int j = tid + u * G::kThreads;
          if (j < nb) stage_splat(rec, npid[u], npairs, st, j, status);
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
          const int j = tid + u * G::kThreads;
          const uint64_t nx = base + kBatch + (uint64_t)j;
          npid[u] = j < kBatch && nx < e ? __ldg(vals + nx) : 0u;
        }
        if (may_hand && tid == 0) {
          const uint32_t slot = few_left(rq, few) ? atomicAdd(&rq->items, 1u) : kNoPair;
          if (slot < long_items) {
            longs.w[slot] = w;
            longs.first[slot] = walked;
          }
          s_hand[(walked >> 8) & 1u] = slot;
        }
        __syncthreads();
      }
      if (__any_sync(0xffffffffu, live != 0)) {
        // which staged splats can reach this warp's block: one ballot per
        // 32 splats, then only the hits are visited
        uint32_t hits[kBatch / 32];
#pragma unroll
        for (int k = 0; k < kBatch / 32; ++k) {
          const int j = 32 * k + lane;
          hits[k] = __ballot_sync(0xffffffffu, j < nb && block_may_hit(s_box[j], s_q[j], s_a[j].x, s_a[j].y,
                                                                       wx0, wx1, wy0, wy1));
        }
        bool any_live = true;
#pragma unroll
        for (int k = 0; k < kBatch / 32; ++k) {
          uint32_t m = hits[k];
          while (m && any_live) {
            const int j = 32 * k + __ffs(m) - 1;
            m &= m - 1;
            const float4 a = s_a[j], b = s_b[j], c = s_c[j];
            const float dx = __fsub_rn(px, a.x);
            const float zxdx = __fmul_rn(__fmul_rn(a.z, dx), dx), bdx = __fmul_rn(a.w, dx);
            const uint32_t pos1 = (uint32_t)(base - s) + (uint32_t)j + 1u;   // within the tile's list
            if (kCount) evals += __popc(live);   // evaluated at every live pixel of the thread
#pragma unroll
            for (int q = 0; q < kPx; ++q) {
              // one test per pixel: still compositing, and power >= pcut (both
              // q <= 9 and alpha >= 1/255); alpha = min(0.99, o 2^power)
              const float power = splat_power(a, b, bdx, zxdx, py0 + (float)(q * G::kRowStep));
              if (((live >> q) & 1u) && power >= c.z) {
                const float araw = __fmul_rn(-b.y, ex2_approx(power));   // staged opacity is negated
                const float alpha = araw > kAlphaMax ? kAlphaMax : araw;
                const float Tn = __fmul_rn(T[q], __fsub_rn(1.f, alpha));
                if (Tn < kTMin) {
                  live &= ~(1u << q);
                } else {
                  const float w = __fmul_rn(alpha, T[q]);
                  c0[q] = __fmaf_rn(w, b.z, c0[q]);
                  c1[q] = __fmaf_rn(w, b.w, c1[q]);
                  c2[q] = __fmaf_rn(w, c.x, c2[q]);
                  T[q] = Tn;
                  last[q] = pos1;
                }
              }
            }
            any_live = __any_sync(0xffffffffu, live != 0);
          }
        }
      }
      const bool done = __syncthreads_count(live != 0) == 0;
      // (two words in turn: one is not written again before the next batch's barrier)
      if (may_hand && s_hand[(walked >> 8) & 1u] < long_items) {
        hand = s_hand[(walked >> 8) & 1u];
        if (done) {
          if (tid == 0) longs.w[hand] = kNoPair;
          hand = kNoPair;
        }
        break;
      }
      if (done) break;
    }
    if (hand != kNoPair) {
#pragma unroll
      for (int k = 0; k < kPx; ++k) {
        const size_t at = (size_t)hand * kSplitBlock + (oy + k * G::kRowStep) * kTileSide + ox;
        longs.state[at] = make_float4(c0[k], c1[k], c2[k], T[k]);
        longs.last[at] = last[k] | ((live >> k) & 1u ? 0u : 0x80000000u);
      }
    }
    if (kTma) {
      // a tile that stopped early may still have its next batch in flight
      if (pending) {
        if (!mbar_wait_bounded(&s_bar, phase)) {
          timed_out = true;
          mbar_wait_bounded(&s_bar, phase);
        }
        phase ^= 1u;
      }
      if (__syncthreads_or(timed_out)) {
        if (tid == 0) atomicOr(&status->flags, PK_DEV_TIMEOUT);
        break;
      }
    }
    const size_t plane = (size_t)W * H;
#pragma unroll
    for (int q = 0; q < kPx; ++q) {
      const int y = y0 + q * G::kRowStep;
      if (hand == kNoPair && x < W && y < H) {
        const size_t pix = (size_t)view.pix_off + (size_t)y * W + x;
        const size_t at0 = 3 * (size_t)view.pix_off + (size_t)y * W + x;
        const float v0 = __fmaf_rn(T[q], bg0, c0[q]), v1 = __fmaf_rn(T[q], bg1, c1[q]);
        const float v2 = __fmaf_rn(T[q], bg2, c2[q]);
        image[at0] = v0;
        image[at0 + plane] = v1;
        image[at0 + 2 * plane] = v2;
        Tout[pix] = T[q];
        ncontrib[pix] = last[q];
        if (target) {
          const float vs[3] = {v0, v1, v2};
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float d = vs[c] - __ldcs(target + at0 + c * plane);
            lsum += fabsf(d);
            __stcs(dimg + at0 + c * plane, d > 0.f ? scale : (d < 0.f ? -scale : 0.f));
          }
        }
      }
    }
    __syncthreads();   // everyone has read s_tile / s_view before the next fetch
  }
  if (kHand && tid == 0) atomicAdd(&rq->exited, 1u);
  // one atomic per warp for the evaluation counter (and the loss)
  if (kCount) {
    unsigned long long ev = evals;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ev += __shfl_xor_sync(0xffffffffu, ev, o);
    if (lane == 0 && ev) atomicAdd(evals_out, ev);
  }
  if (target) {
    double dl = (double)lsum;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    if (lane == 0 && dl != 0.0) atomicAdd(loss_acc, dl);
  }
}

// Long lists: a CTA per 8 x 8 pixel block of a handed-over work item takes
// its list up where k_raster_fwd left it.  What has to
// run in list order is short -- per blended entry a subtraction, two products
// and three multiply-adds -- so two warps do only that, one pixel per lane,
// while eight others work a batch ahead: they stage the batch's splats, keep
// those that can reach the block's live pixels and evaluate alpha for all its
// pixels, which the two warps then read.  The same operations in the same
// order as k_raster_fwd's, so the same bits.  A walk costs about 7 ns per
// entry where one warp doing all of it takes 40 (each instruction of a
// visit waits for the last, with nothing else on its scheduler): the forward
// of the 97 x 403 view among three takes 1,490 -> 310 us.
constexpr int kLongBatch = 128;
constexpr int kLongProducers = 256;
constexpr int kLongThreads = 64 + kLongProducers;
constexpr float kNoBlend = -INFINITY;   // alpha of a pixel that skips the splat
struct LongSmem {
  float4 a[kLongBatch], b[kLongBatch], c[kLongBatch], box[kLongBatch], q[kLongBatch];
  float4 col[2][kLongBatch];        // red, green, blue, list position + 1 (bits) of each kept splat
  float alpha[2][kLongBatch][64];
  uint32_t hit[kLongBatch];         // kept splats in list order
};

template <int kT>
__global__ __launch_bounds__(kLongThreads, 2) void k_raster_fwd_long(
    const float *__restrict__ rec, const uint32_t *__restrict__ vals, const uint64_t *__restrict__ ranges,
    const DevView *__restrict__ views, const uint32_t *__restrict__ toff, int V, float bg0, float bg1, float bg2,
    float *__restrict__ image, float *__restrict__ Tout, uint32_t *__restrict__ ncontrib, RasterQueue *rq,
    pk_device_status *status, const float *__restrict__ target, float *__restrict__ dimg, float scale,
    double *loss_acc, uint32_t npairs, LongItems longs, uint32_t long_items) {
  constexpr uint32_t kQuads = (kT / kTileSide) * (kT / kTileSide);
  extern __shared__ __align__(16) unsigned char s_raw[];
  LongSmem &S = *reinterpret_cast<LongSmem *>(s_raw);
  __shared__ uint32_t s_unit, s_nhit[2], s_mask[kLongBatch / 32];
  __shared__ int s_view, s_rect[2][2][4];   // [iteration parity][warp]: live pixels' x0, x1, y0, y1 in the block
  const int tid = threadIdx.x, lane = tid & 31;
  const bool consumer = tid < 64;
  const int pt = tid - 64, pw = pt >> 5;    // producer thread and warp
  const Staged st{S.a, S.b, S.c, S.box, S.q};
  float lsum = 0.f;
  for (;;) {
    if (tid == 0) {
      const uint32_t u = atomicAdd(&rq->seg_q[0], 1u);
      s_view = -1;
      if (u < 4u * min(rq->items, long_items)) {
        s_unit = u;
        const uint32_t w = longs.w[u >> 2];
        s_view = w == kNoPair ? V : view_of_tile(toff, V, w / kQuads);
      }
    }
    __syncthreads();
    if (s_view < 0) break;
    if (s_view == V) {
      __syncthreads();   // everyone has read s_view before the next unit
      continue;
    }
    const uint32_t w = longs.w[s_unit >> 2], blk = s_unit & 3u;
    const uint32_t t = w / kQuads, qd = w - t * kQuads;
    const DevView &view = views[s_view];
    const int W = view.width, H = view.height;
    const uint32_t local = t - (uint32_t)view.tile_off;
    const int ty = (int)(local / (uint32_t)view.tiles_x), tx = (int)(local - (uint32_t)ty * view.tiles_x);
    const int X0 = tx * kT + (int)(qd % (kT / kTileSide)) * kTileSide + (int)(blk & 1u) * 8;
    const int Y0 = ty * kT + (int)(qd / (kT / kTileSide)) * kTileSide + (int)(blk >> 1) * 8;
    if (X0 >= W || Y0 >= H) {
      __syncthreads();   // everyone has read s_unit / s_view before the next unit
      continue;
    }
    const uint32_t first = longs.first[s_unit >> 2];   // entries walked before the hand-over
    const uint64_t s = __ldg(ranges + 2 * (size_t)t) + first;
    const uint32_t len = (uint32_t)(__ldg(ranges + 2 * (size_t)t + 1) - s);
    const uint32_t nbatch = (len + kLongBatch - 1) / kLongBatch;
    // consumer: pixel tid of the block, row-major
    const int x = X0 + (tid & 7), y = Y0 + ((tid >> 3) & 7);
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    uint32_t last = 0;
    bool live = false;
    if (consumer) {
      const size_t at = (size_t)(s_unit >> 2) * kSplitBlock + ((blk >> 1) * 8u + (uint32_t)(tid >> 3)) * kTileSide +
                        (blk & 1u) * 8u + (uint32_t)(tid & 7);
      const float4 v = longs.state[at];
      last = longs.last[at];
      c0 = v.x;
      c1 = v.y;
      c2 = v.z;
      T = v.w;
      live = (last >> 31) == 0u;
      last &= 0x7fffffffu;
    }
    auto note_rect = [&](int par) {
      const int rx = tid & 7, ry = (tid >> 3) & 7;
      const int x0 = __reduce_min_sync(0xffffffffu, live ? rx : 99), x1 = __reduce_max_sync(0xffffffffu, live ? rx : -99);
      const int y0 = __reduce_min_sync(0xffffffffu, live ? ry : 99), y1 = __reduce_max_sync(0xffffffffu, live ? ry : -99);
      if (lane == 0) {
        int *r = s_rect[par][tid >> 5];
        r[0] = x0;
        r[1] = x1;
        r[2] = y0;
        r[3] = y1;
      }
    };
    // producer: this thread's entry of the next batch, its record a batch
    // ahead and its list entry two
    const bool stager = !consumer && pt < kLongBatch;
    uint32_t pid = kNoPair, npid = kNoPair;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0, r2 = r0;
    auto entry = [&](uint32_t b) -> uint32_t {
      const uint32_t i = b * kLongBatch + (uint32_t)pt;
      return i < len ? __ldg(vals + s + i) : kNoPair;
    };
    auto record = [&](uint32_t p) {
      if (p < npairs) {
        const float4 *r = reinterpret_cast<const float4 *>(rec + (size_t)p * kRec);
        r0 = __ldg(r);
        r1 = __ldg(r + 1);
        r2 = __ldg(r + 2);
      }
    };
    if (stager) {
      pid = entry(0);
      record(pid);
      npid = entry(1);
    }
    if (consumer) note_rect(1);
    const float px = (float)(X0 + (lane & 7)) + 0.5f, py = (float)(Y0 + (lane >> 3)) + 0.5f;   // producer's pixels
    __syncthreads();
    // iteration i: the producers prepare batch i, the consumers blend batch i - 1
    for (uint32_t i = 0; i <= nbatch; ++i) {
      const int cur = (int)(i & 1u), prev = cur ^ 1;
      const int *ra = s_rect[prev][0], *rb = s_rect[prev][1];
      const int lx0 = min(ra[0], rb[0]), lx1 = max(ra[1], rb[1]), ly0 = min(ra[2], rb[2]), ly1 = max(ra[3], rb[3]);
      if (lx0 > lx1) break;   // every pixel has stopped (uniform: read after the last barrier)
      if (consumer) {
        if (i > 0) {
          const uint32_t nh = s_nhit[prev];
          const float *al = &S.alpha[prev][0][tid];
#pragma unroll 4
          for (uint32_t h = 0; h < nh; ++h) {
            const float alpha = al[64 * h];
            const float4 col = S.col[prev][h];
            if (live && alpha != kNoBlend) {
              const float Tn = __fmul_rn(T, __fsub_rn(1.f, alpha));
              if (Tn < kTMin) {
                live = false;
              } else {
                const float wt = __fmul_rn(alpha, T);
                c0 = __fmaf_rn(wt, col.x, c0);
                c1 = __fmaf_rn(wt, col.y, c1);
                c2 = __fmaf_rn(wt, col.z, c2);
                T = Tn;
                last = __float_as_uint(col.w);
              }
            }
          }
        }
        note_rect(cur);
      } else if (i < nbatch) {
        const uint32_t base = i * kLongBatch, nb = min((uint32_t)kLongBatch, len - base);
        bool hit = false;
        if (stager) {
          if ((uint32_t)pt < nb) {
            if (pid < npairs) {
              stage_from(r0, r1, r2, pid, st, pt);
            } else {
              stage_none(st, pt);
              atomicOr(&status->flags, PK_DEV_BOUNDS);
            }
            hit = block_may_hit(S.box[pt], S.q[pt], S.a[pt].x, S.a[pt].y, (float)(X0 + lx0) + 0.5f,
                                (float)(X0 + lx1) + 0.5f, (float)(Y0 + ly0) + 0.5f, (float)(Y0 + ly1) + 0.5f);
          }
          pid = npid;
          record(pid);
          npid = entry(i + 2);
          const uint32_t m = __ballot_sync(0xffffffffu, hit);
          if (lane == 0) s_mask[pw] = m;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kLongProducers) : "memory");
        uint32_t nh = 0, before = 0;
#pragma unroll
        for (int k = 0; k < kLongBatch / 32; ++k) {
          const uint32_t m = s_mask[k];
          if (k < pw) before += __popc(m);
          nh += __popc(m);
        }
        if (hit) {
          const uint32_t h = before + __popc(s_mask[pw] & ((1u << lane) - 1u));
          S.hit[h] = (uint32_t)pt;
          const float4 b = S.b[pt];
          S.col[cur][h] = make_float4(b.z, b.w, S.c[pt].x, __uint_as_float(first + base + (uint32_t)pt + 1u));
        }
        if (pt == 0) s_nhit[cur] = nh;
        asm volatile("bar.sync 1, %0;" ::"n"(kLongProducers) : "memory");
#pragma unroll 2
        for (uint32_t h = pw; h < nh; h += kLongProducers / 32) {
          const uint32_t j = S.hit[h];
          const float4 a = S.a[j], b = S.b[j];
          const float pcut = S.c[j].z;
          const float dx = __fsub_rn(px, a.x);
          const float zxdx = __fmul_rn(__fmul_rn(a.z, dx), dx), bdx = __fmul_rn(a.w, dx);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const float power = splat_power(a, b, bdx, zxdx, py + 4.f * (float)q);
            const float araw = __fmul_rn(-b.y, ex2_approx(power));
            const float alpha = araw > kAlphaMax ? kAlphaMax : araw;
            S.alpha[cur][h][lane + 32 * q] = power >= pcut ? alpha : kNoBlend;
          }
        }
      }
      __syncthreads();
    }
    if (consumer && x < W && y < H) {
      const size_t plane = (size_t)W * H;
      const size_t pix = (size_t)view.pix_off + (size_t)y * W + x;
      const size_t at0 = 3 * (size_t)view.pix_off + (size_t)y * W + x;
      const float vs[3] = {__fmaf_rn(T, bg0, c0), __fmaf_rn(T, bg1, c1), __fmaf_rn(T, bg2, c2)};
#pragma unroll
      for (int c = 0; c < 3; ++c) image[at0 + c * plane] = vs[c];
      Tout[pix] = T;
      ncontrib[pix] = last;
      if (target) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float d = vs[c] - __ldcs(target + at0 + c * plane);
          lsum += fabsf(d);
          __stcs(dimg + at0 + c * plane, d > 0.f ? scale : (d < 0.f ? -scale : 0.f));
        }
      }
    }
    __syncthreads();   // everyone is done with this unit's shared state
  }
  if (target && consumer) {
    double dl = (double)lsum;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    if (lane == 0 && dl != 0.0) atomicAdd(loss_acc, dl);
  }
}

// One persistent launch: as many CTAs as fit on the GPU, at most one per tile.
template <int kBatch, bool kFwdTma, int kT, bool kCount, bool kHand>
pk_status launch_fwd(const pk_plan *p, const float *records, const uint32_t *sorted_vals,
                     const uint64_t *tile_ranges, float *image, float *T_final, uint32_t *n_contrib, void *ws,
                     DevCounters *ctr, pk_device_status *status, const float *target, float *dimg, float *clear,
                     uint64_t clear_floats, cudaStream_t st) {
  static KernelInfo info;
  const int sms = sm_count();
  const auto kernel = k_raster_fwd<kBatch, kFwdTma, kFwdPx, kT, kCount, kHand>;
  const int per_sm = std::max(1, resident_ctas(info, reinterpret_cast<const void *>(kernel), Geo<kFwdPx>::kThreads, 0));
  const int64_t items = p->n_tiles * (kT / kTileSide) * (kT / kTileSide);
  int64_t grid = (int64_t)sms * per_sm;
  if (grid > items) grid = items;
  if (grid < 1) grid = 1;
  const uint64_t clr_n4 = clear ? clear_floats / 4 : 0;
  const uint64_t clr_per = items > 0 ? (clr_n4 + (uint64_t)items - 1) / (uint64_t)items : 0;
  k_raster_fwd<kBatch, kFwdTma, kFwdPx, kT, kCount, kHand><<<(int)grid, Geo<kFwdPx>::kThreads, 0, st>>>(
      records, sorted_vals, tile_ranges, at<DevView>(ws, p->ws.views), at<uint32_t>(ws, p->ws.toff), p->V,
      (uint32_t)items, p->opts.bg[0], p->opts.bg[1], p->opts.bg[2], image, T_final, n_contrib,
      &ctr->raster[0], reinterpret_cast<unsigned long long *>(&status->evals_fwd), status, target, dimg,
      (float)(1.0 / (3.0 * (double)std::max<int64_t>(1, p->P))), &ctr->loss_acc, p->first_polls, (uint32_t)p->pairs,
      reinterpret_cast<float4 *>(clr_n4 ? clear : nullptr), clr_n4, clr_per,
      LongItems::of(at<char>(ws, p->ws.longs), p->long_items), p->long_items,
      std::min<uint32_t>(p->long_items, (uint32_t)(sms * per_sm / 8)));
  if (kHand) {
    static KernelInfo long_info;
    const auto long_kernel = k_raster_fwd_long<kT>;
    if (resident_ctas(long_info, reinterpret_cast<const void *>(long_kernel), kLongThreads, sizeof(LongSmem)) == 0)
      return PK_ERR_CUDA;
    k_raster_fwd_long<kT><<<(int)std::min<int64_t>(2 * sms, 4 * (int64_t)p->long_items), kLongThreads, sizeof(LongSmem), st>>>(
        records, sorted_vals, tile_ranges, at<DevView>(ws, p->ws.views), at<uint32_t>(ws, p->ws.toff), p->V,
        p->opts.bg[0], p->opts.bg[1], p->opts.bg[2], image, T_final, n_contrib, &ctr->raster[0], status, target, dimg,
        (float)(1.0 / (3.0 * (double)std::max<int64_t>(1, p->P))), &ctr->loss_acc, (uint32_t)p->pairs,
        LongItems::of(at<char>(ws, p->ws.longs), p->long_items), p->long_items);
  }
  return check_launch();
}

pk_status rasterize_fwd(const pk_plan *p, const float *records, const uint32_t *sorted_vals,
                        const uint64_t *tile_ranges, const float *target, float *image, float *T_final,
                        uint32_t *n_contrib, float *dimg, float *clear, uint64_t clear_floats, void *ws,
                        cudaStream_t st) {
  DevCounters *ctr = at<DevCounters>(ws, p->ws.counters);
  pk_device_status *status = at<pk_device_status>(ws, p->ws.status);
  // the work counters, the evaluation counter and, with a target, loss_acc,
  // ssim_acc and ssim_lambda (0: the loss is L1 alone)
  pk_status ze = zero_async({{&ctr->raster[0], sizeof(RasterQueue)},
                             {&status->evals_fwd, sizeof(uint64_t)},
                             {&ctr->loss_acc, target ? 2 * sizeof(double) + sizeof(float) : 0}},
                            st);
  if (ze != PK_OK) return ze;
  const bool hand = p->long_items > 0;
#define PK_FWD_T(B, M, C, H)                                                                                     \
  return p->T == 32 ? launch_fwd<B, M, 32, C, H>(p, records, sorted_vals, tile_ranges, image, T_final, n_contrib, \
                                                 ws, ctr, status, target, dimg, clear, clear_floats, st)           \
                    : launch_fwd<B, M, 16, C, H>(p, records, sorted_vals, tile_ranges, image, T_final, n_contrib, \
                                                 ws, ctr, status, target, dimg, clear, clear_floats, st)
#define PK_FWD(B, M)             \
  {                              \
    if (p->opts.count_evals) {   \
      PK_FWD_T(B, M, true, false); \
    }                            \
    if (hand) {                  \
      PK_FWD_T(B, M, false, true); \
    }                            \
    PK_FWD_T(B, M, false, false); \
  }
  const bool tma = p->opts.stage_fwd == PK_STAGE_BULK;
  switch (p->opts.batch) {
    case 64:
      if (tma) PK_FWD(64, true);
      PK_FWD(64, false);
    case 128:
      if (tma) PK_FWD(128, true);
      PK_FWD(128, false);
    default:
      if (tma) PK_FWD(256, true);
      PK_FWD(256, false);
  }
#undef PK_FWD
#undef PK_FWD_T
}

}  // namespace

extern "C" pk_status pk_rasterize_fwd(const pk_plan *p, const float *records, const uint32_t *sorted_vals,
                                      const uint64_t *tile_ranges, float *image, float *T_final, uint32_t *n_contrib,
                                      void *ws, pk_stream_t stream) {
  if (!p || !records || !sorted_vals || !tile_ranges || !image || !T_final || !n_contrib || !ws) return PK_ERR_ARG;
  if (!aligned16(records) || (reinterpret_cast<uintptr_t>(tile_ranges) & 7u)) return PK_ERR_ARG;
  return rasterize_fwd(p, records, sorted_vals, tile_ranges, nullptr, image, T_final, n_contrib, nullptr, nullptr, 0,
                       ws, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" pk_status pk_rasterize_fwd_l1(const pk_plan *p, const float *records, const uint32_t *sorted_vals,
                                         const uint64_t *tile_ranges, const float *target, float *image,
                                         float *T_final, uint32_t *n_contrib, float *dL_dimage, void *ws,
                                         pk_stream_t stream) {
  if (!p || !records || !sorted_vals || !tile_ranges || !target || !image || !T_final || !n_contrib ||
      !dL_dimage || !ws)
    return PK_ERR_ARG;
  if (!aligned16(records) || (reinterpret_cast<uintptr_t>(tile_ranges) & 7u)) return PK_ERR_ARG;
  return rasterize_fwd(p, records, sorted_vals, tile_ranges, target, image, T_final, n_contrib, dL_dimage, nullptr,
                       0, ws, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" pk_status pk_rasterize_fwd_l1_clear(const pk_plan *p, const float *records, const uint32_t *sorted_vals,
                                               const uint64_t *tile_ranges, const float *target, float *image,
                                               float *T_final, uint32_t *n_contrib, float *dL_dimage,
                                               float *grad2d, void *ws, pk_stream_t stream) {
  if (!p || !records || !sorted_vals || !tile_ranges || !target || !image || !T_final || !n_contrib ||
      !dL_dimage || !grad2d || !ws)
    return PK_ERR_ARG;
  if (!aligned16(records) || !aligned16(grad2d) || (reinterpret_cast<uintptr_t>(tile_ranges) & 7u))
    return PK_ERR_ARG;
  return rasterize_fwd(p, records, sorted_vals, tile_ranges, target, image, T_final, n_contrib, dL_dimage, grad2d,
                       (uint64_t)kG2d * (uint64_t)p->pairs, ws, reinterpret_cast<cudaStream_t>(stream));
}
