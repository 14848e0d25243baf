// a1 -- atlas gather (Sec. 4.2 "Fitting UV Maps Directly"; FP16 proxy of
// "Low Precision Optimization").  Live texels of the occupancy mask, in
// row-major order, become the Gaussians 0..N-1 of every frame.
//
// Two kernels: a scan of the per-word popcounts, then one thread per group
// of four texels that reads each channel with one 16-byte (FP32) or 8-byte
// (FP16) load and writes the live ones to the channel-major SoA.
#include <cuda_fp16.h>

#include "pk_common.cuh"
#include "pk_lpo.cuh"

using namespace pk;

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanMaxBlocks = 64;

// woff[i] = number of live texels in mask words [0, i); woff[nwords] = total.
// Block b scans words [b per, (b + 1) per), per a multiple of 1024 so that
// at most kScanMaxBlocks blocks are needed.  It first counts the live texels
// of all words before its own (16-byte loads; they are L2 hits, and at most
// 64 blocks read them), so no block waits for another: one launch of a few
// microseconds where one block walking the whole mask took 11 us at 32 K
// words.
__device__ __forceinline__ uint32_t block_sum(uint32_t v, uint32_t *s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = __reduce_add_sync(0xffffffffu, v);
  if (lane == 0) s[warp] = v;
  __syncthreads();
  v = __reduce_add_sync(0xffffffffu, s[lane]);
  __syncthreads();
  return v;
}

__global__ __launch_bounds__(kScanThreads) void k_word_scan(const uint32_t *__restrict__ occ, int64_t nwords,
                                                            int64_t per, uint32_t *__restrict__ woff,
                                                            pk_device_status *status, int64_t N) {
  __shared__ uint32_t s_warp[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t w0 = (int64_t)blockIdx.x * per, w1 = min(nwords, w0 + per);
  // live texels before this block (w0 is a multiple of 1024)
  uint32_t before = 0;
  if ((reinterpret_cast<uintptr_t>(occ) & 15u) == 0) {
    const uint4 *q = reinterpret_cast<const uint4 *>(occ);
#pragma unroll 4
    for (int64_t i = tid; i < w0 / 4; i += kScanThreads) {
      const uint4 v = __ldg(q + i);
      before += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
    }
  } else {
    for (int64_t i = tid; i < w0; i += kScanThreads) before += __popc(__ldg(occ + i));
  }
  uint32_t carry = block_sum(before, s_warp);
  for (int64_t base = w0; base < w1; base += kScanThreads) {
    const int64_t i = base + tid;
    const uint32_t c = i < w1 ? __popc(__ldg(occ + i)) : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t w = s_warp[lane];   // every warp scans the 32 warp totals
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    const uint32_t mine = __shfl_sync(0xffffffffu, w, (warp + 31) & 31), total = __shfl_sync(0xffffffffu, w, 31);
    if (i < w1) woff[i] = carry + (warp ? mine : 0u) + x - c;
    carry += total;
    __syncthreads();   // before the next chunk's warp totals
  }
  if (w1 == nwords && tid == 0) {   // the last block: the whole mask's count
    woff[nwords] = carry;
    status->live_seen = carry;
    status->nonfinite = 0;   // counted by the gather kernel that follows
    if ((int64_t)carry != N) atomicOr(&status->flags, PK_DEV_LIVE_MISMATCH);
  }
}

void launch_word_scan(const uint32_t *occ, int64_t nwords, uint32_t *woff, pk_device_status *status, int64_t N,
                      cudaStream_t st) {
  int64_t per = (nwords + kScanMaxBlocks - 1) / kScanMaxBlocks;
  per = (per + kScanThreads - 1) / kScanThreads * kScanThreads;
  if (per < kScanThreads) per = kScanThreads;
  const unsigned blocks = (unsigned)((nwords + per - 1) / per);
  k_word_scan<<<blocks ? blocks : 1u, kScanThreads, 0, st>>>(occ, nwords, per, woff, status, N);
}

template <typename Tex>
struct Quad;
template <>
struct Quad<float> {
  using V = float4;
  __device__ static float get(const V &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
  __device__ static float one(const float *p) { return *p; }
};
template <>
struct Quad<__half> {
  using V = uint2;
  __device__ static float get(const V &v, int i) {
    uint32_t w = (i < 2) ? v.x : v.y;
    unsigned short h = (i & 1) ? (unsigned short)(w >> 16) : (unsigned short)(w & 0xffffu);
    return __half2float(__ushort_as_half(h));
  }
  __device__ static float one(const __half *p) { return __half2float(*p); }
};

// The live ones among the (up to) four texels x0 .. x0 + 3 of row y (bit i:
// texel i), whose Gaussians are consecutive from `first`; with `write`,
// writes their texel ids and dynamic flags.
__device__ __forceinline__ uint32_t quad_live(const uint32_t *__restrict__ occ, const uint32_t *__restrict__ dyn,
                                              const uint32_t *__restrict__ woff, int W, int y, int x0, int64_t N,
                                              bool write, uint32_t *__restrict__ texel,
                                              uint8_t *__restrict__ dynflag, int64_t &first) {
  const int64_t w = (int64_t)y * ((W + 31) / 32) + (x0 >> 5);   // one word: x0 is a multiple of 4
  const uint32_t word = occ[w];
  uint32_t live = (word >> (x0 & 31)) & 15u;
  if (x0 + 4 > W) live &= (1u << (W - x0)) - 1u;
  first = woff[w] + __popc(word & ((1u << (x0 & 31)) - 1u));
  int64_t g = first;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!((live >> i) & 1u)) continue;
    if (g >= N) {
      live &= ~(1u << i);
    } else if (write) {
      texel[g] = (uint32_t)((int64_t)y * W + x0 + i);
      dynflag[g] = dyn ? (uint8_t)((dyn[w] >> ((x0 & 31) + i)) & 1u) : (uint8_t)1;
    }
    ++g;
  }
  return live;
}

// The live ones of a group's four values, in order from dst.
__device__ __forceinline__ void store_live(const float (&x)[4], uint32_t live, float *__restrict__ dst) {
  const uint32_t r1 = live & 1u, r2 = r1 + ((live >> 1) & 1u), r3 = r2 + ((live >> 2) & 1u);
  if (live & 1u) dst[0] = x[0];
  if (live & 2u) dst[r1] = x[1];
  if (live & 4u) dst[r2] = x[2];
  if (live & 8u) dst[r3] = x[3];
}

// One thread per 4 consecutive texels of a row.  Loads in flight bound it: a
// group's Gaussians are consecutive, so one pointer per channel and four small
// offsets replace four 64-bit indices (128 registers, two CTAs per SM), and
// three CTAs fit.  1024^2 atlas, 60 % live, 59 channels: FP32 90 -> 77 us
// (395 MB of planes and SoA, 5.1 TB/s), three-level FP16 142 -> 81 us; with
// four CTAs 74 us but the 512^2 atlas 24 -> 29 us.  A warp that puts its
// values in order in shared memory to store whole rows of 32 takes 130 us.
template <typename Tex, bool kVec>
__global__ __launch_bounds__(256, 3) void k_gather(const Tex *__restrict__ atlas, const uint32_t *__restrict__ occ,
                                                   const uint32_t *__restrict__ dyn,
                                                   const uint32_t *__restrict__ woff, int W, int H, int F, int D,
                                                   int64_t N, float *__restrict__ soa, uint32_t *__restrict__ texel,
                                                   uint8_t *__restrict__ dynflag, pk_device_status *status) {
  const int Wq = (W + 3) / 4;
  uint32_t nbad = 0;   // (frame, Gaussian) pairs of this thread with a non-finite texel value
  const int64_t nq = (int64_t)Wq * H;
  const int64_t plane = (int64_t)W * H;
  const int64_t G = (int64_t)F * N;
  for (int64_t qi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; qi < nq; qi += (int64_t)gridDim.x * blockDim.x) {
    const int y = (int)(qi / Wq), x0 = (int)(qi % Wq) * 4;
    int64_t first;
    const uint32_t live = quad_live(occ, dyn, woff, W, y, x0, N, true, texel, dynflag, first);
    if (!live) continue;
    const int64_t pix = (int64_t)y * W + x0;
    for (int f = 0; f < F; ++f) {
      uint32_t bad = 0;   // bit i: texel i has a non-finite value in some channel of frame f
      const Tex *src = atlas + (int64_t)f * D * plane + pix;
      float *dst = soa + (int64_t)f * N + first;
#pragma unroll 4
      for (int c = 0; c < D; ++c, src += plane, dst += G) {
        float x[4];
        if (kVec) {
          const typename Quad<Tex>::V v = __ldg(reinterpret_cast<const typename Quad<Tex>::V *>(src));
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = Quad<Tex>::get(v, i);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = (live >> i) & 1u ? Quad<Tex>::one(src + i) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) bad |= (uint32_t)!isfinite(x[i]) << i;
        store_live(x, live, dst);
      }
      nbad += __popc(bad & live);
    }
  }
  // one atomic per warp
  const uint32_t wbad = __reduce_add_sync(0xffffffffu, nbad);
  if ((threadIdx.x & 31) == 0 && wbad) atomicAdd(reinterpret_cast<unsigned long long *>(&status->nonfinite), wbad);
}

// Low-precision proxy (Sec. 4.2 "Low Precision Optimization"): channel c
// quantised to 16 (position) or 8 bits over [lo_c, hi_c], read either as
// codes ([F][D + 3][H][W] bytes, position as high and low byte planes) or
// by fake-quantising the FP32 masters on the fly.  FP32 steps in the order
// packuv.h states, without fused multiply-adds.
__device__ __forceinline__ float lpo_proxy(uint32_t q, float lo, float delta) {
  return __fadd_rn(lo, __fmul_rn((float)q, delta));
}

// One thread per 4 consecutive texels of a row and group of kChannels
// channels (blockIdx.y = (frame, group)), whose loads are issued together.
// kVec: the codes of four texels are one 4-byte load per plane.  At the
// 1024^2 atlas with 59 channels 116 us with a byte load per texel and all
// channels in one thread, 87 us so, and 63 us with one pointer per channel and
// a group's Gaussians at small offsets from it, as in k_gather.
constexpr int kChannels = 8;
template <bool kCodes, bool kVec>
__global__ __launch_bounds__(256) void k_gather_lpo(const void *__restrict__ src, const float *__restrict__ lohi,
                                                    const uint32_t *__restrict__ occ,
                                                    const uint32_t *__restrict__ dyn,
                                                    const uint32_t *__restrict__ woff, int W, int H, int F, int D,
                                                    int64_t N, float *__restrict__ soa,
                                                    uint32_t *__restrict__ texel, uint8_t *__restrict__ dynflag) {
  __shared__ float s_lo[PK_MAX_CHANNELS], s_delta[PK_MAX_CHANNELS], s_rd[kCodes ? 1 : PK_MAX_CHANNELS];
  for (int c = threadIdx.x; c < D; c += blockDim.x) {
    const float L = c < 3 ? 65535.0f : 255.0f;
    s_lo[c] = lohi[2 * c];
    s_delta[c] = __fdiv_rn(__fsub_rn(lohi[2 * c + 1], lohi[2 * c]), L);
    if (!kCodes) s_rd[c] = lpo_rstep(s_delta[c]);
  }
  __syncthreads();
  const uint32_t Wq = (uint32_t)(W + 3) / 4, nq = Wq * (uint32_t)H;
  const int64_t plane = (int64_t)W * H, G = (int64_t)F * N;
  const int groups = (D + kChannels - 1) / kChannels;
  for (int fg = blockIdx.y; fg < F * groups; fg += gridDim.y) {
    const int f = fg / groups, c0 = (fg - f * groups) * kChannels;
    for (uint32_t qi = blockIdx.x * blockDim.x + threadIdx.x; qi < nq; qi += gridDim.x * blockDim.x) {
      const int y = (int)(qi / Wq), x0 = (int)(qi - (uint32_t)y * Wq) * 4;
      int64_t first;
      const uint32_t live = quad_live(occ, dyn, woff, W, y, x0, N, fg == 0, texel, dynflag, first);
      if (!live) continue;
      const int64_t pix = (int64_t)y * W + x0;
      float *dst = soa + (int64_t)c0 * G + (int64_t)f * N + first;
      if (kCodes) {
        const uint8_t *cb = reinterpret_cast<const uint8_t *>(src) + (int64_t)f * (D + 3) * plane + pix;
        auto four = [&](int64_t at) -> uint32_t {   // the four texels' bytes of a code plane
          if (kVec) return __ldg(reinterpret_cast<const uint32_t *>(cb + at));
          uint32_t v = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if ((live >> i) & 1u) v |= (uint32_t)__ldg(cb + at + i) << (8 * i);
          return v;
        };
        uint32_t lob[kChannels], hib[3];
#pragma unroll
        for (int k = 0; k < kChannels; ++k) {
          const int c = c0 + k;
          lob[k] = c < D ? four((c < 3 ? 2 * c + 1 : c + 3) * plane) : 0u;
          if (k < 3) hib[k] = c < 3 && c < D ? four(2 * c * plane) : 0u;   // position: high bytes
        }
#pragma unroll
        for (int k = 0; k < kChannels; ++k) {
          const int c = c0 + k;
          if (c >= D) break;
          const float lo = s_lo[c], delta = s_delta[c];
          float x[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t q = (lob[k] >> (8 * i)) & 255u;
            if (k < 3) q |= ((hib[k] >> (8 * i)) & 255u) << 8;
            x[i] = lpo_proxy(q, lo, delta);
          }
          store_live(x, live, dst + k * G);
        }
      } else {
#pragma unroll 4
        for (int c = c0; c < min(c0 + kChannels, D); ++c, dst += G) {
          const float lo = s_lo[c], delta = s_delta[c];
          const float *sc = reinterpret_cast<const float *>(src) + ((int64_t)f * D + c) * plane + pix;
          float x[4] = {0.f, 0.f, 0.f, 0.f};
          if (kVec) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(sc));
            x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if ((live >> i) & 1u) x[i] = __ldg(sc + i);
          }
          uint32_t q[4];
          lpo_codes4(x, live, lo, delta, s_rd[c], c < 3 ? 65535.0f : 255.0f, q);
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = lpo_proxy(q[i], lo, delta);
          store_live(x, live, dst);
        }
      }
    }
  }
}

// One thread per group of four texels, one grid row per frame and channel group.
dim3 gather_grid(int W, int H, int F, int D) {
  const int64_t nq = (int64_t)((W + 3) / 4) * H;
  const int64_t blocks = std::min<int64_t>(std::max<int64_t>(1, (nq + 255) / 256), 152 * 64);
  return dim3((unsigned)blocks, (unsigned)std::min(std::max(F, 1) * ((D + kChannels - 1) / kChannels), 65535));
}

}  // namespace

extern "C" pk_status pk_atlas_gather_lpo(const pk_plan *p, const void *src, int32_t src_kind, const float *lohi,
                                         const uint32_t *occ, const uint32_t *dyn, float *soa, uint32_t *texel,
                                         uint8_t *dynflag, void *ws, pk_stream_t stream) {
  if (!p || !src || !lohi || !occ || !soa || !texel || !dynflag || !ws) return PK_ERR_ARG;
  if (src_kind != PK_LPO_CODES && src_kind != PK_LPO_MASTERS) return PK_ERR_ARG;
  if (!aligned16(soa)) return PK_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int W = p->desc.atlas_w, H = p->desc.atlas_h;
  const int64_t nwords = (int64_t)((W + 31) / 32) * H;
  uint32_t *woff = at<uint32_t>(ws, p->ws.woff);
  pk_device_status *status = at<pk_device_status>(ws, p->ws.status);
  launch_word_scan(occ, nwords, woff, status, p->N, st);
  const dim3 blocks = gather_grid(W, H, p->F, p->D);
  // four texels per load: whole groups per row, aligned planes (codes: any caller's pointer)
  const bool vec = (W % 4) == 0 && (reinterpret_cast<uintptr_t>(src) & (src_kind == PK_LPO_CODES ? 3u : 15u)) == 0;
#define PK_LPO(C, V) k_gather_lpo<C, V><<<blocks, 256, 0, st>>>(src, lohi, occ, dyn, woff, W, H, p->F, p->D, p->N, soa, texel, dynflag)
  if (src_kind == PK_LPO_CODES) {
    if (vec) PK_LPO(true, true); else PK_LPO(true, false);
  } else {
    if (vec) PK_LPO(false, true); else PK_LPO(false, false);
  }
#undef PK_LPO
  return check_launch();
}

extern "C" pk_status pk_atlas_gather(const pk_plan *p, const void *atlas, const uint32_t *occ, const uint32_t *dyn,
                                     float *soa, uint32_t *texel, uint8_t *dynflag, void *ws, pk_stream_t stream) {
  if (!p || !atlas || !occ || !soa || !texel || !dynflag || !ws) return PK_ERR_ARG;
  if (!aligned16(atlas) || !aligned16(soa)) return PK_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int W = p->desc.atlas_w, H = p->desc.atlas_h;
  const int64_t nwords = (int64_t)((W + 31) / 32) * H;
  uint32_t *woff = at<uint32_t>(ws, p->ws.woff);
  pk_device_status *status = at<pk_device_status>(ws, p->ws.status);
  launch_word_scan(occ, nwords, woff, status, p->N, st);
  const int64_t nq = (int64_t)((W + 3) / 4) * H;
  int blocks = (int)((nq + 255) / 256);
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (blocks < 1) blocks = 1;
  const bool vec = (W % 4) == 0;
  if (p->desc.texel_type == PK_TEXEL_F16) {
    auto a = reinterpret_cast<const __half *>(atlas);
    if (vec)
      k_gather<__half, true><<<blocks, 256, 0, st>>>(a, occ, dyn, woff, W, H, p->F, p->D, p->N, soa, texel, dynflag, status);
    else
      k_gather<__half, false><<<blocks, 256, 0, st>>>(a, occ, dyn, woff, W, H, p->F, p->D, p->N, soa, texel, dynflag,
                                                      status);
  } else {
    auto a = reinterpret_cast<const float *>(atlas);
    if (vec)
      k_gather<float, true><<<blocks, 256, 0, st>>>(a, occ, dyn, woff, W, H, p->F, p->D, p->N, soa, texel, dynflag,
                                                    status);
    else
      k_gather<float, false><<<blocks, 256, 0, st>>>(a, occ, dyn, woff, W, H, p->F, p->D, p->N, soa, texel, dynflag,
                                                     status);
  }
  return check_launch();
}
