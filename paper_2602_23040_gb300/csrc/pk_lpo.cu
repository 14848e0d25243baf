// Low-precision proxy (Sec. 4.2 "Low Precision Optimization", Supp. "Video
// Coding"): per-channel min/max normalisation over the live texels of every
// frame and the 8-bit plane layout (position as two bytes).  The gather
// that reads the proxy lives with the other gathers.
//
// Both kernels stream the planar FP32 atlas once, kQuads groups of four
// consecutive texels per thread and step, one block row per (frame,
// channel) plane.  HBM bounds them once enough loads are in flight: a
// step's loads are issued together, the texel coordinates advance by
// additions (a 64-bit division per group cost more issue slots than the
// rest of the loop), and the grid is several waves of short blocks, so that
// no block is left over for a wave of its own.  1024^2 atlas, 59
// channels: min / max 105 -> 55 us, encode 144 -> 97 us, and 82 us with the
// four codes of a group formed without branches (pk_lpo.cuh).
#include "pk_common.cuh"
#include "pk_lpo.cuh"

using namespace pk;

namespace {

constexpr int kLpoThreads = 256;
constexpr int kQuads = 4;

// Groups of four texels of a plane.  A block takes runs of kQuads *
// kLpoThreads consecutive groups (64 KB of a plane), gridDim.x runs apart, a
// thread every kLpoThreads-th of a run: (x, y) of its next group, x in groups.
struct QuadWalk {
  int64_t q, nq, jump;   // group index in the plane, groups of the plane, from a run's end to the next run
  int x, y, dx, dy, jx, jy, Wq;
  __device__ __forceinline__ QuadWalk(int W, int H) {
    Wq = (W + 3) >> 2;
    nq = (int64_t)Wq * H;
    q = (int64_t)blockIdx.x * (kLpoThreads * kQuads) + threadIdx.x;
    jump = (int64_t)(gridDim.x - 1) * (kLpoThreads * kQuads);
    y = (int)(q / Wq);
    x = (int)(q - (int64_t)y * Wq);
    dy = kLpoThreads / Wq;
    dx = kLpoThreads - dy * Wq;
    jy = (int)(jump / Wq);
    jx = (int)(jump - (int64_t)jy * Wq);
  }
  __device__ __forceinline__ void next() { move(kLpoThreads, dx, dy); }
  __device__ __forceinline__ void next_run() { move(jump, jx, jy); }
  __device__ __forceinline__ void move(int64_t n, int mx, int my) {
    q += n;
    x += mx;
    y += my;
    if (x >= Wq) {
      x -= Wq;
      ++y;
    }
  }
};

// The texels of the thread's next kQuads groups and their occupancy (bits
// 0..3 of live[k]; 0 past the plane), all loads issued before the first use.
struct QuadBatch {
  float v[kQuads][4];
  uint32_t live[kQuads];
  int x0[kQuads];
  int64_t at[kQuads];   // first texel in the plane
};

__device__ __forceinline__ void load_quads(const float *__restrict__ src, const uint32_t *__restrict__ occ, int W,
                                           QuadWalk &w, QuadBatch &b) {
  const int Wp = (W + 31) >> 5;
  const bool vec = (W & 3) == 0;   // 16-byte aligned rows of four texels
#pragma unroll
  for (int k = 0; k < kQuads; ++k) {
    const bool in = w.q < w.nq;
    b.x0[k] = 4 * w.x;
    b.at[k] = in ? (int64_t)w.y * W + 4 * w.x : -1;
    // the four texels share one occupancy word (x0 is a multiple of 4)
    b.live[k] = in ? (__ldg(occ + (int64_t)w.y * Wp + (w.x >> 3)) >> (4 * (w.x & 7))) & 15u : 0u;
    w.next();
  }
  w.next_run();
#pragma unroll
  for (int k = 0; k < kQuads; ++k) {
    if (vec) {
      const float4 q = b.live[k] ? __ldg(reinterpret_cast<const float4 *>(src + b.at[k])) : make_float4(0.f, 0.f, 0.f, 0.f);
      b.v[k][0] = q.x; b.v[k][1] = q.y; b.v[k][2] = q.z; b.v[k][3] = q.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (b.x0[k] + i >= W) b.live[k] &= ~(1u << i);
        b.v[k][i] = (b.live[k] >> i) & 1u ? __ldg(src + b.at[k] + i) : 0.f;
      }
    }
  }
}

// Order-preserving map of a float onto uint32 (NaN excluded by the caller).
__device__ __forceinline__ uint32_t ordered(float v) {
  const uint32_t b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unordered(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__global__ void k_minmax_init(uint32_t *keys, int D) {
  const int i = threadIdx.x;
  if (i < 2 * D) keys[i] = (i & 1) ? 0u : 0xffffffffu;
}

// Planes fc = f * D + c from blockIdx.y in steps of gridDim.y.
__global__ __launch_bounds__(kLpoThreads) void k_minmax(const float *__restrict__ atlas,
                                                        const uint32_t *__restrict__ occ, int W, int H, int D,
                                                        int64_t planes, uint32_t *keys) {
  __shared__ uint32_t s_lo[kLpoThreads / 32], s_hi[kLpoThreads / 32];
  const int64_t plane = (int64_t)W * H;
  for (int64_t fc = blockIdx.y; fc < planes; fc += gridDim.y) {
    const int c = (int)(fc % D);
    const float *src = atlas + fc * plane;
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (QuadWalk w(W, H); w.q < w.nq;) {
      QuadBatch b;
      load_quads(src, occ, W, w, b);
#pragma unroll
      for (int k = 0; k < kQuads; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float v = b.v[k][i];
          if (!((b.live[k] >> i) & 1u) || v != v) continue;
          const uint32_t key = ordered(v);
          lo = min(lo, key);
          hi = max(hi, key);
        }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
      s_lo[threadIdx.x >> 5] = lo;
      s_hi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 1; k < kLpoThreads / 32; ++k) {
        lo = min(lo, s_lo[k]);
        hi = max(hi, s_hi[k]);
      }
      if (lo != 0xffffffffu) atomicMin(&keys[2 * c], lo);
      if (hi != 0u) atomicMax(&keys[2 * c + 1], hi);
    }
    __syncthreads();   // before the next plane's sums
  }
}

__global__ void k_minmax_final(uint32_t *keys, int D) {
  const int c = threadIdx.x;
  if (c >= D) return;
  const uint32_t lo = keys[2 * c], hi = keys[2 * c + 1];
  float *out = reinterpret_cast<float *>(keys);
  const bool none = lo == 0xffffffffu;
  out[2 * c] = none ? 0.0f : unordered(lo);
  out[2 * c + 1] = none ? 0.0f : unordered(hi);
}

__device__ __forceinline__ void encode_plane(const float *__restrict__ atlas, const uint32_t *__restrict__ occ,
                                             const float *__restrict__ lohi, int W, int H, int D, int64_t fc,
                                             uint8_t *__restrict__ codes) {
  const int f = (int)(fc / D), c = (int)(fc - (int64_t)f * D);
  const int64_t plane = (int64_t)W * H;
  const float L = c < 3 ? 65535.0f : 255.0f;
  const float lo = __ldg(lohi + 2 * c);
  const float delta = __fdiv_rn(__fsub_rn(__ldg(lohi + 2 * c + 1), lo), L);
  const float rd = lpo_rstep(delta);
  const float *src = atlas + fc * plane;
  uint8_t *p0 = codes + ((int64_t)f * (D + 3) + (c < 3 ? 2 * c : c + 3)) * plane;
  uint8_t *p1 = c < 3 ? p0 + plane : nullptr;
  const bool vec = (W & 3) == 0;
  for (QuadWalk w(W, H); w.q < w.nq;) {
    QuadBatch b;
    load_quads(src, occ, W, w, b);
#pragma unroll
    for (int k = 0; k < kQuads; ++k) {
      if (b.at[k] < 0) continue;
      uint32_t q[4];
      lpo_codes4(b.v[k], b.live[k], lo, delta, rd, L, q);
      // low bytes, and the high ones of a position channel
      uint32_t b0 = q[0] | (q[1] << 8) | (q[2] << 16) | (q[3] << 24), b1 = 0;
      if (c < 3) {
        b1 = __byte_perm(__byte_perm(q[0], q[1], 0x0040), __byte_perm(q[2], q[3], 0x0040), 0x5410);
        b0 = __byte_perm(__byte_perm(q[0], q[1], 0x0051), __byte_perm(q[2], q[3], 0x0051), 0x5410);
      }
      if (vec) {
        *reinterpret_cast<uint32_t *>(p0 + b.at[k]) = b0;
        if (p1) *reinterpret_cast<uint32_t *>(p1 + b.at[k]) = b1;
      } else {
        for (int i = 0; i < 4 && b.x0[k] + i < W; ++i) {
          p0[b.at[k] + i] = (uint8_t)(b0 >> (8 * i));
          if (p1) p1[b.at[k] + i] = (uint8_t)(b1 >> (8 * i));
        }
      }
    }
  }
}

// Planes fc = f * D + c as in k_minmax; four texels per thread, written as
// one 4-byte group per code plane when the width allows.
__global__ __launch_bounds__(kLpoThreads) void k_encode(const float *__restrict__ atlas,
                                                        const uint32_t *__restrict__ occ,
                                                        const float *__restrict__ lohi, int W, int H, int D,
                                                        int64_t planes, uint8_t *__restrict__ codes) {
  for (int64_t fc = blockIdx.y; fc < planes; fc += gridDim.y) encode_plane(atlas, occ, lohi, W, H, D, fc, codes);
}

dim3 plane_grid(const pk_plan *p, int64_t planes) {
  const int W = p->desc.atlas_w, H = p->desc.atlas_h;
  const int64_t nq = (int64_t)((W + 3) / 4) * H;
  int64_t bx = (nq + kLpoThreads * kQuads - 1) / (kLpoThreads * kQuads);
  // 32 blocks per SM over all planes: several waves
  const int64_t cap = (152 * 32 + planes - 1) / planes;
  if (bx > cap) bx = cap;
  if (bx < 1) bx = 1;
  return dim3((unsigned)bx, (unsigned)(planes < 65535 ? planes : 65535));
}

}  // namespace

extern "C" pk_status pk_lpo_minmax(const pk_plan *p, const float *atlas, const uint32_t *occ, float *lohi, void *ws,
                                   pk_stream_t stream) {
  if (!p || !atlas || !occ || !lohi || !ws) return PK_ERR_ARG;
  if (!aligned16(atlas) || !aligned16(lohi)) return PK_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  uint32_t *keys = reinterpret_cast<uint32_t *>(lohi);
  k_minmax_init<<<1, 128, 0, st>>>(keys, p->D);
  k_minmax<<<plane_grid(p, (int64_t)p->F * p->D), kLpoThreads, 0, st>>>(atlas, occ, p->desc.atlas_w,
                                                                        p->desc.atlas_h, p->D,
                                                                        (int64_t)p->F * p->D, keys);
  k_minmax_final<<<1, 64, 0, st>>>(keys, p->D);
  return check_launch();
}

extern "C" pk_status pk_lpo_encode(const pk_plan *p, const float *atlas, const uint32_t *occ, const float *lohi,
                                   uint8_t *codes, void *ws, pk_stream_t stream) {
  if (!p || !atlas || !occ || !lohi || !codes || !ws) return PK_ERR_ARG;
  if (!aligned16(atlas) || !aligned16(codes)) return PK_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  k_encode<<<plane_grid(p, (int64_t)p->F * p->D), kLpoThreads, 0, st>>>(atlas, occ, lohi, p->desc.atlas_w,
                                                                        p->desc.atlas_h, p->D,
                                                                        (int64_t)p->F * p->D, codes);
  return check_launch();
}
