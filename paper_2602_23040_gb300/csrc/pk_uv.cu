// UV cells (eq. uvgs2) and Max-K UV pruning (Sec. 4.2 "UV-Based Pruning").
//
// Four launches over n candidate Gaussians and an M x N map (after the
// zeroing of the counts): cell and in-cell slot per Gaussian (one atomic per
// valid Gaussian on the cell's counter), a bucket per cell (each block scans
// its cells' counts and takes its stretch of the bucket array with one
// atomic: the buckets' order among each other does not matter), a scatter of
// the Gaussian indices into the buckets, and the rank of every Gaussian
// within its bucket by opacity (higher first, then lower index): the
// buckets hold a handful of Gaussians, so each Gaussian counts the members
// that beat it.  The cell is the one FP64 gives (atan2, acos); FP64 itself
// runs only where FP32 cannot tell the cell apart (k_uv_cell).
#include "pk_common.cuh"

using namespace pk;

namespace {

constexpr int kUvThreads = 256;
constexpr int kUvScanItems = 2048;   // counts per scan block (8 per thread)
constexpr int kUvCellItems = 8;      // Gaussians per thread of k_uv_cell
constexpr uint32_t kInvalid = 0xFFFFFFFFu;

struct UvScratch {
  size_t slot, offs, taken, bucket, total;
};

UvScratch uv_layout(int64_t n, int64_t cells) {
  UvScratch L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at_ = off;
    off = (off + bytes + 255) & ~size_t(255);
    return at_;
  };
  L.slot = take(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1));
  L.offs = take(sizeof(uint32_t) * (size_t)cells);
  L.taken = take(sizeof(uint32_t));   // bucket entries handed out so far
  L.bucket = take(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1));
  L.total = off;
  return L;
}

// Cell of a Gaussian in FP64, kInvalid without a valid projection.
__device__ __noinline__ uint32_t uv_cell_f64(float xf, float yf, float zf, int M, int N) {
  const double x = xf, y = yf, z = zf;
  const double rho = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)));
  if (!(rho > 0.0) || !isfinite(rho)) return kInvalid;
  const double kPi = 3.14159265358979323846;
  const double su = (kPi + atan2(y, x)) / (2.0 * kPi) * M, sv = acos(z / rho) / kPi * N;
  const double u = floor(su), v = floor(sv);
  return u >= 0.0 && u < M && v >= 0.0 && v < N ? (uint32_t)v * (uint32_t)M + (uint32_t)u : kInvalid;
}

// Cell by FP32 where that is certain to be the FP64 cell; false where it is
// not.  The FP32 coordinates su = (pi + atan2(y, x)) M / 2pi and sv =
// atan2(sqrt(x^2 + y^2), z) N / pi (acos(z / rho) without its cancellation
// at the poles) lie within 3.5e-7 M and 4.4e-7 N of the exact ones: atan2f
// is within 3 ulp (7.2e-7 at pi), the sum with pi, the scale and the product
// add 2^-22 + 1.5 * 2^-23 relative, sqrtf's argument 0.8e-7 of angle.  The
// FP64 coordinates lie within 1e-8 N (acos near the poles).  So a coordinate
// further than 1e-6 M (N) from an integer has the same floor in both.
// The range of the values keeps the squares normal.
__device__ __forceinline__ bool uv_cell_f32(float x, float y, float z, int M, int N, uint32_t &c) {
  const float big = fmaxf(fmaxf(fabsf(x), fabsf(y)), fabsf(z));
  if (!(big > 1e-15f && big < 1e15f) || !isfinite(x) || !isfinite(y) || !isfinite(z)) return false;
  const float su = (3.14159265f + atan2f(y, x)) * (0.15915494f * (float)M);
  const float sv = atan2f(sqrtf(x * x + y * y), z) * (0.31830989f * (float)N);
  const float u = floorf(su), v = floorf(sv);
  const float du = 1e-6f * (float)M, dv = 1e-6f * (float)N;
  if (!(su - u > du && su - u < 1.f - du && sv - v > dv && sv - v < 1.f - dv)) return false;
  if (!(u >= 0.f && u < (float)M && v >= 0.f && v < (float)N)) return false;
  c = (uint32_t)v * (uint32_t)M + (uint32_t)u;
  return true;
}

// The FP64 chain (atan2, acos, divisions) bounds a kernel that runs it for
// every Gaussian: FP64 runs at a small fraction of the FP32 rate here.
// Here each block places its kUvCellItems * 256 Gaussians in FP32 and queues
// the ones within 1e-6 M (N) of a cell's edge -- four in a thousand at 1024^2
// cells -- which its warps then place in FP64, the lanes full, instead of
// one lane of every eighth warp: 143 -> 13.7 us at 629 K Gaussians and 1024^2
// cells (the whole call, with two launches of the scan gone, 183 -> 46 us).
__global__ __launch_bounds__(kUvThreads) void k_uv_cell(const float *__restrict__ soa, int64_t n, int64_t stride,
                                                         int M, int N, uint32_t *__restrict__ cell,
                                                         uint32_t *__restrict__ slot, uint32_t *count) {
  __shared__ uint16_t s_queue[kUvThreads * kUvCellItems];
  __shared__ uint32_t s_n;
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (kUvThreads * kUvCellItems);
  float x[kUvCellItems], y[kUvCellItems], z[kUvCellItems], lg[kUvCellItems];
#pragma unroll
  for (int k = 0; k < kUvCellItems; ++k) {
    const int64_t i = base + k * kUvThreads + threadIdx.x;
    const bool in = i < n;
    x[k] = in ? __ldg(soa + i) : 0.f;
    y[k] = in ? __ldg(soa + stride + i) : 0.f;
    z[k] = in ? __ldg(soa + 2 * stride + i) : 0.f;
    lg[k] = in ? __ldg(soa + 10 * stride + i) : 0.f;
  }
#pragma unroll
  for (int k = 0; k < kUvCellItems; ++k) {
    const int64_t i = base + k * kUvThreads + threadIdx.x;
    if (i >= n) continue;
    uint32_t c = kInvalid;
    if (lg[k] == lg[k] && !uv_cell_f32(x[k], y[k], z[k], M, N, c)) {
      s_queue[atomicAdd(&s_n, 1u)] = (uint16_t)(k * kUvThreads + threadIdx.x);
      continue;
    }
    cell[i] = c;
    if (c != kInvalid) slot[i] = atomicAdd(count + c, 1u);
  }
  __syncthreads();
  const uint32_t queued = s_n;
  for (uint32_t q = threadIdx.x; q < queued; q += kUvThreads) {
    const int64_t i = base + s_queue[q];
    const uint32_t c = uv_cell_f64(__ldg(soa + i), __ldg(soa + stride + i), __ldg(soa + 2 * stride + i), M, N);
    cell[i] = c;
    if (c != kInvalid) slot[i] = atomicAdd(count + c, 1u);
  }
}

// Exclusive scan of one value per thread over the block.
__device__ __forceinline__ uint32_t block_scan_excl(uint32_t x, uint32_t &total, uint32_t *s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < kUvThreads / 32 ? s_warp[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kUvThreads / 32) s_warp[lane] = w;
  }
  __syncthreads();
  total = s_warp[kUvThreads / 32 - 1];
  const uint32_t excl = (warp ? s_warp[warp - 1] : 0u) + inc - x;
  __syncthreads();
  return excl;
}

// First bucket entry of each cell: a block's cells lie one after another,
// the blocks in the order in which they ask.
__global__ __launch_bounds__(kUvThreads) void k_uv_offsets(const uint32_t *__restrict__ count, int64_t cells,
                                                            uint32_t *taken,
                                                            uint32_t *__restrict__ offs) {
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_base;
  constexpr int kPer = kUvScanItems / kUvThreads;
  const int64_t base = (int64_t)blockIdx.x * kUvScanItems + (int64_t)threadIdx.x * kPer;
  uint32_t v[kPer], acc = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    v[k] = base + k < cells ? __ldg(count + base + k) : 0u;
    acc += v[k];
  }
  uint32_t tot;
  uint32_t run = block_scan_excl(acc, tot, s_warp);
  if (threadIdx.x == 0) s_base = tot ? atomicAdd(taken, tot) : 0u;
  __syncthreads();
  run += s_base;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (base + k < cells) offs[base + k] = run;
    run += v[k];
  }
}

__global__ __launch_bounds__(kUvThreads) void k_uv_bucket(const uint32_t *__restrict__ cell,
                                                           const uint32_t *__restrict__ slot,
                                                           const uint32_t *__restrict__ offs, int64_t n,
                                                           uint32_t *__restrict__ bucket) {
  const int64_t i = (int64_t)blockIdx.x * kUvThreads + threadIdx.x;
  if (i >= n) return;
  const uint32_t c = cell[i];
  if (c != kInvalid) bucket[offs[c] + slot[i]] = (uint32_t)i;
}

// Rank of Gaussian i among the Gaussians of its cell: those with a higher
// opacity logit, or an equal logit and a lower index, come first.
__global__ __launch_bounds__(kUvThreads) void k_uv_rank(const float *__restrict__ soa, int64_t stride,
                                                         const uint32_t *__restrict__ cell,
                                                         const uint32_t *__restrict__ offs,
                                                         const uint32_t *__restrict__ count,
                                                         const uint32_t *__restrict__ bucket, int64_t n, int K,
                                                         uint32_t *__restrict__ rank, uint8_t *__restrict__ keep) {
  const int64_t i = (int64_t)blockIdx.x * kUvThreads + threadIdx.x;
  if (i >= n) return;
  const uint32_t c = cell[i];
  if (c == kInvalid) {
    rank[i] = kInvalid;
    keep[i] = 0;
    return;
  }
  const float* logit = soa + 10 * stride;
  const float li = __ldg(logit + i);
  const uint32_t beg = offs[c], cnt = count[c];
  uint32_t r = 0;
  for (uint32_t k = 0; k < cnt; ++k) {
    const uint32_t j = __ldg(bucket + beg + k);
    const float lj = __ldg(logit + j);
    r += (lj > li || (lj == li && j < (uint32_t)i)) ? 1u : 0u;
  }
  rank[i] = r;
  keep[i] = r < (uint32_t)K ? 1 : 0;
}

}  // namespace

extern "C" uint64_t pk_uv_max_k_scratch_bytes(int64_t n, int32_t M, int32_t N) {
  if (n < 0 || M < 1 || N < 1) return 0;
  return uv_layout(n, (int64_t)M * N).total;
}

extern "C" pk_status pk_uv_max_k(const float *soa, int64_t n, int64_t stride, int32_t M, int32_t N, int32_t K,
                                 uint32_t *cell, uint32_t *rank, uint8_t *keep, uint32_t *count, void *scratch,
                                 pk_stream_t stream) {
  if (n < 0 || M < 1 || N < 1 || K < 0 || stride < n) return PK_ERR_ARG;
  const int64_t cells = (int64_t)M * N;
  if (cells >= (int64_t)kInvalid || n >= (int64_t)kInvalid) return PK_ERR_ARG;
  if (!count || !scratch || (n > 0 && (!soa || !cell || !rank || !keep))) return PK_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(scratch) & 255u) return PK_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const UvScratch L = uv_layout(n, cells);
  uint32_t *slot = at<uint32_t>(scratch, L.slot), *offs = at<uint32_t>(scratch, L.offs);
  uint32_t *taken = at<uint32_t>(scratch, L.taken), *bucket = at<uint32_t>(scratch, L.bucket);
  pk_status ze = zero_async({{count, sizeof(uint32_t) * (size_t)cells}, {taken, sizeof(uint32_t)}}, st);
  if (ze != PK_OK) return ze;
  if (n == 0) return PK_OK;
  const unsigned gn = (unsigned)((n + kUvThreads - 1) / kUvThreads);
  const int64_t blocks = (cells + kUvScanItems - 1) / kUvScanItems;
  constexpr int kCellBlock = kUvThreads * kUvCellItems;
  k_uv_cell<<<(unsigned)((n + kCellBlock - 1) / kCellBlock), kUvThreads, 0, st>>>(soa, n, stride, M, N, cell, slot,
                                                                                  count);
  k_uv_offsets<<<(unsigned)blocks, kUvThreads, 0, st>>>(count, cells, taken, offs);
  k_uv_bucket<<<gn, kUvThreads, 0, st>>>(cell, slot, offs, n, bucket);
  k_uv_rank<<<gn, kUvThreads, 0, st>>>(soa, stride, cell, offs, count, bucket, n, K, rank, keep);
  return check_launch();
}
