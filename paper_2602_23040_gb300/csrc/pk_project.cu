// a2 -- per (view, Gaussian) EWA projection and SH colour.
//
// One thread per Gaussian of every frame: its D attributes are read once
// (coalesced, channel-major SoA), activated once, and then projected into
// every view of its frame; each view's record is three 16-byte stores.  The
// atlas is therefore read once per launch however many views the launch holds.
#include "pk_proj_math.cuh"

using namespace pk;

namespace {

constexpr int kProjThreads = 128;

// The SH coefficients of a thread's Gaussian live in shared memory, column
// tid of s_k[NK][kProjThreads], coefficient 3 j + c, four to an access (each
// thread reads only its own column, so no barrier is needed); in registers
// they would cap the occupancy.
// kPair: two views at a time, so that the coefficients' reads (the kernel's
// shared-memory pipe is its busiest) and the latencies of one view's chain
// serve both: 474 -> 418 us at the 52-view rig.  A frame of one view has
// nothing to pair (11.2 us instead of 9.8 for 157 K Gaussians).
template <int L, bool kPair>
__global__ __launch_bounds__(kProjThreads) void k_project(const float *__restrict__ soa, int64_t G, int64_t N,
                                                          const DevView *__restrict__ views,
                                                          const int32_t *__restrict__ fview_off,
                                                          const int32_t *__restrict__ fview_idx, float znear,
                                                          float *__restrict__ rec) {
  constexpr int NB = (L + 1) * (L + 1), NK = (3 * NB + 3) / 4;
  extern __shared__ float4 s_k[];   // [NK][kProjThreads]
  for (int64_t gi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gi < G; gi += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = gi / N, g = gi - f * N;
    auto attr = [&](int c) { return __ldg(soa + (int64_t)c * G + gi); };
    Act a;
    activate(attr, a);
    float4 *mine = s_k + threadIdx.x;
    bool finite = a.finite;   // a Gaussian with a non-finite texel value is culled in every view
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      float kv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        kv[e] = 4 * i + e < 3 * NB ? attr(11 + 4 * i + e) : 0.f;
        finite = finite && isfinite(kv[e]);
      }
      mine[i * kProjThreads] = make_float4(kv[0], kv[1], kv[2], kv[3]);
    }
    const int vb = __ldg(fview_off + f), ve = __ldg(fview_off + f + 1);
    for (int vi = vb; vi < ve; vi += kPair ? 2 : 1) {
      const bool two = kPair && vi + 1 < ve;
      const int v0 = __ldg(fview_idx + vi), v1 = two ? __ldg(fview_idx + vi + 1) : v0;
      Proj p0, p1;
      float d0[3], d1[3], len;
      bool ok0, ok1 = false;
      {
        const ViewCam cam = load_cam(views + v0);
        ok0 = finite && project(a, cam, znear, p0);
        view_dir(a, cam, d0, len);
      }
      if (kPair) {   // (of an odd view out the result is not used)
        const ViewCam cam = load_cam(views + v1);
        ok1 = finite && project(a, cam, znear, p1);
        view_dir(a, cam, d1, len);
      }
      float Y0[NB], Y1[NB], c0[3], c1[3];
      sh_basis<L>(d0[0], d0[1], d0[2], Y0);
      if (kPair) sh_basis<L>(d1[0], d1[1], d1[2], Y1);
#pragma unroll
      for (int c = 0; c < 3; ++c) c0[c] = c1[c] = 0.5f;
#pragma unroll
      for (int i = 0; i < NK; ++i) {
        const float4 q = mine[i * kProjThreads];
        const float kv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * i + e < 3 * NB) {
            const int j = (4 * i + e) / 3, c = (4 * i + e) % 3;
            c0[c] = fmaf(kv[e], Y0[j], c0[c]);
            if (kPair) c1[c] = fmaf(kv[e], Y1[j], c1[c]);
          }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        c0[c] = fmaxf(c0[c], 0.f);
        c1[c] = fmaxf(c1[c], 0.f);
      }
      auto put = [&](int v, bool ok, const Proj &p, const float (&rgb)[3]) {
        float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0, r2 = r0;
        if (ok && isfinite(rgb[0]) && isfinite(rgb[1]) && isfinite(rgb[2]) && isfinite(a.o)) {
          r0 = make_float4(p.m[0], p.m[1], p.conic[0], p.conic[1]);
          r1 = make_float4(p.conic[2], a.o, p.X[2], p.radius);
          r2 = make_float4(rgb[0], rgb[1], rgb[2], 0.f);
        }
        float4 *dst = reinterpret_cast<float4 *>(rec + ((int64_t)v * N + g) * kRec);
        dst[0] = r0;
        dst[1] = r1;
        dst[2] = r2;
      };
      put(v0, ok0, p0, c0);
      if (two) put(v1, ok1, p1, c1);
    }
  }
}

}  // namespace

extern "C" pk_status pk_project_and_sh(const pk_plan *p, const float *soa, float *records, void *ws,
                                       pk_stream_t stream) {
  if (!p || !soa || !records || !ws) return PK_ERR_ARG;
  if (!aligned16(records)) return PK_ERR_ARG;
  if (p->G == 0) return PK_OK;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const DevView *views = at<DevView>(ws, p->ws.views);
  const int32_t *fo = at<int32_t>(ws, p->ws.fview_off), *fi = at<int32_t>(ws, p->ws.fview_idx);
  int64_t blocks = (p->G + kProjThreads - 1) / kProjThreads;
  if (blocks > 152 * 64) blocks = 152 * 64;
  const float zn = p->opts.znear;
  const size_t smem = sizeof(float4) * ((3 * (p->L + 1) * (p->L + 1) + 3) / 4) * kProjThreads;
  // by pairs where the frames have two views or more on average
#define PK_PROJECT(LL)                                                                                            \
  if (p->V >= 2 * p->F)                                                                                           \
    k_project<LL, true><<<(int)blocks, kProjThreads, smem, st>>>(soa, p->G, p->N, views, fo, fi, zn, records);    \
  else                                                                                                            \
    k_project<LL, false><<<(int)blocks, kProjThreads, smem, st>>>(soa, p->G, p->N, views, fo, fi, zn, records);   \
  break
  switch (p->L) {
    case 0: PK_PROJECT(0);
    case 1: PK_PROJECT(1);
    case 2: PK_PROJECT(2);
    default: PK_PROJECT(3);
  }
#undef PK_PROJECT
  return check_launch();
}
