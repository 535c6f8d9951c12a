// march_fwd.cu -- forward march: render and training forward (sm_103a).
//
// Persistent kernel of 8 warps per CTA; a warp owns a bundle of 32 rays at a
// time (an 8 x 4 pixel tile of a camera, or 32 consecutive rays of a list).  The warp walks its rays
// in order and packs their evaluated samples (Sec. 4.1: only samples inside
// the occupancy interval are evaluated) into a 32-entry queue that may span
// rays (packed.cuh); the 32 queued samples are gathered and activated in
// parallel, composited with segmented lane scans (Eq. 1: a product scan of
// 1 - M alpha per ray) and early termination is resolved per ray.  After
// the bundle each lane shades its ray with the deferred MLP (Eq. 4): FP32 on
// CUDA cores, or BF16 on tensor cores for a BF16 scene.
//
// Modes: render (pixels and sample counts); training forward with the loss
// (per-ray state for the backward, MLP, Charbonnier and smoothness terms);
// training forward without the loss (per-ray state only: the fused training
// step lets the MLP backward, which evaluates the MLP anyway, add the loss).
#include <cstdio>

#include <type_traits>

#include "march_fwd.cuh"

namespace omerf {

#ifndef OMERF_FWD_MINB
#define OMERF_FWD_MINB 3  // resident CTAs per SM the register budget is sized for
#endif

// TRAIN: write the per-ray state the backward needs instead of pixels; with
// LOSS also evaluate the deferred MLP and the loss terms (a fused training
// step leaves the loss to the MLP backward, which evaluates the MLP anyway).
template <class FT, bool SPARSE, bool TRAIN, bool LOSS>
__global__ void __launch_bounds__(kThreads, OMERF_FWD_MINB) march_fwd_kernel(const Geo g, const FwdArgs a) {
  // BF16 render: deferred MLP on tensor cores; otherwise FP32 on CUDA cores
  constexpr bool kMMA = std::is_same<FT, __nv_bfloat16>::value && !TRAIN;
  __shared__ __align__(16) float sW[kMMA ? 4 : kSmemMlp];
  __shared__ typename std::conditional<kMMA, MlpFrags, int>::type sFrag;
  __shared__ float sLoss[2][kThreads / 32];
  __shared__ WarpMarch<kMMA> sMarch[kThreads / 32];
  if constexpr (kMMA) {
    build_mlp_frags(g.mlp, sFrag);
  } else if constexpr (!TRAIN || LOSS) {
    load_mlp_padded(g.mlp, sW);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  WarpMarch<kMMA>& ws = sMarch[threadIdx.x >> 5];
  float l_rgb = 0.0f, l_smooth = 0.0f;

  // A camera (of a BF16 scene; FP32 ones are marched by march_cam.cu): the CTA
  // takes super-tiles of 2 x 4 tiles of 8 x 4 pixels (16 x 16 pixels), so that
  // its 8 warps march neighbouring rays together and share L1 lines.  A list:
  // every warp takes its next 32 consecutive rays on its own, without waiting
  // for the CTA's slowest bundle (the rays of a training batch lie anywhere).
  // Without a counter there is one unit per CTA or warp.
  __shared__ unsigned sWork;
  const int warp = threadIdx.x >> 5;
  for (bool first = true;; first = false) {
    unsigned sb;
    if (kMMA && a.use_cam) {
      if (threadIdx.x == 0)
        sWork = a.counter ? atomicAdd(a.counter, 1u) : (first ? blockIdx.x : (unsigned)a.n_super);
      __syncthreads();
      sb = sWork;
      __syncthreads();
    } else {
      sb = first ? blockIdx.x * (kThreads / 32) + warp : (unsigned)a.n_super;
      if (a.counter) {
        if (lane == 0) sb = atomicAdd(a.counter, 1u);
        sb = __shfl_sync(kFull, sb, 0);
      }
    }
    if (sb >= a.n_super) break;

    long rid;
    bool valid;
    float o[3] = {0.0f, 0.0f, 0.0f}, d[3] = {0.0f, 0.0f, 1.0f};
    if (kMMA && a.n_cams > 0) {
      int c = 0;
      while (c + 1 < a.n_cams && (long long)sb >= a.cams[c + 1].super_start) c++;
      const CamRec& cr = a.cams[c];
      const unsigned lsb = (unsigned)((long long)sb - cr.super_start);
      const int sx = (int)(lsb % (unsigned)cr.super_x), sy = (int)(lsb / (unsigned)cr.super_x);
      const int tx = 2 * sx + (warp & 1), ty = 4 * sy + (warp >> 1);
      const int px = tx * 8 + (lane & 7), py = ty * 4 + (lane >> 3);
      valid = px < cr.cam.width && py < cr.cam.height;
      rid = (long)cr.ray_start + (long)py * cr.cam.width + px;
      if (valid) camera_ray(cr.cam, px, py, o, d);
    } else if (kMMA && a.use_cam) {
      const int sx = (int)(sb % (unsigned)a.super_x), sy = (int)(sb / (unsigned)a.super_x);
      const int tx = 2 * sx + (warp & 1), ty = 4 * sy + (warp >> 1);
      const int px = tx * 8 + (lane & 7), py = ty * 4 + (lane >> 3);
      valid = px < a.cam.width && py < a.cam.height;
      rid = (long)py * a.cam.width + px;
      if (valid) camera_ray(a.cam, px, py, o, d);
    } else {
      rid = (long)sb * 32 + lane;
      valid = rid < a.n;
      if (valid) {
        const float* r = a.rays + 6 * rid;
#pragma unroll
        for (int c = 0; c < 3; c++) {
          o[c] = __ldg(r + c);
          d[c] = __ldg(r + 3 + c);
        }
      }
    }
    int klo = 0, khi = -1;
    const bool any = valid && lattice_range(g, o, d, klo, khi);
    march_bundle<FT, SPARSE>(g, lane, o, d, klo, khi, any, ws);
    float F[7];
#pragma unroll
    for (int c = 0; c < 7; c++) F[c] = ws.s.F[lane][c];
    const float T = ws.s.T[lane];
    const int cnt = ws.s.cnt[lane];
    __syncwarp();

    float yd_mma[3] = {0.0f, 0.0f, 0.0f};
    if constexpr (kMMA) {
      mlp_stage_row(ws.m, lane, valid && cnt > 0, F, d);
      mlp_bf16_warp(sFrag, ws.m, lane, yd_mma);
    }
    if (valid && (!TRAIN || LOSS)) {
      float out[3], yd[3] = {0.0f, 0.0f, 0.0f};
      if (cnt == 0) {
#pragma unroll
        for (int j = 0; j < 3; j++) out[j] = g.bg[j];
      } else {
        if constexpr (kMMA) {
#pragma unroll
          for (int j = 0; j < 3; j++) yd[j] = yd_mma[j];
        } else {
          mlp_forward_padded(sW, F, d, yd);
        }
#pragma unroll
        for (int j = 0; j < 3; j++) out[j] = F[j] + yd[j] + T * g.bg[j];
      }
      if (!TRAIN) {
#pragma unroll
        for (int j = 0; j < 3; j++) a.rgb[3 * rid + j] = out[j];
        if (a.count) a.count[rid] = cnt;
      } else {
        float e2 = 0.0f;
#pragma unroll
        for (int j = 0; j < 3; j++) {
          const float e = out[j] - __ldg(a.target + 3 * rid + j);
          e2 = fmaf(e, e, e2);
        }
        l_rgb += sqrtf(e2 + 1e-6f);
        if (cnt > 0) {
          const float dn = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
          for (int k = 0; k < a.K; k++) {
            const float* sp = a.dirs + 3 * ((long)rid * a.K + k);
            float sv[3] = {__ldg(sp), __ldg(sp + 1), __ldg(sp + 2)};
            const float sn = sqrtf(sv[0] * sv[0] + sv[1] * sv[1] + sv[2] * sv[2]);
            const float S = (d[0] * sv[0] + d[1] * sv[1] + d[2] * sv[2]) / (dn * sn);
            float sh[3] = {sv[0] / sn, sv[1] / sn, sv[2] / sn};
            float ys[3];
            mlp_forward_padded(sW, F, sh, ys);
            float q = 0.0f;
#pragma unroll
            for (int j = 0; j < 3; j++) q = fmaf(ys[j] - yd[j], ys[j] - yd[j], q);
            l_smooth = fmaf(S, q, l_smooth);
          }
        }
      }
    }
    if (TRAIN && valid) {
      float4* sv = reinterpret_cast<float4*>(a.saved + (long)kSavedFloats * rid);
      sv[0] = make_float4(F[0], F[1], F[2], F[3]);
      sv[1] = make_float4(F[4], F[5], F[6], T);
      sv[2] = make_float4(__int_as_float(cnt), __int_as_float(klo), __int_as_float(khi), 0.0f);
    }
  }

  if (TRAIN && LOSS) {
    l_rgb = warp_sum(l_rgb);
    l_smooth = warp_sum(l_smooth);
    if (lane == 0) {
      sLoss[0][threadIdx.x >> 5] = l_rgb;
      sLoss[1][threadIdx.x >> 5] = l_smooth;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float s0 = 0.0f, s1 = 0.0f;
      for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
        s0 += sLoss[0][w];
        s1 += sLoss[1][w];
      }
      s0 *= a.lam_rgb;
      s1 *= a.lam_smooth;
      atomicAdd(a.loss + 1, s0);
      atomicAdd(a.loss + 2, s1);
      atomicAdd(a.loss + 0, s0 + s1);
    }
  }
}

#ifndef OMERF_CARVEOUT
#define OMERF_CARVEOUT 1
#endif
int persistent_blocks(const void* kernel, int threads, size_t smem, int num_sms) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
#if OMERF_CARVEOUT
  // The marches' gathers are served from L1, which shares each SM's SRAM
  // with shared memory: ask for the smallest shared-memory carveout that
  // still holds per_sm blocks (with the driver's 1 KB per block), leaving
  // the rest to L1; keep it only if the occupancy still holds.
  cudaFuncAttributes fa;
  int dev = 0, max_smem = 0;
  if (cudaFuncGetAttributes(&fa, kernel) == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess &&
      max_smem > 0) {
    const size_t need = (fa.sharedSizeBytes + smem + 1024) * (size_t)per_sm;
    const int pct = (int)((need * 100 + (size_t)max_smem - 1) / (size_t)max_smem);
    if (pct < 100 && cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct) == cudaSuccess) {
      int again = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&again, kernel, threads, smem) != cudaSuccess ||
          again < per_sm)
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutDefault);
    }
  }
  cudaGetLastError();  // a refused hint is not an error of the launch
#endif
  return per_sm * num_sms;
}

template <class FT, bool SPARSE, bool TRAIN, bool LOSS = TRAIN>
static cudaError_t launch_variant(const omerf_scene* s, const FwdArgs& a, cudaStream_t stream) {
  auto kern = march_fwd_kernel<FT, SPARSE, TRAIN, LOSS>;
  static std::atomic<int> blocks[64];  // per device: resident CTAs of this variant
  const int dev = s->device & 63;
  int nb = blocks[dev].load(std::memory_order_relaxed);
  if (nb == 0) {
    nb = persistent_blocks((const void*)kern, kThreads, 0, s->num_sms);
    blocks[dev].store(nb, std::memory_order_relaxed);
  }
  // units: super-tiles of a camera, one CTA each; bundles of a list, one warp each
  const long want = a.use_cam ? a.n_super : (a.n_super + kThreads / 32 - 1) / (kThreads / 32);
  const int grid = (int)(want < nb ? want : nb);
  FwdArgs b = a;
  // every unit has its CTA or warp: no work counter (and no launch to zero it)
  b.counter = want <= grid ? nullptr : next_counter(s, stream);
  kern<<<grid < 1 ? 1 : grid, kThreads, 0, stream>>>(s->geo, b);
  return cudaGetLastError();
}

cudaError_t launch_march_fwd(const omerf_scene* s, const Cam* cam, const float* rays, long n, float* rgb,
                             int* count, const float* target, const float* dirs, int K, const float lam[3],
                             float* saved, float* loss, cudaStream_t stream) {
  FwdArgs a{};
  const bool train = saved != nullptr;
  int lanes = 0;
  if (cam) {
    a.cam = *cam;
    a.use_cam = 1;
    int sw, sh;
    lanes = cam_lanes(s, n, count != nullptr);
    cam_super(lanes, cam->width, cam->height, a.lw, sw, sh);
    a.super_x = (cam->width + sw - 1) / sw;
    a.n_super = (long)a.super_x * ((cam->height + sh - 1) / sh);
  } else {
    a.use_cam = 0;
    lanes = train ? 0 : list_lanes(s, n);
    const int per = lanes > 0 ? 16 : 32;  // rays of a CTA with 8 lanes per ray, or of a warp
    a.n_super = (n + per - 1) / per;
  }
  a.rays = rays;
  a.n = n;
  a.rgb = rgb;
  a.count = count;
  a.target = target;
  a.dirs = dirs;
  a.K = K;
  if (train) {
    a.lam_rgb = n > 0 ? lam[0] / (float)n : 0.0f;
    a.lam_smooth = n > 0 ? lam[1] / (float)n : 0.0f;
  }
  a.saved = saved;
  a.loss = loss;
  if (a.n_super == 0) return cudaSuccess;
  if (lanes > 0) return launch_render_cam(s, a, lanes, stream);
  const bool bf16 = s->desc.feat_dtype == OMERF_BF16;
  const bool sparse = s->desc.brick > 0;
  if (train && loss) {
    if (bf16) return sparse ? launch_variant<__nv_bfloat16, true, true>(s, a, stream)
                            : launch_variant<__nv_bfloat16, false, true>(s, a, stream);
    return sparse ? launch_variant<float, true, true>(s, a, stream) : launch_variant<float, false, true>(s, a, stream);
  }
  if (train) {
    if (bf16) return sparse ? launch_variant<__nv_bfloat16, true, true, false>(s, a, stream)
                            : launch_variant<__nv_bfloat16, false, true, false>(s, a, stream);
    return sparse ? launch_variant<float, true, true, false>(s, a, stream)
                  : launch_variant<float, false, true, false>(s, a, stream);
  }
  if (bf16) return sparse ? launch_variant<__nv_bfloat16, true, false>(s, a, stream)
                          : launch_variant<__nv_bfloat16, false, false>(s, a, stream);
  return sparse ? launch_variant<float, true, false>(s, a, stream) : launch_variant<float, false, false>(s, a, stream);
}


cudaError_t launch_march_fwd_cams(const omerf_scene* s, const CamRec* cams, int n_cams, int lanes, long n_super, long n,
                                  float* rgb, int* count, cudaStream_t stream) {
  FwdArgs a{};
  a.use_cam = 1;
  a.cams = cams;
  a.n_cams = n_cams;
  a.n_super = n_super;
  a.n = n;
  a.rgb = rgb;
  a.count = count;
  if (a.n_super == 0) return cudaSuccess;
  if (lanes > 0) return launch_render_cam(s, a, lanes, stream);
  // (a BF16 scene)
  return s->desc.brick > 0 ? launch_variant<__nv_bfloat16, true, false>(s, a, stream)
                           : launch_variant<__nv_bfloat16, false, false>(s, a, stream);
}

}  // namespace omerf
