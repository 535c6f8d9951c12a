// march_fwd.cuh -- the packed forward march of one bundle of 32 rays and the
// launch arguments shared by the forward kernels (march_fwd.cu, march_cam.cu).
#pragma once

#include <type_traits>

#include "internal.h"
#include "mlp_mma.cuh"
#include "packed.cuh"

namespace omerf {

// Per-warp shared state of the packed march of one bundle of 32 rays.
struct MarchState {
  WarpQueue q;
  float F[32][8];    // per-ray accumulated [sum w c^d, sum w f]
  float T[32];       // per-ray transmittance so far
  int cnt[32];       // per-ray evaluated samples
};
// With the tensor-core MLP the whole march state doubles as the warp's MLP
// staging area.  Two warp barriers separate the uses: the one after each ray's
// F, T and count are copied to registers, before the MLP rows are staged, and
// the one that ends mlp_bf16_warp, after the outputs are read and before the
// next bundle's state is written (a warp takes its next bundle of a list on its
// own: there is no CTA barrier in between).  The smaller per-warp footprint lets
// the BF16 render take a smaller shared-memory carveout, leaving more of the
// SM's SRAM to L1.
template <bool MMA>
struct WarpMarch {
  MarchState s;
};
template <>
struct WarpMarch<true> {
  union {
    MarchState s;
    MlpStage m;
  };
};

// March the 32 rays of a bundle (lane r owns ray r: o, d, [klo, khi]).
//
// fill:    evaluated samples of consecutive rays are queued, 32 at a time
//          (packed.cuh);
// process: the 32 queued samples are gathered and activated in parallel;
//          compositing is a segmented lane scan (segments = rays) of
//          1 - alpha_hat, early termination is resolved per segment, and
//          the weighted features are summed per segment into the ray's
//          accumulator.
// On return ws.s.F / ws.s.T / ws.s.cnt hold every ray's F, T_N and sample count.
template <class FT, bool SPARSE, class WS>
__device__ __forceinline__ void march_bundle(const Geo& g, int lane, const float o[3], const float d[3], int klo,
                                             int khi, bool any, WS& ws) {
#pragma unroll
  for (int c = 0; c < 8; c++) ws.s.F[lane][c] = 0.0f;
  ws.s.T[lane] = 1.0f;
  ws.s.cnt[lane] = 0;
  queue_ray(g, ws.s.q, lane, o, d, klo, any ? khi : klo - 1, g.n_max);
  unsigned pend = __ballot_sync(kFull, any);
  FillState f;
  __syncwarp();
  while (pend) {
    const int nq = fill_queue(g, lane, pend, f, ws.s.q);
    if (nq == 0) break;
    const bool act = lane < nq;
    const float4 qa = ws.s.q.a[lane], qb = ws.s.q.b[lane];
    const int r = act ? __float_as_int(qb.y) : 32;
    SampleAct s;
    s.ah = 0.0f;
#pragma unroll
    for (int c = 0; c < 7; c++) s.x[c] = 0.0f;
    if (act) {
      const float p[3] = {qa.x, qa.y, qa.z};
      float t[8];
      gather_features<FT, SPARSE>(g, p, t);
      activate(g, t, p[2], make_float2(qa.w, qb.x), s);
    }
    bool head;
    const int segstart = segment_start(lane, r, head);
    // transmittance: segmented inclusive product scan of (1 - alpha_hat)
    const float P = seg_prod_scan(__fsub_rn(1.0f, s.ah), lane, segstart);
    float Pex = __shfl_up_sync(kFull, P, 1);
    if (head) Pex = 1.0f;
    const float Tprev = act ? ws.s.T[r] : 1.0f;
    const float Ti = Tprev * Pex, Tn = Tprev * P;
    // early termination: the first sample of a segment whose T drops below t_thr ends the ray
    const bool term = act && Tn < g.t_thr;
    const unsigned tm = __ballot_sync(kFull, term);
    const unsigned seglt = lanemask_lt() & ~((1u << segstart) - 1u);
    const bool dropped = (tm & seglt) != 0u;
    const bool ok = act && !dropped;
    const float w = ok ? Ti * s.ah : 0.0f;
    float wx[7];
#pragma unroll
    for (int c = 0; c < 7; c++) wx[c] = w * s.x[c];
    seg_sum_scan7(wx, lane, segstart);
    const unsigned okm = __ballot_sync(kFull, ok);
    const int rnext = __shfl_down_sync(kFull, r, 1);
    const bool tail = act && (lane == 31 || rnext != r);
    const unsigned segle = lanemask_le() & ~((1u << segstart) - 1u);
    if (tail) {
#pragma unroll
      for (int c = 0; c < 7; c++) ws.s.F[r][c] += wx[c];
      ws.s.cnt[r] += __popc(okm & segle);
      if (!(tm & segle)) ws.s.T[r] = Tn;
    }
    const bool first_term = term && !dropped;
    if (first_term) ws.s.T[r] = Tn;
    pend &= ~__reduce_or_sync(kFull, first_term ? (1u << r) : 0u);
    __syncwarp();
  }
}

struct FwdArgs {
  Cam cam;
  int use_cam, super_x, lw;  // lw: the super-tiles' form (march_cam.cu)
  const float* rays;
  long n, n_super;
  float* rgb;
  int* count;
  // training
  const float* target;
  const float* dirs;
  int K;
  float lam_rgb, lam_smooth;  // already divided by n
  float* saved;
  float* loss;
  unsigned* counter;
  // multi-camera render (n_cams > 0): device camera records, super-tiles in
  // camera order
  const CamRec* cams;
  int n_cams;
};

// Relative distance from the termination threshold within which the order of
// the transmittance's products could decide a sample: the queue rounds at most
// cnt products by 2^-24 each, march_cam.cu's own transmittance (compensated)
// is good to two roundings.  The factors are the same in both.
__device__ __forceinline__ float ambiguity(int cnt) { return 2.5e-7f + 6.2e-8f * (float)cnt; }

// Camera render with `lanes` lanes per ray (march_cam.cu).
cudaError_t launch_render_cam(const omerf_scene* s, const FwdArgs& a, int lanes, cudaStream_t stream);

}  // namespace omerf
