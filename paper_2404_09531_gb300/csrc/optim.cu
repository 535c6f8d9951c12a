// optim.cu -- fused Adam step over the scene's parameter groups and the
// training schedules of Oblique-MERF (appendix A).
//
// One launch updates every group: the threads walk the concatenation of the
// groups (at most 8), each element reading p, g, m, v and writing p, m, v and,
// for a group with a BF16 shadow (BF16 features with an FP32 master copy),
// the rounded value.  HBM-bound: 28 B per element (30 B with a shadow).
#include <cmath>

#include "internal.h"

namespace omerf {

constexpr int kMaxGroups = 8;

struct AdamArgs {
  float* p[kMaxGroups];
  const float* g[kMaxGroups];
  float* m[kMaxGroups];
  float* v[kMaxGroups];
  __nv_bfloat16* shadow[kMaxGroups];
  long n[kMaxGroups];    // elements
  bool vec[kMaxGroups];  // arrays aligned for 16-byte accesses (the shadow for 8-byte ones)
  long end[kMaxGroups];  // inclusive prefix of the groups' units of 4 elements
  float lr_c[kMaxGroups];  // lr / (1 - beta1^t)
  int n_groups;
  long units;
  float b1, b2, inv_bc2, eps;
};

// One element: p, m, v updated in place.
__device__ __forceinline__ void adam_element(const AdamArgs& a, float lr_c, float g, float& m, float& v, float& p) {
  m = a.b1 * m + (1.0f - a.b1) * g;
  v = a.b2 * v + (1.0f - a.b2) * g * g;
  p = p - lr_c * m / (sqrtf(v * a.inv_bc2) + a.eps);
}

// A thread's unit is four elements of one group: four neighbours with 16-byte
// loads and stores (8-byte for the shadow) and element by element at the
// group's ragged end; in arrays that are not aligned for them, elements 32 apart
// among the 128 of 32 threads, so that a warp's accesses stay contiguous (2^24
// unaligned elements: 140 us with four neighbours, 80 us with these).
// HBM-bound: 47.9 M parameters with BF16 shadows (1.44 GB) take 225 us, 94 %
// of the measured copy bandwidth; 295 us with 4-byte accesses.
__global__ void __launch_bounds__(256) adam_kernel(const AdamArgs a) {
  for (long u = (long)blockIdx.x * blockDim.x + threadIdx.x; u < a.units; u += (long)gridDim.x * blockDim.x) {
    int q = 0;
    while (q < a.n_groups - 1 && u >= a.end[q]) q++;
    const long unit = u - (q ? a.end[q - 1] : 0), j = 4 * unit;
    const float lr_c = a.lr_c[q];
    if (a.vec[q] && j + 4 <= a.n[q]) {
      const float4 g = __ldg(reinterpret_cast<const float4*>(a.g[q] + j));
      float4 m = *reinterpret_cast<const float4*>(a.m[q] + j);
      float4 v = *reinterpret_cast<const float4*>(a.v[q] + j);
      float4 p = *reinterpret_cast<const float4*>(a.p[q] + j);
      adam_element(a, lr_c, g.x, m.x, v.x, p.x);
      adam_element(a, lr_c, g.y, m.y, v.y, p.y);
      adam_element(a, lr_c, g.z, m.z, v.z, p.z);
      adam_element(a, lr_c, g.w, m.w, v.w, p.w);
      *reinterpret_cast<float4*>(a.m[q] + j) = m;
      *reinterpret_cast<float4*>(a.v[q] + j) = v;
      *reinterpret_cast<float4*>(a.p[q] + j) = p;
      if (a.shadow[q]) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(p.x, p.y), hi = __floats2bfloat162_rn(p.z, p.w);
        *reinterpret_cast<uint2*>(a.shadow[q] + j) =
            make_uint2(*reinterpret_cast<const unsigned*>(&lo), *reinterpret_cast<const unsigned*>(&hi));
      }
    } else {
      // the aligned arrays' ragged end, or 128 elements of unaligned arrays
      const long e0 = a.vec[q] ? j : (unit >> 5) * 128 + (unit & 31);
      const int step = a.vec[q] ? 1 : 32;
      float g[4], m[4], v[4], p[4];
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const long e = e0 + k * step;
        if (e >= a.n[q]) continue;
        g[k] = __ldg(a.g[q] + e);
        m[k] = a.m[q][e];
        v[k] = a.v[q][e];
        p[k] = a.p[q][e];
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const long e = e0 + k * step;
        if (e >= a.n[q]) continue;
        adam_element(a, lr_c, g[k], m[k], v[k], p[k]);
        a.m[q][e] = m[k];
        a.v[q][e] = v[k];
        a.p[q][e] = p[k];
        if (a.shadow[q]) a.shadow[q][e] = __float2bfloat16_rn(p[k]);
      }
    }
  }
}

}  // namespace omerf

using namespace omerf;

extern "C" {

omerf_status omerf_adam_step(const omerf_adam_group* groups, int32_t n_groups, float beta1, float beta2, float eps,
                             int64_t step, void* stream) {
  OMERF_API_RANGE();
  if (!groups || n_groups < 1 || n_groups > kMaxGroups) {
    set_error("n_groups must be in 1..%d", kMaxGroups);
    return OMERF_EINVAL;
  }
  if (!(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps >= 0.0f) || step < 1) {
    set_error("need 0 <= beta < 1, eps >= 0 and step >= 1");
    return OMERF_EINVAL;
  }
  AdamArgs a{};
  long total = 0;
  for (int q = 0; q < n_groups; q++) {
    const omerf_adam_group& gr = groups[q];
    if (gr.n < 0 || (gr.n > 0 && (!gr.param || !gr.grad || !gr.m || !gr.v)) || !std::isfinite(gr.lr)) {
      set_error("adam group %d: null array or bad size / learning rate", q);
      return OMERF_EINVAL;
    }
    a.p[q] = gr.param;
    a.g[q] = gr.grad;
    a.m[q] = gr.m;
    a.v[q] = gr.v;
    a.shadow[q] = static_cast<__nv_bfloat16*>(gr.shadow_bf16);
    a.n[q] = gr.n;
    a.vec[q] = aligned(gr.param, 16) && aligned(gr.grad, 16) && aligned(gr.m, 16) && aligned(gr.v, 16) &&
               aligned(gr.shadow_bf16, 8);
    total += a.vec[q] ? (gr.n + 3) / 4 : (gr.n + 127) / 128 * 32;
    a.end[q] = total;
    // bias corrections in double on the host, applied as FP32 constants
    a.lr_c[q] = (float)((double)gr.lr / (1.0 - std::pow((double)beta1, (double)step)));
  }
  a.n_groups = n_groups;
  a.units = total;
  a.b1 = beta1;
  a.b2 = beta2;
  a.inv_bc2 = (float)(1.0 / (1.0 - std::pow((double)beta2, (double)step)));
  a.eps = eps;
  if (total == 0) return OMERF_OK;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long want = (total + 255) / 256;
  const int grid = (int)(want < 8L * sms ? want : 8L * sms);
  OMERF_LAUNCH_FAULT();
  for (int q = 0; q < n_groups; q++) {
    const omerf_adam_group& gr = groups[q];
    const omerf_status st = check_device_ptrs(
        {{gr.param, "param"}, {gr.grad, "grad"}, {gr.m, "m"}, {gr.v, "v"}, {gr.shadow_bf16, "shadow_bf16"}});
    if (st != OMERF_OK) return st;
  }
  adam_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(a);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OMERF_OK : cuda_fail(e, "adam kernel");
}

float omerf_lr_exponential(float lr0, float lr1, int64_t step, int64_t total) {
  if (total <= 0) return lr1;
  const double s = (double)(step < 0 ? 0 : (step > total ? total : step)) / (double)total;
  return (float)((double)lr0 * std::pow((double)lr1 / (double)lr0, s));
}

float omerf_lambda_occ(int64_t step) {
  if (step < 10000) return 0.0f;
  const int64_t k = (step - 10000) / 2000;
  if (k >= 20) return 0.2f;
  const double v = 1e-4 * std::pow(1.5, (double)k);
  return (float)(v < 0.2 ? v : 0.2);
}

}  // extern "C"
