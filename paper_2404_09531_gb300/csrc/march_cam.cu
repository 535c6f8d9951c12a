// march_cam.cu -- FP32 render with a fixed set of lanes per ray: cameras and
// short ray lists (sm_103a).
//
// The L1 data pipe bounds the render: a 256-bit texel load takes one
// wavefront per distinct 128-byte line in each group of four lanes, 20 loads
// per sample, and the packed queue of march_fwd.cu adds a quarter more for
// its shared-memory queue and segmented scans.  Neighbouring pixels march
// through neighbouring texels and evaluate nearly the same number of samples
// (95 % of the lanes stay busy when the 32 rays of an 8 x 4 tile are marched
// one per lane), so a camera needs no queue: every ray is marched by its own
// G lanes, which keep its transmittance and sums in registers.
//   G = 1  one lane per ray; the four lanes of a 2 x 2 pixel quad share a
//          lattice frame, so the lanes of a load group sample one depth (254
//          wavefronts per 32 samples by a replay, 293 without the frame)
//   G = 4, 8  the lanes of a ray take its next samples together: a ray's
//          serial chain is 4 or 8 times shorter and there are 4 or 8 times
//          the warps, for images too small to fill the chip with G = 1
// A frame skips the 32-index windows that the coarse occupancy grid rules
// out, tests a whole window at a time and then takes the evaluated samples.
// Texel pairs are read in even / odd order (216 wavefronts, see even_odd)
// with two channels per FMA.  All forms composite a ray's samples one after
// the other in the same order, so a pixel does not depend on G, nor on
// whether counts are wanted.
//
// Measured on a GB300, 512 x 512 x 32 city, against the packed queue: 8 x
// 1920x1080 29.4 -> 19.4 ms (L1 pipe 81 % busy, 1.9 G instead of 2.7 G
// instructions per frame), 1920x1080 3.75 -> 2.53 ms, 640x360 0.83 -> 0.43 ms (G =
// 8: 0.45, G = 1: 0.78), 64x64 of the 64 x 64 x 16 field with counts 0.113 ->
// 0.030 ms.
//
// Sample counts are those of the packed queue, which training and long ray
// lists use, also where rounding decides them.  The two forms multiply a
// ray's transmittance in different orders: where counts are wanted the
// density is also summed in the queue's order, its transmittance (compensated,
// so that the queue's rounding alone is in doubt) decides the count, and a ray
// that passes the termination threshold within that rounding (1 of 2 x 10^5 in
// the city, 1 of 80 in fog of 0.01 per sample) is counted again in the queue's
// order (see "Counts in the queue's order").
#include "march_fwd.cuh"

namespace omerf {

// Warps per CTA and the pixels of its super-tile (whole or half 8 x 4 tiles).
// CTAs of 4 warps wait less for their slowest tile than CTAs of 8 (an earlier
// state of the kernel: 2.96 against 3.10 ms per 1080p frame; 2 warps 3.05).
template <int G>
struct CamShape;
template <>
struct CamShape<1> {
  static constexpr int kWarps = 4, kW = 16, kH = 8, kRays = kW * kH;
};
template <>
struct CamShape<4> {
  static constexpr int kWarps = 4, kW = 8, kH = 4, kRays = kW * kH;
};
template <>
struct CamShape<8> {
  static constexpr int kWarps = 4, kW = 4, kH = 4, kRays = kW * kH;
};

// Pixel of a lane's ray inside the super-tile.
template <int G>
__device__ __forceinline__ void lane_pixel(int warp, int lane, int& x, int& y) {
  if (G == 1) {  // 8 x 4 pixels per warp, quads of 2 x 2
    const int q = lane >> 2, j = lane & 3;
    x = (warp & 1) * 8 + (q & 3) * 2 + (j & 1);
    y = (warp >> 1) * 4 + (q >> 2) * 2 + (j >> 1);
  } else if (G == 4) {  // 4 x 2 pixels per warp
    const int r = lane >> 2;
    x = (warp & 1) * 4 + (r & 3);
    y = (warp >> 1) * 2 + (r >> 2);
  } else {  // 2 x 2 pixels per warp
    const int r = lane >> 3;
    x = (warp & 1) * 2 + (r & 1);
    y = (warp >> 1) * 2 + (r >> 1);
  }
}

// Images of one or two rows, or of up to four columns (two for G = 8), would
// leave most pixels of such a super-tile empty.  They are cut into sub-tiles of
// 2^lw columns with as many rays as a CTA (G = 4, 8) or a warp (G = 1) takes,
// which holds whole 8 x 4 bundles of the queue, as far as the image has pixels
// there: ray i is the pixel at place i of the bundles' pixels, one bundle after
// the other.  (us, city pixels in one column / row with the queue, plain
// super-tiles and these: 900,000 pixels 2782 / 4798, 8368 / 6502, 824 / 1326;
// 60,000 pixels 212 / 376, 278 / 409, 131 / 194.)
struct SubTile {
  int lw, lbw, lbh;  // log2 of the width, and of the bundles' width and height in the image
  template <int G>
  static constexpr int kLog = G == 8 ? 4 : 5;
};
template <int G>
__device__ __forceinline__ SubTile sub_tile(int lw) {
  return {lw, min(lw, 3), min(SubTile::kLog<G> - lw, 2)};
}
__device__ __forceinline__ void sub_pixel(const SubTile& t, int i, int& x, int& y) {
  const int b = i >> (t.lbw + t.lbh), w = i & ((1 << (t.lbw + t.lbh)) - 1), lnx = t.lw - t.lbw;
  x = ((b & ((1 << lnx) - 1)) << t.lbw) + (w & ((1 << t.lbw) - 1));
  y = ((b >> lnx) << t.lbh) + (w >> t.lbw);
}
// Origin of a warp's sub-tile (G = 1: four of them, along the image) in its super-tile.
template <int G>
__device__ __forceinline__ void sub_origin(int lw, int warp, int& x, int& y) {
  if (G != 1) return;
  if (lw < 0) {
    x += (warp & 1) * 8;
    y += (warp >> 1) * 4;
  } else if (lw < 3) {
    y += warp * (32 >> lw);
  } else {
    x += warp << lw;
  }
}

// The pixels of a super-tile.
static __host__ __device__ __forceinline__ void super_size(int lanes, int lw, int& w, int& h) {
  if (lw < 0) {
    w = lanes == 1 ? CamShape<1>::kW : (lanes == 4 ? CamShape<4>::kW : CamShape<8>::kW);
    h = lanes == 1 ? CamShape<1>::kH : (lanes == 4 ? CamShape<4>::kH : CamShape<8>::kH);
  } else {
    w = 1 << lw;
    h = (lanes == 8 ? 16 : 32) >> lw;
    if (lanes == 1) (lw < 3 ? h : w) *= 4;
  }
}

// The deferred MLP's weights with the units of a layer as the fast axis, so that
// two units share one packed FMA: W1 [34][16], b1 [16], W2 [16][16], b2 [16],
// W3 [16][4 (3 used)], b3 [4 (3 used)].
constexpr int kTW1 = 0, kTB1 = 544, kTW2 = 560, kTB2 = 816, kTW3 = 832, kTB3 = 896, kSmemMlpT = 900;

__device__ __forceinline__ void load_mlp_units(const float* __restrict__ gw, float* __restrict__ sw) {
  for (int i = threadIdx.x; i < kSmemMlpT; i += blockDim.x) {
    float v = 0.0f;
    if (i < kTB1) v = gw[kOffW1 + (i & 15) * 34 + (i >> 4)];
    else if (i < kTW2) v = gw[kOffB1 + i - kTB1];
    else if (i < kTB2) v = gw[kOffW2 + ((i - kTW2) & 15) * 16 + ((i - kTW2) >> 4)];
    else if (i < kTW3) v = gw[kOffB2 + i - kTB2];
    else if (i < kTB3) v = ((i - kTW3) & 3) < 3 ? gw[kOffW3 + ((i - kTW3) & 3) * 16 + ((i - kTW3) >> 2)] : 0.0f;
    else v = i - kTB3 < 3 ? gw[kOffB3 + i - kTB3] : 0.0f;
    sw[i] = v;
  }
}

// N units from u0 of one layer: h = relu(b + sum_i x_i W[i][u]), two units per FMA.
template <int N, int IN>
__device__ __forceinline__ void mlp_units(const float* __restrict__ W, const float* __restrict__ b, int u0,
                                          const float x[IN], float h[N]) {
  float2 acc[N / 2];
#pragma unroll
  for (int q = 0; q < N / 2; q++) acc[q] = *reinterpret_cast<const float2*>(b + u0 + 2 * q);
#pragma unroll
  for (int i = 0; i < IN; i++) {
    const float2 xx = make_float2(x[i], x[i]);
#pragma unroll
    for (int q = 0; q < N / 4; q++) {
      const float4 w = *reinterpret_cast<const float4*>(W + 16 * i + u0 + 4 * q);
      acc[2 * q] = __ffma2_rn(xx, make_float2(w.x, w.y), acc[2 * q]);
      acc[2 * q + 1] = __ffma2_rn(xx, make_float2(w.z, w.w), acc[2 * q + 1]);
    }
    if (N == 2) acc[0] = __ffma2_rn(xx, *reinterpret_cast<const float2*>(W + 16 * i + u0), acc[0]);
  }
#pragma unroll
  for (int q = 0; q < N / 2; q++) {
    h[2 * q] = fmaxf(acc[q].x, 0.0f);
    h[2 * q + 1] = fmaxf(acc[q].y, 0.0f);
  }
}

// G(F, d) with the encoding's angles and the units of each layer spread over
// the G lanes of a ray (every unit summed in the same order whatever G): all
// three outputs for G = 1, output j in y[0] of lane j < 3 else.  Every sine and
// cosine of the encoding is sincosf of its own angle, as in view_encoding:
// doubling those of d is cheaper but loses a factor of ten at 8 d.  All lanes
// of the warp call it for G > 1.
template <int G>
__device__ __forceinline__ void mlp_rays(const float* __restrict__ W, const float F[7], const float d[3], int j,
                                         float y[3]) {
  constexpr int N = 16 / G;
  float x[34], h[N], a[16];
#pragma unroll
  for (int i = 0; i < 7; i++) x[i] = F[i];
  x[7] = d[0];
  x[8] = d[1];
  x[9] = d[2];
  // angle 3 k + c is 2^k d_c: its sine is input 10 + 6 k + c, its cosine 13 + 6 k + c
  float sn[(12 + G - 1) / G], cs[(12 + G - 1) / G];
#pragma unroll
  for (int t = 0; t < (12 + G - 1) / G; t++) {
    const int m = min(t * G + j, 11), k = m / 3, c = m - 3 * k;
    sincosf((float)(1 << k) * (c == 0 ? d[0] : (c == 1 ? d[1] : d[2])), &sn[t], &cs[t]);
  }
#pragma unroll
  for (int m = 0; m < 12; m++) {
    const int at = 10 + 6 * (m / 3) + m % 3;
    x[at] = G == 1 ? sn[m / G] : __shfl_sync(kFull, sn[m / G], m % G, G);
    x[at + 3] = G == 1 ? cs[m / G] : __shfl_sync(kFull, cs[m / G], m % G, G);
  }
  mlp_units<N, 34>(W + kTW1, W + kTB1, N * j, x, h);
#pragma unroll
  for (int u = 0; u < 16; u++) a[u] = G == 1 ? h[u % N] : __shfl_sync(kFull, h[u % N], u / N, G);
  mlp_units<N, 16>(W + kTW2, W + kTB2, N * j, a, h);
#pragma unroll
  for (int u = 0; u < 16; u++) a[u] = G == 1 ? h[u % N] : __shfl_sync(kFull, h[u % N], u / N, G);
  if (G == 1) {
    float2 o[2] = {make_float2(W[kTB3], W[kTB3 + 1]), make_float2(W[kTB3 + 2], 0.0f)};
#pragma unroll
    for (int i = 0; i < 16; i++) {
      const float4 w = *reinterpret_cast<const float4*>(W + kTW3 + 4 * i);
      const float2 xx = make_float2(a[i], a[i]);
      o[0] = __ffma2_rn(xx, make_float2(w.x, w.y), o[0]);
      o[1] = __ffma2_rn(xx, make_float2(w.z, w.w), o[1]);
    }
    y[0] = sigmoidf_(o[0].x);
    y[1] = sigmoidf_(o[0].y);
    y[2] = sigmoidf_(o[1].x);
  } else {
    const int o = min(j, 2);
    float v = W[kTB3 + o];
#pragma unroll
    for (int i = 0; i < 16; i++) v = fmaf(a[i], W[kTW3 + 4 * i + o], v);
    y[0] = sigmoidf_(v);
  }
}

// The evaluated lattice indices of a window, [k0, k0 + 31] clipped to the ray's
// [klo, khi]: every lane of a ray tests 32 / G of them with the decision rule.
// A run of tests without votes or branches in between: one candidate per
// step of the march, with a vote each, took 36 % of a frame's instructions.
template <int G>
__device__ __forceinline__ unsigned window_samples(const Geo& g, const float o[3], const float d[3], int k0, int klo,
                                                   int khi, int j) {
  unsigned m = 0;
#pragma unroll 8
  for (int i = 0; i < 32; i += G) {
    float p[3];
    lattice_point(g, o, d, k0 + i + j, p);
    const bool in = p[0] >= g.lo[0] && p[0] <= g.hi[0] && p[1] >= g.lo[1] && p[1] <= g.hi[1] && p[2] >= g.lo[2] &&
                    p[2] <= g.hi[2];
    float2 zb = make_float2(0.0f, 0.0f);
    if (in) zb = __ldg(g.occ + occ_cell(g, p));
    if (in && zb.x < p[2] && p[2] < zb.y) m |= 1u << (i + j);
  }
  const int lo = max(klo - k0, 0), hi = min(khi - k0, 31);
  return lo > hi ? 0u : m & (~0u << lo) & (~0u >> (31 - hi));
}

// The bits of a ballot that belong to the lanes of this lane's ray.
template <int G>
__device__ __forceinline__ unsigned hits_of(bool v, int base) {
  return (__ballot_sync(kFull, v) >> base) & ((1u << G) - 1u);
}

// Transpose the values of a ray's G lanes in blocks of G: v[b G + i] of lane j
// becomes lane i's v[b G + j].  log2 G exchanges of half the values (12
// shuffles for G = 8, 8 for G = 4) let every lane sum its own channels (a
// broadcast of all values, summed by every lane, took 64 and 32: 641x361
// pixels 484 -> 450 us, 10,007 listed rays 156 -> 148 us).
template <int G>
__device__ __forceinline__ void transpose_lanes(float v[8], int j) {
#pragma unroll
  for (int s = 1; s < G; s <<= 1) {
    const bool bit = j & s;
#pragma unroll
    for (int r = 0; r < 8; r++) {
      if (r & s) continue;
      const float got = __shfl_xor_sync(kFull, bit ? v[r] : v[r | s], s);
      if (bit) v[r] = got;
      else v[r | s] = got;
    }
  }
}

// The sums over a ray's samples are compensated: a ray's samples are taken one
// after the other, where the packed queue's lane scans round a sample's
// contribution about five times whatever the ray's length, and a plain sum
// in order would be coarser (pixels of rays of 700 samples 3.7e-7 off 64-bit
// ones instead of 1.8e-7, root mean square; with the compensation 1.6e-7; it
// costs a 1080p frame 2 % and small images of few samples up to 5 %).
//
// Transmittance T = h + l, the rounding errors of h's products carried along.
struct Through {
  float h = 1.0f, l = 0.0f;
  __device__ __forceinline__ float value() const { return __fadd_rn(h, l); }
  __device__ __forceinline__ void pass(float om) {  // through a sample with 1 - opacity om
    const float p = __fmul_rn(h, om);
    l = fmaf(l, om, fmaf(h, om, -p));
    h = p;
  }
};
// A sum s + c of terms w x: the error of every sum is the term less what it
// changed s by, added up in c beside the chain of s.
__device__ __forceinline__ void add_to(float& s, float& c, float w, float x) {
  const float t = fmaf(w, x, s);
  c = __fadd_rn(c, fmaf(w, x, __fsub_rn(s, t)));
  s = t;
}
// The same for two channels, packed (s - t as t (-1) + s: one rounding).
__device__ __forceinline__ void add_to2(float2& s, float2& c, float w, float x0, float x1) {
  const float2 ww = make_float2(w, w), x = make_float2(x0, x1);
  const float2 t = __ffma2_rn(ww, x, s);
  c = __fadd2_rn(c, __ffma2_rn(ww, x, __ffma2_rn(t, make_float2(-1.0f, -1.0f), s)));
  s = t;
}

// A ray's transmittance T carried through its G lanes' opacities in lane
// order, in place: T becomes the transmittance before this lane's sample, or
// after it (`after`); `last` is the lane whose sample takes it below thr, G if
// none does.
template <int G>
__device__ __forceinline__ void chain(Through& T, Through& after, float ah, bool hit, int j, int base, float thr,
                                      int& last) {
  const float om = __fsub_rn(1.0f, ah);
#pragma unroll
  for (int i = 0; i < G - 1; i++) {
    const float v = __shfl_sync(kFull, om, i, G);
    if (i < j) T.pass(v);
  }
  after = T;
  after.pass(om);
  const unsigned below = hits_of<G>(hit && after.value() < thr, base);
  last = below ? __ffs(below) - 1 : G;
}

// The camera of super-tile sb, its form (see SubTile), pixel origin and first ray.
template <int G>
__device__ __forceinline__ const Cam& tile_camera(const FwdArgs& a, unsigned sb, int& lw, int& x0, int& y0,
                                                  long& ray0) {
  const Cam* cam = &a.cam;
  int super_x = a.super_x;
  lw = a.lw;
  ray0 = 0;
  if (a.n_cams > 0) {
    int c = 0;
    while (c + 1 < a.n_cams && (long long)sb >= a.cams[c + 1].super_start) c++;
    const CamRec& cr = a.cams[c];
    sb = (unsigned)((long long)sb - cr.super_start);
    cam = &cr.cam;
    super_x = cr.super_x;
    lw = cr.lw;
    ray0 = (long)cr.ray_start;
  }
  int w, h;
  super_size(G, lw, w, h);
  x0 = (int)(sb % (unsigned)super_x) * w;
  y0 = (int)(sb / (unsigned)super_x) * h;
  return *cam;
}

__device__ __forceinline__ void load_ray(const float* __restrict__ r, float o[3], float d[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    o[c] = __ldg(r + c);
    d[c] = __ldg(r + 3 + c);
  }
}

// ---------------------------------------------------------------------------
// Counts in the queue's order
//
// The queue takes a bundle's 32 rays (an 8 x 4 tile, bit 8 y + x, or 32
// consecutive rays of a list) one after the other and fills 32 places at a
// time with their evaluated samples; the transmittance of a ray's samples in a
// batch is a lane scan from the ray's first place in it, so its rounding
// depends on where the batches cut the ray and on nothing else.  The place
// where a ray starts follows from the counts of the rays before it and from
// whether their evaluated samples fill the batch they stop in (next_place).
// So an ambiguous ray alone is marched again, 32 samples at a time by a warp,
// and the other rays of its bundle only say how many samples they have beyond
// their last one.  (Marching the whole bundle with the queue kept a CTA
// waiting for one warp: a 333x201 city camera with one such ray took 560 us
// instead of 225, 1280x720 pixels of fog of 0.01 per sample 48 ms, 15 without
// counts.  Now 225 us and 17.1 ms.)
// ---------------------------------------------------------------------------

// Of the bundle's ray r: its count and its evaluated samples up to 31 beyond
// the last counted one (or all of them); samples = -1: to be counted again.
struct BundleCounts {
  int count[32], samples[32];
};

// The queue's places filled after a ray that starts at `place`.
__device__ __forceinline__ int next_place(int place, int count, int samples) {
  const int free = 32 - place;
  if (samples <= free) return (place + samples) & 31;  // all of them fit in
  if (count <= free) return 0;                         // stopped in a batch that it filled
  const int rest = (samples - free) - ((count - free - 1) & ~31);  // for the batch of its last sample
  return rest >= 32 ? 0 : rest;
}

// A ray's evaluated samples after lattice index k, at most `want` (or a few
// more), by its G lanes.  All lanes of the warp call it.
template <int G>
__device__ __noinline__ int samples_after(const Geo& g, float o0, float o1, float o2, float d0, float d1, float d2,
                                          int k, int khi, int want, int j) {
  const float o[3] = {o0, o1, o2}, d[3] = {d0, d1, d2};
  int n = 0;
#pragma unroll 1
  for (int wb = k + 1; __any_sync(kFull, n < want && wb <= khi); wb += 1024) {
    unsigned m = 0;
    if (n < want)
      for (int jw = j; jw < 32 && wb + 32 * jw <= khi; jw += G)
        if (window_maybe(g, o, d, wb + 32 * jw, min(wb + 32 * jw + 31, khi))) m |= 1u << jw;
#pragma unroll
    for (int s = 1; s < G; s <<= 1) m |= __shfl_xor_sync(kFull, m, s);
    while (__any_sync(kFull, n < want && m != 0u)) {
      unsigned e = 0;
      if (n < want && m != 0u) {
        e = window_samples<G>(g, o, d, wb + 32 * (__ffs(m) - 1), k + 1, khi, j);
        m &= m - 1u;
      }
#pragma unroll
      for (int s = 1; s < G; s <<= 1) e |= __shfl_xor_sync(kFull, e, s);
      n += __popc(e);
    }
  }
  return n;
}

// Count a ray (the same one in every lane) as the queue does from `place`, and
// move `place` on.
template <bool SPARSE>
__device__ __forceinline__ int count_in_queue(const Geo& g, const float o[3], const float d[3], float4* sa, float* sb,
                                              int lane, int& place) {
  int klo = 0, khi = -1, count = 0, nq = place, first = place, taken = 0;
  float T = 1.0f;
  bool done = !lattice_range(g, o, d, klo, khi);
  // the batch's places [first, nq): composite them
  auto batch = [&]() {
    __syncwarp();
    const bool act = lane >= first && lane < nq;
    SampleAct s;
    s.ah = 0.0f;
    if (act) {
      const float4 q = sa[lane];
      const float p[3] = {q.x, q.y, q.z};
      float t[8];
      gather_features<float, SPARSE>(g, p, t);
      activate(g, t, p[2], make_float2(q.w, sb[lane]), s);
    }
    const float Tn = T * seg_prod_scan(__fsub_rn(1.0f, s.ah), lane, first);
    const unsigned below = __ballot_sync(kFull, act && Tn < g.t_thr);
    count += below ? __ffs(below) - first : nq - first;
    done = below != 0u;
    T = __shfl_sync(kFull, Tn, nq - 1);
    if (nq == 32) nq = 0;
    first = nq;
    __syncwarp();  // the places are read: they may be filled again
  };
  for (int wb = klo; !done && wb <= khi; wb += 1024) {
    for (unsigned wm = window_mask(g, o, d, wb, khi, lane); wm && !done; wm &= wm - 1u) {
      const int k = wb + 32 * (__ffs(wm) - 1) + lane;
      float p[3];
      float2 zb = make_float2(0.0f, 0.0f);
      int cell = 0;
      const bool ok = k <= khi && lattice_test(g, o, d, k, p, zb, cell);
      for (unsigned m = __ballot_sync(kFull, ok); m && !done;) {
        const int take = min(__popc(m), min(g.n_max - taken, 32 - nq)), rank = __popc(m & lanemask_lt());
        const bool sel = ((m >> lane) & 1u) && rank < take;
        if (sel) {
          sa[nq + rank] = make_float4(p[0], p[1], p[2], zb.x);
          sb[nq + rank] = zb.y;
        }
        m &= ~__ballot_sync(kFull, sel);
        nq += take;
        taken += take;
        const bool last = taken >= g.n_max;
        if (nq == 32) batch();
        if (last) {
          if (nq > first) batch();
          done = true;
        }
      }
    }
  }
  if (!done && nq > first) batch();
  place = nq;
  return count;
}

template <int G>
__device__ __noinline__ bool whole_bundles(const FwdArgs& a, unsigned sb) {
  int lw, x0, y0;
  long ray0;
  tile_camera<G>(a, sb, lw, x0, y0, ray0);
  return lw >= 0;
}

// Count the ambiguous rays of a warp's (G = 1) or a CTA's bundles, and write
// their counts (a call of its own, so that the march keeps its registers).
template <bool SPARSE, int G>
__device__ __noinline__ void count_again(const Geo& g, const FwdArgs& a, unsigned sb, int warp, const BundleCounts& bc,
                                         float4* qa, float* qb) {
  const int lane = threadIdx.x & 31;
  int lw = -1, x0 = 0, y0 = 0, place = 0;
  long ray0 = ((long)sb * CamShape<G>::kRays) & ~31l;
  const Cam* cam = nullptr;
  if (a.use_cam) {
    cam = &tile_camera<G>(a, sb, lw, x0, y0, ray0);
    sub_origin<G>(lw, warp, x0, y0);
  }
  const SubTile st = sub_tile<G>(max(lw, 0));
  const unsigned starts = lw < 0 ? 0u : (1u << (st.lbw + st.lbh)) - 1u;  // of bundles: r & starts == 0
  unsigned again = __ballot_sync(kFull, bc.samples[lane] < 0);
  if (G == 8 && lw >= 0) again &= 0xffffu;  // (the other half of the places is not in use)
#pragma unroll 1
  for (unsigned r = 0; r < 32 && again >> r; r++) {
    if (starts && (r & starts) == 0u) place = 0;
    if (!((again >> r) & 1u)) {
      place = next_place(place, bc.count[r], bc.samples[r]);
      continue;
    }
    // (a ray of the other half is counted for its place only)
    float o[3], d[3];
    bool own = true;
    long id = ray0 + r;
    if (a.use_cam) {
      int px = (x0 & ~7) + (r & 7), py = y0 + (r >> 3);
      if (lw >= 0) {
        sub_pixel(st, r, px, py);
        px += x0;
        py += y0;
      }
      own = G != 8 || lw >= 0 || ((px ^ x0) & 4) == 0;
      id = ray0 + (long)py * cam->width + px;
      camera_ray(*cam, px, py, o, d);
    } else {
      own = G != 8 || (r >> 4) == (sb & 1u);
      load_ray(a.rays + 6 * id, o, d);
    }
    const int n = count_in_queue<SPARSE>(g, o, d, qa, qb, lane, place);
    if (own && lane == 0) a.count[id] = n;
  }
}

// Resident CTAs per SM: a 1080p frame with 5, 6 for G = 1 2.35, 2.37 ms, with
// counts (a second density sum in registers) with 4, 5 2.60, 2.94 ms; 641x361
// with 5, 6 for G = 4 417, 434 us; 320x180 with 6, 7 for G = 8 242, 208 us;
// 10,007 listed rays with counts with 4, 5 for G = 8 180, 144 us.
template <bool SPARSE, int G, bool COUNT>
__global__ void __launch_bounds__(32 * CamShape<G>::kWarps, COUNT ? (G == 1 ? 4 : 5) : (G == 8 ? 7 : 5))
    march_cam_kernel(const __grid_constant__ Geo g, const __grid_constant__ FwdArgs a) {
  constexpr int kFrame = G == 8 ? 8 : 4;           // lanes that share a lattice frame
  constexpr unsigned kFrameMask = (1u << kFrame) - 1u;
  __shared__ __align__(16) float sW[kSmemMlpT];
  // ambiguous counts: the bundles' rays and the places of a batch, per warp that replays
  constexpr int kReplay = COUNT ? (G == 1 ? CamShape<G>::kWarps : 1) : 0;
  __shared__ BundleCounts sCounts[kReplay > 0 ? kReplay : 1];
  __shared__ float4 sQa[kReplay > 0 ? kReplay : 1][COUNT ? 32 : 1];
  __shared__ float sQb[kReplay > 0 ? kReplay : 1][COUNT ? 32 : 1];
  __shared__ unsigned sWork[2];
  load_mlp_units(g.mlp, sW);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int base = lane & ~(kFrame - 1), j = G == 1 ? 0 : lane & (G - 1);
  // (without a counter there is one super-tile per CTA)
  if (threadIdx.x == 0) sWork[0] = a.counter ? atomicAdd(a.counter, 1u) : blockIdx.x;
  __syncthreads();
  for (int it = 0;; it ^= 1) {
    const unsigned sb = sWork[it];
    if (sb >= a.n_super) break;
    if (threadIdx.x == 0) sWork[it ^ 1] = a.counter ? atomicAdd(a.counter, 1u) : (unsigned)a.n_super;

    // G = 8 with counts: half of one of the queue's bundles; if a ray of it is
    // to be counted again, the other half is marched as well (for its counts)
    for (int half = 0;; half++) {
      bool valid;
      long rid;
      int slot;  // the ray's place in its bundle
      float o[3] = {0.0f, 0.0f, 0.0f}, d[3] = {0.0f, 0.0f, 1.0f};
      if (a.use_cam) {
        int px, py, lw, x0, y0;
        long ray0;
        const Cam& cam = tile_camera<G>(a, sb, lw, x0, y0, ray0);
        if (lw < 0) {
          lane_pixel<G>(warp, lane, px, py);
          px += COUNT && G == 8 ? x0 ^ (4 * half) : x0;
          py += y0;
          slot = ((py & 3) << 3) | (px & 7);
        } else {
          slot = G == 1 ? lane : warp * (32 / G) + lane / G;
          sub_pixel(sub_tile<G>(lw), slot, px, py);
          sub_origin<G>(lw, warp, x0, y0);
          px += x0;
          py += y0;
        }
        valid = px < cam.width && py < cam.height;
        rid = ray0 + (long)py * cam.width + px;
        if (valid) camera_ray(cam, px, py, o, d);
      } else {
        rid = (long)(COUNT && G == 8 ? sb ^ (unsigned)half : sb) * CamShape<G>::kRays + warp * (32 / G) + lane / G;
        valid = rid < a.n;
        if (valid) load_ray(a.rays + 6 * rid, o, d);
        slot = (int)(rid & 31);
      }
      int klo = 0, khi = -1;
      bool alive = valid && lattice_range(g, o, d, klo, khi);
      if (!alive) {
        klo = 0x7fffffff;
        khi = -1;
      }
      // the common lattice frame and its blocks of 32 windows from wb
      int wb = klo, ke = khi;
      if (G == 1) {
        wb = min(wb, __shfl_xor_sync(kFull, wb, 1));
        wb = min(wb, __shfl_xor_sync(kFull, wb, 2));
        ke = max(ke, __shfl_xor_sync(kFull, ke, 1));
        ke = max(ke, __shfl_xor_sync(kFull, ke, 2));
      }
      unsigned wm = 0;
      bool need_mask = wb <= ke;
      bool amb = false, done = false, counted = false;
      Through T, Tc;  // of the pixel's densities and of the counts'
      // the sums over the samples and their corrections: all channels for G = 1,
      // channels j and j + 4 of lane j for G = 4 (in F2[0]), channel j for G = 8 (in F)
      float2 F2[4], E2[4];
      float F = 0.0f, E = 0.0f;
#pragma unroll
      for (int c = 0; c < 4; c++) F2[c] = E2[c] = make_float2(0.0f, 0.0f);
      int seen = 0, cnt = 0, kstop = khi;  // kstop: the lattice index where the ray stopped
      int k0 = 0;
      unsigned own = 0, todo = 0;
      for (;;) {
        // A frame whose window is done takes its next one that the coarse grid
        // cannot rule out.  With one lane per ray the frames of a warp do so
        // together (a window is 32 tests for every lane), else each when it has to.
        if (G > 1 || !__any_sync(kFull, todo != 0u)) {
          while (__any_sync(kFull, todo == 0u && need_mask)) {
            const bool now = todo == 0u && need_mask;
            unsigned m = 0;
            if (now && alive) {
              const int nw = min((ke - wb) >> 5, 31);
              for (int jw = j; jw <= nw; jw += G) {
                const int ka = max(wb + 32 * jw, klo), kz = min(wb + 32 * jw + 31, khi);
                if (ka <= kz && window_maybe(g, o, d, ka, kz)) m |= 1u << jw;
              }
            }
#pragma unroll
            for (int s = 1; s < kFrame; s <<= 1) m |= __shfl_xor_sync(kFull, m, s);
            if (now) {
              wm = m;
              need_mask = wm == 0u && wb + 1024 <= ke;
              if (need_mask) wb += 1024;
            }
          }
          if (__any_sync(kFull, todo == 0u && wm != 0u)) {
            // the window's evaluated indices (bit i: index k0 + i): of this
            // lane's ray (own), and of any ray of the frame (todo)
            const bool now = todo == 0u && wm != 0u;
            unsigned m = 0;
            if (now) {
              k0 = wb + 32 * (__ffs(wm) - 1);
              if (alive) m = window_samples<G>(g, o, d, k0, klo, khi, j);
              own = m;
              wm &= wm - 1u;
              need_mask = wm == 0u && wb + 1024 <= ke;
              if (need_mask) wb += 1024;
            }
#pragma unroll
            for (int s = 1; s < kFrame; s <<= 1) m |= __shfl_xor_sync(kFull, m, s);
            if (now) todo = m;
            continue;
          }
          if (!__any_sync(kFull, todo != 0u)) break;
        }
        // G = 1: the frame's next index, for the rays evaluated there; else the
        // ray's next G samples, one per lane
        unsigned left = todo;
        const unsigned had = todo;
        if (G == 1) {
          todo &= todo - 1u;
        } else {
#pragma unroll
          for (int i = 0; i < G - 1; i++) {
            if (i < j) left &= left - 1u;
            todo &= todo - 1u;
          }
          todo &= todo - 1u;
        }
        const int bit = __ffs(left) - 1;
        bool hit = alive && left != 0u && (G != 1 || ((own >> bit) & 1u));
        float p[3] = {0.0f, 0.0f, 0.0f};
        float2 zb = make_float2(0.0f, 0.0f);
        if (hit) {
          lattice_point(g, o, d, k0 + bit, p);
          zb = __ldg(g.occ + occ_cell(g, p));
        }
        if (G == 1) {
          if (hit) {
            float t[8], t0;
            gather_features_eo<SPARSE, COUNT>(g, p, t, t0);
            SampleAct s;
            activate(g, t, p[2], zb, s);
            seen++;
            if (!COUNT || !done) {
              const float w = __fmul_rn(T.value(), s.ah);
#pragma unroll
              for (int c = 0; c < 4; c++) add_to2(F2[c], E2[c], w, s.x[2 * c], c < 3 ? s.x[2 * c + 1] : 0.0f);
              T.pass(__fsub_rn(1.0f, s.ah));
              done = T.value() < g.t_thr;
            }
            if (COUNT && !counted) {
              t[0] = t0;
              activate(g, t, p[2], zb, s);
              Tc.pass(__fsub_rn(1.0f, s.ah));
              cnt = seen;
              counted = Tc.value() < g.t_thr;
              amb |= fabsf(Tc.value() - g.t_thr) < g.t_thr * ambiguity(cnt);
            }
            alive = seen < g.n_max && !(done && (!COUNT || counted));
            if (COUNT && !alive) kstop = k0 + bit;
          }
          const unsigned am = __ballot_sync(kFull, alive);
          if (((am >> base) & kFrameMask) == 0u) {
            todo = wm = 0u;
            need_mask = false;
          }
        } else {
          hit = hit && seen + j < g.n_max;
          SampleAct s;
          s.ah = 0.0f;
          float ahc = 0.0f;
#pragma unroll
          for (int c = 0; c < 7; c++) s.x[c] = 0.0f;
          if (hit) {
            float t[8], t0;
            gather_features_eo<SPARSE, COUNT>(g, p, t, t0);
            activate(g, t, p[2], zb, s);
            if (COUNT) {
              SampleAct sc;
              t[0] = t0;
              activate(g, t, p[2], zb, sc);
              ahc = sc.ah;
            }
          }
          if (!COUNT || __any_sync(kFull, !done)) {
            // transmittance before each lane's sample, in lattice order
            int last;
            Through before = T, after;
            chain<G>(before, after, s.ah, hit, j, base, g.t_thr, last);
            const unsigned kept = hits_of<G>(hit && !done && j <= last, base);
            const float w = __fmul_rn(before.value(), s.ah);
            // lane j sums its channels, sample after sample
            float v[8];
#pragma unroll
            for (int c = 0; c < 8; c++) v[c] = c < 7 ? s.x[c] : 0.0f;
            transpose_lanes<G>(v, j);
#pragma unroll
            for (int i = 0; i < G; i++) {
              const float wi = __shfl_sync(kFull, w, i, G);
              if ((kept >> i) & 1u) {
                if (G == 4) add_to2(F2[0], E2[0], wi, v[i], v[(4 + i) & 7]);
                else add_to(F, E, wi, v[i]);
              }
            }
            const float th = __shfl_sync(kFull, after.h, min(last, G - 1), G);
            const float tl = __shfl_sync(kFull, after.l, min(last, G - 1), G);
            if (!done) {
              T.h = th;
              T.l = tl;
            }
            done = done || last < G;
          }
          if (COUNT && __any_sync(kFull, !counted)) {
            int last;
            Through before = Tc, after;
            chain<G>(before, after, ahc, hit, j, base, g.t_thr, last);
            const bool kept = hit && !counted && j <= last;
            const int n = __popc(hits_of<G>(kept, base));
            if (!counted) cnt = seen + n;
            amb |= kept && fabsf(after.value() - g.t_thr) < g.t_thr * ambiguity(cnt);
            const float th = __shfl_sync(kFull, after.h, min(last, G - 1), G);
            const float tl = __shfl_sync(kFull, after.l, min(last, G - 1), G);
            if (!counted) {
              Tc.h = th;
              Tc.l = tl;
            }
            counted = counted || last < G;
          }
          seen += __popc(hits_of<G>(hit, base));
          if (seen >= g.n_max || (done && (!COUNT || counted))) {
            if (COUNT && alive) kstop = k0 + 31 - __clz(had & ~todo);
            alive = need_mask = false;
            todo = wm = 0u;
          }
        }
      }

      if (COUNT && G > 1) amb = hits_of<G>(amb, lane & ~(G - 1)) != 0u;
      float out[3];
      if (G == 1) {
        if (valid) {
          float yd[3] = {0.0f, 0.0f, 0.0f}, all[7];
#pragma unroll
          for (int c = 0; c < 7; c++) all[c] = c & 1 ? F2[c / 2].y + E2[c / 2].y : F2[c / 2].x + E2[c / 2].x;
          if (seen > 0) mlp_rays<1>(sW, all, d, 0, yd);
#pragma unroll
          for (int c = 0; c < 3; c++) out[c] = seen > 0 ? fmaf(T.value(), g.bg[c], all[c] + yd[c]) : g.bg[c];
#pragma unroll
          for (int c = 0; c < 3; c++) a.rgb[3 * rid + c] = out[c];
          if (COUNT && !amb) a.count[rid] = cnt;
        }
      } else if (half == 0) {
        float y[3] = {0.0f, 0.0f, 0.0f};
        const float Fj = G == 4 ? F2[0].x + E2[0].x : F + E;  // channel j
        if (__any_sync(kFull, seen > 0)) {
          float all[7];
#pragma unroll
          for (int c = 0; c < 7; c++) all[c] = __shfl_sync(kFull, c < G ? Fj : F2[0].y + E2[0].y, c % G, G);
          mlp_rays<G>(sW, all, d, j, y);
        }
        if (valid && j < 3) {
          a.rgb[3 * rid + j] = seen > 0 ? fmaf(T.value(), g.bg[j], Fj + y[0]) : g.bg[j];
          if (COUNT && j == 0 && !amb) a.count[rid] = cnt;
        }
      }
      if constexpr (!COUNT) {
        break;
      } else {
        // does a ray of the bundle have to be counted again?
        if (G == 1 ? !__any_sync(kFull, amb) : !__syncthreads_or(amb) && half == 0) break;
        const int home = G == 1 ? warp : 0;  // the warp that replays, and its places
        BundleCounts& bc = sCounts[home];
        const int more = cnt + 31 - seen;  // wanted beyond the samples it has seen
        const int extra = samples_after<G>(g, o[0], o[1], o[2], d[0], d[1], d[2], kstop, khi,
                                           valid && seen < g.n_max && kstop < khi ? more : 0, j);
        if (j == 0) {
          bc.count[slot] = cnt;
          bc.samples[slot] = amb ? -1 : min(min(seen + extra, g.n_max), cnt + 31);
        }
        // (narrow images' super-tiles hold whole bundles)
        if (G == 8 && half == 0 && !(a.use_cam && whole_bundles<G>(a, sb))) continue;
        if (G == 1) __syncwarp();
        else __syncthreads();
        if (warp == home) count_again<SPARSE, G>(g, a, sb, warp, bc, sQa[home], sQb[home]);
        break;
      }
    }
    __syncthreads();
  }
}

template <bool SPARSE, int G, bool COUNT>
static cudaError_t launch_cam_variant(const omerf_scene* s, const FwdArgs& a, cudaStream_t stream) {
  auto kern = march_cam_kernel<SPARSE, G, COUNT>;
  constexpr int threads = 32 * CamShape<G>::kWarps;
  static std::atomic<int> blocks[64];  // per device: resident CTAs of this variant
  const int dev = s->device & 63;
  int nb = blocks[dev].load(std::memory_order_relaxed);
  if (nb == 0) {
    nb = persistent_blocks((const void*)kern, threads, 0, s->num_sms);
    blocks[dev].store(nb, std::memory_order_relaxed);
  }
  const int grid = (int)(a.n_super < nb ? a.n_super : nb);
  FwdArgs b = a;
  b.counter = a.n_super <= grid ? nullptr : next_counter(s, stream);
  kern<<<grid < 1 ? 1 : grid, threads, 0, stream>>>(s->geo, b);
  return cudaGetLastError();
}

template <int G, bool COUNT>
static cudaError_t launch_cam_group(const omerf_scene* s, const FwdArgs& a, cudaStream_t stream) {
  return s->desc.brick > 0 ? launch_cam_variant<true, G, COUNT>(s, a, stream)
                           : launch_cam_variant<false, G, COUNT>(s, a, stream);
}

// The lines lie where the measured times cross.  In a box of many lattice
// steps' height rays hold more samples and differ more, so that a warp of whole
// rays waits longer for its last one and needs a larger image; and the counting
// form of one lane per ray, with fewer warps per SM, needs a smaller one.
// us with 8 / 4 / 1 lanes, means of three scenes:
//   city (256 steps)  129,600 rays 285 / 301 / 696, 176,400 356 / 356 / 770,
//     518,400 920 / 834 / 966, 705,600 1233 / 1105 / 1153, 921,600 1586 / 1409 /
//     1370; with counts 176,400 426 / 441 / 706, 360,000 808 / 739 / 809, 518,400
//     1130 / 1005 / 979
//   field (64 steps)  65,536 72 / 73 / 115, 102,400 99 / 92 / 146, 262,144 216 /
//     183 / 193, 409,600 323 / 268 / 233; with counts 65,536 89 / 89 / 116,
//     147,456 170 / 144 / 177, 200,704 222 / 182 / 186, 262,144 283 / 226 / 191
// (the city's first line is within 6 % of the better form from 2^17 to 2^18).
// A BF16 scene keeps the packed queue: its deferred MLP rounds F to bfloat16, so
// sums in another order would move pixels by a step of that rounding.
int cam_lanes(const omerf_scene* s, long n, bool count) {
  if (s->desc.feat_dtype != OMERF_F32) return 0;
  const bool tall = s->geo.hi[2] - s->geo.lo[2] > 128.0f * s->geo.step;
  const long eight = tall ? 1 << 17 : 5 << 14;
  const long four = tall ? (count ? 7 << 16 : 3 << 18) : (count ? 3 << 16 : 5 << 16);
  return n < eight ? 8 : (n < four ? 4 : 1);
}

// Rays of a list may lie anywhere: rays of different lengths share a warp, and
// the queue, which packs samples whatever their ray, keeps its lanes busy.  Few
// rays leave the chip idle, and there 8 lanes per ray shorten the chain, but a
// handful of rays goes through the queue with all 32 lanes on one ray.  us with
// the queue / 8 lanes, random city rays with counts: 1 ray 18 / 25, 6 rays 39 /
// 40, 12 rays 63 / 50, 8,192 rays 220 / 105, 16,383 rays 226 / 177, 30,000 rays
// 232 / 229, 40,000 rays 236 / 274; field: 6 rays 22 / 26, 12 rays 31 / 27, 16,383
// rays 86 / 72, 24,576 rays 87 / 80, 30,000 rays 87 / 95.  The upper line lies
// below all crossings.
int list_lanes(const omerf_scene* s, long n) {
  return s->desc.feat_dtype == OMERF_F32 && n > 6 && n < (1 << 14) ? 8 : 0;
}

void cam_super(int lanes, int width, int height, int& lw, int& w, int& h) {
  lw = -1;
  if (lanes == 0) {
    w = h = 16;
    return;
  }
  if (width <= (lanes == 8 ? 2 : 4)) lw = width < 3 ? width - 1 : 2;
  else if (height <= 2) lw = (lanes == 8 ? 5 : 6) - height;
  super_size(lanes, lw, w, h);
}

cudaError_t launch_render_cam(const omerf_scene* s, const FwdArgs& a, int lanes, cudaStream_t stream) {
  if (a.count)
    return lanes == 1 ? launch_cam_group<1, true>(s, a, stream)
                      : (lanes == 4 ? launch_cam_group<4, true>(s, a, stream) : launch_cam_group<8, true>(s, a, stream));
  return lanes == 1 ? launch_cam_group<1, false>(s, a, stream)
                    : (lanes == 4 ? launch_cam_group<4, false>(s, a, stream) : launch_cam_group<8, false>(s, a, stream));
}

}  // namespace omerf
