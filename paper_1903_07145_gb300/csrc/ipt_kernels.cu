// Kernels of one nested-SGD iteration of inverse path tracing:
//   k_prepare   per-segment tables from the parameters (light selection CDF,
//               lobe probabilities): the per-iteration form of the emission-
//               proportional light selection of Appendix E;
//   k_forward   Monte Carlo pixel estimates (Eq. 1-2) with MIS (App. A.2),
//               optionally fused with the residual of the loss (Eq. 3);
//   k_adjoint   derivative paths from an independent sample set (Sec. 3.3),
//               scattering g . dI/dTheta (Eq. 5-6) into per-block shared
//               accumulators;
//   k_finalize  loss and gradient reduction;
//   k_adam      Adam + L1 emission regulariser + clamps (Sec. 4.4-4.5), then
//               the tables for the next iteration;
//   k_philox    the random-number primitive (ray casting: ipt_wavefront.cu).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "ipt_device.cuh"
#include "ipt_internal.h"
#include "ipt_path.cuh"
#include "ipt_wavefront.h"

namespace ipt {

__global__ void k_prepare(const float* params, const float* sparams, uint32_t S, float es,
                          const double* seg_area, SegBuffers t) {
  build_tables(params, sparams, S, es, seg_area, t);
}

// A camera path of the forward pass between two vertices.
struct FwdPath {
  PathRng rng;
  float3 o, d, beta, L;
  float prev_pdf;
  int skip;
  uint32_t k;
};

__device__ __forceinline__ void forward_start(FwdPath& p, const ViewDev& vw, uint32_t px, uint32_t py, uint32_t pid,
                                              uint32_t sample, const PathParams& pp) {
  p.rng.base = make_uint4(pid, sample, pp.set_iter, 0);
  p.rng.key = pp.key;
  p.d = camera_ray(vw, px, py, p.rng, p.o);
  p.beta = f3(1.0f, 1.0f, 1.0f);
  p.L = f3(0.0f, 0.0f, 0.0f);
  p.prev_pdf = 0.0f;
  p.skip = -1;
  p.k = 0;
}

// Traces to the next vertex and shades it; false when the path ends there.
__device__ __forceinline__ bool forward_vertex(const SceneDev& s, const SegDev& t, const PathParams& pp, bool light_on,
                                               FwdPath& p, uint32_t* err) {
  const Hit h = trace_closest(s, p.o, p.d, __int_as_float(0x7f800000), p.skip, err);
  if (h.tri < 0) return false;
  const Vtx v = make_vertex(s, h, p.d, pp.profile);
  if (v.prof > 0.0f) {
    const float wb = emission_weight(t, v, h.t, p.k > 0, light_on, p.prev_pdf, pp.mis);
    if (wb > 0.0f) p.L = p.L + p.beta * xyz(__ldg(&t.emis[v.seg])) * (wb * v.prof);
  }
  if (p.k == pp.max_depth) return false;
  const float4 ua = p.rng.draw(p.k, 0), ub = p.rng.draw(p.k, 1);
  const float4 ma = __ldg(&t.mat_a[v.seg]), mb = __ldg(&t.mat_b[v.seg]);
  const float4 sa = __ldg(&t.samp[v.seg]);
  if (light_on) {
    const NeeResult ne = next_event(s, t, v, ua, ub, pp.profile, pp.mis, sa.y, sa.x, err);
    if (ne.valid) {
      const BrdfVal bv = brdf_eval(ma, mb, v.ns, v.wi, ne.wl);
      // rounded before it is added, as the wavefront keeps it in a queue: the
      // integrators' radiances are equal
      const float3 c = p.beta * bv.f * xyz(__ldg(&t.emis[ne.seg])) * ne.k;
      p.L = f3(__fadd_rn(p.L.x, c.x), __fadd_rn(p.L.y, c.y), __fadd_rn(p.L.z, c.z));
    }
  }
  if (!(dot(v.wi, v.ns) > 0.0f)) return false;
  const float3 wo = bsdf_sample(sa.w, sa.x, v.ns, v.wi, ua.x, ua.y, ua.z);
  const float pdf = bsdf_pdf(sa.y, sa.x, v.ns, v.wi, wo);
  const float co = dot(wo, v.ns);
  if (!(dot(wo, v.ng) > 0.0f) || !(co > 0.0f) || !(pdf > 0.0f)) return false;
  const BrdfVal bv = brdf_eval(ma, mb, v.ns, v.wi, wo);
  p.beta = p.beta * bv.f * (co / pdf);
  p.prev_pdf = pdf;
  p.o = v.x + v.ng * s.eps;
  p.d = wo;
  p.skip = h.tri;
  ++p.k;
  return true;
}

// Radiance estimate of one camera path.
__device__ __forceinline__ float3 forward_path(const SceneDev& s, const SegDev& t, const ViewDev& vw, uint32_t px,
                                               uint32_t py, uint32_t pid, uint32_t sample, const PathParams& pp,
                                               bool light, uint32_t* err) {
  FwdPath p;
  forward_start(p, vw, px, py, pid, sample, pp);
  while (forward_vertex(s, t, pp, pp.nee && light, p, err)) {
  }
  return p.L;
}

__device__ __forceinline__ void add3(float* acc, int i, float3 v) {
  atomicAdd(&acc[i], v.x);
  atomicAdd(&acc[i + 1], v.y);
  atomicAdd(&acc[i + 2], v.z);
}

// Derivative of one camera path, contracted with the pixel's upstream
// gradient gp and scattered into acc (S x 10).  Eq. 5-6 differentiate the
// product of BSDFs along each light path; here each continuing vertex l keeps
// T_l (the throughput with its own weight w_l left out) and U_l (the sum of
// later contributions through T_l), so that d/dTheta_l of the whole path is
// (dw_l/dTheta) . U_l without dividing by w_l.  Emission and the local NEE term
// are differentiated on the spot.  Pdfs and MIS weights are held constant.
template <int MAXD>
__device__ void adjoint_path(const SceneDev& s, const SegDev& t, const ViewDev& vw, uint32_t px, uint32_t py,
                             uint32_t pid, uint32_t sample, const PathParams& pp, bool light, float3 gp,
                             float* acc, uint32_t* err) {
  PathRng rng;
  rng.base = make_uint4(pid, sample, pp.set_iter, 0);
  rng.key = pp.key;
  float3 o;
  float3 d = camera_ray(vw, px, py, rng, o);
  float3 beta = f3(1.0f, 1.0f, 1.0f);
  const bool light_on = pp.nee && light;
  const float es = pp.emission_scale;
  float3 T[MAXD], U[MAXD];
  float AD[MAXD], AS[MAXD], AR[MAXD];
  int SG[MAXD];
  int nv = 0;
  int skip = -1;
  float prev_pdf = 0.0f;
  for (uint32_t k = 0;; ++k) {
    const Hit h = trace_closest(s, o, d, __int_as_float(0x7f800000), skip, err);
    if (h.tri < 0) break;
    const Vtx v = make_vertex(s, h, d, pp.profile);
    float3 C = f3(0.0f, 0.0f, 0.0f);
    if (v.prof > 0.0f) {
      const float wb = emission_weight(t, v, h.t, k > 0, light_on, prev_pdf, pp.mis);
      if (wb > 0.0f) {
        const float f = wb * v.prof;
        C = xyz(__ldg(&t.emis[v.seg])) * f;
        add3(acc, 10 * v.seg + 7, gp * beta * (f * es));  // Eq. 5 at the hit
      }
    }
    const bool last = k == pp.max_depth;
    const float4 ma = __ldg(&t.mat_a[v.seg]), mb = __ldg(&t.mat_b[v.seg]);
    const float4 sa = __ldg(&t.samp[v.seg]);
    float4 ua = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!last) {
      ua = rng.draw(k, 0);
      const float4 ub = rng.draw(k, 1);
      if (light_on) {
        const NeeResult ne = next_event(s, t, v, ua, ub, pp.profile, pp.mis, sa.y, sa.x, err);
        if (ne.valid) {
          const BrdfVal bv = brdf_eval(ma, mb, v.ns, v.wi, ne.wl);
          const float3 Le = xyz(__ldg(&t.emis[ne.seg]));
          C = C + bv.f * Le * ne.k;
          add3(acc, 10 * ne.seg + 7, gp * beta * bv.f * (ne.k * es));        // Eq. 5, light end
          const float3 q = gp * beta * Le * ne.k;                              // Eq. 6, l = this vertex
          add3(acc, 10 * v.seg + 0, q * (1.0f / kPi));
          add3(acc, 10 * v.seg + 3, q * bv.sp.s);
          atomicAdd(&acc[10 * v.seg + 6], dot(q, f3(mb.x, mb.y, mb.z)) * bv.sp.ds_dr);
        }
      }
    }
#pragma unroll
    for (int l = 0; l < MAXD; ++l)
      if (l < nv) U[l] = U[l] + T[l] * C;
    if (last || !(dot(v.wi, v.ns) > 0.0f)) break;
    const float3 wo = bsdf_sample(sa.w, sa.x, v.ns, v.wi, ua.x, ua.y, ua.z);
    const float pdf = bsdf_pdf(sa.y, sa.x, v.ns, v.wi, wo);
    const float co = dot(wo, v.ns);
    if (!(dot(wo, v.ng) > 0.0f) || !(co > 0.0f) || !(pdf > 0.0f)) break;
    const BrdfVal bv = brdf_eval(ma, mb, v.ns, v.wi, wo);
    const float kk = co / pdf;
    const float3 w = bv.f * kk;
#pragma unroll
    for (int l = 0; l < MAXD; ++l) {
      if (l < nv) T[l] = T[l] * w;
      if (l == nv) {
        T[l] = beta;
        U[l] = f3(0.0f, 0.0f, 0.0f);
        AD[l] = kk * (1.0f / kPi);
        AS[l] = kk * bv.sp.s;
        AR[l] = kk * bv.sp.ds_dr;
        SG[l] = v.seg;
      }
    }
    ++nv;
    beta = beta * w;
    prev_pdf = pdf;
    o = v.x + v.ng * s.eps;
    d = wo;
    skip = h.tri;
  }
#pragma unroll
  for (int l = 0; l < MAXD; ++l) {
    if (l < nv) {
      const float3 q = gp * U[l];
      const int sg = SG[l];
      add3(acc, 10 * sg + 0, q * AD[l]);
      add3(acc, 10 * sg + 3, q * AS[l]);
      const float4 mb = __ldg(&t.mat_b[sg]);
      atomicAdd(&acc[10 * sg + 6], dot(q, f3(mb.x, mb.y, mb.z)) * AR[l]);
    }
  }
}

// ---------------------------------------------------------------------------
// Forward kernel: each pixel is handled by `group` lanes of one warp, each
// lane tracing spp / group samples; the lanes' sums are combined with
// butterfly shuffles, so the pixel estimate is deterministic.  kRad: the
// samples' radiances were traced before (k_forward_samples) and are read from
// `rad`; the sums are the same, in the same order, unless pp.serial asks for
// the wavefront's.
// ---------------------------------------------------------------------------

// Adds a pixel's traced radiances one after the other: its group of G lanes
// loads G of them at a time (one lane alone: 12 us for 64 samples of 64
// pixels) and every lane adds all, so each ends with the pixel's sums.  All
// 32 lanes call it together.
template <typename Add>
__device__ __forceinline__ void each_radiance(const float4* rad, bool active, uint32_t sub, uint32_t spp, uint32_t G,
                                              Add add) {
  for (uint32_t s0 = 0; s0 < spp; s0 += G) {
    const float4 r = active && s0 + sub < spp ? rad[s0 + sub] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t n = min(G, spp - s0);
    for (uint32_t j = 0; j < n; ++j) {
      const int src = (int)j;
      add(f3(__shfl_sync(0xffffffffu, r.x, src, (int)G), __shfl_sync(0xffffffffu, r.y, src, (int)G),
             __shfl_sync(0xffffffffu, r.z, src, (int)G)));
    }
  }
}

template <bool kRad>
__global__ void __launch_bounds__(kBlockThreads) k_forward(SceneDev s, SegDev t, const ViewDev* views,
                                                           uint32_t n_views, uint32_t pix_begin, uint32_t n_pix,
                                                           PathParams pp, float* img, float* msq,
                                                           const float* target, float* g_out,
                                                           double* loss_partials, float g_scale, int loss_kind,
                                                           const float4* rad, uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t G = pp.group;
  const uint32_t ppw = 32u / G;
  const uint32_t sub = lane & (G - 1u);
  const uint32_t warps_per_block = blockDim.x >> 5;
  const uint32_t n_tasks = (n_pix + ppw - 1) / ppw;
  const uint32_t stride = gridDim.x * warps_per_block;
  const bool light = any_light(s, t);
  const float inv_spp = 1.0f / (float)pp.spp;
  double loss_acc = 0.0;
  for (uint32_t task = blockIdx.x * warps_per_block + (threadIdx.x >> 5); task < n_tasks; task += stride) {
    const uint32_t local = task * ppw + lane / G;
    const bool active = local < n_pix;
    float3 a = f3(0.f, 0.f, 0.f), a2 = f3(0.f, 0.f, 0.f);
    const auto add = [&](float3 L) {
      a = a + L;
      a2 = a2 + L * L;
    };
    uint32_t pid = pix_begin + local;
    if (active) {
      uint32_t s0 = 0;
      if (pp.pick) {
        pid = pp.pick[local];
        s0 = local * pp.stride;
      }
      const ViewDev& vw = find_view(views, n_views, pid);
      const uint32_t lp = pid - vw.offset;
      const uint32_t px = lp % vw.w, py = lp / vw.w;
      for (uint32_t smp = sub; smp < pp.spp && !(kRad && pp.serial); smp += G) {
        if constexpr (kRad)
          add(xyz(rad[local * pp.spp + smp]));
        else
          add(forward_path(s, t, vw, px, py, pid, s0 + smp, pp, light, err));
      }
    }
    if (kRad && pp.serial) each_radiance(rad + (size_t)local * pp.spp, active, sub, pp.spp, G, add);
    for (uint32_t off = kRad && pp.serial ? 0u : G >> 1; off >= 1; off >>= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, off);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, off);
      a.z += __shfl_xor_sync(0xffffffffu, a.z, off);
      a2.x += __shfl_xor_sync(0xffffffffu, a2.x, off);
      a2.y += __shfl_xor_sync(0xffffffffu, a2.y, off);
      a2.z += __shfl_xor_sync(0xffffffffu, a2.z, off);
    }
    if (active && sub == 0) {
      const float3 mean = a * inv_spp;
      if (img) {
        img[3 * local + 0] = mean.x;
        img[3 * local + 1] = mean.y;
        img[3 * local + 2] = mean.z;
      }
      if (msq) {
        msq[3 * local + 0] = a2.x * inv_spp;
        msq[3 * local + 1] = a2.y * inv_spp;
        msq[3 * local + 2] = a2.z * inv_spp;
      }
      if (target) {
        // a pixel batch reads the target of the drawn pixel (the caller passes
        // the whole target image); otherwise target is indexed like the outputs
        const uint32_t ti = pp.pick ? pid : local;
        const float r[3] = {mean.x - target[3 * ti + 0], mean.y - target[3 * ti + 1],
                            mean.z - target[3 * ti + 2]};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (loss_kind == 0) {
            g_out[3 * local + c] = 2.0f * r[c] * g_scale;
            loss_acc += (double)r[c] * (double)r[c];
          } else {
            g_out[3 * local + c] = (r[c] > 0.0f ? 1.0f : (r[c] < 0.0f ? -1.0f : 0.0f)) * g_scale;
            loss_acc += fabs((double)r[c]);
          }
        }
      }
    }
  }
  if (loss_partials) {
    __shared__ double red[kBlockThreads / 32];
    for (int off = 16; off >= 1; off >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, off);
    if (lane == 0) red[threadIdx.x >> 5] = loss_acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (uint32_t w = 0; w < warps_per_block; ++w) sum += red[w];
      loss_partials[blockIdx.x] = sum;
    }
  }
}

// Small launches (a pixel batch of Sec. 4.5) leave most of the chip idle when a
// pixel's samples share one warp, and last as long as one lane's chain of
// paths in a diverging warp.  Here sample i (of pixel i / spp) is one thread's,
// `lanes` samples to a warp, with the samples spread over all warps that fit.
// Pixel batches on a Cornell box, 8 pixels of 128 samples: 141 -> 36 us
// (derivative pass 52 -> 30 us); on a 4.8k-triangle room 657 -> 81 us, and 512
// pixels of 33 samples, one lane a pixel before, 5.44 -> 0.18 ms.  The 64-scene
// Cornell batch (64 pixels of 64 samples each, 262k samples) gains from the
// blocks being scheduled as they end: a step 0.58 -> 0.34 ms.  kFewWarpsPerSm
// 4, 8, 12, 16: 512 pixels of 33: 0.205, 0.177, 0.173, 0.175 ms; derivative
// pass of 3000 paths: 0.127, 0.121, 0.185, 0.186 ms.
__global__ void __launch_bounds__(kBlockThreads) k_forward_samples(SceneDev s, SegDev t, const ViewDev* views,
                                                                   uint32_t n_views, uint32_t pix_begin, uint32_t n,
                                                                   uint32_t lanes, PathParams pp, float4* rad,
                                                                   uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t i = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * lanes + lane;
  if (lane >= lanes || i >= n) return;
  const uint32_t local = i / pp.spp, smp = i - local * pp.spp;
  uint32_t pid = pix_begin + local, s0 = 0;
  if (pp.pick) {
    pid = pp.pick[local];
    s0 = local * pp.stride;
  }
  const ViewDev& vw = find_view(views, n_views, pid);
  const uint32_t lp = pid - vw.offset;
  const float3 L = forward_path(s, t, vw, lp % vw.w, lp / vw.w, pid, s0 + smp, pp, any_light(s, t), err);
  rad[i] = make_float4(L.x, L.y, L.z, 0.0f);
}

// Pixels [pix_begin, pix_begin + n_pix) of the concatenated views; g_img is
// indexed relative to pix_begin.
template <int MAXD>
__global__ void __launch_bounds__(kBlockThreads, MAXD <= 4 ? 3 : 2) k_adjoint(SceneDev s, SegDev t, const ViewDev* views,
                                                           uint32_t n_views, uint32_t pix_begin, uint32_t n_pix,
                                                           PathParams pp, uint32_t lanes, const float* g_img,
                                                           double* grad_acc, float* gacc, uint32_t* err) {
  // per-block accumulators in shared memory, or (scenes with too many
  // segments for it) one zeroed accumulator in global memory
  extern __shared__ float sgrad_sh[];
  float* sgrad = gacc ? gacc : sgrad_sh;
  const uint32_t n_par = 10u * s.n_seg;
  if (!gacc)
    for (uint32_t i = threadIdx.x; i < n_par; i += blockDim.x) sgrad[i] = 0.0f;
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31u;
  const bool light = any_light(s, t);
  const float inv_spp = 1.0f / (float)pp.spp;
  const auto paths = [&](uint32_t local, uint32_t first, uint32_t step) {
    const uint32_t pid = pp.pick ? pp.pick[local] : pix_begin + local;
    const uint32_t s0 = pp.pick ? local * pp.stride : 0u;
    const float3 gp = f3(g_img[3 * local], g_img[3 * local + 1], g_img[3 * local + 2]) * inv_spp;
    if (gp.x == 0.0f && gp.y == 0.0f && gp.z == 0.0f) return;
    const ViewDev& vw = find_view(views, n_views, pid);
    const uint32_t lp = pid - vw.offset;
    const uint32_t px = lp % vw.w, py = lp / vw.w;
    for (uint32_t smp = first; smp < pp.spp; smp += step)
      adjoint_path<MAXD>(s, t, vw, px, py, pid, s0 + smp, pp, light, gp, sgrad, err);
  };
  // lanes > 0 (few paths): path i is one thread's, `lanes` paths to a warp;
  // otherwise `group` lanes of a warp share a pixel
  uint32_t task = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_tasks, stride = 1u;
  const uint32_t G = pp.group, ppw = 32u / G;
  if (lanes) {
    n_tasks = lane < lanes && task * lanes + lane < n_pix * pp.spp ? task + 1u : 0u;
  } else {
    n_tasks = (n_pix + ppw - 1) / ppw;
    stride = gridDim.x * (blockDim.x >> 5);
  }
  for (; task < n_tasks; task += stride) {
    const uint32_t i = task * lanes + lane;
    const uint32_t local = lanes ? i / pp.spp : task * ppw + lane / G;
    if (local < n_pix) paths(local, lanes ? i % pp.spp : lane & (G - 1u), lanes ? pp.spp : G);
  }
  __syncthreads();
  if (!gacc)
    for (uint32_t i = threadIdx.x; i < n_par; i += blockDim.x) {
      const float v = sgrad[i];
      if (v != 0.0f) atomicAdd(&grad_acc[i], (double)v);
    }
}

// ---------------------------------------------------------------------------
// Batched megakernel: the paths of every scene of a batch's launch table in
// one forward and one adjoint launch (the small pixel batches of Sec. 4.5
// are latency-bound, and a stage-by-stage wavefront pays ~45 launches per
// iteration).  Launch pixel p belongs to the table entry whose pixel range
// holds it; each scene keeps its own Philox key, emission scale, pixel draw,
// target and segment range, so its paths are the ones it traces alone.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t table_scene(const WfScene* tab, uint32_t n, uint32_t p) {
  uint32_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (tab[mid].pix_begin <= p)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ PathParams scene_params(const PathParams& base, const WfScene& e, uint32_t set_iter) {
  PathParams p = base;
  p.key = e.key;
  p.emission_scale = e.es;
  p.set_iter = set_iter;
  p.pick = e.pick;
  return p;
}

// Residual pass: the upstream gradient of every entry and, per block, each
// scene's loss sum (rows[block * n_scenes + scene], the layout of the
// wavefront's reduction).
// Four resident blocks per SM (at most 128 registers), as the single-scene
// forward: the grid is one loss row per block of a full wave.  kRad: reads the
// radiances that k_forward_samples_batch traced, as k_forward does.
template <bool kRad>
__global__ void __launch_bounds__(kBlockThreads, 4)
    k_forward_batch(const WfScene* tab, uint32_t n_scenes, uint32_t total, PathParams pp, uint32_t set,
                    const uint32_t* iter_dev, int loss_kind, double* loss_rows, const float4* rad, uint32_t* err) {
  extern __shared__ double sloss[];
  for (uint32_t i = threadIdx.x; i < n_scenes; i += blockDim.x) sloss[i] = 0.0;
  __syncthreads();
  const uint32_t set_iter = (set << 24) | (*iter_dev & 0xFFFFFFu);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t G = pp.group;
  const uint32_t ppw = 32u / G;
  const uint32_t sub = lane & (G - 1u);
  const uint32_t warps_per_block = blockDim.x >> 5;
  const uint32_t n_tasks = (total + ppw - 1) / ppw;
  const uint32_t stride = gridDim.x * warps_per_block;
  const float inv_spp = 1.0f / (float)pp.spp;
  for (uint32_t task = blockIdx.x * warps_per_block + (threadIdx.x >> 5); task < n_tasks; task += stride) {
    const uint32_t p = task * ppw + lane / G;
    const bool active = p < total;
    float3 a = f3(0.f, 0.f, 0.f);
    uint32_t b = 0, entry = 0, pid = 0;
    if (active) {
      b = table_scene(tab, n_scenes, p);
      const WfScene& e = tab[b];
      entry = p - e.pix_begin + e.pix_base;
      pid = e.pick ? e.pick[entry] : entry;
      if constexpr (kRad) {
        for (uint32_t smp = sub; smp < pp.spp && !pp.serial; smp += G) a = a + xyz(rad[p * pp.spp + smp]);
      } else {
        const uint32_t s0 = e.pick ? entry * pp.stride : 0u;
        const PathParams q = scene_params(pp, e, set_iter);
        const bool light = any_light(e.s, e.t);
        const ViewDev& vw = find_view(e.views, e.n_views, pid);
        const uint32_t lp = pid - vw.offset;
        const uint32_t px = lp % vw.w, py = lp / vw.w;
        for (uint32_t smp = sub; smp < pp.spp; smp += G)
          a = a + forward_path(e.s, e.t, vw, px, py, pid, s0 + smp, q, light, err);
      }
    }
    if (kRad && pp.serial)
      each_radiance(rad + (size_t)p * pp.spp, active, sub, pp.spp, G, [&](float3 L) { a = a + L; });
    for (uint32_t off = kRad && pp.serial ? 0u : G >> 1; off >= 1; off >>= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, off);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, off);
      a.z += __shfl_xor_sync(0xffffffffu, a.z, off);
    }
    if (active && sub == 0) {
      const WfScene& e = tab[b];
      const float3 mean = a * inv_spp;
      const uint32_t ti = e.pick ? pid : entry;
      const float r[3] = {mean.x - e.target[3 * ti + 0], mean.y - e.target[3 * ti + 1], mean.z - e.target[3 * ti + 2]};
      double l = 0.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (loss_kind == 0) {
          e.g_img[3 * entry + c] = 2.0f * r[c] * e.g_scale;
          l += (double)r[c] * (double)r[c];
        } else {
          e.g_img[3 * entry + c] = (r[c] > 0.0f ? 1.0f : (r[c] < 0.0f ? -1.0f : 0.0f)) * e.g_scale;
          l += fabs((double)r[c]);
        }
      }
      atomicAdd(&sloss[b], l);
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n_scenes; i += blockDim.x) loss_rows[(size_t)blockIdx.x * n_scenes + i] = sloss[i];
}

// One sample of a launch pixel a thread (see k_forward_samples).
__global__ void __launch_bounds__(kBlockThreads, 4)
    k_forward_samples_batch(const WfScene* tab, uint32_t n_scenes, uint32_t n, uint32_t lanes, PathParams pp,
                            uint32_t set, const uint32_t* iter_dev, float4* rad, uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t i = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * lanes + lane;
  if (lane >= lanes || i >= n) return;
  const uint32_t p = i / pp.spp, smp = i - p * pp.spp;
  const WfScene& e = tab[table_scene(tab, n_scenes, p)];
  const uint32_t entry = p - e.pix_begin + e.pix_base;
  const uint32_t pid = e.pick ? e.pick[entry] : entry;
  const uint32_t s0 = e.pick ? entry * pp.stride : 0u;
  const PathParams q = scene_params(pp, e, (set << 24) | (*iter_dev & 0xFFFFFFu));
  const ViewDev& vw = find_view(e.views, e.n_views, pid);
  const uint32_t lp = pid - vw.offset;
  const float3 L =
      forward_path(e.s, e.t, vw, lp % vw.w, lp / vw.w, pid, s0 + smp, q, any_light(e.s, e.t), err);
  rad[i] = make_float4(L.x, L.y, L.z, 0.0f);
}

// Derivative pass: every entry's paths into the batch's packed segment
// accumulators (shared per block, or global when they do not fit).
template <int MAXD>
__global__ void __launch_bounds__(kBlockThreads, MAXD <= 4 ? 3 : 2)
    k_adjoint_batch(const WfScene* tab, uint32_t n_scenes, uint32_t total, uint32_t n_par, PathParams pp,
                    uint32_t lanes, uint32_t set, const uint32_t* iter_dev, double* grad_acc, float* gacc, uint32_t* err) {
  extern __shared__ float bgrad_sh[];
  float* acc = gacc ? gacc : bgrad_sh;
  if (!gacc)
    for (uint32_t i = threadIdx.x; i < n_par; i += blockDim.x) acc[i] = 0.0f;
  __syncthreads();
  const uint32_t set_iter = (set << 24) | (*iter_dev & 0xFFFFFFu);
  const uint32_t lane = threadIdx.x & 31u;
  const float inv_spp = 1.0f / (float)pp.spp;
  const auto paths = [&](uint32_t p, uint32_t first, uint32_t step) {
    const WfScene& e = tab[table_scene(tab, n_scenes, p)];
    const uint32_t entry = p - e.pix_begin + e.pix_base;
    const uint32_t pid = e.pick ? e.pick[entry] : entry;
    const uint32_t s0 = e.pick ? entry * pp.stride : 0u;
    const float3 gp = f3(e.g_img[3 * entry], e.g_img[3 * entry + 1], e.g_img[3 * entry + 2]) * inv_spp;
    if (gp.x == 0.0f && gp.y == 0.0f && gp.z == 0.0f) return;
    const PathParams q = scene_params(pp, e, set_iter);
    const bool light = any_light(e.s, e.t);
    const ViewDev& vw = find_view(e.views, e.n_views, pid);
    const uint32_t lp = pid - vw.offset;
    const uint32_t px = lp % vw.w, py = lp / vw.w;
    float* sacc = acc + 10u * e.seg_offset;
    for (uint32_t smp = first; smp < pp.spp; smp += step)
      adjoint_path<MAXD>(e.s, e.t, vw, px, py, pid, s0 + smp, q, light, gp, sacc, err);
  };
  // paths to threads as in k_adjoint
  uint32_t task = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_tasks, stride = 1u;
  const uint32_t G = pp.group, ppw = 32u / G;
  if (lanes) {
    n_tasks = lane < lanes && task * lanes + lane < total * pp.spp ? task + 1u : 0u;
  } else {
    n_tasks = (total + ppw - 1) / ppw;
    stride = gridDim.x * (blockDim.x >> 5);
  }
  for (; task < n_tasks; task += stride) {
    const uint32_t i = task * lanes + lane;
    const uint32_t p = lanes ? i / pp.spp : task * ppw + lane / G;
    if (p < total) paths(p, lanes ? i % pp.spp : lane & (G - 1u), lanes ? pp.spp : G);
  }
  __syncthreads();
  if (!gacc)
    for (uint32_t i = threadIdx.x; i < n_par; i += blockDim.x) {
      const float v = acc[i];
      if (v != 0.0f) atomicAdd(&grad_acc[i], (double)v);
    }
}

__global__ void k_add_to_double(const float* src, uint32_t n, double* dst) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    dst[i] += (double)src[i];
}

// One block: fixed-order sums (deterministic for a fixed grid).
__global__ void k_finalize(const double* loss_partials, int n_partials, double* loss_dev,
                           const double* grad_acc, float* grad_out, uint32_t n_params) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n_partials; i += blockDim.x) s += loss_partials[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w >= 1; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0 && loss_dev) *loss_dev = red[0];
  if (grad_out)
    for (uint32_t i = threadIdx.x; i < n_params; i += blockDim.x) grad_out[i] = (float)grad_acc[i];
}

__global__ void k_grad_out(const double* grad_acc, float* grad_out, uint32_t n_params) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_params; i += gridDim.x * blockDim.x)
    grad_out[i] = (float)grad_acc[i];
}

// Adam on the concatenated parameters of a batch, one block per member,
// followed by that member's tables for the next iteration.
__device__ __forceinline__ void adam_range(float* params, float* m, float* v, const uint8_t* free_mask,
                                           const double* grad_acc, const float* grad_f, uint32_t begin,
                                           uint32_t end, uint32_t g_begin, const AdamHost& a, int step,
                                           uint32_t lane0, uint32_t lanes) {
  const float bc1 = 1.0f - powf(a.beta1, (float)step);
  const float bc2 = 1.0f - powf(a.beta2, (float)step);
  for (uint32_t i = begin + lane0; i < end; i += lanes) {
    if (free_mask && !free_mask[i]) continue;
    const uint32_t j = i % 10u;
    float g = grad_f ? grad_f[i] : (float)grad_acc[g_begin + (i - begin)];
    const float th = params[i];
    if (j >= 7) g += a.l1 * (th > 0.0f ? 1.0f : (th < 0.0f ? -1.0f : 0.0f));
    const float mi = a.beta1 * m[i] + (1.0f - a.beta1) * g;
    const float vi = a.beta2 * v[i] + (1.0f - a.beta2) * g * g;
    m[i] = mi;
    v[i] = vi;
    float nt = th - a.lr * (mi / bc1) / (sqrtf(vi / bc2) + a.eps);
    if (j < 6)
      nt = fminf(fmaxf(nt, 0.0f), 1.0f);
    else if (j == 6)
      nt = fminf(fmaxf(nt, 0.02f), 1.0f);
    else
      nt = fmaxf(nt, 0.0f);
    params[i] = nt;
  }
}

// True on every thread of the block when the loss (nullable) or any of the n
// gradient values (FP64 accumulators, or FP32 when grad_f is given) is NaN or
// infinite.
__device__ __forceinline__ bool block_nonfinite(const double* loss, const double* grad_acc, const float* grad_f,
                                                uint32_t n) {
  bool bad = loss && !isfinite(*loss);
  for (uint32_t i = threadIdx.x; i < n && !bad; i += blockDim.x)
    bad = grad_f ? !isfinite(grad_f[i]) : !isfinite(grad_acc[i]);
  return __syncthreads_or(bad) != 0;
}

// A member whose loss or gradient is not finite keeps its parameters and
// Adam moments (the step is skipped for it alone) and sets the error word.
__global__ void k_adam_batch(const BatchMember* members, float* params, float* m, float* v,
                             const uint8_t* free_mask, const double* grad_acc, const uint32_t* iter_dev,
                             AdamHost a, const double* losses, uint32_t* err) {
  const BatchMember mb = members[blockIdx.x];
  if (!mb.active) return;
  const int step = (int)*iter_dev + 1;
  if (block_nonfinite(losses + blockIdx.x, grad_acc + 10u * mb.grad_offset, nullptr, 10u * mb.n_seg)) {
    if (threadIdx.x == 0) atomicOr(err, kErrNonFinite);
  } else {
    adam_range(params, m, v, free_mask, grad_acc, nullptr, 10u * mb.seg_offset, 10u * (mb.seg_offset + mb.n_seg),
               10u * mb.grad_offset, a, step, threadIdx.x, blockDim.x);
  }
  __syncthreads();
  const float* p = params + 10u * mb.seg_offset;
  build_tables(p, p, mb.n_seg, mb.es, mb.seg_area, mb.tab);
}

__global__ void k_prepare_batch(const BatchMember* members, const float* params) {
  const BatchMember mb = members[blockIdx.x];
  const float* p = params + 10u * mb.seg_offset;
  build_tables(p, p, mb.n_seg, mb.es, mb.seg_area, mb.tab);
}

// Loss of each member from the per-block rows of the launch table (n_tab
// entries: the active members).
__global__ void k_batch_losses(const double* rows, int n_rows, const BatchMember* members, uint32_t n_tab,
                               double* loss) {
  __shared__ double red[256];
  const uint32_t b = blockIdx.x;
  if (!members[b].active) {  // traced nothing this step
    if (threadIdx.x == 0) loss[b] = 0.0;
    return;
  }
  const uint32_t slot = members[b].slot;
  double s = 0.0;
  for (int r = threadIdx.x; r < n_rows; r += blockDim.x) s += rows[(size_t)r * n_tab + slot];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w >= 1; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[b] = red[0] * (double)members[b].inv_n;
}

__global__ void k_tick(uint32_t* counter) { *counter += 1u; }

// With a non-finite loss or gradient the update is skipped: parameters, Adam
// moments and the step count stay those of the last good step, and the
// error word reports it.  The tables are rebuilt either way.
__global__ void k_adam(float* params, float* m, float* v, const uint8_t* free_mask,
                       const double* grad_acc, const float* grad_f, int* step_dev, AdamHost a, uint32_t S,
                       float es, const double* seg_area, SegBuffers t, const double* loss, uint32_t* err) {
  const int step = *step_dev + 1;
  const bool bad = block_nonfinite(loss, grad_acc, grad_f, 10u * S);
  if (!bad) adam_range(params, m, v, free_mask, grad_acc, grad_f, 0, 10u * S, 0u, a, step, threadIdx.x, blockDim.x);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (bad)
      atomicOr(err, kErrNonFinite);
    else
      *step_dev = step;
  }
  build_tables(params, params, S, es, seg_area, t);
}

// The same check for launches over a grid: one block decides, *flag = 1
// when the step must be skipped.
__global__ void __launch_bounds__(1024) k_finite_guard(const double* loss, const double* grad_acc,
                                                       const float* grad_f, uint32_t n, uint32_t* flag,
                                                       uint32_t* err) {
  const bool bad = block_nonfinite(loss, grad_acc, grad_f, n);
  if (threadIdx.x == 0) {
    *flag = bad ? 1u : 0u;
    if (bad) atomicOr(err, kErrNonFinite);
  }
}

// Scenes with many segments (per-triangle parameters): Adam over a grid, the
// per-segment tables over a grid, and the light CDF by one block that keeps
// the sequential FP64 summation order of build_tables.  The terms of
// non-emitting segments are exact zeros, so the running sum changes only at
// emitters: those are added in order by one thread, and every other entry
// takes the running value of the last emitter before it.
constexpr uint32_t kWideSegments = 4096;

__global__ void k_adam_wide(float* params, float* m, float* v, const uint8_t* free_mask, const double* grad_acc,
                            const float* grad_f, const int* step_dev, AdamHost a, uint32_t S, const uint32_t* skip) {
  if (*skip) return;
  const int step = *step_dev + 1;
  adam_range(params, m, v, free_mask, grad_acc, grad_f, 0, 10u * S, 0u, a, step,
             blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void k_tables_seg(const float* params, const float* sparams, uint32_t S, float es, SegBuffers t) {
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
    const float* p = params + 10 * s;
    const float* q = sparams + 10 * s;
    const float r = p[6];
    t.mat_a[s] = make_float4(p[0], p[1], p[2], r);
    t.mat_b[s] = make_float4(p[3], p[4], p[5], fmaxf(r * r, 1e-4f));
    t.emis[s] = make_float4(es * p[7], es * p[8], es * p[9], 0.0f);
    const double ld = lum_d(q[0], q[1], q[2]);
    const double ls = lum_d(q[3], q[4], q[5]);
    const double sum = __dadd_rn(ld, ls);
    const double P = sum > 0.0 ? __ddiv_rn(ls, sum) : 0.0;
    const float rs = q[6];
    t.samp[s] = make_float4(fmaxf(rs * rs, 1e-4f), (float)P, 0.0f, unit_threshold(P, 1.0));
    double le = lum_d(q[7], q[8], q[9]);
    if (!(le > 0.0)) le = 0.0;
    t.lum[s] = le;
  }
}

// One block of 1024 threads; bumps *step_dev when given (after Adam) unless
// *skip says the Adam step was skipped.
__global__ void __launch_bounds__(1024) k_tables_cdf(uint32_t S, const double* seg_area, SegBuffers t,
                                                     int* step_dev, const uint32_t* skip) {
  __shared__ double term[1024];
  __shared__ unsigned nz[32];
  __shared__ double warp_end[32];
  __shared__ double carry, start;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
  if (tid == 0) carry = 0.0;
  for (uint32_t base = 0; base < S; base += 1024u) {
    const uint32_t i = base + tid;
    if (tid == 0) start = carry;
    const double a = i < S ? __dmul_rn(t.lum[i], seg_area[i]) : 0.0;
    term[tid] = a;
    const unsigned m = __ballot_sync(0xffffffffu, a != 0.0);
    if (lane == 0) nz[wid] = m;
    __syncthreads();
    if (tid == 0) {
      double acc = carry;
      for (int w = 0; w < 32; ++w) {
        for (unsigned b = nz[w]; b; b &= b - 1u) {
          const int j = w * 32 + __ffs(b) - 1;
          acc = __dadd_rn(acc, term[j]);
          term[j] = acc;
        }
        warp_end[w] = acc;
      }
      carry = acc;
    }
    __syncthreads();
    // running value after the last emitter at or before this entry
    const unsigned upto = nz[wid] & (0xffffffffu >> (31u - lane));
    double c;
    if (upto)
      c = term[wid * 32 + 31 - __clz(upto)];
    else
      c = wid > 0 ? warp_end[wid - 1] : start;
    if (i < S) t.cdf[i] = c;
    __syncthreads();
  }
  if (tid == 0) {
    *t.W = carry;
    if (step_dev && !(skip && *skip)) *step_dev += 1;
  }
}

__global__ void k_tables_samp(uint32_t S, SegBuffers t) {
  const double W = *t.W;
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
    const double le = t.lum[s];
    t.samp[s].z = (W > 0.0 && le > 0.0) ? (float)(le / W) : 0.0f;
    t.sel[s] = unit_threshold(t.cdf[s], W);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) t.sel[S] = W > 0.0 ? 1.0f : 0.0f;
}

static cudaError_t launch_tables_wide(const SceneBuffers& s, const SegBuffers& t, const float* params,
                                      const float* sparams, int* step_dev, const uint32_t* skip, cudaStream_t st) {
  const int grid = (int)std::min<uint32_t>((s.n_seg + 255u) / 256u, 1024u);
  k_tables_seg<<<grid, 256, 0, st>>>(params, sparams, s.n_seg, s.emission_scale, t);
  k_tables_cdf<<<1, 1024, 0, st>>>(s.n_seg, s.seg_area, t, step_dev, skip);
  k_tables_samp<<<grid, 256, 0, st>>>(s.n_seg, t);
  return cudaGetLastError();
}


__global__ void k_philox(uint32_t n, const uint32_t* ctr, const uint32_t* key, uint32_t* out) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
  const uint4 o = philox4x32_10(c, make_uint2(key[2 * i], key[2 * i + 1]));
  out[4 * i] = o.x;
  out[4 * i + 1] = o.y;
  out[4 * i + 2] = o.z;
  out[4 * i + 3] = o.w;
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
template <int MAXD>
static void adjoint_occupancy(int* out) {
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_adjoint<MAXD>, kBlockThreads, 16384);
}

cudaError_t init_launcher(Launcher* L, int device) {
  cudaError_t e = cudaDeviceGetAttribute(&L->num_sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&L->fwd_blocks_per_sm, k_forward<false>, kBlockThreads, 0);
  if (e != cudaSuccess) return e;
  adjoint_occupancy<2>(&L->adj_blocks_per_sm[0]);
  adjoint_occupancy<4>(&L->adj_blocks_per_sm[1]);
  adjoint_occupancy<6>(&L->adj_blocks_per_sm[2]);
  adjoint_occupancy<8>(&L->adj_blocks_per_sm[3]);
  for (int i = 0; i < 4; ++i)
    if (L->adj_blocks_per_sm[i] < 1) L->adj_blocks_per_sm[i] = 1;
  if (L->fwd_blocks_per_sm < 1) L->fwd_blocks_per_sm = 1;
  e = wf_init(L);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

int loss_partials_capacity(const Launcher& L) { return L.num_sms * L.fwd_blocks_per_sm; }

static int grid_for(uint64_t n_tasks_warps, int blocks_cap) {
  const uint64_t per_block = kBlockThreads / 32;
  uint64_t g = (n_tasks_warps + per_block - 1) / per_block;
  if (g > (uint64_t)blocks_cap) g = blocks_cap;
  if (g < 1) g = 1;
  return (int)g;
}

// Samples per warp of a launch of n samples that runs one sample a thread: as
// few as kFewWarpsPerSm warps on each SM allow, 32 beyond that.
constexpr uint32_t kFewWarpsPerSm = 8;
static uint32_t few_lanes(const Launcher& L, uint64_t n) {
  const uint32_t warps = kFewWarpsPerSm * (uint32_t)L.num_sms;
  return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(32, (n + warps - 1u) / warps));
}

// The residual pass runs one sample a thread up to the capacity of the
// radiance buffer; the derivative pass, whose blocks each clear and flush
// their accumulators, up to kFewAdjointWarps.  Above 8 warps an SM the blocks
// come in more than one wave; with `group` lanes a pixel there instead, 527
// pixels of 129 paths (a 3k-triangle room, depth 5, the whole call) took 31.5
// ms for 0.64, 2060 of 33 8.3 for 0.66, and 2125 of 32 the same 0.66 (5k
// segments: 45 for 1.4, 11.7 for 1.4, and 1.39 for 1.45).
static bool few_forward(const Launcher& L, uint64_t n) { return n <= L.rad_cap; }
static bool few_adjoint(const Launcher& L, uint64_t n) { return n <= 32ull * kFewAdjointWarps * (uint32_t)L.num_sms; }

// In-order sums: a group loads what it can of a pixel's samples at once, its
// size need not divide their number.
static void serial_group(PathParams& pp) {
  pp.serial = true;
  pp.group = 1;
  while (pp.group < 32 && pp.group < pp.spp) pp.group *= 2;
}

static int few_grid(uint32_t n, uint32_t lanes) {
  const uint32_t per_block = lanes * (kBlockThreads / 32u);
  return (int)((n + per_block - 1u) / per_block);
}

cudaError_t launch_prepare(const SceneBuffers& s, const SegBuffers& t, const float* params,
                           const float* sparams, cudaStream_t st) {
  if (s.n_seg > kWideSegments) return launch_tables_wide(s, t, params, sparams ? sparams : params, nullptr, nullptr, st);
  k_prepare<<<1, 256, 0, st>>>(params, sparams ? sparams : params, s.n_seg, s.emission_scale, s.seg_area, t);
  return cudaGetLastError();
}

cudaError_t launch_forward(const Launcher& L, const SceneBuffers& s, const SegBuffers& t,
                           const ViewHost* views_dev, uint32_t n_views, uint32_t pix_begin,
                           uint32_t n_pix, const TraceParams& tp, float* img, float* msq,
                           const float* target, float* g_out, double* loss_partials,
                           float g_scale, int loss_kind, uint32_t* err, cudaStream_t st) {
  PathParams pp = make_path_params(tp, s);
  if (tp.serial_sums) serial_group(pp);
  const uint64_t tasks = (n_pix + (32 / pp.group) - 1) / (32 / pp.group);
  const int cap = L.num_sms * L.fwd_blocks_per_sm;
  // with a loss the grid is fixed, so the partial sums reduce in a fixed order
  const int grid = loss_partials ? cap : grid_for(tasks, cap);
  const SceneDev sd = scene_dev(s);
  const SegDev td = seg_dev(t);
  const ViewDev* vd = reinterpret_cast<const ViewDev*>(views_dev);
  if (few_forward(L, (uint64_t)n_pix * tp.spp)) {
    const uint32_t n = n_pix * tp.spp, lanes = few_lanes(L, n);
    k_forward_samples<<<few_grid(n, lanes), kBlockThreads, 0, st>>>(sd, td, vd, n_views, pix_begin, n, lanes, pp, L.rad,
                                                                  err);
    k_forward<true><<<grid, kBlockThreads, 0, st>>>(sd, td, vd, n_views, pix_begin, n_pix, pp, img, msq, target, g_out,
                                                    loss_partials, g_scale, loss_kind, L.rad, err);
    return cudaGetLastError();
  }
  k_forward<false><<<grid, kBlockThreads, 0, st>>>(sd, td, vd, n_views, pix_begin, n_pix, pp, img, msq, target, g_out,
                                                   loss_partials, g_scale, loss_kind, nullptr, err);
  return cudaGetLastError();
}

cudaError_t launch_adjoint(const Launcher& L, const SceneBuffers& s, const SegBuffers& t,
                           const ViewHost* views_dev, uint32_t n_views, uint32_t pix_begin, uint32_t n_pix,
                           const TraceParams& tp, const float* g_img, double* grad_acc,
                           float* gacc_scratch, uint32_t* err, cudaStream_t st) {
  const PathParams pp = make_path_params(tp, s);
  const uint64_t tasks = (n_pix + (32 / pp.group) - 1) / (32 / pp.group);
  // above wf_max_segments() segments the accumulators move to global memory
  const bool global = s.n_seg > wf_max_segments();
  if (global && !gacc_scratch) return cudaErrorInvalidValue;
  float* gacc = global ? gacc_scratch : nullptr;
  const size_t shmem = global ? 0 : sizeof(float) * 10u * s.n_seg;
  if (global) {
    cudaError_t e = cudaMemsetAsync(gacc, 0, sizeof(float) * 10u * s.n_seg, st);
    if (e != cudaSuccess) return e;
  }
  const ViewDev* vd = reinterpret_cast<const ViewDev*>(views_dev);
  const uint64_t n_paths = (uint64_t)n_pix * tp.spp;
  const uint32_t lanes = few_adjoint(L, n_paths) ? few_lanes(L, n_paths) : 0u;
  const int md = tp.max_depth < 1 ? 1 : (int)tp.max_depth;
#define IPT_LAUNCH_ADJ(D, I)                                                                         \
  {                                                                                                  \
    if (shmem > 48 * 1024)                                                                           \
      cudaFuncSetAttribute(k_adjoint<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shmem);  \
    const int grid = lanes ? few_grid(n_pix * tp.spp, lanes)                                         \
                           : grid_for(tasks, L.num_sms * L.adj_blocks_per_sm[I]);                    \
    k_adjoint<D><<<grid, kBlockThreads, shmem, st>>>(scene_dev(s), seg_dev(t), vd, n_views, pix_begin, n_pix, pp, \
                                                     lanes, g_img, grad_acc, gacc, err);             \
  }
  if (md <= 2)
    IPT_LAUNCH_ADJ(2, 0)
  else if (md <= 4)
    IPT_LAUNCH_ADJ(4, 1)
  else if (md <= 6)
    IPT_LAUNCH_ADJ(6, 2)
  else
    IPT_LAUNCH_ADJ(8, 3)
#undef IPT_LAUNCH_ADJ
  if (global) k_add_to_double<<<(10u * s.n_seg + 255) / 256, 256, 0, st>>>(gacc, 10u * s.n_seg, grad_acc);
  return cudaGetLastError();
}

static PathParams batch_path_params(const TraceParams& tp) {
  PathParams p{};
  p.spp = tp.spp;
  p.group = lanes_per_pixel(tp.spp);
  p.max_depth = tp.max_depth;
  p.nee = tp.nee;
  p.mis = tp.mis;
  p.profile = tp.profile;
  p.stride = tp.sample_stride ? tp.sample_stride : tp.spp;
  return p;
}

cudaError_t launch_forward_batch(const Launcher& L, const WfScene* tab_dev, uint32_t n_scenes, uint32_t total,
                                 const TraceParams& tp, const uint32_t* iter_dev, int loss_kind, double* loss_rows,
                                 uint32_t* err, cudaStream_t st) {
  // one block per loss row: every row of the batch's loss reduction is written
  PathParams pp = batch_path_params(tp);
  if (tp.serial_sums) serial_group(pp);
  const size_t sm = sizeof(double) * n_scenes;
  if (few_forward(L, (uint64_t)total * tp.spp)) {
    const uint32_t n = total * tp.spp, lanes = few_lanes(L, n);
    if (n)
      k_forward_samples_batch<<<few_grid(n, lanes), kBlockThreads, 0, st>>>(tab_dev, n_scenes, n, lanes, pp, tp.set,
                                                                          iter_dev, L.rad, err);
    k_forward_batch<true><<<loss_partials_capacity(L), kBlockThreads, sm, st>>>(
        tab_dev, n_scenes, total, pp, tp.set, iter_dev, loss_kind, loss_rows, L.rad, err);
    return cudaGetLastError();
  }
  k_forward_batch<false><<<loss_partials_capacity(L), kBlockThreads, sm, st>>>(
      tab_dev, n_scenes, total, pp, tp.set, iter_dev, loss_kind, loss_rows, nullptr, err);
  return cudaGetLastError();
}

uint32_t batch_shared_params() { return (96u * 1024u) / (uint32_t)sizeof(float); }

cudaError_t launch_adjoint_batch(const Launcher& L, const WfScene* tab_dev, uint32_t n_scenes, uint32_t total,
                                 uint32_t n_seg, const TraceParams& tp, const uint32_t* iter_dev, double* grad_acc,
                                 float* gacc_scratch, uint32_t* err, cudaStream_t st) {
  const PathParams pp = batch_path_params(tp);
  const uint32_t n_par = 10u * n_seg;
  const bool global = n_par > batch_shared_params();
  if (global && !gacc_scratch) return cudaErrorInvalidValue;
  float* gacc = global ? gacc_scratch : nullptr;
  const size_t shmem = global ? 0 : sizeof(float) * n_par;
  if (global) {
    cudaError_t e = cudaMemsetAsync(gacc, 0, sizeof(float) * n_par, st);
    if (e != cudaSuccess) return e;
  }
  const uint64_t tasks = ((uint64_t)total + (32 / pp.group) - 1) / (32 / pp.group);
  const uint64_t n_paths = (uint64_t)total * tp.spp;
  const uint32_t lanes = few_adjoint(L, n_paths) ? few_lanes(L, n_paths) : 0u;
  const int md = tp.max_depth < 1 ? 1 : (int)tp.max_depth;
#define IPT_LAUNCH_ADJB(D, I)                                                                              \
  {                                                                                                        \
    if (shmem > 48 * 1024)                                                                                 \
      cudaFuncSetAttribute(k_adjoint_batch<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shmem);  \
    const int grid = lanes ? few_grid((uint32_t)n_paths, lanes)                                            \
                           : grid_for(tasks, L.num_sms * L.adj_blocks_per_sm[I]);                          \
    k_adjoint_batch<D><<<grid, kBlockThreads, shmem, st>>>(tab_dev, n_scenes, total, n_par, pp, lanes,     \
                                                           tp.set, iter_dev, grad_acc, gacc, err);         \
  }
  if (md <= 2)
    IPT_LAUNCH_ADJB(2, 0)
  else if (md <= 4)
    IPT_LAUNCH_ADJB(4, 1)
  else if (md <= 6)
    IPT_LAUNCH_ADJB(6, 2)
  else
    IPT_LAUNCH_ADJB(8, 3)
#undef IPT_LAUNCH_ADJB
  if (global) k_add_to_double<<<(n_par + 255) / 256, 256, 0, st>>>(gacc, n_par, grad_acc);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const double* loss_partials, int n_partials, double* loss_dev,
                            const double* grad_acc, float* grad_out, uint32_t n_params,
                            cudaStream_t st) {
  // many parameters (a segment per triangle): the gradient leaves over a grid
  // (100k values: 96 us by the one block)
  const bool wide = grad_out && n_params > 10u * kWideSegments;
  if (wide)
    k_grad_out<<<(int)std::min<uint32_t>((n_params + 255u) / 256u, 1024u), 256, 0, st>>>(grad_acc, grad_out, n_params);
  if (!wide || loss_dev)
    k_finalize<<<1, 256, 0, st>>>(loss_partials, n_partials, loss_dev, grad_acc, wide ? nullptr : grad_out, n_params);
  return cudaGetLastError();
}

cudaError_t launch_adam(const SceneBuffers& s, const SegBuffers& t, float* params, float* m,
                        float* v, const uint8_t* free_mask, const double* grad_acc,
                        const float* grad_f, int* step_dev, const AdamHost& a, const double* loss,
                        uint32_t* guard, uint32_t* err, cudaStream_t st) {
  if (s.n_seg > kWideSegments) {
    k_finite_guard<<<1, 1024, 0, st>>>(loss, grad_acc, grad_f, 10u * s.n_seg, guard, err);
    const int grid = (int)std::min<uint32_t>((10u * s.n_seg + 255u) / 256u, 2048u);
    k_adam_wide<<<grid, 256, 0, st>>>(params, m, v, free_mask, grad_acc, grad_f, step_dev, a, s.n_seg, guard);
    return launch_tables_wide(s, t, params, params, step_dev, guard, st);
  }
  k_adam<<<1, 256, 0, st>>>(params, m, v, free_mask, grad_acc, grad_f, step_dev, a, s.n_seg,
                            s.emission_scale, s.seg_area, t, loss, err);
  return cudaGetLastError();
}

cudaError_t launch_adam_batch(const BatchMember* members, uint32_t n_members, float* params, float* m, float* v,
                              const uint8_t* free_mask, const double* grad_acc, const uint32_t* iter_dev,
                              const AdamHost& a, const double* losses, uint32_t* err, cudaStream_t st) {
  k_adam_batch<<<n_members, 256, 0, st>>>(members, params, m, v, free_mask, grad_acc, iter_dev, a, losses, err);
  return cudaGetLastError();
}

cudaError_t launch_prepare_batch(const BatchMember* members, uint32_t n_members, const float* params,
                                 cudaStream_t st) {
  k_prepare_batch<<<n_members, 256, 0, st>>>(members, params);
  return cudaGetLastError();
}

cudaError_t launch_batch_losses(const double* rows, int n_rows, const BatchMember* members, uint32_t n,
                                uint32_t n_tab, double* loss, cudaStream_t st) {
  k_batch_losses<<<n, 256, 0, st>>>(rows, n_rows, members, n_tab, loss);
  return cudaGetLastError();
}

cudaError_t launch_tick(uint32_t* counter, cudaStream_t st) {
  k_tick<<<1, 1, 0, st>>>(counter);
  return cudaGetLastError();
}

cudaError_t launch_philox(uint32_t n, const uint32_t* ctr, const uint32_t* key, uint32_t* out,
                          cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_philox<<<(n + 255) / 256, 256, 0, st>>>(n, ctr, key, out);
  return cudaGetLastError();
}

}  // namespace ipt
