// Optimiser step of the training loop (Sec. 3.2 "Optimizing 3D GS
// representations"; the paper names neither the optimiser nor the
// activations, so this is the 3DGS practice): Adam on unconstrained raw
// parameters
//   raw = (p, log s, q, log rho),   params = (p, exp(log s), q, exp(log rho)),
// the quaternion staying raw (the projection normalises it).  The gradient
// comes in with respect to params and is carried to raw by the chain rule
// (d/dlog s = s d/ds, d/dlog rho = rho d/drho).
#include <math.h>

#include "gem_internal.cuh"

namespace gem {

// Parameter group of entry m of a Gaussian: 0 centre, 1 scale, 2 rotation,
// 3 density.
__device__ __forceinline__ int group_of(int m) { return m < 3 ? 0 : (m < 6 ? 1 : (m < 10 ? 2 : 3)); }

__device__ __forceinline__ bool is_log(int m) { return (m >= 3 && m < 6) || m == 10; }

// Entry m of Gaussian j (iso: its imposed scale, or NULL).
__device__ __forceinline__ void adam_entry(const AdamArgs &a, int m, unsigned j, float &raw, float &mo,
                                           float &ve, float grad, float &param,
                                           const float *__restrict__ iso) {
  float r = raw;
  if (iso && m >= 3 && m < 6) {
    // isotropic ablation: the scale is the given distance, not learnt
    const float s = iso[j];
    raw = logf(s);
    param = s;
    return;
  }
  const float p = is_log(m) ? expf(r) : r;
  float g = grad;
  if (is_log(m)) g *= p;
  if (!isfinite(g)) g = 0.f;
  const float mm = a.beta1 * mo + (1.f - a.beta1) * g;
  const float vv = a.beta2 * ve + (1.f - a.beta2) * g * g;
  mo = mm;
  ve = vv;
  const float mhat = mm * a.c1, vhat = vv * a.c2;
  r -= a.lr[group_of(m)] * mhat / (sqrtf(vhat) + a.eps);
  raw = r;
  param = is_log(m) ? expf(r) : r;
}

// Bound by HBM: eight arrays of [M][11] floats read or written once.  A
// thread takes kVec consecutive entries (four 16-byte loads in flight, four
// stores) when all five arrays are 16-byte aligned and that leaves the GPU two
// CTAs per SM (at M = 6941 a call takes 2% longer with four entries per thread
// than with one), else one; M <= 2^24, so entry numbers fit 32 bits.
// M = 500000 (176 MB): 35 us with one entry per thread and 64-bit remainders,
// 25 us with four, where a copy of as many bytes takes 26 (a repeated step
// finds part of them in the 129 MB L2).
template <int kVec>
__global__ void __launch_bounds__(256) adam_step_kernel(AdamArgs a, unsigned n,
                                                        float *__restrict__ raw,
                                                        float *__restrict__ mo,
                                                        float *__restrict__ ve,
                                                        const float *__restrict__ grad,
                                                        float *__restrict__ params,
                                                        const float *__restrict__ iso) {
  const unsigned i = (blockIdx.x * blockDim.x + threadIdx.x) * kVec;
  if (i >= n) return;
  unsigned j = i / kNpar;
  int m = (int)(i - j * kNpar);
  if (kVec == 4 && i + 4 <= n) {
    float4 r = *reinterpret_cast<const float4 *>(raw + i), mm = *reinterpret_cast<const float4 *>(mo + i);
    float4 vv = *reinterpret_cast<const float4 *>(ve + i);
    const float4 g = __ldg(reinterpret_cast<const float4 *>(grad + i));
    float4 p;
    auto next = [&]() {
      if (++m == kNpar) m = 0, ++j;
    };
    adam_entry(a, m, j, r.x, mm.x, vv.x, g.x, p.x, iso);
    next();
    adam_entry(a, m, j, r.y, mm.y, vv.y, g.y, p.y, iso);
    next();
    adam_entry(a, m, j, r.z, mm.z, vv.z, g.z, p.z, iso);
    next();
    adam_entry(a, m, j, r.w, mm.w, vv.w, g.w, p.w, iso);
    *reinterpret_cast<float4 *>(raw + i) = r;
    *reinterpret_cast<float4 *>(mo + i) = mm;
    *reinterpret_cast<float4 *>(ve + i) = vv;
    *reinterpret_cast<float4 *>(params + i) = p;
    return;
  }
  for (unsigned k = i; k < n && k < i + kVec; ++k) {
    adam_entry(a, m, j, raw[k], mo[k], ve[k], grad[k], params[k], iso);
    if (++m == kNpar) m = 0, ++j;
  }
}

__global__ void __launch_bounds__(256) activate_kernel(int64_t n, const float *__restrict__ raw,
                                                       float *__restrict__ params) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int m = (int)(i % kNpar);
  params[i] = is_log(m) ? expf(raw[i]) : raw[i];
}

cudaError_t launch_adam(const AdamArgs &a, int64_t M, float *raw, float *m, float *v,
                        const float *grad, float *params, const float *iso, cudaStream_t st) {
  const unsigned n = (unsigned)(M * kNpar);
  const uintptr_t all = (uintptr_t)raw | (uintptr_t)m | (uintptr_t)v | (uintptr_t)grad | (uintptr_t)params;
  if ((all & 15u) == 0 && n >= 2 * 152 * 1024)
    adam_step_kernel<4><<<(n + 1023) / 1024, 256, 0, st>>>(a, n, raw, m, v, grad, params, iso);
  else
    adam_step_kernel<1><<<(n + 255) / 256, 256, 0, st>>>(a, n, raw, m, v, grad, params, iso);
  return cudaGetLastError();
}

cudaError_t launch_activate(int64_t M, const float *raw, float *params, cudaStream_t st) {
  const int64_t n = M * kNpar;
  activate_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, raw, params);
  return cudaGetLastError();
}

}  // namespace gem
