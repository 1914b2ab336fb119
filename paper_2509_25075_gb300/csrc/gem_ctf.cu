// Step a4 of the GEM hot path: Eq. loss and its adjoint.
//
//   I_pred = F^-1(H . F(I^)),  r = I_pred - I,  L = (1/B) sum_b mean(r^2),
//   dL/dI^ = F^-1(H . F(2 r / (B d^2)))   (H real and even: self-adjoint).
//
// Both real images of a view are packed into one complex image
// z = I^ + i I, so F(z) = X + i Y with X = F(I^), Y = F(I) recovered from the
// Hermitian symmetry of real spectra.  In Fourier space
//   P = H X,  R = H X - Y  (= F(r)),  G = H R,
// the loss is (by Parseval) sum |R|^2 / d^4 per image, and one inverse
// transform of W = P + i G returns I_pred (real part) and, times
// 2 / (B d^2), dL/dI^ (imaginary part).  G is transformed unscaled so that
// both halves of W have comparable magnitude and share the FFT's rounding
// fairly.  So each image costs one forward and one inverse complex 2D FFT.
//
// Three passes through a [B][d][d] complex buffer, stored transposed
// (Z[b][kx][y]) so that every FFT runs on contiguous lines:
//   pass 1: FFT along x of kLines rows of z, written transposed;
//   pass 2: FFT along y of the lines kx and d - kx (kLines / 2 pairs per CTA; the
//           first CTA holds the self-paired lines 0 and d/2 in the slots
//           of line 0's pair), CTF, loss, W, inverse FFT along y, written
//           back in place;
//   pass 3: inverse FFT along x of kLines rows, split into I_pred and dL/dI^.
// FFTs are radix-4/2/3 Stockham transforms (gem_fft.cuh), instantiated for
// every side.
//
// Bound by latency (two or three barriers per pass and the reads of the
// spectrum, which stays in L2).  Against a shared-memory round trip per radix
// stage and separate copies in and out, same arithmetic and bits: d 144, B 50,
// transfer arrays, every output: the call 51.7 -> 34.8 us.  The CTF constants
// are worked out beside the first pass (the double-precision chain of one
// thread otherwise opens every CTA of the second) and the losses folded by the
// last CTAs of the second instead of two launches: 34.8 -> 33.5 us there, and
// a d 256, B 64 prediction with CTF parameters 1083 -> 1069 us.
#include <math.h>

#include "gem_fft.cuh"
#include "gem_internal.cuh"

namespace gem {

// Lines per CTA in every pass: 16 up to side 208, else 8 (large images: more,
// smaller CTAs, so the last wave is short).  The line was drawn when a CTA held
// two line buffers (d 384, B 16: 16 lines 0.168 ms, 8 lines 0.125; d 128, B 256:
// 0.151 and 0.167); the second pass's line count is also the order in which an
// image's loss is summed, so it stays.
constexpr int kCtfThreads = 256;
__host__ __device__ constexpr int ctf_lines(int d) { return d <= 208 ? 16 : 8; }

template <int N>
struct CtfSmem {
  float2 lines[ctf_lines(N) * fft_stride(N)];
  float2 tw[N];
};

// A float-float number hi + lo (|lo| <= ulp(hi) / 2).
struct FF {
  float hi, lo;
};

__device__ __forceinline__ FF ff_split(double x) {
  FF r;
  r.hi = (float)x;
  r.lo = (float)(x - (double)r.hi);
  return r;
}

// c * N for an integer-valued float N (|N| < 2^24), reduced modulo 1: the
// product of the high parts is error-free (fmaf), its integer part dropped.
__device__ __forceinline__ FF ff_mul_mod1(FF c, float N) {
  float p = c.hi * N;
  float e = fmaf(c.hi, N, -p);
  FF r;
  r.hi = p - rintf(p);
  r.lo = fmaf(c.lo, N, e);
  return r;
}

__device__ __forceinline__ FF ff_add(FF a, FF b) {
  float s = a.hi + b.hi;
  float bb = s - a.hi;
  float err = (a.hi - (s - bb)) + (b.hi - bb);
  FF r;
  r.hi = s;
  r.lo = err + a.lo + b.lo;
  return r;
}

// Per-image CTF constants for the parameter form, in turns (chi / 2 pi):
//   chi / (2 pi) = lambda/2 dF(angle) k^2 - Cs lambda^3 k^4 / 4 + phase / (2 pi),
// with k = n / (d apix) for the signed bin indices n = (kx, ky).
// dF(angle) k^2 expands into integer multiples (kx^2 + ky^2, kx^2 - ky^2,
// 2 kx ky) of per-image constants, so no angle is formed, and every term is
// a constant times an integer, evaluated in float-float and reduced modulo
// one turn (tens of turns at Nyquist would otherwise cost float32 its
// accuracy).
struct CtfConst {
  FF c1;   // turns per (kx^2 + ky^2), mean defocus
  FF c2;   // turns per (kx^2 - ky^2), astigmatism
  FF c3;   // turns per 2 kx ky, astigmatism
  FF c4;   // turns per (kx^2 + ky^2)^2, spherical aberration
  FF ph;   // phase shift, turns
  float sw, w;  // sqrt(1 - w^2), w
  float bq;     // B-factor damping per (kx^2 + ky^2)
};

__device__ CtfConst ctf_const(const float *__restrict__ prm, int d, float apix) {
  double dU = prm[0], dV = prm[1], volt = (double)prm[3] * 1e3;
  double cs = (double)prm[4] * 1e7, w = prm[5], phase = prm[6], bf = prm[7];
  double lam = 12.2643247 / sqrt(volt * (1.0 + 0.978466e-6 * volt));
  double cf = 1.0 / ((double)d * apix * (double)d * apix);
  double mean = 0.5 * (dU + dV), half = 0.5 * (dU - dV);
  // the astigmatism terms reach a fraction of a turn at Nyquist, so the
  // angle's cosine and sine need float accuracy only (kept off the slow
  // double-precision path, which this single thread runs while its CTA waits)
  float s2a, c2a;
  sincosf(2.f * prm[2], &s2a, &c2a);
  CtfConst c;
  c.c1 = ff_split(0.5 * lam * mean * cf);
  c.c2 = ff_split(0.5 * lam * half * (double)c2a * cf);
  c.c3 = ff_split(0.5 * lam * half * (double)s2a * cf);
  c.c4 = ff_split(-0.25 * cs * lam * lam * lam * cf * cf);
  c.ph = ff_split(phase / (2.0 * 3.14159265358979323846));
  c.sw = (float)sqrt(1.0 - w * w);
  c.w = (float)w;
  c.bq = (float)(bf * cf / 4.0);
  return c;
}

// CTF at signed bin indices (sx, sy).
__device__ __forceinline__ float ctf_at(const CtfConst &c, int sx, int sy) {
  float x2 = (float)(sx * sx), y2 = (float)(sy * sy);
  float n2 = x2 + y2;  // exact (< 2^24)
  FF t = ff_mul_mod1(c.c1, n2);
  t = ff_add(t, ff_mul_mod1(c.c2, x2 - y2));
  t = ff_add(t, ff_mul_mod1(c.c3, (float)(2 * sx * sy)));
  // (n2)^2 as an exact float-float q + qe, then c4 q mod 1 + c4 qe
  float q = n2 * n2;
  float qe = fmaf(n2, n2, -q);
  FF t4 = ff_mul_mod1(c.c4, q);
  t4.lo = fmaf(c.c4.hi, qe, t4.lo);
  t = ff_add(t, t4);
  t = ff_add(t, c.ph);
  float turns = (t.hi - rintf(t.hi)) + t.lo;
  float s, co;
  sincospif(2.f * turns, &s, &co);
  return -(c.sw * s + c.w * co) * __expf(-c.bq * n2);
}

// pass 1: rows y0 .. y0 + L - 1 of z = proj + i images -> FFT along x -> Z[b][kx][y].
// In the parameter form one more CTA per image works out its CTF constants
// (a chain of double-precision operations in one thread), beside the others.
template <int N>
__global__ void __launch_bounds__(kCtfThreads) ctf_pass1_kernel(
    const float *__restrict__ proj, const float *__restrict__ images,
    const float2 *__restrict__ tw, const float *__restrict__ ctf_params, float apix,
    CtfConst *__restrict__ consts, float2 *__restrict__ Z) {
  constexpr int L = ctf_lines(N);
  extern __shared__ __align__(16) unsigned char ctf_sm[];
  CtfSmem<N> &S = *reinterpret_cast<CtfSmem<N> *>(ctf_sm);
  const int y0 = blockIdx.x * L, b = blockIdx.y;
  if (blockIdx.x == N / L) {
    if (threadIdx.x == 0) consts[b] = ctf_const(ctf_params + 8 * b, N, apix);
    return;
  }
  load_twiddles<N, kCtfThreads>(S.tw, tw);
  __syncthreads();
  const float *pr = proj + ((int64_t)b * N + y0) * N;
  const float *im = images + ((int64_t)b * N + y0) * N;
  float2 *zb = Z + (int64_t)b * N * N + y0;
  fft_lines<N, L, kCtfThreads, false, false, false, true>(
      [&](int l, int x) { return make_float2(pr[l * N + x], im[l * N + x]); },
      [&](int l, int kx, float2 v) { zb[kx * N + l] = v; }, S.lines, S.tw);
}

__device__ __forceinline__ int signed_bin(int k, int d) { return k < d / 2 ? k : k - d; }

// Line kx held in slot i of pass-2 CTA blk (see ctf_pass2_kernel).
template <int kHalf>
__device__ __forceinline__ int pass2_line(int blk, int i, int d) {
  const int kx1 = kHalf * blk + (i & (kHalf - 1));
  return i < kHalf ? kx1 : (kx1 == 0 ? d / 2 : d - kx1);
}

// Where the losses go: the CTAs' partials part[b][gridDim.x], the per-image
// losses img[b] (NULL: not wanted), their mean (may be NULL), and counters
// [B + 1] of the CTAs and images that are done, zero between calls.
struct LossOut {
  double *part, *img, *mean;
  double inv_d4;
  unsigned *done;
};

// One warp, after its CTA has stored its partial: the last CTA of an image
// adds the image's partials / d^4, the last image's takes the mean, both in a
// fixed order (deterministic).
__device__ __forceinline__ void fold_loss(const LossOut &lo, int b) {
  const int lane = threadIdx.x & 31, B = (int)gridDim.y, nblk = (int)gridDim.x;
  unsigned prev = 0;
  if (lane == 0) {
    __threadfence();
    prev = atomicAdd(lo.done + b, 1u);
  }
  if (__shfl_sync(0xffffffffu, prev, 0) != (unsigned)nblk - 1) return;
  __threadfence();
  double s = 0.0;
  for (int c = lane; c < nblk; c += 32) s += __ldcg(lo.part + (int64_t)b * nblk + c);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    __stcg(lo.img + b, s * lo.inv_d4);
    lo.done[b] = 0u;  // as the next call expects it
    if (lo.mean) {
      __threadfence();
      prev = atomicAdd(lo.done + B, 1u);
    }
  }
  if (!lo.mean || __shfl_sync(0xffffffffu, prev, 0) != (unsigned)B - 1) return;
  __threadfence();
  double t = 0.0;
  for (int w = 0; w < 8; ++w) {
    double m = 0.0;
    for (int q = 32 * w + lane; q < B; q += 256) m += __ldcg(lo.img + q);
    for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
    t += m;
  }
  if (lane == 0) {
    *lo.mean = t / B;
    lo.done[B] = 0u;
  }
}

// pass 2: slots i < kHalf hold the lines kx1 = kHalf c + i (kx1 < d/2),
// slots kHalf + i their partners d - kx1; line 0 is its own partner, so its
// slot kHalf holds the other self-paired line, d/2.  d is a multiple of
// the line count, so the d / L CTAs of an image hold every line once.
template <int N>
__global__ void __launch_bounds__(kCtfThreads) ctf_pass2_kernel(
    const float2 *__restrict__ tw, const float *__restrict__ ctf,
    const CtfConst *__restrict__ consts, float2 *__restrict__ Z, LossOut lo) {
  constexpr int kLines = ctf_lines(N), kHalf = kLines / 2;  // line pairs per CTA
  constexpr int d = N, hd = N / 2, ls = fft_stride(N);
  extern __shared__ __align__(16) unsigned char ctf_sm[];
  CtfSmem<N> &S = *reinterpret_cast<CtfSmem<N> *>(ctf_sm);
  __shared__ CtfConst cc;
  __shared__ double red[kCtfThreads / 32];
  const int blk = blockIdx.x, b = blockIdx.y;
  load_twiddles<N, kCtfThreads>(S.tw, tw);
  if (consts && threadIdx.x == 0) cc = consts[b];
  float2 *zb = Z + (int64_t)b * d * d;
  __syncthreads();
  float2 *L = S.lines;
  fft_lines<N, kLines, kCtfThreads, false, true, false, false>(
      [&](int i, int y) { return zb[pass2_line<kHalf>(blk, i, d) * d + y]; }, FftNone{}, L, S.tw);
  // combine: thread per (pair i, ky); the first CTA has one more "pair",
  // the self-paired line d/2 in slot kHalf
  float lsum = 0.f;
  const int npair = blk == 0 ? kHalf + 1 : kHalf;
  for (int idx = threadIdx.x; idx < npair * d; idx += blockDim.x) {
    int i = idx / d, ky = idx - i * d;
    int kx = i < kHalf ? kHalf * blk + i : hd;
    bool self = (kx == 0 || kx == hd);
    if (self && ky > hd) continue;
    int mky = ky == 0 ? 0 : d - ky;
    float2 *l1 = L + i * ls;
    float2 *l2 = self ? l1 : L + (kHalf + i) * ls;
    float2 z1 = l1[fft_at(ky)], z2 = l2[fft_at(mky)];
    // X = (z1 + conj z2) / 2,  Y = (z1 - conj z2) / (2 i)
    float2 X = make_float2(0.5f * (z1.x + z2.x), 0.5f * (z1.y - z2.y));
    float2 Yv = make_float2(0.5f * (z1.y + z2.y), -0.5f * (z1.x - z2.x));
    float h;
    if (consts) {
      int sx = signed_bin(kx, d), sy = signed_bin(ky, d);
      h = ctf_at(cc, sx, sy);
      if (kx == hd || ky == hd) {
        int px = signed_bin(kx == 0 ? 0 : d - kx, d), py = signed_bin(mky, d);
        h = 0.5f * (h + ctf_at(cc, px, py));
      }
    } else {
      const float *hb = ctf + (int64_t)b * d * (hd + 1);
      h = hb[(int64_t)ky * (hd + 1) + kx];
      if (self) h = 0.5f * (h + hb[(int64_t)mky * (hd + 1) + kx]);
    }
    float2 P = make_float2(h * X.x, h * X.y);
    float2 Rr = make_float2(P.x - Yv.x, P.y - Yv.y);
    float2 G = make_float2(h * Rr.x, h * Rr.y);
    float r2 = Rr.x * Rr.x + Rr.y * Rr.y;
    bool lone = self && (ky == 0 || ky == hd);
    lsum += lone ? r2 : 2.f * r2;
    // W(k) = P + i G;  W(-k) = conj P + i conj G.  Stored conjugated: the
    // inverse transform runs as conj(FFT(conj .)).
    // (products and sums rounded on their own, whatever the side's instance)
    float2 W = make_float2(__fsub_rn(P.x, G.y), __fadd_rn(P.y, G.x));
    float2 Wm = make_float2(__fadd_rn(P.x, G.y), __fsub_rn(G.x, P.y));
    l1[fft_at(ky)] = make_float2(W.x, -W.y);
    l2[fft_at(mky)] = make_float2(Wm.x, -Wm.y);
  }
  // block reduction of the loss partial in float64
  double lw = (double)lsum;
  for (int o = 16; o > 0; o >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lw;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kCtfThreads / 32; ++w) s += red[w];
    __stcg(lo.part + (int64_t)b * gridDim.x + blk, s);
  }
  // inverse along y (conjugated forward transform)
  fft_lines<N, kLines, kCtfThreads, true, false, false, false>(
      FftNone{},
      [&](int i, int y, float2 v) {
        zb[pass2_line<kHalf>(blk, i, d) * d + y] = make_float2(v.x, -v.y);
      },
      L, S.tw);
  if (lo.img && threadIdx.x < 32) fold_loss(lo, b);
}

// pass 3: rows y0 .. y0 + L - 1 of W (read transposed) -> inverse FFT along x ->
// I_pred = Re / d^2, dL/dI^ = Im (2 / (B d^2)) / d^2.
template <int N>
__global__ void __launch_bounds__(kCtfThreads) ctf_pass3_kernel(
    const float2 *__restrict__ tw, const float2 *__restrict__ Z, float inv_n2,
    float gscale, float *__restrict__ pred, float *__restrict__ dproj) {
  constexpr int L = ctf_lines(N);
  extern __shared__ __align__(16) unsigned char ctf_sm[];
  CtfSmem<N> &S = *reinterpret_cast<CtfSmem<N> *>(ctf_sm);
  const int y0 = blockIdx.x * L, b = blockIdx.y;
  load_twiddles<N, kCtfThreads>(S.tw, tw);
  __syncthreads();
  const float2 *zb = Z + (int64_t)b * N * N + y0;
  const int64_t off = ((int64_t)b * N + y0) * N;
  fft_lines<N, L, kCtfThreads, false, false, true, false>(
      [&](int l, int kx) {
        const float2 v = zb[kx * N + l];
        return make_float2(v.x, -v.y);
      },
      [&](int l, int x, float2 v) {
        if (pred) pred[off + l * N + x] = v.x * inv_n2;
        if (dproj) dproj[off + l * N + x] = -v.y * gscale;
      },
      S.lines, S.tw);
}

size_t ctf_partials(int d) { return (size_t)(d / ctf_lines(d)); }

template <int N>
static cudaError_t ctf_configure_side() {
  const int smem = (int)sizeof(CtfSmem<N>);
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(ctf_pass1_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                smem)) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(ctf_pass2_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                smem)) != cudaSuccess)
    return e;
  return cudaFuncSetAttribute(ctf_pass3_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t ctf_configure(int d) {
  switch (d) {
#define X(N) \
  case N:    \
    return ctf_configure_side<N>();
    GEM_FFT_SIDES(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

template <int N>
static void launch_ctf_passes(int B, float apix, const float2 *tw, const float *proj,
                              const float *ctf, const float *ctf_params, const float *images,
                              float2 *Z, CtfConst *consts, const LossOut &lo, float *pred,
                              float *dproj, cudaStream_t st) {
  const size_t smem = sizeof(CtfSmem<N>);
  const dim3 grid(N / ctf_lines(N), B);
  const float cscale = (float)(2.0 / ((double)B * N * N));
  ctf_pass1_kernel<N><<<dim3(grid.x + (ctf_params ? 1 : 0), B), kCtfThreads, smem, st>>>(
      proj, images, tw, ctf_params, apix, consts, Z);
  ctf_pass2_kernel<N><<<grid, kCtfThreads, smem, st>>>(tw, ctf, ctf_params ? consts : nullptr, Z, lo);
  ctf_pass3_kernel<N><<<grid, kCtfThreads, smem, st>>>(tw, Z, (float)(1.0 / ((double)N * N)),
                                                       (float)(cscale / ((double)N * N)), pred, dproj);
}

cudaError_t launch_ctf_loss(int d, int B, float apix, const float2 *tw,
                            const float *proj, const float *ctf, const float *ctf_params,
                            const float *images, const CtfScratch &s, float *pred,
                            float *dproj, double *loss_img, double *loss, cudaStream_t st) {
  static_assert(sizeof(CtfConst) <= kCtfConstFloats * sizeof(float), "constants of an image");
  // per-image losses land in loss_img, or after the partials when the
  // caller does not want them (lossp holds max_B * partials + max_B doubles)
  LossOut lo;
  lo.part = s.lossp;
  lo.img = loss_img ? loss_img : loss ? s.lossp + (int64_t)B * ctf_partials(d) : nullptr;
  lo.mean = loss;
  lo.inv_d4 = 1.0 / ((double)d * d * (double)d * d);
  lo.done = s.done;
  CtfConst *consts = reinterpret_cast<CtfConst *>(s.consts);
  switch (d) {
#define X(N)                                                                                         \
  case N:                                                                                            \
    launch_ctf_passes<N>(B, apix, tw, proj, ctf, ctf_params, images, s.Z, consts, lo, pred, dproj, st); \
    break;
    GEM_FFT_SIDES(X)
#undef X
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace gem
