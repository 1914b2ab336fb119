// Density query (Eq. query): V(x) = sum_j G_j(x) on the d^3 voxel grid,
// with the contribution threshold of Eq. accu applied per voxel.
//
// Each z-slice of the volume is rendered as an image by the same binning and
// forward rasteriser as the projections.  Restricted to the plane z = z_k, a
// 3D Gaussian is exactly a 2D Gaussian: with P = Sigma^-1 split into its xy
// block P_aa and the rest,
//   (x - p)^T P (x - p) = (a - m)^T P_aa (a - m) + (z - p_z)^2 / Sigma_zz,
//   m = p_a + (Sigma_az / Sigma_zz) (z - p_z)            (Schur complement),
// so the slice record has conic P_aa, centre m(z_k) and log2 amplitude
// log2 A3 - (log2 e / 2) (z_k - p_z)^2 / Sigma_zz.  Slices are independent
// "images" and run in batches of the context's max_B.
//
// A Gaussian exceeds tau in a dozen slices, so each slice gets the list of
// the Gaussians that can matter there (their range of slices is known once
// the threshold is), and only those get a record and enter the binning.  With
// a record of every Gaussian in every slice, the records and the count pass
// over them were 60% of a query (d 256, M 100000, batches of 64 slices:
// 1.27 ms; 0.43 ms now).
#include "gem_internal.cuh"

namespace gem {

__global__ void __launch_bounds__(256) query_prep_kernel(const float *__restrict__ params,
                                                         int64_t M, int norm_mode, int shape,
                                                         float apix, int d, float l2tau,
                                                         QueryPrep *__restrict__ qp,
                                                         uint32_t *__restrict__ range) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const float *th = params + j * kNpar;
  const bool iso = (shape & kIsotropic) != 0, fixed = (shape & kNoRotation) != 0;
  const float s0 = th[3], s1 = iso ? th[3] : th[4], s2 = iso ? th[3] : th[5];
  const float qw = fixed ? 1.f : th[6], qx = fixed ? 0.f : th[7], qy = fixed ? 0.f : th[8],
              qz = fixed ? 0.f : th[9];
  const float rho = th[10];
  const float qn = sqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
  QueryPrep o;
  o.p[0] = th[0];
  o.p[1] = th[1];
  o.p[2] = th[2];
  const float iq = qn > 0.f ? 1.f / qn : 0.f;
  float R[9];
  quat_rot(qw * iq, qx * iq, qy * iq, qz * iq, R);
  const float a0 = s0 * s0, a1 = s1 * s1, a2 = s2 * s2;
  const float b0 = 1.f / a0, b1 = 1.f / a1, b2 = 1.f / a2;
  // P = R diag(1/s^2) R^T (xy block), Sigma = R diag(s^2) R^T (z column)
  o.pxx = R[0] * R[0] * b0 + R[1] * R[1] * b1 + R[2] * R[2] * b2;
  o.pxy = R[0] * R[3] * b0 + R[1] * R[4] * b1 + R[2] * R[5] * b2;
  o.pyy = R[3] * R[3] * b0 + R[4] * R[4] * b1 + R[5] * R[5] * b2;
  // det of that block by Cauchy-Binet (the squared 2x2 minors of the first
  // two rows of R, weighted): positive terms, no cancellation for an
  // elongated Gaussian
  const float m12 = fmaf(R[1], R[5], -R[2] * R[4]);
  const float m20 = fmaf(R[2], R[3], -R[0] * R[5]);
  const float m01 = fmaf(R[0], R[4], -R[1] * R[3]);
  o.pdet = b1 * b2 * m12 * m12 + b0 * b2 * m20 * m20 + b0 * b1 * m01 * m01;
  const float sxz = R[0] * R[6] * a0 + R[1] * R[7] * a1 + R[2] * R[8] * a2;
  const float syz = R[3] * R[6] * a0 + R[4] * R[7] * a1 + R[5] * R[8] * a2;
  const float szz = R[6] * R[6] * a0 + R[7] * R[7] * a1 + R[8] * R[8] * a2;
  o.hz = 1.f / szz;
  o.mx = sxz * o.hz;
  o.my = syz * o.hz;
  // 3D amplitude: rho (peak density, Eq. G) in mode 1; rho / ((2 pi)^3/2
  // |s0 s1 s2|) in mode 0, the density whose line integral is Eq. render
  const float two_pi = 6.283185307179586f;
  o.l2A = norm_mode == 0 ? log2f(rho / (two_pi * sqrtf(two_pi) * fabsf(s0 * s1 * s2)))
                         : log2f(rho);
  const bool ok = qn > 0.f && isfinite(qn) && rho > 0.f && isfinite(rho) && isfinite(o.l2A) &&
                  isfinite(o.pxx) && isfinite(o.pxy) && isfinite(o.pyy) && isfinite(o.hz) &&
                  isfinite(o.mx) && isfinite(o.my) && isfinite(o.p[0]) && isfinite(o.p[1]) &&
                  o.pdet > 0.f && isfinite(o.pdet) &&
                  isfinite(o.p[2]) && a0 > 0.f && a1 > 0.f && a2 > 0.f;
  o.valid = ok ? 1.f : 0.f;
  qp[j] = o;
  // headroom l2A - (log2 e / 2) dz^2 hz > l2tau, widened by far more than the
  // rounding of either side; the record's own test stays exact
  unsigned r = 1u;  // none
  const float head = o.l2A - l2tau;
  if (ok && head > 0.f) {
    const float D = sqrtf(head * (2.f / kLog2e) / o.hz) / apix * (1.f + 1e-4f) + 0.05f;
    const float c = o.p[2] / apix + 0.5f * d;
    const float lo = fmaxf(ceilf(c - D), 0.f), hi = fminf(floorf(c + D), (float)(d - 1));
    if (lo <= hi) r = (unsigned)lo | ((unsigned)hi << 16);
  }
  range[j] = r;
}

// Record of (slice k, Gaussian g), in the layout of Rec.
__device__ __forceinline__ Rec slice_record(const QueryPrep &g, int k, float apix, int d, float l2tau) {
  const float z = ((float)k - 0.5f * d) * apix;
  const float dz = z - g.p[2];
  const float inv = 1.f / apix;
  const float px = fmaf(fmaf(g.mx, dz, g.p[0]), inv, 0.5f * d);
  const float py = fmaf(fmaf(g.my, dz, g.p[1]), inv, 0.5f * d);
  const float a2 = apix * apix;
  const float cxx = g.pxx * a2, cxy = g.pxy * a2, cyy = g.pyy * a2;  // 1/pixel^2
  const float l2A = g.l2A - 0.5f * kLog2e * dz * dz * g.hz;
  const float det = g.pdet * a2 * a2;
  // U^T U = c^2 [[cxx, cxy], [cxy, cyy]] (the record layout of Rec)
  const float u11 = kC * sqrtf(cxx);
  const float u12 = u11 * (cxy / cxx);
  const float u22 = kC2 * sqrtf(det) / u11;
  Rec r;
  if (g.valid != 0.f && det > 0.f && isfinite(l2A) && u11 > 0.f && u22 > 0.f && isfinite(u11) &&
      isfinite(u12) && isfinite(u22)) {
    r.a = make_float4(px, py, u11, u12);
    r.b = make_float4(u22, l2A, -1.f, -1.f);
    const float kap = l2A - l2tau;
    if (kap > 0.f) {
      const float km = (kap + kMargin) * (2.f / kLog2e);
      r.b.z = sqrtf(km * cyy / det);  // covariance xx = cyy / det
      r.b.w = sqrtf(km * cxx / det);
    }
  } else {
    r.a = make_float4(px, py, 0.f, 0.f);
    r.b = make_float4(0.f, -INFINITY, -1.f, -1.f);
  }
  return r;
}

// Few (slice, Gaussian) pairs: a record of every Gaussian in every slice.
__global__ void __launch_bounds__(256) slice_all_kernel(const QueryPrep *__restrict__ qp, int64_t M,
                                                        int k0, float apix, int d, float l2tau,
                                                        Rec *__restrict__ rec) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < M) rec[(int64_t)blockIdx.y * M + j] = slice_record(qp[j], k0 + (int)blockIdx.y, apix, d, l2tau);
}

// Which Gaussians of chunk blockIdx.x (256 of them) meet which slices of the
// batch: one bit per Gaussian, bm[slice][8].
__device__ __forceinline__ void slice_bits(uint32_t *bm, const uint32_t *__restrict__ range, int64_t M,
                                           int k0, int ns, int &lo, int &hi) {
  const int64_t j = (int64_t)blockIdx.x * kChunkT + threadIdx.x;
  const unsigned r = j < M ? range[j] : 1u;
  lo = max((int)(r & 0xffffu) - k0, 0);
  hi = min((int)(r >> 16) - k0, ns - 1);
  if ((r & 0xffffu) > (r >> 16)) hi = lo - 1;
  for (int q = threadIdx.x; q < 8 * ns; q += kChunkT) bm[q] = 0u;
  __syncthreads();
  for (int k = lo; k <= hi; ++k) atomicOr(&bm[8 * k + (threadIdx.x >> 5)], 1u << (threadIdx.x & 31));
  __syncthreads();
}

// How many Gaussians of each chunk meet each slice: cnt[chunk][ns].
__global__ void __launch_bounds__(kChunkT) slice_count_kernel(const uint32_t *__restrict__ range,
                                                              int64_t M, int k0, int ns,
                                                              uint32_t *__restrict__ cnt) {
  extern __shared__ uint32_t bm[];
  int lo, hi;
  slice_bits(bm, range, M, k0, ns, lo, hi);
  for (int k = threadIdx.x; k < ns; k += kChunkT) {
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) n += __popc(bm[8 * k + w]);
    cnt[(int64_t)blockIdx.x * ns + k] = n;
  }
}

// The records and the lists, off[chunk][ns] (exclusive prefix over the
// chunks) saying where each chunk's Gaussians go in a slice's list.
__global__ void __launch_bounds__(kChunkT) slice_write_kernel(
    const QueryPrep *__restrict__ qp, const uint32_t *__restrict__ range, int64_t M, int k0, int ns,
    float apix, int d, float l2tau, const uint32_t *__restrict__ off, Rec *__restrict__ rec,
    uint32_t *__restrict__ sel) {
  extern __shared__ uint32_t bm[];
  int lo, hi;
  slice_bits(bm, range, M, k0, ns, lo, hi);
  if (lo > hi) return;
  const int64_t j = (int64_t)blockIdx.x * kChunkT + threadIdx.x;
  const QueryPrep g = qp[j];
  const int word = threadIdx.x >> 5;
  const uint32_t below = (1u << (threadIdx.x & 31)) - 1u;
  for (int k = lo; k <= hi; ++k) {
    uint32_t pos = off[(int64_t)blockIdx.x * ns + k] + __popc(bm[8 * k + word] & below);
    for (int w = 0; w < word; ++w) pos += __popc(bm[8 * k + w]);
    sel[(int64_t)k * M + pos] = (uint32_t)j;
    rec[(int64_t)k * M + j] = slice_record(g, k0 + k, apix, d, l2tau);
  }
}

// Few Gaussians: a CTA per slice goes over all their ranges, 1024 at a time,
// and writes the slice's records and list itself; one launch where the form
// above takes three.  The counts of a step's warps are double-buffered, so a
// step has one barrier.
constexpr int kSelThreads = 1024;
__global__ void __launch_bounds__(kSelThreads) slice_select_kernel(
    const QueryPrep *__restrict__ qp, const uint32_t *__restrict__ range, int64_t M, int k0, float apix,
    int d, float l2tau, Rec *__restrict__ rec, uint32_t *__restrict__ sel, uint32_t *__restrict__ nsel) {
  __shared__ uint32_t wn[2][kSelThreads / 32];
  const int64_t k = blockIdx.x;
  const unsigned z = (unsigned)(k0 + k);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t before = 0;  // of the earlier steps
  int buf = 0;
  unsigned next = threadIdx.x < M ? range[threadIdx.x] : 1u;  // 1: no slice
  for (int64_t j0 = 0; j0 < M; j0 += kSelThreads, buf ^= 1) {
    const int64_t j = j0 + threadIdx.x;
    const unsigned r = next;
    next = j + kSelThreads < M ? range[j + kSelThreads] : 1u;
    const bool in = (r & 0xffffu) <= z && z <= (r >> 16);
    const unsigned bits = __ballot_sync(0xffffffffu, in);
    if (lane == 0) wn[buf][warp] = __popc(bits);
    __syncthreads();
    const uint32_t mine = wn[buf][lane];
    const uint32_t lower = __reduce_add_sync(0xffffffffu, lane < warp ? mine : 0u);
    if (in) {
      sel[k * M + before + lower + __popc(bits & ((1u << lane) - 1u))] = (uint32_t)j;
      rec[k * M + j] = slice_record(qp[j], (int)z, apix, d, l2tau);
    }
    before += __reduce_add_sync(0xffffffffu, mine);
  }
  if (threadIdx.x == 0) nsel[k] = before;
}

cudaError_t launch_query_prep(const float *params, int64_t M, int norm_mode, int shape, float apix,
                              int d, float l2tau, QueryPrep *qp, uint32_t *range, cudaStream_t st) {
  query_prep_kernel<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(params, M, norm_mode, shape, apix, d,
                                                                 l2tau, qp, range);
  return cudaGetLastError();
}

// Where a record of every Gaussian in every slice and the lists of those that
// can matter meet: us per batch, all and lists, of M Gaussians and n slices.
// d 256: M 16000, n 8: 40, 50; M 20000, n 16: 49, 56; M 50000, n 4: 45, 50, n 8:
// 52, 51; M 100000, n 4: 52, 51, n 8: 66, 58; M 300000, n 1: 54, 59, n 2: 66, 62.
// d 64: M 20000, n 16: 51, 62; M 50000, n 8: 54, 58; M 100000, n 8: 78, 72.
bool slices_all(int64_t M, int nslice) { return M * nslice <= 400000; }

cudaError_t launch_slices_all(const QueryPrep *qp, int64_t M, int k0, int nslice, float apix, int d,
                              float l2tau, Rec *rec, cudaStream_t st) {
  const dim3 grid((unsigned)((M + 255) / 256), (unsigned)nslice);
  slice_all_kernel<<<grid, 256, 0, st>>>(qp, M, k0, apix, d, l2tau, rec);
  return cudaGetLastError();
}

cudaError_t launch_slices(const QueryPrep *qp, const uint32_t *range, int64_t M, int k0, int nslice,
                          float apix, int d, float l2tau, uint32_t *cnt, Rec *rec, uint32_t *sel,
                          uint32_t *nsel, cudaStream_t st) {
  // Where the two forms meet: us per query of 16384 and 16385 Gaussians, 319
  // and 327 at d 256 and 64 slices per batch, 289 and 299 at d 192 and 50, 258
  // and 255 at d 64 and 16 (launches are most of it); at 4351 Gaussians, d
  // 192, 50 slices, one launch 228 and three 279.
  if (M <= 16384) {
    slice_select_kernel<<<nslice, kSelThreads, 0, st>>>(qp, range, M, k0, apix, d, l2tau, rec, sel, nsel);
    return cudaGetLastError();
  }
  const int nch = (int)bin_chunks_tiles(M);
  const size_t smem = (size_t)nslice * 8 * sizeof(uint32_t);  // at most 24 KB (768 slices)
  slice_count_kernel<<<nch, kChunkT, smem, st>>>(range, M, k0, nslice, cnt);
  const cudaError_t e = launch_scan_cols(cnt, nch, nslice, 1, nullptr, nsel, st);
  if (e != cudaSuccess) return e;
  slice_write_kernel<<<nch, kChunkT, smem, st>>>(qp, range, M, k0, nslice, apix, d, l2tau, cnt, rec,
                                                 sel);
  return cudaGetLastError();
}

}  // namespace gem
