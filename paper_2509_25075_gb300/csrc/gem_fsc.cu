// Fourier shell correlation of two maps (Eq. fsc; Sec. 4, Gold-Standard
// Fourier Shell Correlation) and its threshold crossing.
//
//   FSC(r_i) = sum_{k in shell i} F1(k) F2(k)^* /
//              sqrt(sum |F1(k)|^2 . sum |F2(k)|^2),
//
// shell i holding the frequencies with round(|k|) = i (k in signed DFT
// indices, shells 0 .. d/2).  Both real maps ride in one complex volume
// z = X1 + i X2; after the 3D DFT, F1(k) = (Z(k) + Z(-k)^*) / 2 and
// F2(k) = (Z(k) - Z(-k)^*) / (2i).  The 3D DFT is three passes of line FFTs
// in shared memory, each along the contiguous axis, each writing its output
// with the axes rotated so the next axis becomes contiguous:
//   [z][y][x] -> [kx][z][y] -> [ky][kx][z] -> [kz][ky][kx].
// Each pass reads and writes the volume once; its stages meet shared memory
// once or twice (gem_fft.cuh).  Same bits as a round trip per stage: two
// 256^3 maps 664 -> 293 us, the shell sums as they were.
#include <math.h>

#include <algorithm>

#include "gem_fft.cuh"
#include "gem_internal.cuh"
#include "gem_pairsum.cuh"

namespace gem {

constexpr int kFThreads = 256;
// Most blocks of the shell sums: 8 per SM on 152 SMs (as many as fit up to side
// 256; beyond, where shared memory lets 7 down to 2 in, they run in turns).
constexpr int kShellBlocks = 1216;
// Lines per CTA of the transform passes: 16 (their transposed stores then
// fill 128-byte lines) up to sides whose 16 lines leave room for four CTAs
// per SM, else 8.
__host__ __device__ constexpr int fsc_lines(int d) { return d <= 384 ? 16 : 8; }

template <int N>
struct FscSmem {
  float2 lines[fsc_lines(N) * fft_stride(N)];
  float2 tw[N];
};

// x pass: rows y0 .. y0 + L - 1 of slab z of z = X1 + i X2, FFT along x,
// written as A[kx][z][y].
template <int N>
__global__ void __launch_bounds__(kFThreads) fsc_pass_real_kernel(
    const float *__restrict__ X1, const float *__restrict__ X2, const float2 *__restrict__ tw,
    float2 *__restrict__ A) {
  constexpr int L = fsc_lines(N);
  extern __shared__ __align__(16) unsigned char fsc_sm[];
  FscSmem<N> &S = *reinterpret_cast<FscSmem<N> *>(fsc_sm);
  const int y0 = blockIdx.x * L, z = blockIdx.y;
  load_twiddles<N, kFThreads>(S.tw, tw);
  __syncthreads();
  const int64_t base = ((int64_t)z * N + y0) * N;
  const float *x1 = X1 + base, *x2 = X2 + base;
  float2 *out = A + (int64_t)z * N + y0;
  fft_lines<N, L, kFThreads, false, false, false, true>(
      [&](int l, int x) { return make_float2(x1[l * N + x], x2[l * N + x]); },
      [&](int l, int k, float2 v) { out[k * (N * N) + l] = v; }, S.lines, S.tw);
}

// Complex pass: B[k][i0][i1] = FFT along i2 of A[i0][i1][:], lines
// i1 = i1_0 .. i1_0 + L - 1 of slab i0.
template <int N>
__global__ void __launch_bounds__(kFThreads) fsc_pass_cplx_kernel(const float2 *__restrict__ A,
                                                                  const float2 *__restrict__ tw,
                                                                  float2 *__restrict__ Bo) {
  constexpr int L = fsc_lines(N);
  extern __shared__ __align__(16) unsigned char fsc_sm[];
  FscSmem<N> &S = *reinterpret_cast<FscSmem<N> *>(fsc_sm);
  const int i10 = blockIdx.x * L, i0 = blockIdx.y;
  load_twiddles<N, kFThreads>(S.tw, tw);
  __syncthreads();
  const float2 *in = A + ((int64_t)i0 * N + i10) * N;
  float2 *out = Bo + (int64_t)i0 * N + i10;
  fft_lines<N, L, kFThreads, false, false, false, true>(
      [&](int l, int x) { return in[l * N + x]; },
      [&](int l, int k, float2 v) { out[k * (N * N) + l] = v; }, S.lines, S.tw);
}

// Shell of a frequency with squared norm k2: the integer s with
// (s - 1/2)^2 <= k2 < (s + 1/2)^2.  No k2 comes closer to a boundary than
// s^2 - s, whose root lies 1 / (8 s) below it: 3.2e-4 at s = 385, the last
// shell of the largest side, against 4.6e-5 of the root (2^-23 of it) and
// 1.5e-5 of the sum.
__device__ __forceinline__ int shell_of(int k2) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"((float)k2));
  return (int)(r + 0.5f);
}

// One step of an inclusive sum over the run of equal keys ending at each lane:
// add the value o lanes below where that lane belongs to the run.
__device__ __forceinline__ float seg_add(float v, int o, bool take) {
  const float u = __shfl_up_sync(0xffffffffu, v, o);
  return take ? v + u : v;
}

// CTAs of the shell sums that an SM's shared memory holds, at most 8.
__host__ __device__ constexpr int shell_ctas(int n) {
  const int fit = 228 * 1024 / (9 * 3 * (n / 2 + 1) * (int)sizeof(double) + 1024);
  return fit < 8 ? fit : 8;
}
// Rows of a unit of the shell sums.
__host__ __device__ constexpr int shell_rows(int n) { return n % 32 ? 2 : 1; }

// Per-block sums over the shells 0 .. nsh-1 of Re(F1 F2^*), |F1|^2, |F2|^2,
// written to part[blk][3][nsh].  A warp takes 32 consecutive frequencies;
// neighbouring frequencies mostly share a shell, so each run of equal shells
// (at most 32 terms) is summed in float32 by a segmented warp scan and added
// once to the warp's own sums in shared memory.  Within half a row the shell
// is monotone, so the runs of one step have different shells and the sums
// need no atomics.
//
// A sum is a pair of floats, its value and the sum of that value's rounding
// errors, added to without loss (gem_pairsum.cuh) and converted to float64
// when the block is done: this GPU's float64 adds run at a 64th of its float32
// adds, and three of them and their conversions per step were the kernel's
// bound.  What the pair cannot hold (terms more than 48 bits apart, which is
// rare), and runs of 1e30 and more, infinities and NaN, go to float64 sums of
// their own, so nothing is rounded but the float64 additions there and at the
// block's end: fewer than with float64 sums throughout.
//
// Then the instructions bound it, and after them the load: the part of the
// volume inside the last shell (half of it), once.  A unit is the least whole
// number q of rows that 32 divides (two rows on sides like 48 or 432, else
// one), so a warp works out row numbers once per unit, and steps beyond the
// last shell load and sum nothing.  The warp follows a unit with its mirror
// image, which then finds both its operands in L1.  Against one pass over all
// frequencies with divisions, two loads each and float64 atomics: side 256,
// the whole call 293 -> 220 us (287 with float64 sums).  Where a step lies in
// one half of a row (sides that 64 divides), as few registers as leave room
// for the CTAs that the shared memory holds: side 256, 226 -> 220 us.
template <int N>
__global__ void __launch_bounds__(kFThreads, N % 64 == 0 ? shell_ctas(N) : 1)
    fsc_shell_kernel(const float2 *__restrict__ F, int nsh, double *__restrict__ part) {
  constexpr int q = shell_rows(N), h = N / 2, kUnits = N / q;  // units per plane
  static_assert(q * N % 32 == 0, "a unit is whole warps");
  constexpr int kWarps = kFThreads / 32;
  extern __shared__ double big[];  // [3][nsh], then the warps' pairs [kWarps][3][nsh]
  float2 *acc = reinterpret_cast<float2 *>(big + 3 * nsh);
  for (int i = threadIdx.x; i < 3 * nsh; i += kFThreads) big[i] = 0.0;
  for (int i = threadIdx.x; i < kWarps * 3 * nsh; i += kFThreads) acc[i] = make_float2(0.f, 0.f);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2 *mine = acc + warp * 3 * nsh;
  auto add = [&](int s, float num, float p1, float p2) {
    if (p1 < 1e30f && p2 < 1e30f) {  // then |num| is as well
      float2 a = mine[s], b = mine[nsh + s], c = mine[2 * nsh + s];
      num = pair_add(a.x, a.y, num);
      p1 = pair_add(b.x, b.y, p1);
      p2 = pair_add(c.x, c.y, p2);
      mine[s] = a;
      mine[nsh + s] = b;
      mine[2 * nsh + s] = c;
      if (num == 0.f && p1 == 0.f && p2 == 0.f) return;
    }
    atomicAdd(&big[s], (double)num);
    atomicAdd(&big[nsh + s], (double)p1);
    atomicAdd(&big[2 * nsh + s], (double)p2);
  };
  const int lim = nsh * nsh - nsh + 1;  // the last shell is nsh - 1: k2 < lim
  const int nunit = (h + 1) * kUnits, step = gridDim.x * kWarps;
  for (int u2 = 2 * (blockIdx.x * kWarps + warp); u2 < 2 * nunit; u2 += (u2 & 1) ? 2 * step - 1 : 1) {
    int kz = (u2 >> 1) / kUnits, j = (u2 >> 1) - kz * kUnits;
    if (u2 & 1) {  // the mirror image; a plane that is its own is done already
      if (kz == 0 || kz == h) continue;
      kz = N - kz;
      j = j ? kUnits - j : 0;
    }
    const int sz = kz < h ? kz : kz - N, z2 = sz * sz;
    const int mz = kz ? N - kz : 0;
    const int ky0 = j * q;
#pragma unroll 2
    for (int i0 = 0; i0 < q * N; i0 += 32) {
      const int e = i0 + lane, r = q > 1 && e >= N ? 1 : 0;
      const int kx = e - r * N, ky = ky0 + r;
      const int sx = kx < h ? kx : kx - N, sy = ky < h ? ky : ky - N;
      const int k2 = sx * sx + sy * sy + z2;
      const bool in = k2 < lim;
      if (!__any_sync(0xffffffffu, in)) continue;
      int s = nsh;  // out of range: contributes nothing
      float num = 0.f, p1 = 0.f, p2 = 0.f;
      if (in) {
        s = shell_of(k2);
        const int mx = kx ? N - kx : 0, my = ky ? N - ky : 0;
        const float2 Z = F[(kz * N + ky) * N + kx];
        const float2 Zm = F[(mz * N + my) * N + mx];
        const float f1r = 0.5f * (Z.x + Zm.x), f1i = 0.5f * (Z.y - Zm.y);
        const float f2r = 0.5f * (Z.y + Zm.y), f2i = -0.5f * (Z.x - Zm.x);
        num = fmaf(f1r, f2r, f1i * f2i);
        p1 = fmaf(f1r, f1r, f1i * f1i);
        p2 = fmaf(f2r, f2r, f2i * f2i);
      }
      const int prev = __shfl_up_sync(0xffffffffu, s, 1);
      // bit l of m: lanes l - o .. l share a run
      unsigned m = __ballot_sync(0xffffffffu, lane > 0 && prev == s);
      const bool last = lane == 31 || !(m >> (lane + 1) & 1u);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        if (!m) break;
        const bool take = m >> lane & 1u;
        num = seg_add(num, o, take);
        p1 = seg_add(p1, o, take);
        p2 = seg_add(p2, o, take);
        m &= m << o;
      }
      const bool write = last && s < nsh;
      if (h % 32 == 0 || i0 / h == (i0 + 31) / h) {
        if (write) add(s, num, p1, p2);
      } else {  // rows' halves meet here: one half's runs at a time
#pragma unroll
        for (int g = 0; g <= 31 / h + 1; ++g) {
          if (write && e / h == i0 / h + g) add(s, num, p1, p2);
          __syncwarp();
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 3 * nsh; i += kFThreads) {
    double t = big[i];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float2 a = acc[w * 3 * nsh + i];
      t += (double)a.x + (double)a.y;
    }
    part[(size_t)blockIdx.x * 3 * nsh + i] = t;
  }
}

// One block per shell: the block sums in a fixed order.
__global__ void __launch_bounds__(256) fsc_fold_kernel(const double *__restrict__ part, int nblk,
                                                       int nsh, double *__restrict__ tot) {
  const int s = blockIdx.x;
  double a = 0, b = 0, c = 0;
  for (int k = threadIdx.x; k < nblk; k += blockDim.x) {
    const double *p = part + (int64_t)k * 3 * nsh;
    a += p[s];
    b += p[nsh + s];
    c += p[2 * nsh + s];
  }
  __shared__ double red[3][256];
  red[0][threadIdx.x] = a;
  red[1][threadIdx.x] = b;
  red[2][threadIdx.x] = c;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int q = 0; q < 3; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 3) tot[threadIdx.x * nsh + s] = red[threadIdx.x][0];
}

// FSC per shell from the folded sums, and the threshold crossing: the first
// shell i >= 1 with FSC < thr, interpolated linearly between shells i-1 and
// i; resolution = d apix / k* (Angstrom).  No crossing: the Nyquist shell
// d/2 (resolution 2 apix).
__global__ void __launch_bounds__(512) fsc_final_kernel(const double *__restrict__ tot, int nsh,
                                                        int d, float apix, float thr,
                                                        double *__restrict__ fsc,
                                                        double *__restrict__ sums,
                                                        double *__restrict__ resolution) {
  extern __shared__ double f[];  // [nsh]
  __shared__ int first;          // the first shell below the threshold
  if (threadIdx.x == 0) first = nsh;
  for (int s = threadIdx.x; s < nsh; s += blockDim.x) {
    const double a = tot[s], b = tot[nsh + s], c = tot[2 * nsh + s];
    const double den = sqrt(b * c);
    f[s] = den > 0.0 ? a / den : 0.0;
    fsc[s] = f[s];
    if (sums) {
      sums[s] = a;
      sums[nsh + s] = b;
      sums[2 * nsh + s] = c;
    }
  }
  __syncthreads();
  if (!resolution) return;
  for (int s = 1 + threadIdx.x; s < nsh; s += blockDim.x)
    if (f[s] < thr) atomicMin(&first, s);
  __syncthreads();
  if (threadIdx.x == 0) {
    double kstar = (double)(nsh - 1);
    if (first < nsh) {
      const double a = f[first - 1], b = f[first];
      const double frac = a > b ? (a - thr) / (a - b) : 0.0;
      kstar = (first - 1) + fmin(fmax(frac, 0.0), 1.0);
    }
    resolution[0] = kstar > 0.0 ? (double)d * apix / kstar : INFINITY;
  }
}

static int shell_smem(int nsh) { return (kFThreads / 32 + 1) * 3 * nsh * (int)sizeof(double); }

template <int N>
static cudaError_t fsc_configure_side() {
  const int smem = (int)sizeof(FscSmem<N>);
  cudaError_t e = cudaFuncSetAttribute(fsc_pass_real_kernel<N>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fsc_shell_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             shell_smem(N / 2 + 1));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fsc_pass_cplx_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              smem);
}

cudaError_t fsc_configure(int d) {
  switch (d) {
#define X(N) \
  case N:    \
    return fsc_configure_side<N>();
    GEM_FFT_SIDES(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

// A block for every eight units of the half volume: beyond that (sides up to
// 128) blocks would only clear, write and fold empty sums.
static int shell_blocks(int d) {
  constexpr int kWarps = kFThreads / 32;
  return std::min(kShellBlocks, ((d / 2 + 1) * (d / shell_rows(d)) + kWarps - 1) / kWarps);
}

template <int N>
static void launch_fsc_passes(const float2 *tw, const float *X1, const float *X2, float2 *P, float2 *Q,
                              double *part, cudaStream_t st) {
  const size_t smem = sizeof(FscSmem<N>);
  const dim3 g(N / fsc_lines(N), N);
  fsc_pass_real_kernel<N><<<g, kFThreads, smem, st>>>(X1, X2, tw, P);
  fsc_pass_cplx_kernel<N><<<g, kFThreads, smem, st>>>(P, tw, Q);
  fsc_pass_cplx_kernel<N><<<g, kFThreads, smem, st>>>(Q, tw, P);
  const int nsh = N / 2 + 1;
  fsc_shell_kernel<N><<<shell_blocks(N), kFThreads, shell_smem(nsh), st>>>(P, nsh, part);
}

// block partials, then the folded sums
int fsc_partial_count(int d) { return (kShellBlocks + 1) * 3 * (d / 2 + 1); }

cudaError_t launch_fsc(int d, float apix, float thr, const float2 *tw, const float *X1,
                       const float *X2, float2 *P, float2 *Q, double *part, double *fsc,
                       double *sums, double *resolution, cudaStream_t st) {
  switch (d) {
#define X(N)                                          \
  case N:                                             \
    launch_fsc_passes<N>(tw, X1, X2, P, Q, part, st); \
    break;
    GEM_FFT_SIDES(X)
#undef X
    default:
      return cudaErrorInvalidValue;
  }
  const int nsh = d / 2 + 1;
  double *tot = part + (size_t)kShellBlocks * 3 * nsh;
  fsc_fold_kernel<<<nsh, 256, 0, st>>>(part, shell_blocks(d), nsh, tot);
  fsc_final_kernel<<<1, 512, nsh * sizeof(double), st>>>(tot, nsh, d, apix, thr, fsc, sums,
                                                         resolution);
  return cudaGetLastError();
}

}  // namespace gem
