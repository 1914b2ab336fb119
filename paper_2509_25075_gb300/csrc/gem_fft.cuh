// Radix-4/3/2 Stockham FFT of lines held in shared memory, for the fixed set
// of image sides n = 2^a 3^b (multiples of 16 up to 768), shared by the CTF
// step and the Fourier shell correlation.  tw[m] = e^{-2 pi i m / n}.
//
// A line goes through its stages two at a time: a thread holds R1 R2 elements
// in registers, does R2 butterflies of radix R1 and R1 of radix R2, and
// touches shared memory once per pass, not once per stage.  Every side is a
// template parameter, so strides, divisions and twiddle steps are constants.
// The first pass of a transform can read its elements from global memory and
// the last one write there, which leaves one or two round trips through
// shared memory where a pass per stage made four or five, besides a copy in
// and a copy out.  Passes from shared to shared memory run in place: every
// thread has read its elements before the first is written.
#pragma once

#include "gem_internal.cuh"

namespace gem {

// The fused halves are named, so that every instance rounds alike.
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}

template <int R>
__device__ __forceinline__ void butterfly(float2 (&v)[R]) {
  if constexpr (R == 4) {
    float2 a0 = make_float2(v[0].x + v[2].x, v[0].y + v[2].y);
    float2 a1 = make_float2(v[0].x - v[2].x, v[0].y - v[2].y);
    float2 a2 = make_float2(v[1].x + v[3].x, v[1].y + v[3].y);
    float2 a3 = make_float2(v[1].y - v[3].y, v[3].x - v[1].x);  // (v1 - v3) (-i)
    v[0] = make_float2(a0.x + a2.x, a0.y + a2.y);
    v[2] = make_float2(a0.x - a2.x, a0.y - a2.y);
    v[1] = make_float2(a1.x + a3.x, a1.y + a3.y);
    v[3] = make_float2(a1.x - a3.x, a1.y - a3.y);
  } else if constexpr (R == 2) {
    float2 a0 = v[0];
    v[0] = make_float2(a0.x + v[1].x, a0.y + v[1].y);
    v[1] = make_float2(a0.x - v[1].x, a0.y - v[1].y);
  } else if constexpr (R == 3) {
    const float h = 0.8660254037844386f;  // sqrt(3)/2
    float2 t1 = make_float2(v[1].x + v[2].x, v[1].y + v[2].y);
    float2 t2 = make_float2(v[0].x - 0.5f * t1.x, v[0].y - 0.5f * t1.y);
    float2 t3 = make_float2(h * (v[1].y - v[2].y), -h * (v[1].x - v[2].x));
    v[0] = make_float2(v[0].x + t1.x, v[0].y + t1.y);
    v[1] = make_float2(t2.x + t3.x, t2.y + t3.y);
    v[2] = make_float2(t2.x - t3.x, t2.y - t3.y);
  }
}

// Stages of every side, in order, grouped into passes (R2 = 1: one stage).
template <int R1, int R2>
struct FftPass {
  static constexpr int r1 = R1, r2 = R2;
};
template <class... P>
struct FftPasses {};
template <int N>
struct FftDef;
#define GEM_FFT_DEF(N, ...) \
  template <>               \
  struct FftDef<N> {        \
    using passes = FftPasses<__VA_ARGS__>; \
  }
using P33 = FftPass<3, 3>;
using P34 = FftPass<3, 4>;
using P44 = FftPass<4, 4>;
using P42 = FftPass<4, 2>;
using P4 = FftPass<4, 1>;
using P2 = FftPass<2, 1>;
GEM_FFT_DEF(16, P44);
GEM_FFT_DEF(32, P44, P2);
GEM_FFT_DEF(48, P34, P4);
GEM_FFT_DEF(64, P44, P4);
GEM_FFT_DEF(96, P34, P42);
GEM_FFT_DEF(128, P44, P42);
GEM_FFT_DEF(144, P33, P44);
GEM_FFT_DEF(192, P34, P44);
GEM_FFT_DEF(256, P44, P44);
GEM_FFT_DEF(288, P33, P4, P42);
GEM_FFT_DEF(384, P34, P4, P42);
GEM_FFT_DEF(432, P33, P34, P4);
GEM_FFT_DEF(512, P44, P4, P42);
GEM_FFT_DEF(576, P33, P44, P4);
GEM_FFT_DEF(768, P34, P44, P4);
#undef GEM_FFT_DEF

// Calls f(std::integral_constant<int, d>) for the supported side d.
#define GEM_FFT_SIDES(X) \
  X(16) X(32) X(48) X(64) X(96) X(128) X(144) X(192) X(256) X(288) X(384) X(432) X(512) X(576) X(768)

// Place of element i of a line, and the lines' stride: one element of padding
// every 16, so that the strided stores of a pass and the column-wise accesses
// (element k of neighbouring lines) spread over the banks.
__host__ __device__ constexpr int fft_at(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int fft_stride(int n) { return (n + n / 16) | 1; }

// Stages R1 then R2 of one group: element i of v is the line's element
// base + i N / (R1 R2); afterwards v[r R2 + s] is element
// (base / NS) NS R1 R2 + base % NS + (r + R1 s) NS.
template <int N, int NS, int R1, int R2>
__device__ __forceinline__ void fft_group(float2 (&v)[R1 * R2], int base,
                                          const float2 *__restrict__ tw) {
  constexpr int kT1 = N / (NS * R1), kT2 = N / (NS * R1 * R2);
  const int k = NS == 1 ? 0 : base % NS;
  {
    float2 w[R1];
    if (NS > 1) {
#pragma unroll
      for (int r = 1; r < R1; ++r) w[r] = tw[r * k * kT1];
    }
#pragma unroll
    for (int s = 0; s < R2; ++s) {
      float2 u[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) u[r] = NS > 1 && r > 0 ? cmul(v[r * R2 + s], w[r]) : v[r * R2 + s];
      butterfly<R1>(u);
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r * R2 + s] = u[r];
    }
  }
  if constexpr (R2 > 1) {
#pragma unroll
    for (int r = 0; r < R1; ++r) {
      const int k2 = r * NS + k;
      float2 u[R2];
#pragma unroll
      for (int s = 0; s < R2; ++s)
        u[s] = s > 0 && !(NS == 1 && r == 0) ? cmul(v[r * R2 + s], tw[s * k2 * kT2]) : v[r * R2 + s];
      butterfly<R2>(u);
#pragma unroll
      for (int s = 0; s < R2; ++s) v[r * R2 + s] = u[s];
    }
  }
}

// One pass over L lines by T threads.  kInS, kOutS: the elements come from,
// go to the line buffer sm (else ld(line, i) gives an element and
// st(line, i, v) takes one).  kLineFast: neighbouring threads take
// neighbouring lines, else neighbouring elements of a line.
template <int N, int L, int T, int NS, int R1, int R2, bool kInS, bool kOutS, bool kLineFast, class LD,
          class ST>
__device__ __forceinline__ void fft_pass(LD &ld, ST &st, float2 *sm, const float2 *__restrict__ tw) {
  constexpr int G = R1 * R2, NB = N / G, LS = fft_stride(N);
  constexpr int kIter = (L * NB + T - 1) / T;
  auto place = [&](int g, int &line, int &base) {
    if (kLineFast) {
      line = g % L;
      base = g / L;
    } else {
      line = g / NB;
      base = g - line * NB;
    }
  };
  auto load = [&](float2(&v)[G], int line, int base) {
#pragma unroll
    for (int i = 0; i < G; ++i)
      v[i] = kInS ? sm[line * LS + fft_at(base + i * NB)] : ld(line, base + i * NB);
    fft_group<N, NS, R1, R2>(v, base, tw);
  };
  auto store = [&](const float2(&v)[G], int line, int base) {
    const int o = NS == 1 ? base * G : base / NS * (NS * G) + base % NS;
#pragma unroll
    for (int r = 0; r < R1; ++r)
#pragma unroll
      for (int s = 0; s < R2; ++s) {
        const int i = o + (r + R1 * s) * NS;
        if (kOutS)
          sm[line * LS + fft_at(i)] = v[r * R2 + s];
        else
          st(line, i, v[r * R2 + s]);
      }
  };
  if (kInS && kOutS) {  // in place: all is read before the first is written
    float2 v[kIter][G];
#pragma unroll
    for (int it = 0; it < kIter; ++it) {
      const int g = it * T + threadIdx.x;
      int line, base;
      place(g, line, base);
      if (L * NB % T == 0 || g < L * NB) load(v[it], line, base);
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kIter; ++it) {
      const int g = it * T + threadIdx.x;
      int line, base;
      place(g, line, base);
      if (L * NB % T == 0 || g < L * NB) store(v[it], line, base);
    }
  } else {
#pragma unroll 1
    for (int g = threadIdx.x; g < L * NB; g += T) {
      int line, base;
      place(g, line, base);
      float2 v[G];
      load(v, line, base);
      store(v, line, base);
    }
  }
  if (kOutS) __syncthreads();
}

template <int N, int L, int T, bool kInS, bool kOutS, bool kInLineFast, bool kOutLineFast, int NS,
          bool kFirst, class LD, class ST, class P, class... Rest>
__device__ __forceinline__ void fft_run(FftPasses<P, Rest...>, LD &ld, ST &st, float2 *sm,
                                        const float2 *__restrict__ tw) {
  constexpr bool kLast = sizeof...(Rest) == 0;
  fft_pass<N, L, T, NS, P::r1, P::r2, !kFirst || kInS, !kLast || kOutS,
           kFirst ? kInLineFast : (kLast && kOutLineFast)>(ld, st, sm, tw);
  if constexpr (!kLast)
    fft_run<N, L, T, kInS, kOutS, kInLineFast, kOutLineFast, NS * P::r1 * P::r2, false>(
        FftPasses<Rest...>{}, ld, st, sm, tw);
}

// Forward (e^{-2 pi i}) FFT of L lines of length N by the CTA's T threads.
// kInS: the lines lie in sm already (element i of line l at
// l fft_stride(N) + fft_at(i)), else ld gives them; kOutS: they stay there
// (with a barrier at the end), else st takes them.  A one-pass transform
// (N = 16) between ld and st uses no shared memory.
template <int N, int L, int T, bool kInS, bool kOutS, bool kInLineFast, bool kOutLineFast, class LD,
          class ST>
__device__ __forceinline__ void fft_lines(LD ld, ST st, float2 *sm, const float2 *__restrict__ tw) {
  fft_run<N, L, T, kInS, kOutS, kInLineFast, kOutLineFast, 1, true>(typename FftDef<N>::passes{}, ld,
                                                                    st, sm, tw);
}

struct FftNone {
  __device__ float2 operator()(int, int) const { return make_float2(0.f, 0.f); }
  __device__ void operator()(int, int, float2) const {}
};

template <int N, int T>
__device__ __forceinline__ void load_twiddles(float2 *tw_s, const float2 *__restrict__ tw) {
  for (int i = threadIdx.x; i < N; i += T) tw_s[i] = tw[i];
}

}  // namespace gem
