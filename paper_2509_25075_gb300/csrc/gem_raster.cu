// Steps a3 (raster forward) and a5 (raster backward) of the GEM hot path,
// plus the plain dense forms used as the baseline.
//
// A tile's list is in ascending depth and carries, per entry, the mask of
// the 4x4 pixel blocks the Gaussian's region above tau meets (computed once
// by the binning).  A Gaussian therefore costs 16 pixel evaluations per block
// it touches, instead of 256 per tile.  Pixels are evaluated in whitened
// coordinates (Rec): the exponent is l2A - (u11 dx + u12 dy)^2 - (u22 dy)^2.
//
// a3: Eq. render restricted by Eq. accu.  The lists are cut into segments of
//     at most 512 entries, taken from a counter by persistent CTAs of 128
//     threads, which walk them in windows of 256 entries (only the 24 bytes
//     that the evaluation reads are staged).  A window's (block, record) items
//     are laid out block after block, each block's records in list order, and
//     each block gets a share of the threads in proportion to its items.  A
//     thread evaluates the 16 pixels of its block for each of its items
//     (packed float pairs); each pixel sums its block's partial images in
//     thread order, and windows join with Kahan compensation in list order.
//     The result is deterministic and follows the list's depth order window by
//     window.
// a5: the "efficient gradient" of Sec. 1 (iii) / Sec. 3.2: only pairs kept by
//     Eq. accu.  Each warp takes up to 256 entries of a segment, sorts them by
//     block count and first block and runs them in rounds of 32 records, one
//     lane per record: the lanes walk the record's blocks and accumulate
//     six moments of w = g * value in the record's whitened coordinates
//     (rows in packed float pairs: the sums of w, w z1, w z1^2, weighted by
//     z2).  The second moments are taken about the whitened S^, c^2 I:
//     for a wide Gaussian under a smooth upstream gradient the conic and
//     amplitude terms of dL/dS^ nearly cancel, and this form lets that
//     cancellation happen inside an accurate sum instead of in the float32
//     chain rule.  Each block's sums join the lane's totals, and the (tile,
//     Gaussian) partial goes to float64 moments in global memory (L2
//     atomics), so the sum over a Gaussian's tiles loses nothing to
//     rounding.  No barrier couples the warps.  a6 turns the moments into
//     parameter gradients.
#include "gem_internal.cuh"

namespace gem {

constexpr int kThreads = 128;

// (sum, compensation) + x, Kahan; the compensated value is sum - compensation.
__device__ __forceinline__ float2 kahan_add(float2 s, float x) {
  const float y = x - s.y;
  const float t = s.x + y;
  return make_float2(t, (t - s.x) - y);
}
// The 32 x 32 bit matrix whose row r is lane r's x, transposed: lane k gets
// the bits k of all lanes (bit r from lane r), as 32 ballots would give it.
// Five butterfly stages; at distance j the lanes of a pair swap the j-bit
// halves of their 2j-bit groups that lie off the diagonal.
__device__ __forceinline__ unsigned warp_transpose32(unsigned x, int lane) {
  const unsigned hi[5] = {0xffff0000u, 0xff00ff00u, 0xf0f0f0f0u, 0xccccccccu, 0xaaaaaaaau};
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int j = 16 >> s;
    const unsigned y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? ((x & hi[s]) | ((y >> j) & ~hi[s])) : ((x & ~hi[s]) | ((y << j) & hi[s]));
  }
  return x;
}


// One record in one 256-bit load: a warp's gather of 32 records then takes
// one pass over the L1 tags, not one for each half.
__device__ __forceinline__ Rec load_rec(const Rec *p) {
  Rec r;
  asm volatile("ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r.a.x), "=f"(r.a.y), "=f"(r.a.z), "=f"(r.a.w), "=f"(r.b.x), "=f"(r.b.y),
                 "=f"(r.b.z), "=f"(r.b.w)
               : "l"(p));
  return r;
}

constexpr int kWin = 256;       // forward: records per window
constexpr int kSegMax = 512;    // entries of the longest segment

// Tasks of the rasterisers.  A tile's list is cut into segments of S entries
// (the last one shorter); a task is one segment, and the warps that take it
// work on pieces of it, so that nobody walks a long list alone (the longest
// list of a workload holds five to twenty times the mean) and a call with few
// tiles still fills the SMs.  S is a multiple of the forward's window: 512,
// or 256 where that would leave resident CTAs without a segment.  Tasks follow
// the tiles' index order up to the order in which the CTAs here claim their
// ranges, so neighbouring tiles, which share records, are in flight together.
// Empty tiles get their zeros here and no task.
__device__ __forceinline__ int64_t segment_length(int64_t total, int slots) {
  const int64_t S = total / (2 * (int64_t)slots);
  return (max((int64_t)1, min((int64_t)kSegMax, S)) + kWin - 1) / kWin * kWin;
}

// A CTA takes kPer tiles, one per thread, and its eight warps share the zeros of
// the empty ones.
template <int kPer>
__global__ void __launch_bounds__(256) raster_tasks_kernel(const int64_t *__restrict__ tile_start,
                                                           int ntiles, int64_t cap, int d, int slots,
                                                           RasterTasks tk, float *__restrict__ proj) {
  __shared__ unsigned wsum[2][8], base_sh[2], empty[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * kPer, i = (int)threadIdx.x < kPer ? i0 + (int)threadIdx.x : ntiles;
  const int64_t total = tile_start[ntiles];
  // lists that overflowed their capacity are incomplete: every list counts
  // as empty (the status word reports it)
  const bool over = total > cap;
  const int64_t S = segment_length(total, slots);
  int64_t s = 0, len = 0;
  if (i < ntiles) {
    s = tile_start[i];
    len = over ? 0 : tile_start[i + 1] - s;
  }
  unsigned nseg = (unsigned)((len + S - 1) / S);
  // exclusive prefixes of the tasks and of the partial images they need (one
  // per window of tiles with several segments)
  const unsigned nwin = (unsigned)((len + kWin - 1) / kWin);
  unsigned inc = nseg, incp = nseg > 1 ? nwin : 0;
  const unsigned mine = incp;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(0xffffffffu, inc, o), v = __shfl_up_sync(0xffffffffu, incp, o);
    if (lane >= o) {
      inc += u;
      incp += v;
    }
  }
  const unsigned none = __ballot_sync(0xffffffffu, i < ntiles && nseg == 0);
  if (lane == 31) {
    wsum[0][warp] = inc;
    wsum[1][warp] = incp;
    empty[warp] = none;
  }
  __syncthreads();
  unsigned at = inc - nseg, part = incp - mine, all = 0, allp = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w < warp) {
      at += wsum[0][w];
      part += wsum[1][w];
    }
    all += wsum[0][w];
    allp += wsum[1][w];
  }
  if (i0 + threadIdx.x == 0) tk.ctr[kCtrSegment] = (unsigned)S;
  if (threadIdx.x == 0) {
    base_sh[0] = atomicAdd(tk.ctr + kCtrTasks, all);
    base_sh[1] = atomicAdd(tk.ctr + kCtrParts, allp);
  }
  __syncthreads();
  at += base_sh[0];
  part += base_sh[1];
  if (nseg > 0) {
    for (unsigned k = 0; k < nseg; ++k) {
      const int64_t a = s + k * S, n = min(S, s + len - a);
      uint4 *t = tk.task + 2 * (int64_t)(at + k);
      t[0] = make_uint4((unsigned)a, (unsigned)((uint64_t)a >> 32), (unsigned)n, (unsigned)i);
      t[1] = make_uint4(k * (unsigned)(S / kWin), nseg, part, nwin);
    }
  }
  if (proj) {
    const int nt = d / kTile, T = nt * nt;
    for (int k = warp; k < kPer; k += 8) {
      if (!(empty[k >> 5] >> (k & 31) & 1u)) continue;
      const int bt = i0 + k;
      const int b = bt / T, t = bt - b * T;
      float *o = proj + ((int64_t)b * d + (t / nt) * kTile) * d + (t % nt) * kTile;
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4 *>(o + (int64_t)(8 * q + (lane >> 2)) * d + 4 * (lane & 3)) =
            make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

// Shared memory of one forward CTA: a window.
struct FwdWin {
  float4 sa[kWin];                // px, py, u11, u12
  float2 sb[kWin];                // u22, log2 A
  float4 part[kThreads][4];       // the threads' partial images of their blocks
  unsigned char flat[16 * kWin];  // slot of each (block, record) item
  unsigned short cnt[4][16];      // per warp: its records that touch each block
  unsigned short pstart[18];      // block k's items: [pstart[k], pstart[k + 1])
  unsigned short tfirst[18];      // block k's threads: [tfirst[k], tfirst[k + 1])
  uint4 desc[2][2];               // this task's descriptor and the next one's
  int last;                       // whether this is the tile's last segment
};
// Row q of thread v's partial image lies at part[v][q ^ swizzle(v)]:
// eight neighbouring lanes then store to different banks.
__device__ __forceinline__ int part_swizzle(int v) { return (v >> 1) & 3; }
constexpr unsigned kNoSum = 0x80000000u;  // -0: a block without items (a sum of values is never -0)

// a3.  A CTA claims a segment from a counter and walks it in windows of 256
// entries, the next window's entries on their way while one is evaluated.
// Its warps stage a quarter of a window's records each; the lanes' packed
// masks, transposed as a bit matrix, leave each lane one of the words that
// say which of 32 records touch a block; the lane lists its word's records, so
// that the window's (block, record) items lie block after block, each
// block's in list order.  The 128 threads share the items: every non-empty
// block gets at least one (thread range [T_k, T_k+1) with T_k = (non-empty
// blocks before k) + floor((128 - non-empty) start_k / N)), and a block's
// threads take its items interleaved.  A thread evaluates 16 pixels per item
// and leaves one partial image of its block; each pixel sums its block's
// partials in thread order.  A pixel's windows join with Kahan compensation
// in list order: in registers where the tile has one segment, else the windows
// go to `part`, and the CTA that finishes the tile's last segment adds them.
// Nothing depends on which CTA did what, so the result is deterministic and
// in depth order window by window.
//
// What bounds it: issue (70% of the slots) and the L1 (66%), through which
// every entry's 32 scattered bytes come and which serves the evaluation.  The
// records of the next window, of this task or the next, wait in registers (one
// 256-bit load each: two loads of 16 and 8 bytes take two passes over the L1
// tags, and asynchronous copies of the same into a second buffer were slower
// than no prefetch: 655 against 575 us at d 384, M 500000, B 16).  Against one
// CTA per tile, the longest lists first, that loaded a window's records when
// it came to them (us per launch; the sums are the same bits): d 384,
// M 500000, B 16: 680 -> 510; d 128, M 20000, B 256: 388 -> 364; d 256,
// M 100000, B 64: 498 -> 428; d 128, M 50000, B 64, scales 0.3-12 px, whose
// longest lists hold 14000 entries against a mean of 3400: 745-850 -> 442;
// d 64, M 2000, B 32: 37 -> 20; d 64, M 1999, B 9, every pair: 71 -> 41.
// Segments of 256, 1024, 2048 entries: 538, 510, 526 at the first, 381, 371,
// 387 at the second.  Two warps per window, 24 on an SM: 592 and 422; one
// warp, 16 on an SM: 606 and 438.
//
// kCount = true: the same walk, counting kept pairs into kept[0] and
// evaluated pairs into kept[1] instead of writing the projection
// (inspection only, never on the timed path).
template <int kMinB, bool kCount>
__global__ void __launch_bounds__(kThreads, kMinB) raster_fwd_kernel(
    const Rec *__restrict__ rec, const uint2 *__restrict__ list, int64_t M, int d, float l2tau,
    RasterTasks tk, int sms, float *__restrict__ proj, unsigned long long *__restrict__ kept) {
  __shared__ FwdWin W;
  const int nt = d / kTile, T = nt * nt;
  const int hw = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float nl2tau = -l2tau;  // kept: -e < -log2(tau)
  const int ntasks = (int)tk.ctr[kCtrTasks];
  unsigned nkept = 0, neval = 0;
  // A CTA's first three tasks are its own, one of each round of the grid, so
  // that no CTA has two before every CTA has one; from there on thread 0 claims
  // a task two ahead and reads its descriptor one ahead.  A round's tasks go to
  // the SMs in turn (every sms-th CTA is on the same one, as a rule), moved on
  // by one per turn: where lists are alike, full segments and short last ones
  // alternate, and would meet on the same SMs.  (Claims from the second task on:
  // a query of 300 Gaussians, side 96, tau 0: 531 us, now 443; a projection of
  // 2000, side 384, one view, tau 0: 1541, now 1499.)  A task with no entries
  // ends the list.
  auto task_at = [&](int q, uint4 &a, uint4 &c) {
    a = c = make_uint4(0u, 0u, 0u, 0u);
    if (q < ntasks) {
      a = tk.task[2 * (int64_t)q];
      c = tk.task[2 * (int64_t)q + 1];
    }
  };
  auto claim = [&]() { return (int)(atomicAdd(tk.ctr + kCtrFwd, 1u) + 3 * gridDim.x); };
  int nq = 0;
  if (threadIdx.x == 0) {
    const int G = (int)gridDim.x, col = (int)blockIdx.x % sms, row = (int)blockIdx.x / sms;
    auto own = [&](int r) { return r * G + row * sms + (col + row + r) % sms; };
    task_at(own(0), W.desc[0][0], W.desc[0][1]);
    task_at(own(1), W.desc[1][0], W.desc[1][1]);
    nq = own(2);
  }
  __syncthreads();
  // this warp's quarter of a window: slots 64 hw .. 64 hw + 63, two per lane.
  // masks: their block masks, packed; an entry whose Gaussian index is out of
  // range (a list position left unwritten when the lists overflowed their
  // capacity) counts as empty.
  const int slot0 = 64 * hw + lane;
  auto entry = [&](const uint4 &a, int w0, int q) {
    const int i = w0 + slot0 + 32 * q;
    const uint2 *L = list + (int64_t)(((uint64_t)a.y << 32) | a.x);
    return i < (int)a.z ? L[i] : make_uint2(0xffffffffu, 0u);
  };
  Rec r0, r1;  // the next window's records, on their way while this one is evaluated
  auto fetch = [&](const uint4 &a, const uint2 &e0, const uint2 &e1) {
    const Rec *rb = rec + (int64_t)((int)a.w / T) * M;
    unsigned m = 0;
    if (e0.x < (uint64_t)M) {
      m = e0.y & 0xffffu;
      r0 = load_rec(rb + e0.x);
    }
    if (e1.x < (uint64_t)M) {
      m |= e1.y << 16;
      r1 = load_rec(rb + e1.x);
    }
    return m;
  };
  // this thread's pixels when it sums: half a row of block ob
  const int id = threadIdx.x, ob = id >> 3, row = (id >> 1) & 3;
  int cd = 0;  // descriptor in use
  unsigned masks = 0;
  {
    const uint4 a = W.desc[0][0];
    masks = fetch(a, entry(a, 0, 0), entry(a, 0, 1));
  }
  while (W.desc[cd][0].z != 0u) {
    const uint4 t0 = W.desc[cd][0];
    const uint4 t1 = W.desc[cd][1];
    const int ntask = (int)t0.z, bt = (int)t0.w;
    const unsigned nseg = t1.y;
    const int b = bt / T, t = bt - b * T;
    const int tx = t % nt, ty = t / nt;
    const int x0 = tx * kTile, y0 = ty * kTile;
    float *o = proj + ((int64_t)b * d + y0) * d + x0;
    float2 *part = reinterpret_cast<float2 *>(tk.part + (int64_t)t1.z * 256);
    float2 run0 = make_float2(0.f, 0.f), run1 = run0;  // Kahan sums over the windows
    for (int w0 = 0; w0 < ntask; w0 += kWin) {
      const bool lastw = w0 + kWin >= ntask;
      // the next window's entries (this task's or the next one's)
      const uint4 na = lastw ? W.desc[cd ^ 1][0] : t0;
      const int nw0 = lastw ? 0 : w0 + kWin;
      const uint2 e0 = entry(na, nw0, 0), e1 = entry(na, nw0, 1);
      // lane (k, h) = k + 16 h: word 2 hw + h of block k (bit l: slot 32 word + l)
      const int h = lane >> 4;
      const unsigned w = warp_transpose32(masks, lane);
      const int c = __popc(w), o2 = __shfl_xor_sync(0xffffffffu, c, 16);
      if (lane < 16) W.cnt[hw][lane] = (unsigned short)(c + o2);
      W.sa[slot0] = r0.a;
      W.sb[slot0] = make_float2(r0.b.x, r0.b.y);
      W.sa[slot0 + 32] = r1.a;
      W.sb[slot0 + 32] = make_float2(r1.b.x, r1.b.y);
      __syncthreads();
      // the blocks' items and threads (every warp, the same numbers)
      int len = 0, before = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q == hw) before = len;
        len += W.cnt[q][lane & 15];
      }
      int incl = len, ne = len > 0 ? 1 : 0;
#pragma unroll
      for (int s = 1; s < 16; s <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, s, 16);
        const int x = __shfl_up_sync(0xffffffffu, ne, s, 16);
        if ((lane & 15) >= s) {
          incl += v;
          ne += x;
        }
      }
      const int N = __shfl_sync(0xffffffffu, incl, 15), nne = __shfl_sync(0xffffffffu, ne, 15);
      const int st = incl - len;
      // floor(a / N) for a = (128 - nne) st < 2^19, N <= 16 kWin: a / N is a
      // multiple of 1 / N, so (a + 1/2) / N sits at least 1 / (2 N) from
      // an integer, far more than the few-ulp error of the fast division
      const float a = (float)((kThreads - nne) * st) + 0.5f;
      if (hw == 0 && lane < 16) {
        W.pstart[lane] = (unsigned short)st;
        W.tfirst[lane] = (unsigned short)(ne - (len > 0 ? 1 : 0) + (N > 0 ? (int)__fdividef(a, (float)N) : 0));
      }
      if (hw == 0 && lane == 15) {
        W.pstart[16] = (unsigned short)N;
        W.tfirst[16] = kThreads;
      }
      // the records of this lane's word
      {
        unsigned char *f = W.flat + st + before + (h ? o2 : 0);
        const int first = 32 * (2 * hw + h);
        for (unsigned m = w; m; m &= m - 1) *f++ = (unsigned char)(first + __ffs(m) - 1);
      }
      __syncthreads();
      masks = fetch(na, e0, e1);
      {
        // this thread's block is the last one whose range starts at or before
        // it (an empty block's range is empty)
        const int vt = threadIdx.x;
        int k = 0;
#pragma unroll
        for (int s = 8; s >= 1; s >>= 1)
          if (W.tfirst[k + s] <= vt) k += s;
        const int th0 = W.tfirst[k], nth = W.tfirst[k + 1] - th0, end = W.pstart[k + 1];
        // acc[4 h + x]: column x, rows 2 h and 2 h + 1
        float2 acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = make_float2(0.f, 0.f);
        const float X0 = (float)(x0 + 4 * (k & 3)), Y0 = (float)(y0 + 4 * (k >> 2));
        const float2 ys0 = make_float2(Y0, Y0 + 1.f), ys1 = make_float2(Y0 + 2.f, Y0 + 3.f);
        for (int i = W.pstart[k] + vt - th0; i < end; i += nth) {
          const int slot = W.flat[i];
          const float4 A = W.sa[slot];
          const float2 Bv = W.sb[slot];
          // -e = z1^2 + (z2^2 - l2A), z1 = u11 dx + u12 dy (u11 dx fused into
          // the sum), z2 = u22 dy, two rows of a column in one packed operation
          float2 dx[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) dx[x] = f2(__fsub_rn(X0 + (float)x, A.x));
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const float2 dy = add2(g ? ys1 : ys0, f2(-A.y));
            const float2 uy = mul2(f2(A.w), dy);
            const float2 z2 = mul2(f2(Bv.x), dy);
            const float2 nc = fma2(z2, z2, f2(-Bv.y));
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              const float2 z = fma2(f2(A.z), dx[x], uy);
              const float2 f = fma2(z, z, nc);
              if (kCount)
                nkept += (f.x < nl2tau) + (f.y < nl2tau);
              else  // value on kept pairs (value > tau), zero elsewhere
                acc[4 * g + x] = fma2(make_float2(ex2_approx(-f.x), ex2_approx(-f.y)),
                                      make_float2(set_lt(f.x, nl2tau), set_lt(f.y, nl2tau)),
                                      acc[4 * g + x]);
            }
          }
          if (kCount) neval += 16;
        }
        const int sw = part_swizzle(vt);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          W.part[vt][(2 * g) ^ sw] = make_float4(acc[4 * g].x, acc[4 * g + 1].x, acc[4 * g + 2].x, acc[4 * g + 3].x);
          W.part[vt][(2 * g + 1) ^ sw] = make_float4(acc[4 * g].y, acc[4 * g + 1].y, acc[4 * g + 2].y, acc[4 * g + 3].y);
        }
      }
      if (lastw && threadIdx.x == 0) {  // every thread has read this task's descriptor
        task_at(nq, W.desc[cd][0], W.desc[cd][1]);
        nq = claim();
      }
      __syncthreads();
      if (kCount) continue;
      // a pixel's partials in thread order
      float2 sum = make_float2(0.f, 0.f);
      const bool own = W.pstart[ob + 1] > W.pstart[ob];
      if (own) {
        const int v1 = W.tfirst[ob + 1];
        for (int v = W.tfirst[ob]; v < v1; ++v) {
          const float2 x = reinterpret_cast<const float2 *>(&W.part[v][row ^ part_swizzle(v)])[id & 1];
          sum.x += x.x;
          sum.y += x.y;
        }
        if (nseg == 1) {
          run0 = kahan_add(run0, sum.x);
          run1 = kahan_add(run1, sum.y);
        }
      } else {
        sum.x = sum.y = __uint_as_float(kNoSum);
      }
      if (nseg > 1) __stcg(part + (int64_t)(t1.x + w0 / kWin) * 128 + id, sum);
    }
    if (!kCount) {
      float2 *out = reinterpret_cast<float2 *>(o + (4 * (ob >> 2) + row) * d + 4 * (ob & 3)) + (id & 1);
      bool write = nseg == 1;
      if (!write) {
        // the tile's last CTA adds its windows
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) W.last = atomicAdd(tk.done + bt, 1u) == nseg - 1;
        __syncthreads();
        write = W.last;
        if (write) {
          __threadfence();
          if (threadIdx.x == 0) tk.done[bt] = 0u;  // as the next call expects it
#pragma unroll 4
          for (unsigned g = 0; g < t1.w; ++g) {
            const float2 x = __ldcg(part + (int64_t)g * 128 + id);
            if (__float_as_uint(x.x) != kNoSum) {
              run0 = kahan_add(run0, x.x);
              run1 = kahan_add(run1, x.y);
            }
          }
        }
      }
      if (write) *out = make_float2(run0.x - run0.y, run1.x - run1.y);
    }
    cd ^= 1;
  }
  if (kCount) {
    for (int o = 16; o > 0; o >>= 1) {
      nkept += __shfl_xor_sync(0xffffffffu, nkept, o);
      neval += __shfl_xor_sync(0xffffffffu, neval, o);
    }
    if (lane == 0) {
      atomicAdd(kept, (unsigned long long)nkept);
      atomicAdd(kept + 1, (unsigned long long)neval);
    }
  }
}

// The forward's kernel configurations (the autotuner's search space).
static const FwdCfg kFwdCfgs[] = {
    {8, "8 CTAs/SM"}, {7, "7 CTAs/SM"}, {6, "6 CTAs/SM"}, {5, "5 CTAs/SM"},
    {4, "4 CTAs/SM"}, {3, "3 CTAs/SM"}, {2, "2 CTAs/SM"}, {1, "1 CTA/SM"},
};
int fwd_config_count() { return (int)(sizeof(kFwdCfgs) / sizeof(kFwdCfgs[0])); }
const FwdCfg &fwd_config(int i) { return kFwdCfgs[i]; }

static int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

size_t raster_task_count(int64_t cap, int64_t ntiles) {
  // one per tile, and one more per full segment
  return (size_t)(ntiles + cap / kWin + 1);
}

template <bool kCount>
static cudaError_t launch_fwd_any(int cfg, const Rec *rec, const uint2 *list,
                                  const int64_t *tile_start, int64_t cap, int64_t M, int B, int d,
                                  float l2tau, float *proj, unsigned long long *kept,
                                  const RasterTasks &tk, bool fresh, cudaStream_t st) {
  if (cfg < 0 || cfg >= fwd_config_count()) return cudaErrorInvalidValue;
  const int nt = d / kTile, ntiles = nt * nt * B, sms = sm_count();
  if (!fresh) {
    const cudaError_t e = cudaMemsetAsync(tk.ctr, 0, kCtrCount * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
  }
  // small calls: fewer tiles per CTA, so that more CTAs share the zeros
  if (ntiles <= 32 * sms)
    raster_tasks_kernel<32><<<(ntiles + 31) / 32, 256, 0, st>>>(tile_start, ntiles, cap, d, sms * 8, tk, proj);
  else
    raster_tasks_kernel<256><<<(ntiles + 255) / 256, 256, 0, st>>>(tile_start, ntiles, cap, d, sms * 8, tk, proj);
  const int grid = sms * kFwdCfgs[cfg].ctas;
  if (kFwdCfgs[cfg].ctas > 7)
    raster_fwd_kernel<8, kCount><<<grid, kThreads, 0, st>>>(rec, list, M, d, l2tau, tk, sms, proj, kept);
  else
    raster_fwd_kernel<7, kCount><<<grid, kThreads, 0, st>>>(rec, list, M, d, l2tau, tk, sms, proj, kept);
  return cudaGetLastError();
}

cudaError_t launch_raster_fwd(int cfg, const Rec *rec, const uint2 *list,
                              const int64_t *tile_start, int64_t cap, int64_t M, int B, int d,
                              float l2tau, float *proj, const RasterTasks &tk, bool fresh,
                              cudaStream_t st) {
  return launch_fwd_any<false>(cfg, rec, list, tile_start, cap, M, B, d, l2tau, proj, nullptr, tk,
                               fresh, st);
}

cudaError_t launch_count_kept(int cfg, const Rec *rec, const uint2 *list,
                              const int64_t *tile_start, int64_t cap, int64_t M, int B, int d,
                              float l2tau, unsigned long long *kept, const RasterTasks &tk,
                              cudaStream_t st) {
  return launch_fwd_any<true>(cfg, rec, list, tile_start, cap, M, B, d, l2tau, nullptr, kept, tk,
                              false, st);
}

// Sum of two packed pairs, rounded on its own: no product that goes into it is
// contracted with it.
__device__ __forceinline__ float2 add2_apart(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "add.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

// The six moments of w = g * value over the 16 pixels of block k of the tile
// at (x0, y0) for one record (centre A.x, A.y, first row of U in A.z, A.w;
// u22, l2A), in the record's whitened coordinates z1 = u11 dx + u12 dy,
// z2 = u22 dy, added to the running totals (n0, n1), (n2, n3), (n4, n5):
//   n0 = sum w, n1 = sum w z1, n2 = sum w z2,
//   n3 = sum w (z1^2 - c^2), n4 = sum w z1 z2, n5 = sum w (z2^2 - c^2).
// Rows are taken two at a time, one per half of a packed pair, so the row
// terms (z2, and what is weighted by it) pack as naturally as the pixels'
// (a sixth fewer instructions than pairs of columns, whose row terms are
// scalars).  A row's sums are (pixel 0 + pixel 2) + (pixel 1 + pixel 3), and
// the rows are added in order: the gradient's bits do not depend on how the
// pixels are packed.  The second moments are taken about c^2 I, the whitened
// S^, per block.  sg is the g tile: [row pair, column][block] = rows 2 h and
// 2 h + 1 of column c, then of column c + 2.
__device__ __forceinline__ void block_moments(const float4 (*__restrict__ sg)[16], int k, int x0,
                                              int y0, const float4 &A, float u22, float l2A,
                                              float nl2tau, float2 (&n)[3]) {
  // the exponent rounded exactly as the forward rounds it, so that both
  // decide Eq. accu alike
  const float X0 = (float)(x0 + 4 * (k & 3)), Y0 = (float)(y0 + 4 * (k >> 2));
  float2 dx[4];
#pragma unroll
  for (int x = 0; x < 4; ++x) dx[x] = f2(__fsub_rn(X0 + (float)x, A.x));
  float m0, m1, m2, m3, m4, m5;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 dy = add2(make_float2(Y0 + (float)(2 * h), Y0 + (float)(2 * h + 1)), f2(-A.y));
    const float2 uy = mul2(f2(A.w), dy);
    const float2 z2 = mul2(f2(u22), dy);
    const float2 nc = fma2(z2, z2, f2(-l2A));
    float2 s0, s1, s2;  // the rows' sums of w, w z1 and w z1^2
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float4 g4 = sg[2 * h + c][k];
      // -e = z1^2 + (z2^2 - l2A), as in the forward's terms
      const float2 za = fma2(f2(A.z), dx[c], uy), zb = fma2(f2(A.z), dx[c + 2], uy);
      const float2 fa = fma2(za, za, nc), fb = fma2(zb, zb, nc);
      // w = g * value on kept pairs (value > tau), zero elsewhere: g is
      // masked to +0 on the integer pipe, which leaves the FMA pipe (this
      // loop's busiest) the multiply
      const float2 ga = make_float2(keep_or_zero(g4.x, fa.x, nl2tau), keep_or_zero(g4.y, fa.y, nl2tau));
      const float2 gb = make_float2(keep_or_zero(g4.z, fb.x, nl2tau), keep_or_zero(g4.w, fb.y, nl2tau));
      const float2 wa = mul2(ga, make_float2(ex2_approx(-fa.x), ex2_approx(-fa.y)));
      const float2 wb = mul2(gb, make_float2(ex2_approx(-fb.x), ex2_approx(-fb.y)));
      const float2 wza = mul2(wa, za), wzb = mul2(wb, zb);
      const float2 p0 = add2_apart(wa, wb), p1 = add2_apart(wza, wzb);
      const float2 p2 = fma2(wzb, zb, mul2(wza, za));
      s0 = c ? add2(s0, p0) : p0;
      s1 = c ? add2(s1, p1) : p1;
      s2 = c ? add2(s2, p2) : p2;
    }
    // weighted by z2, row after row
    const float2 t = mul2(s0, z2);
    m0 = h ? m0 + s0.x : s0.x;
    m1 = h ? m1 + s1.x : s1.x;
    m3 = h ? m3 + s2.x : s2.x;
    m2 = h ? fmaf(s0.x, z2.x, m2) : t.x;
    m4 = h ? fmaf(s1.x, z2.x, m4) : s1.x * z2.x;
    m5 = h ? fmaf(t.x, z2.x, m5) : t.x * z2.x;
    m0 += s0.y;
    m1 += s1.y;
    m3 += s2.y;
    m2 = fmaf(s0.y, z2.y, m2);
    m4 = fmaf(s1.y, z2.y, m4);
    m5 = fmaf(t.y, z2.y, m5);
  }
  // second moments about c^2 I, then into the totals
  m3 = fmaf(-kC2, m0, m3);
  m5 = fmaf(-kC2, m0, m5);
  n[0] = add2(n[0], make_float2(m0, m1));
  n[1] = add2(n[1], make_float2(m2, m3));
  n[2] = add2(n[2], make_float2(m4, m5));
}

// Entries of a backward unit: 256, or 128 where the lists hold no more than one
// and a half times 256 for every warp of the grid, so that the last units take
// less of the time, or 64 where they hold no more than 32 and most warps would
// have none.  us per backward with units of 64, 128, 256, by entries per
// warp / 256: 0.01 (d 64, M 2000): 20, 21, -; 0.125: 29, 31, -; 0.2: 40, 34, -;
// 0.8 (d 128, M 20000): 71, 72, 90; 1.26: 98, 91, 101; 1.5: 110, 104, 107; 2: 141,
// 128, 127; 4: 279, 218, 202.
__device__ __forceinline__ int unit_length(int64_t total, int nwarps) {
  return total <= 32 * (int64_t)nwarps ? 64 : total <= 384 * (int64_t)nwarps ? 128 : 256;
}

// a5.  Every warp works on its own: a unit is up to 256 consecutive entries of
// a task (a segment of one tile's list), claimed from a counter, with the
// tile's g in the warp's own shared memory, so no barrier couples the warps
// and the units in flight at any time come from neighbouring tiles.  A warp
// sorts each window of its unit by (number of blocks, first block) and runs
// it in rounds of 32 records, one lane per record: the lanes of a round have
// loops of one length, and mostly read the same blocks of g at the same time
// (a broadcast instead of bank conflicts).
//
// The moments of a round are added to memory one lane per record, or six lanes
// per record, which costs the L1 a sixth of the tag lookups and about a tenth
// more instructions.  Six lanes are the better where records have few blocks
// to evaluate between their additions.  us per backward, one lane and six, by
// list entries per (view, Gaussian): 1.24 (d 128, M 20000, B 128): 229, 218;
// 1.75 (d 384, M 300000, B 8): 283, 262; 1.88 (d 128, M 20000) B 32: 93, 97,
// B 96: 221, 206; 2.08, B 32: 101, 106, B 96: 232, 224; 2.45, B 32: 119, 126,
// B 256: 626, 639; 4.2 (scales 0.3-12 px, M 50000, B 64): 723, 758.  The line
// lies at 2.  Each form is an instance of its own: one loop with both took 1 to
// 3% longer.
//
// What bounds it: the L1 (72%: the scattered additions), issue (65% of the
// slots) and the FMA pipe (57% of its cycles), at d 384, M 500000.  Against
// CTAs of four warps that walked a whole tile's list, the longest lists first
// (us per backward, the default configuration then and now): d 384, M 500000,
// B 3: 699, 271; d 128, M 20000, B 256: 677, 623; d 128, M 50000, B 64, scales
// 0.3-12 px: 1084, 715; d 64, M 2000, B 32: 57, 35, but B 320: 115, 121 (the
// step of these: 406, 354).

// One warp's shared memory.  A round's moments have kRed words per record: one
// of padding where that does not cost a CTA.
template <int kPer, int kRed>
struct BwdWarp {
  static constexpr int kWW = 32 * kPer;  // records per window
  static constexpr int kBins = 256;      // (16 - blocks) * 16 + first block
  float4 sg[4][16];                      // g by row pair and column of a block, and block
  float4 sa[kWW];                        // px, py, u11, u12
  float2 sb[kWW];                        // u22, log2 A
  uint32_t sj[kWW];
  unsigned short smask[kWW];
  float red[32 * kRed];                  // a round's moments
  static_assert(sizeof(float4) * kWW >= kBins * sizeof(int), "the bins lie where the records go");
};

// The walk of one warp; spread: the moments of a round are added one lane per
// record, else six.
template <bool spread, int kPer, int kRed>
__device__ __forceinline__ void bwd_walk(
    BwdWarp<kPer, kRed> &S, const Rec *__restrict__ rec, const uint2 *__restrict__ list, int64_t M, int d,
    float l2tau, int64_t total, const float *__restrict__ dproj, double *__restrict__ mom,
    const RasterTasks &tk) {
  constexpr int kWarps = kThreads / 32, kWW = 32 * kPer;
  const int nt = d / kTile, T = nt * nt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float nl2tau = -l2tau;  // kept: -e < -log2(tau)
  float4(*sg)[16] = S.sg;
  float4 *sa = S.sa;
  float2 *sb = S.sb;
  uint32_t *sj = S.sj;
  unsigned short *smask = S.smask;
  float *red = S.red;
  const int lr = lane < 30 ? lane / 6 : 64, lc = lane % 6;  // record and moment a lane adds
  int *bins = reinterpret_cast<int *>(sa);
  const int nwarps = (int)gridDim.x * kWarps;
  const int unit = unit_length(total, nwarps);
  const int per_task = ((int)tk.ctr[kCtrSegment] + unit - 1) / unit;  // units of a task
  const int64_t nunits = (int64_t)tk.ctr[kCtrTasks] * per_task;
  int64_t u = blockIdx.x * kWarps + warp;
  uint4 t0 = make_uint4(0u, 0u, 0u, 0u);
  if (u < nunits) t0 = tk.task[2 * (u / per_task)];
  while (u < nunits) {
    // the next unit is claimed now and its descriptor read while this one runs
    int64_t nu = 0;
    uint4 tn = make_uint4(0u, 0u, 0u, 0u);
    if (lane == 0) nu = (int64_t)atomicAdd(tk.ctr + kCtrBwd, 1u) + nwarps;
    const int off = (int)(u % per_task) * unit;
    const int n = min(unit, (int)t0.z - off);
    const uint2 *L = list + (int64_t)(((uint64_t)t0.y << 32) | t0.x) + off;
    const int bt = (int)t0.w;
    const int b = bt / T, t = bt - b * T;
    const int tx = t % nt, ty = t / nt;
    const int x0 = tx * kTile, y0 = ty * kTile;
    const Rec *rb = rec + (int64_t)b * M;
    double *mb = mom + (int64_t)b * M * 6, *mbl = mb + lc;
    if (n > 0) {
      // the tile's g, stored block by block
      float4 g[2];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        g[h] = __ldg(reinterpret_cast<const float4 *>(
            dproj + ((int64_t)b * d + y0 + 8 * h + (lane >> 2)) * d + x0 + 4 * (lane & 3)));
      __syncwarp();  // the last unit's reads are done
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 8 * h + (lane >> 2), k = 4 * (r >> 2) + (lane & 3), hp = r & 2, lo = r & 1;
        float *u0 = reinterpret_cast<float *>(&sg[hp][k]) + lo;
        float *u1 = reinterpret_cast<float *>(&sg[hp + 1][k]) + lo;
        u0[0] = g[h].x;
        u0[2] = g[h].z;
        u1[0] = g[h].y;
        u1[2] = g[h].w;
      }
    }
    for (int w0 = 0; w0 < n; w0 += kWW) {
      uint2 en[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int i = w0 + 32 * q + lane;
        en[q] = i < n ? L[i] : make_uint2(0xffffffffu, 0u);
      }
      __syncwarp();  // the last window's reads are done
      reinterpret_cast<int4 *>(bins)[lane] = make_int4(0, 0, 0, 0);
      reinterpret_cast<int4 *>(bins)[32 + lane] = make_int4(0, 0, 0, 0);
      __syncwarp();
      int bin[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        // an out-of-range index (an entry left unwritten when the lists
        // overflowed their capacity) counts as empty
        const unsigned m = en[q].x < (uint64_t)M ? en[q].y & 0xffffu : 0u;
        en[q].y = m;
        bin[q] = m ? (16 - __popc(m)) * 16 + __ffs(m) - 1 : -1;
        if (m) atomicAdd(&bins[bin[q]], 1);
      }
      __syncwarp();
      // exclusive scan of the bins, eight per lane
      int nv;
      {
        int4 c[2] = {reinterpret_cast<int4 *>(bins)[2 * lane], reinterpret_cast<int4 *>(bins)[2 * lane + 1]};
        const int sum = c[0].x + c[0].y + c[0].z + c[0].w + c[1].x + c[1].y + c[1].z + c[1].w;
        int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += v;
        }
        nv = __shfl_sync(0xffffffffu, inc, 31);
        int run = inc - sum;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          int4 o;
          o.x = run;
          o.y = o.x + c[h].x;
          o.z = o.y + c[h].y;
          o.w = o.z + c[h].z;
          run = o.w + c[h].w;
          reinterpret_cast<int4 *>(bins)[2 * lane + h] = o;
        }
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < kPer; ++q)
        if (bin[q] >= 0) bin[q] = atomicAdd(&bins[bin[q]], 1);
      __syncwarp();  // the bins make way for the records
#pragma unroll
      for (int q0 = 0; q0 < kPer; q0 += 4) {
        Rec r[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (bin[q0 + q] >= 0) r[q] = load_rec(rb + en[q0 + q].x);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (bin[q0 + q] >= 0) {
            const int pos = bin[q0 + q];
            sa[pos] = r[q].a;
            sb[pos] = make_float2(r[q].b.x, r[q].b.y);
            sj[pos] = en[q0 + q].x;
            smask[pos] = (unsigned short)en[q0 + q].y;
          }
      }
      __syncwarp();
      if (w0 == 0) {
        nu = __shfl_sync(0xffffffffu, nu, 0);
        if (nu < nunits) tn = tk.task[2 * (nu / per_task)];
      }
#pragma unroll 1
      for (int r0 = 0; r0 < nv; r0 += 32) {
        const int slot = r0 + lane;
        if (slot < nv) {
          const float4 A = sa[slot];
          const float2 Bv = sb[slot];
          float2 tot[3];
#pragma unroll
          for (int i = 0; i < 3; ++i) tot[i] = make_float2(0.f, 0.f);
          for (unsigned mm = smask[slot]; mm; mm &= mm - 1)
            block_moments(sg, __ffs(mm) - 1, x0, y0, A, Bv.x, Bv.y, nl2tau, tot);
          if (spread) {
            double *mo = mb + 6ull * sj[slot];
#pragma unroll
            for (int i = 0; i < 6; ++i) atomicAdd(mo + i, (double)(i & 1 ? tot[i / 2].y : tot[i / 2].x));
          } else {
#pragma unroll
            for (int i = 0; i < 6; ++i) red[kRed * lane + i] = i & 1 ? tot[i / 2].y : tot[i / 2].x;
          }
        }
        if (spread) continue;
        __syncwarp();
        // six lanes add one record's six moments, five records at a time: the
        // warp's addresses then lie in five or so lines, not in 32
        const int left = min(32, nv - r0);
        const float *rp = red + kRed * lr + lc;
        const uint32_t *jp = sj + r0 + lr;
#pragma unroll
        for (int i = 0; i < 7; ++i)
          if (5 * i + lr < left) atomicAdd(mbl + 6ull * jp[5 * i], (double)rp[5 * kRed * i]);
        __syncwarp();  // read before the next round's replace them
      }
    }
    if (n <= 0) {
      nu = __shfl_sync(0xffffffffu, nu, 0);
      if (nu < nunits) tn = tk.task[2 * (nu / per_task)];
    }
    u = nu;
    t0 = tn;
  }
}

template <int kPer, int kMinB>
__global__ void __launch_bounds__(kThreads, kMinB) raster_bwd_kernel(
    const Rec *__restrict__ rec, const uint2 *__restrict__ list, int64_t M, int d, float l2tau,
    const int64_t *__restrict__ tile_start, int ntiles, const float *__restrict__ dproj,
    double *__restrict__ mom, RasterTasks tk) {
  // six CTAs of 256-record windows fit an SM's shared memory to the byte
  constexpr int kRed = kPer == 8 && kMinB == 6 ? 6 : 7;
  __shared__ BwdWarp<kPer, kRed> S[kThreads / 32];
  static_assert(kMinB * (sizeof(S) + 1024) <= 228 * 1024, "kMinB CTAs fit an SM's shared memory");
  const int nt = d / kTile;
  const int64_t total = tile_start[ntiles];
  if (total > 2 * (int64_t)(ntiles / (nt * nt)) * M)
    bwd_walk<true, kPer, kRed>(S[threadIdx.x >> 5], rec, list, M, d, l2tau, total, dproj, mom, tk);
  else
    bwd_walk<false, kPer, kRed>(S[threadIdx.x >> 5], rec, list, M, d, l2tau, total, dproj, mom, tk);
}

// The backward's kernel configurations (the autotuner's search space):
// records per lane and window, CTAs per SM.
static const BwdCfg kBwdCfgs[] = {
    {8, 5, "256-record warp windows, 5 CTAs/SM"}, {8, 4, "256-record warp windows, 4 CTAs/SM"},
    {8, 6, "256-record warp windows, 6 CTAs/SM"}, {4, 8, "128-record warp windows, 8 CTAs/SM"},
    {4, 7, "128-record warp windows, 7 CTAs/SM"}, {4, 6, "128-record warp windows, 6 CTAs/SM"},
    {4, 5, "128-record warp windows, 5 CTAs/SM"}, {4, 4, "128-record warp windows, 4 CTAs/SM"},
    {8, 3, "256-record warp windows, 3 CTAs/SM"}, {4, 3, "128-record warp windows, 3 CTAs/SM"},
};
int bwd_config_count() { return (int)(sizeof(kBwdCfgs) / sizeof(kBwdCfgs[0])); }
const BwdCfg &bwd_config(int i) { return kBwdCfgs[i]; }

cudaError_t launch_raster_bwd(int cfg, const Rec *rec, const uint2 *list,
                              const int64_t *tile_start, int64_t M, int B, int d, float l2tau,
                              const float *dproj, double *mom, const RasterTasks &tk,
                              cudaStream_t st) {
  if (cfg < 0 || cfg >= bwd_config_count()) return cudaErrorInvalidValue;
  const BwdCfg &c = kBwdCfgs[cfg];
  const int grid = sm_count() * c.ctas, nt = d / kTile, ntiles = nt * nt * B;
  if (c.per == 8 && c.ctas == 6)
    raster_bwd_kernel<8, 6><<<grid, kThreads, 0, st>>>(rec, list, M, d, l2tau, tile_start, ntiles, dproj, mom, tk);
  else if (c.per == 8)
    raster_bwd_kernel<8, 5><<<grid, kThreads, 0, st>>>(rec, list, M, d, l2tau, tile_start, ntiles, dproj, mom, tk);
  else if (c.ctas >= 7)
    raster_bwd_kernel<4, 8><<<grid, kThreads, 0, st>>>(rec, list, M, d, l2tau, tile_start, ntiles, dproj, mom, tk);
  else
    raster_bwd_kernel<4, 6><<<grid, kThreads, 0, st>>>(rec, list, M, d, l2tau, tile_start, ntiles, dproj, mom, tk);
  return cudaGetLastError();
}

// ------------------------------------------------------ plain dense -----

// One thread per pixel, every Gaussian of the image, no culling.
__global__ void __launch_bounds__(256) dense_fwd_kernel(const Rec *__restrict__ rec, int64_t M,
                                                        int d, float l2tau,
                                                        float *__restrict__ proj) {
  int b = blockIdx.y;
  int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool act = pix < (int64_t)d * d;
  int u = (int)(pix % d), v = (int)(pix / d);
  const Rec *rb = rec + (int64_t)b * M;
  const float nl2tau = -l2tau;
  double acc = 0.0;
  float part = 0.f;
  for (int64_t j = 0; j < M; ++j) {
    Rec r = rb[j];
    float dx = (float)u - r.a.x, dy = (float)v - r.a.y;
    // -e = z1^2 + (z2^2 - l2A), every product rounded (the tiled forms fuse
    // u11 dx into z1's sum, so a pair within that rounding of tau can be kept
    // by one and not by the other)
    float z1 = __fadd_rn(__fmul_rn(r.a.z, dx), __fmul_rn(r.a.w, dy));
    float z2 = __fmul_rn(r.b.x, dy);
    float ff = __fmaf_rn(z1, z1, __fmaf_rn(z2, z2, -r.b.y));
    float val = ex2_approx(-ff);
    part += ff < nl2tau ? val : 0.f;
    if ((j & 127) == 127) {
      acc += part;
      part = 0.f;
    }
  }
  acc += part;
  if (act) proj[(int64_t)b * d * d + pix] = (float)acc;
}

// One thread per (image, Gaussian), every pixel of the image; the same six
// moments as the tiled backward (whitened coordinates, second moments about
// c^2 I, taken per row).
__global__ void __launch_bounds__(128) dense_bwd_kernel(const Rec *__restrict__ rec, int64_t M,
                                                        int d, float l2tau,
                                                        const float *__restrict__ dproj,
                                                        double *__restrict__ mom) {
  int b = blockIdx.y;
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  Rec r = rec[(int64_t)b * M + j];
  const float *g = dproj + (int64_t)b * d * d;
  const float nl2tau = -l2tau;
  float m[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int v = 0; v < d; ++v) {
    float dy = (float)v - r.a.y;
    float uy = __fmul_rn(r.a.w, dy), z2 = __fmul_rn(r.b.x, dy);
    float nc = __fmaf_rn(z2, z2, -r.b.y);
    float r0 = 0.f, r1 = 0.f, r3 = 0.f;
    for (int u = 0; u < d; ++u) {
      float dx = (float)u - r.a.x;
      float z1 = __fadd_rn(__fmul_rn(r.a.z, dx), uy);
      float ff = __fmaf_rn(z1, z1, nc);
      float val = ex2_approx(-ff);
      float gv = ff < nl2tau ? __ldg(g + (int64_t)v * d + u) * val : 0.f;
      r0 += gv;
      float tt = gv * z1;
      r1 += tt;
      r3 = fmaf(tt, z1, r3);
    }
    m[0] += r0;
    m[1] += r1;
    m[2] = fmaf(z2, r0, m[2]);
    m[3] += fmaf(-kC2, r0, r3);
    m[4] = fmaf(z2, r1, m[4]);
    m[5] = fmaf(fmaf(z2, z2, -kC2), r0, m[5]);
  }
  if (!(r.b.z >= 0.f)) {  // no region above tau: no tile, no moments
#pragma unroll
    for (int k = 0; k < 6; ++k) m[k] = 0.f;
  }
  double *mm = mom + ((int64_t)b * M + j) * 6;
#pragma unroll
  for (int k = 0; k < 6; ++k) mm[k] = (double)m[k];
}

cudaError_t launch_dense_fwd(const Rec *rec, int64_t M, int B, int d, float l2tau, float *proj,
                             cudaStream_t st) {
  dim3 grid((unsigned)(((int64_t)d * d + 255) / 256), B);
  dense_fwd_kernel<<<grid, 256, 0, st>>>(rec, M, d, l2tau, proj);
  return cudaGetLastError();
}

cudaError_t launch_dense_bwd(const Rec *rec, int64_t M, int B, int d, float l2tau,
                             const float *dproj, double *mom, cudaStream_t st) {
  dim3 grid((unsigned)((M + 127) / 128), B);
  dense_bwd_kernel<<<grid, 128, 0, st>>>(rec, M, d, l2tau, dproj, mom);
  return cudaGetLastError();
}

}  // namespace gem
