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
//     at most 1024 entries, taken from a counter by persistent CTAs.  Producer
//     warps stage a segment's records (only the 24 bytes the evaluation reads)
//     and, by warp bit transposes of the packed block masks, each block's
//     record set; consumer warps take the window's blocks one after the other
//     and evaluate 32 of a block's records at a time, one record and 16 pixels
//     per lane (packed float pairs).  A pixel's sum within a segment runs
//     over lanes, then by a tree over the 32 lanes; a tile's segments join in
//     list order with Kahan compensation.  The result is deterministic and
//     follows the list's depth order segment by segment.
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

// Barrier id over the given number of threads of the CTA.
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// mbarriers in shared memory: arrivals release, waits acquire.
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
// Waits for the phase of the given parity, at most kWaitTries tries (each
// suspends the thread for a hardware time slice; seconds in all); false when
// it did not complete.
constexpr int kWaitTries = 1 << 22;
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  for (int i = 0; i < kWaitTries; ++i) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

constexpr int kFwdWin = 1024;  // forward: records staged per window

// Tasks of the rasterisers.  A tile's list is cut into segments of S entries
// (the last one shorter); a task is one segment, staged as one window, so
// that no CTA walks a long list alone (the longest list of a workload holds
// five to twenty times the mean) and a call with few tiles still fills the
// SMs.  S is 1024, less (down to 256) where that would leave resident CTAs
// without a segment.  Tasks follow the tiles' index order up to the order in
// which the CTAs here claim their ranges, so neighbouring tiles, which share
// records, are in flight together.  Empty tiles get their zeros here and no
// task.
__device__ __forceinline__ int64_t segment_length(int64_t total, int slots) {
  const int64_t S = total / (2 * (int64_t)slots);
  return (max((int64_t)256, min((int64_t)kFwdWin, S)) + 63) / 64 * 64;
}

__global__ void __launch_bounds__(256) raster_tasks_kernel(const int64_t *__restrict__ tile_start,
                                                           int ntiles, int64_t cap, int d, int slots,
                                                           RasterTasks tk, float *__restrict__ proj) {
  __shared__ unsigned wsum[2][8], base_sh[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 256 + threadIdx.x;
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
  // exclusive prefixes of the tasks and of the partial images they need
  unsigned inc = nseg, incp = nseg > 1 ? nseg : 0;
  const unsigned mine = incp;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(0xffffffffu, inc, o), v = __shfl_up_sync(0xffffffffu, incp, o);
    if (lane >= o) {
      inc += u;
      incp += v;
    }
  }
  if (lane == 31) {
    wsum[0][warp] = inc;
    wsum[1][warp] = incp;
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
  if (i == 0) tk.ctr[kCtrSegment] = (unsigned)S;
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
      t[1] = make_uint4(k, nseg, part, 0u);
    }
  }
  if (proj) {
    const int nt = d / kTile, T = nt * nt;
    for (unsigned e = __ballot_sync(0xffffffffu, i < ntiles && nseg == 0); e; e &= e - 1) {
      const int bt = blockIdx.x * 256 + warp * 32 + __ffs(e) - 1;
      const int b = bt / T, t = bt - b * T;
      float *o = proj + ((int64_t)b * d + (t / nt) * kTile) * d + (t % nt) * kTile;
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4 *>(o + (int64_t)(8 * q + (lane >> 2)) * d + 4 * (lane & 3)) =
            make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

// Shared memory of one forward CTA: two staged windows, the lists of the
// consumer warps, and the barriers.
struct FwdWindow {
  float4 sa[kFwdWin];        // px, py, u11, u12
  float2 sb[kFwdWin];        // u22, log2 A
  unsigned bal[16][33];      // block, 32 records: which touch it
  float out[16][16];         // block, pixel: the window's sums
  int n, bt;                 // entries (-1: no more tasks), image * T + tile
  unsigned seg, nseg, part;  // segment of the tile, how many, first partial image
  int next_block, done;      // blocks handed out, blocks finished
};
template <int kCons>
struct FwdShared {
  uint4 desc[2][2];                      // the producers' current and next task
  FwdWindow win[2];
  unsigned short slots[kCons][kFwdWin];  // a block's records, in list order
  uint64_t full[2], empty[2];            // mbarriers
};

// a3.  One producer warp and kCons consumer warps per CTA, two windows in
// shared memory.  The producer claims tasks and stages their records; the
// lanes' packed masks, transposed as bit matrices, give for every block one
// 32-bit word per 32 records (which of them touch the block).  A consumer
// warp takes the next block of the window, turns the block's words into the
// list of the records that touch it (lane l lists those of 32 slots, in
// order), its 32 lanes evaluate 32 of those records at a time, one record
// and 16 pixels per lane, and the lanes' partial images are added by a
// butterfly that halves the pixels a lane holds at each of four steps.  A
// warp that finds no block left goes on to the other window without waiting
// for its neighbours; the warp that finishes the last block writes the
// window's 256 pixels.  Windows of a tile with several segments go to
// partial images, which the last segment to finish adds in segment order
// (Kahan).  Nothing depends on which warp or CTA did what, so the result is
// deterministic.
//
// What bounds it: issue (about 60% of the slots) and the L1, through which
// every entry's 32 scattered bytes come (one 256-bit load per record: two
// loads of 16 and 8 bytes cost 8% of the launch) and which serves the record
// reads of the evaluation.  Against CTAs of four warps that staged 256
// records between barriers and gave each block a share of the threads
// (us per launch): d 384, M 500000, B 16: 680 -> 467; d 128, M 20000, B 256:
// 388 -> 367; d 256, M 100000, B 64: 498 -> 418; d 128, M 50000, B 64, scales
// 0.3-12 px, whose longest lists hold 14000 entries: 745-850 -> 391; d 64,
// M 2000, B 32: 37 -> 24.  Staging by the consumers between barriers: 553 at
// the first of these; one producer warp with small copies in flight: 494-518;
// windows of 512 records: 610.
//
// kCount = true: the same walk, counting kept pairs into kept[0] and
// evaluated pairs into kept[1] instead of writing the projection
// (inspection only, never on the timed path).
template <int kCons, int kProd, int kMinB, bool kCount>
__global__ void __launch_bounds__(32 * (kCons + kProd), kMinB) raster_fwd_kernel(
    const Rec *__restrict__ rec, const uint2 *__restrict__ list, int64_t M, int d, float l2tau,
    RasterTasks tk, float *__restrict__ proj, unsigned long long *__restrict__ kept) {
  extern __shared__ __align__(16) unsigned char fwd_smem[];
  FwdShared<kCons> &S = *reinterpret_cast<FwdShared<kCons> *>(fwd_smem);
  const int nt = d / kTile, T = nt * nt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&S.full[i], 32 * kProd);
      mbar_init(&S.empty[i], kCons);
    }
  }
  __syncthreads();
  if (warp >= kCons) {
    // ---- producers ----
    const int pw = warp - kCons;
    const bool leader = pw == 0 && lane == 0;
    const int ntasks = (int)tk.ctr[kCtrTasks];
    // the leader claims a task two windows ahead and reads its descriptor one
    // window ahead; t1.w marks the end
    int nq = 0;
    if (leader) {
      const int q = blockIdx.x;
      if (q < ntasks) {
        S.desc[0][0] = tk.task[2 * (int64_t)q];
        S.desc[0][1] = tk.task[2 * (int64_t)q + 1];
      } else {
        S.desc[0][1].w = 1u;
      }
      nq = (int)(atomicAdd(tk.ctr + kCtrFwd, 1u) + gridDim.x);
    }
    for (int it = 0;; ++it) {
      FwdWindow &W = S.win[it & 1];
      named_sync(1, 32 * kProd);
      const uint4 t0 = S.desc[it & 1][0], t1 = S.desc[it & 1][1];
      // the other parity passes at once on a fresh barrier
      if (!mbar_wait(&S.empty[it & 1], ((it >> 1) & 1) ^ 1)) {
        if (lane == 0) atomicOr(tk.status, kStatusTimeout);
        return;
      }
      if (t1.w) {
        if (leader) W.n = -1;
        mbar_arrive(&S.full[it & 1]);
        return;
      }
      uint4 n0 = make_uint4(0u, 0u, 0u, 0u), n1 = make_uint4(0u, 0u, 0u, 1u);
      int nq2 = 0;
      if (leader) {
        if (nq < ntasks) {
          n0 = tk.task[2 * (int64_t)nq];
          n1 = tk.task[2 * (int64_t)nq + 1];
        }
        nq2 = (int)(atomicAdd(tk.ctr + kCtrFwd, 1u) + gridDim.x);
      }
      const uint2 *L = list + (int64_t)(((uint64_t)t0.y << 32) | t0.x);
      const int n = (int)t0.z, bt = (int)t0.w;
      const Rec *rb = rec + (int64_t)(bt / T) * M;
      if (leader) {
        W.n = n;
        W.bt = bt;
        W.seg = t1.x;
        W.nseg = t1.y;
        W.part = t1.z;
        W.next_block = 0;
        W.done = 0;
      }
      // this warp's pairs of 32-entry chunks, all their entries in flight together
      constexpr int kPairs = kFwdWin / 64 / kProd;
      uint2 ent[2 * kPairs];
#pragma unroll
      for (int u = 0; u < 2 * kPairs; ++u) {
        const int slot = 64 * ((u >> 1) * kProd + pw) + 32 * (u & 1) + lane;
        ent[u] = slot < n ? L[slot] : make_uint2(0xffffffffu, 0u);
      }
      // records in batches of kB chunks in flight
      constexpr int kB = kPairs >= 2 ? 4 : 2;
#pragma unroll
      for (int u0 = 0; u0 < 2 * kPairs; u0 += kB) {
        if (64 * ((u0 >> 1) * kProd + pw) >= n) break;
        Rec r[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u) {
          // an entry whose Gaussian index is out of range counts as empty
          if (ent[u0 + u].x < (uint64_t)M)
            r[u] = load_rec(rb + ent[u0 + u].x);
          else
            ent[u0 + u].y = 0u;
        }
        // lane k < 16: block k of the first chunk of a pair, lane 16 + k: of the second
#pragma unroll
        for (int u = 0; u < kB; u += 2)
          W.bal[lane & 15][2 * (((u0 + u) >> 1) * kProd + pw) + (lane >> 4)] =
              warp_transpose32((ent[u0 + u].y & 0xffffu) | (ent[u0 + u + 1].y << 16), lane);
#pragma unroll
        for (int u = 0; u < kB; ++u) {
          const int slot = 64 * (((u0 + u) >> 1) * kProd + pw) + 32 * (u & 1) + lane;
          W.sa[slot] = r[u].a;
          W.sb[slot] = make_float2(r[u].b.x, r[u].b.y);
        }
      }
      if (leader) {
        S.desc[(it + 1) & 1][0] = n0;
        S.desc[(it + 1) & 1][1] = n1;
        nq = nq2;
      }
      __syncwarp();
      mbar_arrive(&S.full[it & 1]);
    }
  }
  // ---- consumers ----
  const float nl2tau = -l2tau;  // kept: -e < -log2(tau)
  unsigned short *slots = S.slots[warp];
  unsigned nkept = 0, neval = 0;
  for (int it = 0;; ++it) {
    FwdWindow &W = S.win[it & 1];
    if (!mbar_wait(&S.full[it & 1], (it >> 1) & 1)) {
      if (lane == 0) atomicOr(tk.status, kStatusTimeout);
      return;
    }
    const int n = W.n;
    if (n < 0) break;
    const int bt = W.bt;
    const int b = bt / T, t = bt - b * T;
    const int tx = t % nt, ty = t / nt;
    const int x0 = tx * kTile, y0 = ty * kTile;
    const int nw = ((n + 63) >> 6) << 1;  // words staged
    for (;;) {
      int k = 0;
      if (lane == 0) k = atomicAdd(&W.next_block, 1);
      k = __shfl_sync(0xffffffffu, k, 0);
      if (k >= 16) break;
      unsigned bits = lane < nw ? W.bal[k][lane] : 0u;
      const int c = __popc(bits);
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int nk = __shfl_sync(0xffffffffu, incl, 31);
      {
        unsigned short *w = slots + (incl - c);
        for (; bits; bits &= bits - 1) *w++ = (unsigned short)(32 * lane + __ffs(bits) - 1);
      }
      __syncwarp();
      // acc[4 h + x]: column x, rows 2 h and 2 h + 1
      float2 acc[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = make_float2(0.f, 0.f);
      const float X0 = (float)(x0 + 4 * (k & 3)), Y0 = (float)(y0 + 4 * (k >> 2));
      const float2 ys0 = make_float2(Y0, Y0 + 1.f), ys1 = make_float2(Y0 + 2.f, Y0 + 3.f);
      for (int i = lane; i < nk; i += 32) {
        const int slot = slots[i];
        const float4 A = W.sa[slot];
        const float2 Bv = W.sb[slot];
        // -e = z1^2 + (z2^2 - l2A), z1 = u11 dx + u12 dy (u11 dx fused into
        // the sum), z2 = u22 dy, two rows of a column in one packed operation
        float2 dx[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) dx[x] = f2(__fsub_rn(X0 + (float)x, A.x));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 dy = add2(h ? ys1 : ys0, f2(-A.y));
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
              acc[4 * h + x] = fma2(make_float2(ex2_approx(-f.x), ex2_approx(-f.y)),
                                    make_float2(set_lt(f.x, nl2tau), set_lt(f.y, nl2tau)),
                                    acc[4 * h + x]);
          }
        }
        if (kCount) neval += 16;
      }
      __syncwarp();  // the slots are read before the next block's replace them
      if (kCount) continue;
      // 16 pixels x 32 lanes -> the pixel of lane pair (2 p, 2 p + 1)
      float v8[8], v4[4], v2[2];
      const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        // lanes with bit 4 clear keep rows 0 and 1, the others rows 2 and 3
        const float2 keep = b4 ? acc[4 + x] : acc[x], give = b4 ? acc[x] : acc[4 + x];
        v8[x] = keep.x + __shfl_xor_sync(0xffffffffu, give.x, 16);
        v8[4 + x] = keep.y + __shfl_xor_sync(0xffffffffu, give.y, 16);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
        v4[x] = (b3 ? v8[4 + x] : v8[x]) + __shfl_xor_sync(0xffffffffu, b3 ? v8[x] : v8[4 + x], 8);
#pragma unroll
      for (int x = 0; x < 2; ++x)
        v2[x] = (b2 ? v4[2 + x] : v4[x]) + __shfl_xor_sync(0xffffffffu, b2 ? v4[x] : v4[2 + x], 4);
      float v1 = (b1 ? v2[1] : v2[0]) + __shfl_xor_sync(0xffffffffu, b1 ? v2[0] : v2[1], 2);
      v1 += __shfl_xor_sync(0xffffffffu, v1, 1);
      if (!(lane & 1)) W.out[k][lane >> 1] = v1;
      // the warp that finishes the window's last block writes its pixels
      __threadfence_block();
      __syncwarp();
      int dn = 0;
      if (lane == 0) dn = atomicAdd(&W.done, 1);
      dn = __shfl_sync(0xffffffffu, dn, 0);
      if (dn != 15) continue;
      __threadfence_block();
      // lane: half a pixel row of the tile, two blocks' rows of four
      const int row = lane >> 1, k0 = 4 * (row >> 2) + 2 * (lane & 1), p0 = 4 * (row & 3);
      float4 v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) v[h] = *reinterpret_cast<const float4 *>(&W.out[k0 + h][p0]);
      const unsigned nseg = W.nseg;
      float4 *o = reinterpret_cast<float4 *>(proj + ((int64_t)b * d + y0 + row) * d + x0 + 8 * (lane & 1));
      if (nseg > 1) {
        float4 *part = reinterpret_cast<float4 *>(tk.part + (int64_t)W.part * 256) + 2 * lane;
        __stcg(part + (int64_t)W.seg * 64, v[0]);
        __stcg(part + (int64_t)W.seg * 64 + 1, v[1]);
        __threadfence();
        __syncwarp();
        unsigned prev = 0;
        if (lane == 0) prev = atomicAdd(tk.done + bt, 1u);
        if (__shfl_sync(0xffffffffu, prev, 0) != nseg - 1) continue;
        __threadfence();
        float2 s[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] = make_float2(0.f, 0.f);
        for (unsigned g = 0; g < nseg; ++g) {
          const float4 a = __ldcg(part + (int64_t)g * 64), c4 = __ldcg(part + (int64_t)g * 64 + 1);
          const float x[8] = {a.x, a.y, a.z, a.w, c4.x, c4.y, c4.z, c4.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) s[j] = kahan_add(s[j], x[j]);
        }
        if (lane == 0) tk.done[bt] = 0u;  // as the next call expects it
        v[0] = make_float4(s[0].x - s[0].y, s[1].x - s[1].y, s[2].x - s[2].y, s[3].x - s[3].y);
        v[1] = make_float4(s[4].x - s[4].y, s[5].x - s[5].y, s[6].x - s[6].y, s[7].x - s[7].y);
      }
      o[0] = v[0];
      o[1] = v[1];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.empty[it & 1]);
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
    {6, 2, 3, "6 consumer and 2 producer warps, 3 CTAs/SM"},
    {8, 2, 3, "8 consumer and 2 producer warps, 3 CTAs/SM"},
    {8, 4, 2, "8 consumer and 4 producer warps, 2 CTAs/SM"},
    {12, 4, 2, "12 consumer and 4 producer warps, 2 CTAs/SM"},
    {10, 2, 2, "10 consumer and 2 producer warps, 2 CTAs/SM"},
    {6, 2, 2, "6 consumer and 2 producer warps, 2 CTAs/SM"},
    {8, 2, 2, "8 consumer and 2 producer warps, 2 CTAs/SM"},
    {12, 4, 1, "12 consumer and 4 producer warps, 1 CTA/SM"},
};
int fwd_config_count() { return (int)(sizeof(kFwdCfgs) / sizeof(kFwdCfgs[0])); }
const FwdCfg &fwd_config(int i) { return kFwdCfgs[i]; }

static int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Partial images that any lists of up to cap entries can need: a tile of
// more than S entries has fewer than 2 len / S segments, and S is at least
// total / (2 slots) (at most 4 slots of them) or 1024.
constexpr int kFwdSlots = 3 * 256;  // CTAs that fit up to 256 SMs
size_t raster_part_count(int64_t cap) {
  return (size_t)(4 * kFwdSlots + 2 * (cap / kFwdWin + 1));
}

template <int kCons, int kProd, int kMinB, bool kCount>
static cudaError_t launch_fwd_one(int grid, const Rec *rec, const uint2 *list, int64_t M, int d,
                                  float l2tau, const RasterTasks &tk, float *proj,
                                  unsigned long long *kept, cudaStream_t st) {
  raster_fwd_kernel<kCons, kProd, kMinB, kCount>
      <<<grid, 32 * (kCons + kProd), sizeof(FwdShared<kCons>), st>>>(rec, list, M, d, l2tau, tk, proj, kept);
  return cudaGetLastError();
}

template <int kCons, int kProd, int kMinB>
static cudaError_t configure_fwd_one() {
  const int smem = (int)sizeof(FwdShared<kCons>);
  const cudaError_t e = cudaFuncSetAttribute(raster_fwd_kernel<kCons, kProd, kMinB, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(raster_fwd_kernel<kCons, kProd, kMinB, true>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t raster_configure() {
  cudaError_t e;
  if ((e = configure_fwd_one<6, 2, 3>()) != cudaSuccess || (e = configure_fwd_one<8, 2, 3>()) != cudaSuccess ||
      (e = configure_fwd_one<8, 4, 2>()) != cudaSuccess || (e = configure_fwd_one<12, 4, 2>()) != cudaSuccess ||
      (e = configure_fwd_one<10, 2, 2>()) != cudaSuccess)
    return e;
  return cudaSuccess;
}

template <bool kCount>
static cudaError_t launch_fwd_any(int cfg, const Rec *rec, const uint2 *list,
                                  const int64_t *tile_start, int64_t cap, int64_t M, int B, int d,
                                  float l2tau, float *proj, unsigned long long *kept,
                                  const RasterTasks &tk, bool fresh, cudaStream_t st) {
  if (cfg < 0 || cfg >= fwd_config_count()) return cudaErrorInvalidValue;
  const FwdCfg &c = kFwdCfgs[cfg];
  const int nt = d / kTile, ntiles = nt * nt * B, sms = sm_count();
  if (!fresh) {
    const cudaError_t e = cudaMemsetAsync(tk.ctr, 0, kCtrCount * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
  }
  raster_tasks_kernel<<<(ntiles + 255) / 256, 256, 0, st>>>(tile_start, ntiles, cap, d,
                                                            min(sms * 3, kFwdSlots), tk, proj);
  const int grid = sms * c.ctas;
  if (c.cons == 6) return launch_fwd_one<6, 2, 3, kCount>(grid, rec, list, M, d, l2tau, tk, proj, kept, st);
  if (c.cons == 10) return launch_fwd_one<10, 2, 2, kCount>(grid, rec, list, M, d, l2tau, tk, proj, kept, st);
  if (c.cons == 12) return launch_fwd_one<12, 4, 2, kCount>(grid, rec, list, M, d, l2tau, tk, proj, kept, st);
  if (c.prod == 4) return launch_fwd_one<8, 4, 2, kCount>(grid, rec, list, M, d, l2tau, tk, proj, kept, st);
  return launch_fwd_one<8, 2, 3, kCount>(grid, rec, list, M, d, l2tau, tk, proj, kept, st);
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

// The six moments of w = g * value over the 16 pixels of block k of the tile
// at (x0, y0) for one record (centre A.x, A.y, first row of U in A.z, A.w;
// u22, l2A), in the record's whitened coordinates z1 = u11 dx + u12 dy,
// z2 = u22 dy, added to the running totals n[0..5], each a pair (upper rows
// of the row pairs, lower rows):
//   n0 = sum w, n1 = sum w z1, n2 = sum w z2,
//   n3 = sum w (z1^2 - c^2), n4 = sum w z1 z2, n5 = sum w (z2^2 - c^2).
// Rows are taken two at a time, one per half of a packed pair, so the row
// terms (z2, and what is weighted by it) pack as naturally as the pixels'
// (a fifth fewer instructions than pairs of columns, whose row terms are
// scalars).  The second moments are taken about c^2 I, the whitened S^, per
// block.  sg is the g tile: [row pair, column pair][block] = rows 2 h and
// 2 h + 1 of column 2 c, then of column 2 c + 1.
__device__ __forceinline__ void block_moments(const float4 (*__restrict__ sg)[16], int k, int x0,
                                              int y0, const float4 &A, float u22, float l2A,
                                              float nl2tau, float2 (&n)[6]) {
  // the exponent rounded exactly as the forward rounds it, so that both
  // decide Eq. accu alike
  const float X0 = (float)(x0 + 4 * (k & 3)), Y0 = (float)(y0 + 4 * (k >> 2));
  float2 dx[4];
#pragma unroll
  for (int x = 0; x < 4; ++x) dx[x] = f2(__fsub_rn(X0 + (float)x, A.x));
  float2 m[6];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 dy = add2(make_float2(Y0 + (float)(2 * h), Y0 + (float)(2 * h + 1)), f2(-A.y));
    const float2 uy = mul2(f2(A.w), dy);
    const float2 z2 = mul2(f2(u22), dy);
    const float2 nc = fma2(z2, z2, f2(-l2A));
    float2 s0, s1, s2;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float4 g4 = sg[2 * h + c][k];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        // -e = z1^2 + (z2^2 - l2A), as in the forward's terms
        const float2 z = fma2(f2(A.z), dx[2 * c + q], uy);
        const float2 f = fma2(z, z, nc);
        // w = g * value on kept pairs (value > tau), zero elsewhere: g is
        // masked to +0 on the integer pipe, which leaves the FMA pipe (this
        // loop's busiest) the multiply
        const float2 gm = make_float2(keep_or_zero(q ? g4.z : g4.x, f.x, nl2tau),
                                      keep_or_zero(q ? g4.w : g4.y, f.y, nl2tau));
        const float2 w = mul2(gm, make_float2(ex2_approx(-f.x), ex2_approx(-f.y)));
        const float2 wz = mul2(w, z);
        s0 = c + q ? add2(s0, w) : w;
        s1 = c + q ? add2(s1, wz) : wz;
        s2 = c + q ? fma2(wz, z, s2) : mul2(wz, z);
      }
    }
    // the rows' sums of w, w z1 and w z1^2, weighted by z2
    const float2 t = mul2(s0, z2);
    m[0] = h ? add2(m[0], s0) : s0;
    m[1] = h ? add2(m[1], s1) : s1;
    m[2] = h ? add2(m[2], t) : t;
    m[3] = h ? add2(m[3], s2) : s2;
    m[4] = h ? fma2(s1, z2, m[4]) : mul2(s1, z2);
    m[5] = h ? fma2(t, z2, m[5]) : mul2(t, z2);
  }
  // second moments about c^2 I, then into the totals
  m[3] = fma2(f2(-kC2), m[0], m[3]);
  m[5] = fma2(f2(-kC2), m[0], m[5]);
#pragma unroll
  for (int i = 0; i < 6; ++i) n[i] = add2(n[i], m[i]);
}

// Entries of a backward unit: 256, less (down to 64) where that would leave
// warps of the grid without one.
__device__ __forceinline__ int unit_length(int64_t total, int nwarps) {
  const int64_t U = (total / nwarps + 31) / 32 * 32;
  return (int)max((int64_t)64, min((int64_t)256, U));
}

// a5.  Every warp works on its own: a unit is up to 256 consecutive entries of
// a task (a segment of one tile's list), claimed from a counter, with the
// tile's g in the warp's own shared memory, so no barrier couples the warps
// and the units in flight at any time come from neighbouring tiles.  A warp
// sorts each window of its unit by (number of blocks, first block) and runs
// it in rounds of 32 records, one lane per record: the lanes of a round have
// loops of one length, and mostly read the same blocks of g at the same time
// (a broadcast instead of bank conflicts).  The moments of a round are added
// to memory six lanes per record, which costs the L1 a sixth of the tag
// lookups of one lane per record and about a tenth more instructions: the
// better of the two at 2.5 list entries per (view, Gaussian) and four blocks
// each (d 128, M 20000, B 256: 0.53 against 0.59 ms), the worse at 4.2 and
// 5.5 (d 128, M 50000, B 64, scales 0.3-12 px: 0.66 against 0.62 ms), where
// a record's evaluation takes longer; the line lies at 3 entries.
//
// What bounds it: the FMA pipe (57% of its cycles) and issue (66%).  Against
// CTAs of four warps that walked a whole tile's list, the longest lists first
// (us per launch, the default configuration then, the one the autotuner
// picked, now): d 384, M 500000, B 16: 1033, 901, 792; d 128, M 20000, B 256:
// 568, 568, 540; d 128, M 50000, B 64, scales 0.3-12 px: 1150, 846, 637;
// d 64, M 2000, B 32: 44, 42, 26.
template <int kPer, int kMinB>
__global__ void __launch_bounds__(kThreads, kMinB) raster_bwd_kernel(
    const Rec *__restrict__ rec, const uint2 *__restrict__ list, int64_t M, int d, float l2tau,
    const int64_t *__restrict__ tile_start, int ntiles, const float *__restrict__ dproj,
    double *__restrict__ mom, RasterTasks tk) {
  constexpr int kWarps = kThreads / 32;
  constexpr int kWW = 32 * kPer;  // records per window
  constexpr int kBins = 256;      // (16 - blocks) * 16 + first block
  __shared__ float4 sg_[kWarps][4][16];  // g by row pair and column pair of a block, and block
  __shared__ float4 sa_[kWarps][kWW];    // px, py, u11, u12
  __shared__ float2 sb_[kWarps][kWW];    // u22, log2 A
  __shared__ uint32_t sj_[kWarps][kWW];
  __shared__ unsigned short smask_[kWarps][kWW];
  __shared__ float red_[kWarps][32 * 7];  // a round's moments, one word of padding per record
  static_assert(sizeof(sa_[0]) >= kBins * sizeof(int), "the bins lie where the records go");
  const int nt = d / kTile, T = nt * nt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float nl2tau = -l2tau;  // kept: -e < -log2(tau)
  float4(*sg)[16] = sg_[warp];
  float4 *sa = sa_[warp];
  float2 *sb = sb_[warp];
  uint32_t *sj = sj_[warp];
  unsigned short *smask = smask_[warp];
  float *red = red_[warp];
  const int lr = lane < 30 ? lane / 6 : 64, lc = lane % 6;  // record and moment a lane adds
  int *bins = reinterpret_cast<int *>(sa);
  const int nwarps = (int)gridDim.x * kWarps;
  const int64_t total = tile_start[ntiles];
  const int unit = unit_length(total, nwarps);
  const int per_task = ((int)tk.ctr[kCtrSegment] + unit - 1) / unit;  // units of a task
  const int64_t nunits = (int64_t)tk.ctr[kCtrTasks] * per_task;
  const bool spread = total > 3 * (int64_t)(ntiles / T) * M;
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
        u0[2] = g[h].y;
        u1[0] = g[h].z;
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
          float2 tot[6];
#pragma unroll
          for (int i = 0; i < 6; ++i) tot[i] = make_float2(0.f, 0.f);
          for (unsigned mm = smask[slot]; mm; mm &= mm - 1)
            block_moments(sg, __ffs(mm) - 1, x0, y0, A, Bv.x, Bv.y, nl2tau, tot);
          if (spread) {
            double *mo = mb + 6ull * sj[slot];
#pragma unroll
            for (int i = 0; i < 6; ++i) atomicAdd(mo + i, (double)(tot[i].x + tot[i].y));
          } else {
#pragma unroll
            for (int i = 0; i < 6; ++i) red[7 * lane + i] = tot[i].x + tot[i].y;
          }
        }
        if (spread) continue;
        __syncwarp();
        // six lanes add one record's six moments, five records at a time: the
        // warp's addresses then lie in five or so lines, not in 32
        const int left = min(32, nv - r0);
        const float *rp = red + 7 * lr + lc;
        const uint32_t *jp = sj + r0 + lr;
#pragma unroll
        for (int i = 0; i < 7; ++i)
          if (5 * i + lr < left) atomicAdd(mbl + 6ull * jp[5 * i], (double)rp[35 * i]);
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
                              const int64_t *tile_start, int64_t cap, int64_t M, int B, int d,
                              float l2tau, const float *dproj, double *mom, const RasterTasks &tk,
                              bool fresh, cudaStream_t st) {
  if (cfg < 0 || cfg >= bwd_config_count()) return cudaErrorInvalidValue;
  const BwdCfg &c = kBwdCfgs[cfg];
  if (!fresh) {  // the tasks stand; only the backward's counter starts again
    const cudaError_t e = cudaMemsetAsync(tk.ctr + kCtrBwd, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
  }
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
    // -e = z1^2 + (z2^2 - l2A), rounded as the tiled forms round it
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
