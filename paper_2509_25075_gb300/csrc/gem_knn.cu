// k nearest neighbours of the Gaussian centres.
//
// The isotropic-scaling ablation (Sec. 4, Design Choices of 3DGS for cryo-EM)
// sets S_j = s_j I with s_j the distance of Gaussian j to its nearest
// neighbour; the same distances serve as a scale initialisation.
//
// Uniform grid: the centres' bounding box is cut into about 3/2 M cubic cells
// (the centres cluster, so most cells are empty and the others hold several);
// a counting sort by cell puts the centres of a cell, and of the cells of a
// row along x, next to each other; each query walks Chebyshev rings of cells
// around its own until the k-th best distance is shorter than anything an
// unvisited ring can hold.  The result is exact: the k smallest
// (distance^2, index) pairs in lexicographic order, which does not depend on
// the order the candidates were met.
#include "gem_internal.cuh"

namespace gem {

constexpr int kKnnBlk = 256;
constexpr int kScanPer = 4096;  // elements per block of the cell-count scan

// Bounding box of the finite centres, and the grid over it.  Every block
// leaves its box in part[blk][6] = (min x, y, z, max x, y, z); the last one to
// finish folds them and picks the cell size: cubes of side h with about
// 3/2 M of them over the box, at most cap cells.
__global__ void __launch_bounds__(kKnnBlk) knn_bbox_kernel(const float *__restrict__ params,
                                                           int64_t M, float *__restrict__ part,
                                                           int64_t cap, int *__restrict__ ticket,
                                                           KnnGrid *__restrict__ g) {
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < M;
       j += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float v = params[j * kNpar + a];
      if (isfinite(v)) {
        lo[a] = fminf(lo[a], v);
        hi[a] = fmaxf(hi[a], v);
      }
    }
  }
  __shared__ float red[kKnnBlk / 32][6];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // box of the block: its threads', then its warps'
  auto fold = [&]() {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
        hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
      }
    if (lane == 0)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        red[warp][a] = lo[a];
        red[warp][3 + a] = hi[a];
      }
    __syncthreads();
  };
  fold();
  if (threadIdx.x < 6) {
    float v = red[0][threadIdx.x];
    for (int w = 1; w < kKnnBlk / 32; ++w)
      v = threadIdx.x < 3 ? fminf(v, red[w][threadIdx.x]) : fmaxf(v, red[w][threadIdx.x]);
    __stcg(part + blockIdx.x * 6 + threadIdx.x, v);
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kKnnBlk)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], __ldcg(part + b * 6 + a));
      hi[a] = fmaxf(hi[a], __ldcg(part + b * 6 + 3 + a));
    }
  fold();
  if (threadIdx.x != 0) return;
  *ticket = 0;  // as the next call expects it
  for (int w = 0; w < kKnnBlk / 32; ++w)
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], red[w][a]);
      hi[a] = fmaxf(hi[a], red[w][3 + a]);
    }
  float ext[3];
  for (int a = 0; a < 3; ++a) {
    if (!(lo[a] <= hi[a])) lo[a] = hi[a] = 0.f;  // no finite centre
    ext[a] = hi[a] - lo[a];
  }
  const float emax = fmaxf(ext[0], fmaxf(ext[1], ext[2]));
  const double target = fmax(1.0, 1.5 * (double)M);
  // side from the volume, kept above emax / 1024 so flat or linear sets of
  // centres do not make the grid explode
  double h = cbrt(fmax((double)ext[0] * ext[1] * ext[2], 0.0) / target);
  h = fmax(h, (double)emax / 1024.0);
  if (!(h > 0.0)) h = 1.0;
  int n[3] = {1, 1, 1};
  bool fits = false;
  for (int it = 0; it < 1024 && !fits; ++it) {
    double cells = 1.0;
    for (int a = 0; a < 3; ++a) {
      double na = floor(ext[a] / h) + 1.0;
      n[a] = na < 1.0e6 ? (int)na : 1000000;
      cells *= n[a];
    }
    fits = cells <= (double)cap;
    // no set of centres needs more than the cube root of the excess; flat and
    // linear ones come closer step by step
    if (!fits) h *= fmax(1.1, cbrt(cells / (double)cap));
  }
  if (!fits || !(h > 0.0) || !isfinite(h)) {  // absurd coordinates: one cell holds all
    n[0] = n[1] = n[2] = 1;
    h = 1.0e30;
  }
  for (int a = 0; a < 3; ++a) g->lo[a] = lo[a];
  g->h = (float)h;
  g->ih = (float)(1.0 / h);
  for (int a = 0; a < 3; ++a) g->n[a] = n[a];
  g->ncell = n[0] * n[1] * n[2];
}

__device__ __forceinline__ int knn_axis_cell(float v, float lo, float ih, int n) {
  int c = (int)floorf((v - lo) * ih);
  return min(max(c, 0), n - 1);
}

// Cell of every centre (non-finite centres go to cell 0 and are never
// reported as neighbours), its place among the cell's members, and per-cell
// counts.
__global__ void __launch_bounds__(kKnnBlk) knn_cell_kernel(const float *__restrict__ params,
                                                           int64_t M,
                                                           const KnnGrid *__restrict__ g,
                                                           int *__restrict__ cell,
                                                           int *__restrict__ rank,
                                                           int *__restrict__ cnt) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const KnnGrid G = *g;
  const float *p = params + j * kNpar;
  int c = 0;
  if (isfinite(p[0]) && isfinite(p[1]) && isfinite(p[2])) {
    int cx = knn_axis_cell(p[0], G.lo[0], G.ih, G.n[0]);
    int cy = knn_axis_cell(p[1], G.lo[1], G.ih, G.n[1]);
    int cz = knn_axis_cell(p[2], G.lo[2], G.ih, G.n[2]);
    c = (cz * G.n[1] + cy) * G.n[0] + cx;
  }
  cell[j] = c;
  rank[j] = atomicAdd(cnt + c, 1);
}

// Exclusive scan of cnt[0 .. ncell) into start (start[ncell] = total), in
// three steps: block sums, scan of the block sums, block scans.
__global__ void __launch_bounds__(1024) knn_scan_sums_kernel(const int *__restrict__ cnt,
                                                             const KnnGrid *__restrict__ g,
                                                             int *__restrict__ bsum) {
  const int n = g->ncell;
  const int64_t base = (int64_t)blockIdx.x * kScanPer;
  int s = 0;
  for (int i = threadIdx.x; i < kScanPer; i += 1024)
    if (base + i < n) s += cnt[base + i];
  s = __reduce_add_sync(0xffffffffu, s);
  __shared__ int ws[32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    int v = __reduce_add_sync(0xffffffffu, ws[threadIdx.x]);
    if (threadIdx.x == 0) bsum[blockIdx.x] = v;
  }
}

__device__ __forceinline__ int block_exclusive_scan(int v, int *ws, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int w = ws[lane], wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int u = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += u;
    }
    ws[lane] = wi - w;
    if (lane == 31) ws[32] = wi;
  }
  __syncthreads();
  int r = ws[warp] + inc - v;
  total = ws[32];
  __syncthreads();
  return r;
}

// bsum[0 .. nb) becomes its exclusive scan; bsum[nb] = the total.
__global__ void __launch_bounds__(1024) knn_scan_top_kernel(int *__restrict__ bsum, int nb) {
  __shared__ int ws[33];
  int carry = 0;
  for (int base = 0; base < nb; base += 1024) {
    int i = base + threadIdx.x;
    int v = i < nb ? bsum[i] : 0;
    int tot;
    int ex = block_exclusive_scan(v, ws, tot);
    if (i < nb) bsum[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) bsum[nb] = carry;
}

__global__ void __launch_bounds__(1024) knn_scan_blocks_kernel(const int *__restrict__ cnt,
                                                               const KnnGrid *__restrict__ g,
                                                               const int *__restrict__ bsum,
                                                               int *__restrict__ start) {
  __shared__ int ws[33];
  const int n = g->ncell;
  const int64_t base = (int64_t)blockIdx.x * kScanPer;
  int carry = bsum[blockIdx.x];
  // 4 elements per thread, in order
  const int64_t i0 = base + 4 * threadIdx.x;
  int v[4], s = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = (i0 + k < n) ? cnt[i0 + k] : 0;
    s += v[k];
  }
  int tot;
  int ex = block_exclusive_scan(s, ws, tot) + carry;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i0 + k < n) start[i0 + k] = ex;
    ex += v[k];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) start[n] = bsum[gridDim.x];
}

// The centres in cell order, each with its index: one coalesced 16-byte load
// per candidate instead of a gather of its parameter row.
__global__ void __launch_bounds__(kKnnBlk) knn_scatter_kernel(const float *__restrict__ params,
                                                              const int *__restrict__ cell,
                                                              const int *__restrict__ rank,
                                                              const int *__restrict__ start,
                                                              int64_t M, float4 *__restrict__ sorted) {
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  const float *p = params + j * kNpar;
  sorted[start[cell[j]] + rank[j]] = make_float4(p[0], p[1], p[2], __int_as_float((int)j));
}

// Squared distance without contraction into FMA, so that it is the same
// number whatever the compiler does.
__device__ __forceinline__ float dist2_rn(float ax, float ay, float az, float bx, float by,
                                          float bz) {
  float dx = __fsub_rn(ax, bx), dy = __fsub_rn(ay, by), dz = __fsub_rn(az, bz);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// The k best (distance^2, index) pairs, ascending in lexicographic order.
template <int K>
struct KBest {
  float d[K];
  int i[K];
  __device__ __forceinline__ void fill(float dist, int index) {
#pragma unroll
    for (int m = 0; m < K; ++m) {
      d[m] = dist;
      i[m] = index;
    }
  }
  // A non-finite candidate's squared distance is infinite or not a number:
  // it is never below d[K - 1], nor equal to it with an index below -1.
  __device__ __forceinline__ bool takes(float d2, int j) const {
    return d2 < d[K - 1] || (d2 == d[K - 1] && j < i[K - 1]);
  }
  __device__ __forceinline__ void insert(float d2, int j) {
    // from the end, each slot takes its left neighbour while the newcomer
    // sorts before it, else the newcomer if it sorts before the slot
#pragma unroll
    for (int m = K - 1; m > 0; --m) {
      const bool before_left = d2 < d[m - 1] || (d2 == d[m - 1] && j < i[m - 1]);
      const bool before_here = d2 < d[m] || (d2 == d[m] && j < i[m]);
      if (before_left) {
        d[m] = d[m - 1];
        i[m] = i[m - 1];
      } else if (before_here) {
        d[m] = d2;
        i[m] = j;
      }
    }
    if (d2 < d[0] || (d2 == d[0] && j < i[0])) {
      d[0] = d2;
      i[0] = j;
    }
  }
  // The best k over the lanes' lists, which hold no index twice (but for the
  // placeholders, which come last), left in every lane.  Distances are not
  // negative, so their bits order as they do.
  __device__ __forceinline__ void merge_warp() {
    KBest<K> all;
#pragma unroll
    for (int m = 0; m < K; ++m) {
      const unsigned mine = __float_as_uint(d[0]);
      const unsigned bd = __reduce_min_sync(0xffffffffu, mine);
      const unsigned bi = __reduce_min_sync(0xffffffffu, mine == bd ? (unsigned)i[0] : 0xffffffffu);
      all.d[m] = __uint_as_float(bd);
      all.i[m] = (int)bi;
      if (mine == bd && (unsigned)i[0] == bi) {  // this lane's head was the best: drop it
#pragma unroll
        for (int q = 0; q + 1 < K; ++q) {
          d[q] = d[q + 1];
          i[q] = i[q + 1];
        }
        d[K - 1] = INFINITY;
        i[K - 1] = -1;
      }
    }
    *this = all;
  }
};

// Looks at the sorted centres qs .. qe - 1 for query (p, i).
template <int K>
__device__ __forceinline__ void knn_visit(KBest<K> &best, const float4 *__restrict__ sorted, int qs,
                                          int qe, const float4 &p, int i) {
  for (int q = qs; q < qe; ++q) {
    const float4 c = sorted[q];
    const float d2 = dist2_rn(p.x, p.y, p.z, c.x, c.y, c.z);
    const int j = __float_as_int(c.w);
    if (best.takes(d2, j) && j != i) best.insert(d2, j);
  }
}

// One thread per centre, in cell order, for its cell and the 26 around it:
// neighbouring threads read the same cells, and the cells of a row along x
// are one run of the sorted centres.  A centre that needs further rings of
// cells walks them in its thread as long as enough of its warp's lanes do; the
// last ones (those in the thin outskirts of the clusters, whose rings hold
// hundreds of mostly empty rows) are finished by the whole warp, one after the
// other, a row per lane: a thread walking them alone is a chain of dependent
// loads.
//
// The line between the two: a ring costs a thread its rows, and the warp about
// 2 + K / 4 + rows / 32 rows' time (the merge of the lanes' lists grows with K)
// for each centre.  With the warp from the second ring on, sets whose centres
// mostly need it (several neighbours, flat sets) waited for 32 searches in a
// row; with constants half and twice these, times are the same within 10% but
// for a few sets.
//
// Bound by the latency of the loads at k = 1, by insertions at k = 16, which
// wait for each other: as many CTAs per SM as the lists leave registers for
// (three instead of four at k = 8: 583 us, not 426, below).
// Calls of M = 300000, us, with one thread per centre, a gather of the
// parameter row per candidate and two bounds per cell; with sorted centres,
// rows, 3/2 M cells and the warp from the second ring on; now:  64 clusters,
// k = 1: 402, 145, 129; k = 4: 626, 486, 245; k = 8: 918, 1034, 426; k = 16: 1743,
// 5889, 1075.  A plane, k = 1: 138, 109, 74; k = 16: 533, 4787, 443.  Uniform,
// k = 8: 559, 854, 233.
template <int K>
__global__ void __launch_bounds__(kKnnBlk, K > 8 ? 3 : K > 4 ? 4 : 5) knn_query_kernel(
    const float4 *__restrict__ sorted, int64_t M, const KnnGrid *__restrict__ g,
    const int *__restrict__ start, float *__restrict__ dist, int32_t *__restrict__ idx) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const KnnGrid G = *g;
  const int n0 = G.n[0], n1 = G.n[1], n2 = G.n[2];
  const int rmax = max(n0, max(n1, n2));
  float4 me = make_float4(0.f, 0.f, 0.f, 0.f);
  if (t < M) me = sorted[t];
  const int i = __float_as_int(me.w);
  KBest<K> best;
  best.fill(INFINITY, -1);
  const bool fin = t < M && isfinite(me.x) && isfinite(me.y) && isfinite(me.z);
  bool done = !fin;
  // everything in rings beyond r lies farther than r * h from the point
  auto enough = [&](const KBest<K> &b, int r) {
    const float reach = (float)r * G.h * (1.f - 1e-4f);
    return b.i[K - 1] >= 0 && b.d[K - 1] <= reach * reach;
  };
  if (fin) {
    const int cx = knn_axis_cell(me.x, G.lo[0], G.ih, n0);
    const int cy = knn_axis_cell(me.y, G.lo[1], G.ih, n1);
    const int cz = knn_axis_cell(me.z, G.lo[2], G.ih, n2);
    const int x0 = max(cx - 1, 0), x1 = min(cx + 1, n0 - 1) + 1;
    if constexpr (K == 1) {
      int qs[9], qe[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const int z = cz + q / 3 - 1, y = cy + q % 3 - 1;
        qs[q] = qe[q] = 0;
        if (z >= 0 && z < n2 && y >= 0 && y < n1) {
          const int *row = start + ((int64_t)z * n1 + y) * n0;
          qs[q] = row[x0];
          qe[q] = row[x1];
        }
      }
#pragma unroll
      for (int q = 0; q < 9; ++q) knn_visit(best, sorted, qs[q], qe[q], me, i);
    } else {
      // many neighbours: the runs in a loop, whose body is the insertion of K
      // compares (nine copies of it do not fit the instruction cache), the own
      // cell first, whose centres are the likeliest to stay in the list; the
      // next run's bounds are loaded meanwhile
      auto bounds = [&](int h, int &qs, int &qe) {
        const int q = h < 3 ? 4 : h < 7 ? h - 3 : h - 2;  // the own row is in three runs
        const int z = cz + q / 3 - 1, y = cy + q % 3 - 1;
        qs = qe = 0;
        if (z >= 0 && z < n2 && y >= 0 && y < n1) {
          const int *row = start + ((int64_t)z * n1 + y) * n0;
          qs = row[h == 0 ? cx : h == 2 ? cx + 1 : x0];
          qe = row[h == 0 ? cx + 1 : h == 1 ? cx : x1];
        }
      };
      int ns, ne;
      bounds(0, ns, ne);
#pragma unroll 1
      for (int h = 0; h < 11; ++h) {
        const int qs = ns, qe = ne;
        if (h < 10) bounds(h + 1, ns, ne);
        knn_visit(best, sorted, qs, qe, me, i);
      }
    }
    done = enough(best, 1) || rmax <= 1;
  }
  // row (z, y) of ring r about cell (cx, cy, cz), cut off at the grid's faces;
  // the inner rows of a ring hold only its two end cells
  auto visit_row = [&](KBest<K> &b, const float4 &p, int pi, int cx, int cy, int cz, int r, int z, int y) {
    const int *row = start + ((int64_t)z * n1 + y) * n0;
    const bool face = z == cz - r || z == cz + r || y == cy - r || y == cy + r;
    const int a = cx - r, c = cx + r;  // the run a .. c, or the cells a and c
    int qs = 0, qe = 0, rs = 0, re = 0;
    if (face || a >= 0) {
      qs = row[max(a, 0)];
      qe = row[face ? min(c, n0 - 1) + 1 : a + 1];
    }
    if (!face && c < n0) {
      rs = row[c];
      re = row[c + 1];
    }
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      knn_visit(b, sorted, qs, qe, p, pi);
      qs = rs;
      qe = re;
    }
  };
  int r0 = 2;
  unsigned todo;
  for (; (todo = __ballot_sync(0xffffffffu, !done)) != 0u; ++r0) {
    const int cx = knn_axis_cell(me.x, G.lo[0], G.ih, n0);
    const int cy = knn_axis_cell(me.y, G.lo[1], G.ih, n1);
    const int cz = knn_axis_cell(me.z, G.lo[2], G.ih, n2);
    const int z0 = max(cz - r0, 0), z1 = min(cz + r0, n2 - 1);
    const int y0 = max(cy - r0, 0), y1 = min(cy + r0, n1 - 1);
    const int rows = __reduce_max_sync(0xffffffffu, done ? 0 : (z1 - z0 + 1) * (y1 - y0 + 1));
    if (__popc(todo) * (2 + K / 4 + rows / 32) < rows) break;
    if (!done) {
      for (int z = z0; z <= z1; ++z)
        for (int y = y0; y <= y1; ++y) visit_row(best, me, i, cx, cy, cz, r0, z, y);
      done = enough(best, r0) || r0 >= rmax;
    }
  }
  for (; todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1;
    float4 p;
    p.x = __shfl_sync(0xffffffffu, me.x, src);
    p.y = __shfl_sync(0xffffffffu, me.y, src);
    p.z = __shfl_sync(0xffffffffu, me.z, src);
    const int pi = __shfl_sync(0xffffffffu, i, src);
    const int cx = knn_axis_cell(p.x, G.lo[0], G.ih, n0);
    const int cy = knn_axis_cell(p.y, G.lo[1], G.ih, n1);
    const int cz = knn_axis_cell(p.z, G.lo[2], G.ih, n2);
    // lane src starts from what it has, the others from placeholders at its
    // k-th distance, which sort behind every centre that close
    KBest<K> b = best;
    for (int r = r0; r <= rmax; ++r) {
      const float kth = __shfl_sync(0xffffffffu, b.d[K - 1], src);
      const int none = kth < INFINITY ? 0x7fffffff : -1;
      if (lane != src) b.fill(kth, none);
      const int z0 = max(cz - r, 0), z1 = min(cz + r, n2 - 1);
      const int y0 = max(cy - r, 0), y1 = min(cy + r, n1 - 1);
      const int ny = y1 - y0 + 1, rows = (z1 - z0 + 1) * ny;
      for (int q = lane; q < rows; q += 32) {
        const int dz = q / ny;
        visit_row(b, p, pi, cx, cy, cz, r, z0 + dz, y0 + (q - dz * ny));
      }
      __syncwarp();
      if (__any_sync(0xffffffffu, lane != src && b.i[0] != none)) b.merge_warp();
      if (__any_sync(0xffffffffu, lane == src && enough(b, r))) break;
    }
    if (lane == src) best = b;
  }
  if (t >= M) return;
#pragma unroll
  for (int m = 0; m < K; ++m) {
    dist[(int64_t)i * K + m] = best.i[m] >= 0 ? sqrtf(best.d[m]) : INFINITY;
    if (idx) idx[(int64_t)i * K + m] = best.i[m];
  }
}

// One instance per k, so that the k best live in registers.
template <int K>
void launch_query(int k, unsigned gm, cudaStream_t st, const float4 *sorted, int64_t M,
                  const KnnGrid *g, const int *start, float *dist, int32_t *idx) {
  if (k == K)
    knn_query_kernel<K><<<gm, kKnnBlk, 0, st>>>(sorted, M, g, start, dist, idx);
  else if constexpr (K < 16)
    launch_query<K + 1>(k, gm, st, sorted, M, g, start, dist, idx);
}

int knn_scan_blocks(int64_t cap) { return (int)((cap + kScanPer - 1) / kScanPer); }

cudaError_t launch_knn(const float *params, int64_t M, int k, const KnnScratch &s, float *dist,
                       int32_t *idx, cudaStream_t st) {
  cudaError_t e;
  const int64_t nbl = (M + kKnnBlk - 1) / kKnnBlk;
  const int nbb = (int)(nbl < 608 ? nbl : 608);  // KnnScratch::part holds 608 boxes
  knn_bbox_kernel<<<nbb, kKnnBlk, 0, st>>>(params, M, s.part, s.cap, s.ticket, s.grid);
  if ((e = cudaMemsetAsync(s.cnt, 0, (size_t)s.cap * sizeof(int), st)) != cudaSuccess) return e;
  const unsigned gm = (unsigned)((M + kKnnBlk - 1) / kKnnBlk);
  knn_cell_kernel<<<gm, kKnnBlk, 0, st>>>(params, M, s.grid, s.cell, s.rank, s.cnt);
  const int nb = knn_scan_blocks(s.cap);
  knn_scan_sums_kernel<<<nb, 1024, 0, st>>>(s.cnt, s.grid, s.bsum);
  knn_scan_top_kernel<<<1, 1024, 0, st>>>(s.bsum, nb);
  knn_scan_blocks_kernel<<<nb, 1024, 0, st>>>(s.cnt, s.grid, s.bsum, s.start);
  knn_scatter_kernel<<<gm, kKnnBlk, 0, st>>>(params, s.cell, s.rank, s.start, M, s.sorted);
  launch_query<1>(k, gm, st, s.sorted, M, s.grid, s.start, dist, idx);
  return cudaGetLastError();
}

}  // namespace gem
