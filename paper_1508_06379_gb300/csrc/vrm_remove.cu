// Particle removal (the outlook of Sec. 6.2): where particles have come closer
// than r h to one another, the one with the smaller key (|Gamma|, index) of
// such a pair is redistributed to its kept neighbours by non-negative
// weights that reproduce the identity's moments of order 0 and 1 (sum g = 1,
// sum g r = 0; the weights come from k_lp_identity in vrm_lp.cu) and removed.
//
//   k_close          candidate flags and the largest neighbour count, one scan
//                    of the 3 x 3 cells (FP32 prefilter on cell-local
//                    coordinates, the FP64 definition dx*dx + dy*dy < (r h)^2,
//                    or <= (R h)^2, for the undecided pairs)
//   k_remove_link    the removed particles' entries (target, weight) in a list
//                    per target
//   k_remove_apply   Gamma_j + sum_i g_ij Gamma_i for every kept j, its entries
//                    sorted by i; no floating-point atomics
//   k_remove_out     the kept particles compacted in index order
// Only the candidates (a tenth of a crowded cloud) are searched for their
// closest non-candidates, and only targets with entries gather anything.  1.1
// million particles with 113,000 candidates: the scan for flags and counts 80
// us, the candidates' search 75, their LPs 101, the entries 25; it was 55 us for
// the flags alone, 315 for sorted rows of all particles, 140 for LPs that chose
// their columns from rows, 72 to look every row through.
#include <climits>

#include "vrm_internal.cuh"

namespace vrm {

// |Gamma| as bits (non-negative: the bit order is the value order).
__device__ __forceinline__ unsigned long long abs_key(double g) {
  return (unsigned long long)__double_as_longlong(g) & 0x7FFFFFFFFFFFFFFFull;
}

__global__ void __launch_bounds__(kBlock) k_close(Consts c, const Grid* __restrict__ gp,
                                                  const int* __restrict__ cell_start,
                                                  const double2* __restrict__ sxy, const float2* __restrict__ sloc,
                                                  const int* __restrict__ sidx, int n,
                                                  const double* __restrict__ gamma, uint8_t* __restrict__ close,
                                                  DevStats* __restrict__ ds) {
  const Grid g = *gp;
  int most = 0;
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (long)gridDim.x * blockDim.x) {
    const int i = sidx[p];
    const double2 pi = sxy[p];
    const float2 li = sloc[p];
    const int cx = grid_cell_x(g, pi.x), cy = grid_cell_y(g, pi.y);
    const unsigned long long ai = abs_key(gamma[i]);
    bool cl = false;
    int cnt = 0;
    for (int by = cy - 1; by <= cy + 1; ++by) {
      if (by < 0 || by >= g.ny) continue;
      const float dvb = (float)(by - cy) - li.y;
      for (int bx = cx - 1; bx <= cx + 1; ++bx) {
        if (bx < 0 || bx >= g.nx) continue;
        const float dub = (float)(bx - cx) - li.x;
        const int cell = by * g.nx + bx;
        const int q0 = cell_start[cell], q1 = cell_start[cell + 1];
        for (int q = q0; q < q1; ++q) {
          const float2 lj = sloc[q];
          const float du = dub + lj.x, dv = dvb + lj.y;
          const float d2f = __fmaf_rn(du, du, dv * dv);
          if (d2f > g.hi_out) continue;
          if (d2f > g.lo_in && d2f < g.hi_in) {
            ++cnt;
            continue;
          }
          const int j = sidx[q];
          if (j == i) continue;
          bool in = d2f < g.lo_out;  // certainly closer than r h
          if (!in) {
            const double2 pj = sxy[q];
            const double d2 = dist2(__dsub_rn(pj.x, pi.x), __dsub_rn(pj.y, pi.y));
            in = d2 < c.lo2;
            if (!in && d2 <= c.hi2) ++cnt;
          }
          if (!in || cl) continue;
          const unsigned long long aj = abs_key(gamma[j]);
          cl = ai < aj || (ai == aj && i < j);
        }
      }
    }
    most = cnt > most ? cnt : most;
    close[i] = cl ? 1 : 0;
  }
  // one atomic per block
  __shared__ int w_most[kBlock / 32];
  most = (int)__reduce_max_sync(0xffffffffu, (unsigned)most);
  if ((threadIdx.x & 31) == 0) w_most[threadIdx.x >> 5] = most;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kBlock / 32; ++w) most = w_most[w] > most ? w_most[w] : most;
    if (most > 0) atomicMax(&ds->max_count, most);
  }
}

// Entry 4 i + slot of every removed i into the list of its target (any order).
__global__ void __launch_bounds__(kBlock) k_remove_link(const int* __restrict__ clist, const int* __restrict__ n_cand,
                                                        const uint8_t* __restrict__ removed,
                                                        const int* __restrict__ cols4, int* __restrict__ head,
                                                        int* __restrict__ next) {
  const int m = *n_cand;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (long)gridDim.x * blockDim.x) {
    const int i = clist[t];
    if (!removed[i]) continue;
    const int4 cc = reinterpret_cast<const int4*>(cols4)[i];
    const int col[4] = {cc.x, cc.y, cc.z, cc.w};
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (col[s] >= 0) next[4 * (long)i + s] = atomicExch(&head[col[s]], 4 * i + s);
  }
}

__global__ void __launch_bounds__(kBlock) k_remove_apply(int n, int k_cap, const double* __restrict__ gamma,
                                                         const uint8_t* __restrict__ removed,
                                                         const double* __restrict__ w4, const int* __restrict__ head,
                                                         const int* __restrict__ next, double* __restrict__ gnew,
                                                         uint8_t* __restrict__ keep, DevStats* __restrict__ ds) {
  for (long j = (long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (long)gridDim.x * blockDim.x) {
    const double gj = gamma[j];
    if ((__double_as_longlong(gj) & 0x7FF0000000000000LL) == 0x7FF0000000000000LL) atomicOr(&ds->nonfinite, 1);
    const bool gone = removed[j] != 0;
    keep[j] = gone ? 0 : 1;
    if (gone) continue;
    // the list's entries in ascending order (the sources differ, so that is
    // the sources' order): the smallest one above the last, a few times.  The
    // sources are neighbours of j, so a list beyond k_cap belongs to a call that
    // ends in the capacity error: it is left alone at its k_cap-th entry (a spot
    // of 20,000 particles puts most of them in one list, 4e8 dependent loads of
    // one thread)
    double acc = gj;
    const int first = head[j];
    if (first >= 0 && next[first] < 0) {  // one entry: most targets that have any
      acc = __dadd_rn(acc, __dmul_rn(w4[first], gamma[first >> 2]));
    } else {
      for (int last = -1; first >= 0;) {
        int best = INT_MAX, seen = 0;
        for (int e = first; e >= 0 && seen <= k_cap; e = next[e], ++seen)
          if (e > last && e < best) best = e;
        if (best == INT_MAX || seen > k_cap) break;
        acc = __dadd_rn(acc, __dmul_rn(w4[best], gamma[best >> 2]));
        last = best;
      }
    }
    gnew[j] = acc;
  }
}

__global__ void __launch_bounds__(kBlock) k_remove_out(const int* __restrict__ n_keep, const int* __restrict__ klist,
                                                       const double* __restrict__ x, const double* __restrict__ y,
                                                       const double* __restrict__ gnew, double* __restrict__ x_out,
                                                       double* __restrict__ y_out, double* __restrict__ g_out) {
  const int m = *n_keep;
  for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (long)gridDim.x * blockDim.x) {
    const int i = klist[k];
    x_out[k] = x[i];
    y_out[k] = y[i];
    g_out[k] = gnew[i];
  }
}

namespace {
int blocks_for(int n) {
  long b = ((long)n + kBlock - 1) / kBlock;
  if (b > 8L * sm_count()) b = 8L * sm_count();
  return b < 1 ? 1 : (int)b;
}
}  // namespace

cudaError_t remove_close_flags(const Consts& c, const Grid* g, const int* cell_start, const double2* sorted_xy,
                               const float2* sorted_loc, const int* sorted_idx, int n, const double* gamma,
                               uint8_t* close, DevStats* ds, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_close<<<blocks_for(n), kBlock, 0, s>>>(c, g, cell_start, sorted_xy, sorted_loc, sorted_idx, n, gamma, close, ds);
  note_launch();
  return cudaGetLastError();
}

cudaError_t remove_apply(const Consts& c, const int* clist, const int* n_cand, int n, const double* gamma,
                         const uint8_t* removed, const int* cols4, const double* w4, int* head, int* next,
                         double* gnew, uint8_t* keep, DevStats* ds, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const cudaError_t e = cudaMemsetAsync(head, 0xFF, sizeof(int) * (size_t)n, s);
  if (e != cudaSuccess) return e;
  k_remove_link<<<blocks_for(n), kBlock, 0, s>>>(clist, n_cand, removed, cols4, head, next);
  note_launch();
  k_remove_apply<<<blocks_for(n), kBlock, 0, s>>>(n, c.k_cap, gamma, removed, w4, head, next, gnew, keep, ds);
  note_launch();
  return cudaGetLastError();
}

cudaError_t remove_out(int n, const int* n_keep, const int* klist, const double* x, const double* y,
                       const double* gnew, double* x_out, double* y_out, double* g_out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_remove_out<<<blocks_for(n), kBlock, 0, s>>>(n_keep, klist, x, y, gnew, x_out, y_out, g_out);
  note_launch();
  return cudaGetLastError();
}

}  // namespace vrm
