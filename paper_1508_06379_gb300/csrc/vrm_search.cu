// Annulus neighbourhoods (Sec. 2, Eq. neighbourhood), 45-degree segment
// masks (Sec. 4.2) and small neighbourhoods (Sec. 4.3) on the cell grid.
//
// One thread per particle, taken in cell order so that the threads of a warp
// read overlapping cells.  Each thread scans the 3 x 3 cells around its own.
// The annulus test of the method is the FP64 definition
//   lo2 <= dx*dx + dy*dy <= hi2,  dx = x_j - x_i,  dy = y_j - y_i,
// every operation rounded separately.  GB300 runs FP64 at 1/60 of its FP32
// rate, so each pair is measured in FP32 on cell-local coordinates (error
// below 1e-5 cell^2): a pair further than the band from both bounds is
// decided in FP32; segments are decided in FP32 unless the offset lies within
// seg_eps of a decision line; the closest member of a segment is chosen in
// FP32 unless another member lies within two bands of it.  Only the
// undecided cases (rare on jittered clouds, frequent on exact lattices) take
// the FP64 definition, so the result is bit-identical to it.
//
// Rows (k_cap apart) are sorted by index for the library's neighbourhood
// calls: the members are collected in shared memory in visiting order and
// sorted in registers by an odd-even merge network of 16, 24 or 32 (a sorted
// insertion per member in local memory doubled the kernel: 205 us for 393,000
// particles, 131 this way; 80 registers and 48 KB a block, three blocks per SM:
// two take 158 us and four 148 before the rows went out as vectors, three 141); a row that overflows keeps the row_cap smallest
// indices.  The step's form over the diffused list (LIST) writes members
// straight to the row in visiting order and cuts it at row_cap: the step then
// repeats with whole rows or reports the capacity error.  The closest particle of every segment is tracked in shared memory
// with ties to the smaller index.
#include <climits>

#include "vrm_internal.cuh"
#include "vrm_smem.cuh"

namespace vrm {

// Exact member test and segment of one candidate pair, for the rare pairs
// the FP32 measure cannot decide.  Returns the segment, or -1 if j is not in
// the annulus of i.
__device__ __forceinline__ int exact_member(const Consts& c, const double2& pi, const double2& pj, bool certain_in,
                                            double* d2_out) {
  const double dx = __dsub_rn(pj.x, pi.x), dy = __dsub_rn(pj.y, pi.y);
  const double d2 = dist2(dx, dy);
  *d2_out = d2;
  if (!certain_in && (d2 < c.lo2 || d2 > c.hi2)) return -1;
  return segment_of(dx, dy);
}

// Small neighbourhood bookkeeping: per segment the smallest FP32 squared
// distance and its particle, and a flag `amb` set when another member of
// the segment lies within 2 bands of it (then the FP32 order may differ from
// the FP64 order, and a second pass decides that segment exactly).
//
// LIST = true: only the particles of `list` (list_count of them; the step's
// diffused set, the only particles whose rows the step reads), each located
// in the sorted arrays through its cell key and rank; threads follow the
// list's order.  Rows are then padded with -1 to the end of their last
// 32-byte sector, so that the sector is written whole.
// ROWS = false (list form only): the rows are not written (the count, mask
// and small neighbourhood are).  skip (list form, optional): flagged particles
// are not members (SKIP).
// Comparators of Batcher's odd-even merge sort of the next power of two, those
// past N left out (entries there would be the largest).
template <int N>
struct SortNet {
  int n = 0;
  unsigned char a[256] = {}, b[256] = {};
  constexpr SortNet() {
    const int P = N <= 16 ? 16 : 32;
    for (int p = 1; p < P; p <<= 1)
      for (int k = p; k >= 1; k >>= 1)
        for (int j = k % p; j + k < P; j += 2 * k)
          for (int i = 0; i < k; ++i)
            if (i + j + k < N && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
              a[n] = (unsigned char)(i + j);
              b[n] = (unsigned char)(i + j + k);
              ++n;
            }
  }
};
template <int N>
__device__ __forceinline__ void sort_row(int (&v)[N]) {
  constexpr SortNet<N> net;
#pragma unroll
  for (int t = 0; t < net.n; ++t) {
    const int x = v[net.a[t]], y = v[net.b[t]];
    v[net.a[t]] = x < y ? x : y;
    v[net.b[t]] = x < y ? y : x;
  }
}
// The m <= N entries of a thread's list (stride nb) sorted into its row.
template <int N>
__device__ __forceinline__ void write_sorted_row(const int* list, int nb, int m, int* __restrict__ row) {
  int v[N];
#pragma unroll
  for (int t = 0; t < N; ++t) v[t] = t < m ? list[t * nb] : INT_MAX;
  sort_row<N>(v);
  const bool whole = ((uintptr_t)row & 15u) == 0;  // (k_cap may be any number)
#pragma unroll
  for (int t = 0; t < N; t += 4) {
    if (whole && t + 4 <= m) {
      *reinterpret_cast<int4*>(row + t) = make_int4(v[t], v[t + 1], v[t + 2], v[t + 3]);
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u < m) row[t + u] = v[t + u];
    }
  }
}

// (The list forms want 64 registers, four blocks per SM: 184 us for 696,000
// particles, 261 at the 80 the compiler takes by itself.)
template <int KCAP, bool LIST = false, bool ROWS = true, bool SKIP = false>
__global__ void __launch_bounds__(kBlock, LIST ? 4 : 3) k_search_all(Consts c, const Grid* __restrict__ gp,
                                                       const int* __restrict__ cell_start,
                                                       const double2* __restrict__ sxy,
                                                       const float2* __restrict__ sloc,
                                                       const int* __restrict__ sidx, int n,
                                                       const int* __restrict__ n_dev,
                                                       int* __restrict__ nbr_count, int* __restrict__ nbr_idx,
                                                       uint8_t* __restrict__ seg_mask, int* __restrict__ small,
                                                       DevStats* __restrict__ ds,
                                                       const int* __restrict__ list = nullptr,
                                                       const int* __restrict__ cell_key = nullptr,
                                                       const int* __restrict__ cell_rank = nullptr,
                                                       const uint8_t* __restrict__ skip = nullptr) {
  if (n_dev) n = *n_dev;
  const Grid g = *gp;
  const int k_cap = c.row_cap < KCAP ? c.row_cap : KCAP;  // entries kept
  const size_t stride = (size_t)c.k_cap;
  const float tie = 2.f * kBand;
  int local_max = 0;
  // closest member of every segment so far (FP32 squared distance, index),
  // one column per thread: read and written with a dynamic segment index
  // (conflict-free: the row stride, the block size, is a multiple of 32
  // words).  Sized by the launch (8 + 8 words per thread), so that a small
  // block leaves the rest of the SM's shared memory to L1.
  extern __shared__ int s_search[];
  const int nb = blockDim.x;
  float* const s_bf = reinterpret_cast<float*>(s_search);
  int* const s_bj = s_search + 8 * nb;
  const int tx = threadIdx.x;
  int* const row_list = s_search + 16 * nb + tx;  // !LIST: the members so far, entry t at t nb
  for (long t0 = (long)blockIdx.x * blockDim.x + threadIdx.x; t0 < n; t0 += (long)gridDim.x * blockDim.x) {
    int i, cx, cy;
    long p;
    if (LIST) {
      i = list[t0];
      const int key = cell_key[i];
      p = cell_start[key] + cell_rank[i];
      cy = key / g.nx;
      cx = key - cy * g.nx;
    } else {
      p = t0;
      i = sidx[p];
    }
    const double2 pi = sxy[p];
    const float2 li = sloc[p];
    if (!LIST) {
      cx = grid_cell_x(g, pi.x);
      cy = grid_cell_y(g, pi.y);
    }
    // LIST: members go straight to the row in visiting order (a row longer
    // than row_cap is cut; the step then repeats with whole rows or reports
    // the capacity error, so no smallest-index rule is needed); otherwise
    // they are collected in shared memory first
    int* const row_out = nbr_idx + (size_t)i * stride;
    int cnt = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      s_bf[t * nb + tx] = 3e38f;
      s_bj[t * nb + tx] = -1;
    }
    unsigned mask = 0, amb = 0;
    for (int by = cy - 1; by <= cy + 1; ++by) {
      if (by < 0 || by >= g.ny) continue;
      const float dvb = (float)(by - cy) - li.y;
      for (int bx = cx - 1; bx <= cx + 1; ++bx) {
        if (bx < 0 || bx >= g.nx) continue;
        const float dub = (float)(bx - cx) - li.x;
        const int cell = by * g.nx + bx;
        const int q0 = cell_start[cell], q1 = cell_start[cell + 1];
        // the next candidate's coordinates and index are loaded while this
        // one is tested (the loop is bound by load latency)
        float2 lnext = q0 < q1 ? sloc[q0] : make_float2(0.f, 0.f);
        int jnext = q0 < q1 ? sidx[q0] : 0;
        for (int q = q0; q < q1; ++q) {
          const float2 lj = lnext;
          const int j = jnext;
          if (q + 1 < q1) {
            lnext = sloc[q + 1];
            jnext = sidx[q + 1];
          }
          const float du = dub + lj.x, dv = dvb + lj.y;
          const float d2f = __fmaf_rn(du, du, dv * dv);
          if (d2f < g.lo_out || d2f > g.hi_out) continue;
          if (j == i) continue;
          if (SKIP && skip[j]) continue;
          const bool certain_in = d2f > g.lo_in && d2f < g.hi_in;
          int s = certain_in ? segment_or_ambiguous(du, dv, g.seg_eps) : -1;
          if (s < 0) {
            double d2;
            s = exact_member(c, pi, sxy[q], certain_in, &d2);
            if (s < 0) continue;
          }
          mask |= 1u << s;
          const float cb = s_bf[s * nb + tx];
          const int cjb = s_bj[s * nb + tx];
          const bool take = cjb < 0 || d2f < cb || (d2f == cb && j < cjb);
          // conservative: the displaced or the new member is close to the best
          const bool close = cjb >= 0 && fabsf(d2f - cb) <= tie;
          if (close) amb |= 1u << s;
          if (take) {
            s_bf[s * nb + tx] = d2f;
            s_bj[s * nb + tx] = j;
          }
          if (LIST) {
            if (ROWS && cnt < k_cap) row_out[cnt] = j;
          } else if (cnt < k_cap) {
            row_list[cnt * nb] = j;
          } else {
            // the row overflows (rare): it keeps the k_cap smallest indices,
            // in order from here on
            if (cnt == k_cap)
              for (int a = 1; a < k_cap; ++a) {
                const int v = row_list[a * nb];
                int b = a;
                while (b > 0 && row_list[(b - 1) * nb] > v) {
                  row_list[b * nb] = row_list[(b - 1) * nb];
                  --b;
                }
                row_list[b * nb] = v;
              }
            if (j < row_list[(k_cap - 1) * nb]) {
              int pos = k_cap - 1;
              while (pos > 0 && row_list[(pos - 1) * nb] > j) {
                row_list[pos * nb] = row_list[(pos - 1) * nb];
                --pos;
              }
              row_list[pos * nb] = j;
            }
          }
          ++cnt;
        }
      }
    }
    int bj[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) bj[t] = s_bj[t * nb + tx];
    if (amb) {
      // exact FP64 order (ties to the smaller index) for the flagged segments
      double bd[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        bd[t] = 1e300;
        if ((amb >> t) & 1u) bj[t] = -1;
      }
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
            if (d2f < g.lo_out || d2f > g.hi_out) continue;
            const int j = sidx[q];
            if (j == i) continue;
            if (SKIP && skip[j]) continue;
            const bool certain_in = d2f > g.lo_in && d2f < g.hi_in;
            double d2;
            const int s = exact_member(c, pi, sxy[q], certain_in, &d2);
            if (s < 0 || !((amb >> s) & 1u)) continue;
            double cb = bd[0];
            int cjb = bj[0];
#pragma unroll
            for (int t = 1; t < 8; ++t) {
              cb = (s == t) ? bd[t] : cb;
              cjb = (s == t) ? bj[t] : cjb;
            }
            if (cjb < 0 || d2 < cb || (d2 == cb && j < cjb)) {
#pragma unroll
              for (int t = 0; t < 8; ++t) {
                bd[t] = (s == t) ? d2 : bd[t];
                bj[t] = (s == t) ? j : bj[t];
              }
            }
          }
        }
      }
    }
    nbr_count[i] = cnt;
    const int m = cnt < k_cap ? cnt : k_cap;
    int* row = nbr_idx + (size_t)i * stride;
    if (!LIST) {
      const unsigned here = __activemask();  // (whoever is here decides for itself)
      if (!__any_sync(here, m > 16))
        write_sorted_row<16>(row_list, nb, m, row);
      else if (KCAP > 16 && !__any_sync(here, m > 24))
        write_sorted_row<(KCAP > 16 ? 24 : 16)>(row_list, nb, m, row);
      else if (KCAP > 24)
        write_sorted_row<(KCAP > 24 ? 32 : 16)>(row_list, nb, m, row);
    }
    if (LIST && ROWS) {
      const int pad = ((m + 7) & ~7) < (int)stride ? ((m + 7) & ~7) : (int)stride;
      for (int t = m; t < pad; ++t) row[t] = -1;
    }
    seg_mask[i] = (uint8_t)mask;
    int4* sm = reinterpret_cast<int4*>(small + (size_t)i * 8);
    sm[0] = make_int4(bj[0], bj[1], bj[2], bj[3]);
    sm[1] = make_int4(bj[4], bj[5], bj[6], bj[7]);
    local_max = cnt > local_max ? cnt : local_max;
  }
  // one atomic per block (one per warp on a single address serialises at L2)
  local_max = (int)__reduce_max_sync(0xffffffffu, (unsigned)local_max);
  __shared__ int w_max[kBlock / 32];
  if ((threadIdx.x & 31) == 0) w_max[threadIdx.x >> 5] = local_max;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) local_max = w_max[w] > local_max ? w_max[w] : local_max;
    if (local_max > 0) atomicMax(&ds->max_count, local_max);
  }
}

// Small clouds: counts, masks and small neighbourhoods of the listed particles
// (k_search_all<., true, false>), a warp per particle: the lanes test
// the candidates, lane s < 8 keeps segment s's closest.  A segment whose two
// closest members are within two bands of each other in FP32 is decided by
// the FP64 order in a second pass.
__global__ void __launch_bounds__(128) k_search_warp(Consts c, const Grid* __restrict__ gp,
                                                     const int* __restrict__ cell_start,
                                                     const double2* __restrict__ sxy,
                                                     const float2* __restrict__ sloc, const int* __restrict__ sidx,
                                                     const int* __restrict__ list, const int* __restrict__ list_count,
                                                     const int* __restrict__ cell_key,
                                                     const int* __restrict__ cell_rank, int* __restrict__ nbr_count,
                                                     uint8_t* __restrict__ seg_mask, int* __restrict__ small,
                                                     DevStats* __restrict__ ds) {
  constexpr unsigned kAll = 0xffffffffu;
  const int m = *list_count;
  const Grid g = *gp;
  const float tie = 2.f * kBand;
  const int lane = threadIdx.x & 31;
  int local_max = 0;
  for (long t = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < m; t += ((long)gridDim.x * blockDim.x) >> 5) {
    const int i = list[t];
    const int key = cell_key[i];
    const int p = cell_start[key] + cell_rank[i];
    const double2 pi = sxy[p];
    const float2 li = sloc[p];
    const int cy = key / g.nx, cx = key - cy * g.nx;
    const WarpCells wc = warp_cells(cell_start, g, cx, cy);
    // candidate k: its segment, or -1 if it is not a neighbour
    auto member = [&](int k, int* j, float* d2f, double* d2) {
      int ox, oy;
      const int q = warp_candidate(wc, k, &ox, &oy);
      const float2 lj = sloc[q];
      *j = sidx[q];
      const float du = ((float)ox - li.x) + lj.x, dv = ((float)oy - li.y) + lj.y;
      *d2f = __fmaf_rn(du, du, dv * dv);
      if (*d2f < g.lo_out || *d2f > g.hi_out || *j == i) return -1;
      const bool certain_in = *d2f > g.lo_in && *d2f < g.hi_in;
      int s = certain_in && !d2 ? segment_or_ambiguous(du, dv, g.seg_eps) : -1;
      double e;
      if (s < 0) s = exact_member(c, pi, sxy[q], certain_in, d2 ? d2 : &e);
      return s;
    };
    int cnt = 0, bj = -1;  // lane s: segment s's closest so far
    float bf = 3e38f;
    unsigned mask = 0, amb = 0;
    for (int k0 = 0; k0 < wc.total; k0 += 32) {
      int j = 0, s = -1;
      float d2f = 3e38f;
      if (k0 + lane < wc.total) s = member(k0 + lane, &j, &d2f, nullptr);
      cnt += __popc(__ballot_sync(kAll, s >= 0));
#pragma unroll 1
      for (int sg = 0; sg < 8; ++sg) {
        const bool mine = s == sg;
        if (!__any_sync(kAll, mine)) continue;
        mask |= 1u << sg;
        const float dmin = __uint_as_float(__reduce_min_sync(kAll, __float_as_uint(mine ? d2f : 3e38f)));
        const unsigned near = __ballot_sync(kAll, mine && d2f - dmin <= tie);
        // (not above dmin rather than equal to it: a NaN offset, which the step
        // refuses in the end, must leave an index too)
        const int jmin = (int)__reduce_min_sync(kAll, mine && !(d2f > dmin) ? (unsigned)j : 0x7FFFFFFFu);
        const float pb = __shfl_sync(kAll, bf, sg);
        const int pj = __shfl_sync(kAll, bj, sg);
        if (__popc(near) > 1 || (pj >= 0 && fabsf(dmin - pb) <= tie)) amb |= 1u << sg;
        if (lane == sg && (pj < 0 || dmin < pb || (dmin == pb && jmin < pj))) {
          bf = dmin;
          bj = jmin;
        }
      }
    }
    while (amb) {
      // exact FP64 order (ties to the smaller index)
      const int sg = __ffs(amb) - 1;
      amb &= amb - 1;
      unsigned long long bd = ~0ull;
      int jd = 0x7FFFFFFF;
      for (int k = lane; k < wc.total; k += 32) {
        int j;
        float d2f;
        double d2 = 0.0;
        if (member(k, &j, &d2f, &d2) != sg) continue;
        const unsigned long long b = (unsigned long long)__double_as_longlong(d2);  // d2 >= +0
        if (b < bd || (b == bd && j < jd)) {
          bd = b;
          jd = j;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long od = __shfl_xor_sync(kAll, bd, o);
        const int oj = __shfl_xor_sync(kAll, jd, o);
        if (od < bd || (od == bd && oj < jd)) {
          bd = od;
          jd = oj;
        }
      }
      if (lane == sg && jd != 0x7FFFFFFF) bj = jd;
    }
    if (lane < 8) small[(size_t)i * 8 + lane] = bj;
    if (lane == 0) {
      nbr_count[i] = cnt;
      seg_mask[i] = (uint8_t)mask;
    }
    local_max = cnt > local_max ? cnt : local_max;
  }
  __shared__ int w_max[4];
  if (lane == 0) w_max[threadIdx.x >> 5] = local_max;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 4; ++w) local_max = w_max[w] > local_max ? w_max[w] : local_max;
    if (local_max > 0) atomicMax(&ds->max_count, local_max);
  }
}

// Small clouds: segment masks, a warp per particle (k_search_masks_list).
__global__ void __launch_bounds__(128) k_masks_warp(Consts c, const Grid* __restrict__ gp,
                                                    const int* __restrict__ cell_start,
                                                    const double2* __restrict__ sxy, const float2* __restrict__ sloc,
                                                    const int* __restrict__ sidx, const int* __restrict__ cell_key,
                                                    const int* __restrict__ cell_rank, const int* __restrict__ list,
                                                    const int* __restrict__ list_count, uint8_t* __restrict__ mask) {
  const int m = *list_count;
  const Grid g = *gp;
  const int lane = threadIdx.x & 31;
  for (long t = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < m; t += ((long)gridDim.x * blockDim.x) >> 5) {
    const int i = list[t];
    const int key = cell_key[i];
    const int p = cell_start[key] + cell_rank[i];
    const double2 pi = sxy[p];
    const float2 li = sloc[p];
    const int cy = key / g.nx, cx = key - cy * g.nx;
    const WarpCells wc = warp_cells(cell_start, g, cx, cy);
    unsigned mk = 0;
    for (int k = lane; k < wc.total; k += 32) {
      int ox, oy;
      const int q = warp_candidate(wc, k, &ox, &oy);
      const float2 lj = sloc[q];
      const float du = ((float)ox - li.x) + lj.x, dv = ((float)oy - li.y) + lj.y;
      const float d2f = __fmaf_rn(du, du, dv * dv);
      if (d2f < g.lo_out || d2f > g.hi_out) continue;
      const bool certain_in = d2f > g.lo_in && d2f < g.hi_in;
      int s = certain_in ? segment_or_ambiguous(du, dv, g.seg_eps) : -1;
      if (s < 0) {
        double d2;
        if (sidx[q] != i) s = exact_member(c, pi, sxy[q], false, &d2);
      }
      if (s >= 0) mk |= 1u << s;
    }
    mk = __reduce_or_sync(0xffffffffu, mk);
    if (lane == 0) mask[i] = (uint8_t)mk;
  }
}

// Grid of the warp-per-particle kernels.
static int warp_grid(int m_bound) {
  const long b = ((long)m_bound + 3) / 4, most = 16L * sm_count();
  return (int)(b < most ? b : most);
}

// Segment masks of the listed particles (the diffused list, in index order:
// lattice order keeps a warp's particles neighbours), each located in the
// sorted arrays through its cell key and rank: FP32 distances on the
// cell-local coordinates, the FP64 definition only for the pairs within the
// band of an annulus bound or a segment line.
__global__ void __launch_bounds__(kBlock) k_search_masks_list(Consts c, const Grid* __restrict__ gp,
                                                              const int* __restrict__ cell_start,
                                                              const double2* __restrict__ sxy,
                                                              const float2* __restrict__ sloc,
                                                              const int* __restrict__ sidx,
                                                              const int* __restrict__ cell_key,
                                                              const int* __restrict__ cell_rank,
                                                              const int* __restrict__ list,
                                                              const int* __restrict__ list_count,
                                                              uint8_t* __restrict__ mask) {
  const int m = *list_count;
  const Grid g = *gp;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (long)gridDim.x * blockDim.x) {
    const int i = list[t];
    const int key = cell_key[i];
    const int p = cell_start[key] + cell_rank[i];
    const double2 pi = sxy[p];
    const float2 li = sloc[p];
    const int cy = key / g.nx, cx = key - cy * g.nx;
    unsigned mk = 0;
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
          if (d2f < g.lo_out || d2f > g.hi_out) continue;
          int s = -1;
          if (d2f > g.lo_in && d2f < g.hi_in) s = segment_or_ambiguous(du, dv, g.seg_eps);
          if (s < 0) {
            const int j = sidx[q];
            if (j == i) continue;
            const double2 pj = sxy[q];
            const double dx = __dsub_rn(pj.x, pi.x), dy = __dsub_rn(pj.y, pi.y);
            const double d2 = dist2(dx, dy);
            if (d2 < c.lo2 || d2 > c.hi2) continue;
            s = segment_of(dx, dy);
          }
          mk |= 1u << s;
        }
      }
    }
    mask[i] = (uint8_t)mk;
  }
}

cudaError_t search_masks_list_dev(const Consts& c, const Grid* g, const int* cell_start, const double2* sorted_xy,
                                  const float2* sorted_loc, const int* sorted_idx, const int* cell_key,
                                  const int* cell_rank, const int* list, const int* list_count, int m_bound,
                                  uint8_t* mask, cudaStream_t s) {
  if (m_bound <= 0) return cudaSuccess;
  if (warp_scans(c, m_bound)) {
    k_masks_warp<<<warp_grid(m_bound), 128, 0, s>>>(c, g, cell_start, sorted_xy, sorted_loc, sorted_idx, cell_key,
                                                    cell_rank, list, list_count, mask);
    note_launch();
    return cudaGetLastError();
  }
  const int blocks = (m_bound + kBlock - 1) / kBlock;
  k_search_masks_list<<<blocks, kBlock, 0, s>>>(c, g, cell_start, sorted_xy, sorted_loc, sorted_idx, cell_key,
                                                cell_rank, list, list_count, mask);
  note_launch();
  return cudaGetLastError();
}

// Dynamic shared memory of k_search_all: a segment's best distance and
// index per thread, eight segments, and the row being collected.
static size_t search_smem(int tb, int list) { return (size_t)tb * (8 * (sizeof(float) + sizeof(int)) + sizeof(int) * list); }

cudaError_t search_all(const Consts& c, const Grid* g, const int* cell_start, const double2* sorted_xy,
                       const float2* sorted_loc, const int* sorted_idx, int n, int* nbr_count, int* nbr_idx,
                       uint8_t* seg_mask, int* small, DevStats* ds, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int tb = c.search_block;
  const int blocks = (int)(((long)n + tb - 1) / tb);
#define VRM_SEARCH_LAUNCH(K)                                                                                      \
  do {                                                                                                            \
    const cudaError_t e = allow_smem<k_search_all<K>>(search_smem(kBlock, K));                                    \
    if (e != cudaSuccess) return e;                                                                               \
    k_search_all<K><<<blocks, tb, search_smem(tb, K), s>>>(c, g, cell_start, sorted_xy, sorted_loc, sorted_idx, n, \
                                                           nullptr, nbr_count, nbr_idx, seg_mask, small, ds);     \
  } while (0)
  if (c.row_cap <= 16)
    VRM_SEARCH_LAUNCH(16);
  else if (c.row_cap <= 24)
    VRM_SEARCH_LAUNCH(24);
  else
    VRM_SEARCH_LAUNCH(VRM_KCAP_MAX);
#undef VRM_SEARCH_LAUNCH
  note_launch();
  return cudaGetLastError();
}

cudaError_t search_list_dev(const Consts& c, const Grid* g, const int* cell_start, const double2* sorted_xy,
                            const float2* sorted_loc, const int* sorted_idx, const int* cell_key,
                            const int* cell_rank, const int* list, const int* list_count, int m_bound,
                            int* nbr_count, int* nbr_idx, uint8_t* seg_mask, int* small, DevStats* ds,
                            cudaStream_t s, bool rows, const uint8_t* skip) {
  if (m_bound <= 0) return cudaSuccess;
  if (!rows && !skip && search_by_warps(c.search_block, m_bound, c.load)) {
    k_search_warp<<<warp_grid(m_bound), 128, 0, s>>>(c, g, cell_start, sorted_xy, sorted_loc, sorted_idx, list,
                                                     list_count, cell_key, cell_rank, nbr_count, seg_mask, small, ds);
    note_launch();
    return cudaGetLastError();
  }
  const int tb = c.search_block;
  const int blocks = (int)(((long)m_bound + tb - 1) / tb);
#define VRM_SEARCH_LAUNCH(K, R, S)                                                                                    \
  k_search_all<K, true, R, S><<<blocks, tb, search_smem(tb, 0), s>>>(                                            \
      c, g, cell_start, sorted_xy, sorted_loc, sorted_idx, m_bound, list_count, nbr_count, nbr_idx, seg_mask, small, \
      ds, list, cell_key, cell_rank, skip)
  if (!rows && skip)
    VRM_SEARCH_LAUNCH(VRM_KCAP_MAX, false, true);
  else if (!rows)
    VRM_SEARCH_LAUNCH(VRM_KCAP_MAX, false, false);  // rows not written: the cap only bounds the count
  else if (c.row_cap <= 16)
    VRM_SEARCH_LAUNCH(16, true, false);
  else if (c.row_cap <= 24)
    VRM_SEARCH_LAUNCH(24, true, false);
  else
    VRM_SEARCH_LAUNCH(VRM_KCAP_MAX, true, false);
#undef VRM_SEARCH_LAUNCH
  note_launch();
  return cudaGetLastError();
}

}  // namespace vrm
