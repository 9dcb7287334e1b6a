// Kernels for small clouds (capacity at most kSmallCap), where a step is a
// chain of launches that each leave most of the GPU idle: one block does what
// ten kernels do for larger ones.  k_front_small: growth control (the exact
// radix select of vrm_reduce.cu), the diffused list, the bounding box, the
// cell grid's geometry and its cleared counts.  k_open_small: the first open
// list and the state of the insertion rounds.  Both leave every array as the
// separate kernels leave it, bit for bit.
//
// Bound by latency and, from some ten thousand particles on, by the one SM's
// issue: 870 particles take 13 us, 20,449 43 us and 32,041 80 us, the ten
// kernels of the front 75 us either way.  k_front_small_cluster shares the
// particles out to the eight blocks of a cluster: each takes its own into its
// shared memory and sums their digits, the blocks exchange digit sums,
// candidates and counts through distributed shared memory, and every block
// takes the same decisions (20,449 particles: 25 us); its seven cluster
// barriers make it slower for few particles.  The open list and the rounds'
// state take 5 and 12 us against 17.
#include <cooperative_groups.h>

#include "vrm_internal.cuh"
#include "vrm_smem.cuh"

namespace vrm {

namespace {

constexpr int kFsThreads = 1024;
constexpr int kFsWarps = kFsThreads / 32;
// From this capacity on the front takes a cluster: steps of 3,600 particles
// (8,224 of capacity) 221 us in one block and 229 in a cluster, of 10,000
// (21,024) 228 and 222, of 20,449 302 and 281, of 32,041 377 and 327.
constexpr int kFsClusterCap = 16384;
// a block's keys, kept in shared memory
template <int C>
constexpr int kFsKeys = C == 1 ? kFsClusterCap : kSmallCap / C;
// The first selection takes the keys' top 16 bits (sixteenths of a binade)
// below those of the largest key: q is 0 more than 96 binades below it.
constexpr int kFsBins = 97 * 16;
constexpr int kFsPieces = 7;  // 16-bit pieces of a sum of q (at most 96 + 16 bits)
constexpr int kFsCluster = 8;  // blocks of the clustered form
constexpr int kFsList = 256;  // candidates for the threshold that are compared pairwise
template <int C>
constexpr size_t kFsSmem = sizeof(unsigned long long) * (kFsKeys<C> + kFsWarps) +
                           sizeof(unsigned) * (kFsPieces + 1) * (kFsBins + (C > 1 ? (kFsBins + C - 1) / C : 0));

struct FrontSmallArgs {
  const double *gamma, *x, *y;
  int cap;
  const int* n_dev;
  double c_bound, Rh, lo2, hi2;
  int ncell_cap;
  uint8_t* diffused;
  int *dlist, *dcount;
  DevStats* ds;
  Grid* g;
  int *cell_count, *cell_ts;
};

__device__ __forceinline__ u128 warp_scan_u128(u128 acc) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long lo = __shfl_up_sync(0xffffffffu, (unsigned long long)acc, o);
    const unsigned long long hi = __shfl_up_sync(0xffffffffu, (unsigned long long)(acc >> 64), o);
    if (lane >= o) acc += ((u128)hi << 64) | (u128)lo;
  }
  return acc;
}
__device__ __forceinline__ u128 shfl_u128(u128 v, int src) {
  const unsigned long long lo = __shfl_sync(0xffffffffu, (unsigned long long)v, src);
  const unsigned long long hi = __shfl_sync(0xffffffffu, (unsigned long long)(v >> 64), src);
  return ((u128)hi << 64) | (u128)lo;
}

// Inclusive scan of one u128 per thread over the block; *total: the sum.
__device__ u128 block_scan_u128(u128 v, u128* total) {
  __shared__ unsigned long long s_lo[kFsWarps], s_hi[kFsWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const u128 acc = warp_scan_u128(v);
  __syncthreads();  // the totals of an earlier scan are read
  if (lane == 31) {
    s_lo[w] = (unsigned long long)acc;
    s_hi[w] = (unsigned long long)(acc >> 64);
  }
  __syncthreads();
  const u128 sums = warp_scan_u128(((u128)s_hi[lane] << 64) | (u128)s_lo[lane]);
  *total = shfl_u128(sums, 31);
  const u128 before = shfl_u128(sums, w > 0 ? w - 1 : 0);
  return (w > 0 ? before : (u128)0) + acc;
}

// Exclusive prefix over the warps of one int per warp (s[0..31] written, a
// barrier passed), and the total.
__device__ __forceinline__ int warps_before(const int* s, int w, int* total) {
  const int lane = threadIdx.x & 31;
  int v = s[lane], incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  *total = __shfl_sync(0xffffffffu, incl, 31);
  return __shfl_sync(0xffffffffu, incl - v, w);
}

// Sums of q by digit in shared memory, 16-bit pieces: h[piece][bin], counts last.
struct DigitSums {
  unsigned* h;
  int bins;
  __device__ void clear() {
    for (int k = threadIdx.x; k < (kFsPieces + 1) * bins; k += kFsThreads) h[k] = 0;
  }
  __device__ void add(int bin, u128 s, unsigned count) {
#pragma unroll
    for (int k = 0; k < kFsPieces; ++k) {
      const unsigned p = (unsigned)(s >> (16 * k)) & 0xFFFFu;
      if (p) atomicAdd(&h[k * bins + bin], p);
    }
    atomicAdd(&h[kFsPieces * bins + bin], count);
  }
  __device__ u128 sum(int bin) const {
    u128 s = 0;
#pragma unroll
    for (int k = 0; k < kFsPieces; ++k) s += (u128)h[k * bins + bin] << (16 * k);
    return s;
  }
  __device__ unsigned count(int bin) const { return h[kFsPieces * bins + bin]; }
};

__device__ __forceinline__ bool finite_bits(double v) {
  return (__double2hiint(v) & 0x7FF00000) != 0x7FF00000;
}

// Sums of q over a run of keys that share a digit, hence the exponent: their
// significands added (at most kSmallCap / kFsThreads of 53 bits), shifted once.
struct Run {
  int digit = -1, sh = 0;
  unsigned count = 0;
  unsigned long long sum = 0;
  __device__ void start(int d, unsigned long long key, int E) {
    digit = d;
    const int ebits = (int)(key >> 52);
    sh = (ebits ? ebits - 1075 : -1074) + 96 - E;  // as q_of_key
    count = 0;
    sum = 0;
  }
  __device__ void add(unsigned long long key) {
    const unsigned long long frac = key & 0xFFFFFFFFFFFFFull;
    const unsigned long long M = (key >> 52) ? (frac | 0x10000000000000ull) : frac;
    sum += sh >= 0 ? M : (sh <= -64 ? 0ull : M >> (-sh));
    ++count;
  }
  __device__ void flush(DigitSums& h) {
    if (digit >= 0) h.add(digit, sh > 0 ? (u128)sum << sh : (u128)sum, count);
  }
};

// The blocks of a cluster of C (1: one block) as k_front_small uses them.
template <int C>
__device__ __forceinline__ void all_sync() {
  if constexpr (C > 1)
    cooperative_groups::this_cluster().sync();
  else
    __syncthreads();
}
template <int C, class T>
__device__ __forceinline__ T* of_block(T* p, int r) {
  if constexpr (C > 1)
    return cooperative_groups::this_cluster().map_shared_rank(p, r);
  else
    return p;
}
// Every block's digit sums become those of all blocks: block r adds up its
// share of the bins into `merged`, then every block copies all shares.
template <int C, int BINS>
__device__ __forceinline__ void merge_sums(unsigned* h, unsigned* merged, int rank) {
  all_sync<C>();
  if constexpr (C > 1) {
    constexpr int kShare = (BINS + C - 1) / C;
    for (int k = threadIdx.x; k < kShare * (kFsPieces + 1); k += kFsThreads) {
      const int piece = k / kShare, b = rank * kShare + k % kShare;
      unsigned v = 0;
      if (b < BINS) {
#pragma unroll
        for (int r = 0; r < C; ++r) v += of_block<C>(h, r)[piece * BINS + b];
      }
      merged[k] = v;
    }
    all_sync<C>();
    for (int k = threadIdx.x; k < BINS * (kFsPieces + 1); k += kFsThreads) {
      const int piece = k / BINS, b = k % BINS;
      h[k] = of_block<C>(merged, b / kShare)[piece * kShare + b % kShare];
    }
    __syncthreads();
  }
}

template <int C>
__device__ __forceinline__ void front_small_block(const FrontSmallArgs& a) {
  extern __shared__ unsigned long long s_dyn[];
  unsigned long long* const s_key = s_dyn;
  unsigned* const s_merged = reinterpret_cast<unsigned*>(s_dyn + kFsKeys<C> + kFsWarps) + (kFsPieces + 1) * kFsBins;
  __shared__ unsigned long long s_x[5];
  __shared__ int s_xflag, s_xties, s_xgt;
  const int rank = C > 1 ? (int)blockIdx.x : 0;
  DigitSums H{reinterpret_cast<unsigned*>(s_dyn + kFsKeys<C> + kFsWarps), kFsBins};
  __shared__ unsigned long long s_red[5][kFsWarps], s_tau[2], s_rem[2], s_T;
  __shared__ unsigned long long s_list[kFsList], s_qlo[kFsList], s_qhi[kFsList];
  __shared__ int s_flag[kFsWarps], s_sel, s_cnt, s_ktie, s_gt[kFsWarps], s_tie[kFsWarps], s_nlist;
  __shared__ Grid s_grid;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // the block's share of the particles: [c0, c0 + n) of n_all
  const int n_all = *a.n_dev, per = (n_all + C - 1) / C;
  const int c0 = rank * per < n_all ? rank * per : n_all, n = n_all - c0 < per ? n_all - c0 : per;
  // The particles in 32 segments of 32 `chunk`s: warp w takes segment w where a
  // warp works together, and where every thread takes a chunk of its own, lane
  // l of warp w has chunk w of segment l, so that a warp's lanes are far apart
  // in the cloud and rarely add to the same digit at once.  A segment's keys
  // are shifted by its number, which spreads those lanes over the banks.
  const int chunk = (n + kFsThreads - 1) / kFsThreads;
  const int seg = 32 * chunk;
  auto key_of = [&](int i, int sg) { return s_key[i + sg]; };

  // keys, their maximum, the bounding box (ordered bit patterns)
  unsigned long long amax = 0, mnx = ~0ull, mxx = 0, mny = ~0ull, mxy = 0;
  int flags = 0;  // 1: a circulation is NaN or Inf, 2: a position is
#pragma unroll 4
  for (int i = tid; i < n; i += kFsThreads) {
    unsigned long long b = (unsigned long long)__double_as_longlong(a.gamma[c0 + i]) & 0x7FFFFFFFFFFFFFFFull;
    const double xi = a.x[c0 + i], yi = a.y[c0 + i];
    if (b >= 0x7FF0000000000000ull) {
      flags |= 1;
      b = 0;
    }
    s_key[i + i / seg] = b;
    amax = b > amax ? b : amax;
    // (exponent bits: a test in FP64 would take the one SM's FP64 pipe 10 us for
    // 20,449 particles)
    if (!finite_bits(xi) || !finite_bits(yi)) {
      flags |= 2;
    } else {
      const unsigned long long ox = ordered_bits(xi), oy = ordered_bits(yi);
      mnx = ox < mnx ? ox : mnx;
      mxx = ox > mxx ? ox : mxx;
      mny = oy < mny ? oy : mny;
      mxy = oy > mxy ? oy : mxy;
    }
  }
  H.clear();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long t;
    t = __shfl_xor_sync(0xffffffffu, amax, o);
    amax = t > amax ? t : amax;
    t = __shfl_xor_sync(0xffffffffu, mnx, o);
    mnx = t < mnx ? t : mnx;
    t = __shfl_xor_sync(0xffffffffu, mxx, o);
    mxx = t > mxx ? t : mxx;
    t = __shfl_xor_sync(0xffffffffu, mny, o);
    mny = t < mny ? t : mny;
    t = __shfl_xor_sync(0xffffffffu, mxy, o);
    mxy = t > mxy ? t : mxy;
  }
  flags = __reduce_or_sync(0xffffffffu, flags);
  if (lane == 0) {
    s_red[0][w] = amax;
    s_red[1][w] = mnx;
    s_red[2][w] = mxx;
    s_red[3][w] = mny;
    s_red[4][w] = mxy;
    s_flag[w] = flags;
  }
  __syncthreads();
  if (tid == kFsThreads - 32) {
    for (int k = 0; k < kFsWarps; ++k) {
      amax = s_red[0][k] > amax ? s_red[0][k] : amax;
      mnx = s_red[1][k] < mnx ? s_red[1][k] : mnx;
      mxx = s_red[2][k] > mxx ? s_red[2][k] : mxx;
      mny = s_red[3][k] < mny ? s_red[3][k] : mny;
      mxy = s_red[4][k] > mxy ? s_red[4][k] : mxy;
      flags |= s_flag[k];
    }
    s_x[0] = amax;
    s_x[1] = mnx;
    s_x[2] = mxx;
    s_x[3] = mny;
    s_x[4] = mxy;
    s_xflag = flags;
  }
  all_sync<C>();
  amax = 0;
#pragma unroll
  for (int r = 0; r < C; ++r) {
    const unsigned long long t = of_block<C>(s_x, r)[0];
    amax = t > amax ? t : amax;
  }
  if (rank == 0 && tid == kFsThreads - 32) {  // the last warp's first lane: the grid, beside the selection
#pragma unroll
    for (int r = 1; r < C; ++r) {
      const unsigned long long* const o = of_block<C>(s_x, r);
      mnx = o[1] < mnx ? o[1] : mnx;
      mxx = o[2] > mxx ? o[2] : mxx;
      mny = o[3] < mny ? o[3] : mny;
      mxy = o[4] > mxy ? o[4] : mxy;
      flags |= *of_block<C>(&s_xflag, r);
    }
    if (flags & 1) atomicOr(&a.ds->nonfinite, 1);
    s_grid = grid_geometry(mnx, mxx, mny, mxy, (flags & 2) != 0, n_all, a.Rh, a.lo2, a.hi2, a.ncell_cap);
    *a.g = s_grid;
  }

  // the threshold key T: particles above it diffuse, and of those equal to it
  // all but the first k_tie
  bool all_out = amax == 0 || !(a.c_bound < 1.0);
  unsigned long long T = 0;
  int k_tie = 0;
  if (!all_out) {
    const int E = exponent_of_key(amax);
    const int top = (int)(amax >> 48), bin0 = top >= kFsBins ? top - kFsBins + 1 : 0;
    // consecutive particles often share a digit: a thread sums its run of them
    // before the shared atomics
    const int i0 = lane * seg + w * chunk, i1 = i0 + chunk < n ? i0 + chunk : n;
    {
      Run run;
      for (int i = i0; i < i1; ++i) {
        const unsigned long long key = key_of(i, lane);
        const int bin = (int)(key >> 48) - bin0;
        if (bin < 0) continue;  // q = 0
        if (bin != run.digit) {
          run.flush(H);
          run.start(bin, key, E);
        }
        run.add(key);
      }
      run.flush(H);
    }
    merge_sums<C, kFsBins>(H.h, s_merged, rank);
    const int b0 = 2 * tid;
    const u128 v0 = b0 < kFsBins ? H.sum(b0) : (u128)0, v1 = b0 + 1 < kFsBins ? H.sum(b0 + 1) : (u128)0;
    u128 total;
    const u128 incl = block_scan_u128(v0 + v1, &total);
    if (tid == 0) {
      const u128 t = dbl_floor_to_u128(__dmul_rn(a.c_bound, u128_to_dbl(total)));
      s_tau[0] = (unsigned long long)t;
      s_tau[1] = (unsigned long long)(t >> 64);
    }
    __syncthreads();
    u128 tau = ((u128)s_tau[1] << 64) | (u128)s_tau[0];
    if (total <= tau) {
      all_out = true;
    } else {
      const u128 e0 = incl - v0 - v1, e1 = incl - v1;
      const bool h0 = e0 <= tau && e1 > tau, h1 = e1 <= tau && incl > tau;
      if (h0 || h1) {
        const u128 rem = tau - (h0 ? e0 : e1);
        s_sel = bin0 + b0 + (h0 ? 0 : 1);
        s_cnt = (int)H.count(b0 + (h0 ? 0 : 1));
        s_rem[0] = (unsigned long long)rem;
        s_rem[1] = (unsigned long long)(rem >> 64);
      }
      __syncthreads();
      unsigned long long prefix = (unsigned long long)s_sel;
      int count = s_cnt;
      tau = ((u128)s_rem[1] << 64) | (u128)s_rem[0];
      DigitSums B{H.h, 256};
      int pass = 2;
      for (; pass < 8 && count > kFsList; ++pass) {
        __syncthreads();
        B.clear();
        __syncthreads();
        const int shift = 56 - 8 * pass;
        Run run;
        for (int i = i0; i < i1; ++i) {
          const unsigned long long key = key_of(i, lane);
          if ((key >> (shift + 8)) != prefix) continue;
          const int d = (int)((key >> shift) & 0xFF);
          if (d != run.digit) {
            run.flush(B);
            run.start(d, key, E);
          }
          run.add(key);
        }
        run.flush(B);
        merge_sums<C, 256>(B.h, s_merged, rank);
        const u128 v = tid < 256 ? B.sum(tid) : (u128)0;
        u128 all;
        const u128 inc = block_scan_u128(v, &all);
        if (tid < 256 && inc > tau && inc - v <= tau) {
          const u128 rem = tau - (inc - v);
          s_sel = tid;
          s_cnt = (int)B.count(tid);
          s_rem[0] = (unsigned long long)rem;
          s_rem[1] = (unsigned long long)(rem >> 64);
        }
        __syncthreads();
        prefix = (prefix << 8) | (unsigned long long)s_sel;
        count = s_cnt;
        tau = ((u128)s_rem[1] << 64) | (u128)s_rem[0];
      }
      if (pass == 8) {
        // every byte chosen: of the particles with key T the first k_tie by
        // index stay out, k_tie = max k <= count with k q_T <= the rest
        if (tid == 0) {
          const u128 qT = q_of_key(prefix, E);
          unsigned long long lo = 0, hi = (unsigned long long)count;
          while (lo < hi) {
            const unsigned long long mid = (lo + hi + 1) / 2;
            if ((u128)mid * qT <= tau) lo = mid;
            else hi = mid - 1;
          }
          s_T = prefix;
          s_ktie = (int)lo;
        }
      } else {
        // the few particles with these leading bytes, compared pairwise: T is
        // the key at which the sum of the q up to it passes the rest
        const int shift = 64 - 8 * pass;
        if (tid == 0) s_nlist = 0;
        all_sync<C>();
        unsigned long long *const l_key = of_block<C>(s_list, 0), *const l_lo = of_block<C>(s_qlo, 0),
                           *const l_hi = of_block<C>(s_qhi, 0);
        int* const l_n = of_block<C>(&s_nlist, 0);
        for (int i = i0; i < i1; ++i) {
          const unsigned long long key = key_of(i, lane);
          if ((key >> shift) != prefix) continue;
          const int k = atomicAdd(l_n, 1);
          const u128 q = q_of_key(key, E);
          l_key[k] = key;
          l_lo[k] = (unsigned long long)q;
          l_hi[k] = (unsigned long long)(q >> 64);
        }
        all_sync<C>();
        if (rank == 0 && tid < count) {
          const unsigned long long mine = s_list[tid];
          u128 less = 0, q = 0;
          unsigned same = 0;
          for (int k = 0; k < count; ++k) {
            const unsigned long long o = s_list[k];
            const u128 qo = ((u128)s_qhi[k] << 64) | (u128)s_qlo[k];
            if (o < mine) less += qo;
            if (o == mine) {
              ++same;
              q = qo;
            }
          }
          if (less <= tau && less + q * same > tau) {
            // of the particles with key T the first k_tie by index stay out,
            // k_tie = max k with k q_T <= the rest (every such thread agrees)
            unsigned lo = 0, hi = same;
            while (lo < hi) {
              const unsigned mid = (lo + hi + 1) / 2;
              if (q * mid <= tau - less) lo = mid;
              else hi = mid - 1;
            }
            s_T = mine;
            s_ktie = (int)lo;
          }
        }
      }
      all_sync<C>();
      T = *of_block<C>(&s_T, 0);
      k_tie = *of_block<C>(&s_ktie, 0);
    }
  }

  // flags and the diffused list (ascending): warp w takes segment w
  const int r0 = w * seg, r1 = r0 + seg < n ? r0 + seg : n;
  int gt = 0, ties = 0;
#pragma unroll 4
  for (int base = r0; base < r1; base += 32) {
    const int i = base + lane;
    const unsigned long long key = i < r1 ? key_of(i, w) : 0;
    gt += __popc(__ballot_sync(0xffffffffu, i < r1 && !all_out && key > T));
    ties += __popc(__ballot_sync(0xffffffffu, i < r1 && !all_out && key == T));
  }
  if (lane == 0) {
    s_gt[w] = gt;
    s_tie[w] = ties;
  }
  __syncthreads();
  int all_ties, total;
  int tie_at = warps_before(s_tie, w, &all_ties);  // ties before this warp's segment
  if (C > 1) {
    if (tid == 0) s_xties = all_ties;
    all_sync<C>();
    for (int r = 0; r < rank; ++r) tie_at += *of_block<C>(&s_xties, r);
  }
  {
    // ties of rank k_tie and above diffuse
    const int first = tie_at > k_tie ? tie_at : k_tie;
    if (lane == 0) s_gt[w] = gt + (tie_at + ties > first ? tie_at + ties - first : 0);
  }
  __syncthreads();
  int at = warps_before(s_gt, w, &total);
  if (C > 1) {
    if (tid == 0) s_xgt = total;
    all_sync<C>();
    total = 0;
#pragma unroll
    for (int r = 0; r < C; ++r) {
      const int t = *of_block<C>(&s_xgt, r);
      if (r < rank) at += t;
      total += t;
    }
  }
#pragma unroll 4
  for (int base = r0; base < r1; base += 32) {
    const int i = base + lane;
    const unsigned long long key = i < r1 ? key_of(i, w) : 0;
    const bool tie = i < r1 && !all_out && key == T;
    const unsigned tb = __ballot_sync(0xffffffffu, tie);
    const bool d = i < r1 && !all_out && (key > T || (tie && tie_at + __popc(tb & ((1u << lane) - 1u)) >= k_tie));
    const unsigned db = __ballot_sync(0xffffffffu, d);
    if (i < r1) a.diffused[c0 + i] = d;
    if (d) a.dlist[at + __popc(db & ((1u << lane) - 1u))] = c0 + i;
    at += __popc(db);
    tie_at += __popc(tb);
  }
  const int g_tid = rank * kFsThreads + tid, g_threads = C * kFsThreads;
  {  // flags past the particles: 0, in words where they are whole
    const uintptr_t d0 = (uintptr_t)a.diffused;
    const int head = (int)(((d0 + n_all + 15) & ~(uintptr_t)15) - d0);
    const int v0 = head < a.cap ? head : a.cap, v1 = v0 + ((a.cap - v0) & ~15);
    for (int i = v0 + 16 * g_tid; i < v1; i += 16 * g_threads)
      *reinterpret_cast<uint4*>(a.diffused + i) = make_uint4(0, 0, 0, 0);
    for (int i = n_all + g_tid; i < v0; i += g_threads) a.diffused[i] = 0;
    for (int i = v1 + g_tid; i < a.cap; i += g_threads) a.diffused[i] = 0;
  }
  if (g_tid == 0) *a.dcount = total;
  // the grid's cells empty (s_grid was written before the barriers above)
  const int ncell = of_block<C>(&s_grid, 0)->ncell;
  if (C > 1) all_sync<C>();  // no block ends while another reads it
  for (int k = g_tid; k < ncell; k += g_threads) a.cell_count[k] = 0;
  for (int k = g_tid; k <= ncell / kScanTile; k += g_threads) a.cell_ts[k] = 0;
}

__global__ void __launch_bounds__(kFsThreads) k_front_small(const __grid_constant__ FrontSmallArgs a) {
  front_small_block<1>(a);
}
__global__ void __cluster_dims__(kFsCluster, 1, 1) __launch_bounds__(kFsThreads)
    k_front_small_cluster(const __grid_constant__ FrontSmallArgs a) {
  front_small_block<kFsCluster>(a);
}

// Open list of the first round (the diffused particles whose mask is not
// full, ascending), the counts of its proposals, its active positions and
// the state of the rounds (as open_list and rounds_init).
constexpr int kOpenTiles = kSmallCap / kScanTile + 1;
__global__ void __launch_bounds__(kFsThreads) k_open_small(const int* __restrict__ dlist, const int* __restrict__ dcount,
                                                           const uint8_t* __restrict__ mask, int* __restrict__ open,
                                                           int* __restrict__ n_open, int* __restrict__ cnt,
                                                           int* __restrict__ act0, int* __restrict__ cnt_ts,
                                                           StepState* st, cudaGraphConditionalHandle h, int graph) {
  __shared__ int s_w[kFsWarps], s_ts[kOpenTiles];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int m = *dcount;
  for (int k = tid; k < kOpenTiles; k += kFsThreads) s_ts[k] = 0;
  // 256 diffused particles at a time per warp, their loads issued together;
  // the empty segments of the first kOpenKeep batches stay in registers
  constexpr int U = 8, kOpenKeep = 2;
  const int range = ((m + kFsWarps - 1) / kFsWarps + 31) & ~31;
  const int r0 = w * range, r1 = r0 + range < m ? r0 + range : m;
  int idx[kOpenKeep][U];
  unsigned emp[kOpenKeep][U];
  auto load = [&](int base, int (&id)[U], unsigned (&em)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = base + 32 * u + lane;
      id[u] = t < r1 ? dlist[t] : -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) em[u] = id[u] >= 0 ? ~(unsigned)mask[id[u]] & 0xFFu : 0u;
  };
  int c = 0;
#pragma unroll
  for (int b = 0; b < kOpenKeep; ++b) {
    load(r0 + 32 * U * b, idx[b], emp[b]);
#pragma unroll
    for (int u = 0; u < U; ++u) c += __popc(__ballot_sync(0xffffffffu, emp[b][u] != 0));
  }
  for (int base = r0 + 32 * U * kOpenKeep; base < r1; base += 32 * U) {
    int id[U];
    unsigned em[U];
    load(base, id, em);
#pragma unroll
    for (int u = 0; u < U; ++u) c += __popc(__ballot_sync(0xffffffffu, em[u] != 0));
  }
  if (lane == 0) s_w[w] = c;
  __syncthreads();
  int total, at = warps_before(s_w, w, &total);
  auto put = [&](const int (&id)[U], const unsigned (&em)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned b = __ballot_sync(0xffffffffu, em[u] != 0);
      if (em[u]) {
        const int p = at + __popc(b & ((1u << lane) - 1u));
        open[p] = id[u];
        cnt[p] = __popc(em[u]);
        act0[p] = p;
        atomicAdd(&s_ts[p >> kScanTileLog], __popc(em[u]));
      }
      at += __popc(b);
    }
  };
#pragma unroll
  for (int b = 0; b < kOpenKeep; ++b) put(idx[b], emp[b]);
  for (int base = r0 + 32 * U * kOpenKeep; base < r1; base += 32 * U) {
    int id[U];
    unsigned em[U];
    load(base, id, em);
    put(id, em);
  }
  __syncthreads();
  for (int k = tid; k <= total >> kScanTileLog; k += kFsThreads) cnt_ts[k] = s_ts[k];
  if (tid == 0) {
    *n_open = total;
    rounds_start(st, total, h, graph);
  }
}

}  // namespace

cudaError_t front_small(const double* gamma, const double* x, const double* y, int cap, const int* n_dev,
                        double c_bound, double Rh, double lo2, double hi2, int ncell_cap, uint8_t* diffused,
                        int* dlist, int* dcount, DevStats* ds, Grid* g, int* cell_count, int* cell_ts,
                        cudaStream_t s) {
  const FrontSmallArgs a{gamma, x, y, cap, n_dev, c_bound, Rh, lo2, hi2, ncell_cap, diffused, dlist, dcount, ds, g,
                         cell_count, cell_ts};
  cudaError_t e;
  if (cap >= kFsClusterCap) {
    if ((e = allow_smem<k_front_small_cluster>(kFsSmem<kFsCluster>)) != cudaSuccess) return e;
    k_front_small_cluster<<<kFsCluster, kFsThreads, kFsSmem<kFsCluster>, s>>>(a);
  } else {
    if ((e = allow_smem<k_front_small>(kFsSmem<1>)) != cudaSuccess) return e;
    k_front_small<<<1, kFsThreads, kFsSmem<1>, s>>>(a);
  }
  note_launch();
  return cudaGetLastError();
}

cudaError_t open_small(const int* dlist, const int* dcount, const uint8_t* mask, int* n_open, const RoundBufs& rb,
                       StepState* st, cudaGraphConditionalHandle handle, bool graph, cudaStream_t s) {
  k_open_small<<<1, kFsThreads, 0, s>>>(dlist, dcount, mask, rb.open, n_open, rb.cnt, rb.act0, rb.cnt_ts, st, handle,
                                        graph ? 1 : 0);
  note_launch();
  return cudaGetLastError();
}

}  // namespace vrm
