// Smoothed Biot-Savart velocity by direct summation (Sec. 5, Eq.
// smoothkernel): u_h(x) = sum_j Gamma_j K_eps(x - x_j),
//   K_eps(x) = (-y, x) / (2 pi |x|^2) (1 - exp(-|x/eps|^2)),
// written as K_eps(x) = (-y, x) phi(q) / (2 pi eps^2), q = |x|^2/eps^2,
// phi(q) = (1 - exp(-q))/q (phi(0) = 1, so a particle does not move itself).
//
// GB300 runs FP32 at 62x its FP64 rate, so the pair terms are FP32: every
// position is split into an fp32 pair hi + lo (hi = fp32(x), lo =
// fp32(x - hi)), the offset is (hi_t - hi_s) + (lo_t - lo_s), accurate to
// about 1e-14 of |x| like an FP64 difference; phi by its Taylor series
// 1 - q/2 + q^2/6 - q^3/24 + q^4/120 - q^5/720 for q < 0.1 (truncation below
// 2e-10) and (1 - expf(-q)) / q above; terms summed in fp32 over tiles of
// 256 sources, tile sums added in FP64.  Relative error of a velocity about
// 1e-6 of sum_j |Gamma_j K_eps|.
//
// Work split: a block takes 128 T targets (T per thread, in pairs) and a few
// consecutive tiles of sources, so that small problems still fill the GPU;
// it writes every tile's fp32 sums to a workspace, and k_bs_sum adds a
// target's tile sums in FP64 in tile order, so the result does not depend on
// the split.  What bounds the kernel is instruction issue, so the pair terms
// are computed for two targets at once with the packed fp32 instructions
// (add, mul, fma .f32x2: the same roundings as the scalar ones), and where
// every pair of a warp and a tile has q >= 17.5 (decided from the bounding
// boxes of the tile and of the warp's targets) exp(-q) < 2^-25, 1 - exp(-q)
// is exactly 1 in binary32 and phi is the correctly rounded 1/q: the hardware
// reciprocal and one Newton step (Markstein, IBM J. Res. Dev. 34, 1990: exact
// after one step from a 1-ulp estimate but for isolated significands, of
// which the hardware estimate leaves none: every binary32 in [0.1, 2^101)
// compared with __frcp_rn).  That is 14 packed instructions and two
// reciprocals per two pairs; the parts of a tile near a warp's targets take
// the general form, where a vote per source skips the exponential as long as
// all lanes are far.  The FMA pipe binds it (a packed instruction takes it for
// two cycles: 14 cycles a pair of the 18 measured).  251,001 sources at 40,000
// targets: 5.36 ms (31.1 ms with one target per thread, a branch at q = 0.1,
// __frcp_rn and one block per 256 targets); all pairs far: 4.95 ms, and 5.51
// ms with scalar instructions in place of the packed ones; targets in random
// order: 6.6 ms.
#include "vrm_internal.cuh"

namespace vrm {

namespace {
constexpr int kTile = 256;     // sources per tile: the length of the fp32 sums
constexpr int kBsThreads = 128;
// q from which 1 - expf(-q) == 1.0f (exp(-q) < 2^-25 for q > 17.33), with
// room for the rounding of the box distances
constexpr float kFarQ = 17.5f;
// beyond it the reciprocals would leave the range the Newton step is exact in
constexpr float kFarQMax = 1e30f;
}

__global__ void k_bs_split(const double* __restrict__ x, const double* __restrict__ y,
                           const double* __restrict__ g, int n_bound, const int* __restrict__ n_dev,
                           float4* __restrict__ pos, float* __restrict__ gf) {
  const int n = n_dev ? *n_dev : n_bound;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const double xi = x[i], yi = y[i];
    const float xh = __double2float_rn(xi), yh = __double2float_rn(yi);
    const float xl = __double2float_rn(xi - (double)xh), yl = __double2float_rn(yi - (double)yh);
    pos[i] = make_float4(xh, yh, xl, yl);
    if (gf) gf[i] = g ? __double2float_rn(g[i]) : 0.0f;
  }
}

__device__ __forceinline__ float phi_series(float q) {
  float p = fmaf(q, -1.0f / 720.0f, 1.0f / 120.0f);
  p = fmaf(q, p, -1.0f / 24.0f);
  p = fmaf(q, p, 1.0f / 6.0f);
  p = fmaf(q, p, -0.5f);
  return fmaf(q, p, 1.0f);
}
__device__ __forceinline__ float phi_of(float q) {
  if (q < 0.1f) return phi_series(q);
  return (1.0f - expf(-q)) * __frcp_rn(q);
}

__device__ __forceinline__ float rcp_hw(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

// One tile of sources as the pair loop reads it: every value twice (for the
// two targets of a pair), positions negated.
struct BsTile {
  ulonglong2 hi[kTile];  // (-xh, -xh), (-yh, -yh)
  ulonglong2 lo[kTile];  // (-xl, -xl), (-yl, -yl)
  f32x2 g[kTile];        // (gamma, gamma)
  float box[4][4];       // per 64 sources: min x, max x, min y, max y (of the hi parts)
};

__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Offsets and q of the pair of targets p from source k of the tile.
template <int P>
struct BsTargets {
  f32x2 xh[P], yh[P], xl[P], yl[P];
};
template <int P>
__device__ __forceinline__ void bs_pair(const BsTargets<P>& t, int p, const ulonglong2& hi, const ulonglong2& lo,
                                        f32x2 ie, f32x2& dx, f32x2& dy, f32x2& q) {
  dx = add2(add2(t.xh[p], hi.x), add2(t.xl[p], lo.x));
  dy = add2(add2(t.yh[p], hi.y), add2(t.yl[p], lo.y));
  q = mul2(fma2(dx, dx, mul2(dy, dy)), ie);
}
// -1/q of a pair with q in [0.1, kFarQMax], correctly rounded.
__device__ __forceinline__ f32x2 bs_neg_rcp(f32x2 q, f32x2 one) {
  float q0, q1;
  unpack2(q, q0, q1);
  const f32x2 nr = pack2(rcp_hw(-q0), rcp_hw(-q1));
  return fma2(nr, fma2(q, nr, one), nr);
}

// Whether every pair of the warp's targets (box x0..x1, y0..y1) and the 64
// sources of `box` has q in [kFarQ, kFarQMax]: from the distance of the boxes
// (the hi parts are within 2^-24 of the positions; 1e-6 of the coordinates
// covers that and the roundings here) and their largest extent.  A NaN or
// infinite coordinate fails the test or spoils both forms alike.
__device__ __forceinline__ bool bs_all_far(const float* box, float x0, float x1, float y0, float y1, float inv_eps2) {
  const float sx0 = box[0], sx1 = box[1], sy0 = box[2], sy1 = box[3];
  const float mag = fmaxf(fmaxf(fmaxf(fabsf(x0), fabsf(x1)), fmaxf(fabsf(y0), fabsf(y1))),
                          fmaxf(fmaxf(fabsf(sx0), fabsf(sx1)), fmaxf(fabsf(sy0), fabsf(sy1))));
  const float gx = fmaxf(fmaxf(sx0 - x1, x0 - sx1), 0.0f), gy = fmaxf(fmaxf(sy0 - y1, y0 - sy1), 0.0f);
  const float gap = 0.99999f * sqrtf(fmaf(gx, gx, gy * gy)) - 1e-6f * mag;
  return gap > 0.0f && gap * gap * inv_eps2 > kFarQ && 8.0f * mag * mag * inv_eps2 < kFarQMax;
}

template <int T>
__global__ void __launch_bounds__(kBsThreads) k_bs_direct(const float4* __restrict__ src, const float* __restrict__ gs,
                                                          int n, int tile0, int tiles, int tiles_per_block,
                                                          const float4* __restrict__ tgt, int m, float inv_eps2,
                                                          float2* __restrict__ part) {
  constexpr int P = T / 2;
  __shared__ BsTile s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the warp's 32 T consecutive targets, lane-contiguous; past the end the last one again
  const long t0 = (long)blockIdx.x * (kBsThreads * T) + warp * (32 * T) + lane;
  BsTargets<P> tg;
  float x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const long ta = t0 + 64 * p, tb = ta + 32;
    const float4 a = tgt[ta < m ? ta : m - 1], b = tgt[tb < m ? tb : m - 1];
    tg.xh[p] = pack2(a.x, b.x);
    tg.yh[p] = pack2(a.y, b.y);
    tg.xl[p] = pack2(a.z, b.z);
    tg.yl[p] = pack2(a.w, b.w);
    x0 = fminf(x0, fminf(a.x, b.x));
    x1 = fmaxf(x1, fmaxf(a.x, b.x));
    y0 = fminf(y0, fminf(a.y, b.y));
    y1 = fmaxf(y1, fmaxf(a.y, b.y));
  }
  x0 = warp_min(x0);
  x1 = warp_max(x1);
  y0 = warp_min(y0);
  y1 = warp_max(y1);
  const f32x2 ie = pack2(inv_eps2, inv_eps2), one = pack2(1.0f, 1.0f);
  const int first = blockIdx.y * tiles_per_block;
  const int last = min(first + tiles_per_block, tiles);
  // the sources of the first tile (two per thread); a missing one gets
  // circulation 0 at the tile's first source
  float4 np[2];
  float ng[2];
  auto fetch = [&](int tile) {
    const int base = (tile0 + tile) * kTile;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = base + 2 * (int)threadIdx.x + r;
      np[r] = src[k < n ? k : base];
      ng[r] = k < n ? gs[k] : 0.0f;
    }
  };
  if (first < last) fetch(first);
  for (int tile = first; tile < last; ++tile) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k = 2 * threadIdx.x + r;
      s.hi[k] = make_ulonglong2(pack2(-np[r].x, -np[r].x), pack2(-np[r].y, -np[r].y));
      s.lo[k] = make_ulonglong2(pack2(-np[r].z, -np[r].z), pack2(-np[r].w, -np[r].w));
      s.g[k] = pack2(ng[r], ng[r]);
    }
    {
      const float bx0 = warp_min(fminf(np[0].x, np[1].x)), bx1 = warp_max(fmaxf(np[0].x, np[1].x));
      const float by0 = warp_min(fminf(np[0].y, np[1].y)), by1 = warp_max(fmaxf(np[0].y, np[1].y));
      if (lane == 0) {
        s.box[warp][0] = bx0;
        s.box[warp][1] = bx1;
        s.box[warp][2] = by0;
        s.box[warp][3] = by1;
      }
    }
    __syncthreads();
    if (tile + 1 < last) fetch(tile + 1);
    f32x2 au[P], nav[P];
#pragma unroll
    for (int p = 0; p < P; ++p) au[p] = nav[p] = 0ULL;
    const int cnt = min(kTile, n - (tile0 + tile) * kTile);
    for (int part64 = 0; 64 * part64 < cnt; ++part64) {
      const int k0 = 64 * part64, k1 = min(k0 + 64, cnt);
      if (bs_all_far(s.box[part64], x0, x1, y0, y1, inv_eps2)) {
#pragma unroll 8
        for (int k = k0; k < k1; ++k) {
          const ulonglong2 hi = s.hi[k], lo = s.lo[k];
          const f32x2 g = s.g[k];
#pragma unroll
          for (int p = 0; p < P; ++p) {
            f32x2 dx, dy, q;
            bs_pair<P>(tg, p, hi, lo, ie, dx, dy, q);
            const f32x2 nw = mul2(g, bs_neg_rcp(q, one));
            au[p] = fma2(dy, nw, au[p]);
            nav[p] = fma2(dx, nw, nav[p]);
          }
        }
      } else {
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
          const ulonglong2 hi = s.hi[k], lo = s.lo[k];
          const f32x2 g = s.g[k];
          f32x2 dx[P], dy[P], q[P];
          bool near = false;
#pragma unroll
          for (int p = 0; p < P; ++p) {
            bs_pair<P>(tg, p, hi, lo, ie, dx[p], dy[p], q[p]);
            float q0, q1;
            unpack2(q[p], q0, q1);
            near = near || !(q0 > kFarQ && q0 < kFarQMax) || !(q1 > kFarQ && q1 < kFarQMax);
          }
          if (!__any_sync(0xffffffffu, near)) {
#pragma unroll
            for (int p = 0; p < P; ++p) {
              const f32x2 nw = mul2(g, bs_neg_rcp(q[p], one));
              au[p] = fma2(dy[p], nw, au[p]);
              nav[p] = fma2(dx[p], nw, nav[p]);
            }
          } else {
            bool big = false;
#pragma unroll
            for (int p = 0; p < P; ++p) {
              float q0, q1;
              unpack2(q[p], q0, q1);
              big = big || !(q0 < kFarQMax) || !(q1 < kFarQMax);
            }
            const bool odd = __any_sync(0xffffffffu, big);  // NaN, infinite or huge offsets
#pragma unroll
            for (int p = 0; p < P; ++p) {
              float q0, q1, e0, e1;
              unpack2(q[p], q0, q1);
              f32x2 nphi;
              if (odd) {
                nphi = pack2(-phi_of(q0), -phi_of(q1));
              } else {  // phi_of without its branch
                unpack2(mul2(pack2(1.0f - expf(-q0), 1.0f - expf(-q1)), bs_neg_rcp(q[p], one)), e0, e1);
                nphi = pack2(q0 < 0.1f ? -phi_series(q0) : e0, q1 < 0.1f ? -phi_series(q1) : e1);
              }
              const f32x2 nw = mul2(g, nphi);
              au[p] = fma2(dy[p], nw, au[p]);
              nav[p] = fma2(dx[p], nw, nav[p]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
      float u0, u1, v0, v1;
      unpack2(au[p], u0, u1);
      unpack2(nav[p], v0, v1);
      const long ta = t0 + 64 * p, tb = ta + 32;
      if (ta < m) part[(size_t)tile * m + ta] = make_float2(u0, -v0);
      if (tb < m) part[(size_t)tile * m + tb] = make_float2(u1, -v1);
    }
  }
}

// Adds a target's tile sums in FP64 in tile order; the sums so far come from
// u, v unless this is the first group of tiles, and are scaled after the last.
__global__ void k_bs_sum(const float2* __restrict__ part, int tiles, int m, int first, int last, double c0,
                         double* __restrict__ u, double* __restrict__ v) {
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (long)gridDim.x * blockDim.x) {
    double U = first ? 0.0 : u[t], V = first ? 0.0 : v[t];
#pragma unroll 8
    for (int k = 0; k < tiles; ++k) {
      const float2 a = part[(size_t)k * m + t];
      U += (double)a.x;
      V += (double)a.y;
    }
    u[t] = last ? U * c0 : U;
    v[t] = last ? V * c0 : V;
  }
}

cudaError_t bs_split(const double* x, const double* y, const double* g, int n_bound, const int* n_dev, float4* pos,
                     float* gf, cudaStream_t s) {
  if (n_bound <= 0) return cudaSuccess;
  int blocks = (n_bound + kBlock - 1) / kBlock;
  if (blocks > 8 * sm_count()) blocks = 8 * sm_count();
  k_bs_split<<<blocks, kBlock, 0, s>>>(x, y, g, n_bound, n_dev, pos, gf);
  note_launch();
  return cudaGetLastError();
}


// Tile sums kept at a time: the workspace holds kBsPart of them (256 MB), or
// one per target where there are more targets than that; larger problems go
// through their sources in groups of tiles.
constexpr size_t kBsPart = (size_t)32 << 20;
static long bs_tiles(int n) { return ((long)n + kTile - 1) / kTile; }

size_t bs_part_count(int n, int m) {
  if (n <= 0 || m <= 0) return 0;
  const size_t all = (size_t)bs_tiles(n) * (size_t)m, most = kBsPart > (size_t)m ? kBsPart : (size_t)m;
  return all < most ? all : most;
}

cudaError_t bs_direct(const float4* src, const float* gs, int n, const float4* tgt, int m, double eps, float2* part,
                      double* u, double* v, cudaStream_t s) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  const float inv_eps2 = (float)(1.0 / (eps * eps));
  const double c0 = 1.0 / (2.0 * 3.141592653589793 * eps * eps);
  const int all = (int)bs_tiles(n), group = (int)(bs_part_count(n, m) / (size_t)m);
  // four targets per thread read a source half as often as two, but need
  // enough (target block, tile) pairs to fill the GPU's 8 blocks per SM: 900
  // sources at 900 targets (16 blocks of 256 targets) take 0.053 ms, 0.109 ms
  // before; 160,000 at 300 targets 0.19 ms, 16.9 ms before
  const long slots = 8L * sm_count();
  const bool wide = (((long)m + 4 * kBsThreads - 1) / (4 * kBsThreads)) * all >= slots;
  const int T = wide ? 4 : 2;
  const int tb = (int)(((long)m + T * kBsThreads - 1) / (T * kBsThreads));
  for (int tile0 = 0; tile0 < all; tile0 += group) {
    const int tiles = all - tile0 < group ? all - tile0 : group;
    // about eight waves of blocks, so that a late block costs little
    long per = (long)tiles * tb / (8 * slots);
    per = per < 1 ? 1 : per;
    if (((long)tiles + per - 1) / per > 65535) per = ((long)tiles + 65534) / 65535;
    const dim3 grid(tb, (unsigned)((tiles + per - 1) / per));
    if (T == 4)
      k_bs_direct<4><<<grid, kBsThreads, 0, s>>>(src, gs, n, tile0, tiles, (int)per, tgt, m, inv_eps2, part);
    else
      k_bs_direct<2><<<grid, kBsThreads, 0, s>>>(src, gs, n, tile0, tiles, (int)per, tgt, m, inv_eps2, part);
    note_launch();
    int blocks = (m + 127) / 128;
    if (blocks > 16 * sm_count()) blocks = 16 * sm_count();
    k_bs_sum<<<blocks, 128, 0, s>>>(part, tiles, m, tile0 == 0, tile0 + tiles >= all, c0, u, v);
    note_launch();
  }
  return cudaGetLastError();
}

}  // namespace vrm
