// The weight-proposal network of the learned path and its training, on the
// tensor cores (tcgen05, bf16 operands, fp32 accumulators in TMEM).
//
// Network: 96 inputs (the K = 32 neighbour slots' scaled offsets xi_x, xi_y
// and mask; padded to 128 columns with zeros) -> 256 -> 256 -> 256 -> 32,
// GELU (tanh form) after each hidden layer.  Parameters are kept as one fp32
// vector [W1 (256x96), b1, W2 (256x256), b2, W3, b3, W4 (32x256), b4]; the
// GEMMs read bf16 copies (W1 padded to 256x128) and, for the backward pass,
// transposed bf16 copies.
//
// Inference is one kernel (k_mlp_fused), a training step four:
//   k_gather     the batch's rows, their transposes and the mask sums
//   k_chain      per 128-row tile the forward pass, the loss gradient and the
//                backward pass down to the first layer, with the tile's
//                activations in shared memory
//   k_weight_grad  the weight gradients of every layer, split over the batch
//   k_update     the splits and the biases summed in a fixed order (training is
//                deterministic), AdamW, and the bf16 copies of the weights
// A batch of 4096 rows takes 81 us (540 us with a kernel per product, whose 32
// CTAs stored row by row, a one-block loss and separate sums: 23 launches),
// 512 rows 69 us (369), 16,384 rows 119 us (1119).
// The products are tcgen05 MMAs (M = 128, K = 16) on K-major bf16 tiles that
// TMA or the epilogues leave in shared memory in the 128-byte swizzle, with
// fp32 accumulators in TMEM.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <new>

#include "vrm_internal.cuh"
#include "vrm_mlp.cuh"
#include "vrm_smem.cuh"
#include "vrm_umma.cuh"

using namespace vrm;
using bf16 = __nv_bfloat16;

namespace {

constexpr int kIn = 96;       // features
constexpr int kInPad = 128;   // feature row stride
constexpr int kHid = 256;
constexpr int kOut = 32;
constexpr int kOutPad = 64;   // dY row stride (one K slab)
constexpr int kBM = 128;      // rows per tile
constexpr int kBK = 64;       // K per slab
constexpr long long kWaitCycles = 2000000000LL;  // about one second
constexpr long long kDrainCycles = 4000000LL;    // about 2 ms

// Copies that nothing waited for (after a wait that gave up) arrive before the
// CTA ends.
__device__ __forceinline__ void wait_for_copies() {
  const long long t0 = clock64();
  while (clock64() - t0 < kDrainCycles) {
  }
}

constexpr long kOffW1 = 0, kOffB1 = kOffW1 + (long)kHid * kIn;
constexpr long kOffW2 = kOffB1 + kHid, kOffB2 = kOffW2 + (long)kHid * kHid;
constexpr long kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + (long)kHid * kHid;
constexpr long kOffW4 = kOffB3 + kHid, kOffB4 = kOffW4 + (long)kOut * kHid;
constexpr long kParams = kOffB4 + kOut;
static_assert(kParams == VRM_MLP_PARAMS, "parameter count");

// GELU in its tanh form, 0.5 z (1 + tanh(c (z + a z^3))) with c = sqrt(2/pi),
// a = 0.044715, on the hardware tanh (tanh.approx.f32, relative error about
// 2^-11, below the bf16 rounding of the activations).
constexpr float kGeluC = 0.7978845608028654f, kGeluA = 0.044715f;
__device__ __forceinline__ float tanh_hw(float u) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
  return t;
}
// c (z + a z^3) as z (c + (c a) z^2): five fp32 operations and the tanh.
constexpr float kGeluCA = kGeluC * kGeluA;
// Of a pair z0, z1 (half the instructions), rounded to bf16 with z0 in the low half.
__device__ __forceinline__ uint32_t gelu_bf16x2(f32x2 z) {
  const f32x2 t = fma2(pack2(kGeluCA, kGeluCA), mul2(z, z), pack2(kGeluC, kGeluC));
  const f32x2 hz = mul2(pack2(0.5f, 0.5f), z);
  float u0, u1;
  unpack2(mul2(z, t), u0, u1);
  unpack2(fma2(hz, pack2(tanh_hw(u0), tanh_hw(u1)), hz), u0, u1);
  const __nv_bfloat162 r = __floats2bfloat162_rn(u0, u1);
  return *reinterpret_cast<const uint32_t*>(&r);
}
// d/dz of the same, of a pair: 0.5 (1 + t) + 0.5 z (1 - t^2) c (1 + 3 a z^2).
__device__ __forceinline__ f32x2 gelu_grad2(f32x2 z) {
  const f32x2 one = pack2(1.0f, 1.0f), half = pack2(0.5f, 0.5f), cc = pack2(kGeluC, kGeluC);
  const f32x2 z2 = mul2(z, z);
  float u0, u1;
  unpack2(mul2(cc, fma2(mul2(pack2(kGeluA, kGeluA), z), z2, z)), u0, u1);
  const float t0 = tanh_hw(u0), t1 = tanh_hw(u1);
  const f32x2 t = pack2(t0, t1);
  const f32x2 du = mul2(cc, fma2(pack2(3.0f * kGeluA, 3.0f * kGeluA), z2, one));
  return fma2(mul2(mul2(half, z), du), fma2(pack2(-t0, -t1), t, one), mul2(half, add2(one, t)));
}

// ---- fused inference ------------------------------------------------------------------
//
// The whole network for 256-row tiles in one persistent kernel of CTA pairs; a
// tile's activations never leave shared memory.  A CTA holds 128 of the rows
// and half of every weight slab; one MMA of the pair covers both.  Two tiles
// are in flight per pair (slots 0 and 1: activation tiles H[0], H[1], TMEM
// columns 0-255 and 256-511) so that the MMAs of one overlap the epilogue of
// the other:
//   warp 17 (one thread): streams the CTA's halves of the weight slabs (64
//     input columns of one layer: 128 rows of W1, W2, W3, 16 of W4) through a
//     5-stage ring with TMA as stages come free, ahead of the MMAs (a weight
//     slab is loaded once per slot);
//   warp 16 of the leading CTA (one thread): issues the MMAs layer by layer,
//     alternating the slots;
//   warp 18 (one thread): loads a slot's next input as its last layer's MMAs
//     complete;
//   warps 0-15: the epilogue of each (slot, layer) as its accumulator
//     completes: warp w reads TMEM lanes 32 (w mod 4), columns 64 (w div 4),
//     adds the bias, applies GELU and writes bf16 back into the slot's
//     activation tile in the MMA operand layout (128-byte swizzle), which the
//     next layer reads as A; the last layer writes the 32 proposals.
// Barriers (xfull, actr and wfull count in the leading CTA for both, accf and
// wempty are signalled in both): xfull (a slot's input tiles loaded), accf (the
// layer's MMAs are complete: commit), actr (the layer's epilogue is done: 32
// warp arrivals, so the next layer may overwrite TMEM and read the
// activations), hfree (the last layer's MMAs are complete: the next input may
// replace the tile; both CTAs), wfull and wempty (ring).  Every wait is bounded;
// one that gives up raises its CTA's abort flag, which every role checks before
// its next wait, and the error flag in global memory.
//
// A call of 500,000 rows takes 201 to 211 us, 168 of them the kernel (314 us with a 128-row tile per CTA and one thread
// for weights, inputs and MMAs; 243 us with a thread for the weights, biases by
// vector and GELU on pairs).  What the rest gave, in clocks of the MMA thread
// per 128-row tile: issue 4,600 -> 1,100 with an elected thread (a branch on
// the lane makes every MMA wait for its operands to move to uniform
// registers); the pair halves what shared memory takes in and L2 gives out per
// MMA, 448 KB a tile before.  The arrivals keep their default scope (CTA):
// what orders the activations, which only MMAs read, is the proxy fence before
// the arrival and not its release, and one released at cluster scope waits for
// all the CTA's stores (300 us).
// What bounds it now (tensor pipe 45%, FMA pipe 42% busy; clocks read in the
// kernel): of a tile's 11,000 clocks the epilogues take 9,000, three
// times about 3,000, at 1,600 of the FMA pipe (six operations a value) and
// 2,400 of shared memory (64 KB of A, 64 KB of the half weight slabs read, 64 KB
// of them and 64 KB of activations written).  Epilogue warps split between the
// slots instead took 250 us: two warps a scheduler do not cover the latencies.

constexpr int kEpiWarps = 16;
constexpr int kFusedThreads = (kEpiWarps + 3) * 32;
constexpr int kRing = 5;
constexpr int kSlabsPerTile = 14;  // W1: 2, W2: 4, W3: 4, W4: 4
constexpr int kSlabsPerPair = 2 * kSlabsPerTile;
constexpr uint32_t kSlabBytes = kBM * kBK * 2;  // one 128-row activation slab, or half a weight slab
constexpr uint32_t kRingBytes = 256 * kBK * 2;  // one 256-row weight slab
constexpr int kBiases = 3 * kHid + kOut;
constexpr size_t kFusedSmem = 1024 + (2 * 4 + kRing) * (size_t)kSlabBytes + kBiases * sizeof(float) + 256;

// Layer and K slab of the g-th weight slab a single tile consumes.
__device__ __forceinline__ void slab_of(int s, int* layer, int* kb) {
  if (s < 2) {
    *layer = 0, *kb = s;
  } else if (s < 6) {
    *layer = 1, *kb = s - 2;
  } else if (s < 10) {
    *layer = 2, *kb = s - 6;
  } else {
    *layer = 3, *kb = s - 10;
  }
}

// Layer and K slab of the g-th weight slab the producer consumes: whole
// pairs of tiles take each layer's slabs twice (slot 0, then slot 1); a
// last unpaired tile takes them once.
__device__ __forceinline__ void slab_at(int g, int pairs, int* layer, int* kb) {
  if (g < pairs * kSlabsPerPair) {
    const int r = g % kSlabsPerPair;
    if (r < 4) {
      *layer = 0, *kb = r & 1;
    } else if (r < 12) {
      *layer = 1, *kb = (r - 4) & 3;
    } else if (r < 20) {
      *layer = 2, *kb = (r - 12) & 3;
    } else {
      *layer = 3, *kb = (r - 20) & 3;
    }
  } else {
    slab_of(g - pairs * kSlabsPerPair, layer, kb);
  }
}

struct FusedArgs {
  const float* bias;  // theta: b1, b2, b3, b4 at their offsets
  float* Y;           // [rows x 32]
  int rows;           // bound
  const int* rows_dev;
  int* error;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kFusedThreads, 1)
    k_mlp_fused(const __grid_constant__ CUtensorMap tx, const __grid_constant__ CUtensorMap tw1,
                const __grid_constant__ CUtensorMap tw2, const __grid_constant__ CUtensorMap tw3,
                const __grid_constant__ CUtensorMap tw4, FusedArgs a) {
  extern __shared__ uint8_t smem_raw[];
  int rows = a.rows;
  if (a.rows_dev) {
    const int r = *a.rows_dev;
    rows = r < rows ? r : rows;
  }
  const int ntiles = (rows + 2 * kBM - 1) / (2 * kBM);
  const int pair = (int)blockIdx.x >> 1, npair = (int)gridDim.x >> 1;
  const int rank = (int)umma::cluster_rank();
  if (pair >= ntiles) return;  // both CTAs
  const int my_tiles = (ntiles - 1 - pair) / npair + 1;
  const int pairs_full = my_tiles / 2;
  const int npairs = (my_tiles + 1) / 2;
  const int total = pairs_full * kSlabsPerPair + (my_tiles & 1) * kSlabsPerTile;

  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* H = base;                              // 2 slots x 4 slabs x 16 KB
  uint8_t* ring = base + 8 * (size_t)kSlabBytes;  // kRing x 16 KB
  float* s_bias = (float*)(ring + (size_t)kRing * kSlabBytes);  // b1, b2, b3, b4
  uint64_t* bars = (uint64_t*)(s_bias + kBiases);
  uint64_t* xfull = bars;
  uint64_t* accf = bars + 2;
  uint64_t* actr = bars + 4;
  uint64_t* hfree = bars + 6;
  uint64_t* wfull = bars + 8;
  uint64_t* wempty = bars + 8 + kRing;
  uint64_t* drain = bars + 8 + 2 * kRing;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      umma::mbar_init(&xfull[s], 1);
      umma::mbar_init(&accf[s], 1);
      umma::mbar_init(&actr[s], 2 * kEpiWarps);
      umma::mbar_init(&hfree[s], 1);
    }
    for (int s = 0; s < kRing; ++s) {
      umma::mbar_init(&wfull[s], 1);
      umma::mbar_init(&wempty[s], 1);
    }
    umma::mbar_init(drain, 1);
    *abort_flag = 0;
    umma::fence_barrier_init();
  }
  for (int k = threadIdx.x; k < kBiases; k += kFusedThreads)
    s_bias[k] = a.bias[(k < kHid ? kOffB1 : k < 2 * kHid ? kOffB2 : k < 3 * kHid ? kOffB3 : kOffB4) + k % kHid];
  __syncwarp();
  if (warp == 0) umma::tmem_alloc_pair(tmem_slot, 512);
  umma::fence_before_sync();
  __syncthreads();
  umma::cluster_sync();
  umma::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const int last_tile = (rows - 1) / kBM;  // 128-row tiles of the input

  if (warp == kEpiWarps + 1) {
    // ---- weight slabs (one thread) ----
    if (umma::elect_one()) {
      const CUtensorMap* wmap[4] = {&tw1, &tw2, &tw3, &tw4};
      for (int g = 0; g < total; ++g) {
        int layer, kb;
        slab_at(g, pairs_full, &layer, &kb);
        const int st = g % kRing;
        if (g >= kRing && (*abort_flag || !umma::mbar_wait(&wempty[st], (uint32_t)(g / kRing - 1) & 1u,
                                                                   2 * kWaitCycles))) {
          *abort_flag = 1;
          break;
        }
        const int half = layer == 3 ? kOut / 2 : kBM;  // rows of this CTA
        if (rank == 0) umma::mbar_arrive_expect_tx(&wfull[st], 2u * (uint32_t)half * kBK * 2);
        umma::tma_load_2d_pair(ring + (size_t)st * kSlabBytes, wmap[layer], umma::lead_addr(&wfull[st]), kb * kBK,
                               rank * half);
      }
      // Every commit arrives in this CTA before it ends: the leading CTA sees its
      // own arrivals, not its peer's, so each waits for those it gets (here and
      // beside the inputs; accf is waited for by the epilogues).  And every MMA
      // issued completes before the TMEM is released.
      for (int g = total < kRing ? 0 : total - kRing; g < total && !*abort_flag; ++g)
        if (!umma::mbar_wait(&wempty[g % kRing], (uint32_t)(g / kRing) & 1u, 2 * kWaitCycles)) *abort_flag = 1;
      if (!umma::mbar_wait(drain, 0u, 2 * kWaitCycles)) *abort_flag = 1;
    }
  } else if (warp == kEpiWarps + 2) {
    // ---- input tiles (one thread) ----
    if (umma::elect_one()) {
      for (int i = 0; i < my_tiles; ++i) {
        const int s = i & 1;
        if (i >= 2 && (*abort_flag || !umma::mbar_wait(&hfree[s], (uint32_t)(i / 2 - 1) & 1u, 2 * kWaitCycles))) {
          *abort_flag = 1;
          break;
        }
        // over the slot's activations; a half beyond the last row loads the
        // last rows again and stores nothing
        uint8_t* h = H + (size_t)s * 4 * kSlabBytes;
        const int t = 2 * (pair + i * npair) + rank;
        const int row0 = (t < last_tile ? t : last_tile) * kBM;
        const uint32_t bar = umma::lead_addr(&xfull[s]);
        if (rank == 0) umma::mbar_arrive_expect_tx(&xfull[s], 4u * kSlabBytes);
        umma::tma_load_2d_pair(h, &tx, bar, 0, row0);
        umma::tma_load_2d_pair(h + kSlabBytes, &tx, bar, kBK, row0);
      }
      for (int i = my_tiles < 2 ? 0 : my_tiles - 2; i < my_tiles && !*abort_flag; ++i)
        if (!umma::mbar_wait(&hfree[i & 1], (uint32_t)(i / 2) & 1u, 2 * kWaitCycles)) *abort_flag = 1;
    }
  } else if (warp == kEpiWarps) {
    // ---- MMA issue (one thread of the pair) ----
    if (rank == 0 && umma::elect_one()) {
      bool fail = false;
      int g = 0;
      for (int p = 0; p < npairs && !fail; ++p) {
        const int nslot = (2 * p + 1 < my_tiles) ? 2 : 1;
        for (int l = 0; l < 4 && !fail; ++l) {
          for (int s = 0; s < nslot && !fail; ++s) {
            if (*abort_flag) {
              fail = true;
              break;
            }
            const int e = 4 * p + l;  // epilogues of this slot that must be done
            if (e > 0 && !umma::mbar_wait(&actr[s], (uint32_t)(e - 1) & 1u, kWaitCycles)) {
              fail = true;
              break;
            }
            if (l == 0 && !umma::mbar_wait(&xfull[s], (uint32_t)p & 1u, kWaitCycles)) {
              fail = true;
              break;
            }
            umma::fence_after_sync();
            const uint32_t idesc = umma::idesc_bf16(2 * kBM, l == 3 ? kOut : kHid);
            const int nk = l == 0 ? 2 : 4;
            uint8_t* h = H + (size_t)s * 4 * kSlabBytes;
            for (int kb = 0; kb < nk; ++kb, ++g) {
              const int st = g % kRing;
              if (!umma::mbar_wait(&wfull[st], (uint32_t)(g / kRing) & 1u, kWaitCycles)) {
                fail = true;
                break;
              }
              umma::fence_after_sync();
              const uint64_t da = umma::desc_sw128(umma::smem_u32(h + (size_t)kb * kSlabBytes));
              const uint64_t db = umma::desc_sw128(umma::smem_u32(ring + (size_t)st * kSlabBytes));
#pragma unroll
              for (int k = 0; k < kBK / 16; ++k)
                umma::mma_bf16_pair(tmem + (uint32_t)(s * 256), da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
              umma::mma_commit_pair(&wempty[st]);
            }
            if (fail) break;
            umma::mma_commit_pair(&accf[s]);
            if (l == 3) umma::mma_commit_pair(&hfree[s]);
          }
        }
      }
      if (fail) *abort_flag = 1;
      umma::mma_commit_pair(drain);  // (after a failure too)
    }
  } else {
    // ---- epilogue warps ----
    const int q = warp & 3, cg = warp >> 2;
    const int r = q * 32 + lane;  // row within the CTA's half of the tile
    bool stop = false;
    for (int p = 0; p < npairs && !stop; ++p) {
      const int nslot = (2 * p + 1 < my_tiles) ? 2 : 1;
      for (int l = 0; l < 4 && !stop; ++l) {
        for (int s = 0; s < nslot; ++s) {
          if (*abort_flag) {
            stop = true;
            break;
          }
          if (!umma::mbar_wait(&accf[s], (uint32_t)(4 * p + l) & 1u, 2 * kWaitCycles)) {
            *abort_flag = 1;
            stop = true;
            break;
          }
          umma::fence_after_sync();
          const uint32_t trow = tmem + (uint32_t)(s * 256) + ((uint32_t)(q * 32) << 16);
          const uint32_t done = umma::lead_addr(&actr[s]);
          if (l < 3) {
            // 32 columns at a time, bias and GELU on pairs of columns
            const ulonglong2* b = reinterpret_cast<const ulonglong2*>(s_bias + l * kHid + cg * 64);
            uint8_t* slab = H + ((size_t)s * 4 + cg) * kSlabBytes + (size_t)r * 128;
            uint32_t va[32], vb[32];
            umma::tmem_request32(trow + (uint32_t)(cg * 64), va);
            umma::tmem_wait32(va);
            umma::tmem_request32(trow + (uint32_t)(cg * 64 + 32), vb);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              if (half == 1) umma::tmem_wait32(vb);
              const uint32_t* v = half == 0 ? va : vb;
#pragma unroll
              for (int u = 0; u < 4; ++u) {  // eight columns: one 16-byte chunk of the operand
                uint32_t hv[4];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                  const ulonglong2 b4 = b[half * 8 + 2 * u + k];
                  const uint32_t* vv = &v[8 * u + 4 * k];
                  hv[2 * k] = gelu_bf16x2(add2(pack2(__uint_as_float(vv[0]), __uint_as_float(vv[1])), b4.x));
                  hv[2 * k + 1] = gelu_bf16x2(add2(pack2(__uint_as_float(vv[2]), __uint_as_float(vv[3])), b4.y));
                }
                *reinterpret_cast<uint4*>(slab + (((half * 4 + u) ^ (r & 7)) << 4)) =
                    make_uint4(hv[0], hv[1], hv[2], hv[3]);
              }
            }
            umma::fence_proxy_async_smem();  // the activation writes feed the next MMAs (async proxy)
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive_cluster(done);
          } else {
            // the accumulator is free once it is read; the proposals are stored after that
            float v[16];
            const int c0 = (cg & 1) * 16;
            if (cg < 2) umma::tmem_ld16(trow + (uint32_t)c0, v);
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive_cluster(done);
            const int row = ((pair + (2 * p + s) * npair) * 2 + rank) * kBM + r;
            if (cg < 2 && row < rows) {
              const float* b = s_bias + 3 * kHid + c0;
              float4* dst = reinterpret_cast<float4*>(a.Y + (size_t)row * kOut + c0);
#pragma unroll
              for (int i = 0; i < 4; ++i)
                dst[i] = make_float4(v[4 * i] + b[4 * i], v[4 * i + 1] + b[4 * i + 1], v[4 * i + 2] + b[4 * i + 2],
                                     v[4 * i + 3] + b[4 * i + 3]);
            }
          }
        }
      }
    }
  }
  __syncwarp();
  umma::fence_before_sync();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0 && a.error) atomicExch(a.error, 1);
    wait_for_copies();
  }
  umma::cluster_sync();  // the peer is as far: nothing it sent here is under way
  if (warp == 0) {
    umma::fence_after_sync();
    umma::tmem_dealloc_pair(tmem, 512);
  }
}

// ---- small kernels -----------------------------------------------------------------

// ---- training -------------------------------------------------------------------
//
// Batch assembly: rows idx[r] (or r) of the data set into X [B x 128],
// X^T [128 x B] and T [B x 32], and the sum of each 32-row block's mask; rows
// >= rows are zero (their mask is 0, so they add nothing to the loss or the
// gradients).  One block per 32 rows, transposed through shared memory, so
// that every store is coalesced (aligned: X_all starts on a 4-byte boundary).
constexpr int kGatherRows = 32;
__global__ void __launch_bounds__(256) k_gather(const bf16* __restrict__ X_all, const float* __restrict__ T_all,
                                                const int* __restrict__ idx, int rows, int B, bf16* __restrict__ Xb,
                                                bf16* __restrict__ Xbt, float* __restrict__ Tb,
                                                float* __restrict__ cnt, bool aligned) {
  __shared__ uint32_t tile[kGatherRows][kInPad / 2 + 1];
  __shared__ float part[8];
  const int tid = threadIdx.x, r0 = blockIdx.x * kGatherRows;
  float m = 0.0f;
  for (int t = tid; t < kGatherRows * (kInPad / 2); t += 256) {  // pairs of columns
    const int r = t / (kInPad / 2), c = t % (kInPad / 2), row = r0 + r;
    uint32_t v = 0;
    if (row < rows) {
      const bf16* src = X_all + (size_t)(idx ? idx[row] : row) * kInPad + 2 * c;
      if (aligned) {
        v = *reinterpret_cast<const uint32_t*>(src);
      } else {
        const uint16_t* h = reinterpret_cast<const uint16_t*>(src);
        v = (uint32_t)h[0] | (uint32_t)h[1] << 16;
      }
    }
    reinterpret_cast<uint32_t*>(Xb)[(size_t)row * (kInPad / 2) + c] = v;
    tile[r][c] = v;
    if (c >= kOut && c < 3 * kOut / 2) {  // columns 64..95
      const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&v);
      m += __bfloat162float(b.x) + __bfloat162float(b.y);
    }
  }
  for (int t = tid; t < kGatherRows * kOut; t += 256) {
    const int row = r0 + t / kOut;
    Tb[(size_t)r0 * kOut + t] =
        row < rows ? T_all[(size_t)(idx ? idx[row] : row) * kOut + t % kOut] : 0.0f;
  }
  for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  if ((tid & 31) == 0) part[tid >> 5] = m;
  __syncthreads();
  for (int t = tid; t < kInPad * (kGatherRows / 2); t += 256) {  // pairs of rows of X^T
    const int c = t / (kGatherRows / 2), r = 2 * (t % (kGatherRows / 2));
    const uint32_t a = tile[r][c / 2], b = tile[r + 1][c / 2];
    const uint32_t v = c & 1 ? (a >> 16) | (b & 0xFFFF0000u) : (a & 0xFFFFu) | (b << 16);
    reinterpret_cast<uint32_t*>(Xbt + (size_t)c * B + r0)[r / 2] = v;
  }
  if (tid == 0) {
    float sum = 0.0f;
    for (int w = 0; w < 8; ++w) sum += part[w];
    cnt[blockIdx.x] = sum;
  }
}

// Forward and backward pass of 128-row tiles, seven products in a row:
//   0-2  Z = A W^T + b, A = GELU(Z)         (A in shared memory, in place)
//   3    Y = A W4^T + b4, dY = 2 M (Y - T) / sum(M) and the tile's loss
//   4    dZ3 = (dY W4) GELU'(Z3)
//   5, 6 dZ2 = (dZ3 W3) GELU'(Z2), dZ1 = (dZ2 W2) GELU'(Z1)
// One thread of warp 17 streams the weight slabs through a ring with TMA, one of
// warp 16 loads the inputs and issues the MMAs; warps 0-15 run each product's
// epilogue (warp w: TMEM lanes 32 (w mod 4), columns 64 (w div 4)) and write the
// next operand in the swizzled layout.  Products accumulate in alternating
// halves of the TMEM (chain_half), so that what an epilogue stores goes out
// after the operand is handed over, under the next product: pre-activations Z1
// and Z2, which come back to the same thread, tile by tile with the rows
// contiguous (Z3 stays in its half until product 4), and what k_weight_grad
// reads (A^T, dZ^T, dY^T), transposed, 64 bytes of a row per warp.
// The chain is bound by its epilogues: of 63,000 clocks for a tile those up to
// the hand-over take 4,000 (forward) and 6,500 (backward) a product, the MMAs
// 2,000, and the stores 5,000 beside them (192 KB a product from one SM).  A step
// of 4096 rows went from 95 to 81 us with the stores after the hand-over, elected
// threads, a thread for the weights, biases in shared memory (each is used once
// by a tile: a load from L2 every time) and Z3 kept.
// Barriers: xfull (input tile loaded), wfull / wempty (ring), accf (a
// product's MMAs are complete), actr (its epilogue is done: 16 warps).  Every
// wait is bounded, as in k_mlp_fused.
constexpr int kChainThreads = (kEpiWarps + 2) * 32;
constexpr int kChainRing = 4;
constexpr size_t kChainSmem =
    1024 + 4 * (size_t)kSlabBytes + (size_t)kChainRing * kRingBytes + kBiases * sizeof(float) + 256;

struct ChainMaps {
  CUtensorMap w[7];  // W1, W2, W3, W4, W4^T, W3^T, W2^T
};
struct ChainArgs {
  const float* theta;
  const bf16* Xb;
  const float* Tb;
  const float* cnt;   // mask sums of the batch's 32-row blocks
  float* Z[2];        // [tile][256][128]
  bf16* At[3];        // A1^T, A2^T, A3^T [256 x B]
  bf16* dZt[3];       // dZ1^T, dZ2^T, dZ3^T [256 x B]
  bf16* dYt;          // [128 x B], rows >= 32 stay 0
  float* lossp;       // [tiles][8]
  int B;
  int* error;
};

// Half of the TMEM that product p accumulates in.
__device__ __forceinline__ uint32_t chain_half(int p) { return p == 1 || p == 3 || p == 4 || p == 6 ? 256u : 0u; }
__device__ __forceinline__ int chain_k(int p) { return p == 0 ? 2 : p == 4 ? 1 : 4; }  // K slabs of product p

__global__ void __launch_bounds__(kChainThreads, 1)
    k_chain(const __grid_constant__ CUtensorMap tx, const __grid_constant__ ChainMaps maps,
            const __grid_constant__ ChainArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const int ntiles = a.B / kBM;
  const int my_tiles = (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* H = base;                              // 4 slabs x 16 KB
  uint8_t* ring = base + 4 * (size_t)kSlabBytes;  // kChainRing x 32 KB
  float* s_bias = (float*)(ring + (size_t)kChainRing * kRingBytes);  // b1, b2, b3, b4
  uint64_t* bars = (uint64_t*)(s_bias + kBiases);
  uint64_t *xfull = bars, *accf = bars + 1, *actr = bars + 2, *drain = bars + 3;
  uint64_t *wfull = bars + 4, *wempty = bars + 4 + kChainRing;
  uint32_t* tmem_slot = (uint32_t*)(bars + 4 + 2 * kChainRing);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    umma::mbar_init(xfull, 1);
    umma::mbar_init(accf, 1);
    umma::mbar_init(actr, kEpiWarps);
    umma::mbar_init(drain, 1);
    for (int s = 0; s < kChainRing; ++s) {
      umma::mbar_init(&wfull[s], 1);
      umma::mbar_init(&wempty[s], 1);
    }
    *abort_flag = 0;
    umma::fence_barrier_init();
  }
  for (int k = threadIdx.x; k < kBiases; k += kChainThreads)
    s_bias[k] = a.theta[(k < kHid ? kOffB1 : k < 2 * kHid ? kOffB2 : k < 3 * kHid ? kOffB3 : kOffB4) + k % kHid];
  __syncwarp();
  if (warp == 0) umma::tmem_alloc(tmem_slot, 512);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = *tmem_slot;

  if (warp == kEpiWarps + 1) {
    // ---- weight slabs (one thread) ----
    if (umma::elect_one()) {
      int g = 0;
      bool fail = false;
      for (int i = 0; i < my_tiles && !fail; ++i) {
        for (int p = 0; p < 7 && !fail; ++p) {
          const int nk = chain_k(p);
          for (int kb = 0; kb < nk; ++kb, ++g) {
            const int st = g % kChainRing;
            if (g >= kChainRing && (*abort_flag || !umma::mbar_wait(&wempty[st], (uint32_t)(g / kChainRing - 1) & 1u,
                                                                    2 * kWaitCycles))) {
              *abort_flag = 1;
              fail = true;
              break;
            }
            umma::mbar_arrive_expect_tx(&wfull[st], p == 3 ? (uint32_t)kOut * kBK * 2 : kRingBytes);
            umma::tma_load_2d(ring + (size_t)st * kRingBytes, &maps.w[p], &wfull[st], kb * kBK, 0);
          }
        }
      }
      // the last commit of every ring stage lands before the CTA ends
      for (int k = g < kChainRing ? 0 : g - kChainRing; k < g && !fail && !*abort_flag; ++k)
        if (!umma::mbar_wait(&wempty[k % kChainRing], (uint32_t)(k / kChainRing) & 1u, 2 * kWaitCycles))
          *abort_flag = 1;
    }
  } else if (warp == kEpiWarps) {
    // ---- inputs and MMA issue (one thread) ----
    if (umma::elect_one()) {
      auto load_x = [&](int tile) {
        umma::mbar_arrive_expect_tx(xfull, 2u * kSlabBytes);
        umma::tma_load_2d(H, &tx, xfull, 0, tile * kBM);
        umma::tma_load_2d(H + kSlabBytes, &tx, xfull, kBK, tile * kBM);
      };
      load_x(blockIdx.x);
      int g = 0;
      bool fail = false;
      for (int i = 0; i < my_tiles && !fail; ++i) {
        for (int p = 0; p < 7 && !fail; ++p) {
          const int e = 7 * i + p;  // epilogues that must be done
          if (*abort_flag || (e > 0 && !umma::mbar_wait(actr, (uint32_t)(e - 1) & 1u, kWaitCycles))) {
            fail = true;
            break;
          }
          if (p == 0) {
            // the last product of the tile before has read its operand (its
            // epilogue is done): the next input may replace it
            if (i > 0) load_x(blockIdx.x + i * gridDim.x);
            if (!umma::mbar_wait(xfull, (uint32_t)i & 1u, kWaitCycles)) {
              fail = true;
              break;
            }
          }
          umma::fence_after_sync();
          const uint32_t idesc = umma::idesc_bf16(kBM, p == 3 ? kOut : kHid);
          const int nk = chain_k(p);
          for (int kb = 0; kb < nk; ++kb, ++g) {
            const int st = g % kChainRing;
            if (!umma::mbar_wait(&wfull[st], (uint32_t)(g / kChainRing) & 1u, kWaitCycles)) {
              fail = true;
              break;
            }
            umma::fence_after_sync();
            const uint64_t da = umma::desc_sw128(umma::smem_u32(H + (size_t)kb * kSlabBytes));
            const uint64_t db = umma::desc_sw128(umma::smem_u32(ring + (size_t)st * kRingBytes));
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k) 
              umma::mma_bf16(tmem + chain_half(p), da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
            umma::mma_commit(&wempty[st]);
          }
          if (!fail) umma::mma_commit(accf);
        }
      }
      if (fail) *abort_flag = 1;
      umma::mma_commit(drain);
      if (!umma::mbar_wait(drain, 0u, kWaitCycles)) *abort_flag = 1;
    }
  } else {
    const int q = warp & 3, cg = warp >> 2;
    const int r = q * 32 + lane;  // row within the tile
    float inv = 0.0f;
    if (cg < 2) {  // sum of the batch's mask (whole numbers: exact in any order below 2^24)
      float c = 0.0f;
      for (int k = lane; k < a.B / kGatherRows; k += 32) c += a.cnt[k];
      for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      inv = 1.0f / fmaxf(c, 1.0f);
    }
    uint8_t* const hrow = H + (size_t)cg * kSlabBytes + (size_t)r * 128;  // this thread's 64 columns
    // the next operand is written: its MMAs may start
    auto handed = [&]() {
      umma::fence_proxy_async_smem();
      umma::fence_before_sync();
      __syncwarp();
      if (lane == 0) umma::mbar_arrive(actr);
    };
    bool stop = false;
    for (int i = 0; i < my_tiles && !stop; ++i) {
      const int tile = blockIdx.x + i * gridDim.x;
      const int row = tile * kBM + r;
      for (int p = 0; p < 7; ++p) {
        const int e = 7 * i + p;
        const uint32_t trow = tmem + chain_half(p) + ((uint32_t)(q * 32) << 16);
        const bool fwd = p < 3;
        const int l = fwd ? p : 6 - p;  // layer whose Z this is (p != 3)
        float* const zt = a.Z[p < 2 || p > 4 ? l : 0] + ((size_t)tile * kHid + cg * 64) * kBM + r;
        bf16* const ot = (fwd ? a.At[l] : a.dZt[p == 3 ? 0 : l]) + (size_t)(cg * 64) * a.B + row;
        // what the epilogue reads from memory is requested ahead of the MMAs' end
        float z[32];  // Z's first 32 columns; p == 3: 16 targets and, as bits, the mask
        if (p > 4) {
#pragma unroll
          for (int k = 0; k < 32; ++k) z[k] = zt[(size_t)k * kBM];
        } else if (p == 3 && cg < 2) {
          const float4* tt = reinterpret_cast<const float4*>(a.Tb + (size_t)row * kOut + cg * 16);
          const float4* xm = reinterpret_cast<const float4*>(a.Xb + (size_t)row * kInPad + 2 * kOut + cg * 16);
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const float4 t4 = k < 4 ? tt[k] : xm[k - 4];
            z[4 * k] = t4.x, z[4 * k + 1] = t4.y, z[4 * k + 2] = t4.z, z[4 * k + 3] = t4.w;
          }
        }
        if (*abort_flag) {
          stop = true;
          break;
        }
        if (!umma::mbar_wait(accf, (uint32_t)e & 1u, 2 * kWaitCycles)) {
          *abort_flag = 1;
          stop = true;
          break;
        }
        umma::fence_after_sync();
        if (p == 3) {
          uint32_t gv[8];
          float loss = 0.0f;
          const int c0 = cg * 16;
          if (cg < 2) {
            float v[16];
            umma::tmem_ld16(trow + (uint32_t)c0, v);
#pragma unroll
            for (int n = 0; n < 16; n += 2) {
              const uint32_t mk = __float_as_uint(z[16 + n / 2]);  // two mask entries
              const float y0 = v[n] + s_bias[3 * kHid + c0 + n];
              const float y1 = v[n + 1] + s_bias[3 * kHid + c0 + n + 1];
              const float d0 = __uint_as_float(mk << 16) * (y0 - z[n]);
              const float d1 = __uint_as_float(mk & 0xFFFF0000u) * (y1 - z[n + 1]);
              loss += d0 * d0;
              loss += d1 * d1;
              const __nv_bfloat162 g = __floats2bfloat162_rn(2.0f * d0 * inv, 2.0f * d1 * inv);
              gv[n / 2] = *reinterpret_cast<const uint32_t*>(&g);
            }
          } else {
#pragma unroll
            for (int n = 0; n < 8; ++n) gv[n] = 0u;
          }
          // dY: columns 16 cg .. 16 cg + 15 of the first slab (zeros from 32 on)
          uint8_t* const drow = H + (size_t)r * 128;
#pragma unroll
          for (int u = 0; u < 2; ++u)
            *reinterpret_cast<uint4*>(drow + (((2 * cg + u) ^ (r & 7)) << 4)) =
                make_uint4(gv[4 * u], gv[4 * u + 1], gv[4 * u + 2], gv[4 * u + 3]);
          handed();
          if (cg < 2) {
            uint16_t* const dy = reinterpret_cast<uint16_t*>(a.dYt) + (size_t)c0 * a.B + row;
#pragma unroll
            for (int n = 0; n < 16; ++n) dy[(size_t)n * a.B] = (uint16_t)(gv[n / 2] >> (16 * (n & 1)));
            for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
            if (lane == 0) a.lossp[(size_t)tile * 8 + warp] = loss;
          }
        } else {
          const ulonglong2* const b = reinterpret_cast<const ulonglong2*>(s_bias + l * kHid + cg * 64);
          uint32_t hv[32];  // the operand's 64 columns
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            uint32_t v[32];
            umma::tmem_request32(trow + (uint32_t)(cg * 64 + 32 * half), v);
            if (p == 4) {  // Z3 is still where product 2 left it, without the bias
              uint32_t zv[32];
              umma::tmem_request32(tmem + chain_half(2) + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * 64 + 32 * half),
                                   zv);
              umma::tmem_wait32(zv);
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                const ulonglong2 b4 = b[8 * half + (k >> 1)];
                unpack2(add2(pack2(__uint_as_float(zv[2 * k]), __uint_as_float(zv[2 * k + 1])), k & 1 ? b4.y : b4.x),
                        z[2 * k], z[2 * k + 1]);
              }
            } else if (!fwd && half == 1) {
#pragma unroll
              for (int k = 0; k < 32; ++k) z[k] = zt[(size_t)(32 + k) * kBM];
            }
            umma::tmem_wait32(v);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              if (fwd) {
                const ulonglong2 b4 = b[8 * half + (k >> 1)];
                hv[16 * half + k] = gelu_bf16x2(
                    add2(pack2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])), k & 1 ? b4.y : b4.x));
              } else {
                float g0, g1;
                unpack2(mul2(pack2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])),
                             gelu_grad2(pack2(z[2 * k], z[2 * k + 1]))),
                        g0, g1);
                const __nv_bfloat162 g = __floats2bfloat162_rn(g0, g1);
                hv[16 * half + k] = *reinterpret_cast<const uint32_t*>(&g);
              }
            }
            if (p < 6) {
#pragma unroll
              for (int u = 0; u < 4; ++u)
                *reinterpret_cast<uint4*>(hrow + (((4 * half + u) ^ (r & 7)) << 4)) =
                    make_uint4(hv[16 * half + 4 * u], hv[16 * half + 4 * u + 1], hv[16 * half + 4 * u + 2],
                               hv[16 * half + 4 * u + 3]);
            }
          }
          handed();
          // the stores run under the next product (which accumulates in the
          // other half of the TMEM)
          uint16_t* const o16 = reinterpret_cast<uint16_t*>(ot);
#pragma unroll
          for (int k = 0; k < 64; ++k) o16[(size_t)k * a.B] = (uint16_t)(hv[k >> 1] >> (16 * (k & 1)));
          if (p < 2) {
#pragma unroll 1
            for (int c0 = 0; c0 < 64; c0 += 32) {
              uint32_t v[32];
              umma::tmem_request32(trow + (uint32_t)(cg * 64 + c0), v);
              umma::tmem_wait32(v);
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                const ulonglong2 b4 = b[c0 / 4 + (k >> 1)];
                float z0, z1;
                unpack2(add2(pack2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])), k & 1 ? b4.y : b4.x), z0,
                        z1);
                zt[(size_t)(c0 + 2 * k) * kBM] = z0;
                zt[(size_t)(c0 + 2 * k + 1) * kBM] = z1;
              }
            }
          }
        }
      }
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0 && a.error) atomicExch(a.error, 1);
    wait_for_copies();
  }
  if (warp == 0) {
    umma::fence_after_sync();
    umma::tmem_dealloc(tmem, 512);
  }
}

// Weight gradients: dW[M x N] = dZ^T A with the batch as K, split over
// blockIdx.x; blockIdx.y is one 128-row piece of a layer's gradient:
//   0, 1 W1 (N = 128, the padded inputs), 2, 3 W2, 4, 5 W3, 6 W4 (32 rows)
// One thread loads both operands' slabs with TMA through a two-stage ring (two
// CTAs per SM) and issues the MMAs; the four warps write the accumulator
// transposed, part[split][piece][column][row], so that a warp's store is 128
// contiguous bytes.
constexpr int kPieces = 7;
constexpr int kWgStages = 2;
constexpr uint32_t kWgStageBytes = kSlabBytes + kRingBytes;
constexpr size_t kWgSmem = 1024 + (size_t)kWgStages * kWgStageBytes + 128;
constexpr long long kPartSplit = (long long)kPieces * kHid * kBM;  // floats of one split

struct WgMaps {
  CUtensorMap a[4], b[4];  // per layer: dZ^T (dY^T), activations^T
};

__global__ void __launch_bounds__(128, 2)
    k_weight_grad(const __grid_constant__ WgMaps maps, int k_slabs, float* __restrict__ part, int* __restrict__ error) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(base + (size_t)kWgStages * kWgStageBytes);
  uint64_t *full = bars, *empty = bars + kWgStages, *done = bars + 2 * kWgStages;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * kWgStages + 1);
  __shared__ int s_fail;
  const int piece = blockIdx.y, layer = piece >> 1, m0 = (piece & 1) * kBM;
  const int N = layer == 0 ? kInPad : kHid;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int s = 0; s < kWgStages; ++s) {
      umma::mbar_init(&full[s], 1);
      umma::mbar_init(&empty[s], 1);
    }
    umma::mbar_init(done, 1);
    umma::fence_barrier_init();
  }
  if (warp == 0) umma::tmem_alloc(tmem_slot, 256);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  if (warp == 0 && umma::elect_one()) {
    bool ok = true;
    const int k0 = blockIdx.x * k_slabs;
    const uint32_t idesc = umma::idesc_bf16(kBM, N);
    auto load = [&](int kb) {
      const int s = kb % kWgStages;
      uint8_t* sa = base + (size_t)s * kWgStageBytes;
      umma::mbar_arrive_expect_tx(&full[s], kSlabBytes + (uint32_t)N * kBK * 2);
      umma::tma_load_2d(sa, &maps.a[layer], &full[s], (k0 + kb) * kBK, m0);
      umma::tma_load_2d(sa + kSlabBytes, &maps.b[layer], &full[s], (k0 + kb) * kBK, 0);
    };
    for (int s = 0; s < kWgStages && s < k_slabs; ++s) load(s);
    for (int kb = 0; kb < k_slabs && ok; ++kb) {
      const int s = kb % kWgStages;
      const uint32_t par = (uint32_t)(kb / kWgStages) & 1u;
      if (!umma::mbar_wait(&full[s], par, kWaitCycles)) {
        ok = false;
        break;
      }
      umma::fence_after_sync();
      uint8_t* sa = base + (size_t)s * kWgStageBytes;
      const uint64_t da = umma::desc_sw128(umma::smem_u32(sa)), db = umma::desc_sw128(umma::smem_u32(sa + kSlabBytes));
#pragma unroll
      for (int k = 0; k < kBK / 16; ++k) umma::mma_bf16(tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
      umma::mma_commit(&empty[s]);
      if (kb + kWgStages < k_slabs) {
        if (!umma::mbar_wait(&empty[s], par, kWaitCycles)) {
          ok = false;
          break;
        }
        load(kb + kWgStages);
      }
    }
    umma::mma_commit(done);
    // the last commit of every stage
    for (int s = 0; s < kWgStages && s < k_slabs; ++s)
      ok = ok && umma::mbar_wait(&empty[s], (uint32_t)((k_slabs - 1 - s) / kWgStages) & 1u, kWaitCycles);
    if (!ok) s_fail = 1;
  }
  const bool got = umma::mbar_wait(done, 0, 2 * kWaitCycles);
  umma::fence_after_sync();
  const bool failed = __syncthreads_or(!got || s_fail) != 0;  // uniform: the TMEM loads below are warp-wide
  if (failed) {
    if (threadIdx.x == 0 && error) atomicExch(error, 1);
    wait_for_copies();
  } else if (layer < 3 || warp == 0) {
    float* const out = part + (size_t)blockIdx.x * kPartSplit + (size_t)piece * kHid * kBM + warp * 32 + lane;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 32) {
      float v[32];
      umma::tmem_ld32(trow + (uint32_t)c0, v);
#pragma unroll
      for (int k = 0; k < 32; ++k) out[(size_t)(c0 + k) * kBM] = v[k];
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    umma::fence_after_sync();
    umma::tmem_dealloc(tmem, 256);
  }
}

// AdamW (decoupled weight decay): c1 = 1 - beta1^t, c2 = 1 - beta2^t.
struct AdamwArgs {
  float lr, b1, b2, eps, wd, c1, c2;
};
__device__ __forceinline__ float adamw_one(const AdamwArgs& o, float* theta, float* m, float* v, float gi) {
  const float mi = o.b1 * *m + (1.0f - o.b1) * gi;
  const float vi = o.b2 * *v + (1.0f - o.b2) * gi * gi;
  *m = mi;
  *v = vi;
  const float mh = mi / o.c1, vh = vi / o.c2;
  const float th = *theta - o.lr * (mh / (sqrtf(vh) + o.eps) + o.wd * *theta);
  *theta = th;
  return th;
}
__global__ void k_adamw(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                        const float* __restrict__ g, long n, AdamwArgs o) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    adamw_one(o, theta + i, m + i, v + i, g[i]);
}

// The last kernel of a gradient or training step.  Blocks 0..159 take one
// 32 x 32 tile of a weight matrix each: the splits' partial sums (rows
// contiguous) added in split order, transposed through shared memory, then
// the gradient written (grad given) or AdamW applied and the bf16 copies of
// the weight and of its transpose written.  The next blocks take eight bias
// entries each, a warp summing a row of dZ^T lane by lane, and the last one
// sums the tiles' losses.
constexpr int kUpdTiles = 24 + 64 + 64 + 8;
constexpr int kUpdBias = (3 * kHid + kOut) / 8;
struct UpdArgs {
  const float* part;
  int splits;
  const bf16* dZt[3];
  const bf16* dYt;
  const float* lossp;
  const float* cnt;
  int B;
  float *theta, *m, *v, *grad, *loss;
  bf16 *W[4], *Wt[4];  // Wt[0] null: W1 has no transposed copy
  AdamwArgs opt;
};

__global__ void __launch_bounds__(256) k_update(const __grid_constant__ UpdArgs a) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int b = blockIdx.x;
  if (b < kUpdTiles) {
    __shared__ float tile[32][33];
    const int layer = b < 24 ? 0 : b < 88 ? 1 : b < 152 ? 2 : 3;
    const int t = b - (layer == 0 ? 0 : layer == 1 ? 24 : layer == 2 ? 88 : 152);
    const int tc = layer == 0 ? 3 : 8;  // tiles across
    const int r0 = 32 * (t / tc), c0 = 32 * (t % tc);
    const long off = layer == 0 ? kOffW1 : layer == 1 ? kOffW2 : layer == 2 ? kOffW3 : kOffW4;
    const int cols = layer == 0 ? kIn : kHid;
    const float* p = a.part + ((size_t)(2 * layer + r0 / kBM) * kHid + c0 + ty) * kBM + r0 % kBM + tx;
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
    for (int k = 0; k < a.splits; ++k, p += kPartSplit)
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += p[(size_t)(8 * u) * kBM];
#pragma unroll
    for (int u = 0; u < 4; ++u) tile[ty + 8 * u][tx] = s[u];  // [column][row]
    __syncthreads();
    if (a.grad) {
#pragma unroll
      for (int u = 0; u < 4; ++u) a.grad[off + (long)(r0 + ty + 8 * u) * cols + c0 + tx] = tile[tx][ty + 8 * u];
      return;
    }
    float th[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + ty + 8 * u;
      const long i = off + (long)r * cols + c0 + tx;
      th[u] = adamw_one(a.opt, a.theta + i, a.m + i, a.v + i, tile[tx][ty + 8 * u]);
      a.W[layer][(long)r * (layer == 0 ? kInPad : kHid) + c0 + tx] = __float2bfloat16_rn(th[u]);
    }
    if (layer == 0) return;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) tile[tx][ty + 8 * u] = th[u];
    __syncthreads();
    const int ld = layer == 3 ? kOutPad : kHid;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      a.Wt[layer][(long)(c0 + ty + 8 * u) * ld + r0 + tx] = __float2bfloat16_rn(tile[ty + 8 * u][tx]);
  } else if (b < kUpdTiles + kUpdBias) {
    const int w = (b - kUpdTiles) * 8 + ty;  // b1, b2, b3, b4
    const int layer = w / kHid, n = w % kHid;
    const bf16* row = (layer < 3 ? a.dZt[layer] : a.dYt) + (size_t)n * a.B;
    float s = 0.0f;
#pragma unroll 8
    for (int r = tx; r < a.B; r += 32) s += __bfloat162float(row[r]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tx == 0) {
      const long i = (layer == 0 ? kOffB1 : layer == 1 ? kOffB2 : layer == 2 ? kOffB3 : kOffB4) + n;
      if (a.grad)
        a.grad[i] = s;
      else
        adamw_one(a.opt, a.theta + i, a.m + i, a.v + i, s);
    }
  } else {
    __shared__ float red[2][8];
    float l = 0.0f, c = 0.0f;
    for (int k = threadIdx.x; k < a.B / kBM * 8; k += 256) l += a.lossp[k];
    for (int k = threadIdx.x; k < a.B / kGatherRows; k += 256) c += a.cnt[k];
    for (int o = 16; o > 0; o >>= 1) {
      l += __shfl_xor_sync(0xffffffffu, l, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (tx == 0) {
      red[0][ty] = l;
      red[1][ty] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) {
        l += red[0][w];
        c += red[1][w];
      }
      a.loss[0] = l * (1.0f / fmaxf(c, 1.0f));
      a.loss[1] = c;
    }
  }
}

// bf16 weights for the products from the fp32 parameters: W1 padded to 256 x 128,
// W2, W3, W4, and transposed copies W2^T, W3^T (256 x 256), W4^T (256 x 64).
__global__ void k_refresh(const float* __restrict__ th, bf16* __restrict__ W1, bf16* __restrict__ W2,
                          bf16* __restrict__ W3, bf16* __restrict__ W4, bf16* __restrict__ W2t,
                          bf16* __restrict__ W3t, bf16* __restrict__ W4t) {
  const long n1 = (long)kHid * kInPad, n2 = (long)kHid * kHid, n4 = (long)kHid * kOutPad;
  const long total = n1 + 2 * n2 + n4;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    if (t < n1) {
      const int r = (int)(t / kInPad), c = (int)(t % kInPad);
      W1[t] = __float2bfloat16_rn(c < kIn ? th[kOffW1 + (long)r * kIn + c] : 0.0f);
    } else if (t < n1 + n2) {
      const long u = t - n1;
      const int r = (int)(u / kHid), c = (int)(u % kHid);
      const bf16 w = __float2bfloat16_rn(th[kOffW2 + u]);
      W2[u] = w;
      W2t[(long)c * kHid + r] = w;
    } else if (t < n1 + 2 * n2) {
      const long u = t - n1 - n2;
      const int r = (int)(u / kHid), c = (int)(u % kHid);
      const bf16 w = __float2bfloat16_rn(th[kOffW3 + u]);
      W3[u] = w;
      W3t[(long)c * kHid + r] = w;
    } else {
      const long u = t - n1 - 2 * n2;  // W4^T entry (c, r): c < 256, r < 64
      const int c = (int)(u / kOutPad), r = (int)(u % kOutPad);
      const bf16 w = __float2bfloat16_rn(r < kOut ? th[kOffW4 + (long)r * kHid + c] : 0.0f);
      W4t[u] = w;
      if (r < kOut) W4[(long)r * kHid + c] = w;
    }
  }
}

// ---- host side ----------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  });
  return fn;
}

// Tensor map of a row-major bf16 matrix [rows x cols] read in boxes of
// 64 columns x box_rows rows with 128-byte swizzle.  The caller keeps every
// box inside the matrix (rows a multiple of box_rows, cols of 64).
bool make_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn || !ptr || ((uintptr_t)ptr & 15u) || cols % 64 || rows % box_rows) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int blocks_for_n(long n, int threads) {
  long b = (n + threads - 1) / threads;
  const long cap = 8L * sm_count();
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

struct vrm_mlp {
  int B = 0;       // training batch rows (multiple of 128)
  int splits = 1;  // K splits of the weight-gradient products
  int* err = nullptr;
  float *theta = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr, *part = nullptr, *loss = nullptr;
  bf16 *W1 = nullptr, *W2 = nullptr, *W3 = nullptr, *W4 = nullptr, *W2t = nullptr, *W3t = nullptr, *W4t = nullptr;
  bf16 *Xb = nullptr, *Xbt = nullptr;
  float *Tb = nullptr, *cnt = nullptr, *lossp = nullptr;
  float* Z[2] = {};
  bf16 *At[3] = {}, *dZt[3] = {}, *dYt = nullptr;
  CUtensorMap mW1, mW2, mW3, mW4;  // weights as B operands
  CUtensorMap half[4];             // the same, half of the rows at a time (CTA pairs)
  CUtensorMap mX;
  ChainMaps chain;
  WgMaps wg;
};

namespace vrm {

cudaError_t mlp_acts_alloc(MlpActs* a, int rows) {
  mlp_acts_free(a);
  const int rp = (rows + kBM - 1) / kBM * kBM;
  cudaError_t e = cudaMalloc(&a->X, (size_t)rp * kInPad * sizeof(bf16));
  if (e == cudaSuccess) e = cudaMemset(a->X, 0, (size_t)rp * kInPad * sizeof(bf16));
  if (e != cudaSuccess) {
    mlp_acts_free(a);
    return e;
  }
  if (!make_map(&a->mX, a->X, rp, kInPad, kBM)) {
    mlp_acts_free(a);
    return cudaErrorInvalidValue;
  }
  a->rows_pad = rp;
  return cudaSuccess;
}

void mlp_acts_free(MlpActs* a) {
  if (a->X) cudaFree(a->X);
  a->X = nullptr;
  a->rows_pad = 0;
}

bool mlp_input_map(CUtensorMap* m, const bf16* X, int rows_pad) { return make_map(m, X, rows_pad, kInPad, kBM); }

cudaError_t mlp_forward(vrm_mlp* net, const CUtensorMap& mX, int rows, const int* rows_dev, float* Y,
                        cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  const cudaError_t r = allow_smem<k_mlp_fused>(kFusedSmem);
  if (r != cudaSuccess) return r;
  const int ntiles = (rows + 2 * kBM - 1) / (2 * kBM), npair = sm_count() / 2;
  const int grid = 2 * (ntiles < npair ? ntiles : npair);
  FusedArgs fa;
  fa.bias = net->theta;
  fa.Y = Y;
  fa.rows = rows;
  fa.rows_dev = rows_dev;
  fa.error = net->err;
  k_mlp_fused<<<grid, kFusedThreads, kFusedSmem, s>>>(mX, net->half[0], net->half[1], net->half[2], net->half[3],
                                                      fa);
  note_launch();
  return cudaGetLastError();
}

}  // namespace vrm

namespace {

void free_mlp(vrm_mlp* n) {
  void* ptrs[] = {n->err, n->theta, n->m, n->v, n->grad, n->part, n->loss, n->W1, n->W2, n->W3, n->W4, n->W2t,
                  n->W3t, n->W4t, n->Xb, n->Xbt, n->Tb, n->cnt, n->lossp, n->Z[0], n->Z[1], n->At[0],
                  n->At[1], n->At[2], n->dZt[0], n->dZt[1], n->dZt[2], n->dYt};
  for (void* p : ptrs)
    if (p) cudaFree(p);
}

template <typename T>
cudaError_t zalloc(T** p, size_t count) {
  cudaError_t e = cudaMalloc((void**)p, sizeof(T) * count);
  if (e == cudaSuccess) e = cudaMemset(*p, 0, sizeof(T) * count);
  return e;
}

// Forward and backward pass of the current batch (Xb, Xbt, Tb) up to the
// partial weight gradients.
cudaError_t forward_backward(vrm_mlp* n, cudaStream_t s) {
  cudaError_t r = allow_smem<k_chain>(kChainSmem);
  if (r == cudaSuccess) r = allow_smem<k_weight_grad>(kWgSmem);
  if (r != cudaSuccess) return r;
  ChainArgs a;
  a.theta = n->theta;
  a.Xb = n->Xb;
  a.Tb = n->Tb;
  a.cnt = n->cnt;
  for (int l = 0; l < 3; ++l) {
    if (l < 2) a.Z[l] = n->Z[l];
    a.At[l] = n->At[l];
    a.dZt[l] = n->dZt[l];
  }
  a.dYt = n->dYt;
  a.lossp = n->lossp;
  a.B = n->B;
  a.error = n->err;
  const int tiles = n->B / kBM;
  k_chain<<<tiles < sm_count() ? tiles : sm_count(), kChainThreads, kChainSmem, s>>>(n->mX, n->chain, a);
  note_launch();
  k_weight_grad<<<dim3(n->splits, kPieces), 128, kWgSmem, s>>>(n->wg, n->B / kBK / n->splits, n->part, n->err);
  note_launch();
  return cudaGetLastError();
}

// The gradient of the batch into n->grad (opt null), or one AdamW step with it.
cudaError_t update(vrm_mlp* n, const AdamwArgs* opt, cudaStream_t s) {
  UpdArgs a;
  memset(&a, 0, sizeof(a));
  a.part = n->part;
  a.splits = n->splits;
  for (int l = 0; l < 3; ++l) a.dZt[l] = n->dZt[l];
  a.dYt = n->dYt;
  a.lossp = n->lossp;
  a.cnt = n->cnt;
  a.B = n->B;
  a.theta = n->theta;
  a.m = n->m;
  a.v = n->v;
  a.loss = n->loss;
  bf16* w[4] = {n->W1, n->W2, n->W3, n->W4};
  bf16* wt[4] = {nullptr, n->W2t, n->W3t, n->W4t};
  for (int l = 0; l < 4; ++l) {
    a.W[l] = w[l];
    a.Wt[l] = wt[l];
  }
  if (opt)
    a.opt = *opt;
  else
    a.grad = n->grad;
  k_update<<<kUpdTiles + kUpdBias + 1, 256, 0, s>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t refresh(vrm_mlp* n, cudaStream_t s) {
  const long total = (long)kHid * kInPad + 2L * kHid * kHid + (long)kHid * kOutPad;
  k_refresh<<<blocks_for_n(total, 256), 256, 0, s>>>(n->theta, n->W1, n->W2, n->W3, n->W4, n->W2t, n->W3t, n->W4t);
  note_launch();
  return cudaGetLastError();
}

cudaError_t gather(vrm_mlp* n, const bf16* X, const float* T, const int* idx, int rows, cudaStream_t s) {
  k_gather<<<n->B / kGatherRows, 256, 0, s>>>(X, T, idx, rows, n->B, n->Xb, n->Xbt, n->Tb, n->cnt,
                                                   ((uintptr_t)X & 3u) == 0);
  note_launch();
  return cudaGetLastError();
}

vrm_status check_err(vrm_mlp* n, cudaStream_t s) {
  int h = 0;
  if (cudaMemcpyAsync(&h, n->err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return VRM_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return VRM_ERR_CUDA;
  return h ? VRM_ERR_CUDA : VRM_OK;
}

bool adamw_ok(const vrm_adamw* a) {
  return a && a->lr >= 0 && a->beta1 >= 0 && a->beta1 < 1 && a->beta2 >= 0 && a->beta2 < 1 && a->eps >= 0 &&
         a->weight_decay >= 0 && std::isfinite(a->lr);
}

AdamwArgs adamw_args(const vrm_adamw* a, int32_t t) {
  const double c1 = 1.0 - std::pow((double)a->beta1, (double)t);
  const double c2 = 1.0 - std::pow((double)a->beta2, (double)t);
  return AdamwArgs{a->lr, a->beta1, a->beta2, a->eps, a->weight_decay, (float)c1, (float)c2};
}

}  // namespace

extern "C" {

vrm_status vrm_mlp_create(int32_t batch_rows, vrm_mlp** out) {
  if (!out) return VRM_ERR_ARG;
  *out = nullptr;
  if (batch_rows < kBM || batch_rows % kBM || batch_rows > (1 << 20)) return VRM_ERR_ARG;
  if (!encode_fn()) return VRM_ERR_UNSUPPORTED;
  vrm_mlp* n = new (std::nothrow) vrm_mlp();
  if (!n) return VRM_ERR_CUDA;
  const int B = batch_rows;
  n->B = B;
  // weight-gradient products: K = B split in at most 64 equal pieces of whole
  // 128-row blocks (a prime number of blocks above 64 goes unsplit: a step of
  // 67 blocks takes 146 us, of 127 259, between 83 for 64 and 110 for 128)
  int splits = 1;
  for (int d = 64; d >= 1; --d)
    if ((B / 128) % d == 0) {
      splits = d;
      break;
    }
  n->splits = splits;
  cudaError_t e = cudaSuccess;
#define MLP_ALLOC(p, cnt) \
  if (e == cudaSuccess) e = zalloc(&(n->p), (size_t)(cnt))
  MLP_ALLOC(err, 1);
  MLP_ALLOC(theta, kParams);
  MLP_ALLOC(m, kParams);
  MLP_ALLOC(v, kParams);
  MLP_ALLOC(grad, kParams);
  MLP_ALLOC(part, (size_t)splits * kPartSplit);
  MLP_ALLOC(loss, 2);
  MLP_ALLOC(W1, (size_t)kHid * kInPad);
  MLP_ALLOC(W2, (size_t)kHid * kHid);
  MLP_ALLOC(W3, (size_t)kHid * kHid);
  MLP_ALLOC(W4, (size_t)kOut * kHid);
  MLP_ALLOC(W2t, (size_t)kHid * kHid);
  MLP_ALLOC(W3t, (size_t)kHid * kHid);
  MLP_ALLOC(W4t, (size_t)kHid * kOutPad);
  MLP_ALLOC(Xb, (size_t)B * kInPad);
  MLP_ALLOC(Xbt, (size_t)kInPad * B);
  MLP_ALLOC(Tb, (size_t)B * kOut);
  MLP_ALLOC(cnt, B / kGatherRows);
  MLP_ALLOC(lossp, (size_t)B / kBM * 8);
  for (int l = 0; l < 3; ++l) {
    if (l < 2) MLP_ALLOC(Z[l], (size_t)B * kHid);
    MLP_ALLOC(At[l], (size_t)kHid * B);
    MLP_ALLOC(dZt[l], (size_t)kHid * B);
  }
  MLP_ALLOC(dYt, (size_t)kBM * B);
#undef MLP_ALLOC
  bool ok = e == cudaSuccess;
  // B operands: boxes of N rows; A operands: 128-row boxes
  ok = ok && make_map(&n->half[0], n->W1, kHid, kInPad, kBM) && make_map(&n->half[1], n->W2, kHid, kHid, kBM) &&
       make_map(&n->half[2], n->W3, kHid, kHid, kBM) && make_map(&n->half[3], n->W4, kOut, kHid, kOut / 2);
  ok = ok && make_map(&n->mW1, n->W1, kHid, kInPad, 256) && make_map(&n->mW2, n->W2, kHid, kHid, 256) &&
       make_map(&n->mW3, n->W3, kHid, kHid, 256) && make_map(&n->mW4, n->W4, kOut, kHid, 32) &&
       make_map(&n->mX, n->Xb, B, kInPad, kBM);
  CUtensorMap* cw = n->chain.w;
  ok = ok && make_map(&cw[4], n->W4t, kHid, kOutPad, 256) && make_map(&cw[5], n->W3t, kHid, kHid, 256) &&
       make_map(&cw[6], n->W2t, kHid, kHid, 256);
  cw[0] = n->mW1, cw[1] = n->mW2, cw[2] = n->mW3, cw[3] = n->mW4;
  for (int l = 0; l < 3; ++l)
    ok = ok && make_map(&n->wg.a[l], n->dZt[l], kHid, B, kBM) && make_map(&n->wg.b[l + 1], n->At[l], kHid, B, 256);
  ok = ok && make_map(&n->wg.a[3], n->dYt, kBM, B, kBM) && make_map(&n->wg.b[0], n->Xbt, kInPad, B, 128);
  if (!ok) {
    free_mlp(n);
    delete n;
    cudaGetLastError();
    return e == cudaSuccess ? VRM_ERR_UNSUPPORTED : VRM_ERR_CUDA;
  }
  *out = n;
  return VRM_OK;
}

void vrm_mlp_destroy(vrm_mlp* n) {
  if (!n) return;
  free_mlp(n);
  delete n;
}

vrm_status vrm_mlp_set_params(vrm_mlp* n, const float* theta, cudaStream_t s) {
  if (!n || !theta) return VRM_ERR_ARG;
  if (cudaMemcpyAsync(n->theta, theta, sizeof(float) * kParams, cudaMemcpyDefault, s) != cudaSuccess)
    return VRM_ERR_CUDA;
  if (cudaMemsetAsync(n->m, 0, sizeof(float) * kParams, s) != cudaSuccess) return VRM_ERR_CUDA;
  if (cudaMemsetAsync(n->v, 0, sizeof(float) * kParams, s) != cudaSuccess) return VRM_ERR_CUDA;
  if (refresh(n, s) != cudaSuccess) return VRM_ERR_CUDA;
  return VRM_OK;
}

vrm_status vrm_mlp_get_params(const vrm_mlp* n, float* theta, cudaStream_t s) {
  if (!n || !theta) return VRM_ERR_ARG;
  if (cudaMemcpyAsync(theta, n->theta, sizeof(float) * kParams, cudaMemcpyDefault, s) != cudaSuccess)
    return VRM_ERR_CUDA;
  return VRM_OK;
}

vrm_status vrm_mlp_forward(vrm_mlp* n, const uint16_t* X, int32_t rows, float* Y, cudaStream_t s) {
  if (!n || rows < 0 || (rows > 0 && (!X || !Y)) || ((uintptr_t)X & 15u)) return VRM_ERR_ARG;
  if (rows == 0) return VRM_OK;
  const int rp = (rows + kBM - 1) / kBM * kBM;
  CUtensorMap mX;
  if (!vrm::mlp_input_map(&mX, reinterpret_cast<const bf16*>(X), rp)) return VRM_ERR_ARG;
  if (vrm::mlp_forward(n, mX, rows, nullptr, Y, s) != cudaSuccess) return VRM_ERR_CUDA;
  return check_err(n, s);
}

vrm_status vrm_mlp_grads(vrm_mlp* n, const uint16_t* X, const float* T, int32_t rows, float* grad, float* loss,
                         cudaStream_t s) {
  if (!n || !X || !T || rows < 1 || rows > n->B) return VRM_ERR_ARG;
  if (gather(n, reinterpret_cast<const bf16*>(X), T, nullptr, rows, s) != cudaSuccess) return VRM_ERR_CUDA;
  if (forward_backward(n, s) != cudaSuccess || update(n, nullptr, s) != cudaSuccess) return VRM_ERR_CUDA;
  if (grad && cudaMemcpyAsync(grad, n->grad, sizeof(float) * kParams, cudaMemcpyDefault, s) != cudaSuccess)
    return VRM_ERR_CUDA;
  if (loss && cudaMemcpyAsync(loss, n->loss, sizeof(float) * 2, cudaMemcpyDefault, s) != cudaSuccess)
    return VRM_ERR_CUDA;
  return check_err(n, s);
}

vrm_status vrm_mlp_train_step(vrm_mlp* n, const uint16_t* X_all, const float* T_all, const int32_t* batch_idx,
                              int32_t rows, const vrm_adamw* hp, int32_t t, float* loss, cudaStream_t s) {
  if (!n || !X_all || !T_all || rows < 1 || rows > n->B || t < 1 || !adamw_ok(hp)) return VRM_ERR_ARG;
  if (gather(n, reinterpret_cast<const bf16*>(X_all), T_all, batch_idx, rows, s) != cudaSuccess) return VRM_ERR_CUDA;
  const AdamwArgs o = adamw_args(hp, t);
  if (forward_backward(n, s) != cudaSuccess || update(n, &o, s) != cudaSuccess) return VRM_ERR_CUDA;
  if (loss && cudaMemcpyAsync(loss, n->loss, sizeof(float) * 2, cudaMemcpyDefault, s) != cudaSuccess)
    return VRM_ERR_CUDA;
  return VRM_OK;
}

vrm_status vrm_mlp_adamw(vrm_mlp* n, const float* grad, const vrm_adamw* hp, int32_t t, cudaStream_t s) {
  if (!n || !grad || t < 1 || !adamw_ok(hp)) return VRM_ERR_ARG;
  k_adamw<<<blocks_for_n(kParams, 256), 256, 0, s>>>(n->theta, n->m, n->v, grad, kParams, adamw_args(hp, t));
  note_launch();
  if (refresh(n, s) != cudaSuccess) return VRM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? VRM_OK : VRM_ERR_CUDA;
}

vrm_status vrm_mlp_error(vrm_mlp* n, cudaStream_t s) {
  if (!n) return VRM_ERR_ARG;
  return check_err(n, s);
}

}  // extern "C"
