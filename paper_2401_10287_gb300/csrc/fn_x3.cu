// FP32 products on the 5th-generation tensor cores, to FP32 accuracy: the stream layers, the mean-field
// term and the orbitals of the FP32 local-energy pass.
//
// Every FP32 operand is the exact sum of three BF16 parts, x = x0 + x1 + x2 (8 significant
// bits each; rows by truncation, weights by rounding).  Of the nine partial products six are kept,
// x0 w0, x0 w1, x1 w0, x0 w2, x1 w1, x2 w0.  Truncated rows leave |x1| < 2^-7 |x| and |x2| < 2^-15 |x|,
// rounded weights |w1| <= 2^-8 |w| and |w2| <= 2^-17 |w|, so the three dropped products are below 2^-22.4
// of the product (8 million normal pairs: at most 2^-22.6, root mean square 2^-25.7, with the sign of
// the row's remainder); one FP32 rounding is up to 2^-24.  The tensor core adds in FP32 but truncates,
// so the leading products x0 w0 have an accumulator of their own and the five small ones another: one
// truncated addition per 16 k instead of one rounded addition per k.  Measured against FP64 (1024 x
// 128, k = 320, tanh-like rows, weights N(0, 1/k)): relative RMS error 2.9e-7, the sequential
// FP32 FMA chain 3.2e-7; k = 64: 0.8e-7 and 1.5e-7.
//
// Infinities: the leading part of an infinite operand is infinite and its further parts are NaN
// (inf - inf), so an infinite leading sum is the result, as in FP32.
//
// One CTA of 640 threads per SM:
//   warp 0         TMA: the three parts of a k-block's weights (3 x nt x 64, prepared in BF16)
//   warp 1         allocates tensor memory; one lane issues five tcgen05.mma per 16 k: x0 times
//                  the stacked [w0; w1] (N = 2 nt: both accumulators), x1 w0, x1 w1, x2 w0, x0 w2
//   warps 4..11    read the FP32 rows of the next k-block (any row addresses: gathered electrons
//                  of one spin), split them and write the parts into the swizzled operand tiles
//   warps 12..19   epilogue: a TMEM lane quarter and nt / 2 columns each; a warp first moves its
//                  sums to registers and hands the accumulators back, so that the MMAs of the
//                  next item run under the rest
// Two stages of 2 x 48 KB operand tiles.  Activations stay FP32 in memory and are split in the
// kernel: stored parts would move 6 instead of 4 bytes an element.
//
// Measured, N2 network (4 x 256, k_self 320) at 4096 walkers, per FP32 local-energy call: layers
// 35.1 ms on the FMA pipe -> 9.8 (0.13 PFLOP/s of FP32 products, 0.77 PFLOP/s of BF16 MMAs), mean
// field 3.0 -> 0.8, orbitals 6.6 -> 1.7; the call 48.1 -> 15.7.  What binds the layer kernel: about
// 106 KB per k-block into each SM (32 KB of rows, 48 KB of weights, residual and mean field),
// 17000 cycles per 128 x 128 item against 10400 for its MMAs alone; the first layer (one
// k-block) is bound by the epilogue, 8800 cycles per item.
#include <algorithm>

#include "fn_internal.cuh"
#include "fn_tc.cuh"
#include "fn_x3.cuh"

namespace fn {
namespace x3 {

using namespace tc;

constexpr int kNt = 128;                         // output columns per CTA
constexpr int kStages = 2;
constexpr int kPart = 128 * 128;                 // bytes of one operand tile: 128 rows x 64 bf16
constexpr int kStageBytes = 6 * kPart;           // x0 x1 x2 w0 w1 w2
constexpr int kThreads = 640;
constexpr int kConvWarps = 8;
constexpr int kTileBytes = 2048;                 // epilogue staging tile: 32 rows x 16 floats, two per warp
constexpr int kLaunchRegs = 96;
constexpr int kRegsLow = 40, kRegsConv = 64, kRegsEpi = 152;
// The launch holds 640 x 96 registers; the warpgroups' shares after setmaxnreg must fit.
static_assert(128 * (kRegsLow + 2 * kRegsConv + 2 * kRegsEpi) <= kThreads * kLaunchRegs, "register split above the launch");
constexpr size_t kSmem = 1024 + kStages * kStageBytes + kEpiWarps * 2 * kTileBytes + 256;

// The three BF16 parts of two floats, packed in pairs: each part is the leading 16 bits of what the
// earlier ones leave (truncation, so that packing is one byte permutation; the remainders are
// exact, the third one has at most 8 bits).
__device__ __forceinline__ void split3(uint64_t x, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  uint32_t a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(x));
  p0 = __byte_perm(a, b, 0x7632);
  const uint64_t r = sub_f2(x, pack_f2(__uint_as_float(a & 0xffff0000u), __uint_as_float(b & 0xffff0000u)));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(r));
  p1 = __byte_perm(a, b, 0x7632);
  const uint64_t q = sub_f2(r, pack_f2(__uint_as_float(a & 0xffff0000u), __uint_as_float(b & 0xffff0000u)));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(q));
  p2 = __byte_perm(a, b, 0x7632);
}

// 16 floats of one row to the warp's staging tile and out as a TMA tile store (rows x 16
// columns; 64-byte swizzle: 16-byte chunk c of row r sits at chunk c ^ (r / 2 mod 4), so that eight
// rows fall into different banks); the tile's previous store has been waited for.
__device__ __forceinline__ void store_tile(const CUtensorMap* map, float4* stg, int lane, const float (&v)[16], int x, int y) {
#pragma unroll
  for (int q = 0; q < 4; ++q) stg[4 * lane + (q ^ ((lane >> 1) & 3))] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  fence_proxy_async();
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(map, stg, x, y);
    bulk_commit();
  }
}

__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) *(float4*)(v + 4 * q) = __ldg((const float4*)p + q);
}
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&a)[8], uint32_t (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void load16(const float* p, float (&v)[16]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) *(float4*)(v + 4 * q) = __ldg((const float4*)p + q);
}

// Items of a CTA: the layer kernel walks over the T slabs of a row tile (h and sum z^2 of the
// tile stay in tensor memory); the GEMM and the orbitals take (slab, row tile) pairs.
template <int EPI>
__global__ void __launch_bounds__(kThreads, 1)
    k_x3(const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmX,
         const __grid_constant__ CUtensorMap tmY, Args a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float4* ystage = (float4*)(base + kStages * kStageBytes);
  uint64_t* full = (uint64_t*)((unsigned char*)ystage + kEpiWarps * 2 * kTileBytes);
  uint64_t* empty = full + kStages;
  uint64_t* accf = empty + kStages;              // [2]
  uint64_t* acce = accf + 2;                     // [2]
  uint64_t* mma_done = acce + 2;
  uint64_t* resf = mma_done + 1;                 // [8 warps][2 tiles] residual tile has arrived
  uint32_t* tmem_slot = (uint32_t*)(resf + 2 * kEpiWarps);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  // accumulators: one pair (leading | small, 2 x 128 columns) in the layer kernel, which keeps h
  // and sum z^2 in the other 256 columns; two pairs otherwise
  constexpr int NBUF = EPI == kLayer ? 1 : 2;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Shape& sh = a.sh;
  const int ctile = blockIdx.x, nkb = a.nkb, T = sh.T;
  const int my_tiles = a.tiles > (int)blockIdx.y ? (a.tiles - 1 - (int)blockIdx.y) / (int)gridDim.y + 1 : 0;
  const int inner = EPI == kLayer ? T : 1;       // items per tile
  const int n_items = my_tiles * inner;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full + s, 1 + kConvWarps); mbar_init(empty + s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf + b, 1); mbar_init(acce + b, kEpiWarps); }
    mbar_init(mma_done, 1);
    for (int w = 0; w < 2 * kEpiWarps; ++w) mbar_init(resf + w, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  pdl_wait();
  pdl_launch();
  const uint32_t tmem = *tmem_slot;
  const uint64_t deadline = globaltimer() + kWaitNs * 8 * (uint64_t)(my_tiles > 0 ? my_tiles : 1);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLow));
    if (warp == 0 && lane == 0) {
      int stage = 0, issued = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int item = 0; item < n_items && ok; ++item)
        for (int kb = 0; kb < nkb; ++kb) {
          if (*abort_flag || !mbar_wait(empty + stage, phase ^ 1u, deadline)) { ok = false; break; }
          mbar_expect_tx(full + stage, 3 * kPart);
          unsigned char* sB = base + stage * kStageBytes + 3 * kPart;
          for (int p = 0; p < 3; ++p)
            tma_load_2d(sB + p * kPart, &tmB, full + stage, p * a.ldw + kb * kBlockK, a.brow0 + ctile * kNt);
          ++issued;
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(a.status, kStatusTimeout);
      }
      // bounded wait for the copies in flight
      const uint64_t dl2 = globaltimer() + kWaitNs;
      for (int q = issued > kStages ? issued - kStages : 0; q < issued; ++q)
        mbar_wait(full + (q % kStages), (uint32_t)((q / kStages) & 1), dl2);
    } else if (warp == 1 && lane == 0) {
      const uint32_t id2 = idesc_bf16(128, 2 * kNt), id1 = idesc_bf16(128, kNt);
      const uint32_t base_u = smem_u32(base);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int item = 0; item < n_items && ok; ++item) {
        const int buf = NBUF == 2 ? item & 1 : 0;
        const uint32_t use = (uint32_t)(item / NBUF);
        if (*abort_flag || !mbar_wait(acce + buf, (use & 1u) ^ 1u, deadline)) { ok = false; break; }
        fence_after();
        const uint32_t d = tmem + (uint32_t)(buf * 2 * kNt), ds = d + kNt;
        for (int kb = 0; kb < nkb; ++kb) {
          if (*abort_flag || !mbar_wait(full + stage, phase, deadline)) { ok = false; break; }
          fence_after();
          const uint32_t s0 = base_u + (uint32_t)(stage * kStageBytes);
          const uint64_t x0 = sdesc(s0), x1 = sdesc(s0 + kPart), x2 = sdesc(s0 + 2 * kPart), w0 = sdesc(s0 + 3 * kPart),
                         w1 = sdesc(s0 + 4 * kPart), w2 = sdesc(s0 + 5 * kPart);
#pragma unroll
          for (int k4 = 0; k4 < kBlockK / 16; ++k4) {
            const uint64_t o = (uint64_t)(2 * k4);
            mma_bf16(d, x0 + o, w0 + o, id2, (kb != 0 || k4 != 0) ? 1u : 0u);
            mma_bf16(ds, x1 + o, w0 + o, id1, 1u);
            mma_bf16(ds, x1 + o, w1 + o, id1, 1u);
            mma_bf16(ds, x2 + o, w0 + o, id1, 1u);
            mma_bf16(ds, x0 + o, w2 + o, id1, 1u);
          }
          mma_commit(empty + stage);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (ok) mma_commit(accf + buf);
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(a.status, kStatusTimeout);
      }
      mma_commit(mma_done);
      mbar_wait(mma_done, 0u, globaltimer() + kWaitNs);
    }
  } else if (warp < 4 + kConvWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsConv));
    // a warp converts 16 rows of a k-block, four at a time (8 lanes x 8 floats cover a row's 64
    // columns); the next k-block's loads are issued as soon as the registers are free
    const int rw = (warp - 4) * 16, hl = lane >> 3, kl = 8 * (lane & 7);
    uint32_t soff[2];                            // swizzled offset of row rw + 4 i + hl, i mod 2 (+ 1024 for i >= 2)
#pragma unroll
    for (int i = 0; i < 2; ++i) soff[i] = (uint32_t)((rw + 4 * i + hl) * 128 + (((lane & 7) ^ ((4 * i + hl) & 7)) << 4));
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    const float* src = nullptr;                  // element 0 of the item's first row
    int roff = -1;                               // row rw + lane % 16 relative to it, -1: zero row
    auto next_item = [&](int item) {
      const int tile = (int)blockIdx.y + (item / inner) * (int)gridDim.y, r = rw + (lane & 15);
      if (EPI == kLayer) {
        src = a.A + ((int64_t)(item % inner) * sh.R + (int64_t)tile * 128) * a.lda;
        roff = r < sh.wpt * sh.N ? r * a.lda : -1;
      } else if (EPI == kPlain) {
        src = a.A + (int64_t)tile * 128 * a.lda;
        roff = (int64_t)tile * 128 + r < a.rows ? r * a.lda : -1;
      } else {
        const int t = tile / a.rtiles, w0 = (tile - t * a.rtiles) * a.wpc, w = w0 + r / a.n_s;
        const int64_t row0 = tile_row(w0, 0, sh.N, sh.wpt);
        src = a.A + ((int64_t)t * sh.R + row0) * a.lda;
        roff = r < a.wpc * a.n_s && w < sh.B ? (int)(tile_row(w, a.e0 + r % a.n_s, sh.N, sh.wpt) - row0) * a.lda : -1;
      }
    };
    ulonglong2 v[4][2];                          // 4 rows x 8 floats
    auto load = [&](int kb) {
      const int k = kb * kBlockK + kl;
      const float* p = src + k;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int o = __shfl_sync(0xffffffffu, roff, 4 * i + hl);
#pragma unroll
        for (int q = 0; q < 2; ++q)
          v[i][q] = o >= 0 && k + 4 * q < a.kd ? __ldg((const ulonglong2*)(p + o + 4 * q)) : make_ulonglong2(0ull, 0ull);
      }
    };
    if (n_items > 0) {
      next_item(0);
      load(0);
    }
    for (int item = 0; item < n_items && ok; ++item) {
      for (int kb = 0; kb < nkb; ++kb) {
        // warp-uniform, so that no lane waits for one that has given up
        const bool got = !*abort_flag && mbar_wait(empty + stage, phase ^ 1u, deadline);
        if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
        unsigned char* sA = base + stage * kStageBytes;
        const int left = a.kd - kb * kBlockK - kl;
        if (left < 8) {                          // columns beyond the contraction length
          const uint64_t keep1 = 0xffffffffull;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[i][0].x = left < 1 ? 0ull : (left < 2 ? v[i][0].x & keep1 : v[i][0].x);
            v[i][0].y = left < 3 ? 0ull : (left < 4 ? v[i][0].y & keep1 : v[i][0].y);
            v[i][1].x = left < 5 ? 0ull : (left < 6 ? v[i][1].x & keep1 : v[i][1].x);
            v[i][1].y = left < 7 ? 0ull : v[i][1].y & keep1;
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint4 p0, p1, p2;
          split3(v[i][0].x, p0.x, p1.x, p2.x);
          split3(v[i][0].y, p0.y, p1.y, p2.y);
          split3(v[i][1].x, p0.z, p1.z, p2.z);
          split3(v[i][1].y, p0.w, p1.w, p2.w);
          unsigned char* dst = sA + soff[i & 1] + (i >> 1) * 1024;
          *(uint4*)dst = p0;
          *(uint4*)(dst + kPart) = p1;
          *(uint4*)(dst + 2 * kPart) = p2;
        }
        if (kb + 1 < nkb) {
          load(kb + 1);
        } else if (item + 1 < n_items) {
          next_item(item + 1);
          load(0);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(full + stage);
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicOr(a.status, kStatusTimeout);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    const int q = warp & 3, r = q * 32 + lane;   // TMEM lane quarter; this thread's row
    const int ew = warp - 4 - kConvWarps;
    const int c0 = (ew >> 2) * 64;               // first of this warp's 64 columns
    const int n0 = ctile * kNt + c0;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    float4* stg0 = ystage + ew * (2 * kTileBytes / 16);
    constexpr int kTile4 = kTileBytes / 16;
    const int npieces = max(0, min(4, (a.ncols - n0 + 15) / 16));
    for (int item = 0; item < n_items; ++item) {
      const int buf = NBUF == 2 ? item & 1 : 0;
      const uint32_t use = (uint32_t)(item / NBUF);
      const int tile = (int)blockIdx.y + (item / inner) * (int)gridDim.y;
      const bool ok = !*abort_flag && mbar_wait(accf + buf, use & 1u, deadline);
      if (epilogue_any(!ok)) {
        if (ew == 0 && lane == 0) {
          *abort_flag = 1;
          atomicOr(a.status, kStatusTimeout);
        }
        // the residual tile fetched for this item is still in flight
        if (EPI == kLayer && a.residual && item > 0 && lane == 0) mbar_wait(resf + 2 * ew, 0u, globaltimer() + kWaitNs);
        break;
      }
      fence_after();
      float z[4][16];
      const uint32_t acc = tmem + lane_base + (uint32_t)(buf * 2 * kNt + c0);
      uint64_t odd = 0;                          // becomes NaN with the first value that is not finite
#pragma unroll
      for (int pc = 0; pc < 4; ++pc) {
        uint32_t u[16], s[16];
        tmem_ld16_nowait(acc + 16 * pc, u);
        tmem_ld16_nowait(acc + kNt + 16 * pc, s);
        tmem_wait_ld32(u, s);
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          const uint64_t v = add_f2(pack_f2(__uint_as_float(u[j]), __uint_as_float(u[j + 1])),
                                    pack_f2(__uint_as_float(s[j]), __uint_as_float(s[j + 1])));
          odd = fma_f2(v, 0ull, odd);
          unpack_f2(v, z[pc][j], z[pc][j + 1]);
        }
      }
      float odd0, odd1;
      unpack_f2(odd, odd0, odd1);
      if (__any_sync(0xffffffffu, !(odd0 + odd1 == 0.f))) {
        // An infinite operand has its value in the leading products; its further parts are NaN.
#pragma unroll
        for (int pc = 0; pc < 4; ++pc) {
          uint32_t u[16];
          tmem_ld16(acc + 16 * pc, u);
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (isinf(__uint_as_float(u[j]))) z[pc][j] = __uint_as_float(u[j]);
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce + buf);

      if (EPI == kLayer) {
        const int t = item % inner, wl = r / sh.N, w = tile * sh.wpt + wl;
        const bool valid = wl < sh.wpt && w < sh.B;
        const int64_t row = (int64_t)t * sh.R + (int64_t)tile * 128 + r;
        const float* mrow = a.Mterm + ((int64_t)t * sh.B + (valid ? w : 0)) * a.ncols + n0;
        const uint32_t th = tmem + lane_base + (uint32_t)(2 * kNt + c0);      // h; sum z^2 128 columns on
        // The residual (the layer input's columns of this thread) comes as TMA tiles of 32 rows x
        // 16 columns, one piece ahead, into the two staging tiles that the output leaves from:
        // row-per-thread global loads would cost a cache line per lane.
        auto fetch = [&](int it, int piece, int parity) {      // lane 0: residual tile of (item, piece)
          const int tl = (int)blockIdx.y + (it / inner) * (int)gridDim.y;
          mbar_expect_tx(resf + 2 * ew + parity, kTileBytes);
          tma_load_2d(stg0 + parity * kTile4, &tmX, resf + 2 * ew + parity, n0 + 16 * piece,
                      (int)((int64_t)(it % inner) * sh.R + (int64_t)tl * 128 + q * 32));
        };
        if (item == 0 && a.residual && lane == 0) fetch(0, 0, 0);
        bool got = true;
#pragma unroll
        for (int pc = 0; pc < 4; ++pc) {
          float4* stg = stg0 + (pc & 1) * kTile4;
          float m[16];
          load16(mrow + 16 * pc, m);
          // the other tile's store (previous piece) has been read: fetch the next residual there
          if (lane == 0) {
            bulk_wait_read0();
            if (a.residual && (pc < 3 || item + 1 < n_items)) fetch(pc < 3 ? item : item + 1, pc < 3 ? pc + 1 : 0, (pc + 1) & 1);
          }
          __syncwarp();
          // a tile's barrier completes twice per item: the phase parity of piece pc is pc >> 1
          if (a.residual) {
            const bool in = mbar_wait(resf + 2 * ew + (pc & 1), (uint32_t)(pc >> 1), deadline);
            got = __all_sync(0xffffffffu, in) && got;
          }
          float (&out)[16] = z[pc];              // in place
#pragma unroll
          for (int hc = 0; hc < 2; ++hc) {       // 8 columns at a time (register budget)
            const int cc = 16 * pc + 8 * hc;
            uint32_t hv[8], sq[8];
            if (t > 0) {
              tmem_ld8_nowait(th + cc, hv);
              tmem_ld8_nowait(th + kNt + cc, sq);
            }
            float res[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) res[j] = 0.f;
            if (a.residual) {
              *(float4*)res = stg[4 * lane + ((2 * hc) ^ ((lane >> 1) & 3))];
              *(float4*)(res + 4) = stg[4 * lane + ((2 * hc + 1) ^ ((lane >> 1) & 3))];
            }
            if (t == 0) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float h = tanhf(z[pc][8 * hc + j] + m[8 * hc + j]);
                out[8 * hc + j] = h + res[j];
                hv[j] = __float_as_uint(h);
                sq[j] = 0u;
              }
              tmem_st8(th + cc, hv);
              tmem_st8(th + kNt + cc, sq);
            } else {
              tmem_wait_ld16(hv, sq);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float zj = z[pc][8 * hc + j] + m[8 * hc + j], h = __uint_as_float(hv[j]), d = 1.f - h * h,
                            s2 = __uint_as_float(sq[j]);
                if (t < T - 1) {
                  out[8 * hc + j] = d * zj + res[j];
                  sq[j] = __float_as_uint(s2 + zj * zj);
                } else {
                  out[8 * hc + j] = d * zj - 2.f * h * d * s2 + res[j];
                }
              }
              if (t < T - 1) tmem_st8(th + kNt + cc, sq);
            }
          }
          if (!valid)
#pragma unroll
            for (int j = 0; j < 16; ++j) out[j] = 0.f;
          store_tile(&tmY, stg, lane, out, n0 + 16 * pc, (int)(row - lane));
        }
        if (!got && lane == 0) {                 // expired wait: reported; every warp ends at its next one
          *abort_flag = 1;
          atomicOr(a.status, kStatusTimeout);
        }
        __syncwarp();
        tmem_wait_st();
      } else if (EPI == kPlain) {
        const int64_t m = (int64_t)tile * 128 + r;
#pragma unroll
        for (int pc = 0; pc < 4; ++pc) {
          if (pc >= npieces) break;              // warp-uniform
          if (m < a.bias_rows) {
            float b[16];
            load16(a.bias + n0 + 16 * pc, b);
#pragma unroll
            for (int j = 0; j < 16; ++j) z[pc][j] += b[j];
          }
          if (lane == 0) bulk_wait_read0();
          __syncwarp();
          store_tile(&tmY, stg0, lane, z[pc], n0 + 16 * pc, tile * 128 + q * 32);   // rows past the end are clipped
        }
      } else {
        // phi = (w . h + g) env; a row's elements of one orbital lie n_s apart from the next
        // electron's: consecutive lanes write consecutive words
        const int t = tile / a.rtiles, w = (tile - t * a.rtiles) * a.wpc + r / a.n_s, jj = r % a.n_s;
        if (r < a.wpc * a.n_s && w < sh.B) {
          const int ldp = a.K * sh.N;
          const int64_t row = tile_row(w, a.e0 + jj, sh.N, sh.wpt);
          const int own = t - 1 - 3 * (a.e0 + jj), slot = t == 0 ? 0 : (own >= 0 && own < 3 && t < T - 1 ? 1 + own : -1);
          const float* env = a.envv + (int64_t)(a.poff + n0) * sh.R + row;
          float* keep = a.orbP + (row * 4 + (slot < 0 ? 0 : slot)) * ldp + a.poff;
          const int nn = a.n_s * a.n_s;
          int i = n0 % a.n_s;                    // orbital ko = k n_s + i
          float* phi = a.Phi + (int64_t)w * a.PW + a.phi_off + (int64_t)t * nn + jj + (int64_t)(n0 / a.n_s) * T * nn;
#pragma unroll
          for (int pc = 0; pc < 4; ++pc) {
            float ev[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) ev[j] = n0 + 16 * pc + j < a.ncols ? __ldg(env + (int64_t)(16 * pc + j) * sh.R) : 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int ko = n0 + 16 * pc + j;
              if (ko >= a.ncols) break;
              float p = z[pc][j];
              if (t == 0) p += a.bias[ko];
              if (slot >= 0) keep[ko] = p;
              phi[i * a.n_s] = p * ev[j];
              if (++i == a.n_s) { i = 0; phi += (int64_t)T * nn; }
            }
          }
        }
      }
    }
    if (lane == 0) bulk_wait0();                 // the output stores have completed
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---- prepared weights: [n][part][ldw] BF16, columns kd .. ldw - 1 zero ------------------
__global__ void k_split_weights(const float* __restrict__ blob, SplitList list, __nv_bfloat16* __restrict__ out) {
  pdl_wait();
  pdl_launch();
  const SplitEntry e = list.e[blockIdx.y];
  const int64_t n = (int64_t)e.rows * e.ldw;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / e.ldw;
    const int k = (int)(i - r * e.ldw);
    float v = 0.f;
    if (k < e.len1) v = blob[e.src1 + r * e.src_ld + k];
    else if (k < e.kd) v = blob[e.src2 + r * e.src_ld + (k - e.len1)];
    __nv_bfloat16* o = out + e.dst + r * 3 * e.ldw + k;
    __nv_bfloat16 p0 = __float2bfloat16_rn(v);
    if (__hisinf(p0) && !isinf(v)) p0 = __float2bfloat16_rz(v);   // the largest finite values stay finite
    const float r1 = v - __bfloat162float(p0);
    const __nv_bfloat16 p1 = __float2bfloat16_rn(r1);
    o[0] = p0;
    o[e.ldw] = p1;
    o[2 * e.ldw] = __float2bfloat16_rn(r1 - __bfloat162float(p1));
  }
}

void launch_split_weights(const float* blob, const SplitList& list, void* out, cudaStream_t st) {
  launch_k(false, k_split_weights, dim3(32, list.n), 256, 0, st, blob, list, (__nv_bfloat16*)out);
}

// The register split needs the full launch allocation: a kernel compiled to another count cannot run.
template <int EPI>
static bool registers_fit() {
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, k_x3<EPI>) == cudaSuccess) return fa.numRegs == kLaunchRegs;
  cudaGetLastError();
  return false;
}

bool available() {
  static const bool ok = tc_available() && registers_fit<kLayer>() && registers_fit<kPlain>() && registers_fit<kOrbital>();
  return ok;
}

template <int EPI>
static bool launch(const Args& a, const void* W, int64_t w_rows, const float* X, int64_t ldx, float* Y, int64_t y_cols, int64_t y_rows, int64_t ldy,
                   int sm_count, cudaStream_t st) {
  CUtensorMap tb, tx, ty;
  if (!make_map(&tb, W, 3 * (int64_t)a.ldw, w_rows, 3 * (int64_t)a.ldw, kNt)) return false;
  if (Y) {
    if (!make_tile_map_f32(&ty, Y, y_cols, y_rows, ldy)) return false;
  } else {
    ty = tb;
  }
  if (X) {
    if (!make_tile_map_f32(&tx, X, ldx, y_rows, ldx)) return false;
  } else {
    tx = tb;
  }
  const int ctiles = (a.ncols + kNt - 1) / kNt;
  const dim3 grid(ctiles, std::min(a.tiles, std::max(1, sm_count / ctiles)));
  cudaFuncSetAttribute(k_x3<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  launch_k(false, k_x3<EPI>, grid, kThreads, kSmem, st, tb, tx, ty, a);
  return true;
}

bool launch_layer(const Shape& sh, const float* X, int ldx, int k_self, const void* W, int ldw, const float* Mterm,
                  float* Y, int ldy, int residual, int h1, int* status, int sm_count, cudaStream_t st) {
  Args a{};
  a.sh = sh; a.tiles = sh.tiles; a.nkb = (k_self + kBlockK - 1) / kBlockK; a.kd = k_self; a.ncols = h1; a.ldw = ldw;
  a.A = X; a.lda = ldx; a.Mterm = Mterm; a.residual = residual; a.status = status;
  return launch<kLayer>(a, W, h1, residual ? X : nullptr, ldx, Y, ldy, (int64_t)sh.T * sh.R, ldy, sm_count, st);
}

bool launch_gemm(int64_t rows, int k, const float* A, int lda, const void* W, int ldw, int ncols, float* C,
                 const float* bias, int bias_rows, int* status, int sm_count, cudaStream_t st) {
  Args a{};
  a.sh.T = 1; a.rows = rows; a.tiles = (int)((rows + 127) / 128); a.nkb = (k + kBlockK - 1) / kBlockK; a.kd = k;
  a.ncols = ncols; a.ldw = ldw; a.A = A; a.lda = lda; a.bias = bias; a.bias_rows = bias_rows; a.status = status;
  return launch<kPlain>(a, W, ncols, nullptr, 0, C, ncols, rows, ncols, sm_count, st);
}

bool launch_orbitals(const Shape& sh, int spin, const float* HL, int h1, const void* W, int ldw, const float* bias,
                     int K, float* Phi, int64_t PW, const float* envv, float* orbP, int* status, int sm_count,
                     cudaStream_t st) {
  Args a{};
  a.sh = sh; a.n_s = spin ? sh.n_dn : sh.n_up; a.e0 = spin ? sh.n_up : 0; a.wpc = 128 / a.n_s;
  a.rtiles = (sh.B + a.wpc - 1) / a.wpc; a.tiles = a.rtiles * sh.T;
  a.nkb = (h1 + kBlockK - 1) / kBlockK; a.kd = h1; a.ncols = K * a.n_s; a.ldw = ldw; a.A = HL; a.lda = h1;
  a.K = K; a.poff = spin ? K * sh.n_up : 0; a.Phi = Phi; a.PW = PW;
  a.phi_off = spin ? (int64_t)K * sh.T * sh.n_up * sh.n_up : 0;
  a.envv = envv; a.orbP = orbP; a.bias = bias; a.status = status;
  return launch<kOrbital>(a, W, a.ncols, nullptr, 0, nullptr, 0, 0, 0, sm_count, st);
}

}  // namespace x3
}  // namespace fn
