// Register-tiled GEMM core of the FP32 and FP64 modes (no tensor cores: FP32 operands keep
// their 24 bits and FP64 theirs).  C[BM x BN] += A[BM x k] B[k x BN]:
//   * a CTA is WM warps stacked along the rows; a warp covers 4 TM rows x 8 TN columns, its
//     lanes 4 (rows) x 8 (columns), a lane TM x TN accumulators.  FP32 uses packed two-lane
//     FMAs (one instruction for two columns), so that shared-memory loads and address
//     arithmetic fit into the issue slots the FMA pipe leaves free;
//   * A stays row-major in shared memory (rows of 64 bytes of k, padded to 80 bytes: the 4
//     rows a warp reads together fall into different banks), so global tiles arrive by
//     16-byte asynchronous copies without a transpose; B rows are read as 16-byte vectors,
//     8 lanes x 16 bytes = one 128-byte wavefront;
//   * a ring of 3 stages, one CTA barrier per stage; the caller streams any number of
//     (slab, k-block) stages through it, so that the loads of the next slab run under the
//     epilogue of the present one.
// Copies fall back to single elements where a row stride is not a multiple of 16 bytes.
#pragma once
#include <stdint.h>

#include "fn_device.cuh"

namespace fn {
namespace simt {

constexpr int kStages = 3;
constexpr int kRowBytes = 64;                    // bytes of k per stage and row
constexpr int kRowPad = 80;                      // shared-memory stride of an A row

template <typename T> struct Vec;                // 16-byte vectors
template <> struct Vec<float> { using type = float4; static constexpr int n = 4; };
template <> struct Vec<double> { using type = double2; static constexpr int n = 2; };

template <typename T, int TM, int TN, int WM>
struct Tile {
  static constexpr int V = Vec<T>::n;
  static constexpr int BK = kRowBytes / (int)sizeof(T);
  static constexpr int BM = 4 * TM * WM, BN = 8 * TN;
  static constexpr int kThreads = 32 * WM;
  static constexpr int kABytes = BM * kRowPad;
  static constexpr int kStageBytes = kABytes + BK * BN * (int)sizeof(T);
  static constexpr int kRingBytes = kStages * kStageBytes;
};

// Asynchronous copy of `bytes` (<= N) bytes, the rest of the N zero-filled.
template <int N>
__device__ __forceinline__ void cp_zfill(uint32_t dst, const void* src, int bytes) {
  if constexpr (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(N), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One stage of A and B (k0 the first k of the stage, kd the contraction length).
//   A: rows_src(row) is the address of a tile row's element 0 (nullptr: zero row); with AT the
//      matrix is stored k-major, element (row, k) at rows_src(row) + k lda.
//   B: [kd][ldb], columns n0 .. ncols - 1; with BT stored n-major, element (k, n) at
//      n ldb + k.
// A transposed operand is copied element by element (adjacent threads on adjacent addresses).
template <typename Tl, typename T, bool VEC, bool AT, bool BT, typename RowSrc>
__device__ __forceinline__ void load_stage(unsigned char* stage, RowSrc rows_src, int64_t lda, int k0, int kd,
                                           int rows, const T* B, int64_t ldb, int n0, int ncols) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(stage), sb = sa + Tl::kABytes;
  constexpr int S = (int)sizeof(T);
  if constexpr (AT) {
#pragma unroll
    for (int q = 0; q < (Tl::BM * Tl::BK + Tl::kThreads - 1) / Tl::kThreads; ++q) {
      const int e = threadIdx.x + q * Tl::kThreads, row = e % Tl::BM, kk = e / Tl::BM;
      if (Tl::BM * Tl::BK % Tl::kThreads && e >= Tl::BM * Tl::BK) break;
      const bool in = row < rows && k0 + kk < kd;
      cp_zfill<S>(sa + row * kRowPad + kk * S, in ? (const void*)(rows_src(row) + (int64_t)(k0 + kk) * lda) : (const void*)B,
                  in ? S : 0);
    }
  } else {
    constexpr int CB = VEC ? 16 : S, CE = CB / S, CA = kRowBytes / CB;     // copies of CB bytes, CA per row
#pragma unroll
    for (int q = 0; q < (Tl::BM * CA + Tl::kThreads - 1) / Tl::kThreads; ++q) {
      const int e = threadIdx.x + q * Tl::kThreads, row = e / CA, k = k0 + (e % CA) * CE;
      if (Tl::BM * CA % Tl::kThreads && e >= Tl::BM * CA) break;
      const T* p = rows_src(row);
      const int left = p ? (kd - k) * S : 0;
      const int bytes = left < 0 ? 0 : (left < CB ? left : CB);
      cp_zfill<CB>(sa + row * kRowPad + (e % CA) * CB, bytes ? (const void*)(p + k) : (const void*)B, bytes);
    }
  }
  if constexpr (BT) {
#pragma unroll
    for (int q = 0; q < (Tl::BN * Tl::BK + Tl::kThreads - 1) / Tl::kThreads; ++q) {
      const int e = threadIdx.x + q * Tl::kThreads, kk = e % Tl::BK, n = e / Tl::BK;
      if (Tl::BN * Tl::BK % Tl::kThreads && e >= Tl::BN * Tl::BK) break;
      const bool in = n0 + n < ncols && k0 + kk < kd;
      cp_zfill<S>(sb + (kk * Tl::BN + n) * S, in ? (const void*)(B + (int64_t)(n0 + n) * ldb + k0 + kk) : (const void*)B,
                  in ? S : 0);
    }
  } else {
    constexpr int CB = VEC ? 16 : S, CE = CB / S, CN = Tl::BN / CE;
#pragma unroll
    for (int q = 0; q < (Tl::BK * CN + Tl::kThreads - 1) / Tl::kThreads; ++q) {
      const int e = threadIdx.x + q * Tl::kThreads, kk = e / CN, n = (e % CN) * CE;
      if (Tl::BK * CN % Tl::kThreads && e >= Tl::BK * CN) break;
      const int left = (k0 + kk < kd) ? (ncols - n0 - n) * S : 0;
      const int bytes = left < 0 ? 0 : (left < CB ? left : CB);
      cp_zfill<CB>(sb + (kk * Tl::BN + n) * S,
                   bytes ? (const void*)(B + (int64_t)(k0 + kk) * ldb + n0 + n) : (const void*)B, bytes);
    }
  }
}

template <typename T, int TM, int TN, bool TWO> struct Acc;

// FP32: accumulators as pairs of adjacent columns.  TWO: sums in two levels, each stage's products
// from zero in v and then added to s, so that a contraction of k terms rounds like one of 16 and one
// of k / 16 terms instead of one chain of k.  The value passes need it: the determinants multiply the
// roundings of their matrices by the inverse, and one chain over k = 128 .. 256 was most of the
// error of an FP32 gradient.  One packed addition per 16 FMAs; the first product of a stage is a
// multiplication, so nothing is cleared between stages.
template <int TM, int TN, bool TWO>
struct Acc<float, TM, TN, TWO> {
  uint64_t v[TM][TN / 2], s[TWO ? TM : 1][TWO ? TN / 2 : 1];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int p = 0; p < TN / 2; ++p) (TWO ? s[TWO ? i : 0][TWO ? p : 0] : v[i][p]) = 0ull;
  }
  __device__ __forceinline__ float get(int i, int j) const {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(TWO ? s[TWO ? i : 0][TWO ? j >> 1 : 0] : v[i][j >> 1]));
    return (j & 1) ? hi : lo;
  }
  // sa: this lane's row 0 of the stage's A tile; sb: this lane's column 0 of the B tile
  template <int BK, int BN>
  __device__ __forceinline__ void step(const unsigned char* sa, const float* sb) {
#pragma unroll
    for (int k = 0; k < BK; k += 2) {
      float2 a[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *(const float2*)(sa + 4 * i * kRowPad + k * 4);
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        uint64_t b[TN / 2];
#pragma unroll
        for (int g = 0; g < TN / 4; ++g) {
          const ulonglong2 u = *(const ulonglong2*)(sb + (k + kk) * BN + 32 * g);
          b[2 * g] = u.x;
          b[2 * g + 1] = u.y;
        }
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          uint64_t aa;
          const float s = kk ? a[i].y : a[i].x;
          asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(s));
#pragma unroll
          for (int p = 0; p < TN / 2; ++p) {
            if (TWO && k == 0 && kk == 0)
              asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v[i][p]) : "l"(aa), "l"(b[p]));
            else
              asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v[i][p]) : "l"(aa), "l"(b[p]));
          }
        }
      }
    }
    if constexpr (TWO)
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int p = 0; p < TN / 2; ++p) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s[i][p]) : "l"(v[i][p]));
  }
};

template <int TM, int TN, bool TWO>
struct Acc<double, TM, TN, TWO> {
  double v[TM][TN];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) v[i][j] = 0.0;
  }
  __device__ __forceinline__ double get(int i, int j) const { return v[i][j]; }
  template <int BK, int BN>
  __device__ __forceinline__ void step(const unsigned char* sa, const double* sb) {
#pragma unroll
    for (int k = 0; k < BK; k += 2) {
      double2 a[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *(const double2*)(sa + 4 * i * kRowPad + k * 8);
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        double b[TN];
#pragma unroll
        for (int g = 0; g < TN / 2; ++g) {
          const double2 u = *(const double2*)(sb + (k + kk) * BN + 16 * g);
          b[2 * g] = u.x;
          b[2 * g + 1] = u.y;
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) v[i][j] += (kk ? a[i].y : a[i].x) * b[j];
      }
    }
  }
};

// Lane coordinates: row of accumulator i is row0() + 4 i, column of accumulator j is
// col(j) (16-byte groups of V adjacent columns, 8 V apart).
template <typename Tl> __device__ __forceinline__ int lane_row0() {
  return (threadIdx.x >> 5) * (Tl::BM * 32 / Tl::kThreads) + ((threadIdx.x & 31) >> 3);
}
template <typename Tl> __device__ __forceinline__ int lane_col(int j) {
  return (threadIdx.x & 7) * Tl::V + (j / Tl::V) * 8 * Tl::V + j % Tl::V;
}

// Streams stages 0 .. n_stages - 1 through the ring: load(stage index, buffer) issues one
// stage's copies, done(acc, slab) is called after every `nk` stages with the finished
// accumulators (cleared afterwards).  TWO: two-level FP32 sums.
template <typename Tl, typename T, int TM, int TN, bool TWO, typename Load, typename Done>
__device__ __forceinline__ void stream(unsigned char* ring, int nk, int n_slabs, Load load, Done done) {
  const int total = nk * n_slabs;
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < total) load(s, ring + s * Tl::kStageBytes);
    cp_commit();
  }
  Acc<T, TM, TN, TWO> acc;
  acc.clear();
  const int a_off = lane_row0<Tl>() * kRowPad, b_off = Tl::kABytes + lane_col<Tl>(0) * (int)sizeof(T);
  int buf = 0, kb = 0, slab = 0;
  for (int it = 0; it < total; ++it) {
    cp_wait<kStages - 2>();
    __syncthreads();                              // stage `it` has arrived; stage it - 1 is consumed
    const int nb = buf == 0 ? kStages - 1 : buf - 1;
    if (it + kStages - 1 < total) load(it + kStages - 1, ring + nb * Tl::kStageBytes);
    cp_commit();
    const unsigned char* st = ring + buf * Tl::kStageBytes;
    acc.template step<Tl::BK, Tl::BN>(st + a_off, (const T*)(st + b_off));
    buf = buf == kStages - 1 ? 0 : buf + 1;
    if (++kb == nk) {
      done(acc, slab);
      acc.clear();
      kb = 0;
      ++slab;
    }
  }
}

}  // namespace simt
}  // namespace fn
