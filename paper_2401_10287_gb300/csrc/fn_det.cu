// Determinant stage and local-energy assembly (one CTA per walker).
//
// For every determinant k and spin block of n x n orbitals A (psi = sum_k
// det A_k,up det A_k,down, empty blocks have determinant 1):
//   * LU with partial pivoting in shared memory, one warp per spin block, lane =
//     matrix row, warp shuffles pick the first maximal |pivot|;
//   * C = A^{-1} by substitution, lane = right-hand-side column;
//   * for every coordinate t (one thread per (block, t) item):
//       g_t = tr(C d_t A),   q_t = tr((C d_t A)^2) = sum_i B_ii^2 + 2 sum_{i<j} B_ij B_ji,
//     and tr(C lap A) for the Laplacian slab, so that
//       d_t log|det A| = g_t,   lap log|det A| = tr(C lap A) - sum_t q_t;
//   * the K terms combine by a signed log-sum-exp with rho_k = D_k / psi:
//       grad log|psi| = sum_k rho_k g_k,
//       lap log|psi| = sum_k rho_k (lap_k + |g_k|^2) - |grad log|psi||^2,
//   * E_L = -1/2 (|grad|^2 + lap) + V_ee + V_ne + V_nn (Eqs. 2-3).
// All of it runs in the Det type (FP64 in the FP64 and BF16-mixed modes); FP32 mode takes FP64 for
// the energies of few electrons and for the gradient's seeds of blocks of at most 8 x 8.
#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "fn_device.cuh"
#include "fn_internal.cuh"
#include "fn_lu.cuh"
#include "fn_small.cuh"
#include "fn_tc.cuh"

namespace fn {

struct DetArgs {
  const void* Phi;
  int64_t PW;
  int K;
  double* e_local;
  double* log_psi;
  int8_t* sign;
  void* inv_out;      // value-pass backward seed rho_k A^{-T}, [B][K (nu^2 + nd^2)], or null
  const double* charges;
  double v_nn;
  int* status;
};

// One thread factorises one small matrix held in shared memory with element (i, j) at
// A[(i n + j) ST] (ST = number of matrices interleaved, so neighbouring threads touch
// neighbouring words).  Partial pivoting picks the first maximal |pivot|; the
// determinant is tracked as mantissa * 2^exponent so that a single log per matrix is
// needed; the pivot reciprocals are kept for the inverse.
template <typename Det>
__device__ void thread_lu(Det* A, int n, int ST, int* perm, Det* rcp, Det* ld_out, Det* sign_out) {
  Det sgn = 1, mant = 1;
  int expo = 0;
  bool singular = false;
  for (int i = 0; i < n; ++i) perm[i * ST] = i;
  for (int c = 0; c < n; ++c) {
    int piv = c;
    auto best = abs_key(A[(c * n + c) * ST]);
    for (int r = c + 1; r < n; ++r) {
      const auto v = abs_key(A[(r * n + c) * ST]);
      if (v > best) { best = v; piv = r; }
    }
    if (best == 0) { singular = true; break; }
    if (piv != c) {
      for (int j = 0; j < n; ++j) {
        const Det t = A[(c * n + j) * ST];
        A[(c * n + j) * ST] = A[(piv * n + j) * ST];
        A[(piv * n + j) * ST] = t;
      }
      const int tp = perm[c * ST]; perm[c * ST] = perm[piv * ST]; perm[piv * ST] = tp;
      sgn = -sgn;
    }
    const Det p = A[(c * n + c) * ST];
    const Det rp = (Det)1 / p;
    rcp[c * ST] = rp;
    int e;
    mant *= frexp(p, &e);
    expo += e;
    int e2;
    mant = frexp(mant, &e2);
    expo += e2;
    for (int r = c + 1; r < n; ++r) {
      const Det f = A[(r * n + c) * ST] * rp;
      A[(r * n + c) * ST] = f;
      for (int j = c + 1; j < n; ++j) A[(r * n + j) * ST] -= f * A[(c * n + j) * ST];
    }
  }
  if (singular) {
    *ld_out = 0;
    *sign_out = 0;
    return;
  }
  *sign_out = mant < 0 ? -sgn : sgn;
  *ld_out = f_log(f_abs(mant)) + (Det)expo * (Det)0.6931471805599453;
}

// C = A^{-1} from the factors of thread_lu (same interleaving): column j of C solves
// L U x = e_{perm^-1(j)}.
template <typename Det>
__device__ void thread_inverse(const Det* A, const int* perm, const Det* rcp, int n, int ST, Det* C) {
  for (int j = 0; j < n; ++j) {
    for (int i = 0; i < n; ++i) {
      Det y = perm[i * ST] == j ? (Det)1 : (Det)0;
      for (int k = 0; k < i; ++k) y -= A[(i * n + k) * ST] * C[(k * n + j) * ST];
      C[(i * n + j) * ST] = y;
    }
    for (int i = n - 1; i >= 0; --i) {
      Det x = C[(i * n + j) * ST];
      for (int k = i + 1; k < n; ++k) x -= A[(i * n + k) * ST] * C[(k * n + j) * ST];
      C[(i * n + j) * ST] = x * rcp[i * ST];
    }
  }
}

// Tangent item for an n x n block with n known at compile time: B = C D row by row with n
// independent accumulators (no serial dot-product chains), then g = tr B and q = tr(B^2)
// from the registers.  C is interleaved with stride ST; D is the slab in global memory.
template <int NN, typename Det, typename PhiT>
__device__ __forceinline__ void tangent_item_fixed(const Det* __restrict__ Cm, int ST, const PhiT* __restrict__ D,
                                                   Det* g_out, Det* q_out) {
  Det B[NN][NN];
  Det d[NN][NN];
#pragma unroll
  for (int m = 0; m < NN; ++m)
#pragma unroll
    for (int j = 0; j < NN; ++j) d[m][j] = widen<Det, PhiT>(D[m * NN + j]);
#pragma unroll
  for (int i = 0; i < NN; ++i) {
#pragma unroll
    for (int j = 0; j < NN; ++j) B[i][j] = 0;
#pragma unroll
    for (int m = 0; m < NN; ++m) {
      const Det c = Cm[(int64_t)(i * NN + m) * ST];
#pragma unroll
      for (int j = 0; j < NN; ++j) B[i][j] += c * d[m][j];
    }
  }
  Det g = 0, q = 0;
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    g += B[i][i];
    q += B[i][i] * B[i][i];
#pragma unroll
    for (int j = i + 1; j < NN; ++j) q += (Det)2 * B[i][j] * B[j][i];
  }
  *g_out = g;
  *q_out = q;
}

// Same for any n (serial dots; used for blocks larger than 8).
template <typename Det, typename PhiT>
__device__ void tangent_item_any(const Det* __restrict__ Cm, int ST, const PhiT* __restrict__ D, int n, Det* g_out,
                                 Det* q_out) {
  Det g = 0, q = 0;
  for (int i = 0; i < n; ++i) {
    for (int j = i; j < n; ++j) {
      Det bij = 0;
      for (int m = 0; m < n; ++m) bij += Cm[(int64_t)(i * n + m) * ST] * widen<Det, PhiT>(D[m * n + j]);
      if (j == i) {
        g += bij;
        q += bij * bij;
      } else {
        Det bji = 0;
        for (int m = 0; m < n; ++m) bji += Cm[(int64_t)(j * n + m) * ST] * widen<Det, PhiT>(D[m * n + i]);
        q += (Det)2 * bij * bji;
      }
    }
  }
  *g_out = g;
  *q_out = q;
}

template <typename Det, typename PhiT>
__device__ __forceinline__ void tangent_item(const Det* Cm, int ST, const PhiT* D, int n, Det* g, Det* q) {
  switch (n) {
    case 1: tangent_item_fixed<1>(Cm, ST, D, g, q); break;
    case 2: tangent_item_fixed<2>(Cm, ST, D, g, q); break;
    case 3: tangent_item_fixed<3>(Cm, ST, D, g, q); break;
    case 4: tangent_item_fixed<4>(Cm, ST, D, g, q); break;
    case 5: tangent_item_fixed<5>(Cm, ST, D, g, q); break;
    case 6: tangent_item_fixed<6>(Cm, ST, D, g, q); break;
    case 7: tangent_item_fixed<7>(Cm, ST, D, g, q); break;
    case 8: tangent_item_fixed<8>(Cm, ST, D, g, q); break;
    default: tangent_item_any(Cm, ST, D, n, g, q); break;
  }
}

// ---- double-FP32 tangent products (BF16-mixed mode) -------------------------------------
// In the BF16-mixed mode the orbital tangents D are FP32 values and C = A^-1 is FP64.  The
// products B = C D, g = tr B and q = tr(B^2) are evaluated in double-FP32 arithmetic on the
// FP32 pipe, which on this part runs 64 times as many operations per clock as the FP64
// pipe: C = c_hi + c_lo (two FP32 values, 48 significant bits), every D entry is exact in
// FP32, each product c_hi d is split exactly by an FMA (Dekker's two-product), sums are
// accumulated with Knuth's error-free two-sum and the small terms (c_lo d, the rounding
// errors) in a second FP32 word.  The result carries about 46 significant bits, converted to
// FP64 at the end; the LU, the inverse and every later step stay FP64.
__device__ __forceinline__ void ff_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (sh, sl) += (xh, xl) * (yh, yl) * scale, scale = 1 or 2 (exact)
__device__ __forceinline__ void ff_fma_acc(float xh, float xl, float yh, float yl, float scale, float& sh,
                                           float& sl) {
  const float p = __fmul_rn(xh, yh);
  float pe = __fmaf_rn(xh, yh, -p);
  pe = __fmaf_rn(xh, yl, __fmaf_rn(xl, yh, pe));
  float s, e;
  ff_two_sum(sh, __fmul_rn(p, scale), s, e);
  sh = s;
  sl = __fadd_rn(sl, __fmaf_rn(pe, scale, e));
}

template <int NN>
__device__ __forceinline__ void tangent_item_ff(const float* __restrict__ Ch, const float* __restrict__ Cl, int ST,
                                                const float* __restrict__ D, double* g_out, double* q_out) {
  float bh[NN][NN], bl[NN][NN];
#pragma unroll
  for (int i = 0; i < NN; ++i)
#pragma unroll
    for (int j = 0; j < NN; ++j) { bh[i][j] = 0.f; bl[i][j] = 0.f; }
#pragma unroll
  for (int m = 0; m < NN; ++m) {
    float d[NN];
#pragma unroll
    for (int j = 0; j < NN; ++j) d[j] = D[m * NN + j];
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      const float ch = Ch[(i * NN + m) * ST], cl = Cl[(i * NN + m) * ST];
#pragma unroll
      for (int j = 0; j < NN; ++j) {
        const float p = __fmul_rn(ch, d[j]);
        const float pe = __fmaf_rn(ch, d[j], -p);
        float s, e;
        ff_two_sum(bh[i][j], p, s, e);
        bh[i][j] = s;
        bl[i][j] = __fmaf_rn(cl, d[j], __fadd_rn(bl[i][j], __fadd_rn(e, pe)));
      }
    }
  }
  float gh = 0.f, gl = 0.f, qh = 0.f, ql = 0.f;
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    float s, e;
    ff_two_sum(gh, bh[i][i], s, e);
    gh = s;
    gl = __fadd_rn(gl, __fadd_rn(e, bl[i][i]));
    ff_fma_acc(bh[i][i], bl[i][i], bh[i][i], bl[i][i], 1.f, qh, ql);
#pragma unroll
    for (int j = i + 1; j < NN; ++j) ff_fma_acc(bh[i][j], bl[i][j], bh[j][i], bl[j][i], 2.f, qh, ql);
  }
  *g_out = (double)gh + (double)gl;
  *q_out = (double)qh + (double)ql;
}

template <typename Det, typename PhiT>
__device__ __forceinline__ bool tangent_item_split(const float* Ch, const float* Cl, int ST, const PhiT* D, int n,
                                                   Det* g, Det* q) {
  if constexpr (std::is_same<Det, double>::value && std::is_same<PhiT, float>::value) {
    switch (n) {
      case 1: tangent_item_ff<1>(Ch, Cl, ST, D, g, q); return true;
      case 2: tangent_item_ff<2>(Ch, Cl, ST, D, g, q); return true;
      case 3: tangent_item_ff<3>(Ch, Cl, ST, D, g, q); return true;
      case 4: tangent_item_ff<4>(Ch, Cl, ST, D, g, q); return true;
      case 5: tangent_item_ff<5>(Ch, Cl, ST, D, g, q); return true;
      case 6: tangent_item_ff<6>(Ch, Cl, ST, D, g, q); return true;
      case 7: tangent_item_ff<7>(Ch, Cl, ST, D, g, q); return true;
      case 8: tangent_item_ff<8>(Ch, Cl, ST, D, g, q); return true;
      default: return false;
    }
  }
  return false;
}

// Local-energy pass: one CTA per walker.  Threads 0..2K-1 factorise and invert the
// (determinant, spin) blocks; then every thread takes (block, coordinate) items
// g_t = tr(C d_t A), q_t = tr((C d_t A)^2) and tr(C lap A); then the determinant terms
// are combined and E_L assembled.
template <typename Det, typename Wlk, typename PhiT>
__global__ void __launch_bounds__(128) k_det_energy(const Wlk* r, const double* __restrict__ nuc,
                                                    Shape sh, DetArgs a) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int w = blockIdx.x, tid = threadIdx.x;
  const int N = sh.N, T = sh.T, K = a.K, NC = 3 * N, NM = 2 * K;
  const int ST = (int)round_up(NM, 32);
  const int ns[2] = {sh.n_up, sh.n_dn};
  const int nmax = max(ns[0], ns[1]);
  Det* A = (Det*)smem_raw;                                // [nmax^2][ST]
  Det* C = A + (int64_t)nmax * nmax * ST;                 // [nmax^2][ST]
  Det* rcp = C + (int64_t)nmax * nmax * ST;               // [nmax][ST]
  Det* ld2 = rcp + (int64_t)nmax * ST;                   // [NM]
  Det* sg2 = ld2 + NM;                                   // [NM]
  Det* gt = sg2 + NM;                                    // [NM][NC]
  Det* qt = gt + NM * NC;                                // [NM][NC]
  Det* lt = qt + NM * NC;                                // [NM]
  Det* gradk = lt + NM;                                  // [K][NC]
  Det* lapk = gradk + K * NC;                            // [K]
  Det* rho = lapk + K;                                   // [K]
  Det* red = rho + K;                                    // [128]
  int* perm = (int*)(red + 128);                         // [nmax][ST]
  // double-FP32 copies of C (BF16-mixed mode): [nmax^2][ST] high words, then low words
  constexpr bool kSplit = std::is_same<Det, double>::value && std::is_same<PhiT, float>::value;
  float* Ch = (float*)(perm + (int64_t)nmax * ST);
  float* Cl = Ch + (int64_t)nmax * nmax * ST;
  const PhiT* Phi = (const PhiT*)a.Phi + (int64_t)w * a.PW;
  const int64_t blk_off[2] = {0, (int64_t)K * T * ns[0] * ns[0]};
  // value slabs of every block, interleaved by block (thread 2k + spin)
  for (int sp = 0; sp < 2; ++sp) {
    const int nn = ns[sp] * ns[sp];
    for (int e = tid; e < K * nn; e += blockDim.x) {
      const int k = e / nn, idx = e % nn;
      A[(int64_t)idx * ST + 2 * k + sp] = widen<Det, PhiT>(Phi[blk_off[sp] + (int64_t)k * T * nn + idx]);
    }
  }
  __syncthreads();
  if (tid < NM) {
    const int n = ns[tid & 1];
    if (n == 0) {
      ld2[tid] = 0;
      sg2[tid] = 1;
    } else {
      thread_lu<Det>(A + tid, n, ST, perm + tid, rcp + tid, ld2 + tid, sg2 + tid);
      if (sg2[tid] != 0) thread_inverse<Det>(A + tid, perm + tid, rcp + tid, n, ST, C + tid);
      else for (int e = 0; e < n * n; ++e) C[(int64_t)e * ST + tid] = 0;
      if (kSplit && n <= 8) {
        for (int e = 0; e < n * n; ++e) {
          const double c = (double)C[(int64_t)e * ST + tid];
          const float ch = __double2float_rn(c);
          Ch[(int64_t)e * ST + tid] = ch;
          Cl[(int64_t)e * ST + tid] = __double2float_rn(c - (double)ch);
        }
      }
    }
  }
  __syncthreads();
  // items: (block p, coordinate t < NC) and (block p, Laplacian)
  const int per = NC + 1;
  for (int it = tid; it < NM * per; it += blockDim.x) {
    const int p = it / per, tr = it % per;
    const int k = p >> 1, sp = p & 1, n = ns[sp];
    if (n == 0) {
      if (tr < NC) { gt[p * NC + tr] = 0; qt[p * NC + tr] = 0; } else { lt[p] = 0; }
      continue;
    }
    const Det* Cm = C + p;
    const int t = tr < NC ? 1 + tr : T - 1;
    const PhiT* D = Phi + blk_off[sp] + (int64_t)k * T * n * n + (int64_t)t * n * n;
    if (tr < NC) {
      Det g, q;
      if (!tangent_item_split<Det, PhiT>(Ch + p, Cl + p, ST, D, n, &g, &q)) tangent_item<Det, PhiT>(Cm, ST, D, n, &g, &q);
      gt[p * NC + tr] = g;
      qt[p * NC + tr] = q;
    } else {
      Det l = 0;
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) l += Cm[(int64_t)(j * n + i) * ST] * widen<Det, PhiT>(D[i * n + j]);
      lt[p] = l;
    }
  }
  __syncthreads();
  for (int e = tid; e < K * NC; e += blockDim.x) {
    const int k = e / NC, t = e % NC;
    gradk[e] = gt[(2 * k) * NC + t] + gt[(2 * k + 1) * NC + t];
  }
  for (int k = tid; k < K; k += blockDim.x) {
    Det qs = 0;
    for (int t = 0; t < NC; ++t) qs += qt[(2 * k) * NC + t] + qt[(2 * k + 1) * NC + t];
    lapk[k] = lt[2 * k] + lt[2 * k + 1] - qs;
  }
  __syncthreads();
  if (tid == 0) {
    Det m = -INFINITY;
    for (int k = 0; k < K; ++k) {
      const Det sk = sg2[2 * k] * sg2[2 * k + 1];
      if (sk != 0 && ld2[2 * k] + ld2[2 * k + 1] > m) m = ld2[2 * k] + ld2[2 * k + 1];
    }
    Det S = 0;
    for (int k = 0; k < K; ++k) {
      const Det sk = sg2[2 * k] * sg2[2 * k + 1];
      rho[k] = sk != 0 ? sk * f_exp(ld2[2 * k] + ld2[2 * k + 1] - m) : (Det)0;
      S += rho[k];
    }
    for (int k = 0; k < K; ++k) rho[k] = S != 0 ? rho[k] / S : (Det)0;
    red[0] = m + f_log(f_abs(S));
    red[1] = S > 0 ? 1 : (S < 0 ? -1 : 0);
  }
  __syncthreads();
  const double lpsi = (double)red[0];
  const int sgn = (int)red[1];
  __syncthreads();
  // E_kin = -1/2 (|grad log psi|^2 + lap log psi) = -1/2 sum_k rho_k (lap_k + |g_k|^2)
  Det kin = 0;
  for (int k = tid; k < K; k += blockDim.x) {
    Det g2 = 0;
    for (int t = 0; t < NC; ++t) g2 += gradk[k * NC + t] * gradk[k * NC + t];
    kin += rho[k] * (lapk[k] + g2);
  }
  double pot = 0.0;
  const Wlk* rw = r + (int64_t)w * N * 3;
  for (int p = tid; p < N * N; p += blockDim.x) {
    const int i = p / N, j = p % N;
    if (j <= i) continue;
    const double dx = (double)rw[3 * i] - (double)rw[3 * j], dy = (double)rw[3 * i + 1] - (double)rw[3 * j + 1],
                 dz = (double)rw[3 * i + 2] - (double)rw[3 * j + 2];
    pot += 1.0 / sqrt(dx * dx + dy * dy + dz * dz);
  }
  for (int p = tid; p < N * sh.M; p += blockDim.x) {
    const int i = p / sh.M, m = p % sh.M;
    const double dx = (double)rw[3 * i] - nuc[3 * m], dy = (double)rw[3 * i + 1] - nuc[3 * m + 1],
                 dz = (double)rw[3 * i + 2] - nuc[3 * m + 2];
    pot -= a.charges[m] / sqrt(dx * dx + dy * dy + dz * dz);
  }
  red[tid] = (Det)(-0.5) * kin + (Det)pot;
  __syncthreads();
  for (int off = 64; off > 0; off >>= 1) {
    if (tid < off) red[tid] += red[tid + off];
    __syncthreads();
  }
  if (tid == 0) {
    const double e = (double)red[0] + a.v_nn;
    a.e_local[w] = e;
    if (a.log_psi) a.log_psi[w] = lpsi;
    if (a.sign) a.sign[w] = (int8_t)sgn;
    if (sgn == 0) atomicOr(a.status, kStatusSingular);
    else if (!isfinite(e) || !isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
  }
}

// ---- local-energy pass on 8-lane groups (BF16-mixed mode, blocks of up to 8 electrons) ----
// One CTA of 128 threads per walker, in 16 groups of 8 lanes; lane r of a group holds row r
// of one (determinant, spin) block.  Every lane works in every phase, so no thread waits on
// a barrier while a few others factorise, and no thread holds a whole matrix in registers:
//   1. Gauss-Jordan elimination with partial pivoting, in place, in FP64 registers, the pivot
//      row found by a group reduction and broadcast by shuffles.  (Column c of the row takes the
//      inverse's column of the pivot row once c is eliminated: the numbers of the elimination of
//      [A | I] with two thirds of its FP64 operations and shuffles.)  The rows are not swapped:
//      the lane that supplies column c's pivot ends with row c of C = A^-1.  The unused rows
//      receive the updates of an LU factorisation, so the pivots are those of the one-thread
//      LU (log|det| agrees with it to rounding, 1e-14 in log|psi| measured).  The same lanes
//      form the Laplacian trace tr(C lap A) in FP64 and store C as double-FP32 rows.
//   2. Tangent items (block, two coordinates): lane r forms row r of B = C d_t A in double-FP32
//      arithmetic (the operations of the one-thread items: from the same C they give the
//      same entries), then g = tr B and q = tr(B^2) from the rows staged in shared memory
//      and a double-FP32 reduction over the group.  The two coordinates are the two words of
//      packed FP32 instructions: half the issue slots for the same roundings.
//      N2, 4096 walkers: [A | I] and one coordinate per instruction 2.30 ms, this 1.74 (Si-, 1031
//      walkers: 1.24 -> 0.84); what is left is FP64 and the chains of the double-FP32 sums.
//   3. The determinant terms are combined and E_L assembled as in k_det_energy.
constexpr int kGrpN = 8;                 // rows per group (largest block of this kernel)
constexpr int kGrpCP = kGrpN + 1;        // padded row of a staged C copy (floats)
constexpr int kGrpBS = kGrpN + 1;        // padded row of a staged B row (pairs: two coordinates)

__host__ __device__ inline size_t smem_det_energy_grp(int N, int K) {
  const int NM = 2 * K, NC = 3 * N;
  return sizeof(double) * ((size_t)2 * NM * NC + 3 * NM + (size_t)K * NC + 2 * K + 128) +
         sizeof(float) * ((size_t)NM * 2 * kGrpN * kGrpCP + 2 * 16 * 8 * kGrpBS);
}

// (s, e) = a - np, the rounding error of the difference in e; np holds the negated second term
// (packed FP32 has no negated operand: products are formed negated and subtracted, the same roundings).
__device__ __forceinline__ void ff2_two_diff(uint64_t a, uint64_t np, uint64_t& s, uint64_t& e) {
  s = tc::sub_f2(a, np);
  const uint64_t bb = tc::sub_f2(s, a);
  e = tc::sub_f2(tc::sub_f2(a, tc::sub_f2(s, bb)), tc::add_f2(np, bb));
}

// (h, l) += the (h, l) of the lane `off` away (double-FP32 sum, error-free on the high words)
__device__ __forceinline__ void ff2_add_xor(uint64_t& h, uint64_t& l, int off) {
  const uint64_t oh = __shfl_xor_sync(0xffffffffu, h, off), ol = __shfl_xor_sync(0xffffffffu, l, off);
  const uint64_t s = tc::add_f2(h, oh), bb = tc::sub_f2(s, h);
  const uint64_t e = tc::add_f2(tc::sub_f2(h, tc::sub_f2(s, bb)), tc::sub_f2(oh, bb));
  h = s;
  l = tc::add_f2(tc::add_f2(l, ol), e);
}

// Row r of B = C D for two consecutive tangent slabs of an M x M block (D1 = D0 + M^2), the slabs in
// the words of a pair: M double-FP32 accumulators each, the operations and order of
// tangent_item_ff's inner loop.
template <int M>
__device__ __forceinline__ void ff_row2(const float* __restrict__ chr, const float* __restrict__ clr,
                                        const float* __restrict__ D0, uint64_t (&bh)[kGrpN], uint64_t (&bl)[kGrpN]) {
  const float* D1 = D0 + M * M;
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const float c = chr[m], l = clr[m];
    const uint64_t ch = tc::pack_f2(c, c), nch = tc::pack_f2(-c, -c), cl = tc::pack_f2(l, l);
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const uint64_t d = tc::pack_f2(D0[m * M + j], D1[m * M + j]);
      const uint64_t np = tc::mul_f2(nch, d), pe = tc::fma_f2(ch, d, np);
      uint64_t sum, e;
      ff2_two_diff(bh[j], np, sum, e);
      bh[j] = sum;
      bl[j] = tc::fma_f2(cl, d, tc::add_f2(bl[j], tc::add_f2(e, pe)));
    }
  }
}

template <typename Wlk>
__global__ void __launch_bounds__(128, 4) k_det_energy_grp(const Wlk* r, const double* __restrict__ nuc,
                                                           Shape sh, DetArgs a) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int w = blockIdx.x, tid = threadIdx.x;
  const int N = sh.N, T = sh.T, K = a.K, NC = 3 * N, NM = 2 * K;
  const int ns[2] = {sh.n_up, sh.n_dn};
  // g and q of every item as double-FP32 pairs (converted to FP64 in the reductions, where
  // every lane of a warp has work: an FP64 instruction costs the same warp slot with one
  // active lane as with 32)
  float2* gt = (float2*)smem_raw;                         // [NM][NC]
  float2* qt = gt + NM * NC;                              // [NM][NC]
  double* lt = (double*)(qt + NM * NC);                   // [NM]
  double* ld2 = lt + NM;                                  // [NM]
  double* sg2 = ld2 + NM;                                 // [NM]
  double* gradk = sg2 + NM;                               // [K][NC]
  double* lapk = gradk + K * NC;                          // [K]
  double* rho = lapk + K;                                 // [K]
  double* red = rho + K;                                  // [128]
  float* Cs = (float*)(red + 128);                        // [NM][2][8][9]: rows of C, high then low words
  uint64_t* Bs = (uint64_t*)(Cs + NM * 2 * kGrpN * kGrpCP);               // [16 groups][8 rows][9 pairs]: B rows of an item
  const float* Phi = (const float*)a.Phi + (int64_t)w * a.PW;
  const int64_t blk_off[2] = {0, (int64_t)K * T * ns[0] * ns[0]};
  const int lane = tid & 31, gid = tid >> 3, rr = tid & 7;
  const int gbase = lane & ~7;                            // the group's first lane in the warp

  // 1. factorisation, 16 blocks at a time (every lane runs every shuffle)
  for (int p0 = 0; p0 < NM; p0 += 16) {
    const int p = p0 + gid;
    const bool live = p < NM;
    const int n = live ? ns[p & 1] : 0;
    const float* Ab = Phi + blk_off[p & 1] + (int64_t)(p >> 1) * T * n * n;     // value slab of the block
    double av[kGrpN];
#pragma unroll
    for (int j = 0; j < kGrpN; ++j) av[j] = (rr < n && j < n) ? widen<double, float>(Ab[rr * n + j]) : 0.0;
    bool used = rr >= n, singular = false;
    int mycol = -1, pc[kGrpN];
    double mant = 1.0;
    int expo = 0;
#pragma unroll
    for (int c = 0; c < kGrpN; ++c) {
      const bool col = c < n;
      // pivot: the unused row of largest |a_c| (the first such row on ties)
      unsigned long long key = (!used && col) ? abs_key(av[c]) : 0ull;
      int li = rr;
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, off);
        const int ol = __shfl_xor_sync(0xffffffffu, li, off);
        if (ok > key || (ok == key && ol < li)) { key = ok; li = ol; }
      }
      pc[c] = li;
      if (col && key == 0ull) singular = true;
      double pa[kGrpN];
#pragma unroll
      for (int j = 0; j < kGrpN; ++j) pa[j] = __shfl_sync(0xffffffffu, av[j], gbase + li);
      if (col && !singular) {
        const double piv = pa[c];
        const double rp = 1.0 / piv;
        int e;
        mant *= frexp(piv, &e);
        expo += e;
        int e2;
        mant = frexp(mant, &e2);
        expo += e2;
        if (rr == li) {
#pragma unroll
          for (int j = 0; j < kGrpN; ++j) av[j] = j == c ? rp : pa[j] * rp;
          used = true;
          mycol = c;
        } else {
          const double f = av[c] * rp;
#pragma unroll
          for (int j = 0; j < kGrpN; ++j) av[j] = j == c ? -f : av[j] - f * pa[j];
        }
      }
    }
    // log|det| and its sign: the pivots' product (mantissa x 2^exponent) and the parity of
    // the permutation column c -> pivot row pc[c]
    int par = 0;
#pragma unroll
    for (int i = 0; i < kGrpN; ++i)
#pragma unroll
      for (int j = i + 1; j < kGrpN; ++j)
        if (j < n && pc[i] > pc[j]) par ^= 1;
    if (live && rr == 0) {
      if (n == 0) {
        ld2[p] = 0;
        sg2[p] = 1;
      } else if (singular) {
        ld2[p] = 0;
        sg2[p] = 0;
      } else {
        const double sgn = par ? -1.0 : 1.0;
        sg2[p] = mant < 0 ? -sgn : sgn;
        ld2[p] = log(fabs(mant)) + (double)expo * 0.6931471805599453;
      }
    }
    // row `row` of C (zero for a singular block) as double-FP32 words, and this row's part of
    // tr(C lap A) = sum_i C[row][i] lap A[i][row]
    const int row = singular ? rr : mycol;
    double lpart = 0.0;
    if (live && rr < n && row >= 0 && row < n) {
      float* ch = Cs + ((int64_t)(p * 2) * kGrpN + row) * kGrpCP;
      float* cl = ch + kGrpN * kGrpCP;
      const float* Dl = Phi + blk_off[p & 1] + (int64_t)(p >> 1) * T * n * n + (int64_t)(T - 1) * n * n;
      double* vv = (double*)Bs + (gid * 8 + rr) * kGrpBS;       // the row in the order of its columns
#pragma unroll
      for (int m = 0; m < kGrpN; ++m)
        if (m < n) vv[pc[m]] = av[m];
#pragma unroll
      for (int m = 0; m < kGrpN; ++m) {
        if (m < n) {
          const double c = singular ? 0.0 : vv[m];
          const float h = __double2float_rn(c);
          ch[m] = h;
          cl[m] = __double2float_rn(c - (double)h);
          lpart += c * widen<double, float>(Dl[m * n + row]);
        }
      }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) lpart += __shfl_xor_sync(0xffffffffu, lpart, off);
    if (live && rr == 0) lt[p] = lpart;
  }
  __syncthreads();

  // 2. tangent items: each group takes two coordinates (tr0, tr0 + 1) of a block per step,
  // four groups per warp
  const int NP2 = (NC + 1) / 2;                           // coordinate pairs per block
  for (int base = (tid >> 5) * 4; base < NM * NP2; base += 16) {
    const int it = base + ((tid >> 3) & 3);
    const bool live = it < NM * NP2;
    const int p = live ? it / NP2 : 0;
    const int tr0 = live ? 2 * (it - p * NP2) : 0;
    const bool two = tr0 + 1 < NC;
    const int n = live ? ns[p & 1] : 0;
    uint64_t bh[kGrpN], bl[kGrpN];                        // (zero bits: 0.f, 0.f)
#pragma unroll
    for (int j = 0; j < kGrpN; ++j) { bh[j] = 0; bl[j] = 0; }
    uint64_t* brow = Bs + (gid * 8 + rr) * kGrpBS;
    {
      // the orbital tangents are read once, from DRAM: start the pair of blocks this group
      // takes two steps later on its way into L2 (up to four 128-byte lines)
      const int it2 = it + 32;
      if (rr < 4 && it2 < NM * NP2) {
        const int p2 = it2 / NP2, n2 = ns[p2 & 1];
        const float* D2 = Phi + blk_off[p2 & 1] + (int64_t)(p2 >> 1) * T * n2 * n2 +
                          (int64_t)(1 + 2 * (it2 - p2 * NP2)) * n2 * n2;
        if (rr * 32 < 2 * n2 * n2) asm volatile("prefetch.L2 [%0];" ::"l"(D2 + rr * 32));
      }
    }
    if (rr < n) {
      // (a block's last odd coordinate is the second word of its pair and keeps no other)
      const float* D = Phi + blk_off[p & 1] + (int64_t)(p >> 1) * T * n * n + (int64_t)(1 + tr0 - (two ? 0 : 1)) * n * n;
      const float* chr = Cs + ((int64_t)(p * 2) * kGrpN + rr) * kGrpCP;
      const float* clr = chr + kGrpN * kGrpCP;
      switch (n) {
        case 1: ff_row2<1>(chr, clr, D, bh, bl); break;
        case 2: ff_row2<2>(chr, clr, D, bh, bl); break;
        case 3: ff_row2<3>(chr, clr, D, bh, bl); break;
        case 4: ff_row2<4>(chr, clr, D, bh, bl); break;
        case 5: ff_row2<5>(chr, clr, D, bh, bl); break;
        case 6: ff_row2<6>(chr, clr, D, bh, bl); break;
        case 7: ff_row2<7>(chr, clr, D, bh, bl); break;
        default: ff_row2<8>(chr, clr, D, bh, bl); break;
      }
    }
    // g: this row's diagonal entry; q: sum_j B[rr][j] B[j][rr]; the high words, then the low words,
    // pass through the group's staging rows
    uint64_t gh = 0, gl = 0, qh = 0, ql = 0, ch[kGrpN], cl[kGrpN];
    const uint64_t* bcol = Bs + (gid * 8) * kGrpBS + rr;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (rr < n) {
#pragma unroll
        for (int j = 0; j < kGrpN; ++j) brow[j] = half ? bl[j] : bh[j];
      }
      __syncwarp();
      if (rr < n) {
        (half ? gl : gh) = bcol[rr * kGrpBS];
#pragma unroll
        for (int j = 0; j < kGrpN; ++j)
          if (j < n) (half ? cl : ch)[j] = bcol[j * kGrpBS];
      }
      __syncwarp();
    }
    if (rr < n) {
      const uint64_t minus = tc::pack_f2(-1.f, -1.f);
#pragma unroll
      for (int j = 0; j < kGrpN; ++j)
        if (j < n) {                                      // ff_fma_acc of both words
          const uint64_t nb = tc::mul_f2(bh[j], minus), np = tc::mul_f2(nb, ch[j]);
          const uint64_t pe = tc::fma_f2(bh[j], cl[j], tc::fma_f2(bl[j], ch[j], tc::fma_f2(bh[j], ch[j], np)));
          uint64_t sum, e;
          ff2_two_diff(qh, np, sum, e);
          qh = sum;
          ql = tc::add_f2(ql, tc::add_f2(pe, e));
        }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      ff2_add_xor(gh, gl, off);
      ff2_add_xor(qh, ql, off);
    }
    if (live && rr == 0) {
      float h0, h1, l0, l1;
      tc::unpack_f2(gh, h0, h1);
      tc::unpack_f2(gl, l0, l1);
      if (two) gt[p * NC + tr0] = make_float2(h0, l0);
      gt[p * NC + tr0 + (two ? 1 : 0)] = make_float2(h1, l1);
      tc::unpack_f2(qh, h0, h1);
      tc::unpack_f2(ql, l0, l1);
      if (two) qt[p * NC + tr0] = make_float2(h0, l0);
      qt[p * NC + tr0 + (two ? 1 : 0)] = make_float2(h1, l1);
    }
  }
  __syncthreads();
  // 3. the determinant terms and E_L (as in k_det_energy)
  for (int e = tid; e < K * NC; e += blockDim.x) {
    const int k = e / NC, t = e % NC;
    const float2 g0 = gt[(2 * k) * NC + t], g1 = gt[(2 * k + 1) * NC + t];
    gradk[e] = ((double)g0.x + (double)g0.y) + ((double)g1.x + (double)g1.y);
  }
  for (int k = tid; k < K; k += blockDim.x) {
    double qs = 0;
    for (int t = 0; t < NC; ++t) {
      const float2 q0 = qt[(2 * k) * NC + t], q1 = qt[(2 * k + 1) * NC + t];
      qs += ((double)q0.x + (double)q0.y) + ((double)q1.x + (double)q1.y);
    }
    lapk[k] = lt[2 * k] + lt[2 * k + 1] - qs;
  }
  __syncthreads();
  if (tid == 0) {
    double m = -INFINITY;
    for (int k = 0; k < K; ++k) {
      const double sk = sg2[2 * k] * sg2[2 * k + 1];
      if (sk != 0 && ld2[2 * k] + ld2[2 * k + 1] > m) m = ld2[2 * k] + ld2[2 * k + 1];
    }
    double S = 0;
    for (int k = 0; k < K; ++k) {
      const double sk = sg2[2 * k] * sg2[2 * k + 1];
      rho[k] = sk != 0 ? sk * f_exp(ld2[2 * k] + ld2[2 * k + 1] - m) : (double)0;
      S += rho[k];
    }
    for (int k = 0; k < K; ++k) rho[k] = S != 0 ? rho[k] / S : (double)0;
    red[0] = m + f_log(f_abs(S));
    red[1] = S > 0 ? 1 : (S < 0 ? -1 : 0);
  }
  __syncthreads();
  const double lpsi = (double)red[0];
  const int sgn = (int)red[1];
  __syncthreads();
  // E_kin = -1/2 (|grad log psi|^2 + lap log psi) = -1/2 sum_k rho_k (lap_k + |g_k|^2)
  double kin = 0;
  for (int k = tid; k < K; k += blockDim.x) {
    double g2 = 0;
    for (int t = 0; t < NC; ++t) g2 += gradk[k * NC + t] * gradk[k * NC + t];
    kin += rho[k] * (lapk[k] + g2);
  }
  double pot = 0.0;
  const Wlk* rw = r + (int64_t)w * N * 3;
  for (int p = tid; p < N * N; p += blockDim.x) {
    const int i = p / N, j = p % N;
    if (j <= i) continue;
    const double dx = (double)rw[3 * i] - (double)rw[3 * j], dy = (double)rw[3 * i + 1] - (double)rw[3 * j + 1],
                 dz = (double)rw[3 * i + 2] - (double)rw[3 * j + 2];
    pot += 1.0 / sqrt(dx * dx + dy * dy + dz * dz);
  }
  for (int p = tid; p < N * sh.M; p += blockDim.x) {
    const int i = p / sh.M, m = p % sh.M;
    const double dx = (double)rw[3 * i] - nuc[3 * m], dy = (double)rw[3 * i + 1] - nuc[3 * m + 1],
                 dz = (double)rw[3 * i + 2] - nuc[3 * m + 2];
    pot -= a.charges[m] / sqrt(dx * dx + dy * dy + dz * dz);
  }
  red[tid] = (double)(-0.5) * kin + (double)pot;
  __syncthreads();
  for (int off = 64; off > 0; off >>= 1) {
    if (tid < off) red[tid] += red[tid + off];
    __syncthreads();
  }
  if (tid == 0) {
    const double e = (double)red[0] + a.v_nn;
    a.e_local[w] = e;
    if (a.log_psi) a.log_psi[w] = lpsi;
    if (a.sign) a.sign[w] = (int8_t)sgn;
    if (sgn == 0) atomicOr(a.status, kStatusSingular);
    else if (!isfinite(e) || !isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
  }
}


// Value pass (log|psi|, plus the backward seed rho_k A^{-T} when requested): one CTA per
// walker, one thread per (determinant, spin) block.
template <typename Det, typename PhiT>
__global__ void k_det_value(Shape sh, DetArgs a) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int w = blockIdx.x, tid = threadIdx.x;
  const int K = a.K, NM = 2 * K, ST = blockDim.x;
  const int ns[2] = {sh.n_up, sh.n_dn};
  const int nmax = max(ns[0], ns[1]);
  const bool want_inv = a.inv_out != nullptr;
  Det* A = (Det*)smem_raw;                                // [nmax^2][ST]
  Det* C = A + (int64_t)nmax * nmax * ST;                 // [nmax^2][ST] (inverse)
  Det* rcp = C + (want_inv ? (int64_t)nmax * nmax * ST : 0);   // [nmax][ST]
  Det* ld2 = rcp + (int64_t)nmax * ST;                   // [NM]
  Det* sg2 = ld2 + NM;
  Det* rho = sg2 + NM;                                   // [K]
  int* perm = (int*)(rho + K);                           // [nmax][ST]
  const PhiT* Phi = (const PhiT*)a.Phi + (int64_t)w * a.PW;
  const int64_t blk_off[2] = {0, (int64_t)K * ns[0] * ns[0]};
  const int64_t per = (int64_t)K * (ns[0] * ns[0] + ns[1] * ns[1]);
  Det* io = want_inv ? (Det*)a.inv_out + (int64_t)w * per : nullptr;
  // coalesced staging: block (k, spin) -> thread 2k + spin
  for (int e = tid; e < per; e += blockDim.x) {
    const int sp = e < blk_off[1] ? 0 : 1;
    const int n = ns[sp];
    const int64_t q = e - blk_off[sp];
    const int k = (int)(q / (n * n)), idx = (int)(q % (n * n));
    A[(int64_t)idx * ST + 2 * k + sp] = widen<Det, PhiT>(Phi[e]);
  }
  __syncthreads();
  if (tid < NM) {
    const int k = tid >> 1, sp = tid & 1, n = ns[sp];
    if (n == 0) {
      ld2[tid] = 0;
      sg2[tid] = 1;
    } else {
      thread_lu<Det>(A + tid, n, ST, perm + tid, rcp + tid, ld2 + tid, sg2 + tid);
      if (want_inv) {
        if (sg2[tid] != 0) thread_inverse<Det>(A + tid, perm + tid, rcp + tid, n, ST, C + tid);
        else for (int e = 0; e < n * n; ++e) C[(int64_t)e * ST + tid] = 0;
      }
    }
    (void)k;
  }
  __syncthreads();
  if (tid == 0) {
    Det m = -INFINITY;
    for (int k = 0; k < K; ++k) {
      const Det sk = sg2[2 * k] * sg2[2 * k + 1];
      if (sk != 0 && ld2[2 * k] + ld2[2 * k + 1] > m) m = ld2[2 * k] + ld2[2 * k + 1];
    }
    Det S = 0;
    for (int k = 0; k < K; ++k) {
      const Det sk = sg2[2 * k] * sg2[2 * k + 1];
      rho[k] = sk != 0 ? sk * f_exp(ld2[2 * k] + ld2[2 * k + 1] - m) : (Det)0;
      S += rho[k];
    }
    for (int k = 0; k < K; ++k) rho[k] = S != 0 ? rho[k] / S : (Det)0;
    const double lpsi = (double)(m + f_log(f_abs(S)));
    const int sgn = S > 0 ? 1 : (S < 0 ? -1 : 0);
    if (a.log_psi) a.log_psi[w] = lpsi;
    if (a.sign) a.sign[w] = (int8_t)sgn;
    if (sgn == 0) atomicOr(a.status, kStatusSingular);
    else if (!isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
  }
  if (want_inv) {
    __syncthreads();
    for (int e = tid; e < per; e += blockDim.x) {
      const int sp = e < blk_off[1] ? 0 : 1;
      const int n = ns[sp];
      const int64_t q = e - blk_off[sp];
      const int k = (int)(q / (n * n)), idx = (int)(q % (n * n));
      const int i = idx / n, j = idx % n;
      io[e] = rho[k] * C[(int64_t)(j * n + i) * ST + 2 * k + sp];        // rho_k A^{-T}
    }
  }
}

// Value pass without the backward seed, blocks of at most 8 x 8: one thread per
// (determinant, spin) block, 128 / (2K) walkers per CTA, no shared-memory staging.  Each
// block's determinant is kept as mantissa x 2^exponent; a walker's K terms
// D_k = det A_k,up det A_k,down are summed after scaling by 2^(e_k - max e), so that
// log|psi| = log|S| + (max e) ln 2 takes one logarithm per walker and no exponential
// (the same signed log-sum-exp, without forming log|D_k|).
template <typename Det, typename PhiT>
__global__ void __launch_bounds__(128, 3) k_det_value_small(Shape sh, DetArgs a) {
  pdl_wait();
  pdl_launch();
  __shared__ Det mt2[128];
  __shared__ int ex2[128];
  const int K = a.K, NM = 2 * K;
  const int per_cta = 128 / NM;
  const int wl = threadIdx.x / NM, p = threadIdx.x % NM;
  const int w = blockIdx.x * per_cta + wl;
  const int ns[2] = {sh.n_up, sh.n_dn};
  if (wl < per_cta && w < sh.B) {
    const int k = p >> 1, sp = p & 1, n = ns[sp];
    if (n == 0) {
      mt2[threadIdx.x] = (Det)1;
      ex2[threadIdx.x] = 0;
    } else {
      const PhiT* A = (const PhiT*)a.Phi + (int64_t)w * a.PW + (sp ? (int64_t)K * ns[0] * ns[0] : 0) +
                      (int64_t)k * n * n;
      lu_regs_any<Det, PhiT>(A, n, mt2 + threadIdx.x, ex2 + threadIdx.x);
    }
  }
  __syncthreads();
  if (threadIdx.x < per_cta) {
    const int w2 = blockIdx.x * per_cta + threadIdx.x;
    if (w2 < sh.B) {
      const Det* mt = mt2 + threadIdx.x * NM;
      const int* ex = ex2 + threadIdx.x * NM;
      int emax = INT_MIN;
      for (int k = 0; k < K; ++k)
        if (mt[2 * k] * mt[2 * k + 1] != 0 && ex[2 * k] + ex[2 * k + 1] > emax) emax = ex[2 * k] + ex[2 * k + 1];
      Det S = 0;
      for (int k = 0; k < K; ++k) {
        const Det mk = mt[2 * k] * mt[2 * k + 1];
        if (mk != 0) S += ldexp(mk, ex[2 * k] + ex[2 * k + 1] - emax);
      }
      const int sgn = S > 0 ? 1 : (S < 0 ? -1 : 0);
      const double lpsi = sgn == 0 ? (double)f_log(f_abs(S)) : (double)(f_log(f_abs(S)) + (Det)emax * (Det)0.6931471805599453);
      if (a.log_psi) a.log_psi[w2] = lpsi;
      if (a.sign) a.sign[w2] = (int8_t)sgn;
      if (sgn == 0) atomicOr(a.status, kStatusSingular);
      else if (!isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
    }
  }
}

// Gradient's value pass, blocks of at most 8 x 8 in FP64 (in every mode): log|psi| as in
// k_det_value_small, and the backward seed rho_k A^{-T}.  One thread inverts one block in registers
// (Gauss-Jordan in place, partial pivoting by predicated row swaps; the column permutation of the
// inverse goes into the store addresses), 128 / (2K) walkers per CTA.  FP32 mode takes it because rho
// from FP32 logarithms of D_k is off by 6e-8 |log D_k| and the inverse by its own roundings (N2, 1024
// walkers, worst of 20 gradients: 1.4e-5 of the norm with the FP32 stage, 1.2e-5 with this).  The factors in shared memory with two
// substitutions per column took 488 us for the 131072 7 x 7 blocks of 4096 N2 walkers, bound by the
// latency of 8 warps per SM; in registers they take 269 us (n^3 multiply-adds are about 80 us of the
// FP64 pipe, the rest is the predicated swaps and scattered 8-byte stores).
template <int NN, int C>
struct GjStep {
  static __device__ __forceinline__ void run(double (&a)[NN][NN], int (&piv)[NN], double& mant, int& expo,
                                             bool& singular) {
    auto best = abs_key(a[C][C]);
    int pr = C;
#pragma unroll
    for (int r = C + 1; r < NN; ++r) {
      const auto v = abs_key(a[r][C]);
      if (v > best) { best = v; pr = r; }
    }
    if (best == 0) singular = true;
    piv[C] = pr;
#pragma unroll
    for (int r = C + 1; r < NN; ++r) {
      const bool sw = r == pr;
#pragma unroll
      for (int j = 0; j < NN; ++j) {
        const double t = a[C][j];
        a[C][j] = sw ? a[r][j] : t;
        a[r][j] = sw ? t : a[r][j];
      }
    }
    const double p = a[C][C], rp = 1.0 / p;
    int e, e2;
    mant *= frexp(pr != C ? -p : p, &e);
    mant = frexp(mant, &e2);
    expo += e + e2;
    a[C][C] = 1.0;
#pragma unroll
    for (int j = 0; j < NN; ++j) a[C][j] *= rp;
#pragma unroll
    for (int r = 0; r < NN; ++r) {
      if (r == C) continue;
      const double f = a[r][C];
      a[r][C] = 0.0;
#pragma unroll
      for (int j = 0; j < NN; ++j) a[r][j] -= f * a[C][j];
    }
    GjStep<NN, C + 1>::run(a, piv, mant, expo, singular);
  }
};
template <int NN>
struct GjStep<NN, NN> {
  static __device__ __forceinline__ void run(double (&)[NN][NN], int (&)[NN], double&, int&, bool&) {}
};

// out[i n + j] = (A^{-1})[j][i]; det A = mant 2^expo (mant = 0 and a zero inverse if singular)
template <int NN, typename PhiT, typename Out>
__device__ __forceinline__ void invert_regs(const PhiT* __restrict__ Ag, Out* __restrict__ out, double* mant_out,
                                            int* expo_out) {
  double a[NN][NN], mant = 1.0;
  int piv[NN], expo = 0;
  bool singular = false;
#pragma unroll
  for (int i = 0; i < NN; ++i)
#pragma unroll
    for (int j = 0; j < NN; ++j)   // (FP32 mode keeps subnormal entries, which the bitwise widening drops)
      a[i][j] = sizeof(Out) == 4 ? widen_all<double, PhiT>(Ag[i * NN + j]) : widen<double, PhiT>(Ag[i * NN + j]);
  GjStep<NN, 0>::run(a, piv, mant, expo, singular);
  // the row swaps of A are column swaps of its inverse, undone last to first: column c of `a` is
  // column col[c] of A^{-1}
  int col[NN];
#pragma unroll
  for (int c = 0; c < NN; ++c) col[c] = c;
#pragma unroll
  for (int c = 0; c < NN; ++c) {
#pragma unroll
    for (int r = c + 1; r < NN; ++r) {
      const bool sw = piv[c] == r;
      const int t = col[c];
      col[c] = sw ? col[r] : t;
      col[r] = sw ? t : col[r];
    }
  }
#pragma unroll
  for (int c = 0; c < NN; ++c)
#pragma unroll
    for (int j = 0; j < NN; ++j) out[col[c] * NN + j] = (Out)(singular ? 0.0 : a[j][c]);
  *mant_out = singular ? 0.0 : mant;
  *expo_out = singular ? 0 : expo;
}

template <typename PhiT, typename Out>
__global__ void __launch_bounds__(128, 2) k_det_seed_small(Shape sh, DetArgs a) {
  pdl_wait();
  pdl_launch();
  __shared__ double mt2[128], rho[64];
  __shared__ int ex2[128];
  const int K = a.K, NM = 2 * K, per_cta = 128 / NM;
  const int wl = threadIdx.x / NM, p = threadIdx.x % NM, w0 = blockIdx.x * per_cta, w = w0 + wl;
  const int ns[2] = {sh.n_up, sh.n_dn};
  const int64_t dn_off = (int64_t)K * ns[0] * ns[0], per = dn_off + (int64_t)K * ns[1] * ns[1];
  Out* io = (Out*)a.inv_out;
  if (wl < per_cta && w < sh.B) {
    const int k = p >> 1, sp = p & 1, n = ns[sp];
    const int64_t off = (sp ? dn_off : 0) + (int64_t)k * n * n;
    const PhiT* A = (const PhiT*)a.Phi + (int64_t)w * a.PW + off;
    Out* out = io + (int64_t)w * per + off;
    double* m = mt2 + threadIdx.x;
    int* e = ex2 + threadIdx.x;
    switch (n) {
      case 0: *m = 1.0; *e = 0; break;
      case 1: invert_regs<1, PhiT, Out>(A, out, m, e); break;
      case 2: invert_regs<2, PhiT, Out>(A, out, m, e); break;
      case 3: invert_regs<3, PhiT, Out>(A, out, m, e); break;
      case 4: invert_regs<4, PhiT, Out>(A, out, m, e); break;
      case 5: invert_regs<5, PhiT, Out>(A, out, m, e); break;
      case 6: invert_regs<6, PhiT, Out>(A, out, m, e); break;
      case 7: invert_regs<7, PhiT, Out>(A, out, m, e); break;
      default: invert_regs<8, PhiT, Out>(A, out, m, e); break;
    }
  }
  __syncthreads();
  if (threadIdx.x < per_cta && w0 + (int)threadIdx.x < sh.B) {
    const int w2 = w0 + threadIdx.x;
    const double* mt = mt2 + threadIdx.x * NM;
    const int* ex = ex2 + threadIdx.x * NM;
    int emax = INT_MIN;
    for (int k = 0; k < K; ++k)
      if (mt[2 * k] * mt[2 * k + 1] != 0 && ex[2 * k] + ex[2 * k + 1] > emax) emax = ex[2 * k] + ex[2 * k + 1];
    double S = 0;
    for (int k = 0; k < K; ++k) {
      const double mk = mt[2 * k] * mt[2 * k + 1];
      const double t = mk != 0 ? ldexp(mk, ex[2 * k] + ex[2 * k + 1] - emax) : 0.0;
      rho[threadIdx.x * K + k] = t;
      S += t;
    }
    for (int k = 0; k < K; ++k) rho[threadIdx.x * K + k] = S != 0 ? rho[threadIdx.x * K + k] / S : 0.0;
    const int sgn = S > 0 ? 1 : (S < 0 ? -1 : 0);
    const double lpsi = sgn == 0 ? log(fabs(S)) : log(fabs(S)) + (double)emax * 0.6931471805599453;
    if (a.log_psi) a.log_psi[w2] = lpsi;
    if (a.sign) a.sign[w2] = (int8_t)sgn;
    if (sgn == 0) atomicOr(a.status, kStatusSingular);
    else if (!isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
  }
  __syncthreads();
  // scale by rho_k, consecutive elements per lane (the inverses of this CTA are in L2)
  const int nw = min(per_cta, sh.B - w0);
  for (int v = 0; v < nw; ++v) {
    Out* o = io + (int64_t)(w0 + v) * per;
    for (int e = threadIdx.x; e < (int)per; e += blockDim.x) {
      const int k = e < dn_off ? e / (ns[0] * ns[0]) : (e - (int)dn_off) / (ns[1] * ns[1]);
      o[e] = (Out)(rho[v * K + k] * (double)o[e]);
    }
  }
}

// ---- local-energy pass for small blocks --------------------------------------------------
// Blocks of at most 4 x 4 and at most 8 electrons (hydrogen, lithium hydride and its ions,
// atoms up to oxygen): one thread per (walker, determinant, spin) block does the
// Gauss-Jordan inversion with partial pivoting (first maximal |pivot|), the determinant as
// mantissa x 2^exponent, every tangent trace g_t = tr(C d_t A), the sum over t of
// q_t = tr((C d_t A)^2) and tr(C lap A), all in registers; one thread per walker then combines
// the K terms and assembles E_L.  128 / (2K) walkers share a CTA, so a small walker does not
// occupy a CTA of idle threads.
template <int NMAX, typename Det, typename Wlk, typename PhiT>
__global__ void __launch_bounds__(128) k_det_energy_small(const Wlk* r, const double* __restrict__ nuc,
                                                          Shape sh, DetArgs a) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int K = a.K, NM = 2 * K, NC = 3 * sh.N, T = sh.T;
  const int per_cta = 128 / NM;
  const int wl = threadIdx.x / NM, p = threadIdx.x % NM;
  const int w = blockIdx.x * per_cta + wl;
  const int ns[2] = {sh.n_up, sh.n_dn};
  // per walker of the CTA: gt [NM][NC], lt [NM], qs [NM], mant [NM]; then expo [NM] ints
  const int stride = NM * (NC + 3);
  Det* sd = (Det*)smem_raw;
  int* sexp = (int*)(sd + (int64_t)per_cta * stride);
  if (wl < per_cta && w < sh.B) {
    Det* gt = sd + (int64_t)wl * stride + p * NC;
    Det* lt = sd + (int64_t)wl * stride + NM * NC + p;
    Det* qs = lt + NM;
    Det* mt = qs + NM;
    const int k = p >> 1, sp = p & 1, n = ns[sp];
    if (n == 0) {
      for (int t = 0; t < NC; ++t) gt[t] = 0;
      *lt = 0; *qs = 0; *mt = 1;
      sexp[wl * NM + p] = 0;
    } else {
      const PhiT* blk = (const PhiT*)a.Phi + (int64_t)w * a.PW + (sp ? (int64_t)K * T * ns[0] * ns[0] : 0) +
                        (int64_t)k * T * n * n;
      // [A | I] -> [I | A^-1]
      Det M[NMAX][2 * NMAX];
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NMAX; ++j) M[i][j] = 0;
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
#pragma unroll
        for (int j = 0; j < NMAX; ++j)
          if (i < n && j < n) M[i][j] = widen_all<Det, PhiT>(blk[i * n + j]);
#pragma unroll
      for (int i = 0; i < NMAX; ++i) M[i][NMAX + i] = (i < n) ? (Det)1 : (Det)0;
      Det sgn = 1, mant = 1;
      int expo = 0;
      bool singular = false;
#pragma unroll
      for (int c = 0; c < NMAX; ++c) {
        if (c < n) {
          int piv = c;
          auto best = abs_key(M[c][c]);
#pragma unroll
          for (int i = c + 1; i < NMAX; ++i)
            if (i < n && abs_key(M[i][c]) > best) { best = abs_key(M[i][c]); piv = i; }
          if (best == 0) singular = true;
#pragma unroll
          for (int i = c + 1; i < NMAX; ++i)
            if (i == piv) {
#pragma unroll
              for (int j = 0; j < 2 * NMAX; ++j) { const Det tmp = M[c][j]; M[c][j] = M[i][j]; M[i][j] = tmp; }
            }
          if (piv != c) sgn = -sgn;
          const Det pv = M[c][c];
          int e;
          mant *= frexp(pv, &e);
          expo += e;
          int e2;
          mant = frexp(mant, &e2);
          expo += e2;
          const Det rp = (Det)1 / pv;
#pragma unroll
          for (int j = 0; j < 2 * NMAX; ++j) M[c][j] *= rp;
#pragma unroll
          for (int i = 0; i < NMAX; ++i)
            if (i != c && i < n) {
              const Det f = M[i][c];
#pragma unroll
              for (int j = 0; j < 2 * NMAX; ++j) M[i][j] -= f * M[c][j];
            }
        }
      }
      *mt = singular ? (Det)0 : sgn * mant;
      sexp[wl * NM + p] = singular ? 0 : expo;
      // C = A^-1 in M[.][NMAX ..]; tangent items
      Det qsum = 0;
      for (int t = 0; t < NC; ++t) {
        const PhiT* D = blk + (int64_t)(1 + t) * n * n;
        Det Bm[NMAX][NMAX];
#pragma unroll
        for (int i = 0; i < NMAX; ++i)
#pragma unroll
          for (int j = 0; j < NMAX; ++j) {
            Det s = 0;
#pragma unroll
            for (int m = 0; m < NMAX; ++m)
              if (m < n && j < n) s += M[i][NMAX + m] * widen_all<Det, PhiT>(D[m * n + j]);
            Bm[i][j] = s;
          }
        Det g = 0, q = 0;
#pragma unroll
        for (int i = 0; i < NMAX; ++i) {
          if (i < n) {
            g += Bm[i][i];
            q += Bm[i][i] * Bm[i][i];
#pragma unroll
            for (int j = i + 1; j < NMAX; ++j)
              if (j < n) q += (Det)2 * Bm[i][j] * Bm[j][i];
          }
        }
        gt[t] = singular ? (Det)0 : g;
        qsum += q;
      }
      const PhiT* DL = blk + (int64_t)(T - 1) * n * n;
      Det l = 0;
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
#pragma unroll
        for (int j = 0; j < NMAX; ++j)
          if (i < n && j < n) l += M[j][NMAX + i] * widen_all<Det, PhiT>(DL[i * n + j]);
      *lt = singular ? (Det)0 : l;
      *qs = singular ? (Det)0 : qsum;
    }
  }
  __syncthreads();
  if (threadIdx.x < per_cta) {
    const int wc = threadIdx.x;
    const int w2 = blockIdx.x * per_cta + wc;
    if (w2 < sh.B) {
      const Det* gtw = sd + (int64_t)wc * stride;
      const Det* ltw = gtw + NM * NC;
      const Det* qsw = ltw + NM;
      const Det* mtw = qsw + NM;
      const int* ew = sexp + wc * NM;
      int emax = INT_MIN;
      for (int kk = 0; kk < K; ++kk)
        if (mtw[2 * kk] * mtw[2 * kk + 1] != 0 && ew[2 * kk] + ew[2 * kk + 1] > emax) emax = ew[2 * kk] + ew[2 * kk + 1];
      Det S = 0;
      for (int kk = 0; kk < K; ++kk) {
        const Det mk = mtw[2 * kk] * mtw[2 * kk + 1];
        if (mk != 0) S += ldexp(mk, ew[2 * kk] + ew[2 * kk + 1] - emax);
      }
      // E_kin = -1/2 sum_k rho_k (lap_k + |g_k|^2), rho_k = D_k / psi
      Det kin = 0;
      for (int kk = 0; kk < K; ++kk) {
        const Det mk = mtw[2 * kk] * mtw[2 * kk + 1];
        if (mk == 0 || S == 0) continue;
        const Det rho = ldexp(mk, ew[2 * kk] + ew[2 * kk + 1] - emax) / S;
        Det g2 = 0;
        for (int t = 0; t < NC; ++t) {
          const Det g = gtw[(2 * kk) * NC + t] + gtw[(2 * kk + 1) * NC + t];
          g2 += g * g;
        }
        kin += rho * (ltw[2 * kk] + ltw[2 * kk + 1] - qsw[2 * kk] - qsw[2 * kk + 1] + g2);
      }
      double pot = 0.0;
      const Wlk* rw = r + (int64_t)w2 * sh.N * 3;
      for (int i = 0; i < sh.N; ++i)
        for (int j = i + 1; j < sh.N; ++j) {
          const double dx = (double)rw[3 * i] - (double)rw[3 * j], dy = (double)rw[3 * i + 1] - (double)rw[3 * j + 1],
                       dz = (double)rw[3 * i + 2] - (double)rw[3 * j + 2];
          pot += 1.0 / sqrt(dx * dx + dy * dy + dz * dz);
        }
      for (int i = 0; i < sh.N; ++i)
        for (int m = 0; m < sh.M; ++m) {
          const double dx = (double)rw[3 * i] - nuc[3 * m], dy = (double)rw[3 * i + 1] - nuc[3 * m + 1],
                       dz = (double)rw[3 * i + 2] - nuc[3 * m + 2];
          pot -= a.charges[m] / sqrt(dx * dx + dy * dy + dz * dz);
        }
      const int sgn = S > 0 ? 1 : (S < 0 ? -1 : 0);
      const double lpsi = sgn == 0 ? (double)f_log(f_abs(S)) : (double)(f_log(f_abs(S)) + (Det)emax * (Det)0.6931471805599453);
      const double e = (double)((Det)(-0.5) * kin) + pot + a.v_nn;
      a.e_local[w2] = e;
      if (a.log_psi) a.log_psi[w2] = lpsi;
      if (a.sign) a.sign[w2] = (int8_t)sgn;
      if (sgn == 0) atomicOr(a.status, kStatusSingular);
      else if (!isfinite(e) || !isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
    }
  }
}

inline size_t smem_det_energy_small(int det_bytes, int N, int K) {
  const int NM = 2 * K, per_cta = 128 / NM;
  return (size_t)per_cta * ((size_t)det_bytes * NM * (3 * N + 3) + sizeof(int) * NM);
}

// The BF16-mixed local-energy pass uses the 8-lane-group kernel for blocks of up to 8
// electrons; FN_DET_KERNEL=thread selects the one-thread-per-block kernel instead (the same
// pivots; C = A^-1 by forward and back substitution instead of Gauss-Jordan; the results
// agree to rounding).
static bool det_grp_enabled() {
  const char* v = getenv("FN_DET_KERNEL");
  return !(v && strcmp(v, "thread") == 0);
}

template <class Mode>
void launch_det_energy(const fn_system* s, const void* walkers, const Shape& sh, double* e_local, double* log_psi,
                       int8_t* sign, bool keep_inverse, cudaStream_t st) {
  using Det = typename Mode::Det; using Wlk = typename Mode::Wlk; using PhiT = typename Mode::PhiT;
  DetArgs a{};
  a.Phi = s->ws.Phi;
  a.PW = phi_walker_stride(s, sh.T);
  a.K = s->cfg.n_dets;
  a.e_local = e_local;
  a.log_psi = log_psi;
  a.sign = sign;
  a.inv_out = keep_inverse ? s->ws.dPhi : nullptr;
  a.charges = s->d_charges;
  a.v_nn = s->v_nn;
  a.status = s->ws.status;
  const bool full = sh.T > 1 && e_local != nullptr;
  const bool ov = overlap_launches(sh, Mode::kMode == FN_FP64 ? 8 : 4);
  const int nmax = std::max(s->n_up, s->n_dn), K = s->cfg.n_dets;
  ProfScope ps(s->prof, full ? kProfDetFull : kProfDetValue, st);
  if (full && nmax <= 4 && s->N <= 8) {
    // FP64 in every mode.  A determinant that nearly vanishes beside a psi that does not leaves terms
    // 1/d^2 that cancel to 1/d between lap_k and |g_k|^2; in FP32 they decided the error of the FP32
    // energies of few-electron walkers (one such walker up to 0.99 of the 2-norm over 2500).  LiH-,
    // 4096 walkers: 72 -> 189 us of a 1.8 ms call, error against 64 bits 1.0e-6 -> 0.4e-6 in the 2-norm.
    const int per_cta = 128 / (2 * K);
    const size_t smem = smem_det_energy_small(sizeof(double), s->N, K);
    cudaFuncSetAttribute(k_det_energy_small<4, double, Wlk, PhiT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_k(ov, k_det_energy_small<4, double, Wlk, PhiT>, (unsigned)((sh.B + per_cta - 1) / per_cta), 128, smem, st,
             (const Wlk*)walkers, s->d_nuclei, sh, a);
  } else if (full && std::is_same<Det, double>::value && std::is_same<PhiT, float>::value && nmax <= kGrpN &&
             det_grp_enabled()) {
    const size_t smem = smem_det_energy_grp(s->N, K);
    cudaFuncSetAttribute(k_det_energy_grp<Wlk>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_k(ov, k_det_energy_grp<Wlk>, sh.B, 128, smem, st, (const Wlk*)walkers, s->d_nuclei, sh, a);
  } else if (full) {
    const size_t smem = smem_det_energy(sizeof(Det), nmax, s->N, K,
                                        std::is_same<Det, double>::value && std::is_same<PhiT, float>::value);
    cudaFuncSetAttribute(k_det_energy<Det, Wlk, PhiT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_k(ov, k_det_energy<Det, Wlk, PhiT>, sh.B, 128, smem, st, (const Wlk*)walkers, s->d_nuclei, sh, a);
  } else if (!keep_inverse && nmax <= 8) {
    const int per_cta = 128 / (2 * K);
    launch_k(ov, k_det_value_small<Det, PhiT>, (unsigned)((sh.B + per_cta - 1) / per_cta), 128, 0, st, sh, a);
  } else if (nmax <= 8) {
    const int per_cta = 128 / (2 * K);
    launch_k(ov, k_det_seed_small<PhiT, Det>, (unsigned)((sh.B + per_cta - 1) / per_cta), 128, 0, st, sh, a);
  } else {
    const int threads = (int)round_up(2 * K, 32);
    const size_t vsmem = smem_det_value(sizeof(Det), nmax, K, keep_inverse);
    cudaFuncSetAttribute(k_det_value<Det, PhiT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vsmem);
    launch_k(ov, k_det_value<Det, PhiT>, sh.B, threads, vsmem, st, sh, a);
  }
}

template <class Mode>
void launch_log_psi(const fn_system* s, const void* walkers, int B, double* log_psi, int8_t* sign, cudaStream_t st) {
  if (small_covers(s, B)) {
    launch_small_log_psi(s, walkers, B, log_psi, sign, st);
    return;
  }
  const Shape sh = make_shape(s, B, 1);
  launch_forward<Mode>(s, walkers, sh, false, st);
  launch_det_energy<Mode>(s, walkers, sh, nullptr, log_psi, sign, false, st);
}

template void launch_log_psi<ModeF64>(const fn_system*, const void*, int, double*, int8_t*, cudaStream_t);
template void launch_log_psi<ModeF32>(const fn_system*, const void*, int, double*, int8_t*, cudaStream_t);
template void launch_log_psi<ModeBF16>(const fn_system*, const void*, int, double*, int8_t*, cudaStream_t);
template void launch_det_energy<ModeF64>(const fn_system*, const void*, const Shape&, double*, double*, int8_t*,
                                         bool, cudaStream_t);
template void launch_det_energy<ModeF32>(const fn_system*, const void*, const Shape&, double*, double*, int8_t*,
                                         bool, cudaStream_t);
template void launch_det_energy<ModeBF16>(const fn_system*, const void*, const Shape&, double*, double*, int8_t*,
                                          bool, cudaStream_t);

}  // namespace fn
