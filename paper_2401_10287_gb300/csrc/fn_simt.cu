// FP32 and FP64 stream layers, orbitals and GEMMs on the register-tiled core of
// fn_simt.cuh.
#include "fn_simt.cuh"

#include <algorithm>

#include "fn_device.cuh"
#include "fn_internal.cuh"
#include "fn_simt_launch.cuh"

namespace fn {
namespace simt {

template <typename T> __device__ __forceinline__ void load_vec(const T* p, T (&v)[Vec<T>::n]) {
  *(typename Vec<T>::type*)v = *(const typename Vec<T>::type*)p;
}
template <typename T> __device__ __forceinline__ void store_vec(T* p, const T (&v)[Vec<T>::n]) {
  *(typename Vec<T>::type*)p = *(const typename Vec<T>::type*)v;
}
// V adjacent elements, of which the first `live` exist
template <typename T, bool VEC>
__device__ __forceinline__ void load_group(const T* p, int live, T (&v)[Vec<T>::n]) {
  if constexpr (VEC) load_vec(p, v);
  else
#pragma unroll
    for (int e = 0; e < Vec<T>::n; ++e) v[e] = e < live ? p[e] : (T)0;
}
template <typename T, bool VEC>
__device__ __forceinline__ void store_group(T* p, int live, const T (&v)[Vec<T>::n]) {
  if constexpr (VEC) store_vec(p, v);
  else
#pragma unroll
    for (int e = 0; e < Vec<T>::n; ++e)
      if (e < live) p[e] = v[e];
}

// ---------------------------------------------------------------------------------------
// stream layer: a CTA owns the rows of `wps` whole walkers and BN output columns and walks
// over the tangent slabs: value (h = tanh z), gradients ((1 - h^2) z_t, sum z_t^2),
// Laplacian ((1 - h^2) z - 2 h (1 - h^2) sum z_t^2).  h and the sums stay in registers, the
// ring keeps loading across slabs, the spin means of the output are summed in electron
// order from a staged copy.
// Bound by the FMA pipe: N2 network at 4096 walkers, 104 -> 35 ms per FP32 local-energy
// call for its four layers (1.26 TFLOP); that width now takes the tensor cores (fn_x3.cu).
// ---------------------------------------------------------------------------------------
template <typename T, int TM, int TN, int WM, bool FULL, bool VEC>
__global__ void __launch_bounds__(32 * WM) k_layer(Shape sh, LayerArgs a, int wps, int subs) {
  pdl_wait();
  pdl_launch();
  using Tl = Tile<T, TM, TN, WM>;
  constexpr int V = Tl::V, G = TN / V, LDY = Tl::BN + V;
  constexpr bool TWO = sizeof(T) == 4 && !FULL;                 // (with tangents the registers hold h and sum z^2)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ys = (T*)(smem_raw + Tl::kRingBytes);                      // [BM][LDY] staged outputs
  // column tiles run fastest, so that the CTAs that share input rows run together
  const int nct = (a.h1 + Tl::BN - 1) / Tl::BN, rb = blockIdx.x / nct, n0 = (blockIdx.x % nct) * Tl::BN;
  const int tile = rb / subs, sub = rb % subs;
  const int w0 = tile * sh.wpt + sub * wps;
  const int nw = min(min(wps, sh.wpt - sub * wps), sh.B - w0);
  if (nw <= 0) return;
  const int rows = nw * sh.N;
  const int64_t row0 = (int64_t)tile * kTileRows + (int64_t)sub * wps * sh.N;
  const T* X = (const T*)a.X + row0 * a.ldx;
  T* Y = (T*)a.Y + row0 * a.ldy;
  const T* Mt = (const T*)a.Mterm;
  const T* W = (const T*)a.VsT;
  const int64_t xslab = sh.R * a.ldx, yslab = sh.R * a.ldy, mslab = (int64_t)sh.B * a.h1;
  const int nk = (a.k_self + Tl::BK - 1) / Tl::BK;
  const int r0 = lane_row0<Tl>();
  int lk = 0;
  const T* Xl = X;
  auto load = [&](int, unsigned char* stage) {
    const T* Xt = Xl;
    load_stage<Tl, T, VEC, false, false>(
        stage, [&](int row) { return row < rows ? Xt + (int64_t)row * a.ldx : (const T*)nullptr; }, a.ldx,
        lk * Tl::BK, a.k_self, rows, W, a.h1, n0, a.h1);
    if (++lk == nk) { lk = 0; Xl += xslab; }
  };
  T hv[FULL ? TM : 1][FULL ? TN : 1], sq[FULL ? TM : 1][FULL ? TN : 1];
  auto done = [&](const Acc<T, TM, TN, TWO>& acc, int t) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int rl = r0 + 4 * i;
      if (rl < rows) {
        const int w = w0 + rl / sh.N;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const int cl = lane_col<Tl>(g * V), col = n0 + cl, live = a.h1 - col;
          if (live <= 0) continue;
          T m[V], res[V], out[V];
          load_group<T, VEC>(Mt + t * mslab + (int64_t)w * a.h1 + col, live, m);
          if (a.residual) load_group<T, VEC>(X + t * xslab + (int64_t)rl * a.ldx + col, live, res);
#pragma unroll
          for (int e = 0; e < V; ++e) {
            const int j = g * V + e;
            const T z = acc.get(i, j) + m[e];
            if (!FULL || t == 0) {
              const T h = f_tanh(z);
              if constexpr (FULL) { hv[i][j] = h; sq[i][j] = 0; }
              out[e] = h;
            } else if constexpr (FULL) {
              const T h = hv[i][j], d = (T)1 - h * h;
              if (t < sh.T - 1) {
                out[e] = d * z;
                sq[i][j] += z * z;
              } else {
                out[e] = d * z - (T)2 * h * d * sq[i][j];
              }
            }
          }
          if (!FULL && a.act_out) store_group<T, VEC>((T*)a.act_out + (row0 + rl) * a.h1 + col, live, out);
          if (a.residual)
#pragma unroll
            for (int e = 0; e < V; ++e) out[e] += res[e];
          store_group<T, VEC>(Y + t * yslab + (int64_t)rl * a.ldy + col, live, out);
          if (a.Hbar_out) store_vec(ys + rl * LDY + cl, out);
        }
      }
    }
    if (a.Hbar_out) {
      __syncthreads();
      T* Hb = (T*)a.Hbar_out + ((int64_t)t * sh.B + w0) * 2 * a.h1;
      for (int e = threadIdx.x; e < nw * 2 * Tl::BN; e += Tl::kThreads) {
        const int cl = e % Tl::BN, ws = e / Tl::BN, wl = ws >> 1, s = ws & 1, col = n0 + cl;
        if (col >= a.h1) continue;
        const int lo = s ? sh.n_up : 0, hi = s ? sh.N : sh.n_up;
        T sum = 0;
        for (int i = lo; i < hi; ++i) sum += ys[(wl * sh.N + i) * LDY + cl];
        Hb[(int64_t)ws * a.h1 + col] = hi > lo ? sum / (T)(hi - lo) : (T)0;
      }
      // the barrier of the next slab's first stage orders these reads before the next staging
    }
  };
  stream<Tl, T, TM, TN, TWO>(smem_raw, nk, sh.T, load, done);
}

template <typename T, int TM, int TN, int WM>
static void layer_cfg(const Shape& sh, const LayerArgs& a, bool vec, cudaStream_t st) {
  using Tl = Tile<T, TM, TN, WM>;
  const int wps = std::min(sh.wpt, Tl::BM / sh.N), subs = (sh.wpt + wps - 1) / wps;
  const size_t smem = Tl::kRingBytes + sizeof(T) * Tl::BM * (Tl::BN + Tl::V);
  const unsigned grid = (unsigned)((a.h1 + Tl::BN - 1) / Tl::BN) * sh.tiles * subs;
  auto go = [&](auto kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_k(false, kernel, grid, Tl::kThreads, smem, st, sh, a, wps, subs);
  };
  if (sh.T > 1) vec ? go(k_layer<T, TM, TN, WM, true, true>) : go(k_layer<T, TM, TN, WM, true, false>);
  else vec ? go(k_layer<T, TM, TN, WM, false, true>) : go(k_layer<T, TM, TN, WM, false, false>);
}

// Cost of a tile shape: CTAs on the busiest SM (at least the number that fills its FMA
// pipe) x tile area / the shape's relative FMA rate.  FP32: the small tile has a quarter of the sums per
// loaded operand, taken as half the rate.  Time with one tile only over the rule's, FP32 log|psi|: large
// 1.48 to 2.2 up to 8192 rows, 1.00 to 1.26 at 65536; small 1.00 to 1.02 up to 4096 rows, 1.09 for N2 (4 x 256) at
// 32760 rows and more, 0.93 to 0.95 for LiH (4 x 128) and 0.88 for C (3 x 64) at 65536, 0.89 for N2 at 16380.
// FP64, where either tile saturates the pipe: large 1.2 to 1.8 up to 8192 rows (idle SMs), small 1.00 to 1.14; one warp
// more or less per SM decides, which the equal rates count.
template <typename Tl>
static double tile_cost(int64_t ctas, int sm_count, int fill, double rate) {
  const int64_t per_sm = std::max<int64_t>((ctas + sm_count - 1) / sm_count, fill);
  return (double)per_sm * Tl::BM * Tl::BN / rate;
}

template <typename T>
void launch_layer(const Shape& sh, const LayerArgs& a, int sm_count, cudaStream_t st) {
  constexpr int V = Vec<T>::n;
  const bool vec = a.ldx % V == 0 && a.ldy % V == 0 && a.h1 % V == 0;
  auto ctas = [&](int BM, int BN) {
    const int wps = std::min(sh.wpt, BM / sh.N);
    return (int64_t)sh.tiles * ((sh.wpt + wps - 1) / wps) * ((a.h1 + BN - 1) / BN);
  };
  if constexpr (sizeof(T) == 4) {
    using Big = Tile<T, 8, 8, 4>; using Small = Tile<T, 4, 4, 2>;
    if (tile_cost<Big>(ctas(Big::BM, Big::BN), sm_count, 2, 1.0) <=
        tile_cost<Small>(ctas(Small::BM, Small::BN), sm_count, 4, 0.5))
      layer_cfg<T, 8, 8, 4>(sh, a, vec, st);
    else
      layer_cfg<T, 4, 4, 2>(sh, a, vec, st);
  } else {
    using Big = Tile<T, 4, 4, 8>; using Small = Tile<T, 4, 4, 2>;
    if (tile_cost<Big>(ctas(Big::BM, Big::BN), sm_count, 1, 1.0) <=
        tile_cost<Small>(ctas(Small::BM, Small::BN), sm_count, 1, 1.0))
      layer_cfg<T, 4, 4, 8>(sh, a, vec, st);
    else
      layer_cfg<T, 4, 4, 2>(sh, a, vec, st);
  }
}

// ---------------------------------------------------------------------------------------
// orbitals: phi^k_i(r_j) = (w_ki . h_j + g_ki) env_ki(r_j) of one spin, one slab per grid z.
// A CTA takes the rows (electrons of the spin) of whole walkers and BN orbitals; the matrix
// elements are staged in shared memory and written in the order of Phi, whose n_s x n_s
// blocks are contiguous.  The value pass evaluates the envelope for its elements; the
// full pass reads the values of k_envelope (once per electron and orbital instead of once
// per slab), and the own-coordinate and Laplacian envelope terms are added afterwards from
// the projections kept in orbP (k_orbital_fixup).
// ---------------------------------------------------------------------------------------
// sum_m pi_m exp(-|sigma_m d_m|); d[q * ld] = coordinate q mod 3 of the distance to nucleus q / 3
template <typename T>
__device__ __forceinline__ T env_value(const T* pi, const T* sig, int aniso, int M, const T* d, int ld) {
  T env = 0;
  for (int m = 0; m < M; ++m) {
    const T d0 = d[3 * m * ld], d1 = d[(3 * m + 1) * ld], d2 = d[(3 * m + 2) * ld];
    T s;
    if (!aniso) {
      s = sig[m] * f_sqrt(d0 * d0 + d1 * d1 + d2 * d2);
    } else {
      const T* S = sig + m * 9;
      const T u0 = S[0] * d0 + S[1] * d1 + S[2] * d2, u1 = S[3] * d0 + S[4] * d1 + S[5] * d2,
              u2 = S[6] * d0 + S[7] * d1 + S[8] * d2;
      s = f_sqrt(u0 * u0 + u1 * u1 + u2 * u2);
    }
    env += pi[m] * f_exp(-s);
  }
  return env;
}

// Envelope values of every electron's own-spin orbitals, orbital-major [K N][R]: the rows of an
// orbital are adjacent, so that a kernel with one electron row per lane reads whole lines.  A CTA
// takes one 128-row tile (thread = row) and 16 orbitals, whose parameters every thread of a spin
// reads at the same time.
constexpr int kEnvOrbs = 16;
template <typename T>
__global__ void __launch_bounds__(kTileRows) k_envelope(Shape sh, OrbArgs a) {
  pdl_wait();
  pdl_launch();
  __shared__ T ds[3 * kMaxNuclei][kTileRows];
  const int tile = blockIdx.x, rl = threadIdx.x, wl = rl / sh.N, j = rl - wl * sh.N, w = tile * sh.wpt + wl;
  if (wl >= sh.wpt || w >= sh.B) return;                        // no barrier below: each thread reads its own column
  const T* rj = (const T*)a.walkers + ((int64_t)w * sh.N + j) * 3;
  for (int q = 0; q < 3 * sh.M; ++q) ds[q][rl] = (T)((double)rj[q % 3] - a.nuclei[q]);
  const int spin = j < sh.n_up ? 0 : 1, n_ko = a.K * (spin ? sh.n_dn : sh.n_up), nc = a.aniso ? 9 : 1;
  T* out = (T*)a.envv + (int64_t)(spin ? a.K * sh.n_up : 0) * sh.R + (int64_t)tile * kTileRows + rl;
  for (int ko = blockIdx.y * kEnvOrbs; ko < min(n_ko, (int)(blockIdx.y + 1) * kEnvOrbs); ++ko)
    out[(int64_t)ko * sh.R] = env_value<T>((const T*)a.pi[spin] + (int64_t)ko * sh.M,
                                           (const T*)a.sig[spin] + (int64_t)ko * sh.M * nc, a.aniso, sh.M, &ds[0][rl],
                                           kTileRows);
}

template <typename T, int TM, int TN, int WM, bool FULL, bool VEC>
__global__ void __launch_bounds__(32 * WM) k_orbitals(Shape sh, OrbArgs a, int spin) {
  pdl_wait();
  pdl_launch();
  using Tl = Tile<T, TM, TN, WM>;
  constexpr int V = Tl::V, G = TN / V, LDY = Tl::BN + V;
  constexpr bool TWO = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ys = (T*)(smem_raw + Tl::kRingBytes);                      // [BM][LDY]
  T* ds = ys + Tl::BM * LDY;                                    // value pass: [BM][3 M] electron - nucleus
  const int n_s = spin ? sh.n_dn : sh.n_up, e0 = spin ? sh.n_up : 0, n_ko = a.K * n_s, t = blockIdx.z;
  const int nct = (n_ko + Tl::BN - 1) / Tl::BN, n0 = (blockIdx.x % nct) * Tl::BN;
  const int wpc = Tl::BM / n_s, w0 = blockIdx.x / nct * wpc, nw = min(wpc, sh.B - w0), rows = nw * n_s;
  const T* H = (const T*)a.HL + (int64_t)t * sh.R * a.h1;
  if (!FULL) {
    for (int e = threadIdx.x; e < rows * 3 * sh.M; e += Tl::kThreads) {
      const int rl = e / (3 * sh.M), q = e % (3 * sh.M);
      const T* rj = (const T*)a.walkers + ((int64_t)(w0 + rl / n_s) * sh.N + e0 + rl % n_s) * 3;
      ds[rl * 3 * sh.M + q] = (T)((double)rj[q % 3] - a.nuclei[q]);
    }
  }
  auto row_of = [&](int rl) { return tile_row(w0 + rl / n_s, e0 + rl % n_s, sh.N, sh.wpt); };
  const int nk = (a.h1 + Tl::BK - 1) / Tl::BK;
  auto load = [&](int s, unsigned char* stage) {
    load_stage<Tl, T, VEC, false, false>(
        stage, [&](int rl) { return rl < rows ? H + row_of(rl) * a.h1 : (const T*)nullptr; }, a.h1, s * Tl::BK, a.h1,
        rows, (const T*)a.wT[spin], n_ko, n0, n_ko);
  };
  const int r0 = lane_row0<Tl>(), poff = spin ? a.K * sh.n_up : 0, ldp = a.K * sh.N;
  auto done = [&](const Acc<T, TM, TN, TWO>& acc, int) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int rl = r0 + 4 * i;
      if (rl >= rows) continue;
      const int64_t row = row_of(rl);
      // slot of orbP this (row, slab) fills: the value projection, or one along an own coordinate
      const int own = t - 1 - 3 * (e0 + rl % n_s), slot = t == 0 ? 0 : (own >= 0 && own < 3 ? 1 + own : -1);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int cl = lane_col<Tl>(g * V), ko = n0 + cl;
#pragma unroll
        for (int e = 0; e < V; ++e) {
          if (ko + e >= n_ko) continue;
          T p = acc.get(i, g * V + e);
          if (t == 0) p += ((const T*)a.g[spin])[ko + e];
          T env;
          if constexpr (FULL) {
            env = ((const T*)a.envv)[(int64_t)(poff + ko + e) * sh.R + row];
            if (slot >= 0 && t < sh.T - 1) ((T*)a.orbP)[(row * 4 + slot) * ldp + poff + ko + e] = p;
          } else {
            const int nc = a.aniso ? 9 : 1;
            env = env_value<T>((const T*)a.pi[spin] + (int64_t)(ko + e) * sh.M,
                               (const T*)a.sig[spin] + (int64_t)(ko + e) * sh.M * nc, a.aniso, sh.M,
                               ds + rl * 3 * sh.M, 1);
          }
          ys[rl * LDY + cl + e] = p * env;
        }
      }
    }
    __syncthreads();
    T* Phi = (T*)a.Phi + (int64_t)w0 * a.PW + (spin ? (int64_t)a.K * sh.T * sh.n_up * sh.n_up : 0);
    const int ncol = min(Tl::BN, n_ko - n0), nn = n_s * n_s;
    for (int e = threadIdx.x; e < rows * ncol; e += Tl::kThreads) {
      const int jj = e % n_s, q = e / n_s, c = q % ncol, wl = q / ncol, ko = n0 + c, k = ko / n_s, i = ko - k * n_s;
      Phi[wl * a.PW + ((int64_t)k * sh.T + t) * nn + i * n_s + jj] = ys[(wl * n_s + jj) * LDY + c];
    }
  };
  stream<Tl, T, TM, TN, TWO>(smem_raw, nk, 1, load, done);
}

template <typename T, int TM, int TN, int WM>
static void orbitals_cfg(const Shape& sh, const OrbArgs& a, int spin, cudaStream_t st) {
  using Tl = Tile<T, TM, TN, WM>;
  constexpr int V = Tl::V;
  const int n_s = spin ? sh.n_dn : sh.n_up, n_ko = a.K * n_s, wpc = Tl::BM / n_s;
  const bool full = sh.T > 1, vec = a.h1 % V == 0 && n_ko % V == 0;
  const size_t smem = Tl::kRingBytes + sizeof(T) * Tl::BM * (Tl::BN + V + (full ? 0 : 3 * sh.M));
  const dim3 grid((unsigned)((n_ko + Tl::BN - 1) / Tl::BN) * ((sh.B + wpc - 1) / wpc), 1, sh.T);
  auto go = [&](auto kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_k(false, kernel, grid, Tl::kThreads, smem, st, sh, a, spin);
  };
  if (full) vec ? go(k_orbitals<T, TM, TN, WM, true, true>) : go(k_orbitals<T, TM, TN, WM, true, false>);
  else vec ? go(k_orbitals<T, TM, TN, WM, false, true>) : go(k_orbitals<T, TM, TN, WM, false, false>);
}

template <typename T>
void launch_envelope(const Shape& sh, const OrbArgs& a, cudaStream_t st) {
  const int n_ko = a.K * std::max(sh.n_up, sh.n_dn);
  launch_k(false, k_envelope<T>, dim3(sh.tiles, (n_ko + kEnvOrbs - 1) / kEnvOrbs), kTileRows, 0, st, sh, a);
}

template <typename T>
void launch_orbitals(const Shape& sh, const OrbArgs& a, int sm_count, cudaStream_t st) {
  if (sh.T > 1) launch_envelope<T>(sh, a, st);
  for (int spin = 0; spin < 2; ++spin) {
    const int n_s = spin ? sh.n_dn : sh.n_up;
    if (!n_s) continue;
    auto ctas = [&](int BM, int BN) {
      return (int64_t)((sh.B + BM / n_s - 1) / (BM / n_s)) * ((a.K * n_s + BN - 1) / BN) * sh.T;
    };
    using Small = Tile<T, 4, 4, 2>;
    if constexpr (sizeof(T) == 4) {
      using Big = Tile<T, 8, 8, 4>;
      if (tile_cost<Big>(ctas(Big::BM, Big::BN), sm_count, 2, 1.0) <=
          tile_cost<Small>(ctas(Small::BM, Small::BN), sm_count, 4, 0.5))
        orbitals_cfg<T, 8, 8, 4>(sh, a, spin, st);
      else
        orbitals_cfg<T, 4, 4, 2>(sh, a, spin, st);
    } else {
      using Big = Tile<T, 4, 4, 8>;
      if (tile_cost<Big>(ctas(Big::BM, Big::BN), sm_count, 1, 1.0) <=
          tile_cost<Small>(ctas(Small::BM, Small::BN), sm_count, 1, 1.0))
        orbitals_cfg<T, 4, 4, 8>(sh, a, spin, st);
      else
        orbitals_cfg<T, 4, 4, 2>(sh, a, spin, st);
    }
  }
}

// ---------------------------------------------------------------------------------------
// plain GEMM: C(m,n) (+)= sum_k A(m,k) B(k,n) + bias[n] (rows m < bias_rows), K split over
// gridDim.z (atomic accumulation).  AT: A(m,k) = A[k lda + m]; BT: B(k,n) = B[n ldb + k].
// ---------------------------------------------------------------------------------------
template <typename T, int TM, int TN, int WM, bool AT, bool BT, bool VEC>
__global__ void __launch_bounds__(32 * WM) k_gemm(GemmArgs<T> g) {
  pdl_wait();
  pdl_launch();
  using Tl = Tile<T, TM, TN, WM>;
  constexpr int V = Tl::V, G = TN / V;
  constexpr bool TWO = sizeof(T) == 4 && !AT && !BT;             // the value pass's products
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nct = (g.N + Tl::BN - 1) / Tl::BN, n0 = (blockIdx.x % nct) * Tl::BN;
  const int64_t m0 = (int64_t)(blockIdx.x / nct) * Tl::BM;
  const int rows = (int)min((int64_t)Tl::BM, g.M - m0);
  const int nk_all = (g.K + Tl::BK - 1) / Tl::BK, chunk = (nk_all + gridDim.z - 1) / gridDim.z;
  const int kb0 = blockIdx.z * chunk, nk = min(chunk, nk_all - kb0);
  if (nk <= 0) return;
  const T* A = g.A + (AT ? m0 : m0 * g.lda);
  auto load = [&](int s, unsigned char* stage) {
    load_stage<Tl, T, VEC, AT, BT>(
        stage, [&](int row) { return row < rows ? A + (AT ? (int64_t)row : (int64_t)row * g.lda) : (const T*)nullptr; },
        g.lda, (kb0 + s) * Tl::BK, g.K, rows, g.B, g.ldb, n0, g.N);
  };
  const int r0 = lane_row0<Tl>();
  auto done = [&](const Acc<T, TM, TN, TWO>& acc, int) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int rl = r0 + 4 * i;
      if (rl >= rows) continue;
      const int64_t m = m0 + rl;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const int col = n0 + lane_col<Tl>(q * V), live = g.N - col;
        if (live <= 0) continue;
        T out[V];
#pragma unroll
        for (int e = 0; e < V; ++e) out[e] = acc.get(i, q * V + e);
        if (g.bias && m < g.bias_rows && blockIdx.z == 0)
#pragma unroll
          for (int e = 0; e < V; ++e)
            if (e < live) out[e] += g.bias[col + e];
        T* c = g.C + m * g.ldc + col;
        if (g.atomic) {
#pragma unroll
          for (int e = 0; e < V; ++e)
            if (e < live) atomicAdd(c + e, out[e]);
        } else if (VEC && live >= V) {
          store_vec(c, out);
        } else {
#pragma unroll
          for (int e = 0; e < V; ++e)
            if (e < live) c[e] = out[e];
        }
      }
    }
  };
  stream<Tl, T, TM, TN, TWO>(smem_raw, nk, 1, load, done);
}

template <typename T, int TM, int TN, int WM>
static void gemm_cfg(const GemmArgs<T>& g, bool at, bool bt, int split, bool vec, cudaStream_t st) {
  using Tl = Tile<T, TM, TN, WM>;
  const dim3 grid((unsigned)((g.N + Tl::BN - 1) / Tl::BN * ((g.M + Tl::BM - 1) / Tl::BM)), 1, split);
  auto go = [&](auto kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Tl::kRingBytes);
    launch_k(false, kernel, grid, Tl::kThreads, Tl::kRingBytes, st, g);
  };
  if (at) vec ? go(k_gemm<T, TM, TN, WM, true, false, true>) : go(k_gemm<T, TM, TN, WM, true, false, false>);
  else if (bt) vec ? go(k_gemm<T, TM, TN, WM, false, true, true>) : go(k_gemm<T, TM, TN, WM, false, true, false>);
  else vec ? go(k_gemm<T, TM, TN, WM, false, false, true>) : go(k_gemm<T, TM, TN, WM, false, false, false>);
}

template <typename T>
void launch_gemm(GemmArgs<T> g, bool at, bool bt, int max_split, int sm_count, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0) return;
  constexpr int V = Vec<T>::n;
  const bool vec = g.lda % V == 0 && g.ldb % V == 0 && g.ldc % V == 0 &&
                   (((uintptr_t)g.A | (uintptr_t)g.B | (uintptr_t)g.C) & 15) == 0;
  auto pick = [&](auto tile, int fill, double rate, int* split) {
    using Tl = decltype(tile);
    const int64_t tiles = ((g.M + Tl::BM - 1) / Tl::BM) * ((g.N + Tl::BN - 1) / Tl::BN);
    const int64_t nk = (g.K + Tl::BK - 1) / Tl::BK;
    // split K until every SM has `fill` CTAs, each at least 4 stages deep
    const int64_t want = std::max<int64_t>(1, ((int64_t)fill * sm_count + tiles - 1) / tiles);
    *split = (int)std::max<int64_t>(1, std::min<int64_t>({want, (int64_t)max_split, nk / 4}));
    return tile_cost<Tl>(tiles * *split, sm_count, fill, rate) / *split;
  };
  // FP64: each SM quarter has a pipe of its own that one warp saturates, so a product takes as long as
  // the busiest SM's warps per quarter; K is split as that comes out shortest, with as few parts as give
  // it to 2 %.  (Just enough CTAs for the SMs left quarters idle and some SMs with two: the weight
  // gradients of a 320 x 256 layer ran 160 CTAs of two warps.  Products of the N2 gradient, 1618 walkers:
  // 39.6 -> 28.6 ms; mean field with one part, 1618 and 3000 rows: 1.26 and 2.15 ms as before.)
  auto pick64 = [&](auto tile, int* split) {
    using Tl = decltype(tile);
    const int64_t tiles = ((g.M + Tl::BM - 1) / Tl::BM) * ((g.N + Tl::BN - 1) / Tl::BN);
    const int64_t nk = (g.K + Tl::BK - 1) / Tl::BK;
    const int64_t most = std::max<int64_t>(1, std::min<int64_t>({(int64_t)max_split, nk / 4, 256}));
    constexpr int warps = Tl::kThreads / 32;
    double best = 0.0;
    for (int64_t s = 1; s <= most; ++s) {
      const int64_t per_sm = (tiles * s + sm_count - 1) / sm_count;
      const double per_quarter = std::max(1.0, per_sm * warps / 4.0);
      const double cost = per_quarter * (Tl::BM * Tl::BN / warps) * (double)((nk + s - 1) / s);
      if (s == 1 || cost < 0.98 * best) {
        best = cost;
        *split = (int)s;
      }
    }
    return best;
  };
  int sb, ss;
  if constexpr (sizeof(T) == 4) {
    const double big = pick(Tile<T, 8, 8, 4>{}, 2, 1.0, &sb), small = pick(Tile<T, 4, 4, 2>{}, 4, 0.5, &ss);
    g.atomic = g.atomic || (big <= small ? sb : ss) > 1;
    if (big <= small) gemm_cfg<T, 8, 8, 4>(g, at, bt, sb, vec, st);
    else gemm_cfg<T, 4, 4, 2>(g, at, bt, ss, vec, st);
  } else {
    const double big = pick64(Tile<T, 4, 4, 8>{}, &sb), small = pick64(Tile<T, 4, 4, 2>{}, &ss);
    g.atomic = g.atomic || (big <= small ? sb : ss) > 1;
    if (big <= small) gemm_cfg<T, 4, 4, 8>(g, at, bt, sb, vec, st);
    else gemm_cfg<T, 4, 4, 2>(g, at, bt, ss, vec, st);
  }
}

template void launch_layer<float>(const Shape&, const LayerArgs&, int, cudaStream_t);
template void launch_layer<double>(const Shape&, const LayerArgs&, int, cudaStream_t);
template void launch_envelope<float>(const Shape&, const OrbArgs&, cudaStream_t);
template void launch_orbitals<float>(const Shape&, const OrbArgs&, int, cudaStream_t);
template void launch_orbitals<double>(const Shape&, const OrbArgs&, int, cudaStream_t);
template void launch_gemm<float>(GemmArgs<float>, bool, bool, int, int, cudaStream_t);
template void launch_gemm<double>(GemmArgs<double>, bool, bool, int, int, cudaStream_t);

}  // namespace simt
}  // namespace fn
