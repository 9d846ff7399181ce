// Launch interface of the FP32/FP64 kernels of fn_simt.cu.
#pragma once
#include "fn_internal.cuh"

namespace fn {
namespace simt {

struct LayerArgs {
  const void* X; int ldx; int k_self;
  const void* VsT;      // [k_self][h1]
  const void* Mterm;    // [T][B][h1]
  void* Y; int ldy;     // output [T][R][ldy]
  int residual;
  void* Hbar_out;       // [T][B][2 h1] or null
  void* act_out;        // [R][h1] tanh values (value pass) or null
  int h1;
};

struct OrbArgs {
  const void* HL;               // [T][R][h1]
  const void* wT[2]; const void* g[2]; const void* pi[2]; const void* sig[2];
  void* Phi;                    // [B][PW]
  int64_t PW;                   // elements per walker
  int h1, K, aniso;
  const void* walkers;          // [B][N][3]
  const double* nuclei;
  void* envv;                   // full pass: [K N][R] envelope values
  void* orbP;                   // full pass: [R][4][K N] value and own-coordinate projections
};

template <typename T>
struct GemmArgs {
  int64_t M;
  int N, K;
  const T* A; int64_t lda;
  const T* B; int64_t ldb;
  T* C; int64_t ldc;
  const T* bias; int64_t bias_rows;
  int atomic;
};

// One stream layer over all slabs of sh; the tile shape is chosen from the number of CTAs.
template <typename T> void launch_layer(const Shape& sh, const LayerArgs& a, int sm_count, cudaStream_t st);
// Envelope values of every electron's own-spin orbitals into a.envv.
template <typename T> void launch_envelope(const Shape& sh, const OrbArgs& a, cudaStream_t st);
// Orbital matrices of every slab; in the full pass without the envelope-derivative terms
// (which k_orbital_fixup adds from orbP).
template <typename T> void launch_orbitals(const Shape& sh, const OrbArgs& a, int sm_count, cudaStream_t st);
// max_split > 1 allows splitting K over CTAs, whose results are added atomically to C.
template <typename T>
void launch_gemm(GemmArgs<T> g, bool at, bool bt, int max_split, int sm_count, cudaStream_t st);

}  // namespace simt
}  // namespace fn
