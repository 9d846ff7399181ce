// Launch interface of the FP32 tensor-core kernels of fn_x3.cu.
#pragma once
#include "fn_internal.cuh"

namespace fn {
namespace x3 {

enum { kLayer = 0, kPlain = 1, kOrbital = 2 };

struct Args {
  Shape sh;
  int tiles;                     // row tiles of 128 (orbitals: rtiles per slab x T); CTA rows stride over them
  int nkb, kd, ncols, ldw;       // k-blocks of 64, contraction length, output columns, weight part stride
  int brow0;                     // first weight row
  const float* A; int lda;       // FP32 rows
  const float* Mterm; int residual;                  // layer
  int64_t rows; const float* bias; int bias_rows;    // GEMM: rows and bias; orbitals: bias g
  int n_s, e0, wpc, rtiles, K, poff;                 // orbitals: electrons of the spin, walkers per row tile
  float* Phi; int64_t PW, phi_off;
  const float* envv; float* orbP;
  int* status;
};

// One weight matrix: `rows` rows of kd columns, columns [0, len1) from blob[src1 + r src_ld + k] and the
// rest from blob[src2 + r src_ld + k - len1]; its parts go to out[dst + (3 r + part) ldw + k].
struct SplitEntry {
  int64_t src1, src2, src_ld, dst;
  int len1, kd, ldw, rows;
};
struct SplitList {
  SplitEntry e[2 * kMaxLayers + 2];
  int n;
};

// Whether these kernels can run: the driver encodes tensor maps and every kernel has the registers
// its split needs.  Decided when a handle is created; without them FP32 passes stay on the FMA pipe.
bool available();
void launch_split_weights(const float* blob, const SplitList& list, void* out, cudaStream_t st);
// false: a tensor map could not be built (nothing launched)
bool launch_layer(const Shape& sh, const float* X, int ldx, int k_self, const void* W, int ldw, const float* Mterm,
                  float* Y, int ldy, int residual, int h1, int* status, int sm_count, cudaStream_t st);
bool launch_gemm(int64_t rows, int k, const float* A, int lda, const void* W, int ldw, int ncols, float* C,
                 const float* bias, int bias_rows, int* status, int sm_count, cudaStream_t st);
bool launch_orbitals(const Shape& sh, int spin, const float* HL, int h1, const void* W, int ldw, const float* bias,
                     int K, float* Phi, int64_t PW, const float* envv, float* orbP, int* status, int sm_count,
                     cudaStream_t st);

}  // namespace x3
}  // namespace fn
