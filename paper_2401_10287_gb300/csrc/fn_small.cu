// Value pass and Metropolis chain of a small network in one kernel (FP64 mode).
//
// A small network (H2, LiH with 16..64 columns) leaves every kernel of the general path with a
// few CTAs, and a Metropolis step is ten of them: 0.28 ms per step for 256 H2 walkers, almost
// all of it idle.  Walkers never interact, so a CTA takes a few whole walkers through every
// stage, features to determinants, with all activations in shared memory, and through every
// step of the chain: propose, evaluate, accept.  One thread per (walker, electron, column) of a
// layer; the mean-field product, common to a walker's electrons, is split over their threads.
//
// The FP64 pipe takes one warp instruction in 64 cycles per SM quarter, so one warp per quarter
// saturates it and the dot products need no further splitting; weights come from L1/L2 (the
// prepared layouts of the general path), which that pace hides.
// H2 (2 x 32 / 8, one determinant), 256 walkers, start + 20 steps + E_L: 6.7 -> 1.34 ms (the chain 0.58 ms).
#include <climits>

#include <algorithm>

#include "fn_device.cuh"
#include "fn_internal.cuh"
#include "fn_lu.cuh"
#include "fn_rng.cuh"
#include "fn_small.cuh"

namespace fn {

constexpr int kSmallThreads = 256;       // at most
constexpr int kSmallSteps = 256;         // Metropolis steps per launch (bounds a kernel's duration)

struct SmallArgs {
  int N, n_up, n_dn, M, L, h1, h2, K, aniso, G;
  int d_h[kMaxLayers], d_g[kMaxLayers], k_self[kMaxLayers];
  const double* VsT[kMaxLayers]; const double* UT[kMaxLayers]; const double* b[kMaxLayers];
  const double* W[kMaxLayers]; const double* c[kMaxLayers];
  const double* wT[2]; const double* g[2]; const double* pi[2]; const double* sig[2];
  const double* nuc;
  int B, n_steps;
  double* walkers; double* lp; int8_t* sign;
  double step_size; uint64_t seed, walker_offset; uint32_t step0;
  unsigned long long* accepted;
  int* status;
};

// Shared-memory layout (elements of double, per CTA of G walkers).
struct SmallLayout {
  int r, rp, h[2], hbar, pm, g[2], gm, phi, mant, expo, lp, lpn, total;
};
__host__ __device__ inline SmallLayout small_layout(const SmallArgs& a) {
  const int hw = a.h1 > 4 * a.M ? a.h1 : 4 * a.M, gw = a.h2 > 4 ? a.h2 : 4;
  SmallLayout s;
  int o = 0;
  auto take = [&](int n) { const int v = o; o += n * a.G; return v; };
  s.r = take(3 * a.N);
  s.rp = take(3 * a.N);
  s.h[0] = take(a.N * hw);
  s.h[1] = take(a.N * hw);
  s.hbar = take(2 * hw);
  s.pm = take(a.N * a.h1);
  s.g[0] = take(a.N * a.N * gw);
  s.g[1] = take(a.N * a.N * gw);
  s.gm = take(a.N * 2 * gw);
  s.phi = take(a.K * (a.n_up * a.n_up + a.n_dn * a.n_dn));
  s.mant = take(2 * a.K);
  s.expo = take(a.K);                    // 2K ints
  s.lp = take(1);
  s.lpn = take(1);
  s.total = o;
  return s;
}

// log|psi| and sign of the CTA's nw walkers at positions r (shared memory) -> lp_out, sign.
__device__ void small_eval(const SmallArgs& a, const SmallLayout& s, double* sm, int nw, const double* r,
                           double* lp_out, int8_t* sign_out) {
  const int tid = threadIdx.x, nt = blockDim.x, N = a.N, M = a.M;
  const int hw = max(a.h1, 4 * M), gw = max(a.h2, 4);
  double *h = sm + s.h[0], *h2 = sm + s.h[1], *g = sm + s.g[0], *g2 = sm + s.g[1];
  double *hbar = sm + s.hbar, *pm = sm + s.pm, *gm = sm + s.gm, *phi = sm + s.phi;
  // features; element (w, i, c) of h at (w N + i) hw + c, (w, i, j, c) of g at ((w N + i) N + j) gw + c
  for (int e = tid; e < nw * N * M; e += nt) {
    const int m = e % M, wi = e / M;
    const double* p = r + 3 * wi;
    const double d0 = p[0] - a.nuc[3 * m], d1 = p[1] - a.nuc[3 * m + 1], d2 = p[2] - a.nuc[3 * m + 2];
    double* o = h + wi * hw + 4 * m;
    o[0] = d0; o[1] = d1; o[2] = d2; o[3] = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
  }
  for (int e = tid; e < nw * N * N; e += nt) {
    const int j = e % N, wi = e / N, w = wi / N, i = wi - w * N;
    double d[4] = {0.0, 0.0, 0.0, 0.0};
    if (i != j) {
      const double *p = r + 3 * wi, *q = r + 3 * (w * N + j);
      d[0] = p[0] - q[0]; d[1] = p[1] - q[1]; d[2] = p[2] - q[2];
      d[3] = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    }
    double* o = g + e * gw;
    for (int c = 0; c < 4; ++c) o[c] = d[c];
  }
  __syncthreads();
  for (int l = 0; l < a.L; ++l) {
    const int dh = a.d_h[l], dg = a.d_g[l], h1 = a.h1;
    // spin means of h (per walker) and of g (per electron)
    for (int e = tid; e < nw * 2 * dh; e += nt) {
      const int c = e % dh, ws = e / dh, w = ws >> 1, lo = (ws & 1) ? a.n_up : 0, hi = (ws & 1) ? N : a.n_up;
      double v = 0.0;
      for (int i = lo; i < hi; ++i) v += h[(w * N + i) * hw + c];
      hbar[w * 2 * hw + (ws & 1) * dh + c] = hi > lo ? v / (double)(hi - lo) : 0.0;
    }
    for (int e = tid; e < nw * N * 2 * dg; e += nt) {
      const int c = e % dg, q = e / dg, wi = q >> 1, lo = (q & 1) ? a.n_up : 0, hi = (q & 1) ? N : a.n_up;
      double v = 0.0;
      for (int j = lo; j < hi; ++j) v += g[(wi * N + j) * gw + c];
      gm[wi * 2 * gw + (q & 1) * dg + c] = hi > lo ? v / (double)(hi - lo) : 0.0;
    }
    __syncthreads();
    // z without the mean-field term into h2, and electron i's share of the mean-field product
    const double *V = a.VsT[l], *U = a.UT[l];
    for (int e = tid; e < nw * N * h1; e += nt) {
      const int n = e % h1, wi = e / h1, w = wi / N, i = wi - w * N;
      const double *hi_ = h + wi * hw, *gi = gm + wi * 2 * gw, *hb = hbar + w * 2 * hw;
      double z = 0.0, m = i == 0 ? a.b[l][n] : 0.0;
      for (int k = 0; k < dh; ++k) z += hi_[k] * V[(int64_t)k * h1 + n];
      for (int k = 0; k < 2 * dg; ++k) z += gi[k] * V[(int64_t)(dh + k) * h1 + n];
      for (int k = 2 * dh * i / N; k < 2 * dh * (i + 1) / N; ++k) m += hb[k] * U[(int64_t)k * h1 + n];
      h2[wi * hw + n] = z;
      pm[wi * h1 + n] = m;
    }
    // next pair activations
    if (l < a.L - 1) {
      const double *W = a.W[l], *cc = a.c[l];
      for (int e = tid; e < nw * N * N * a.h2; e += nt) {
        const int c = e % a.h2, p = e / a.h2;
        double v = cc[c];
        for (int k = 0; k < dg; ++k) v += W[c * dg + k] * g[p * gw + k];
        v = tanh(v);
        g2[p * gw + c] = l > 0 ? v + g[p * gw + c] : v;
      }
    }
    __syncthreads();
    for (int e = tid; e < nw * N * h1; e += nt) {
      const int n = e % h1, wi = e / h1, w = wi / N;
      double z = h2[wi * hw + n];
      for (int i = 0; i < N; ++i) z += pm[(w * N + i) * h1 + n];
      const double v = tanh(z);
      h2[wi * hw + n] = l > 0 ? v + h[wi * hw + n] : v;
    }
    __syncthreads();
    { double* t = h; h = h2; h2 = t; }
    if (l < a.L - 1) { double* t = g; g = g2; g2 = t; }
  }
  // orbital matrices: element (k, i, j) of a spin block at (k n + i) n + j
  const int up2 = a.n_up * a.n_up, per = up2 + a.n_dn * a.n_dn;
  for (int e = tid; e < nw * a.K * per; e += nt) {
    const int w = e / (a.K * per);
    int q = e - w * a.K * per;
    const int sp = q < a.K * up2 ? 0 : 1, n = sp ? a.n_dn : a.n_up;
    if (sp) q -= a.K * up2;
    const int ko = q / n, jj = q - ko * n, n_ko = a.K * n;
    const int wi = w * N + (sp ? a.n_up : 0) + jj;
    double p = a.g[sp][ko];
    for (int c = 0; c < a.h1; ++c) p += h[wi * hw + c] * a.wT[sp][(int64_t)c * n_ko + ko];
    const double* pr = r + 3 * wi;
    double env = 0.0;
    for (int m = 0; m < M; ++m) {
      const double d0 = pr[0] - a.nuc[3 * m], d1 = pr[1] - a.nuc[3 * m + 1], d2 = pr[2] - a.nuc[3 * m + 2];
      double t;
      if (!a.aniso) {
        t = a.sig[sp][ko * M + m] * sqrt(d0 * d0 + d1 * d1 + d2 * d2);
      } else {
        const double* S = a.sig[sp] + (ko * M + m) * 9;
        const double u0 = S[0] * d0 + S[1] * d1 + S[2] * d2, u1 = S[3] * d0 + S[4] * d1 + S[5] * d2,
                     u2 = S[6] * d0 + S[7] * d1 + S[8] * d2;
        t = sqrt(u0 * u0 + u1 * u1 + u2 * u2);
      }
      env += a.pi[sp][ko * M + m] * exp(-t);
    }
    phi[e] = p * env;
  }
  __syncthreads();
  double* mant = sm + s.mant;
  int* expo = (int*)(sm + s.expo);
  for (int e = tid; e < nw * 2 * a.K; e += nt) {
    const int w = e / (2 * a.K), q = e - w * 2 * a.K, k = q >> 1, sp = q & 1, n = sp ? a.n_dn : a.n_up;
    if (n == 0) {
      mant[e] = 1.0;
      expo[e] = 0;
    } else {
      lu_regs_any<double, double>(phi + w * a.K * per + (sp ? a.K * up2 : 0) + k * n * n, n, mant + e, expo + e);
    }
  }
  __syncthreads();
  // the signed sum of the determinants, as in k_det_value_small
  for (int w = tid; w < nw; w += nt) {
    const double* mt = mant + w * 2 * a.K;
    const int* ex = expo + w * 2 * a.K;
    int emax = INT_MIN;
    for (int k = 0; k < a.K; ++k)
      if (mt[2 * k] * mt[2 * k + 1] != 0 && ex[2 * k] + ex[2 * k + 1] > emax) emax = ex[2 * k] + ex[2 * k + 1];
    double S = 0.0;
    for (int k = 0; k < a.K; ++k) {
      const double mk = mt[2 * k] * mt[2 * k + 1];
      if (mk != 0) S += ldexp(mk, ex[2 * k] + ex[2 * k + 1] - emax);
    }
    const int sgn = S > 0 ? 1 : (S < 0 ? -1 : 0);
    const double lpsi = sgn == 0 ? log(fabs(S)) : log(fabs(S)) + (double)emax * 0.6931471805599453;
    lp_out[w] = lpsi;
    if (sign_out) sign_out[w] = (int8_t)sgn;
    if (sgn == 0) atomicOr(a.status, kStatusSingular);
    else if (!isfinite(lpsi)) atomicOr(a.status, kStatusNonFinite);
  }
  __syncthreads();
}

// log|psi| and sign of every walker (n_steps = 0), or n_steps Metropolis steps from d_log_psi.
__global__ void __launch_bounds__(kSmallThreads) k_small(SmallArgs a) {
  pdl_wait();
  pdl_launch();
  extern __shared__ __align__(16) double small_smem[];
  double* sm = small_smem;
  const SmallLayout s = small_layout(a);
  const int w0 = blockIdx.x * a.G, nw = min(a.G, a.B - w0), N = a.N, n3 = 3 * N, tid = threadIdx.x, nt = blockDim.x;
  double *r = sm + s.r, *rp = sm + s.rp, *lp = sm + s.lp, *lpn = sm + s.lpn;
  for (int e = tid; e < nw * n3; e += nt) r[e] = a.walkers[(int64_t)w0 * n3 + e];
  if (a.n_steps == 0) {
    __syncthreads();
    small_eval(a, s, sm, nw, r, lpn, a.sign ? a.sign + w0 : nullptr);
    for (int w = tid; w < nw; w += nt) a.lp[w0 + w] = lpn[w];
    return;
  }
  for (int w = tid; w < nw; w += nt) lp[w] = a.lp[w0 + w];
  int taken = 0;                                 // accepted moves of the walkers of this thread
  const int pairs = (n3 + 1) / 2;
  for (int k = 0; k < a.n_steps; ++k) {
    const uint32_t step = a.step0 + (uint32_t)k;
    __syncthreads();
    for (int e = tid; e < nw * pairs; e += nt) { // a Box-Muller pair moves two coordinates
      const int w = e / pairs, j = 2 * (e - w * pairs);
      double z0, z1;
      normal_pair((uint32_t)(j >> 1), (uint32_t)(a.walker_offset + w0 + w), step, (uint32_t)kStreamProposal, a.seed, &z0, &z1);
      rp[w * n3 + j] = __dadd_rn(r[w * n3 + j], __dmul_rn(z0, a.step_size));
      if (j + 1 < n3) rp[w * n3 + j + 1] = __dadd_rn(r[w * n3 + j + 1], __dmul_rn(z1, a.step_size));
    }
    __syncthreads();
    small_eval(a, s, sm, nw, rp, lpn, nullptr);
    for (int w = tid; w < nw; w += nt) {
      const double log_u = log_uniform_accept((uint32_t)(a.walker_offset + w0 + w), step, a.seed);
      const double d = __dmul_rn(2.0, __dadd_rn(lpn[w], -lp[w]));
      if (log_u <= d) {                          // ties accept; NaN proposals are rejected
        for (int c = 0; c < n3; ++c) r[w * n3 + c] = rp[w * n3 + c];
        lp[w] = lpn[w];
        ++taken;
      }
    }
  }
  __syncthreads();
  for (int e = tid; e < nw * n3; e += nt) a.walkers[(int64_t)w0 * n3 + e] = r[e];
  for (int w = tid; w < nw; w += nt) a.lp[w0 + w] = lp[w];
  if (a.accepted && taken) atomicAdd(a.accepted, (unsigned long long)taken);
}

static SmallArgs small_args(const fn_system* s) {
  SmallArgs a{};
  const double* prep = (const double*)s->ws.prep;
  a.N = s->N; a.n_up = s->n_up; a.n_dn = s->n_dn; a.M = s->M; a.L = s->cfg.n_layers;
  a.h1 = s->cfg.h1; a.h2 = s->cfg.h2; a.K = s->cfg.n_dets; a.aniso = s->cfg.envelope == FN_ENV_ANISOTROPIC;
  for (int l = 0; l < a.L; ++l) {
    a.d_h[l] = s->layer[l].d_h; a.d_g[l] = s->layer[l].d_g; a.k_self[l] = s->layer[l].k_self;
    a.VsT[l] = prep + s->prep.VsT[l]; a.UT[l] = prep + s->prep.UT[l]; a.b[l] = prep + s->prep.b[l];
    if (l < a.L - 1) { a.W[l] = prep + s->prep.W[l]; a.c[l] = prep + s->prep.c[l]; }
  }
  for (int q = 0; q < 2; ++q) {
    a.wT[q] = prep + s->prep.wT[q]; a.g[q] = prep + s->prep.g[q];
    a.pi[q] = prep + s->prep.pi[q]; a.sig[q] = prep + s->prep.sig[q];
  }
  a.nuc = s->d_nuclei;
  a.status = s->ws.status;
  // walkers per CTA: about 128 threads of layer outputs
  a.G = std::max(1, std::min(8, 128 / (a.N * a.h1)));
  return a;
}

// Where it is the faster path (log|psi| and a Metropolis step, against the general kernels, FP64; networks
// 2 x 16 / 8, 2 x 32 / 8, 4 x 48 / 16, 3 x 64 / 16 and / 32 with 1 to 16 determinants): one or two electrons
// at every batch (65536 walkers: 1.01 to 2.7 x).  With more, dot products without register tiling lose once
// the general kernels have CTAs enough: LiH 1.03 to 1.2 x at 2048 to 4096 walkers, 0.75 to 0.92 at 65536;
// C 1.04 to 1.26 at 2048, 0.63 to 0.94 at 65536; O 1.17 to 1.4 at 1024, 0.88 to 1.05 at 2048, 0.62 to 0.86 at
// 65536.  At 16 columns the general tiles are half padding: up to four electrons win at every batch (1.15 x),
// C at 16384 (1.06), O at 4096 (1.08).
static bool small_wins(int N, int h1, int B) {
  if (N <= (h1 <= 16 ? 4 : 2)) return true;
  return (int64_t)B * N <= (h1 <= 16 ? 65536 : 12288);
}

bool small_covers(const fn_system* s, int B) {
  if (s->cfg.precision != FN_FP64 || s->N > 8 || s->cfg.h1 > 64 || s->cfg.n_dets > 16) return false;
  return small_wins(s->N, s->cfg.h1, B) && small_layout(small_args(s)).total * sizeof(double) <= 96 * 1024;
}

static void launch(const SmallArgs& a, cudaStream_t st) {
  const int threads = (int)std::min<int64_t>(kSmallThreads, round_up((int64_t)a.G * a.N * a.h1, 32));
  const size_t smem = small_layout(a).total * sizeof(double);
  cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_k(false, k_small, (unsigned)((a.B + a.G - 1) / a.G), threads, smem, st, a);
}

void launch_small_log_psi(const fn_system* s, const void* walkers, int B, double* log_psi, int8_t* sign, cudaStream_t st) {
  SmallArgs a = small_args(s);
  a.B = B;
  a.walkers = (double*)const_cast<void*>(walkers);
  a.lp = log_psi;
  a.sign = sign;
  ProfScope ps(s->prof, kProfLayerValue, st);
  launch(a, st);
}

void launch_small_mcmc(const fn_system* s, void* walkers, double* log_psi, int B, int n_steps, double step_size,
                       uint64_t seed, uint64_t step_offset, int64_t* accept, cudaStream_t st) {
  SmallArgs a = small_args(s);
  a.B = B;
  a.walkers = (double*)walkers;
  a.lp = log_psi;
  a.step_size = step_size;
  a.seed = seed;
  a.walker_offset = s->walker_offset;
  a.accepted = (unsigned long long*)accept;
  ProfScope ps(s->prof, kProfSampler, st);
  for (int k = 0; k < n_steps; k += kSmallSteps) {
    a.step0 = (uint32_t)(step_offset + (uint64_t)k);
    a.n_steps = std::min(kSmallSteps, n_steps - k);
    launch(a, st);
  }
}

}  // namespace fn
