// internal.h — declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/ps_poisson.h"
#include "common.cuh"

namespace ps {

// Launch with programmatic stream serialisation (see pdl_wait, common.cuh): the launch
// latency overlaps the end of the kernel ahead of it. Most of a small solve's launches are
// skipped kernels of the refinement loop after convergence, 2.1 µs each (4.1 with 2000
// CTAs) without it. Solves without → with: 32^3 FP64 55 → 45 µs, 512×256×144 refined
// 817 → 708 µs, 128^3 RK3 step 1645 → 1311 µs, 1024^3 32.21 → 32.09 ms.
template <class... P, class... A>
cudaError_t launch_k(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

enum { BC_P = 0, BC_NN = 1, BC_DD = 2, BC_ND = 3, BC_DN = 4, BC_FD = 5 /* z only: face unknowns */ };
// ND and DN share the DCT-IV line transform: DN is the ND problem on the reversed
// line, so on the physical side of a transform the two reals x_{2p} and x_{n−1−2p}
// trade places; the spectral side, the tables and the eigenvalues are ND's.
__host__ __device__ inline bool bc_iv(int bc) { return bc == BC_ND || bc == BC_DN; }
// Longest x or y line: lines of n ≤ 1024 run in the register-resident transform
// kernels; longer ones in the shared-memory kernel, one line per CTA (two buffers
// of n/2 + 1 complex values: 131 KB for an FP64 line of 8192)
constexpr int kMaxN = 8192;
constexpr int kSMs = 152;  // of the part this is written for (rules on how far work is split)
constexpr int kMaxStages = 6;   // of a generic line FFT (radices up to 9: m ≤ 4096 needs 4)
extern thread_local char g_launch_diag[256];  // configuration of the last failed launch
// Test hook (ps_inject_alloc_failures): true while injected device-allocation failures
// remain; each call consumes one.
bool take_injected_alloc_failure();

// One Stockham stage of a generic line FFT of m points: radix r, nb = m/r butterflies,
// ns the product of the earlier radices, tws = m/(ns·r), mg = ⌈2^32/ns⌉ (0 for ns = 1).
struct FftStage {
  int r, nb, ns, tws;
  unsigned mg;
};
// A line's tables and FFT stages (device memory), made at plan creation. The split and
// BC factors of xform_dev.cuh with their constants folded in, [0] backward, [1] forward:
//   t0: k ≤ m/2: forward −(i/2)e^{−2πik/2m}, backward i·e^{+2πik/2m}/2m (FD: the forward one
//       both ways); DCT-IV: e^{−iπk/n}, k < m;
//   t1: NN, DD: q ≤ m: forward 2e^{−iπq/2n}, backward ½e^{+iπq/2n}; DCT-IV: k < m:
//       e^{−iπ(4k+1)/4n} times 2 (forward) or 1/n (backward); else null.
template <class T>
struct LineTab {
  const FftStage* stage;
  int nstages;
  unsigned mg_m, mg_h;      // reciprocals of m and n/2
  T inv2m;                  // 1/(2m)
  const cplx<T>* w;         // e^{−2πit/m}, t < m
  const cplx<T>* t0[2];
  const cplx<T>* t1[2];
};

// Arguments of one batch of line transforms (x or y).
template <class T>
struct XformArgs {
  const void* in;
  void* out;
  int n, m;          // line length and half length
  int axis;          // 0 = x (contiguous rows), 1 = y (strided by nx)
  int nx, ny, nz;
  int nlines;        // x: nz*ny rows
  int lgL;           // log2 of the lines per tile (set by the launcher)
  int bc;
  LineTab<T> tab;
  const T* plane_scale;     // per-z factor on load (fwd) / store (bwd), or null
  int accumulate;           // store: out = out + v
  const int* skip;          // if non-null and *skip != 0 the kernel returns at once
  unsigned long long* amax; // FP64 output: atomicMax of |transform output| bit patterns, or null
  float* out2;              // FP64 output: also store the FP32 transform output here, or null
  const float* base32;      // FP64 output: out = widen(base32) + v instead of (out +) v, or null
};

template <class T, class TI, class TO, bool FWD>
cudaError_t launch_xform(XformArgs<T> a, cudaStream_t st);

// z tridiagonal solves of Eq. 5, one per (q_x, q_y) column.
template <class T>
struct ZArgs {
  T* data;                  // [nz][ny][nx], spectral in x and y; overwritten with Φ̂
  T* scr_c;                 // scratch, nx*ny*nz (eliminated upper diagonal)
  T* scr_u;                 // scratch of a periodic z (carried coefficients), or null
  int nx, ny, nz;
  const T* lamx;            // λ_qx/Δx², nx
  const T* lamy;            // λ_qy/Δy², ny
  const T* za;              // a_k (sub-diagonal; a_0 = wrap coupling when periodic)
  const T* zc;              // c_k (super-diagonal; c_{n−1} = wrap coupling when periodic)
  const T* zg;              // excess g_k = −(a_k + b_k + c_k) ≥ 0 of the diagonal without λ (a Dirichlet
                            // end, the Helmholtz shift), from its terms, not by subtraction
  const T* dzf;             // cell widths (weights of the singular column)
  int periodic;
  int singular;             // column (0,0) is singular: handled by the fix-up kernel
  const int* skip;
  // FP32 path: the columns q_x < lowx, q_y < lowy (the worst-conditioned, see tridiag.cu;
  // the singular one among them) are solved in double-float by extra CTAs of the same
  // launch (0: none).
  int lowx, lowy;
  const double *lamx64, *lamy64, *dzf64;
  const float2* zdf;        // per plane (a_k, c_k, g_k) in double-float
  float ga, ge0, ge1;       // the excess g_k in its terms: every row's (the shift), the first and last row's extra
  double* scr64;            // 2·nz·lowx·lowy doubles
};

constexpr int ZK = 16;  // planes per checkpoint of the FP32 z sweeps (tridiag.cu)
__host__ __device__ inline int zckpt_chunks(int rows) { return (rows + ZK - 1) / ZK; }
cudaError_t launch_zsolve64(ZArgs<double> a, cudaStream_t st);     // FP64, the singular column included
cudaError_t launch_zsolve_ckpt(ZArgs<float> a, cudaStream_t st);   // FP32
cudaError_t launch_zsingular(ZArgs<float> a, cudaStream_t st);     // FP32, no rectangle

// Residuals of the refinement (residual.cu): incremental passes on an FP32
// operand with a double-float base, and the exact pass from the FP64 solution.
struct ResidArgs {
  const double* p;          // exact pass: the stored FP64 solution
  const double* f;          // exact pass and incremental pass 0: the right-hand side
  float* r;                 // exact pass: FP32 residual out (n_x·n_y·n_z floats)
  const float* u;           // incremental: FP32 operand (Φ_0 in pass 0, the last correction later)
  const float* rh_in;       // incremental pass ≥ 1: r_{m−1} = rh + rl
  const float* rl_in;
  float* rh_out;            // incremental: r_m = rh + rl out, or both null (norms only)
  float* rl_out;
  int nx, ny, nz;
  int bcx, bcy, bcz;        // ends: see residual.cu
  df idx2, idy2;            // 1/Δx², 1/Δy²
  const float2* zlo;        // coefficient of (Φ_{k−1} − Φ_k), ghost rules folded in
  const float2* zhi;        // coefficient of (Φ_{k+1} − Φ_k)
  const float2* zres;       // passes m ≥ 1: per plane (a_k, c_k, w_c) in double-float, the
                            // Dirichlet ghost sign folded into a_0 / c_{n−1} (see residual.cu)
  double asum;              // max over planes of Σ_j |w_j| (the 7 coefficients of a row)
  df nalpha;                // −α of a Helmholtz plan (A − α·I), double-float; zero otherwise
  const float* wz;          // Δz^f_k (weights of the mean, singular problems)
  const float* mu;          // double-float volume-weighted mean of f (singular)
  const unsigned long long* pmax_bits;  // bit pattern of max|operand| (sets the fixed-point scale)
  int singular;
  unsigned* red;            // per-call reduction words (see residual.cu)
  float* partial;           // per-block double-float weighted sums (2 floats per block) ×2
  int nblocks;
  int zchunk;               // planes per CTA (set by the launcher)
  const int* skip;
};

// CTAs (= partial sums) of a residual pass: which = 0 pass 0 (two-level split),
// 1 three-level split (pass 0 repeated, exact pass), 2 passes m ≥ 1
int residual_blocks(int nx, int ny, int nz, int which);
cudaError_t launch_residual_inc(const ResidArgs& a, int pass, int split3, cudaStream_t st);
cudaError_t launch_residual_exact(const ResidArgs& a, cudaStream_t st);

// Control block at the start of the workspace.
struct Ctrl {
  int converged;            // set when ‖r‖ ≤ rtol·‖f_c‖ (refinement done)
  int iterations;
  int status;
  int vskip;                // 1: the exact confirmation pass is not needed
  unsigned red[8];          // reduction words of the current residual pass (r: 0–1, f: 2–3)
  double rel, rnorm, fnorm;
  float mu[2];              // double-float weighted mean of f, set by the first finalize
  double mf;                // the same mean in FP64
  unsigned long long pmax;  // bit pattern of max|Φ| after the first FP32 solve
  unsigned long long dmax;  // bit pattern of max|e| of the last correction
  double bnd;               // accumulated drift bound of the incremental residual
  int skip_redo;            // 0: pass 0 is repeated with the three-level split
  int nomat0;               // 0: the loop ended at pass 0, p is written from Φ_0
  int skip_out;             // 0: a pass m ≥ 1 found no convergence; it is repeated with its output
  int met;                  // 1: the first correction reached rtol and another one was asked for
  unsigned long long dmax_prev;  // max|e| of the correction the current pass used
  double rel1, rnorm1;      // the first correction's residual when met is set
  int undo;                 // 1: the second correction missed rtol after met; it is taken back from p
};

cudaError_t launch_finalize(Ctrl* ctrl, const float* partial, int nblocks, double wsum_total,
                            int singular, double rtol, int iteration, int attempt, int last,
                            double anorm, const int* skip, ps_info* info, cudaStream_t st);
// After the loop: p = Φ_0 (widened exactly) if it ended at pass 0; p −= e if the second
// correction is taken back (Ctrl::undo); else nothing.
cudaError_t launch_settle(const float* u0, const float* e, double* p, size_t n, const Ctrl* ctrl, cudaStream_t st);
cudaError_t launch_finalize_exact(Ctrl* ctrl, const float* partial, int nblocks, double wsum_total,
                                  int singular, double rtol, ps_info* info, cudaStream_t st);
cudaError_t launch_info_plain(ps_info* info, cudaStream_t st);

// Staggered divergence / gradient of the projection step and their adjoints.
template <class T>
struct ProjArgs {
  int nx, ny, nz;
  int per[3];
  T idx, idy;
  const T* idzf;
  const T* idzc;
};
// op: 0 f = D u; 1 u = u* − G φ; 2 h = Gᵀ g; 3 out = g − Dᵀ s
template <class T>
cudaError_t launch_projection(int op, const ProjArgs<T>& a, const void* x0, const void* x1, void* y,
                              cudaStream_t st);

// One RK3 substep around the solve (navier_stokes.cu): the predictor (2a) and the
// pressure update (2d). idzf[k] = 1/Δz^f_k; idzc[k] = 1/(centre distance between
// cells k−1 and k), idzc[0] the periodic wrap.
template <class T>
struct NsArgs {
  int nx, ny, nz;
  int per_x, per_y, per_z;  // axis periodic (else no-slip walls at both ends)
  T idx, idy, idx2, idy2;   // 1/Δx, 1/Δy, 1/Δx², 1/Δy²
  T qx, qy;                 // ¼/Δx, ¼/Δy (flux differences of products of two sums)
  const T* idzf;
  const T* idzc;
  T nu, dt, alpha, beta, gamma;
  // FP64 fields: idx, idy, idx2, idy2, qx, qy, nu, dt, alpha, beta, gamma split into
  // hi + lo floats on the host (the predictor's double-float constants, read as
  // operands from the parameter bank instead of held in registers)
  float2 dc[11];
};
template <class T>
cudaError_t launch_ns_predict(const NsArgs<T>& a, const void* u3, const void* p, const void* ad_prev,
                              void* ustar, void* ad_out, cudaStream_t st);
template <class T>
cudaError_t launch_ns_pressure(size_t N, double scale, void* p, void* phi, cudaStream_t st);

// Record a message for ps_last_error(plan).
void set_plan_error(ps_plan* plan, const char* msg);

// The FP32 tables of a plan (used by the batched solve).
double ps_plan_internal_alpha(const ps_plan* p);  // the plan's Helmholtz shift (0: Poisson)
void ps_plan_internal_tables(const ps_plan* p, LineTab<float>* tx, LineTab<float>* ty,
                             const float** lamx, const float** lamy, const float** za, const float** zg,
                             const float** zc, const float** dzf, const double** dzf64, const float2** zdf, const float2** zlo, const float2** zhi,
                             df* idx2, df* idy2, double* wsum_total);

}  // namespace ps
