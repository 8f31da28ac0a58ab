// Tensor-network contractions of one site (H_eff, K_eff, environment updates)
// and the Lanczos local exponential, as free functions over device pointers.
// The engine and the handle-free C-ABI entry points share them.
#pragma once
#include <functional>
#include <memory>

#include "linalg.cuh"
#include "tc_gemm.cuh"

// Everything one-site contractions read: environments, MPO site, dimensions.
struct SiteOp {
  const cplx* L = nullptr;     // ml x wl x ml
  const cplx* R = nullptr;     // mr x wr x mr
  const WSparse* W = nullptr;  // MPO site (sparse lists on device)
  int ml = 0, mr = 0, wl = 0, wr = 0, d = 2;
  long long env_key = -1;      // identifies the (L, R) content for operand caching; -1 = never cache
};

struct F64EnvDigits;  // digits of the environments of the FP64 tensor-core path (tc_f64.cu)
struct TcSliceCache;  // sliced operands of the BF16 tensor-core path (tc_bf16.cu)

// Work buffers reused across calls (drawn from a pool).
struct Scratch {
  DevicePool* pool = nullptr;
  DArr t1, t2, t3;
  TcEnvCache tc;
  std::shared_ptr<TcSliceCache> tcs;
  std::shared_ptr<F64EnvDigits> f64;
};

// Algorithmic flop count of one H_eff apply (8 real flops per complex multiply-add):
// 8 [ml d mr (ml wl + mr wr) + ml mr nnz(W)]
double heff_flops(const SiteOp& op);

// y[a,s,b] = sum L[a,w,a'] W[w,s,s',v] x[a',s',b'] R[b,v,b']
void heff_fp64(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y);
void heff_tf32x3(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y);
// The same on the BF16 exact-slice tensor-core GEMM with S = 3 or 4 slices per operand.
void heff_bf16s(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y, int S);
// Slices per operand of a BF16 precision mode (BF16X6: 3, BF16X10: 4).
int bf16_slices(int precision);
// (output tile, 128-entry K chunk) pairs the BF16 tensor-core GEMMs visited on the current
// device since the library loaded: out[0] all of them, out[1] the ones multiplied (the rest
// had an all-zero A or B tile and were skipped).  Synchronises the device.
void gemm_chunk_pairs(long long out[2]);
bool prec_is_bf16(int precision);
void heff_apply_prec(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y, int precision);
// C = opA(A) opB(B) (complex, alpha = 1, beta = 0) on the tensor cores (split TF32,
// FP32 accumulation, FP64 output).
void zgemm_tc(cudaStream_t st, Scratch& s, int opA, int opB, int M, int N, int K, const cplx* A, long long lda,
              const cplx* B, long long ldb, cplx* C, long long ldc);
// C = opA(A) opB(B) on the BF16 exact-slice tensor-core GEMM (S slices, FP64 output).
void zgemm_bf16s(cudaStream_t st, Scratch& s, int S, int opA, int opB, int M, int N, int K, const cplx* A,
                 long long lda, const cplx* B, long long ldb, cplx* C, long long ldc);
// FP64 on the tensor cores by exact 8-bit digits (tc_f64.cu): whether a complex product of this
// size belongs there, C = alpha opA(A) opB(B) + beta C, and H_eff.
bool f64_on_tensor_cores(long long M, long long N, long long K);
void zgemm_f64s(cudaStream_t st, Scratch& s, int opA, int opB, int M, int N, int K, cplx alpha, const cplx* A,
                long long lda, const cplx* B, long long ldb, cplx beta, cplx* C, long long ldc);
void heff_f64s(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y);
// The FP64 product by size: exact digits on the tensor cores, or the CUDA-core GEMM.
void zgemm_fp64(cudaStream_t st, Scratch& s, int opA, int opB, int M, int N, int K, cplx alpha, const cplx* A,
                long long lda, const cplx* B, long long ldb, cplx beta, cplx* C, long long ldc);
// The error word of the tensor-core kernels' bounded waits (read by tc_check); marks it pending.
int* tc_error_word(cudaStream_t st, Scratch& s);
// The tensor-core GEMM of `precision` (zgemm_tc for the TF32 modes, zgemm_bf16s for
// the BF16 modes) when the product is large enough to fill its tiles, the FP64
// GEMM otherwise (alpha = 1, beta = 0).
void zgemm_prec(cudaStream_t st, Scratch& s, int precision, int opA, int opB, int M, int N, int K, const cplx* A,
                long long lda, const cplx* B, long long ldb, cplx* C, long long ldc);
// Reads the tensor-core error word of the launches since the last check (synchronises);
// throws TDVP_ERR_TIMEOUT when a bounded device wait ran out.
void tc_check(cudaStream_t st, Scratch& s);

// y[a,c] = sum L[a,w,a'] x[a',b'] R[c,w,b']   (x: ml x mr; L: ml x w x ml; R: mr x w x mr)
void keff_fp64(cudaStream_t st, Scratch& s, const cplx* L, int ml, const cplx* R, int mr, int w, const cplx* x,
               cplx* y, int precision = TDVP_PREC_FP64);

// Lout[b,v,b'] = sum conj(A[a,s,b]) L[a,w,a'] W[w,s,s',v] A[a',s',b']
void env_left_fp64(cudaStream_t st, Scratch& s, const cplx* L, const WSparse& W, const cplx* A, int ml, int mr,
                   int d, cplx* Lout, int precision = TDVP_PREC_FP64);
// Rout[a,w,a'] = sum conj(B[a,s,b]) W[w,s,s',v] R[b,v,b'] B[a',s',b']
void env_right_fp64(cudaStream_t st, Scratch& s, const cplx* R, const WSparse& W, const cplx* B, int ml, int mr,
                    int d, cplx* Rout, int precision = TDVP_PREC_FP64);

// Lanczos exponential with full re-orthogonalisation applied twice:
// out = exp(-i delta Op) x (kind 0) or exp(-delta Op) x (kind 1), Op Hermitian.
// Returns the Krylov dimension used; throws LANCZOS_NOT_CONVERGED when nmax
// steps do not bring the error estimate below tol.
struct LanczosWork {
  DArr V, w, c, y;
  RawBuf live;             // bitmap of the nonzero 32-entry groups of the basis
  double* real = nullptr;  // device: alpha[64], beta[65], nrm2[2] at 130, scratch norms; |x|^2 at 255 and
                           // from 256 the error estimates of each iteration of a batch
  void init(DevicePool* pool);
  void release();
};
// hint (may be null): the Krylov dimension of the previous run of the same operator kind; read
// to size the first batch of iterations a small local problem launches without a host round
// trip each, and updated to this run's dimension.  Results do not depend on it.
// scr: whose error word the operator's bounded waits set; once it is set the run ends with
// TDVP_ERR_TIMEOUT at its next stopping test (the word is left for tc_check).
int lanczos_expm(cudaStream_t st, DevicePool* pool, Blas1& blas, LanczosWork& lw, const Scratch& scr,
                 const std::function<void(const cplx*, cplx*)>& op, const cplx* x, cplx* out, long long n,
                 double delta, int kind, double tol, int nmax, int* hint = nullptr);
