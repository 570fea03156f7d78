// Internal declarations of the device eigen path (eig.cu, eig_host.cu, modes.cu).
#pragma once
#include "internal.cuh"

namespace foa {

constexpr int kMaxSweeps = 32;  // Jacobi sweeps at most (the launch asks for 30)

// Cross-CTA synchronisation state of the cooperative Jacobi SVD, zeroed before every launch.
struct GridBar {
  unsigned count;                 // grid barrier: arrivals
  unsigned gen;                   // grid barrier: generation
  unsigned rot[kMaxSweeps];       // rotations applied in each sweep (summed over CTAs)
};

// integer scalars of one eigen-decomposition (device)
enum { ISC_R = 0, ISC_STATUS = 1, ISC_ERR = 2, ISC_ROT = 3, ISC_SWEEPS = 4, ISC_QR = 5, ISC_ITS = 6, ISC_RES = 7,
       ISC_N = 16 };  // QR: no values from the simultaneous iteration; RES: values that invit_kernel did not confirm
// rows of the sorted output block (each ld long)
enum { OUT_LRE = 0, OUT_LIM = 1, OUT_IND = 2, OUT_ARE = 3, OUT_AIM = 4, OUT_N = 5 };

struct EigArgs {
  const double *Hs;   // Hessenberg matrix whose eigenpairs are wanted (r x r, ld)
  const double *Q;    // G = Q Hs Q^T (when have_q)
  const double *U;    // U_r (m x r, ld) when have_u
  const double *H;    // H-bar of the stream (ldH), for the truncated indicator
  int ldH;
  const double *wr, *wi;
  const double *anorm;  // roots_setup_kernel's scal
  double *M;          // Hs transposed and flipped about its antidiagonal (r x r, ld)
  double *vec;        // inverse iteration: Re z, Im z, Re w, Im w planes of ld x ld (eigenvectors of Hs)
  double *tw;         // per-CTA scratch
  double *yr, *yi;    // y_i = U_r z_i (m x r, ld), unsorted
  double *ysr, *ysi;  // sorted y columns
  double *ind, *amp_re, *amp_im;
  double *out;        // OUT_N x ld sorted scalars
  int *perm;
  int *isc;
  int ld, m;
  int have_q, have_u;
  const double *hlast_p;  // h_{m+1,m} (device)
  const double *b11_p;    // beta_{1,1} (device)
};

// Simultaneous iteration for the eigenvalues (eig_roots.cu)
constexpr int kRootSteps32 = 14; // steps in FP32
constexpr int kRootSteps = 20;   // and in FP64, at most; what has not converged by then goes to the QR iteration
constexpr int kRootMinOrder = 6;   // below this order the QR iteration's few steps are as quick
constexpr int kRootMin32 = 64;    // below this one an FP64 step costs little more than its launch (5 us at order 10)
struct RootArgs {
  const double *H;    // Hessenberg matrix (ld)
  double *invsub;     // -1 / h_{i,i-1}
  float *Hf, *invsubf;  // the same rounded to FP32
  double *zr, *zi;    // 2 x ld: the values before and after a step
  double *dold;       // size of each value's last correction
  int *conv, *left;   // per value: converged (1 in FP32, 2 in FP64); per FP64 step: values that had not
  int *part;          // per value: the one nearest to its conjugate
  double *scal;       // see roots_setup_kernel
  double *wr, *wi;
  int *isc;
  int ld, min_n;
};
cudaError_t launch_roots(const RootArgs &a, int m, int sms, cudaStream_t s);
cudaError_t launch_invit(const EigArgs &e, bool after_qr, cudaStream_t s);
cudaError_t launch_vectors(const EigArgs &e, int vgrid, cudaStream_t s);

// one push-time indicator (device ring written by the indicator stream)
struct IndRecord {
  int32_t push;   // 1-based index of the push that scheduled it
  int32_t m;      // size of the projected matrix
  double value;   // max over the n_lead leading modes
};

struct EigWork {
  int K = 0;
  int vgrid = 0;
  double *A = nullptr, *U = nullptr, *sig_raw = nullptr, *sig = nullptr, *G = nullptr, *Q = nullptr, *T = nullptr,
         *Aqr = nullptr, *wr = nullptr, *wi = nullptr, *yr = nullptr, *yi = nullptr, *ysr = nullptr, *ysi = nullptr,
         *ind = nullptr, *amp_re = nullptr, *amp_im = nullptr, *out = nullptr, *rscal = nullptr, *vec = nullptr,
         *tw = nullptr, *yplanes = nullptr, *invsub = nullptr, *zr = nullptr, *zi = nullptr, *dold = nullptr;
  float *bop = nullptr;  // pre-split Y operand of the tensor-core mode product
  double *scal = nullptr;  // untruncated path: h_{m+1,m} and beta_11, copied with H_m
  int *perm = nullptr, *isc = nullptr, *conv = nullptr, *left = nullptr, *part = nullptr;
  float *hf = nullptr;  // K x K, then K
  GridBar *gb = nullptr;
};

constexpr int kSvdHalf = 128;           // threads that hold a column pair of A, and as many for J
constexpr int kSvdThreads = 2 * kSvdHalf;
constexpr int kSvdRows = (kMaxK + kSvdHalf - 1) / kSvdHalf;
constexpr long long kGridSpinCycles = 1ll << 32;  // bounded wait of a grid barrier (about 2 s at 2 GHz)
__global__ void svd_jacobi_kernel(const double *B, int ldb, int m, double *A, double *J, int lda, double *sig, int *isc,
                                  GridBar *gb, int max_sweeps, double tol, long long spin_limit, int skip_cta);
__global__ void svd_finish_kernel(const double *J, int ld, int m, const double *sig_in, double *U, double *sig,
                                  int *isc, double rank_tol);
__global__ void project_t_kernel(const double *H, int ldh, int m, const double *U, int ldu, const int *isc,
                                 double *T, int ldt);
__global__ void project_g_kernel(const double *U, int ldu, int m, const int *isc, const double *T, int ldt, double *G,
                                 int ldg);
__global__ void copy_h_kernel(const double *H, int ldh, int m, double *G, int ldg, int *isc, const double *B,
                              double *scal);
__global__ void hessenberg_kernel(double *G, int ldg, double *Q, int ldq, const int *isc);
__global__ void hqr_kernel(double *Ag, int lda, const int *isc_in, double *wr, double *wi, int *isc,
                           int smem_elems);
__global__ void order_kernel(EigArgs e, int nsel);

// v 2^(1023 - e) as a float (e a biased exponent, at least v's): -2 < result < 2, 0 below 2^-126
__device__ __forceinline__ float scaled_float(double v, int e) {
  const int hi = __double2hiint(v), ex = ((hi >> 20) & 0x7ff) - e + 127;
  if (ex <= 0) return 0.f;
  return __int_as_float((hi & 0x80000000) | (ex << 23) | ((hi & 0xfffff) << 3) | (unsigned(__double2loint(v)) >> 29));
}

// sum over the CTA, in a fixed order; red: one double per warp
__device__ __forceinline__ double block_sum(double v, double *red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  const int nw = blockDim.x >> 5;
  for (int i = 0; i < nw; ++i) t += red[i];
  __syncthreads();
  return t;
}

size_t modes_tc_bop_bytes(int kmax);
// modes.cu: Phi = V Y (Y: m x ncols real planes, ld), written to phi (ld_phi)
int launch_modes(foa_dmd *h, int m, const double *Y, int ldy, int ncols, void *phi, int64_t ld_phi);

}  // namespace foa
