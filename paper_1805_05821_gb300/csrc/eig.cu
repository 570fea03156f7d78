// Device eigen path of FOA-based DMD (the eigen extraction of Alg. 1 and Alg. 3), all in FP64:
//
//   eig_svd.cu         singular values and left singular vectors of beta_m (Sec. 3.2.2 rank truncation).
//   project_t/g_kernel G = U_r^T H_m U_r (copy_h_kernel: G = H_m without truncation).
//   hessenberg_kernel  Householder reduction of G to upper Hessenberg form G = Q Hs Q^T.
//   eig_roots.cu       eigenvalues of Hs by simultaneous iteration, all SMs at work.
//   hqr_kernel         where that does not apply or converge: the Francis double-shift QR iteration
//                      (single CTA; the sequential steps of the EISPACK routine hqr).
//   eig_vectors.cu     per eigenvalue: right and left eigenvectors of Hs by inverse iteration, and
//                      from them z, the amplitude, the error indicator and y = U_r z.
//   order_kernel       ordering by |c| (conjugate pairs share the larger |c|), |lambda|, Im.
//
// The modes Phi = V y_i are formed by the GEMM in modes.cu.
#include <cmath>
#include <cstring>
#include <vector>

#include "api_internal.cuh"
#include "eig_internal.cuh"

namespace foa {

__device__ __forceinline__ int block_max_int(int v, int *red) {
  for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  int t = red[0];
  const int nw = blockDim.x >> 5;
  for (int i = 1; i < nw; ++i) t = max(t, red[i]);
  __syncthreads();
  return t;
}

// ------------------------------------------------------------------------------ projection
// T = H_m U_r (m x r), then G = U_r^T T (r x r).  Without truncation G = H_m.
__global__ void project_t_kernel(const double *H, int ldh, int m, const double *U, int ldu, const int *isc,
                                 double *T, int ldt) {
  const int r = isc[ISC_R];
  const int64_t total = int64_t(m) * r;
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int i = int(e % m), c = int(e / m);
    double s = 0.0;
    const int k0 = i > 0 ? i - 1 : 0;  // H_m is upper Hessenberg
    for (int k = k0; k < m; ++k) s += H[i + int64_t(k) * ldh] * U[k + int64_t(c) * ldu];
    T[i + int64_t(c) * ldt] = s;
  }
}
__global__ void project_g_kernel(const double *U, int ldu, int m, const int *isc, const double *T, int ldt, double *G,
                                 int ldg) {
  const int r = isc[ISC_R];
  const int64_t total = int64_t(r) * r;
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int i = int(e % r), c = int(e / r);
    double s = 0.0;
    for (int k = 0; k < m; ++k) s += U[k + int64_t(i) * ldu] * T[k + int64_t(c) * ldt];
    G[i + int64_t(c) * ldg] = s;
  }
}
// G = H_m (Hessenberg part), and the two entries of the stream's state the untruncated eigen path
// still needs (h_{m+1,m} for the indicators, beta_11 for the amplitudes), so that nothing after this
// kernel reads H-bar or beta.
__global__ void copy_h_kernel(const double *H, int ldh, int m, double *G, int ldg, int *isc, const double *B,
                              double *scal) {
  for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < int64_t(m) * m;
       e += int64_t(gridDim.x) * blockDim.x) {
    const int i = int(e % m), c = int(e / m);
    G[i + int64_t(c) * ldg] = (i <= c + 1) ? H[i + int64_t(c) * ldh] : 0.0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    isc[ISC_R] = m;
    scal[0] = H[m + int64_t(m - 1) * ldh];
    scal[1] = B[0];
  }
}

// ------------------------------------------------------------------------------ Hessenberg
// Householder reduction G = Q Hs Q^T (single CTA).  Q accumulated explicitly.
__global__ void hessenberg_kernel(double *G, int ldg, double *Q, int ldq, const int *isc) {
  const int n = isc[ISC_R];
  extern __shared__ double sh[];
  double *v = sh;            // n
  double *red = sh + n;      // 32
  __shared__ double s_beta;
  for (int64_t e = threadIdx.x; e < int64_t(n) * n; e += blockDim.x) {
    const int i = int(e % n), c = int(e / n);
    Q[i + int64_t(c) * ldq] = (i == c) ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int k = 0; k + 2 < n; ++k) {
    // reflector for G[k+1:n, k] (identity when the entries below G[k+1,k] are already zero)
    double ss = 0.0;
    for (int i = k + 2 + threadIdx.x; i < n; i += blockDim.x) {
      const double x = G[i + int64_t(k) * ldg];
      ss += x * x;
    }
    ss = block_sum(ss, red);
    if (ss == 0.0) continue;
    const double alpha = G[(k + 1) + int64_t(k) * ldg];
    const double nrm = sqrt(alpha * alpha + ss);
    const double beta = alpha >= 0.0 ? -nrm : nrm;  // new G[k+1,k]
    const double v0 = alpha - beta;
    // v = [1, x(k+2:)/v0], tau = (beta - alpha)/beta
    for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) v[i] = (i == k + 1) ? 1.0 : G[i + int64_t(k) * ldg] / v0;
    if (threadIdx.x == 0) s_beta = (beta - alpha) / beta;
    __syncthreads();
    const double tau = s_beta;
    // G <- (I - tau v v^T) G : columns k..n-1
    for (int c = k + threadIdx.x; c < n; c += blockDim.x) {
      double d = 0.0;
      for (int i = k + 1; i < n; ++i) d += v[i] * G[i + int64_t(c) * ldg];
      d *= tau;
      for (int i = k + 1; i < n; ++i) G[i + int64_t(c) * ldg] -= d * v[i];
    }
    __syncthreads();
    // G <- G (I - tau v v^T) : all rows;  Q <- Q (I - tau v v^T)
    for (int row = threadIdx.x; row < 2 * n; row += blockDim.x) {
      double *M = row < n ? G : Q;
      const int ldm = row < n ? ldg : ldq;
      const int i = row < n ? row : row - n;
      double d = 0.0;
      for (int c = k + 1; c < n; ++c) d += M[i + int64_t(c) * ldm] * v[c];
      d *= tau;
      for (int c = k + 1; c < n; ++c) M[i + int64_t(c) * ldm] -= d * v[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      G[(k + 1) + int64_t(k) * ldg] = beta;
      for (int i = k + 2; i < n; ++i) G[i + int64_t(k) * ldg] = 0.0;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------ QR iteration
// Eigenvalues of the upper Hessenberg Hs (n x n) by the Francis double-shift QR iteration with
// deflation.  The sequential core follows the published routine hqr of Martin, Peters and
// Wilkinson ("The QR algorithm for real Hessenberg matrices", Numer. Math. 14 (1970) 219-231;
// Handbook for Automatic Computation vol. II, contribution II/14; EISPACK hqr): the negligible-
// subdiagonal search, the exceptional shifts after 10 and 20 iterations without deflation
// (0.75 s and -0.4375 s^2), the search for two small consecutive subdiagonals and the bulge-
// chasing sweep with its p, q, r, x, y, z, w quantities (Golub & Van Loan, Sec. 7.5, give the
// same method).  Works in place on a copy A.  A conjugate pair is stored +Im first.
//
// Layout: the band |j - i| <= 3 (every entry the bulge chase reads, 7 n doubles) lives in shared
// memory; the rest of A in shared memory when n^2 fits the smem_elems doubles offered, else in
// global memory.  Sweep step k applies reflector k to rows k..k+2 (columns k..nn) and then to
// columns k..k+2 (rows l..k+3).  Warp 0 takes the corner, rows/columns k..k+3 (all band
// entries): lanes 0-3 the row update of columns k..k+3, then the column update of rows k..k+3,
// and lane 0 forms reflector k+1 from column k; the other warps apply reflector k to rows k..k+2
// of columns k+4..nn and to columns k..k+2 of rows l..k-1, a fixed thread per column and per
// row.  Those entries are never read by the chase within the sweep, so one CTA barrier per step
// suffices, and every entry receives the same updates in the same order as the sequential sweep.
__global__ void hqr_kernel(double *Ag, int lda, const int *isc_in, double *wr, double *wi, int *isc,
                           int smem_elems) {
  const int n = isc_in[ISC_R];
  if (!isc_in[ISC_QR] && !isc_in[ISC_RES]) return;
  extern __shared__ double sh[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int T1 = blockDim.x - 32;  // threads outside warp 0
  double *a = Ag;
  int ld = lda;
  double *band = sh + smem_elems;  // entry (i, j), |j - i| <= 3, at band[7 i + j - i + 3]
  if (int64_t(n) * n <= int64_t(smem_elems)) {
    a = sh;
    ld = n;
    for (int64_t e = tid; e < int64_t(n) * n; e += blockDim.x) {
      const int i = int(e % n), c = int(e / n);
      a[i + int64_t(c) * n] = Ag[i + int64_t(c) * lda];
    }
  }
  for (int e = tid; e < 7 * n; e += blockDim.x) {
    const int i = e / 7, j = i + e % 7 - 3;
    band[e] = (j >= 0 && j < n) ? Ag[i + int64_t(j) * lda] : 0.0;
  }
#define AA(i, j) (*((((j) - (i)) <= 3 && ((i) - (j)) <= 3) ? &band[7 * (i) + (j) - (i) + 3] : &a[(i) + int64_t(j) * ld]))
  __shared__ double red[32];
  __shared__ int ired[32];
  __shared__ double sp, sq, sx, st_, sw, sanorm;
  __shared__ int snn, sits, sskip, sfail;
  __shared__ double rfl[2][5];  // reflector of step k in slot k & 1: x, y, z, q, r
  __shared__ int rskip[2];
  __syncthreads();
  double an = 0.0;
  for (int64_t e = tid; e < int64_t(n) * n; e += blockDim.x) {
    const int i = int(e % n), c = int(e / n);
    if (i <= c + 1) an += fabs(AA(i, c));
  }
  an = block_sum(an, red);
  if (tid == 0) {
    sanorm = an;
    snn = n - 1;
    st_ = 0.0;
    sits = 0;
    sfail = 0;
  }
  __syncthreads();
  const double eps = 2.220446049250313e-16;
  // Reflector of step k from (p, q, r) (the first step m gets them already scaled); records it in
  // slot k & 1 and writes A(k, k-1).  Lane 0 of warp 0 only.  Past the first step (p, q, r) are
  // scaled by the power of two x nearest below max(|p|, |q|, |r|), which is exact: on GB300 a
  // dependent FP64 operation takes about 64 cycles and a division about 420, and the reflector is
  // the chase's critical path, so the division by |p| + |q| + |r| of the sequential routine is
  // replaced; the reflector (p/s, q/s, r/s, q/p, r/p) does not depend on the scale.
  auto reflector = [&](int k, int m, int l, double p, double q, double r, double x) {
    bool go = true;
    if (k != m) {
      const double mx = fmax(fabs(p), fmax(fabs(q), fabs(r)));
      const long long eb = (__double_as_longlong(mx) >> 52) & 0x7ff;  // biased exponent of mx
      if (mx != 0.0 && eb != 0 && eb < 2046) {
        x = __longlong_as_double(eb << 52);                        // 2^(e), e the exponent of mx
        const double ix = __longlong_as_double((2046 - eb) << 52);  // 2^(-e)
        p *= ix;
        q *= ix;
        r *= ix;
      } else if (mx != 0.0) {  // subnormal or near-overflow maximum: the division as in hqr
        x = fabs(p) + fabs(q) + fabs(r);
        const double ix = 1.0 / x;
        p *= ix;
        q *= ix;
        r *= ix;
      } else {
        go = false;
      }
    }
    double s = 0.0;
    if (go) {
      s = copysign(sqrt(p * p + q * q + r * r), p);
      if (s == 0.0) go = false;
    }
    const int b = k & 1;
    if (go) {
      if (k == m) {
        if (l != m) AA(k, k - 1) = -AA(k, k - 1);
      } else {
        AA(k, k - 1) = -s * x;
      }
      p += s;
      const double is = 1.0 / s, ip = 1.0 / p;
      rfl[b][0] = p * is;
      rfl[b][1] = q * is;
      rfl[b][2] = r * is;
      rfl[b][3] = q * ip;
      rfl[b][4] = r * ip;
      rskip[b] = 0;
    } else {
      rskip[b] = 1;
    }
  };
  while (true) {
    const int nn = snn;
    if (nn < 0 || sfail) break;
    // largest l in [1, nn] whose subdiagonal is negligible (0 if none)
    int cand = 0;
    for (int l = 1 + tid; l <= nn; l += blockDim.x) {
      double s = fabs(AA(l - 1, l - 1)) + fabs(AA(l, l));
      if (s == 0.0) s = sanorm;
      if (fabs(AA(l, l - 1)) <= eps * s) cand = max(cand, l);
    }
    const int l = block_max_int(cand, ired);
    if (tid == 0 && l > 0) AA(l, l - 1) = 0.0;
    __syncthreads();
    if (l == nn) {
      if (tid == 0) {
        wr[nn] = AA(nn, nn) + st_;
        wi[nn] = 0.0;
        snn = nn - 1;
        sits = 0;
      }
      __syncthreads();
      continue;
    }
    if (l == nn - 1) {
      if (tid == 0) {
        const double y = AA(nn - 1, nn - 1), x = AA(nn, nn) + st_;
        const double w = AA(nn, nn - 1) * AA(nn - 1, nn);
        const double p = 0.5 * (y - AA(nn, nn));
        const double q = p * p + w;
        double z = sqrt(fabs(q));
        if (q >= 0.0) {
          z = p + copysign(z, p);
          wr[nn - 1] = wr[nn] = x + z;
          if (z != 0.0) wr[nn] = x - w / z;
          wi[nn - 1] = wi[nn] = 0.0;
        } else {
          wr[nn - 1] = wr[nn] = x + p;
          wi[nn - 1] = z;
          wi[nn] = -z;
        }
        snn = nn - 2;
        sits = 0;
      }
      __syncthreads();
      continue;
    }
    if (sits >= 60) {
      if (tid == 0) sfail = 1;
      __syncthreads();
      break;
    }
    // shifts
    if (tid == 0) {
      double x = AA(nn, nn), y = AA(nn - 1, nn - 1), w = AA(nn, nn - 1) * AA(nn - 1, nn);
      if (sits == 10 || sits == 20) {
        st_ += x;
        sx = x;
        const double s = fabs(AA(nn, nn - 1)) + fabs(AA(nn - 1, nn - 2));
        x = y = 0.75 * s;
        w = -0.4375 * s * s;
        sskip = 1;  // diagonal shift pending
      } else {
        sskip = 0;
      }
      sp = x;  // keep x, y, w
      sq = y;
      sw = w;
      sits = sits + 1;
    }
    __syncthreads();
    if (sskip) {
      const double xs = sx;
      for (int i = tid; i <= nn; i += blockDim.x) AA(i, i) -= xs;
      __syncthreads();
    }
    const double X = sp, Y = sq, W = sw;
    // largest m in [l, nn-2] where two consecutive subdiagonals are small (or m = l)
    int mc = l;
    for (int m = l + 1 + tid; m <= nn - 2; m += blockDim.x) {
      const double z = AA(m, m);
      const double r = X - z, s = Y - z;
      double p = (r * s - W) / AA(m + 1, m) + AA(m, m + 1);
      double q = AA(m + 1, m + 1) - z - r - s;
      double rr = AA(m + 2, m + 1);
      const double sc = fabs(p) + fabs(q) + fabs(rr);
      p /= sc;
      q /= sc;
      rr /= sc;
      const double u = fabs(AA(m, m - 1)) * (fabs(q) + fabs(rr));
      const double v = fabs(p) * (fabs(AA(m - 1, m - 1)) + fabs(z) + fabs(AA(m + 1, m + 1)));
      if (u <= eps * v) mc = max(mc, m);
    }
    const int m = block_max_int(mc, ired);
    for (int i = m + 2 + tid; i <= nn; i += blockDim.x) {
      AA(i, i - 2) = 0.0;
      if (i != m + 2) AA(i, i - 3) = 0.0;
    }
    __syncthreads();
    if (tid == 0) {
      const double z = AA(m, m);
      const double r = X - z, s = Y - z;
      double p = (r * s - W) / AA(m + 1, m) + AA(m, m + 1);
      double q = AA(m + 1, m + 1) - z - r - s;
      double rr = AA(m + 2, m + 1);
      const double sc = fabs(p) + fabs(q) + fabs(rr);
      reflector(m, m, l, p / sc, q / sc, rr / sc, 0.0);
    }
    __syncthreads();
    // double-shift QR sweep on rows/columns l..nn, starting at m; one barrier per step
    for (int k = m; k <= nn - 1; ++k) {
      const int b = k & 1;
      const bool three = (k != nn - 1);
      const bool skip = rskip[b] != 0;
      const double x = rfl[b][0], y = rfl[b][1], z = rfl[b][2], q = rfl[b][3], r = rfl[b][4];
      if (tid < 32) {
        // ---- warp 0: the corner, then the next reflector
        double fw = 0.0;  // lane 1 + i: row k + 1 + i of column k after the step
        if (!skip) {
          const int jj = k + lane;
          if (lane < 4 && jj <= nn) {
            double p = AA(k, jj) + q * AA(k + 1, jj);
            if (three) {
              p += r * AA(k + 2, jj);
              AA(k + 2, jj) -= p * z;
            }
            AA(k + 1, jj) -= p * y;
            AA(k, jj) -= p * x;
          }
          __syncwarp();
          const int i = k + lane;
          if (lane < 4 && i <= nn && i <= k + 3) {
            double p = x * AA(i, k) + y * AA(i, k + 1);
            if (three) {
              p += z * AA(i, k + 2);
              AA(i, k + 2) -= p * r;
            }
            AA(i, k + 1) -= p * q;
            const double aik = AA(i, k) - p;
            AA(i, k) = aik;
            fw = aik;
          }
        } else {
          const int i = k + lane;
          if (lane >= 1 && lane < 4 && i <= nn) fw = AA(i, k);
        }
        const double f0 = __shfl_sync(0xffffffffu, fw, 1);
        const double f1 = __shfl_sync(0xffffffffu, fw, 2);
        const double f2 = __shfl_sync(0xffffffffu, fw, 3);
        if (lane == 0 && k + 1 <= nn - 1) reflector(k + 1, m, l, f0, f1, (k + 1 != nn - 1) ? f2 : 0.0, 0.0);
      } else if (!skip) {
        // ---- the other warps: columns k+4..nn (rows k..k+2) and rows l..k-1 (columns k..k+2),
        // at most two of each a thread (n <= 512 < 2 T1); every load issued before any update,
        // so the step waits for one memory round trip
        const int t1 = tid - 32;
        const int j0 = k + 4 + ((t1 - (k + 4)) % T1 + T1) % T1, j1 = j0 + T1;
        const int i0 = l + ((t1 - l) % T1 + T1) % T1, i1 = i0 + T1;
        const bool hj0 = j0 <= nn, hj1 = j1 <= nn, hi0 = i0 <= k - 1, hi1 = i1 <= k - 1;
        double c0[3] = {0.0, 0.0, 0.0}, c1[3] = {0.0, 0.0, 0.0}, r0[3] = {0.0, 0.0, 0.0}, r1[3] = {0.0, 0.0, 0.0};
        if (hj0) {
          c0[0] = AA(k, j0), c0[1] = AA(k + 1, j0);
          if (three) c0[2] = AA(k + 2, j0);
        }
        if (hj1) {
          c1[0] = AA(k, j1), c1[1] = AA(k + 1, j1);
          if (three) c1[2] = AA(k + 2, j1);
        }
        if (hi0) {
          r0[0] = AA(i0, k), r0[1] = AA(i0, k + 1);
          if (three) r0[2] = AA(i0, k + 2);
        }
        if (hi1) {
          r1[0] = AA(i1, k), r1[1] = AA(i1, k + 1);
          if (three) r1[2] = AA(i1, k + 2);
        }
        auto rowupd = [&](double (&v)[3], int jj) {
          double p = v[0] + q * v[1];
          if (three) {
            p += r * v[2];
            AA(k + 2, jj) = v[2] - p * z;
          }
          AA(k + 1, jj) = v[1] - p * y;
          AA(k, jj) = v[0] - p * x;
        };
        auto colupd = [&](double (&v)[3], int i) {
          double p = x * v[0] + y * v[1];
          if (three) {
            p += z * v[2];
            AA(i, k + 2) = v[2] - p * r;
          }
          AA(i, k + 1) = v[1] - p * q;
          AA(i, k) = v[0] - p;
        };
        if (hj0) rowupd(c0, j0);
        if (hj1) rowupd(c1, j1);
        if (hi0) colupd(r0, i0);
        if (hi1) colupd(r1, i1);
      }
      __syncthreads();
    }
  }
  if (tid == 0) isc[ISC_STATUS] = sfail ? FOA_DMD_ENOCONV : FOA_DMD_OK;
#undef AA
}

// ------------------------------------------------------------------------------ ordering
// key_i = |c_i| (a conjugate pair takes the larger of its two), order by key desc, |lambda| desc,
// Im desc, index asc.  Writes the sorted eigenvalues, indicators, amplitudes and y columns.
__global__ void order_kernel(EigArgs e, int nsel) {
  const int r = e.isc[ISC_R];
  const int m = e.m;
  extern __shared__ double sh[];
  double *key = sh, *lab = sh + r;
  int *pos = reinterpret_cast<int *>(sh + 2 * r);
  // |c| and |lambda| are not negative: their bits compare as integers (the FP64 pipe takes 64 cycles)
  const long long *ki = reinterpret_cast<const long long *>(key), *li = reinterpret_cast<const long long *>(lab);
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    double k = hypot(e.amp_re[i], e.amp_im[i]);
    if (e.wi[i] > 0.0 && i + 1 < r) k = fmax(k, hypot(e.amp_re[i + 1], e.amp_im[i + 1]));
    if (e.wi[i] < 0.0 && i > 0) k = fmax(k, hypot(e.amp_re[i - 1], e.amp_im[i - 1]));
    key[i] = k;
    lab[i] = hypot(e.wr[i], e.wi[i]);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    int rank = 0;
    for (int k = 0; k < r; ++k) {
      bool before;
      if (ki[k] != ki[i]) before = ki[k] > ki[i];
      else if (li[k] != li[i]) before = li[k] > li[i];
      else if (e.wi[k] != e.wi[i]) before = e.wi[k] > e.wi[i];
      else before = k < i;
      rank += before;
    }
    pos[i] = rank;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < r; i += blockDim.x) {
    const int p = pos[i];
    e.out[OUT_LRE * e.ld + p] = e.wr[i];
    e.out[OUT_LIM * e.ld + p] = e.wi[i];
    e.out[OUT_IND * e.ld + p] = e.ind[i];
    e.out[OUT_ARE * e.ld + p] = e.amp_re[i];
    e.out[OUT_AIM * e.ld + p] = e.amp_im[i];
    e.perm[p] = i;
  }
  __syncthreads();
  // sorted y columns 0..min(nsel, r)-1 (perm has r entries)
  for (int64_t t = threadIdx.x; t < int64_t(min(nsel, r)) * m; t += blockDim.x) {
    const int c = int(t / m), i = int(t % m);
    const int src = e.perm[c];
    e.ysr[i + int64_t(c) * e.ld] = e.yr[i + int64_t(src) * e.ld];
    e.ysi[i + int64_t(c) * e.ld] = e.yi[i + int64_t(src) * e.ld];
  }
}

}  // namespace foa
