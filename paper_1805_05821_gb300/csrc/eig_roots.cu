// Eigenvalues of the projected matrix by simultaneous iteration (Ehrlich-Aberth) on Hyman's form of
// the characteristic polynomial.
//
//   roots_setup_kernel   norms, traces, the start circle, and whether the iteration applies
//   roots_step_kernel    one step of all eigenvalues: one CTA each
//   roots_finish_kernel  conjugate pairs, checks, hand-over to the QR iteration where one fails
//
// For an upper Hessenberg H with nonzero subdiagonals, x_{n-1} = 1 and rows n-1 .. 1 of (H - z) x = 0
// give x_{n-2} .. x_0 by back substitution with the subdiagonal as divisor, and row 0 leaves
// p(z) = det(H - z) up to a constant factor (Hyman 1957; Wilkinson, The Algebraic Eigenvalue Problem,
// ch. 7 par. 11: the value is that of a matrix with small relative changes of its entries).  The
// derivative follows from the same recurrence, and all eigenvalues are improved together by
//   z_i <- z_i - N_i / (1 - N_i sum_{j != i} 1 / (z_i - z_j)),   N = p / p'
// (Ehrlich 1967; Aberth, Math. Comp. 27 (1973) 339-344), each from the values of the step before, so
// the result does not depend on the order in which CTAs run.  They start on a circle around the mean
// eigenvalue tr(H) / n whose radius is the geometric mean of |lambda - tr(H)/n|, from the determinant:
// the Ritz values of a flow's snapshots lie near such a circle, and it takes 4 to 13 steps, 4.0 to 6.5
// evaluations per eigenvalue (dense random matrices: 30 steps, 16 evaluations).
//
// Why not the QR iteration: its chain of about 0.75 n^2 dependent 3 x 3 reflectors runs on one SM at
// the latency of GB300's FP64 pipe (64 cycles an operation).  Here every eigenvalue is independent
// within a step, so the work, 2 n^2 FP64 FMAs an evaluation, spreads over all SMs and is bound by
// their FP64 rate (2 FMAs a clock and SM).  At n = 255 the eigenvalues took 103 ms and take 3.9 ms; at
// n = 96 13.5 and 0.5 ms.  Spectra that the iteration does not resolve (multiple
// eigenvalues, long real intervals) and matrices with negligible subdiagonals go to hqr_kernel.
#include "api_internal.cuh"
#include "eig_internal.cuh"

namespace foa {

constexpr int kRootThreads = 128;  // four lanes per row: Re x, Im x, Re x', Im x' of Hyman's recurrence
constexpr double kEps = 2.220446049250313e-16;

__device__ __forceinline__ double block_sum_n(double v, double *red, int nthreads) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  named_bar_sync(1, nthreads);
  if (l == 0) red[w] = v;
  named_bar_sync(1, nthreads);
  double t = 0.0;
  for (int i = 0; i < (nthreads >> 5); ++i) t += red[i];
  named_bar_sync(1, nthreads);
  return t;
}

struct HymanShared {
  double x[2][4];   // Re x_i, Im x_i, Re x'_i, Im x'_i of the current row, double-buffered
  double scale[2];  // power of two applied to that row (and to every running sum)
};

// Hyman's recurrence for the n x n Hessenberg H (column-major, ld) at z, on kRootThreads threads.
// Thread 4 r + c carries component c of the running sums of rows r, r + 32, ..: row i needs
// sum_{k > i} h_ik x_k when its turn comes.  Column k of H is loaded one row ahead of its use.
// On return s.x[*out] holds (p, p') up to a common factor; the return value is the base-2 exponent
// of the factors applied (for the determinant).
template <int NB>
__device__ __forceinline__ int hyman(const double *__restrict__ H, int ld, int n, const double *__restrict__ invsub,
                                     double zr, double zi, HymanShared &s, int *out) {
  const int tid = threadIdx.x, comp = tid & 3, slot = tid >> 2;
  double acc[NB], h[NB];
  const double zo = (comp & 1) ? -zi : zi;  // (h_ii - z) x: the shift's imaginary part times the partner component
  int e2 = 0, buf = 0;
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    acc[u] = 0.0;
    const int r = slot + 32 * u;
    h[u] = r < n ? __ldg(H + r + int64_t(n - 1) * ld) : 0.0;
  }
  if (tid < 4) s.x[0][tid] = tid == 0 ? 1.0 : 0.0;
  if (tid == 0) s.scale[0] = 1.0;
  named_bar_sync(1, kRootThreads);
#pragma unroll
  for (int ub = NB - 1; ub >= 0; --ub) {
    for (int ii = min(31, n - 1 - 32 * ub); ii >= 0; --ii) {
      const int i = 32 * ub + ii;
      const double own = s.x[buf][comp], other = s.x[buf][comp ^ 1], base = s.x[buf][comp & 1];
      const double sc = s.scale[buf];
      double hn[NB];  // column i-1
#pragma unroll
      for (int u = 0; u <= ub; ++u) {
        const int r = slot + 32 * u;
        hn[u] = (i > 0 && r < i) ? __ldg(H + r + int64_t(i - 1) * ld) : 0.0;
      }
      if (sc != 1.0) {
#pragma unroll
        for (int u = 0; u <= ub; ++u) acc[u] *= sc;
        e2 += sc < 1.0 ? 300 : -200;
      }
      if ((ii >> 3) == (tid >> 5)) {  // the warp that owns row i closes it
        double v = fma(h[ub] - zr, own, acc[ub]);
        v = fma(zo, other, v);
        if (comp >= 2) v -= base;
        const double nx = i > 0 ? v * __ldg(invsub + i) : v;
        // keep |x|, |x'| within 2^+-300: the running sums stay far inside the range of a double
        int ex = (__double2hiint(nx) >> 20) & 0x7ff;
        ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 1));
        ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, 2));
        const double f = i == 0 ? 1.0 : ex > 1023 + 300 ? 0x1p-300 : (ex < 1023 - 300 && ex > 0) ? 0x1p+200 : 1.0;
        if (slot == ii) {
          s.x[buf ^ 1][comp] = nx * f;
          if (comp == 0) s.scale[buf ^ 1] = f;
        }
      }
#pragma unroll
      for (int u = 0; u < ub; ++u) acc[u] = fma(h[u], own, acc[u]);
      if (slot < ii) acc[ub] = fma(h[ub], own, acc[ub]);
#pragma unroll
      for (int u = 0; u <= ub; ++u) h[u] = hn[u];
      named_bar_sync(1, kRootThreads);
      buf ^= 1;
    }
  }
  *out = buf;
  return e2;
}

__device__ __forceinline__ int hyman_any(const double *H, int ld, int n, const double *invsub, double zr, double zi,
                                         HymanShared &s, int *out) {
  if (n <= 64) return hyman<2>(H, ld, n, invsub, zr, zi, s, out);
  if (n <= 128) return hyman<4>(H, ld, n, invsub, zr, zi, s, out);
  if (n <= 256) return hyman<8>(H, ld, n, invsub, zr, zi, s, out);
  if (n <= 384) return hyman<12>(H, ld, n, invsub, zr, zi, s, out);
  return hyman<16>(H, ld, n, invsub, zr, zi, s, out);
}

// One CTA.  scal: [0] sum |h_ij| over the Hessenberg part (also the pivot floor of the inverse
// iteration), [1] tr H, [2] tr H^2, [3] ||H - tr(H)/n||_F / sqrt(n); z[0] gets the start circle.
__global__ void __launch_bounds__(512) roots_setup_kernel(RootArgs a) {
  const int n = a.isc[ISC_R];
  const int tid = threadIdx.x;
  __shared__ double red[32];
  __shared__ int bad;
  __shared__ HymanShared hs;
  __shared__ double s_rad;
  if (tid == 0) bad = (n < a.min_n) ? 1 : 0;
  for (int k = tid; k < kRootSteps; k += 512) a.left[k] = 0;
  __syncthreads();
  double an = 0.0, fr = 0.0, t1 = 0.0, t2 = 0.0, mx = 0.0, ls = 0.0;
  for (int c = tid >> 5; c < n; c += 16)  // a warp per column
    for (int i = tid & 31; i <= min(c + 1, n - 1); i += 32) {
      const double v = fabs(a.H[i + int64_t(c) * a.ld]);
      an += v;
      fr = fma(v, v, fr);
      mx = fmax(mx, v);
    }
  for (int i = tid; i < n; i += 512) {
    const double d = a.H[i + int64_t(i) * a.ld];
    t1 += d;
    t2 = fma(d, d, t2);
    if (i > 0) {
      const double sub = a.H[i + int64_t(i - 1) * a.ld], up = a.H[i - 1 + int64_t(i) * a.ld];
      const double s = fabs(a.H[i - 1 + int64_t(i - 1) * a.ld]) + fabs(d);
      t2 = fma(2.0 * sub, up, t2);
      a.invsub[i] = -1.0 / sub;
      // a negligible subdiagonal (the QR iteration's test) splits the matrix: left to that iteration
      if (!(fabs(sub) > kEps * s)) bad = 1;
      ls += log2(fabs(sub));
    }
  }
  named_bar_sync(1, 512);
  an = block_sum_n(an, red, 512);
  fr = block_sum_n(fr, red, 512);
  t1 = block_sum_n(t1, red, 512);
  t2 = block_sum_n(t2, red, 512);
  ls = block_sum_n(ls, red, 512);
  for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) red[tid >> 5] = mx;
  __syncthreads();
  mx = red[0];
  for (int w = 1; w < 16; ++w) mx = fmax(mx, red[w]);
  // recurrence growth is bounded where every divisor is within 2^60 of the largest entry
  for (int i = 1 + tid; i < n; i += 512)
    if (!(fabs(a.H[i + int64_t(i - 1) * a.ld]) > 0x1p-60 * mx)) bad = 1;
  if (tid == 0 && !(mx > 0x1p-200 && mx < 0x1p+200)) bad = 1;
  __syncthreads();
  const double c = t1 / n;
  const double fro = sqrt(fmax(0.0, fr - t1 * c) / n);
  if (tid == 0) {
    a.scal[0] = an;
    a.scal[1] = t1;
    a.scal[2] = t2;
    a.scal[3] = fro;
    a.isc[ISC_QR] = bad;
  }
  if (bad) return;
  if (tid < kRootThreads) {
    int b;
    const int e2 = hyman_any(a.H, a.ld, n, a.invsub, c, 0.0, hs, &b);
    if (tid == 0) {
      const double v = fabs(hs.x[b][0]);
      double rad = v > 0.0 ? exp2((log2(v) + double(e2) + ls) / n) : 0.0;
      s_rad = fmin(fmax(rad, 1e-2 * fro), fro);
    }
  }
  __syncthreads();
  for (int i = tid; i < n; i += 512) {
    double sn, cs;
    sincospi(2.0 * (i + 0.35) / n, &sn, &cs);
    a.zr[i] = fma(s_rad, cs, c);
    a.zi[i] = s_rad * sn;
    a.dold[i] = 1e300;
    a.conv[i] = 0;
  }
}

// Step `it`: CTA i improves eigenvalue i from the values in buffer it & 1 into the other one.
__global__ void __launch_bounds__(kRootThreads) roots_step_kernel(RootArgs a, int it) {
  const int n = a.isc[ISC_R], i = blockIdx.x;
  if (i >= n || a.isc[ISC_QR] || (it > 0 && a.left[it - 1] == 0)) return;
  const int tid = threadIdx.x, K = a.ld;
  const double *zri = a.zr + (it & 1) * K, *zii = a.zi + (it & 1) * K;
  double *zro = a.zr + ((it & 1) ^ 1) * K, *zio = a.zi + ((it & 1) ^ 1) * K;
  const double zr = zri[i], zi = zii[i];
  if (a.conv[i]) {
    if (tid == 0) {
      zro[i] = zr;
      zio[i] = zi;
    }
    return;
  }
  __shared__ HymanShared hs;
  __shared__ double red[kRootThreads / 32];
  double sr = 0.0, si = 0.0;
  for (int j = tid; j < n; j += kRootThreads)
    if (j != i) {
      const double dr = zr - zri[j], di = zi - zii[j];
      const double q = 1.0 / fma(dr, dr, di * di);
      sr = fma(dr, q, sr);
      si = fma(-di, q, si);
    }
  int b;
  hyman_any(a.H, K, n, a.invsub, zr, zi, hs, &b);
  sr = block_sum_n(sr, red, kRootThreads);
  si = block_sum_n(si, red, kRootThreads);
  if (tid == 0) {
    // d = p / (p' - p S)
    const double pr = hs.x[b][0], pi = hs.x[b][1];
    const double qr = hs.x[b][2] - (pr * sr - pi * si), qi = hs.x[b][3] - (pr * si + pi * sr);
    double dr, di;
    if (fabs(qr) >= fabs(qi)) {  // Smith's division
      const double t = qi / qr, d = fma(qi, t, qr);
      dr = fma(pi, t, pr) / d;
      di = fma(-pr, t, pi) / d;
    } else {
      const double t = qr / qi, d = fma(qr, t, qi);
      dr = fma(pr, t, pi) / d;
      di = fma(pi, t, -pr) / d;
    }
    const bool fin = isfinite(dr) && isfinite(di);
    if (!fin) dr = di = 0.0;
    zro[i] = zr - dr;
    zio[i] = zi - di;
    // The correction shrinks at least quadratically: below 1e-12 the value after it is as near as the
    // arithmetic allows.  An ill-conditioned eigenvalue's corrections stop shrinking at its own
    // rounding level, above that.
    const double ad = hypot(dr, di), scl = hypot(zr, zi) + 1e-3 * a.scal[3];
    const bool done = fin && (ad <= 1e-12 * scl || (ad < 1e-7 * scl && ad > 0.5 * a.dold[i]));
    a.dold[i] = ad;
    if (done) a.conv[i] = 1;
    else atomicAdd(&a.left[it], 1);
  }
}

// Pair the values, check them, and store them as the QR iteration does (a conjugate pair side by
// side, +Im first).  They stand if all converged, each value's nearest conjugate has that value as
// its own nearest one (a real eigenvalue is its own), and both traces agree: a value found twice in
// place of another one would change them.  Otherwise isc[ISC_QR] asks for the QR iteration.
__global__ void __launch_bounds__(512) roots_finish_kernel(RootArgs a) {
  const int n = a.isc[ISC_R], tid = threadIdx.x, K = a.ld;
  if (a.isc[ISC_QR]) return;
  __shared__ double zr[kMaxK], zi[kMaxK], red[32];
  __shared__ short part[kMaxK];
  __shared__ int bad, last;
  if (tid == 0) {
    bad = 0;
    last = -1;
    for (int k = 0; k < kRootSteps; ++k)
      if (a.left[k] == 0) {
        last = k;
        break;
      }
    a.isc[ISC_ITS] = last + 1;
  }
  __syncthreads();
  if (last < 0) {
    if (tid == 0) a.isc[ISC_QR] = 1;
    return;
  }
  const int buf = (last & 1) ^ 1;
  double t1 = 0.0, t2 = 0.0;
  for (int i = tid; i < n; i += 512) {
    zr[i] = a.zr[buf * K + i];
    zi[i] = a.zi[buf * K + i];
    t1 += zr[i];
    t2 += zr[i] * zr[i] - zi[i] * zi[i];
  }
  named_bar_sync(1, 512);
  t1 = block_sum_n(t1, red, 512);
  t2 = block_sum_n(t2, red, 512);
  const double nf = a.scal[3] * sqrt(double(n)) + fabs(a.scal[1]) / n;  // about ||H||_F
  if (tid == 0 && (!(fabs(t1 - a.scal[1]) <= 1e-11 * nf * n) || !(fabs(t2 - a.scal[2]) <= 1e-11 * nf * nf * n))) bad = 1;
  for (int i = tid; i < n; i += 512) {
    double best = 1e300;
    int arg = i;
    for (int j = 0; j < n; ++j) {
      const double dr = zr[j] - zr[i], di = zi[j] + zi[i];
      const double d = fma(dr, dr, di * di);
      if (d < best) {
        best = d;
        arg = j;
      }
    }
    part[i] = short(arg);
  }
  __syncthreads();
  for (int i = tid; i < n; i += 512)
    if (part[part[i]] != i ||
        (part[i] == i ? fabs(zi[i]) > 1e-8 * (fabs(zr[i]) + 1e-3 * a.scal[3]) : !(zi[i] * zi[part[i]] < 0.0)))
      bad = 1;
  __syncthreads();
  if (bad) {
    if (tid == 0) a.isc[ISC_QR] = 1;
    return;
  }
  // position: pairs and real values in the order of their first index
  for (int i = tid; i < n; i += 512) {
    const int p = part[i], lead = min(i, p);
    int pos = 0;
    for (int j = 0; j < lead; ++j) pos += (part[j] >= j) ? (part[j] > j ? 2 : 1) : 0;
    if (p == i) {
      a.wr[pos] = zr[i];
      a.wi[pos] = 0.0;
    } else if (zi[i] > 0.0) {
      const double re = 0.5 * (zr[i] + zr[p]), im = 0.5 * (zi[i] - zi[p]);
      a.wr[pos] = a.wr[pos + 1] = re;
      a.wi[pos] = im;
      a.wi[pos + 1] = -im;
    }
  }
  if (tid == 0) a.isc[ISC_STATUS] = FOA_DMD_OK;
}

cudaError_t launch_roots(const RootArgs &a, int m, cudaStream_t s) {
  roots_setup_kernel<<<1, 512, 0, s>>>(a);
  if (m >= a.min_n) {
    for (int it = 0; it < kRootSteps; ++it) roots_step_kernel<<<m, kRootThreads, 0, s>>>(a, it);
    roots_finish_kernel<<<1, 512, 0, s>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace foa
