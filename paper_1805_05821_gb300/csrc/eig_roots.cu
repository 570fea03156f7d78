// Eigenvalues of the projected matrix by simultaneous iteration (Ehrlich-Aberth) on Hyman's form of
// the characteristic polynomial.
//
//   roots_setup_kernel   norms, traces, and whether the iteration applies
//   roots_start_kernel   the start circle
//   roots_step32_kernel  one step of all eigenvalues in FP32, one CTA each
//   roots_step_kernel    the same in FP64
//   roots_pair_kernel    each value's nearest conjugate
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
// evaluations per eigenvalue (dense random matrices 7 steps at order 10, 15 at 48 and 30, FP32 ones included, at
// 200).
//
// Why not the QR iteration: its chain of about 0.75 n^2 dependent 3 x 3 reflectors runs on one SM at
// the latency of GB300's FP64 pipe (64 cycles an operation).  Here every eigenvalue is independent
// within a step, so the work, 2 n^2 FP64 FMAs an evaluation, spreads over all SMs and is bound by
// their FP64 rate (2 FMAs a clock and SM) or, where there are few, by the recurrence's latency.  The
// eigenvalues of n = 255 took 103 ms and take 1.7 ms, of n = 96 13.5 and 0.6 ms (14 steps in FP32 at
// 57 us, four to eight in FP64 at 131 us; FP64 alone 2.1 ms).  Spectra that the iteration does not resolve (multiple
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

__device__ __forceinline__ float nan_of(float) { return __int_as_float(0x7fc00000); }
__device__ __forceinline__ double nan_of(double) { return __longlong_as_double(0x7ff8000000000000ll); }

template <typename T> struct HymanShared {
  T x[4][8][4];  // of the last four groups of 8 rows: Re x_i, Im x_i, Re x'_i, Im x'_i
  T next[4][4];  // the same of the row below each group (p, p' after the last one)
  T scale[4];    // power of two applied within the group
};

// Biased exponent, and the limits between which |x|, |x'| are kept (a power of two is applied to them
// and to the running sums outside): after 4 rows of a double's recurrence, or one of a float's, sums
// and values are still far inside the type's range for the divisors that roots_setup_kernel lets pass.
template <typename T> struct Range;
template <> struct Range<double> {
  static constexpr int kBias = 1023, kHi = 1023 + 300, kLo = 1023 - 300, kEvery = 4;
  static __device__ __forceinline__ int ex(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
  static __device__ __forceinline__ double down() { return 0x1p-300; }
  static __device__ __forceinline__ double up() { return 0x1p+200; }
};
template <> struct Range<float> {
  static constexpr int kBias = 127, kHi = 127 + 30, kLo = 127 - 30, kEvery = 1;
  static __device__ __forceinline__ int ex(float v) { return (__float_as_int(v) >> 23) & 0xff; }
  static __device__ __forceinline__ float down() { return 0x1p-40f; }
  static __device__ __forceinline__ float up() { return 0x1p+30f; }
};

// Hyman's recurrence for the n x n Hessenberg H (column-major, ld) at z, on kRootThreads threads.
// Thread 4 r + c carries component c of the running sums of rows r, r + 32, ..: row i needs
// sum_{k > i} h_ik x_k when its turn comes, so warp w owns rows 8 w .. 8 w + 7 of every 32.
//
// The rows are closed in groups of 8, each by the warp that owns them: within a group x goes from row
// to row by shuffles, and one CTA barrier per group hands the 8 values to the other warps, which add
// them to their rows (8 columns of H at a time) while the next owner, which brings its own 8 rows up to
// date first, closes the next group.  A row costs four dependent operations (64 cycles each in FP64)
// and the shuffles.  (One barrier per row, every warp's additions between two rows: 1650 cycles a row
// in FP64, 200 us for one evaluation at n = 255; by groups 110 us.)
// On return s.next[*out] holds (p, p') up to a common factor; the return value is the base-2 exponent
// of the factors applied (for the determinant).
template <typename T, int NB>
__device__ __forceinline__ int hyman(const T *__restrict__ H, int ld, int n, const T *__restrict__ invsub, T zr, T zi,
                                     HymanShared<T> &s, int *out) {
  using R = Range<T>;
  const int tid = threadIdx.x, comp = tid & 3, slot = tid >> 2, warp = tid >> 5, lane = tid & 31;
  const int row8 = slot & 7;  // row within the warp's group
  T acc[NB], hb[8], hp[8];
  const T zo = (comp & 1) ? -zi : zi;  // (h_ii - z) x: the shift's imaginary part times the partner component
  int e2 = 0, g = 0, pbase = 0;        // groups closed; first row of the last one
#pragma unroll
  for (int u = 0; u < NB; ++u) acc[u] = T(0);
  // columns c0 .. c0+7 of one row
  auto load8 = [&](T (&h)[8], int row, int c0) {
#pragma unroll
    for (int r = 0; r < 8; ++r)
      h[r] = (row >= 0 && row < n && c0 + r < n) ? __ldg(H + row + int64_t(c0 + r) * ld) : T(0);
  };
  auto add8 = [&](T a, const T (&h)[8], int b) {
#pragma unroll
    for (int r = 0; r < 8; ++r) a = fma(h[r], s.x[b][r][comp], a);
    return a;
  };
  // the group with first column c0 (values in buffer b) to row blocks u < ub, one block's entries
  // under way while the block before it is added
  T hn[8];
  auto add_block = [&](int ub, int c0, int b) {
    T h[8];
    load8(h, ub > 0 ? slot : -1, c0);
#pragma unroll
    for (int u = 0; u < NB - 1; ++u) {
      if (u >= ub) break;
      load8(hn, u + 1 < ub ? 32 * (u + 1) + slot : -1, c0);
      acc[u] = add8(acc[u], h, b);
#pragma unroll
      for (int r = 0; r < 8; ++r) h[r] = hn[r];
    }
  };
  const int top = (n - 1) >> 3;  // the first group
  if (warp == (top & 3)) load8(hb, 8 * top + row8, 8 * top);
  if (tid < 32) s.x[0][tid >> 2][tid & 3] = T(0);        // rows past n of the first group
  __syncwarp();
  if (tid < 4) s.next[3][tid] = tid == 0 ? T(1) : T(0);  // x_{n-1} = 1, as if handed on by a group before
  named_bar_sync(1, kRootThreads);
#pragma unroll
  for (int ub = NB - 1; ub >= 0; --ub) {
    for (int w4 = 3; w4 >= 0; --w4) {
      const int base = 32 * ub + 8 * w4;
      if (base >= n) continue;
      const int b = g & 3, pb = (g + 3) & 3;
      const bool owner = warp == w4;
      if (g > 0) {
        const T sc = s.scale[pb];
        if (R::ex(sc) != R::kBias) {
#pragma unroll
          for (int u = 0; u <= ub; ++u) acc[u] *= sc;
          e2 -= R::ex(sc) - R::kBias;
        }
      }
      if (owner) {
        if (g > 0) acc[ub] = add8(acc[ub], hp, pb);
#pragma unroll
        for (int r = 0; r < 8; ++r)
          if (row8 == r) hb[r] -= zr;
        T nx = s.next[pb][comp], own = nx, other = s.next[pb][comp ^ 1], xb = s.next[pb][comp & 1];
        T scale = T(1);
        int ex = 0;
#pragma unroll
        for (int r = 7; r >= 0; --r) {
          const int i = base + r;
          if (i >= n) continue;
          const T is = i > 0 ? __ldg(invsub + i) : T(1);
          if (lane < 4) s.x[b][r][comp] = own;
          // row i is closed by its quad, the rows above it take column i
          if (row8 <= r) acc[ub] = fma(hb[r], own, acc[ub]);
          T v = fma(zo, other, acc[ub]);
          if (comp >= 2) v -= xb;
          nx = v * is;
          ex = max(ex, row8 == r ? R::ex(nx) : 0);
          if (r % R::kEvery == 0) {
            ex = __reduce_max_sync(0xffffffffu, ex);
            if (i > 0 && (ex > R::kHi || (ex < R::kLo && ex > 0))) {
              const T f = ex > R::kHi ? R::down() : R::up();
              nx *= f;
              acc[ub] *= f;
              scale *= f;
              __syncwarp();
              for (int q = r; q < 8; ++q)
                if (lane < 4 && base + q < n) s.x[b][q][comp] *= f;
              // the power applied stays representable however long the group
              if (R::ex(scale) < 8 || R::ex(scale) > 2 * R::kBias - 8) scale = nan_of(T(0));
            }
            ex = 0;
          }
          own = __shfl_sync(0xffffffffu, nx, 4 * r + comp);
          other = __shfl_sync(0xffffffffu, nx, 4 * r + (comp ^ 1));
          xb = __shfl_sync(0xffffffffu, nx, 4 * r + (comp & 1));
        }
        if (lane < 4) s.next[b][comp] = own;
        if (lane == 0) s.scale[b] = scale;
      } else if (g > 0) {
        if (warp < w4) {
          load8(hn, 32 * ub + slot, pbase);
          acc[ub] = add8(acc[ub], hn, pb);
        }
        add_block(ub, pbase, pb);
      }
      // the next owner fetches its 8 rows' entries in this group's columns and in its own
      const int nbase = base - 8;
      if (nbase >= 0 && warp == (w4 + 3) % 4) {
        load8(hp, nbase + row8, base);
        load8(hb, nbase + row8, nbase);
      }
      named_bar_sync(1, kRootThreads);
      if (owner && g > 0) add_block(ub, pbase, pb);
      pbase = base;
      ++g;
    }
  }
  *out = (g + 3) & 3;
  return e2 - (R::ex(s.scale[*out]) - R::kBias);
}

template <typename T>
__device__ __forceinline__ int hyman_any(const T *H, int ld, int n, const T *invsub, T zr, T zi, HymanShared<T> &s,
                                         int *out) {
  if (n <= 64) return hyman<T, 2>(H, ld, n, invsub, zr, zi, s, out);
  if (n <= 128) return hyman<T, 4>(H, ld, n, invsub, zr, zi, s, out);
  if (n <= 256) return hyman<T, 8>(H, ld, n, invsub, zr, zi, s, out);
  if (n <= 384) return hyman<T, 12>(H, ld, n, invsub, zr, zi, s, out);
  return hyman<T, 16>(H, ld, n, invsub, zr, zi, s, out);
}

// One CTA.  scal: [0] sum |h_ij| over the Hessenberg part (also the pivot floor of the inverse
// iteration), [1] tr H, [2] tr H^2, [3] ||H - tr(H)/n||_F / sqrt(n), [4] log2 of the subdiagonals' product,
// [5] ||H||_F.
__global__ void __launch_bounds__(512) roots_setup_kernel(RootArgs a) {
  const int n = a.isc[ISC_R];
  const int tid = threadIdx.x;
  __shared__ double red[32];
  __shared__ int bad;
  if (tid == 0) bad = (n < a.min_n) ? 1 : 0;
  for (int k = tid; k < kRootSteps; k += 512) a.left[k] = 0;
  __syncthreads();
  double an = 0.0, fr = 0.0, t1 = 0.0, t2 = 0.0, mx = 0.0, ls = 0.0;
  for (int c = tid >> 5; c < n; c += 16)  // a warp per column
    for (int i = tid & 31; i <= min(c + 1, n - 1); i += 32) {
      const double h = a.H[i + int64_t(c) * a.ld], v = fabs(h);
      a.Hf[i + int64_t(c) * a.ld] = float(h);
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
      a.invsubf[i] = float(-1.0 / sub);
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
  // and H, the divisors' reciprocals and the values fit FP32 (a projected matrix has the snapshots' ratio
  // as its scale, so others hardly occur)
  if (tid == 0 && !(mx > 0x1p-60 && mx < 0x1p+60)) bad = 1;
  __syncthreads();
  const double c = t1 / n;
  const double fro = sqrt(fmax(0.0, fr - t1 * c) / n);
  if (tid == 0) {
    a.scal[0] = an;
    a.scal[1] = t1;
    a.scal[2] = t2;
    a.scal[3] = fro;
    a.scal[4] = ls;
    a.scal[5] = sqrt(fr);
    a.isc[ISC_QR] = bad;
  }
}

// The start circle: its radius from the determinant of H - tr(H)/n.
__global__ void __launch_bounds__(kRootThreads) roots_start_kernel(RootArgs a) {
  pdl_wait();
  pdl_trigger();
  const int n = a.isc[ISC_R], tid = threadIdx.x;
  if (a.isc[ISC_QR]) return;
  __shared__ HymanShared<float> hs;
  const double c = a.scal[1] / n, fro = a.scal[3];
  int b;
  const int e2 = hyman_any<float>(a.Hf, a.ld, n, a.invsubf, float(c), 0.f, hs, &b);
  const float v = fabsf(hs.next[b][0]);
  const double det = v == 0.f ? 0.0 : v <= 3e38f ? exp2((double(log2f(v)) + double(e2) + a.scal[4]) / n) : fro;
  const double rad = fmin(fmax(det, 1e-2 * fro), fro);
  for (int i = tid; i < n; i += kRootThreads) {
    double sn, cs;
    sincospi(2.0 * (i + 0.35) / n, &sn, &cs);
    a.zr[i] = fma(rad, cs, c);
    a.zi[i] = rad * sn;
    a.dold[i] = 1e300;
    a.conv[i] = 0;
  }
}

// Steps after which a spectrum of n values is given up if none of them has converged: repeated eigenvalues,
// whose corrections shrink by a third to two thirds a step.  (Where the iteration succeeds the first value
// converges in step 4 to 9; the steps that are left out cost up to 12 us each at order 10, and the QR
// iteration that follows them 260.)
__device__ __forceinline__ int patience(int n) { return 8 + min(n, 32) / 8; }
__device__ __forceinline__ bool given_up(const RootArgs &a, int n) { return a.left[patience(n) - 1] == n; }

// The FP64 step after which no value was left, -1 if there is none
__device__ __forceinline__ int last_step(const RootArgs &a, int n) {
  if (given_up(a, n)) return -1;
  for (int k = 0; k < kRootSteps; ++k)
    if (a.left[k] == 0) return k;
  return -1;
}

// The correction p / (p' - p S) of one eigenvalue (Smith's division); S = sum 1 / (z_i - z_j)
template <typename T>
__device__ __forceinline__ void correction(T pr, T pi, T qr, T qi, T sr, T si, T &dr, T &di) {
  qr -= pr * sr - pi * si;
  qi -= pr * si + pi * sr;
  if (fabs(qr) >= fabs(qi)) {
    const T t = qi / qr, d = fma(qi, t, qr);
    dr = fma(pi, t, pr) / d;
    di = fma(-pr, t, pi) / d;
  } else {
    const T t = qr / qi, d = fma(qr, t, qi);
    dr = fma(pr, t, pi) / d;
    di = fma(pi, t, -pr) / d;
  }
}

// Step `it` of the first phase, in FP32: CTA i improves eigenvalue i from the values in buffer it & 1
// into the other one.  Far from the eigenvalues the corrections need no more, and an FP32 operation
// takes 4 cycles where an FP64 one takes 64: 57 us a step at n = 255 against 131.  What FP32 makes of
// a value only decides where the FP64 phase starts from: a value that it cannot improve stays.
__global__ void __launch_bounds__(kRootThreads) roots_step32_kernel(RootArgs a, int it) {
  pdl_wait();
  pdl_trigger();
  const int n = a.isc[ISC_R], i = blockIdx.x;
  if (i >= n || a.isc[ISC_QR]) return;
  const int tid = threadIdx.x, K = a.ld;
  const double *zri = a.zr + (it & 1) * K, *zii = a.zi + (it & 1) * K;
  double *zro = a.zr + ((it & 1) ^ 1) * K, *zio = a.zi + ((it & 1) ^ 1) * K;
  const float zr = float(zri[i]), zi = float(zii[i]);
  if (a.conv[i]) {
    if (tid == 0) {
      zro[i] = zr;
      zio[i] = zi;
    }
    return;
  }
  __shared__ HymanShared<float> hs;
  __shared__ float red[kRootThreads / 32][2];
  float sr = 0.f, si = 0.f;
  for (int j = tid; j < n; j += kRootThreads)
    if (j != i) {
      const float dr = zr - float(zri[j]), di = zi - float(zii[j]);
      const float q = 1.f / fmaf(dr, dr, di * di);
      sr = fmaf(dr, q, sr);
      si = fmaf(-di, q, si);
    }
  sr = warp_sum(sr);
  si = warp_sum(si);
  if ((tid & 31) == 0) {
    red[tid >> 5][0] = sr;
    red[tid >> 5][1] = si;
  }
  int b;
  hyman_any<float>(a.Hf, K, n, a.invsubf, zr, zi, hs, &b);
  if (tid == 0) {
    sr = (red[0][0] + red[1][0]) + (red[2][0] + red[3][0]);
    si = (red[0][1] + red[1][1]) + (red[2][1] + red[3][1]);
    float dr, di;
    correction(hs.next[b][0], hs.next[b][1], hs.next[b][2], hs.next[b][3], sr, si, dr, di);
    const bool fin = isfinite(dr) && isfinite(di);
    if (!fin) dr = di = 0.f;
    zro[i] = zr - dr;
    zio[i] = zi - di;
    const float ad = hypotf(dr, di), scl = hypotf(zr, zi) + 1e-3f * float(a.scal[3]);
    if (fin && (ad <= 3e-5f * scl || (ad < 1e-2f * scl && ad > 0.5f * float(a.dold[i])))) a.conv[i] = 1;
    a.dold[i] = fin ? ad : 1e30f;
  }
}

// Step `it` of the second phase, in FP64.
__global__ void __launch_bounds__(kRootThreads) roots_step_kernel(RootArgs a, int it) {
  pdl_wait();
  pdl_trigger();
  const int n = a.isc[ISC_R], i = blockIdx.x;
  if (i >= n || a.isc[ISC_QR] || (it > 0 && a.left[it - 1] == 0) || given_up(a, n)) return;
  const int tid = threadIdx.x, K = a.ld;
  const double *zri = a.zr + (it & 1) * K, *zii = a.zi + (it & 1) * K;
  double *zro = a.zr + ((it & 1) ^ 1) * K, *zio = a.zi + ((it & 1) ^ 1) * K;
  const double zr = zri[i], zi = zii[i];
  if (a.conv[i] == 2) {
    if (tid == 0) {
      zro[i] = zr;
      zio[i] = zi;
    }
    return;
  }
  __shared__ HymanShared<double> hs;
  __shared__ double red[kRootThreads / 32];
  double sr = 0.0, si = 0.0, s2 = 0.0;
  for (int j = tid; j < n; j += kRootThreads)
    if (j != i) {
      const double dr = zr - zri[j], di = zi - zii[j];
      const double q = 1.0 / fma(dr, dr, di * di);
      sr = fma(dr, q, sr);
      si = fma(-di, q, si);
      s2 += q;
    }
  int b;
  hyman_any<double>(a.H, K, n, a.invsub, zr, zi, hs, &b);
  sr = block_sum_n(sr, red, kRootThreads);
  si = block_sum_n(si, red, kRootThreads);
  s2 = block_sum_n(s2, red, kRootThreads);
  if (tid == 0) {
    double dr, di;
    correction(hs.next[b][0], hs.next[b][1], hs.next[b][2], hs.next[b][3], sr, si, dr, di);
    const bool fin = isfinite(dr) && isfinite(di);
    if (!fin) dr = di = 0.0;
    zro[i] = zr - dr;
    zio[i] = zi - di;
    // What a correction d leaves is at most about d^2 sum_j |e_j| / |z_i - z_j|^2, e_j the errors of the
    // other values (none above the spectrum's own size): nothing, once d^2 s2 is below 1e-16.  An
    // ill-conditioned eigenvalue's corrections stop shrinking at its own rounding level instead.
    const double ad = hypot(dr, di), scl = hypot(zr, zi) + 1e-3 * a.scal[3];
    const double before = it > 0 ? a.dold[i] : 1e300;
    const bool done = fin && ad < 1e-7 * scl && (ad * ad * s2 <= 1e-16 || ad <= 1e-12 * scl || ad > 0.5 * before);
    a.dold[i] = ad;
    if (done) a.conv[i] = 2;
    else atomicAdd(&a.left[it], 1);
  }
}

// For each value the one nearest to its conjugate, and its nearest neighbour: a warp per value
__global__ void __launch_bounds__(256) roots_pair_kernel(RootArgs a) {
  pdl_wait();
  pdl_trigger();
  const int n = a.isc[ISC_R], i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (a.isc[ISC_QR] || i >= n) return;
  const int last = last_step(a, n);
  if (last < 0) return;
  const double *zr = a.zr + ((last & 1) ^ 1) * a.ld, *zi = a.zi + ((last & 1) ^ 1) * a.ld;
  double best = 1e300, near = 1e300;
  int arg = i;
  for (int j = lane; j < n; j += 32) {
    const double dr = zr[j] - zr[i], di = zi[j] + zi[i], ds = zi[j] - zi[i];
    const double d = fma(dr, dr, di * di);
    if (j != i) near = fmin(near, fma(dr, dr, ds * ds));
    if (d < best) {
      best = d;
      arg = j;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
    if (ob < best || (ob == best && oa < arg)) {
      best = ob;
      arg = oa;
    }
  }
  // two values this close may be one eigenvalue found twice
  if (!(near > 1e-18 * a.scal[3] * a.scal[3])) a.isc[ISC_QR] = 1;
  if (lane == 0) a.part[i] = arg;
}

// Pair the values, check them, and store them as the QR iteration does (a conjugate pair side by
// side, +Im first).  They are passed on if all converged, no two are within 1e-9 of the spectrum's size,
// each value's nearest conjugate has that value as its own nearest one (a real eigenvalue is its
// own), and both traces agree: a value found twice in place of another one would change them.  Otherwise
// isc[ISC_QR] asks for the QR iteration.  Whether each is as accurate as the QR iteration's decides the
// inverse iteration (invit_kernel), which takes the pairs' means as they are stored here.
__global__ void __launch_bounds__(512) roots_finish_kernel(RootArgs a) {
  pdl_wait();
  const int n = a.isc[ISC_R], tid = threadIdx.x, K = a.ld;
  if (a.isc[ISC_QR]) return;
  __shared__ double zr[kMaxK], zi[kMaxK], red[32];
  __shared__ short part[kMaxK];
  __shared__ int bad, last;
  if (tid == 0) {
    bad = 0;
    last = last_step(a, n);
    a.isc[ISC_ITS] = last >= 0 ? last + 1 : given_up(a, n) ? patience(n) : kRootSteps;
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
  for (int i = tid; i < n; i += 512) part[i] = short(a.part[i]);
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

// Up to one CTA per SM the steps follow one another as programmatic dependent launches (each waits before it
// reads anything), so that a step that finds nothing left to do costs little more than its launch:
// order 10 332 -> 292 us, order 100 925 -> 838 us.  Beyond that the next step's waiting CTAs unbalance the
// running one's second CTAs over the SMs (order 255 3.47 -> 3.64 ms).
cudaError_t launch_roots(const RootArgs &a, int m, int sms, cudaStream_t s) {
  roots_setup_kernel<<<1, 512, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (m < a.min_n) return e;
  static_assert(kRootSteps32 % 2 == 0, "the FP64 phase starts from buffer 0");
  auto go = [&](auto k, int grid, int block, auto... args) {
    if (e != cudaSuccess) return;
    if (m <= sms) {
      e = launch_pdl(k, grid, block, 0, s, args...);
    } else {
      k<<<grid, block, 0, s>>>(args...);
      e = cudaGetLastError();
    }
  };
  go(roots_start_kernel, 1, kRootThreads, a);
  for (int it = 0; it < (m >= kRootMin32 ? kRootSteps32 : 0); ++it) go(roots_step32_kernel, m, kRootThreads, a, it);
  for (int it = 0; it < kRootSteps; ++it) go(roots_step_kernel, m, kRootThreads, a, it);
  go(roots_pair_kernel, (m + 7) / 8, 256, a);
  go(roots_finish_kernel, 1, 512, a);
  return e;
}

}  // namespace foa
