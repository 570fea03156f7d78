// Singular values and left singular vectors of the upper-triangular beta_m (the rank truncation of
// Sec. 3.2.2), FP64:
//
//   svd_jacobi_kernel  one-sided (Hestenes) Jacobi on the rows of beta_m, a cooperative grid with one
//                      CTA per pair of the round-robin ordering
//   svd_finish_kernel  order by sigma, count the rank, put the vectors in that order
#include "api_internal.cuh"
#include "eig_internal.cuh"

namespace foa {

// ------------------------------------------------------------------------------ grid barrier
// Only used in cooperative launches (all CTAs co-resident), by the T threads threadIdx.x < T of each
// CTA (named barrier 1).  Bounded spin: a CTA that has waited spin_limit clock cycles for the others
// records FOA_DMD_ETIMEOUT and returns false, and its caller returns at once, so a CTA that never
// arrives ends the whole grid within the limit.
template <int T>
__device__ bool grid_barrier(GridBar *gb, int *err, long long spin_limit) {
  __shared__ int ok;
  named_bar_sync(1, T);
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned *vgen = &gb->gen;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(&gb->count, 1u);
    if (arrived == gridDim.x - 1) {
      gb->count = 0u;
      __threadfence();
      atomicAdd(&gb->gen, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (clock64() - t0 > spin_limit) {
          ok = 0;
          atomicExch(err, FOA_DMD_ETIMEOUT);
          break;
        }
      }
    }
    __threadfence();
  }
  named_bar_sync(1, T);
  return ok != 0;
}

// A matrix element with the number of the round that wrote it, moved as one 16-byte access, so that a
// reader that sees the round it waits for has the value too: no flag, no fence, one trip through L2.
__device__ __forceinline__ void st_tagged(double *p, double v, long long tag) {
  asm volatile("{\n .reg .b128 q;\n mov.b128 q, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], q;\n}\n" ::"l"(p),
               "l"(__double_as_longlong(v)), "l"(tag)
               : "memory");
}
__device__ __forceinline__ void ld_tagged(const double *p, double &v, long long &tag) {
  long long b;
  asm volatile("{\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%2];\n mov.b128 {%0, %1}, q;\n}\n"
               : "=l"(b), "=l"(tag)
               : "l"(p)
               : "memory");
  v = __longlong_as_double(b);
}

// This thread's rows of columns a and b (tagged elements) once both carry `tag`: bounded wait.
__device__ __forceinline__ bool load_pair(const double *a, const double *b, int t, int m, long long tag,
                                          double (&x)[kSvdRows], double (&y)[kSvdRows], long long spin_limit) {
  const long long t0 = clock64();
  while (true) {
    bool there = true;
    long long g[2 * kSvdRows];
#pragma unroll
    for (int u = 0; u < kSvdRows; ++u) {
      const int k = t + u * kSvdHalf;
      x[u] = y[u] = 0.0;
      g[2 * u] = g[2 * u + 1] = tag;
      if (k < m) {
        ld_tagged(a + 2 * k, x[u], g[2 * u]);
        ld_tagged(b + 2 * k, y[u], g[2 * u + 1]);
      }
    }
#pragma unroll
    for (int u = 0; u < 2 * kSvdRows; ++u) there = there && g[u] == tag;
    if (there) return true;
    if (clock64() - t0 > spin_limit) return false;
  }
}

__device__ __forceinline__ float sqrt_approx(float v) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

struct Rotation {
  double c, s;
  int go;
};

// The rotation that makes columns with squared norms sa, sb and product sg orthogonal, none (go = 0)
// where |sg| <= tol sqrt(sa sb).  zeta = (sb - sa) / (2 sg), t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
// c = 1 / sqrt(1 + t^2), s = c t.  The angle is formed in FP32: an error of 1e-7 in t leaves a product
// 1e-7 times the old one, which the next sweep removes (the number of sweeps is the same, measured on
// the fields' beta at m = 255 and 383); what has to be exact is c^2 + s^2 = 1, and c comes from that t
// in FP64 by one third-order step y + y e (1/2 + 3/8 e), e = 1 - u y^2, from the FP32 root.  With
// division and square roots in FP64 this took about 2400 cycles of every round, now about 700.
__device__ __forceinline__ Rotation rotation(double sa, double sb, double sg, float tol2) {
  Rotation r{1.0, 0.0, 0};
  const int ea = (__double2hiint(sa) >> 20) & 0x7ff, eb = (__double2hiint(sb) >> 20) & 0x7ff;
  const int eg = (__double2hiint(sg) >> 20) & 0x7ff;
  if (ea == 0 || eb == 0 || eg == 0) return r;
  const float fa = scaled_float(sa, ea), fb = scaled_float(sb, eb), fg = scaled_float(sg, eg);
  const int ex = 2 * eg - ea - eb;
  if (ex < -122 || ldexpf(__fdividef(fg * fg, fa * fb), ex) <= tol2) return r;
  r.go = 1;
  const double d = sb - sa;
  const int ed = (__double2hiint(d) >> 20) & 0x7ff;
  double t;
  float ft;
  if (eg + 60 < ed) {  // |zeta| beyond FP32's squares: t = 1 / (2 zeta)
    t = sg / d;
    ft = 0.f;
  } else {
    const int e = max(ed, eg);
    const float z = __fdividef(scaled_float(d, e), 2.f * scaled_float(sg, e));
    ft = __fdividef(copysignf(1.f, z), fabsf(z) + sqrt_approx(fmaf(z, z, 1.f)));
    t = ft;
  }
  const double u = fma(t, t, 1.0), y = rsqrtf(fmaf(ft, ft, 1.f));
  const double e = fma(-u * y, y, 1.0);
  r.c = fma(y * e, fma(0.375, e, 0.5), y);
  r.s = r.c * t;
  return r;
}

// ------------------------------------------------------------------------------ SVD
// One-sided Jacobi on the columns of A = beta_m^T: A J = U' Sigma with J orthogonal, so beta_m = J Sigma
// U'^T, and the left singular vectors of beta_m are the columns of J, the product of the rotations
// (A and J hold tagged elements, see st_tagged).  beta_m is the R factor of the snapshots: its rows fall off in size and are nearly
// orthogonal from the start, its columns are not: 12 and 13 sweeps for the fields' beta at m = 255
// and 383 against 15 and 16 on the columns, and 13 against 23 where the noise lies at 1e-7.
//
// A CTA takes one column pair at a time (one a round: the grid has (m+1)/2 <= 256 CTAs).  Threads 0-127
// (four warps, one per SM sub-partition) hold the pair of A, form its three products (a reduce-scatter
// over the lanes, 6 FP64 additions instead of 15, then the four warps), the rotation (every warp for
// itself) and the new columns; threads 128-255 follow with the same rotations on J, out of a ring in
// shared memory, so that J stays off the chain from round to round.
//
// What bounds it is that chain: a round's columns come from two other CTAs of the round before.  Every
// element carries its round (st_tagged), and a thread reads its rows until they are those of the last
// round: one trip through L2 from the neighbours' stores to these loads, where a flag behind a fence took
// three (the store's acknowledgement, the flag, the data).  A column has one owner in each round, who
// alone rewrites it, so it cannot be overwritten before it is read; nothing depends on which CTA takes
// which pair.  One grid barrier per sweep sums the rotation counts for the convergence test.
// m = 383, 13 sweeps: 24.2 ms (with flags 35 ms; the one-group kernel on beta's columns, 16 sweeps,
// 41 ms).
//
// skip_cta (normally -1) and spin_limit serve foa_dmd_test_wait_fault: CTA skip_cta returns before
// its first grid-barrier arrival, as a CTA that died would, and the others give up after
// spin_limit cycles.
constexpr int kRing = 16;  // rotations J may lag behind A

__global__ void __launch_bounds__(kSvdThreads, 2) svd_jacobi_kernel(const double *B, int ldb, int m, double *A, double *J,
                                                                    int lda, double *sig, int *isc, GridBar *gb,
                                                                    int max_sweeps, double tol, long long spin_limit,
                                                                    int skip_cta) {
  int *err = isc + ISC_ERR;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t gtid = int64_t(blockIdx.x) * blockDim.x + tid;
  const int64_t gthreads = int64_t(gridDim.x) * blockDim.x;
  __shared__ Rotation ring[kRing];
  __shared__ volatile int produced, consumed, total, abort_;
  __shared__ double red[2][kSvdHalf / 32][3];
  __shared__ int nrot;
  if (tid == 0) {
    produced = consumed = abort_ = 0;
    total = -1;  // pairs in all, once known
  }
  for (int64_t e = gtid; e < int64_t(m) * m; e += gthreads) {
    const int r = int(e % m), c = int(e / m);
    st_tagged(A + 2 * (r + int64_t(c) * lda), (c <= r) ? B[c + int64_t(r) * ldb] : 0.0, 0);
    st_tagged(J + 2 * (r + int64_t(c) * lda), (c == r) ? 1.0 : 0.0, 0);
  }
  if (gtid == 0) isc[ISC_ROT] = 0;
  if (int(blockIdx.x) == skip_cta) return;  // failure injection only (uniform over the CTA)
  if (!grid_barrier<kSvdThreads>(gb, err, spin_limit)) return;
  const int mp = m + (m & 1);  // players of the round-robin schedule (m may be odd: one dummy)
  const int npairs = mp / 2;
  if (max_sweeps > kMaxSweeps) max_sweeps = kMaxSweeps;
  auto columns = [&](int p, int rnd, int &i, int &j) {
    const int pa = p, pb = mp - 1 - p;
    i = pa == 0 ? 0 : 1 + (pa - 1 + rnd) % (mp - 1);
    j = pb == 0 ? 0 : 1 + (pb - 1 + rnd) % (mp - 1);
    return i < m && j < m;  // uniform over the CTA
  };
  auto store_pair = [&](double *a, double *b, const double (&x)[kSvdRows], const double (&y)[kSvdRows], const Rotation &r,
                        int t, long long tag) {
#pragma unroll
    for (int u = 0; u < kSvdRows; ++u) {
      const int k = t + u * kSvdHalf;
      if (k < m) {
        st_tagged(a + 2 * k, r.go ? r.c * x[u] - r.s * y[u] : x[u], tag);
        st_tagged(b + 2 * k, r.go ? r.s * x[u] + r.c * y[u] : y[u], tag);
      }
    }
  };
  // the column that meets the dummy this round: handed on unchanged
  auto pass_on = [&](double *M, int c, int t, long long tag) {
    double x[kSvdRows], y[kSvdRows];
    double *a = M + 2 * int64_t(c) * lda;
    const bool ok = load_pair(a, a, t, m, tag, x, y, spin_limit);
#pragma unroll
    for (int u = 0; u < kSvdRows; ++u) {
      const int k = t + u * kSvdHalf;
      if (k < m) st_tagged(a + 2 * k, x[u], tag + 1);
    }
    return ok;
  };

  if (tid >= kSvdHalf) {
    // ---------------------------------------------------------------- J: the same rotations, behind A
    const int t = tid - kSvdHalf;
    int n = 0;  // pairs done by this CTA
    for (int rd = 0, rnd = 0;; ++rd, rnd = rnd == mp - 2 ? 0 : rnd + 1)
      for (int p = blockIdx.x; p < npairs; p += gridDim.x, ++n) {
        bool stop = false;
        const long long t0 = clock64();
        while (produced <= n) {
          if (abort_ || (total >= 0 && n >= total)) {
            stop = true;
            break;
          }
          if (clock64() - t0 > 2 * spin_limit) {
            atomicExch(err, FOA_DMD_ETIMEOUT);
            stop = true;
            break;
          }
        }
        __threadfence_block();
        const Rotation r = ring[n % kRing];
        if (named_bar_or(2, kSvdHalf, abort_ || (stop && produced <= n))) return;
        if (t == 0) consumed = n + 1;
        int i, j;
        bool ok = true;
        if (columns(p, rnd, i, j)) {
          double *ji = J + 2 * int64_t(i) * lda, *jj = J + 2 * int64_t(j) * lda;
          double x[kSvdRows], y[kSvdRows];
          ok = load_pair(ji, jj, t, m, rd, x, y, spin_limit);
          store_pair(ji, jj, x, y, r, t, rd + 1);
        } else if (i < m || j < m) {
          ok = pass_on(J, i < m ? i : j, t, rd);
        }
        if (!ok) {
          atomicExch(err, FOA_DMD_ETIMEOUT);
          abort_ = 1;
        }
      }
  }

  // ------------------------------------------------------------------ A
  const int warp = tid >> 5;
  const float tol2 = float(tol * tol);
  int gr = 0, rd = 0;  // pairs done by this CTA, rounds
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    int myrot = 0;  // rotations applied by this CTA in the sweep
    for (int rnd = 0; rnd < mp - 1; ++rnd, ++rd) {
      for (int p = blockIdx.x; p < npairs; p += gridDim.x, ++gr) {
        int i, j;
        Rotation r{1.0, 0.0, 0};
        const bool both = columns(p, rnd, i, j);
        double *ai = A + 2 * int64_t(i) * lda, *aj = A + 2 * int64_t(j) * lda;
        double x[kSvdRows], y[kSvdRows];
        bool ok;
        if (both) ok = load_pair(ai, aj, tid, m, rd, x, y, spin_limit);
        else ok = (i < m || j < m) ? pass_on(A, i < m ? i : j, tid, rd) : true;
        const long long t0 = clock64();
        while (ok && gr - consumed >= kRing)  // room in J's ring
          if (abort_ || clock64() - t0 > 2 * spin_limit) ok = false;
        if (both) {
          double al = 0.0, be = 0.0, ga = 0.0;
#pragma unroll
          for (int u = 0; u < kSvdRows; ++u)
            if (u * kSvdHalf < m) {
              al = fma(x[u], x[u], al);
              be = fma(y[u], y[u], be);
              ga = fma(x[u], y[u], ga);
            }
          // reduce-scatter: lanes 0-7 end with al's sum, 8-15 with be's, 16-23 with ga's
          const bool hi = lane & 16, h8 = lane & 8;
          double k0 = hi ? ga : al, k1 = hi ? 0.0 : be;
          k0 += __shfl_xor_sync(0xffffffffu, hi ? al : ga, 16);
          k1 += __shfl_xor_sync(0xffffffffu, hi ? be : 0.0, 16);
          double v = h8 ? k1 : k0;
          v += __shfl_xor_sync(0xffffffffu, h8 ? k0 : k1, 8);
#pragma unroll
          for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if ((lane & 7) == 0 && lane < 24) red[gr & 1][warp][lane >> 3] = v;
        }
        if (named_bar_or(1, kSvdHalf, !ok)) {
          if (tid == 0) atomicExch(err, FOA_DMD_ETIMEOUT);
          abort_ = 1;
          return;
        }
        if (both) {
          const double(*rw)[3] = red[gr & 1];
          const double v = lane < 3 ? (rw[0][lane] + rw[1][lane]) + (rw[2][lane] + rw[3][lane]) : 0.0;
          r = rotation(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 1), __shfl_sync(0xffffffffu, v, 2),
                       tol2);
          store_pair(ai, aj, x, y, r, tid, rd + 1);
          myrot += r.go;
        }
        if (tid == 0) {
          ring[gr % kRing] = r;
          __threadfence_block();
          produced = gr + 1;
        }
      }
    }
    if (tid == 0 && myrot) atomicAdd(&gb->rot[sweep], unsigned(myrot));
    if (!grid_barrier<kSvdHalf>(gb, err, spin_limit)) {  // every CTA has finished the sweep and added its count
      abort_ = 1;
      return;
    }
    if (tid == 0) nrot = int(*(volatile unsigned *)&gb->rot[sweep]);
    named_bar_sync(1, kSvdHalf);
    if (nrot == 0) break;
  }
  if (tid == 0) total = gr;
  if (gtid == 0) isc[ISC_SWEEPS] = sweep;
  // column norms (one warp per column)
  const int warp_g = blockIdx.x * (kSvdHalf / 32) + warp, nwarps = gridDim.x * (kSvdHalf / 32);
  for (int c = warp_g; c < m; c += nwarps) {
    const double *ac = A + 2 * int64_t(c) * lda;
    double sq = 0.0;
    for (int k = lane; k < m; k += 32) {
      const double v = __ldcg(ac + 2 * k);
      sq += v * v;
    }
    sq = warp_sum(sq);
    if (lane == 0) sig[c] = sqrt(sq);
  }
}

// Sort singular values descending (stable by index), put the vectors (the columns of J) in that order,
// and count the retained rank r = #{sigma_i > tol sigma_1} (at least 1).  Every CTA ranks all values
// (bits of non-negative doubles compare as integers) and moves its share of the columns.
__global__ void __launch_bounds__(512) svd_finish_kernel(const double *J, int ld, int m, const double *sig_in, double *U,
                                                         double *sig, int *isc, double rank_tol) {
  __shared__ long long s[kMaxK];
  __shared__ short pos[kMaxK];
  __shared__ int cnt;
  const int tid = threadIdx.x;
  for (int i = tid; i < m; i += blockDim.x) s[i] = __double_as_longlong(sig_in[i]);
  if (tid == 0) cnt = 0;
  __syncthreads();
  long long smax = 0;
  for (int i = tid; i < m; i += blockDim.x) {
    int rank = 0;
    for (int k = 0; k < m; ++k) rank += (s[k] > s[i]) || (s[k] == s[i] && k < i);
    pos[i] = short(rank);
  }
  for (int k = 0; k < m; ++k) smax = s[k] > smax ? s[k] : smax;
  __syncthreads();
  for (int c = blockIdx.x; c < m; c += gridDim.x)
    for (int r = tid; r < m; r += blockDim.x) U[r + int64_t(pos[c]) * ld] = J[2 * (r + int64_t(c) * ld)];
  if (blockIdx.x != 0) return;
  for (int i = tid; i < m; i += blockDim.x) {
    const double v = __longlong_as_double(s[i]);
    sig[pos[i]] = v;
    if (v > rank_tol * __longlong_as_double(smax)) atomicAdd(&cnt, 1);
  }
  __syncthreads();
  if (tid == 0) isc[ISC_R] = cnt < 1 ? 1 : cnt;
}

}  // namespace foa
