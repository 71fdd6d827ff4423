// lbm_vn.cu -- linear (von Neumann) stability analysis of Sec. IV on the
// device (include/lbm_vn.h).
//
// k_vn_jacobian: one block of 16 threads per case. Thread j pushes the dual
//   number f + eps e_j through the per-node collision code of the step kernels
//   (d2v16::transform / conserved / collide) at f = f^eq(state); the
//   derivative part of the result is column j of the collision Jacobian
//   d(Delta f^coll)/df = -dt M^-1 S_hat (M - dfhat^eq/df) of Sec. IV.
// k_vn_eig: L = 4, 8 or 16 threads per matrix (32 / L matrices per warp, a warp
//   per block, the matrices in shared memory). G = diag(Lax-Wendroff symbol of
//   Eq. A.1) + Jacobian, then Householder reduction to upper Hessenberg form
//   and explicit single-shift complex QR sweeps (Wilkinson shift from the
//   trailing 2 x 2 block, exceptional shifts after 10 and 20 sweeps without
//   deflation, deflation where |h_{l,l-1}| <= u (|h_{l-1,l-1}| + |h_{l,l}|), u =
//   2^-52), the textbook complex Schur iteration (Golub and Van Loan, Matrix
//   Computations, Secs. 7.4-7.5), in FP64. Every loop is bounded; a matrix
//   that does not converge within 30 x 16 sweeps gets NaN results.

#include <cuda_runtime.h>

#include <cmath>
#include <string>

#include "../../include/lbm_vn.h"
#include "coeffs.h"
#include "d2v16.cuh"

using namespace d2v16;

namespace {

thread_local std::string g_vn_error = "no error";

int vfail(int code, const std::string& m) {
  g_vn_error = m;
  return code;
}
int vcuda(cudaError_t e, const char* what) {
  return vfail(e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA,
               std::string(what) + ": " + cudaGetErrorString(e));
}
#define VCK(call)                                  \
  do {                                             \
    cudaError_t e_ = (call);                       \
    if (e_ != cudaSuccess) return vcuda(e_, #call); \
  } while (0)

// ---------------------------------------------------------------------------
// Forward-mode dual numbers: (value, derivative along one direction)
// ---------------------------------------------------------------------------
struct Dual {
  double v, d;
  Dual() = default;
  __device__ Dual(double x) : v(x), d(0.0) {}
  __device__ Dual(double x, double dx) : v(x), d(dx) {}
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return Dual(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return Dual(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) {
  return Dual(a.v * b.v, a.d * b.v + a.v * b.d);
}
__device__ __forceinline__ Dual operator*(double k, Dual b) { return Dual(k * b.v, k * b.d); }
// (1/x)' = -x' / x^2
__device__ __forceinline__ Dual recip(Dual x) {
  const double r = d2v16::recip(x.v);
  return Dual(r, -x.d * r * r);
}

// Lax-Wendroff weights of Eq. A.1 per population (set_advection).
struct LW {
  double a0[16], aE[16], aW[16], aN[16], aS[16];
};

constexpr int SWEEPS_PER_EIG = 30;  // average QR sweeps allowed per eigenvalue

__global__ void __launch_bounds__(16) k_vn_jacobian(const lbm_vn_case* cases, const Coeffs<double> base,
                                                    double dt, double* Jc) {
  __shared__ Coeffs<double> K;
  const int c = blockIdx.x, j = threadIdx.x;
  const lbm_vn_case cs = cases[c];
  if (j == 0) {
    K = base;
    set_rates(K, dt, cs.s);
  }
  __syncthreads();
  bool ok = cs.rho > 0.0 && cs.T > 0.0 && isfinite(cs.rho) && isfinite(cs.T) &&
            isfinite(cs.u) && isfinite(cs.v);
  for (int k = 0; k < 16; ++k) ok = ok && isfinite(cs.s[k]);
  double* col = Jc + (size_t)c * 256;
  if (!ok) {
    for (int i = 0; i < 16; ++i) col[i * 16 + j] = nan("");
    return;
  }
  const double rho = cs.rho, jx = rho * cs.u, jy = rho * cs.v;
  const double e = rho * cs.T + 0.5 * rho * (cs.u * cs.u + cs.v * cs.v);
  double f0[16];
  feq<double, double>(K, rho, jx, jy, e, f0);
  Dual f[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) f[i] = Dual(f0[i], i == j ? 1.0 : 0.0);
  Groups<Dual> g;
  transform(f, g);
  const Cons<Dual> m = conserved(K, g);
  Dual df[16];
  collide(K, g, m, df);
#pragma unroll
  for (int i = 0; i < 16; ++i) col[i * 16 + j] = df[i].d;
}

// ---------------------------------------------------------------------------
// Complex arithmetic and the 16 x 16 eigenvalue solver
// ---------------------------------------------------------------------------
struct cplx {
  double re, im;
};
__device__ __forceinline__ cplx mk(double r, double i) { return cplx{r, i}; }
__device__ __forceinline__ cplx operator+(cplx a, cplx b) { return mk(a.re + b.re, a.im + b.im); }
__device__ __forceinline__ cplx operator-(cplx a, cplx b) { return mk(a.re - b.re, a.im - b.im); }
__device__ __forceinline__ cplx operator-(cplx a) { return mk(-a.re, -a.im); }
__device__ __forceinline__ cplx operator*(cplx a, cplx b) {
  return mk(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
__device__ __forceinline__ cplx operator*(double k, cplx a) { return mk(k * a.re, k * a.im); }
__device__ __forceinline__ cplx conj(cplx a) { return mk(a.re, -a.im); }
__device__ __forceinline__ double cabs(cplx a) { return hypot(a.re, a.im); }
__device__ __forceinline__ double cabs1(cplx a) { return fabs(a.re) + fabs(a.im); }
__device__ __forceinline__ double norm2(cplx a) { return a.re * a.re + a.im * a.im; }
// 1 / sqrt(x) for positive normal x: the hardware's approximation y and one
// third-order step of the series of (1 - e)^(-1/2), e = 1 - x y^2: y (1 + e / 2
// + 3 e^2 / 8), which leaves e^3 (below 2^-60): five FP64 operations.
__device__ __forceinline__ double rsq(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ bool is_zero(double x) {  // without the FP64 units
  return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) == 0;
}
// The solver scales its matrix to entries below 2 in magnitude, so squares
// cannot overflow; sums of squares from TINY on have lost nothing to underflow (their
// bits end above 2^-1022).
constexpr double TINY = 0x1p-960;
// Principal square root of z = x + i y, |z| = r: t = sqrt((r + |x|) / 2),
// (t, y / (2 t)) when x >= 0, else (|y| / (2 t), sign(y) t); 0 for |z|^2 <
// TINY. Used for shifts only, which may be guesses.
__device__ __forceinline__ cplx csqrt(cplx z) {
  const double n2 = norm2(z);
  if (!(n2 >= TINY)) return mk(0.0, 0.0);
  const double u = 0.5 * fma(n2, rsq(n2), fabs(z.re));
  const double iu = rsq(u), t = u * iu, o = 0.5 * z.im * iu;
  return z.re >= 0.0 ? mk(t, o) : mk(fabs(o), copysign(t, z.im));
}
// Givens rotation G = [[c, s], [-conj(s), c]], c real, with G (a, b)^T = (r, 0)^T:
// c = |a| / n, s = a conj(b) / (|a| n), r = a n / |a|, n^2 = |a|^2 + |b|^2: all
// from w = 1 / (|a| n), one reciprocal square root.
__device__ __forceinline__ void givens(cplx a, cplx b, double& c, cplx& s, cplx& r) {
  const double na2 = norm2(a), nb2 = norm2(b), n2 = na2 + nb2;
  const double q = na2 * n2;
  if (__double2hiint(q) >= __double2hiint(TINY)) {
    const double w = rsq(q);
    c = na2 * w;
    s = w * (a * conj(b));
    r = (n2 * w) * a;
    return;
  }
  // |a| n is tiny or not a number: the rotation from the components' norms
  const double aa = cabs(a), ab = cabs(b);
  if (ab == 0.0) {
    c = 1.0;
    s = mk(0.0, 0.0);
    r = a;
  } else if (aa == 0.0) {
    c = 0.0;
    s = (1.0 / ab) * conj(b);
    r = mk(ab, 0.0);
  } else {
    const double n = hypot(aa, ab);
    const cplx ph = (1.0 / aa) * a;
    c = aa / n;
    s = ph * ((1.0 / n) * conj(b));
    r = n * ph;
  }
}

// One matrix in shared memory. Rows are one element (16 bytes) longer than the
// matrix, so that neighbouring rows start in different banks, and the whole is
// 64 bytes past a multiple of 512, so that the threads of a warp that access
// the same element of their matrices do too.
struct EigWork {
  cplx A[16][17];
  cplx v[16];      // Householder vector
  cplx pad[36];
};
static_assert(sizeof(EigWork) % 512 == 64, "bank offset between matrices");

// FP64 instructions of a warp cost the same whatever its number of active
// threads (19 clocks per SM, and 64 between two of one warp), so a warp runs
// its matrices in step: loops have bounds common to the warp, with the
// matrices' own ranges as conditions inside.
constexpr unsigned FULL = 0xffffffffu;
__device__ __forceinline__ int warp_max(int v) { return __reduce_max_sync(FULL, v); }
__device__ __forceinline__ int warp_min(int v) { return __reduce_min_sync(FULL, v); }
__device__ __forceinline__ int exponent(double x) { return __double2hiint(x) >> 20 & 0x7ff; }
template <int L>
__device__ __forceinline__ int group_max(int v) {
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(FULL, v, o));
  return v;
}

// Eigenvalues of W.A by the L threads of a group (thread l0 = 0 .. L - 1 of it,
// rows and columns l0, l0 + L, ...). On a true return (the same in the group)
// the eigenvalues are W.A's diagonal. Every thread of the warp calls it;
// `active` is false for groups without a matrix.
template <int L>
__device__ bool eig16(EigWork& W, int l0, bool active) {
  constexpr double U = 2.220446049250313e-16;  // 2^-52
  constexpr int N = 16 / L;                    // rows and columns per thread
  __syncwarp();
  // Largest exponent of an entry (as the high words' bits) and whether any is
  // non-zero, without the FP64 units.
  int top = 0;
  unsigned any = 0;
  for (int j = 0; j < N; ++j)
    for (int i = 0; i < 16; ++i) {
      const cplx a = W.A[l0 + L * j][i];
      const int hr = __double2hiint(a.re) & 0x7fffffff, hm = __double2hiint(a.im) & 0x7fffffff;
      top = max(top, max(hr, hm));
      any |= hr | hm | __double2loint(a.re) | __double2loint(a.im);
    }
  top = group_max<L>(top);
  any = (unsigned)group_max<L>(any != 0);
  const bool finite = top < 0x7ff00000;
  // 2^e with the largest component / 2^e in [1, 2): an exact scaling (e
  // clamped so that 2^-e stays a normal number)
  const int e = any ? max(-1000, min(1000, (top >> 20) - 1023)) : 0;
  const double scale = __hiloint2double((1023 + e) << 20, 0);
  const double inv_scale = __hiloint2double((1023 - e) << 20, 0);
  active = active && finite;
  for (int j = 0; j < N; ++j)
    for (int i = 0; i < 16; ++i) W.A[l0 + L * j][i] = inv_scale * W.A[l0 + L * j][i];

  // Householder reduction to upper Hessenberg form: A <- H A H, H = I - tau v v^H.
#pragma unroll 1
  for (int c = 0; c < 14; ++c) {
    __syncwarp();
    double tail = 0.0;
#pragma unroll 1
    for (int i = c + 2; i < 16; ++i) tail += norm2(W.A[i][c]);
    // Entries below 2^-480 beside ones of order 1 are left where they are (they
    // are not read again). The same decision in the group.
    const bool doit = tail >= TINY;
    const cplx x0 = W.A[c + 1][c];
    // An x0 that small counts as zero in everything that follows: the reflection has to
    // be one (its own inverse), or it changes the eigenvalues of the whole matrix.
    const double x2 = norm2(x0);
    const bool phase = x2 >= TINY;
    const double n0 = phase ? x2 : 0.0;
    const double i0 = rsq(x2);
    const double ax0 = phase ? n0 * i0 : 0.0;
    const cplx ph = phase ? i0 * x0 : mk(1.0, 0.0);
    const double s2 = n0 + tail, sigma = s2 * rsq(s2);
    const double tau = d2v16::recip(fma(sigma, ax0, s2));
    for (int j = 0; j < N; ++j) {
      const int l = l0 + L * j;
      if (l >= c + 1) W.v[l] = l == c + 1 ? (ax0 + sigma) * ph : W.A[l][c];
    }
    __syncwarp();
    if (doit) {
#pragma unroll 1
      for (int j = (c + 1) / L; j < N; ++j) {  // column l: A[:, l] -= tau v (v^H A[:, l])
        const int l = l0 + L * j;
        if (l > c) {
          cplx w = mk(0.0, 0.0);
#pragma unroll 1
          for (int i = c + 1; i < 16; ++i) w = w + conj(W.v[i]) * W.A[i][l];
          w = tau * w;
#pragma unroll 1
          for (int i = c + 1; i < 16; ++i) W.A[i][l] = W.A[i][l] - W.v[i] * w;
        }
      }
      for (int j = 0; j < N; ++j) {
        const int l = l0 + L * j;
        if (l == c + 1) W.A[l][c] = -(sigma * ph);
        else if (l > c + 1) W.A[l][c] = mk(0.0, 0.0);
      }
    }
    __syncwarp();
    if (doit) {
#pragma unroll 1
      for (int j = 0; j < N; ++j) {  // row l: A[l, :] -= tau (A[l, :] v) v^H
        const int l = l0 + L * j;
        cplx z = mk(0.0, 0.0);
#pragma unroll 1
        for (int i = c + 1; i < 16; ++i) z = z + W.A[l][i] * W.v[i];
        z = tau * z;
#pragma unroll 1
        for (int i = c + 1; i < 16; ++i) W.A[l][i] = W.A[l][i] - z * conj(W.v[i]);
      }
    }
  }
  __syncwarp();
  // max |a_ij|_1, as the bits of a non-negative double (their order as
  // integers): the deflation reference of a zero diagonal.
  long long nb = 0;
  for (int j = 0; j < N; ++j)
    for (int i = 0; i < 16; ++i) nb = max(nb, __double_as_longlong(cabs1(W.A[l0 + L * j][i])));
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) nb = max(nb, __shfl_xor_sync(FULL, nb, o));
  const double nrm = __longlong_as_double(nb);

  // Shifted QR sweeps on the active block [lo, hi].
  int hi = active ? 15 : 0, its = 0, total = 0, lo = 0;
  bool converged = active;
#pragma unroll 1
  while (true) {
    // Deflate until every unfinished matrix has an active block of two or more.
#pragma unroll 1
    while (true) {
      __syncwarp();
      int best = 0;
      unsigned small = 0;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const int l = l0 + L * j;
        // An entry within 2^-48 of the largest component on the diagonal (by
        // exponents, off the FP64 units) is not small; the others are looked at, and all
        // beside a diagonal so small that the difference has no meaning.
        bool look = false;
        if (l >= 1 && l <= hi) {
          const cplx p = W.A[l - 1][l - 1], q = W.A[l][l], o = W.A[l][l - 1];
          const int ed = max(max(exponent(p.re), exponent(p.im)), max(exponent(q.re), exponent(q.im)));
          look = max(exponent(o.re), exponent(o.im)) <= ed - 48 || ed <= 48;
        }
        if (!__any_sync(FULL, look)) continue;
        if (look) {
          double ref = cabs1(W.A[l - 1][l - 1]) + cabs1(W.A[l][l]);
          if (is_zero(ref)) ref = nrm;
          if (cabs1(W.A[l][l - 1]) <= U * ref) {
            best = l;
            small |= 1u << j;
          }
        }
      }
      lo = group_max<L>(best);
      __syncwarp();
#pragma unroll
      for (int j = 0; j < N; ++j)
        if (small >> j & 1u) W.A[l0 + L * j][l0 + L * j - 1] = mk(0.0, 0.0);
      const bool deflated = hi > 0 && lo == hi;
      if (deflated) {
        --hi;
        its = 0;
      }
      if (!__any_sync(FULL, deflated)) break;
    }
    if (hi > 0 && total >= SWEEPS_PER_EIG * 16) {
      converged = false;
      hi = 0;
    }
    if (!__any_sync(FULL, hi > 0)) break;
    __syncwarp();
    const bool run = hi > 0;
    cplx mu = mk(0.0, 0.0);
    if (run) {
      const cplx d = W.A[hi][hi], sub = W.A[hi][hi - 1];
      // Eigenvalue of [[a, b], [sub, d]] nearer d: d + h -+ sqrt(h^2 + b sub),
      // h = (a - d)/2, written as d - b sub / (h +- sqrt(...)) with the larger
      // denominator (no cancellation); where that is nearly nothing, d.
      const cplx a = W.A[hi - 1][hi - 1], b = W.A[hi - 1][hi];
      const cplx h = 0.5 * (a - d);
      const cplx bc = b * sub;
      const cplx r = csqrt(h * h + bc);
      const cplx den = (h.re * r.re + h.im * r.im) >= 0.0 ? h + r : h - r;
      const double n2 = norm2(den);
      mu = n2 >= TINY ? d - d2v16::recip(n2) * (bc * conj(den)) : d;
      if (its == 10 || its == 20) mu = mk(d.re + 0.75 * fabs(sub.re), d.im);
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int l = l0 + L * j;
      if (run && l >= lo && l <= hi) W.A[l][l] = W.A[l][l] - mu;
    }
    // H - mu I = Q R, rows k, k + 1 rotated in turn; R Q: columns k - 1, k
    // rotated one turn later, once row k is final (their rows end at k).
    const int k0 = warp_min(run ? lo : 16), k1 = warp_max(run ? hi : 0);
    double cp = 1.0;  // the previous rotation
    cplx sp = mk(0.0, 0.0);
#pragma unroll 1
    for (int k = k0; k <= k1; ++k) {
      __syncwarp();
      const bool rot = run && k >= lo && k < hi;       // a rotation of rows k, k + 1
      const bool col = run && k > lo && k <= hi;       // columns k - 1, k
      double c = 1.0;
      cplx s = mk(0.0, 0.0), r = mk(0.0, 0.0);
      if (rot) givens(W.A[k][k], W.A[k + 1][k], c, s, r);
      __syncwarp();
#pragma unroll 1
      for (int j = k / L; j <= k1 / L; ++j) {
        const int l = l0 + L * j;
        if (rot && l > k && l <= hi) {
          const cplx x = W.A[k][l], y = W.A[k + 1][l];
          W.A[k][l] = c * x + s * y;
          W.A[k + 1][l] = c * y - conj(s) * x;
        } else if (rot && l == k) {
          W.A[k][k] = r;
          W.A[k + 1][k] = mk(0.0, 0.0);
        }
      }
      __syncwarp();
#pragma unroll 1
      for (int j = k0 / L; j <= k / L; ++j) {
        const int l = l0 + L * j;
        if (col && l >= lo && l <= k) {
          const cplx x = W.A[l][k - 1], y = W.A[l][k];
          W.A[l][k - 1] = cp * x + conj(sp) * y;
          W.A[l][k] = cp * y - sp * x;
        }
      }
      cp = c;
      sp = s;
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int l = l0 + L * j;
      if (run && l >= lo && l <= hi) W.A[l][l] = W.A[l][l] + mu;
    }
    ++its;
    ++total;
  }
  __syncwarp();
  for (int j = 0; j < N; ++j) W.A[l0 + L * j][l0 + L * j] = scale * W.A[l0 + L * j][l0 + L * j];
  __syncwarp();
  return converged;
}

// Input modes of k_vn_eig.
enum { SRC_VN = 0, SRC_MATRIX = 1 };

// The phases (sin, cos of k_x dx and of k_y dy) of a wave vector.
struct Phases {
  double sx, cx, sy, cy;
};
__device__ __forceinline__ Phases phases(const double* k, double dx, double dy) {
  Phases p;
  sincos(k[0] * dx, &p.sx, &p.cx);
  sincos(k[1] * dy, &p.sy, &p.cy);
  return p;
}
// Entry r of the Lax-Wendroff symbol: a0 + aE e^{i tx} + aW e^{-i tx} + aN e^{i ty} +
// aS e^{-i ty}
__device__ __forceinline__ cplx symbol(const LW& lw, int r, const Phases& p) {
  return mk(lw.a0[r] + (lw.aE[r] + lw.aW[r]) * p.cx + (lw.aN[r] + lw.aS[r]) * p.cy,
            (lw.aE[r] - lw.aW[r]) * p.sx + (lw.aN[r] - lw.aS[r]) * p.sy);
}

// G of every (case, wave vector): the case's Jacobian and the symbol on the diagonal.
// Bound by the writes (4 KB a matrix, 8-byte stores since G may be aligned to doubles
// only). A block writes GM matrices, whose phases and diagonals are computed in full
// warps first: an FP64 instruction costs a warp the same whatever its active threads.
// 32 x 1024 matrices with the call's allocations: 264 us; 408 us when k_vn_eig wrote them
// in blocks of a warp, 300 in blocks of four.
constexpr int GM = 8, GM_T = 256;
__global__ void __launch_bounds__(GM_T) k_vn_matrices(long long nitems, int nk, const double* __restrict__ Jc,
                                                      const double* __restrict__ kvec, LW lw, double dx,
                                                      double dy, double* __restrict__ G) {
  __shared__ Phases ph[GM];
  __shared__ cplx diag[GM][16];
  const long long item0 = (long long)blockIdx.x * GM;
  const int n = (int)min((long long)GM, nitems - item0), t = threadIdx.x;
  if (t < n) ph[t] = phases(kvec + 2 * ((item0 + t) % nk), dx, dy);
  __syncthreads();
  if (t < 16 * n) {
    const int m = t >> 4, r = t & 15;
    diag[m][r] = mk(Jc[(item0 + m) / nk * 256 + 17 * r], 0.0) + symbol(lw, r, ph[m]);
  }
  __syncthreads();
  for (int m = 0; m < n; ++m) {
    const double* J = Jc + (item0 + m) / nk * 256;
    double* g = G + (item0 + m) * 512;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = (t + h * GM_T) >> 1, r = i >> 4;  // entry i, its real (t even) or imaginary part
      const bool on = (i & 15) == r;
      g[t + h * GM_T] = t & 1 ? (on ? diag[m][r].im : 0.0) : (on ? diag[m][r].re : J[i]);
    }
  }
}

// One matrix per L threads. SRC_VN: G of item (case, wave vector) from the
// case's collision Jacobian and the Lax-Wendroff symbol. SRC_MATRIX: the item's input
// matrix.
//
// Bound by the FP64 units. With 8 matrices per warp (L = 4) the scalar part of
// each rotation and shift serves 8 matrices and few threads idle: 3.2 M matrices/s
// on a map of 32 x 1024 (FP64 pipe 82 % busy); two per warp
// (16 threads each, idle outside the active block, shifts and rotations
// computed by all, the norms by one thread) 1.2 M. Rotations from one reciprocal
// square root instead of two, shifts and reflections from reciprocal square roots
// and the deflation test first by exponents: 11.5 -> 10.4 ms on that map.
template <int L>
__global__ void __launch_bounds__(32) k_vn_eig(int src, long long nitems, int nk,
                                               const double* __restrict__ Jc,
                                               const double* __restrict__ kvec, LW lw, double dx,
                                               double dy, const double* __restrict__ Ain,
                                               double* omega, double* radius,
                                               unsigned long long* failed) {
  constexpr int M = 32 / L;  // matrices per warp
  __shared__ EigWork work[M];
  const int grp = threadIdx.x / L, l0 = threadIdx.x % L;
  const long long item = (long long)blockIdx.x * M + grp;
  const bool have = item < nitems;
  EigWork& W = work[grp];
  if (!have) {
    for (int i = l0; i < 256; i += L) W.A[i >> 4][i & 15] = mk(0.0, 0.0);
  } else if (src == SRC_VN) {
    const long long c = item / nk;
    const int q = (int)(item - c * nk);
    const double* J = Jc + c * 256;
    const Phases p = phases(kvec + 2 * q, dx, dy);
    for (int i = l0; i < 256; i += L) {
      cplx a = mk(J[i], 0.0);
      const int r = i >> 4;
      if ((i & 15) == r) a = a + symbol(lw, r, p);
      W.A[r][i & 15] = a;
    }
  } else {
    const double* a = Ain + item * 512;
    for (int i = l0; i < 256; i += L) W.A[i >> 4][i & 15] = mk(a[2 * i], a[2 * i + 1]);
  }
  const bool ok = eig16<L>(W, l0, have);
  double r = ok ? 0.0 : nan("");
#pragma unroll 1
  for (int l = l0; l < 16; l += L) {
    const cplx w = ok ? W.A[l][l] : mk(nan(""), nan(""));
    if (omega && have) {
      omega[item * 32 + 2 * l] = w.re;
      omega[item * 32 + 2 * l + 1] = w.im;
    }
    if (ok) r = fmax(r, cabs(w));
  }
#pragma unroll
  for (int off = L / 2; off > 0; off >>= 1) r = fmax(r, __shfl_xor_sync(FULL, r, off));
  if (l0 == 0 && have) {
    if (radius) radius[item] = ok ? r : nan("");
    if (!ok && failed) atomicAdd(failed, 1ull);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct DevBuf {
  void* p = nullptr;
  cudaStream_t s = nullptr;
  ~DevBuf() {
    if (p) cudaFreeAsync(p, s);
  }
};

int check_grid(double dx, double dy, double dt) {
  if (!(std::isfinite(dx) && dx > 0.0 && std::isfinite(dy) && dy > 0.0 && std::isfinite(dt) &&
        dt > 0.0))
    return vfail(LBM_ERR_INVALID, "dx, dy and dt must be finite and > 0");
  return LBM_OK;
}

int check_cases(const lbm_vn_case* cases, int n) {
  for (int c = 0; c < n; ++c) {
    const lbm_vn_case& k = cases[c];
    bool ok = std::isfinite(k.rho) && k.rho > 0.0 && std::isfinite(k.T) && k.T > 0.0 &&
              std::isfinite(k.u) && std::isfinite(k.v);
    for (int i = 0; i < 16; ++i) ok = ok && std::isfinite(k.s[i]);
    if (!ok) return vfail(LBM_ERR_INVALID, "case " + std::to_string(c) +
                                               ": needs finite rates, rho > 0 and T > 0");
  }
  return LBM_OK;
}

int check_k(const double* k, int nk) {
  for (int q = 0; q < 2 * nk; ++q)
    if (!std::isfinite(k[q])) return vfail(LBM_ERR_INVALID, "non-finite wave vector");
  return LBM_OK;
}

// Copies n bytes of host data to a new device buffer (or aliases device data).
int stage_in(const void* src, size_t n, int on_device, cudaStream_t s, DevBuf& buf,
             const void** out) {
  if (on_device) {
    *out = src;
    return LBM_OK;
  }
  buf.s = s;
  VCK(cudaMallocAsync(&buf.p, n, s));
  VCK(cudaMemcpyAsync(buf.p, src, n, cudaMemcpyHostToDevice, s));
  *out = buf.p;
  return LBM_OK;
}

int alloc_out(void* host, size_t n, int on_device, cudaStream_t s, DevBuf& buf, void** out) {
  if (!host) {
    *out = nullptr;
    return LBM_OK;
  }
  if (on_device) {
    *out = host;
    return LBM_OK;
  }
  buf.s = s;
  VCK(cudaMallocAsync(&buf.p, n, s));
  *out = buf.p;
  return LBM_OK;
}

int copy_out(void* host, const void* dev, size_t n, int on_device, cudaStream_t s) {
  if (host && !on_device) VCK(cudaMemcpyAsync(host, dev, n, cudaMemcpyDeviceToHost, s));
  return LBM_OK;
}

// Threads per matrix: a warp's time grows with its matrices, so batches that
// do not give every SM four warps (one per partition) take fewer matrices per
// warp. Measured with 16 / 8 / 4 threads (before the last change): 1200 matrices
// 1.36 / 1.61 / 2.10 ms, 1600 1.70 / 1.59 / 2.10, 2400 2.26 / 1.82 / 2.34, 4800 3.92 /
// 2.76 / 2.44, 32768 23.9 / 15.7 / 11.5.
int launch_eig(int src, long long nitems, int nk, const double* Jc, const double* kvec, const LW& lw,
               double dx, double dy, const double* Ain, double* omega, double* radius,
               unsigned long long* failed, cudaStream_t s) {
  int dev = 0, sms = 0;
  VCK(cudaGetDevice(&dev));
  VCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const long long warps = 4ll * sms;
  auto grid = [&](int m) { return (unsigned)((nitems + m - 1) / m); };
  if (nitems <= 2 * warps)
    k_vn_eig<16><<<grid(2), 32, 0, s>>>(src, nitems, nk, Jc, kvec, lw, dx, dy, Ain, omega, radius, failed);
  else if (nitems <= 4 * warps)
    k_vn_eig<8><<<grid(4), 32, 0, s>>>(src, nitems, nk, Jc, kvec, lw, dx, dy, Ain, omega, radius, failed);
  else
    k_vn_eig<4><<<grid(8), 32, 0, s>>>(src, nitems, nk, Jc, kvec, lw, dx, dy, Ain, omega, radius, failed);
  VCK(cudaGetLastError());
  return LBM_OK;
}
// Items of one call: the grid of eight matrices per warp must stay below 2^31.
bool too_many(long long nitems) { return (nitems + 7) / 8 > 0x7FFFFFFFLL; }

// Shared body of lbm_vn_matrices (G != nullptr) and lbm_vn_spectrum.
int vn_run(const lbm_vn_case* cases, int ncases, const double* k, int nk, double dx, double dy,
           double dt, double* G, double* radius, double* omega, int on_device, void* stream,
           long long* nonconverged) {
  if (ncases < 1 || nk < 1 || !cases || !k)
    return vfail(LBM_ERR_INVALID, "need ncases >= 1, nk >= 1, cases and k");
  int rc = check_grid(dx, dy, dt);
  if (rc != LBM_OK) return rc;
  if (!on_device) {
    if ((rc = check_cases(cases, ncases)) != LBM_OK) return rc;
    if ((rc = check_k(k, nk)) != LBM_OK) return rc;
  }
  const long long nitems = (long long)ncases * nk;
  if (too_many(nitems)) return vfail(LBM_ERR_INVALID, "too many items");
  Coeffs<double> K;
  if (!lattice_constants(K)) return vfail(LBM_ERR_CUDA, "singular lattice block");
  set_advection(K, dt, dx, dy);
  LW lw;
  for (int i = 0; i < 16; ++i) {
    lw.a0[i] = K.a0[i];
    lw.aE[i] = K.aE[i];
    lw.aW[i] = K.aW[i];
    lw.aN[i] = K.aN[i];
    lw.aS[i] = K.aS[i];
  }
  cudaStream_t s = (cudaStream_t)stream;
  DevBuf bc, bk, bj, bg, br, bo, bf;
  const void *dcases = nullptr, *dk = nullptr;
  if ((rc = stage_in(cases, sizeof(lbm_vn_case) * ncases, on_device, s, bc, &dcases)) ||
      (rc = stage_in(k, sizeof(double) * 2 * nk, on_device, s, bk, &dk)))
    return rc;
  bj.s = s;
  VCK(cudaMallocAsync(&bj.p, sizeof(double) * 256 * (size_t)ncases, s));
  void *dG = nullptr, *dr = nullptr, *dw = nullptr;
  if ((rc = alloc_out(G, sizeof(double) * 512 * (size_t)nitems, on_device, s, bg, &dG)) ||
      (rc = alloc_out(radius, sizeof(double) * (size_t)nitems, on_device, s, br, &dr)) ||
      (rc = alloc_out(omega, sizeof(double) * 32 * (size_t)nitems, on_device, s, bo, &dw)))
    return rc;
  unsigned long long* dfail = nullptr;
  if (nonconverged) {
    bf.s = s;
    VCK(cudaMallocAsync(&bf.p, sizeof(unsigned long long), s));
    dfail = (unsigned long long*)bf.p;
    VCK(cudaMemsetAsync(dfail, 0, sizeof(unsigned long long), s));
  }
  k_vn_jacobian<<<ncases, 16, 0, s>>>((const lbm_vn_case*)dcases, K, dt, (double*)bj.p);
  VCK(cudaGetLastError());
  if (G) {
    k_vn_matrices<<<(unsigned)((nitems + GM - 1) / GM), GM_T, 0, s>>>(nitems, nk, (const double*)bj.p, (const double*)dk,
                                                                    lw, dx, dy, (double*)dG);
    VCK(cudaGetLastError());
  } else if ((rc = launch_eig(SRC_VN, nitems, nk, (const double*)bj.p, (const double*)dk, lw, dx, dy, nullptr,
                              (double*)dw, (double*)dr, dfail, s)) != LBM_OK) {
    return rc;
  }
  if ((rc = copy_out(G, dG, sizeof(double) * 512 * (size_t)nitems, on_device, s)) ||
      (rc = copy_out(radius, dr, sizeof(double) * (size_t)nitems, on_device, s)) ||
      (rc = copy_out(omega, dw, sizeof(double) * 32 * (size_t)nitems, on_device, s)))
    return rc;
  unsigned long long nf = 0;
  if (nonconverged) VCK(cudaMemcpyAsync(&nf, dfail, sizeof(nf), cudaMemcpyDeviceToHost, s));
  if (!on_device || nonconverged) VCK(cudaStreamSynchronize(s));
  if (nonconverged) *nonconverged = (long long)nf;
  return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_vn_matrices(const lbm_vn_case* cases, int ncases, const double* k, int nk, double dx,
                    double dy, double dt, double* G, int on_device, void* cuda_stream) {
  if (!G) return vfail(LBM_ERR_INVALID, "G is required");
  return vn_run(cases, ncases, k, nk, dx, dy, dt, G, nullptr, nullptr, on_device, cuda_stream,
                nullptr);
}

int lbm_vn_spectrum(const lbm_vn_case* cases, int ncases, const double* k, int nk, double dx,
                    double dy, double dt, double* radius, double* omega, int on_device,
                    void* cuda_stream, long long* nonconverged) {
  if (!radius && !omega && !nonconverged)
    return vfail(LBM_ERR_INVALID, "no output requested");
  return vn_run(cases, ncases, k, nk, dx, dy, dt, nullptr, radius, omega, on_device, cuda_stream,
                nonconverged);
}

int lbm_eig16(const double* A, long long n, double* omega, double* radius, int on_device,
              void* cuda_stream, long long* nonconverged) {
  if (n < 1 || !A) return vfail(LBM_ERR_INVALID, "need n >= 1 and A");
  if (!omega && !radius && !nonconverged) return vfail(LBM_ERR_INVALID, "no output requested");
  if (too_many(n)) return vfail(LBM_ERR_INVALID, "too many matrices");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  DevBuf ba, bo, br, bf;
  const void* dA = nullptr;
  int rc;
  if ((rc = stage_in(A, sizeof(double) * 512 * (size_t)n, on_device, s, ba, &dA))) return rc;
  void *dw = nullptr, *dr = nullptr;
  if ((rc = alloc_out(omega, sizeof(double) * 32 * (size_t)n, on_device, s, bo, &dw)) ||
      (rc = alloc_out(radius, sizeof(double) * (size_t)n, on_device, s, br, &dr)))
    return rc;
  unsigned long long* dfail = nullptr;
  if (nonconverged) {
    bf.s = s;
    VCK(cudaMallocAsync(&bf.p, sizeof(unsigned long long), s));
    dfail = (unsigned long long*)bf.p;
    VCK(cudaMemsetAsync(dfail, 0, sizeof(unsigned long long), s));
  }
  LW lw = {};
  if ((rc = launch_eig(SRC_MATRIX, n, 1, nullptr, nullptr, lw, 1.0, 1.0, (const double*)dA,
                       (double*)dw, (double*)dr, dfail, s)) != LBM_OK)
    return rc;
  if ((rc = copy_out(omega, dw, sizeof(double) * 32 * (size_t)n, on_device, s)) ||
      (rc = copy_out(radius, dr, sizeof(double) * (size_t)n, on_device, s)))
    return rc;
  unsigned long long nf = 0;
  if (nonconverged) VCK(cudaMemcpyAsync(&nf, dfail, sizeof(nf), cudaMemcpyDeviceToHost, s));
  if (!on_device || nonconverged) VCK(cudaStreamSynchronize(s));
  if (nonconverged) *nonconverged = (long long)nf;
  return LBM_OK;
}

const char* lbm_vn_last_error(void) { return g_vn_error.c_str(); }

}  // extern "C"
