// Small dense problems of the eigensolver, one CTA each: the Rayleigh-Ritz eigenproblem on the
// trial basis and the SVQB transforms that orthonormalise a block from its Gram matrix
// (declarations and layout conventions in blockops.cuh).
//
// The Hermitian eigensolver is direct: Householder reduction to a real tridiagonal matrix,
// bisection of the wanted eigenvalues, inverse iteration, back-transformation. What bounds it is
// the FP64 pipe of one SM: a warp's FP64 instruction occupies its quarter of the SM for 64 cycles
// whatever its active lanes and however independent (measured; 2 lanes a clock and SM), so
//   - long sums run with full warps, short serial chains (norms, square roots) on one warp, and
//     chains that do not depend on one another on different quarters of the SM;
//   - bisection, which needs no last bit, counts eigenvalues in double-float arithmetic on the
//     FP32 pipes (5x the FP64 rate); inverse iteration and Rayleigh quotients are FP64.
// Measured on one GB300, Rayleigh-Ritz with 72 basis vectors and 24 pairs: 1.21 ms (reduction 0.50,
// bisection 0.06, inverse iteration 0.11, back-transformation 0.24, P coefficients 0.30), m = 12
// with 4 pairs 0.11 ms. Cyclic Jacobi in double-float arithmetic, which this replaced, took 6.2
// and 0.30 ms (8 to 13 sweeps of 71 rounds at about 19k cycles) and left residuals near 1e-10 on
// matrices with entries near 10^3; errors are now those of FP64 (residuals 2e-16 |A|).
#include <algorithm>
#include <cmath>
#include <string>

#include "blockops.cuh"

namespace iwf {

namespace {

constexpr int kSmallThreads = 512;
constexpr int kLu = kMaxSmall * kMaxBlock;   // one LU array or the eigenvectors of T, in doubles

struct SmallShared {
  double2 A[kMaxSmall * kMaxSmall];   // matrix, then its reflectors below the diagonal
  double2 V[kMaxSmall * kMaxSmall];   // work: LU factors and eigenvectors of T; small products
  double2 B[kMaxSmall * kMaxBlock];   // n x k eigenvectors; m x b P coefficients
  double2 v[2][kMaxSmall], p[kMaxSmall], wv[kMaxSmall];  // Householder vectors, A v, w
  double2 ph[kMaxSmall];              // phases that make T real
  double d[kMaxSmall], e[kMaxSmall];  // T: diagonal, off-diagonal (then scaled to |T| < 1)
  double tau[kMaxSmall];
  float4 t[kMaxSmall];                // scaled d and e^2 as float pairs
  long long lam[32];                  // eigenvalues of scaled T in units of 2^-55
  double w[kMaxBlock];                // eigenvalues, ascending
  double scale[kMaxBlock];            // SVQB column scales
  double2 al;                         // of the column in work: alpha, its square, 1 / |alpha|,
  double a2, ra, tot, nrm;            // |x|^2, |x|
  int idx[kMaxSmall];
  int keep[kMaxBlock];
  double r, r2;
  int flag, reflect, dev;
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// s + a b and s + conj(a) b
__device__ __forceinline__ double2 cmac(double2 a, double2 b, double2 s) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, s.x)), fma(a.x, b.y, fma(a.y, b.x, s.y)));
}
__device__ __forceinline__ double2 cmac_conj(double2 a, double2 b, double2 s) {
  return make_double2(fma(a.x, b.x, fma(a.y, b.y, s.x)), fma(a.x, b.y, fma(-a.y, b.x, s.y)));
}

// Element e < n (n + 1) / 2 of the lower triangle of an n x n matrix, folded so that rows r and
// n - 1 - r share n + 1 consecutive e (no division-free row search, equal work per thread).
__device__ __forceinline__ void fold(int e, int n, int& row, int& col) {
  const int a = e / (n + 1), b = e - a * (n + 1);
  if (b < n - a) { row = n - 1 - a; col = b; }
  else { row = a; col = b - (n - a); }
}

// ---- Householder reduction ------------------------------------------------------------------
// A <- H A H for Hermitian reflectors H = I - tau v v^H, tau = 2 / |v|^2 (real), column by column:
// x = the column below the diagonal, alpha = x_0 = |alpha| u, v = x + u |x| e_0, so that H x =
// -u |x| e_0 and tau = 1 / (|x|^2 + |alpha| |x|). The off-diagonals' phases are gathered in ph:
// A = (H_0 H_1 ...) diag(ph) T diag(ph)^H (...)^H with T real. v replaces its column.
// A step costs 4 r^2 multiply-adds for A v and 4 r^2 for the rank-two update of one triangle
// (mirrored by stores), r = n - 1 - i, and a serial FP64 chain: warp 0 updates the next column
// first and starts that column's chain while the other warps finish the update.
__device__ void householder_chain(SmallShared& sh, int n, int i) {
  const int lane = threadIdx.x & 31, r = n - 1 - i;
  const double2* col = sh.A + (i + 1) * n + i;
  double s2 = 0.0;                                     // |x_1|^2 + ...
  for (int x = 1 + lane; x < r; x += 32) {
    const double2 c = col[x * n];
    s2 = fma(c.x, c.x, fma(c.y, c.y, s2));
  }
  for (int o = 16; o; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  const double2 al = col[0];
  const double a2 = fma(al.x, al.x, al.y * al.y);
  // above about 1e-290 (compared as integers: an FP64 comparison costs as much as a product);
  // a NaN, of either sign, goes on
  const auto nonzero = [](double v) { return (__double2hiint(v) & 0x7fffffff) > 0x03000000; };
  const bool reflect = nonzero(s2), has_al = nonzero(a2);
  const double tot = s2 + a2;
  // lane 1: 1 / |alpha|, the others 1 / |x|
  const double q = lane == 1 ? (has_al ? a2 : 1.0) : (reflect || has_al ? tot : 1.0);
  const double rq = rsqrt(q);
  const double ra = __shfl_sync(0xffffffffu, rq, 1), rn = __shfl_sync(0xffffffffu, rq, 0);
  const double nrm = tot * rn, f = fma(nrm, ra, 1.0);  // v_0 = alpha (1 + |x| / |alpha|)
  double2* v = sh.v[i & 1];
  for (int x = lane; x < r; x += 32)
    v[x] = x > 0 ? col[x * n] : has_al ? make_double2(al.x * f, al.y * f) : make_double2(nrm, 0.0);
  if (lane == 0) {
    sh.al = al; sh.a2 = has_al ? a2 : 0.0; sh.ra = ra; sh.tot = tot; sh.nrm = nrm;
    sh.reflect = reflect;
  }
}

__device__ void tridiagonalise(SmallShared& sh, int n) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double2* A = sh.A;
  double2 phase = make_double2(1.0, 0.0);              // thread 32's running product
  if (tid == 32) sh.ph[0] = phase;
  if (warp == 0 && n > 1) householder_chain(sh, n, 0);
  __syncthreads();
  for (int i = 0; i + 1 < n; ++i) {
    const int r = n - 1 - i;
    const bool reflect = sh.reflect;
    if (tid == 32) {                                   // off-diagonal and its phase, -u or u
      const double al_abs = sh.a2 * sh.ra;
      double2 u = make_double2(1.0, 0.0);
      if (sh.a2 != 0.0) u = make_double2(sh.al.x * sh.ra, sh.al.y * sh.ra);
      if (reflect) u = make_double2(-u.x, -u.y);
      sh.e[i] = reflect ? sh.nrm : al_abs;
      phase = cmul(phase, u);
      sh.ph[i + 1] = phase;
    }
    if (tid == kSmallThreads - 1)
      sh.tau[i] = reflect ? 1.0 / fma(sh.a2 * sh.ra, sh.nrm, sh.tot) : 0.0;
    const double2* v = sh.v[i & 1];
    if (reflect) {
      // p = A v, tpr threads a row: the warps in use spread evenly over the SM's quarters
      const int tpr = (r <= 16 || (r > 32 && r <= 48)) ? 8 : 4;
      const int row = tid / tpr, part = tid & (tpr - 1);
      if ((warp << 5) < r * tpr) {
        double2 s = make_double2(0.0, 0.0);
        if (row < r) {
          const double2* a = A + (i + 1 + row) * n + i + 1;
          for (int y = part; y < r; y += tpr) s = cmac(a[y], v[y], s);
        }
        for (int o = tpr >> 1; o; o >>= 1) {
          s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
          s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (row < r && part == 0) sh.p[row] = s;
      }
      __syncthreads();
      // w = tau p - K v, K = tau^2 / 2 (v^H p): each of three warps sums K for itself
      if (warp < 3 && (warp << 5) < r) {
        double k = 0.0;
        for (int x = lane; x < r; x += 32) {
          const double2 c = v[x], b = sh.p[x];
          k = fma(c.x, b.x, fma(c.y, b.y, k));
        }
        for (int o = 16; o; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
        const double tau = sh.tau[i];
        k *= 0.5 * tau * tau;
        if (tid < r) {
          const double2 c = v[tid], b = sh.p[tid];
          sh.wv[tid] = make_double2(fma(-k, c.x, tau * b.x), fma(-k, c.y, tau * b.y));
        }
      }
      __syncthreads();
      // A -= v w^H + w v^H on the lower triangle, mirrored; v into its column
      const auto update = [&](int x, int y) {
        const double2 vx = v[x], vy = v[y], wx = sh.wv[x], wy = sh.wv[y];
        double2 c = A[(i + 1 + x) * n + i + 1 + y];
        c.x = fma(-vx.x, wy.x, fma(-vx.y, wy.y, fma(-wx.x, vy.x, fma(-wx.y, vy.y, c.x))));
        c.y = fma(vx.x, wy.y, fma(-vx.y, wy.x, fma(wx.x, vy.y, fma(-wx.y, vy.x, c.y))));
        if (x == y) c.y = 0.0;
        A[(i + 1 + x) * n + i + 1 + y] = c;
        if (y > 0) A[(i + 1 + y) * n + i + 1 + x] = make_double2(c.x, -c.y);
      };
      if (warp == 0) {
        for (int x = lane; x < r; x += 32) update(x, 0);
        __syncwarp();
      } else {
        // small triangles stay off warp 0's quarter of the SM
        const int cnt = r * (r - 1) / 2;
        const bool aside = cnt <= 384;
        const int first = aside ? ((warp >> 2) * 3 + (warp & 3) - 1) * 32 + lane : tid - 32;
        const int stride = aside ? 384 : kSmallThreads - 32;
        if (!aside || (warp & 3) != 0)
          for (int e = first; e < cnt; e += stride) {
            int x, y;
            fold(e, r - 1, x, y);
            update(x + 1, y + 1);
          }
        for (int x = tid - 32; x < r; x += kSmallThreads - 32) A[(i + 1 + x) * n + i] = v[x];
      }
    } else {
      __syncthreads();                                 // the chain overwrites what was just read
    }
    if (warp == 0 && i + 2 < n) householder_chain(sh, n, i + 1);
    __syncthreads();
  }
  for (int i = tid; i < n; i += kSmallThreads) sh.d[i] = A[i * n + i].x;
  __syncthreads();
}

// ---- eigenvalues of T -----------------------------------------------------------------------
struct DF { float h, l; };
__device__ __forceinline__ DF df_norm(float s, float e) {   // |s| >= |e|
  DF o;
  o.h = s + e;
  o.l = e - (o.h - s);
  return o;
}
__device__ __forceinline__ DF df_sub(DF a, DF b) {
  const float s = a.h - b.h;
  const float bb = s - a.h;
  const float e = (a.h - (s - bb)) - (b.h + bb);
  return df_norm(s, e + (a.l - b.l));
}
__device__ __forceinline__ DF df_div(DF a, DF b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b.h));
  const float t = a.h * r;
  const float p = t * b.h, err = fmaf(t, b.h, -p);
  const float rem = ((a.h - p) - err) + fmaf(-t, b.l, a.l);
  return df_norm(t, rem * r);
}
__device__ __forceinline__ DF df_of(double x) {
  DF o;
  o.h = (float)x;
  o.l = (float)(x - (double)o.h);
  return o;
}
// x 2^-55 as a float pair
__device__ __forceinline__ DF df_fixed(long long x) {
  const float h = __ll2float_rn(x);
  const float l = __ll2float_rn(x - __float2ll_rn(h));
  const float s = __int_as_float((127 - 55) << 23);
  return DF{h * s, l * s};
}

// Scales T to |T| < 3/4 by a power of two (returned; 0: T is zero, -1: not finite) and writes the
// k smallest eigenvalues of scaled T to lam, within 2^-46 or so. Half-warp j owns eigenvalue j:
// its lanes count the eigenvalues below 15 points (Sturm sequence q_i = (d_i - x) - e_{i-1}^2 /
// q_{i-1}), 4 bits a pass: 5 passes in FP32, then 9 in double-float arithmetic.
__device__ double bisect(SmallShared& sh, int n, int k) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) sh.flag = 0;
  __syncthreads();
  for (int i = tid; i < n; i += kSmallThreads) {
    int m = (int)(__double2hiint(sh.d[i]) & 0x7fffffff) >> 20;
    if (i + 1 < n) m = max(m, (int)(__double2hiint(sh.e[i]) & 0x7fffffff) >> 20);
    atomicMax(&sh.flag, m);
  }
  __syncthreads();
  const int maxe = sh.flag;                            // |entries| < 2^(maxe - 1022)
  __syncthreads();
  if (maxe == 2047) return -1.0;
  if (maxe == 0) return 0.0;
  const int se = min(2046, 1023 + 1022 - maxe - 2);    // biased exponent of the scale
  const double scale = __hiloint2double(max(1, se) << 20, 0);
  for (int i = tid; i < n; i += kSmallThreads) {
    const double dv = sh.d[i] * scale, ev = i + 1 < n ? sh.e[i] * scale : 0.0;
    const DF a = df_of(dv), b = df_of(ev * ev);
    sh.d[i] = dv;
    sh.e[i] = ev;
    sh.t[i] = make_float4(a.h, a.l, b.h, b.l);
  }
  __syncthreads();
  const int j = tid >> 4, t = tid & 15;
  if (j < k) {
    const unsigned mask = 0xffffu << (lane & 16);
    const auto narrow = [&](long long& lo, long long step, int below) {
      const unsigned b = __ballot_sync(mask, t < 15 && below <= j);
      lo += step * __popc(b & mask);
    };
    long long lo = -(1LL << 55), step = 1LL << 52;
    for (int pass = 0; pass < 5; ++pass, step >>= 4) {   // the leading bits in FP32
      const float x = df_fixed(lo + step * (t + 1)).h;
      int below = 0;
      float c = 0.f;                                   // e_{i-1}^2 / q_{i-1}
      for (int i = 0; i < n; ++i) {
        const float4 r = sh.t[i];
        float q = (r.x - x) - c;
        if (fabsf(q) < 1e-20f) q = -1e-20f;
        below += q < 0.f;
        float rq;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rq) : "f"(q));
        c = r.z * rq;
      }
      narrow(lo, step, below);
    }
    // FP32 counts belong to a matrix within 2^-22 of T: widen the interval (2^-19 now) 16 times
    step <<= 4;
    lo -= 7 * step + (step >> 1);
    for (int pass = 0; pass < 9; ++pass, step >>= 4) {
      const DF x = df_fixed(lo + step * (t + 1));
      int below = 0;
      DF c{0.f, 0.f};
      for (int i = 0; i < n; ++i) {
        const float4 r = sh.t[i];
        DF q = df_sub(df_sub(DF{r.x, r.y}, x), c);
        if (fabsf(q.h) < 1e-30f) q = DF{-1e-30f, 0.f};
        below += q.h < 0.f;
        c = df_div(DF{r.z, r.w}, q);
      }
      narrow(lo, step, below);
    }
    if (t == 0) sh.lam[j] = lo + 8 * step;             // (step is a sixteenth of the last one)
  }
  __syncthreads();
  return scale;
}

// ---- eigenvectors of T ----------------------------------------------------------------------
// 1 / x for 1e-30 < |x| < 1e30: Newton steps from the FP32 reciprocal.
__device__ __forceinline__ double recip(double x) {
  double r = (double)(1.f / (float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// One warp, lane j: T - lam_j = P L U (partial pivoting; 1/U_ii, two superdiagonals and the
// multipliers kept, row exchanges in two words), then solves with a right-hand side that is
// pseudo-random the first time, normalised. z: n x k, lane j's vector in column j.
struct LuRows { unsigned long long lo, hi; };
__device__ __forceinline__ bool row_swapped(const LuRows& s, int i) {
  return ((i < 64 ? s.lo >> i : s.hi >> (i - 64)) & 1ull) != 0;
}
__device__ LuRows factor(const SmallShared& sh, double* lu, int n, int k, int j, double lam) {
  double* rp = lu;
  double *u1 = lu + kLu, *u2 = lu + 2 * kLu, *ml = lu + 3 * kLu;
  LuRows sw{0, 0};
  constexpr double tiny = 1e-17;
  double p = sh.d[0] - lam, q = n > 1 ? sh.e[0] : 0.0;
  for (int i = 0; i + 1 < n; ++i) {
    const double b = sh.e[i], dn = sh.d[i + 1] - lam, en = sh.e[i + 1];
    const bool swap = fabs(b) > fabs(p);
    double piv = swap ? b : p;
    if (!(fabs(piv) > tiny)) piv = piv < 0.0 ? -tiny : tiny;
    const double r = recip(piv);
    const double m = (swap ? p : b) * r;
    rp[i * k + j] = r;
    u1[i * k + j] = swap ? dn : q;
    u2[i * k + j] = swap ? en : 0.0;
    ml[i * k + j] = m;
    if (swap) {
      if (i < 64) sw.lo |= 1ull << i; else sw.hi |= 1ull << (i - 64);
      p = fma(-m, dn, q);
      q = -m * en;
    } else {
      p = fma(-m, q, dn);
      q = en;
    }
  }
  if (!(fabs(p) > tiny)) p = p < 0.0 ? -tiny : tiny;
  rp[(n - 1) * k + j] = recip(p);
  return sw;
}
__device__ void solve(const double* lu, double* z, int n, int k, int j, LuRows sw) {
  const double* rp = lu;
  const double *u1 = lu + kLu, *u2 = lu + 2 * kLu, *ml = lu + 3 * kLu;
  double y = z[j];
  for (int i = 0; i + 1 < n; ++i) {
    const double nx = z[(i + 1) * k + j];
    const bool s = row_swapped(sw, i);
    const double top = s ? nx : y, bot = s ? y : nx;
    z[i * k + j] = top;
    y = fma(-ml[i * k + j], top, bot);
  }
  double x2 = 0.0, x1 = y * rp[(n - 1) * k + j], s2 = x1 * x1;
  z[(n - 1) * k + j] = x1;
  for (int i = n - 2; i >= 0; --i) {
    const double x = fma(-u1[i * k + j], x1, fma(-u2[i * k + j], x2, z[i * k + j])) * rp[i * k + j];
    z[i * k + j] = x;
    s2 = fma(x, x, s2);
    x2 = x1;
    x1 = x;
  }
  const double f = rsqrt(s2);
  for (int i = 0; i < n; ++i) z[i * k + j] *= f;
}

// Modified Gram-Schmidt, twice, on the columns of z (n x k): for clusters of eigenvalues, where
// inverse iteration alone returns nearly parallel vectors. c: k doubles.
__device__ void orthonormalise_mgs(double* z, double* c, int n, int k) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int pass = 0; pass < 2; ++pass)
    for (int l = 0; l < k; ++l) {
      for (int j = l + warp; j < k; j += kSmallThreads / 32) {
        double s = 0.0;
        for (int i = lane; i < n; i += 32) s = fma(z[i * k + l], z[i * k + j], s);
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) c[j] = s;
      }
      __syncthreads();
      const double f = c[l] > 0.0 ? rsqrt(c[l]) : 0.0;
      for (int j = l + warp; j < k; j += kSmallThreads / 32)
        for (int i = lane; i < n; i += 32) {
          const double zl = z[i * k + l];
          if (j > l) z[i * k + j] = fma(-c[j] * f * f, zl, z[i * k + j]);
        }
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += kSmallThreads) z[i * k + l] *= f;
      __syncthreads();
    }
}

// E = z^T z - I (k x k) and its largest entry (in units of float bits: sh.dev).
__device__ void gram_defect(SmallShared& sh, const double* z, double* E, int n, int k) {
  if (threadIdx.x == 0) sh.dev = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < k * (k + 1) / 2; e += kSmallThreads) {
    int a, b;
    fold(e, k, a, b);
    double s = a == b ? -1.0 : 0.0;
    for (int i = 0; i < n; ++i) s = fma(z[i * k + a], z[i * k + b], s);
    E[a * k + b] = s;
    E[b * k + a] = s;
    atomicMax(&sh.dev, __float_as_int(fabsf((float)s)));
  }
  __syncthreads();
}

// The k <= kMaxBlock smallest eigenpairs of the Hermitian n x n matrix in sh.A (row-major, leading
// dimension n): sh.w ascending, eigenvectors as the columns of sh.B (row-major, leading dimension
// k), orthonormal to FP64 rounding. sh.A and sh.V are overwritten.
__device__ void herm_eig(SmallShared& sh, int n, int k) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int e = tid; e < n * (n + 1) / 2; e += kSmallThreads) {   // A = (A + A^H) / 2
    int i, j;
    fold(e, n, i, j);
    const double2 a = sh.A[i * n + j], c = sh.A[j * n + i];
    const double2 m = make_double2(0.5 * (a.x + c.x), i == j ? 0.0 : 0.5 * (a.y - c.y));
    sh.A[i * n + j] = m;
    sh.A[j * n + i] = make_double2(m.x, -m.y);
  }
  __syncthreads();
  tridiagonalise(sh, n);
  const double scale = bisect(sh, n, k);
  if (scale <= 0.0) {                                  // zero, or not finite
    const double bad = scale < 0.0 ? nan("") : 0.0;
    for (int e = tid; e < n * k; e += kSmallThreads)
      sh.B[e] = make_double2(e / k == e % k ? 1.0 + bad : bad, bad);
    for (int j = tid; j < k; j += kSmallThreads) sh.w[j] = bad;
    __syncthreads();
    return;
  }
  double* lu = reinterpret_cast<double*>(sh.V);
  double *z = lu + 4 * kLu, *E = lu + 5 * kLu, *c = E + kMaxBlock * kMaxBlock;
  static_assert(5 * kLu + kMaxBlock * kMaxBlock + kMaxBlock <= 2 * kMaxSmall * kMaxSmall, "work");
  LuRows sw{0, 0};
  if (warp == 0) {
    // close eigenvalues are kept 2^-47 apart, so that their solves differ
    constexpr long long kApart = 1LL << 8;
    const long long raw = lane < k ? sh.lam[lane] : (1LL << 56) + (long long)lane * (1LL << 50);
    const long long prev = __shfl_up_sync(0xffffffffu, raw, 1);
    long long a = raw - lane * kApart;
    for (int o = 1; o < 32; o <<= 1) {
      const long long b = __shfl_up_sync(0xffffffffu, a, o);
      if (lane >= o) a = max(a, b);
    }
    const double lam = (double)(a + lane * kApart) * (1.0 / 36028797018963968.0);
    const bool close = lane > 0 && lane < k && raw - prev < (1LL << 25);
    const int any = __any_sync(0xffffffffu, close);
    if (lane == 0) sh.flag = any;
    if (lane < k) {
      for (int i = 0; i < n; ++i) {                    // (mixed by xxHash32's multipliers and shifts)
        unsigned h = (unsigned)(i * 2654435761u) ^ ((unsigned)lane * 2246822519u + 374761393u);
        h ^= h >> 15; h *= 2246822519u; h ^= h >> 13; h *= 3266489917u; h ^= h >> 16;
        z[i * k + lane] = (double)((float)(int)h * 4.656612873e-10f);
      }
      sw = factor(sh, lu, n, k, lane, lam);
      solve(lu, z, n, k, lane, sw);
    }
  }
  __syncthreads();
  const bool clustered = sh.flag != 0;
  __syncthreads();
  if (clustered) orthonormalise_mgs(z, c, n, k);
  if (warp == 0 && lane < k) solve(lu, z, n, k, lane, sw);
  __syncthreads();
  if (clustered) orthonormalise_mgs(z, c, n, k);
  for (int rep = 0; rep < 3; ++rep) {
    gram_defect(sh, z, E, n, k);
    const float dev = __int_as_float(sh.dev);
    if (rep > 0 && dev < 1e-14f) break;
    if (!(dev < 1e-3f)) orthonormalise_mgs(z, c, n, k);
    else if (dev > 1e-16f) {
      // one Newton-Schulz step z (I - E / 2): the defect squares
      double corr[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + u * kSmallThreads;
        corr[u] = 0.0;
        if (e < n * k) {
          const int i = e / k, j = e - i * k;
          for (int l = 0; l < k; ++l) corr[u] = fma(z[i * k + l], E[l * k + j], corr[u]);
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + u * kSmallThreads;
        if (e < n * k) z[e] = fma(-0.5, corr[u], z[e]);
      }
      __syncthreads();
    }
    if (dev < 1e-8f) break;                            // the defect left is below 1e-16
  }
  static_assert(kLu <= 4 * kSmallThreads, "correction registers");
  // Rayleigh quotients and back-transformation: four lanes a vector (part), eight vectors a warp,
  // so that a shared-memory phase reads eight neighbouring columns
  const int j = warp * 8 + (lane & 7), part = lane >> 3;
  if (warp * 8 < k) {
    const bool live = j < k;
    double q = 0.0;
    for (int i = part; live && i < n; i += 4) {
      const double zi = z[i * k + j];
      double s = sh.d[i] * zi;
      if (i + 1 < n) s = fma(2.0 * sh.e[i], z[(i + 1) * k + j], s);
      q = fma(s, zi, q);
    }
    q += __shfl_xor_sync(0xffffffffu, q, 8);
    q += __shfl_xor_sync(0xffffffffu, q, 16);
    if (live && part == 0) sh.w[j] = q / scale;
    // rows part, part + 4, ... of the vector in registers, three at a time behind a branch that the
    // whole warp takes: an FP64 instruction that is only predicated off still costs its 64 cycles
    constexpr int kPer = kMaxSmall / 4, kStep = 3;
    double2 y[kPer];
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int i = part + 4 * t;
      const double zi = live && i < n ? z[i * k + j] : 0.0;
      y[t] = i < n ? make_double2(sh.ph[i].x * zi, sh.ph[i].y * zi) : make_double2(0.0, 0.0);
    }
    for (int c0 = n - 3; c0 >= 0; --c0) {              // the last column has no reflector
      const double tau = sh.tau[c0];
      if (tau == 0.0) continue;
      const double2* a = sh.A + c0;
      double2 s = make_double2(0.0, 0.0);
      const auto entry = [&](int i) {                  // 0 outside the reflector
        const double2 v = a[min(i, n - 1) * n];
        const bool in = i > c0 && i < n;
        return make_double2(in ? v.x : 0.0, in ? v.y : 0.0);
      };
#pragma unroll
      for (int t0 = 0; t0 < kPer; t0 += kStep)
        if (4 * (t0 + kStep) > c0 + 1 && 4 * t0 < n) {
#pragma unroll
          for (int t = t0; t < t0 + kStep; ++t) s = cmac_conj(entry(part + 4 * t), y[t], s);
        }
      s.x += __shfl_xor_sync(0xffffffffu, s.x, 8);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, 8);
      s.x += __shfl_xor_sync(0xffffffffu, s.x, 16);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, 16);
      s = make_double2(-tau * s.x, -tau * s.y);
#pragma unroll
      for (int t0 = 0; t0 < kPer; t0 += kStep)
        if (4 * (t0 + kStep) > c0 + 1 && 4 * t0 < n) {
#pragma unroll
          for (int t = t0; t < t0 + kStep; ++t) y[t] = cmac(entry(part + 4 * t), s, y[t]);
        }
    }
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int i = part + 4 * t;
      if (live && i < n) sh.B[i * k + j] = y[t];
    }
  }
  __syncthreads();
}

// T = M^{-1/2} for a Hermitian b x b matrix M = I + E on the columns with on[j], zero in the
// others, when E is small enough for its series (entries below 1e-6: 0.27 |E|^4 < 1e-18), which
// holds for blocks that were orthonormalised once; false otherwise. M must be zero outside the
// columns that are on. W: b x b work.
__device__ bool inv_sqrt_series(SmallShared& sh, const double2* M, double2* T, double2* W, int b,
                                const double* on) {
  if (threadIdx.x == 0) sh.dev = 0;
  __syncthreads();
  const auto entry = [&](int e) {                      // E
    double2 v = M[e];
    if (e / b == e % b && on[e / b] > 0.0) v.x -= 1.0;
    return v;
  };
  for (int e = threadIdx.x; e < b * b; e += kSmallThreads) {
    const double2 v = entry(e);
    const float m = fmaxf(fabsf((float)v.x), fabsf((float)v.y));
    atomicMax(&sh.dev, m == m ? __float_as_int(m) : 0x7f800000);
  }
  __syncthreads();
  const float dev = __int_as_float(sh.dev);
  if (!(dev < 1e-6f)) { __syncthreads(); return false; }
  const bool second = dev > 1e-9f;                     // else |E|^2 is below 1e-16
  if (second) {
    for (int e = threadIdx.x; e < b * b; e += kSmallThreads) {
      const int i = e / b, j = e - i * b;
      double2 s = make_double2(0.0, 0.0);
      for (int l = 0; l < b; ++l) s = cmac(entry(i * b + l), entry(l * b + j), s);
      W[e] = s;
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < b * b; e += kSmallThreads) {
    const int i = e / b, j = e - i * b;
    const double2 v = entry(e);
    double2 t = make_double2((i == j && on[i] > 0.0 ? 1.0 : 0.0) - 0.5 * v.x, -0.5 * v.y);
    if (second) {
      double2 s = make_double2(0.0, 0.0);              // E^3
      for (int l = 0; l < b; ++l) s = cmac(entry(i * b + l), W[l * b + j], s);
      t.x += 0.375 * W[e].x - 0.3125 * s.x;
      t.y += 0.375 * W[e].y - 0.3125 * s.y;
    }
    T[e] = t;
  }
  __syncthreads();
  return true;
}

// T (b x b) for the Cholesky factorisation with diagonal pivoting of a Hermitian matrix M (full,
// overwritten): T^H M T = I on the columns kept. The largest pivot left comes next, so that columns
// with a pivot not above drop, which depend on those before them, come last: their column of T is
// zero and sh.keep 0. Without pivoting small pivots arise early and amplify what follows: columns of
// a nearly dependent block came out 8e-9 off the space they had been projected out of, where the
// eigenvectors of M leave 6e-12 and this order 2e-11 (24 powers of x on [0, 1], drop 1e-14 of the
// largest eigenvalue). T is built along with the factor, as Gram-Schmidt on the unit vectors: 24
// steps of one square root and one update each. b <= 32.
__device__ void cholesky_transform(SmallShared& sh, double2* M, double2* T, int b, double drop) {
  const int tid = threadIdx.x;
  int* perm = sh.idx;                                  // the order of the pivots
  for (int e = tid; e < b * b; e += kSmallThreads) T[e] = make_double2(e / b == e % b ? 1.0 : 0.0, 0.0);
  for (int k = tid; k < b; k += kSmallThreads) perm[k] = k;
  __syncthreads();
  for (int k = 0; k < b; ++k) {
    if (tid < 32) {
      // by the high words, as integers: close enough for an order
      const int pos = k + tid;
      const int c = pos < b ? perm[pos] : 0;
      const int key = pos < b ? max(0, __double2hiint(M[c * b + c].x)) : -1;
      const int best = __ffs(__ballot_sync(0xffffffffu, key == __reduce_max_sync(0xffffffffu, key))) - 1;
      if (tid == best) {
        const double piv = M[c * b + c].x;
        const bool ok = piv > drop;
        const double r = ok ? rsqrt(piv) : 0.0;
        sh.scale[c] = r;
        sh.r2 = r * r;
        sh.keep[c] = ok;
        perm[pos] = perm[k];
        perm[k] = c;
      }
    }
    __syncthreads();
    const int ck = perm[k];
    if (sh.keep[ck]) {
      const double r2 = sh.r2;
      const int rest = b - 1 - k, tri = rest * (rest + 1) / 2;
      for (int e = tid; e < tri + (k + 1) * rest; e += kSmallThreads) {
        int i, j;
        if (e < tri) {                                 // M_ij -= conj(M_ki) M_kj / M_kk, mirrored
          fold(e, rest, j, i);
          i += k + 1; j += k + 1;
        } else {                                       // T_ij -= T_ik M_kj / M_kk
          i = (e - tri) / rest;
          j = k + 1 + (e - tri) - i * rest;
        }
        const int ci = perm[i], cj = perm[j];
        const double2 m = M[ck * b + cj];
        const double2 g = make_double2(-m.x * r2, -m.y * r2);
        if (e < tri) {
          const double2 u = cmac_conj(M[ck * b + ci], g, M[ci * b + cj]);
          M[ci * b + cj] = u;
          if (ci != cj) M[cj * b + ci] = make_double2(u.x, -u.y);
        } else {
          T[ci * b + cj] = cmac(T[ci * b + ck], g, T[ci * b + cj]);
        }
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < b * b; e += kSmallThreads) {
    const double f = sh.scale[e % b];
    T[e] = make_double2(T[e].x * f, T[e].y * f);
  }
  __syncthreads();
}

// Orthonormalising transform of a block Y from its Gram matrix: Y T is orthonormal on the columns
// that are kept; dependent columns of T are zero with their mask entry 0. With D =
// diag(G)^{-1/2}: T = D (D G D)^{-1/2} from its series when the block is orthonormal up to 1e-6
// already, else from the pivoted Cholesky factorisation of D G D, which costs a fraction of the
// eigenproblem of SVQB (41 against 617 us at b = 24, 10 against 78 at 4). Dependent are columns whose pivot is at most drop times a bound of the
// largest eigenvalue (the largest absolute row sum), which takes the place of SVQB's test of the
// eigenvalues. As there, a second application to the result removes the rounding that small pivots
// amplify.
__global__ void __launch_bounds__(kSmallThreads, 1)
svqb_kernel(Batch bt, const double2* G, int b, double drop, double2* T, int* mask, int* status) {
  extern __shared__ __align__(16) unsigned char raw[];
  SmallShared& sh = *reinterpret_cast<SmallShared*>(raw);
  const int tid = threadIdx.x;
  const int prob = blockIdx.x;
  if (bt.active && !bt.active[prob]) return;
  G += (size_t)prob * kCapG;
  T += (size_t)prob * kCapT;
  mask += (size_t)prob * kMaxBlock;
  if (status) status += prob;
  double* D = sh.d;
  for (int i = tid; i < b; i += kSmallThreads) {
    const double g = G[i * b + i].x;
    D[i] = g > 1e-300 ? 1.0 / sqrt(g) : 0.0;
  }
  __syncthreads();
  for (int e = tid; e < b * b; e += kSmallThreads) {
    const double di = D[e / b], dj = D[e % b];
    const double2 g = G[e];
    const bool on = di > 0.0 && dj > 0.0;
    sh.A[e] = make_double2(on ? g.x * di * dj : 0.0, on ? g.y * di * dj : 0.0);
  }
  __syncthreads();
  const bool series = inv_sqrt_series(sh, sh.A, sh.B, sh.V, b, D);
  if (!series) {
    if (tid == 0) sh.flag = 0;
    __syncthreads();
    for (int i = tid >> 5; i < b; i += kSmallThreads / 32) {
      const int j = tid & 31;
      const double2 v = j < b ? sh.A[i * b + j] : make_double2(0.0, 0.0);
      float r = fabsf((float)v.x) + fabsf((float)v.y);
      for (int o = 16; o; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
      if (j == 0 && r < 1e3f) atomicMax(&sh.flag, __float_as_int(r));
    }
    __syncthreads();
    cholesky_transform(sh, sh.A, sh.B, b, drop * (double)__int_as_float(sh.flag));
  }
  for (int e = tid; e < b * b; e += kSmallThreads) {
    const double f = D[e / b];
    T[e] = make_double2(sh.B[e].x * f, sh.B[e].y * f);
  }
  for (int k = tid; k < b; k += kSmallThreads) mask[k] = (series ? D[k] > 0.0 : sh.keep[k] != 0) ? 1 : 0;
  if (tid == 0 && status) *status = 0;
}

// G (b x b) = X^H Y for m x b matrices.
__device__ void small_gram(const double2* X, const double2* Y, double2* G, int m, int b) {
  for (int e = threadIdx.x; e < b * b; e += kSmallThreads) {
    const int r = e / b, c = e - r * b;
    double2 s = make_double2(0, 0);
    for (int i = 0; i < m; ++i) s = cmac_conj(X[i * b + r], Y[i * b + c], s);
    G[e] = s;
  }
  __syncthreads();
}
// The same for Y = X: one triangle, mirrored.
__device__ void small_gram_herm(const double2* Y, double2* G, int m, int b) {
  for (int e = threadIdx.x; e < b * (b + 1) / 2; e += kSmallThreads) {
    int r, c;
    fold(e, b, r, c);
    double2 s = make_double2(0, 0);
    for (int i = 0; i < m; ++i) s = cmac_conj(Y[i * b + r], Y[i * b + c], s);
    if (r == c) s.y = 0.0;
    G[r * b + c] = s;
    G[c * b + r] = make_double2(s.x, -s.y);
  }
  __syncthreads();
}
// Y -= X G (m x b, in place).
__device__ void small_subtract(const double2* X, const double2* G, double2* Y, int m, int b) {
  for (int e = threadIdx.x; e < m * b; e += kSmallThreads) {
    const int i = e / b, c = e - i * b;
    double2 s = make_double2(0, 0);
    for (int r = 0; r < b; ++r) s = cmac(X[i * b + r], G[r * b + c], s);
    const double2 y = Y[e];
    Y[e] = make_double2(y.x - s.x, y.y - s.y);
  }
  __syncthreads();
}
// Z = Y T (m x b; Z is not Y).
__device__ void small_multiply(const double2* Y, const double2* T, double2* Z, int m, int b) {
  for (int e = threadIdx.x; e < m * b; e += kSmallThreads) {
    const int i = e / b, c = e - i * b;
    double2 s = make_double2(0, 0);
    for (int r = 0; r < b; ++r) s = cmac(Y[i * b + r], T[r * b + c], s);
    Z[e] = s;
  }
  __syncthreads();
}

// First round of the P coefficients: Y = the columns in sh.B (m x b, rows below x_rows zero) minus
// their projection on the orthonormal X in sh.A, scaled to unit norm and orthonormalised by
// modified Gram-Schmidt; back to sh.B. Columns of norm up to 1e-12, and columns within 1e-7 of the
// span of those before them, become zero with sh.keep 0. In FP64: double-float arithmetic took
// 105 us less at 72 x 24, but left the span 1e-14 to 1e-13 off (now 4e-16).
__device__ void p_columns_near(SmallShared& sh, int m, int b, int x_rows) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kWarps = kSmallThreads / 32;
  const int ld = m | 1;                                // column-major, odd stride: no conflicts
  double2* X = sh.V;
  double2* Y = X + kMaxBlock * (kMaxSmall + 1);
  double2* G = Y + kMaxBlock * (kMaxSmall + 1);
  static_assert(2 * kMaxBlock * (kMaxSmall + 1) + kMaxBlock * kMaxBlock <= kMaxSmall * kMaxSmall, "work");
  for (int e = tid; e < m * b; e += kSmallThreads) {
    const int i = e / b, c = e - i * b;
    X[c * ld + i] = sh.A[e];
    Y[c * ld + i] = sh.B[e];
  }
  __syncthreads();
  // G = X^H Y: Hermitian, since Y is X with rows zeroed
  for (int e = tid; e < b * (b + 1) / 2; e += kSmallThreads) {
    int r, c;
    fold(e, b, r, c);
    double2 s = make_double2(0.0, 0.0);
    for (int i = x_rows; i < m; ++i) s = cmac_conj(X[r * ld + i], Y[c * ld + i], s);
    if (r == c) s.y = 0.0;
    G[r * b + c] = s;
    G[c * b + r] = make_double2(s.x, -s.y);
  }
  __syncthreads();
  for (int e = tid; e < m * b; e += kSmallThreads) {
    const int c = e / m, i = e - c * m;
    double2 s = Y[c * ld + i];
    for (int r = 0; r < b; ++r) {
      const double2 g = G[r * b + c];
      s = cmac(X[r * ld + i], make_double2(-g.x, -g.y), s);
    }
    Y[c * ld + i] = s;
  }
  __syncthreads();
  // eight lanes a column, four columns a warp: an FP64 instruction costs a warp the same with any
  // number of lanes, and a sum over 32 lanes would take as many of them as the products
  const int part = lane & 7, sub = lane >> 3;
  const auto dots = [&](const double2* a, int j, bool live) {   // a^H y_j in the column's lanes
    double2 s = make_double2(0.0, 0.0);
    for (int i = part; live && i < m; i += 8) s = cmac_conj(a[i], Y[j * ld + i], s);
    for (int o = 4; o; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    return s;
  };
  for (int c0 = 4 * warp; c0 < b; c0 += 4 * kWarps) {  // unit columns
    const int c = c0 + sub;
    const bool live = c < b;
    const double n2 = dots(Y + min(c, b - 1) * ld, c, live).x;
    const double f = n2 > 1e-24 ? rsqrt(n2) : 0.0;
    for (int i = part; live && i < m; i += 8)
      Y[c * ld + i] = make_double2(Y[c * ld + i].x * f, Y[c * ld + i].y * f);
  }
  __syncthreads();
  for (int l = 0; l < b; ++l) {
    const double2* yl = Y + l * ld;
    for (int j0 = l + 4 * warp; j0 < b; j0 += 4 * kWarps) {
      const int j = j0 + sub;
      const double2 s = dots(yl, j, j < b);
      if (part == 0 && j < b) G[j] = s;
    }
    __syncthreads();
    const double n2 = G[l].x;
    const bool on = n2 > 1e-14;
    const double f = on ? rsqrt(n2) : 0.0, f2 = f * f;
    for (int j = l + 1 + 4 * warp + sub; on && j < b; j += 4 * kWarps) {
      const double2 g = make_double2(-G[j].x * f2, -G[j].y * f2);
      for (int i = part; i < m; i += 8) Y[j * ld + i] = cmac(yl[i], g, Y[j * ld + i]);
    }
    __syncthreads();
    for (int i = tid; i < m; i += kSmallThreads) Y[l * ld + i] = make_double2(yl[i].x * f, yl[i].y * f);
    if (tid == 0) sh.keep[l] = on;
  }
  __syncthreads();
  for (int e = tid; e < m * b; e += kSmallThreads) {
    const int i = e / b, c = e - i * b;
    sh.B[e] = Y[c * ld + i];
  }
  __syncthreads();
}

// Rayleigh-Ritz on the orthonormal basis S (m columns, `mask` marks the active ones):
// eigenpairs of the compacted Hermitian A; theta and Cx (m x b) take the lowest b.
// Cp: Cx with its first x_rows rows zeroed (the W and P parts), orthogonalised against Cx
// and orthonormalised in the coefficient space, so that S Cp is orthonormal and orthogonal
// to S Cx; dependent columns are zero with mask_p = 0.
__global__ void __launch_bounds__(kSmallThreads, 1)
rr_kernel(Batch bt, const double2* Ain, int m, int b, const int* mask, int x_rows,
          double* theta, double2* Cx, double2* Cp, int* mask_p, int* status) {
  extern __shared__ __align__(16) unsigned char raw[];
  SmallShared& sh = *reinterpret_cast<SmallShared*>(raw);
  const int tid = threadIdx.x;
  const int prob = blockIdx.x;
  if (bt.active && !bt.active[prob]) return;
  Ain += (size_t)prob * kCapG;
  mask += (size_t)prob * kMaxSmall;
  theta += (size_t)prob * kMaxBlock;
  Cx += (size_t)prob * kCapC;
  Cp += (size_t)prob * kCapC;
  mask_p += (size_t)prob * kMaxBlock;
  status += prob;
  if (tid < 32) {                                      // indices of the active columns, in order
    int na = 0;
    for (int i0 = 0; i0 < m; i0 += 32) {
      const int i = i0 + tid;
      const bool on = i < m && mask[i];
      const unsigned b = __ballot_sync(0xffffffffu, on);
      if (on) sh.idx[na + __popc(b & ((1u << tid) - 1u))] = i;
      na += __popc(b);
    }
    if (tid == 0) sh.flag = na;
  }
  __syncthreads();
  const int na = sh.flag;
  __syncthreads();
  if (na < b) {
    if (tid == 0) *status = 1;
    return;
  }
  for (int e = tid; e < na * na; e += kSmallThreads) {
    const int i = e / na, j = e % na;
    sh.A[e] = Ain[sh.idx[i] * m + sh.idx[j]];
  }
  __syncthreads();
  herm_eig(sh, na, b);
  // Cx (m x b), kept in shared memory (A) too: rows of inactive columns are zero
  for (int e = tid; e < m * b; e += kSmallThreads) sh.A[e] = make_double2(0, 0);
  for (int k = tid; k < b; k += kSmallThreads) theta[k] = sh.w[k];
  __syncthreads();
  for (int e = tid; e < na * b; e += kSmallThreads) sh.A[sh.idx[e / b] * b + e % b] = sh.B[e];
  __syncthreads();
  for (int e = tid; e < m * b; e += kSmallThreads) {
    const double2 c = sh.A[e];
    Cx[e] = c;
    sh.B[e] = (e / b) < x_rows ? make_double2(0, 0) : c;
  }
  __syncthreads();
  // Cp in two rounds of (orthogonalise against Cx, then orthonormalise). The first scales the
  // columns to unit norm (down to 1e-12) and orthonormalises them by Gram-Schmidt. The second
  // removes what normalising tiny columns left of Cx in them, and restores orthonormality to
  // rounding: one projection, one Gram matrix and, since the columns are orthonormal to better than
  // 1e-6, a series.
  p_columns_near(sh, m, b, x_rows);
  double2* X = sh.A;
  double2 *M = sh.A + kLu, *T = M + kMaxBlock * kMaxBlock;
  static_assert(kLu + 2 * kMaxBlock * kMaxBlock <= kMaxSmall * kMaxSmall, "work");
  small_gram(X, sh.B, sh.V, m, b);
  small_subtract(X, sh.V, sh.B, m, b);
  small_gram_herm(sh.B, M, m, b);
  for (int k = tid; k < b; k += kSmallThreads) sh.d[k] = sh.keep[k] ? 1.0 : 0.0;
  __syncthreads();
  const bool series = inv_sqrt_series(sh, M, T, sh.V, b, sh.d);
  if (!series) cholesky_transform(sh, M, T, b, 1e-2);
  small_multiply(sh.B, T, Cp, m, b);
  for (int k = tid; k < b; k += kSmallThreads) mask_p[k] = sh.keep[k];
  if (tid == 0) *status = 0;
}

template <typename K>
iwf_status small_smem(K* kernel) {
  static bool done[64] = {};
  int dev = 0;
  IWF_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !done[dev]) {
    IWF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(SmallShared)));
    if (dev >= 0 && dev < 64) done[dev] = true;
  }
  return IWF_OK;
}

}  // namespace

iwf_status svqb_small(const Batch& bt, const double2* G, int b, double drop, double2* T,
                      int* mask, int* status, cudaStream_t s) {
  IWF_TRY(small_smem(svqb_kernel));
  svqb_kernel<<<bt.nprob, kSmallThreads, sizeof(SmallShared), s>>>(bt, G, b, drop, T, mask, status);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

iwf_status rayleigh_ritz_small(const Batch& bt, const double2* A, int m, int b, const int* mask,
                               int x_rows, double* theta, double2* Cx, double2* Cp,
                               int* mask_p, int* status, cudaStream_t s) {
  IWF_TRY(small_smem(rr_kernel));
  rr_kernel<<<bt.nprob, kSmallThreads, sizeof(SmallShared), s>>>(bt, A, m, b, mask, x_rows, theta,
                                                                 Cx, Cp, mask_p, status);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

}  // namespace iwf
