// Block kernels of the eigensolver (declarations and layout conventions in blockops.cuh).
#include <algorithm>
#include <cmath>

#include "blockops.cuh"

namespace iwf {

namespace {

constexpr int kGramRows = 16;      // rows staged per Gram tile
constexpr int kGramTx = 24;        // 24 x 24 threads, 3 x 3 outputs each -> up to 72 x 72
constexpr int kGramThreads = kGramTx * kGramTx;
constexpr int kRedWarps = 8;       // warps that share the slots of a reduction

template <typename T> struct Acc { using type = double; };
template <> struct Acc<float> { using type = float; };

// ---- double-float arithmetic ------------------------------------------------------------
// A double x is carried as an unevaluated sum hi + lo of two floats (hi = x rounded to float,
// lo = the rest rounded to float: 48 significant bits). Products of two such pairs are formed
// with the exact float product error from fma (Dekker); sums keep their rounding error with
// TwoSum (Knuth). FP64 on this GPU runs at 1/62 of the FP32 rate, so a complex multiply-add in
// this form (about 48 FP32 operations) costs about a fifth of its 4 FP64 fmas.
struct DF4 { float rh, rl, ih, il; };              // complex: re (hi, lo), im (hi, lo)

__device__ __forceinline__ DF4 df_split(double2 v) {
  DF4 o;
  split_bits(v.x, o.rh, o.rl);
  split_bits(v.y, o.ih, o.il);
  return o;
}
__device__ __forceinline__ double df_value(float h, float l) { return (double)h + (double)l; }

// G_partial[cta] = sum over this CTA's rows of conj(A_i,a) * B_i,c.
// 24 x 24 threads; each owns a U x V micro-tile (outputs ty + 24u, tx + 24v), so the
// launch picks U = ceil(ma/24), V = ceil(mb/24) and no thread multiplies padding.
// HERM (the product is Hermitian, ma == mb): only the 24 x 24 output blocks u <= v are
// formed; reduce_partials mirrors the others.
template <typename T, int U, int V, bool HERM>
__global__ void __launch_bounds__(kGramThreads)
gram_kernel(Batch bt, BlockList A, BlockList B, int ma, int mb, long long N, double2* partial) {
  static_assert(U > 0 && V > 0 && (!HERM || U == V), "tile");
  using V2 = typename Cplx<T>::type;
  using AT = typename Acc<T>::type;
  const int prob = blockIdx.y;
  if (bt.active && !bt.active[prob]) return;
  const size_t poff = (size_t)prob * bt.pstride;
  for (int i = 0; i < A.nb; ++i) A.p[i] = reinterpret_cast<const V2*>(A.p[i]) + poff;
  for (int i = 0; i < B.nb; ++i) B.p[i] = reinterpret_cast<const V2*>(B.p[i]) + poff;
  __shared__ V2 sa[kGramRows][kMaxSmall + 1];
  __shared__ V2 sb[kGramRows][kMaxSmall + 1];
  const int tx = threadIdx.x % kGramTx, ty = threadIdx.x / kGramTx;
  // running sums across tiles: double for double blocks; for float blocks a float pair
  // (hi, lo) kept with TwoSum, because adding into doubles would put one FP64 addition per
  // output and tile on the slow FP64 pipe
  AT sumr[U][V], sumi[U][V], lor[U][V], loi[U][V];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < V; ++v) { sumr[u][v] = 0; sumi[u][v] = 0; lor[u][v] = 0; loi[u][v] = 0; }
  const long long ntiles = (N + kGramRows - 1) / kGramRows;
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long r0 = t * kGramRows;
    for (int e = threadIdx.x; e < kGramRows * ma; e += blockDim.x) {
      const int k = e / kGramRows, r = e % kGramRows;
      V2 v; v.x = 0; v.y = 0;
      if (r0 + r < N) v = col_ptr<T>(A, k, N)[r0 + r];
      sa[r][k] = v;
    }
    for (int e = threadIdx.x; e < kGramRows * mb; e += blockDim.x) {
      const int k = e / kGramRows, r = e % kGramRows;
      V2 v; v.x = 0; v.y = 0;
      if (r0 + r < N) v = col_ptr<T>(B, k, N)[r0 + r];
      sb[r][k] = v;
    }
    __syncthreads();
    AT accr[U][V], acci[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) { accr[u][v] = 0; acci[u][v] = 0; }
    for (int r = 0; r < kGramRows; ++r) {
      V2 av[U], bv[V];
#pragma unroll
      for (int u = 0; u < U; ++u) av[u] = sa[r][min(ty + kGramTx * u, kMaxSmall)];
#pragma unroll
      for (int v = 0; v < V; ++v) bv[v] = sb[r][min(tx + kGramTx * v, kMaxSmall)];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          if (HERM && u > v) continue;
          // conj(a) * b: re = ax bx + ay by, im = ax by - ay bx
          accr[u][v] = fma((AT)av[u].x, (AT)bv[v].x, accr[u][v]);
          accr[u][v] = fma((AT)av[u].y, (AT)bv[v].y, accr[u][v]);
          acci[u][v] = fma((AT)av[u].x, (AT)bv[v].y, acci[u][v]);
          acci[u][v] = fma(-(AT)av[u].y, (AT)bv[v].x, acci[u][v]);
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < V; ++v) {
        if (HERM && u > v) continue;
        if constexpr (sizeof(AT) == 4) {
          float t, e;
          two_sum(sumr[u][v], accr[u][v], t, e); sumr[u][v] = t; lor[u][v] += e;
          two_sum(sumi[u][v], acci[u][v], t, e); sumi[u][v] = t; loi[u][v] += e;
        } else {
          sumr[u][v] += accr[u][v]; sumi[u][v] += acci[u][v];
        }
      }
    __syncthreads();
  }
  double2* out = partial + ((size_t)prob * gridDim.x + blockIdx.x) * ma * mb;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int a = ty + kGramTx * u, c = tx + kGramTx * v;
      if (a < ma && c < mb && !(HERM && u > v))
        out[a * mb + c] = make_double2((double)sumr[u][v] + (double)lor[u][v],
                                       (double)sumi[u][v] + (double)loi[u][v]);
    }
}

// Double-float variant of gram_kernel for complex-double blocks: the staged rows are split into
// float pairs once, every product and sum runs on the FP32 pipes into one double-float
// accumulator per output (TwoSum keeps each addition exact in the high part), and the CTA's
// total is written as double.
template <int U, int V, bool HERM>
__global__ void __launch_bounds__(kGramThreads)
gram_df_kernel(Batch bt, BlockList A, BlockList B, int ma, int mb, long long N, double2* partial) {
  static_assert(!HERM || U == V, "tile");
  const int prob = blockIdx.y;
  if (bt.active && !bt.active[prob]) return;
  const size_t poff = (size_t)prob * bt.pstride;
  for (int i = 0; i < A.nb; ++i) A.p[i] = reinterpret_cast<const double2*>(A.p[i]) + poff;
  for (int i = 0; i < B.nb; ++i) B.p[i] = reinterpret_cast<const double2*>(B.p[i]) + poff;
  __shared__ DF4 sa[kGramRows][kMaxSmall + 1];
  __shared__ DF4 sb[kGramRows][kMaxSmall + 1];
  const int tx = threadIdx.x % kGramTx, ty = threadIdx.x / kGramTx;
  float srh[U][V], srl[U][V], sih[U][V], sil[U][V];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < V; ++v) { srh[u][v] = srl[u][v] = sih[u][v] = sil[u][v] = 0.f; }
  const long long ntiles = (N + kGramRows - 1) / kGramRows;
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long r0 = t * kGramRows;
    for (int e = threadIdx.x; e < kGramRows * ma; e += blockDim.x) {
      const int k = e / kGramRows, r = e % kGramRows;
      double2 v = make_double2(0.0, 0.0);
      if (r0 + r < N) v = col_ptr<double>(A, k, N)[r0 + r];
      sa[r][k] = df_split(v);
    }
    for (int e = threadIdx.x; e < kGramRows * mb; e += blockDim.x) {
      const int k = e / kGramRows, r = e % kGramRows;
      double2 v = make_double2(0.0, 0.0);
      if (r0 + r < N) v = col_ptr<double>(B, k, N)[r0 + r];
      sb[r][k] = df_split(v);
    }
    __syncthreads();
    for (int r = 0; r < kGramRows; ++r) {
      DF4 av[U], bv[V];
#pragma unroll
      for (int u = 0; u < U; ++u) av[u] = sa[r][min(ty + kGramTx * u, kMaxSmall)];
#pragma unroll
      for (int v = 0; v < V; ++v) bv[v] = sb[r][min(tx + kGramTx * v, kMaxSmall)];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < V; ++v) {
          if (HERM && u > v) continue;
          // conj(a) * b: re = ar br + ai bi, im = ar bi - ai br
          df_mac(srh[u][v], srl[u][v], av[u].rh, av[u].rl, bv[v].rh, bv[v].rl);
          df_mac(srh[u][v], srl[u][v], av[u].ih, av[u].il, bv[v].ih, bv[v].il);
          df_mac(sih[u][v], sil[u][v], av[u].rh, av[u].rl, bv[v].ih, bv[v].il);
          df_mac(sih[u][v], sil[u][v], -av[u].ih, -av[u].il, bv[v].rh, bv[v].rl);
        }
    }
    __syncthreads();
  }
  double2* out = partial + ((size_t)prob * gridDim.x + blockIdx.x) * ma * mb;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int a = ty + kGramTx * u, c = tx + kGramTx * v;
      if (a < ma && c < mb && !(HERM && u > v))
        out[a * mb + c] = make_double2(df_value(srh[u][v], srl[u][v]), df_value(sih[u][v], sil[u][v]));
    }
}

// Sum the per-CTA partials in a fixed order (deterministic); problem blockIdx.y. A CTA takes 32
// entries, its eight warps every eighth slot each: one thread an entry walked 608 slots one FP64
// addition after another (130 us at 72 x 72).
// herm: entries in 24 x 24 blocks below the block diagonal were not formed; they are the
// conjugates of their mirror images (mb = row length).
__global__ void reduce_partials(Batch bt, const double2* partial, int slots, int count,
                                double2* out, bool herm, int mb) {
  const int prob = blockIdx.y;
  if (bt.active && !bt.active[prob]) return;
  __shared__ double2 part[kRedWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  const bool live = e < count;
  int src = live ? e : 0;
  bool conj = false;
  if (herm && live) {
    const int a = e / mb, c = e % mb;
    if (a / kGramTx > c / kGramTx) { src = c * mb + a; conj = true; }
  }
  const double2* pp = partial + (size_t)prob * slots * count;
  double re = 0, im = 0;
  for (int s = warp; s < slots; s += kRedWarps) {
    const double2 v = pp[(size_t)s * count + src];
    re += v.x; im += v.y;
  }
  part[warp][lane] = make_double2(re, im);
  __syncthreads();
  if (warp > 0 || !live) return;
  for (int w = 1; w < kRedWarps; ++w) { re += part[w][lane].x; im += part[w][lane].y; }
  out[(size_t)prob * kCapG + e] = make_double2(re, conj ? -im : im);
}

constexpr int kUpdRows = 16;
constexpr int kUpdThreads = kUpdRows * kMaxBlock;

// out1[:, j] (=|-=) sum_k S[:, k] C1[k, j]; out2 likewise with C2. C row-major m x q.
template <typename T, bool SUB>
__global__ void __launch_bounds__(kUpdThreads)
update_kernel(Batch bt, BlockList S, int m, long long N, const double2* C1, const double2* C2,
              int cstride, int q, typename Cplx<T>::type* out1, typename Cplx<T>::type* out2) {
  using V2 = typename Cplx<T>::type;
  using AT = typename Acc<T>::type;
  const int prob = blockIdx.y;
  if (bt.active && !bt.active[prob]) return;
  const size_t poff = (size_t)prob * bt.pstride;
  for (int i = 0; i < S.nb; ++i) S.p[i] = reinterpret_cast<const V2*>(S.p[i]) + poff;
  out1 += poff;
  if (out2) out2 += poff;
  C1 += (size_t)prob * cstride;
  if (C2) C2 += (size_t)prob * cstride;
  extern __shared__ __align__(16) unsigned char upd_raw[];
  using C2T = typename Cplx<AT>::type;            // coefficients in the arithmetic type
  C2T* sc1 = reinterpret_cast<C2T*>(upd_raw);
  C2T* sc2 = sc1 + kMaxSmall * kMaxBlock;
  constexpr int rows = kUpdRows;                  // one thread per (row, j)
  __shared__ V2 ss[rows][kMaxSmall + 1];
  for (int e = threadIdx.x; e < m * q; e += blockDim.x) {
    C2T c; c.x = (AT)C1[e].x; c.y = (AT)C1[e].y;
    sc1[e] = c;
    if (C2) { C2T c2; c2.x = (AT)C2[e].x; c2.y = (AT)C2[e].y; sc2[e] = c2; }
  }
  const int r = threadIdx.x / kMaxBlock, j = threadIdx.x % kMaxBlock;  // r < kUpdRows
  const long long ntiles = (N + rows - 1) / rows;
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long r0 = t * rows;
    __syncthreads();
    for (int e = threadIdx.x; e < rows * m; e += blockDim.x) {
      const int k = e / rows, rr = e % rows;
      V2 v; v.x = 0; v.y = 0;
      if (r0 + rr < N) v = col_ptr<T>(S, k, N)[r0 + rr];
      ss[rr][k] = v;
    }
    __syncthreads();
    if (j < q && r0 + r < N) {
      AT a1r = 0, a1i = 0, a2r = 0, a2i = 0;
      for (int k = 0; k < m; ++k) {
        const V2 sv = ss[r][k];
        const C2T c1 = sc1[k * q + j];
        a1r = fma((AT)sv.x, (AT)c1.x, a1r);
        a1r = fma(-(AT)sv.y, (AT)c1.y, a1r);
        a1i = fma((AT)sv.x, (AT)c1.y, a1i);
        a1i = fma((AT)sv.y, (AT)c1.x, a1i);
        if (C2) {
          const C2T c2 = sc2[k * q + j];
          a2r = fma((AT)sv.x, (AT)c2.x, a2r);
          a2r = fma(-(AT)sv.y, (AT)c2.y, a2r);
          a2i = fma((AT)sv.x, (AT)c2.y, a2i);
          a2i = fma((AT)sv.y, (AT)c2.x, a2i);
        }
      }
      const size_t gi = (size_t)j * N + r0 + r;
      if (SUB) {
        V2 o = out1[gi];
        o.x = (T)((AT)o.x - a1r); o.y = (T)((AT)o.y - a1i);
        out1[gi] = o;
      } else {
        V2 o; o.x = (T)a1r; o.y = (T)a1i;
        out1[gi] = o;
        if (C2) { V2 o2; o2.x = (T)a2r; o2.y = (T)a2i; out2[gi] = o2; }
      }
    }
  }
}

// Double-float variant of update_kernel for complex-double blocks (same layout and
// semantics; see gram_df_kernel for the arithmetic). One output element per thread is a sum of
// at most 72 products, kept in one double-float accumulator.
template <bool SUB>
__global__ void __launch_bounds__(kUpdThreads)
update_df_kernel(Batch bt, BlockList S, int m, long long N, const double2* C1, const double2* C2,
                 int cstride, int q, double2* out1, double2* out2) {
  const int prob = blockIdx.y;
  if (bt.active && !bt.active[prob]) return;
  const size_t poff = (size_t)prob * bt.pstride;
  for (int i = 0; i < S.nb; ++i) S.p[i] = reinterpret_cast<const double2*>(S.p[i]) + poff;
  out1 += poff;
  if (out2) out2 += poff;
  C1 += (size_t)prob * cstride;
  if (C2) C2 += (size_t)prob * cstride;
  extern __shared__ __align__(16) unsigned char upd_raw[];
  DF4* sc1 = reinterpret_cast<DF4*>(upd_raw);
  DF4* sc2 = sc1 + kMaxSmall * kMaxBlock;
  constexpr int rows = kUpdRows;
  __shared__ DF4 ss[rows][kMaxSmall + 1];
  for (int e = threadIdx.x; e < m * q; e += blockDim.x) {
    sc1[e] = df_split(C1[e]);
    if (C2) sc2[e] = df_split(C2[e]);
  }
  const int r = threadIdx.x / kMaxBlock, j = threadIdx.x % kMaxBlock;
  const long long ntiles = (N + rows - 1) / rows;
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long r0 = t * rows;
    __syncthreads();
    for (int e = threadIdx.x; e < rows * m; e += blockDim.x) {
      const int k = e / rows, rr = e % rows;
      double2 v = make_double2(0.0, 0.0);
      if (r0 + rr < N) v = col_ptr<double>(S, k, N)[r0 + rr];
      ss[rr][k] = df_split(v);
    }
    __syncthreads();
    if (j < q && r0 + r < N) {
      float a1rh = 0, a1rl = 0, a1ih = 0, a1il = 0, a2rh = 0, a2rl = 0, a2ih = 0, a2il = 0;
      for (int k = 0; k < m; ++k) {
        const DF4 sv = ss[r][k];
        const DF4 c1 = sc1[k * q + j];
        // s * c: re = sr cr - si ci, im = sr ci + si cr
        df_mac(a1rh, a1rl, sv.rh, sv.rl, c1.rh, c1.rl);
        df_mac(a1rh, a1rl, -sv.ih, -sv.il, c1.ih, c1.il);
        df_mac(a1ih, a1il, sv.rh, sv.rl, c1.ih, c1.il);
        df_mac(a1ih, a1il, sv.ih, sv.il, c1.rh, c1.rl);
        if (C2) {
          const DF4 c2 = sc2[k * q + j];
          df_mac(a2rh, a2rl, sv.rh, sv.rl, c2.rh, c2.rl);
          df_mac(a2rh, a2rl, -sv.ih, -sv.il, c2.ih, c2.il);
          df_mac(a2ih, a2il, sv.rh, sv.rl, c2.ih, c2.il);
          df_mac(a2ih, a2il, sv.ih, sv.il, c2.rh, c2.rl);
        }
      }
      const size_t gi = (size_t)j * N + r0 + r;
      if (SUB) {
        double2 o = out1[gi];
        o.x -= df_value(a1rh, a1rl);
        o.y -= df_value(a1ih, a1il);
        out1[gi] = o;
      } else {
        out1[gi] = make_double2(df_value(a1rh, a1rl), df_value(a1ih, a1il));
        if (C2) out2[gi] = make_double2(df_value(a2rh, a2rl), df_value(a2ih, a2il));
      }
    }
  }
}

constexpr int kResThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kResThreads)
residual_kernel(Batch bt, const typename Cplx<T>::type* X, const typename Cplx<T>::type* HX,
                const double* theta, const double* lam, const double* shift, const double* off2,
                typename Cplx<T>::type* W, long long N, int b, double* partial) {
  using V2 = typename Cplx<T>::type;
  using AT = typename Acc<T>::type;
  const int prob = blockIdx.y;
  if (bt.active && !bt.active[prob]) return;
  const size_t poff = (size_t)prob * bt.pstride;
  X += poff; HX += poff; W += poff;
  theta += (size_t)prob * kMaxBlock;
  const double sh = shift[prob], o2 = off2[prob];
  __shared__ double red[kResThreads / 32][kMaxBlock];  // b <= kMaxBlock
  AT acc[kMaxBlock];
#pragma unroll
  for (int j = 0; j < kMaxBlock; ++j) acc[j] = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
       i += (long long)gridDim.x * blockDim.x) {
    const double h = lam[i] + sh;
    const T mi = (T)(h / (h * h + o2));
#pragma unroll
    for (int j = 0; j < kMaxBlock; ++j) {
      if (j >= b) break;
      const size_t gi = (size_t)j * N + i;
      const V2 x = X[gi], h = HX[gi];
      const T th = (T)theta[j];
      V2 r; r.x = h.x - th * x.x; r.y = h.y - th * x.y;
      acc[j] += (AT)r.x * (AT)r.x + (AT)r.y * (AT)r.y;
      V2 w; w.x = mi * r.x; w.y = mi * r.y;
      W[gi] = w;
    }
  }
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
#pragma unroll
  for (int j = 0; j < kMaxBlock; ++j) {
    if (j >= b) break;
    double v = (double)acc[j];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < b) {
    double v = 0;
    for (int w = 0; w < kResThreads / 32; ++w) v += red[w][threadIdx.x];
    partial[((size_t)prob * gridDim.x + blockIdx.x) * b + threadIdx.x] = v;
  }
}

// One CTA a problem: lane j sums column j, its warps every kRedWarps-th slot.
__global__ void resid_finish(Batch bt, const double* partial, int slots, int b, double* resid) {
  const int prob = blockIdx.x;
  if (bt.active && !bt.active[prob]) return;
  __shared__ double part[kRedWarps][32];
  const int j = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double s = 0;
  for (int c = warp; j < b && c < slots; c += kRedWarps) s += partial[((size_t)prob * slots + c) * b + j];
  part[warp][j] = s;
  __syncthreads();
  if (warp > 0 || j >= b) return;
  for (int w = 1; w < kRedWarps; ++w) s += part[w][j];
  resid[(size_t)prob * kMaxBlock + j] = sqrt(s);
}

template <typename Tin, typename Tout>
__global__ void convert_kernel(const Tin* in, Tout* out, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = (Tout)in[i];
}

// splitmix64 (Steele, Lea, Flood 2014) as a counter-based generator of start vectors.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

template <typename T>
__global__ void random_kernel(typename Cplx<T>::type* X, long long count, unsigned long long seed) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const unsigned long long a = splitmix64(seed ^ (2ull * (unsigned long long)i));
    const unsigned long long c = splitmix64(seed ^ (2ull * (unsigned long long)i + 1ull));
    typename Cplx<T>::type v;
    v.x = (T)((double)(a >> 11) * (1.0 / 9007199254740992.0) - 0.5);
    v.y = (T)((double)(c >> 11) * (1.0 / 9007199254740992.0) - 0.5);
    X[i] = v;
  }
}

// flag = 1 when any of the count doubles is NaN or infinite
__global__ void nonfinite_kernel(const double* x, long long count, int* flag) {
  int bad = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x)
    bad |= !isfinite(x[i]);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

__global__ void mask_kernel(int nprob, int* mask, int off, int b, int value, const int* src) {
  const int prob = blockIdx.x;
  const int j = threadIdx.x;
  if (prob >= nprob || j >= b) return;
  mask[(size_t)prob * kMaxSmall + off + j] = src ? src[(size_t)prob * kMaxBlock + j] : value;
}

int grid_for(long long work, int per_block) {
  long long g = (work + per_block - 1) / per_block;
  if (g > 4 * 152) g = 4 * 152;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

template <typename T>
iwf_status gram(const Batch& bt, const BlockList& A, const BlockList& B, long long N, double2* out,
                double2* partial, int slots_per_prob, cudaStream_t s, bool herm) {
  const int ma = A.nb * A.b, mb = B.nb * B.b;
  if (ma > kMaxSmall || mb > kMaxSmall) return fail(IWF_ERR_ARG, "gram: too many columns");
  if (herm && ma != mb) return fail(IWF_ERR_ARG, "gram: a Hermitian product must be square");
  if (sizeof(T) == 8 && bt.engine == kEngineTensor)
    return gram_tc(bt, A, B, N, out, reinterpret_cast<double*>(partial), slots_per_prob, bt.err, s,
                   herm);
  const bool df = sizeof(T) == 8 && bt.engine == kEngineDF;
  // at least eight tiles a CTA where that still gives every SM one (a partial of up to 83 KB for
  // each 16-row tile cost more than the tile); in FP64 the tile costs more, and as many CTAs as
  // there are slots even out the last wave (20736 rows, 72 x 72: 932 us in 162 CTAs, 560 in 608)
  const long long tiles = (N + kGramRows - 1) / kGramRows;
  const long long want = sizeof(T) == 8 && !df
                             ? tiles
                             : std::max<long long>((152 + bt.nprob - 1) / bt.nprob, tiles / 8);
  const int g = (int)std::min<long long>(std::min<long long>(tiles, want), slots_per_prob);
  const int U = (ma + kGramTx - 1) / kGramTx, V = (mb + kGramTx - 1) / kGramTx;
  const dim3 grid(g, bt.nprob);
  switch (U * 4 + V + (herm ? 100 : 0)) {
#define IWF_GRAM(U_, V_, H_) \
    case U_ * 4 + V_ + (H_ ? 100 : 0): \
      if (df) gram_df_kernel<U_, V_, H_><<<grid, kGramThreads, 0, s>>>(bt, A, B, ma, mb, N, partial); \
      else gram_kernel<T, U_, V_, H_><<<grid, kGramThreads, 0, s>>>(bt, A, B, ma, mb, N, partial); \
      break;
    IWF_GRAM(1, 1, false) IWF_GRAM(1, 2, false) IWF_GRAM(1, 3, false) IWF_GRAM(2, 1, false)
    IWF_GRAM(2, 2, false) IWF_GRAM(2, 3, false) IWF_GRAM(3, 1, false) IWF_GRAM(3, 2, false)
    IWF_GRAM(3, 3, false) IWF_GRAM(1, 1, true) IWF_GRAM(2, 2, true) IWF_GRAM(3, 3, true)
#undef IWF_GRAM
    default: return fail(IWF_ERR_ARG, "gram: shape");
  }
  IWF_CUDA(cudaGetLastError());
  count_launch();
  const int cnt = ma * mb;
  reduce_partials<<<dim3((cnt + 31) / 32, bt.nprob), 32 * kRedWarps, 0, s>>>(bt, partial, g, cnt,
                                                                           out, herm, mb);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

template <typename T>
iwf_status block_update(const Batch& bt, const BlockList& S, long long N, const double2* C1,
                        const double2* C2, int cstride, int q, void* out1, void* out2,
                        bool subtract, cudaStream_t s, const double* norms) {
  // (the static attribute flags below are per instantiation of T)
  using V2 = typename Cplx<T>::type;
  const int m = S.nb * S.b;
  if (m > kMaxSmall || q > kMaxBlock || q < 1) return fail(IWF_ERR_ARG, "block_update: shape");
  if (cstride < m * q) return fail(IWF_ERR_ARG, "block_update: coefficient stride too small");
  if (sizeof(T) == 8 && bt.engine == kEngineTensor)
    return update_tc(bt, S, N, C1, C2, cstride, q, reinterpret_cast<double2*>(out1),
                     reinterpret_cast<double2*>(out2), subtract, bt.err, s, norms);
  int g0 = grid_for(N, kUpdRows);
  if (bt.nprob > 1) g0 = std::max(1, std::min(g0, (8 * 152 + bt.nprob - 1) / bt.nprob));
  const dim3 g(g0, bt.nprob);
  const size_t dyn = 2 * sizeof(double2) * kMaxSmall * kMaxBlock;
  static bool attr[2] = {false, false};
  if (!attr[subtract]) {
    if (subtract)
      IWF_CUDA(cudaFuncSetAttribute(update_kernel<T, true>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    else
      IWF_CUDA(cudaFuncSetAttribute(update_kernel<T, false>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    attr[subtract] = true;
  }
  if (sizeof(T) == 8 && bt.engine == kEngineDF) {
    static bool attr_df[2] = {false, false};
    if (!attr_df[subtract]) {
      if (subtract)
        IWF_CUDA(cudaFuncSetAttribute(update_df_kernel<true>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
      else
        IWF_CUDA(cudaFuncSetAttribute(update_df_kernel<false>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
      attr_df[subtract] = true;
    }
    if (subtract)
      update_df_kernel<true><<<g, kUpdThreads, dyn, s>>>(bt, S, m, N, C1, nullptr, cstride, q,
                                                         reinterpret_cast<double2*>(out1), nullptr);
    else
      update_df_kernel<false><<<g, kUpdThreads, dyn, s>>>(bt, S, m, N, C1, C2, cstride, q,
                                                          reinterpret_cast<double2*>(out1),
                                                          reinterpret_cast<double2*>(out2));
    IWF_CUDA(cudaGetLastError());
    count_launch();
    return IWF_OK;
  }
  if (subtract)
    update_kernel<T, true><<<g, kUpdThreads, dyn, s>>>(bt, S, m, N, C1, nullptr, cstride, q,
                                                       reinterpret_cast<V2*>(out1), nullptr);
  else
    update_kernel<T, false><<<g, kUpdThreads, dyn, s>>>(bt, S, m, N, C1, C2, cstride, q,
                                                        reinterpret_cast<V2*>(out1),
                                                        reinterpret_cast<V2*>(out2));
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

template <typename T>
iwf_status residual_precond(const Batch& bt, const void* X, const void* HX, const double* theta,
                            const double* lam, const double* shift, const double* off2,
                            void* W, long long N, int b, double* partial, int slots_per_prob,
                            double* resid, cudaStream_t s) {
  using V2 = typename Cplx<T>::type;
  int g = grid_for(N, kResThreads);
  if (g > slots_per_prob) g = slots_per_prob;
  residual_kernel<T><<<dim3(g, bt.nprob), kResThreads, 0, s>>>(
      bt, reinterpret_cast<const V2*>(X), reinterpret_cast<const V2*>(HX), theta, lam, shift,
      off2, reinterpret_cast<V2*>(W), N, b, partial);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  resid_finish<<<bt.nprob, 32 * kRedWarps, 0, s>>>(bt, partial, g, b, resid);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

template <typename Tin, typename Tout>
iwf_status convert_block(const void* in, void* out, long long count, cudaStream_t s) {
  convert_kernel<Tin, Tout><<<grid_for(count, 256), 256, 0, s>>>(
      reinterpret_cast<const Tin*>(in), reinterpret_cast<Tout*>(out), count);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

template <typename T>
iwf_status random_block(void* X, long long N, int b, unsigned long long seed, cudaStream_t s) {
  const long long count = N * b;
  random_kernel<T><<<grid_for(count, 256), 256, 0, s>>>(
      reinterpret_cast<typename Cplx<T>::type*>(X), count, seed);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

iwf_status any_nonfinite(const double* x, long long count, int* flag, cudaStream_t s) {
  IWF_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), s));
  nonfinite_kernel<<<grid_for(count, 256), 256, 0, s>>>(x, count, flag);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

iwf_status set_mask(const Batch& bt, int* mask, int off, int b, int value, const int* src,
                    cudaStream_t s) {
  mask_kernel<<<bt.nprob, 32, 0, s>>>(bt.nprob, mask, off, b, value, src);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

template iwf_status gram<double>(const Batch&, const BlockList&, const BlockList&, long long,
                                 double2*, double2*, int, cudaStream_t, bool);
template iwf_status gram<float>(const Batch&, const BlockList&, const BlockList&, long long,
                                double2*, double2*, int, cudaStream_t, bool);
template iwf_status block_update<double>(const Batch&, const BlockList&, long long, const double2*,
                                         const double2*, int, int, void*, void*, bool,
                                         cudaStream_t, const double*);
template iwf_status block_update<float>(const Batch&, const BlockList&, long long, const double2*,
                                        const double2*, int, int, void*, void*, bool,
                                        cudaStream_t, const double*);
template iwf_status residual_precond<double>(const Batch&, const void*, const void*, const double*,
                                             const double*, const double*, const double*, void*,
                                             long long, int, double*, int, double*, cudaStream_t);
template iwf_status residual_precond<float>(const Batch&, const void*, const void*, const double*,
                                            const double*, const double*, const double*, void*,
                                            long long, int, double*, int, double*, cudaStream_t);
template iwf_status convert_block<double, float>(const void*, void*, long long, cudaStream_t);
template iwf_status convert_block<float, double>(const void*, void*, long long, cudaStream_t);
template iwf_status random_block<double>(void*, long long, int, unsigned long long, cudaStream_t);
template iwf_status random_block<float>(void*, long long, int, unsigned long long, cudaStream_t);

}  // namespace iwf
