// Direct-convolution apply: H~ psi = Lambda psi + sum_m Vg_m psi(k* - m), the cyclic
// convolution on the K* grid with the potential's folded modes that F V F^{-1} equals
// (Sec. 3.3, Sec. 4.1; App. C for the folding). One pass, one read of psi and one write of
// H psi, no workspace; its cost grows with the number of modes, that of the transforms does
// not. iwf_apply takes it for potentials with few modes (every potential of the paper is a sum
// of cosines: 4 to 12 modes), iwf_apply_stencil always.
//
// In window order, grid point k* of slice o (k_II window position pos) sits at k_I window
// position w_j = (k*_j - lo_j(o)) mod 2K_j. The neighbour k* - m lies in slice o' with
// pos'_j = (pos_j - m_{II,j}) mod 2L_j, at k_I window position
// (w_j + lo_j(o) - lo_j(o') - m_{I,j}) mod 2K_j: each mode is a cyclic shift of whole slices,
// fixed per (slice, mode) pair.
#include <algorithm>
#include <cstdint>
#include <string>
#include <type_traits>

#include "common.cuh"

namespace iwf {

namespace {

constexpr int kStencilMaxModes = 256;
constexpr int kDirectThreads = 256;

template <typename T> struct SVec2;
template <> struct SVec2<double> { using type = double2; };
template <> struct SVec2<float> { using type = float2; };

struct DirectArgs {
  Geom g;
  const int* lo;          // MII x d
  const int* modes;       // nm x n, folded, none of them the constant
  const double2* coef;    // nm per problem
  const double* cst;      // constant term per problem (null: c0)
  double c0;
  int nm;
  const void* psi;
  void* out;
  const void* lam;
  long long ld;           // N
  int vpp;                // vectors per problem
  int groups;             // vector groups of a problem
  const int* active;      // problem p skipped when active[p] == 0 (may be null)
  int S, P;               // slices per CTA, threads per slice
  int parts;              // CTAs that share a slice (1 when S > 1)
  unsigned mag1, mag2;    // ceil(2^32 / len) of the faster k_I axes
};

// Running sum of c x over modes for one point and vector. Complex float: the two parts of x move
// through one packed multiply-add per coefficient part, sum cr (xr, xi) and sum ci (xr, xi), and
// are combined once at the end; complex double: four multiply-adds (two for real c). Lambda psi,
// the larger term by far for most points, is added last, so that the modes round against their
// own sum (added first, errors against 64 bits doubled: 8.4e-8 in complex float at 32^4).
template <typename T, bool REAL> struct ModeSum;
template <bool REAL> struct ModeSum<double, REAL> {
  double r = 0.0, i = 0.0;
  __device__ __forceinline__ void add(double2 c, double2 x) {
    r = fma(c.x, x.x, r);
    i = fma(c.x, x.y, i);
    if constexpr (!REAL) {
      r = fma(-c.y, x.y, r);
      i = fma(c.y, x.x, i);
    }
  }
  __device__ __forceinline__ double2 plus(double l, double2 p) const {
    return make_double2(fma(l, p.x, r), fma(l, p.y, i));
  }
};
__device__ __forceinline__ unsigned long long pack_f32x2(float a, float b) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ float2 unpack_f32x2(unsigned long long v) {
  float2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(v));
  return o;
}
__device__ __forceinline__ void fma_f32x2(unsigned long long& acc, unsigned long long c,
                                          unsigned long long x) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(c), "l"(x));
}
template <bool REAL> struct ModeSum<float, REAL> {
  unsigned long long a = 0, b = 0;
  __device__ __forceinline__ void add(float2 c, float2 x) {
    const unsigned long long xv = pack_f32x2(x.x, x.y);
    fma_f32x2(a, pack_f32x2(c.x, c.x), xv);
    if constexpr (!REAL) fma_f32x2(b, pack_f32x2(c.y, c.y), xv);
  }
  __device__ __forceinline__ float2 plus(float l, float2 p) const {
    float2 u = unpack_f32x2(a);
    if constexpr (!REAL) {
      const float2 w = unpack_f32x2(b);
      u = make_float2(u.x - w.y, u.y + w.x);
    }
    return make_float2(fmaf(l, p.x, u.x), fmaf(l, p.y, u.y));
  }
};

// CTA: blockIdx.x = S neighbouring slices (one, unless slices are smaller than a CTA), or one of
// `parts` shares of a slice where there are few slices; blockIdx.y = (problem, group of NV vectors).
// Thread (s, t) owns positions t, t + P, ... of slice s (with parts, every parts-th run of P) in NV
// vectors, so that a mode's index arithmetic is paid once for NV vectors; the neighbours of U modes
// are loaded before they are used.
// Measured on 16 vectors, transforms before and this kernel now: complex double, 32^4, 8 real
// modes 4330 -> 514 us (bound by the FP64 pipe: 18 operations a point, 480 us at its peak), Example
// 4.1's 1280 x 2048 23.85 -> 0.74 ms (also FP64); complex float, 32^4, 8 complex modes 184 ->
// 91 us (8 real ones 80), 16^6, 12 modes 15.1 -> 1.5 ms (issue and L1 latency together; ncu at 32^4,
// complex modes: issue 57 %, L1 56 %, DRAM 33 %, L2 32 %). NV = 2 or 8 were 30 % slower in complex float (index arithmetic;
// registers), U = 2 slower on 16^6, and patches of 2 x 2 to 4 x 8 slices a CTA, so that neighbour
// slices come from its own L1, no faster anywhere. psi itself is loaded after the modes: held in
// registers meanwhile it costs occupancy (111 us). Complex
// float runs with register bounds, none of which spills: three k_I axes for five CTAs an SM (16^6:
// 1.50 against 1.94 ms), two for four (8 complex modes at 32^4 92 us, 98 with three CTAs, 125 with
// the two that 92 registers allow; 22^4, 24 vectors 41, 45 and 55 us), the others for three, since
// four spill (1280 x 2048 185 against 446 us with one, at 175 registers).
// D: number of k_I axes when it is 1, 2 or 3; 0 handles any d. REAL: every coefficient is real.
template <typename T, int D, int NV, int U, bool REAL>
__global__ void __launch_bounds__(kDirectThreads, sizeof(T) == 8 ? 1 : D == 3 ? 5 : D == 2 ? 4 : 3)
direct_kernel(DirectArgs a) {
  using V2 = typename SVec2<T>::type;
  using Off = typename std::conditional<(D > 0), unsigned, size_t>::type;  // byte offsets
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Geom& g = a.g;
  const int d = D > 0 ? D : g.d, nII = g.n - d;
  const int prob = blockIdx.y / a.groups, group = blockIdx.y - prob * a.groups;
  if (a.active && !a.active[prob]) return;
  const int S = a.S, nm = a.nm;
  constexpr int W = D > 0 ? 4 : IWF_MAX_N;             // words per (mode, slice): slice, shifts
  V2* s_c = reinterpret_cast<V2*>(smem_raw);
  int* s_m = reinterpret_cast<int*>(smem_raw + (size_t)((nm + 1) & ~1) * sizeof(V2));
  const int MI = (int)g.MI;
  const int run = blockIdx.x % (unsigned)a.parts;
  const int o0 = (int)(blockIdx.x / (unsigned)a.parts) * S;
  for (int e = threadIdx.x; e < nm * S; e += blockDim.x) {
    const int q = e / S, o = o0 + e - q * S;
    if (o >= g.MII) continue;
    // k_II window position of slice o (C order, last k_II axis fastest), shifted by -m_II
    int rem = o, op = 0, stride = 1;
    for (int j = nII - 1; j >= 0; --j) {
      const int len = g.lens[d + j];
      const int pos = rem % len;
      rem /= len;
      int np = pos - a.modes[q * g.n + d + j];
      if (np < 0) np += len;
      op += np * stride;
      stride *= len;
    }
    s_m[e * W] = D > 0 ? op * MI : op;
    for (int j = 0; j < d; ++j) {
      const int len = g.lens[j];
      int sh = (a.lo[(size_t)o * d + j] - a.lo[(size_t)op * d + j] - a.modes[q * g.n + j]) % len;
      if (sh < 0) sh += len;
      s_m[e * W + 1 + j] = sh;
    }
  }
  for (int q = threadIdx.x; q < nm; q += blockDim.x) {
    const double2 c = a.coef[(size_t)prob * nm + q];
    V2 cv; cv.x = (T)c.x; cv.y = (T)c.y;
    s_c[q] = cv;
  }
  __syncthreads();
  const int s = threadIdx.x / a.P, t = threadIdx.x - s * a.P;
  const int o = o0 + s;
  if (s >= S || o >= g.MII) return;
  const T cst = (T)(a.cst ? a.cst[prob] : a.c0);
  const T* __restrict__ lam = reinterpret_cast<const T*>(a.lam) + (size_t)o * MI;
  const int l0 = g.lens[0], l1 = D >= 2 ? g.lens[1] : 1, l2 = D == 3 ? g.lens[2] : 1;
  const int* meta = s_m + s * W;
  const int v0 = prob * a.vpp + group * NV;
  const int nv = min(NV, a.vpp - group * NV);
  const char* base[NV];                                // the last group repeats its last vector
#pragma unroll
  for (int v = 0; v < NV; ++v)
    base[v] = reinterpret_cast<const char*>(a.psi) + (size_t)(v0 + min(v, nv - 1)) * a.ld * sizeof(V2);
  const auto load = [&](int v, Off i) { return __ldg(reinterpret_cast<const V2*>(base[v] + i)); };
  V2* out = reinterpret_cast<V2*>(a.out) + (size_t)v0 * a.ld + (size_t)o * MI;
  for (int w = run * a.P + t; w < MI; w += a.parts * a.P) {
    // coordinates of position w along the k_I axes (C order)
    int w0 = w, w1 = 0, w2 = 0;
    int wc[IWF_MAX_N];
    if (D == 2) {
      w0 = (int)__umulhi((unsigned)w, a.mag1);
      w1 = w - w0 * l1;
    } else if (D == 3) {
      const int r = (int)__umulhi((unsigned)w, a.mag2);
      w2 = w - r * l2;
      w0 = (int)__umulhi((unsigned)r, a.mag1);
      w1 = r - w0 * l1;
    } else if (D == 0) {
      int rr = w;
      for (int j = d - 1; j >= 0; --j) { wc[j] = rr % g.lens[j]; rr /= g.lens[j]; }
    }
    const auto offset = [&](int q) -> Off {            // of mode q's neighbour of position w
      if constexpr (D > 0) {
        const int4 m = *reinterpret_cast<const int4*>(meta + q * S * W);
        int x = w0 + m.y;
        if (x >= l0) x -= l0;
        if constexpr (D >= 2) {
          int y = w1 + m.z;
          if (y >= l1) y -= l1;
          x = x * l1 + y;
        }
        if constexpr (D == 3) {
          int z = w2 + m.w;
          if (z >= l2) z -= l2;
          x = x * l2 + z;
        }
        return (unsigned)(m.x + x) * (unsigned)sizeof(V2);
      } else {
        const int* m = meta + q * S * W;
        int x = 0;
        for (int j = 0; j < d; ++j) {
          int y = wc[j] + m[1 + j];
          if (y >= g.lens[j]) y -= g.lens[j];
          x = x * g.lens[j] + y;
        }
        return ((size_t)m[0] * MI + x) * sizeof(V2);
      }
    };
    T l = lam[w];
    if (cst != T(0)) l += cst;
    const Off own = ((Off)o * (Off)MI + (Off)w) * (Off)sizeof(V2);
    ModeSum<T, REAL> acc[NV];
    int q0 = 0;
    for (; q0 + U <= nm; q0 += U) {
      V2 x[U][NV];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const Off i = offset(q0 + u);
#pragma unroll
        for (int v = 0; v < NV; ++v) x[u][v] = load(v, i);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const V2 c = s_c[q0 + u];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v].add(c, x[u][v]);
      }
    }
    for (; q0 < nm; ++q0) {
      const Off i = offset(q0);
      const V2 c = s_c[q0];
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v].add(c, load(v, i));
    }
    // streaming stores: H psi is not read again here, psi's lines are
#pragma unroll
    for (int v = 0; v < NV; ++v)
      if (v < nv) __stcs(out + (size_t)v * a.ld + w, acc[v].plus(l, load(v, own)));
  }
}

template <typename T, int D, int NV>
iwf_status launch_direct(DirectArgs a, bool real, int nprob, cudaStream_t s) {
  using V2 = typename SVec2<T>::type;
  constexpr int U = 4;
  a.groups = (a.vpp + NV - 1) / NV;
  const long long slices = (a.g.MII + a.S - 1) / a.S;
  // A slice is shared among CTAs where there are fewer than four an SM: a window of few slices
  // (8^4 x 16, 48 real modes, 4 vectors: 16 CTAs, 390 us where the transforms take 164) otherwise
  // leaves the chip idle (now 45 us). With four or more, sharing only repeats the shifts' set-up.
  const long long rounds = (a.g.MI + a.P - 1) / a.P;
  a.parts = 1;
  if (rounds > 1) {
    int sms = 0, dev = 0;
    IWF_CUDA(cudaGetDevice(&dev));
    IWF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const long long want = 4LL * sms / std::max(1LL, slices * nprob * a.groups);
    a.parts = (int)std::max(1LL, std::min(want, rounds));
  }
  const long long blocks = slices * a.parts;
  if ((long long)nprob * a.groups > 65535 || blocks > 2147483647LL)
    return fail(IWF_ERR_UNSUPPORTED, "direct apply: too many slices or vectors");
  const size_t smem = (size_t)((a.nm + 1) & ~1) * sizeof(V2) +
                      (size_t)a.nm * a.S * (D > 0 ? 4 : IWF_MAX_N) * sizeof(int);
  const dim3 grid((unsigned)blocks, (unsigned)(nprob * a.groups));
  const int threads = (a.S * a.P + 31) / 32 * 32;
  if (real) direct_kernel<T, D, NV, U, true><<<grid, threads, smem, s>>>(a);
  else direct_kernel<T, D, NV, U, false><<<grid, threads, smem, s>>>(a);
  IWF_CUDA(cudaGetLastError());
  count_launch();
  return IWF_OK;
}

template <typename T, int D>
iwf_status launch_direct_d(const DirectArgs& a, bool real, int nprob, cudaStream_t s) {
  if (a.vpp == 1) return launch_direct<T, D, 1>(a, real, nprob, s);
  if (a.vpp == 2) return launch_direct<T, D, 2>(a, real, nprob, s);
  return launch_direct<T, D, 4>(a, real, nprob, s);
}

template <typename T>
iwf_status run_direct(const iwf_plan* p, DirectArgs a, bool real, int nprob, cudaStream_t s) {
  using V2 = typename SVec2<T>::type;
  const Geom& g = p->g;
  a.g = g;
  a.lo = p->d_lo;
  a.ld = g.N;
  a.lam = sizeof(T) == 8 ? (const void*)p->d_lam64 : (const void*)p->d_lam32;
  // threads of a slice: 256 or 128, whichever leaves fewer idle in its last round; slices that
  // small share a CTA, as many as its threads hold and shared memory has room for
  const auto rounds = [&](int n) { return (g.MI + n - 1) / n * n; };
  a.P = (int)std::min<long long>(g.MI, rounds(128) < rounds(256) ? 128 : 256);
  a.S = (int)std::max<long long>(1, std::min<long long>(128 / a.P, g.MII));
  a.S = std::max(1, std::min(a.S, 1024 / std::max(1, a.nm)));
  const auto mag = [](int l) { return (unsigned)(((1ull << 32) + l - 1) / l); };
  a.mag1 = g.d >= 2 ? mag(g.lens[1]) : 0;
  a.mag2 = g.d >= 3 ? mag(g.lens[2]) : 0;
  // 32-bit offsets and divisions by multiplication where the sizes allow them (the quotients
  // are exact for positions below 2^18: positions x (len - 1) < 2^32)
  const bool small = (size_t)g.N * sizeof(V2) < (1ull << 32) && g.MI <= (1 << 18);
  switch (small && g.d <= 3 ? g.d : 0) {
    case 1: return launch_direct_d<T, 1>(a, real, nprob, s);
    case 2: return launch_direct_d<T, 2>(a, real, nprob, s);
    case 3: return launch_direct_d<T, 3>(a, real, nprob, s);
    default: return launch_direct_d<T, 0>(a, real, nprob, s);
  }
}

}  // namespace

iwf_status apply_direct(const iwf_plan* p, int precision, const void* psi, void* hpsi, int nvec,
                        cudaStream_t stream, const ApplyBatch* batch) {
  DirectArgs a{};
  a.psi = psi;
  a.out = hpsi;
  bool real = p->stencil_real;
  int nprob = 1;
  if (batch) {
    a.modes = batch->modes; a.coef = batch->coef; a.cst = batch->cst; a.nm = batch->nm;
    a.vpp = batch->vecs_per_prob;
    a.active = batch->active;
    real = batch->real;
    nprob = nvec / batch->vecs_per_prob;
  } else {
    a.modes = p->d_stencil_m; a.coef = p->d_stencil_c; a.nm = p->stencil_nm; a.c0 = p->vconst;
    a.vpp = nvec;
  }
  return precision == IWF_PREC_F64 ? run_direct<double>(p, a, real, nprob, stream)
                                   : run_direct<float>(p, a, real, nprob, stream);
}

iwf_status apply_stencil_impl(iwf_plan* p, int precision, const void* psi, void* hpsi, int nvec,
                              cudaStream_t stream) {
  if (nvec < 0) return fail(IWF_ERR_ARG, "iwf_apply_stencil: nvec < 0");
  if (nvec == 0) return IWF_OK;
  if (!psi || !hpsi) return fail(IWF_ERR_ARG, "iwf_apply_stencil: null vector pointer");
  if (precision != IWF_PREC_F64 && precision != IWF_PREC_C64)
    return fail(IWF_ERR_ARG, "iwf_apply_stencil: unknown precision");
  if (p->pot_kind == 0) return fail(IWF_ERR_ARG, "iwf_apply_stencil: no potential set");
  if (nvec > 65535) return fail(IWF_ERR_ARG, "iwf_apply_stencil: nvec > 65535");
  if (p->stencil_nm + (p->stencil_const ? 1 : 0) > kStencilMaxModes)
    return fail(IWF_ERR_UNSUPPORTED, "iwf_apply_stencil: more than " +
                std::to_string(kStencilMaxModes) + " folded modes (use iwf_apply)");
  const size_t bytes = (size_t)p->g.N * nvec * (precision == IWF_PREC_F64 ? 16 : 8);
  const uintptr_t ua = reinterpret_cast<uintptr_t>(psi), ub = reinterpret_cast<uintptr_t>(hpsi);
  if (ua < ub + bytes && ub < ua + bytes) return fail(IWF_ERR_ARG, "iwf_apply_stencil: psi and hpsi overlap");
  if (p->g.lens[p->g.d - 1] > 32) return fail(IWF_ERR_UNSUPPORTED, "iwf_apply_stencil: axis longer than 32");
  if (p->g.MII > 2147483647LL) return fail(IWF_ERR_UNSUPPORTED, "iwf_apply_stencil: too many slices");
  return apply_direct(p, precision, psi, hpsi, nvec, stream, nullptr);
}

}  // namespace iwf
