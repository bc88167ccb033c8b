// Device parts shared by the Rayleigh-Ritz chain (rr_wide.cu) and the dense
// symmetric eigensolver (eigh.cu): arithmetic templated on double or dfl, the
// work layout of a pencil, and the eigenpairs of a symmetric tridiagonal
// matrix (location by FP32 Sturm counts, Rayleigh-quotient iteration per
// isolated vector, clusters).  Internal linkage: each translation unit has
// its own kernels.
#pragma once

#include <cfloat>

#include "dfloat.cuh"
#include "internal.h"

namespace dgdft {

namespace {

// ---------------------------------------------------------------- arithmetic

__device__ __forceinline__ double rt_add(double a, double b) { return a + b; }
__device__ __forceinline__ double rt_sub(double a, double b) { return a - b; }
__device__ __forceinline__ double rt_mul(double a, double b) { return a * b; }
__device__ __forceinline__ double rt_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double rt_fnma(double a, double b, double c) { return fma(-a, b, c); }
__device__ __forceinline__ double rt_neg(double a) { return -a; }
__device__ __forceinline__ double rt_abs(double a) { return fabs(a); }
__device__ __forceinline__ double rt_rcp(double a) { return 1.0 / a; }
__device__ __forceinline__ double rt_rsqrt(double a) { return rsqrt(a); }
__device__ __forceinline__ double rt_val(double a) { return a; }
__device__ __forceinline__ double rt_mag(double a) { return fabs(a); }
__device__ __forceinline__ bool rt_pos(double a) { return a > 0.0 && isfinite(a); }
__device__ __forceinline__ bool rt_nonneg(double a) { return a >= 0.0; }
__device__ __forceinline__ dfl rt_add(dfl a, dfl b) { return dfl_add(a, b); }
__device__ __forceinline__ dfl rt_sub(dfl a, dfl b) { return dfl_sub(a, b); }
__device__ __forceinline__ dfl rt_mul(dfl a, dfl b) { return dfl_mul(a, b); }
__device__ __forceinline__ dfl rt_fma(dfl a, dfl b, dfl c) { return dfl_fma(a, b, c); }
__device__ __forceinline__ dfl rt_fnma(dfl a, dfl b, dfl c) { return dfl_fnma(a, b, c); }
__device__ __forceinline__ dfl rt_neg(dfl a) { return dfl_neg(a); }
__device__ __forceinline__ dfl rt_abs(dfl a) { return dfl_abs(a); }
__device__ __forceinline__ dfl rt_rcp(dfl a) { return dfl_rcp(a); }
__device__ __forceinline__ dfl rt_rsqrt(dfl a) { return dfl_rsqrt(a); }
__device__ __forceinline__ double rt_val(dfl a) { return dfl_val(a); }
__device__ __forceinline__ float rt_mag(dfl a) { return fabsf(a.h); }
__device__ __forceinline__ bool rt_pos(dfl a) { return a.h > 0.0f && isfinite(a.h); }
__device__ __forceinline__ bool rt_nonneg(dfl a) { return a.h >= 0.0f; }
__device__ __forceinline__ float rt_sub(float a, float b) { return a - b; }
__device__ __forceinline__ float rt_mul(float a, float b) { return a * b; }
__device__ __forceinline__ float rt_fnma(float a, float b, float c) { return fmaf(-a, b, c); }
__device__ __forceinline__ float rt_neg(float a) { return -a; }
__device__ __forceinline__ float rt_rcp(float a) { return 1.0f / a; }
__device__ __forceinline__ float rt_mag(float a) { return fabsf(a); }
__device__ __forceinline__ bool rt_nonneg(float a) { return a >= 0.0f; }

template <class T> struct RtOf;
template <> struct RtOf<double> {
  static __device__ __forceinline__ double of(double x) { return x; }
  static __device__ __forceinline__ double off(float x) { return (double)x; }
  static __device__ __forceinline__ float to_f(double x) { return (float)x; }
  static constexpr double eps = 2.220446049250313e-16;
};
template <> struct RtOf<dfl> {
  static __device__ __forceinline__ dfl of(double x) { return dfl_of(x); }  // FP64 instructions
  static __device__ __forceinline__ dfl off(float x) { return {x, 0.0f}; }
  static __device__ __forceinline__ float to_f(dfl x) { return x.h + x.l; }
  static constexpr double eps = 1.4210854715202004e-14;  // 2^-46
};
template <> struct RtOf<float> {
  static __device__ __forceinline__ float off(float x) { return x; }
};

// Solutions of an inverse iteration reach 1 / (eps |T|) and, inside a cluster,
// its square, whose own square leaves the FP32 range of a pair: pairs are
// kept scaled by 2^-46 (exactly), doubles need none.
template <class T> struct RtScale;
template <> struct RtScale<double> {
  static constexpr double inv = 1.0;
  static constexpr double window = 1e-5;  // rrw_fix_kernel: eps / window bounds the loss of orthogonality
  static __device__ __forceinline__ double down(double x) { return x; }
};
template <> struct RtScale<dfl> {
  static constexpr double inv = 1.4210854715202004e-14;
  static constexpr double window = 3e-5;
  static __device__ __forceinline__ dfl down(dfl x) { return dfl_scale2(x, 1.4210854715202004e-14f); }
};

__device__ __forceinline__ double rt_shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ dfl rt_shfl(dfl v, int src) {
  return {__shfl_sync(0xffffffffu, v.h, src), __shfl_sync(0xffffffffu, v.l, src)};
}
__device__ __forceinline__ double rt_down(unsigned mask, double v, int o, int w) {
  return __shfl_down_sync(mask, v, o, w);
}
__device__ __forceinline__ dfl rt_down(unsigned mask, dfl v, int o, int w) {
  return {__shfl_down_sync(mask, v.h, o, w), __shfl_down_sync(mask, v.l, o, w)};
}
__device__ __forceinline__ double rt_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dfl rt_xor(dfl v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
}
// sum over the warp, the same value in every lane
template <class T> __device__ __forceinline__ T rt_warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = rt_add(v, rt_down(0xffffffffu, v, o, 32));
  return rt_shfl(v, 0);
}

// ---------------------------------------------------------------- layout

constexpr int RW_THREADS = 512;
constexpr int RW_WARPS = RW_THREADS / 32;
constexpr int RW_CL_MAX = 16;
// Of |T|: closer eigenvalue estimates form a cluster.  The FP32 Sturm counts
// locate an eigenvalue to 2e-8 .. 7e-8 |T| (measured on LOBPCG pencils of 16 to
// 312 columns), so a vector that moved by over half of this found another one.
constexpr float RW_ORTOL = 5e-7f;

// Work of one pencil; every matrix has leading dimension ld = the largest
// pencil the task can form.
template <class T> struct WideWork {
  T *L, *LT, *X, *C, *Z, *scr, *d, *e, *rinv, *scal;
  double *lam, *sh;
  int* st;  // [0] n of the accepted pencil (0: nothing to do), [1] 1 when blocks were dropped,
            // [2] 1 for a standard problem (no L)
  int ld;
};

__host__ __device__ inline size_t wide_work_doubles(int n, int m) {
  return (size_t)4 * n * n + (size_t)5 * n * m + 4 * (size_t)n + 2 * (size_t)m + 16;
}

template <class T> __device__ __forceinline__ WideWork<T> wide_carve(const RRTask& t) {
  WideWork<T> w;
  const int ld = (t.mode == RR_FIXED) ? t.n_fixed : (t.mode == RR_INITIAL) ? t.m : 3 * t.m;
  const size_t nn = (size_t)ld * ld, nm = (size_t)ld * t.m;
  T* p = reinterpret_cast<T*>(t.work);
  w.ld = ld;
  w.L = p;
  w.LT = p + nn;
  w.X = p + 2 * nn;
  w.C = p + 3 * nn;
  w.Z = p + 4 * nn;
  w.scr = w.Z + nm;  // 4 values per row and vector
  w.d = w.scr + 4 * nm;
  w.e = w.d + ld;
  w.rinv = w.e + ld;
  w.scal = w.rinv + ld;
  w.lam = reinterpret_cast<double*>(w.scal + ld);
  w.sh = w.lam + t.m;
  w.st = reinterpret_cast<int*>(w.sh + t.m);
  return w;
}

// element (r, c) of the symmetric pencil matrix M: the Gram blocks are formed
// for the upper block triangle, diagonal blocks are averaged with their
// transpose
__device__ __forceinline__ double wide_sym(const double* M, int ldm, int r, int c, int bm) {
  const int br = (r >= bm) + (r >= 2 * bm), bc = (c >= bm) + (c >= 2 * bm);  // at most three blocks
  if (br < bc) return M[r + (size_t)c * ldm];
  if (br > bc) return M[c + (size_t)r * ldm];
  return 0.5 * (M[r + (size_t)c * ldm] + M[c + (size_t)r * ldm]);
}

// ---------------------------------------------------------------- eigenvalue estimates

constexpr int BI_WARPS = 4, BI_PER = 2;  // warps per CTA, eigenvalues per warp

// Lowest m eigenvalues of the tridiagonal matrix to FP32 accuracy: a warp
// splits the bracket of an eigenvalue into 33 parts a round by 32 Sturm counts
// and carries two eigenvalues at once, whose chains of divisions overlap.
// Five rounds: 33^-5 of the Gershgorin interval, FP32 resolution.
template <class T>
__global__ void __launch_bounds__(32 * BI_WARPS) rrw_bisect_kernel(const RRTask* __restrict__ tasks) {
  const RRTask Tk = tasks[blockIdx.y];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int n = W.st[0], m = Tk.m;
  if (n == 0 || (int)blockIdx.x * BI_WARPS * BI_PER >= m) return;
  extern __shared__ __align__(16) unsigned char rw_raw[];
  float* d = reinterpret_cast<float*>(rw_raw);
  float* e2 = d + n;
  __shared__ float rg[3][BI_WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float glo = FLT_MAX, ghi = -FLT_MAX, gno = 0.0f;
  for (int i = tid; i < n; i += 32 * BI_WARPS) {
    const float di = RtOf<T>::to_f(W.d[i]), ei = RtOf<T>::to_f(W.e[i]);
    const float r = (i > 0 ? fabsf(RtOf<T>::to_f(W.e[i - 1])) : 0.0f) + (i < n - 1 ? fabsf(ei) : 0.0f);
    d[i] = di;
    e2[i] = ei * ei;
    glo = fminf(glo, di - r);
    ghi = fmaxf(ghi, di + r);
    gno = fmaxf(gno, fabsf(di) + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    glo = fminf(glo, __shfl_xor_sync(0xffffffffu, glo, o));
    ghi = fmaxf(ghi, __shfl_xor_sync(0xffffffffu, ghi, o));
    gno = fmaxf(gno, __shfl_xor_sync(0xffffffffu, gno, o));
  }
  if (lane == 0) {
    rg[0][warp] = glo;
    rg[1][warp] = ghi;
    rg[2][warp] = gno;
  }
  __syncthreads();
  for (int w = 0; w < BI_WARPS; ++w) {
    glo = fminf(glo, rg[0][w]);
    ghi = fmaxf(ghi, rg[1][w]);
    gno = fmaxf(gno, rg[2][w]);
  }
  const float pad = 1e-6f * fmaxf(gno, 1e-30f);
  const int j0 = (blockIdx.x * BI_WARPS + warp) * BI_PER;
  float lo[BI_PER], hi[BI_PER];
#pragma unroll
  for (int q = 0; q < BI_PER; ++q) {
    lo[q] = glo - pad;
    hi[q] = ghi + pad;
  }
  for (int round = 0; round < 5; ++round) {
    float x[BI_PER], q0[BI_PER];
    int cnt[BI_PER];
#pragma unroll
    for (int q = 0; q < BI_PER; ++q) {
      x[q] = lo[q] + (hi[q] - lo[q]) * ((float)(lane + 1) / 33.0f);
      q0[q] = 1.0f;
      cnt[q] = 0;
    }
    float eprev = 0.0f;
    for (int i = 0; i < n; ++i) {
      const float di = d[i];
#pragma unroll
      for (int q = 0; q < BI_PER; ++q) {
        float v = di - x[q] - __fdividef(eprev, q0[q]);
        if (fabsf(v) < 1e-30f) v = -1e-30f;
        cnt[q] += v < 0.0f;
        q0[q] = v;
      }
      eprev = e2[i];
    }
#pragma unroll
    for (int q = 0; q < BI_PER; ++q) {
      const unsigned above = __ballot_sync(0xffffffffu, cnt[q] > j0 + q);
      const int f = above ? __ffs(above) - 1 : 32;  // first point with more than j eigenvalues below it
      const float xf = __shfl_sync(0xffffffffu, x[q], min(f, 31));
      const float xb = __shfl_sync(0xffffffffu, x[q], max(f - 1, 0));
      if (f < 32) hi[q] = xf;
      if (f > 0) lo[q] = xb;
    }
  }
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < BI_PER; ++q)
      if (j0 + q < m) W.sh[j0 + q] = 0.5 * ((double)lo[q] + (double)hi[q]);
}

// ---------------------------------------------------------------- eigenvectors

__device__ __forceinline__ float wide_hash(unsigned a, unsigned b) {
  unsigned h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (float)(h & 0xFFFFFF) * (1.0f / 8388608.0f) - 1.0f;
}

template <class T> __device__ __forceinline__ T wide_cut(T p, float tiny) {
  if (rt_mag(p) < tiny) p = RtOf<T>::off(rt_nonneg(p) ? tiny : -tiny);
  return p;
}

// Solve (T - lq I) x = b by elimination with partial pivoting, one thread.
// d, e in U; b(i) gives the right-hand side, out(i, x_i) takes the solution
// from the last row to the first.  scr[(4 i + c) stride]: the finished rows
// (reciprocal pivot, two entries right of it, right-hand side).
template <class U, class Mat, class Rhs, class Out>
__device__ __forceinline__ void wide_tri_solve(const Mat& d, const Mat& e, int n, U lq, float tiny, U* scr, size_t stride,
                                               Rhs b, Out out) {
  U c0 = rt_sub(d[0], lq), c1 = (n > 1) ? e[0] : RtOf<U>::off(0.0f);
  U bi = b(0);
  for (int i = 0; i + 1 < n; ++i) {
    const U sub = e[i];
    const U n0 = rt_sub(d[i + 1], lq);
    const U n1 = (i + 2 < n) ? e[i + 1] : RtOf<U>::off(0.0f);
    const U bn = b(i + 1);
    const bool swap = rt_mag(sub) > rt_mag(c0);
    const U p0 = wide_cut(swap ? sub : c0, tiny);
    const U rp = rt_rcp(p0);
    const U mlt = rt_mul(swap ? c0 : sub, rp);
    const U p1 = swap ? n0 : c1, p2 = swap ? n1 : RtOf<U>::off(0.0f), pb = swap ? bn : bi;
    c0 = rt_fnma(mlt, p1, swap ? c1 : n0);
    c1 = swap ? rt_neg(rt_mul(mlt, n1)) : n1;
    bi = rt_fnma(mlt, pb, swap ? bi : bn);
    U* s = scr + (size_t)(4 * i) * stride;
    s[0] = rp;
    s[stride] = p1;
    s[2 * stride] = p2;
    s[3 * stride] = pb;
  }
  U x1 = rt_mul(bi, rt_rcp(wide_cut(c0, tiny))), x2 = RtOf<U>::off(0.0f);
  out(n - 1, x1);
  for (int i = n - 2; i >= 0; --i) {
    const U* s = scr + (size_t)(4 * i) * stride;
    U t = rt_fnma(s[2 * stride], x2, s[3 * stride]);
    t = rt_fnma(s[stride], x1, t);
    const U x = rt_mul(t, s[0]);
    out(i, x);
    x2 = x1;
    x1 = x;
  }
}

// the matrix as float: a staged copy, or converted on the way
template <class T, bool STAGED> struct FloatOf {
  const T* t;
  const float* f;
  __device__ __forceinline__ float operator[](int i) const { return STAGED ? f[i] : RtOf<T>::to_f(t[i]); }
};

// |T| by Gershgorin, in FP32, for every thread of the CTA (blockDim <= 1024)
template <class T> __device__ float wide_gnorm(const T* d, const T* e, int n, float* red) {
  float g = 0.0f;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    g = fmaxf(g, (float)rt_mag(d[i]) + (i > 0 ? (float)rt_mag(e[i - 1]) : 0.0f) +
                     (i + 1 < n ? (float)rt_mag(e[i]) : 0.0f));
  for (int o = 16; o > 0; o >>= 1) g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = g;
  __syncthreads();
  g = red[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) g = fmaxf(g, red[w]);
  __syncthreads();
  return fmaxf(g, 1e-30f);
}

// does estimate j sit within the cluster threshold of estimate j - 1?
__device__ __forceinline__ bool wide_joins(const double* sh, int j, double ortol) {
  return j > 0 && sh[j] - sh[j - 1] <= ortol;
}

// The shift of the next step: the Rayleigh quotient, or the located estimate
// while the quotient is farther from it than the location error (a start that
// happens to hold little of its eigenvector would otherwise be drawn to a
// neighbour: seen in 1 of 80 pencils of a monolayer solve).
template <class T> __device__ __forceinline__ T near_estimate(T rq, double sh, double ortol) {
  return fabs(rt_val(rq) - sh) <= 0.5 * ortol ? rq : RtOf<T>::of(sh);
}

constexpr int VE_THREADS = 128, VE_VECS = 8;

// Shared memory of rrw_vec_kernel with NV vectors per CTA; staged: the matrix
// as T and as float beside them.
inline size_t vec_smem(int n, int nv, bool staged) { return 8 * (size_t)n * 5 * nv + (staged ? 24 * (size_t)n : 0); }

// Eigenvectors of isolated eigenvalues, NV per CTA, one per lane of warp 0: an FP32 inverse iteration from a random start, then Rayleigh-quotient
// iterations in T until the residual 1 / |x| is at rounding (two as a rule).
// With (T - s) x = b the Rayleigh quotient of x is s + x.b / x.x, so a step
// needs no product with T.  What bounds it is the chain of eliminations (a
// reciprocal per row: 440 cycles in FP64), so few vectors share a CTA and the
// finished rows and the vectors stay in shared memory (from global memory a
// row waited ~700 cycles on top).  The four warps share the normalisations.
// STAGED: the matrix in shared memory too (n <= 608 with eight vectors); large
// matrices leave it to the L1 cache and take fewer vectors per CTA.
template <class T, int NV, bool STAGED>
__global__ void __launch_bounds__(VE_THREADS) rrw_vec_kernel(const RRTask* __restrict__ tasks) {
  const RRTask Tk = tasks[blockIdx.y];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int n = W.st[0], m = Tk.m, ld = W.ld;
  if (n == 0 || (int)blockIdx.x * NV >= m) return;
  extern __shared__ __align__(16) unsigned char rw_raw[];
  T* scr = reinterpret_cast<T*>(rw_raw);  // 4 n x NV
  T* zs = scr + (size_t)4 * n * NV;       // n x NV
  T *ds = zs + (size_t)n * NV, *es = ds + n;
  float *df = reinterpret_cast<float*>(es + n), *ef = df + n;
  const T *d = STAGED ? ds : W.d, *e = STAGED ? es : W.e;
  __shared__ float redf[VE_THREADS / 32];
  __shared__ T s_scale[NV], s_lam[NV];
  __shared__ int s_more, s_on[NV];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (STAGED) {
    for (int i = tid; i < n; i += VE_THREADS) {
      ds[i] = W.d[i];
      es[i] = W.e[i];
      df[i] = RtOf<T>::to_f(W.d[i]);
      ef[i] = RtOf<T>::to_f(W.e[i]);
    }
    __syncthreads();
  }
  const float gnorm = wide_gnorm(d, e, n, redf);
  const double ortol = (double)RW_ORTOL * (double)gnorm;
  const int q0 = blockIdx.x * NV, nq = min(NV, m - q0);
  const int q = q0 + lane;
  if (tid < NV) {
    const bool on = lane < nq && !wide_joins(W.sh, q, ortol) && !(q + 1 < m && wide_joins(W.sh, q + 1, ortol));
    s_on[lane] = on;
    if (on) {
      T* z = zs + lane;
      float amax = 0.0f;
      // (float values in the same 8-byte slots as the steps in T)
      const FloatOf<T, STAGED> dl{d, df}, el{e, ef};
      wide_tri_solve<float>(
          dl, el, n, (float)W.sh[q], 1.2e-7f * gnorm, reinterpret_cast<float*>(scr + lane), 2 * (size_t)NV,
          [&](int i) { return wide_hash(i, q + 7919u * blockIdx.y); },
          [&](int i, float x) {
            amax = fmaxf(amax, fabsf(x));
            z[i * NV] = RtOf<T>::off(x);
          });
      // scaled by the largest entry, so that the squares below stay in range
      s_scale[lane] = RtOf<T>::off(amax > 0.0f ? 1.0f / amax : 1.0f);
    }
  }
  __syncthreads();
  // Rayleigh quotients and norms in T
  for (int v = warp; v < nq; v += VE_THREADS / 32) {
    if (!s_on[v]) continue;
    T* zv = zs + v;
    const T sc = s_scale[v];
    T xx = RtOf<T>::off(0.0f), xt = RtOf<T>::off(0.0f);
    for (int i = lane; i < n; i += 32) {
      const T x = rt_mul(zv[i * NV], sc);
      T t = rt_mul(d[i], x);
      if (i > 0) t = rt_fma(e[i - 1], rt_mul(zv[(i - 1) * NV], sc), t);
      if (i + 1 < n) t = rt_fma(e[i], rt_mul(zv[(i + 1) * NV], sc), t);
      xx = rt_fma(x, x, xx);
      xt = rt_fma(x, t, xt);
    }
    xx = rt_warp_sum(xx);
    xt = rt_warp_sum(xt);
    if (lane == 0) s_lam[v] = near_estimate(rt_mul(xt, rt_rcp(xx)), W.sh[q0 + v], ortol);
    const T s2 = rt_mul(sc, rt_rsqrt(xx));
    for (int i = lane; i < n; i += 32) zv[i * NV] = rt_mul(zv[i * NV], s2);
  }
  __syncthreads();
  const float tiny = fmaxf((float)(RtOf<T>::eps * gnorm), 1e-36f);
  const double done = 256.0 * RtOf<T>::eps * (double)gnorm;
  for (int it = 0; it < 6; ++it) {
    if (tid == 0) s_more = 0;
    __syncthreads();
    if (tid < NV && s_on[lane]) {
      T* z = zs + lane;
      const T lq = s_lam[lane];
      T xx = RtOf<T>::off(0.0f), xb = RtOf<T>::off(0.0f);
      wide_tri_solve<T>(
          d, e, n, lq, tiny, scr + lane, (size_t)NV, [&](int i) { return z[i * NV]; },
          [&](int i, T xi) {
            const T x = RtScale<T>::down(xi);
            xb = rt_fma(x, z[i * NV], xb);
            xx = rt_fma(x, x, xx);
            z[i * NV] = x;
          });
      const T inv = rt_rsqrt(xx);
      s_scale[lane] = inv;
      const T rq = rt_fma(RtScale<T>::down(rt_mul(xb, inv)), inv, lq);
      s_lam[lane] = near_estimate(rq, W.sh[q], ortol);
      if (rt_val(inv) * RtScale<T>::inv > done) s_more = 1;
    }
    __syncthreads();
    for (int v = warp; v < nq; v += VE_THREADS / 32) {
      if (!s_on[v]) continue;
      T* zv = zs + v;
      const T s2 = s_scale[v];
      for (int i = lane; i < n; i += 32) zv[i * NV] = rt_mul(zv[i * NV], s2);
    }
    const int more = s_more;
    __syncthreads();
    if (!more) break;
  }
  for (int v = warp; v < nq; v += VE_THREADS / 32) {
    if (!s_on[v]) continue;
    for (int i = lane; i < n; i += 32) W.Z[i + (size_t)(q0 + v) * ld] = zs[i * NV + v];
    if (lane == 0) W.lam[q0 + v] = rt_val(s_lam[v]);
  }
}

inline size_t fix_smem(int n, int m) { return 16 * (size_t)n + 24 * (size_t)m + 16; }

// Clusters: estimates closer than the threshold, and all m vectors when two
// isolated ones turn out to be the same.  The estimates are refined in FP64
// (32 Sturm counts a round), kept at least 10 eps |T| apart, and every step
// of the inverse iteration is followed by modified Gram-Schmidt inside each
// cluster.  One CTA per task; most tasks have no cluster and return at once.
template <class T>
__global__ void __launch_bounds__(256) rrw_fix_kernel(const RRTask* __restrict__ tasks) {
  const RRTask Tk = tasks[blockIdx.x];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int n = W.st[0], m = Tk.m, ld = W.ld;
  if (n == 0) return;
  extern __shared__ __align__(16) unsigned char rw_raw[];
  T* d = reinterpret_cast<T*>(rw_raw);
  T* e = d + n;
  double* sh = reinterpret_cast<double*>(e + n);         // m: estimates
  double* lam = sh + m;                                  // m: eigenvalues
  int* cstart = reinterpret_cast<int*>(lam + m);         // m
  int* join = cstart + m;                                // m + 1
  __shared__ float redf[8];
  __shared__ T red[8];
  __shared__ int any, same;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = 8;
  for (int i = tid; i < n; i += 256) {
    d[i] = W.d[i];
    e[i] = W.e[i];
  }
  for (int j = tid; j < m; j += 256) {
    sh[j] = W.sh[j];
    lam[j] = W.lam[j];
  }
  if (tid == 0) any = same = 0;
  __syncthreads();
  const float gnorm = wide_gnorm(d, e, n, redf);
  const double ortol = (double)RW_ORTOL * (double)gnorm;
  // join[j]: estimate j is within the threshold of estimate j - 1
  for (int j = tid; j <= m; j += 256) {
    const bool jn = j < m && wide_joins(sh, j, ortol);
    join[j] = jn;
    if (jn) any = 1;
  }
  __syncthreads();
  auto in_cluster = [&](int j) { return join[j] || join[j + 1]; };
  // an isolated vector that left its estimate for another eigenvalue, or two
  // of them with one eigenvalue (unit vectors of distinct eigenvalues are
  // orthogonal to rounding)
  for (int j = tid; j < m; j += 256) {
    if (in_cluster(j)) continue;
    if (!(fabs(lam[j] - sh[j]) <= 0.5 * ortol)) same = 1;
    if (j + 1 < m && !in_cluster(j + 1) && !(lam[j + 1] - lam[j] > 1e-9 * (double)gnorm)) same = 1;
  }
  __syncthreads();
  const bool all = same != 0;
  if (any || all) {
  // refined shifts of the cluster members
  const double tinyd = DBL_MIN / DBL_EPSILON;
  for (int j = warp; j < m; j += NW) {
    if (!all && !in_cluster(j)) continue;
    double lo = sh[j] - 4e-6 * (double)gnorm, hi = sh[j] + 4e-6 * (double)gnorm;
    for (int round = 0; round < 9; ++round) {
      const double x = lo + (hi - lo) * ((double)(lane + 1) / 33.0);
      int c = 0;
      double qv = 1.0, ep = 0.0;
      for (int i = 0; i < n; ++i) {
        qv = rt_val(d[i]) - x - ep / qv;
        if (fabs(qv) < tinyd) qv = -tinyd;
        c += qv < 0.0;
        ep = rt_val(e[i]);
        ep *= ep;
      }
      const unsigned above = __ballot_sync(0xffffffffu, c > j);
      const int f = above ? __ffs(above) - 1 : 32;
      const double xf = __shfl_sync(0xffffffffu, x, min(f, 31));
      const double xb = __shfl_sync(0xffffffffu, x, max(f - 1, 0));
      if (f < 32) hi = xf;
      if (f > 0) lo = xb;
    }
    if (lane == 0) lam[j] = 0.5 * (lo + hi);
  }
  __syncthreads();
  if (tid == 0) {
    const double sep = 10.0 * RtOf<T>::eps * (double)gnorm;
    for (int j = 0; j < m; ++j) {
      cstart[j] = -1;
      if (!all && !in_cluster(j)) continue;
      const bool joins = all ? j > 0 : join[j] != 0;
      cstart[j] = joins ? cstart[j - 1] : j;
      if (joins) lam[j] = fmax(lam[j], lam[j - 1] + sep);
    }
  }
  __syncthreads();
  const float tiny = fmaxf((float)(RtOf<T>::eps * gnorm), 1e-36f);
  for (int it = 0; it < 3; ++it) {
    for (int q = tid; q < m; q += 256) {
      if (cstart[q] < 0) continue;
      T* z = W.Z + (size_t)q * ld;
      if (it == 0)
        for (int i = 0; i < n; ++i) z[i] = RtOf<T>::off(wide_hash(i, q + 7919u * blockIdx.x));
      T xx = RtOf<T>::off(0.0f);
      wide_tri_solve<T>(
          d, e, n, RtOf<T>::of(lam[q]), tiny, W.scr + q, (size_t)m, [&](int i) { return z[i]; },
          [&](int i, T xi) {
            const T x = RtScale<T>::down(xi);
            xx = rt_fma(x, x, xx);
            z[i] = x;
          });
      const T inv = rt_rsqrt(xx);
      for (int i = 0; i < n; ++i) z[i] = rt_mul(z[i], inv);
    }
    __syncthreads();
    for (int j = 0; j < m; ++j) {
      if (cstart[j] < 0) continue;  // uniform across the block
      T* zj = W.Z + (size_t)j * ld;
      T part = RtOf<T>::off(0.0f);
      for (int i = tid; i < n; i += 256) part = rt_fma(zj[i], zj[i], part);
      part = rt_warp_sum(part);
      if (lane == 0) red[warp] = part;
      __syncthreads();
      T s = red[0];
      for (int w = 1; w < NW; ++w) s = rt_add(s, red[w]);
      const T inv = rt_rsqrt(s);
      for (int i = tid; i < n; i += 256) zj[i] = rt_mul(zj[i], inv);
      __syncthreads();
      int kend = j + 1;
      while (kend < m && cstart[kend] == cstart[j]) ++kend;
      for (int k = j + 1 + warp; k < kend; k += NW) {
        T* zk = W.Z + (size_t)k * ld;
        T s2 = RtOf<T>::off(0.0f);
        for (int i = lane; i < n; i += 32) s2 = rt_fma(zj[i], zk[i], s2);
        s2 = rt_warp_sum(s2);
        for (int i = lane; i < n; i += 32) zk[i] = rt_fnma(s2, zj[i], zk[i]);
      }
      __syncthreads();
    }
  }
  // eigenvalues as Rayleigh quotients of the unit vectors
  for (int j = warp; j < m; j += NW) {
    if (cstart[j] < 0) continue;
    const T* zj = W.Z + (size_t)j * ld;
    T s = RtOf<T>::off(0.0f);
    for (int i = lane; i < n; i += 32) {
      T t = rt_mul(d[i], zj[i]);
      if (i > 0) t = rt_fma(e[i - 1], zj[i - 1], t);
      if (i + 1 < n) t = rt_fma(e[i], zj[i + 1], t);
      s = rt_fma(zj[i], t, s);
    }
    s = rt_warp_sum(s);
    if (lane == 0) W.lam[j] = lam[j] = rt_val(s);
  }
  __syncthreads();
  }
  // Vectors found one by one are orthogonal to eps |T| / gap: a Gram-Schmidt
  // pass over each run of near eigenvalues (a warp per run) takes care of the
  // close ones.
  const double win = RtScale<T>::window * (double)gnorm;
  auto near = [&](int j) { return j > 0 && lam[j] - lam[j - 1] <= win; };
  for (int j0 = warp; j0 < m; j0 += NW) {
    if (near(j0)) continue;
    for (int k = j0 + 1; k < m && near(k); ++k) {
      T* zk = W.Z + (size_t)k * ld;
      for (int p = k - 1; p >= j0 && lam[k] - lam[p] <= win; --p) {
        const T* zp = W.Z + (size_t)p * ld;
        T s = RtOf<T>::off(0.0f);
        for (int i = lane; i < n; i += 32) s = rt_fma(zp[i], zk[i], s);
        s = rt_warp_sum(s);
        for (int i = lane; i < n; i += 32) zk[i] = rt_fnma(s, zp[i], zk[i]);
      }
    }
  }
}

}  // namespace

}  // namespace dgdft
