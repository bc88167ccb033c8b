// Lowest eigenpairs of one dense symmetric FP64 matrix over the whole GPU (the
// DIAG route of Sec. II.B for the density: n = n_elem J up to 4096).
//
// What bounds it.  One-sided Jacobi took 13 to 16 sweeps of ~11 n^3 FP64
// operations with a grid barrier per round of pairs: 544 ms at n = 1440.
// Householder tridiagonalisation needs 4/3 n^3 and one grid barrier per
// column; the eigenpairs of the tridiagonal matrix come from the kernels of
// the Rayleigh-Ritz chain (rr_wide.cuh), and the back-transformation costs 2
// n^2 m.  All of it is FP64 work at the FP64 pipe's rate (1.2 TFLOP/s).
//
// eigh_tri_kernel deals the rows cyclically to one CTA per SM.  Up to n ~ 1,900
// they fit the SMs' shared memory together; larger matrices stay in global
// memory (L2).  A step: every CTA forms the reflector of the pivot row from
// its own copy (four warps, one per SM sub-partition: FP64 vector work on more
// warps only queues), applies the previous rank-two update to its rows and
// multiplies them by the reflector in one pass, and publishes its products
// and, from the owner, the next pivot row through L2; after the grid barrier
// (2,300 cycles) every CTA forms the update vector and the new pivot row.
// With s = sqrt(2) v the reflection is I - s s^T and the update C - s u^T -
// u s^T, u = p - (s.p / 2) s, p = C s: six FP64 operations per entry of a
// vector.  Measured, n = 1440, m = 720: 544 -> 29 ms (tridiagonalisation 17.7,
// back-transformation 5.6, vectors 5.2, location 0.2); n = 4096 with half of
// the vectors 519 ms; n = 72 (one pencil on two CTAs) 3.6 -> 0.5 ms.
#include <cooperative_groups.h>

#include <algorithm>

#include "rr_wide.cuh"

namespace dgdft {

namespace {

constexpr int EH_THREADS = 512, EH_VW = 4;

// A <- (A + A^T) / 2
__global__ void eigh_sym_kernel(double* __restrict__ A, int n) {
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < (size_t)n * n; q += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(q / n), j = (int)(q - (size_t)i * n);
    if (j >= i) continue;
    const double s = 0.5 * (A[q] + A[(size_t)j * n + i]);
    A[q] = s;
    A[(size_t)j * n + i] = s;
  }
}

__global__ void eigh_state_kernel(const RRTask* __restrict__ task) {
  const WideWork<double> W = wide_carve<double>(*task);
  W.st[0] = W.ld;
  W.st[1] = 0;
  W.st[2] = 1;
}

__host__ __device__ inline int eigh_ld(int n) { return n | 1; }
size_t eigh_smem(int n, int ncta, bool rows) {
  const size_t R = (n + ncta - 1) / ncta;
  return 8 * (4 * (size_t)n + (rows ? R * eigh_ld(n) : 0)) + 256;
}

// rows: the CTA's rows in shared memory, else in place in W.C.  xchg: two sets
// of (n products, n entries of the next pivot row).  Reflector k (unit, H = I
// - 2 v v^T) goes to column k of W.X.
template <bool ROWS>
__global__ void __launch_bounds__(EH_THREADS, 1) eigh_tri_kernel(const RRTask* __restrict__ task,
                                                                 double* __restrict__ xchg) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  const WideWork<double> W = wide_carve<double>(*task);
  const int n = W.ld, G = gridDim.x, rank = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int VT = 32 * EH_VW, NW = EH_THREADS / 32;
  extern __shared__ __align__(16) unsigned char eh_raw[];
  double* sb = reinterpret_cast<double*>(eh_raw);  // 2: s of this step and the one before
  double* uv = sb + 2 * (size_t)n;
  double* rcur = uv + n;
  double* S = ROWS ? rcur + n : W.C;
  const size_t ldS = ROWS ? eigh_ld(n) : n;
  __shared__ double red[2][EH_VW], sx0;
  const int R = (n - rank + G - 1) / G;
  auto row_of = [&](int t) { return S + (ROWS ? (size_t)t : (size_t)(rank + G * t)) * ldS; };
  auto vsum = [&](double s, int slot) {
    s = warp_sum(s);
    if (lane == 0) red[slot][warp] = s;
    asm volatile("bar.sync 1, %0;" ::"n"(VT) : "memory");
    s = red[slot][0];
#pragma unroll
    for (int w = 1; w < EH_VW; ++w) s += red[slot][w];
    return s;
  };
  if (ROWS)
    for (int t = warp; t < R; t += NW)
      for (int j = lane; j < n; j += 32) S[t * ldS + j] = W.C[(size_t)(rank + G * t) * n + j];
  if (warp < EH_VW)
    for (int j = tid; j < n; j += VT) rcur[j] = W.C[j];
  __syncthreads();
  for (int k = 0; k + 2 < n; ++k) {
    const int par = k & 1;
    double* s = sb + (size_t)par * n;
    const double* so = sb + (size_t)(par ^ 1) * n;
    double* gp = xchg + (size_t)par * 2 * n;
    double* gr = gp + n;
    double s1 = 0.0;  // s[k+1]
    if (warp < EH_VW) {
      double a = 0.0;
      const int j0 = tid + (k + 1 - tid + VT - 1) / VT * VT;  // this thread's first entry past k
      const int jb = k + 1 > tid ? j0 : tid;
      for (int j = jb; j < n; j += VT) a = fma(rcur[j], rcur[j], a);
      if (tid == 0) sx0 = rcur[k + 1];
      const double xx = vsum(a, 0);
      const double x0 = sx0;
      double alpha = x0, inv = 0.0;
      if (xx > 0.0 && isfinite(xx)) {
        const double nx = xx * rsqrt(xx);
        alpha = x0 >= 0.0 ? -nx : nx;
        // |x - alpha e_1|^2 / 2 = |x|^2 + |x| |x_0|, no cancellation
        inv = rsqrt(fma(nx, fabs(x0), xx));
      }
      s1 = (x0 - alpha) * inv;
      if (rank == 0 && tid == 0) {
        W.d[k] = rcur[k];
        W.e[k] = alpha;
      }
      const bool mine = rank == k % G;
      for (int j = jb; j < n; j += VT) {
        const double sj = j == k + 1 ? s1 : rcur[j] * inv;
        s[j] = sj;
        if (mine) W.X[(size_t)k * n + j] = sj * 0.70710678118654752440;
      }
    }
    __syncthreads();
    // own rows past k: previous update, product with s; a warp per row
    const int t0 = k + 1 > rank ? (k + 1 - rank + G - 1) / G : 0;
    for (int t = t0 + warp; t < R; t += NW) {
      const int i = rank + G * t;
      double* row = row_of(t);
      double acc0 = 0.0, acc1 = 0.0;
      const double si = so[i], ui = uv[i];
      const bool next = i == k + 1;
      for (int jb = k + 1; jb < n; jb += 64) {
        const int ja = jb + lane, jc = ja + 32;
        double c0 = ja < n ? row[ja] : 0.0, c1 = 0.0;
        const bool two = jb + 32 < n;  // uniform
        if (two) c1 = jc < n ? row[jc] : 0.0;
        if (k > 0) {
          if (ja < n) {
            c0 = fma(-ui, so[ja], fma(-si, uv[ja], c0));
            row[ja] = c0;
          }
          if (two && jc < n) {
            c1 = fma(-ui, so[jc], fma(-si, uv[jc], c1));
            row[jc] = c1;
          }
        }
        if (ja < n) acc0 = fma(c0, s[ja], acc0);
        if (two && jc < n) acc1 = fma(c1, s[jc], acc1);
        if (next) {
          if (ja < n) gr[ja] = c0;
          if (jc < n) gr[jc] = c1;
        }
      }
      const double p = warp_sum(acc0 + acc1);
      if (lane == 0) gp[i] = p;
    }
    grid.sync();
    if (warp < EH_VW) {
      const int j0 = tid + (k + 1 - tid + VT - 1) / VT * VT;
      const int jb = k + 1 > tid ? j0 : tid;
      double a = 0.0;
      for (int j = jb; j < n; j += VT) {
        const double p = __ldcg(gp + j);
        uv[j] = p;
        rcur[j] = __ldcg(gr + j);
        a = fma(s[j], p, a);
      }
      const double K = 0.5 * vsum(a, 1);
      const double u1 = fma(-K, s1, uv[k + 1]);
      asm volatile("bar.sync 1, %0;" ::"n"(VT) : "memory");  // uv[k + 1] is read by all before it changes
      for (int j = jb; j < n; j += VT) {
        const double sj = s[j], u = fma(-K, sj, uv[j]);
        uv[j] = u;
        rcur[j] = fma(-u1, sj, fma(-s1, u, rcur[j]));
      }
      asm volatile("bar.sync 1, %0;" ::"n"(VT) : "memory");
    }
  }
  __syncthreads();
  if (rank == 0 && tid == 0 && n >= 2) {
    W.d[n - 2] = rcur[n - 2];
    W.e[n - 2] = rcur[n - 1];
  }
  if (rank == (n - 1) % G && tid == 0) {
    double c = row_of((n - 1) / G)[n - 1];
    if (n >= 3) c = fma(-2.0 * sb[(size_t)((n - 3) & 1) * n + n - 1], uv[n - 1], c);
    W.d[n - 1] = c;
    W.e[n - 1] = 0.0;
  }
}

// y = H_0 ... H_{n-3} z for NV eigenvectors per CTA held in shared memory, a
// warp per vector; the reflectors come through shared memory, EK at a time,
// the next ones on their way.
size_t eigh_back_smem(int n, int vecs, int ek) { return 8 * (size_t)n * (vecs + 2 * ek); }

template <int NV, int EK>
__global__ void __launch_bounds__(32 * NV) eigh_back_kernel(const RRTask* __restrict__ task) {
  const RRTask Tk = *task;
  const WideWork<double> W = wide_carve<double>(Tk);
  const int n = W.ld, m = Tk.m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ __align__(16) unsigned char eh_raw[];
  double* buf = reinterpret_cast<double*>(eh_raw);  // 2 x EK reflectors
  double* z = buf + (size_t)2 * EK * n + (size_t)warp * n;
  const int c = blockIdx.x * NV + warp;
  auto stage = [&](int k0) {  // reflectors k0 .. k0 + EK - 1
    double* b = buf + (size_t)((k0 / EK) & 1) * EK * n;
    for (int u = 0; u < EK; ++u) {
      const int k = k0 + u;
      if (k + 2 >= n) continue;
      for (int i = k + 1 + tid; i < n; i += 32 * NV)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(shared_addr(b + (size_t)u * n + i)),
                     "l"(W.X + (size_t)k * n + i)
                     : "memory");
    }
    cp_async_commit();
  };
  if (c < m)
    for (int i = lane; i < n; i += 32) z[i] = W.Z[(size_t)c * n + i];
  const int ktop = n > 2 ? (n - 3) / EK * EK : -EK;
  if (ktop >= 0) stage(ktop);
  for (int k0 = ktop; k0 >= 0; k0 -= EK) {
    if (k0 > 0) {
      stage(k0 - EK);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const double* b = buf + (size_t)((k0 / EK) & 1) * EK * n;
    if (c < m)
      for (int u = EK - 1; u >= 0; --u) {
        const int k = k0 + u;
        if (k + 2 >= n) continue;
        const double* v = b + (size_t)u * n;
        double s0 = 0.0, s1 = 0.0;
        int i = k + 1 + lane;
        for (; i + 32 < n; i += 64) {
          s0 = fma(v[i], z[i], s0);
          s1 = fma(v[i + 32], z[i + 32], s1);
        }
        if (i < n) s0 = fma(v[i], z[i], s0);
        const double s = 2.0 * warp_sum(s0 + s1);
        for (int q = k + 1 + lane; q < n; q += 32) z[q] = fma(-s, v[q], z[q]);
      }
    __syncthreads();
  }
  if (c >= m) return;
  for (int i = lane; i < n; i += 32) Tk.Y[(size_t)c * Tk.ldy + i] = z[i];
  if (lane == 0) Tk.theta[c] = W.lam[c];
}

}  // namespace

size_t eigh_work_doubles(int n, int m) { return wide_work_doubles(n, m) + 4 * (size_t)n; }

double* eigh_matrix(const RRTask& t) { return t.work + (size_t)3 * t.n_fixed * t.n_fixed; }

cudaError_t launch_eigh(const RRTask& h, const RRTask* d_task, cudaStream_t st) {
  const int n = h.n_fixed, m = h.m;
  eigh_sym_kernel<<<1024, 256, 0, st>>>(eigh_matrix(h), n);
  eigh_state_kernel<<<1, 1, 0, st>>>(d_task);
  if (n <= 608) {
    launch_rr_standard(d_task, n, m, st);
    return cudaGetLastError();
  }
  int dev = 0, nsm = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  double* xchg = h.work + wide_work_doubles(n, m);
  const bool rows = eigh_smem(n, nsm, true) + 512 <= (size_t)optin;
  void* args[] = {(void*)&d_task, (void*)&xchg};
  const void* tri = rows ? (const void*)eigh_tri_kernel<true> : (const void*)eigh_tri_kernel<false>;
  const void* big[] = {tri, (const void*)rrw_vec_kernel<double, 2, false>, (const void*)rrw_vec_kernel<double, 1, false>,
                       (const void*)rrw_fix_kernel<double>, (const void*)eigh_back_kernel<8, 4>,
                       (const void*)eigh_back_kernel<2, 2>};
  for (const void* k : big) opt_in_dynamic_smem(k);
  cudaError_t e = cudaLaunchCooperativeKernel(tri, dim3(nsm), dim3(EH_THREADS), args, eigh_smem(n, nsm, rows), st);
  if (e != cudaSuccess) return e;
  const int per = BI_WARPS * BI_PER;
  rrw_bisect_kernel<double><<<dim3((m + per - 1) / per, 1), 32 * BI_WARPS, 8 * (size_t)n, st>>>(d_task);
  if (vec_smem(n, 2, false) + 2048 <= (size_t)optin)
    rrw_vec_kernel<double, 2, false><<<dim3((m + 1) / 2, 1), VE_THREADS, vec_smem(n, 2, false), st>>>(d_task);
  else
    rrw_vec_kernel<double, 1, false><<<dim3(m, 1), VE_THREADS, vec_smem(n, 1, false), st>>>(d_task);
  rrw_fix_kernel<double><<<1, 256, fix_smem(n, m), st>>>(d_task);
  // eight vectors share a CTA's reads of the reflectors while they fit (n <=
  // 1,800); two and shorter stages hold up to 4096
  if (eigh_back_smem(n, 8, 4) + 1024 <= (size_t)optin)
    eigh_back_kernel<8, 4><<<(m + 7) / 8, 256, eigh_back_smem(n, 8, 4), st>>>(d_task);
  else
    eigh_back_kernel<2, 2><<<(m + 1) / 2, 64, eigh_back_smem(n, 2, 2), st>>>(d_task);
  return cudaGetLastError();
}

}  // namespace dgdft
