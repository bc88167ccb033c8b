// Rayleigh-Ritz of a LOBPCG pencil (Sec. II.B, operation 4) spread over many
// SMs: a chain of kernels instead of one CTA per pencil.
//
// What bounds it.  On this part a warp's FP64 instruction holds its SM
// sub-partition for 64 cycles (0.5 lane per cycle; an SM with all four busy
// takes one per 19 cycles), so an FP64 1/x or 1/sqrt(x) costs 440 cycles and a
// five-step shuffle sum 520.  One CTA per pencil is then bound by one SM's
// FP64 pipe (n^3 multiply-adds and more: 76 ms at n = 432, m = 144) or, for
// small n, by FP64 work done redundantly by all of its warps (1.07 ms at
// n = 40).  In pair arithmetic (dfl: 2^-46 relative, far below the ~1e-7 that
// the FP32 stage's Gram blocks carry; a multiply-add costs 17 FP32
// instructions) one CTA took 2.2 ms at n = 144, over half of it in products
// that need no barrier.
//
// The split.  What carries a dependency across the whole matrix runs in one
// thread-block cluster per pencil (rrw_chol_kernel, rrw_tri_kernel): rows are
// dealt cyclically to its CTAs and stay in shared memory, a step's column (or
// matrix-vector product) is written into every CTA's shared memory, and a
// step needs one cluster barrier; scalars are formed by one warp of each CTA.
// What has independent columns (both triangular solves, the
// back-transformation and L^-T) gives a column to a warp of the whole GPU,
// held in registers.  The eigenvalues are located by FP32 Sturm counts, a warp
// per eigenvalue; isolated eigenvectors take one FP32 inverse iteration and
// then Rayleigh-quotient iterations, a thread per vector; close eigenvalues
// are located to full precision and orthogonalised in one CTA
// (rrw_fix_kernel).  The arithmetic type T is double or dfl, as the caller
// asks.
//
// Nothing spins: the cluster barriers are the hardware's, every CTA of a
// cluster takes the same decisions from the same data, and each loop is
// bounded by the matrix size.
//
// Measured (cycles at 2.07 GHz, one pencil).  FP64, n = 432, m = 144, 16 CTAs:
// factorisation 1.6 M, solves 2 x 0.5 M, tridiagonalisation 7.5 M (17,400 a
// step: 8,050 the pass over the rows, 3,380 the reflector, 3,400 the barrier
// and its messages), location 0.15 M, vectors 1.5 M, back-transformation
// 1.25 M.  dfl, n = 144, m = 48, 4 CTAs: 0.33 M, 2 x 0.05 M, 1.1 M, 0.05 M,
// 0.2 M, 0.16 M.  FP64, n = 48, one CTA: 0.07 M, 2 x 0.02 M, 0.25 M, 0.02 M,
// 0.08 .. 0.18 M, 0.06 M.
#include "rr_wide.cuh"

namespace dgdft {

namespace {

// ---------------------------------------------------------------- clusters

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// a step's barrier: the cluster's, or the CTA's own where a pencil has one CTA
__device__ __forceinline__ void cl_sync(int cs) {
  if (cs > 1) {
    cl_arrive();
    cl_wait();
  } else {
    __syncthreads();
  }
}
// store into the same shared-memory location of CTA `dst` of the cluster
template <class T> __device__ __forceinline__ void cl_store(T* p, T v, int dst) {
  static_assert(sizeof(T) == 8, "8-byte values");
  unsigned long long bits;
  memcpy(&bits, &v, 8);
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(shared_addr(p)), "r"(dst));
  asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(bits) : "memory");
}

size_t chol_smem(int n, int cs) {
  const size_t R = (n + cs - 1) / cs;
  return 8 * (R * (n | 1) + 3 * (size_t)n + R + 2 * (size_t)n) + 128;
}
// row stride of the tridiagonalisation: 8 (mod 16) values, two rows' starts
// 16 banks apart
__host__ __device__ inline int tri_ld(int n) { return (n + 7) / 16 * 16 + 8; }
size_t tri_smem(int n, int cs) {
  const size_t R = (n + cs - 1) / cs;
  return 8 * (R * tri_ld(n) + 7 * (size_t)n + R) + 512;
}

// ---------------------------------------------------------------- Cholesky

// Equilibrated B = D B D = L L^T, D = diag(B)^-1/2, with the pivot-ratio
// condition check and the LOBPCG fallbacks (without P, then X alone, then a
// restart), one cluster of cs CTAs per task.  CTA `rank` holds rows i = rank +
// cs t up to the diagonal.  Step k: every CTA finishes its rows' entries of
// column k (still unscaled, c_i) and writes them to all CTAs; while they
// travel, the rest of the rows take the update of step k - 1; after the
// barrier c_kk is the pivot and f_i = c_i / c_kk.  Columns are scaled to L by
// 1 / sqrt(c_kk) once, at the end.  Three column buffers: a CTA that has
// arrived may still read column k - 2 while others already write column k.
// ONE (a pencil per CTA, n <= 160): warp 0 finishes column k + 1 and its pivot
// while the other warps update the rest with column k; one CTA barrier per step.
template <class T, bool ONE>
__global__ void __launch_bounds__(RW_THREADS, 1) rrw_chol_kernel(const RRTask* __restrict__ tasks, int cs, int nmax) {
  const int rank = blockIdx.x % cs;
  const RRTask Tk = tasks[blockIdx.x / cs];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = Tk.m;
  // the state words are read by every CTA of the cluster before any writes them
  const bool active = !Tk.state || Tk.state[ST_ACTIVE];
  const bool stale = Tk.state && (Tk.state[ST_ERROR] & ERR_TIMEOUT);
  const bool has_p = Tk.mode == RR_LOBPCG && Tk.state[ST_HAS_P];
  const bool can_restart =
      Tk.mode == RR_LOBPCG && Tk.restart_max > 0 && Tk.state && Tk.state[ST_NRESTART] < Tk.restart_max;
  cl_sync(cs);
  if (!active || stale) {
    if (rank == 0 && tid == 0) {
      W.st[0] = 0;
      // a wait in this iteration's Gram launch ran out: its products are stale
      if (active) Tk.state[ST_ACTIVE] = 0;
    }
    return;
  }
  extern __shared__ __align__(16) unsigned char rw_raw[];
  T* col = reinterpret_cast<T*>(rw_raw);            // 3 columns
  T* pd = col + 3 * (size_t)nmax;                   // pivots
  T* scal = pd + nmax;
  T* f = scal + nmax;
  T* S = f + (nmax + cs - 1) / cs;
  __shared__ int sflag, sfail, spiv[2];
  int n = (Tk.mode == RR_FIXED) ? Tk.n_fixed : (Tk.mode == RR_INITIAL) ? m : (has_p ? 3 * m : 2 * m);
  const int bm = (Tk.mode == RR_FIXED) ? n : m;
  bool dropped = false;
  for (;;) {
    const int R = (n - rank + cs - 1) / cs, ldS = n | 1;
    if (tid == 0) sflag = spiv[0] = spiv[1] = 0;
    cl_sync(cs);  // the previous attempt's columns are done with
    for (int i = tid; i < n; i += RW_THREADS) {
      const double bii = Tk.B[i + (size_t)i * Tk.ld];
      if (!(bii > 0.0) || !isfinite(bii)) {
        sflag = 1;
        scal[i] = RtOf<T>::off(0.0f);
      } else {
        scal[i] = RtOf<T>::of(1.0 / sqrt(bii));
      }
    }
    __syncthreads();
    bool bad = sflag != 0;  // the same in every CTA
    for (int t = warp; t < R; t += RW_WARPS) {
      const int i = rank + cs * t;
      const T si = scal[i];
      for (int j = lane; j <= i; j += 32)
        S[t * ldS + j] = rt_mul(rt_mul(RtOf<T>::of(wide_sym(Tk.B, Tk.ld, i, j, bm)), si), scal[j]);
    }
    __syncthreads();
    if constexpr (ONE) {
      // pivot k by warp 0: L_kk apart in pd (as its square) and f (its
      // reciprocal), column k scaled
      auto pivot = [&](int k) {
        const T p = S[k * ldS + k];
        if (!rt_pos(p)) {
          if (lane == 0) spiv[k & 1] = 1;
          return;
        }
        const T rs = rt_rsqrt(p);
        if (lane == 0) {
          pd[k] = p;
          f[k] = rs;
        }
        for (int i = k + 1 + lane; i < n; i += 32) S[i * ldS + k] = rt_mul(S[i * ldS + k], rs);
      };
      if (warp == 0 && !bad) pivot(0);
      __syncthreads();
      for (int k = 0; k + 1 < n; ++k) {
        // uniform: pivot k was formed before the last barrier, pivot k + 1
        // reports in the other word
        if (bad || spiv[k & 1]) break;
        const int j1 = k + 1;
        if (warp == 0) {
          const T lj = S[j1 * ldS + k];
          for (int i = j1 + lane; i < n; i += 32) S[i * ldS + j1] = rt_fnma(S[i * ldS + k], lj, S[i * ldS + j1]);
          __syncwarp();
          pivot(j1);
        } else {
          // NB rows i, i + 15, ... at a time: their chains interleave, and they
          // share the loads of column k
          auto rows = [&](auto nb_c, int i0) {
            constexpr int NB = decltype(nb_c)::value;
            T li[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) li[b] = S[(i0 + (RW_WARPS - 1) * b) * ldS + k];
            for (int j = j1 + 1 + lane; j <= i0 + (RW_WARPS - 1) * (NB - 1); j += 32) {
              const T lj = S[j * ldS + k];
              T c[NB];
#pragma unroll
              for (int b = 0; b < NB; ++b) c[b] = rt_fnma(li[b], lj, S[(i0 + (RW_WARPS - 1) * b) * ldS + j]);
#pragma unroll
              for (int b = 0; b < NB; ++b)
                if (j <= i0 + (RW_WARPS - 1) * b) S[(i0 + (RW_WARPS - 1) * b) * ldS + j] = c[b];
            }
          };
          int i = j1 + warp;
          for (; i + 3 * (RW_WARPS - 1) < n; i += 4 * (RW_WARPS - 1)) rows(std::integral_constant<int, 4>(), i);
          for (; i + (RW_WARPS - 1) < n; i += 2 * (RW_WARPS - 1)) rows(std::integral_constant<int, 2>(), i);
          if (i < n) rows(std::integral_constant<int, 1>(), i);
        }
        __syncthreads();
      }
      bad = bad || spiv[0] || spiv[1];
      __syncthreads();
    } else
    for (int k = 0; k < n && !bad; ++k) {
      T* cb = col + (size_t)(k % 3) * nmax;
      const T* cp = col + (size_t)((k + 2) % 3) * nmax;
      for (int dst = warp; dst < cs; dst += RW_WARPS)
        for (int t = lane; t < R; t += 32) {
          const int i = rank + cs * t;
          if (i < k) continue;
          T v = S[t * ldS + k];
          if (k > 0) v = rt_fnma(f[t], cp[k], v);
          if (cs > 1) cl_store(cb + i, v, dst);
          else cb[i] = v;
        }
      if (cs > 1) cl_arrive();
      if (k > 0)
        for (int t = warp; t < R; t += RW_WARPS) {
          const int i = rank + cs * t;
          const T ft = f[t];
          for (int j = k + 1 + lane; j <= i; j += 32) S[t * ldS + j] = rt_fnma(ft, cp[j], S[t * ldS + j]);
        }
      if (cs > 1) cl_wait();
      __syncthreads();  // this CTA's warps are done with f and column k - 1
      const T p = cb[k];
      if (!rt_pos(p)) {
        bad = true;
        break;
      }
      if (tid < R) {
        const int i = rank + cs * tid;
        const T inv = rt_rcp(p);
        if (i >= k) {
          const T c = cb[i];
          S[tid * ldS + k] = c;
          f[tid] = rt_mul(c, inv);
        }
      }
      if (tid == 0) pd[k] = p;
      __syncthreads();
    }
    // condition: ratio of the extreme pivots.  The last LOBPCG resort (X
    // alone) takes any positive-definite B: its Rayleigh-Ritz
    // re-orthonormalises a block that has drifted
    if (!bad && warp == 0) {
      double lo = DBL_MAX, hi = 0.0;
      for (int k = lane; k < n; k += 32) {
        const double p = rt_val(pd[k]);
        lo = fmin(lo, p);
        hi = fmax(hi, p);
      }
      for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      }
      const bool last_resort = Tk.mode == RR_LOBPCG && n == m;
      const double lim = last_resort ? (Tk.restart_max > 0 ? 1e6 : 1e300) : Tk.cond_max;
      if (lane == 0) sfail = hi / lo > lim;
    }
    __syncthreads();
    if (!bad && !sfail) break;
    __syncthreads();
    if (Tk.mode == RR_LOBPCG && n > m) {
      // without P; then X alone, a rotation of the current block (the next
      // iteration brings a new W)
      n = (n == 3 * m) ? 2 * m : m;
      dropped = true;
      continue;
    }
    if (rank == 0) {
      if (can_restart) {
        // no usable pencil, not even X alone: keep X (Y = [I; 0]) and let
        // the restart step perturb it and drop P (Ritz values unchanged)
        const int nr = 3 * m;
        for (int idx = tid; idx < nr * m; idx += RW_THREADS) {
          const int r = idx % nr, c = idx / nr;
          const double y = (r == c) ? 1.0 : 0.0;
          Tk.Y[r + (size_t)c * Tk.ldy] = y;
          if (Tk.Yf) Tk.Yf[r + (size_t)c * Tk.ldy] = (float)y;
        }
      }
      if (tid == 0) {
        W.st[0] = 0;
        if (can_restart) {
          Tk.state[ST_RESTART] = 1;
          Tk.state[ST_NRESTART] += 1;
          Tk.state[ST_FALLBACK] += 1;
        } else if (Tk.state) {
          Tk.state[ST_ERROR] |= ERR_CHOL;
          Tk.state[ST_ACTIVE] = 0;
        } else {
          Tk.theta[0] = __longlong_as_double(0x7ff8000000000000LL);
        }
      }
    }
    return;
  }
  // L (strictly lower, by columns) and its transpose, 1 / L_kk apart
  for (int k = tid; k < n; k += RW_THREADS) {
    const T rs = ONE ? f[k] : rt_rsqrt(pd[k]);
    pd[k] = rs;
    if (rank == 0) {
      W.rinv[k] = rs;
      W.scal[k] = scal[k];
    }
  }
  if (rank == 0 && tid == 0) {
    W.st[0] = n;
    W.st[1] = dropped;
    W.st[2] = 0;
  }
  __syncthreads();
  const int R = (n - rank + cs - 1) / cs, ldS = n | 1;
  for (int t = warp; t < R; t += RW_WARPS) {
    const int i = rank + cs * t;
    for (int k = lane; k < n; k += 32) {
      const T v = (k >= i) ? RtOf<T>::off(0.0f) : ONE ? S[t * ldS + k] : rt_mul(S[t * ldS + k], pd[k]);
      W.LT[k + (size_t)i * W.ld] = v;
      if (!ONE) W.L[i + (size_t)k * W.ld] = v;
    }
  }
  if (ONE)
    for (int k = warp; k < n; k += RW_WARPS)
      for (int i = lane; i < n; i += 32) W.L[i + (size_t)k * W.ld] = (i > k) ? S[i * ldS + k] : RtOf<T>::off(0.0f);
}

// ---------------------------------------------------------------- triangular solves

// Columns k0 .. k0 + KC - 1 of an n x n matrix (leading dimension ld) into
// shared memory, asynchronously, by a CTA of 128 threads; rows from n on stay
// as they are (the readers' registers for them hold zeros, and the buffers
// start as zeros).
constexpr int KC = 8;
template <class T>
__device__ __forceinline__ void stage_columns(T* buf, int ldb, const T* M, int ld, int n, int k0) {
  for (int c = threadIdx.x >> 5; c < KC; c += 4) {
    const int k = k0 + c;
    if (k >= 0 && k < n)
      for (int i = threadIdx.x & 31; i < n; i += 32)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(shared_addr(buf + c * ldb + i)),
                     "l"(M + i + (size_t)k * ld)
                     : "memory");
  }
  cp_async_commit();
}

// pass 0: column c of X = L^-1 (D A D), stored transposed; pass 1: column c of
// C = L^-1 X^T = L^-1 (D A D) L^-T.  A warp per column, row 32 r + lane in
// register r; step k broadcasts x_k and subtracts x_k times column k of L
// (zero up to row k).  The four warps of a CTA take the columns of L from
// shared memory, KC at a time, the next KC on their way: straight from L2 a
// step waited ~900 cycles for its column.  The loop over KC stays rolled: the
// register index needs the outer loop unrolled, and both unrolled do not fit
// the instruction cache.
template <class T, int NR>
__global__ void __launch_bounds__(128) rrw_solve_kernel(const RRTask* __restrict__ tasks, int pass) {
  const RRTask Tk = tasks[blockIdx.y];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int n = W.st[0];
  if ((int)blockIdx.x * 4 >= n) return;  // the whole CTA
  const int lane = threadIdx.x & 31, c = blockIdx.x * 4 + (threadIdx.x >> 5);
  constexpr int ldb = 32 * NR;
  extern __shared__ __align__(16) unsigned char rw_raw[];
  T* buf = reinterpret_cast<T*>(rw_raw);  // 2 x KC columns
  const T zero = RtOf<T>::off(0.0f);
  for (int i = threadIdx.x; i < 2 * KC * ldb; i += 128) buf[i] = zero;
  __syncthreads();
  stage_columns(buf, ldb, W.L, W.ld, n, 0);
  const int bm = (Tk.mode == RR_FIXED) ? n : Tk.m;
  T x[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int i = 32 * r + lane;
    if (i >= n || c >= n) x[r] = zero;
    else if (pass == 0)
      x[r] = rt_mul(rt_mul(RtOf<T>::of(wide_sym(Tk.A, Tk.ld, i, c, bm)), W.scal[i]), W.scal[c]);
    else x[r] = W.X[i + (size_t)c * W.ld];
  }
#pragma unroll
  for (int rk = 0; rk < NR; ++rk) {
    T rinv = (32 * rk + lane < n) ? W.rinv[32 * rk + lane] : zero;
    for (int l0 = 0; l0 < 32; l0 += KC) {
      const int k0 = 32 * rk + l0;
      if (k0 >= n) break;  // uniform
      const T* cur = buf + ((k0 / KC) & 1) * KC * ldb;
      if (k0 + KC < n) {
        stage_columns(buf + (((k0 / KC) & 1) ^ 1) * KC * ldb, ldb, W.L, W.ld, n, k0 + KC);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
#pragma unroll 1
      for (int u = 0; u < KC; ++u) {
        if (k0 + u >= n) break;
        const T xk = rt_mul(rt_shfl(x[rk], l0 + u), rt_shfl(rinv, l0 + u));
#pragma unroll
        for (int r = rk; r < NR; ++r) x[r] = rt_fnma(cur[u * ldb + 32 * r + lane], xk, x[r]);
        if (lane == l0 + u) x[rk] = xk;
      }
      __syncthreads();
    }
  }
  if (c >= n) return;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int i = 32 * r + lane;
    if (i >= n) continue;
    if (pass == 0) W.X[c + (size_t)i * W.ld] = x[r];
    else W.C[i + (size_t)c * W.ld] = x[r];
  }
}

// ---------------------------------------------------------------- tridiagonalisation

// Householder tridiagonalisation of C, one cluster of cs CTAs per task; CTA
// `rank` holds the full rows i = rank + cs t.  Every CTA knows the current
// pivot row, so it forms the reflector v itself; one pass over its rows
// applies the previous step's rank-two update and multiplies by v; the
// products p_i and the next pivot row go to all CTAs; after the barrier each
// forms w = 2 p - 2 (v.p) v and updates the pivot row.  One cluster barrier
// per step.  Work on the vectors belongs to the first VW warps, which agree
// through a barrier of their own: on all 16 warps its FP64 instructions would
// queue (19 cycles each), and the CTA's barriers cost more than the work.
// Reflector k (unit, H = I - 2 v v^T) goes to column k of W.X.
// The pass gives small matrices (LPR = 8) eight lanes per row, so that four
// rows' sums take three shuffle steps together (the rows of the four start 16
// banks apart); larger ones (LPR = 32) a warp per RG rows, which share the
// loads of the vectors and fold their sums: 6 additions for four rows, 5 for two.
template <class T, int VW, int LPR, int RG>
__global__ void __launch_bounds__(RW_THREADS, 1) rrw_tri_kernel(const RRTask* __restrict__ tasks, int cs, int nmax) {
  const int rank = blockIdx.x % cs;
  const RRTask Tk = tasks[blockIdx.x / cs];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int n = W.st[0], ld = W.ld;
  if (n == 0) return;  // the same for the whole cluster
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int VT = 32 * VW, EPT = 5;  // entries of a vector per thread of the group (n <= 160 VW)
  extern __shared__ __align__(16) unsigned char rw_raw[];
  T* vb = reinterpret_cast<T*>(rw_raw);  // 2 vectors: v of this step and the one before
  T* pb = vb + 2 * (size_t)nmax;         // 2: products of all rows
  T* rb = pb + 2 * (size_t)nmax;         // 2: next pivot row
  T* wv = rb + 2 * (size_t)nmax;
  T* psm = wv + nmax;
  T* S = psm + (nmax + cs - 1) / cs;
  __shared__ T red[2][VW], sx0;
  const int R = (n - rank + cs - 1) / cs, ldS = tri_ld(n);
  const T half = RtOf<T>::off(0.5f), zero = RtOf<T>::off(0.0f), two = RtOf<T>::off(2.0f);
  auto vsync = [&]() {
    if (VW > 1) asm volatile("bar.sync 1, %0;" ::"n"(VT) : "memory");
    else __syncwarp();
  };
  // sum over the vector group, the same value in all of its threads
  auto vsum = [&](T s, int slot) {
    s = rt_warp_sum(s);
    if (VW > 1 && lane == 0) red[slot][warp] = s;
    vsync();
    if (VW > 1) {
      s = red[slot][0];
#pragma unroll
      for (int w = 1; w < VW; ++w) s = rt_add(s, red[slot][w]);
    }
    return s;
  };
  if (cs == 1) {
    for (int i = warp; i < n; i += RW_WARPS)
      for (int j = lane; j < n; j += 32) S[i * ldS + j] = W.C[j + (size_t)i * ld];
    __syncthreads();
    for (int i = warp; i < n; i += RW_WARPS)
      for (int j = lane; j < i; j += 32) {
        const T c = rt_mul(half, rt_add(S[i * ldS + j], S[j * ldS + i]));
        S[i * ldS + j] = c;
        S[j * ldS + i] = c;
      }
  } else {
    for (int t = warp; t < R; t += RW_WARPS) {
      const int i = rank + cs * t;
      for (int j = lane; j < n; j += 32)
        S[t * ldS + j] = rt_mul(half, rt_add(W.C[j + (size_t)i * ld], W.C[i + (size_t)j * ld]));
    }
  }
  // the group's vectors stay in registers: entry tid + VT q in slot q, slots
  // wholly at or below the pivot are skipped
  T rc[EPT], vr[EPT], v1 = zero;
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    const int j = tid + VT * q;
    rc[q] = (warp < VW && j < n) ? rt_mul(half, rt_add(W.C[j], W.C[(size_t)j * ld])) : zero;
    vr[q] = zero;
  }
  if (rank == 0 && tid == 0) W.d[0] = rc[0];
  cl_sync(cs);  // every CTA runs before any writes into another's shared memory
  for (int k = 0; k + 2 < n; ++k) {
    const int par = k & 1;
    T* v = vb + (size_t)par * nmax;
    const T* vo = vb + (size_t)(par ^ 1) * nmax;
    if (warp < VW) {
      // reflector of the pivot row: x = row[k+1..], alpha = -sign(x_0) |x|,
      // v = (x - alpha e_1) / |x - alpha e_1| (zero when x = 0)
      T s = zero;
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int j = tid + VT * q;
        if (VT * (q + 1) <= k + 1 || VT * q >= n) continue;  // uniform
        if (j == k + 1) sx0 = rc[q];
        if (j <= k) rc[q] = zero;
        s = rt_fma(rc[q], rc[q], s);
      }
      const T xx = vsum(s, 0);
      const T x0 = sx0;
      T alpha = x0, inv = zero;
      if (rt_pos(xx)) {
        const T nx = rt_mul(xx, rt_rsqrt(xx));
        alpha = rt_nonneg(x0) ? rt_neg(nx) : nx;
        // |x - alpha e_1|^2 = 2 (|x|^2 + |x| |x_0|), no cancellation
        inv = rt_rsqrt(rt_mul(two, rt_fma(nx, rt_abs(x0), xx)));
      }
      v1 = rt_mul(rt_sub(x0, alpha), inv);
      if (rank == 0 && tid == 0) W.e[k] = alpha;
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int j = tid + VT * q;
        if (VT * (q + 1) <= k + 1 || VT * q >= n) continue;
        vr[q] = (j == k + 1) ? v1 : rt_mul(rc[q], inv);
        if (j > k && j < n) {
          v[j] = vr[q];
          if (rank == k % cs) W.X[j + (size_t)k * ld] = vr[q];
        }
      }
    }
    __syncthreads();
    // own rows: previous update, product with v
    const int t0 = k + 1 > rank ? (k + 1 - rank + cs - 1) / cs : 0;  // first row past k
    T* pout = cs > 1 ? psm : pb + (size_t)par * nmax;
    if constexpr (LPR == 32) {
      // NB rows tb + 16 b of this warp (a constant, so that their chains
      // interleave)
      auto rows = [&](auto nb_c, int tb) {
        constexpr int NB = decltype(nb_c)::value;
        T vi[NB], wi[NB], acc[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const int i = rank + cs * (tb + RW_WARPS * b);
          vi[b] = vo[i];
          wi[b] = wv[i];
          acc[b] = zero;
        }
        for (int jb = k + 1; jb < n; jb += 32) {
          const int j = jb + lane;
          const bool in = j < n;
          const T vj = in ? v[j] : zero, voj = in ? vo[j] : zero, wj = in ? wv[j] : zero;
          T c[NB];
#pragma unroll
          for (int b = 0; b < NB; ++b) c[b] = in ? S[(tb + RW_WARPS * b) * ldS + j] : zero;
          if (k > 0) {
#pragma unroll
            for (int b = 0; b < NB; ++b) c[b] = rt_fnma(wi[b], voj, rt_fnma(vi[b], wj, c[b]));
            if (in) {
#pragma unroll
              for (int b = 0; b < NB; ++b) S[(tb + RW_WARPS * b) * ldS + j] = c[b];
            }
          }
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[b] = rt_fma(c[b], vj, acc[b]);
        }
        // folded sums: after the first log2(NB) exchanges a lane carries one row
        if constexpr (NB >= 2) {
          const bool up = lane & 16;
#pragma unroll
          for (int b = 0; b < NB / 2; ++b) {
            const T keep = up ? acc[b + NB / 2] : acc[b], give = up ? acc[b] : acc[b + NB / 2];
            acc[b] = rt_add(keep, rt_xor(give, 16));
          }
        }
        if constexpr (NB >= 4) {
          const bool up = lane & 8;
          const T keep = up ? acc[1] : acc[0], give = up ? acc[0] : acc[1];
          acc[0] = rt_add(keep, rt_xor(give, 8));
        }
        constexpr int LG = 32 / NB;  // lanes that hold one row's sum
#pragma unroll
        for (int o = LG / 2; o > 0; o >>= 1) acc[0] = rt_add(acc[0], rt_xor(acc[0], o));
        const int b = lane / LG;
        if ((lane & (LG - 1)) == 0) pout[cs > 1 ? tb + RW_WARPS * b : rank + cs * (tb + RW_WARPS * b)] = acc[0];
      };
      int tb = t0 + warp;
      if constexpr (RG >= 4)
        for (; tb + 3 * RW_WARPS < R; tb += 4 * RW_WARPS) rows(std::integral_constant<int, 4>(), tb);
      for (; tb + RW_WARPS < R; tb += 2 * RW_WARPS) rows(std::integral_constant<int, 2>(), tb);
      if (tb < R) rows(std::integral_constant<int, 1>(), tb);
    } else {
      const int ll = tid & (LPR - 1);
      const unsigned mask = ((1u << (LPR & 31)) - 1u) << (lane & ~(LPR - 1));
      for (int t = t0 + tid / LPR; t < R; t += RW_THREADS / LPR) {
        const int i = rank + cs * t;
        T* row = S + t * ldS;
        T acc = zero;
        const T vi = vo[i], wi = wv[i];
        for (int jb = k + 1; jb < n; jb += LPR) {
          const int j = jb + ll;
          if (j >= n) break;
          T c = row[j];
          if (k > 0) {
            c = rt_fnma(wi, vo[j], rt_fnma(vi, wv[j], c));
            row[j] = c;
          }
          acc = rt_fma(c, v[j], acc);
        }
        __syncwarp(mask);
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) acc = rt_add(acc, rt_down(mask, acc, o, LPR));
        if (ll == 0) pout[cs > 1 ? t : i] = acc;
      }
    }
    const T* rnew = rb + (size_t)par * nmax;
    if (cs > 1) {
      __syncthreads();
      for (int q = tid; q < R * cs; q += RW_THREADS) {
        const int dst = q / R, t = q - dst * R, i = rank + cs * t;
        if (i > k) cl_store(pb + (size_t)par * nmax + i, psm[t], dst);
      }
      if (rank == (k + 1) % cs) {
        const T* row = S + ((k + 1) / cs) * ldS;
        const int len = n - k - 1;
        for (int q = tid; q < len * cs; q += RW_THREADS) {
          const int dst = q / len, j = k + 1 + (q - dst * len);
          cl_store(rb + (size_t)par * nmax + j, row[j], dst);
        }
      }
    } else {
      rnew = S + (size_t)(k + 1) * ldS;
    }
    cl_sync(cs);
    if (warp < VW) {
      const T* p = pb + (size_t)par * nmax;
      T pr[EPT], s = zero;
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int j = tid + VT * q;
        if (VT * (q + 1) <= k + 1 || VT * q >= n) continue;
        pr[q] = (j > k && j < n) ? p[j] : zero;
        rc[q] = (j > k && j < n) ? rnew[j] : zero;
        s = rt_fma(vr[q], pr[q], s);
      }
      const T p1 = p[k + 1];
      const T K2 = rt_mul(two, vsum(s, 1));
      const T w1 = rt_fnma(K2, v1, rt_mul(two, p1));
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        const int j = tid + VT * q;
        if (VT * (q + 1) <= k + 1 || VT * q >= n) continue;
        const T wj = rt_fnma(K2, vr[q], rt_mul(two, pr[q]));
        rc[q] = rt_fnma(w1, vr[q], rt_fnma(v1, wj, rc[q]));
        if (j > k && j < n) wv[j] = wj;
        if (j == k + 1 && rank == 0) W.d[k + 1] = rc[q];
      }
    }
  }
  __syncthreads();
  // row n - 2 is the pivot row now
  if (rank == 0 && warp < VW && n >= 2) {
#pragma unroll
    for (int q = 0; q < EPT; ++q)
      if (tid + VT * q == n - 1) W.e[n - 2] = rc[q];
  }
  if (rank == (n - 1) % cs && tid == 0) {
    T c = S[((n - 1) / cs) * ldS + n - 1];
    if (n >= 3) {
      const T vl = vb[(size_t)((n - 3) & 1) * nmax + n - 1], wl = wv[n - 1];
      c = rt_fnma(wl, vl, rt_fnma(vl, wl, c));
    }
    W.d[n - 1] = c;
    W.e[n - 1] = zero;
  }
}

// ---------------------------------------------------------------- back-transformation

// y = D L^-T H_0 ... H_{n-3} z, a warp per eigenvector held in registers (row
// 32 r + lane in register r); reflectors, then rows of L, come through shared
// memory as in rrw_solve_kernel, from the last to the first.
template <class T, int NR>
__global__ void __launch_bounds__(128) rrw_back_kernel(const RRTask* __restrict__ tasks) {
  const RRTask Tk = tasks[blockIdx.y];
  const WideWork<T> W = wide_carve<T>(Tk);
  const int n = W.st[0], m = Tk.m, ld = W.ld;
  if (n == 0 || (int)blockIdx.x * 4 >= m) return;  // the whole CTA
  const int lane = threadIdx.x & 31, c = blockIdx.x * 4 + (threadIdx.x >> 5);
  const int n_out = (Tk.mode == RR_LOBPCG) ? 3 * m : n;
  constexpr int ldb = 32 * NR;
  extern __shared__ __align__(16) unsigned char rw_raw[];
  T* buf = reinterpret_cast<T*>(rw_raw);  // 2 x KC columns
  const T zero = RtOf<T>::off(0.0f);
  for (int i = threadIdx.x; i < 2 * KC * ldb; i += 128) buf[i] = zero;
  __syncthreads();
  const int ktop = (n - 1) / KC * KC;  // first of the last KC columns
  stage_columns(buf + ((ktop / KC) & 1) * KC * ldb, ldb, W.X, ld, n, ktop);
  T z[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int i = 32 * r + lane;
    z[r] = (i < n && c < m) ? W.Z[i + (size_t)c * ld] : zero;
  }
#pragma unroll
  for (int rk = NR - 1; rk >= 0; --rk) {
    // reflectors k = 32 rk + 31 .. 32 rk touch rows > k only
    for (int l0 = 32 - KC; l0 >= 0; l0 -= KC) {
      const int k0 = 32 * rk + l0;
      if (k0 > ktop) continue;  // uniform
      const T* cur = buf + ((k0 / KC) & 1) * KC * ldb;
      if (k0 > 0) {
        stage_columns(buf + (((k0 / KC) & 1) ^ 1) * KC * ldb, ldb, W.X, ld, n, k0 - KC);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      if constexpr (std::is_same<T, dfl>::value) {
        // two reflectors at a time: v_k and v_{k-1} act as z - 2 s1 v_k -
        // 2 s2 v_{k-1}, s1 = v_k.z, s2 = v_{k-1}.z - 2 s1 v_{k-1}.v_k, so that
        // the latencies of the three sums overlap
#pragma unroll 1
        for (int u = KC - 1; u > 0; u -= 2) {
          const int k = k0 + u;
          if (k + 1 >= n) continue;  // uniform; column n - 2 holds no reflector
          T va[NR], vc[NR], s1 = zero, s2 = zero, g = zero;
#pragma unroll
          for (int r = rk; r < NR; ++r) {
            const T wa = cur[u * ldb + 32 * r + lane], wc = cur[(u - 1) * ldb + 32 * r + lane];
            va[r] = (k + 2 < n && (r > rk || lane > l0 + u)) ? wa : zero;
            vc[r] = (r > rk || lane > l0 + u - 1) ? wc : zero;
            s1 = rt_fma(va[r], z[r], s1);
            s2 = rt_fma(vc[r], z[r], s2);
            g = rt_fma(va[r], vc[r], g);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            s1 = rt_add(s1, rt_down(0xffffffffu, s1, o, 32));
            s2 = rt_add(s2, rt_down(0xffffffffu, s2, o, 32));
            g = rt_add(g, rt_down(0xffffffffu, g, o, 32));
          }
          s1 = rt_shfl(rt_add(s1, s1), 0);
          s2 = rt_shfl(rt_add(s2, s2), 0);
          g = rt_shfl(g, 0);
          s2 = rt_fnma(rt_add(s1, s1), g, s2);
#pragma unroll
          for (int r = rk; r < NR; ++r) z[r] = rt_fnma(s2, vc[r], rt_fnma(s1, va[r], z[r]));
        }
      } else
#pragma unroll 1
      for (int u = KC - 1; u >= 0; --u) {
        const int k = k0 + u;
        if (k + 2 >= n) continue;  // uniform
        T v[NR], s = zero;
#pragma unroll
        for (int r = rk; r < NR; ++r) {
          const T w = cur[u * ldb + 32 * r + lane];
          v[r] = (r > rk || lane > l0 + u) ? w : zero;  // W.X holds other data up to row k
          s = rt_fma(v[r], z[r], s);
        }
        s = rt_warp_sum(s);
        s = rt_add(s, s);
#pragma unroll
        for (int r = rk; r < NR; ++r) z[r] = rt_fnma(s, v[r], z[r]);
      }
      __syncthreads();
    }
  }
  const bool plain = W.st[2] != 0;
  if (!plain) stage_columns(buf + ((ktop / KC) & 1) * KC * ldb, ldb, W.LT, ld, n, ktop);
#pragma unroll
  for (int rk = NR - 1; rk >= 0; --rk) {
    if (plain) break;  // uniform
    T rinv = (32 * rk + lane < n) ? W.rinv[32 * rk + lane] : zero;
    for (int l0 = 32 - KC; l0 >= 0; l0 -= KC) {
      const int k0 = 32 * rk + l0;
      if (k0 > ktop) continue;  // uniform
      const T* cur = buf + ((k0 / KC) & 1) * KC * ldb;
      if (k0 > 0) {
        stage_columns(buf + (((k0 / KC) & 1) ^ 1) * KC * ldb, ldb, W.LT, ld, n, k0 - KC);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
#pragma unroll 1
      for (int u = KC - 1; u >= 0; --u) {
        if (k0 + u >= n) continue;  // uniform
        const T yk = rt_mul(rt_shfl(z[rk], l0 + u), rt_shfl(rinv, l0 + u));
        // rows of L are zero from the diagonal on
#pragma unroll
        for (int r = 0; r <= rk; ++r) z[r] = rt_fnma(cur[u * ldb + 32 * r + lane], yk, z[r]);
        if (lane == l0 + u) z[rk] = yk;
      }
      __syncthreads();
    }
  }
  if (c >= m) return;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int i = 32 * r + lane;
    if (i >= n) continue;
    const double y = rt_val(plain ? z[r] : rt_mul(z[r], W.scal[i]));
    Tk.Y[i + (size_t)c * Tk.ldy] = y;
    if (Tk.Yf) Tk.Yf[i + (size_t)c * Tk.ldy] = (float)y;
  }
  for (int i = n + lane; i < n_out; i += 32) {
    Tk.Y[i + (size_t)c * Tk.ldy] = 0.0;
    if (Tk.Yf) Tk.Yf[i + (size_t)c * Tk.ldy] = 0.0f;
  }
  if (lane == 0) {
    Tk.theta[c] = W.lam[c];
    if (c == 0 && W.st[1] && Tk.state) Tk.state[ST_FALLBACK] += 1;
  }
}

// ---------------------------------------------------------------- host

size_t optin_smem() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return (size_t)optin;
}

template <class K> void allow_clusters(K kernel) {
  opt_in_dynamic_smem((const void*)kernel);
  cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// CTAs per pencil: enough shared memory first; then more while a pencil is
// large enough to keep them busy and all tasks' clusters still fit the chip.
// Cycles per step of the tridiagonalisation: FP64, n = 144: 12,400 with 4 CTAs,
// 10,300 with 8; n = 48: 4,900 with one, where a cluster barrier and its
// messages cost 1,600.  dfl, n = 144: 11,400 with one, 7,600 with 4 (the pass
// over the rows falls from 7,700 to 2,300; a further halving is eaten by the
// messages).
int cluster_size(int n, int ntask, bool dfloat) {
  int cs = n > 160 ? 2 : 1;  // the one-CTA factorisation holds up to 160 columns
  const size_t cap = optin_smem();
  auto fits = [&](int c) { return tri_smem(n, c) + 1024 <= cap && chol_smem(n, c) + 1024 <= cap; };
  while (cs < RW_CL_MAX && !fits(cs)) cs *= 2;
  if (!fits(cs)) return 0;
  if (n <= 64) return cs;
  if (dfloat) {
    while (cs < 4 && n > 48 * cs && ntask * cs * 2 <= 112) cs *= 2;
    return cs;
  }
  while (cs < RW_CL_MAX && n > 24 * cs && ntask * cs * 2 <= 112) cs *= 2;
  return cs;
}

template <class T, int NR>
void launch_columns(const RRTask* t, int ntask, int n_max, int m_max, int stage, cudaStream_t st) {
  const size_t sm = (size_t)2 * KC * 32 * NR * 8;
  if (stage < 2) rrw_solve_kernel<T, NR><<<dim3((n_max + 3) / 4, ntask), 128, sm, st>>>(t, stage);
  else rrw_back_kernel<T, NR><<<dim3((m_max + 3) / 4, ntask), 128, sm, st>>>(t);
}

template <class T>
void dispatch_columns(const RRTask* t, int ntask, int n_max, int m_max, int stage, cudaStream_t st) {
  const int nr = (n_max + 31) / 32;
  if (nr <= 2) launch_columns<T, 2>(t, ntask, n_max, m_max, stage, st);
  else if (nr <= 3) launch_columns<T, 3>(t, ntask, n_max, m_max, stage, st);
  else if (nr <= 5) launch_columns<T, 5>(t, ntask, n_max, m_max, stage, st);
  else if constexpr (std::is_same<T, double>::value) {
    if (nr <= 8) launch_columns<T, 8>(t, ntask, n_max, m_max, stage, st);
    else if (nr <= 11) launch_columns<T, 11>(t, ntask, n_max, m_max, stage, st);
    else if (nr <= 14) launch_columns<T, 14>(t, ntask, n_max, m_max, stage, st);
    else launch_columns<T, 19>(t, ntask, n_max, m_max, stage, st);
  }
}

void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int ntask, int cs, size_t smem, cudaStream_t st) {
  cfg = {};
  cfg.gridDim = dim3((unsigned)(cs * ntask));
  cfg.blockDim = dim3(RW_THREADS);
  cfg.stream = st;
  cfg.dynamicSmemBytes = smem;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

// from C to the eigenvectors
template <class T> void launch_standard(const RRTask* t, int ntask, int n_max, int m_max, int cs, cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cluster_config(cfg, at, ntask, cs, tri_smem(n_max, cs), st);
  if constexpr (std::is_same<T, dfl>::value) {
    cudaLaunchKernelEx(&cfg, rrw_tri_kernel<T, 1, 32, 4>, t, cs, n_max);
  } else {
    if (n_max <= 64) cudaLaunchKernelEx(&cfg, rrw_tri_kernel<T, 1, 8, 1>, t, cs, n_max);
    else cudaLaunchKernelEx(&cfg, rrw_tri_kernel<T, 4, 32, 2>, t, cs, n_max);
  }
  const int per = BI_WARPS * BI_PER;
  rrw_bisect_kernel<T><<<dim3((m_max + per - 1) / per, ntask), 32 * BI_WARPS, 8 * (size_t)n_max, st>>>(t);
  rrw_vec_kernel<T, VE_VECS, true>
      <<<dim3((m_max + VE_VECS - 1) / VE_VECS, ntask), VE_THREADS, vec_smem(n_max, VE_VECS, true), st>>>(t);
  rrw_fix_kernel<T><<<ntask, 256, fix_smem(n_max, m_max), st>>>(t);
  dispatch_columns<T>(t, ntask, n_max, m_max, 2, st);
}

template <class T> void launch_chain(const RRTask* t, int ntask, int n_max, int m_max, int cs, cudaStream_t st) {
  // the factorisation has a third of the products: where one CTA's shared
  // memory and pipe suffice it spares the cluster barriers
  const int ccs = (n_max <= (std::is_same<T, dfl>::value ? 160 : 96)) ? 1 : cs;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cluster_config(cfg, at, ntask, ccs, chol_smem(n_max, ccs), st);
  if (ccs == 1) cudaLaunchKernelEx(&cfg, rrw_chol_kernel<T, true>, t, ccs, n_max);
  else cudaLaunchKernelEx(&cfg, rrw_chol_kernel<T, false>, t, ccs, n_max);
  dispatch_columns<T>(t, ntask, n_max, m_max, 0, st);
  dispatch_columns<T>(t, ntask, n_max, m_max, 1, st);
  launch_standard<T>(t, ntask, n_max, m_max, cs, st);
}

}  // namespace

size_t rr_wide_work_doubles(int n_max, int m) { return wide_work_doubles(n_max, m); }

void init_rr_wide_kernels() {
  allow_clusters(rrw_chol_kernel<double, false>);
  opt_in_dynamic_smem((const void*)rrw_chol_kernel<double, true>);
  opt_in_dynamic_smem((const void*)rrw_chol_kernel<dfl, true>);
  opt_in_dynamic_smem((const void*)rrw_tri_kernel<double, 1, 8, 1>);
  allow_clusters(rrw_tri_kernel<double, 4, 32, 2>);
  allow_clusters(rrw_tri_kernel<dfl, 1, 32, 4>);
  opt_in_dynamic_smem((const void*)rrw_vec_kernel<double, VE_VECS, true>);
  opt_in_dynamic_smem((const void*)rrw_vec_kernel<dfl, VE_VECS, true>);
  opt_in_dynamic_smem((const void*)rrw_solve_kernel<double, 14>);
  opt_in_dynamic_smem((const void*)rrw_solve_kernel<double, 19>);
  opt_in_dynamic_smem((const void*)rrw_back_kernel<double, 14>);
  opt_in_dynamic_smem((const void*)rrw_back_kernel<double, 19>);
}

bool rr_wide_eligible(int n_max, int m_max, int ntask, bool dfloat) {
  if (n_max < 1 || m_max < 1 || m_max > n_max || n_max > 19 * 32 || (dfloat && (n_max > RR_DF_NMAX || m_max > RR_DF_MMAX)))
    return false;
  return cluster_size(n_max, ntask, dfloat) > 0;
}

void launch_rr_wide(const RRTask* d_tasks, int ntask, cudaStream_t st, int n_max, int m_max, bool dfloat) {
  const int cs = cluster_size(n_max, ntask, dfloat);
  if (dfloat) launch_chain<dfl>(d_tasks, ntask, n_max, m_max, cs, st);
  else launch_chain<double>(d_tasks, ntask, n_max, m_max, cs, st);
}

// The lowest m_max eigenpairs of one FP64 symmetric matrix that the caller has
// put into the task's C (set_standard_kernel): n <= 608.
void launch_rr_standard(const RRTask* d_task, int n, int m, cudaStream_t st) {
  launch_standard<double>(d_task, 1, n, m, cluster_size(n, 1, false), st);
}

}  // namespace dgdft
