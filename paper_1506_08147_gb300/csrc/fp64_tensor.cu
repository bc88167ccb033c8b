// The FP64 stage's Gram products and block updates on the tensor cores, by
// exact digit splitting (digits.cuh) into eight digits.  With seven the
// products of a step of four elements came out 1.4 to 3 times as far from a
// 64-bit reference as an FP64 chain's (residuals; X' is one block plus small
// ones, which a chain rounds once or twice); eight cost a quarter more.
//
// What bounds them.  On the FP64 pipe (1.2 TFLOP/s) a pencil's 12 products of 48
// columns and 122,880 rows took 4 ms per element, an update of three blocks 1.1
// ms; with pairs on the FP32 pipes (the mixed form) a fifth of that.  Here the
// integer instructions of the digit splitting and of reading the sums do, and
// the products issued beside them.  Four elements, an SCF step: the Gram
// products 77 -> 8 ms (nine launches), the updates 45 -> 10 (14 launches); one element of
// 4,096 rows and 16 columns: 31 -> 12.5 us and 36 -> 13 us a launch, so the
// SIMT kernels are not kept for small blocks either.  The orthonormalisation
// (36 elements of 13,440 points, 40 columns): Gram 0.97 and update 1.30 ms a
// launch on the FP64 pipe, a step 82.3 -> 78.8 ms without them.
#include <algorithm>

#include "dig_gram.cuh"
#include "internal.h"

namespace dgdft {

namespace {

constexpr int GT = 64;  // columns of a product's tile, as the partials are laid out

// The distinct blocks of a job's pairs: exponents of their columns are found
// once.
struct DigGramJob {
  GramJob<double> job;
  BRef<double> u[2 * MAX_PAIRS];
  int ncols[2 * MAX_PAIRS], needs_p[2 * MAX_PAIRS];
  int ia[MAX_PAIRS], ib[MAX_PAIRS];
  int nu, stride;  // exponents per block
};

__device__ __forceinline__ int dig_ld(const ElemDev<double>& e, const BRef<double>& r, int ld_in, int rows) {
  return r.ptr ? (ld_in > 0 ? ld_in : rows) : e.ng;
}

// grid (columns, distinct blocks, elements)
__global__ void __launch_bounds__(256) gram_colexp_kernel(const ElemDev<double>* __restrict__ elems, DigGramJob dj,
                                                          int* __restrict__ exps) {
  const ElemDev<double>& e = elems[blockIdx.z];
  const int b = blockIdx.y, c = blockIdx.x;
  if (!e.state[ST_ACTIVE] || (dj.needs_p[b] && !e.state[ST_HAS_P])) return;
  if (c >= (dj.ncols[b] > 0 ? dj.ncols[b] : e.m)) return;
  const int rows = dj.job.rows > 0 ? dj.job.rows : e.ng;
  const double* col = resolve(e, dj.u[b]) + (size_t)c * dig_ld(e, dj.u[b], dj.job.ld_in, rows);
  int ex = 64;
#pragma unroll 8
  for (int p = threadIdx.x; p < rows; p += 256) ex = max(ex, dig_exp(col[p]));
  __shared__ int red[8];
  for (int o = 16; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ex;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) ex = max(ex, red[w]);
    exps[((size_t)blockIdx.z * dj.nu + b) * dj.stride + c] = ex;
  }
}

// Gram products of a job: item (element, row chunk, pair and tile), the pairs of
// a chunk one after another, so that the blocks they share come from L2.
// Partials as gram_reduce_kernel reads them.  A persistent grid.
template <int NB, int RT, bool DB>
__global__ void __launch_bounds__(DIG_THREADS, 1) gram_dig_kernel(const ElemDev<double>* __restrict__ elems,
                                                                  DigGramJob dj, double* __restrict__ partial,
                                                                  size_t pstride, int kchunk, int nchunk, int tiles_a,
                                                                  int tiles_b, int nel, const int* __restrict__ exps) {
  extern __shared__ __align__(1024) unsigned char dig_raw[];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t slot;
  __shared__ int abort_s;
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dig_raw + 1023) & ~(uintptr_t)1023);
  const GramJob<double>& job = dj.job;
  if (threadIdx.x == 0) abort_s = 0;
  DigCta cta;
  dig_open(cta, bar, &slot);
  const int ntile = tiles_a * tiles_b, ny = job.npairs * ntile;
  const long long total = (long long)ny * nchunk * nel;
  for (long long it = blockIdx.x; it < total; it += gridDim.x) {
    const int el = (int)(it / ((long long)ny * nchunk)), rem = (int)(it - (long long)el * ny * nchunk);
    const int chunk = rem / ny, y = rem - chunk * ny, pair = y / ntile, t = y - pair * ntile;
    const ElemDev<double>& e = elems[el];
    if (!e.state[ST_ACTIVE] || (job.needs_p[pair] && !e.state[ST_HAS_P])) continue;
    const int ca = job.ncols_a > 0 ? job.ncols_a : e.m, cb = job.ncols_b > 0 ? job.ncols_b : e.m;
    const int rows = job.rows > 0 ? job.rows : e.ng;
    const int a0 = t / tiles_b * GT, b0 = t % tiles_b * GT;
    if (a0 >= ca || b0 >= cb || chunk * kchunk >= rows) continue;
    DigGramOp op;
    op.ldx = dig_ld(e, job.a[pair], job.ld_in, rows);
    op.ldy = dig_ld(e, job.b[pair], job.ld_in, rows);
    op.X = resolve(e, job.a[pair]) + (size_t)a0 * op.ldx;
    op.Y = resolve(e, job.b[pair]) + (size_t)b0 * op.ldy;
    op.w = op.v = nullptr;
    op.ex = exps + ((size_t)el * dj.nu + dj.ia[pair]) * dj.stride + a0;
    op.ey = exps + ((size_t)el * dj.nu + dj.ib[pair]) * dj.stride + b0;
    op.J1 = min(GT, ca - a0);
    op.nB = min(GT, cb - b0);
    op.p0 = chunk * kchunk;
    op.p1 = min(rows, op.p0 + kchunk);
    op.sym = op.X == op.Y && op.ldx == op.ldy && op.J1 == op.nB;
    dig_gram_chunk<NB, RT, DB, false, DIG8>(cta, op, base, NB, nullptr, &abort_s,
                                      partial + el * pstride + ((size_t)chunk * ny + y) * (GT * GT), GT);
    __syncthreads();
    if (abort_s) {
      if (threadIdx.x == 0) atomicOr(&e.state[ST_ERROR], ERR_TIMEOUT);
      break;
    }
  }
  dig_close(cta, bar + 1, abort_s != 0);
}

// Block update out = alpha sum_i in_i Y_i + beta out: tiles of 128 grid rows, K the
// inputs' columns one after another in stages of 64, N up to 64 output columns.
// Digits of a row count from its largest contribution: column k of the inputs
// counts as scaled by the largest entry of row k of Y (a power of two), and row
// k of Y by its inverse, so that inputs of very different norms (X, W, P) keep
// all the digits that reach the result.  A CTA takes a contiguous range of
// (element, column chunk, tile).
constexpr int UPD_K = 1024;  // inputs' columns at most


// What a block update reads and writes for one element and its output columns
// from c0 on; nout <= 0: nothing.
struct UpdDesc {
  const double *in[3], *Y;  // Y: at the first of the output columns
  double* out;              // likewise
  int nin, nc, ld[3], yrow[3], ldy, ldo, rows, nout;
  double alpha, beta;
};

// the solver's updates
struct UpdElems {
  const ElemDev<double>* elems;
  TsmmJob<double> job;
  __device__ UpdDesc operator()(int el, int c0) const {
    const ElemDev<double>& e = elems[el];
    UpdDesc d;
    d.nout = 0;
    if (!e.state[ST_ACTIVE]) return d;
    d.nc = job.ncols > 0 ? job.ncols : e.m;
    d.rows = job.rows > 0 ? job.rows : e.ng;
    d.nout = d.nc - c0;
    d.nin = 0;
    for (int in = 0; in < job.nin; ++in) {
      if (job.needs_p[in] && !e.state[ST_HAS_P]) continue;
      const double* p = resolve(e, job.in[in]);
      const int ld = dig_ld(e, job.in[in], job.ld_in, d.rows), yr = job.yrow[in] * d.nc;
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (q == d.nin) {
          d.in[q] = p;
          d.ld[q] = ld;
          d.yrow[q] = yr;
        }
      ++d.nin;
    }
    switch (job.y_id) {
      case Y_RR: d.Y = e.Y; d.ldy = job.ldy > 0 ? job.ldy : 3 * e.m; break;
      case Y_GXW: d.Y = e.gxw; d.ldy = job.ldy > 0 ? job.ldy : e.m; break;
      default: d.Y = job.y_ptr; d.ldy = job.ldy; break;
    }
    d.Y += (size_t)(job.ycol * d.nc + c0) * d.ldy;
    d.ldo = dig_ld(e, job.out, job.ld_in, d.rows);
    d.out = resolve(e, job.out) + (size_t)c0 * d.ldo;
    d.alpha = job.alpha;
    d.beta = job.beta;
    return d;
  }
  __device__ void timeout(int el) const { atomicOr(&elems[el].state[ST_ERROR], ERR_TIMEOUT); }
};

// the orthonormalisation's A Y
struct UpdOrtho {
  const OrthoTask* tasks;
  int* err;
  __device__ UpdDesc operator()(int el, int c0) const {
    const OrthoTask T = tasks[el];
    UpdDesc d;
    d.nin = 1;
    d.nc = T.K > 0 ? T.K : T.J;
    d.in[0] = T.a;
    d.ld[0] = d.ldo = d.rows = T.rows;
    d.yrow[0] = 0;
    d.ldy = d.nc;
    d.Y = T.y + (size_t)c0 * d.ldy;
    d.out = T.out + (size_t)c0 * T.rows;
    d.nout = T.J - c0;
    d.alpha = 1.0;
    d.beta = 0.0;
    return d;
  }
  __device__ void timeout(int) const { atomicOr(err, 1); }
};

template <int NB, class Src>
__global__ void __launch_bounds__(DIG_THREADS, 1) update_dig_kernel(Src src, int nel, int nct, int tiles) {
  extern __shared__ __align__(1024) unsigned char dig_raw[];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t slot;
  __shared__ int es[4][DIG_M], ec[NB], abort_s;
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dig_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t abase = smem_u32(base), bbase = abase + DIG8 * DIG_A_BYTES;
  unsigned char* bsm = base + DIG8 * DIG_A_BYTES;
  const double** cp = reinterpret_cast<const double**>(bsm + DIG8 * NB * 128);  // columns of the inputs
  int* fk = reinterpret_cast<int*>(cp + UPD_K);                                 // scales of the columns
  int* yi = fk + UPD_K;                                                         // rows of Y
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & 127, kq = tid >> 7;
  if (tid == 0) abort_s = 0;
  DigCta cta;
  dig_open(cta, bar, &slot);
  const long long total = (long long)nel * nct * tiles, per = (total + gridDim.x - 1) / gridDim.x;
  const long long end = min(total, (blockIdx.x + 1) * per);
  long long have = -1, known = -1;
  int K = 0;
  UpdDesc d;  // of the element and output columns at hand
  for (long long it = blockIdx.x * per; it < end; ++it) {
    const int el = (int)(it / ((long long)nct * tiles)), rem = (int)(it - (long long)el * nct * tiles);
    const int ct = rem / tiles, tile = rem - ct * tiles;
    if (it / tiles != known) {
      known = it / tiles;
      d = src(el, ct * NB);
    }
    const int r0 = tile * DIG_M, rows = d.rows;
    if (d.nout <= 0 || r0 >= rows) continue;
    const int nB = min(NB, d.nout), ldy = d.ldy;
    const double* Y = d.Y;
    if (it / tiles != have) {
      have = it / tiles;
      K = 0;
      for (int in = 0; in < d.nin; ++in) {
        for (int k = tid; k < d.nc; k += DIG_THREADS) {
          cp[K + k] = d.in[in] + (size_t)k * d.ld[in];
          yi[K + k] = d.yrow[in] + k;
        }
        K += d.nc;
      }
      __syncthreads();
      for (int k = warp; k < K; k += DIG_THREADS / 32) {
        int f = 0;
        for (int c = lane; c < nB; c += 32) f = max(f, dig_exp(Y[yi[k] + (size_t)c * ldy]));
        for (int o = 16; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
        if (lane == 0) fk[k] = f == 0 ? -4096 : f - 1023;  // (a row of zeros takes nothing)
      }
      __syncthreads();
      for (int c = warp; c < nB; c += DIG_THREADS / 32) {
        int f = 64;
        for (int k = lane; k < K; k += 32) {
          const int ex = dig_exp(Y[yi[k] + (size_t)c * ldy]);
          f = max(f, ex == 0x7ff ? 1 << 20 : ex == 0 ? 0 : ex - fk[k]);
        }
        for (int o = 16; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
        if (lane == 0) ec[c] = f;
      }
    }
    const int r = r0 + row;
    int er = 64;
    if (r < rows) {
#pragma unroll 4
      for (int k = kq; k < K; k += 4) {
        const int ex = dig_exp(cp[k][r]);
        er = max(er, ex == 0x7ff ? 1 << 20 : ex == 0 ? 0 : ex + fk[k]);
      }
    }
    es[kq][row] = er;
    __syncthreads();
    er = max(max(es[0][row], es[1][row]), max(es[2][row], es[3][row]));
    const uint32_t ta = cta.tmem + ((uint32_t)((warp & 3) * 32) << 16);
    long long hs[NB / 4], ls[NB / 4];
#pragma unroll
    for (int q = 0; q < NB / 4; ++q) hs[q] = ls[q] = 0;
    const int nks = (K + DIG_K - 1) / DIG_K;
    for (int ks = 0; ks < nks; ++ks) {
      const int k0 = ks * DIG_K, kn = min(DIG_K, (K - k0 + 15) / 16 * 16);  // columns in use
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int g = kq * 2 + h;
        if (g * 8 >= kn) continue;
        double x[8];
        int s[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = k0 + g * 8 + u;
          x[u] = (k < K && r < rows) ? cp[k][r] : 0.0;
          s[u] = k < K ? fk[k] : 0;
        }
        uint4 dg[DIG8];
        dig8_split8s(x, s, er, dg);
#pragma unroll
        for (int i = 0; i < DIG8; ++i) *reinterpret_cast<uint4*>(base + i * DIG_A_BYTES + dig_off(row, g)) = dg[i];
      }
      if (tid < NB * 8) {
        const int c = tid >> 3, g = tid & 7;
        double x[8];
        int s[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = k0 + g * 8 + u;
          x[u] = (k < K && c < nB) ? Y[yi[k] + (size_t)c * ldy] : 0.0;
          s[u] = k < K ? -fk[k] : 0;
        }
        uint4 dg[DIG8];
        dig8_split8s(x, s, c < nB ? ec[c] : 64, dg);
#pragma unroll
        for (int i = 0; i < DIG8; ++i) *reinterpret_cast<uint4*>(bsm + i * NB * 128 + dig_off(c, g)) = dg[i];
      }
      dig_publish();
      dig_launch<NB, DIG8>(cta, abase, DIG_A_BYTES, bbase, kn / 16, ks % DIG_WINDOW == 0);
      dig_wait(cta, &abort_s);
      if (ks % DIG_WINDOW == DIG_WINDOW - 1 || ks == nks - 1) {
#pragma unroll
        for (int q = 0; q < NB / 16; ++q) {
          const int j = (warp >> 2) * 4 + 16 * q;
          if (j >= nB) continue;
          long long hi[4], lo[4];
          dig8_drain4<NB>(ta + j, hi, lo);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            hs[4 * q + u] += hi[u];
            ls[4 * q + u] += lo[u];
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      }
    }
    const int lr = (warp & 3) * 32 + lane;  // row of this lane
    const int e2 = max(max(es[0][lr], es[1][lr]), max(es[2][lr], es[3][lr]));
    if (r0 + lr < rows) {
      double* O = d.out + r0 + lr;
#pragma unroll
      for (int q = 0; q < NB / 4; ++q) {
        const int c = (warp >> 2) * 4 + 16 * (q / 4) + (q & 3);
        if (c >= nB) continue;
        double v = dig8_value_sum(hs[q], ls[q], e2, ec[c]);
        if (d.alpha == -1.0) v = -v;
        else if (d.alpha != 1.0) v *= d.alpha;
        double* o = O + (size_t)c * d.ldo;
        if (d.beta == 1.0) v += *o;
        else if (d.beta != 0.0) v += d.beta * *o;
        *o = v;
      }
    }
    __syncthreads();  // es, the scales and the accumulators are read
    if (abort_s) {
      if (tid == 0) src.timeout(el);
      break;
    }
  }
  dig_close(cta, bar + 1, abort_s != 0);
}

// exponents of the columns of every task; grid (columns, 1, tasks)
__global__ void __launch_bounds__(256) ortho_exp_kernel(const OrthoTask* __restrict__ tasks, int stride,
                                                        int* __restrict__ exps) {
  const OrthoTask T = tasks[blockIdx.z];
  const int c = blockIdx.x;
  if (c >= T.J) return;
  int ex = 64;
#pragma unroll 8
  for (int p = threadIdx.x; p < T.rows; p += 256) ex = max(ex, dig_exp(T.a[p + (size_t)c * T.rows]));
  __shared__ int red[8];
  ex = __reduce_max_sync(0xffffffffu, ex);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ex;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) ex = max(ex, red[w]);
    exps[blockIdx.z * stride + c] = ex;
  }
}

// A^T A of the orthonormalisation: item (task, row chunk, pair of 64-column tiles
// on or above the diagonal), partials J x J as ortho_gram_reduce_kernel reads
// them.
template <int NB, int RT, bool DB>
__global__ void __launch_bounds__(DIG_THREADS, 1) ortho_gram_kernel(const OrthoTask* __restrict__ tasks, int ntask,
                                                                    int chunk, int nchunk, int nt, size_t stride,
                                                                    const int* __restrict__ exps, int estride,
                                                                    double* __restrict__ partial, int* err) {
  extern __shared__ __align__(1024) unsigned char dig_raw[];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t slot;
  __shared__ int abort_s;
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dig_raw + 1023) & ~(uintptr_t)1023);
  if (threadIdx.x == 0) abort_s = 0;
  DigCta cta;
  dig_open(cta, bar, &slot);
  const int ny = nt * nt;
  const long long total = (long long)ny * nchunk * ntask;
  for (long long it = blockIdx.x; it < total; it += gridDim.x) {
    const int k = (int)(it / ((long long)ny * nchunk)), rem = (int)(it - (long long)k * ny * nchunk);
    const int ch = rem / ny, y = rem - ch * ny, a0 = y / nt * GT, b0 = y % nt * GT;
    const OrthoTask T = tasks[k];
    if (a0 > b0 || b0 >= T.J || ch * chunk >= T.rows) continue;
    DigGramOp op;
    op.ldx = op.ldy = T.rows;
    op.X = T.a + (size_t)a0 * T.rows;
    op.Y = T.a + (size_t)b0 * T.rows;
    op.w = op.v = nullptr;
    op.ex = exps + k * estride + a0;
    op.ey = exps + k * estride + b0;
    op.J1 = min(GT, T.J - a0);
    op.nB = min(GT, T.J - b0);
    op.p0 = ch * chunk;
    op.p1 = min(T.rows, op.p0 + chunk);
    op.sym = a0 == b0;
    dig_gram_chunk<NB, RT, DB, false, DIG8>(cta, op, base, NB, nullptr, &abort_s,
                                            partial + ((size_t)k * nchunk + ch) * stride + (size_t)a0 * T.J + b0, T.J);
    __syncthreads();
    if (abort_s) break;
  }
  if (abort_s && threadIdx.x == 0) atomicOr(err, 1);
  dig_close(cta, bar + 1, abort_s != 0);
}

__global__ void ortho_gram_reduce_kernel(const OrthoTask* __restrict__ tasks, int chunk, int nchunk, size_t stride,
                                         const double* __restrict__ partial) {
  const OrthoTask T = tasks[blockIdx.z];
  const int J = T.J, nch = (T.rows + chunk - 1) / chunk;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < J * J; q += gridDim.x * blockDim.x) {
    int i = q / J, j = q - (q / J) * J;
    const int oi = i, oj = j;
    if (i > j) {
      const int t = i;
      i = j;
      j = t;
    }
    double s = 0.0;
#pragma unroll 8
    for (int ch = 0; ch < nch; ++ch) s += partial[((size_t)blockIdx.z * nchunk + ch) * stride + i * J + j];
    T.out[oi + (size_t)oj * J] = s;
  }
}

template <int NB> constexpr size_t upd_smem() {
  return (size_t)DIG8 * DIG_A_BYTES + (size_t)DIG8 * NB * 128 + UPD_K * (sizeof(void*) + 2 * sizeof(int)) + 1024;
}

bool same_ref(const BRef<double>& a, const BRef<double>& b) {
  return a.ptr == b.ptr && (a.ptr || (a.sel == b.sel && a.next == b.next));
}

template <int NB> void opt_in_nb() {
  constexpr size_t buf = (size_t)DIG8 * 2 * NB * 128;
  constexpr bool two = 2 * buf + 1024 <= DIG_SMEM_MAX;
  dig_opt_in(gram_dig_kernel<NB, NB <= 32 ? 1 : 2, two>, (two ? 2 : 1) * buf + 1024);
  dig_opt_in(update_dig_kernel<NB, UpdElems>, upd_smem<NB>());
  dig_opt_in(update_dig_kernel<NB, UpdOrtho>, upd_smem<NB>());
  dig_opt_in(ortho_gram_kernel<NB, NB <= 32 ? 1 : 2, two>, (two ? 2 : 1) * buf + 1024);
}

}  // namespace

void init_fp64_tensor_kernels() {
  opt_in_nb<16>();
  opt_in_nb<32>();
  opt_in_nb<48>();
  opt_in_nb<64>();
}

// kchunk rows per chunk (at most 2^20), nchunk of them; `exps` holds
// gram_dig_ints(job, ...) integers.
size_t gram_dig_ints(const GramJob<double>& job, int ca, int cb, int nel) {
  return (size_t)nel * 2 * job.npairs * std::max(ca, cb);
}

void launch_gram_dig(const Batch<double>& b, const GramJob<double>& job, double* partial, size_t pstride, int kchunk,
                     int nchunk, int ca, int cb, int* exps, cudaStream_t st) {
  DigGramJob dj{};
  dj.job = job;
  dj.stride = std::max(ca, cb);
  auto index = [&](const BRef<double>& r, int ncols, int needs) {
    for (int i = 0; i < dj.nu; ++i)
      if (same_ref(dj.u[i], r)) {
        dj.needs_p[i] &= needs;
        dj.ncols[i] = std::max(dj.ncols[i], ncols);
        return i;
      }
    dj.u[dj.nu] = r;
    dj.ncols[dj.nu] = ncols;
    dj.needs_p[dj.nu] = needs;
    return dj.nu++;
  };
  for (int k = 0; k < job.npairs; ++k) {
    dj.ia[k] = index(job.a[k], job.ncols_a, job.needs_p[k]);
    dj.ib[k] = index(job.b[k], job.ncols_b, job.needs_p[k]);
  }
  gram_colexp_kernel<<<dim3(dj.stride, dj.nu, b.s.nel), 256, 0, st>>>(b.d_elems, dj, exps);
  const int ta = (ca + GT - 1) / GT, tb = (cb + GT - 1) / GT;
  const int w = std::min(GT, dj.stride);
  const long long total = (long long)job.npairs * ta * tb * nchunk * b.s.nel;
  const int grid = (int)std::min<long long>(total, sm_count());
  auto go = [&](auto nbc) {
    constexpr int NB = decltype(nbc)::value;
    constexpr size_t buf = (size_t)DIG8 * 2 * NB * 128;
    constexpr bool two = 2 * buf + 1024 <= DIG_SMEM_MAX;
    gram_dig_kernel<NB, NB <= 32 ? 1 : 2, two><<<grid, DIG_THREADS, (two ? 2 : 1) * buf + 1024, st>>>(
        b.d_elems, dj, partial, pstride, kchunk, nchunk, ta, tb, b.s.nel, exps);
  };
  switch ((w + 15) / 16) {
    case 1: go(std::integral_constant<int, 16>()); break;
    case 2: go(std::integral_constant<int, 32>()); break;
    case 3: go(std::integral_constant<int, 48>()); break;
    default: go(std::integral_constant<int, 64>()); break;
  }
}

bool launch_update_dig(const Batch<double>& b, const TsmmJob<double>& job, cudaStream_t st) {
  const int nc = job.ncols > 0 ? job.ncols : b.s.max_m;
  const int rows = job.rows > 0 ? job.rows : b.s.max_ng;
  if (job.nin * nc > UPD_K || job.from2 >= 0) return false;
  const int nb = chunk_cols(nc), nct = (nc + nb - 1) / nb, tiles = (rows + DIG_M - 1) / DIG_M;
  const int grid = (int)std::min<long long>((long long)tiles * nct * b.s.nel, sm_count());
  auto go = [&](auto nbc) {
    constexpr int NB = decltype(nbc)::value;
    update_dig_kernel<NB, UpdElems><<<grid, DIG_THREADS, upd_smem<NB>(), st>>>(UpdElems{b.d_elems, job}, b.s.nel, nct,
                                                                               tiles);
  };
  switch (nb) {
    case 16: go(std::integral_constant<int, 16>()); break;
    case 32: go(std::integral_constant<int, 32>()); break;
    case 48: go(std::integral_constant<int, 48>()); break;
    default: go(std::integral_constant<int, 64>()); break;
  }
  return true;
}

// rows per chunk of the orthonormalisation's Gram, by the rows alone: a single
// element's 13,440 rows make 53 chunks
static int ortho_chunk(int rows) { return std::min(1024, std::max(128, (rows / 64 + 127) / 128 * 128)); }

size_t ortho_partial_doubles(int ntask, int max_rows, int max_J) {
  const int chunk = ortho_chunk(max_rows), nchunk = (max_rows + chunk - 1) / chunk;
  return (size_t)ntask * nchunk * max_J * max_J + ((size_t)ntask * max_J + 1) / 2 + 1;
}

void launch_ortho_gram(const OrthoTask* d_tasks, int ntask, int max_rows, int max_J, double* partial, int* err,
                       cudaStream_t st) {
  if (ntask <= 0) return;
  const int chunk = ortho_chunk(max_rows), nchunk = (max_rows + chunk - 1) / chunk;
  const size_t stride = (size_t)max_J * max_J;
  int* exps = reinterpret_cast<int*>(partial + ntask * nchunk * stride);
  ortho_exp_kernel<<<dim3(max_J, 1, ntask), 256, 0, st>>>(d_tasks, max_J, exps);
  const int nt = (max_J + GT - 1) / GT;
  const int grid = (int)std::min<long long>((long long)nt * nt * nchunk * ntask, sm_count());
  auto go = [&](auto nbc) {
    constexpr int NB = decltype(nbc)::value;
    constexpr size_t buf = (size_t)DIG8 * 2 * NB * 128;
    constexpr bool two = 2 * buf + 1024 <= DIG_SMEM_MAX;
    ortho_gram_kernel<NB, NB <= 32 ? 1 : 2, two><<<grid, DIG_THREADS, (two ? 2 : 1) * buf + 1024, st>>>(
        d_tasks, ntask, chunk, nchunk, nt, stride, exps, max_J, partial, err);
  };
  switch ((std::min(GT, max_J) + 15) / 16) {
    case 1: go(std::integral_constant<int, 16>()); break;
    case 2: go(std::integral_constant<int, 32>()); break;
    case 3: go(std::integral_constant<int, 48>()); break;
    default: go(std::integral_constant<int, 64>()); break;
  }
  ortho_gram_reduce_kernel<<<dim3((max_J * max_J + 255) / 256, 1, ntask), 256, 0, st>>>(d_tasks, chunk, nchunk, stride,
                                                                                       partial);
}

void launch_ortho_apply(const OrthoTask* d_tasks, int ntask, int max_rows, int max_J, int* err, cudaStream_t st) {
  if (ntask <= 0) return;
  const int nb = chunk_cols(max_J), nct = (max_J + nb - 1) / nb, tiles = (max_rows + DIG_M - 1) / DIG_M;
  const int grid = (int)std::min<long long>((long long)tiles * nct * ntask, sm_count());
  auto go = [&](auto nbc) {
    constexpr int NB = decltype(nbc)::value;
    update_dig_kernel<NB, UpdOrtho><<<grid, DIG_THREADS, upd_smem<NB>(), st>>>(UpdOrtho{d_tasks, err}, ntask, nct, tiles);
  };
  switch (nb) {
    case 16: go(std::integral_constant<int, 16>()); break;
    case 32: go(std::integral_constant<int, 32>()); break;
    case 48: go(std::integral_constant<int, 48>()); break;
    default: go(std::integral_constant<int, 64>()); break;
  }
}

}  // namespace dgdft
