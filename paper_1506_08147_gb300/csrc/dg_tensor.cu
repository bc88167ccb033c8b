// Contractions of the DG Hamiltonian assembly on the tensor cores (FP64 by
// digit splitting, digits.cuh): a small matrix along one axis of every
// element's array (interpolation, differentiation, orthonormalisation) and
// the weighted Gram products.
//
// What bounds them.  On the FP64 pipe both ran at 84 to 96 % of its 1.2
// TFLOP/s, with pairs on the FP32 pipes at two to three times that.  Here integer
// instructions do (64 lanes a cycle and SM): a CTA of 512 threads spends 3,060
// cycles on the digits of 128 x 64 values, 590 to 700 on the products of 16
// values with 48 columns, 6,400 on joining 128 x 40 sums to FP64 and writing
// them.  In the Gram products (one 64-point stage of 40 columns: 5,300 cycles)
// the split and the reads of the next stage run beside the products.
// 36 elements of 107,520 points, 40 columns: interpolation 30.7 -> 3.6 ms, mass
// matrices, basis and gradients 54 -> 8.9, volume products 31.6 -> 6.7, the whole
// assembly 124 (61 with pairs) -> 24.2.
#include <algorithm>

#include "dg_tensor.h"
#include "dig_gram.cuh"
#include "internal.h"

namespace dgdft {

namespace {

// ---------------------------------------------------------------- axis passes

struct AxisShape {
  const double* const* in;   // per element
  double* const* out;
  const uint4* img;          // digit images of the matrix
  const int* fexp;           // exponents of its rows
  long long img_stride, f_stride;  // per element (0: one matrix for all)
  int n_in, n_out, S, nel;
  long long O;
  int nc, nks;               // chunks of NB output rows, stages of 64 inputs
  int resident;              // all images fit the shared memory beside A
  const int* shift;          // input i of element e enters as in 2^-shift[e n_in + i] (NULL: as it is)
  int* err;
};

// image (chunk c, stage k) of the matrix A (n_out x n_in, row-major): seven digit
// tiles of NB rows, one after another, rows beyond n_out zero.  A warp per row.
__global__ void __launch_bounds__(128) axis_image_kernel(const double* __restrict__ A, long long a_stride, int n_out,
                                                         int n_in, int nb, int nc, int nks, uint4* __restrict__ img,
                                                         long long img_stride, int* __restrict__ fexp,
                                                         long long f_stride, const int* __restrict__ shift) {
  const int r = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nc * nb) return;
  const double* row = A + blockIdx.y * a_stride + (long long)r * n_in;
  const int* sh = shift ? shift + (long long)blockIdx.y * n_in : nullptr;
  auto at = [&](int i) { return sh ? scalbn(row[i], sh[i]) : row[i]; };
  int e = 0;
  if (r < n_out)
    for (int i = lane; i < n_in; i += 32) e = max(e, dig_exp(at(i)));
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  e = max(e, 64);
  if (lane == 0) fexp[blockIdx.y * f_stride + r] = e;
  const int c = r / nb, n = r - c * nb;
  uint4* dst = img + blockIdx.y * img_stride;
  for (int g = lane; g < nks * 8; g += 32) {
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = g * 8 + u;
      x[u] = (r < n_out && i < n_in) ? at(i) : 0.0;
    }
    uint4 q[DIG];
    dig_split8(x, e, q);
    const int ks = g >> 3;
#pragma unroll
    for (int d = 0; d < DIG; ++d)
      dst[((long long)(c * nks + ks) * DIG + d) * nb * 8 + (dig_off(n, g & 7) >> 4)] = q[d];
  }
}

// out[o][r][s] = sum_i A[r][i] in[o][i][s] for every element: tiles of 128 lines
// (o, s), s fastest, as the rows of the product; K the axis; N the output
// rows in chunks of NB.  Thread t splits values 16 (t / 128) .. + 15 of line t %
// 128 of every stage.  A persistent grid over (element, tile).  NKS: stages of
// 64 inputs, whose values stay in registers for all chunks; 0: any number of
// inputs (more than 128), read again for each chunk and summed over exact
// windows of 128.
template <int NB, int NKS>
__global__ void __launch_bounds__(DIG_THREADS, 1) axis_tensor_kernel(AxisShape jb) {
  extern __shared__ __align__(1024) unsigned char dig_raw[];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t slot;
  __shared__ int es[4][DIG_M], fs[DIG_M], abort_s;
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dig_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t abase = smem_u32(base), bbase = abase + DIG * DIG_A_BYTES;
  constexpr int IMG = DIG * NB * 8;  // uint4 per image
  uint4* bsm = reinterpret_cast<uint4*>(base + DIG * DIG_A_BYTES);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & 127, kq = tid >> 7;
  if (tid == 0) abort_s = 0;
  DigCta cta;
  dig_open(cta, bar, &slot);
  const long long lines = jb.O * jb.S, tiles = (lines + DIG_M - 1) / DIG_M;
  const long long total = tiles * jb.nel;
  const int nin = jb.n_in, nout = jb.n_out, S = jb.S;
  int have = -1;  // element whose images are resident
  constexpr int NV = NKS ? NKS : 1;
  double v[NV][16];
  // this thread's values of item `it`: the next item's are on their way while
  // this one's products run and its sums are read
  auto load = [&](long long it) {
    if (NKS == 0 || it >= total) return;
    const int el = (int)(it / tiles);
    const long long g = (it - el * tiles) * DIG_M + row;
    const bool valid = g < lines;
    const long long o = valid ? g / S : 0, s = valid ? g - o * S : 0;
    const double* src = jb.in[el] + o * nin * S + s;
#pragma unroll
    for (int ks = 0; ks < NKS; ++ks)
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int i = ks * DIG_K + kq * 16 + u;
        v[ks][u] = (valid && i < nin) ? src[(long long)i * S] : 0.0;
      }
  };
  load(blockIdx.x);
  for (long long it = blockIdx.x; it < total; it += gridDim.x) {
    const int el = (int)(it / tiles);
    const long long g = (it - el * tiles) * DIG_M + row;
    const bool valid = g < lines;
    const long long o = valid ? g / S : 0, s = valid ? g - o * S : 0;
    const double* src = jb.in[el] + o * nin * S + s;
    int e = 64;
    if (NKS == 0)
      for (int i = kq; i < nin; i += 4) e = max(e, valid ? dig_exp(src[(long long)i * S]) : 0);
    if (NKS && jb.shift) {
      const int* sh = jb.shift + (long long)el * nin;
#pragma unroll
      for (int ks = 0; ks < NKS; ++ks)
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int i = ks * DIG_K + kq * 16 + u;
          if (i < nin) v[ks][u] = dig_scale(v[ks][u], -sh[i]);
        }
    }
#pragma unroll
    for (int ks = 0; ks < NKS; ++ks)
#pragma unroll
      for (int u = 0; u < 16; ++u) e = max(e, dig_exp(v[ks][u]));
    es[kq][row] = e;
    const int mel = jb.img_stride ? el : 0;
    const uint4* img = jb.img + mel * jb.img_stride;
    const int* fexp = jb.fexp + mel * jb.f_stride;
    if (have != mel) {
      if (jb.resident)
        for (int q = tid; q < jb.nc * jb.nks * IMG; q += DIG_THREADS) bsm[q] = img[q];
      if (tid < DIG_M) fs[tid] = tid < jb.nc * NB ? dig_row_exp(fexp[tid]) : 0;
      have = mel;
    }
    __syncthreads();
    e = max(max(es[0][row], es[1][row]), max(es[2][row], es[3][row]));
    const uint32_t ta = cta.tmem + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's lane quarter
    for (int c = 0; c < jb.nc; ++c) {
      long long hs[NKS ? 1 : NB / 4], ls[NKS ? 1 : NB / 4];
      if (NKS == 0) {
#pragma unroll
        for (int q = 0; q < NB / 4; ++q) hs[q] = ls[q] = 0;
        for (int ks = 0; ks < jb.nks; ++ks) {
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int i = ks * DIG_K + kq * 16 + u;
            v[0][u] = (valid && i < nin) ? src[(long long)i * S] : 0.0;
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = v[0][8 * h + u];
            uint4 q[DIG];
            dig_split8(x, e, q);
#pragma unroll
            for (int d = 0; d < DIG; ++d)
              *reinterpret_cast<uint4*>(base + d * DIG_A_BYTES + dig_off(row, kq * 2 + h)) = q[d];
          }
          for (int q = tid; q < IMG; q += DIG_THREADS) bsm[q] = img[(long long)(c * jb.nks + ks) * IMG + q];
          dig_publish();
          dig_launch<NB>(cta, abase, DIG_A_BYTES, bbase, min(4, (nin - ks * DIG_K + 15) / 16), ks % DIG_WINDOW == 0);
          dig_wait(cta, &abort_s);
          if (ks % DIG_WINDOW == DIG_WINDOW - 1 || ks == jb.nks - 1) {
#pragma unroll
            for (int q = 0; q < NB / 16; ++q) {
              long long hi[4], lo[4];
              dig_drain4<NB>(ta + (warp >> 2) * 4 + 16 * q, hi, lo);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                hs[(4 * q + u) % (NKS ? 1 : NB / 4)] += hi[u];
                ls[(4 * q + u) % (NKS ? 1 : NB / 4)] += lo[u];
              }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          }
        }
      }
#pragma unroll
      for (int ks = 0; ks < NKS; ++ks) {
        if (NKS > 1 || c == 0) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = v[ks][8 * h + u];
            uint4 q[DIG];
            dig_split8(x, e, q);
#pragma unroll
            for (int d = 0; d < DIG; ++d)
              *reinterpret_cast<uint4*>(base + d * DIG_A_BYTES + dig_off(row, kq * 2 + h)) = q[d];
          }
        }
        uint32_t b = bbase;
        if (jb.resident) {
          b += (uint32_t)((c * jb.nks + ks) * IMG * 16);
        } else {
          for (int q = tid; q < IMG; q += DIG_THREADS) bsm[q] = img[(long long)(c * jb.nks + ks) * IMG + q];
        }
        dig_publish();
        const int nk16 = min(4, (nin - ks * DIG_K + 15) / 16);
        dig_launch<NB>(cta, abase, DIG_A_BYTES, b, nk16, ks == 0);
        // the values are split for the last time
        if (ks == NKS - 1 && c == (NKS > 1 ? jb.nc - 1 : 0)) load(it + gridDim.x);
        dig_wait(cta, &abort_s);
      }
      // the sums of lane quarter warp % 4, every fourth group of four columns
      const int r = (warp & 3) * 32 + lane;  // line of this lane
      const int er = dig_row_exp(max(max(es[0][r], es[1][r]), max(es[2][r], es[3][r])));
      const long long gr = (it - el * tiles) * DIG_M + r;
      const long long orow = gr / S, srow = gr - orow * S;
      double* dst = jb.out[el] + orow * nout * S + srow;
#pragma unroll
      for (int q = 0; q < NB / 16; ++q) {
        const int c0 = (warp >> 2) * 4 + 16 * q, j0 = c * NB + c0;
        if (j0 >= nout) continue;
        long long t[4];
        if (NKS) dig_join4<NB>(ta + c0, t);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = j0 + u;
          if (j >= nout || gr >= lines) continue;
          if (NKS) dst[(long long)j * S] = dig_value(t[u], er, fs[j]);
          else
            dst[(long long)j * S] = dig_value_sum<DIG>(hs[(4 * q + u) % (NKS ? 1 : NB / 4)],
                                                  ls[(4 * q + u) % (NKS ? 1 : NB / 4)], er, fs[j]);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();  // es and the accumulators are read
    if (abort_s) break;
  }
  if (abort_s && tid == 0) atomicExch(jb.err, 1);
  dig_close(cta, bar + 1, abort_s != 0);
}

// ---------------------------------------------------------------- Gram products

// exponents: of w v x for the columns of X (a bound: factors' exponents add up,
// one more per product), of the columns of Y; a CTA per column, which takes
// both of a column that stands on both sides
__global__ void __launch_bounds__(256) gram_exp_kernel(const TGramTask* __restrict__ tasks, int* __restrict__ exps) {
  const TGramTask T = tasks[blockIdx.y];
  const int c = blockIdx.x;
  const bool both = T.X == T.Y && T.ldx == T.ldy && T.J1 == T.J2;
  if (c >= T.J1 + (T.sym || both ? 0 : T.J2)) return;
  const bool left = c < T.J1;
  const double* col = left ? T.X + (size_t)c * T.ldx : T.Y + (size_t)(c - T.J1) * T.ldy;
  int e = 64, f = 64;
#pragma unroll 4
  for (int p = threadIdx.x; p < T.n; p += 256) {
    int ex = dig_exp(col[p]);
    f = max(f, ex);
    if (left) {
      // (a zero factor leaves a bound that is too small to matter)
      const int ew = dig_exp(T.w[p]);
      const int ev = T.v ? dig_exp(T.v[p]) : 1022;
      const bool zero = ex == 0 || ew == 0 || ev == 0, inf = ex == 0x7ff || ew == 0x7ff || ev == 0x7ff;
      ex = inf ? 0x7ff : zero ? 0 : ex + ew + ev - 2044;
    }
    e = max(e, ex);
  }
  __shared__ int red[2][8];
  for (int o = 16; o > 0; o >>= 1) {
    e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = e;
    red[1][threadIdx.x >> 5] = f;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      e = max(e, red[0][w]);
      f = max(f, red[1][w]);
    }
    exps[T.exp0 + c] = min(e, 0x7ff);
    if (left && both && !T.sym) exps[T.exp0 + T.J1 + c] = f;
  }
}

// X^T diag(w v) Y, item (task, row chunk, chunk of NB columns of Y); sym: (w X)^T
// (w X).  DB: two operand buffers, where at most 112 columns have to fit.
// Partials as dg_gram_reduce_kernel reads them.
template <int NB, int RT, bool DB>
__global__ void __launch_bounds__(DIG_THREADS, 1) gram_tensor_kernel(const TGramTask* __restrict__ tasks,
                                                                     const int* __restrict__ items, int nitems, int arows,
                                                                     const int* __restrict__ exps,
                                                                     double* __restrict__ partial, int* err) {
  extern __shared__ __align__(1024) unsigned char dig_raw[];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t slot;
  __shared__ int abort_s;
  __shared__ DigWeight ws[2][DIG_K];  // weights of this stage and the next
  unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)dig_raw + 1023) & ~(uintptr_t)1023);
  if (threadIdx.x == 0) abort_s = 0;
  DigCta cta;
  dig_open(cta, bar, &slot);
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const TGramTask T = tasks[items[3 * it]];
    const int chunk = items[3 * it + 1], j0 = items[3 * it + 2] * NB;
    DigGramOp op;
    op.X = T.X;
    op.Y = T.Y + (size_t)j0 * T.ldy;
    op.ldx = T.ldx;
    op.ldy = T.ldy;
    op.w = T.w;
    op.v = T.v;
    op.ex = exps + T.exp0;
    op.ey = op.ex + T.J1 + j0;
    op.J1 = T.J1;
    op.nB = min(NB, T.J2 - j0);
    op.p0 = chunk * T.chunk;
    op.p1 = min(T.n, op.p0 + T.chunk);
    op.sym = T.sym != 0;
    dig_gram_chunk<NB, RT, DB, true, DIG>(cta, op, base, arows, ws, &abort_s,
                                     partial + T.part + (size_t)chunk * T.J1 * T.J2 + j0, T.J2);
    __syncthreads();
    if (abort_s) break;
  }
  if (abort_s && threadIdx.x == 0) atomicExch(err, 1);
  dig_close(cta, bar + 1, abort_s != 0);
}

size_t dig_smem(int nb, int images) { return (size_t)DIG * DIG_A_BYTES + (size_t)images * DIG * nb * 128 + 1024; }

template <int NB> void launch_axis_nb(const AxisShape& s, int grid, size_t smem, cudaStream_t st) {
  if (s.nks > 2) {
    dig_opt_in(axis_tensor_kernel<NB, 0>, smem);
    axis_tensor_kernel<NB, 0><<<grid, DIG_THREADS, smem, st>>>(s);
  } else if (s.nks == 1) {
    dig_opt_in(axis_tensor_kernel<NB, 1>, smem);
    axis_tensor_kernel<NB, 1><<<grid, DIG_THREADS, smem, st>>>(s);
  } else {
    dig_opt_in(axis_tensor_kernel<NB, 2>, smem);
    axis_tensor_kernel<NB, 2><<<grid, DIG_THREADS, smem, st>>>(s);
  }
}

template <int NB, bool DB>
void launch_gram_nb(const TGramTask* t, const int* items, int ni, const int* exps, double* part, int* err, int arows,
                    int rows, size_t smem, int grid, cudaStream_t st) {
  auto go = [&](auto k) {
    dig_opt_in(k, smem);
    k<<<grid, DIG_THREADS, smem, st>>>(t, items, ni, arows, exps, part, err);
  };
  if (!DB) go(gram_tensor_kernel<NB, 3, DB>);
  else if (rows <= 64) go(gram_tensor_kernel<NB, 1, DB>);
  else go(gram_tensor_kernel<NB, 2, DB>);
}

}  // namespace

size_t axis_image_bytes(int n_in, int n_out, int nmat) {
  const int nb = chunk_cols(n_out), nc = (n_out + nb - 1) / nb, nks = (n_in + DIG_K - 1) / DIG_K;
  return (size_t)nmat * ((size_t)nc * nks * DIG * nb * 128 + sizeof(int) * (size_t)nc * nb) + 256;
}

cudaError_t launch_axis_tensor(const double* const* in, double* const* out, int nel, const double* A, long long a_stride,
                               int n_in, int n_out, int S, long long O, const int* shift, void* scratch, int* err,
                               cudaStream_t st) {
  const int nb = chunk_cols(n_out), nc = (n_out + nb - 1) / nb, nks = (n_in + DIG_K - 1) / DIG_K;
  const int nmat = a_stride ? nel : 1;
  AxisShape s{};
  s.in = in;
  s.out = out;
  s.n_in = n_in;
  s.n_out = n_out;
  s.S = S;
  s.nel = nel;
  s.O = O;
  s.nc = nc;
  s.nks = nks;
  s.err = err;
  uint4* img = static_cast<uint4*>(scratch);
  const long long istr = (long long)nc * nks * DIG * nb * 8;
  int* fexp = reinterpret_cast<int*>(img + istr * nmat);
  s.img = img;
  s.fexp = fexp;
  s.img_stride = a_stride ? istr : 0;
  s.f_stride = a_stride ? nc * nb : 0;
  axis_image_kernel<<<dim3((nc * nb + 3) / 4, nmat), 128, 0, st>>>(A, a_stride, n_out, n_in, nb, nc, nks, img, istr,
                                                                   fexp, nc * nb, shift);
  s.shift = shift;
  s.resident = dig_smem(nb, nc * nks) <= DIG_SMEM_MAX;
  const size_t smem = dig_smem(nb, s.resident ? nc * nks : 1);
  const long long tiles = (O * S + DIG_M - 1) / DIG_M * nel;
  const int grid = (int)std::min<long long>(tiles, sm_count());
  switch (nb) {
    case 16: launch_axis_nb<16>(s, grid, smem, st); break;
    case 32: launch_axis_nb<32>(s, grid, smem, st); break;
    case 48: launch_axis_nb<48>(s, grid, smem, st); break;
    default: launch_axis_nb<64>(s, grid, smem, st); break;
  }
  return cudaGetLastError();
}

int gram_tensor_chunk(long long n) {
  // 16 chunks of at least 512 points, a multiple of the 128 of an exact window;
  // at most 8,192 points.  By the points alone: the order of the sums must not
  // depend on how many elements a batch holds.
  const long long c = std::min<long long>(8192, std::max<long long>(512, (n + 15) / 16));
  return (int)((c + 127) / 128 * 128);
}

void gram_tensor_items(const TGramTask* tasks, int ntask, std::vector<int>& items) {
  int mj = 1;
  for (int t = 0; t < ntask; ++t) mj = std::max(mj, tasks[t].J2);
  const int nb = chunk_cols(mj);
  items.clear();
  for (int t = 0; t < ntask; ++t)
    for (int c = 0; c * tasks[t].chunk < tasks[t].n; ++c)
      for (int j = 0; j * nb < tasks[t].J2; ++j) {
        items.push_back(t);
        items.push_back(c);
        items.push_back(j);
      }
}

cudaError_t launch_gram_tensor(const TGramTask* d_tasks, int ntask, const int* d_items, int nitems, int maxJ1, int maxJ2,
                               int* d_exps, double* partial, int* err, cudaStream_t st) {
  gram_exp_kernel<<<dim3(maxJ1 + maxJ2, ntask), 256, 0, st>>>(d_tasks, d_exps);
  const int nb = chunk_cols(maxJ2), arows = (maxJ1 + 15) / 16 * 16, rows = maxJ1 + std::min(nb, maxJ2);
  const int grid = std::min(nitems, sm_count());
  const size_t buf = (size_t)DIG * (arows + nb) * 128;
  const bool two = 2 * buf + 1024 <= DIG_SMEM_MAX;
  auto go = [&](auto n) {
    if (two) launch_gram_nb<decltype(n)::value, true>(d_tasks, d_items, nitems, d_exps, partial, err, arows, rows, 2 * buf + 1024, grid, st);
    else launch_gram_nb<decltype(n)::value, false>(d_tasks, d_items, nitems, d_exps, partial, err, arows, rows, buf + 1024, grid, st);
  };
  switch (nb) {
    case 16: go(std::integral_constant<int, 16>()); break;
    case 32: go(std::integral_constant<int, 32>()); break;
    case 48: go(std::integral_constant<int, 48>()); break;
    default: go(std::integral_constant<int, 64>()); break;
  }
  return cudaGetLastError();
}

}  // namespace dgdft
