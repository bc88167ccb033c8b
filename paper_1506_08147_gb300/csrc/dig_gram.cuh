// One chunk of a Gram product X^T diag(w v) Y on the tensor cores by digit
// splitting (digits.cuh): the loop that the DG assembly and the FP64 solver
// share.
#pragma once

#include "digits.cuh"

namespace dgdft {

namespace {

struct DigGramOp {
  const double *X, *Y;  // column-major; first column of the tile
  int ldx, ldy;
  const double *w, *v;  // weights of X (WEIGHT only; v may be null)
  const int *ex, *ey;   // exponents of the columns (with the weights for X), at least 64
  int J1, nB;           // columns of X (at most 128) and of Y (at most NB)
  int p0, p1;           // points
  bool sym;             // Y = X and nB = J1: one operand for both sides (`arows` = NB)
};

// Rows of the product are the columns of X (`arows` in shared memory), K the
// points, N the columns of Y.  A thread splits groups of eight points g, g + 8,
// .. of one column (neighbouring threads read neighbouring points: with eight
// points in a row the reads alone took 4,200 cycles a stage of 80 columns):
// group t, t + 512, ... of (columns x 8) per stage.  DB: two buffers of operands,
// so that a stage's products run while the next one is split; otherwise one.
// D digits (weights: seven).  Exact integer sums over the whole chunk (at most 2^20
// points), then FP64
// to out[r ldout + c].  All threads of the CTA; ends without a barrier.
template <int NB, int RT, bool DB, bool WEIGHT, int D>
__device__ __forceinline__ void dig_gram_chunk(DigCta& cta, const DigGramOp& T, unsigned char* base, int arows,
                                               DigWeight (*ws)[DIG_K], int* abort_s, double* out, int ldout) {
  const int astep = arows * 128, boff = D * astep, buf = boff + D * NB * 128;
  const uint32_t abase = smem_u32(base);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows = T.J1 + (T.sym ? 0 : T.nB), p1 = T.p1;
  double v[RT][8];
  auto load = [&](int p) {
#pragma unroll
    for (int k = 0; k < RT; ++k) {
      const int q = tid + k * DIG_THREADS, r = q >> 3, pt = p + (q & 7);
      const double* col = r < T.J1 ? T.X + (size_t)r * T.ldx : T.Y + (size_t)(r - T.J1) * T.ldy;
#pragma unroll
      for (int u = 0; u < 8; ++u) v[k][u] = (r < rows && pt + 8 * u < p1) ? col[pt + 8 * u] : 0.0;
    }
  };
  // weight of point p + tid, tid < 64
  auto weight = [&](int p) {
    const int pt = p + tid;
    double w = (tid < DIG_K && pt < p1) ? T.w[pt] : 0.0;
    if (T.v && tid < DIG_K && pt < p1) w *= T.v[pt];
    return w;
  };
  int ek[RT];  // exponents of this thread's columns
#pragma unroll
  for (int k = 0; k < RT; ++k) {
    const int r = (tid + k * DIG_THREADS) >> 3;
    ek[k] = r >= rows ? 64 : r < T.J1 ? T.ex[r] : T.ey[r - T.J1];
  }
  long long hs[NB / 4], ls[NB / 4];
#pragma unroll
  for (int q = 0; q < NB / 4; ++q) hs[q] = ls[q] = 0;
  if (WEIGHT) {
    if (tid < DIG_K) ws[0][tid] = dig_weight(weight(T.p0));
    __syncthreads();
  }
  const int nst = (p1 - T.p0 + DIG_K - 1) / DIG_K;
  // the products of stage st are done; the sums of a window are read (by the
  // warps whose rows and columns are in use)
  auto finish = [&](int st) {
    dig_wait(cta, abort_s);
    if ((st % DIG_WINDOW) != DIG_WINDOW - 1 && st != nst - 1) return;
    const uint32_t ta = cta.tmem + ((uint32_t)((warp & 3) * 32) << 16);
    if ((warp & 3) * 32 < T.J1) {
#pragma unroll
      for (int q = 0; q < NB / 16; ++q) {
        const int c0 = (warp >> 2) * 4 + 16 * q;
        if (c0 >= T.nB) continue;
        long long hi[4], lo[4];
        if constexpr (D == DIG8) dig8_drain4<NB>(ta + c0, hi, lo);
        else dig_drain4<NB>(ta + c0, hi, lo);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          hs[4 * q + u] += hi[u];
          ls[4 * q + u] += lo[u];
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  };
  load(T.p0);
  for (int st = 0; st < nst; ++st) {
    const int p = T.p0 + st * DIG_K, off = DB ? (st & 1) * buf : 0;
    if (!DB && st > 0) finish(st - 1);
#pragma unroll
    for (int k = 0; k < RT; ++k) {
      const int q = tid + k * DIG_THREADS, r = q >> 3, g = q & 7;
      if (r >= rows) continue;
      const bool left = r < T.J1;
      uint4 d[D];
      if constexpr (D == DIG8) {
        const int s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        dig8_split8s(v[k], s, ek[k], d);
      } else if (WEIGHT && left) {
        dig_split8w(v[k], &ws[st & 1][g], 8, ek[k], d);
      } else {
        dig_split8(v[k], ek[k], d);
      }
      unsigned char* dst = base + off + (left ? dig_off(r, g) : boff + dig_off(r - T.J1, g));
      const int step = left ? astep : NB * 128;
#pragma unroll
      for (int i = 0; i < D; ++i) *reinterpret_cast<uint4*>(dst + i * step) = d[i];
    }
    double wn = 0.0;
    if (WEIGHT) wn = weight(p + DIG_K);
    if (st + 1 < nst) load(p + DIG_K);
    if (DB && st > 0) finish(st - 1);
    if (WEIGHT && tid < DIG_K) ws[(st + 1) & 1][tid] = dig_weight(wn);
    dig_publish();
    dig_launch<NB, D>(cta, abase + off, astep, abase + off + (T.sym ? 0 : boff), 4, (st % DIG_WINDOW) == 0);
  }
  if (nst > 0) finish(nst - 1);
  const int r = (warp & 3) * 32 + lane;
  if (r < T.J1) {
    const int e = T.ex[r];
#pragma unroll
    for (int q = 0; q < NB / 16; ++q)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = (warp >> 2) * 4 + 16 * q + u;
        if (c >= T.nB) continue;
        out[(size_t)r * ldout + c] = dig_value_sum<D>(hs[4 * q + u], ls[4 * q + u], e, T.sym ? T.ex[c] : T.ey[c]);
      }
  }
}

}  // namespace

}  // namespace dgdft
