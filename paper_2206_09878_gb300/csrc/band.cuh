// Banded-LU solves and banded evaluations shared by the forward and adjoint y-kernels.
#pragma once
#include "lmvd_internal.h"

namespace lmvd {

// ------------------------------------------------------------------ band LU access
// element (i, q) of L, (i, r) of U, 1 / U(i, i) for factor mode mf (ignored for shared factors)
__device__ inline double lu_lo(const DLU& f, int i, int q, int mf) {
  return __ldg(f.lo + (f.mstride ? ((size_t)(i * f.K + q - 1) * f.mstride + mf) : (size_t)(i * f.K + q - 1)));
}
__device__ inline double lu_up(const DLU& f, int i, int r, int mf) {
  return __ldg(f.up + (f.mstride ? ((size_t)(i * f.K + r - 1) * f.mstride + mf) : (size_t)(i * f.K + r - 1)));
}
__device__ inline double lu_invd(const DLU& f, int i, int mf) {
  return __ldg(f.invd + (f.mstride ? ((size_t)i * f.mstride + mf) : (size_t)i));
}

// Banded solves with the LU factors, for right-hand sides stored complex [row][mode]. Every y-system
// matrix is real, so the real and imaginary parts of a right-hand side are independent recurrences. With
// many modes a thread solves both parts of one mode (band_solve_cd, band_solve_T_cd): the FP64 pipe is
// saturated and each factor is loaded once per mode. With few modes it solves one part (band_solve_piped,
// band_solve_T_piped), which halves each thread's chain of dependent FP64 operations, the bound there
// (GB300 retires 2 FP64 lanes per clock per SM, so a lone warp's dependent FP64 instruction costs ~64
// cycles). A warp's accesses stay contiguous in both (32 modes, or 16 modes x 2 parts, of one row).

// L U x = in, then out = x (+ add). out may alias in; add may be null.
__device__ inline void band_solve_cd(const DLU& f, int m, int mf, const cd* in, const cd* add, cd* out, size_t M) {
  if (!LMVD_IN(m, M) || (f.mstride && !LMVD_IN(mf, f.mstride)) || !LMVD_IN(f.K, KMAX + 1)) return;
  cd win[KMAX];
#pragma unroll
  for (int q = 0; q < KMAX; ++q) win[q] = cd{};
  for (int i = 0; i < f.n; ++i) {
    cd v = in[(size_t)i * M + m];
    const int nl = __ldg(f.nl + i);
#pragma unroll
    for (int q = 1; q <= KMAX; ++q)
      if (q <= nl) v = fma_rc(-lu_lo(f, i, q, mf), win[q - 1], v);
#pragma unroll
    for (int q = KMAX - 1; q > 0; --q) win[q] = win[q - 1];
    win[0] = v;
    out[(size_t)i * M + m] = v;
  }
#pragma unroll
  for (int q = 0; q < KMAX; ++q) win[q] = cd{};
  for (int i = f.n - 1; i >= 0; --i) {
    const size_t o = (size_t)i * M + m;
    cd v = out[o];
    const int nu = __ldg(f.nu + i);
#pragma unroll
    for (int r = 1; r <= KMAX; ++r)
      if (r <= nu) v = fma_rc(-lu_up(f, i, r, mf), win[r - 1], v);
    v = lu_invd(f, i, mf) * v;
#pragma unroll
    for (int q = KMAX - 1; q > 0; --q) win[q] = win[q - 1];
    win[0] = v;
    out[o] = add ? v + add[o] : v;
  }
}

// The same solve for one real part, for grids with few Fourier modes (1 - 14 warps per SM): element i of the column is
// at in[i rs], out[i rs] and add[i rs]. With so few warps nothing hides a load or an instruction of another warp, so a
// row costs its latencies: 183 us for 129 rows at 128 x 128 modes as band_solve_cd writes it (a value, its row's profile,
// then its factors, one after the other; 300 instructions a row). All but a few rows at each end have the same
// number of factors (DLU::lin, uin), so those rows run in a sweep that knows it: no tests, the window in registers,
// pointers that walk, values and factors of the next 6 or 8 rows in flight: 65 us (m^c system, 3 factors per mode:
// 86 us), with the FP64 pipe, which takes 64 cycles of an SM sub-partition per warp instruction, 40% busy. Loads ahead
// by single rows instead of blocks gained nothing (they share scoreboards, and a wait is for the newest), nor did 4
// rows reach (71 / 98 us).
template <bool DIAG>
constexpr int kBandRows = DIAG ? 6 : 8;  // rows per block: what the registers of a sweep with / without diagonals allow
__device__ __forceinline__ void band_push(double (&win)[KMAX], double v) {
#pragma unroll
  for (int q = KMAX - 1; q > 0; --q) win[q] = win[q - 1];
  win[0] = v;
}
// rows i0, i0 + step, ... (cnt of them) of the sweep with L (UP = false) or U, any number of factors per row
template <bool UP>
__device__ __forceinline__ void band_rows(const DLU& f, int mf, const double* x, const double* add, double* out,
                                          long long rs, int i0, int cnt, double (&win)[KMAX]) {
  for (int s = 0; s < cnt; ++s) {
    const int i = UP ? i0 - s : i0 + s, n = __ldg((UP ? f.nu : f.nl) + i);
    double v = x[i * rs];
    double fq[KMAX];
#pragma unroll
    for (int q = 1; q <= KMAX; ++q) fq[q - 1] = q <= f.K ? (UP ? lu_up(f, i, q, mf) : lu_lo(f, i, q, mf)) : 0.0;
#pragma unroll
    for (int q = 1; q <= KMAX; ++q)
      if (q <= n) v = fma(-fq[q - 1], win[q - 1], v);
    if (UP) v = lu_invd(f, i, mf) * v;
    band_push(win, v);
    out[i * rs] = UP && add ? v + add[i * rs] : v;
  }
}
// Pointers walking the rows of a sweep (a step adds to each, no index is multiplied out): values, factors (fq apart
// within a row), reciprocal diagonals, addends.
template <bool UP, int NB>
struct BandWalk {
  const double *x, *f, *d, *a;
  long long sx, sf, sd, fq;
  __device__ __forceinline__ BandWalk(const DLU& lu, int mf, const double* x0, const double* add, long long rs, int i0,
                                      int dir) {
    const long long ms = lu.mstride ? (long long)lu.mstride : 1, o = lu.mstride ? mf : 0;
    fq = ms;
    sx = dir * rs;
    sf = dir * (lu.K * ms);
    sd = dir * ms;
    x = x0 + i0 * rs;
    f = (UP ? lu.up : lu.lo) + i0 * (lu.K * ms) + o;
    d = lu.invd + i0 * ms + o;
    a = add ? add + i0 * rs : nullptr;
  }
};
template <bool UP, int NB>
struct BandBlock {
  static constexpr int BAND_ROWS = kBandRows<UP>;
  double v[BAND_ROWS], f[BAND_ROWS][NB], d[BAND_ROWS], a[BAND_ROWS];
  __device__ __forceinline__ void load(BandWalk<UP, NB>& w) {
#pragma unroll
    for (int u = 0; u < BAND_ROWS; ++u) {
      v[u] = *w.x;
      w.x += w.sx;
      const double* p = w.f;
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        f[u][q] = __ldg(p);
        p += w.fq;
      }
      w.f += w.sf;
      if (UP) {
        d[u] = __ldg(w.d);
        w.d += w.sd;
        a[u] = 0.0;
        if (w.a) {
          a[u] = *w.a;
          w.a += w.sx;
        }
      }
    }
  }
};
// the same for rows with exactly NB factors
template <bool UP, int NB>
__device__ __forceinline__ void band_rows_nb(const DLU& f, int mf, const double* x, const double* add, double* out,
                                             long long rs, int i0, int cnt, double (&win)[KMAX]) {
  constexpr int BAND_ROWS = kBandRows<UP>;
  const int full = cnt / BAND_ROWS * BAND_ROWS;
  BandBlock<UP, NB> cur, nxt;
  BandWalk<UP, NB> w(f, mf, x, add, rs, i0, UP ? -1 : 1);
  double* o = out + i0 * rs;
  if (full) cur.load(w);
#pragma unroll 1
  for (int s = 0; s < full; s += BAND_ROWS) {
    if (s + BAND_ROWS < full) nxt.load(w);
    double h[BAND_ROWS + KMAX];  // h[KMAX + u]: row u's value; before it the window, oldest first
#pragma unroll
    for (int q = 0; q < KMAX; ++q) h[q] = win[KMAX - 1 - q];
#pragma unroll
    for (int u = 0; u < BAND_ROWS; ++u) {
      double v = cur.v[u];
#pragma unroll
      for (int q = 1; q <= NB; ++q) v = fma(-cur.f[u][q - 1], h[KMAX + u - q], v);
      if (UP) v = cur.d[u] * v;
      h[KMAX + u] = v;
      if (UP && add) v += cur.a[u];
      *o = v;
      o += w.sx;
    }
#pragma unroll
    for (int q = 0; q < KMAX; ++q) win[KMAX - 1 - q] = h[BAND_ROWS + q];
    cur = nxt;
  }
  band_rows<UP>(f, mf, x, add, out, rs, UP ? i0 - full : i0 + full, cnt - full, win);
}
template <bool UP>
__device__ __forceinline__ void band_sweep(const DLU& f, int mf, const double* x, const double* add, double* out,
                                           long long rs) {
  double win[KMAX];
#pragma unroll
  for (int q = 0; q < KMAX; ++q) win[q] = 0.0;
  const int nb = UP ? f.uin.n : f.lin.n, r0 = UP ? f.uin.r0 : f.lin.r0, r1 = UP ? f.uin.r1 : f.lin.r1;
  const int head = UP ? f.n - r1 : r0, mid = r1 - r0, first = UP ? f.n - 1 : 0;
  const int i0 = UP ? r1 - 1 : r0;
  band_rows<UP>(f, mf, x, add, out, rs, first, head, win);
  switch (nb) {
    case 1: band_rows_nb<UP, 1>(f, mf, x, add, out, rs, i0, mid, win); break;
    case 2: band_rows_nb<UP, 2>(f, mf, x, add, out, rs, i0, mid, win); break;
    case 3: band_rows_nb<UP, 3>(f, mf, x, add, out, rs, i0, mid, win); break;
    case 4: band_rows_nb<UP, 4>(f, mf, x, add, out, rs, i0, mid, win); break;
    default: band_rows<UP>(f, mf, x, add, out, rs, i0, mid, win);
  }
  band_rows<UP>(f, mf, x, add, out, rs, UP ? r0 - 1 : r1, f.n - head - mid, win);
}
__device__ __forceinline__ void band_solve_piped(const DLU& f, int mf, const double* in, const double* add, double* out,
                                                 long long rs) {
  if ((f.mstride && !LMVD_IN(mf, f.mstride)) || !LMVD_IN(f.K, KMAX + 1)) return;
  band_sweep<false>(f, mf, in, nullptr, out, rs);
  band_sweep<true>(f, mf, out, add, out, rs);
}

// Solve A^T x = in with the factors A = L U of A (no pivoting): A^T = U^T L^T, so a forward sweep with
// U^T (lower triangular, diagonal of U) is followed by a backward sweep with L^T (unit upper). Entries of
// the factors outside their profile are stored as zeros, so the sweeps run over K. Rows of the result
// outside [zlo, zhi] are stored as zero (the recurrence itself uses the unmodified values). out may
// alias in.
__device__ inline void band_solve_T_cd(const DLU& f, int m, int mf, const cd* in, cd* out, size_t M, int zlo,
                                       int zhi) {
  if (!LMVD_IN(m, M) || (f.mstride && !LMVD_IN(mf, f.mstride)) || !LMVD_IN(f.K, KMAX + 1)) return;
  cd win[KMAX];
#pragma unroll
  for (int q = 0; q < KMAX; ++q) win[q] = cd{};
  for (int i = 0; i < f.n; ++i) {
    cd v = in[(size_t)i * M + m];
#pragma unroll
    for (int r = 1; r <= KMAX; ++r)
      if (r <= f.K && i - r >= 0) v = fma_rc(-lu_up(f, i - r, r, mf), win[r - 1], v);
    v = lu_invd(f, i, mf) * v;
#pragma unroll
    for (int q = KMAX - 1; q > 0; --q) win[q] = win[q - 1];
    win[0] = v;
    out[(size_t)i * M + m] = v;
  }
#pragma unroll
  for (int q = 0; q < KMAX; ++q) win[q] = cd{};
  for (int i = f.n - 1; i >= 0; --i) {
    const size_t o = (size_t)i * M + m;
    cd v = out[o];
#pragma unroll
    for (int q = 1; q <= KMAX; ++q)
      if (q <= f.K && i + q < f.n) v = fma_rc(-lu_lo(f, i + q, q, mf), win[q - 1], v);
#pragma unroll
    for (int q = KMAX - 1; q > 0; --q) win[q] = win[q - 1];
    win[0] = v;
    out[o] = (i < zlo || i > zhi) ? cd{} : v;
  }
}

// band_solve_T_cd for one real part (see band_solve_piped): the sweep with U^T uses row i - r's factor r, the one with
// L^T row i + q's factor q; factors outside the profile are zeros and are skipped in the rows at the ends. Away from
// the ends a row has the interior number of factors.
template <bool UP>
__device__ __forceinline__ void band_rows_T(const DLU& f, int mf, const double* x, double* out, long long rs, int i0,
                                            int cnt, int zlo, int zhi, double (&win)[KMAX]) {
  for (int s = 0; s < cnt; ++s) {
    const int i = UP ? i0 + s : i0 - s;
    double v = x[i * rs];
    double fq[KMAX];
#pragma unroll
    for (int q = 1; q <= KMAX; ++q) {
      const int o = UP ? i - q : i + q;
      fq[q - 1] = q <= f.K && o >= 0 && o < f.n ? (UP ? lu_up(f, o, q, mf) : lu_lo(f, o, q, mf)) : 0.0;
    }
#pragma unroll
    for (int q = 1; q <= KMAX; ++q)
      if ((__double_as_longlong(fq[q - 1]) << 1) != 0) v = fma(-fq[q - 1], win[q - 1], v);
    if (UP) v = lu_invd(f, i, mf) * v;
    band_push(win, v);
    out[i * rs] = !UP && (i < zlo || i > zhi) ? 0.0 : v;
  }
}
template <bool UP, int NB>
__device__ __forceinline__ void band_rows_nb_T(const DLU& f, int mf, const double* x, double* out, long long rs, int i0,
                                               int cnt, int zlo, int zhi, double (&win)[KMAX]) {
  // row i's factor q is row i - q's (UP) or i + q's: the first one's walk, with a row's step added per factor
  constexpr int BAND_ROWS = kBandRows<UP>;
  const int full = cnt / BAND_ROWS * BAND_ROWS;
  BandBlock<UP, NB> cur, nxt;
  BandWalk<UP, NB> w(f, mf, x, nullptr, rs, i0, UP ? 1 : -1);
  w.f += (UP ? -1 : 1) * (f.K * w.fq);
  w.fq += (UP ? -1 : 1) * (f.K * w.fq);
  double* o = out + i0 * rs;
  if (full) cur.load(w);
#pragma unroll 1
  for (int s = 0; s < full; s += BAND_ROWS) {
    if (s + BAND_ROWS < full) nxt.load(w);
    double h[BAND_ROWS + KMAX];
#pragma unroll
    for (int q = 0; q < KMAX; ++q) h[q] = win[KMAX - 1 - q];
#pragma unroll
    for (int u = 0; u < BAND_ROWS; ++u) {
      double v = cur.v[u];
#pragma unroll
      for (int q = 1; q <= NB; ++q) v = fma(-cur.f[u][q - 1], h[KMAX + u - q], v);
      if (UP) v = cur.d[u] * v;
      h[KMAX + u] = v;
      const int i = UP ? i0 + s + u : i0 - s - u;
      *o = !UP && (i < zlo || i > zhi) ? 0.0 : v;
      o += w.sx;
    }
#pragma unroll
    for (int q = 0; q < KMAX; ++q) win[KMAX - 1 - q] = h[BAND_ROWS + q];
    cur = nxt;
  }
  band_rows_T<UP>(f, mf, x, out, rs, UP ? i0 + full : i0 - full, cnt - full, zlo, zhi, win);
}
template <bool UP>
__device__ __forceinline__ void band_sweep_T(const DLU& f, int mf, const double* x, double* out, long long rs, int zlo,
                                             int zhi) {
  double win[KMAX];
#pragma unroll
  for (int q = 0; q < KMAX; ++q) win[q] = 0.0;
  // rows whose K neighbours i - r (UP) or i + q lie in the interior range
  const int nb = UP ? f.uin.n : f.lin.n;
  const int lo = UP ? f.uin.r0 + f.K : f.lin.r0, hi = UP ? f.uin.r1 : f.lin.r1 - f.K;
  const int r0 = lo < hi ? lo : 0, r1 = lo < hi ? hi : 0;
  const int head = UP ? r0 : f.n - r1, mid = r1 - r0, i0 = UP ? r0 : r1 - 1;
  band_rows_T<UP>(f, mf, x, out, rs, UP ? 0 : f.n - 1, head, zlo, zhi, win);
  switch (nb) {
    case 1: band_rows_nb_T<UP, 1>(f, mf, x, out, rs, i0, mid, zlo, zhi, win); break;
    case 2: band_rows_nb_T<UP, 2>(f, mf, x, out, rs, i0, mid, zlo, zhi, win); break;
    case 3: band_rows_nb_T<UP, 3>(f, mf, x, out, rs, i0, mid, zlo, zhi, win); break;
    case 4: band_rows_nb_T<UP, 4>(f, mf, x, out, rs, i0, mid, zlo, zhi, win); break;
    default: band_rows_T<UP>(f, mf, x, out, rs, i0, mid, zlo, zhi, win);
  }
  band_rows_T<UP>(f, mf, x, out, rs, UP ? r1 : r0 - 1, f.n - head - mid, zlo, zhi, win);
}
__device__ __forceinline__ void band_solve_T_piped(const DLU& f, int mf, const double* in, double* out, long long rs,
                                                   int zlo, int zhi) {
  if ((f.mstride && !LMVD_IN(mf, f.mstride)) || !LMVD_IN(f.K, KMAX + 1)) return;
  band_sweep_T<true>(f, mf, in, out, rs, zlo, zhi);
  band_sweep_T<false>(f, mf, out, out, rs, zlo, zhi);
}

__device__ inline double band_row_real(const DBand& B, int i, const double* x) {
  double acc = 0.0;
  if (!LMVD_IN(i, B.rows)) return acc;
  const int c = B.c0[i];
  const double* v = B.v + (size_t)i * B.w;
  const int n = __ldg(B.cnt + i);
  for (int q = 0; q < n; ++q)
    if (LMVD_IN(c + q, B.cols)) acc = fma(__ldg(v + q), x[c + q], acc);
  return acc;
}

}  // namespace lmvd
