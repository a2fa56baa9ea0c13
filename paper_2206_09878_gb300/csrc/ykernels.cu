// Kernels along the inhomogeneous direction y: one thread per Fourier mode (kx, kz) walks the
// B-spline rows, so a warp reads 32 consecutive modes of one row (coalesced, [y][kz][kx] layout).
//
// Paper: Sec. 4.1 (m^d, Eq. phi_poisson, md_recon), Sec. 4.2 (m^c, Eq. COM_fourier, CF_fourier,
// mc_recon, mc_mean), Sec. 4.4 (Eq. DNS_system, Algorithm 2), Sec. 3.2-3.3 (Eq. dzdt_guesses,
// midpoint RK2), Appendix C (B-spline spaces and the exact derivative map D*).
#include "band.cuh"
#include "ykernels.h"

namespace lmvd {

LMVD_DEFINE_OOB_TAKE(yk)

// ------------------------------------------------------------------ step 1-2 inputs: values at g
// out[0..7] = z, dz/dx, dz/dz, dz/dy, lap z, m1^d, m2^d, m3^d at the Greville points of the order-p space.
// m1^d, m3^d follow Eq. md_recon with d m2^d / dy evaluated directly from the order-(p+1) space;
// the k = 0 mode carries the plane means (and m2^d = 0).
// Rows are split into gridDim.y chunks (row_range), so that a grid with few modes still has enough
// threads, each with its own loads in flight.
__global__ void k_eval_p1(Grid g, DBand B0g, DBand B1g, DBand B2g, DBand Sg0, DBand Sg1, const cd* z,
                          const cd* om, const cd* m2, const double* mm1, const double* mm3, Fields8 out) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  int r0, r1;
  row_range(g.ny, blockIdx.y, gridDim.y, r0, r1);
  if (is_nyquist(g, m)) {
    for (int i = r0; i < r1; ++i)
      for (int f = 0; f < 8; ++f) out.p[f][(size_t)i * M + m] = mk(0, 0);
    return;
  }
  double k1, k3;
  wavenumbers(g, m, k1, k3);
  const double k2 = k1 * k1 + k3 * k3;
  const double ik2 = m == 0 ? 0.0 : 1.0 / k2, a1 = k1 * ik2, a3 = k3 * ik2;
  for (int i = r0; i < r1; ++i) {
    const size_t o = (size_t)i * M + m;
    const cd zg = band_row(B0g, i, z, M, m);
    const cd zy = band_row(B1g, i, z, M, m);
    const cd zyy = band_row(B2g, i, z, M, m);
    out.p[0][o] = zg;
    out.p[1][o] = k1 * times_i(zg);
    out.p[2][o] = k3 * times_i(zg);
    out.p[3][o] = zy;
    out.p[4][o] = fma_rc(-k2, zg, zyy);
    if (m == 0) {
      out.p[5][o] = mk(band_row_real(B0g, i, mm1), 0.0);
      out.p[6][o] = mk(0, 0);
      out.p[7][o] = mk(band_row_real(B0g, i, mm3), 0.0);
    } else {
      const cd dm2 = band_row(Sg1, i, m2, M, m);
      const cd omg = band_row(B0g, i, om, M, m);
      out.p[5][o] = times_i(fma_rc(a1, dm2, (-a3) * omg));
      out.p[6][o] = band_row(Sg0, i, m2, M, m);
      out.p[7][o] = times_i(fma_rc(a3, dm2, a1 * omg));
    }
  }
}

// ------------------------------------------------------------------ generic values at points
// job blockIdx.y: out = B in (or out += B in), rows B.rows split into gridDim.z chunks; Nyquist modes
// zero (or unchanged).
__global__ void k_eval(Grid g, EvalJobs jobs) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const EvalJob& jb = jobs.j[blockIdx.y];
  const size_t M = g.M;
  const bool ny = is_nyquist(g, m);
  int r0, r1;
  row_range(jb.B.rows, blockIdx.z, gridDim.z, r0, r1);
  if (jb.acc) {
    if (ny) return;
    for (int i = r0; i < r1; ++i) jb.out[(size_t)i * M + m] = jb.out[(size_t)i * M + m] + band_row(jb.B, i, jb.in, M, m);
    return;
  }
  for (int i = r0; i < r1; ++i)
    jb.out[(size_t)i * M + m] = ny ? mk(0, 0) : band_row(jb.B, i, jb.in, M, m);
}

// ------------------------------------------------------------------ evaluations in double-float
// The precision path (precision = 1) evaluates the B-spline sums that feed the inverse transforms in
// double-float on the FP32 pipe: the band entries come as pairs (DBand.vf), each complex double input is split
// with integer operations, the products are accumulated without renormalisation (error <= ~w 2^-48 of the sum
// of |terms|), and the result is renormalised. The per-mode multipliers (i k1, 1/k^2, ...) are applied in
// double-float too, so these kernels issue no FP64 instruction per term.

// acc + b * x without renormalisation: TwoProd by FMA, TwoSum of the high parts, low parts summed
__device__ __forceinline__ df dfma_lazy(df b, df x, df acc) {
  const float p = __fmul_rn(b.hi, x.hi);
  float e = __fmaf_rn(b.hi, x.hi, -p);
  e = __fmaf_rn(b.hi, x.lo, e);
  e = __fmaf_rn(b.lo, x.hi, e);
  float s, t;
  two_sum(acc.hi, p, s, t);
  return df{s, __fadd_rn(__fadd_rn(acc.lo, e), t)};
}
__device__ __forceinline__ df drenorm(df a) {
  float s, e;
  two_sum(a.hi, a.lo, s, e);
  return df{s, e};
}
__device__ __forceinline__ cdf cd_to_cdf(cd x) { return cdf{df_from_double_int(x.re), df_from_double_int(x.im)}; }
// The values these evaluations produce feed only the inverse transforms: they are stored as renormalised
// pairs (cdf, the same 16 bytes as a complex double) and the z-pass converts the pairs to its fixed point
// (fft_inverse, fft_inverse_mul with df_in), with fewer instructions than a double's bits need.
__device__ __forceinline__ void put_df(cd* p, size_t o, cdf v) {
  reinterpret_cast<cdf*>(p)[o] = cdf{drenorm(v.re), drenorm(v.im)};
}
__device__ __forceinline__ void put_df(cd* p, size_t o, cd v) { reinterpret_cast<cdf*>(p)[o] = cd_to_cdf(v); }

// A thread walks the rows of one mode, and a band's first column c0[i] never decreases and grows by at
// most one per row (Greville points are at most one knot interval apart), so each input coefficient is
// split into a double-float pair once and kept in a register window of the W columns c .. c + W - 1
// (W = the band width) instead of once per band entry that reads it.
template <int W>
struct DfWin {
  cdf v[W];
  int c = -(1 << 30);
  cd pre;             // the raw coefficient of column pre_col, loaded one row ahead
  int pre_col = -1;
  __device__ __forceinline__ cdf fetch(const cd* x, size_t M, int m, int col, int cols) const {
    if (col == pre_col) return cd_to_cdf(pre);
    return (col < cols && LMVD_IN(col, cols)) ? cd_to_cdf(x[(size_t)col * M + m]) : cdf{};
  }
  __device__ __forceinline__ void load(const cd* x, size_t M, int m, int c0, int cols) {
    c = c0;
#pragma unroll
    for (int q = 0; q < W; ++q) v[q] = fetch(x, M, m, c0 + q, cols);
  }
  // move the window to start at column c0
  __device__ __forceinline__ void seek(const cd* x, size_t M, int m, int c0, int cols) {
    if (c0 < c || c0 > c + 2) {
      load(x, M, m, c0, cols);
      return;
    }
    while (c < c0) {
#pragma unroll
      for (int q = 0; q < W - 1; ++q) v[q] = v[q + 1];
      v[W - 1] = fetch(x, M, m, c + W, cols);
      ++c;
    }
  }
  // issue the load of the column the next row's window adds (its first column is c_next), so that its
  // latency overlaps this row's arithmetic; a thread otherwise has a single load in flight
  __device__ __forceinline__ void prefetch(const cd* x, size_t M, int m, int c_next, int cols) {
    const int col = c_next + W - 1;
    if (c_next > c && col > c + W - 1 && col != pre_col && col < cols && LMVD_IN(col, cols)) {
      pre = x[(size_t)col * M + m];
      pre_col = col;
    }
  }
  // sum over q < w of b[q] v[q] (lazy accumulation)
  __device__ __forceinline__ cdf dot(const DBand& B, int i) const {
    const float2* b = reinterpret_cast<const float2*>(B.vf) + (size_t)i * B.w;
    df ar{0.f, 0.f}, ai{0.f, 0.f};
#pragma unroll
    for (int q = 0; q < W; ++q)
      if (q < B.w) {
        const float2 bq = __ldg(b + q);
        const df bb{bq.x, bq.y};
        ar = dfma_lazy(bb, v[q].re, ar);
        ai = dfma_lazy(bb, v[q].im, ai);
      }
    return cdf{ar, ai};
  }
};
__device__ __forceinline__ cdf cdf_add_lazy(cdf a, cdf b) { return cdf{dadd_lazy(a.re, b.re), dadd_lazy(a.im, b.im)}; }
__device__ __forceinline__ df df_of(double x) { return df_from_double_int(x); }

// k_eval_p1 in double-float (same outputs, same layout, FP64 values); WB: width of the order-p bands (B0g,
// B1g, B2g, one window each for z and Omega2), WS: of the order-(p+1) ones (Sg0, Sg1; one window for m2)
template <int WB, int WS>
__global__ void __launch_bounds__(128) k_eval_p1_df(Grid g, DBand B0g, DBand B1g, DBand B2g, DBand Sg0, DBand Sg1,
                                                    const cd* z, const cd* om, const cd* m2, const double* mm1,
                                                    const double* mm3, Fields8 out) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  int r0, r1;
  row_range(g.ny, blockIdx.y, gridDim.y, r0, r1);
  if (is_nyquist(g, m)) {
    for (int i = r0; i < r1; ++i)
      for (int f = 0; f < 8; ++f) put_df(out.p[f], (size_t)i * M + m, mk(0, 0));
    return;
  }
  if (m == 0) {  // the plane means and the k = 0 z values: one mode, kept in FP64
    for (int i = r0; i < r1; ++i) {
      const size_t o = (size_t)i * M;
      put_df(out.p[0], o, band_row(B0g, i, z, M, 0));
      put_df(out.p[1], o, mk(0, 0));
      put_df(out.p[2], o, mk(0, 0));
      put_df(out.p[3], o, band_row(B1g, i, z, M, 0));
      put_df(out.p[4], o, band_row(B2g, i, z, M, 0));
      put_df(out.p[5], o, mk(band_row_real(B0g, i, mm1), 0.0));
      put_df(out.p[6], o, mk(0, 0));
      put_df(out.p[7], o, mk(band_row_real(B0g, i, mm3), 0.0));
    }
    return;
  }
  double k1d, k3d;
  wavenumbers(g, m, k1d, k3d);
  const double k2d = k1d * k1d + k3d * k3d;
  // per-mode multipliers, split once (one FP64 division per mode, none per row)
  const df k1 = df_of(k1d), k3 = df_of(k3d), nk2 = df_of(-k2d), ik2 = df_of(1.0 / k2d);
  const df nk1 = dneg(k1), nk3 = dneg(k3);
  DfWin<WB> wz, wo;
  DfWin<WS> wm;
  for (int i = r0; i < r1; ++i) {
    if (!LMVD_IN(i, B0g.rows) || !LMVD_IN(i, Sg0.rows)) continue;
    const size_t o = (size_t)i * M + m;
    const int cb = __ldg(B0g.c0 + i), cs = __ldg(Sg0.c0 + i);
    wz.seek(z, M, m, cb, B0g.cols);
    wo.seek(om, M, m, cb, B0g.cols);
    wm.seek(m2, M, m, cs, Sg0.cols);
    if (i + 1 < r1) {
      const int nb = __ldg(B0g.c0 + i + 1), ns = __ldg(Sg0.c0 + i + 1);
      wz.prefetch(z, M, m, nb, B0g.cols);
      wo.prefetch(om, M, m, nb, B0g.cols);
      wm.prefetch(m2, M, m, ns, Sg0.cols);
    }
    const cdf zg = wz.dot(B0g, i), zy = wz.dot(B1g, i), zyy = wz.dot(B2g, i);
    const cdf dm2 = wm.dot(Sg1, i), omg = wo.dot(B0g, i);
    const cdf zgr{drenorm(zg.re), drenorm(zg.im)};
    put_df(out.p[0], o, zgr);
    put_df(out.p[1], o, cdf{dmul(nk1, zgr.im), dmul(k1, zgr.re)});   // i k1 z
    put_df(out.p[2], o, cdf{dmul(nk3, zgr.im), dmul(k3, zgr.re)});   // i k3 z
    put_df(out.p[3], o, zy);
    put_df(out.p[4], o, cdf_add_lazy(cdf{dmul(nk2, zgr.re), dmul(nk2, zgr.im)}, zyy));  // -k^2 z + z''
    const cdf dmr{drenorm(dm2.re), drenorm(dm2.im)}, omr{drenorm(omg.re), drenorm(omg.im)};
    // m1^d = (i k1 dm2 - i k3 om) / k^2, m3^d = (i k3 dm2 + i k1 om) / k^2 (Eq. md_recon)
    const df a1 = ddot2(k1, dmr.re, nk3, omr.re), b1 = ddot2(k1, dmr.im, nk3, omr.im);
    const df a3 = ddot2(k3, dmr.re, k1, omr.re), b3 = ddot2(k3, dmr.im, k1, omr.im);
    put_df(out.p[5], o, cdf{dmul(ik2, dneg(b1)), dmul(ik2, a1)});
    put_df(out.p[6], o, wm.dot(Sg0, i));
    put_df(out.p[7], o, cdf{dmul(ik2, dneg(b3)), dmul(ik2, a3)});
  }
}

// k_eval in double-float (jobs without accumulation into out; values as double-float pairs); W: the widest
// band of the jobs
template <int W>
__global__ void __launch_bounds__(128) k_eval_df(Grid g, EvalJobs jobs) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const EvalJob& jb = jobs.j[blockIdx.y];
  const size_t M = g.M;
  const bool ny = is_nyquist(g, m);
  int r0, r1;
  row_range(jb.B.rows, blockIdx.z, gridDim.z, r0, r1);
  DfWin<W> win;
  for (int i = r0; i < r1; ++i) {
    if (ny) {
      put_df(jb.out, (size_t)i * M + m, mk(0, 0));
      continue;
    }
    win.seek(jb.in, M, m, __ldg(jb.B.c0 + i), jb.B.cols);
    if (i + 1 < r1) win.prefetch(jb.in, M, m, __ldg(jb.B.c0 + i + 1), jb.B.cols);
    put_df(jb.out, (size_t)i * M + m, win.dot(jb.B, i));
  }
}

// k_mc_values in double-float (values as double-float pairs); WS: width of the order-(p+1) bands
template <int WS>
__global__ void __launch_bounds__(128) k_mc_values_df(Grid g, DBand Sg0, DBand Sg1, const cd* rtv, const cd* m2c, cd* v1,
                                                      cd* v2, cd* v3) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  int r0, r1;
  row_range(g.ny, blockIdx.y, gridDim.y, r0, r1);
  if (m == 0 || is_nyquist(g, m)) {  // k = 0: one mode, kept in FP64
    for (int i = r0; i < r1; ++i) {
      const size_t o = (size_t)i * M + m;
      put_df(v1, o, mk(0, 0));
      put_df(v2, o, m == 0 ? band_row(Sg0, i, m2c, M, 0) : mk(0, 0));
      put_df(v3, o, mk(0, 0));
    }
    return;
  }
  double k1, k3;
  wavenumbers(g, m, k1, k3);
  const double ik2 = 1.0 / (k1 * k1 + k3 * k3);
  const df a1 = df_of(k1 * ik2), a3 = df_of(k3 * ik2);
  DfWin<WS> win;
  for (int i = r0; i < r1; ++i) {
    const size_t o = (size_t)i * M + m;
    win.seek(m2c, M, m, __ldg(Sg0.c0 + i), Sg0.cols);
    if (i + 1 < r1) win.prefetch(m2c, M, m, __ldg(Sg0.c0 + i + 1), Sg0.cols);
    const cdf t = cdf_add_lazy(cd_to_cdf(rtv[o]), win.dot(Sg1, i));
    const df tr = drenorm(t.re), ti = drenorm(t.im);
    put_df(v1, o, cdf{dmul(a1, dneg(ti)), dmul(a1, tr)});
    put_df(v2, o, win.dot(Sg0, i));
    put_df(v3, o, cdf{dmul(a3, dneg(ti)), dmul(a3, tr)});
  }
}

// launchers for spline orders 4..8 (band widths 4..9); api.cu brackets them with its launch accounting
void launch_eval_p1_df(int p, dim3 grid, int tpb, cudaStream_t st, const Grid& g, const DBand& B0g, const DBand& B1g,
                       const DBand& B2g, const DBand& Sg0, const DBand& Sg1, const cd* z, const cd* om, const cd* m2,
                       const double* mm1, const double* mm3, const Fields8& out) {
  switch (p) {
#define LMVD_P1(P) \
    case P: launch_next(k_eval_p1_df<P, P + 1>, grid, tpb, 0, st, g, B0g, B1g, B2g, Sg0, Sg1, z, om, m2, mm1, mm3, out); break;
    LMVD_P1(4) LMVD_P1(5) LMVD_P1(6) LMVD_P1(7) LMVD_P1(8)
#undef LMVD_P1
  }
}
void launch_eval_df(int w, dim3 grid, int tpb, cudaStream_t st, const Grid& g, const EvalJobs& jobs) {
  switch (w) {
#define LMVD_EV(W) \
    case W: launch_next(k_eval_df<W>, grid, tpb, 0, st, g, jobs); break;
    LMVD_EV(4) LMVD_EV(5) LMVD_EV(6) LMVD_EV(7) LMVD_EV(8) LMVD_EV(9)
#undef LMVD_EV
  }
}
void launch_mc_values_df(int p, dim3 grid, int tpb, cudaStream_t st, const Grid& g, const DBand& Sg0, const DBand& Sg1,
                         const cd* rtv, const cd* m2c, cd* v1, cd* v2, cd* v3) {
  switch (p) {
#define LMVD_MV(P) \
    case P: launch_next(k_mc_values_df<P + 1>, grid, tpb, 0, st, g, Sg0, Sg1, rtv, m2c, v1, v2, v3); break;
    LMVD_MV(4) LMVD_MV(5) LMVD_MV(6) LMVD_MV(7) LMVD_MV(8)
#undef LMVD_MV
  }
}

// ------------------------------------------------------------------ banded solves
// job blockIdx.y: out = A^{-1} in (+ add), factors shared or per mode (DLU.mstride); used for the
// collocation (interpolation) solves and the per-mode systems. out may alias in. Nyquist modes are set to
// zero. k_solve_cd: one thread per mode (band_solve_cd).
__global__ void k_solve_cd(Grid g, DLU lu, SolveJobs jobs) {
  grid_wait();
  const size_t m = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (m >= g.M) return;
  const SolveJob& jb = jobs.j[blockIdx.y];
  if (is_nyquist(g, (int)m)) {
    for (int i = 0; i < lu.n; ++i) jb.out[(size_t)i * g.M + m] = mk(0, 0);
    return;
  }
  band_solve_cd(lu, (int)m, lu.mstride ? factor_mode(g, (int)m) : 0, jb.in, jb.add, jb.out, g.M);
}
// One thread per (mode, real part), loads pipelined (band_solve_piped); a job may have its own factors, and a job of
// real columns (modes = 0: the plane means) has one thread per column, `part` elements apart.
__global__ void __launch_bounds__(128) k_solve_piped(Grid g, const __grid_constant__ PipedJobs jobs) {
  grid_wait();
  const PipedJob& jb = jobs.j[blockIdx.y];
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const int m = (int)(t >> 1), comp = (int)(t & 1);
  if (m >= (jb.modes ? jb.modes : 1)) return;
  const long long o = jb.modes ? (long long)t : comp * jb.part, rs = jb.modes ? 2ll * jb.modes : 1;
  const DLU lu = jb.lu;
  if (jb.modes && is_nyquist(g, m)) {
    for (int i = 0; i < lu.n; ++i) jb.out[o + i * rs] = 0.0;
    return;
  }
  band_solve_piped(lu, lu.mstride ? factor_mode(g, m) : 0, jb.in + o, jb.add ? jb.add + o : nullptr, jb.out + o, rs);
}

// ------------------------------------------------------------------ m^c from rho_t
// Eq. COM_fourier + CF_fourier with m_par eliminated: rows 1..ny-1 collocate
// (B*'' - k^2 B*) m2^c = -B' rho_t at the interior order-(p+1) Greville points, rows 0 and ny hold the
// boundary rows (walls: m2^c(+-1) = 0; potential matching: the Robin rows), all with zero right-hand side.
// Then m_par = i (rho_t + D* m2^c) / k (exact mass conservation in B-coefficient space) and
// Eq. mc_recon m1^c = k1/k m_par, m3^c = k3/k m_par.
// k = 0 (Eq. mc_mean): D* <m2^c> = -<rho_t> with <m2^c>(+1) = 0; <m1^c> = <m3^c> = 0.
// k_mc_rhs writes the right-hand side into m2c, the banded solve runs in place with per-mode factors (those of k = 0
// are the summation of Eq. mc_mean), k_mc_values gives the values of m^c at g for the transforms, k_mc_post the
// coefficients of m1^c and m3^c.

// rows 0..ny split over gridDim.y chunks
__global__ void k_mc_rhs(Grid g, DBand Bs1, const double* dstar, const cd* rt, cd* m2c) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  const int ny = g.ny;
  int r0, r1;
  row_range(ny + 1, blockIdx.y, gridDim.y, r0, r1);
  const bool zero = is_nyquist(g, m);
  for (int i = r0; i < r1; ++i) {
    cd v = mk(0, 0);
    if (m == 0) {
      if (i < ny) v = (1.0 / __ldg(dstar + i)) * rt[(size_t)i * M];
    } else if (!zero && i > 0 && i < ny) {
      const cd d = band_row(Bs1, i, rt, M, m);
      v = mk(-d.re, -d.im);
    }
    m2c[(size_t)i * M + m] = v;
  }
}

// rows 0..ny-1 split over gridDim.y chunks
__global__ void k_mc_post(Grid g, const double* dstar, const cd* rt, cd* m1c, const cd* m2c, cd* m3c) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  const int ny = g.ny;
  int r0, r1;
  row_range(ny, blockIdx.y, gridDim.y, r0, r1);
  if (m == 0 || is_nyquist(g, m)) {
    for (int i = r0; i < r1; ++i) m1c[(size_t)i * M + m] = m3c[(size_t)i * M + m] = mk(0, 0);
    return;
  }
  double k1, k3;
  wavenumbers(g, m, k1, k3);
  const double k = sqrt(k1 * k1 + k3 * k3), ik = 1.0 / k;
  for (int i = r0; i < r1; ++i) {
    if (!LMVD_IN(i + 1, ny + 1)) continue;
    const cd x = m2c[(size_t)i * M + m], xn = m2c[(size_t)(i + 1) * M + m];
    const cd dm = __ldg(dstar + i) * (xn - x);
    const cd mpar = ik * times_i(rt[(size_t)i * M + m] + dm);
    m1c[(size_t)i * M + m] = (k1 * ik) * mpar;
    m3c[(size_t)i * M + m] = (k3 * ik) * mpar;
  }
}

// Values of m^c at g: v2 = B* m2^c, (v1, v3) = i (k1, k3) / k^2 (rho_t + d m2^c / dy) with rtv the values of rho_t; zero
// v1, v3 at k = 0. Rows split over gridDim.y chunks.
__global__ void k_mc_values(Grid g, DBand Sg0, DBand Sg1, const cd* rtv, const cd* m2c, cd* v1, cd* v2, cd* v3) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  int r0, r1;
  row_range(g.ny, blockIdx.y, gridDim.y, r0, r1);
  const bool zero = is_nyquist(g, m);
  double a1 = 0.0, a3 = 0.0;
  if (m != 0 && !zero) {
    double k1, k3;
    wavenumbers(g, m, k1, k3);
    const double ik2 = 1.0 / (k1 * k1 + k3 * k3);
    a1 = k1 * ik2;
    a3 = k3 * ik2;
  }
  for (int i = r0; i < r1; ++i) {
    const size_t o = (size_t)i * M + m;
    cd w = mk(0, 0), t = mk(0, 0);
    if (!zero) {
      w = band_row(Sg0, i, m2c, M, m);
      if (m != 0) t = times_i(rtv[o] + band_row(Sg1, i, m2c, M, m));
    }
    v1[o] = a1 * t;
    v2[o] = w;
    v3[o] = a3 * t;
  }
}

// ------------------------------------------------------------------ RHS streams (Eq. DNS_system)
// sv[0..8] = C11 - C22, C12, C13, C23, C33 - C22, u1, u2, u3, rho at the Greville points (values).
// With H_i = d_j C_ij + mu lap u_i - g rho delta_i2 (the (1/3) grad div u part of the viscous force and C22 delta_ij
// are gradients and cancel in both curls):
//   RHS_Omega2 = i k3 H1 - i k1 H3 = st0 + d/dy st1 + d2/dy2 st2,
//   RHS_phi2 = -k^2 H2 - d/dy (i k1 H1 + i k3 H3) = st3 + d/dy st4 + d2/dy2 st5 + d3/dy3 st6,
// so only st1..st6 need B-spline coefficients (st0 is already the value at g).
// k = 0: st1 = <C12>, st2 = mu <u1>, st4 = <C23>, st5 = mu <u3> carry the mean equations
// (Eq. mean_m1m3); the k = 0 values of all seven streams vanish otherwise.
// One thread per mode and row chunk: the multipliers are formed once per mode.
__global__ void k_rhs_combine(Grid g, double mu, double grav, Fields9C sv, Fields7 st) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  int r0, r1;
  row_range(g.ny, blockIdx.y, gridDim.y, r0, r1);
  if (is_nyquist(g, m)) {
    for (int i = r0; i < r1; ++i)
      for (int q = 0; q < 7; ++q) st.p[q][(size_t)i * M + m] = mk(0, 0);
    return;
  }
  if (m == 0) {
    for (int i = r0; i < r1; ++i) {
      const size_t o = (size_t)i * M;
      const cd C12 = sv.p[1][o], C23 = sv.p[3][o], u1 = sv.p[5][o], u3 = sv.p[7][o];
      st.p[0][o] = st.p[3][o] = st.p[6][o] = mk(0, 0);
      st.p[1][o] = C12;
      st.p[2][o] = mu * u1;
      st.p[4][o] = C23;
      st.p[5][o] = mu * u3;
    }
    return;
  }
  double k1, k3;
  wavenumbers(g, m, k1, k3);
  const double k11 = k1 * k1, k33 = k3 * k3, k13 = k1 * k3, k2 = k11 + k33, kd = k11 - k33, m2 = mu * k2, m4 = m2 * k2;
  for (int i = r0; i < r1; ++i) {
    const size_t o = (size_t)i * M + m;
    const cd D11 = sv.p[0][o], C12 = sv.p[1][o], C13 = sv.p[2][o], C23 = sv.p[3][o], D33 = sv.p[4][o], u1 = sv.p[5][o],
             u2 = sv.p[6][o], u3 = sv.p[7][o], rho = sv.p[8][o];
    const cd w13 = times_i(fma_rc(k3, u1, (-k1) * u3));      // i k3 u1 - i k1 u3
    const cd d13 = times_i(fma_rc(k1, u1, k3 * u3));         // i k1 u1 + i k3 u3
    const cd c1223 = times_i(fma_rc(k1, C12, k3 * C23));     // i k1 C12 + i k3 C23
    const cd nc = mk(-c1223.re, -c1223.im);
    st.p[0][o] = fma_rc(-m2, w13, fma_rc(kd, C13, k13 * (D33 - D11)));
    st.p[1][o] = times_i(fma_rc(k3, C12, (-k1) * C23));
    st.p[2][o] = mu * w13;
    st.p[3][o] = fma_rc(m4, u2, k2 * fma_rc(grav, rho, nc));
    st.p[4][o] = fma_rc(m2, d13, fma_rc(k33, D33, fma_rc(2.0 * k13, C13, k11 * D11)));
    st.p[5][o] = fma_rc(-m2, u2, nc);
    st.p[6][o] = (-mu) * d13;
  }
}

// RHS values from the streams (st1..st6 now B coefficients): R_Omega2 at g (ny rows), R_phi2 at g*
// (ny + 1 rows), and for k = 0 the mean RHS (2 ny reals).
// Rows 0..ny (R_phi2 has ny + 1) are split into gridDim.y chunks.
__global__ void k_rhs_eval(Grid g, DBand B1g, DBand B2g, DBand Bs0, DBand Bs1, DBand Bs2, DBand Bs3, Fields7C st,
                           cd* r_om, cd* r_phi, double* r_m) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  const int ny = g.ny;
  int r0, r1;
  row_range(ny + 1, blockIdx.y, gridDim.y, r0, r1);
  if (m == 0 || is_nyquist(g, m)) {
    for (int i = r0; i < r1; ++i) {
      if (i < ny) r_om[(size_t)i * M + m] = mk(0, 0);
      r_phi[(size_t)i * M + m] = mk(0, 0);
      if (m == 0 && i < ny) {
        r_m[i] = (band_row(B1g, i, st.p[1], M, 0) + band_row(B2g, i, st.p[2], M, 0)).re;
        r_m[ny + i] = (band_row(B1g, i, st.p[4], M, 0) + band_row(B2g, i, st.p[5], M, 0)).re;
      }
    }
    return;
  }
  for (int i = r0; i < r1; ++i) {
    if (i < ny)
      r_om[(size_t)i * M + m] = st.p[0][(size_t)i * M + m] + band_row(B1g, i, st.p[1], M, m) +
                                band_row(B2g, i, st.p[2], M, m);
    r_phi[(size_t)i * M + m] = band_row(Bs0, i, st.p[3], M, m) + band_row(Bs1, i, st.p[4], M, m) +
                               band_row(Bs2, i, st.p[5], M, m) + band_row(Bs3, i, st.p[6], M, m);
  }
}

// ------------------------------------------------------------------ RK2 update (step 6)
// Midpoint RK2 in low-storage form at the collocation points, X^{s+1} = X^s + dt (al R^s + be R^{s-1}), with boundary
// rows:
//  * Omega2 (blockIdx.z = 0) and m2^d (blockIdx.z = 2) in increments of the coefficients: the interior rows of their
//    solves are those that evaluate X^s, so evaluating X^s and solving is X^s itself, and X^{s+1} = X^s + A^{-1} r with r
//    the increments and, in the boundary rows, minus those rows applied to X^s. Omega2: increments at g, Dirichlet
//    rows (interpolation LU). m2^d (Eq. phi_poisson): increments of phi2 = (B*'' - k^2 B*) m2^d at g*_2 .. g*_{ny-2}, four
//    boundary rows of A(k) (no-slip or potential matching); k = 0: zero.
//  * z (blockIdx.z = 1): t = z + dt (al zdot + be zdot_prev) evaluated at g, Neumann rows dz/dy = 0 (Neumann LU). Its
//    coefficients would be t but for the walls; but the next guess divides differences of z by dt, so z keeps the
//    rounding of an evaluation and a solve. Each t is formed once and kept in a window of W coefficients.
//  * plane means <m1>, <m3> (blockIdx.z = 3, one thread per row and component): values at g advanced, boundary rows zero.
// This kernel writes the right-hand sides into the new fields; rows split over gridDim.y chunks.
template <int W>
__global__ void k_update_rhs(Grid g, DBand B0g, const __grid_constant__ UpdateArgs a) {
  grid_wait();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  const int ny = g.ny;
  const int job = blockIdx.z;
  const double dal = a.dt * a.al, dbe = a.dt * a.be;
  if (job == 3) {
    if (blockIdx.y != 0 || m >= 2 * ny) return;
    const int c = m / ny, i = m - c * ny;
    const double v = i > 0 && i < ny - 1 ? band_row_real(B0g, i, c == 0 ? a.mm1 : a.mm3) +
                                               (dal * a.r_m[m] + dbe * a.r_m_prev[m])
                                         : 0.0;
    (c == 0 ? a.mm1_new : a.mm3_new)[i] = v;
    return;
  }
  if (m >= (int)g.M) return;
  const size_t M = g.M;
  const int rows = job == 2 ? ny + 1 : ny;
  int r0, r1;
  row_range(rows, blockIdx.y, gridDim.y, r0, r1);
  cd* out = job == 0 ? a.om_new : (job == 1 ? a.z_new : a.m2_new);
  if (is_nyquist(g, m) || (job != 1 && m == 0)) {
    for (int i = r0; i < r1; ++i) out[(size_t)i * M + m] = mk(0, 0);
    return;
  }
  if (job == 1) {
    auto t = [&](int i) {
      if (!LMVD_IN(i, B0g.cols)) return mk(0, 0);
      const size_t o = (size_t)i * M + m;
      return a.z[o] + a.dt * (a.al * a.zdot[o] + a.be * a.zdot_prev[o]);
    };
    cd w[W];
    int c = -(1 << 30);
    for (int i = r0; i < r1; ++i) {
      cd v = mk(0, 0);
      if (i > 0 && i < ny - 1 && LMVD_IN(i, B0g.rows)) {
        const int ci = __ldg(B0g.c0 + i);
        if (ci == c + 1) {
#pragma unroll
          for (int q = 0; q + 1 < W; ++q) w[q] = w[q + 1];
          w[W - 1] = t(ci + W - 1);
        } else if (ci != c) {
#pragma unroll
          for (int q = 0; q < W; ++q) w[q] = t(ci + q);
        }
        c = ci;
        const int n = __ldg(B0g.cnt + i);
#pragma unroll
        for (int q = 0; q < W; ++q)
          if (q < n) v = fma_rc(__ldg(B0g.v + (size_t)i * W + q), w[q], v);
      }
      out[(size_t)i * M + m] = v;
    }
    return;
  }
  const cd* x = job == 0 ? a.om : a.m2;
  const cd* r = job == 0 ? a.r_om : a.r_phi;
  const cd* rp = job == 0 ? a.r_om_prev : a.r_phi_prev;
  const int nb = job == 0 ? 1 : 2;  // boundary rows at each end
  for (int i = r0; i < r1; ++i) {
    const size_t o = (size_t)i * M + m;
    cd v;
    if (i >= nb && i < rows - nb) {
      const cd p = rp[o], q = r[o];
      v = mk(fma(dal, q.re, dbe * p.re), fma(dal, q.im, dbe * p.im));
    } else if (job == 0) {
      v = band_row(B0g, i, x, M, m);
      v = mk(-v.re, -v.im);
    } else {
      double k1, k3;
      wavenumbers(g, m, k1, k3);
      const double k2 = k1 * k1 + k3 * k3, k = sqrt(k2);
      v = mk(0, 0);
      for (int q = -a.md.K; q <= a.md.K; ++q) {
        const int j = i + q;
        if (j < 0 || j >= a.md.n) continue;
        const size_t e = (size_t)i * (2 * a.md.K + 1) + q + a.md.K;
        const double c = __ldg(a.md.A2 + e) - k2 * __ldg(a.md.A0 + e) + k * __ldg(a.md.A1 + e);
        if (LMVD_IN(j, ny + 1)) v = fma_rc(-c, x[(size_t)j * M + m], v);
      }
    }
    out[o] = v;
  }
}

void launch_update_rhs(int p, dim3 grid, int tpb, cudaStream_t st, const Grid& g, const DBand& B0g, const UpdateArgs& a) {
  switch (p) {
#define LMVD_UP(P) \
    case P: launch_next(k_update_rhs<P>, grid, tpb, 0, st, g, B0g, a); break;
    LMVD_UP(4) LMVD_UP(5) LMVD_UP(6) LMVD_UP(7) LMVD_UP(8)
#undef LMVD_UP
  }
}

// ------------------------------------------------------------------ failure detection
// Sets bit 0 of *flag if array blockIdx.y of the job list holds a non-finite double (inf or nan: all
// exponent bits set). Integer tests on the bit pattern keep this off the FP64 pipe; one atomic per warp.
__global__ void k_check_finite(CheckJobs jobs, unsigned* flag) {
  grid_wait();
  const CheckJob jb = pick(jobs.j, (int)blockIdx.y);
  bool bad = false;
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < jb.n; o += (size_t)gridDim.x * blockDim.x)
    bad |= (__double_as_longlong(jb.p[o]) & 0x7FF0000000000000ll) == 0x7FF0000000000000ll;
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1u);
}

// ------------------------------------------------------------------ diagnostics (lmvd_diagnostics)
// Block sums then one atomicAdd per block (the record is not bitwise reproducible; it is diagnostic only).
__device__ inline void block_add(double v, double* out) {
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(out, v);
  }
}

// out[0] += |a - b|^2, out[1] += |a|^2 over n complex entries
__global__ void k_diff_norms(size_t n, const cd* a, const cd* b, double* out) {
  grid_wait();
  double d = 0.0, s = 0.0;
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    const cd x = a[o], y = b[o];
    const double dr = x.re - y.re, di = x.im - y.im;
    d += dr * dr + di * di;
    s += x.re * x.re + x.im * x.im;
  }
  block_add(d, out);
  block_add(s, out + 1);
}

// Mass conservation of m^c in B-coefficient space (Sec. 4.2): out[0] += |rho_t + i k1 m1 + i k3 m3 + D* m2|^2,
// out[1] += |rho_t|^2, over all rows and modes (k = 0 included: D* <m2^c> = -<rho_t>)
__global__ void k_mass_norms(Grid g, const double* dstar, const cd* rt, const cd* m1, const cd* m2, const cd* m3,
                             double* out) {
  grid_wait();
  const size_t n = (size_t)g.ny * g.M;
  double d = 0.0, s = 0.0;
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(o % g.M), i = (int)(o / g.M);
    double k1, k3;
    wavenumbers(g, m, k1, k3);
    const cd r = rt[o];
    const cd dm = __ldg(dstar + i) * (m2[o + g.M] - m2[o]);
    const cd res = r + times_i(k1 * m1[o] + k3 * m3[o]) + dm;
    d += res.re * res.re + res.im * res.im;
    s += r.re * r.re + r.im * r.im;
  }
  block_add(d, out);
  block_add(s, out + 1);
}

// Kinetic energy (1/2) integral of |m|^2 / rho over the domain and max |m|^2 over the grid, m = m^d + m^c on the
// padded grid. A plane's mean of a product on the 3/2 grid is the k = 0 coefficient of the dealiased product;
// the y-integral uses the quadrature weights of the Greville interpolant (wq), and the x-z area lx lz is
// applied on the host.
__global__ void k_energy_norms(Grid g, const double* wq, Fields3C md, Fields3C mc, const double* invrho, double* ke,
                               unsigned long long* m2max) {
  grid_wait();
  const size_t n = (size_t)g.ny * g.P;
  double e = 0.0, mx = 0.0;
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    double mm = 0.0;
    for (int c = 0; c < 3; ++c) {
      const double m = md.p[c][o] + mc.p[c][o];
      mm = fma(m, m, mm);
    }
    e = fma(0.5 * __ldg(wq + o / g.P) * mm, invrho[o], e);
    mx = fmax(mx, mm);
  }
  block_add(e / (double)g.P, ke);
  for (int q = 16; q > 0; q >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, q));
  if ((threadIdx.x & 31) == 0) atomicMax(m2max, (unsigned long long)__double_as_longlong(mx));
}

// bit 1 of *flag if the last (the kf-th) fixed-point application, recorded at diag[2 kf], diag[2 kf + 1],
// still changed dz/dt by half its size or more
__global__ void k_fp_check(const double* diag, int kf, unsigned* flag) {
  grid_wait();
  if (kf < 1) return;
  const double d = diag[2 * kf], s = diag[2 * kf + 1];
  if (d >= 0.25 * s && d > 0.0) atomicOr(flag, 2u);
}

// ------------------------------------------------------------------ elementwise helpers
// BDF-like guess (Eq. dzdt_guesses): zdot = (a0 z^s + a1 z^{s-1} + a2 z^{s-2} + a3 z^{s-3}) / dt.
__global__ void k_bdf(size_t n, double a0, double a1, double a2, double a3, double idt, const cd* z, const cd* h0,
                      const cd* h1, const cd* h2, cd* out) {
  grid_wait();
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x)
    out[o] = idt * (a0 * z[o] + a1 * h0[o] + a2 * h1[o] + a3 * h2[o]);
}

// start-up history: zh_q = z - c_q dt zdot
__global__ void k_backfill(size_t n, double c0, double c1, double c2, const cd* z, const cd* zdot, cd* h0, cd* h1,
                           cd* h2) {
  grid_wait();
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    const cd zz = z[o], d = zdot[o];
    h0[o] = zz - c0 * d;
    h1[o] = zz - c1 * d;
    h2[o] = zz - c2 * d;
  }
}

// zero the Nyquist slots of a spectral field and, if zero_mean, its k = 0 slot
__global__ void k_sanitize(Grid g, int rows, cd* f, int zero_mean) {
  grid_wait();
  const size_t n = (size_t)rows * g.M;
  for (size_t o = blockIdx.x * (size_t)blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(o % g.M);
    if (is_nyquist(g, m) || (zero_mean && m == 0)) f[o] = mk(0, 0);
  }
}

// ------------------------------------------------------------------ per-mode factorisation
// LU (no pivoting) of A(k) = A2 - k^2 A0 + k A1 for the factor modes (kx, kz >= 0), mf = jz * nxh + kx,
// jz = 0..nz/2 (stride Mh = (nz/2 + 1) nxh); A2, A0, A1 in diagonal band storage (half-width K, shared),
// profile nl/nu shared; entries outside the profile are stored as zeros. k = 0 and Nyquist modes get
// identity factors, or with mean_rows the k = 0 mode those of x_i - x_{i+1} = r_i (x_{n-1} = r_{n-1}).
__global__ void k_factor(Grid g, int n, int K, const double* A2, const double* A0, const double* A1, const int* nl,
                         const int* nu, double* lo, double* up, double* invd, int mean_rows) {
  grid_wait();
  const size_t Mh = (size_t)(g.nz / 2 + 1) * g.nxh;
  const int mf = blockIdx.x * blockDim.x + threadIdx.x;
  if (mf >= (int)Mh) return;
  const int jz = mf / g.nxh, kx = mf - jz * g.nxh;
  const int W = 2 * K + 1;
  if (mf == 0 || kx == g.nx / 2 || jz == g.nz / 2) {
    for (int i = 0; i < n; ++i) {
      for (int q = 0; q < K; ++q) lo[(size_t)(i * K + q) * Mh + mf] = up[(size_t)(i * K + q) * Mh + mf] = 0.0;
      invd[(size_t)i * Mh + mf] = 1.0;
      if (mean_rows && mf == 0 && i < n - 1) up[(size_t)(i * K) * Mh] = -1.0;
    }
    return;
  }
  const double k1 = 6.283185307179586476925286766559 / g.lx * kx;
  const double k3 = 6.283185307179586476925286766559 / g.lz * jz;
  const double k2 = k1 * k1 + k3 * k3, k = sqrt(k2);
  double row[2 * KMAX + 1];
  for (int i = 0; i < n; ++i) {
    for (int q = 0; q < W; ++q)
      row[q] = A2[(size_t)i * W + q] - k2 * A0[(size_t)i * W + q] + k * A1[(size_t)i * W + q];
    for (int q = nl[i]; q >= 1; --q) {
      const int c = i - q;
      const double l = row[K - q] * invd[(size_t)c * Mh + mf];
      lo[(size_t)(i * K + q - 1) * Mh + mf] = l;
      row[K - q] = 0.0;
      for (int r = 1; r <= nu[c]; ++r) row[K - q + r] -= l * up[(size_t)(c * K + r - 1) * Mh + mf];
    }
    invd[(size_t)i * Mh + mf] = 1.0 / row[K];
    for (int r = 1; r <= K; ++r) up[(size_t)(i * K + r - 1) * Mh + mf] = r <= nu[i] ? row[K + r] : 0.0;
    for (int q = nl[i] + 1; q <= K; ++q) lo[(size_t)(i * K + q - 1) * Mh + mf] = 0.0;
  }
}

}  // namespace lmvd
