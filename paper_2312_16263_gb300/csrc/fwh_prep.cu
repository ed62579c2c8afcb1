// Observer-independent source-time series of the FW-H integrand ("compute
// Noise", Sec. III B), per panel and source sample:
//   Qn  = rho' (U.n) + (1 + rho') (u'.n)                  (Eq. Qn_New_nd)
//   L_c = p' n_c + (1 + rho') u'_c (U.n + u'.n)           (Eq. Li_New_nd)
// in pulsation-expanded form (no cancellation of O(1) terms in FP32), their
// second-order source-time derivatives (central inside, one-sided 3-point at
// the first and last frame), and the cubic B-spline coefficients of the
// natural spline of all eight series, used by the spline interpolation onto
// the observer grid ("interp pressure signal").  The spline of the per-panel
// signal sum_s c_s F_s has coefficients sum_s c_s beta(F_s) by linearity, so
// they are computed once per panel instead of once per (panel, observer).
//
// With m the natural-spline second derivatives, tridiag(1, 4, 1) m = (6/dt^2)
// D2 F on rows 1 .. N - 2 and m_0 = m_{N-1} = 0, the coefficients are
// beta = F - m dt^2 / 6.  Extending F by point reflection about its end
// values, F(-k) = 2 F(0) - F(k) and likewise at N - 1, makes the end
// conditions hold by symmetry (and gives the ghost coefficients beta_{-1},
// beta_N), so the solve is the infinite Toeplitz inverse, which factors as
//   tridiag(1, 4, 1)^-1 = -rho (1 - rho z)^-1 (1 - rho z^-1)^-1,  rho = sqrt 3 - 2,
// a causal recursion y_k = r_k + rho y_{k-1} followed by an anti-causal one
// x_k = y_k + rho x_{k+1}:
//   beta_k = F_k + rho x_k   with r = D2 F          (FP32: no loss at low frequency)
//   beta_k = F_0 - 6 rho x_k with r = F - F_0       (FP64: fewer operations; F_0
//                                                    a constant, see below)
// A recursion started H samples outside the 64-row block it serves errs by
// |rho|^H (H = 16 for FP32, 32 for FP64: below rounding), so blocks are
// independent.  At the record ends both start exactly: y_0 is a sum over the
// first H samples of the reflected series, and beta_{N-1} = F_{N-1} gives
// x_{N-1}.
//
// Away from the record ends the solve commutes with the central difference, so
// a derivative series' coefficients are the central differences d_k =
// (beta_{k+1} - beta_{k-1}) / (2 dt) of its value series' coefficients: four
// filters, not eight.  Near an end they differ by a solution of the
// homogeneous system: beta'_k = d_k + (D_0 - d_0) rho^k from the start (D_0 the
// one-sided derivative, d_0 = (beta_1 - beta_0) / dt), and likewise from the end.
//
// A mean of F far above its changes (a mean pressure on a flat face) must not round
// into the differences.  FP32 forms d_k from the differences of F and of x, not of the
// rounded beta (a fluctuation under a mean of 1000 amplitudes: error 4e-5, 6e-4 with
// differences of beta; no time lost).  FP64 filters F less its value at the work
// unit's first sample, which the integrands' last multiply-adds subtract: 5e-14, and
// 1.2e-12 with the filter's gain folded into the normals, which saved a multiply-add
// per value (32768 panels x 2048 steps 5.28 against 5.70 ms, 2048 x 256 113 against
// 118 us).
//
// Kernels: k_prep_iir_int (FP32) and k_prep_f64_int (FP64), persistent CTAs that
// walk consecutive blocks of a panel group; k_prep_iir for records too short for
// them (under H + 3 samples), all eight series by index arithmetic.  All
// take the panels in the caller's order, so field reads are coalesced also
// for a reordered surface; the rows of X go where the panel's place is.
#include "fwh_internal.cuh"

#include <algorithm>
#include <atomic>

#include <cstdint>

namespace fwh {

namespace {

constexpr double kRho = -0.26794919243112270647;  // sqrt(3) - 2

constexpr int kIirPanels = 8;
constexpr int kIirChunk = 64;
constexpr int kIirJ = 32;
constexpr int kIirThreads = kIirPanels * 8 * (kIirChunk / kIirJ);
constexpr int kIirH = Prec<float>::halo;
template <typename T>
constexpr int iir_rows() { return kIirChunk + 2 * Prec<T>::halo + 6; }  // bound on the staged rows
constexpr int kIirQ = 8;  // integrand stride in a staged row ([4 integrands][8 panels])
constexpr int kIirRow = 4 * kIirQ;                   // staged row stride (values)

// ---------------------------------------------------------------------------
// FP32 prep: one thread owns one (panel, integrand) over a whole 64-row block
// and stores the pair (derivative, value) of each sample, 8 of the 32 bytes of
// an X row.  Bound by HBM: 20 bytes in and 32 out per (panel, sample), 5.1 TB/s
// (75 % of a copy's).  The blocks at the record ends take the same filters with
// exact starts (edge_block); as a kernel of their own that filtered all eight
// reflected series they took 0.32 of 0.88 ms at 32768 panels x 2048 steps; the
// whole prep now takes 0.68.
// ---------------------------------------------------------------------------
constexpr int kIntPanels = 16;
constexpr int kIntThreads = kIntPanels * 4;
constexpr int kIntRow = kIntPanels * 4;              // staged row: [panel][integrand]
constexpr int kIntRows = kIirChunk + 2 * kIirH + 3;  // samples c0 - H - 2 .. c0 + 64 + H
constexpr int kIntKeep = kIntRows - kIirChunk;       // rows shared by consecutive blocks
// fields of 64 frames in flight, or (record ends) y of 81 rows of the window
constexpr int kIntRaw = kIirChunk * 5 * kIntPanels + kIntRow;
static_assert(kIntRaw >= (kIirChunk + kIirH + 1) * kIntRow, "y of an end block fits");
constexpr int kIntUnit = 8;                          // most blocks per work unit

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 4 : 0;  // zero fill
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_async8(double *dst, const double *src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 8 : 0;  // zero fill
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// rho^k, k < kIirH + 4 (below FP32 rounding from there on).
struct RhoPow {
  float v[kIirH + 4];
  constexpr RhoPow() : v() {
    double p = 1.0;
    for (int i = 0; i < kIirH + 4; ++i, p *= kRho) v[i] = (float)p;
  }
};
__constant__ RhoPow c_rho_pow = RhoPow();

// A block at a record end: bc[k kIntRow] is the integrand of sample c0 + k (valid
// inside the record), ys[(k + 1) kIntRow] takes y, xr is the thread's pair in the
// block's first X row, `room` the rows of X from there on.  Compact loops: a
// small problem has little else to do, and unrolled code reaches it through
// cold instruction caches (24 us for 64 panels x 48 steps unrolled, 18 so).
__device__ __forceinline__ void edge_block(const float *bc, float *ys, float *xr, int c0, int N,
                                           float inv2h, int room, bool store) {
  constexpr int H = kIirH, C = kIirChunk;
  constexpr float rho = (float)kRho;
  auto B = [&](int k) -> float { return bc[k * kIntRow]; };
  auto y = [&](int k) -> float & { return ys[(k + 1) * kIntRow]; };
  const bool start = c0 < 0;                    // c0 = -1: sample 0 at k = 1
  const int top = min(C + H, N - 1 - c0);       // the anti-causal recursion starts here
  float yy = 0.f;
  int k = -1 - H;
  if (start) {  // y of sample 0 from the reflected series
    for (int j = H; j >= 1; --j) yy = (yy - (B(j + 2) - 2.f * B(j + 1) + B(j))) * rho;
    y(-1) = y(0) = 0.f;
    y(1) = yy;
    k = 2;
  }
  {
    float Bm = B(k - 1), B0 = B(k);
#pragma unroll 4
    for (; k < top; ++k) {
      const float Bp = B(k + 1);
      yy = (Bp - 2.f * B0 + Bm) + rho * yy;
      if (k >= -1) y(k) = yy;
      Bm = B0;
      B0 = Bp;
    }
  }
  float D0 = 0.f, ex = 0.f;  // one-sided derivative at sample 0, its excess over the central one
  if (start) {
    float x1 = 0.f;
    for (int j = H + 2; j >= 2; --j) x1 = y(j) + rho * x1;
    D0 = (-3.f * B(1) + 4.f * B(2) - B(3)) * inv2h;
    ex = D0 - fmaf(rho, x1, B(2) - B(1)) * (2.f * inv2h);
  }
  // coefficients, integrand and recursion at k + 1 and k + 2
  float xx = 0.f, b1v = 0.f, b2v = 0.f, F1 = 0.f, F2 = 0.f, x1 = 0.f, x2 = 0.f;
  float cr = 0.f, DN = 0.f, d2 = 0.f;
#pragma unroll 2
  for (k = top; k >= -1; --k) {
    const int sk = c0 + k;
    if (k < top) xx = y(k) + rho * xx;
    const float F0 = B(k), bk = fmaf(rho, xx, F0);
    cr *= rho;
    if (sk == N - 2) {
      DN = (3.f * F1 - 4.f * F0 + B(k - 1)) * inv2h;
      cr = DN - fmaf(rho, x1 - xx, F1 - F0) * (2.f * inv2h);
    }
    // sample se = sk + 1, row e of the block, is now complete
    const int e = k + 1, se = sk + 1;
    float d = fmaf(rho, x2 - xx, F2 - F0) * inv2h + cr;
    if (start && se < H + 4 && se > 0) d += ex * c_rho_pow.v[se];
    if (e < C && se <= N - 2 && store) {
      float2 *row = reinterpret_cast<float2 *>(xr + e * kSer);
      constexpr int NR = kSer / 2;  // a row in pairs
      if (!(start && e <= 1)) *row = make_float2(d, b1v);
      if (start && e == 1) {  // sample 0 and the ghost before it
        row[0] = make_float2(D0, b1v);
        row[-NR] = make_float2(2.f * D0 - d2, 2.f * b1v - b2v);
      }
      if (se == N - 2) {  // the last sample, the ghost after it and a zero row
        const float bN = B(e + 1);
        if (e + 1 < room) row[NR] = make_float2(DN, bN);
        if (e + 2 < room) row[2 * NR] = make_float2(2.f * DN - d, 2.f * bN - b1v);
        if (e + 3 < room) row[3 * NR] = make_float2(0.f, 0.f);
      }
    }
    d2 = d;
    b2v = b1v;
    b1v = bk;
    F2 = F1;
    F1 = F0;
    x2 = x1;
    x1 = xx;
  }
}

__global__ void __launch_bounds__(kIntThreads, 4) k_prep_iir_int(PrepArgs<float> a, int unit) {
  constexpr int NP = kIntPanels, H = kIirH, C = kIirChunk;
  constexpr float rho = -0.267949192431122706f;  // sqrt(3) - 2
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *sb = reinterpret_cast<float *>(smem_raw);  // [kIntRows][NP][4] integrands
  float *raw = sb + kIntRows * kIntRow;             // [C rows][5][NP] fields in flight
  const int tid = threadIdx.x;
  const int n_pg = (a.P + NP - 1) / NP;
  const int n_blk = a.c_hi - a.c_lo;
  const int n_us = (n_blk + unit - 1) / unit;
  const long n_units = (long)n_pg * n_us;
  // phase A thread: panel pa, rows tid / NP + 4 u
  const int pa = tid % NP;
  // phase B thread: integrand qi of panel pl
  const int qi = tid & 3;
  const int pl = tid >> 2;
  const float inv2h = (float)(0.5 / a.dt);
  const bool vec = (a.P & 3) == 0 && ((size_t)a.fields & 15) == 0;  // 16-byte copies of 4 panels
  for (long u = blockIdx.x; u < n_units; u += gridDim.x) {
    // panel group fastest: concurrent units read neighbouring segments of the same rows
    const int p0 = (int)(u % n_pg) * NP;
    const int b0 = a.c_lo + (int)(u / n_pg) * unit;
    const int b1 = min(a.c_hi, b0 + unit);
    const int p = p0 + pa;
    const bool live = p < a.P;
    float n0 = 0.f, n1 = 0.f, n2 = 0.f, Un = 0.f;
    if (live) {
      const double *n = a.n + 3 * (size_t)(a.place ? a.place[p] : p);
      n0 = (float)n[0];
      n1 = (float)n[1];
      n2 = (float)n[2];
      Un = (float)(a.ca * n[0] + a.sa * n[1]);
    }
    const int pb = p0 + pl;
    const bool live_b = pb < a.P;
    // row of component rc % 5 of frame r0 + rc / 5 (rows outside the record are
    // copied from its ends and not used)
    auto src_row = [&](int r0, int rc) -> size_t {
      return (size_t)min(max(r0 + rc / 5, 0), a.nt - 1) * 5 + rc % 5;
    };
    // copy field rows [r0, r0 + n) of the group into raw (n <= C)
    auto issue = [&](int r0, int n) {
      if (vec) {
        for (int e = tid; e < n * 5 * (NP / 4); e += kIntThreads) {
          const int q4 = e % (NP / 4), rc = e / (NP / 4);  // rc = row * 5 + component
          const int pq = p0 + 4 * q4;
          if (pq < a.P)
            cp_async16(raw + rc * NP + 4 * q4, a.fields + src_row(r0, rc) * a.P + pq);
          else
            *reinterpret_cast<float4 *>(raw + rc * NP + 4 * q4) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      } else {
        const int po = live ? p : 0;
        for (int rc = tid / NP; rc < n * 5; rc += kIntThreads / NP)
          cp_async4(raw + rc * NP + pa, a.fields + src_row(r0, rc) * a.P + po, live);
      }
    };
    // integrands of the n rows in raw into window rows [w0, w0 + n)
    auto integrands = [&](int w0, int n) {
      for (int r = tid / NP; r < n; r += kIntThreads / NP) {
        const float *f = raw + r * 5 * NP + pa;
        const float rho_ = f[0], u0v = f[NP], u1 = f[2 * NP], u2 = f[3 * NP], pp = f[4 * NP];
        const float un = u0v * n0 + u1 * n1 + u2 * n2;
        const float r1 = 1.f + rho_;
        const float utn = Un + un;
        float4 q;
        q.x = rho_ * Un + r1 * un;             // Qn   (Eq. Qn_New_nd)
        q.y = pp * n0 + r1 * u0v * utn;        // L_1  (Eq. Li_New_nd)
        q.z = pp * n1 + r1 * u1 * utn;
        q.w = pp * n2 + r1 * u2 * utn;
        *reinterpret_cast<float4 *>(sb + (size_t)(w0 + r) * kIntRow + pa * 4) = q;
      }
    };
    float *const xp = a.X + ((size_t)(live_b ? (a.place ? a.place[pb] : pb) : 0) * a.x_ld) * kSer + 2 * qi;
    // window of block b (first sample c0): samples c0 - H - 2 .. c0 + C + H;
    // load its first C rows, then the rest, so that later blocks only add C
    {
      const int lo = b0 * C - 1 - H - 2;
      __syncthreads();  // the previous unit is done with raw and sb
      issue(lo, C);
      cp_async_wait_all();
      __syncthreads();
      integrands(0, C);
      __syncthreads();
      issue(lo + C, kIntKeep);
      cp_async_wait_all();
      __syncthreads();
      integrands(C, kIntKeep);
      __syncthreads();
    }
    for (int b = b0; b < b1; ++b) {
      const int c0 = b * C - 1;  // first sample: row b C holds it
      const bool more = b + 1 < b1;
      const bool edge = c0 < 0 || c0 + C + H >= a.nt - 1;
      // rows of the next window, in flight meanwhile (a record end keeps y in raw)
      if (more && !edge) issue(c0 + C + H + 1, C);
      // ---- phase B: filters of block b ----------------------------------------
      float *const xr = xp + (size_t)(b * C - a.row0) * kSer;
      const float *bc = sb + (size_t)(H + 2) * kIntRow + pl * 4 + qi;
      auto B = [&](int k) -> float { return bc[k * kIntRow]; };  // k relative to c0
      if (edge) {
        edge_block(bc, raw + pl * 4 + qi, xr, c0, a.nt, inv2h, a.row0 + a.x_ld - b * C, live_b);
      } else {
        float y[C + H + 1];
        float yy = 0.f;
        float Bm = B(-2 - H), B0 = B(-1 - H);
#pragma unroll
        for (int k = -1 - H; k <= C + H - 1; ++k) {
          const float Bp = B(k + 1);
          yy = (Bp - 2.f * B0 + Bm) + rho * yy;
          if (k >= -1) y[k + 1] = yy;
          Bm = B0;
          B0 = Bp;
        }
        // integrand F and recursion x at k + 1 and k + 2
        float xx = 0.f, x1 = 0.f, x2 = 0.f, F1 = 0.f, F2 = 0.f;
#pragma unroll
        for (int k = C + H - 1; k >= -1; --k) {
          xx = y[k + 1] + rho * xx;
          if (k <= C) {
            const float F0 = B(k);
            if (k <= C - 2 && live_b)
              *reinterpret_cast<float2 *>(xr + (k + 1) * kSer) =
                  make_float2(fmaf(rho, x2 - xx, F2 - F0) * inv2h, fmaf(rho, x1, F1));
            F2 = F1;
            F1 = F0;
            x2 = x1;
            x1 = xx;
          }
        }
      }
      if (!more) break;
      // ---- slide the window by C rows and add the rows now in raw --------------
      __syncthreads();  // every thread is done reading the window
      if (edge) issue(c0 + C + H + 1, C);
      for (int e = tid; e < kIntKeep * kIntRow / 4; e += kIntThreads)
        reinterpret_cast<float4 *>(sb)[e] = reinterpret_cast<const float4 *>(sb + C * kIntRow)[e];
      cp_async_wait_all();
      __syncthreads();
      integrands(kIntKeep, C);
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 prep of the interior blocks, on the FP64 pipe: a thread owns one
// (panel, integrand) and walks the blocks of a work unit in source time.  Its
// column of the window holds y (the causal recursion, carried on from block to
// block, in place of the integrand), so per sample the integrands are formed
// once, the causal step runs once and the anti-causal one 1.5 times (64 + 34
// rows per 64): about 36 FP64 operations per (panel, sample).  The record ends
// are handled in place.  Field rows arrive 32 at a time, half of a block's ahead
// of the block, so that three CTAs fit an SM and hide each other's chains.
// 32768 panels x 2048 steps: 5.7 ms (6.8 with 64 rows in flight and two CTAs; 8.7
// with a kernel of its own for the record ends; 15.2 by windowed elimination, 142
// operations and 128-byte rows).
// ---------------------------------------------------------------------------
constexpr int kF64H = Prec<double>::halo;
constexpr int kF64Raw = 32;  // field rows in flight
static_assert(kF64H <= kF64Raw, "the rows a unit starts on are issued at once");
constexpr int kF64Rows = kIirChunk + kF64H + 2;  // samples c0 - 1 .. c0 + 64 + H
constexpr int kF64Keep = kF64Rows - kIirChunk;

// Field rows in flight to shared memory: [n rows][5][NP].
template <int NP>
__device__ __forceinline__ void issue_rows_f64(const double *fields, int P, int nt, int p0, int r0,
                                               int n, double *raw, bool vec) {
  const int tid = threadIdx.x;
  // (rows outside the record are copied from its ends and not used)
  auto src_row = [&](int rc) -> size_t {
    return (size_t)min(max(r0 + rc / 5, 0), nt - 1) * 5 + rc % 5;
  };
  if (vec) {  // 16-byte copies of 2 panels
    for (int e = tid; e < n * 5 * (NP / 2); e += kIntThreads) {
      const int q2 = e % (NP / 2), rc = e / (NP / 2);
      const int pq = p0 + 2 * q2;
      if (pq < P)
        cp_async16(raw + rc * NP + 2 * q2, fields + src_row(rc) * P + pq);
      else
        *reinterpret_cast<double2 *>(raw + rc * NP + 2 * q2) = make_double2(0.0, 0.0);
    }
  } else {
    const int pa = tid % NP;
    const bool live = p0 + pa < P;
    for (int rc = tid / NP; rc < n * 5; rc += kIntThreads / NP)
      cp_async8(raw + rc * NP + pa, fields + src_row(rc) * P + (live ? p0 + pa : 0), live);
  }
}

__global__ void __launch_bounds__(kIntThreads) k_prep_f64_int(PrepArgs<double> a, int unit) {
  constexpr int NP = kIntPanels, C = kIirChunk, H = kF64H, R = kF64Rows;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *win = reinterpret_cast<double *>(smem_raw);  // [R][NP][4]
  double *raw = win + R * kIntRow;                     // [kF64Raw][5][NP]
  double *base = raw + kF64Raw * 5 * NP;               // [NP][4]: F0
  const int tid = threadIdx.x;
  const int n_pg = (a.P + NP - 1) / NP;
  const int n_us = (a.c_hi - a.c_lo + unit - 1) / unit;
  const long n_units = (long)n_pg * n_us;
  const int pa = tid % NP;               // integrand phase: panel, rows tid / NP + 4 u
  const int qi = tid & 3, pl = tid >> 2; // filter phase: integrand, panel
  // What is filtered is F - F0, F0 the integrand of the unit's first sample: the
  // differences then round with the changes of F, not with its mean (see above).
  // Coefficients are F0 + kGain x, their differences kGain times those of x.
  constexpr double kGain = -6.0 * kRho, kUngain = 1.0 / kGain;
  const double inv2h = 0.5 / a.dt, g2h = kGain * inv2h;
  const bool vec = (a.P & 1) == 0 && ((size_t)a.fields & 15) == 0;
  for (long u = blockIdx.x; u < n_units; u += gridDim.x) {
    const int p0 = (int)(u % n_pg) * NP;
    const int b0 = a.c_lo + (int)(u / n_pg) * unit;
    const int b1 = min(a.c_hi, b0 + unit);
    const int p = p0 + pa, pb = p0 + pl;
    double n0 = 0, n1 = 0, n2 = 0, Un = 0;
    if (p < a.P) {
      const double *n = a.n + 3 * (size_t)(a.place ? a.place[p] : p);
      n0 = n[0];
      n1 = n[1];
      n2 = n[2];
      Un = a.ca * n0 + a.sa * n1;
    }
    const bool live_b = pb < a.P;
    double *const xp =
        a.X + ((size_t)(live_b ? (a.place ? a.place[pb] : pb) : 0) * a.x_ld) * kSer + 2 * qi;
    double *const col = win + pl * 4 + qi;
    // integrands, less F0, of the n rows in raw into window rows [w0, w0 + n)
    double q0[4] = {0.0, 0.0, 0.0, 0.0};  // F0 of this thread's panel (integrand phase)
    auto form = [&](int r, double (&q)[4]) {
      const double *f = raw + r * 5 * NP + pa;
      const double rho_ = f[0], u0 = f[NP], u1 = f[2 * NP], u2 = f[3 * NP], pp = f[4 * NP];
      const double un = u0 * n0 + u1 * n1 + u2 * n2;
      const double r1 = 1.0 + rho_;
      const double t = r1 * (Un + un);
      q[0] = fma(rho_, Un, fma(r1, un, -q0[0]));  // Qn
      q[1] = fma(pp, n0, fma(u0, t, -q0[1]));     // L_1
      q[2] = fma(pp, n1, fma(u1, t, -q0[2]));
      q[3] = fma(pp, n2, fma(u2, t, -q0[3]));
    };
    auto integrands = [&](int w0, int n) {
      for (int r = tid / NP; r < n; r += kIntThreads / NP) {
        double q[4];
        form(r, q);
        double *w = win + (w0 + r) * kIntRow + pa * 4;
        *reinterpret_cast<double2 *>(w) = make_double2(q[0], q[1]);
        *reinterpret_cast<double2 *>(w + 2) = make_double2(q[2], q[3]);
      }
    };
    auto issue = [&](int sample, int n) {
      issue_rows_f64<NP>(a.fields, a.P, a.nt, p0, sample, n, raw, vec);
    };
    // integrands of n samples from `sample` on into window rows from w0 on; the
    // first min(n, kF64Raw) are in flight already (`first`: the unit's first rows)
    auto fill = [&](int sample, int w0, int n, bool first = false) {
      for (int r = 0; r < n; r += kF64Raw) {
        const int m = min(kF64Raw, n - r);
        if (r > 0) issue(sample + r, m);
        cp_async_wait_all();
        __syncthreads();
        if (first && r == 0) {
          double q[4];
          form(0, q);
          for (int c = 0; c < 4; ++c) {
            q0[c] = q[c];
            if (tid < NP) base[4 * pa + c] = q[c];
          }
        }
        integrands(w0 + r, m);
        __syncthreads();
      }
    };
    const int lo = b0 * C - 2;  // sample c0 - 1 of the first block
    const int N = a.nt;
    double yy = 0.0;
    double f1 = 0.0, f2 = 0.0, f3 = 0.0;  // F - F0 at the last three samples passed
    // causal recursion over window rows [r0, R), whose row r holds sample s0 + r;
    // it stops being used at sample N - 1
    auto causal = [&](int r0, int s0) {
      if (s0 + R <= N) {
#pragma unroll 8
        for (int r = r0; r < R; ++r) {
          yy = fma(kRho, yy, col[r * kIntRow]);
          col[r * kIntRow] = yy;
        }
        f1 = fma(-kRho, col[(R - 2) * kIntRow], col[(R - 1) * kIntRow]);
        f2 = fma(-kRho, col[(R - 3) * kIntRow], col[(R - 2) * kIntRow]);
        f3 = fma(-kRho, col[(R - 4) * kIntRow], col[(R - 3) * kIntRow]);
      } else {
        for (int r = r0; r < R && s0 + r < N; ++r) {
          f3 = f2;
          f2 = f1;
          f1 = col[r * kIntRow];
          yy = fma(kRho, yy, f1);
          col[r * kIntRow] = yy;
        }
      }
    };
    double e0 = 0.0, D0 = 0.0;  // F - F0 and the one-sided derivative at sample 0
    __syncthreads();  // the previous unit is done with raw and win
    if (b0 > 0) {
      issue(lo - H, H);
      fill(lo - H, 0, H, true);  // the samples the causal recursion starts on
      for (int r = 0; r < H; ++r) {
        f3 = f2;
        f2 = f1;
        f1 = col[r * kIntRow];
        yy = fma(kRho, yy, f1);
      }
      __syncthreads();
    }
    issue(lo, kF64Raw);
    fill(lo, 0, R, b0 == 0);
    const double Fb = base[pl * 4 + qi];
    if (b0 > 0) {
      causal(0, lo);
    } else {  // rows 0 and 1 lie before the record; y_0 from the reflected series
      e0 = col[2 * kIntRow];
      D0 = (-3.0 * e0 + 4.0 * col[3 * kIntRow] - col[4 * kIntRow]) * inv2h;
      for (int j = H; j >= 1; --j) yy = kRho * (col[(2 + j) * kIntRow] + yy);
      yy = e0 * ((1.0 + kRho) / (1.0 - kRho)) - yy;
      f1 = e0;
      col[2 * kIntRow] = yy;
      causal(3, lo);
    }
    for (int b = b0; b < b1; ++b) {
      const bool more = b + 1 < b1;
      if (more) issue(b * C - 2 + R, kF64Raw);
      double *const xr = xp + (size_t)(b * C - a.row0) * kSer;
      const int s0 = b * C - 2;  // sample of window row 0
      double xx = 0.0, c1 = 0.0, c2 = 0.0;  // x, and x one and two samples on
      if (b > 0 && s0 + R < N) {
#pragma unroll 14
        for (int r = R - 1; r >= C + 2; --r) xx = fma(kRho, xx, col[r * kIntRow]);
#pragma unroll
        for (int r = C + 1; r >= C; --r) {
          xx = fma(kRho, xx, col[r * kIntRow]);
          c2 = c1;
          c1 = xx;
        }
#pragma unroll 16
        for (int r = C - 1; r >= 0; --r) {  // window row r: sample c0 - 1 + r
          xx = fma(kRho, xx, col[r * kIntRow]);
          if (live_b)
            *reinterpret_cast<double2 *>(xr + r * kSer) =
                make_double2((c2 - xx) * g2h, fma(kGain, c1, Fb));
          c2 = c1;
          c1 = xx;
        }
      } else {
        // a record end: row r of X holds sample s0 + 1 + r
        double pw = 0.0;  // excess of D0 over the central difference, times rho^sample
        if (b == 0) {
          double x1 = 0.0;
          for (int r = H + 3; r >= 3; --r) x1 = fma(kRho, x1, col[r * kIntRow]);
          pw = D0 - (kGain * x1 - e0) * (2.0 * inv2h);
          for (int i = 0; i < H + 4; ++i) pw *= kRho;  // below rounding from sample H + 4 on
        }
        const double ir = 1.0 / kRho;
        // (used where f1 is sample N - 1)
        const double DN = (3.0 * f1 - 4.0 * f2 + f3) * inv2h, xN = kUngain * f1;
        double cr = 0.0, d2 = 0.0;
        for (int r = R - 1; r >= 0; --r) {
          const int sr = s0 + r;
          if (sr > N - 1) continue;
          xx = sr == N - 1 ? xN : fma(kRho, xx, col[r * kIntRow]);
          if (sr == N - 2)
            cr = DN - (c1 - xx) * (2.0 * g2h);
          else if (sr > N - 3 - (H + 4))  // below rounding further on
            cr *= kRho;
          else
            cr = 0.0;
          const int se = sr + 1;  // the sample now complete, in X row r
          double d = (c2 - xx) * g2h;
          if (cr != 0.0) d += cr;
          if (b == 0 && se < H + 4) {
            pw *= ir;
            d += pw;
          }
          if (r < C && live_b && se <= N - 2) {
            double *row = xr + r * kSer;
            const double v = fma(kGain, c1, Fb);
            if (se > 0) *reinterpret_cast<double2 *>(row) = make_double2(d, v);
            if (se == 0) {  // sample 0 and the ghost before it
              *reinterpret_cast<double2 *>(row) = make_double2(D0, v);
              *reinterpret_cast<double2 *>(row - kSer) =
                  make_double2(2.0 * D0 - d2, fma(kGain, 2.0 * c1 - c2, Fb));
            }
            if (se == N - 2) {  // the last sample, the ghost after it and a zero row
              const int room = a.row0 + a.x_ld - b * C - r;  // rows of X from this one on
              if (room > 1) *reinterpret_cast<double2 *>(row + kSer) = make_double2(DN, f1 + Fb);
              if (room > 2)
                *reinterpret_cast<double2 *>(row + 2 * kSer) =
                    make_double2(2.0 * DN - d, fma(kGain, 2.0 * xN - c1, Fb));
              if (room > 3) *reinterpret_cast<double2 *>(row + 3 * kSer) = make_double2(0.0, 0.0);
            }
          }
          d2 = d;
          c2 = c1;
          c1 = xx;
        }
      }
      if (!more) break;
      // slide the thread's column by C rows, then add the rows now in raw
      for (int r = 0; r < kF64Keep; ++r) col[r * kIntRow] = col[(r + C) * kIntRow];
      fill(s0 + R, kF64Keep, C);
      causal(kF64Keep, s0 + C);
    }
  }
}

// Prep of records shorter than H + 3 samples (compact code): thread (series,
// half, panel) filters 32 rows of one of the eight series, r = D2 F on the
// odd-periodic extension of any number of periods; the eight threads of a panel
// write one X row per step.
template <typename T>
__global__ void __launch_bounds__(kIirThreads, sizeof(T) == 4 ? 6 : 2) k_prep_iir(PrepArgs<T> a) {
  constexpr int NP = kIirPanels, H = Prec<T>::halo, J = kIirJ, ROWS = iir_rows<T>();
  constexpr T rho = (T)kRho;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // staged integrands, two copies [rows][4 (stride kIirQ)][NP]: the second
  // with its columns rotated by two, read by the threads of the upper half
  // block (rows 32 apart would otherwise share a bank)
  T *sb = reinterpret_cast<T *>(smem_raw);
  T *sb2 = sb + ROWS * kIirRow;
  const int tid = threadIdx.x;
  const int n_blk = a.c_hi - a.c_lo;  // 1D grid: block fastest, then panel tiles
  const int blk = a.c_lo + (int)(blockIdx.x % n_blk);
  const int c0 = blk * kIirChunk - 1;  // first sample
  const int p0 = (int)(blockIdx.x / n_blk) * NP;
  const int N = a.nt;
  // phase B thread: series s, half h (samples c0 + 32 h ..), panel pl
  const int s = tid & 7;
  const int h = (tid >> 3) & 1;
  const int pl = tid >> 4;
  const int pb = p0 + pl;
  const bool live_b = pb < a.P;
  T *xr = a.X + ((size_t)(live_b ? (a.place ? a.place[pb] : pb) : 0) * a.x_ld +
                 (blk * kIirChunk - a.row0) + J * h) * kSer + s;
  auto put = [&](int t, T v) {
    if (live_b) xr[t * kSer] = v;
  };
  if (c0 > N) {  // past the record's ghost sample
    for (int t = 0; t < J; ++t) put(t, T(0));
    return;
  }
  // staged integrand rows: the tile's filter reach plus FD neighbours, and
  // for a tile at the record end the rows its window folds back onto
  const int reach_lo = c0 - H - 3, reach_hi = c0 + kIirChunk + H + 3;
  const int lo = max(0, min(reach_lo, 2 * (N - 1) - reach_hi));
  const int hi = min(N, reach_hi);
  // ---- phase A: integrands ------------------------------------------------
  {
    const int pl_a = tid % NP;
    const int p = p0 + pl_a;
    const bool live = p < a.P;
    T n0 = 0, n1 = 0, n2 = 0, Un = 0;
    if (live) {
      const double *n = a.n + 3 * (size_t)(a.place ? a.place[p] : p);
      n0 = (T)n[0];
      n1 = (T)n[1];
      n2 = (T)n[2];
      Un = (T)(a.ca * n[0] + a.sa * n[1]);
    }
    // all field loads of this thread's rows first, then the integrands
    constexpr int RS = kIirThreads / NP;               // row stride between passes
    constexpr int RPT = (ROWS + RS - 1) / RS;          // passes
    T fv[RPT][5];
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      const int i = lo + tid / NP + u * RS;
      const bool ok = live && i < hi;
      const T *b = a.fields + (size_t)(ok ? i : 0) * 5 * a.P + (live ? p : 0);
#pragma unroll
      for (int c = 0; c < 5; ++c) fv[u][c] = ok ? b[(size_t)c * a.P] : T(0);
    }
    const int rot = (pl_a + 2) & (NP - 1);
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      const int i = lo + tid / NP + u * RS;
      if (i >= hi) break;
      const T rho_ = fv[u][0], u0 = fv[u][1], u1 = fv[u][2], u2 = fv[u][3], pp = fv[u][4];
      const T un = u0 * n0 + u1 * n1 + u2 * n2;
      const T r1 = T(1) + rho_;
      const T utn = Un + un;
      const T q0 = rho_ * Un + r1 * un;            // Qn   (Eq. Qn_New_nd)
      const T q1 = pp * n0 + r1 * u0 * utn;        // L_1  (Eq. Li_New_nd)
      const T q2 = pp * n1 + r1 * u1 * utn;
      const T q3 = pp * n2 + r1 * u2 * utn;
      T *row = sb + (size_t)(i - lo) * kIirRow;
      T *row2 = sb2 + (size_t)(i - lo) * kIirRow;
      row[pl_a] = q0;
      row[kIirQ + pl_a] = q1;
      row[2 * kIirQ + pl_a] = q2;
      row[3 * kIirQ + pl_a] = q3;
      row2[rot] = q0;
      row2[kIirQ + rot] = q1;
      row2[2 * kIirQ + rot] = q2;
      row2[3 * kIirQ + rot] = q3;
    }
  }
  __syncthreads();
  // ---- phase B: coefficients, stored straight to X ---------------------------
  const int ks = c0 + J * h;
  const bool deriv = (s & 1) == 0;
  const int qi = s >> 1;
  const T *col = (h ? sb2 + ((pl + 2) & (NP - 1)) : sb + pl) + qi * kIirQ -
                 (ptrdiff_t)lo * kIirRow;  // B(i) = col[i * kIirRow]
  const T inv2h = (T)(0.5 / a.dt);
  auto B = [&](int i) -> T { return col[(ptrdiff_t)i * kIirRow]; };
  // Series at frame i: one-sided derivatives at the first and last frame.
  auto F = [&](int i) -> T {
    if (!deriv) return B(i);
    if (i == 0) return (T(-3) * B(0) + T(4) * B(1) - B(2)) * inv2h;
    if (i == N - 1) return (T(3) * B(N - 1) - T(4) * B(N - 2) + B(N - 3)) * inv2h;
    return (B(i + 1) - B(i - 1)) * inv2h;
  };
  const int L2 = 2 * (N - 1);
  auto r_at = [&](int kk) -> T {
    int km = kk % L2;
    if (km < 0) km += L2;
    T sg = T(1);
    if (km >= N - 1) {
      km = L2 - km;
      sg = T(-1);
    }
    if (km == 0 || km == N - 1) return T(0);
    return sg * (F(km + 1) - T(2) * F(km) + F(km - 1));
  };
  T ye[J + H];
  T yy = T(0);
#pragma unroll 1
  for (int t = 0; t < J + 2 * H; ++t) {
    yy = r_at(ks - H + t) + rho * yy;
    if (t >= H) ye[t - H] = yy;
  }
  T xx = T(0);
#pragma unroll 1
  for (int t = J + H - 1; t >= 0; --t) {
    xx = ye[t] + rho * xx;
    if (t >= J) continue;
    const int k = ks + t;
    T v = T(0);
    if (k < 0)
      v = T(2) * F(0) - F(-k) + rho * xx;
    else if (k < N)
      v = F(k) + rho * xx;
    else if (k == N)
      v = T(2) * F(N - 1) - F(N - 2) + rho * xx;
    put(t, v);
  }
}

// ---------------------------------------------------------------------------
// Adjoint of the prep followed by the Jacobian of the integrands.  With S the
// (symmetric) map from a series to its coefficients and D the time difference,
// the gradient of an integrand is S Xbar_v + D^T S Xbar_d (Xbar_v, Xbar_d: its
// value and derivative series' rows of Xbar), and the four integrand gradients
// of a (panel, sample) map to the five field gradients.
//
// S and D commute away from the ends, so one filter per integrand on
//   w = Xbar_v + D^T Xbar_d,
// in the form -6 rho (1 - rho z)^-1 (1 - rho z^-1)^-1.  The ends transpose the
// forward's: with a0 = sum rho^k Xbar_d,k (the sum that D_0 - d_0 multiplies
// there), the two samples of d_0 see Xbar_d,0 - a0 instead of Xbar_d,0, a0 goes
// through D_0's one-sided weights straight into the gradient, the recursions
// run on the odd extension of w (zero at the end samples), and the end sample's
// own gradient is w minus the moment next to it; likewise aN.
//
// A thread owns one (panel, integrand) and walks the blocks of a work unit: its
// column of the window holds the causal recursion's y (carried on from block
// to block), then the integrand gradients, in place; the Jacobian phase takes
// (sample, panel) pairs, so field reads and gradient writes are coalesced.
// Each thread's Xbar rows of the next 16 samples are in flight while it works on
// these, and half of the block's fields are copied to shared memory behind the
// anti-causal pass, the other half behind the first half's gradients (six CTAs
// an SM instead of five, three instead of two in FP64).  Bound by HBM and the
// latency of the chains together.  16384 panels x 1024 steps: 0.23 ms (0.36 with
// the record ends in a kernel of their own that filtered all eight series, and
// all the fields at once); FP64, 5151 x 701: 0.40 ms (0.68).
// ---------------------------------------------------------------------------
template <typename T> struct Pair;
template <> struct Pair<float> { using V = float2; };
template <> struct Pair<double> { using V = double2; };

// Field gradients from the integrand gradients (qb: Qn, lb: L_c) of a
// (panel, sample) with fields f = rho', u' and normal n.
template <typename T>
__device__ __forceinline__ void put_grad(T *g, size_t P, const T *f, T qb, T lb0, T lb1, T lb2,
                                         T n0, T n1, T n2, T Un) {
  const T un = f[1] * n0 + f[2] * n1 + f[3] * n2;
  const T utn = Un + un;   // total u . n
  const T r1 = T(1) + f[0];
  const T lu = lb0 * f[1] + lb1 * f[2] + lb2 * f[3];
  const T t = qb + lu;
  g[0] = t * utn;                              // d/drho'
  g[P] = r1 * (t * n0 + lb0 * utn);            // d/du'_1
  g[2 * P] = r1 * (t * n1 + lb1 * utn);
  g[3 * P] = r1 * (t * n2 + lb2 * utn);
  g[4 * P] = lb0 * n0 + lb1 * n1 + lb2 * n2;   // d/dp' (dL_c/dp' = n_c)
}

constexpr int kAdjFieldRows = 32;  // field rows of a block staged at a time

template <typename T>
__global__ void __launch_bounds__(kIntThreads, sizeof(T) == 4 ? 6 : 2)
    k_prep_adj_int(PrepAdjArgs<T> a, int n_blk, int unit) {
  constexpr int NP = kIntPanels, C = kIirChunk, H = Prec<T>::halo, R = C + H;
  constexpr int BT = 16;  // rows in flight per thread
  constexpr int FR = kAdjFieldRows;
  static_assert(C % BT == 0 && H % BT == 0 && C % FR == 0, "row batches");
  using V = typename Pair<T>::V;
  constexpr T rho = (T)kRho, six = (T)(-6.0 * kRho);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *win = reinterpret_cast<T *>(smem_raw);  // [R][NP][4]: samples c0 .. c0 + R - 1
  T *fld = win + R * kIntRow;                // [FR][4][NP]: rho', u' of the block
  const int tid = threadIdx.x;
  const int n_pg = (a.P + NP - 1) / NP;
  const int n_us = (n_blk + unit - 1) / unit;
  const long n_units = (long)n_pg * n_us;
  const int N = a.nt;
  const int pa = tid % NP;               // Jacobian phase: panel, rows tid / NP + 4 u
  const int qi = tid & 3, pl = tid >> 2; // filter phase: integrand, panel
  const T inv2h = (T)(0.5 / a.dt);
  const size_t P = a.P;
  for (long u = blockIdx.x; u < n_units; u += gridDim.x) {
    const int p0 = (int)(u % n_pg) * NP;
    const int b0 = (int)(u / n_pg) * unit;
    const int b1 = min(n_blk, b0 + unit);
    const int p = p0 + pa, pb = min(p0 + pl, a.P - 1);
    const bool live = p < a.P;
    T n0 = 0, n1 = 0, n2 = 0, Un = 0;
    if (live) {
      const double *n = a.n + 3 * (size_t)(a.place ? a.place[p] : p);
      n0 = (T)n[0];
      n1 = (T)n[1];
      n2 = (T)n[2];
      Un = (T)(a.ca * n[0] + a.sa * n[1]);
    }
    // (derivative, value) pair of sample k
    const T *const xb = a.Xbar + (size_t)(a.place ? a.place[pb] : pb) * a.xb_ld * kSer + 2 * qi;
    auto X = [&](int k) -> V { return __ldg(reinterpret_cast<const V *>(xb + (size_t)k * kSer)); };
    T *const col = win + pl * 4 + qi;
    T yy = T(0);
    int k;               // next sample of the causal recursion
    const int k_last = min((b1 - 1) * C + R, N - 1);  // last sample it reads
    V cur;
    T dm;                // derivative gradient one sample back
    T a0 = T(0), w0 = T(0);             // the start's sum, w of sample 0
    T aN = T(0), wN = T(0), yN = T(0);  // the end's sum, w of the last sample, y before it
    if (b0 > 0) {
      k = b0 * C - H;
      cur = X(k);
      dm = X(k - 1).x;
    } else {  // exact start: y of sample 0 on the odd extension of w
      k = 0;
      T e = T(0);
      V x1 = V{}, x2 = V{};
#pragma unroll
      for (int j = H + 1; j >= 0; --j) {
        const V x = X(j);
        a0 = fma(rho, a0, x.x);
        if (j >= 1 && j < H) e = rho * (e + fma(x.x - x2.x, inv2h, x1.y));
        if (j > 0) {
          x2 = x1;
          x1 = x;
        } else {
          const T d0 = T(2) * (x.x - a0);  // what sample 1 sees as the one before it
          e = rho * (e + fma(d0 - x2.x, inv2h, x1.y));
          w0 = fma(-inv2h, x1.x + d0, x.y);
          cur.x = d0;
          cur.y = -e;
          dm = x1.x;  // no difference: the first step gives y_0 = -e itself
        }
      }
    }
    if (k_last == N - 1) {
#pragma unroll
      for (int j = H + 2; j >= 0; --j) aN = fma(rho, aN, X(N - 1 - j).x);
    }
    V nx[BT];            // the next batch, in flight
    auto fetch = [&]() {
#pragma unroll
      for (int i = 0; i < BT; ++i) nx[i] = X(min(k + 1 + i, k_last));
    };
    // BT samples of the recursion; y of each to col (row `w` on) unless w < 0
    auto causal = [&](int w) {
      V x[BT];
#pragma unroll
      for (int i = 0; i < BT; ++i) x[i] = nx[i];
      const int k0 = k;
      k += BT;
      fetch();
      if (k0 + BT < N - 1) {
#pragma unroll
        for (int i = 0; i < BT; ++i) {
          yy = fma(rho, yy, fma(dm - x[i].x, inv2h, cur.y));
          if (w >= 0) col[(w + i) * kIntRow] = yy;
          dm = cur.x;
          cur = x[i];
        }
      } else {  // x of sample N - 1 is zero: so is y from there on
#pragma unroll
        for (int i = 0; i < BT; ++i) {
          const bool last = k0 + i == N - 2;
          const T xn = last ? T(2) * (x[i].x - aN) : x[i].x;
          yy = k0 + i <= N - 2 ? fma(rho, yy, fma(dm - xn, inv2h, cur.y)) : T(0);
          if (last) {
            yN = yy;
            wN = fma(inv2h, cur.x + xn, x[i].y);
          }
          if (w >= 0) col[(w + i) * kIntRow] = yy;
          dm = cur.x;
          cur = x[i];
        }
      }
    };
    fetch();
    // fields of FR samples from row r0 of a block on, in flight to shared memory
    // (read by the Jacobian phase)
    auto issue_fields = [&](int b, int r0) {
      const T *f0 = a.fields + (live ? p : 0);
#pragma unroll 4
      for (int rc = tid / NP; rc < 4 * FR; rc += kIntThreads / NP) {
        const T *src = f0 + ((size_t)min(b * C + r0 + (rc >> 2), N - 1) * 5 + (rc & 3)) * P;
        if constexpr (sizeof(T) == 4)
          cp_async4(fld + rc * NP + pa, src, live);
        else
          cp_async8(fld + rc * NP + pa, src, live);
      }
    };
    __syncthreads();  // the previous unit's Jacobian phase is done with win
    if (b0 > 0)
      for (int i = 0; i < H; i += BT) causal(-1);
    for (int i = 0; i < R; i += BT) causal(i);
    for (int b = b0; b < b1; ++b) {
      issue_fields(b, 0);
      T xx = T(0);
#pragma unroll 16
      for (int r = R - 1; r >= C; --r) xx = fma(rho, xx, col[r * kIntRow]);
#pragma unroll 16
      for (int r = C - 1; r >= 0; --r) {
        xx = fma(rho, xx, col[r * kIntRow]);
        col[r * kIntRow] = six * xx;
      }
      if (b == 0) {
        col[0] = w0 - col[kIntRow] * T(1.0 / 6.0) - T(3) * inv2h * a0;
        col[kIntRow] += T(4) * inv2h * a0;
        col[2 * kIntRow] -= inv2h * a0;
      }
      const int rN = N - 1 - b * C;  // row of the last sample
      if (rN < C + 2) {
        if (rN < C) col[rN * kIntRow] = wN + rho * yN + T(3) * inv2h * aN;
        if (rN >= 1 && rN <= C) col[(rN - 1) * kIntRow] -= T(4) * inv2h * aN;
        if (rN >= 2) col[(rN - 2) * kIntRow] += inv2h * aN;
      }
      for (int r0 = 0; r0 < C; r0 += FR) {
        if (r0 > 0) {
          __syncthreads();  // every thread is done with the fields before these
          issue_fields(b, r0);
        }
        cp_async_wait_all();
        __syncthreads();
        if (live) {
#pragma unroll 4
          for (int r = r0 + tid / NP; r < min(r0 + FR, N - b * C); r += kIntThreads / NP) {
            const T *f = fld + (r - r0) * 4 * NP + pa;
            const T fv[4] = {f[0], f[NP], f[2 * NP], f[3 * NP]};
            const T *q = win + r * kIntRow + pa * 4;
            put_grad<T>(a.grad_fields + (size_t)(b * C + r) * 5 * P + p, P, fv, q[0], q[1], q[2],
                        q[3], n0, n1, n2, Un);
          }
        }
      }
      if (b + 1 == b1) break;
      __syncthreads();  // every thread is done with the gradients
      for (int r = 0; r < H; ++r) col[r * kIntRow] = col[(r + C) * kIntRow];
      for (int i = 0; i < C; i += BT) causal(H + i);
    }
  }
}

// Records shorter than H + 3 samples: all eight series, S with the natural ends as
//   G_s = Xbar_s - D2^T A Xbar_s,
// A = tridiag(1, 4, 1)^-1 on rows 1 .. N - 2 by the same pair of recursions on
// the odd-periodic extension of Xbar_s (zero at 0 and N - 1), then D^T with its
// one-sided end rows.  Tile: 8 panels x 64 samples; thread (half, panel,
// series) filters samples [32 half - 3, 32 half + 35) of the tile; the
// per-sample gradients meet in shared memory and the Jacobian phase writes
// per (sample, panel).
//
// Every CTA first stages (cp.async) its Xbar rows c0 - 3 - H .. c0 + 64 + H + 2
// as the odd-periodic extension itself (rows mapped by reflection, zero at 0
// and N - 1, negated where reflected), and rows c0 - 2 .. c0 + 65 as they are
// (zero outside the record), so every thread runs the same unrolled filter.
// Per panel the rows are 8 values, the panel stride padded to 8 or 24 mod 32
// words so that the 4 panels x 8 series one warp reads in a step spread over
// the banks.  The per-sample gradients reuse the staging space once every
// thread has filtered.
constexpr int kAdjZ = kIirJ + 6;             // A Xbar values a thread keeps
constexpr int kAdjVRows = kIirChunk + 4;     // c0 - 2 .. c0 + C + 1
constexpr int kAdjVPS = kAdjVRows * 8 + 8;   // panel strides (values)
template <typename T>
constexpr int adj_mps() { return iir_rows<T>() * 8 + 8; }
static_assert((adj_mps<float>() % 32 == 8 || adj_mps<float>() % 32 == 24) &&
                  (kAdjVPS % 32 == 8 || kAdjVPS % 32 == 24),
              "bank spread of the staged rows");
static_assert(kIirPanels * adj_mps<float>() >= kIirChunk * 8 * kIirPanels,
              "gradients fit the staging");

__device__ __forceinline__ void cp_async16_zfill(void *dst, const void *src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = ok ? 16 : 0;  // zero fill
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n)
               : "memory");
}

// o[t] is the contribution of sample ks + t, from z = A Xbar (index 0 is sample
// ks - 3) and xv[8 t], Xbar of sample ks - 2 + t (zero outside the record),
// with the natural ends (no moment at 0 and N - 1), D^T's one-sided end rows,
// and zero past N - 1.  ks is a multiple of 32, so the start end can only
// enter as sample 0 = ks; the far end's G is picked out of the unrolled G by a
// select.
template <typename T>
__device__ __forceinline__ void adj_values_ends(T (&z)[kAdjZ], const T *xv, bool deriv, int ks,
                                                int N, T inv2h, T (&o)[kIirJ]) {
  constexpr int J = kIirJ;
#pragma unroll
  for (int t = 0; t < kAdjZ; ++t) {
    const int i = ks - 3 + t;
    if (i <= 0 || i >= N - 1) z[t] = T(0);
  }
  T G[J + 4];  // samples ks - 2 .. ks + J + 1
#pragma unroll
  for (int t = 0; t < J + 4; ++t) G[t] = xv[8 * t] - (z[t] - T(2) * z[t + 1] + z[t + 2]);
  T gN = T(0);  // G at sample N - 1, when it lies in the thread's range
#pragma unroll
  for (int t = 0; t < J + 4; ++t)
    if (ks - 2 + t == N - 1) gN = G[t];
#pragma unroll
  for (int t = 0; t < J; ++t) {
    const int i = ks + t;
    T c;
    if (!deriv) {
      c = G[t + 2];
    } else {
      c = T(0);
      if (i - 1 >= 1 && i - 1 <= N - 2) c += G[t + 1] * inv2h;
      if (i + 1 >= 1 && i + 1 <= N - 2) c -= G[t + 3] * inv2h;
      if (i <= 2) c += (i == 0 ? T(-3) : (i == 1 ? T(4) : T(-1))) * inv2h * G[2];  // here ks = 0
      if (i >= N - 3) c += (i == N - 1 ? T(3) : (i == N - 2 ? T(-4) : T(1))) * inv2h * gN;
    }
    o[t] = i < N ? c : T(0);
  }
}

// 1D grid, block fastest.
template <typename T>
__global__ void __launch_bounds__(kIirThreads, sizeof(T) == 4 ? 5 : 2)
    k_prep_adj_iir(PrepAdjArgs<T> a) {
  constexpr int NP = kIirPanels, H = Prec<T>::halo, J = kIirJ;
  constexpr int NR = kAdjZ + 2 * H;  // samples each thread filters
  constexpr int MR = iir_rows<T>(), MPS = adj_mps<T>();
  constexpr int PC = kSer * sizeof(T) / 16, VP = 16 / sizeof(T);  // 16-byte pieces of a row
  constexpr T rho = (T)kRho;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *sm = reinterpret_cast<T *>(smem_raw);  // [NP][MPS] (later the gradients), [NP][kAdjVPS]
  T *sv = sm + NP * MPS;
  T *cs = sm;
  const int tid = threadIdx.x;
  const int n_ct = (a.nt + kIirChunk - 1) / kIirChunk;
  const int c0 = (int)(blockIdx.x % n_ct) * kIirChunk;
  const int p0 = (int)(blockIdx.x / n_ct) * NP;
  const int N = a.nt;
  const int L2 = 2 * (N - 1);
  // sample k of the odd-periodic extension as a row of the record: km in
  // [0, N - 1], reflected when the extension's sign is negative
  auto ext_row = [&](int k, bool &reflected) -> int {
    int km = k % L2;
    if (km < 0) km += L2;
    reflected = km > N - 1;
    return reflected ? L2 - km : km;
  };
  auto panel = [&](int pl) -> const T * {
    const int q = min(p0 + pl, a.P - 1);
    return a.Xbar + (size_t)(a.place ? a.place[q] : q) * a.xb_ld * kSer;
  };
  for (int pl = 0; pl < NP; ++pl) {
    const T *xp = panel(pl);
    for (int rq = tid; rq < PC * MR; rq += kIirThreads) {
      bool refl;
      const int km = ext_row(c0 - 3 - H + rq / PC, refl);
      cp_async16_zfill(sm + pl * MPS + VP * rq, xp + (size_t)km * kSer + VP * (rq % PC),
                       km != 0 && km != N - 1);
    }
    for (int rq = tid; rq < PC * kAdjVRows; rq += kIirThreads) {
      const int i = c0 - 2 + rq / PC;
      const bool in = i >= 0 && i < N;
      cp_async16_zfill(sv + pl * kAdjVPS + VP * rq, xp + (size_t)(in ? i : 0) * kSer + VP * (rq % PC),
                       in);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // negate the reflected rows
  for (int e3 = tid; e3 < NP * MR; e3 += kIirThreads) {
    const int pl = e3 / MR, r = e3 - pl * MR;
    bool refl;
    ext_row(c0 - 3 - H + r, refl);
    if (refl) {
      T *q = sm + pl * MPS + 8 * r;
      for (int v = 0; v < kSer; ++v) q[v] = -q[v];
    }
  }
  __syncthreads();
  {
    const int s = tid & 7;
    const int pl = (tid >> 3) % NP;
    const int h = tid / (8 * NP);
    const int ks = c0 + J * h;
    const bool deriv = (s & 1) == 0;
    const T inv2h = (T)(0.5 / a.dt);
    // Xbar slot s of sample ks - 3 - H + t: staged row ks - c0 + t
    const T *xm = sm + pl * MPS + (ks - c0) * 8 + s;
    T y[kAdjZ + H];
    T yy = T(0);
#pragma unroll
    for (int t = 0; t < NR; ++t) {
      yy = xm[8 * t] + rho * yy;
      if (t >= H) y[t - H] = yy;
    }
    T xx = T(0);
    T z[kAdjZ];
#pragma unroll
    for (int t = kAdjZ + H - 1; t >= 0; --t) {
      xx = y[t] + rho * xx;
      if (t < kAdjZ) z[t] = -rho * xx;
    }
    T o[J];
    // Xbar slot s of sample ks - 2 + t: staged row ks - c0 + t
    adj_values_ends<T>(z, sv + pl * kAdjVPS + (ks - c0) * 8 + s, deriv, ks, N, inv2h, o);
    __syncthreads();  // every thread is done with the staged rows
    // [sample][panel][series]
    T *out = cs + (size_t)(ks - c0) * 8 * NP + pl * 8 + s;
#pragma unroll
    for (int t = 0; t < J; ++t) out[t * 8 * NP] = o[t];
  }
  __syncthreads();
  // ---- integrand gradients -> field gradients, per (sample, panel) ----------
  // thread: panel tid % NP, samples tid / NP + 16 it; the field loads of all
  // its samples are issued before any of them is used
  {
    constexpr int IT = kIirChunk * NP / kIirThreads;
    constexpr int RS = kIirThreads / NP;  // sample stride
    const int pl = tid % NP, p = p0 + pl;
    if (p < a.P) {
      const double *n = a.n + 3 * (size_t)(a.place ? a.place[p] : p);
      const T n0 = (T)n[0], n1 = (T)n[1], n2 = (T)n[2];
      const T Un = (T)(a.ca * n[0] + a.sa * n[1]);
      const size_t P = a.P;
      T f[IT][4];
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const int i = c0 + tid / NP + RS * it;
        const T *fb = a.fields + (size_t)min(i, N - 1) * 5 * P + p;
#pragma unroll
        for (int q = 0; q < 4; ++q) f[it][q] = fb[q * P];
      }
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const int ir = tid / NP + RS * it;
        if (c0 + ir >= N) continue;
        const T *c = cs + (size_t)ir * 8 * NP + pl * 8;
        put_grad<T>(a.grad_fields + (size_t)(c0 + ir) * 5 * P + p, P, f[it], c[0] + c[1],
                    c[2] + c[3], c[4] + c[5], c[6] + c[7], n0, n1, n2, Un);
      }
    }
  }
}

}  // namespace

// Persistent CTAs of a walking kernel over `blocks` blocks of n_pg panel groups:
// as many as fit the GPU at once, and the blocks of a work unit (at most
// kIntUnit), by the rounds of units each CTA takes times a unit's cost, its
// blocks and `start` blocks' worth of rows to start on (0.68 ms at 32768 panels
// x 2048 steps; 0.71 with the units that fill the GPU twice).  A small problem
// gets one block a unit, so that its blocks run side by side.
template <auto kern>
cudaError_t persistent_grid(size_t smem, double start, long n_pg, int blocks,
                            int *unit, long *grid) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // CTAs that fit the device, looked up once per kernel and device
  constexpr int kMaxDev = 64;
  static std::atomic<int> fits[kMaxDev];
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  int fit = dev < kMaxDev ? fits[dev].load(std::memory_order_relaxed) : 0;
  if (fit == 0) {
    int sms = 0, per_sm = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kIntThreads, smem)) !=
        cudaSuccess)
      return e;
    fit = std::max(per_sm, 1) * sms;
    if (dev < kMaxDev) fits[dev].store(fit, std::memory_order_relaxed);
  }
  double best = 0.0;
  *unit = 0;
  for (int u = 1; u <= kIntUnit && u <= std::max(blocks, 1); ++u) {
    const long units = n_pg * ((blocks + u - 1) / u);
    const double cost = (double)((units + fit - 1) / fit) * (u + start);
    if (*unit == 0 || cost < best) {
      best = cost;
      *unit = u;
    }
  }
  *grid = std::min<long>(n_pg * ((blocks + *unit - 1) / *unit), (long)fit);
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_prep(const PrepArgs<T> &a0, cudaStream_t s) {
  constexpr int C = kIirChunk;
  static_assert(C == kRowBlk && C - 1 >= Prec<T>::halo + 2, "only block 0 reaches before the record");
  PrepArgs<T> a = a0;
  const int n_rb = (int)(x_rows(a.nt) / C);
  if (a.c_hi == 0) {
    a.c_lo = 0;
    a.c_hi = n_rb;
  }
  if (a.c_lo < 0 || a.c_hi > n_rb || a.c_lo >= a.c_hi || a.c_lo * C < a.row0 ||
      a.c_hi * C > a.row0 + a.x_ld)
    return cudaErrorInvalidValue;
  cudaError_t e;
  // the walking kernels' exact starts reach H + 1 samples into the record and
  // take the two ends' corrections apart (rho^(nt - 1) below rounding)
  if (a.nt >= Prec<T>::halo + 3) {
    const long n_pg = (a.P + kIntPanels - 1) / kIntPanels;
    const int n_blk = a.c_hi - a.c_lo;
    long grid = 0;
    int unit = 1;
    if constexpr (sizeof(T) == 4) {
      const size_t smem = ((size_t)kIntRows * kIntRow + (size_t)kIntRaw) * sizeof(T);
      if ((e = persistent_grid<k_prep_iir_int>(smem, 0.6, n_pg, n_blk, &unit, &grid)) !=
          cudaSuccess)
        return e;
      k_prep_iir_int<<<(unsigned)grid, kIntThreads, smem, s>>>(a, unit);
    } else {
      const size_t smem =
          ((size_t)kF64Rows * kIntRow + (size_t)kF64Raw * 5 * kIntPanels + 4 * kIntPanels) * sizeof(T);
      if ((e = persistent_grid<k_prep_f64_int>(smem, 1.0, n_pg, n_blk, &unit, &grid)) !=
          cudaSuccess)
        return e;
      k_prep_f64_int<<<(unsigned)grid, kIntThreads, smem, s>>>(a, unit);
    }
    return cudaGetLastError();
  }
  const size_t smem = (size_t)2 * iir_rows<T>() * kIirRow * sizeof(T);
  e = cudaFuncSetAttribute(k_prep_iir<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long blocks = (long)(a.c_hi - a.c_lo) * ((a.P + kIirPanels - 1) / kIirPanels);
  if (blocks > INT32_MAX) return cudaErrorInvalidValue;
  k_prep_iir<T><<<(unsigned)blocks, kIirThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prep_adjoint(const PrepAdjArgs<T> &a, cudaStream_t s) {
  constexpr int H = Prec<T>::halo, C = kIirChunk;
  const int n_ct = (a.nt + C - 1) / C;
  const long tiles = (a.P + kIirPanels - 1) / kIirPanels;
  if (n_ct <= 0 || tiles <= 0) return cudaSuccess;
  cudaError_t e;
  if (a.nt >= H + 3) {  // as in launch_prep
    const long n_pg = (a.P + kIntPanels - 1) / kIntPanels;
    const size_t smem =
        ((size_t)(C + H) * kIntRow + (size_t)kAdjFieldRows * 4 * kIntPanels) * sizeof(T);
    long grid = 0;
    int unit = 1;
    if ((e = persistent_grid<k_prep_adj_int<T>>(smem, 0.5, n_pg, n_ct, &unit, &grid)) !=
        cudaSuccess)
      return e;
    k_prep_adj_int<T><<<(unsigned)grid, kIntThreads, smem, s>>>(a, n_ct, unit);
    return cudaGetLastError();
  }
  const long ends = (long)n_ct * tiles;
  if (ends > INT32_MAX) return cudaErrorInvalidValue;
  const size_t smem = (size_t)kIirPanels * (adj_mps<T>() + kAdjVPS) * sizeof(T);
  e = cudaFuncSetAttribute(k_prep_adj_iir<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem);
  if (e != cudaSuccess) return e;
  k_prep_adj_iir<T><<<(unsigned)ends, kIirThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template cudaError_t launch_prep<float>(const PrepArgs<float> &, cudaStream_t);
template cudaError_t launch_prep<double>(const PrepArgs<double> &, cudaStream_t);
template cudaError_t launch_prep_adjoint<float>(const PrepAdjArgs<float> &, cudaStream_t);
template cudaError_t launch_prep_adjoint<double>(const PrepAdjArgs<double> &, cudaStream_t);

}  // namespace fwh
