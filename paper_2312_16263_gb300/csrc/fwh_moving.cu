// General moving surface (Sec. II B): the permeable-surface Farassat 1A
// integrals of Eqs. pT and pL for panels that move in a medium at rest, with
// the retarded time of Eq. tau, FP64 throughout.
//
// Unlike the wind-tunnel form, the distance r, the radiation direction r-hat
// and the Mach numbers change with source time, so every (panel, observer)
// has its own source-time signal and its own arrival times: the spline that
// carries a panel's signal onto the observer grid cannot be shared between
// observers.  Three kernels, all bound by the FP64 pipe (2 operations a clock
// and SM), so what they save is operations:
//  * k_mseries, per (panel, run of frames): the observer-independent series Q_n
//    (Eq. Qn), L_i (Eq. Li), the surface Mach vector M = v / c0, their
//    second-order source-time derivatives (Sec. III B), M.M and L.M, one
//    16-value row per frame; each frame's integrands are formed once;
//  * k_mwindow, per observer: the earliest and latest arrival over panels of
//    the first and last frame (the window t_start, t_end and N_o);
//  * k_mscatter, per (observer, panel), a thread each.  Ascending in source
//    time it evaluates, at every frame, the delay Delta (the positive root of
//    |b + w Delta| = c0 Delta, b = x0 + w tau - y) and the bracket g of Eqs.
//    pT + pL, and runs the forward elimination of the natural spline's cubic
//    B-spline coefficients, beta_{i-1} + 4 beta_i + beta_{i+1} = 6 F_i with
//    beta = F at both ends (g and Delta: two scratch columns).  Descending, the
//    back substitution yields the coefficients in registers, four at a time,
//    while the thread walks the observer bins downwards: the bin t_j lies in
//    the interval whose arrival times tau + Delta bracket it, tau* is the root
//    of a cubic there by Newton's method (three steps from the chord, the last
//    one in FP64; the two before it need not be exact, and their FP32 parts leave
//    the FP64 pipe alone: against long double the result is that of three FP64
//    steps, to rounding up to tip Mach numbers of 0.9 at 30 frames a revolution,
//    1e-11 at 18), and the spline of g at tau* goes to a shared-memory tile from
//    which each warp sums its panels, one FP64 atomic per warp and bin.  Delays
//    and bin times count from the delay at the panel's first frame: that halves
//    the rounding of the arrivals, which is the error that is left.
// About 131 FP64 operations per (panel, sample, observer); bound by the FP64 pipe.
// Spinning sphere of 8192 panels x 2048 frames x 16 observers: 63.6 ms for
// k_mscatter (135.4 with moments, four columns, divisions in Newton's method
// and a shuffle sum per bin: about 380 operations), 1.84 ms for k_mseries (5.65
// with each frame's integrands formed three times), 65.5 ms a call (164).
// Scratch: two FP64 columns of nt per (panel, observer) of a launch; the host
// splits the observers into launches by the scratch budget.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/fwh.h"
#include "fwh_internal.cuh"

fwh_status fwh_fail_handle(fwh_handle h, fwh_status st, const char *msg);

namespace {

constexpr int kMRow = 16;     // series row: Qn, Qn', L(3), L'(3), M(3), M'(3), M.M, L.M
constexpr int kMRun = 16;     // frames per series thread
constexpr int kMTile = 128;   // panels per scatter CTA
constexpr int kMBins = 16;    // bins a warp sums at a time
constexpr double kInv4Pi = 0.079577471545947667884441881686257181;

struct MovArgs {
  const double *y, *n, *v;    // [nt][P][3]
  const double *dS;           // [P]
  const double *fields;       // [nt][5][P]
  const double *x0, *w;       // [O][3], [3]
  double c0, rho0, dt;
  int P, nt, O;
  double *S;                  // [nt][kMRow][P] series (panel fastest)
  double *ts, *te;            // [O] window
  int *nv;                    // [O]
  double *p_out;              // [O][nt]
  double *scratch;            // [2][nt][P * n_obs of the launch]
  int o_lo, n_obs;            // observers of this launch
};

// Q_n (Eq. Qn) and L_i (Eq. Li with P_ij = p' delta_ij) of panel p at frame i.
__device__ __forceinline__ void mv_integrands(const MovArgs &a, int p, int i, double &qn,
                                              double L[3]) {
  const double *n = a.n + ((size_t)i * a.P + p) * 3, *v = a.v + ((size_t)i * a.P + p) * 3;
  const double *f = a.fields + (size_t)i * 5 * a.P + p;
  const double rho = a.rho0 + f[0];
  const double u[3] = {f[(size_t)a.P], f[2 * (size_t)a.P], f[3 * (size_t)a.P]};
  const double pp = f[4 * (size_t)a.P];
  double q = 0.0, un = 0.0, vn = 0.0;
  for (int c = 0; c < 3; ++c) {
    q += (a.rho0 * v[c] + rho * (u[c] - v[c])) * n[c];
    un += u[c] * n[c];
    vn += v[c] * n[c];
  }
  qn = q;
  for (int c = 0; c < 3; ++c) L[c] = pp * n[c] + rho * u[c] * (un - vn);
}

// Frames [i0, i0 + kMRun) of one panel; (q, L, v) of the frames i - 1, i, i + 1 slide
// through registers (central differences inside, one-sided at the ends).
struct MvFrame {
  double q, L[3], v[3];
};
__device__ __forceinline__ MvFrame mv_frame(const MovArgs &a, int p, int i) {
  MvFrame f;
  mv_integrands(a, p, i, f.q, f.L);
  for (int c = 0; c < 3; ++c) f.v[c] = a.v[((size_t)i * a.P + p) * 3 + c];
  return f;
}

__global__ void __launch_bounds__(256) k_mseries(MovArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.P) return;
  const double inv2h = 0.5 / a.dt, ic0 = 1.0 / a.c0;
  for (int i0 = blockIdx.y * kMRun; i0 < a.nt; i0 += gridDim.y * kMRun) {  // grid y <= 65535
    const int i1 = min(a.nt, i0 + kMRun);
    MvFrame fm{}, f = mv_frame(a, p, i0), fp{};
    if (i0 > 0) fm = mv_frame(a, p, i0 - 1);
    for (int i = i0; i < i1; ++i) {
      if (i + 1 < a.nt) fp = mv_frame(a, p, i + 1);
      MvFrame d;
      if (i == 0 || i == a.nt - 1) {  // one-sided three-point
        const double sg = i == 0 ? 1.0 : -1.0;
        const MvFrame g1 = i == 0 ? fp : fm, g2 = mv_frame(a, p, i == 0 ? 2 : a.nt - 3);
        d.q = sg * (-3.0 * f.q + 4.0 * g1.q - g2.q);
        for (int c = 0; c < 3; ++c) {
          d.L[c] = sg * (-3.0 * f.L[c] + 4.0 * g1.L[c] - g2.L[c]);
          d.v[c] = sg * (-3.0 * f.v[c] + 4.0 * g1.v[c] - g2.v[c]);
        }
      } else {
        d.q = fp.q - fm.q;
        for (int c = 0; c < 3; ++c) {
          d.L[c] = fp.L[c] - fm.L[c];
          d.v[c] = fp.v[c] - fm.v[c];
        }
      }
      const size_t P = a.P;
      double *row = a.S + (size_t)i * kMRow * P + p;  // value q at row[q P]
      row[0] = f.q;
      row[P] = d.q * inv2h;
      double M2 = 0.0, LM = 0.0;
      for (int c = 0; c < 3; ++c) {
        const double M = f.v[c] * ic0;
        M2 = fma(M, M, M2);
        LM = fma(f.L[c], M, LM);
        row[(2 + c) * P] = f.L[c];
        row[(5 + c) * P] = d.L[c] * inv2h;
        row[(8 + c) * P] = M;
        row[(11 + c) * P] = d.v[c] * inv2h * ic0;
      }
      row[14 * P] = M2;
      row[15 * P] = LM;
      fm = f;
      f = fp;
    }
  }
}

// Delay Delta of one source sample: the non-negative root of
// (c0^2 - w.w) Delta^2 - 2 (b.w) Delta - b.b = 0 (Eq. tau, r = c0 Delta).
__device__ __forceinline__ double mv_delay(const MovArgs &a, const double x0[3], double tau,
                                           const double *y, double b[3]) {
  for (int c = 0; c < 3; ++c) b[c] = x0[c] + a.w[c] * tau - y[c];
  const double ww = a.w[0] * a.w[0] + a.w[1] * a.w[1] + a.w[2] * a.w[2];
  const double bw = b[0] * a.w[0] + b[1] * a.w[1] + b[2] * a.w[2];
  const double bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
  const double q = a.c0 * a.c0 - ww;
  return (bw + sqrt(bw * bw + q * bb)) / q;
}

__global__ void __launch_bounds__(256) k_mwindow(MovArgs a) {
  const int o = blockIdx.x;
  const double x0[3] = {a.x0[3 * o], a.x0[3 * o + 1], a.x0[3 * o + 2]};
  const double tau1 = (double)(a.nt - 1) * a.dt;
  double ts = -1e300, te = 1e300;
  for (int p = threadIdx.x; p < a.P; p += blockDim.x) {
    double b[3];
    const double d0 = mv_delay(a, x0, 0.0, a.y + (size_t)p * 3, b);
    const double d1 = mv_delay(a, x0, tau1, a.y + ((size_t)(a.nt - 1) * a.P + p) * 3, b);
    ts = fmax(ts, d0);
    te = fmin(te, tau1 + d1);
  }
  for (int off = 16; off > 0; off >>= 1) {
    ts = fmax(ts, __shfl_xor_sync(0xffffffffu, ts, off));
    te = fmin(te, __shfl_xor_sync(0xffffffffu, te, off));
  }
  __shared__ double sts[8], ste[8];
  const int wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sts[wid] = ts;
    ste[wid] = te;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
      ts = fmax(ts, sts[i]);
      te = fmin(te, ste[i]);
    }
    double v = __dadd_rn(floor(__ddiv_rn(__dsub_rn(te, ts), a.dt)), 1.0);
    v = fmax(0.0, fmin((double)a.nt, v));
    a.ts[o] = ts;
    a.te[o] = te;
    a.nv[o] = (int)v;
  }
}

constexpr int kPiv = 64;  // pivots of tridiag(1, 4, 1); constant to FP64 rounding from row 63 on

// Reciprocal of a number of ordinary size: Newton's method from the FP32 one.
__device__ __forceinline__ double recip(double x) {
  double y = (double)__frcp_rn((float)x);
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// REST: observers at rest (w = 0), whose distance needs no quadratic.
template <bool REST>
__global__ void __launch_bounds__(kMTile, 7) k_mscatter(MovArgs a) {
  const int ob = blockIdx.y;               // observer within the launch
  const int o = a.o_lo + ob;
  const int p = blockIdx.x * kMTile + threadIdx.x;
  const int lane = threadIdx.x & 31, N = a.nt;
  const bool live = p < a.P;
  const int pp = live ? p : a.P - 1;
  const size_t P = a.P, ld = P * a.n_obs;  // scratch row stride
  double *const ZG = a.scratch + (size_t)ob * P + pp, *const ZD = ZG + (size_t)N * ld;
  const double c0 = a.c0, ic0 = 1.0 / c0, h = a.dt;
  __shared__ double ipiv[kPiv];
  __shared__ double tile[kMTile / 32][kMBins][33];
  if (threadIdx.x == 0) {
    double piv = 4.0;
    ipiv[0] = 0.0;
    for (int i = 1; i < kPiv; ++i) {
      if (i > 1) piv = 4.0 - ipiv[i - 1];
      ipiv[i] = 1.0 / piv;
    }
  }
  __syncthreads();
  const double x0[3] = {a.x0[3 * o], a.x0[3 * o + 1], a.x0[3 * o + 2]};
  double iq = 0.0, q = 0.0, w[3] = {0.0, 0.0, 0.0};
  if constexpr (!REST) {
    for (int c = 0; c < 3; ++c) w[c] = a.w[c];
    q = c0 * c0 - (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    iq = 1.0 / q;
  }
  // signal g and delay Delta at every frame (Eqs. pT, pL, tau) and the forward
  // elimination of both, of Delta less its value dl0 at the first frame (bin times
  // less dl0 below): a far observer's distance then rounds neither the spline nor the
  // arrivals.  Threads past the last panel only join the sums below
  double g = 0.0, dl = 0.0, zg = 0.0, zd = 0.0, dl0 = 0.0;
  for (int i = 0; live && i < N; ++i) {
    const double *rw = a.S + (size_t)i * kMRow * P + pp;
    double row[kMRow];
#pragma unroll
    for (int v = 0; v < kMRow; ++v) row[v] = rw[(size_t)v * P];
    const double *y = a.y + ((size_t)i * P + pp) * 3;
    double r, ir, rh[3];
    if constexpr (REST) {
      const double b[3] = {x0[0] - y[0], x0[1] - y[1], x0[2] - y[2]};
      const double bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
      ir = rsqrt(bb);
      r = bb * ir;
      dl = r * ic0;
      for (int c = 0; c < 3; ++c) rh[c] = b[c] * ir;
    } else {
      const double tau = (double)i * h;
      double b[3];
      for (int c = 0; c < 3; ++c) b[c] = fma(w[c], tau, x0[c]) - y[c];
      const double bw = b[0] * w[0] + b[1] * w[1] + b[2] * w[2];
      const double bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
      dl = (bw + sqrt(fma(q, bb, bw * bw))) * iq;
      r = c0 * dl;
      ir = 1.0 / r;
      for (int c = 0; c < 3; ++c) rh[c] = fma(w[c], dl, b[c]) * ir;
    }
    double Mr = row[8] * rh[0], Mdr = row[11] * rh[0], Lr = row[2] * rh[0], Ldr = row[5] * rh[0];
#pragma unroll
    for (int c = 1; c < 3; ++c) {
      Mr = fma(row[8 + c], rh[c], Mr);
      Mdr = fma(row[11 + c], rh[c], Mdr);
      Lr = fma(row[2 + c], rh[c], Lr);
      Ldr = fma(row[5 + c], rh[c], Ldr);
    }
    const double iD = recip(1.0 - Mr);
    const double k = fma(r, Mdr, c0 * (Mr - row[14]));
    // [Qn' + L'_r / c0] / (r D^2) + [L_r - L.M + (Qn + L_r / c0) k / D] / (r^2 D^2)
    const double u = ir * iD * iD;
    const double near = fma(fma(Lr, ic0, row[0]), k * iD, Lr - row[15]);
    g = u * fma(near, ir, fma(Ldr, ic0, row[1]));
    const double ip = ipiv[min(i, kPiv - 1)];
    if (i == 0) {
      zg = g;
      dl0 = dl;
      dl = 0.0;
    } else {
      dl -= dl0;
      zg = fma(6.0, g, -zg) * ip;
      zd = fma(6.0, dl, -zd) * ip;
    }
    ZG[(size_t)i * ld] = zg;
    ZD[(size_t)i * ld] = zd;
  }
  // interval k: coefficients B[0..3] = beta_{k-1} .. beta_{k+2} of both splines
  double G[4] = {0.0, 0.0, 0.0, 0.0}, D[4] = {0.0, 0.0, 0.0, 0.0};
  int k = N - 2;
  auto below = [&](int i, const double *Z, const double *B) -> double {  // beta_i from B[1] = beta_{i+1}
    if (i < 0) return 2.0 * B[1] - B[2];
    return fma(-B[1], ipiv[min(i, kPiv - 1)], Z[(size_t)i * ld]);
  };
  if (live) {
    G[2] = g;
    D[2] = dl;
    G[1] = fma(-g, ipiv[min(N - 2, kPiv - 1)], ZG[(size_t)(N - 2) * ld]);
    D[1] = fma(-dl, ipiv[min(N - 2, kPiv - 1)], ZD[(size_t)(N - 2) * ld]);
    G[3] = 2.0 * G[2] - G[1];
    D[3] = 2.0 * D[2] - D[1];
    G[0] = below(k - 1, ZG, G);
    D[0] = below(k - 1, ZD, D);
  }
  // observer bins downwards: every thread walks the same j; each warp sums its
  // panels kMBins at a time and adds them with one atomic a bin
  const int nv = a.nv[o];
  const double ts = a.ts[o] - dl0, scale = a.dS[pp] * (kInv4Pi / 6.0);
  double(*tl)[33] = tile[threadIdx.x >> 5];
  double ak = fma((double)k, h, (D[0] + 4.0 * D[1] + D[2]) * (1.0 / 6.0));  // arrival of node k
  for (int j1 = nv; j1 > 0; j1 -= kMBins) {
    const int j0 = max(0, j1 - kMBins);
    for (int j = j1 - 1; j >= j0; --j) {
      double val = 0.0;
      if (live) {
        const double tj = fma((double)j, h, ts);
        while (k > 0 && ak > tj) {
          --k;
          G[3] = G[2]; G[2] = G[1]; G[1] = G[0];
          D[3] = D[2]; D[2] = D[1]; D[1] = D[0];
          G[0] = below(k - 1, ZG, G);
          D[0] = below(k - 1, ZD, D);
          ak = fma((double)k, h, (D[0] + 4.0 * D[1] + D[2]) * (1.0 / 6.0));
        }
        // arrival - t_j on the interval: e + p1 f + p2 f^2 + p3 f^3
        const double e = ak - tj;
        const double p1 = fma(0.5, D[2] - D[0], h);
        const double p2 = fma(0.5, D[0] + D[2], -D[1]);
        const double p3 = fma(0.5, D[1] - D[2], (D[3] - D[0]) * (1.0 / 6.0));
        // Newton's method, three steps from the chord, each clamped to the interval:
        // the first in FP32, the second an FP64 residual over an FP32 slope, the
        // last in FP64
        const float r1 = (float)p1, r2 = (float)p2, r3 = (float)p3, re = (float)e;
        auto slope = [&](float x) { return fmaf(fmaf(3.f * r3, x, 2.f * r2), x, r1); };
        float ff = fminf(1.f, fmaxf(0.f, __fdividef(-re, r1 + r2 + r3)));
        ff -= __fdividef(fmaf(fmaf(fmaf(r3, ff, r2), ff, r1), ff, re), slope(ff));
        ff = fminf(1.f, fmaxf(0.f, ff));
        auto residual = [&](double x) { return fma(fma(fma(p3, x, p2), x, p1), x, e); };
        double f = (double)ff;
        f -= (double)__fdividef((float)residual(f), slope(ff));
        f = fmin(1.0, fmax(0.0, f));
        f = fma(-residual(f), recip(fma(fma(3.0 * p3, f, 2.0 * p2), f, p1)), f);
        f = fmin(1.0, fmax(0.0, f));
        const double c = 1.0 - f, f2 = f * f, c2 = c * c;
        val = (c2 * c) * G[0];
        val = fma(fma(f2, fma(3.0, f, -6.0), 4.0), G[1], val);
        val = fma(fma(c2, fma(3.0, c, -6.0), 4.0), G[2], val);
        val = fma(f2 * f, G[3], val) * scale;
      }
      tl[j - j0][lane] = val;
    }
    __syncwarp();
    {  // lane: bin lane % kMBins over half of the warp's panels
      static_assert(kMBins == 16, "two lanes a bin");
      const int b = lane & 15, l0 = lane & 16;
      double v = 0.0;
      if (b < j1 - j0) {
#pragma unroll
        for (int l = 0; l < 16; ++l) v += tl[b][l0 + l];
      }
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      if (lane < j1 - j0) atomicAdd(a.p_out + (size_t)o * N + j0 + lane, v);
    }
    __syncwarp();
  }
}

// Scratch budget of one call (bytes; 0: the default of 16 GiB), process-wide.
std::atomic<int64_t> g_mov_scratch{0};
constexpr int64_t kMovScratchDefault = (int64_t)16 << 30;

// Scratch comes from a pool of the library's own, one per device, which keeps
// up to kPoolKeep bytes between calls (mapping the 6.4 GB of the benchmark case anew on
// every call took 14 ms).  The process can have them back at any time: the driver
// takes them for a cudaMalloc that would otherwise run out (2 GiB free and 6 kept: 4
// GiB are served, for torch's allocator as well); fwh_set_moving_scratch gives them
// back to other processes.  The pool orders reuse between streams itself.
constexpr uint64_t kPoolKeep = (uint64_t)8 << 30;
constexpr int kMaxDev = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kMaxDev] = {};

cudaError_t mov_pool(cudaMemPool_t *pool) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (!g_pool[dev]) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t np = nullptr;
    if ((e = cudaMemPoolCreate(&np, &props)) != cudaSuccess) return e;
    uint64_t keep = kPoolKeep;
    if ((e = cudaMemPoolSetAttribute(np, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
      cudaMemPoolDestroy(np);
      return e;
    }
    g_pool[dev] = np;
  }
  *pool = g_pool[dev];
  return cudaSuccess;
}

bool on_device(const void *p) {
  if (!p) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

fwh_status failm(fwh_status st, const std::string &m) {
  return fwh_fail_handle(nullptr, st, m.c_str());
}

}  // namespace

extern "C" fwh_status fwh_set_moving_scratch(int64_t bytes) {
  if (bytes < 0) return failm(FWH_ERR_ARG, "scratch budget must be >= 0 bytes");
  g_mov_scratch.store(bytes);
  std::lock_guard<std::mutex> lk(g_pool_mu);
  for (cudaMemPool_t p : g_pool)
    if (p && cudaMemPoolTrimTo(p, 0) != cudaSuccess) cudaGetLastError();
  return FWH_OK;
}

extern "C" fwh_status fwh_forward_moving(int64_t P, int64_t nt, const double *y,
                                         const double *normals, const double *velocities,
                                         const double *areas, double c0, double rho0,
                                         double dt, const double *fields, int64_t O,
                                         const double *x0, const double *w, double *p_out,
                                         double *t_start, int64_t *n_valid, void *stream) {
  if (P < 1 || P > (1 << 30)) return failm(FWH_ERR_ARG, "n_panels out of range");
  if (nt < 3 || nt > (1 << 24)) return failm(FWH_ERR_ARG, "nt must be in [3, 2^24]");
  if (O < 1 || O > 65535) return failm(FWH_ERR_ARG, "n_obs must be in [1, 65535]");
  if (!y || !normals || !velocities || !areas || !fields || !x0 || !w || !p_out)
    return failm(FWH_ERR_ARG, "NULL argument");
  if (!(c0 > 0.0) || !(rho0 > 0.0) || !(dt > 0.0) || !std::isfinite(c0) || !std::isfinite(dt))
    return failm(FWH_ERR_ARG, "c0, rho0 and dt must be > 0");
  std::vector<double> wh(3);
  if (on_device(w)) {
    if (cudaMemcpy(wh.data(), w, 3 * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess)
      return failm(FWH_ERR_CUDA, "cannot read w");
  } else {
    wh.assign(w, w + 3);
  }
  if (!(wh[0] * wh[0] + wh[1] * wh[1] + wh[2] * wh[2] < c0 * c0))
    return failm(FWH_ERR_ARG, "observer speed |w| must be below c0");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const size_t geo = (size_t)nt * P * 3 * sizeof(double);
  const size_t fb = (size_t)nt * 5 * P * sizeof(double);
  const size_t ob = (size_t)O * nt * sizeof(double);
  std::vector<void *> tmp;
  cudaMemPool_t pool = nullptr;
  cudaError_t e = mov_pool(&pool);
  auto dev_in = [&](const double *src, size_t bytes) -> const double * {
    if (e != cudaSuccess) return nullptr;
    if (on_device(src)) return src;
    void *d = nullptr;
    if ((e = cudaMallocFromPoolAsync(&d, bytes, pool, s)) != cudaSuccess) return nullptr;
    tmp.push_back(d);
    e = cudaMemcpyAsync(d, src, bytes, cudaMemcpyHostToDevice, s);
    return static_cast<const double *>(d);
  };
  auto dev_buf = [&](size_t bytes) -> void * {
    if (e != cudaSuccess) return nullptr;
    void *d = nullptr;
    if ((e = cudaMallocFromPoolAsync(&d, bytes, pool, s)) != cudaSuccess) return nullptr;
    tmp.push_back(d);
    return d;
  };
  MovArgs a{};
  a.y = dev_in(y, geo);
  a.n = dev_in(normals, geo);
  a.v = dev_in(velocities, geo);
  a.dS = dev_in(areas, (size_t)P * sizeof(double));
  a.fields = dev_in(fields, fb);
  a.x0 = dev_in(x0, (size_t)O * 3 * sizeof(double));
  double *dw = static_cast<double *>(dev_buf(3 * sizeof(double)));
  if (e == cudaSuccess) e = cudaMemcpyAsync(dw, wh.data(), 3 * sizeof(double), cudaMemcpyHostToDevice, s);
  a.w = dw;
  a.c0 = c0;
  a.rho0 = rho0;
  a.dt = dt;
  a.P = (int)P;
  a.nt = (int)nt;
  a.O = (int)O;
  a.S = static_cast<double *>(dev_buf((size_t)P * nt * kMRow * sizeof(double)));
  a.ts = static_cast<double *>(dev_buf((size_t)O * sizeof(double)));
  a.te = static_cast<double *>(dev_buf((size_t)O * sizeof(double)));
  a.nv = static_cast<int *>(dev_buf((size_t)O * sizeof(int)));
  const bool o_dev = on_device(p_out);
  a.p_out = o_dev ? p_out : static_cast<double *>(dev_buf(ob));
  // observers per launch: the budget counts four columns of nt per (panel,
  // observer), of which two are used (at least one observer per launch)
  const size_t per_obs = (size_t)4 * nt * P * sizeof(double);
  const int64_t budget = g_mov_scratch.load() > 0 ? g_mov_scratch.load() : kMovScratchDefault;
  const int n_obs = (int)std::max<size_t>(1, std::min<size_t>((size_t)O, (size_t)budget / per_obs));
  a.scratch = static_cast<double *>(dev_buf(per_obs / 2 * n_obs));
  if (e == cudaSuccess) e = cudaMemsetAsync(a.p_out, 0, ob, s);
  if (e == cudaSuccess) {
    const int64_t runs = (nt + kMRun - 1) / kMRun;
    const dim3 grid((unsigned)((P + 255) / 256), (unsigned)std::min<int64_t>(runs, 65535));
    k_mseries<<<grid, 256, 0, s>>>(a);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    k_mwindow<<<(unsigned)O, 256, 0, s>>>(a);
    e = cudaGetLastError();
  }
  for (int o0 = 0; e == cudaSuccess && o0 < O; o0 += n_obs) {
    a.o_lo = o0;
    a.n_obs = (int)std::min<int64_t>(n_obs, O - o0);
    dim3 grid((unsigned)((P + kMTile - 1) / kMTile), (unsigned)a.n_obs);
    if (wh[0] == 0.0 && wh[1] == 0.0 && wh[2] == 0.0)
      k_mscatter<true><<<grid, kMTile, 0, s>>>(a);
    else
      k_mscatter<false><<<grid, kMTile, 0, s>>>(a);
    e = cudaGetLastError();
  }
  std::vector<double> hts;
  std::vector<int> hnv;
  if (e == cudaSuccess && (t_start || n_valid)) {
    hts.resize(O);
    hnv.resize(O);
    e = cudaMemcpyAsync(hts.data(), a.ts, O * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(hnv.data(), a.nv, O * sizeof(int), cudaMemcpyDeviceToHost, s);
  }
  if (e == cudaSuccess && !o_dev) e = cudaMemcpyAsync(p_out, a.p_out, ob, cudaMemcpyDeviceToHost, s);
  for (void *d : tmp) cudaFreeAsync(d, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return failm(e == cudaErrorMemoryAllocation ? FWH_ERR_OOM : FWH_ERR_CUDA,
                 std::string("fwh_forward_moving: ") + cudaGetErrorString(e));
  }
  for (int64_t o = 0; o < O; ++o) {
    if (t_start) t_start[o] = hts[o];
    if (n_valid) n_valid[o] = hnv[o];
  }
  return FWH_OK;
}
