// Power spectral density of the far-field signals (Sec. IV C): Welch's
// method -- segments of L samples with 50 % overlap, a Hanning window on each,
// the squared magnitude of each segment's discrete Fourier transform averaged
// over the segments -- then the span correction of Eq. PSD_corr,
//   PSD_corr = PSD + 10 log10(b_exp / b_m)   (dB),  i.e. PSD x b_exp / b_m.
//
// A cluster of up to eight CTAs per signal (one where there are signals
// enough to fill the GPU); each CTA takes pairs of segments, and the cluster
// adds its CTAs' sums through distributed shared memory, in rank order.  The
// segments are transformed two at a time: segment a is the real and segment b
// the imaginary part of one complex sequence z, and with Z its transform,
//   A_k = (Z_k + conj Z_{L-k}) / 2,   B_k = (Z_k - conj Z_{L-k}) / (2 i),
// so one complex FFT of length L serves two segments.  The FFT is an
// iterative radix-2 decimation-in-time transform in shared memory (input
// written in bit-reversed order, log2 L butterfly stages; twiddles exp(-2 pi i
// j / L) tabulated once per CTA from an eighth of the circle, the window from
// them).  Everything is FP64, so the FP64 pipe (2 operations a clock and SM)
// and the barriers between stages set the pace: six fused operations a
// butterfly.  72 signals x 2048 samples, L = 512 (four pairs each, so four CTAs a
// signal): 29 us for the kernel, 33 us a call; 67 and 290 us with one CTA a
// signal, a sine and two cosines per table entry and a device copy of the
// lengths.
// Bytes per signal: its N valid samples are read once per segment they fall
// in (twice with the 50 % overlap), L / 2 + 1 values are written.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>

#include "../../include/fwh.h"
#include "fwh_internal.cuh"

fwh_status fwh_fail_handle(fwh_handle h, fwh_status st, const char *msg);

namespace {

constexpr int kPsdThreads = 256;
constexpr int kPsdMaxSeg = 4096;
constexpr int kPsdByValue = 1024;  // signals whose lengths travel with the launch

namespace cg = cooperative_groups;

struct PsdArgs {
  const double *p;          // [n_sig][ld]
  const long long *n_valid; // [n_sig] or null (every signal has ld samples)
  long long ld;
  int L, log2L;
  double fs, span, p_ref;
  int detrend;
  double *out;              // [n_sig][L / 2 + 1]
};

// Host lengths of up to kPsdByValue signals as a kernel parameter (no device
// buffer, copy or synchronisation); n = 0: use PsdArgs::n_valid.
struct PsdLengths {
  int n;
  int len[kPsdByValue];
};

__device__ __forceinline__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();  // red may still be read by a previous sum
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];  // same order in every thread
  return s;
}

__global__ void __launch_bounds__(kPsdThreads)
    k_psd(PsdArgs a, const __grid_constant__ PsdLengths lens) {
  extern __shared__ __align__(16) double2 sm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), cs = (int)cluster.num_blocks();
  const int L = a.L, half = L >> 1, tid = threadIdx.x, T = blockDim.x;
  double2 *z = sm;                                        // [L]
  double2 *tw = z + L;                                    // [L / 2]
  double *acc = reinterpret_cast<double *>(tw + half);    // [L / 2 + 1]
  double *red = acc + half + 1;                           // [T / 32]
  const int sig = blockIdx.x / cs;
  long long n = lens.n ? lens.len[sig] : a.n_valid ? a.n_valid[sig] : a.ld;
  n = n < 0 ? 0 : (n > a.ld ? a.ld : n);
  const int K = n < L ? 0 : (int)((n - L) / half) + 1;  // segments
  // twiddles (cos, -sin)(2 pi j / L), j < L / 2, from the first eighth
  for (int j = tid; j <= L / 8; j += T) {
    double s, c;
    sincospi(2.0 * (double)j / (double)L, &s, &c);
    tw[j] = make_double2(c, -s);
    if (j > 0) tw[half - j] = make_double2(-c, -s);
    tw[L / 4 - j] = make_double2(s, -c);
    tw[L / 4 + j] = make_double2(-s, -c);
  }
  __syncthreads();
  // periodic Hanning window 0.5 - 0.5 cos(2 pi i / L)
  auto hann = [&](int i) -> double {
    return i < half ? 0.5 - 0.5 * tw[i].x : 0.5 + 0.5 * tw[i - half].x;
  };
  double w2 = 0.0;
  for (int i = tid; i < L; i += T) {
    const double w = hann(i);
    w2 += w * w;
  }
  for (int k = tid; k <= half; k += T) acc[k] = 0.0;
  const double wsum2 = block_sum(w2, red);
  const double *x = a.p + (long long)sig * a.ld;
  const double iL = 1.0 / L;
  for (int s = 2 * rank; s < K; s += 2 * cs) {
    const bool hb = s + 1 < K;
    const double *xa = x + (long long)s * half, *xb = x + (long long)(s + 1) * half;
    double ma = 0.0, mb = 0.0;
    if (a.detrend) {
      double sa = 0.0, sb = 0.0;
      for (int i = tid; i < L; i += T) {
        sa += xa[i];
        if (hb) sb += xb[i];
      }
      ma = block_sum(sa, red) * iL;
      mb = block_sum(sb, red) * iL;
    }
    for (int i = tid; i < L; i += T) {
      const double w = hann(i);
      z[__brev((unsigned)i) >> (32 - a.log2L)] =
          make_double2(w * (xa[i] - ma), hb ? w * (xb[i] - mb) : 0.0);
    }
    __syncthreads();
    // the first two stages (twiddles 1 and -i) on four neighbours at once
    for (int b = tid; b < L / 4; b += T) {
      double2 *q = z + 4 * b;
      const double2 q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3];
      const double2 e0 = make_double2(q0.x + q1.x, q0.y + q1.y);
      const double2 e1 = make_double2(q0.x - q1.x, q0.y - q1.y);
      const double2 f0 = make_double2(q2.x + q3.x, q2.y + q3.y);
      const double2 f1 = make_double2(q2.x - q3.x, q2.y - q3.y);
      q[0] = make_double2(e0.x + f0.x, e0.y + f0.y);
      q[1] = make_double2(e1.x + f1.y, e1.y - f1.x);
      q[2] = make_double2(e0.x - f0.x, e0.y - f0.y);
      q[3] = make_double2(e1.x - f1.y, e1.y + f1.x);
    }
    __syncthreads();
    for (int h = 4, step = L / 8; h < L; h <<= 1, step >>= 1) {
      for (int b = tid; b < half; b += T) {
        const int pos = b & (h - 1);
        const int i = ((b - pos) << 1) + pos, j = i + h;
        const double2 w = tw[pos * step], zj = z[j], zi = z[i];
        const double xr = fma(w.x, zj.x, fma(-w.y, zj.y, zi.x));
        const double xi = fma(w.x, zj.y, fma(w.y, zj.x, zi.y));
        z[i] = make_double2(xr, xi);
        z[j] = make_double2(fma(2.0, zi.x, -xr), fma(2.0, zi.y, -xi));
      }
      __syncthreads();
    }
    for (int k = tid; k <= half; k += T) {
      const double2 zk = z[k & (L - 1)], zm = z[(L - k) & (L - 1)];
      // |A_k|^2 + |B_k|^2 = (|Z_k|^2 + |Z_{L-k}|^2) / 2
      acc[k] += 0.5 * (zk.x * zk.x + zk.y * zk.y + zm.x * zm.x + zm.y * zm.y);
    }
    __syncthreads();
  }
  if (cs > 1) cluster.sync();
  double *o = a.out + (long long)sig * (half + 1);
  const double norm = K > 0 ? 1.0 / ((double)K * a.fs * wsum2) : 0.0;
  for (int k = rank * T + tid; k <= half; k += cs * T) {
    double v = nan("");
    if (K > 0) {
      v = acc[k];
      if (cs > 1) {
        v = 0.0;
        for (int r = 0; r < cs; ++r) v += cluster.map_shared_rank(acc, r)[k];
      }
      v *= norm;
      if (k > 0 && k < half) v *= 2.0;  // one-sided
      v *= a.span;                       // Eq. PSD_corr
      if (a.p_ref > 0.0) v = 10.0 * log10(v / (a.p_ref * a.p_ref));
    }
    o[k] = v;
  }
  if (cs > 1) cluster.sync();  // peers may still be reading this CTA's sums
}

bool on_device(const void *p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

fwh_status fail(fwh_status st, const std::string &m) { return fwh_fail_handle(nullptr, st, m.c_str()); }

}  // namespace

extern "C" fwh_status fwh_psd(int64_t n_sig, const double *p, int64_t ld, const int64_t *n_valid,
                              double fs, int64_t nperseg, int detrend, double span_ratio,
                              double p_ref, double *psd, void *stream) {
  if (n_sig < 1 || n_sig > 0x7fffffff) return fail(FWH_ERR_ARG, "n_sig must be in [1, 2^31)");
  if (!p || !psd) return fail(FWH_ERR_ARG, "p or psd is NULL");
  if (ld < 1) return fail(FWH_ERR_ARG, "ld must be >= 1");
  if (!(fs > 0.0) || !std::isfinite(fs)) return fail(FWH_ERR_ARG, "fs must be > 0");
  if (nperseg < 16 || nperseg > kPsdMaxSeg || (nperseg & (nperseg - 1)))
    return fail(FWH_ERR_ARG, "nperseg must be a power of two in [16, 4096]");
  if (detrend != 0 && detrend != 1) return fail(FWH_ERR_ARG, "detrend must be 0 or 1");
  if (!(span_ratio > 0.0) || !std::isfinite(span_ratio))
    return fail(FWH_ERR_ARG, "span_ratio must be > 0");
  if (!(p_ref >= 0.0) || !std::isfinite(p_ref)) return fail(FWH_ERR_ARG, "p_ref must be >= 0");
  const bool nv_dev = n_valid && on_device(n_valid);
  if (n_valid && !nv_dev)
    for (int64_t i = 0; i < n_sig; ++i)
      if (n_valid[i] < 0 || n_valid[i] > ld)
        return fail(FWH_ERR_ARG, "n_valid[" + std::to_string(i) + "] outside [0, ld]");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int L = (int)nperseg;
  int log2L = 0;
  while ((1 << log2L) < L) ++log2L;
  const size_t in_bytes = (size_t)n_sig * ld * sizeof(double);
  const size_t out_bytes = (size_t)n_sig * (L / 2 + 1) * sizeof(double);
  const bool p_dev = on_device(p), o_dev = on_device(psd);
  void *dp = nullptr, *dn = nullptr, *dout = nullptr;
  cudaError_t e = cudaSuccess;
  auto release = [&]() {
    if (dp) cudaFreeAsync(dp, s);
    if (dn) cudaFreeAsync(dn, s);
    if (dout) cudaFreeAsync(dout, s);
  };
  if (!p_dev && (e = cudaMallocAsync(&dp, in_bytes, s)) == cudaSuccess)
    e = cudaMemcpyAsync(dp, p, in_bytes, cudaMemcpyHostToDevice, s);
  // host lengths travel with the launch where they fit
  PsdLengths lens;
  lens.n = 0;
  if (n_valid && !nv_dev && n_sig <= kPsdByValue && ld <= INT32_MAX) {
    lens.n = (int)n_sig;
    for (int64_t i = 0; i < n_sig; ++i) lens.len[i] = (int)n_valid[i];
  }
  const bool nv_copy = n_valid && !nv_dev && lens.n == 0;
  if (e == cudaSuccess && nv_copy &&
      (e = cudaMallocAsync(&dn, (size_t)n_sig * sizeof(int64_t), s)) == cudaSuccess)
    e = cudaMemcpyAsync(dn, n_valid, (size_t)n_sig * sizeof(int64_t), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && !o_dev) e = cudaMallocAsync(&dout, out_bytes, s);
  PsdArgs a{};
  a.p = p_dev ? p : static_cast<const double *>(dp);
  a.n_valid = reinterpret_cast<const long long *>(n_valid ? (nv_dev ? n_valid : dn) : nullptr);
  a.ld = ld;
  a.L = L;
  a.log2L = log2L;
  a.fs = fs;
  a.span = span_ratio;
  a.p_ref = p_ref;
  a.detrend = detrend;
  a.out = o_dev ? psd : static_cast<double *>(dout);
  const size_t smem = (size_t)L * sizeof(double2) + (size_t)(L / 2) * sizeof(double2) +
                      (size_t)(L / 2 + 1) * sizeof(double) +
                      (kPsdThreads / 32) * sizeof(double);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_psd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) {
    // CTAs per signal: one per pair of segments up to eight, as long as the
    // grid does not pass about four CTAs an SM (more signals than that fill
    // the GPU by themselves, and a cluster only adds its tables and barriers)
    const int64_t pairs = ld < L ? 1 : ((ld - L) / (L / 2) + 2) / 2;
    int cs = 1;
    while (cs < 8 && cs < pairs && n_sig * cs * 2 <= 4 * 152) cs *= 2;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n_sig * cs));
    cfg.blockDim = dim3(kPsdThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_psd, a, lens);
  }
  if (e == cudaSuccess && !o_dev) e = cudaMemcpyAsync(psd, dout, out_bytes, cudaMemcpyDeviceToHost, s);
  release();
  if (e == cudaSuccess && (!o_dev || !p_dev || nv_copy)) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(e == cudaErrorMemoryAllocation ? FWH_ERR_OOM : FWH_ERR_CUDA,
                std::string("fwh_psd: ") + cudaGetErrorString(e));
  }
  return FWH_OK;
}
