// Adjoint of the forward scatter: a conflict-free gather over observers.
//
// The forward adds, for panel p, observer o and sample s (row s + 1 of X),
// w_t G_s to the bin of interval s + 1 - t, t = 0 .. 3, with G_s = c . X[s].
// Its transpose, for the gradient g of the loss with respect to p_out (zero
// outside the valid bins 0 <= j < N_o), is
//   q = w3 g[s-2-i0] + w2 g[s-1-i0] + w1 g[s-i0] + w0 g[s+1-i0]
//   Xbar[p][s][v] = sum_o c_v q,
// so each (panel, sample) output is owned by one lane and summed over the
// observers in registers, 12 multiply-adds per (panel, sample, observer).
// The ghost rows beta_{-1} = 2 beta_0 - beta_1 and beta_nt = 2 beta_{nt-1} -
// beta_{nt-2} hand their gradients to the two samples next to them, times 2
// and -1: a warp whose chunk holds one of those sums the ghost's gradient with
// its lanes over the observers, beside the main loop.  An observer whose valid
// bins the chunk cannot reach is left out (its g there is zero).  Two forms:
// k_adjoint_set (FP32) gathers per panel set from a window of g staged in
// shared memory, with atomics only to add the partial sums of several
// 36-observer groups; k_adjoint (FP64) is one CTA per panel reading g from
// L2, without atomics.  Nothing from the forward pass is stored: only the
// per-(p, o) records (geometry, computed once per observer set), the plan and
// g are read.
#include "fwh_internal.cuh"

namespace fwh {

namespace {

// g converted to T with zeros outside [0, N_o): Gt[o][j], j < g_ld.
template <typename T>
__global__ void k_grad_pad(const double *grad_p, const int *n_valid, T *Gt, int O, int nt,
                           int g_ld) {
  for (int o = blockIdx.y; o < O; o += gridDim.y) {  // grid y is capped at 65535
    const int nv = n_valid[o];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < g_ld; j += gridDim.x * blockDim.x)
      Gt[(size_t)o * g_ld + j] = (j < nv && j < nt) ? (T)grad_p[(size_t)o * nt + j] : T(0);
  }
}

// q of a sample from g at the intervals s - 2 .. s + 1.
template <typename T>
__device__ __forceinline__ T gather_q(const T *w, T gm2, T gm1, T g0, T g1) {
  return fma(w[0], g1, fma(w[1], g0, fma(w[2], gm1, w[3] * gm2)));
}
// Sums v[8] over the warp; every lane gets all eight.
template <typename T>
__device__ __forceinline__ void warp_sum8(T (&v)[kSer]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int n = kSer / 2, m = 16; n >= 1; n >>= 1, m >>= 1)
#pragma unroll
    for (int i = 0; i < n; ++i) {  // hand one half of the components to lane ^ m
      const T send = lane & m ? v[i] : v[i + n];
      v[i] = (lane & m ? v[i + n] : v[i]) + __shfl_xor_sync(0xffffffffu, send, m);
    }
  T r = v[0];  // component lane >> 2
  r += __shfl_xor_sync(0xffffffffu, r, 2);
  r += __shfl_xor_sync(0xffffffffu, r, 1);
#pragma unroll
  for (int s = 0; s < kSer; ++s) v[s] = __shfl_sync(0xffffffffu, r, 4 * s);
}
// Ghost rows next to the samples of [k0, k0 + ch): bit 0 the one before the
// record, bit 1 the one after it.
__device__ __forceinline__ int ghosts(int k0, int ch, int nt) {
  return (k0 < 2 ? 1 : 0) | (k0 < nt && k0 + ch >= nt - 1 ? 2 : 0);
}
// The share of ghost row `end` (0 or 1) that sample s takes.
template <typename T>
__device__ __forceinline__ T ghost_share(int end, int s, int nt) {
  const int d = end ? nt - 1 - s : s;
  return d == 0 ? T(2) : d == 1 ? T(-1) : T(0);
}

// FP64: one CTA per (panel, group of 8 chunks of 64 samples), one warp per
// chunk.  The panel's records are staged in shared memory in tiles of
// kObsTile observers (read back as broadcasts), and each lane loads the
// gradient bins of the next observer while it accumulates the current one.
constexpr int kObsTile = 128;

__global__ void __launch_bounds__(256) k_adjoint(AdjArgs<double> a) {
  constexpr int TK = 2, CH = 32 * TK;
  __shared__ __align__(16) double srec[kObsTile * kRec];
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const int nch = (a.nt + CH - 1) / CH;
  const int ngrp = (nch + 7) / 8;
  const int p = blockIdx.x / ngrp;
  const int ch = (blockIdx.x % ngrp) * 8 + w;
  const bool live = ch < nch;  // warps past the last chunk only help staging
  const int k0 = ch * CH;
  double acc[TK][kSer];
#pragma unroll
  for (int j = 0; j < TK; ++j)
#pragma unroll
    for (int s = 0; s < kSer; ++s) acc[j][s] = 0.0;
  const double *rec0 = a.coef + (size_t)p * a.O * kRec;
  for (int ob = 0; ob < a.O; ob += kObsTile) {
    const int no = min(kObsTile, a.O - ob);
    __syncthreads();
    for (int idx = threadIdx.x; idx < no * kRec; idx += blockDim.x)
      srec[idx] = rec0[(size_t)ob * kRec + idx];
    __syncthreads();
    if (!live) continue;
    auto bins = [&](int o, double (&g)[TK][4]) {
      const int i0 = (int)srec[o * kRec + slot::i0];
      const double *G = a.Gt + (size_t)(ob + o) * a.g_ld;
#pragma unroll
      for (int j = 0; j < TK; ++j)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int jb = k0 + lane + 32 * j - 2 + t - i0;  // bin of interval s - 2 + t
          g[j][t] = jb >= 0 && jb < a.g_ld ? __ldg(G + jb) : 0.0;
        }
    };
    for (int of = 0; of < no; of += 32) {
      // observers of the 32 from `of` on with a valid bin in reach
      bool on = false;
      if (of + lane < no) {
        const int i0 = (int)srec[(of + lane) * kRec + slot::i0];
        on = k0 - 2 - i0 < a.n_valid[ob + of + lane] && k0 + CH - i0 >= 0;
      }
      unsigned left = __ballot_sync(0xffffffffu, on);
      if (!left) continue;
      double g[TK][4];
      bins(of + __ffs(left) - 1, g);
      while (left) {
        const int o = of + __ffs(left) - 1;
        left &= left - 1;
        double gn[TK][4];
        if (left) bins(of + __ffs(left) - 1, gn);
        double c[12];
#pragma unroll
        for (int s = 0; s < 12; ++s) c[s] = srec[o * kRec + s];
#pragma unroll
        for (int j = 0; j < TK; ++j) {
          const double q = gather_q(c + slot::w, g[j][0], g[j][1], g[j][2], g[j][3]);
#pragma unroll
          for (int s = 0; s < kSer; ++s) acc[j][s] = fma(c[s], q, acc[j][s]);
        }
        if (left) {
#pragma unroll
          for (int j = 0; j < TK; ++j)
#pragma unroll
            for (int t = 0; t < 4; ++t) g[j][t] = gn[j][t];
        }
      }
    }
  }
  if (!live) return;
  const int gh = ghosts(k0, CH, a.nt);
  for (int e = 0; e < 2; ++e)
    if (gh >> e & 1) {
      double v[kSer] = {};
      for (int o = lane; o < a.O; o += 32) {
        const double *r = rec0 + (size_t)o * kRec, *w4 = r + slot::w;
        const double *G = a.Gt + (size_t)o * a.g_ld;
        auto bin = [&](int k) {  // g of interval k
          const int j = k - (int)r[slot::i0];
          return j >= 0 && j < a.g_ld ? __ldg(G + j) : 0.0;
        };
        const double q = e ? fma(w4[2], bin(a.nt - 1), w4[3] * bin(a.nt - 2)) : w4[0] * bin(0);
#pragma unroll
        for (int s = 0; s < kSer; ++s) v[s] = fma(r[s], q, v[s]);
      }
      warp_sum8(v);
#pragma unroll
      for (int j = 0; j < TK; ++j) {
        const double f = ghost_share<double>(e, k0 + lane + 32 * j, a.nt);
#pragma unroll
        for (int s = 0; s < kSer; ++s) acc[j][s] = fma(f, v[s], acc[j][s]);
      }
    }
  double *out = a.Xbar + ((size_t)p * a.xb_ld + k0 + lane) * kSer;
#pragma unroll
  for (int j = 0; j < TK; ++j)
#pragma unroll
    for (int s = 0; s < kSer; s += 4)
      stg256(out + (size_t)j * 32 * kSer + s, __double_as_longlong(acc[j][s]),
             __double_as_longlong(acc[j][s + 1]), __double_as_longlong(acc[j][s + 2]),
             __double_as_longlong(acc[j][s + 3]));
}

// Set form (FP32).  Work item = (panel set, observer group, 128-sample
// chunk), numbered observer group fastest, then chunk, then the sets in
// descending size.  The gradient bins every (panel, observer) of the set can
// touch in the chunk are staged in shared memory once per item, quarter-split
// as the forward's windows (slot Y, the bin of interval k0 - 2 + Y at the
// set's largest shift, in quarter Y & 3 at word Y >> 2), so the records'
// byte offsets serve here too.  Each warp then takes panels of the set in
// turn; a lane holds four consecutive samples, reads the seven bins they
// touch per observer (conflict-free) and accumulates the eight components of
// its Xbar rows as register pairs with packed FMAs.  Each warp stages the
// group's records of its next panel in shared memory (cp.async, a double
// buffer per warp) while it works on the current one, so the inner loop reads
// every record as a shared-memory broadcast instead of waiting on L2.  One
// observer group writes Xbar directly, 32 bytes a lane and store; several add
// their partial sums with vector atomics into a zeroed Xbar.
// Bound by instruction issue and shared-memory bandwidth together (issue 61 %,
// shared-memory wavefronts 55 %, DRAM 11 %).  Eight warps a CTA so that 16 fit an
// SM beside the windows (four: 12, 2 % slower).  16384 panels x 1024 steps x 36
// observers: 0.50 ms; 0.58 with the ghosts' share computed for every sample of an
// edge chunk and every observer taken in every chunk (FP64, 5151 x 701 x 19:
// 1.78 -> 1.49 ms).  Runs of six: the gradient's error against 64 bits is 2.2e-6
// there (3.2e-6 with one running sum).
constexpr int kAdjGroup = 36;    // observers per item
constexpr int kAdjRun = 6;       // observers summed from zero at a time
constexpr int kAdjWarps = 8;
constexpr int kAdjTK = 4;        // samples per lane (chunk 128)

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
// 4-byte copy, zero fill when !ok (src is then not read)
__device__ __forceinline__ void cp_async4_zf(float *dst, const float *src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void red_add_v4(float *addr, float4 v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(addr), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}

template <bool kAtomic>
__global__ void __launch_bounds__(kAdjWarps * 32) k_adjoint_set(AdjArgs<float> a) {
  constexpr int CH = 32 * kAdjTK;
  extern __shared__ __align__(16) float gw[];  // [kAdjGroup][win], then the record buffers
  __shared__ int s_obs[kAdjGroup];             // the group's observers with a bin in reach
  const int win = a.win, H = win >> 2;
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const int ng = (a.O + kAdjGroup - 1) / kAdjGroup;
  const int nch = (a.nt + CH - 1) / CH;
  const int item = blockIdx.x;
  const int g = item % ng;
  const int rest = item / ng;
  const int ch = rest % nch;
  const int sidx = a.set_order[rest / nch];
  const int k0 = ch * CH;
  const int gh = ghosts(k0, CH, a.nt);
  const int o0 = g * kAdjGroup;
  const int *i0max = a.i0max_tab + (size_t)sidx * a.O + o0;
  int no = 0;  // observers with a valid bin in reach of the set's samples here
  for (int of = 0; of < min(kAdjGroup, a.O - o0); of += 32) {
    const int o = of + lane;
    bool on = false;
    if (o < min(kAdjGroup, a.O - o0)) {
      const int i0 = i0max[o];
      on = k0 - 2 - i0 < a.n_valid[o0 + o] && k0 + CH - i0 + a.slack >= 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (on && w == 0) s_obs[no + __popc(m & ((1u << lane) - 1))] = o;
    no += __popc(m);
  }
  __syncthreads();
  const int p_begin = a.set_begin[sidx], p_end = a.set_begin[sidx + 1];
  // stage the window of each observer of the group (cp.async: every copy in
  // flight at once; zero outside the record)
  for (int o = 0; o < no; ++o) {
    const int base = k0 - 2 - i0max[s_obs[o]];
    const float *G = a.Gt + (size_t)(o0 + s_obs[o]) * a.g_ld;
    for (int t = threadIdx.x; t < win; t += blockDim.x) {
      const int j = base + t;
      const bool ok = j >= 0 && j < a.g_ld;
      cp_async4_zf(gw + o * win + (t & 3) * H + (t >> 2), G + (ok ? j : 0), ok);
    }
  }
  cp_async_commit();
  // this warp's record double buffer: [2][kAdjGroup][kRec]
  float *rb = gw + (size_t)kAdjGroup * win + (size_t)w * 2 * kAdjGroup * kRec;
  auto stage = [&](int p, int buf) {  // the group's records of panel p, 16 bytes a copy
    const float *src = a.coef + ((size_t)p * a.O + o0) * kRec;
    float *dst = rb + (size_t)buf * kAdjGroup * kRec;
    for (int c = lane; c < no * (kRec / 4); c += 32)
      cp_async16(dst + 4 * c, src + s_obs[c / (kRec / 4)] * kRec + 4 * (c % (kRec / 4)));
    cp_async_commit();
  };
  const int shift = a.slot_shift;  // the records' offsets are in slots of 2^shift bytes
  int buf = 0;
  if (p_begin + w < p_end) stage(p_begin + w, 0);
  cp_async_wait<0>();  // the window (and this warp's first records)
  __syncthreads();
  for (int p = p_begin + w; p < p_end; p += kAdjWarps) {
    const bool more = p + kAdjWarps < p_end;
    if (more) {
      stage(p + kAdjWarps, buf ^ 1);
      cp_async_wait<1>();  // this panel's copy has landed (the next one may still fly)
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    // The spline's adjoint amplifies rounding noise in Xbar, so a panel's sum
    // over the group's observers is taken in runs of kAdjRun, each from zero:
    // a third of the rounding of one running sum of 36.
    f32x2 sum[kAdjTK][kSer / 2];
#pragma unroll
    for (int j = 0; j < kAdjTK; ++j)
#pragma unroll
      for (int s = 0; s < kSer / 2; ++s) sum[j][s] = 0ull;
    const float *rec = rb + (size_t)buf * kAdjGroup * kRec;
    for (int or0 = 0; or0 < no; or0 += kAdjRun) {
      f32x2 acc[kAdjTK][kSer / 2];
#pragma unroll
      for (int j = 0; j < kAdjTK; ++j)
#pragma unroll
        for (int s = 0; s < kSer / 2; ++s) acc[j][s] = 0ull;
      const int oe = min(no, or0 + kAdjRun);
#pragma unroll 3
      for (int o = or0; o < oe; ++o) {
        const ulonglong2 c01 = *reinterpret_cast<const ulonglong2 *>(rec + o * kRec);
        const ulonglong2 c23 = *reinterpret_cast<const ulonglong2 *>(rec + o * kRec + 4);
        const float4 wv = *reinterpret_cast<const float4 *>(rec + o * kRec + slot::w);
        const uint4 qo = *reinterpret_cast<const uint4 *>(rec + o * kRec + slot::q0);
        const f32x2 c[4] = {c01.x, c01.y, c23.x, c23.y};
        const float wt[4] = {wv.x, wv.y, wv.z, wv.w};
        const float *gp = gw + o * win + lane;
        const float *A[4] = {gp + (qo.x >> shift), gp + (qo.y >> shift), gp + (qo.z >> shift),
                             gp + (qo.w >> shift)};
        float gv[7];  // bins of intervals s - 2 .. s + 4 of the lane's first sample s
#pragma unroll
        for (int i = 0; i < 7; ++i) gv[i] = A[i & 3][i >> 2];
#pragma unroll
        for (int j = 0; j < kAdjTK; ++j) {
          const f32x2 q2 = f2_dup(gather_q(wt, gv[j], gv[j + 1], gv[j + 2], gv[j + 3]));
#pragma unroll
          for (int s = 0; s < kSer / 2; ++s) acc[j][s] = f2_fma(c[s], q2, acc[j][s]);
        }
      }
#pragma unroll
      for (int j = 0; j < kAdjTK; ++j)
#pragma unroll
        for (int s = 0; s < kSer / 2; ++s) sum[j][s] = f2_add(sum[j][s], acc[j][s]);
    }
    for (int e = 0; e < 2; ++e)
      if (gh >> e & 1) {
        float v[kSer] = {};
        for (int o = lane; o < no; o += 32) {
          const float *r = rec + o * kRec;
          const unsigned *qo = reinterpret_cast<const unsigned *>(r + slot::q0);
          auto bin = [&](int k) {  // g of interval k
            const int y = k - k0 + 2;
            return gw[o * win + (qo[y & 3] >> shift) + (y >> 2)];
          };
          const float *w4 = r + slot::w;
          const float q =
              e ? fmaf(w4[2], bin(a.nt - 1), w4[3] * bin(a.nt - 2)) : w4[0] * bin(0);
#pragma unroll
          for (int s = 0; s < kSer; ++s) v[s] = fmaf(r[s], q, v[s]);
        }
        warp_sum8(v);
        f32x2 v2[kSer / 2];
#pragma unroll
        for (int s = 0; s < kSer / 2; ++s) v2[s] = f2_pack(v[2 * s], v[2 * s + 1]);
#pragma unroll
        for (int j = 0; j < kAdjTK; ++j) {
          const f32x2 f = f2_dup(ghost_share<float>(e, k0 + 4 * lane + j, a.nt));
#pragma unroll
          for (int s = 0; s < kSer / 2; ++s) sum[j][s] = f2_fma(f, v2[s], sum[j][s]);
        }
      }
    float *out = a.Xbar + ((size_t)p * a.xb_ld + k0 + 4 * lane) * kSer;
#pragma unroll
    for (int j = 0; j < kAdjTK; ++j) {
      if (kAtomic) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float4 v;
          f2_split(sum[j][2 * h], v.x, v.y);
          f2_split(sum[j][2 * h + 1], v.z, v.w);
          red_add_v4(out + j * kSer + 4 * h, v);
        }
      } else {
        stg256(out + j * kSer, sum[j][0], sum[j][1], sum[j][2], sum[j][3]);
      }
    }
    __syncwarp();  // every lane is done with this buffer before it is refilled
    buf ^= 1;
  }
}

}  // namespace

template <typename T>
cudaError_t launch_adjoint(const AdjArgs<T> &a, cudaStream_t s) {
  dim3 gg((a.g_ld + 255) / 256, a.O < 65535 ? a.O : 65535);
  k_grad_pad<T><<<gg, 256, 0, s>>>(a.grad_p, a.n_valid, a.Gt, a.O, a.nt, a.g_ld);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if constexpr (sizeof(T) == 4) {
    constexpr int CH = 32 * kAdjTK;
    const int ng = (a.O + kAdjGroup - 1) / kAdjGroup;
    const long items = (long)a.nsets * ng * ((a.nt + CH - 1) / CH);
    if (items <= 0) return cudaSuccess;
    if (items > INT32_MAX) return cudaErrorInvalidValue;
    const size_t smem = ((size_t)kAdjGroup * a.win + (size_t)kAdjWarps * 2 * kAdjGroup * kRec) *
                        sizeof(float);
    auto kern = ng > 1 ? k_adjoint_set<true> : k_adjoint_set<false>;
    if (ng > 1) {
      e = cudaMemsetAsync(a.Xbar, 0, (size_t)a.P * a.xb_ld * kSer * sizeof(float), s);
      if (e != cudaSuccess) return e;
    }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)items, kAdjWarps * 32, smem, s>>>(a);
  } else {
    const long blocks = (long)a.P * (((a.nt + 63) / 64 + 7) / 8);
    if (blocks <= 0) return cudaSuccess;
    if (blocks > INT32_MAX) return cudaErrorInvalidValue;
    k_adjoint<<<(unsigned)blocks, 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

template cudaError_t launch_adjoint<float>(const AdjArgs<float> &, cudaStream_t);
template cudaError_t launch_adjoint<double>(const AdjArgs<double> &, cudaStream_t);

}  // namespace fwh
