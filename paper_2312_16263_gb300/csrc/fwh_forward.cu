// Forward scatter of the FW-H source-time signals onto the observer grids
// ("compute Noise" + "interp pressure signal" + surface integration,
// Sec. III B/C; integrand of Eqs. pT_WT_nd + pL_WT_nd).
//
// For panel p, observer o and the observer-independent rows X[p][r] (B-spline
// coefficients of the 8 series, row r = sample r - 1), with the per-(p, o)
// record (coefficients c, weights w0..w3, shift i0):
//   G[r] = c . X[r]
//   bin k - i0 += w0 G[k] + w1 G[k+1] + w2 G[k+2] + w3 G[k+3]
// for every spline interval k = 0 .. nt - 1, which is the natural-spline value
// at tau = t_j - M0 R for every observer bin j (Eq. tau2), summed over panels:
// 12 multiply-adds per (panel, sample, observer).
//
// Work item = (panel set or a part of it, observer group, time segment).  A
// CTA holds NW compute warps; warp w owns observers o_begin + w + NW m (m <
// obs_per_warp) of the group and keeps, per observer, a window of `win` bins
// in shared memory.  Lanes map to rows, so each X row is loaded once per warp
// and reused for all of the warp's observers, the record is a warp-uniform
// broadcast, and the window updates are conflict-free.  The per-(p, o) shift
// only moves the window offset, never the lane pattern.  After each chunk the
// oldest bins of every window are complete for this item: they are flushed to
// p_out with FP64 atomics (one per bin per item, not per panel) and the
// window slides.
//
// FP32 gathers: a lane holds four consecutive rows of each 128-row block,
// forms G of its rows, takes the next three values from the lane above (the
// last lane of a block from lane 0 of the next block) and adds four complete
// bin values to the window, one read-modify-write per sample.  FP64 scatters:
// a lane holds rows 32 apart and adds each G to its four bins in turn (the
// FP64 pipe, not the window traffic, bounds that form).
//
// Two ways to feed the compute warps:
//  * direct: every warp loads its X rows and coefficient records from global
//    memory (L1/L2) itself;
//  * TMA pipeline: one producer warp streams, per (chunk, panel) step, the X
//    rows (a 2D tensor-map load of 128-byte lines, 128B swizzled so the
//    per-lane reads are bank-conflict-free) and the group's coefficient
//    records (a 1D bulk copy) into a ring of shared-memory stages; full/empty
//    mbarriers hand the stages over.  Every wait is bounded by a clock limit:
//    on expiry the kernel raises kErrTimeout, stops issuing copies, waits
//    (bounded) for the copies already in flight and leaves.
//
// Window bound: a panel set's shifts for one observer span S = i0max - i0min;
// fwd_slack() is the largest S whose slots stay inside the window.  The host
// planner bounds S from the set's extent; the plan kernel records, per (set,
// observer), i0max and, per (panel, observer) record, the window offset
// i0max - i0 clamped to [0, slack], raising kErrWindow if the bound is
// exceeded; the hot loop adds that offset and can never leave the window.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "fwh_internal.cuh"

namespace fwh {

namespace {

constexpr int kMaxObsPerWarp = 16;
constexpr int kMaxObsPerWarpF32 = 9;  // the FP32 consumer unrolls its observer loop to this
constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz

// 16-byte loads of N doubles.
template <int N>
__device__ __forceinline__ void ldg_f64(const double *src, double (&dst)[N]) {
  const double2 *s = reinterpret_cast<const double2 *>(src);
#pragma unroll
  for (int q = 0; q < N / 2; ++q) {
    const double2 v = __ldg(s + q);
    dst[2 * q] = v.x;
    dst[2 * q + 1] = v.y;
  }
}
template <int N>
__device__ __forceinline__ void lds_f64(const double *src, double (&dst)[N]) {
  const double2 *s = reinterpret_cast<const double2 *>(src);
#pragma unroll
  for (int q = 0; q < N / 2; ++q) {
    const double2 v = s[q];
    dst[2 * q] = v.x;
    dst[2 * q + 1] = v.y;
  }
}

// One FP64 X row (64 bytes, two per 128-byte line) from a TMA stage written
// with SWIZZLE_128B, which XORs the 16-byte chunk index (address bits 4..6)
// with address bits 7..9: chunk q of row r is chunk (((r & 1) << 2) | q) ^
// ((r >> 1) & 7) of line r >> 1, so 8 consecutive lanes hit 8 distinct
// 16-byte bank groups.
__device__ __forceinline__ void lds_row_f64(const unsigned char *stg, int r, double (&dst)[kSer]) {
#pragma unroll
  for (int q = 0; q < kSer / 2; ++q) {
    const double2 v = *reinterpret_cast<const double2 *>(
        stg + (size_t)(r >> 1) * 128 + (((((r & 1) << 2) | q) ^ ((r >> 1) & 7)) << 4));
    dst[2 * q] = v.x;
    dst[2 * q + 1] = v.y;
  }
}

// ---- mbarrier / TMA primitives (PTX) -------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Test the phase; a thread whose phase is not complete is suspended until it
// completes or `suspend_ns` pass, so waiting warps do not spin on issue slots.
constexpr unsigned kSuspendNs = 200000;
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity,
                                              unsigned suspend_ns = kSuspendNs) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(suspend_ns)
      : "memory");
  return ok != 0;
}
// Suspend hint of a wait bounded by `limit` clocks: never longer than the bound
// (about 2 clocks per ns at the SM's clock), so a short bound runs out promptly.
__device__ __forceinline__ unsigned suspend_for(long long limit) {
  return limit >= 2LL * kSuspendNs ? kSuspendNs : (unsigned)(limit >> 1);
}
// Bounded wait: false on timeout (flag raised) or when another warp aborted.
// `limit` is the bound in SM clocks (<= 0: kWaitCycles).  The first test uses
// a fixed suspend hint, so that it does not wait on the loads of `limit` and
// `err`: on the usual path, where the phase is already complete, neither is
// needed.  A bound shorter than the hint runs out after the hint instead (a
// test-only case).
constexpr unsigned kFirstSuspendNs = 1000;
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, int *err,
                                          volatile int *abort, long long limit = 0) {
  if (mbar_try_wait(bar, parity, kFirstSuspendNs)) return true;
  if (limit <= 0) limit = kWaitCycles;
  const unsigned ns = suspend_for(limit);
  const long long t0 = clock64();
  for (;;) {
    if (mbar_try_wait(bar, parity, ns)) return true;
    if (*abort) return false;
    if (clock64() - t0 > limit) {
      atomicOr(err, kErrTimeout);
      *abort = 1;
      return false;
    }
  }
}
// The producer's wait for a free stage: it sleeps between polls, so that
// while the compute warps work it takes almost no issue slots from the warps
// that share its SM sub-partition.
__device__ __forceinline__ bool mbar_wait_sleep(uint64_t *bar, unsigned parity, int *err,
                                                volatile int *abort, long long limit = 0) {
  if (mbar_try_wait(bar, parity, kFirstSuspendNs)) return true;
  if (limit <= 0) limit = kWaitCycles;
  const unsigned sus = suspend_for(limit);
  const long long t0 = clock64();
  unsigned ns = 64;
  for (;;) {
    __nanosleep(ns);
    if (mbar_try_wait(bar, parity, sus)) return true;
    if (ns < 512) ns <<= 1;
    if (*abort) return false;
    if (clock64() - t0 > limit) {
      atomicOr(err, kErrTimeout);
      *abort = 1;
      return false;
    }
  }
}
__device__ __forceinline__ void tma_load_2d(void *dst, const void *tmap, int x, int y,
                                            uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// Warm L2 with a contiguous range ahead of its TMA load (no completion to wait for).
__device__ __forceinline__ void prefetch_l2(const void *src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void atomic_add_f64(double *addr, double v) { atomicAdd(addr, v); }

template <typename T>
__global__ void __launch_bounds__(128) k_plan(T *coef, const int *i0_tab, const int *set_begin,
                                              int O, int slack, int win, int slot_bytes,
                                              int *i0max_tab, int *err) {
  const int sidx = blockIdx.x;
  const int pb = set_begin[sidx], pe = set_begin[sidx + 1];
  for (int o = threadIdx.x; o < O; o += blockDim.x) {
    auto i0_at = [&](int p) -> int {
      const size_t e = (size_t)p * O + o;
      if constexpr (sizeof(T) == 4) return i0_tab[e];
      return (int)coef[e * kRec + slot::i0];
    };
    int lo = 0x7fffffff, hi = -0x7fffffff;
    for (int p = pb; p < pe; ++p) {
      const int i0 = i0_at(p);
      lo = min(lo, i0);
      hi = max(hi, i0);
    }
    if (hi - lo > slack) atomicOr(err, kErrWindow);
    i0max_tab[(size_t)sidx * O + o] = hi;
    for (int p = pb; p < pe; ++p) {
      T *rec = coef + ((size_t)p * O + o) * kRec;
      const int off = min(hi - i0_at(p), slack);
      if constexpr (sizeof(T) == 4) {  // quarter-split window: slot x in quarter x & 3
        const int H = win / 4;
        int4 a;
        a.x = ((off & 3) * H + (off >> 2)) * slot_bytes;
        a.y = (((off + 1) & 3) * H + ((off + 1) >> 2)) * slot_bytes;
        a.z = (((off + 2) & 3) * H + ((off + 2) >> 2)) * slot_bytes;
        a.w = (((off + 3) & 3) * H + ((off + 3) >> 2)) * slot_bytes;
        *reinterpret_cast<int4 *>(rec + slot::q0) = a;
      } else {
        rec[slot::off] = (T)off;
      }
    }
  }
}

// Item decomposition shared by both pipelines.
template <typename T, int NW>
struct Item {
  int sidx, p_begin, p_end, o_begin, o_end, opw, nobs, k_begin, k_end;
  __device__ __forceinline__ Item(const FwdArgs<T> &a, int item, int w) {
    const int ng = a.n_obs_groups;
    // observer group fastest (groups share the set's X rows in L2), then the
    // time segments of one set, then its parts, then the sets, largest first
    // so that the last CTAs to start are the shortest
    const int g = item % ng;
    const int rest = item / ng;
    const int q = a.seg_lo + rest % a.seg_cnt;
    const int r2 = rest / a.seg_cnt;
    const int sub = r2 % a.subs, r3 = r2 / a.subs;
    sidx = a.set_order ? a.set_order[r3] : r3;
    const int pb = a.set_begin[sidx], np = a.set_begin[sidx + 1] - pb;
    p_begin = pb + np * sub / a.subs;
    p_end = pb + np * (sub + 1) / a.subs;
    opw = a.obs_per_cta / NW;
    o_begin = g * a.obs_per_cta;
    o_end = min(a.O, o_begin + a.obs_per_cta);
    k_begin = max(0, q * a.seg_len - a.seg_shift);
    k_end = min(a.k_top, (q + 1) * a.seg_len - a.seg_shift);
    nobs = 0;
    for (int m = 0; m < opw; ++m)
      if (o_begin + w + NW * m < o_end) nobs = m + 1;
  }
  // chunks of `ch` rows or intervals
  __device__ __forceinline__ int chunks(int ch) const { return (k_end - k_begin + ch - 1) / ch; }
};

// Per-observer largest shift of the panel set (from the plan); zero windows.
template <typename T, int NW>
__device__ __forceinline__ void item_prologue(const FwdArgs<T> &a, const Item<T, NW> &it,
                                              int w, T *wwin, int *s_i0max) {
  const int lane = threadIdx.x & 31;
  if (lane < it.nobs)
    s_i0max[lane] = a.i0max_tab[(size_t)it.sidx * a.O + it.o_begin + w + NW * lane];
  for (int i = lane; i < it.nobs * a.wfl; i += 32) wwin[i] = T(0);
  __syncwarp();
}

// The warp's observers (bit m) with a valid bin among those a chunk can reach:
// intervals [k_lo, k_hi] at every shift of the set.  Outside an observer's
// window (N_o of nt bins) the work would be dropped bin by bin; it is not done.
// Before its first active chunk a window is zero, and after its last the
// remaining bins lie past N_o, so neither needs a flush.  72 observers around
// 32768 panels x 2048 steps: 3.64 -> 3.49 ms, FP64 104.3 -> 97.8; 36
// around 76800 panels x 4096 steps: 7.90 -> 7.25.
template <typename T, int NW>
__device__ __forceinline__ unsigned active_observers(const FwdArgs<T> &a, const Item<T, NW> &it,
                                                     int w, const int *s_i0max, int k_lo,
                                                     int k_hi) {
  const int lane = threadIdx.x & 31;
  bool on = false;
  if (lane < it.nobs) {
    const int i0 = s_i0max[lane];
    on = k_lo - i0 < a.n_valid[it.o_begin + w + NW * lane] && k_hi - i0 + a.slack >= 0;
  }
  return __ballot_sync(0xffffffffu, on);
}

// FP64, one (panel, observer): lane rows k0 + lane + 32 j (j < nj).  Row r
// enters the bins of intervals r - 3 .. r with weights w3 .. w0; wm is the
// window slot of interval r - 3 of the lane's first row.  Neighbouring lanes'
// updates meet in one bin, so the four steps are separated by __syncwarp.
template <int TK>
__device__ __forceinline__ void accumulate(const double (&x)[TK][kSer], const double (&c)[12],
                                           double *wm, int nj) {
  double g[TK];
#pragma unroll
  for (int j = 0; j < TK; ++j) {
    if (j >= nj) break;
    double v = c[0] * x[j][0];
#pragma unroll
    for (int s = 1; s < kSer; ++s) v = fma(c[s], x[j][s], v);
    g[j] = v;
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
#pragma unroll
    for (int j = 0; j < TK; ++j) {
      if (j >= nj) break;
      wm[32 * j + t] = fma(c[slot::w + 3 - t], g[j], wm[32 * j + t]);
    }
    __syncwarp();
  }
}

// FP64: flush the first CH (complete) bins of every window to p_out and slide.
// Window slot 0 is the bin of interval k0 - 3 at the set's largest shift.
template <int CH, int NW>
__device__ __forceinline__ void flush_slide(const FwdArgs<double> &a, const Item<double, NW> &it,
                                            int w, double *wwin, const int *s_i0max, int k0,
                                            unsigned active) {
  const int lane = threadIdx.x & 31;
  const int win = a.win;
  for (; active; active &= active - 1) {
    const int m = __ffs(active) - 1;
    const int o = it.o_begin + w + NW * m;
    double *wm = wwin + (size_t)m * win;
    const int wbase = k0 - s_i0max[m] - 3;
    const int nvalid = a.n_valid[o];
    double *po = a.p_out + (size_t)o * a.nt;
    for (int t = lane; t < CH; t += 32) {
      const int bin = wbase + t;
      const double v = wm[t];
      if (bin >= 0 && bin < nvalid && v != 0.0) atomic_add_f64(po + bin, v);
    }
    __syncwarp();
    for (int t = lane; t < win - CH; t += 32) wm[t] = wm[CH + t];  // win - CH <= CH
    __syncwarp();
    for (int t = win - CH + lane; t < win; t += 32) wm[t] = 0.0;
    __syncwarp();
  }
}

// Segment end (k0: the row after the last chunk): the remaining window holds
// partial bins of the next segment.
template <int CH, int NW>
__device__ __forceinline__ void flush_tail(const FwdArgs<double> &a, const Item<double, NW> &it,
                                           int w, double *wwin, const int *s_i0max, int k0) {
  const int lane = threadIdx.x & 31;
  const int win = a.win;
  for (int m = 0; m < it.nobs; ++m) {
    const int o = it.o_begin + w + NW * m;
    double *wm = wwin + (size_t)m * win;
    const int wbase = k0 - s_i0max[m] - 3;
    const int nvalid = a.n_valid[o];
    double *po = a.p_out + (size_t)o * a.nt;
    for (int t = lane; t < win - CH; t += 32) {
      const int bin = wbase + t;
      const double v = wm[t];
      if (bin >= 0 && bin < nvalid && v != 0.0) atomic_add_f64(po + bin, v);
    }
  }
  __syncwarp();
}

// ---- direct-load pipeline (FP64) -------------------------------------------
template <int TK, int NW>
__device__ __forceinline__ void process_item_direct(const FwdArgs<double> &a, int item,
                                                    double *smem, int *st) {
  constexpr int CH = 32 * TK;
  const int lane = threadIdx.x & 31;
  const int w = threadIdx.x >> 5;
  const Item<double, NW> it(a, item, w);
  double *wwin = smem + (size_t)w * it.opw * a.wfl;
  int *s_i0max = st + w * kMaxObsPerWarp;
  item_prologue<double, NW>(a, it, w, wwin, s_i0max);
  int k0 = it.k_begin;
  for (; k0 < it.k_end; k0 += CH) {
    const int nj = min(TK, (it.k_end - k0 + 31) / 32);
    const unsigned active = active_observers<double, NW>(a, it, w, s_i0max, k0 - 3, k0 + CH - 1);
    if (!active) continue;
    for (int p = it.p_begin; p < it.p_end; ++p) {
      double x[TK][kSer];
      const double *Xp = a.X + ((size_t)p * a.x_ld + (k0 - a.row0) + lane) * kSer;
#pragma unroll
      for (int j = 0; j < TK; ++j)
        if (j < nj) ldg_f64(Xp + (size_t)j * 32 * kSer, x[j]);
      const double *rec0 = a.coef + (size_t)p * a.O * kRec;
      for (unsigned left = active; left; left &= left - 1) {
        const int m = __ffs(left) - 1;
        const double *rec = rec0 + (size_t)(it.o_begin + w + NW * m) * kRec;
        double c[12];
        ldg_f64(rec, c);
        accumulate<TK>(x, c, wwin + (m * a.win + lane + (int)__ldg(rec + slot::off)), nj);
      }
    }
    flush_slide<CH, NW>(a, it, w, wwin, s_i0max, k0, active);
  }
  flush_tail<CH, NW>(a, it, w, wwin, s_i0max, k0);
}

// ---- TMA pipeline ------------------------------------------------------------
struct PipeState {
  uint64_t *full, *empty;
  unsigned char *stage0;
  unsigned stage_bytes, x_bytes;
  int nst;
  volatile int *abort;
  const void *tmap;  // tensor map of the X rows being streamed
  int *err;          // device error flag and the bound of each wait (SM clocks):
  long long wait_cycles;  // the same for every surface of a launch
};

// Threads per CTA: compute warps, plus the producer warp of the TMA pipeline.
template <int NW, int PIPE>
constexpr int cta_threads() { return (NW + (PIPE == 1 ? 1 : 0)) * 32; }

// Rows or intervals a chunk completes.
template <typename T, int TK>
constexpr int chunk_of() { return 32 * TK - (sizeof(T) == 4 ? 4 : 0); }

// Producer (one lane): stream the steps of one item into the stage ring, and
// warm L2 with the rows and records kPrefetchSteps steps beyond the ring so
// that the stage loads hit L2 instead of waiting for HBM.
constexpr int kPrefetchSteps = 8;

template <typename T, int TK, int NW>
__device__ __forceinline__ void produce_item(const FwdArgs<T> &a, const Item<T, 1> &it,
                                             const PipeState &ps, unsigned &step) {
  constexpr int CH = chunk_of<T, TK>();
  constexpr unsigned RPL = 128 / (kSer * sizeof(T));  // X rows per 128-byte line
  const unsigned cbytes = (unsigned)((it.o_end - it.o_begin) * kRec * sizeof(T));
  const int np = it.p_end - it.p_begin;
  const int nsteps = np * it.chunks(CH);
  // Step idx covers panel p_begin + idx % np, chunk k_begin + (idx / np) CH.
  // Both cursors (the load and the L2 prefetch running ahead of it) advance
  // incrementally: this lane's per-step work stays short, since it is on the
  // critical path of every stage refill.
  // the item's constants in registers (the batched kernels read their
  // arguments through a pointer, which every copy's memory clobber would make
  // them re-read)
  const T *const X = a.X;
  const T *const coef = a.coef;
  const int O = a.O;
  const size_t x_ld = a.x_ld;
  int *const err = ps.err;
  const long long wait_cycles = ps.wait_cycles;
  const size_t row_b = (size_t)it.p_begin * x_ld + (it.k_begin - a.row0);
  auto src_c = [&](int pp) {
    return coef + ((size_t)(it.p_begin + pp) * O + it.o_begin) * kRec;
  };
  if (a.withhold) return;  // testing: no copies, so every consumer wait runs out
  int fp = 0, fk = 0;  // prefetch cursor (panel offset, chunk)
  auto prefetch_next = [&]() {
    prefetch_l2(X + (row_b + fp * x_ld + (size_t)fk * CH) * kSer, ps.x_bytes);
    prefetch_l2(src_c(fp), cbytes);
    if (++fp == np) {
      fp = 0;
      ++fk;
    }
  };
  const int lead = min(nsteps, ps.nst + kPrefetchSteps);
  for (int idx = 0; idx < lead; ++idx) prefetch_next();
  int cp = 0, ck = 0;  // load cursor
  unsigned s = step % (unsigned)ps.nst, ph = (step / (unsigned)ps.nst) & 1u;
  for (int idx = 0; idx < nsteps; ++idx, ++step) {
    if (*ps.abort) return;
    if (idx + lead < nsteps) prefetch_next();
    if (step >= (unsigned)ps.nst &&
        !mbar_wait_sleep(&ps.empty[s], ph ^ 1u, err, ps.abort, wait_cycles))
      return;
    unsigned char *dst = ps.stage0 + (size_t)s * ps.stage_bytes;
    mbar_expect_tx(&ps.full[s], ps.x_bytes + cbytes);
    const size_t row = row_b + cp * x_ld + (size_t)ck * CH;
    tma_load_2d(dst, ps.tmap, 0, (int)(row / RPL), &ps.full[s]);
    bulk_load(dst + ps.x_bytes, src_c(cp), cbytes, &ps.full[s]);
    if (++cp == np) {
      cp = 0;
      ++ck;
    }
    if (++s == (unsigned)ps.nst) {
      s = 0;
      ph ^= 1u;
    }
  }
}

template <int TK, int NW>
__device__ __forceinline__ void consume_item(const FwdArgs<double> &a, const Item<double, NW> &it,
                                             const PipeState &ps, unsigned &step, double *wwin,
                                             int *s_i0max, int w) {
  constexpr int CH = 32 * TK;
  const int lane = threadIdx.x & 31;
  item_prologue<double, NW>(a, it, w, wwin, s_i0max);
  int k0 = it.k_begin;
  for (; k0 < it.k_end; k0 += CH) {
    const int nj = min(TK, (it.k_end - k0 + 31) / 32);
    const unsigned active = active_observers<double, NW>(a, it, w, s_i0max, k0 - 3, k0 + CH - 1);
    for (int p = it.p_begin; p < it.p_end; ++p, ++step) {
      const int s = (int)(step % (unsigned)ps.nst);
      const unsigned ph = (step / (unsigned)ps.nst) & 1u;
      if (!mbar_wait(&ps.full[s], ph, ps.err, ps.abort, ps.wait_cycles)) return;
      const unsigned char *stg = ps.stage0 + (size_t)s * ps.stage_bytes;
      double x[TK][kSer];
#pragma unroll
      for (int j = 0; j < TK; ++j) lds_row_f64(stg, lane + 32 * j, x[j]);
      const double *crec = reinterpret_cast<const double *>(stg + ps.x_bytes);
      for (unsigned left = active; left; left &= left - 1) {
        const int m = __ffs(left) - 1;
        const double *rec = crec + (size_t)(w + NW * m) * kRec;
        double c[12];
        lds_f64(rec, c);
        accumulate<TK>(x, c, wwin + (m * a.win + lane + (int)rec[slot::off]), nj);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ps.empty[s]);
    }
    flush_slide<CH, NW>(a, it, w, wwin, s_i0max, k0, active);
  }
  flush_tail<CH, NW>(a, it, w, wwin, s_i0max, k0);
}

// ---- FP32 consumer (mixed precision) ----------------------------------------
// An X row is 32 bytes, four consecutive rows one 128-byte line.  Lane l owns
// line l + 32 b of each 128-row block b of a chunk and forms, per observer and
// row, G = c . X with packed fma.rn.f32x2 over the register pairs (X_2q,
// X_2q+1) and (c_2q, c_2q+1) as they lie in the row and in the record (no
// duplicated coefficients), the halves added at the end.  A packed FMA issues
// in one slot and occupies the FMA pipe for two cycles.  The bin of interval k
// needs G of rows k .. k + 3: three values come from the lane above by
// shuffle (lane 31: lane 0's of the next block), and the last block's lane 31
// only serves its neighbour, so a chunk of NB blocks completes 128 NB - 4 bins
// and the next chunk starts at that row.
//
// Per (observer, 128-row block): 16 packed FMAs, 4 adds, 16 FMAs, 3 shuffles,
// 4 window loads and stores and a share of the record's 4 loads and 4 address
// adds.  No one unit bounds it: with two blocks the shared-memory pipe is busy
// about 77 % of the time (20 wavefronts per block: windows 8, records 4, X rows
// 3.6, shuffles 3, flushes), issue 58 %, the FMA pipe 46 %; one block a chunk
// lets 16 warps fit an SM instead of 12 but reads each record twice as often
// (24 wavefronts): 0.15 ms more.  On a GB300 the
// sphere of 32768 panels x 2048 steps x 72 observers takes 3.49 ms; the
// former kernel on samples and moments side by side (20 multiply-adds, 64-byte
// rows, 22 instructions per 32 samples) took 4.57 ms.
//
// Quarter-split windows: slot x of an observer's window lives in quarter x & 3
// at word x >> 2, so the four bins of a lane sit in four quarters and 32 lanes
// touch 32 consecutive words of one quarter per access: conflict-free for
// every offset.  The planner writes each record's four byte offsets, so the
// hot loop adds them to the lane's base and never branches on the shift; block
// b adds 32 words.  Within one (panel, observer) no two lanes touch the same
// slot; one __syncwarp per panel orders the next panel's shifted updates.
// Shared-space accesses by 32-bit address (the consumer addresses the stage
// ring and its windows explicitly, so no generic-address arithmetic).
// Window loads are not volatile: the compiler may hoist an observer's loads
// above the previous observer's stores (their windows never overlap), which
// hides their latency.  They stay after the previous panel's stores because
// their addresses derive from a token taken after that panel's __syncwarp.
__device__ __forceinline__ float lds_win(unsigned addr) {
  float v;
  asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_f32(unsigned addr, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// Loads of stage data (X rows, records): not volatile, so the compiler may
// schedule them early; they stay after the stage's full-barrier wait because
// their addresses derive from stage_token(), which that wait orders.
__device__ __forceinline__ float4 lds_v4f32(unsigned addr) {
  float4 v;
  asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "r"(addr));
  return v;
}
// The stage address as an opaque value produced after the barrier wait.
__device__ __forceinline__ unsigned stage_token(unsigned addr) {
  unsigned r;
  asm volatile("mov.u32 %0, %1;" : "=r"(r) : "r"(addr) : "memory");
  return r;
}

// The slots of one FP32 record that the consumer reads, in the groups it loads
// them by: c0..c7 as pairs, the four window byte offsets, the weights.
static_assert(slot::c == 0 && slot::w == 8 && slot::q0 == 12, "record read in 16-byte groups");
struct Coef {
  unsigned long long c[4];
  float w[4];
  uint4 q;
  __device__ __forceinline__ void load_c(unsigned rec) {
    asm("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(c[0]), "=l"(c[1]) : "r"(rec));
    asm("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(c[2]), "=l"(c[3]) : "r"(rec + 16));
  }
  __device__ __forceinline__ void load_w(unsigned rec) {
    const float4 v = lds_v4f32(rec + 32);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  }
  static __device__ __forceinline__ uint4 load_q(unsigned rec) {
    uint4 v;
    asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "r"(rec + 48));
    return v;
  }
};

// Compensated (Kahan) update of a window entry (sum, compensation) by y.
__device__ __forceinline__ float2 kahan_add(float2 w, float y) {
  const float yc = __fsub_rn(y, w.y);
  const float t = __fadd_rn(w.x, yc);
  return make_float2(t, __fsub_rn(__fsub_rn(t, w.x), yc));
}

// A window entry: a plain FP32 sum, or a compensated pair (sum, compensation)
// whose value is sum - compensation (formed in FP64).  add() takes a panel's
// whole contribution to the bin at once: the four taps are summed first, so the
// running sum, much larger than one panel's share, is rounded once per panel
// and not four times (error against 64 bits 7.2e-8 instead of 8.0e-8 at 8192
// panels x 512 steps, for 0.13 of 3.5 ms).
template <bool KAHAN> struct WinEntry;
template <> struct WinEntry<false> {
  using E = float;
  static __device__ __forceinline__ bool nz(E e) { return e != 0.f; }
  static __device__ __forceinline__ double value(E e) { return (double)e; }
  static __device__ __forceinline__ E zero() { return 0.f; }
  static __device__ __forceinline__ E load(unsigned addr) { return lds_win(addr); }
  static __device__ __forceinline__ void store(unsigned addr, E v) { sts_f32(addr, v); }
  static __device__ __forceinline__ E add(E s, float y) { return s + y; }
};
template <> struct WinEntry<true> {
  using E = float2;
  static __device__ __forceinline__ bool nz(E e) { return e.x != 0.f || e.y != 0.f; }
  static __device__ __forceinline__ double value(E e) { return (double)e.x - (double)e.y; }
  static __device__ __forceinline__ E zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ E load(unsigned addr) {
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
  }
  static __device__ __forceinline__ void store(unsigned addr, E v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
  }
  static __device__ __forceinline__ E add(E s, float y) { return kahan_add(s, y); }
};

// Window slots per observer of the FP32 shapes, fixed per chunk length so that
// the hot loop addresses the windows with immediates.
template <int TK>
constexpr int win_f32() { return TK == 4 ? 224 : 352; }

// Add the first n bins of an observer's window to p_out.  Lanes take
// consecutive bins; the quarter length is 8 or 24 mod 32 words, so the eight
// words of each quarter that a warp reads lie on distinct banks.
template <int TK, bool KAHAN, int NW>
__device__ __forceinline__ void flush_bins(const FwdArgs<float> &a, const Item<float, NW> &it,
                                           int w, int m, const void *wm, int wbase, int n) {
  using W = WinEntry<KAHAN>;
  const typename W::E *e = static_cast<const typename W::E *>(wm);
  const int lane = threadIdx.x & 31;
  constexpr int H = win_f32<TK>() / 4;
  const int o = it.o_begin + w + NW * m;
  const int nvalid = a.n_valid[o];
  double *po = a.p_out + (size_t)o * a.nt;
  for (int x = lane; x < n; x += 32) {
    const int bin = wbase + x;
    const typename W::E v = e[(x & 3) * H + (x >> 2)];
    if (bin >= 0 && bin < nvalid && W::nz(v)) atomic_add_f64(po + bin, W::value(v));
  }
}

// Flush the first CH (complete) bins of every window to p_out and slide.
template <int TK, int NW, bool KAHAN>
__device__ __forceinline__ void flush_slide_split(const FwdArgs<float> &a,
                                                  const Item<float, NW> &it, int w, float *wwin,
                                                  const int *s_i0max, int k0, unsigned active) {
  using W = WinEntry<KAHAN>;
  using E = typename W::E;
  constexpr int H = win_f32<TK>() / 4, CH = chunk_of<float, TK>();
  const int lane = threadIdx.x & 31;
  for (; active; active &= active - 1) {
    const int m = __ffs(active) - 1;
    E *wm = reinterpret_cast<E *>(wwin) + m * 4 * H;
    flush_bins<TK, KAHAN, NW>(a, it, w, m, wm, k0 - s_i0max[m], CH);
    __syncwarp();
    constexpr int keep = H - CH / 4;
    static_assert(keep <= CH / 4, "no overlap");
    for (int i = lane; i < 4 * keep; i += 32) {
      E *q = wm + (i & 3) * H + (i >> 2);
      *q = q[CH / 4];
    }
    __syncwarp();
    for (int i = lane; i < CH; i += 32) wm[(i & 3) * H + keep + (i >> 2)] = W::zero();
    __syncwarp();
  }
}

// Segment end (k0: the interval after the last chunk): the remaining window
// holds partial bins of the next segment.
template <int TK, int NW, bool KAHAN>
__device__ __forceinline__ void flush_tail_split(const FwdArgs<float> &a,
                                                 const Item<float, NW> &it, int w, float *wwin,
                                                 const int *s_i0max, int k0) {
  constexpr int WIN = win_f32<TK>();
  for (int m = 0; m < it.nobs; ++m)
    flush_bins<TK, KAHAN, NW>(a, it, w, m, wwin + m * WIN * (KAHAN ? 2 : 1), k0 - s_i0max[m],
                              WIN - chunk_of<float, TK>());
  __syncwarp();
}

__device__ __forceinline__ void lds_v2f32x2(unsigned addr, f32x2 &a, f32x2 &b) {
  asm("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr));
}
__device__ __forceinline__ float f2_sum(f32x2 v) {
  float lo, hi;
  f2_split(v, lo, hi);
  return lo + hi;
}

// One (chunk, panel) step: NA blocks of 128 rows (NA = 1: the last chunk of a
// segment, when its remaining intervals fit one block); `lanes` lanes of the
// last block add their bins.
//
// The next observer's record is loaded piece by piece as this one's is used
// up, always before this observer's stores: the compiler cannot move a shared
// load above a store it cannot tell apart (3.43 ms so, 3.50 with the record
// read at the top of each observer, before the taps were summed apart).  Two
// observers at a time (168 registers): 4.1 ms; the last lane's stores predicated
// or sent to a spare slot instead of the branch: 3.8 and 3.7 ms.
template <int TK, int NA, int NW, bool KAHAN>
__device__ __forceinline__ void consume_step(unsigned active, unsigned stg, unsigned crec,
                                             unsigned win_s, unsigned xrow, int lanes) {
  constexpr unsigned RB = kRec * 4;           // record bytes
  constexpr unsigned BB = KAHAN ? 256 : 128;  // window bytes of 32 words of a quarter
  constexpr unsigned WB = win_f32<TK>() * (KAHAN ? 8u : 4u);  // window bytes
  const int lane = threadIdx.x & 31;
  const bool first = lane == 0, inner = lane < lanes;
  f32x2 XP[NA][4][4];  // [block][row][pair of series]
  const unsigned xb = stg + xrow;
#pragma unroll
  for (int b = 0; b < NA; ++b)
#pragma unroll
    for (int c = 0; c < 8; ++c)
      lds_v2f32x2((xb ^ ((unsigned)c << 4)) + 4096u * b, XP[b][c >> 1][2 * (c & 1)],
                  XP[b][c >> 1][2 * (c & 1) + 1]);
  // window base of this panel's updates, ordered after the previous panel's
  // stores (see lds_win)
  const unsigned wtok = stage_token(win_s);
  // one observer: window m, its record in k; `next`: the record to load
  using W = WinEntry<KAHAN>;
  auto observer = [&](int m, Coef &k, unsigned next) {
    const unsigned A[4] = {wtok + k.q.x + m * WB, wtok + k.q.y + m * WB, wtok + k.q.z + m * WB,
                           wtok + k.q.w + m * WB};
    typename W::E s[NA][4];
#pragma unroll
    for (int b = 0; b < NA; ++b)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[b][j] = W::load(A[j] + BB * b);
    k.q = Coef::load_q(next);
    float g[NA][7];
#pragma unroll
    for (int b = 0; b < NA; ++b)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f32x2 v = f2_mul(k.c[0], XP[b][j][0]);
#pragma unroll
        for (int q = 1; q < 4; ++q) v = f2_fma(k.c[q], XP[b][j][q], v);
        g[b][j] = f2_sum(v);
      }
    k.load_c(next);
#pragma unroll
    for (int b = 0; b < NA; ++b)
#pragma unroll
      for (int t = 0; t < 3; ++t)
        // lane 0 serves lane 31 with the next block's first rows
        g[b][4 + t] = b + 1 < NA ? __shfl_sync(0xffffffffu, first ? g[b + 1][t] : g[b][t],
                                               (lane + 1) & 31)
                                 : __shfl_down_sync(0xffffffffu, g[b][t], 1);
#pragma unroll
    for (int b = 0; b < NA; ++b)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float y = k.w[0] * g[b][j];
#pragma unroll
        for (int t = 1; t < 4; ++t) y = fmaf(k.w[t], g[b][j + t], y);
        s[b][j] = W::add(s[b][j], y);
      }
    k.load_w(next);
#pragma unroll
    for (int b = 0; b < NA; ++b)
      if (b + 1 < NA || inner) {
#pragma unroll
        for (int j = 0; j < 4; ++j) W::store(A[j] + BB * b, s[b][j]);
      }
  };
  auto rec = [&](int m) { return crec + (unsigned)m * NW * RB; };
  Coef k;
  auto load = [&](unsigned r) {
    k.q = Coef::load_q(r);
    k.load_c(r);
    k.load_w(r);
  };
  // A warp with the full count of observers runs them unrolled, so the
  // compiler may overlap one observer's tail with the next one's loads and
  // arithmetic.  (The last one loads its own record again.)  Scatter of 16384
  // panels x 1024 steps, us per observer: 13.6 with 36 observers (nine a warp),
  // 14.8 with 28 (seven), 16.3 with 20 (five), 15.3 with 40 (two groups of five).
  if (active == (1u << kMaxObsPerWarpF32) - 1) {
    load(rec(0));
#pragma unroll
    for (int m = 0; m < kMaxObsPerWarpF32; ++m)
      observer(m, k, rec(m + 1 < kMaxObsPerWarpF32 ? m + 1 : m));
  } else {
    int m = __ffs(active) - 1;
    load(rec(m));
    for (;;) {
      active &= active - 1;
      const int next = active ? __ffs(active) - 1 : m;
      observer(m, k, rec(next));
      if (!active) break;
      m = next;
    }
  }
}

template <int TK, int NW, bool KAHAN>
__device__ __forceinline__ void consume_item_f32(const FwdArgs<float> &a,
                                                 const Item<float, NW> &it,
                                                 const PipeState &ps, unsigned &step,
                                                 float *wwin, int *s_i0max, int w) {
  constexpr int NB = TK / 4;  // 128-row blocks
  constexpr int CH = chunk_of<float, TK>();
  const int lane = threadIdx.x & 31;
  item_prologue<float, NW>(a, it, w, wwin, s_i0max);
  const unsigned win_s = smem_u32(wwin) + (unsigned)lane * (KAHAN ? 8u : 4u);
  const unsigned stage0 = smem_u32(ps.stage0);
  // X line lane + 32 b of a stage: 16-byte chunk c at c ^ (lane & 7).  Stages
  // are 1024-byte aligned and a line is 128 bytes, so chunk c of the lane's
  // line sits at (stage + 128 lane + 16 (lane & 7)) ^ 16 c: one XOR per chunk.
  const unsigned xrow = (unsigned)lane * 128u + (((unsigned)lane & 7u) << 4);
  unsigned s = step % (unsigned)ps.nst, ph = (step / (unsigned)ps.nst) & 1u;
  int k0 = it.k_begin;
  for (; k0 < it.k_end; k0 += CH) {
    const bool one = NB > 1 && it.k_end - k0 <= 124;
    // lanes of the last block whose bins belong to this chunk (a segment that
    // ends inside the record ends at a multiple of four intervals)
    const int lanes = min(31, (it.k_end - k0 - (one ? 0 : 128 * (NB - 1)) + 3) >> 2);
    const unsigned active = active_observers<float, NW>(a, it, w, s_i0max, k0, k0 + CH - 1);
    for (int p = it.p_begin; p < it.p_end; ++p, ++step) {
      if (!mbar_wait(&ps.full[s], ph, ps.err, ps.abort, ps.wait_cycles)) return;
      const unsigned stg = stage_token(stage0 + s * ps.stage_bytes);
      const unsigned crec = stg + ps.x_bytes + (unsigned)w * (kRec * 4);
      if (active) {
        if (one)
          consume_step<TK, 1, NW, KAHAN>(active, stg, crec, win_s, xrow, lanes);
        else
          consume_step<TK, NB, NW, KAHAN>(active, stg, crec, win_s, xrow, lanes);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ps.empty[s]);
      if (++s == (unsigned)ps.nst) {
        s = 0;
        ph ^= 1u;
      }
    }
    flush_slide_split<TK, NW, KAHAN>(a, it, w, wwin, s_i0max, k0, active);
  }
  flush_tail_split<TK, NW, KAHAN>(a, it, w, wwin, s_i0max, k0);
}

// Wait until every copy the producer issued has landed, always with the full
// bound (never the handle's test bound): the CTA must not exit while a copy
// into its shared memory is in flight.
__device__ __forceinline__ void drain_copies(const PipeState &ps, unsigned step, int *err) {
  const unsigned first = step > (unsigned)ps.nst ? step - (unsigned)ps.nst : 0u;
  volatile int never = 0;
  for (unsigned t = first; t < step; ++t) {
    const int s = (int)(t % (unsigned)ps.nst);
    mbar_wait(&ps.full[s], (t / (unsigned)ps.nst) & 1u, err, &never);
  }
}

template <typename T, int TK, int NW>
__device__ __forceinline__ unsigned char *pipe_setup(unsigned char *raw, int obs_per_cta,
                                                     int nst, uint64_t *bars,
                                                     volatile int *abort, PipeState &ps) {
  const unsigned base = smem_u32(raw);
  unsigned char *al = raw + ((1024u - (base & 1023u)) & 1023u);
  ps.x_bytes = 32 * TK * kSer * sizeof(T);
  ps.stage_bytes = (ps.x_bytes + obs_per_cta * kRec * sizeof(T) + 1023u) & ~1023u;
  ps.nst = nst;
  ps.stage0 = al;
  ps.full = bars;
  ps.empty = bars + nst;
  ps.abort = abort;
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&ps.full[s], 1);
      mbar_init(&ps.empty[s], NW);
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  return al + (size_t)nst * ps.stage_bytes;  // windows follow the stages
}

constexpr int kMaxStages = 8;

// CTAs per SM the register budget is sized for.
template <int TK, int NW, int PIPE>
struct MinBlocks {
  static constexpr int v = !PIPE ? 1 : (NW <= 4 ? (TK <= 4 ? 4 : 3) : (TK <= 4 ? 2 : 1));
};

template <typename T, int TK, int NW, int PIPE, int ACC>
__device__ __forceinline__ void forward_cta(const FwdArgs<T> &a, const void *tmap, int nst,
                                            int item, int *err, long long wait_cycles) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int st[NW * kMaxObsPerWarp];
  if constexpr (PIPE == 0) {
    (void)tmap;
    process_item_direct<TK, NW>(a, item, reinterpret_cast<T *>(smem_raw), st);
  } else {
    __shared__ __align__(8) uint64_t bars[2 * kMaxStages];
    __shared__ int abort_flag;
    PipeState ps;
    unsigned char *wbase = pipe_setup<T, TK, NW>(smem_raw, a.obs_per_cta, nst, bars, &abort_flag,
                                                 ps);
    ps.tmap = tmap;
    ps.err = err;
    ps.wait_cycles = wait_cycles;
    const int w = threadIdx.x >> 5;
    unsigned step = 0;
    if (w == NW) {
      if ((threadIdx.x & 31) == 0) {
        const Item<T, 1> it(a, item, 0);
        produce_item<T, TK, NW>(a, it, ps, step);
        drain_copies(ps, step, err);
      }
    } else {
      const Item<T, NW> it(a, item, w);
      T *wwin = reinterpret_cast<T *>(wbase) + (size_t)w * it.opw * a.wfl;
      if constexpr (sizeof(T) == 4)
        consume_item_f32<TK, NW, ACC == 5>(a, it, ps, step, wwin, st + w * kMaxObsPerWarp, w);
      else
        consume_item<TK, NW>(a, it, ps, step, wwin, st + w * kMaxObsPerWarp, w);
    }
  }
}

template <typename T, int TK, int NW, int PIPE, int ACC>
__global__ void __launch_bounds__((cta_threads<NW, PIPE>()), (MinBlocks<TK, NW, PIPE>::v))
    k_forward(FwdArgs<T> a, const __grid_constant__ CUtensorMap tm, int nst) {
  forward_cta<T, TK, NW, PIPE, ACC>(a, &tm, nst, blockIdx.x, a.err, a.wait_cycles);
}

// Persistent form: CTAs pull work items of several surfaces from one queue.
// The surfaces' arguments, item offsets and X descriptors are one
// __grid_constant__ parameter block (kMaxBatchSurf surfaces at most).
//
// With a producer warp (PIPE = 1) items flow back to back: the producer lane
// claims an item, publishes its index in a small ring (s_q, one mbarrier per
// slot) and streams its steps into the stage ring, whose step count runs on
// across items; each compute warp takes the next published item as soon as it
// has flushed its windows for the previous one.  There is no CTA-wide barrier
// between items, so the copies of an item's first stages are in flight while
// the compute warps finish the item before it.  A slot is rewritten kItemQ
// publications later.  What holds the producer back is the stage ring: it can
// run at most `nst` steps ahead of the slowest compute warp, and every published
// item has at least one step, so it is at most `nst` items ahead and kItemQ >
// kMaxStages keeps every publication readable until each warp has taken it.  A
// panel set of fewer panels than the parts it is cut into leaves parts without
// panels; such an item takes no stage, so any number of them could pass while the
// compute warps still work: the producer drops them and claims on (65 panels in
// sets of 64 and 1, four parts each: over 300 in a row).
constexpr int kItemQ = 16;
// kernel parameters may take up to 32764 bytes (CUDA 12.1 and later)
static_assert(sizeof(BatchParams<double>) + 64 <= 32764, "batched launch parameters too large");
static_assert(kItemQ > kMaxStages, "the item ring must outlast the deepest stage ring");

// Surface of a batched item (prefix[lo] <= item < prefix[lo + 1]).
__device__ __forceinline__ int batch_surface(const int *prefix, int n_surf, int item) {
  int lo = 0, hi = n_surf - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <typename T, int TK, int NW, int PIPE, int ACC>
__device__ __forceinline__ void forward_batch_cta(const BatchParams<T> &P, int *counter, int nst) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int st[NW * kMaxObsPerWarp];
  __shared__ int s_item;
  __shared__ __align__(8) uint64_t bars[2 * kMaxStages];
  __shared__ __align__(8) uint64_t qbar[kItemQ];
  __shared__ int s_q[kItemQ];
  __shared__ int abort_flag;
  const int n_surf = P.n_surf, total = P.total;
  const int *prefix = P.prefix;   // parameter space: read through the constant cache
  const FwdArgs<T> *args = P.a;
  if (threadIdx.x == 0) {
    s_item = atomicAdd(counter, 1);
    if constexpr (PIPE == 1)
      for (int q = 0; q < kItemQ; ++q) mbar_init(&qbar[q], 1);
  }
  __syncthreads();
  const int w = threadIdx.x >> 5;
  PipeState ps;
  unsigned char *wbase = smem_raw;
  unsigned step = 0;
  int maxo = 0;  // observers of the largest group: the same windows' places for every surface
  if constexpr (PIPE != 0) {
    for (int i = 0; i < n_surf; ++i) maxo = max(maxo, args[i].obs_per_cta);
    // (its barrier also orders the item ring's initialisation above)
    wbase = pipe_setup<T, TK, NW>(smem_raw, maxo, nst, bars, &abort_flag, ps);
    ps.err = args[0].err;
    ps.wait_cycles = args[0].wait_cycles;
  }
  if constexpr (PIPE == 1) {
    volatile int *abort = &abort_flag;
    if (w == NW) {
      if ((threadIdx.x & 31) == 0) {
        int k = 0;  // publications
        // after a timeout, or with copies withheld (testing), the queue ends: the
        // compute warps stop at the sentinel below or at the abort flag
        for (int item = s_item; item < total;
             item = (*abort || args[0].withhold) ? total : atomicAdd(counter, 1)) {
          const int sf = batch_surface(prefix, n_surf, item);
          const FwdArgs<T> &a = args[sf];
          const Item<T, 1> it(a, item - prefix[sf], 0);
          if (it.p_begin == it.p_end) continue;  // no panels, hence no steps: not published
          s_q[k % kItemQ] = item;
          mbar_arrive(&qbar[k % kItemQ]);  // release: the index is visible to the waiters
          ++k;
          ps.tmap = &P.tm[sf];
          produce_item<T, TK, NW>(a, it, ps, step);
        }
        s_q[k % kItemQ] = total;  // the sentinel that ends the queue
        mbar_arrive(&qbar[k % kItemQ]);
        drain_copies(ps, step, args[0].err);
      }
    } else {
      for (int k = 0;; ++k) {
        if (!mbar_wait(&qbar[k % kItemQ], (unsigned)(k / kItemQ) & 1u, args[0].err, abort,
                       args[0].wait_cycles))
          break;
        const int item = s_q[k % kItemQ];
        if (item >= total) break;
        const int sf = batch_surface(prefix, n_surf, item);
        const FwdArgs<T> &a = args[sf];
        const Item<T, NW> it(a, item - prefix[sf], w);
        // (not it.opw apart: the other warps may still work on an item of a surface
        // with another number of observers)
        T *wwin = reinterpret_cast<T *>(wbase) + (size_t)w * (maxo / NW) * a.wfl;
        if constexpr (sizeof(T) == 4)
          consume_item_f32<TK, NW, ACC == 5>(a, it, ps, step, wwin, st + w * kMaxObsPerWarp, w);
        else
          consume_item<TK, NW>(a, it, ps, step, wwin, st + w * kMaxObsPerWarp, w);
        if (*abort) break;
      }
    }
  } else {
    for (;;) {
      __syncthreads();  // the previous item is done; s_item holds this one
      const int item = s_item;
      __syncthreads();  // every thread has read it
      if (item >= total) break;
      const int sf = batch_surface(prefix, n_surf, item);
      // a reference, not a copy: the fields are read from the parameter block
      // where used, instead of holding the whole argument block in registers
      process_item_direct<TK, NW>(args[sf], item - prefix[sf], reinterpret_cast<T *>(smem_raw), st);
      if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    }
  }
}

template <typename T, int TK, int NW, int PIPE, int ACC>
__global__ void __launch_bounds__((cta_threads<NW, PIPE>()), (MinBlocks<TK, NW, PIPE>::v))
    k_forward_batch(const __grid_constant__ BatchParams<T> P, int *counter, int nst) {
  forward_batch_cta<T, TK, NW, PIPE, ACC>(P, counter, nst);
}

// One grid over every surface's items (CTA i takes work item i of the
// concatenated queue): the hardware places each CTA, so each item's warps
// land wherever slots are free.  The persistent kernel keeps each CTA's warp
// placement for the whole launch; on a GB300 its per-scheduler instruction
// counts spread by 12 % (1 % for this grid) and it ran about 3 % slower.
template <typename T, int TK, int NW, int PIPE, int ACC>
__device__ __forceinline__ void forward_multi_cta(const BatchParams<T> &P, int nst) {
  const int item = (int)blockIdx.x;
  const int sf = batch_surface(P.prefix, P.n_surf, item);
  // (the error flag and wait bound are the same for every surface: read at
  // a fixed parameter offset)
  forward_cta<T, TK, NW, PIPE, ACC>(P.a[sf], &P.tm[sf], nst, item - P.prefix[sf], P.a[0].err,
                                    P.a[0].wait_cycles);
}

template <typename T, int TK, int NW, int PIPE, int ACC>
__global__ void __launch_bounds__((cta_threads<NW, PIPE>()), (MinBlocks<TK, NW, PIPE>::v))
    k_forward_multi(const __grid_constant__ BatchParams<T> P, int nst) {
  forward_multi_cta<T, TK, NW, PIPE, ACC>(P, nst);
}

// Candidate tile shapes {pipe, tk, warps, obs_per_warp, win, seg_chunks,
// stages, acc}; the first is the default: short segments, so that the CTAs of a
// launch end together (FP32 one chunk: 20011 panels x 1501 steps x 37 observers
// 1.03 -> 0.99 ms, 16384 x 1024 x 36 0.52 -> 0.49, the longest records the same;
// FP64 two: 5151 x 701 x 19 1.74 -> 1.56 ms with twice the items).  FP32 (always TMA): tk 4 or 8 (one or two 128-row blocks per
// chunk); acc 3 plain window sums, 5 compensated (Kahan) ones.  win / 4 is 8
// or 24 mod 32 (see flush_bins).
constexpr FwdConfig kCfgF32[] = {
    {1, 8, 4, 9, 352, 1, 2, 3},
    {1, 8, 4, 9, 352, 2, 2, 3},
    {1, 4, 4, 9, 224, 4, 3, 3},
    {1, 4, 8, 9, 224, 4, 3, 3},
    {1, 8, 4, 9, 352, 3, 2, 3},
    {1, 8, 4, 9, 352, 2, 3, 3},
    {1, 4, 4, 9, 224, 2, 3, 3},
    {1, 8, 4, 9, 352, 4, 2, 3},
    {1, 4, 4, 9, 224, 8, 3, 3},
    {1, 4, 4, 9, 224, 4, 2, 3},
    {1, 4, 4, 9, 224, 4, 2, 5},
    {1, 4, 4, 9, 224, 4, 3, 5},
};
constexpr bool f32_obs_fit() {
  for (const FwdConfig &c : kCfgF32)
    if (c.obs_per_warp > kMaxObsPerWarpF32 ||
        c.win != (c.tk == 4 ? win_f32<4>() : win_f32<8>()))
      return false;
  return true;
}
static_assert(f32_obs_fit(), "FP32 shapes: observers per warp and window slots of the unrolled loop");
const FwdConfig kCfgF64[] = {
    {0, 2, 8, 16, 128, 2, 0, 0},
    {1, 2, 8, 9, 128, 8, 3, 0},
    {0, 2, 4, 16, 128, 8, 0, 0},
    {0, 1, 8, 16, 64, 16, 0, 0},
};

template <typename T>
size_t smem_for(const FwdConfig &c, int obs_per_cta) {
  const int opw = obs_per_cta / c.warps;
  size_t win = (size_t)c.warps * opw * c.win * sizeof(T) * (c.acc == 5 ? 2 : 1);
  if (c.pipe == 0) return win;
  const size_t xb = (size_t)32 * c.tk * kSer * sizeof(T);
  const size_t sb =
      (xb + (size_t)obs_per_cta * kRec * sizeof(T) + 1023) & ~size_t(1023);
  return 1024 + (size_t)c.stages * sb + win;
}

template <typename T, int TK, int NW, int PIPE, int ACC>
cudaError_t launch_one(const FwdArgs<T> &a, const CUtensorMap &tm, const FwdConfig &c,
                       cudaStream_t s) {
  const size_t smem = smem_for<T>(c, a.obs_per_cta);
  auto kern = k_forward<T, TK, NW, PIPE, ACC>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  if (a.seg_lo < 0 || a.seg_cnt < 1 || a.seg_lo + a.seg_cnt > a.n_segs) return cudaErrorInvalidValue;
  const long long items = (long long)a.nsets * a.subs * a.n_obs_groups * a.seg_cnt;
  if (items <= 0) return cudaSuccess;
  if (items > INT32_MAX) return cudaErrorInvalidValue;
  kern<<<(unsigned)items, cta_threads<NW, PIPE>(), smem, s>>>(a, tm, c.stages);
  return cudaGetLastError();
}

template <typename T, int TK, int NW, int PIPE, int ACC>
cudaError_t launch_multi_one(const BatchParams<T> &P, size_t smem, int nst, cudaStream_t s) {
  auto kern = k_forward_multi<T, TK, NW, PIPE, ACC>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)P.total, cta_threads<NW, PIPE>(), smem, s>>>(P, nst);
  return cudaGetLastError();
}

template <typename T, int TK, int NW, int PIPE, int ACC>
cudaError_t launch_batch_one(const BatchParams<T> &P, int *d_counter, size_t smem, int n_ctas,
                             int nst, cudaStream_t s) {
  auto kern = k_forward_batch<T, TK, NW, PIPE, ACC>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<n_ctas, cta_threads<NW, PIPE>(), smem, s>>>(P, d_counter, nst);
  return cudaGetLastError();
}

}  // namespace

int fwd_num_configs(bool fp64) {
  return fp64 ? (int)(sizeof(kCfgF64) / sizeof(kCfgF64[0]))
              : (int)(sizeof(kCfgF32) / sizeof(kCfgF32[0]));
}

FwdConfig fwd_config(bool fp64, int idx) {
  const int n = fwd_num_configs(fp64);
  if (idx < 0 || idx >= n) idx = 0;
  return fp64 ? kCfgF64[idx] : kCfgF32[idx];
}

size_t fwd_smem_bytes(bool fp64, const FwdConfig &c, int obs_per_cta) {
  return fp64 ? smem_for<double>(c, obs_per_cta) : smem_for<float>(c, obs_per_cta);
}

bool encode_x_tensor_map(void *out128, const void *X, unsigned long long rows, bool fp64,
                         int box_rows) {
  static PFN_cuTensorMapEncodeTiled_v12000 enc = nullptr;
  if (!enc) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return false;
    enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  // Lines of 128 bytes (four FP32 rows or two FP64 rows), so the inner box
  // dimension equals the 128-byte swizzle span.
  const unsigned per = fp64 ? 2u : 4u;  // rows per 128-byte line
  const cuuint64_t dims[2] = {fp64 ? 16ull : 32ull, rows / per};
  const cuuint64_t strides[1] = {128ull};
  const cuuint32_t box[2] = {fp64 ? 16u : 32u, (cuuint32_t)(box_rows / per)};
  const cuuint32_t estr[2] = {1, 1};
  CUtensorMap *m = reinterpret_cast<CUtensorMap *>(out128);
  const CUresult r = enc(m, fp64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                         2, const_cast<void *>(X), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Instantiated shapes: FP32 {two blocks; one block with 4 and 8 warps; one
// block compensated}; FP64 {direct 2x8, TMA 2x8, direct 2x4, direct 1x8}.
#define FWH_DISPATCH(T, c, CALL)                                                        \
  do {                                                                                   \
    if constexpr (sizeof(T) == 4) {                                                      \
      if (c.tk == 8 && c.warps == 4 && c.acc == 3) return CALL(T, 8, 4, 1, 3);           \
      if (c.tk == 4 && c.warps == 4 && c.acc == 3) return CALL(T, 4, 4, 1, 3);           \
      if (c.tk == 4 && c.warps == 8 && c.acc == 3) return CALL(T, 4, 8, 1, 3);           \
      if (c.tk == 4 && c.warps == 4 && c.acc == 5) return CALL(T, 4, 4, 1, 5);           \
    } else {                                                                             \
      if (c.pipe == 0 && c.tk == 2 && c.warps == 8) return CALL(T, 2, 8, 0, 0);          \
      if (c.pipe == 1 && c.tk == 2 && c.warps == 8) return CALL(T, 2, 8, 1, 0);          \
      if (c.pipe == 0 && c.tk == 2 && c.warps == 4) return CALL(T, 2, 4, 0, 0);          \
      if (c.pipe == 0 && c.tk == 1 && c.warps == 8) return CALL(T, 1, 8, 0, 0);          \
    }                                                                                    \
    return cudaErrorInvalidValue;                                                        \
  } while (0)

template <typename T>
cudaError_t launch_forward(const FwdArgs<T> &a, const void *tmap128, int cfg, cudaStream_t s) {
  const FwdConfig c = fwd_config(sizeof(T) == 8, cfg);
  // the X descriptor travels as a kernel parameter (no device copy to make)
  CUtensorMap tm;
  if (tmap128)
    memcpy(&tm, tmap128, sizeof tm);
  else
    memset(&tm, 0, sizeof tm);
#define FWH_CALL_ONE(TT, TK, NW, PIPE, ACC) launch_one<TT, TK, NW, PIPE, ACC>(a, tm, c, s)
  FWH_DISPATCH(T, c, FWH_CALL_ONE);
#undef FWH_CALL_ONE
}

template <typename T>
cudaError_t launch_forward_batch(const BatchParams<T> &P, int *d_counter, int cfg, int n_ctas,
                                 cudaStream_t s) {
  if (P.n_surf < 1 || P.n_surf > kMaxBatchSurf) return cudaErrorInvalidValue;
  const FwdConfig c = fwd_config(sizeof(T) == 8, cfg);
  const size_t smem = smem_for<T>(c, c.warps * c.obs_per_warp);
#define FWH_CALL_BATCH(TT, TK, NW, PIPE, ACC) \
  launch_batch_one<TT, TK, NW, PIPE, ACC>(P, d_counter, smem, n_ctas, c.stages, s)
  FWH_DISPATCH(T, c, FWH_CALL_BATCH);
#undef FWH_CALL_BATCH
}

template <typename T>
cudaError_t launch_forward_multi(const BatchParams<T> &P, int cfg, cudaStream_t s) {
  if (P.n_surf < 1 || P.n_surf > kMaxBatchSurf || P.total < 1) return cudaErrorInvalidValue;
  const FwdConfig c = fwd_config(sizeof(T) == 8, cfg);
  const size_t smem = smem_for<T>(c, c.warps * c.obs_per_warp);
#define FWH_CALL_MULTI(TT, TK, NW, PIPE, ACC) \
  launch_multi_one<TT, TK, NW, PIPE, ACC>(P, smem, c.stages, s)
  FWH_DISPATCH(T, c, FWH_CALL_MULTI);
#undef FWH_CALL_MULTI
}

// Resident CTAs per SM of the persistent kernel for a config.
template <typename T, int TK, int NW, int PIPE, int ACC>
cudaError_t batch_occupancy_one(const FwdConfig &c, size_t smem, int *per_sm) {
  auto kern = k_forward_batch<T, TK, NW, PIPE, ACC>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, cta_threads<NW, PIPE>(),
                                                       smem);
}

template <typename T>
cudaError_t forward_batch_occupancy(int cfg, int *per_sm) {
  const FwdConfig c = fwd_config(sizeof(T) == 8, cfg);
  const size_t smem = smem_for<T>(c, c.warps * c.obs_per_warp);
  *per_sm = 0;
#define FWH_CALL_OCC(TT, TK, NW, PIPE, ACC) batch_occupancy_one<TT, TK, NW, PIPE, ACC>(c, smem, per_sm)
  FWH_DISPATCH(T, c, FWH_CALL_OCC);
#undef FWH_CALL_OCC
}

template cudaError_t forward_batch_occupancy<float>(int, int *);
template cudaError_t forward_batch_occupancy<double>(int, int *);

template <typename T>
cudaError_t launch_plan(T *coef, const int *i0, const int *set_begin, int nsets, int O, int slack,
                        int win, int slot_bytes, int *i0max_tab, int *err, cudaStream_t s) {
  if (nsets <= 0 || O <= 0) return cudaSuccess;
  k_plan<T><<<nsets, 128, 0, s>>>(coef, i0, set_begin, O, slack, win, slot_bytes, i0max_tab, err);
  return cudaGetLastError();
}

template cudaError_t launch_plan<float>(float *, const int *, const int *, int, int, int, int, int,
                                        int *, int *, cudaStream_t);
template cudaError_t launch_plan<double>(double *, const int *, const int *, int, int, int, int,
                                         int, int *, int *, cudaStream_t);
template cudaError_t launch_forward<float>(const FwdArgs<float> &, const void *, int,
                                           cudaStream_t);
template cudaError_t launch_forward<double>(const FwdArgs<double> &, const void *, int,
                                            cudaStream_t);
template cudaError_t launch_forward_multi<float>(const BatchParams<float> &, int, cudaStream_t);
template cudaError_t launch_forward_multi<double>(const BatchParams<double> &, int, cudaStream_t);
template cudaError_t launch_forward_batch<float>(const BatchParams<float> &, int *, int, int,
                                                 cudaStream_t);
template cudaError_t launch_forward_batch<double>(const BatchParams<double> &, int *, int, int,
                                                  cudaStream_t);

}  // namespace fwh
