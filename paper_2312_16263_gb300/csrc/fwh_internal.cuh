// Internal declarations of the GB300 FW-H library (not part of the C ABI).
//
// The natural cubic spline of a panel's source signal is carried in its
// cubic B-spline coefficients: with F_k the samples and m_k the spline's
// second derivatives, beta_k = F_k - m_k dt^2 / 6, and at k + f (0 <= f < 1)
// the spline is
//   w0 beta_{k-1} + w1 beta_k + w2 beta_{k+1} + w3 beta_{k+2},
//   w0 = (1 - f)^3 / 6, w1 = (4 - 6 f^2 + 3 f^3) / 6,
//   w2 = (1 + 3 f + 3 f^2 - 3 f^3) / 6, w3 = f^3 / 6,
// with beta_{-1} = 2 beta_0 - beta_1 and beta_nt = 2 beta_{nt-1} - beta_{nt-2}
// (the natural ends).  One eight-value dot product and four weights per
// (panel, sample, observer): 12 multiply-adds, where samples and moments side
// by side take 20 and twice the bytes.
//
// Data layout in HBM (P = panels in the library's spatial order, O =
// observers, T = float or double):
//   fields   [nt][5][P]      caller's pulsations (original panel order)
//   X        [P][x_ld][8] T  per panel the B-spline coefficients of the eight
//                            observer-independent series, interleaved as
//                              Qn', Qn, L1', L1, L2', L2, L3', L3
//                            (' = source-time derivative).  Row r holds
//                            sample row0 + r - 1, so that a record's first
//                            row is the end value beta_{-1}; x_ld is a
//                            multiple of 64 rows.  The row after the ghost's
//                            (sample nt + 1) is zero; the rows after that are
//                            not written, and only reach bins past every
//                            observer's window.  Whole records: row0 = 0 and
//                            x_ld >= nt + 3
//   Xbar     [P][xb_ld][8] T gradient with respect to beta_0 .. beta_{nt-1}
//   coef     [P][O][16] T    per (panel, observer) record (slots in
//                            namespace slot): the 8 integrand coefficients
//                            (same order as X), the weights w0..w3, then for
//                            FP64 the shift i0 and the window offset
//                            i0max(set) - i0, for FP32 the four byte offsets
//                            of that window offset (written by the planner)
//   i0       [P][O] int      FP32: the integer shifts
//   p_out    [O][nt] double  caller's output
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fwh {

constexpr int kRec = 16;          // values per coef record
constexpr int kSer = 8;           // values per X row
constexpr int kRowBlk = 64;       // X rows per prep block

// X rows of a whole record of nt samples (samples -1 .. nt + 1, up to a whole block).
inline int64_t x_rows(int64_t nt) { return (nt + 3 + kRowBlk - 1) / kRowBlk * kRowBlk; }
// Bytes past the last X row that an L2 prefetch of a whole chunk may touch.
constexpr size_t kXPad = 16384;

// Slots of a coefficient record (kRec values, both precisions).
namespace slot {
constexpr int c = 0;    // c0..c7: coefficients of the eight series, in X's order
constexpr int w = 8;    // w0..w3: B-spline weights of beta_{k-1} .. beta_{k+2}
constexpr int i0 = 12;  // FP64: integer shift (a value)
constexpr int off = 13; // FP64: window offset i0max(set) - i0, written by the planner
// FP32 records, written by the planner: byte offsets, in an observer's window
// (slot x in quarter x & 3, word x >> 2), of the slots off, off + 1, off + 2, off + 3
constexpr int q0 = 12;
}  // namespace slot
constexpr int kWarp = 32;

// Halo (samples) of the windowed natural-spline solves: the influence of a
// window edge decays as (2 - sqrt 3)^k, below 1e-18 for k = 32 and below
// 1e-9 (under FP32 rounding) for k = 16.
template <typename T> struct Prec;
template <> struct Prec<float> { static constexpr int halo = 16; };
template <> struct Prec<double> { static constexpr int halo = 32; };

#ifdef __CUDACC__
// Packed FP32 pairs (fma.rn.f32x2 and friends): element-wise IEEE round-to-
// nearest operations on two floats held in a 64-bit register pair.  One
// packed FMA issues in one slot and keeps the FMA pipe busy for two cycles.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 f2_dup(float x) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ void f2_split(f32x2 v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// 32 bytes to global memory in one store (a whole sector per lane).
__device__ __forceinline__ void stg256(void *dst, unsigned long long a, unsigned long long b,
                                       unsigned long long c, unsigned long long d) {
  asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "l"(a), "l"(b), "l"(c),
               "l"(d)
               : "memory");
}
#endif

// Device error flags (bitmask written by kernels, read by the host).
enum : int {
  kErrWindow = 1,      // a panel set's arrival spread exceeded the window
  kErrTimeout = 2,     // a bounded wait gave up
  kErrQueue = 4,       // persistent queue inconsistency
};

struct GeomArgs {
  const double *y;      // [P][3] sorted centroids
  const double *n;      // [P][3] sorted normals
  const double *dS;     // [P]
  const double *x;      // [O][3]
  int P, O;
  double mach, ca, sa, dt;
  double *Rmax, *Rmin;  // [O]
};

template <typename T>
struct PrepArgs {
  const T *fields;      // [nt][5][P] original order
  const int *place;     // [P] original panel index -> sorted position (null: the same)
  const double *n;      // [P][3] sorted normals
  T *X;                 // [P][x_ld][8]
  int P, nt;
  int x_ld;             // X rows per panel
  int row0;             // record row held by X row 0 (a multiple of 64)
  double ca, sa, dt;
  int c_lo, c_hi;       // 64-row blocks [c_lo, c_hi) to prepare (0, 0: the whole record)
                        // (rows nt .. nt + 2 are written with the block of row nt - 1)
};

template <typename T>
struct FwdArgs {
  const T *X;           // [P][x_ld][8]
  const T *coef;        // [P][O][16]
  double *p_out;        // [O][nt]
  const int *n_valid;   // [O]
  const int *set_begin; // [nsets + 1] panel-set boundaries (sorted order)
  const int *set_order; // [nsets] sets by descending panel count (null: index order)
  const int *i0max_tab; // [nsets][O] largest shift of each (panel set, observer)
  int *err;
  int nsets, O, nt;
  int x_ld;             // X rows per panel
  int row0;             // record row held by X row 0
  int k_top;            // FP32: spline intervals (nt); FP64: rows that reach a bin (nt + 2)
  int obs_per_cta, n_obs_groups;
  int subs;             // work items a panel set is cut into
  int seg_len, n_segs;
  int seg_shift;        // segment q ends at interval (q + 1) seg_len - seg_shift (a multiple of 4)
  int seg_lo, seg_cnt;  // this launch covers time segments [seg_lo, seg_lo + seg_cnt)
  int win;              // window slots per observer
  int slack;            // largest spread of shifts within a panel set
  int wfl;              // values per observer window: win, or 2 win for compensated
                        // FP32 windows (a sum and its compensation per slot)
  long long wait_cycles; // bound of each pipeline wait in SM clocks (the handle's limit)
  int withhold;         // testing: the copy pipeline issues no copies (every wait runs out)
};

// Surfaces in one batched call (their arguments sit in each CTA's shared memory).
constexpr int kMaxBatchSurf = 32;

template <typename T>
struct AdjArgs {
  const T *coef;        // [P][O][16]
  T *Gt;                // [O][g_ld] workspace: grad_p in T, zero outside [0, N_o)
  const double *grad_p; // [O][nt]
  const int *n_valid;   // [O]
  T *Xbar;              // [P][xb_ld][8] gradient w.r.t. the B-spline coefficients
  int P, O, nt, g_ld, xb_ld;
  // FP32: the forward plan
  const int *set_begin; // [nsets + 1] panel-set boundaries (sorted order)
  const int *set_order; // [nsets] sets by descending panel count
  const int *i0max_tab; // [nsets][O] largest shift of each (panel set, observer)
  int nsets, win;       // win: window slots per observer
  int slot_shift;       // log2 of the plan's bytes per window slot (2, or 3 if compensated)
  int slack;            // largest spread of shifts within a panel set
};

template <typename T>
struct PrepAdjArgs {
  const T *fields;      // [nt][5][P] original order
  const int *place;     // [P] original panel index -> sorted position (null: the same)
  const double *n;      // [P][3] sorted normals
  const T *Xbar;        // [P][xb_ld][8]
  T *grad_fields;       // [nt][5][P] original order
  int P, nt, xb_ld;
  double ca, sa, dt;
};

// ---- launchers (defined in the .cu files) --------------------------------
cudaError_t launch_window(const GeomArgs &a, cudaStream_t s);
// N_o per observer (Eq. t_end) from R_max / R_min, rounded as the host does.
cudaError_t launch_nvalid(const double *Rmax, const double *Rmin, int O, double mach, double dt,
                          int nt, int *n_valid, cudaStream_t s);
template <typename T>
cudaError_t launch_coef(const GeomArgs &a, T *coef, int *i0, cudaStream_t s);
template <typename T>
cudaError_t launch_prep(const PrepArgs<T> &a, cudaStream_t s);
template <typename T>
cudaError_t launch_prep_adjoint(const PrepAdjArgs<T> &a, cudaStream_t s);
template <typename T>
cudaError_t launch_adjoint(const AdjArgs<T> &a, cudaStream_t s);

// Forward tile configurations (index into a table in fwh_forward.cu).
struct FwdConfig {
  int pipe;           // 0: direct loads, 1: TMA + mbarrier pipeline (producer warp)
  int tk;             // X rows per lane per chunk
  int warps;          // compute warps per CTA
  int obs_per_warp;   // max observers per warp
  int win;            // window slots per observer
  int seg_chunks;     // chunks per time segment
  int stages;         // pipeline stages (pipe = 1)
  int acc;            // FP64: 0.  FP32 window sums: 3 plain, 5 compensated (Kahan)
};
// Source samples a chunk completes: FP64 lanes hold rows 32 apart; FP32 lanes
// hold four consecutive rows per 128-row block, and the last lane's serve only
// its neighbour.
inline int fwd_chunk(bool fp64, const FwdConfig &c) { return 32 * c.tk - (fp64 ? 0 : 4); }
// Largest spread of shifts within a panel set that a config's window holds
// (FP32: also the adjoint's window of a 128-row chunk).
constexpr int kAdjReach = 131;
inline int fwd_slack(bool fp64, const FwdConfig &c) {
  const int need = fp64 ? 32 * c.tk + 3 : 32 * c.tk - 4;
  return c.win - (fp64 || need > kAdjReach ? need : kAdjReach);
}
// Bytes of dynamic shared memory a config needs for `obs_per_cta` observers.
size_t fwd_smem_bytes(bool fp64, const FwdConfig &c, int obs_per_cta);
// CTAs of the persistent batch kernel that fit on one SM for config `cfg`.
template <typename T>
cudaError_t forward_batch_occupancy(int cfg, int *per_sm);
// Encode the TMA descriptor of X ([rows][8] elements of 4 or 8 bytes) into a
// host buffer of 128 bytes; returns false if the driver refuses.
bool encode_x_tensor_map(void *out128, const void *X, unsigned long long rows, bool fp64,
                         int box_rows);
int fwd_num_configs(bool fp64);
FwdConfig fwd_config(bool fp64, int idx);
// tmap128: host copy of the X tensor map (128 bytes) for TMA configs, passed
// to the kernel as a parameter; may be null for direct-load configs.
template <typename T>
cudaError_t launch_forward(const FwdArgs<T> &a, const void *tmap128, int cfg_idx,
                           cudaStream_t s);
// Planner kernel: per (panel set, observer) the largest shift i0max into
// i0max_tab and, per record, the window offset i0max - i0 clamped to [0,
// slack], as a value (FP64) or as the byte offsets of its four slots in the
// quarter-split window of `win` slots of slot_bytes (FP32).  A set whose
// shifts span more than slack raises kErrWindow.
template <typename T>
cudaError_t launch_plan(T *coef, const int *i0, const int *set_begin, int nsets, int O, int slack,
                        int win, int slot_bytes, int *i0max_tab, int *err, cudaStream_t s);

// Batched persistent forward: the arguments of one launch, passed by value
// as a __grid_constant__ kernel parameter (under 9 KB at kMaxBatchSurf
// surfaces), so that the kernel reads them from the constant bank and hands
// the descriptors' parameter-space addresses to its tensor copies.
struct alignas(64) TmapBytes {
  unsigned char b[128];   // a CUtensorMap (encoded by encode_x_tensor_map)
};
template <typename T>
struct alignas(64) BatchParams {
  TmapBytes tm[kMaxBatchSurf];      // X descriptor of each surface
  FwdArgs<T> a[kMaxBatchSurf];      // arguments of each surface
  int prefix[kMaxBatchSurf + 1];    // first work item of each surface; [n_surf] = total
  int n_surf, total;
};
template <typename T>
cudaError_t launch_forward_batch(const BatchParams<T> &params, int *d_counter, int cfg_idx,
                                 int n_ctas, cudaStream_t s);
// The same work items as one ordinary grid (one CTA per item, no queue).
template <typename T>
cudaError_t launch_forward_multi(const BatchParams<T> &params, int cfg_idx, cudaStream_t s);

}  // namespace fwh
