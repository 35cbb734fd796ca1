// Deterministic reductions and row-group helpers shared by the solve kernels.
//
// Every dot product is a fixed-grid two-stage reduction: each block folds its
// threads in a fixed order, the last block to finish folds the per-block
// partials in block order and applies the next PCG recurrence step on the
// device (dot_finalize).  Results are therefore identical run to run.  The dot
// products of the recurrence leave only their partials (DOT_PART): every block
// of the kernel that needs them (p.q: the x/r update; r.r and r.z: the p
// update) folds them itself, in the same order.  On small instances that costs it
// less than the fence, counter and re-read of a last block cost the kernel
// before; on large ones it is one FP64 addition per partial and block, so the
// consumer has few blocks (p update) or the fold is done once beside other work
// (rr_test).
#pragma once

#include "common.cuh"

namespace mg {

// Threads of the kernels that end in a dot product.  FP64 issues at about 1.6
// lanes per clock and SM, so a warp's FP64 instruction holds its SM for 20
// clocks: blocks of 128 spread the FP64 work of an instance of 20,000 rows over
// every SM (256-row blocks left a third of them idle).
constexpr int kDotThreads = 128;

enum DotMode {
  DOT_STORE = 0,  // *out = s
  DOT_BNORM,      // |b|^2; zero right-hand side finishes at once
  DOT_RZ0,        // initial r.z
  DOT_PART,       // block partials only (p.q, r.r, r.z)
  DOT_RR,         // r.r's partials and the test on it
  DOT_TR          // |b - A x|^2
};

struct DotCtx {
  double *partials;
  unsigned int *counter;
  PcgScalars *sc;
  double *out;
  int mode;
  double rtol;
  int maxiter;
};

// the end of a PCG iteration by its r.r: tolerance, NaN or the iteration cap;
// true with the status when the solve ends
static __device__ __forceinline__ bool rr_ends(double rr, double thr2, int iters, int maxiter,
                                               int *status) {
  if (rr == rr && rr > thr2 && iters < maxiter) return false;
  *status = !(rr == rr) ? MGPBD_E_BREAKDOWN : (rr <= thr2 ? MGPBD_OK : MGPBD_W_NOT_CONVERGED);
  return true;
}

static __device__ void dot_finalize(const DotCtx &c, double s) {
  PcgScalars *sc = c.sc;
  switch (c.mode) {
    case DOT_STORE:
      *c.out = s;
      break;
    case DOT_BNORM:
      sc->bnorm2 = s;
      sc->thr2 = c.rtol * c.rtol * s;
      sc->rr = s;
      if (s == 0.0) {
        sc->done = 1;
        sc->status = MGPBD_OK;
      } else if (!(s == s) || isinf(s)) {
        sc->done = 1;
        sc->status = MGPBD_E_BREAKDOWN;
      }
      break;
    case DOT_RZ0:
      sc->rz[0] = s;
      if (!(s > 0.0)) {
        sc->done = 1;
        sc->status = MGPBD_E_BREAKDOWN;
      }
      break;
    case DOT_TR:
      sc->tr2 = s;
      break;
    case DOT_RR:
      sc->rr = s;
      if (rr_ends(s, sc->thr2, sc->iters, c.maxiter, &sc->status)) sc->done = 1;
      break;
    case DOT_PART:
      break;
  }
}

// Sum of one value per thread of a block of kDotThreads: through shared memory
// and one warp, nine FP64 additions instead of five per warp and a serial tail.
// The result is in thread 0.  LARGER: over the first kDotThreads of a larger
// block (the guard costs a launch of few blocks up to 2 us, so the others go
// without it).
template <bool LARGER = false>
static __device__ __forceinline__ double block_sum(double v) {
  __shared__ double sd[kDotThreads];
  if (!LARGER || threadIdx.x < kDotThreads) sd[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x >= 32) return 0.0;
#pragma unroll
  for (int k = 32; k < kDotThreads; k += 32) v += sd[threadIdx.x + k];
  return warp_sum(v);
}

// sum over the partials of a reduction of vn blocks by one block, in a fixed
// order whatever block does it; the result is in thread 0
template <bool LARGER = false>
static __device__ __forceinline__ double fold_partials(const double *partials, int vn) {
  double s = 0.0;
  if (!LARGER || threadIdx.x < kDotThreads)
    for (int b = threadIdx.x; b < vn; b += 4 * kDotThreads) {
      double t[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        t[k] = b + k * kDotThreads < vn ? __ldcg(partials + b + k * kDotThreads) : 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) s += t[k];
    }
  return block_sum<LARGER>(s);
}

// The test on r.r by block 0 (of at least kDotThreads threads) of a kernel
// behind the x/r update, after its own share of the work, so that the rest of the
// V-cycle does not run once the solve has ended.  Other blocks of the kernel may
// find the flag raised in their midst: they read it a warp at a time and have no
// barrier behind it.  sc = nullptr: no test.
struct RRTest {
  PcgScalars *sc = nullptr;
  const double *part = nullptr;
  int n = 0, maxiter = 0;
};

static __device__ __forceinline__ void rr_test(const RRTest &t) {
  if (!t.sc || blockIdx.x != 0) return;
  const double rr = fold_partials<true>(t.part, t.n);
  int st;
  if (threadIdx.x == 0) {
    t.sc->rr = rr;
    if (rr_ends(rr, t.sc->thr2, t.sc->iters, t.maxiter, &st)) {
      t.sc->status = st;
      t.sc->done = 1;
    }
  }
}

// block reduce of one value per thread in a fixed order, then the last block
// folds the partials (fixed order) and finalizes.  vb and vn are the block's
// index and the number of blocks of its reduction: the launch's own, or one
// instance's share of a launch that serves several instances (the partition
// into blocks, and so every rounding, is the instance's own either way).
static __device__ void block_dot_finish_vg(double v, const DotCtx &c, int vb, int vn) {
  __shared__ bool last;
  const double s = block_sum(v);
  if (threadIdx.x == 0) c.partials[vb] = s;
  if (c.mode == DOT_PART) return;
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned t = atomicAdd(c.counter, 1u);
    last = (t == (unsigned)vn - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const double t = fold_partials(c.partials, vn);
  if (threadIdx.x == 0) {
    dot_finalize(c, t);
    *c.counter = 0;
  }
}

static __device__ __forceinline__ void block_dot_finish(double v, const DotCtx &c) {
  block_dot_finish_vg(v, c, blockIdx.x, gridDim.x);
}

static __device__ __forceinline__ bool is_done(const PcgScalars *sc) {
  return ((volatile const PcgScalars *)sc)->done != 0;
}

// the same for a warp as a whole
static __device__ __forceinline__ bool warp_is_done(const PcgScalars *sc) {
  return sc && __any_sync(0xffffffffu, is_done(sc));
}

template <int G, class T>
__device__ __forceinline__ T group_sum(T v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of three values over the G lanes of a group (G >= 4) by
// reduce-scatter with a zero fourth slot: two exchange steps leave each lane
// one component summed over four lanes, butterflies finish it.  Lane g ends
// with component 2 * [g & G/2] + [g & G/4]; log2(G) + 1 adds per lane instead
// of 3 log2(G) for three butterflies (the FP64 vertex pass is bound by them).
template <int G, class T>
__device__ __forceinline__ T group_sum3(T a0, T a1, T a2, int g) {
  static_assert(G >= 4 && G <= 32, "group of 4..32 lanes");
  constexpr int o1 = G / 2, o2 = G / 4;
  const bool h1 = (g & o1) != 0, h2 = (g & o2) != 0;
  T k0 = h1 ? a2 : a0, k1 = h1 ? (T)0 : a1;  // kept: components (0,1) or (2,3)
  T s0 = h1 ? a0 : a2, s1 = h1 ? a1 : (T)0;  // sent to the partner
  k0 += __shfl_xor_sync(0xffffffffu, s0, o1);
  k1 += __shfl_xor_sync(0xffffffffu, s1, o1);
  T k = h2 ? k1 : k0, s = h2 ? k0 : k1;
  k += __shfl_xor_sync(0xffffffffu, s, o2);
#pragma unroll
  for (int o = o2 / 2; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  return k;
}

template <int G>
__device__ __forceinline__ int group_sum3_component(int g) {
  return 2 * ((g & (G / 2)) != 0) + ((g & (G / 4)) != 0);
}

// partial row dot of lane g of a G-lane group (no shuffles: callers reduce).
// Four entries per trip are loaded before any is used, so a lane has four
// gathers in flight; the sum order is the plain lane-strided order.
template <int G, class VT, class AT, class XT>
__device__ __forceinline__ AT row_dot(const int64_t *ptr, const int32_t *col, const VT *val,
                                      const XT *x, int i, int g) {
  AT acc = 0;
  int64_t k = ptr[i] + g;
  const int64_t e = ptr[i + 1];
  for (; k + 3 * G < e; k += 4 * G) {
    const int32_t c0 = col[k], c1 = col[k + G], c2 = col[k + 2 * G], c3 = col[k + 3 * G];
    const VT v0 = val[k], v1 = val[k + G], v2 = val[k + 2 * G], v3 = val[k + 3 * G];
    const XT x0 = x[c0], x1 = x[c1], x2 = x[c2], x3 = x[c3];
    acc = fma((AT)v0, (AT)x0, acc);
    acc = fma((AT)v1, (AT)x1, acc);
    acc = fma((AT)v2, (AT)x2, acc);
    acc = fma((AT)v3, (AT)x3, acc);
  }
  for (; k < e; k += G) acc = fma((AT)val[k], (AT)x[col[k]], acc);
  return acc;
}

// The same sum in two halves: row_pre loads the row's extent and the first
// four entries of each lane (static during a solve), row_fin gathers x and
// adds them and the rest in the order of row_dot.  In a launch chain row_pre
// runs before chain_wait, so that the gathers are the only loads behind it;
// most rows of the coarse levels have at most four entries per lane.
template <class VT>
struct RowPre {
  int64_t k, e;
  int32_t c[4];
  VT v[4];
};

template <int G, class VT>
__device__ __forceinline__ RowPre<VT> row_pre(const int64_t *ptr, const int32_t *col,
                                              const VT *val, int64_t i, int g, bool valid) {
  RowPre<VT> p;
  p.k = p.e = 0;
  if (valid) {
    p.k = ptr[i] + g;
    p.e = ptr[i + 1];
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (p.k + j * G < p.e) {
      p.c[j] = col[p.k + j * G];
      p.v[j] = val[p.k + j * G];
    }
  return p;
}

template <int G, class AT, class VT, class XT>
__device__ __forceinline__ AT row_fin(const RowPre<VT> &p, const int32_t *col, const VT *val,
                                      const XT *x) {
  AT acc = 0;
  XT xv[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (p.k + j * G < p.e) xv[j] = x[p.c[j]];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (p.k + j * G < p.e) acc = fma((AT)p.v[j], (AT)xv[j], acc);
  int64_t k = p.k + 4 * G;
  for (; k + 3 * G < p.e; k += 4 * G) {
    const int32_t c0 = col[k], c1 = col[k + G], c2 = col[k + 2 * G], c3 = col[k + 3 * G];
    const VT v0 = val[k], v1 = val[k + G], v2 = val[k + 2 * G], v3 = val[k + 3 * G];
    const XT x0 = x[c0], x1 = x[c1], x2 = x[c2], x3 = x[c3];
    acc = fma((AT)v0, (AT)x0, acc);
    acc = fma((AT)v1, (AT)x1, acc);
    acc = fma((AT)v2, (AT)x2, acc);
    acc = fma((AT)v3, (AT)x3, acc);
  }
  for (; k < p.e; k += G) acc = fma((AT)val[k], (AT)x[col[k]], acc);
  return acc;
}

// The gate between the loads a kernel may make early and the rest: `open`
// waits for the chain's predecessor on its first call and reads the solve's
// done flag beside the loads that follow it; `closed` tells whether the solve
// has finished (checked before anything is written).  Behind a check that has
// been made already (the plain form of a kernel, the cooperative tail) NoGate
// does nothing, and the bodies that differ take their lean form (kEarly).
struct ChainGate {
  static constexpr bool kEarly = true;
  const PcgScalars *sc;
  int state = -1;
  __device__ __forceinline__ explicit ChainGate(const PcgScalars *s) : sc(s) {}
  __device__ __forceinline__ void open() {
    if (state < 0) {
      chain_wait();
      state = sc ? ((volatile const PcgScalars *)sc)->done : 0;
    }
  }
  __device__ __forceinline__ bool closed() const { return state != 0; }
};
struct NoGate {
  static constexpr bool kEarly = false;
  __device__ __forceinline__ void open() {}
  __device__ __forceinline__ bool closed() const { return false; }
};

// Runs body(gate) in a kernel's early form, or in its plain form behind the
// wait and the flag.
template <bool EARLY, class F>
__device__ __forceinline__ void behind_gate(const PcgScalars *sc, F body,
                                            const RRTest &test = RRTest()) {
  if constexpr (EARLY) {
    body(ChainGate(sc));
  } else {
    chain_wait();
    if (warp_is_done(sc)) return;
    body(NoGate{});
    rr_test(test);
  }
}

// Rows handled by G-lane groups, 32/G rows per warp per trip, over warps
// w0, w0 + nw, ...  The loop bound is uniform across the warp, so full-mask
// shuffles inside are safe; `valid` marks groups past the last row.  Which
// warp takes a row never changes that row's arithmetic.
#define GROUP_ROWS_OVER(G, n, w0, nw)                                             \
  const int lane_ = threadIdx.x & 31;                                             \
  const int g = lane_ & ((G) - 1);                                                \
  const int sub_ = lane_ / (G);                                                   \
  const int64_t warp_ = (w0);                                                     \
  const int64_t nwarp_ = (nw);                                                    \
  for (int64_t base_ = warp_ * (32 / (G)), i = base_ + sub_; base_ < (n);         \
       base_ += nwarp_ * (32 / (G)), i = base_ + sub_)                            \
    if (const bool valid = i < (n); true)

// the same over every warp of the launch
#define GROUP_ROWS(G, n)                                                          \
  GROUP_ROWS_OVER(G, n, (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5,    \
                  ((int64_t)gridDim.x * blockDim.x) >> 5)

// the launch's own warps as (first warp, number of warps)
#define HW_WARPS                                                                  \
  (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5,                          \
      ((int64_t)gridDim.x * blockDim.x) >> 5

// the warps of virtual block vb of a grid of vn blocks
#define VG_WARPS(vb, vn)                                                          \
  ((int64_t)(vb) * blockDim.x + threadIdx.x) >> 5, ((int64_t)(vn) * blockDim.x) >> 5

// blocks of a kernel of kDotThreads that leaves one partial per block
inline int dot_blocks(int64_t blocks, const void *kernel) {
  return partial_blocks(blocks, wave_blocks(kernel, kDotThreads));
}

// the test on r.r for the launch being made, if one is due
inline RRTest take_rr_test(Handle *h) {
  RRTest t;
  if (h->rr_test) t = RRTest{h->sc, h->partials, h->n_rr, h->p.pcg_maxiter};
  h->rr_test = false;
  return t;
}

// matrix-free level-0 products (mfree.cu)
bool mf_early(const Handle *h, bool fp64);  // the V-cycle's passes run in their early form
mgpbd_status mf_apply_pq(Handle *h, const double *p, double *q, const DotCtx &c);
mgpbd_status mf_apply_pq_form(Handle *h, bool pairs, const double *p, double *q,
                              const DotCtx &c);
mgpbd_status mf_residual64(Handle *h, const double *x, const double *b, double *r);
mgpbd_status mf_split(Handle *h, const double *a, float2 *out, int64_t n);
template <class T>
mgpbd_status mf_level0(Handle *h, int mode, const T *x, const T *b, const T *dinv, T omega,
                       T *out);
constexpr int kMfSweep = 0, kMfResid = 1, kMfApply = 3, kMfResidMember = 6;
mgpbd_status mf_autotune(Handle *h);

// The last level-0 sweep of a top V-cycle can write the preconditioned
// residual z = x_new straight in FP64 and fold r.z into the PCG scalars.
struct TopOut {
  const double *r;  // FP64 residual the V-cycle was applied to
  double *z;        // FP64 output
  DotCtx c;         // r.z reduction (when dot is set)
  bool dot;
};
template <class T>
mgpbd_status mf_level0_final(Handle *h, const T *x, const T *b, const T *dinv, T omega,
                             const TopOut &o);

}  // namespace mg
