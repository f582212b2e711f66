// One kernel per check block for LPs that fit on the SMs: K iterations, the
// check, the multiplier search, the restart decision and the restart, with
// the matrix and the owned part of every vector in shared memory.  A larger LP
// takes the whole grid (cooperative launch); a small one, and every problem of a
// batch of small ones, a cluster of 1 to 8 blocks.
//
// What bounds a small or medium LP in the two-launches-per-iteration path is
// neither bytes nor FP64 but the chain of each launch: scheduling, the slice
// record, the index, the gather, the epilogue (3-7 us per pass however few
// nonzeros it has), and 23 more launches per check.  Here a launch lives for
// the whole block: P thread blocks, each owning every P-th slice of A^T and of
// A, read their slices once into shared memory; a pass is then gathers from
// L2, FMAs and one grid barrier.  Row sums run in exactly the order of
// process_item (same lanes, same chain, same butterfly), so the iterates are
// those of the per-pass kernels bit for bit.
//
// Measured on GB300, 5k x 25k with 246k nonzeros, FP64, P = 152, cycles per
// iteration: column pass 3,800, barrier 3,300 (the averages included), row pass
// 3,800, barrier 2,600 (6.8 us; the per-pass kernels 13.6 us).  The passes are bound
// by the latency of random gathers from L2 (L1 18% busy, L2 13%), the barriers by
// the release fence and two trips to L2; FP64 is 30% busy.  Tagging every exchanged
// value with the number of its pass, so that gathers wait for their own operand and
// no barrier is needed, was slower: the tagged words bypass L1 and the repeated
// gathers fill it (9,500 cycles per pass).  FP64 instructions are the other scarce
// thing: one of a warp holds its quarter of the SM for 76 cycles whatever the number
// of active lanes.  So sums over the block go through transposed butterflies,
// scalars are computed by one warp, and the owned rows and columns are laid out one
// per thread where the averages and the check's terms are formed.
//
// In a cluster every block holds whole copies of xhat and y in shared memory and
// the owners store into all of them, so a pass of 200 x 400 takes 1,600 cycles and
// a barrier 700 instead of 2,500: 64 iterations and a check, 0.25 ms on 8 blocks
// (0.33 on the grid, 0.49 with the per-pass kernels).  What bounds a batch is the
// FP64 pipe: 512 problems of 200 x 400 run at 20,400 cycles per iteration with four
// blocks per SM; the pipe is busy for 84% of an SM's active cycles, all of them where
// four blocks run (512 blocks give some SMs three: 70% of elapsed).
//
// The multiplier lambda* of Section 6.3 is found by Newton's method on
// F(mu) = sum min(d^2, mu g^2) = r^2, mu = lambda^2: F is concave and piecewise
// linear, so from mu = 0 the iterates increase to mu* and are exact once the
// set of clamped coordinates repeats (5 or 6 steps on the LPs measured).  Each
// step is one scan of the block's own breakpoints, one reduction and one
// barrier; a radix pass needs a histogram of 256 buckets and two barriers.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "lp_internal.h"
#include "spmv_core.cuh"

namespace lpg {
namespace {

constexpr int kGridThreads = 512;      // threads per block of the grid kernel
constexpr int kClusterThreads = 256;   // and of the cluster kernel
constexpr int kU = 8;                  // gathers in flight per lane
constexpr int kLeanU = 4;              // where the registers of two blocks per SM hold no more
constexpr int kStatusIterLimit = 4;
constexpr int kBarLines = kResBarLines;  // arrival counters of the grid barrier
constexpr unsigned long long kWaitNs = 2000000000ull;  // longest wait at a barrier

// One local slice: first element (in shared memory, or from the problem's first
// element on when the matrix stays in global memory), first local row,
// steps << 16 | log2 of the lanes per row << 8 | rows, and its global number.
struct __align__(16) LSlice {
  int32_t soff, slot0;
  uint32_t shape;
  int32_t gid;
  __device__ __forceinline__ int steps() const { return (int)(shape >> 16); }
  __device__ __forceinline__ int lg() const { return (int)((shape >> 8) & 255u); }
  __device__ __forceinline__ int rows() const { return (int)(shape & 255u); }
};

// Position in the local list (most steps first) of a warp's slice of a round:
// the first round goes up the warps and the later ones come down, so the warps
// with the longest slices get the shortest of the rest, or none.
template <int NT>
__device__ __forceinline__ int pick(int round, int warp) {
  constexpr int W = NT / kWarp;
  return round == 0 ? warp : round * W + W - 1 - warp;
}

// Scalars of the problem, read once by one thread.
struct Scalars {
  double tau, sigma, omega, norm_b, norm_c, tol, beta, rho_stored, last_r, mix_s;
  int64_t t0, restarts, tau0, fixed_len;
  int32_t K, scheme, due, returned;
};

struct Header {
  int32_t ncl, nrl;  // local columns and rows
  int32_t nce, nre;  // elements
  int32_t dead;      // a wait ran out
  // Results of one warp: an FP64 instruction of a warp occupies its quarter of
  // the SM for 76 cycles (measured), a square root or a division dozens of
  // them, so the other warps read the results here.
  int32_t status, returned, restart, use_cur;
  int32_t done[2];
  int32_t count[2];  // coordinates clamped at the last Newton step
  double sw, isw, inv;
  double kkt[2][5], r2[2], lam[2], rho_r[2];
  double rho, r, mix_s;
  Scalars sc;
};

template <typename T>
struct Sm {  // shared-memory arrays of a block
  Header *h;
  LSlice *cs, *rs;
  double *red;  // [warps][32] sums of the warps
  double *tot;  // [32] sums over the blocks
  double *nw;   // [8] Newton sums
  double *w;    // [K] averaging weights
  T *ex, *ey;   // cluster kernel: this block's copies of xhat and y
  int32_t *crow, *rrow;     // permuted index of each local column and row
  double *cs0, *cs1, *rs0, *rs1;  // check sums of both candidates
  // FP64: c, x, xbar, order keys of the bounds.  Mixed: cf, dx, dxbar, lf, uf
  T *c, *x, *b, *y;
  double *xb, *yb;
  long long *lk, *uk;
  float *lf, *uf, *lo, *hi;
  int32_t *rt;
  int32_t *cidx, *ridx;
  T *cval, *rval;
};

// What one group of blocks works on: a problem's slices, block `rank` of P
// owning every P-th of them, and its ranges in the permuted index spaces.
struct Share {
  int c0, nc, r0, nr, stride;       // this block's slices: c0 + i stride, i < nc; rows alike
  int cfirst, rfirst;               // the problem's first slices
  int col0, ncol, row0, nrow;
  int rank, P;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(unsigned *p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// How the blocks of a group exchange xhat and y and wait for one another.
// Grid: the vectors lie in global memory.  The barrier of a cooperative launch
// is kBarLines arrival counters that only grow, a 128-byte line each (152
// arrivals at one address cost 900 cycles more), block b on counter b mod
// kBarLines; one lane of warp 0 waits on each.  Block-wide barriers on both
// sides order the other threads' accesses.  The wait is bounded: after kWaitNs
// the block gives up, and every other block's wait runs out the same way.
template <typename T>
struct GridLink {
  static constexpr bool kCluster = false;
  unsigned *counter;
  unsigned gen;  // barriers passed since the counters were zero
  int32_t *dead;
  T *gx, *gy;
  __device__ __forceinline__ const T *x() const { return gx; }
  __device__ __forceinline__ const T *y() const { return gy; }
  __device__ __forceinline__ void put_x(int j, T v) const { gx[j] = v; }
  __device__ __forceinline__ void put_y(int i, T v) const { gy[i] = v; }
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    ++gen;
    if (threadIdx.x == 0) red_release(counter + (blockIdx.x % kBarLines) * 32);
  }
  __device__ __forceinline__ bool wait() {
    const int P = (int)gridDim.x, lane = (int)threadIdx.x;
    if (lane < kBarLines) {
      // blocks that arrive at this lane's counter
      const unsigned want = gen * (unsigned)((P - lane + kBarLines - 1) / kBarLines);
      const unsigned *p = counter + lane * 32;
      int spins = 0;
      unsigned long long t0 = 0;
      while ((int)(ld_acquire(p) - want) < 0) {
        if ((++spins & 255) == 0) {
          const unsigned long long t = now_ns();
          if (t0 == 0) t0 = t;
          if (t - t0 > kWaitNs) {
            *(volatile int32_t *)dead = 1;
            break;
          }
        }
      }
    }
    __syncthreads();
    return *(volatile int32_t *)dead == 0;
  }
  __device__ __forceinline__ bool sync() {
    arrive();
    return wait();
  }
};

__device__ __forceinline__ void put_shared(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void put_shared(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// Cluster: every block keeps whole copies of the two vectors in shared memory;
// an owner stores its element into all of them (distributed shared memory) and
// the hardware's cluster barrier orders the passes (no polling).
template <typename T>
struct ClusterLink {
  static constexpr bool kCluster = true;
  int C;
  T *ex, *ey;  // copies, indexed by permuted column - col0 and row - row0
  int col0, row0;
  uint32_t ax, ay;  // their shared-memory addresses
  __device__ __forceinline__ const T *x() const { return ex; }
  __device__ __forceinline__ const T *y() const { return ey; }
  __device__ __forceinline__ void put(uint32_t addr, T v) const {
    for (int c = 0; c < C; ++c) {
      uint32_t to;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(addr), "r"(c));
      put_shared(to, v);
    }
  }
  __device__ __forceinline__ void put_x(int j, T v) const {
    if (C == 1) ex[j - col0] = v;
    else put(ax + (uint32_t)sizeof(T) * (uint32_t)(j - col0), v);
  }
  __device__ __forceinline__ void put_y(int i, T v) const {
    if (C == 1) ey[i - row0] = v;
    else put(ay + (uint32_t)sizeof(T) * (uint32_t)(i - row0), v);
  }
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    if (C > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  }
  __device__ __forceinline__ bool wait() {
    if (C > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    return true;
  }
  __device__ __forceinline__ bool sync() {
    arrive();
    return wait();
  }
};

// Row sum of one slice, in the order of process_item: `a` is the lane's
// starting value (-c or -b in the row's first lane), ip and vp the lane's
// indices and values.  All lanes of a row return its sum.  The gathers are
// plain loads: the barrier's acquire makes L1 safe to use.  SHIFT: vec starts at
// element `base` of the index space (padding, index 0, reads element base).
template <bool SHIFT, int UR = kU, typename T>
__device__ __forceinline__ T slice_sum(T a, const int32_t *ip, const T *vp, int steps, int lg,
                                       const T *vec, int base) {
  if constexpr (SHIFT) {  // streamed from global memory: indices and values load together
    constexpr int U = 4;
    for (int t = 0; t < steps; t += U) {
      int j[U];
      T c[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < steps) {
          j[u] = __ldg(ip + kWarp * (t + u));
          c[u] = __ldg(vp + kWarp * (t + u));
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < steps) a = fma_t(c[u], vec[max(j[u] - base, 0)], a);
    }
  } else {
    for (int t = 0; t < steps; t += UR) {
      T g[UR];
#pragma unroll
      for (int u = 0; u < UR; ++u)
        if (t + u < steps) g[u] = vec[ip[kWarp * (t + u)]];
#pragma unroll
      for (int u = 0; u < UR; ++u)
        if (t + u < steps) a = fma_t(vp[kWarp * (t + u)], g[u], a);
    }
  }
  for (int o = (1 << lg) >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
  return a;
}

// Sums of the check, both candidates at once, from plain arrays (written
// before a barrier, whose acquire lets plain loads use L1) and FP64 values;
// sval: the resident values, or null to read them from global memory.  base: the
// first element that the resident indices count from.
template <int NT, bool RES>
__device__ __forceinline__ void check_sums(const LSlice *sl, int count, const int32_t *sidx,
                                           const double *sval, const SellMat &A,
                                           int base, const double *v0, const double *v1,
                                           double *o0, double *o1) {
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x >> 5;
  for (int q = 0, i; (i = pick<NT>(q, warp)) < count; ++q) {
    const LSlice s = sl[i];
    const int lg = s.lg(), steps = s.steps();
    const int64_t off = A.info[s.gid].off;
    const int32_t *ip = (RES ? sidx + s.soff : A.idx + off) + lane;
    const double *vp = (sval ? sval + s.soff : A.val + off) + lane;
    double a0 = 0.0, a1 = 0.0;
    for (int t = 0; t < steps; t += 4) {
      double g[4], h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u < steps) {
          const int j = ip[kWarp * (t + u)] + (RES ? base : 0);
          g[u] = v0[j];
          h[u] = v1[j];
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u < steps) {
          const double v = vp[kWarp * (t + u)];
          a0 = fma(v, g[u], a0);
          a1 = fma(v, h[u], a1);
        }
    }
    for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
      a0 += __shfl_xor_sync(kFull, a0, o);
      a1 += __shfl_xor_sync(kFull, a1, o);
    }
    const int r = lane >> lg;
    if ((lane & ((1 << lg) - 1)) == 0 && r < s.rows()) {
      o0[s.slot0 + r] = a0;
      o1[s.slot0 + r] = a1;
    }
  }
}

// Sum over the P blocks of quantity q's partials, by one warp, fixed order.
__device__ __forceinline__ double sum_parts(const double *part, int stride, int q, int P) {
  const int lane = threadIdx.x & (kWarp - 1);
  double s = 0.0;
  for (int p = lane; p < P; p += kWarp) s += __ldcg(part + (size_t)p * stride + q);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  return s;
}

// Local slices of one operator, most steps first: records, and the numbers of
// local rows and elements.  One warp.
template <bool RES>
__device__ void build_slices(const SellMat &A, int first, int count, int stride, int pfirst,
                             LSlice *sl, int32_t *nslot, int32_t *nelem) {
  const int lane = threadIdx.x & (kWarp - 1);
  int slot = 0, el = 0;
  for (int i0 = 0; i0 < count; i0 += kWarp) {
    const int i = i0 + lane;
    int rows = 0, steps = 0, lg = 0, rank = 0, goff = 0;
    if (i < count) {
      const SliceInfo a = A.info[first + i * stride];
      rows = A.info[first + i * stride + 1].row0 - a.row0;
      steps = a.len_g >> 3;
      lg = a.len_g & 7;
      if (!RES) goff = (int)(a.off - A.info[pfirst].off);
      for (int j = 0; j < count; ++j) {
        const int o = A.info[first + j * stride].len_g >> 3;
        rank += (o > steps || (o == steps && j < i)) ? 1 : 0;
      }
    }
    int ps = rows, pl = steps;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
      const int u = __shfl_up_sync(kFull, ps, o), v = __shfl_up_sync(kFull, pl, o);
      if (lane >= o) {
        ps += u;
        pl += v;
      }
    }
    if (i < count)
      sl[rank] = LSlice{RES ? el + kWarp * (pl - steps) : goff, slot + ps - rows,
                        (uint32_t)steps << 16 | (uint32_t)lg << 8 | (uint32_t)rows,
                        first + i * stride};
    slot += __shfl_sync(kFull, ps, kWarp - 1);
    el += kWarp * __shfl_sync(kFull, pl, kWarp - 1);
  }
  if (lane == 0) {
    *nslot = slot;
    *nelem = el;
  }
}

__device__ __forceinline__ unsigned char *carve(unsigned char *&p, size_t bytes) {
  unsigned char *q = p;
  p += (bytes + 15) & ~size_t(15);
  return q;
}

// The permuted indices of the local rows, and (RES) the local slices' elements
// into shared memory, their indices counted from `base` on (padding: 0).
template <typename T, int NT, bool RES>
__device__ __forceinline__ void load_slices(const SellMat &A, const T *gval, const LSlice *sl,
                                            int count, int base, int32_t *row, int32_t *sidx,
                                            T *sval) {
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x >> 5;
  constexpr int VC = 16 / sizeof(T);  // values per 16-byte chunk
  for (int i = warp; i < count; i += NT / kWarp) {
    const LSlice s = sl[i];
    const SliceInfo g = A.info[s.gid];
    for (int r = lane; r < s.rows(); r += kWarp) row[s.slot0 + r] = g.row0 + r;
    if (!RES) continue;
    const int len = s.steps() * kWarp;
    const int4 *gi = reinterpret_cast<const int4 *>(A.idx + g.off);
    int4 *si = reinterpret_cast<int4 *>(sidx + s.soff);
    for (int e = lane; e < len / 4; e += kWarp) {
      const int4 j = __ldg(gi + e);
      si[e] = make_int4(max(j.x - base, 0), max(j.y - base, 0), max(j.z - base, 0),
                        max(j.w - base, 0));
    }
    const int4 *gv = reinterpret_cast<const int4 *>(gval + g.off);
    int4 *sv = reinterpret_cast<int4 *>(sval + s.soff);
    for (int e = lane; e < len / VC; e += kWarp) sv[e] = __ldg(gv + e);
  }
}

// Bytes of shared memory per local column and row.
template <typename T>
constexpr size_t col_bytes() {
  return sizeof(T) == 8 ? 4 + 8 + 8 + 8 + 16 : 4 + 4 + 4 + 8 + 8 + 16;
}
template <typename T>
constexpr size_t row_bytes() {
  return sizeof(T) == 8 ? 4 + 8 + 8 + 8 + 4 : 4 + 4 + 4 + 8 + 8 + 16;
}

// The layout of run_block's shared memory: the arrays whose sizes are known from
// the start, and, once the header tells the numbers of local rows and elements,
// those behind them.
template <typename T, int NT, bool CLUSTER>
__device__ __forceinline__ unsigned char *lay_lists(Sm<T> &S, unsigned char *p, const Share &sh,
                                                    int K) {
  S.h = (Header *)carve(p, sizeof(Header));
  if (CLUSTER) {  // at the same place in every block: owners store into all of them
    S.ex = (T *)carve(p, sizeof(T) * sh.ncol);
    S.ey = (T *)carve(p, sizeof(T) * sh.nrow);
  }
  S.cs = (LSlice *)carve(p, sizeof(LSlice) * sh.nc);
  S.rs = (LSlice *)carve(p, sizeof(LSlice) * sh.nr);
  S.red = (double *)carve(p, sizeof(double) * (NT / kWarp) * 32);
  S.tot = (double *)carve(p, sizeof(double) * 32);
  S.nw = (double *)carve(p, sizeof(double) * 8);
  S.w = (double *)carve(p, sizeof(double) * K);
  return p;
}

template <typename T, bool RES>
__device__ __forceinline__ void lay_arrays(Sm<T> &S, unsigned char *p, int ncl, int nrl) {
  S.crow = (int32_t *)carve(p, 4 * (size_t)ncl);
  S.rrow = (int32_t *)carve(p, 4 * (size_t)nrl);
  S.c = (T *)carve(p, sizeof(T) * ncl);
  S.x = (T *)carve(p, sizeof(T) * ncl);
  S.xb = (double *)carve(p, 8 * (size_t)ncl);
  S.b = (T *)carve(p, sizeof(T) * nrl);
  S.y = (T *)carve(p, sizeof(T) * nrl);
  S.yb = (double *)carve(p, 8 * (size_t)nrl);
  if constexpr (sizeof(T) == 4) {
    S.lf = (float *)carve(p, 4 * (size_t)ncl);
    S.uf = (float *)carve(p, 4 * (size_t)ncl);
    S.lo = (float *)carve(p, 4 * (size_t)nrl);
    S.hi = (float *)carve(p, 4 * (size_t)nrl);
    S.cs0 = (double *)carve(p, 8 * (size_t)ncl);
    S.cs1 = (double *)carve(p, 8 * (size_t)ncl);
    S.rs0 = (double *)carve(p, 8 * (size_t)nrl);
    S.rs1 = (double *)carve(p, 8 * (size_t)nrl);
  } else {
    S.lk = (long long *)carve(p, 8 * (size_t)ncl);
    S.uk = (long long *)carve(p, 8 * (size_t)ncl);
    S.rt = (int32_t *)carve(p, 4 * (size_t)nrl);
    // the check comes after the state has gone back to global memory
    S.cs0 = S.xb;
    S.cs1 = S.c;
    S.rs0 = S.yb;
    S.rs1 = S.b;
  }
  S.cidx = S.ridx = nullptr;
  S.cval = S.rval = nullptr;
  if constexpr (RES) {
    S.cidx = (int32_t *)carve(p, 4 * (size_t)S.h->nce);
    S.cval = (T *)carve(p, sizeof(T) * S.h->nce);
    S.ridx = (int32_t *)carve(p, 4 * (size_t)S.h->nre);
    S.rval = (T *)carve(p, sizeof(T) * S.h->nre);
  }
}

// Mixed precision: the radius of a restart scales the next correction (mix_s),
// whose data are rounded to FP32, so its last bits must not depend on the
// kernel.  These sums of (z - z0)^2 over the columns and the rows repeat the
// order of the per-pass kernels' check.  A block reads rows that others own, so
// the parts are formed before the check's barrier: behind it the owners may
// already be writing the restart point (a search that needs no step has no
// further barrier).
//
// Of the owned rows of one slice, lane by lane.
__device__ __forceinline__ double slice_dist2(const SellMat &A, int slice, const double *z,
                                              const double *z0, double q) {
  const int lane = threadIdx.x & (kWarp - 1);
  const SliceInfo a = A.info[slice];
  const int lg = a.len_g & 7, row = a.row0 + (lane >> lg);
  if ((lane & ((1 << lg) - 1)) == 0 && row < A.info[slice + 1].row0) {
    const double d = z[row] - z0[row];
    q = fma(d, d, q);
  }
  return q;
}

// Single problem (check_kernel, block_reduce_store_mask, check_finalize_kernel):
// the check's blocks of 8 warps, their sums one entry each of out.
template <int NT>
__device__ __forceinline__ void radius_parts(const ResidentArgs &a, const Share &sh, double *red,
                                             int cand, double *out) {
  constexpr int G = NT / kBlock, W = kWarpsPerBlock;
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x >> 5, g = warp / W, w = warp % W;
  const int gc = a.cs.cols_grid, gr = a.cs.rows_grid;
  for (int v0 = sh.rank * G; v0 < gc + gr; v0 += sh.P * G) {
    const int v = v0 + g;
    double q = 0.0;
    if (v < gc) {
      const double *x = cand ? a.v.x : a.v.xbar;
      for (int it = v * W + w; it < a.AT.nslices; it += gc * W) q = slice_dist2(a.AT, it, x, a.v.x0, q);
    } else if (v < gc + gr) {
      const double *y = cand ? a.v.y : a.v.ybar;
      for (int it = (v - gc) * W + w; it < a.A.nslices; it += gr * W)
        q = slice_dist2(a.A, it, y, a.v.y0, q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(kFull, q, o);
    if (lane == 0) red[warp] = q;
    __syncthreads();
    if (lane == 0 && w == 0 && v < gc + gr) {
      double s = 0.0;
      for (int i = 0; i < W; ++i) s += red[g * W + i];
      __stcg(out + v, s);
    }
    __syncthreads();
  }
}

// The sum of entries [lo, hi) of part (of n), by the first kBlock threads; all
// threads of the block call it.
__device__ __forceinline__ double radius_total(const double *part, int n, int lo, int hi,
                                               double *red) {
  const int tid = (int)threadIdx.x;
  if (tid < kBlock) {
    double s = 0.0;
    for (int p = tid; p < n; p += kBlock) s += p >= lo && p < hi ? __ldcg(part + p) : 0.0;
    red[tid] = s;
  }
  __syncthreads();
  for (int o = kBlock / 2; o > 0; o >>= 1) {
    if (tid < o) red[tid] += red[tid + o];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}

// A batch's problem (b_check_kernel, b_finalize_kernel): one entry of out per
// chunk of 8 slices, the chunks shared out over the warps of the cluster.
template <int NT>
__device__ __forceinline__ void radius_chunks(const Share &sh, const SellMat &A, int s0, int s1,
                                              const double *z, const double *z0, double *out) {
  constexpr int W = NT / kWarp;
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x >> 5;
  const int nch = (s1 - s0 + kCheckChunk - 1) / kCheckChunk;
  for (int c = sh.rank * W + warp; c < nch; c += sh.P * W) {
    double q = 0.0;
    const int e = min(s1, s0 + (c + 1) * kCheckChunk);
    for (int s = s0 + c * kCheckChunk; s < e; ++s) q = slice_dist2(A, s, z, z0, q);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(kFull, q, o);
    if (lane == 0) __stcg(out + c, q);
  }
}

__device__ __forceinline__ const float *values(const SellMat &A, float) { return A.valf; }
__device__ __forceinline__ const double *values(const SellMat &A, double) { return A.val; }

// ------------------------------------------------------- state of a problem

// The single problem's state (DevState), its weights and trace.
struct SingleIO {
  static constexpr bool kBatch = false;
  DevState *st;
  double *w, *trace;
  unsigned gen = 0;
  __device__ __forceinline__ bool running() const { return st->status == kRunning; }
  __device__ __forceinline__ int iterations() const { return st->K; }
  __device__ void load(Scalars &c) const {
    c = Scalars{st->tau,    st->sigma,      st->omega,  st->norm_b, st->norm_c,
                st->tol,    st->beta,       st->rho_stored, st->last_r, st->mix_s,
                st->t0,     st->restarts,   st->tau0,   st->fixed_len,
                st->K,      st->scheme,     1,          st->returned};
  }
  __device__ void expired() const { st->status = kStatusTimeout; }
  __device__ void record(const Header &h, int64_t t) const {
    st->bar_gen = gen;
    st->iters += h.sc.K;
    st->checks += 1;
    for (int i = 0; i < 5; ++i) {
      st->kkt_a[i] = h.kkt[0][i];
      st->kkt_c[i] = h.kkt[1][i];
    }
    st->returned = h.returned;
    if (h.status != kRunning) {  // not over another block's expired wait
      atomicCAS(&st->status, kRunning, h.status);
      return;
    }
    if (trace && st->trace_count < st->trace_cap) {
      double *row = trace + 6 * st->trace_count;
      row[0] = (double)st->iters;
      row[1] = h.rho;
      row[2] = (double)h.restart;
      row[3] = h.kkt[0][4];
      row[4] = h.kkt[1][4];
      row[5] = h.r;
    }
    st->trace_count += 1;
    st->last_rho = h.rho;
    st->last_r = h.r;
    st->use_cur = h.use_cur;
    st->restart_now = h.restart;
    st->t0 = h.restart ? 0 : t;
    if (h.restart) {
      st->rho_stored = h.rho;
      st->restarts += 1;
      st->mix_s = h.mix_s;
    }
  }
};

// A problem of a batch (BInst): counters, restart rule and iteration limit as
// in the batch's check chain (b_pre_check, b_finalize, b_decide).
struct BatchIO {
  static constexpr bool kBatch = true;
  BInst *B;
  BGlobal *G;
  __device__ __forceinline__ bool running() const { return B->status == kRunning; }
  __device__ __forceinline__ int iterations() const { return G->Kb; }
  __device__ void load(Scalars &c) const {
    c = Scalars{B->tau,   B->sigma,     B->omega,      B->norm_b, B->norm_c,
                G->tol,   G->beta,      B->rho_stored, B->last_r, B->mix_s,
                B->t0,    B->restarts,  B->tau0,       B->fixed_len,
                G->Kb,    G->scheme,    B->since + G->Kb >= B->K ? 1 : 0, B->returned};
  }
  __device__ void expired() const {}
  __device__ void record(const Header &h, int64_t t) const {
    B->iters += h.sc.K;
    B->since += h.sc.K;
    B->due = h.sc.due;
    B->restart_now = 0;
    B->use_cur = 0;
    if (h.sc.due) {
      B->checks += 1;
      for (int i = 0; i < 5; ++i) {
        B->kkt_a[i] = h.kkt[0][i];
        B->kkt_c[i] = h.kkt[1][i];
      }
      B->returned = h.returned;
      if (h.status != kRunning) {
        B->status = h.status;
        return;
      }
      B->last_rho = h.rho;
      B->last_r = h.r;
      B->use_cur = h.use_cur;
      B->restart_now = h.restart;
      B->since = 0;
    }
    B->t0 = h.restart ? 0 : t;
    if (h.restart) {
      B->rho_stored = h.rho;
      B->restarts += 1;
      B->mix_s = h.mix_s;
    }
    if (B->iters >= B->iter_cap) B->status = kStatusIterLimit;  // the check's restart still happens
    else atomicAdd(&G->running, 1);
  }
};

// ------------------------------------------------------------------ the block
//
// K iterations and, when due, the check of one problem by the blocks of one
// group.  T: float for mixed precision.  RES: the block's slices stay in shared
// memory (else they are read from global memory in every pass).  LEAN: 64
// registers per thread, so what the check needs is laid out again after the
// iterations instead of being kept through them, and 4 gathers are in flight
// (5k x 25k in mixed precision, us per iteration: 7.5 without either, 7.2 with the
// first, 7.0 with both, 6.9 with 128 registers).
template <typename T, int NT, bool RES, bool LEAN, class IO, class Link>
__device__ __forceinline__ void run_block(unsigned char *smem, const ResidentArgs &a,
                                          const Share &sh, IO &io, Link &link) {
  constexpr bool MIX = sizeof(T) == 4;
  constexpr bool SHIFT = Link::kCluster && !RES;  // resident indices count from the problem's first
  constexpr int W = NT / kWarp;
  constexpr int U = LEAN ? kLeanU : kU;
  const int P = sh.P, tid = (int)threadIdx.x;
  const int lane = tid & (kWarp - 1), warp = tid >> 5;
  const int nc = sh.nc, nr = sh.nr, K = io.iterations();

  // ---- layout of shared memory
  Sm<T> S;
  unsigned char *const behind = lay_lists<T, NT, Link::kCluster>(S, smem, sh, K);
  if (warp == 0)
    build_slices<RES>(a.AT, sh.c0, nc, sh.stride, sh.cfirst, S.cs, &S.h->ncl, &S.h->nce);
  else if (warp == 1)
    build_slices<RES>(a.A, sh.r0, nr, sh.stride, sh.rfirst, S.rs, &S.h->nrl, &S.h->nre);
  else if (warp == 2 && lane == 0) {
    Scalars sc;
    io.load(sc);
    S.h->sc = sc;
    S.h->dead = 0;
    const double sw = sqrt(sc.omega);
    S.h->sw = sw;
    S.h->isw = 1.0 / sw;
    S.h->inv = MIX ? 1.0 / sc.mix_s : 1.0;
  }
  __syncthreads();
  const int ncl = S.h->ncl, nrl = S.h->nrl;
  for (int k = tid; k < K; k += NT) S.w[k] = 1.0 / (double)(S.h->sc.t0 + k + 1);
  lay_arrays<T, RES>(S, behind, ncl, nrl);
  const int32_t *cidx, *ridx;  // indexed by LSlice::soff
  const T *cval, *rval;
  if constexpr (RES) {
    cidx = S.cidx;
    cval = S.cval;
    ridx = S.ridx;
    rval = S.rval;
  } else {
    const int64_t oc = a.AT.info[sh.cfirst].off, orr = a.A.info[sh.rfirst].off;
    cidx = a.AT.idx + oc;
    cval = values(a.AT, T(0)) + oc;
    ridx = a.A.idx + orr;
    rval = values(a.A, T(0)) + orr;
  }

  // ---- owned state
  load_slices<T, NT, RES>(a.AT, values(a.AT, T(0)), S.cs, nc, sh.row0, S.crow, S.cidx, S.cval);
  load_slices<T, NT, RES>(a.A, values(a.A, T(0)), S.rs, nr, sh.col0, S.rrow, S.ridx, S.rval);
  __syncthreads();
  if constexpr (Link::kCluster) {
    link.ex = S.ex;
    link.ey = S.ey;
    link.ax = (uint32_t)__cvta_generic_to_shared(S.ex);
    link.ay = (uint32_t)__cvta_generic_to_shared(S.ey);
    for (int i = tid; i < sh.nrow; i += NT) {
      if constexpr (MIX) S.ey[i] = a.mv.dy[sh.row0 + i];
      else S.ey[i] = a.v.y[sh.row0 + i];
    }
  } else {
    link.gen = io.st->bar_gen;
    link.dead = &S.h->dead;
  }
  for (int s = tid; s < nrl; s += NT) {
    const int i = S.rrow[s];
    if constexpr (MIX) {
      S.y[s] = a.mv.dy[i];
      S.b[s] = a.mv.bf[i];
      S.yb[s] = a.mv.dybar[i];
      S.lo[s] = a.mv.ylo[i];
      S.hi[s] = a.mv.yhi[i];
    } else {
      S.y[s] = a.v.y[i];
      S.b[s] = a.v.b[i];
      S.yb[s] = a.v.ybar[i];
      S.rt[s] = (int)a.v.row_type[i];
    }
  }
  for (int s = tid; s < ncl; s += NT) {
    const int j = S.crow[s];
    if constexpr (MIX) {
      S.c[s] = a.mv.cf[j];
      S.x[s] = a.mv.dx[j];
      S.xb[s] = a.mv.dxbar[j];
      S.lf[s] = a.mv.lf[j];
      S.uf[s] = a.mv.uf[j];
    } else {
      S.c[s] = a.v.c[j];
      S.x[s] = a.v.x[j];
      S.xb[s] = a.v.xbar[j];
      S.lk[s] = a.v.lbk[j];
      S.uk[s] = a.v.ubk[j];
    }
  }
  const T tau = (T)S.h->sc.tau, sigma = (T)S.h->sc.sigma;
  // a cluster's blocks store into one another's copies only once all of them
  // have started and filled theirs
  if (Link::kCluster) link.sync();
  else __syncthreads();

  // ---- K iterations.  The averages, which nothing waits for, are updated
  // between a barrier's arrival and its wait.
  bool lost = false;
  for (int k = 0; k < K; ++k) {
    const double w = S.w[k];
    for (int q = 0, i; (i = pick<NT>(q, warp)) < nc; ++q) {
      const LSlice sl = S.cs[i];
      const int lg = sl.lg(), r = lane >> lg, s = sl.slot0 + r;
      const bool owner = (lane & ((1 << lg) - 1)) == 0 && r < sl.rows();
      const T neg_g = slice_sum<SHIFT, U>(owner ? -S.c[s] : T(0), cidx + sl.soff + lane,
                                       cval + sl.soff + lane, sl.steps(), lg, link.y(), sh.row0);
      if (owner) {
        const T x = S.x[s];
        T xn;
        if constexpr (MIX) {
          xn = fminf(fmaxf(fmaf(tau, neg_g, x), S.lf[s]), S.uf[s]);
        } else {
          long long key = ord_key(__double_as_longlong(fma(tau, neg_g, x)));
          const long long lk = S.lk[s], uk = S.uk[s];
          key = key < lk ? lk : key;
          key = key > uk ? uk : key;
          xn = __longlong_as_double(ord_key(key));
        }
        link.put_x(S.crow[s], fma_t(T(2), xn, -x));
        S.x[s] = xn;
      }
    }
    link.arrive();
    for (int s = tid; s < ncl; s += NT) {
      const double xb = S.xb[s];
      S.xb[s] = fma(w, (double)S.x[s] - xb, xb);
    }
    if (!link.wait()) {
      lost = true;
      break;
    }
    for (int q = 0, i; (i = pick<NT>(q, warp)) < nr; ++q) {
      const LSlice sl = S.rs[i];
      const int lg = sl.lg(), r = lane >> lg, s = sl.slot0 + r;
      const bool owner = (lane & ((1 << lg) - 1)) == 0 && r < sl.rows();
      const T res = slice_sum<SHIFT, U>(owner ? -S.b[s] : T(0), ridx + sl.soff + lane,
                                     rval + sl.soff + lane, sl.steps(), lg, link.x(), sh.col0);
      if (owner) {
        const T y = S.y[s];
        T yn;
        if constexpr (MIX) {
          yn = fminf(fmaxf(fmaf(-sigma, res, y), S.lo[s]), S.hi[s]);
        } else {
          long long bits = __double_as_longlong(fma(-sigma, res, y));
          const int t = S.rt[s];
          if (t == 1 && bits < 0) bits = 0;
          else if (t == 2 && bits > 0) bits = 0;
          yn = __longlong_as_double(bits);
        }
        link.put_y(S.rrow[s], yn);
        S.y[s] = yn;
      }
    }
    if (k + 1 < K) link.arrive();  // the barrier after the publication covers the last pass
    else __syncthreads();
    for (int s = tid; s < nrl; s += NT) {
      const double yb = S.yb[s];
      S.yb[s] = fma(w, (double)S.y[s] - yb, yb);
    }
    if (k + 1 < K && !link.wait()) {
      lost = true;
      break;
    }
  }

  if constexpr (LEAN) {
    int zero = 0;
    asm volatile("" : "+r"(zero));  // keeps the compiler from carrying the pointers over
    lay_arrays<T, RES>(S, lay_lists<T, NT, Link::kCluster>(S, smem + zero, sh, K), S.h->ncl, S.h->nrl);
  }

  // ---- publish the iterate and the average (in mixed precision also in FP64)
  const double inv = S.h->inv;
  for (int s = tid; s < ncl; s += NT) {
    const int j = S.crow[s];
    if constexpr (MIX) {
      a.mv.dx[j] = S.x[s];
      a.mv.dxbar[j] = S.xb[s];
      const double x0 = a.v.x0[j], l = a.v.lb[j], u = a.v.ub[j];
      a.v.x[j] = fmin(fmax(fma((double)S.x[s], inv, x0), l), u);
      a.v.xbar[j] = fmin(fmax(fma(S.xb[s], inv, x0), l), u);
    } else {
      a.v.x[j] = S.x[s];
      a.v.xbar[j] = S.xb[s];
    }
  }
  for (int s = tid; s < nrl; s += NT) {
    const int i = S.rrow[s];
    if constexpr (MIX) {
      a.mv.dy[i] = S.y[s];
      a.mv.dybar[i] = S.yb[s];
      const int t = a.v.row_type[i];
      const double lo = (t == 1) ? 0.0 : -INFINITY, hi = (t == 2) ? 0.0 : INFINITY;
      const double y0 = a.v.y0[i];
      a.v.y[i] = fmin(fmax(fma((double)S.y[s], inv, y0), lo), hi);
      a.v.ybar[i] = fmin(fmax(fma(S.yb[s], inv, y0), lo), hi);
    } else {
      a.v.y[i] = S.y[s];
      a.v.ybar[i] = S.yb[s];
    }
  }
  if (lost || !link.sync()) {
    if (tid == 0) io.expired();
    return;
  }
  const int64_t t = S.h->sc.t0 + K;
  if (!S.h->sc.due) {
    if (sh.rank == 0 && tid == 0) {
      S.h->restart = 0;
      io.record(*S.h, t);
    }
    return;
  }

  // ---- check: A^T [ybar, y], A [xbar, x] and their epilogues
  const int scheme = S.h->sc.scheme;
  const bool gap_a = scheme == kSchemeAdaptive || scheme == kSchemeFlexible;
  const bool gap_c = scheme == kSchemeFlexible;
  const GapOut go[2] = {GapOut{a.cs.keys[0], a.cs.d2[0], a.cs.g2[0], a.cs.gd[0]},
                        GapOut{a.cs.keys[1], a.cs.d2[1], a.cs.g2[1], a.cs.gd[1]}};
  {
    const double *sc = nullptr, *sr = nullptr;
    if constexpr (!MIX && RES) {
      sc = S.cval;
      sr = S.rval;
    }
    check_sums<NT, RES>(S.cs, nc, S.cidx, sc, a.AT, sh.row0, a.v.ybar, a.v.y, S.cs0, S.cs1);
    check_sums<NT, RES>(S.rs, nr, S.ridx, sr, a.A, sh.col0, a.v.xbar, a.v.x, S.rs0, S.rs1);
  }
  __syncthreads();
  // owned columns, then (from a whole warp on) owned rows, one per thread
  const int rfirst = (ncl + kWarp - 1) & ~(kWarp - 1), nown = rfirst + nrl;
  const int busy = min(W, (nown + kWarp - 1) / kWarp);
  double *part = a.part + (size_t)P * kResPart * (blockIdx.x / P);
  const int ncand = gap_c ? 2 : gap_a ? 1 : 0;
  const int nrad = a.cs.cols_grid + a.cs.rows_grid;
  if constexpr (MIX) {
    for (int c = 0; c < ncand; ++c) {
      double *rp = a.rpart + (size_t)c * nrad;
      if constexpr (IO::kBatch) {
        const BInst &B = *io.B;
        radius_chunks<NT>(sh, a.AT, B.cs0, B.cs1, c ? a.v.x : a.v.xbar, a.v.x0, rp + B.cc0);
        radius_chunks<NT>(sh, a.A, B.rs0, B.rs1, c ? a.v.y : a.v.ybar, a.v.y0,
                          rp + a.cs.cols_grid + B.rc0);
      } else {
        radius_parts<NT>(a, sh, S.red, c, rp);
      }
    }
  }
  if (warp < busy) {
    CheckColsEpi ce{};
    CheckRowsEpi re{};
    ce.sw = re.sw = S.h->sw;
    ce.isw = re.isw = S.h->isw;
    re.off = a.n;
#pragma unroll
    for (int i = 0; i < NQ; ++i) ce.q[i] = 0.0;
    for (int s = tid; s < ncl; s += NT) {
      const int j = S.crow[s];
      const CheckColsEpi::Pre pre{a.v.c[j], a.v.lb[j], a.v.ub[j], 0.0, 0.0, a.v.x0[j]};
      const bool lf = dbits(pre.lb) != kNegInfBits, uf = dbits(pre.ub) != kPosInfBits;
      const double lam_a = pre.c - S.cs0[s], lam_c = pre.c - S.cs1[s];
      const double xa = a.v.xbar[j], xc = a.v.x[j];
      if (MIX) {
        a.mv.lam[0][j] = lam_a;
        a.mv.lam[1][j] = lam_c;
      }
      ce.candidate(j, lam_a, xa, pre, lf, uf, Q_RD2_A, Q_DOBJ_A, Q_POBJ_A, Q_RRX_A, Q_D2_A,
                   Q_GD_A, Q_G2INF_A, gap_a, go[0]);
      ce.candidate(j, lam_c, xc, pre, lf, uf, Q_RD2_C, Q_DOBJ_C, Q_POBJ_C, Q_RRX_C, Q_D2_C,
                   Q_GD_C, Q_G2INF_C, gap_c, go[1]);
      if (!(finite_d(lam_a) && finite_d(lam_c) && finite_d(xa) && finite_d(xc))) ce.q[Q_BAD] = 1.0;
    }
#pragma unroll
    for (int i = 0; i < NQ; ++i) re.q[i] = ce.q[i];
    for (int e = tid; e < nown; e += NT) {
      if (e < rfirst) continue;
      const int s = e - rfirst, i = S.rrow[s];
      const CheckRowsEpi::Pre pre{a.v.b[i], 0.0, 0.0, a.v.y0[i], (int)a.v.row_type[i]};
      const double ax_a = S.rs0[s], ax_c = S.rs1[s], ya = a.v.ybar[i], yc = a.v.y[i];
      const double va = ax_a - pre.b, vc = ax_c - pre.b;
      if (MIX) {
        a.mv.gy[0][i] = va;
        a.mv.gy[1][i] = vc;
      }
      re.candidate(i, va, ya, pre, Q_RP2_A, Q_DOBJ_A, Q_RRY_A, Q_D2_A, Q_GD_A, Q_G2INF_A, gap_a,
                   go[0]);
      re.candidate(i, vc, yc, pre, Q_RP2_C, Q_DOBJ_C, Q_RRY_C, Q_D2_C, Q_GD_C, Q_G2INF_C, gap_c,
                   go[1]);
      if (!(finite_d(ax_a) && finite_d(ax_c) && finite_d(ya) && finite_d(yc))) re.q[Q_BAD] = 1.0;
    }
    // sums of the warp, of the block, of the group
    double u[16], v[4];
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = re.q[i];
    v[0] = re.q[16];
    v[1] = re.q[17];
    v[2] = re.q[18];
    v[3] = 0.0;
    const double su = warp_sum_multi<16>(u), sv = warp_sum_multi<4>(v);
    if ((lane & 1) == 0) S.red[warp * 32 + (lane >> 1)] = su;
    if ((lane & 7) == 0) S.red[warp * 32 + 16 + (lane >> 3)] = sv;
  }
  __syncthreads();
  if (tid < NQ) {
    double s = 0.0;
    for (int i = 0; i < busy; ++i) s += S.red[i * 32 + tid];
    if (P > 1) __stcg(part + (size_t)sh.rank * kResPart + tid, s);
    else S.tot[tid] = s;
  }
  if (P > 1) {
    if (!link.sync()) {
      if (tid == 0) io.expired();
      return;
    }
    for (int i = warp; i < NQ; i += W) {
      const double s = sum_parts(part, kResPart, i, P);
      if (lane == 0) S.tot[i] = s;
    }
  }
  __syncthreads();

  if constexpr (MIX) {
    for (int c = 0; c < ncand; ++c) {
      double rx, ry;
      const double *rp = a.rpart + (size_t)c * nrad;
      if constexpr (IO::kBatch) {
        const BInst &B = *io.B;
        rx = sum_parts(rp + B.cc0, 1, 0, B.cc1 - B.cc0);
        ry = sum_parts(rp + a.cs.cols_grid + B.rc0, 1, 0, B.rc1 - B.rc0);
      } else {
        rx = radius_total(rp, nrad, 0, a.cs.cols_grid, S.red);
        ry = radius_total(rp, nrad, a.cs.cols_grid, nrad, S.red);
      }
      if (tid == 0) {
        S.tot[c ? Q_RRX_C : Q_RRX_A] = rx;
        S.tot[c ? Q_RRY_C : Q_RRY_A] = ry;
      }
    }
    __syncthreads();
  }

  // ---- termination and search setup: lane 0 for the average, lane 1 for the
  // current iterate; every block decides from the same sums, one records
  const double *tot = S.tot;
  if (warp == 0) {
    const Scalars &sc = S.h->sc;
    const int c = lane & 1;
    double k5[5];
    kkt_from(tot, Q_RP2_A + c, Q_RD2_A + c, Q_POBJ_A + c, Q_DOBJ_A + c, sc.norm_b, sc.norm_c, k5);
    const double rel = k5[4], rel_a = __shfl_sync(kFull, rel, 0), rel_c = __shfl_sync(kFull, rel, 1);
    int status = kRunning, returned = 0;
    if (tot[Q_BAD] > 0.0 || !isfinite(rel_a) || !isfinite(rel_c)) {
      status = kStatusNumerical;
      returned = sc.returned;
    } else if (rel_a <= sc.tol) {
      status = kStatusOK;
    } else if (rel_c <= sc.tol) {
      status = kStatusOK;
      returned = 1;
    } else {
      returned = (rel_a <= rel_c) ? 0 : 1;
    }
    double r2 = 0.0, rho_r = 0.0;
    int done = 1;
    if (status == kRunning && (c ? gap_c : gap_a)) {
      const double om = sc.omega;
      const double r = sqrt(om * tot[c ? Q_RRX_C : Q_RRX_A] + tot[c ? Q_RRY_C : Q_RRY_A] / om);
      r2 = r * r;
      done = (r == 0.0);
      if (!done && tot[c ? Q_G2INF_C : Q_G2INF_A] == 0.0 && tot[c ? Q_D2_C : Q_D2_A] <= r2) {
        done = 1;  // the full clamp lies inside the ball
        rho_r = tot[c ? Q_GD_C : Q_GD_A];
      }
    }
    if (lane < 2) {
#pragma unroll
      for (int i = 0; i < 5; ++i) S.h->kkt[c][i] = k5[i];
      S.h->r2[c] = r2;
      S.h->rho_r[c] = rho_r;
      S.h->lam[c] = 0.0;
      S.h->count[c] = -1;
      S.h->done[c] = done;
      if (c == 0) {
        S.h->status = status;
        S.h->returned = returned;
      }
    }
  }
  __syncthreads();

  // ---- multiplier search: Newton steps on the block's own breakpoints
  for (int step = 0; step < kNewtonMax; ++step) {
    const bool done0 = S.h->done[0] != 0, done1 = S.h->done[1] != 0;
    if (done0 && done1) break;
    if (warp < busy) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (c ? done1 : done0) continue;
        const uint64_t lk = (uint64_t)dbits(S.h->lam[c]);
        double u[4] = {0.0, 0.0, 0.0, 0.0};
        int cnt = 0;
        auto add = [&](int64_t e) {
          const uint64_t key = go[c].keys[e];
          const double d2 = go[c].d2[e], gd = go[c].gd[e], g2 = go[c].g2[e];
          const bool in = key <= lk;
          u[0] += in ? d2 : 0.0;
          u[1] += in ? gd : 0.0;
          u[2] += in || key == kNoKey ? 0.0 : g2;
          cnt += in ? 1 : 0;
        };
        for (int s = tid; s < ncl; s += NT) add(S.crow[s]);
        for (int e = tid; e < nown; e += NT)
          if (e >= rfirst) add((int64_t)a.n + S.rrow[e - rfirst]);
        const double su = warp_sum_multi<4>(u);
        cnt = __reduce_add_sync(kFull, cnt);
        if ((lane & 7) == 0) S.red[warp * 32 + 4 * c + (lane >> 3)] = lane == 24 ? (double)cnt : su;
      }
    }
    __syncthreads();
    // two buffers in turn: a block may still read the last step's sums
    double *np = a.npart + (size_t)(blockIdx.x / P) * 2 * P * 8 + (size_t)(step & 1) * P * 8;
    if (tid < 8 && !(tid < 4 ? done0 : done1)) {
      double s = 0.0;
      for (int i = 0; i < busy; ++i) s += S.red[i * 32 + tid];
      if (P > 1) __stcg(np + (size_t)sh.rank * 8 + tid, s);
      else S.nw[tid] = s;
    }
    if (P > 1) {
      if (!link.sync()) {
        if (tid == 0) io.expired();
        return;
      }
      if (warp < 8 && !(warp < 4 ? done0 : done1)) {
        const double s = sum_parts(np, 8, warp, P);
        if (lane == 0) S.nw[warp] = s;
      }
    }
    __syncthreads();
    if (warp == 0 && lane < 2 && !(lane ? done1 : done0)) {
      const int c = lane;
      const double A = S.nw[4 * c], E = S.nw[4 * c + 1];
      const double B = S.nw[4 * c + 2] + tot[c ? Q_G2INF_C : Q_G2INF_A];
      const int same = (int)S.nw[4 * c + 3];
      S.h->done[c] = newton_next(A, E, B, same, S.h->r2[c], step, S.h->lam[c], S.h->rho_r[c],
                                 S.h->count[c]);
    }
    __syncthreads();
  }

  // ---- restart decision (Eq. adaptive-restart-scheme / flexible / fixed)
  if (tid == 0) {
    const Scalars &sc = S.h->sc;
    double rho = NAN, r = sc.last_r;
    int use_cur = 0, restart = 0;
    if (S.h->status == kRunning) {
      if (gap_a) {
        r = sqrt(S.h->r2[0]);
        rho = S.h->r2[0] > 0.0 ? S.h->rho_r[0] / r : 0.0;
        if (gap_c) {
          const double rc = sqrt(S.h->r2[1]);
          const double rho_c = S.h->r2[1] > 0.0 ? S.h->rho_r[1] / rc : 0.0;
          if (rho_c < rho) {
            use_cur = 1;
            rho = rho_c;
            r = rc;
          }
        }
        restart = (sc.restarts == 0) ? (t >= sc.tau0) : (rho <= sc.beta * sc.rho_stored);
      } else if (scheme == kSchemeFixed) {
        restart = (t >= sc.fixed_len);
      }
    }
    S.h->rho = rho;
    S.h->r = r;
    S.h->use_cur = use_cur;
    S.h->restart = restart;
    S.h->mix_s = (restart && MIX && r > 0.0 && isfinite(r)) ? fmin(1.0 / r, 1e12) : sc.mix_s;
    if (sh.rank == 0) {
      if constexpr (!Link::kCluster) io.gen = link.gen;
      io.record(*S.h, t);
    }
  }
  __syncthreads();
  const int use_cur = S.h->use_cur, restart = S.h->restart;
  const double mix_s = S.h->mix_s;
  if (S.h->status != kRunning) return;
  if (sh.rank == 0 && a.w)  // the next block's weights, for iterations outside this kernel
    for (int k = tid; k < K; k += NT) a.w[k] = 1.0 / (double)((restart ? 0 : t) + k + 1);
  if (!restart && !use_cur) return;

  // ---- restart (or the flexible scheme's replacement of the average), owned part
  for (int s = tid; s < ncl; s += NT) {
    const int j = S.crow[s];
    const double x = (use_cur ? a.v.x : a.v.xbar)[j];
    a.v.xbar[j] = x;
    if (restart) {
      a.v.x0[j] = x;
      a.v.x[j] = x;
    }
    if constexpr (MIX) {
      if (restart) {
        a.mv.cf[j] = (float)(mix_s * a.mv.lam[use_cur][j]);
        a.mv.lf[j] = (float)(mix_s * (a.v.lb[j] - x));
        a.mv.uf[j] = (float)(mix_s * (a.v.ub[j] - x));
        a.mv.dx[j] = 0.0f;
        a.mv.dxhat[j] = 0.0f;
        a.mv.dxbar[j] = 0.0;
      } else {
        a.mv.dxbar[j] = (double)S.x[s];
      }
    }
  }
  for (int s = tid; s < nrl; s += NT) {
    const int i = S.rrow[s];
    const double y = (use_cur ? a.v.y : a.v.ybar)[i];
    a.v.ybar[i] = y;
    if (restart) {
      a.v.y0[i] = y;
      a.v.y[i] = y;
    }
    if constexpr (MIX) {
      if (restart) {
        const int ty = a.v.row_type[i];
        const double lo = (ty == 1) ? 0.0 : -INFINITY, hi = (ty == 2) ? 0.0 : INFINITY;
        a.mv.bf[i] = (float)(-mix_s * a.mv.gy[use_cur][i]);
        a.mv.ylo[i] = (float)(mix_s * (lo - y));
        a.mv.yhi[i] = (float)(mix_s * (hi - y));
        a.mv.dy[i] = 0.0f;
        a.mv.dybar[i] = 0.0;
      } else {
        a.mv.dybar[i] = (double)S.y[s];
      }
    }
  }
}

// ------------------------------------------------------------------ adjoint
//
// The whole of lp_backward (lp_batch_backward: of one problem) by the blocks of
// one group: for every recorded block of K iterations, last first, the forward
// steps from its checkpoint with their clamp and projection masks, then one
// adjoint step per iteration in reverse (the recurrence of AdjColsEpi and
// AdjRowsEpi).  Launched pass by pass this took four launches per iteration, 6 us
// each; here a pass costs what it does in run_block (2k x 5k, 512 iterations, setup,
// forward and backward: 12.1 ms instead of 19.3).  The running averages are recomputed only for the last
// block, whose end is the state that the call leaves behind.
template <int NT, class Link>
__device__ __forceinline__ void run_adjoint(unsigned char *smem, const AdjointArgs &q,
                                            const Share &sh, int problem, double tau, double sigma,
                                            unsigned gen, Link &link) {
  const ResidentArgs &a = q.r;
  const int tid = (int)threadIdx.x, lane = tid & (kWarp - 1), warp = tid >> 5;
  const int nc = sh.nc, nr = sh.nr, K = q.K;
  unsigned char *p = smem;
  Header *h = (Header *)carve(p, sizeof(Header));
  double *ex = nullptr, *ey = nullptr;
  if (Link::kCluster) {  // at the same place in every block: owners store into all of them
    ex = (double *)carve(p, 8 * (size_t)sh.ncol);
    ey = (double *)carve(p, 8 * (size_t)sh.nrow);
  }
  LSlice *cs = (LSlice *)carve(p, sizeof(LSlice) * nc), *rs = (LSlice *)carve(p, sizeof(LSlice) * nr);
  double *w = (double *)carve(p, sizeof(double) * K);
  if (warp == 0) build_slices<true>(a.AT, sh.c0, nc, sh.stride, sh.cfirst, cs, &h->ncl, &h->nce);
  else if (warp == 1) build_slices<true>(a.A, sh.r0, nr, sh.stride, sh.rfirst, rs, &h->nrl, &h->nre);
  if (tid == 0) h->dead = 0;
  __syncthreads();
  const int ncl = h->ncl, nrl = h->nrl;
  auto array = [&](int count) { return (double *)carve(p, 8 * (size_t)count); };
  int32_t *crow = (int32_t *)carve(p, 4 * (size_t)ncl), *rrow = (int32_t *)carve(p, 4 * (size_t)nrl);
  int32_t *rt = (int32_t *)carve(p, 4 * (size_t)nrl);
  double *c = array(ncl), *x = array(ncl), *xb = array(ncl), *ax = array(ncl), *axb = array(ncl),
         *ac = array(ncl);
  long long *lk = (long long *)array(ncl), *uk = (long long *)array(ncl);
  double *b = array(nrl), *y = array(nrl), *yb = array(nrl), *ay = array(nrl), *ayb = array(nrl),
         *ab = array(nrl);
  int32_t *cidx = (int32_t *)carve(p, 4 * (size_t)h->nce);
  double *cval = array(h->nce);
  int32_t *ridx = (int32_t *)carve(p, 4 * (size_t)h->nre);
  double *rval = array(h->nre);
  load_slices<double, NT, true>(a.AT, a.AT.val, cs, nc, sh.row0, crow, cidx, cval);
  load_slices<double, NT, true>(a.A, a.A.val, rs, nr, sh.col0, rrow, ridx, rval);
  __syncthreads();
  if constexpr (Link::kCluster) {
    link.ex = ex;
    link.ey = ey;
    link.ax = (uint32_t)__cvta_generic_to_shared(ex);
    link.ay = (uint32_t)__cvta_generic_to_shared(ey);
  } else {
    link.gen = gen;
    link.dead = &h->dead;
  }
  for (int s = tid; s < ncl; s += NT) {
    const int j = crow[s];
    c[s] = a.v.c[j];
    lk[s] = a.v.lbk[j];
    uk[s] = a.v.ubk[j];
    ax[s] = 0.0;
    axb[s] = q.adj.axb[j];
    ac[s] = 0.0;
  }
  for (int s = tid; s < nrl; s += NT) {
    const int i = rrow[s];
    b[s] = a.v.b[i];
    rt[s] = (int)a.v.row_type[i];
    ay[s] = 0.0;
    ayb[s] = q.adj.ayb[i];
    ab[s] = 0.0;
  }
  __syncthreads();
  // sum of one local column / row slice, with its owner lane's slot (-1: none)
  auto col_sum = [&](int i, bool init, int *slot) {
    const LSlice sl = cs[i];
    const int lg = sl.lg(), r = lane >> lg, s = sl.slot0 + r;
    *slot = (lane & ((1 << lg) - 1)) == 0 && r < sl.rows() ? s : -1;
    return slice_sum<false>(init && *slot >= 0 ? -c[s] : 0.0, cidx + sl.soff + lane,
                            cval + sl.soff + lane, sl.steps(), lg, link.y(), 0);
  };
  auto row_sum = [&](int i, bool init, int *slot) {
    const LSlice sl = rs[i];
    const int lg = sl.lg(), r = lane >> lg, s = sl.slot0 + r;
    *slot = (lane & ((1 << lg) - 1)) == 0 && r < sl.rows() ? s : -1;
    return slice_sum<false>(init && *slot >= 0 ? -b[s] : 0.0, ridx + sl.soff + lane,
                            rval + sl.soff + lane, sl.steps(), lg, link.x(), 0);
  };

  bool ok = true;
  for (int64_t blk = q.blocks - 1; ok && blk >= 0; --blk) {
    const double *ck = q.ckpt + blk * q.slot;
    const bool final = blk == q.blocks - 1;
    const int64_t t0 = q.t0[blk * q.count + problem];
    const int restarted = q.restarted[blk * q.count + problem];
    for (int k = tid; k < K; k += NT) w[k] = 1.0 / (double)(t0 + k + 1);
    for (int s = tid; s < ncl; s += NT) {
      const int j = crow[s];
      x[s] = ck[j];
      if (final) xb[s] = ck[(int64_t)a.n + a.m + j];
    }
    for (int s = tid; s < nrl; s += NT) {
      const int i = rrow[s];
      y[s] = ck[(int64_t)a.n + i];
      if (final) yb[s] = ck[2 * (int64_t)a.n + a.m + i];
    }
    // a cluster's first stores into the other blocks' copies wait until all have started
    if (Link::kCluster) ok = link.sync();
    else __syncthreads();
    for (int s = tid; s < nrl; s += NT) link.put_y(rrow[s], y[s]);
    ok = ok && link.sync();
    // ---- forward steps with masks
    for (int k = 0; ok && k < K; ++k) {
      for (int r = 0, i, s; (i = pick<NT>(r, warp)) < nc; ++r) {
        const double neg_g = col_sum(i, true, &s);
        if (s >= 0) {
          const double xo = x[s];
          long long key = ord_key(__double_as_longlong(fma(tau, neg_g, xo)));
          const long long lo = lk[s], hi = uk[s];
          q.mask_x[(int64_t)k * a.n + crow[s]] = key > lo && key < hi ? 1 : 0;
          key = key < lo ? lo : key;
          key = key > hi ? hi : key;
          const double xn = __longlong_as_double(ord_key(key));
          link.put_x(crow[s], fma(2.0, xn, -xo));
          x[s] = xn;
          if (final) xb[s] = fma(w[k], xn - xb[s], xb[s]);
        }
      }
      if (!(ok = link.sync())) break;
      for (int r = 0, i, s; (i = pick<NT>(r, warp)) < nr; ++r) {
        const double res = row_sum(i, true, &s);
        if (s >= 0) {
          long long bits = __double_as_longlong(fma(-sigma, res, y[s]));
          const int t = rt[s];
          q.mask_y[(int64_t)k * q.mstride + rrow[s]] =
              t == 0 || (t == 1 && bits > 0) || (t == 2 && bits < 0) ? 1 : 0;
          if ((t == 1 && bits < 0) || (t == 2 && bits > 0)) bits = 0;
          const double yn = __longlong_as_double(bits);
          if (k + 1 < K) link.put_y(rrow[s], yn);  // the last y is gathered by nobody
          y[s] = yn;
          if (final) yb[s] = fma(w[k], yn - yb[s], yb[s]);
        }
      }
      if (k + 1 < K) ok = link.sync();
    }
    if (!ok) break;
    __syncthreads();
    if (final) {  // the state of the recorded solve (its last check may have restarted)
      for (int s = tid; s < ncl; s += NT) {
        a.v.x[crow[s]] = restarted ? xb[s] : x[s];
        a.v.xbar[crow[s]] = xb[s];
      }
      for (int s = tid; s < nrl; s += NT) {
        a.v.y[rrow[s]] = restarted ? yb[s] : y[s];
        a.v.ybar[rrow[s]] = yb[s];
      }
    }
    // ---- start of the reverse block: its restart, then u of its last step
    if (restarted)
      for (int s = tid; s < ncl; s += NT) {
        axb[s] += ax[s];
        ax[s] = 0.0;
      }
    for (int s = tid; s < nrl; s += NT) {
      if (restarted) {
        ayb[s] += ay[s];
        ay[s] = 0.0;
      }
      const double up =
          q.mask_y[(int64_t)(K - 1) * q.mstride + rrow[s]] ? fma(w[K - 1], ayb[s], ay[s]) : 0.0;
      ab[s] = fma(sigma, up, ab[s]);
      ayb[s] = (1.0 - w[K - 1]) * ayb[s];
      ay[s] = up;  // holds u between the passes
      link.put_y(rrow[s], up);
    }
    ok = link.sync();
    // ---- adjoint steps
    for (int k = K - 1; ok && k >= 0; --k) {
      const double wk = w[k], wp = k > 0 ? w[k - 1] : 0.0;
      for (int r = 0, i, s; (i = pick<NT>(r, warp)) < nc; ++r) {
        const double atu = col_sum(i, false, &s);
        if (s >= 0) {
          const double adj_xhat = -sigma * atu;
          const double adj_xp = fma(2.0, adj_xhat, fma(wk, axb[s], ax[s]));
          const double vv = q.mask_x[(int64_t)k * a.n + crow[s]] ? adj_xp : 0.0;
          link.put_x(crow[s], vv);
          ax[s] = vv - adj_xhat;
          ac[s] = fma(-tau, vv, ac[s]);
          axb[s] = (1.0 - wk) * axb[s];
        }
      }
      if (!(ok = link.sync())) break;
      for (int r = 0, i, s; (i = pick<NT>(r, warp)) < nr; ++r) {
        const double av = row_sum(i, false, &s);
        if (s >= 0) {
          const double ayk = fma(tau, av, ay[s]);
          if (k > 0) {
            const double up =
                q.mask_y[(int64_t)(k - 1) * q.mstride + rrow[s]] ? fma(wp, ayb[s], ayk) : 0.0;
            link.put_y(rrow[s], up);
            ab[s] = fma(sigma, up, ab[s]);
            ayb[s] = (1.0 - wp) * ayb[s];
            ay[s] = up;
          } else {
            ay[s] = ayk;
          }
        }
      }
      if (k > 0) ok = link.sync();
    }
    __syncthreads();
  }
  if (!ok) {
    if (tid == 0) *q.expired = 1;
    return;
  }
  for (int s = tid; s < ncl; s += NT) q.adj.ac[crow[s]] = ac[s];
  for (int s = tid; s < nrl; s += NT) q.adj.ab[rrow[s]] = ab[s];
  if (Link::kCluster) link.sync();  // no block leaves while another may store into its copies
}

__global__ void __launch_bounds__(kGridThreads, 1)
    adjoint_kernel(const __grid_constant__ AdjointArgs q) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ResidentArgs &a = q.r;
  const int P = (int)gridDim.x, b = (int)blockIdx.x;
  const Share sh{b, (a.AT.nslices - b + P - 1) / P, b, (a.A.nslices - b + P - 1) / P, P, 0, 0,
                 0, a.n, 0, a.m, b, P};
  GridLink<double> link{a.bar, 0u, nullptr, q.adj.v, q.adj.u};
  run_adjoint<kGridThreads>(smem, q, sh, 0, a.st->tau, a.st->sigma, q.gen, link);
}

__global__ void __launch_bounds__(kClusterThreads, 2)
    adjoint_cluster_kernel(const __grid_constant__ AdjointArgs q) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ResidentArgs &a = q.r;
  const int C = a.cluster, rank = (int)blockIdx.x % C, problem = (int)blockIdx.x / C;
  ClusterLink<double> link{};
  link.C = C;
  if (a.inst) {
    const BInst &B = a.inst[problem];
    const Share sh{B.cs0 + rank, (B.cs1 - B.cs0 - rank + C - 1) / C,
                   B.rs0 + rank, (B.rs1 - B.rs0 - rank + C - 1) / C,
                   C, B.cs0, B.rs0, B.col0, B.ncol, B.row0, B.nrow, rank, C};
    link.col0 = sh.col0;
    link.row0 = sh.row0;
    run_adjoint<kClusterThreads>(smem, q, sh, problem, B.tau, B.sigma, 0u, link);
  } else {
    const Share sh{rank, (a.AT.nslices - rank + C - 1) / C, rank, (a.A.nslices - rank + C - 1) / C,
                   C, 0, 0, 0, a.n, 0, a.m, rank, C};
    run_adjoint<kClusterThreads>(smem, q, sh, 0, a.st->tau, a.st->sigma, 0u, link);
  }
}

// One problem over the whole grid (cooperative launch).  A cooperative grid starts
// once all of its blocks find room, so with one block per SM LPs that are solved on
// several streams wait for one another; PER_SM = 2 lets an SM hold blocks of two of
// them (plan_resident has the rule and the figures): in FP64 with half the threads,
// in mixed precision, whose blocks own more slices, with half the registers.
template <typename T, int NT, int PER_SM>
__global__ void __launch_bounds__(NT, PER_SM)
    resident_kernel(const __grid_constant__ ResidentArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  SingleIO io{a.st, a.w, a.trace};
  if (!io.running()) return;
  const int P = (int)gridDim.x, b = (int)blockIdx.x;
  const Share sh{b, (a.AT.nslices - b + P - 1) / P, b, (a.A.nslices - b + P - 1) / P, P, 0, 0,
                 0, a.n, 0, a.m, b, P};
  GridLink<T> link{a.bar, 0u, nullptr, nullptr, nullptr};
  if constexpr (sizeof(T) == 4) {
    link.gx = a.mv.dxhat;
    link.gy = a.mv.dy;
  } else {
    link.gx = a.v.xhat;
    link.gy = a.v.y;
  }
  run_block<T, NT, true, (NT * PER_SM > kGridThreads)>(smem, a, sh, io, link);
}

// One problem per cluster of a.cluster blocks: the single problem, or the
// problems of a batch.
template <typename T, bool RES, class IO>
__global__ void __launch_bounds__(kClusterThreads, RES ? 2 : 4)
    cluster_kernel(const __grid_constant__ ResidentArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int C = a.cluster, rank = (int)blockIdx.x % C;
  ClusterLink<T> link{};
  link.C = C;
  if constexpr (std::is_same<IO, SingleIO>::value) {
    SingleIO io{a.st, a.w, a.trace};
    if (!io.running()) return;
    const Share sh{rank, (a.AT.nslices - rank + C - 1) / C, rank, (a.A.nslices - rank + C - 1) / C,
                   C, 0, 0, 0, a.n, 0, a.m, rank, C};
    run_block<T, kClusterThreads, RES, false>(smem, a, sh, io, link);
  } else {
    BatchIO io{a.inst + blockIdx.x / C, a.glob};
    if (!io.running()) return;
    const BInst &B = *io.B;
    const Share sh{B.cs0 + rank, (B.cs1 - B.cs0 - rank + C - 1) / C,
                   B.rs0 + rank, (B.rs1 - B.rs0 - rank + C - 1) / C,
                   C, B.cs0, B.rs0, B.col0, B.ncol, B.row0, B.nrow, rank, C};
    link.col0 = sh.col0;
    link.row0 = sh.row0;
    run_block<T, kClusterThreads, RES, false>(smem, a, sh, io, link);
  }
}

template <typename F>
bool set_smem(F *kernel, int bytes) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) ==
      cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}

// The grid kernel of a precision, for one block per SM or two.
using ResidentKernel = void (*)(ResidentArgs);
ResidentKernel resident_of(bool mixed, bool lean) {
  static const ResidentKernel k[4] = {
      resident_kernel<double, kGridThreads, 1>, resident_kernel<double, kGridThreads / 2, 2>,
      resident_kernel<float, kGridThreads, 1>, resident_kernel<float, kGridThreads, 2>};
  return k[(mixed ? 2 : 0) + (lean ? 1 : 0)];
}
int resident_threads(bool mixed, bool lean) {
  return lean && !mixed ? kGridThreads / 2 : kGridThreads;
}

// The cluster kernel of a precision, residency and kind of problem.
using ClusterKernel = void (*)(ResidentArgs);
ClusterKernel cluster_of(bool mixed, bool res, bool batch) {
  static const ClusterKernel k[8] = {
      cluster_kernel<double, false, SingleIO>, cluster_kernel<double, false, BatchIO>,
      cluster_kernel<double, true, SingleIO>,  cluster_kernel<double, true, BatchIO>,
      cluster_kernel<float, false, SingleIO>,  cluster_kernel<float, false, BatchIO>,
      cluster_kernel<float, true, SingleIO>,   cluster_kernel<float, true, BatchIO>};
  return k[(mixed ? 4 : 0) + (res ? 2 : 0) + (batch ? 1 : 0)];
}

// The multiplier search of the per-pass check in one cooperative launch: Newton
// steps (newton_next) over N breakpoints, one grid barrier each.  lambda only
// rises, so a coordinate once clamped stays clamped: its d^2 and d g go into the
// thread's running sums at the step that clamps it, and a step reads the keys
// and g^2 (16 bytes per coordinate, from L2) and adds the g^2 of the others,
// one FP64 addition per coordinate.  1.2M coordinates: 70 us alone with a cold
// L2, 240 for the 16 launches of the radix search; one block per SM, because the
// barrier and the sums over blocks grow with their number.
constexpr int kNewtonThreads = 1024;
struct SearchArgs {
  CheckScratch cs;
  DevState *st;
  int64_t N;
  int32_t nsearch;
};

__global__ void __launch_bounds__(kNewtonThreads, 1) search_kernel(SearchArgs a) {
  constexpr int W = kNewtonThreads / kWarp, U = 4;
  __shared__ LSearch L[2];
  __shared__ double red[W][8], nw[8];
  __shared__ int32_t dead;
  const int tid = threadIdx.x, lane = tid & (kWarp - 1), warp = tid >> 5;
  const int P = (int)gridDim.x;
  if (a.st->status != kRunning) return;  // nothing here changes it but a wait that runs out
  GridLink<double> link{a.cs.bar, a.st->bar_gen, &dead, nullptr, nullptr};
  if (tid < 2) {
    L[tid] = a.st->ls[tid];
    if (tid >= a.nsearch) L[tid].done = 1;
  }
  if (tid == 0) dead = 0;
  __syncthreads();
  const unsigned gen0 = link.gen;
  double clamped[2][2] = {{0.0, 0.0}, {0.0, 0.0}};  // this thread's sums of d^2, d g
  uint64_t last[2] = {0ull, 0ull};                  // keys below are in them
  int seen[2] = {0, 0};                             // and their number
  int count[2] = {-1, -1};                          // thread 0's
  for (int step = 0; step < kNewtonMax; ++step) {
    const bool done0 = L[0].done != 0, done1 = L[1].done != 0;
    if (done0 && done1) break;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (c ? done1 : done0) continue;
      const uint64_t *__restrict__ keys = a.cs.keys[c];
      const double *__restrict__ d2 = a.cs.d2[c], *__restrict__ gd = a.cs.gd[c];
      const double *__restrict__ g2 = a.cs.g2[c];
      const uint64_t to = (uint64_t)dbits(L[c].lambda) + 1;  // clamped: keys below to
      double above = 0.0;
      const int64_t stride = (int64_t)P * kNewtonThreads;
      for (int64_t e0 = (int64_t)blockIdx.x * kNewtonThreads + tid; e0 < a.N; e0 += U * stride) {
        uint64_t k[U];
        double g[U];
#pragma unroll
        for (int r = 0; r < U; ++r) {
          const int64_t e = e0 + r * stride;
          k[r] = e < a.N ? keys[e] : kNoKey;
          g[r] = e < a.N ? g2[e] : 0.0;
        }
#pragma unroll
        for (int r = 0; r < U; ++r) {
          if (k[r] < to) {
            if (k[r] >= last[c]) {
              const int64_t e = e0 + r * stride;
              clamped[c][0] += d2[e];
              clamped[c][1] += gd[e];
              ++seen[c];
            }
          } else if (k[r] != kNoKey) {
            above += g[r];
          }
        }
      }
      last[c] = to;
      double u[4] = {clamped[c][0], clamped[c][1], above, 0.0};
      const double su = warp_sum_multi<4>(u);
      const int cnt = __reduce_add_sync(kFull, seen[c]);
      if ((lane & 7) == 0) red[warp][4 * c + (lane >> 3)] = lane == 24 ? (double)cnt : su;
    }
    __syncthreads();
    // two buffers in turn: a block may still read the last step's sums
    double *np = a.cs.npart + (size_t)(step & 1) * P * 8;
    if (tid < 8 && !(tid < 4 ? done0 : done1)) {
      double s = 0.0;
      for (int i = 0; i < W; ++i) s += red[i][tid];
      __stcg(np + (size_t)blockIdx.x * 8 + tid, s);
    }
    if (!link.sync()) {
      if (tid == 0) a.st->status = kStatusTimeout;
      return;
    }
    if (warp < 8 && !(warp < 4 ? done0 : done1)) {
      const double s = sum_parts(np, 8, warp, P);
      if (lane == 0) nw[warp] = s;
    }
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        LSearch &l = L[c];
        if (!l.done)
          l.done = newton_next(nw[4 * c], nw[4 * c + 1], nw[4 * c + 2] + l.f_hi,
                               (int)nw[4 * c + 3], l.r2, step, l.lambda, l.rho_r, count[c]);
      }
    }
    __syncthreads();
  }
  // every block has read the state: each passed a barrier after that
  if (blockIdx.x == 0 && link.gen != gen0 && tid < 2) {
    if (tid < a.nsearch) {
      L[tid].done = 1;
      a.st->ls[tid] = L[tid];
    }
    if (tid == 0) a.st->bar_gen = link.gen;
  }
}

}  // namespace

// Bytes of shared memory of a block that owns nc + nr slices with ncl columns and nrl rows and
// (cluster kernel) copies of ncol and nrow exchanged elements, without resident elements (the
// carving of run_block).
size_t resident_fixed_bytes(int nc, int nr, int ncl, int nrl, int K, bool mixed, int ncol,
                            int nrow) {
  const size_t lists = sizeof(LSlice) * ((size_t)nc + nr);
  const size_t state = mixed ? col_bytes<float>() * ncl + row_bytes<float>() * nrl
                             : col_bytes<double>() * ncl + row_bytes<double>() * nrl;
  const size_t copies = (mixed ? 4 : 8) * ((size_t)ncol + nrow);
  const int warps = (ncol > 0 ? kClusterThreads : kGridThreads) / kWarp;
  return sizeof(Header) + lists + state + copies + sizeof(double) * (warps * 32 + 40 + (size_t)K) +
         16 * 28;
}

// The same for the adjoint kernels (the carving of run_adjoint).
size_t adjoint_fixed_bytes(int nc, int nr, int ncl, int nrl, int K, int ncol, int nrow) {
  return sizeof(Header) + sizeof(LSlice) * ((size_t)nc + nr) + (4 + 8 * 8) * (size_t)ncl +
         (8 + 6 * 8) * (size_t)nrl + 8 * ((size_t)ncol + nrow) + 8 * (size_t)K + 16 * 28;
}

// Largest dynamic shared memory of the kernels on the current device; 0 when it cannot launch
// them (no cooperative launch).
size_t resident_smem_limit(int device, bool mixed) {
  int coop = 0, optin = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) !=
          cudaSuccess ||
      !coop) {
    cudaGetLastError();
    return 0;
  }
  for (int lean = 0; lean < 2; ++lean)
    if (!set_smem(resident_of(mixed, lean != 0), optin)) return 0;
  for (int i = 0; i < 4; ++i)
    if (!set_smem(cluster_of(mixed, i & 1, i & 2), optin)) return 0;
  if (!mixed && !(set_smem(adjoint_kernel, optin) && set_smem(adjoint_cluster_kernel, optin)))
    return 0;
  return (size_t)optin;
}

// Whether P blocks with smem bytes each can be resident at once.
bool resident_fits(int P, int nsm, size_t smem, bool mixed, bool lean) {
  int per_sm = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, resident_of(mixed, lean), resident_threads(mixed, lean), smem);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (int64_t)per_sm * nsm >= P;
}

bool search_fits(int P, int nsm) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, search_kernel, kNewtonThreads, 0) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (int64_t)per_sm * nsm >= P;
}

cudaError_t launch_search(const CheckScratch &cs, int64_t N, int nsearch, DevState *st,
                          cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cs.search_blocks);
  cfg.blockDim = dim3(kNewtonThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, search_kernel, SearchArgs{cs, st, N, nsearch});
}

cudaError_t launch_resident(const ResidentArgs &a, int P, size_t smem, bool mixed, bool lean,
                            cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P);
  cfg.blockDim = dim3((unsigned)resident_threads(mixed, lean));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, resident_of(mixed, lean), a);
}

namespace {
cudaLaunchConfig_t cluster_config(int problems, int C, size_t smem, cudaLaunchAttribute *at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(problems * C));
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = smem;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}
}  // namespace

// lp_backward's recurrence over all recorded blocks: one problem on P blocks, or
// one cluster per problem.
cudaError_t launch_adjoint(const AdjointArgs &q, int P, size_t smem, cudaStream_t s) {
  cudaLaunchAttribute at[1];
  if (q.r.cluster > 0) {
    cudaLaunchConfig_t cfg = cluster_config(q.count, q.r.cluster, smem, at);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, adjoint_cluster_kernel, q);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P);
  cfg.blockDim = dim3(kGridThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, adjoint_kernel, q);
}

// Whether P blocks of the adjoint kernel with smem bytes each can be resident at once.
bool adjoint_fits(int P, int nsm, size_t smem) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, adjoint_kernel, kGridThreads, smem) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (int64_t)per_sm * nsm >= P;
}

// How many clusters of C blocks with smem bytes each the device holds at once (0: none).
namespace {
int active_clusters(const void *kernel, int C, size_t smem) {
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = cluster_config(1, C, smem, at);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}
}  // namespace

int cluster_active(int C, size_t smem, bool mixed, bool res, bool batch) {
  return active_clusters((const void *)cluster_of(mixed, res, batch), C, smem);
}

int adjoint_active(int C, size_t smem) {
  return active_clusters((const void *)adjoint_cluster_kernel, C, smem);
}

cudaError_t launch_cluster(const ResidentArgs &a, int problems, size_t smem, bool mixed, bool res,
                           cudaStream_t s) {
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = cluster_config(problems, a.cluster, smem, at);
  cfg.stream = s;
  return cudaLaunchKernelEx(&cfg, cluster_of(mixed, res, a.inst != nullptr), a);
}

}  // namespace lpg
