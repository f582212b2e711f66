// One kernel per check block for LPs that fit on the SMs: K iterations, the
// check, the multiplier search, the restart decision and the restart, with
// the matrix and the owned part of every vector in shared memory.
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
// iteration: column pass 4,200, barrier 3,000, row pass 4,200, barrier 3,000
// (7 us; the per-pass kernels 13.6 us).  The passes are bound by random
// gathers from L2 (0.8 to 1 per cycle and SM; from L1, when a block gathers
// the same line twice, 2.4), the barriers by the release fence and two trips
// to L2 (2,500 cycles at 152 blocks with nothing else to do, 1,600 at 7).
// Tagging every exchanged value with the number of its pass, so that gathers
// wait for their own operand and no barrier is needed, was slower: the tagged
// words bypass L1 and the repeated gathers fill it (9,500 cycles per pass).
// So was copying the whole gathered vector into shared memory before a pass.
// FP64 instructions are the other scarce thing: one of a warp holds its quarter
// of the SM for 76 cycles whatever the number of active lanes.  So sums over
// the block go through transposed butterflies, scalars are computed by one
// warp, and the owned rows and columns are laid out one per thread where the
// averages and the check's terms are formed.
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

#include "lp_internal.h"
#include "spmv_core.cuh"

namespace lpg {
namespace {

constexpr int kRT = 512;               // threads per block
constexpr int kRW = kRT / kWarp;       // warps per block
constexpr int kU = 8;                  // gathers in flight per lane
constexpr int kNewtonMax = 1024;       // Newton steps (each clamps at least one more coordinate)
constexpr int kStatusTimeout = 6;
constexpr int kBarLines = kResBarLines;  // arrival counters of the grid barrier
constexpr unsigned long long kWaitNs = 2000000000ull;  // longest wait at a barrier

// One local slice: first element in shared memory, first local row,
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
__device__ __forceinline__ int pick(int round, int warp) {
  return round == 0 ? warp : round * kRW + kRW - 1 - warp;
}

struct Header {
  int32_t ncl, nrl;  // local columns and rows
  int32_t nce, nre;  // elements
  int32_t dead;      // a wait ran out
  // Scalars computed by one warp: an FP64 instruction of a warp occupies its
  // quarter of the SM for 76 cycles (measured), a square root or a division dozens
  // of them, so the other warps read the results here.
  int32_t status, returned, restart, use_cur;
  int32_t done[2];
  int32_t count[2];  // coordinates clamped at the last Newton step
  double sw, isw, inv;
  double kkt[2][5], r2[2], lam[2], rho_r[2];
  double rho, r, mix_s;
};

template <typename T>
struct Sm {  // shared-memory arrays of a block
  Header *h;
  LSlice *cs, *rs;
  double *red;  // [kRW][32] sums of the warps
  double *tot;  // [32] sums of the grid
  double *nw;   // [8] Newton sums
  double *w;    // [K] averaging weights
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

// Barrier over the P resident blocks of a cooperative launch: kBarLines arrival
// counters that only grow, a 128-byte line each (152 arrivals at one address
// cost 900 cycles more), block b on counter b mod kBarLines; one lane of warp 0
// waits on each.  Block-wide barriers on both sides order the other threads'
// accesses.  The wait is bounded: after kWaitNs the block gives up, and every
// other block's wait runs out the same way.
struct GridBar {
  unsigned *counter;
  unsigned gen;  // barriers passed since the counters were zero
  int32_t *dead;
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    ++gen;
    if (threadIdx.x == 0) red_release(counter + (blockIdx.x % kBarLines) * 32);
  }
  __device__ __forceinline__ bool sync() {
    arrive();
    return wait();
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
};

// Row sum of one slice, in the order of process_item: `a` is the lane's
// starting value (-c or -b in the row's first lane), ip and vp the lane's
// indices and values in shared memory.  All lanes of a row return its sum.
// The gathers are plain loads: the barrier's acquire makes L1 safe to use.
template <typename T>
__device__ __forceinline__ T slice_sum(T a, const int32_t *ip, const T *vp, int steps, int lg,
                                       const T *vec) {
  for (int t = 0; t < steps; t += kU) {
    T g[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (t + u < steps) g[u] = vec[ip[kWarp * (t + u)]];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (t + u < steps) a = fma_t(vp[kWarp * (t + u)], g[u], a);
  }
  for (int o = (1 << lg) >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
  return a;
}

// Sums of the check, both candidates at once, from plain arrays (written
// before a grid barrier, whose acquire lets plain loads use L1) and FP64 values.
__device__ __forceinline__ void check_sums(const LSlice *sl, int count, const int32_t *sidx,
                                           const double *sval, const SellMat &A,
                                           const double *v0, const double *v1, double *o0,
                                           double *o1) {
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x >> 5;
  for (int q = 0, i; (i = pick(q, warp)) < count; ++q) {
    const LSlice s = sl[i];
    const int lg = s.lg(), steps = s.steps();
    const int32_t *ip = sidx + s.soff + lane;
    const double *vp = (sval ? sval + s.soff : A.val + A.info[s.gid].off) + lane;
    double a0 = 0.0, a1 = 0.0;
    for (int t = 0; t < steps; t += 4) {
      double g[4], h[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u < steps) {
          const int j = ip[kWarp * (t + u)];
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

// Sums of N per-thread values over the warp (N a power of two <= 32): the
// transposed butterfly issues N - 1 + log2(32 / N) additions instead of 5 N.
// Lane l returns the sum of value l / (32 / N).
template <int N>
__device__ __forceinline__ double warp_sum_multi(double (&v)[N]) {
  const int lane = threadIdx.x & (kWarp - 1);
  int o = 16;
#pragma unroll
  for (int half = N / 2; half > 0; half >>= 1, o >>= 1) {
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const double keep = hi ? v[i + half] : v[i], send = hi ? v[i] : v[i + half];
      v[i] = keep + __shfl_xor_sync(kFull, send, o);
    }
  }
  double s = v[0];
  for (; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  return s;
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

// Local slices of one operator (every P-th of the global ones), most steps
// first: records, and the numbers of local rows and elements.  One warp.
__device__ void build_slices(const SellMat &A, int blk, int P, LSlice *sl, int32_t *nslot,
                             int32_t *nelem) {
  const int lane = threadIdx.x & (kWarp - 1);
  int slot = 0, el = 0;
  const int count = (A.nslices - blk + P - 1) / P;
  for (int i0 = 0; i0 < count; i0 += kWarp) {
    const int i = i0 + lane;
    int rows = 0, steps = 0, lg = 0, rank = 0;
    if (i < count) {
      const SliceInfo a = A.info[blk + i * P];
      rows = A.info[blk + i * P + 1].row0 - a.row0;
      steps = a.len_g >> 3;
      lg = a.len_g & 7;
      for (int j = 0; j < count; ++j) {
        const int o = A.info[blk + j * P].len_g >> 3;
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
      sl[rank] = LSlice{el + kWarp * (pl - steps), slot + ps - rows,
                        (uint32_t)steps << 16 | (uint32_t)lg << 8 | (uint32_t)rows, blk + i * P};
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

// Copies the local slices of one operator, and the permuted indices of their
// rows, into shared memory.
template <typename T>
__device__ __forceinline__ void load_slices(const SellMat &A, const T *gval,
                                            const LSlice *sl, int count, int32_t *row,
                                            int32_t *sidx, T *sval) {
  const int lane = threadIdx.x & (kWarp - 1), warp = threadIdx.x >> 5;
  constexpr int VC = 16 / sizeof(T);  // values per 16-byte chunk
  for (int i = warp; i < count; i += kRW) {
    const LSlice s = sl[i];
    const SliceInfo g = A.info[s.gid];
    for (int r = lane; r < s.rows(); r += kWarp) row[s.slot0 + r] = g.row0 + r;
    const int len = s.steps() * kWarp;
    const int4 *gi = reinterpret_cast<const int4 *>(A.idx + g.off);
    int4 *si = reinterpret_cast<int4 *>(sidx + s.soff);
    for (int e = lane; e < len / 4; e += kWarp) si[e] = __ldg(gi + e);
    const int4 *gv = reinterpret_cast<const int4 *>(gval + g.off);
    int4 *sv = reinterpret_cast<int4 *>(sval + s.soff);
    for (int e = lane; e < len / VC; e += kWarp) sv[e] = __ldg(gv + e);
  }
}

// Bytes of shared memory per local column and row.
template <typename T>
constexpr size_t col_bytes() {
  return 4 + 16 + sizeof(T) * 2 + 8 + 2 * sizeof(T);
}
template <typename T>
constexpr size_t row_bytes() {
  return 4 + 16 + sizeof(T) * 2 + 8 + (sizeof(T) == 8 ? 4 : 8);
}

template <typename T>
__global__ void __launch_bounds__(kRT, 1) resident_kernel(const __grid_constant__ ResidentArgs a) {
  constexpr bool MIX = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char smem[];
  const int P = (int)gridDim.x, blk = (int)blockIdx.x, tid = (int)threadIdx.x;
  const int lane = tid & (kWarp - 1), warp = tid >> 5;
  DevState *st = a.st;
  if (st->status != kRunning) return;
  const int K = st->K;
  const int nc = (a.AT.nslices - blk + P - 1) / P, nr = (a.A.nslices - blk + P - 1) / P;

  // ---- layout of shared memory
  Sm<T> S;
  unsigned char *p = smem;
  S.h = (Header *)carve(p, sizeof(Header));
  S.cs = (LSlice *)carve(p, sizeof(LSlice) * nc);
  S.rs = (LSlice *)carve(p, sizeof(LSlice) * nr);
  S.red = (double *)carve(p, sizeof(double) * kRW * 32);
  S.tot = (double *)carve(p, sizeof(double) * 32);
  S.nw = (double *)carve(p, sizeof(double) * 8);
  S.w = (double *)carve(p, sizeof(double) * K);
  if (warp == 0) build_slices(a.AT, blk, P, S.cs, &S.h->ncl, &S.h->nce);
  else if (warp == 1) build_slices(a.A, blk, P, S.rs, &S.h->nrl, &S.h->nre);
  if (warp == 2) {
    const double sw = sqrt(st->omega);
    if (lane == 0) {
      S.h->dead = 0;
      S.h->sw = sw;
      S.h->isw = 1.0 / sw;
      S.h->inv = MIX ? 1.0 / st->mix_s : 1.0;
    }
  }
  for (int k = tid; k < K; k += kRT) S.w[k] = a.w[k];
  __syncthreads();
  const int ncl = S.h->ncl, nrl = S.h->nrl;
  S.crow = (int32_t *)carve(p, 4 * (size_t)ncl);
  S.rrow = (int32_t *)carve(p, 4 * (size_t)nrl);
  S.cs0 = (double *)carve(p, 8 * (size_t)ncl);
  S.cs1 = (double *)carve(p, 8 * (size_t)ncl);
  S.rs0 = (double *)carve(p, 8 * (size_t)nrl);
  S.rs1 = (double *)carve(p, 8 * (size_t)nrl);
  S.c = (T *)carve(p, sizeof(T) * ncl);
  S.x = (T *)carve(p, sizeof(T) * ncl);
  S.xb = (double *)carve(p, 8 * (size_t)ncl);
  S.b = (T *)carve(p, sizeof(T) * nrl);
  S.y = (T *)carve(p, sizeof(T) * nrl);
  S.yb = (double *)carve(p, 8 * (size_t)nrl);
  if constexpr (MIX) {
    S.lf = (float *)carve(p, 4 * (size_t)ncl);
    S.uf = (float *)carve(p, 4 * (size_t)ncl);
    S.lo = (float *)carve(p, 4 * (size_t)nrl);
    S.hi = (float *)carve(p, 4 * (size_t)nrl);
  } else {
    S.lk = (long long *)carve(p, 8 * (size_t)ncl);
    S.uk = (long long *)carve(p, 8 * (size_t)ncl);
    S.rt = (int32_t *)carve(p, 4 * (size_t)nrl);
  }
  S.cidx = (int32_t *)carve(p, 4 * (size_t)S.h->nce);
  S.cval = (T *)carve(p, sizeof(T) * S.h->nce);
  S.ridx = (int32_t *)carve(p, 4 * (size_t)S.h->nre);
  S.rval = (T *)carve(p, sizeof(T) * S.h->nre);

  // ---- owned state
  const T *gvc, *gvr;
  if constexpr (MIX) {
    gvc = a.AT.valf;
    gvr = a.A.valf;
  } else {
    gvc = a.AT.val;
    gvr = a.A.val;
  }
  load_slices<T>(a.AT, gvc, S.cs, nc, S.crow, S.cidx, S.cval);
  load_slices<T>(a.A, gvr, S.rs, nr, S.rrow, S.ridx, S.rval);
  __syncthreads();
  T *gx, *gy;  // the exchanged vectors
  if constexpr (MIX) {
    gx = a.mv.dxhat;
    gy = a.mv.dy;
  } else {
    gx = a.v.xhat;
    gy = a.v.y;
  }
  for (int s = tid; s < nrl; s += kRT) {
    const int i = S.rrow[s];
    T y;
    if constexpr (MIX) {
      y = a.mv.dy[i];
      S.b[s] = a.mv.bf[i];
      S.yb[s] = a.mv.dybar[i];
      S.lo[s] = a.mv.ylo[i];
      S.hi[s] = a.mv.yhi[i];
    } else {
      y = a.v.y[i];
      S.b[s] = a.v.b[i];
      S.yb[s] = a.v.ybar[i];
      S.rt[s] = (int)a.v.row_type[i];
    }
    S.y[s] = y;
  }
  for (int s = tid; s < ncl; s += kRT) {
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
  const T tau = (T)st->tau, sigma = (T)st->sigma;
  GridBar bar{a.bar, st->bar_gen, &S.h->dead};
  __syncthreads();

  // ---- K iterations.  The averages, which nothing waits for, are updated
  // between a barrier's arrival and its wait.
  bool lost = false;
  for (int k = 0; k < K; ++k) {
    const double w = S.w[k];
    for (int q = 0, i; (i = pick(q, warp)) < nc; ++q) {
      const LSlice sl = S.cs[i];
      const int lg = sl.lg(), r = lane >> lg, s = sl.slot0 + r;
      const bool owner = (lane & ((1 << lg) - 1)) == 0 && r < sl.rows();
      const T neg_g = slice_sum<T>(owner ? -S.c[s] : T(0), S.cidx + sl.soff + lane,
                                   S.cval + sl.soff + lane, sl.steps(), lg, gy);
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
        gx[S.crow[s]] = fma_t(T(2), xn, -x);
        S.x[s] = xn;
      }
    }
    bar.arrive();
    for (int s = tid; s < ncl; s += kRT) {
      const double xb = S.xb[s];
      S.xb[s] = fma(w, (double)S.x[s] - xb, xb);
    }
    if (!bar.wait()) {
      lost = true;
      break;
    }
    for (int q = 0, i; (i = pick(q, warp)) < nr; ++q) {
      const LSlice sl = S.rs[i];
      const int lg = sl.lg(), r = lane >> lg, s = sl.slot0 + r;
      const bool owner = (lane & ((1 << lg) - 1)) == 0 && r < sl.rows();
      const T res = slice_sum<T>(owner ? -S.b[s] : T(0), S.ridx + sl.soff + lane,
                                 S.rval + sl.soff + lane, sl.steps(), lg, gx);
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
        gy[S.rrow[s]] = yn;
        S.y[s] = yn;
      }
    }
    if (k + 1 < K) bar.arrive();  // the barrier after the publication covers the last pass
    else __syncthreads();
    for (int s = tid; s < nrl; s += kRT) {
      const double yb = S.yb[s];
      S.yb[s] = fma(w, (double)S.y[s] - yb, yb);
    }
    if (k + 1 < K && !bar.wait()) {
      lost = true;
      break;
    }
  }

  // ---- publish the FP64 iterate and average
  const double inv = S.h->inv;
  for (int s = tid; s < ncl; s += kRT) {
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
  for (int s = tid; s < nrl; s += kRT) {
    const int i = S.rrow[s];
    if constexpr (MIX) {
      a.mv.dybar[i] = S.yb[s];
      const int t = a.v.row_type[i];
      const double lo = (t == 1) ? 0.0 : -INFINITY, hi = (t == 2) ? 0.0 : INFINITY;
      const double y0 = a.v.y0[i];
      a.v.y[i] = fmin(fmax(fma((double)S.y[s], inv, y0), lo), hi);
      a.v.ybar[i] = fmin(fmax(fma(S.yb[s], inv, y0), lo), hi);
    } else {
      a.v.ybar[i] = S.yb[s];
    }
  }
  if (lost || !bar.sync()) {
    if (tid == 0) st->status = kStatusTimeout;
    return;
  }

  // ---- check: A^T [ybar, y], A [xbar, x] and their epilogues
  const int scheme = st->scheme;
  const bool gap_a = scheme == kSchemeAdaptive || scheme == kSchemeFlexible;
  const bool gap_c = scheme == kSchemeFlexible;
  const double om = st->omega;
  const GapOut go[2] = {GapOut{a.cs.keys[0], a.cs.d2[0], a.cs.g2[0], a.cs.gd[0]},
                        GapOut{a.cs.keys[1], a.cs.d2[1], a.cs.g2[1], a.cs.gd[1]}};
  {
    const double *sc = nullptr, *sr = nullptr;
    if constexpr (!MIX) {
      sc = S.cval;
      sr = S.rval;
    }
    check_sums(S.cs, nc, S.cidx, sc, a.AT, a.v.ybar, a.v.y, S.cs0, S.cs1);
    check_sums(S.rs, nr, S.ridx, sr, a.A, a.v.xbar, a.v.x, S.rs0, S.rs1);
  }
  __syncthreads();
  // owned columns, then (from a whole warp on) owned rows, one per thread
  const int rfirst = (ncl + kWarp - 1) & ~(kWarp - 1), nown = rfirst + nrl;
  const int busy = min(kRW, (nown + kWarp - 1) / kWarp);
  if (warp < busy) {
    CheckColsEpi ce{};
    CheckRowsEpi re{};
    ce.sw = re.sw = S.h->sw;
    ce.isw = re.isw = S.h->isw;
    re.off = a.n;
#pragma unroll
    for (int i = 0; i < NQ; ++i) ce.q[i] = 0.0;
    for (int s = tid; s < ncl; s += kRT) {
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
    for (int e = tid; e < nown; e += kRT) {
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
    // block sums, then grid sums
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
    __stcg(a.part + (size_t)blk * kResPart + tid, s);
  }
  // the state that the decision needs, read before the last barrier that every
  // block passes: block 0 writes it after that
  const double norm_b = st->norm_b, norm_c = st->norm_c, tol = st->tol, last_r = st->last_r,
               beta = st->beta, rho_stored = st->rho_stored, mix_old = st->mix_s;
  const int64_t t0 = st->t0, restarts = st->restarts, tau0 = st->tau0, fixed_len = st->fixed_len;
  const int was_returned = st->returned;
  if (!bar.sync()) {
    if (tid == 0) st->status = kStatusTimeout;
    return;
  }
  for (int i = warp; i < NQ; i += kRW) {
    const double s = sum_parts(a.part, kResPart, i, P);
    if (lane == 0) S.tot[i] = s;
  }
  __syncthreads();

  // ---- termination and search setup: lane 0 for the average, lane 1 for the
  // current iterate; every block decides from the same sums, block 0 records
  const double *tot = S.tot;
  if (warp == 0) {
    const int c = lane & 1;
    double k5[5];
    kkt_from(tot, Q_RP2_A + c, Q_RD2_A + c, Q_POBJ_A + c, Q_DOBJ_A + c, norm_b, norm_c, k5);
    const double rel = k5[4], rel_a = __shfl_sync(kFull, rel, 0), rel_c = __shfl_sync(kFull, rel, 1);
    int status = kRunning, returned = 0;
    if (tot[Q_BAD] > 0.0 || !isfinite(rel_a) || !isfinite(rel_c)) {
      status = kStatusNumerical;
      returned = was_returned;
    } else if (rel_a <= tol) {
      status = kStatusOK;
    } else if (rel_c <= tol) {
      status = kStatusOK;
      returned = 1;
    } else {
      returned = (rel_a <= rel_c) ? 0 : 1;
    }
    double r2 = 0.0, rho_r = 0.0;
    int done = 1;
    if (status == kRunning && (c ? gap_c : gap_a)) {
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
        for (int s = tid; s < ncl; s += kRT) add(S.crow[s]);
        for (int e = tid; e < nown; e += kRT)
          if (e >= rfirst) add((int64_t)a.n + S.rrow[e - rfirst]);
        const double su = warp_sum_multi<4>(u);
        cnt = __reduce_add_sync(kFull, cnt);
        if ((lane & 7) == 0) S.red[warp * 32 + 4 * c + (lane >> 3)] = lane == 24 ? (double)cnt : su;
      }
    }
    __syncthreads();
    // two buffers in turn: a block may still read the last step's sums
    double *np = a.npart + (size_t)(step & 1) * P * 8;
    if (tid < 8 && !(tid < 4 ? done0 : done1)) {
      double s = 0.0;
      for (int i = 0; i < busy; ++i) s += S.red[i * 32 + tid];
      __stcg(np + (size_t)blk * 8 + tid, s);
    }
    if (!bar.sync()) {
      if (tid == 0) st->status = kStatusTimeout;
      return;
    }
    if (warp < 8 && !(warp < 4 ? done0 : done1)) {
      const double s = sum_parts(np, 8, warp, P);
      if (lane == 0) S.nw[warp] = s;
    }
    __syncthreads();
    if (warp == 0 && lane < 2 && !(lane ? done1 : done0)) {
      const int c = lane;
      const double A = S.nw[4 * c], E = S.nw[4 * c + 1];
      const double B = S.nw[4 * c + 2] + tot[c ? Q_G2INF_C : Q_G2INF_A];
      const int same = (int)S.nw[4 * c + 3];
      if (!(B > 0.0)) {
        S.h->rho_r[c] = E;
        S.h->done[c] = 1;
      } else {
        const double ln = sqrt(fmax(S.h->r2[c] - A, 0.0) / B);
        S.h->rho_r[c] = E + ln * B;
        // the clamped set repeats (or rounding stops the increase): exact
        if (same == S.h->count[c] || (step > 0 && !(ln > S.h->lam[c]))) S.h->done[c] = 1;
        S.h->count[c] = same;
        S.h->lam[c] = ln;
      }
    }
    __syncthreads();
  }

  // ---- restart decision (Eq. adaptive-restart-scheme / flexible / fixed)
  const int status = S.h->status;
  const int64_t t = t0 + K;
  if (tid == 0) {
    double rho = NAN, r = last_r;
    int use_cur = 0, restart = 0;
    if (status == kRunning) {
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
        restart = (restarts == 0) ? (t >= tau0) : (rho <= beta * rho_stored);
      } else if (scheme == kSchemeFixed) {
        restart = (t >= fixed_len);
      }
    }
    S.h->rho = rho;
    S.h->r = r;
    S.h->use_cur = use_cur;
    S.h->restart = restart;
    S.h->mix_s = (restart && MIX && r > 0.0 && isfinite(r)) ? fmin(1.0 / r, 1e12) : mix_old;
  }
  __syncthreads();
  const int use_cur = S.h->use_cur, restart = S.h->restart;
  const double mix_s = S.h->mix_s;
  const int64_t t0n = restart ? 0 : t;
  if (blk == 0) {
    if (tid == 0) {
      st->bar_gen = bar.gen;
      st->iters += K;
      st->checks += 1;
      for (int i = 0; i < 5; ++i) {
        st->kkt_a[i] = S.h->kkt[0][i];
        st->kkt_c[i] = S.h->kkt[1][i];
      }
      st->returned = S.h->returned;
      if (status != kRunning) {
        st->status = status;
      } else {
        if (a.trace && st->trace_count < st->trace_cap) {
          double *row = a.trace + 6 * st->trace_count;
          row[0] = (double)st->iters;
          row[1] = S.h->rho;
          row[2] = (double)restart;
          row[3] = S.h->kkt[0][4];
          row[4] = S.h->kkt[1][4];
          row[5] = S.h->r;
        }
        st->trace_count += 1;
        st->last_rho = S.h->rho;
        st->last_r = S.h->r;
        st->use_cur = use_cur;
        st->restart_now = restart;
        st->t0 = t0n;
        if (restart) {
          st->rho_stored = S.h->rho;
          st->restarts += 1;
          st->mix_s = mix_s;
        }
      }
    }
    if (status == kRunning)
      for (int k = tid; k < K; k += kRT) a.w[k] = 1.0 / (double)(t0n + k + 1);
  }
  if (status != kRunning || (!restart && !use_cur)) return;

  // ---- restart (or the flexible scheme's replacement of the average), owned part
  for (int s = tid; s < ncl; s += kRT) {
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
  for (int s = tid; s < nrl; s += kRT) {
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

}  // namespace

// Bytes of shared memory of a block that owns nc + nr slices with ncl columns and nrl rows,
// without resident elements (the carving of resident_kernel).
size_t resident_fixed_bytes(int nc, int nr, int ncl, int nrl, int K, bool mixed) {
  const size_t lists = sizeof(LSlice) * ((size_t)nc + nr);
  const size_t state = mixed ? col_bytes<float>() * ncl + row_bytes<float>() * nrl
                             : col_bytes<double>() * ncl + row_bytes<double>() * nrl;
  return sizeof(Header) + lists + state + sizeof(double) * (kRW * 32 + 40 + (size_t)K) + 16 * 26;
}

// Largest dynamic shared memory of the kernel on the current device; 0 when it cannot launch
// cooperatively.
size_t resident_smem_limit(int device, bool mixed) {
  int coop = 0, optin = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) !=
          cudaSuccess ||
      !coop) {
    cudaGetLastError();
    return 0;
  }
  const cudaError_t e =
      mixed ? cudaFuncSetAttribute(resident_kernel<float>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, optin)
            : cudaFuncSetAttribute(resident_kernel<double>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return (size_t)optin;
}

// Whether P blocks with smem bytes each can be resident at once.
bool resident_fits(int P, int nsm, size_t smem, bool mixed) {
  int per_sm = 0;
  const cudaError_t e =
      mixed ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resident_kernel<float>, kRT, smem)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resident_kernel<double>, kRT,
                                                            smem);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (int64_t)per_sm * nsm >= P;
}

cudaError_t launch_resident(const ResidentArgs &a, int P, size_t smem, bool mixed,
                            cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P);
  cfg.blockDim = dim3(kRT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return mixed ? cudaLaunchKernelEx(&cfg, resident_kernel<float>, a)
               : cudaLaunchKernelEx(&cfg, resident_kernel<double>, a);
}

}  // namespace lpg
