// Inner solve of the Poisson refinement loop (eq. 1.1 discretised by eq. 7 /
// eq. "laplace"): conjugate gradients on the SPD two-point part A_T of the diamond
// operator (per face the term |S_f|^2 / ((x_R - x_L) . S_f) (P_R - P_L)), A_T delta = r,
// in T = float or double with FP64 dot products, as ONE persistent cooperative kernel.
//
// A mesh may hold several independent parts (an ensemble of meshes packed into one
// index space); every part has its own CG scalars, stopping test and barrier, and a launch of
// the CG alone (k_cg) leaves the parts that the outer loop does not flag active as they are.
//
// Work split: a part's cells are cut into equal contiguous "sub-chunks", one to each of the
// blocks that are its own; small parts are one sub-chunk each, and a block solves several of
// them in turn (share_blocks in api.cu). Every sum is formed per sub-chunk (block tree), then
// over the part's sub-chunks in a fixed order by every block of the part, so that they take the
// same decisions and results are bitwise reproducible for a given grid. The same sub-chunks
// give the per-part norms of the outer loop (k_residual_norm, k_norm_partial).
//
// Barriers are bounded: a wait longer than one second (or the limit set by the
// test hook fvgb_test_barrier) sets a status word and every block leaves; the host
// reports FVGB_ETIMEOUT.
#include <cuda_runtime.h>

#include "grid_sync.cuh"
#include "internal.h"

namespace fvgb {
namespace {

// Block-wide FP64 sum in a fixed order, valid in thread 0. Every thread's value goes to
// shared memory; four warps (one per SM sub-partition) each add a quarter of them, lane
// by lane in index order and then by a shuffle tree, and thread 0 adds the four results.
// GB300 issues FP64 adds at a small fraction of the FP32 rate, so the sum keeps the FP64
// instructions on its critical path few and spread over the four sub-partitions.
// sh holds blockDim.x doubles (blockDim.x a multiple of 128).
__device__ __forceinline__ double block_sum(double v, double* sh) {
  __syncthreads();                      // the previous call's readers are done with sh
  sh[threadIdx.x] = v;
  __syncthreads();
  double t = 0.0;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int quarter = blockDim.x >> 2;
  if (w < 4) {
    const double* q = sh + w * quarter;
    t = q[l];
    for (int j = l + 32; j < quarter; j += 32) t += q[j];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  __syncthreads();                      // every quarter read before the results overwrite sh
  if (w < 4 && l == 0) sh[w] = t;
  __syncthreads();
  if (threadIdx.x == 0) t = (sh[0] + sh[1]) + (sh[2] + sh[3]);
  return t;
}

template <typename T>
struct SolveArgs {
  // two-point operator scaled to unit diagonal, D^-1/2 A_T D^-1/2, in T, cell-major [N][4]
  const int32_t* at_nbr;
  const T* at_scoef;
  const T* at_isd;          // [N] D^-1/2: the CG solves for D^1/2 x from D^-1/2 r
  const double* r_in;       // [N] right-hand side (FP64 outer residual)
  double* phi;              // the correction is added here
  T* cx;
  T* cr;
  T* cp;
  T* cq;
  // parts
  int n_part;
  int n_sc;
  const int32_t* blk_work;  // [G+1] first entry of each block in work
  const WorkPiece* work;    // [n_sc]
  const int* active;        // [P] parts to solve
  double* buf;              // [4][n_sc] partial sums, used in turn
  Barrier* bar;             // [P + 1]: the launch's status, then the parts' barriers
  double inner_tol2;
  int maxit_inner;
  int* out_inner;           // [P] iterations per part
  int* out_status;          // [0]: 0 ok, 6 non-finite / breakdown; [1]: iterations run
  int skip_block;           // test hook: this block never arrives at a barrier (-1: none)
  unsigned long long barrier_ns;  // limit of a barrier wait
};

constexpr int kLaneSlots = 5;        // partial sums a lane loads at once (160 blocks)

// A block's piece of a part, and the barrier of the blocks that share the part. The parts of an
// ensemble never wait for one another: every part has its own blocks, counter, scalars and
// stopping tests.
struct OneBlock {
  int part, sc, sc0, sc1;              // the part, this piece, the part's pieces
  int64_t lo, hi;
  Barrier* bar;
  int* status;
  bool arrive;                         // test hook: false leaves out this block's arrivals
  unsigned target;
};
template <typename T>
__device__ OneBlock one_block(const SolveArgs<T>& a, int q) {
  const WorkPiece w = a.work[q];
  OneBlock k;
  k.sc = w.sc;
  k.part = w.part;
  k.sc0 = w.sc0;
  k.sc1 = w.sc1;
  k.lo = w.lo;
  k.hi = w.hi;
  k.bar = a.bar + 1 + k.part;
  k.status = &a.bar->status;
  k.arrive = a.skip_block != (int)blockIdx.x;
  k.target = 0;
  return k;
}

// One exchange of a part's blocks: acc of every thread -> block sum (four warps, one per SM
// sub-partition, a quarter each: GB300 issues FP64 adds at a small fraction of the FP32 rate,
// so the FP64 instructions on the critical path are few and spread) -> buf; warp 0 waits,
// sums the partials from registers and hands the total to use(total) (every lane of warp 0);
// one block barrier at the end. False when a wait ran out.
template <typename T, typename F>
__device__ __forceinline__ bool exchange_one(const SolveArgs<T>& a, double* buf, OneBlock& k, double acc, double* sh,
                                             int* s_ok, F use) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int quarter = blockDim.x >> 2;
  k.target += k.sc1 - k.sc0;
  sh[threadIdx.x] = acc;
  __syncthreads();                   // and every row of the phase is written before the arrival
  if (w < 4) {
    const double* q = sh + w * quarter;
    double t = q[l];
    for (int j = l + 32; j < quarter; j += 32) t += q[j];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (l == 0) sh[blockDim.x + w] = t;
    asm volatile("bar.sync 1, 128;" ::: "memory");
  }
  if (w == 0) {
    if (l == 0) {
      const double* q = sh + blockDim.x;
      __stcg(buf + k.sc, (q[0] + q[1]) + (q[2] + q[3]));
      if (k.arrive) grid_arrive(k.bar);
    }
    __syncwarp();
    const bool ok = grid_wait(k.bar, k.status, k.target, a.barrier_ns);
    double t = 0.0;
    if (ok) {
      double v[kLaneSlots];
#pragma unroll
      for (int q = 0; q < kLaneSlots; ++q) v[q] = k.sc0 + l + 32 * q < k.sc1 ? __ldcg(buf + k.sc0 + l + 32 * q) : 0.0;
#pragma unroll
      for (int q = 0; q < kLaneSlots; ++q) t += v[q];
      for (int sc = k.sc0 + l + 32 * kLaneSlots; sc < k.sc1; sc += 32) t += __ldcg(buf + sc);
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      use(t);
    }
    if (l == 0) *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// Loads of the operator and of the vectors in the two phases.
// kStream (a working set well above L2): what an iteration reads once (operator) or reads and
// writes once without a neighbour's look (x) is marked to leave L2 first, so that r, p and q
// stay; 6M cells FP32 84.6 -> 70.3 us an iteration. Smaller sets live in L2 as they are and
// the marks cost them (750,000 cells 13.4 -> 14.5 us), and in FP64 the phase waits for the
// FP64 pipe more than for memory (6M cells 145 us without, 159 with the marks).
template <bool kStream>
__device__ __forceinline__ int4 load_op(const int4* p) {
  if constexpr (!kStream) return __ldg(p);
  unsigned long long pol;
  int4 v;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.s32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
  return v;
}
// r, own rows and neighbours', comes through load_synced: neighbours are mostly rows of the same
// warps, so L1 takes most of the gathers' traffic: 6M cells FP32 68.5 -> 64.5 us, 750,000 cells
// 13.4 -> 11.8 us an iteration against loads that pass L1 by.

// Four operator coefficients of one row, loaded with vector loads.
template <typename T>
struct Coef4;
template <>
struct Coef4<float> {
  float c[4];
  template <bool kStream>
  __device__ __forceinline__ void load(const float* p, int64_t i) {
    const int4 v = load_op<kStream>(reinterpret_cast<const int4*>(p) + i);
    c[0] = __int_as_float(v.x); c[1] = __int_as_float(v.y); c[2] = __int_as_float(v.z); c[3] = __int_as_float(v.w);
  }
};
template <>
struct Coef4<double> {
  double c[4];
  template <bool kStream>
  __device__ __forceinline__ void load(const double* p, int64_t i) {
    const double2 v0 = __ldg(reinterpret_cast<const double2*>(p) + 2 * i);
    const double2 v1 = __ldg(reinterpret_cast<const double2*>(p) + 2 * i + 1);
    c[0] = v0.x; c[1] = v0.y; c[2] = v1.x; c[3] = v1.y;
  }
};

// Rows per thread per trip. Both phases load the next trip's rows before they work on this
// one's, so that the loads of one trip are always in flight: two FP32 rows of 48 bytes or one
// FP64 row of 80 for each of 512 threads. 6M cells FP64 168 -> 146 us an iteration, 750,000
// cells 23.1 -> 20.7 us (more rows a trip without the overlap were no faster, and more rows
// with it spill). A phase's first rows are loaded before the exchange in front of it: 10,000
// cells FP64 7.4 -> 7.0, 750,000 FP64 20.8 -> 19.9, FP32 11.5 -> 10.8 us an iteration.
template <typename T>
__host__ __device__ constexpr int unroll_rows() { return sizeof(T) == 4 ? 2 : 1; }
// the r phase holds two values a row
template <typename T>
__host__ __device__ constexpr int unroll_rows_r() { return sizeof(T) == 4 ? 8 : 4; }

// A thread's rows are lo + threadIdx.x + 512 k in every phase, so its first rows of a phase can
// be loaded before the exchange that the phase waits for: only neighbours' r come from other
// blocks.

// CG phase 1 on rows [lo, hi): r -= alpha q; returns the thread's sum of r^2. (The matching
// x += alpha p is deferred to the next phase 2, which reads p anyway, or to the final pass:
// the same additions in the same order, without streaming x and p through this phase.)
template <typename T>
struct CgRowsR {
  static constexpr int U = unroll_rows_r<T>();
  T r[U], q[U];
  __device__ __forceinline__ void load(const SolveArgs<T>& a, int64_t lo, int n, int b) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = b + u * kCgThreads;
      if (i < n) { r[u] = a.cr[lo + i]; q[u] = a.cq[lo + i]; }
    }
  }
};
template <typename T>
__device__ __forceinline__ T cg_phase_r(const SolveArgs<T>& a, int64_t lo, int64_t hi, T alpha, CgRowsR<T>& w) {
  constexpr int U = CgRowsR<T>::U;
  T* R = a.cr + lo;
  const int n = (int)(hi - lo), bd = kCgThreads;
  T acc = T(0);
  for (int b = threadIdx.x; b < n; b += U * bd) {
    T rn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) rn[u] = w.r[u] - alpha * w.q[u];
    w.load(a, lo, n, b + U * bd);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = b + u * bd;
      if (i < n) {
        R[i] = rn[u];
        acc += rn[u] * rn[u];
      }
    }
  }
  return acc;
}

// The final pass on rows [lo, hi): the deferred x += alpha p of the part's last phase 1
// (pending), then back from the scaled unknowns onto the potential, phi += D^-1/2 x.
template <typename T>
__device__ __forceinline__ void cg_phase_x(const SolveArgs<T>& a, int64_t lo, int64_t hi, bool pending, T alpha) {
  const T* __restrict__ X = a.cx;
  const T* __restrict__ P = a.cp;
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const T x = pending ? X[i] + alpha * P[i] : X[i];
    a.phi[i] += (double)(x * __ldg(a.at_isd + i));
  }
}

// CG phase 2 on rows [lo, hi): x += alpha p (the previous phase 1's update, with the old p),
// p = r + beta p, q = S r + beta q (= S p, S = D^-1/2 A_T D^-1/2 with unit diagonal);
// returns the thread's sum of p.q.
template <typename T, bool kStream>
struct CgRows {
  static constexpr int U = unroll_rows<T>();
  T r[U], p[U], q[U], x[U];
  int4 nb[U];
  Coef4<T> c[U];
  __device__ __forceinline__ void load(const SolveArgs<T>& a, int64_t lo, int n, int b) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = b + u * kCgThreads;
      if (i < n) {
        nb[u] = load_op<kStream>(reinterpret_cast<const int4*>(a.at_nbr) + lo + i);
        c[u].template load<kStream>(a.at_scoef + 4 * lo, i);
        r[u] = load_synced(a.cr + lo + i);
        p[u] = a.cp[lo + i];
        q[u] = a.cq[lo + i];
        x[u] = kStream ? __ldcs(a.cx + lo + i) : a.cx[lo + i];
      }
    }
  }
};

template <typename T, bool kStream>
__device__ __forceinline__ T cg_phase_pq(const SolveArgs<T>& a, int64_t lo, int64_t hi, T beta, T alpha,
                                         CgRows<T, kStream>& w0) {
  constexpr int U = CgRows<T, kStream>::U;
  T* P = a.cp + lo;
  T* Q = a.cq + lo;
  T* X = a.cx + lo;
  const T* R0 = a.cr;
  const int n = (int)(hi - lo), bd = kCgThreads;
  T acc = T(0);
  // rows w of trip b; the next trip's go to nx behind this trip's gathers
  auto work = [&](const CgRows<T, kStream>& w, CgRows<T, kStream>& nx, int b) {
    T g[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (b + u * bd < n) {
        g[u][0] = load_synced(R0 + w.nb[u].x);
        g[u][1] = load_synced(R0 + w.nb[u].y);
        g[u][2] = load_synced(R0 + w.nb[u].z);
        g[u][3] = load_synced(R0 + w.nb[u].w);
      }
    }
    nx.load(a, lo, n, b + U * bd);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = b + u * bd;
      if (i < n) {
        T y = w.r[u];                   // unit diagonal
        y -= w.c[u].c[0] * g[u][0];
        y -= w.c[u].c[1] * g[u][1];
        y -= w.c[u].c[2] * g[u][2];
        y -= w.c[u].c[3] * g[u][3];
        const T pn = w.r[u] + beta * w.p[u];
        const T qn = y + beta * w.q[u];
        const T xn = w.x[u] + alpha * w.p[u];
        if (kStream) __stcs(X + i, xn);
        else X[i] = xn;
        P[i] = pn;
        Q[i] = qn;
        acc += pn * qn;
      }
    }
  };
  CgRows<T, kStream> w1;
  int b = threadIdx.x;
  while (b < n) {
    work(w0, w1, b);
    b += U * bd;
    if (b >= n) break;
    work(w1, w0, b);
    b += U * bd;
  }
  return acc;
}

// Shared memory of the kernels.
template <typename T>
struct OneShared {
  double sh[kCgThreads + 4];
  double total;
  T alpha, beta;
  int state;                           // 0 running, 1 converged, 2 breakdown, 3 idle
  int ok;
};

// CG on one part: scalars in shared memory, one exchange per phase. Returns false when a
// wait ran out; its: iterations.
template <typename T, bool kStream>
__device__ bool cg_one(const SolveArgs<T>& a, OneBlock& k, OneShared<T>& s, bool act, int& its) {
  const int64_t lo = k.lo, hi = k.hi;
  its = 0;
  double* const buf0 = a.buf;
  double* const buf1 = a.buf + a.n_sc;
  bool pending = false, ok;
  double rr = 0.0, rr0 = 0.0;          // warp 0's
  T acc = T(0);
  const int n = (int)(hi - lo);
  // r = D^-1/2 rhs, p = q = x = 0; the first p/q phase (beta = 0) then gives p = r, q = S r
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const T ri = act ? (T)(a.r_in[i] * (double)__ldg(a.at_isd + i)) : T(0);
    a.cr[i] = ri;
    a.cp[i] = T(0);
    a.cq[i] = T(0);
    a.cx[i] = T(0);
    acc += ri * ri;
  }
  CgRows<T, kStream> w;
  CgRowsR<T> wr;
  w.load(a, lo, n, threadIdx.x);
  ok = exchange_one(a, buf0, k, (double)acc, s.sh, &s.ok, [&](double t) {
    rr = rr0 = t;
    s.state = !act || t == 0.0 ? 3 : (t > 0.0 ? 0 : 2);
    s.alpha = s.beta = T(0);
  });
  while (ok && s.state == 0) {
    acc = cg_phase_pq<T, kStream>(a, lo, hi, s.beta, s.alpha, w);
    pending = false;                   // x += alpha p of the last r phase is applied
    wr.load(a, lo, n, threadIdx.x);
    ok = exchange_one(a, buf1, k, (double)acc, s.sh, &s.ok, [&](double pq) {
      if (!(pq > 0.0) || !isfinite(pq)) s.state = 2;
      else s.alpha = (T)(rr / pq);
    });
    if (!ok || s.state != 0 || its >= a.maxit_inner) break;
    acc = cg_phase_r<T>(a, lo, hi, s.alpha, wr);
    pending = true;
    ++its;
    w.load(a, lo, n, threadIdx.x);
    ok = exchange_one(a, buf0, k, (double)acc, s.sh, &s.ok, [&](double rrn) {
      if (!isfinite(rrn)) s.state = 2;
      else if (rrn <= a.inner_tol2 * rr0) s.state = 1;
      else s.beta = (T)(rrn / rr);
      rr = rrn;
    });
    if (its >= a.maxit_inner) break;
  }
  if (ok) cg_phase_x<T>(a, lo, hi, pending, s.alpha);
  return ok;
}

// One 512-thread block per SM (measured faster than two smaller-register blocks: fewer
// arrivals and partial sums, more rows in flight per thread).
template <typename T, bool kStream>
__global__ void __launch_bounds__(kCgThreads, kCgBlocksPerSm) k_cg(SolveArgs<T> a) {
  __shared__ OneShared<T> s;
  // (the end read once: with the load in the condition the phases' schedule changes, 750,000 cells
  // FP64 41.6 -> 43.9 ms a solve)
  for (int q = a.blk_work[blockIdx.x], q1 = a.blk_work[blockIdx.x + 1]; q < q1; ++q) {
    OneBlock k = one_block(a, q);
    int its = 0;
    const bool ok = cg_one<T, kStream>(a, k, s, a.active[k.part] != 0, its);
    if (k.sc == k.sc0 && threadIdx.x == 0) {      // out_status was zeroed with the barriers
      a.out_inner[k.part] = its;
      if (ok && s.state == 2) atomicMax(&a.out_status[0], 6);
      atomicMax(&a.out_status[1], its);
    }
    __syncthreads();
    if (!ok) break;
  }
}

// ---- a whole solve in one launch -----------------------------------------------
// The refinement loop of api.cu's solve_impl on the device: r = b - A phi on the full diamond
// operator, its norm, the stopping test, then the CG above with the correction added to phi
// in its last pass. An outer step as separate launches is six kernels and a host
// synchronisation around the CG, some 60 us on 10,000 cells against 60 us of CG; here it is
// three grid barriers. In an ensemble every part runs its own loop on its own blocks, where
// the launches' loop ran each inner solve to the slowest part's last iteration (16 meshes of 20k
// to 200k cells, mixed: 22.8 -> 9.2 ms a step). The operator is applied in two passes: vertex
// values, then per cell its faces' fluxes (each formed from both sides, the operations and their
// order those of k_face and k_update, so the residual has the same bits).
struct ResidualArgs {
  int64_t N, F, Fi;
  const int64_t* sptr;
  const int32_t* sidx;
  const double* alpha;
  const double* vdir;
  const int32_t* cell_face;
  const int4* nbr;                     // the other cell of every face slot (the cell itself on the boundary)
  const int32_t* fvert;
  const double* coef;
  const int8_t* bkind;
  const double* b;
  double* phi;
  double* uv;
  double* r;
  double rtol;
  int maxit_outer;
  int primed;                          // r holds b - A phi already
  const int* latched;                  // status word to check first, or null
  const int32_t* vert_begin;           // [P + 1] vertices of each part
  SolveInfoDev* info;                  // over all parts
  double* rel;                         // per part
  double* bn2;
  int* outer;
  int* inner;
  int* stat;
};

__device__ __forceinline__ void residual_vertices(const ResidualArgs& g, const OneBlock& k) {
  constexpr int U = 8;
  const int64_t end = g.vert_begin[k.part + 1];
  for (int64_t v = g.vert_begin[k.part] + (k.sc - k.sc0) * (int64_t)blockDim.x + threadIdx.x; v < end;
       v += (k.sc1 - k.sc0) * (int64_t)blockDim.x) {
    const int64_t b0 = g.sptr[v >> 5];
    const int width = (int)((g.sptr[(v >> 5) + 1] - b0) >> 5);
    const int32_t* col = g.sidx + b0 + (v & 31);
    const double* wcol = g.alpha + b0 + (v & 31);
    double s = 0.0;
    for (int c = 0; c < width; c += U) {
      int32_t j[U];
      double w[U], x[U];
#pragma unroll
      for (int q = 0; q < U; ++q) j[q] = c + q < width ? __ldg(col + 32 * (c + q)) : -1;
#pragma unroll
      for (int q = 0; q < U; ++q) {
        w[q] = j[q] >= 0 ? __ldg(wcol + 32 * (c + q)) : 0.0;
        x[q] = j[q] >= 0 ? load_synced(g.phi + j[q]) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (j[q] >= 0) s = __fma_rn(w[q], x[q], s);
    }
    const double d = g.vdir[v];
    g.uv[v] = d == d ? 0.0 : s;
  }
}

// r = b - A phi on the block's rows; returns the thread's sum of r^2
template <int D>
__device__ __forceinline__ double residual_rows(const ResidualArgs& g, int64_t lo, int64_t hi) {
  double sum = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    int32_t e[D + 1], vx[D + 1][3];
    double c[D + 1][3], o[D + 1], uvx[D + 1][3];
    bool on[D + 1], bnd[D + 1];
#pragma unroll
    for (int k = 0; k <= D; ++k) e[k] = g.cell_face[k * g.N + i];
    const int4 nb4 = __ldg(g.nbr + i);
    const int nb[4] = {nb4.x, nb4.y, nb4.z, nb4.w};
    const double me = load_synced(g.phi + i);
#pragma unroll
    for (int k = 0; k <= D; ++k) {
      const int64_t f = e[k] >= 0 ? e[k] : ~e[k];
      bnd[k] = f >= g.Fi;
      on[k] = !bnd[k] || g.bkind[f - g.Fi] == FVGB_BC_DIRICHLET;
      o[k] = bnd[k] ? 0.0 : load_synced(g.phi + nb[k]);
#pragma unroll
      for (int q = 0; q < D; ++q) {
        c[k][q] = __ldg(g.coef + q * g.F + f);
        vx[k][q] = __ldg(g.fvert + q * g.F + f);
      }
    }
#pragma unroll
    for (int k = 0; k <= D; ++k)
#pragma unroll
      for (int q = 0; q < D; ++q) uvx[k][q] = on[k] ? load_synced(g.uv + vx[k][q]) : 0.0;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k <= D; ++k) {
      const bool left = e[k] >= 0;
      const double ul = left ? me : o[k], ur = left ? o[k] : me;
      double q = __dmul_rn(c[k][0], __dsub_rn(ur, ul));
      if constexpr (D == 3) {
        q = __fma_rn(c[k][1], __dsub_rn(uvx[k][0], uvx[k][2]), q);
        q = __fma_rn(c[k][2], __dsub_rn(uvx[k][1], uvx[k][2]), q);
      } else {
        q = __fma_rn(c[k][1], __dsub_rn(uvx[k][1], uvx[k][0]), q);
      }
      if (on[k]) acc += left ? -q : q;
    }
    const double r = g.b[i] - acc;
    g.r[i] = r;
    sum += r * r;
  }
  return sum;
}

// barrier of the part's blocks without sums; false when the wait ran out
template <typename T>
__device__ bool one_barrier(const SolveArgs<T>& a, OneBlock& k) {
  bool ok = true;
  k.target += k.sc1 - k.sc0;
  __syncthreads();
  if (threadIdx.x < 32) {
    if (threadIdx.x == 0 && k.arrive) grid_arrive(k.bar);
    __syncwarp();
    ok = grid_wait(k.bar, k.status, k.target, a.barrier_ns);
  }
  return __syncthreads_and(ok) != 0;
}

// the refinement loop of one part
template <typename T, int D, bool kStream>
__device__ SolveInfoDev solve_part(const SolveArgs<T>& a, const ResidualArgs& g, OneBlock& k, OneShared<T>& s) {
  SolveInfoDev out{0, 0, 0, 0, 0.0, 0.0};
  double* const buf0 = a.buf + 2 * (size_t)a.n_sc;   // the CG uses the first two
  double* const buf1 = buf0 + a.n_sc;
  auto total = [&](double t) { s.total = t; };
  bool ok = true, run = true;
  double sum = 0.0, rel = 0.0;
  const int latched = g.latched ? *g.latched : 0;
  if (latched != 0) {                       // uniform over the grid: nothing writes it meanwhile
    out.latched = latched;
    run = false;
  } else {
    for (int64_t i = k.lo + threadIdx.x; i < k.hi; i += blockDim.x) sum += g.b[i] * g.b[i];
    ok = exchange_one(a, buf1, k, sum, s.sh, &s.ok, total);
    out.bn2 = ok ? s.total : 0.0;
    if (!isfinite(out.bn2)) { out.status = 6; run = false; }
  }
  const double bn2 = out.bn2;
  if (ok && run && bn2 == 0.0) {            // the solution is 0 (and then the residual 0)
    for (int64_t i = k.lo + threadIdx.x; i < k.hi; i += blockDim.x) {
      g.phi[i] = 0.0;
      g.r[i] = 0.0;
    }
    run = false;
  }
  for (int outer = 0; ok && run; ++outer) {
    sum = 0.0;
    if (outer == 0 && g.primed) {
      for (int64_t i = k.lo + threadIdx.x; i < k.hi; i += blockDim.x) sum += g.r[i] * g.r[i];
    } else {
      if (outer > 0 && !(ok = one_barrier(a, k))) break;      // phi of every block
      residual_vertices(g, k);
      if (!(ok = one_barrier(a, k))) break;                    // vertex values of every block
      sum = residual_rows<D>(g, k.lo, k.hi);
    }
    if (!(ok = exchange_one(a, outer & 1 ? buf1 : buf0, k, sum, s.sh, &s.ok, total))) break;
    rel = sqrt(s.total / bn2);
    out.outer = outer;
    out.rel = rel;
    if (!isfinite(rel)) { out.status = 6; break; }
    if (!(rel > g.rtol)) break;
    if (outer >= g.maxit_outer) { out.status = 5; break; }
    int its = 0;
    ok = cg_one<T, kStream>(a, k, s, true, its);
    out.inner += its;
    if (ok && s.state == 2) { out.outer = outer + 1; out.status = 6; break; }
  }
  if (!ok) out.status = 7;
  return out;
}

template <typename T, int D, bool kStream>
__global__ void __launch_bounds__(kCgThreads, kCgBlocksPerSm) k_solve(SolveArgs<T> a, ResidualArgs g) {
  __shared__ OneShared<T> s;
  for (int q = a.blk_work[blockIdx.x], q1 = a.blk_work[blockIdx.x + 1]; q < q1; ++q) {
    OneBlock k = one_block(a, q);
    const SolveInfoDev out = solve_part<T, D, kStream>(a, g, k, s);
    if (k.sc == k.sc0 && threadIdx.x == 0) {
      g.rel[k.part] = out.rel;
      g.bn2[k.part] = out.bn2;
      g.outer[k.part] = out.outer;
      g.inner[k.part] = out.inner;
      g.stat[k.part] = out.status;
      __threadfence();
      // the last part to finish sums up over all, in part order
      if (atomicAdd(&a.bar->count, 1u) == (unsigned)a.n_part - 1) {
        __threadfence();
        SolveInfoDev all{0, 0, 0, out.latched, 0.0, 0.0};
        for (int p = 0; p < a.n_part; ++p) {
          all.outer = max(all.outer, __ldcg(g.outer + p));
          all.inner = max(all.inner, __ldcg(g.inner + p));
          all.status = max(all.status, __ldcg(g.stat + p));
          all.rel = fmax(all.rel, __ldcg(g.rel + p));
          all.bn2 += __ldcg(g.bn2 + p);
        }
        *g.info = all;
      }
    }
    __syncthreads();
  }
}

// kStream in FP32 once an iteration's operator and vectors (48 bytes a cell) are beyond L2.
template <typename T>
bool cg_streams(const fvgb_mesh_s* m) { return sizeof(T) == 4 && 48 * m->topo.N > m->l2_bytes; }

// a kernel, not a memset: the same engine as its neighbours in the stream or graph
__global__ void k_barrier_reset(Barrier* bar, int n, int* cg_info) {
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    bar[p].count = 0;
    bar[p].status = 0;
  }
  if (threadIdx.x < 2) cg_info[threadIdx.x] = 0;
}

// Per part the sum of its sub-chunks' partial sums, in order.
__global__ void __launch_bounds__(kCgThreads) k_part_sumsq_final(const double* __restrict__ buf,
    const int32_t* __restrict__ part_sc, int n_part, double* __restrict__ out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int p = warp; p < n_part; p += nw) {
    double t = 0.0;
    for (int sc = part_sc[p] + lane; sc < part_sc[p + 1]; sc += 32) t += buf[sc];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) out[p] = t;
  }
}

// Per-part sums of r0 (r0 - r1), (r0 - r1)^2, r0^2 and r1^2 over the same sub-chunks, for
// the scale of a correction whose operator image is r0 - r1 (partials per sub-chunk: four
// block sums, in buf[k * n_sc + sc]).
__global__ void __launch_bounds__(kCgThreads) k_part_dots_partial(const double* __restrict__ r0,
    const double* __restrict__ r1, const int64_t* __restrict__ sc_begin, int n_sc, double* __restrict__ buf) {
  __shared__ double sh[kCgThreads];
  const int sc = blockIdx.x;
  double a = 0.0, b = 0.0, c0 = 0.0, c1 = 0.0;
  for (int64_t i = sc_begin[sc] + threadIdx.x; i < sc_begin[sc + 1]; i += blockDim.x) {
    const double x = r0[i], y = r1[i];
    const double d = x - y;
    a += x * d;
    b += d * d;
    c0 += x * x;
    c1 += y * y;
  }
  a = block_sum(a, sh);
  b = block_sum(b, sh);
  c0 = block_sum(c0, sh);
  c1 = block_sum(c1, sh);
  if (threadIdx.x == 0) {
    buf[sc] = a;
    buf[n_sc + sc] = b;
    buf[2 * n_sc + sc] = c0;
    buf[3 * n_sc + sc] = c1;
  }
}

}  // namespace

cudaError_t launch_barrier_reset(fvgb_mesh_s* m, cudaStream_t s) {
  k_barrier_reset<<<1, 32, 0, s>>>(m->barrier, m->parts.n_part + 1, m->d_cg_info);
  count_launch();
  return cudaGetLastError();
}

int solve_grid_size(fvgb_mesh_s* m) {
  const void* kernels[] = {(const void*)k_cg<float, false>, (const void*)k_cg<float, true>,
                           (const void*)k_cg<double, false>,
                           (const void*)k_solve<float, 2, false>, (const void*)k_solve<float, 3, false>,
                           (const void*)k_solve<float, 2, true>, (const void*)k_solve<float, 3, true>,
                           (const void*)k_solve<double, 2, false>, (const void*)k_solve<double, 3, false>};
  int per_sm = kCgBlocksPerSm;
  for (const void* k : kernels) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kCgThreads, 0) != cudaSuccess) return 0;
    per_sm = n < per_sm ? n : per_sm;
  }
  return per_sm < 1 ? 0 : per_sm * m->num_sms;
}

cudaError_t launch_part_dots(fvgb_mesh_s* m, const double* r0, const double* r1, double* out, cudaStream_t s) {
  const PartsDev& pd = m->parts;
  k_part_dots_partial<<<pd.n_sc, kCgThreads, 0, s>>>(r0, r1, pd.sc_begin, pd.n_sc, pd.buf);
  for (int k = 0; k < 4; ++k)
    k_part_sumsq_final<<<1, kCgThreads, 0, s>>>(pd.buf + k * pd.n_sc, pd.part_sc, pd.n_part, out + k * pd.n_part);
  count_launch(5);
  return cudaGetLastError();
}

namespace {
template <typename T>
SolveArgs<T> solve_args(fvgb_mesh_s* m, int bcset, const double* r, double inner_rtol, int maxit, double* phi) {
  GeoDev<T>& g = geo_of<T>(m);
  Work<T>& w = work_of<T>(m);
  SolveArgs<T> a;
  a.at_nbr = g.bc[bcset].at_nbr; a.at_scoef = g.bc[bcset].at_scoef; a.at_isd = g.bc[bcset].at_isd;
  a.r_in = r;
  a.phi = phi;
  a.cx = w.cg_x; a.cr = w.cg_r; a.cp = w.cg_p; a.cq = w.cg_q;
  const PartsDev& pd = m->parts;
  a.n_part = pd.n_part; a.n_sc = pd.n_sc;
  a.blk_work = pd.blk_work; a.work = pd.work;
  a.active = pd.active; a.buf = pd.buf;
  a.bar = m->barrier;
  a.inner_tol2 = inner_rtol * inner_rtol;
  a.maxit_inner = maxit;
  a.out_inner = pd.out_inner;
  a.out_status = m->d_cg_info;
  a.skip_block = m->test_skip_block;
  a.barrier_ns = m->test_barrier_ns > 0 ? m->test_barrier_ns : kBarrierTimeoutNs;
  return a;
}

template <typename T>
cudaError_t launch_whole(fvgb_mesh_s* m, int bcset, ResidualArgs& g, const double* r, const fvgb_solve_opts* o,
                         cudaStream_t s) {
  SolveArgs<T> a = solve_args<T>(m, bcset, r, o->inner_rtol, o->maxit_inner, g.phi);
  cudaError_t e = launch_barrier_reset(m, s);
  if (e != cudaSuccess) return e;
  void* args[] = {&a, &g};
  const void* k = m->topo.dim == 3 ? (const void*)k_solve<T, 3, false> : (const void*)k_solve<T, 2, false>;
  if constexpr (sizeof(T) == 4) {
    if (cg_streams<T>(m)) k = m->topo.dim == 3 ? (const void*)k_solve<T, 3, true> : (const void*)k_solve<T, 2, true>;
  }
  count_launch();
  return cudaLaunchCooperativeKernel(k, dim3(m->solve_grid), dim3(kCgThreads), args, 0, s);
}
}  // namespace

template <typename T>
cudaError_t launch_cg(fvgb_mesh_s* m, int bcset, const double* r, double inner_rtol, int maxit, double* phi,
                      cudaStream_t s) {
  SolveArgs<T> a = solve_args<T>(m, bcset, r, inner_rtol, maxit, phi);
  cudaError_t e = launch_barrier_reset(m, s);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  count_launch();
  const void* k = (const void*)k_cg<T, false>;
  if constexpr (sizeof(T) == 4) {
    if (cg_streams<T>(m)) k = (const void*)k_cg<T, true>;
  }
  return cudaLaunchCooperativeKernel(k, dim3(m->solve_grid), dim3(kCgThreads), args, 0, s);
}

// The whole solve in one launch. A single mesh up to kSolveOneMax cells; a solve to 1e-8 against
// separate launches: 10,368 cells FP64 3.46 -> 2.26 ms, 384,000 13.4 -> 11.9 (mixed 9.7 -> 8.8);
// 750,000 equal; 1.3M 38.8 -> 43.1: one 512-thread block an SM streams the operator's passes slower
// than their own kernels. An ensemble gains more, since no part waits for another's inner solve
// (mixed / FP64, ms: 16 x 162,000 74 -> 52 / 164 -> 109, 8 x 750,000 213 -> 175 / 430 -> 394,
// 2 x 750,000 52 -> 44 / 107 -> 101; 2 x 3M mixed 227 -> 226), but in FP64, bound by its issue,
// not with few parts of more than kSolveOneMean64 cells (2 x 1.3M 181 -> 207, 4 x 1.3M 389 -> 409,
// 2 x 3M 456 -> 513). (CUDA-event timing of the CG wants its own launches.)
constexpr int64_t kSolveOneMax = 600000, kSolveOneMean64 = 1000000;

bool solve_one_ok(const fvgb_mesh_s* m, const fvgb_solve_opts* o) {
  if (o->inner != 0 || m->time_cg) return false;
  const int64_t N = m->topo.N, P = m->parts.n_part;
  return P == 1 ? N <= kSolveOneMax : o->prec != FVGB_FP64 || N <= kSolveOneMean64 * P;
}

cudaError_t launch_solve_one(fvgb_mesh_s* m, int bcset, const double* b, double* phi, double* r, bool primed,
                             const fvgb_solve_opts* o, bool check_latched, SolveInfoDev* info, double* rel,
                             int* outer, int* inner, cudaStream_t s) {
  const TopoDev& t = m->topo;
  const BCDev<double>& bc = m->g64.bc[bcset];
  ResidualArgs g;
  g.N = t.N; g.F = t.F; g.Fi = t.Fi;
  g.sptr = t.vsell.ptr; g.sidx = t.vsell.idx;
  g.alpha = m->g64.valpha; g.vdir = bc.vdir;
  g.cell_face = t.cell_face; g.nbr = reinterpret_cast<const int4*>(bc.at_nbr);
  g.fvert = t.fvert; g.coef = m->g64.coef; g.bkind = bc.bkind;
  g.b = b; g.phi = phi; g.uv = m->w64.uv; g.r = r;
  g.rtol = o->rtol; g.maxit_outer = o->maxit_outer;
  g.primed = primed ? 1 : 0;
  g.latched = check_latched ? m->d_status : nullptr;
  g.info = info;
  g.vert_begin = m->parts.vert_begin;
  g.rel = rel; g.outer = outer; g.inner = inner;
  g.bn2 = m->parts.bn2; g.stat = m->parts.stat;
  const bool fp32 = o->prec == FVGB_FP32 || o->prec == FVGB_MIXED;
  return fp32 ? launch_whole<float>(m, bcset, g, r, o, s) : launch_whole<double>(m, bcset, g, r, o, s);
}

template cudaError_t launch_cg<double>(fvgb_mesh_s*, int, const double*, double, int, double*, cudaStream_t);
template cudaError_t launch_cg<float>(fvgb_mesh_s*, int, const double*, double, int, double*, cudaStream_t);

}  // namespace fvgb
