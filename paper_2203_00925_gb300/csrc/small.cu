// Explicit time steps on small meshes (fvgb_fv_step, first-order upwind): all steps and
// stages of a call in one cooperative launch.
//
// A stage of a small mesh is three kernels (vertex values, face fluxes, update) of some four
// microseconds each, nearly all of it launch and dependent-load latency. Here every block keeps
// its cells' part of the mesh for the whole call - star lists and weights in shared memory, face
// data in registers - and a stage is: gather u, barrier. Four lanes work on a cell: lane k
// forms the least-squares value of the cell's vertex k and the flux of its face k (opposite
// vertex k); the lanes exchange vertex values and fluxes by shuffles. Vertex values and fluxes
// are formed once per cell around them instead of once, with the same operations in the same
// order, so the results are the bits of the three kernels.
//
// 200 Euler steps of 5,000 triangles, FP64: 2.46 ms as 600 launches, 0.577 ms in one (2.9 us a
// step: a grid barrier of 1.2 us, the chain of dependent FP64 operations and one L2 gather).
#include <cuda_runtime.h>

#include <algorithm>

#include "grid_sync.cuh"
#include "internal.h"
#include "rounded.cuh"

namespace fvgb {
namespace {

constexpr int kSmallThreads = 512;
constexpr int kSmallCells = kSmallThreads / 4;   // cells of a block
constexpr int kSmallStages = 8;                  // stages of a step (fvgb_fv_step's limit)

template <typename T>
struct SmallArgs {
  int64_t N, F, Fi;
  const int32_t* cell_face;
  const int32_t* fL;
  const int32_t* fR;
  const int32_t* fvert;
  const int32_t* cverts;
  const int64_t* sptr;        // stars
  const int32_t* sidx;
  const T* alpha;
  const T* vdir;
  const T* S;
  const T* coef;
  const int8_t* bkind;
  const T* bval;
  const T* inv_vol;
  const T* src;
  const T* vel;
  T vc[3];
  T diff;
  T* u;
  T* w[2];
  int nsteps, nstage;
  T adt[kSmallStages];
  int star_max;
  Barrier* bar;
  unsigned arrivals;              // that a barrier waits for: the blocks (test hook: one more)
  unsigned long long barrier_ns;  // limit of a barrier wait
  int* status;
};

template <typename T, int D>
__global__ void __launch_bounds__(kSmallThreads) k_small_steps(SmallArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  T* const sw = reinterpret_cast<T*>(smem);                       // [star_max][threads] weights
  int32_t* const sj = reinterpret_cast<int32_t*>(sw + (size_t)a.star_max * blockDim.x);
  constexpr int kInterior = 3, kNone = 4;
  const int64_t c0 = blockIdx.x * a.N / gridDim.x, c1 = (blockIdx.x + 1) * a.N / gridDim.x;
  const int k = threadIdx.x & 3;
  const int64_t i = c0 + (threadIdx.x >> 2);
  const bool cell = i < c1;
  const bool lane = cell && k <= D;          // this lane has a vertex and a face
  const bool diff = a.diff != T(0);
  // the vertex: its star into shared memory
  int width = 0;
  T vfix = T(0);
  bool fixed = false;
  if (lane && diff) {
    const int32_t v = a.cverts[i * (D + 1) + k];
    const int64_t b0 = a.sptr[v >> 5];
    width = (int)((a.sptr[(v >> 5) + 1] - b0) >> 5);
    for (int c = 0; c < width; ++c) {
      sj[c * blockDim.x + threadIdx.x] = a.sidx[b0 + (v & 31) + 32 * c];
      sw[c * blockDim.x + threadIdx.x] = a.alpha[b0 + (v & 31) + 32 * c];
    }
    vfix = a.vdir[v];
    fixed = vfix == vfix;
  }
  // the face: neighbour, kind, coefficients, V_f . S_f, and the lanes of its vertices
  int kind = kNone, lanes[3] = {0, 0, 0};
  int64_t other = 0;
  bool left = true;                          // this cell is the face's L
  T gb = T(0), cf[3] = {T(0), T(0), T(0)}, vn = T(0);
  if (lane) {
    const int32_t e = a.cell_face[k * a.N + i];
    left = e >= 0;
    const int64_t f = left ? e : ~e;
    const int32_t L = a.fL[f], R = f < a.Fi ? a.fR[f] : -1;
    other = left ? R : L;
    if (f < a.Fi) {
      kind = kInterior;
    } else {
      kind = a.bkind[f - a.Fi];
      gb = a.bval[f - a.Fi];
      other = i;
    }
    T vf[3];
#pragma unroll
    for (int q = 0; q < D; ++q) {
      cf[q] = a.coef[q * a.F + f];
      if (a.vel) {
        const T vl = a.vel[q * a.N + L], vr = R >= 0 ? a.vel[q * a.N + R] : vl;
        vf[q] = mul_rn(T(0.5), add_rn(vl, vr));
      } else {
        vf[q] = a.vc[q];
      }
    }
    vn = fma_rn(vf[1], a.S[a.F + f], mul_rn(vf[0], a.S[f]));
    if (D == 3) vn = fma_rn(vf[2], a.S[2 * a.F + f], vn);
#pragma unroll
    for (int q = 0; q < D; ++q) {
      const int32_t v = a.fvert[q * a.F + f];
#pragma unroll
      for (int p = 0; p <= D; ++p)
        if (a.cverts[i * (D + 1) + p] == v) lanes[q] = p;
    }
  }
  const bool uses_vertices = diff && (kind == kInterior || kind == FVGB_BC_DIRICHLET);
  const T inv_vol = cell ? a.inv_vol[i] : T(0);
  const T src = cell && a.src ? a.src[i] : T(0);
  T base = cell ? a.u[i] : T(0);             // the cell's value at the start of the step
  T ui = base;
  const T* in = a.u;
  unsigned target = 0;
  const int total = a.nsteps * a.nstage;
  int bad = 0;
  for (int s = 0, stage = 0; s < total; ++s) {
    T* out = s + 1 == total ? a.u : a.w[s & 1];
    // gathers: the star of the vertex (four in flight) and the face's other cell
    const T uo = kind == kInterior ? load_synced(in + other) : T(0);
    T uv = T(0);
    {
      int c = 0;
      for (; c + 4 <= width; c += 4) {
        T g[4], w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          g[q] = load_synced(in + sj[(c + q) * blockDim.x + threadIdx.x]);
          w[q] = sw[(c + q) * blockDim.x + threadIdx.x];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) uv = fma_rn(w[q], g[q], uv);
      }
      for (; c < width; ++c)
        uv = fma_rn(sw[c * blockDim.x + threadIdx.x], load_synced(in + sj[c * blockDim.x + threadIdx.x]), uv);
      if (fixed) uv = vfix;
    }
    const T va = __shfl_sync(0xffffffffu, uv, lanes[0], 4), vb = __shfl_sync(0xffffffffu, uv, lanes[1], 4),
            vcc = __shfl_sync(0xffffffffu, uv, lanes[2], 4);
    T Ff = T(0);
    if (kind != kNone && kind != FVGB_BC_WALL) {
      const T far = kind == kInterior ? uo : (kind == FVGB_BC_DIRICHLET ? gb : ui);
      const T ul = left ? ui : far, ur = left ? far : ui;
      Ff = mul_rn(vn, vn >= T(0) ? ul : ur);
      if (uses_vertices) {
        T q = mul_rn(cf[0], sub_rn(ur, ul));
        if constexpr (D == 3) {
          q = fma_rn(cf[1], sub_rn(va, vcc), q);
          q = fma_rn(cf[2], sub_rn(vb, vcc), q);
        } else {
          q = fma_rn(cf[1], sub_rn(vb, va), q);
        }
        Ff = fma_rn(-a.diff, q, Ff);
      }
    }
    if (left) Ff = -Ff;                       // entering minus leaving
    T acc = T(0);
#pragma unroll
    for (int q = 0; q <= D; ++q) acc += __shfl_sync(0xffffffffu, Ff, q, 4);
    const T r = acc * inv_vol + src;
    const T v = base + a.adt[stage] * r;
    ui = v;
    if (++stage == a.nstage) { stage = 0; base = v; }
    if (cell && k == 0) {
      out[i] = v;
      if (!isfinite(v)) bad = 1;
    }
    in = out;
    if (s + 1 == total) break;
    target += a.arrivals;
    __syncthreads();
    bool ok = true;
    if (threadIdx.x < 32) {
      if (threadIdx.x == 0) grid_arrive(a.bar);
      __syncwarp();
      ok = grid_wait(a.bar, &a.bar->status, target, a.barrier_ns);
    }
    if (!__syncthreads_and(ok)) {             // latched: reported by fvgb_sync
      if (threadIdx.x == 0) atomicOr(a.status, 2);
      break;
    }
  }
  if (bad) atomicOr(a.status, 1);
}

template <typename T>
size_t small_smem(const fvgb_mesh_s* m, int threads) {
  return (size_t)m->topo.star_max * threads * (sizeof(T) + sizeof(int32_t));
}

int small_threads(const fvgb_mesh_s* m) {
  const int64_t G = m->num_sms;
  const int64_t cells = (m->topo.N + G - 1) / G;
  return (int)((4 * cells + 31) / 32 * 32);
}

template <typename T>
const void* small_kernel(const fvgb_mesh_s* m) {
  return m->topo.dim == 3 ? (const void*)k_small_steps<T, 3> : (const void*)k_small_steps<T, 2>;
}

}  // namespace

// Whether a call of ``stages`` stages in all runs as one launch: at least two stages, at most
// kSmallCells cells a block with one block an SM (four lanes a cell hold their face data in
// registers), and stars that fit shared memory. The line is what a block can hold, not where the
// two meet: 19,208 triangles take 5.0 us a step in one launch (FP32 2.3), 19,602 take 12.4 in
// three kernels a stage (FP32 12.4).
bool step_small_ok(const fvgb_mesh_s* m, int64_t stages) {
  return m->small_ok && stages >= 2 && stages < (int64_t(1) << 22);
}

// At upload: are the mesh's blocks within the kernel's limits, and its shared memory.
cudaError_t prepare_small(fvgb_mesh_s* m) {
  m->small_ok = false;
  const bool fp32 = is_fp32(m);
  const int threads = small_threads(m);
  if (threads > kSmallThreads) return cudaSuccess;
  const size_t smem = fp32 ? small_smem<float>(m, threads) : small_smem<double>(m, threads);
  int limit = 0;
  cudaError_t e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, m->device);
  if (e != cudaSuccess || smem > (size_t)limit) return e;
  const void* k = fp32 ? small_kernel<float>(m) : small_kernel<double>(m);
  if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, limit))) return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem))) return e;
  m->small_ok = per_sm >= 1;
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_small_steps(fvgb_mesh_s* m, const fvgb_tcoef* tc, T* u, double dt, int nsteps,
                               const double* alpha, int nstage, cudaStream_t s) {
  const TopoDev& t = m->topo;
  GeoDev<T>& g = geo_of<T>(m);
  Work<T>& w = work_of<T>(m);
  const BCDev<T>& b = g.bc[tc->bcset];
  SmallArgs<T> a;
  a.N = t.N; a.F = t.F; a.Fi = t.Fi;
  a.cell_face = t.cell_face; a.fL = t.fL; a.fR = t.fR; a.fvert = t.fvert; a.cverts = t.cverts;
  a.sptr = t.vsell.ptr; a.sidx = t.vsell.idx;
  a.alpha = g.valpha; a.vdir = b.vdir; a.S = g.S; a.coef = g.coef;
  a.bkind = b.bkind; a.bval = b.bval; a.inv_vol = g.inv_vol;
  a.src = (const T*)tc->src_dev;
  a.vel = (const T*)tc->vel_dev;
  for (int q = 0; q < 3; ++q) a.vc[q] = (T)tc->vel_const[q];
  a.diff = (T)tc->diff;
  a.u = u;
  a.w[0] = w.stage; a.w[1] = w.tmp;
  a.nsteps = nsteps; a.nstage = nstage;
  for (int q = 0; q < nstage; ++q) a.adt[q] = (T)(alpha[q] * dt);
  a.star_max = t.star_max;
  a.bar = m->barrier;
  const unsigned grid = (unsigned)std::min<int64_t>(m->num_sms, t.N);
  a.arrivals = grid + (m->test_skip_block >= 0 ? 1 : 0);
  a.barrier_ns = m->test_barrier_ns > 0 ? m->test_barrier_ns : kBarrierTimeoutNs;
  a.status = m->d_status;
  const int threads = small_threads(m);
  cudaError_t e = launch_barrier_reset(m, s);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  count_launch();
  return cudaLaunchCooperativeKernel(small_kernel<T>(m), dim3(grid), dim3(threads), args, small_smem<T>(m, threads), s);
}

template cudaError_t launch_small_steps<float>(fvgb_mesh_s*, const fvgb_tcoef*, float*, double, int, const double*, int, cudaStream_t);
template cudaError_t launch_small_steps<double>(fvgb_mesh_s*, const fvgb_tcoef*, double*, double, int, const double*, int, cudaStream_t);

}  // namespace fvgb
