// kern_1d_cluster.cu -- a whole multi-step advance of a small 1D mesh on one
// thread-block cluster.
//
// Every CTA of the cluster owns `per` neighbouring cells, one thread each, and
// keeps their state in registers for all the steps of the call.  W is put in
// shared memory before each RK stage; a cell's neighbours are read from
// whichever CTA owns them (distributed shared memory), and the CTAs meet at the
// hardware's cluster barrier, twice a step:
//   W(U^n) and the CTA's CFL speeds to shared memory          cluster barrier
//   dt from all speeds, K = L[U^n], W(U^n + dt K)             cluster barrier
//   L[U^n + dt K], U^{n+1}
// Two more threads per CTA form the face values of the cells beyond its ends, so
// that each face is computed by the CTA above it and, at a seam, once more by the
// CTA below (the same bits).  Cells, faces, dt and time are computed by the
// functions of the multi-launch path, so they are bitwise the same; the step
// totals, which only the call's last step leaves behind, agree to rounding.
// Steps after t_end is reached change nothing but dt = 0 and the totals of the
// final state: the first of them is taken and the rest are not.
//
// What bounds it: one warp's chain of FP64 operations (an SM retires two FP64
// lanes a clock, and the chain has some 200 a stage), so the cells spread over
// the 16 SMs of the largest cluster.  Against the grid-wide
// cooperative launch (kern_1d_advance.cu, two grid barriers of 3 us and the
// state through L2): FP64 22 -> 11.2 us a step from 32 to 512 cells and 25 ->
// 23.5 at 4088, FP32 22 -> 2.8 and 25 -> 4.6; Sod's 256 cells in FP64 to t = 0.2
// in calls of 64 steps, 4.44 -> 1.73 ms (a quarter of it from the 52 steps past
// the end).
#include <cooperative_groups.h>

#include "finalize.cuh"
#include "registry.h"
#include "stage_kernel.cuh"

namespace gh {

namespace cg = cooperative_groups;

namespace {

constexpr int MAX_THREADS = 288;  // 256 cells and the two end threads, in whole warps

template <class T, int SOLVER>
__global__ void __launch_bounds__(MAX_THREADS)
    hydro_1d_cluster_kernel(StageArgs<T> A, FinalizeArgs F, int nsteps, const T* uin, T* uout, int per) {
  using Base = StageKernel<1, T, SOLVER, 1, 32, 1, false>;
  constexpr int NV = 3;
  extern __shared__ __align__(16) unsigned char smem_c[];
  cg::cluster_group cluster = cg::this_cluster();
  const int n = A.n[0], rank = blockIdx.x, ranks = gridDim.x, nwarps = blockDim.x >> 5;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  double* const speeds = reinterpret_cast<double*>(smem_c);          // [nwarps], one per warp
  double* const sums = speeds + MAX_THREADS / 32;                    // [nwarps][NV]
  T* const w_s = reinterpret_cast<T*>(sums + NV * MAX_THREADS / 32);  // W: [2 stages][NV][per]
  T* const hi_s = w_s + 2 * NV * per;                                // upper face values of cells -1 .. per - 1
  T* const f_s = hi_s + NV * (per + 1);                              // fluxes of faces 0 .. per

  const int base = rank * per, cnt = min(per, n - base);
  const bool own = t < cnt;
  const bool below = t == per + 1;           // the thread of cell base - 1
  const bool part = t <= cnt || below;       // t == cnt: the thread of cell base + cnt
  const int i = below ? -1 : t;
  // the cell and its neighbours: where their W is, mirrored or not
  const T* at[3];
  bool flip[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int src = part ? bc_map(base + i + d - 1, n, A.bc_lo[0], A.bc_hi[0], flip[d]) : base;
    if (!part) flip[d] = false;
    const int owner = src / per;
    at[d] = cluster.map_shared_rank(w_s + (src - owner * per), owner);
  }
  const Geo<T> g = Base::geo(A, 0, base + i);
  const T iw = A.iw[0][min(base + t, n + 1) + 2];

  T u[NV] = {T(1), T(0), T(1)}, w[NV] = {T(1), T(0), T(1)};
  if (own) {
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = uin[(size_t)v * n + base + t];
  }
  bool bad = false;

  // W of `s` into shared memory for stage b
  auto publish = [&](const T (&s)[NV], int b) {
    recover<1>(s, w);
    if (own) {
      bad |= Base::nonphysical(w, A.gm1);
#pragma unroll
      for (int v = 0; v < NV; ++v) w_s[(b * NV + v) * per + t] = w[v];
    }
  };
  // minus the flux divergence (and the source) of the own cell from stage b's W
  auto rhs = [&](int b, T (&L)[NV]) {
    T lo[NV];
    if (part) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int o = (b * NV + v) * per;
        T wm = at[0][o], wc = own ? w[v] : at[1][o], wp = at[2][o], hi;
        if (v == 1) {
          wm = flip[0] ? -wm : wm;
          wc = flip[1] ? -wc : wc;
          wp = flip[2] ? -wp : wp;
        }
        face_pair(limited_slope(wm, wc, wp, g), g.h, wc, lo[v], hi);
        if (own || below) hi_s[v * (per + 1) + i + 1] = hi;
      }
    }
    __syncthreads();
    if (t <= cnt) {
      T wl[NV], f[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) wl[v] = hi_s[v * (per + 1) + t];
      face_flux<T, 1, 0, SOLVER>(wl, lo, A.gamma, A.gm1, f);
#pragma unroll
      for (int v = 0; v < NV; ++v) f_s[v * (per + 1) + t] = f[v];
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NV; ++v)
      L[v] = own ? mul_rn(sub_rn(f_s[v * (per + 1) + t], f_s[v * (per + 1) + t + 1]), iw) : T(0);
    if (A.has_source) Base::add_source(A, w, L);
  };

  double time = F.scal[SCAL_T], dt = 0.0, speed_inv = 0.0;
  for (int s = 0; s < nsteps; ++s) {
    publish(u, 0);
    T sp = T(0);
    if (own) sp = mul_rn(add_rn(fabs(w[1]), sound_speed(A.gamma, mul_rn(A.gm1, w[2]), w[0])), iw);
    const double ws = (double)warp_max(sp);
    if (lane == 0) speeds[warp] = ws;
    cluster.sync();
    // every warp takes the maximum over all warps of the cluster: the same dt
    unsigned long long mb = 0;
    for (int k = lane; k < ranks * nwarps; k += 32) {
      const int r = k / nwarps;
      const double x = *cluster.map_shared_rank(speeds + (k - r * nwarps), r);
      const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
      mb = b > mb ? b : mb;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long b = __shfl_xor_sync(0xffffffffu, mb, o);
      mb = b > mb ? b : mb;
    }
    dt = fin::step_dt(F, mb, time);
    const bool done = F.t_end > 0.0 && time >= F.t_end;  // this step and all later ones change nothing
    const bool last = done || s == nsteps - 1;
    if (last) {
      speed_inv = 1.0 / __longlong_as_double((long long)mb);
      if (F.part_tot) {  // totals of U^n: warps here, CTAs at the end
        const double dx = own ? A.wd[0][base + t] : 0.0;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const double x = warp_sum(own ? (double)u[v] * dx : 0.0);
          if (lane == 0) sums[warp * NV + v] = x;
        }
      }
    }
    if (done) break;
    time += dt;
    const T d = (T)dt;
    T K[NV], L[NV], u1[NV];
    rhs(0, K);
#pragma unroll
    for (int v = 0; v < NV; ++v) u1[v] = fma_rn(d, K[v], u[v]);
    publish(u1, 1);
    cluster.sync();
    rhs(1, L);
    const T hd = half_of(d);
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = fma_rn(hd, add_rn(K[v], L[v]), u[v]);
  }
  if (own) {
#pragma unroll
    for (int v = 0; v < NV; ++v) uout[(size_t)v * n + base + t] = u[v];
  }
  if (bad) atomicOr(A.status, STATUS_NONPHYS);
  cluster.sync();  // the totals of every CTA
  if (rank == 0 && t == 0) {
    F.scal[SCAL_DT] = dt;
    F.scal[SCAL_T] = time;
    F.scal[SCAL_DTCFL] = speed_inv;
  }
  if (rank == 0 && F.part_tot && t < NV) {
    double acc = 0.0;
    for (int r = 0; r < ranks; ++r) {
      const double* q = cluster.map_shared_rank(sums, r);
      for (int k = 0; k < nwarps; ++k) acc += q[k * NV + t];
    }
    F.scal[SCAL_TOT + t] = acc;
  }
  cluster.sync();  // shared memory of a CTA stays until the others have read it
}

template <class T>
const void* pick(int solver) {
  if (solver == SOLVER_HLL) return reinterpret_cast<const void*>(&hydro_1d_cluster_kernel<T, SOLVER_HLL>);
  if (solver == SOLVER_HLLC) return reinterpret_cast<const void*>(&hydro_1d_cluster_kernel<T, SOLVER_HLLC>);
  return nullptr;
}

}  // namespace

bool cluster_1d_plan(bool fp64, int solver, int n, Cluster1D* out) {
  const void* fn = fp64 ? pick<double>(solver) : pick<float>(solver);
  if (!fn) return false;
  constexpr int MAX_RANKS = 16;
  int per = (n + MAX_RANKS - 1) / MAX_RANKS;
  if (per < 8) per = 8;
  const int ranks = (n + per - 1) / per, threads = (per + 2 + 31) / 32 * 32;
  if (threads > MAX_THREADS) return false;
  const size_t es = fp64 ? sizeof(double) : sizeof(float);
  const size_t smem = (1 + 3) * (MAX_THREADS / 32) * sizeof(double) + (size_t)(2 * 3 * per + 2 * 3 * (per + 1)) * es;
  if (ranks > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  out->fn = fn;
  out->per = per;
  out->ranks = ranks;
  out->threads = threads;
  out->smem = smem;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  cluster_1d_config(*out, nullptr, &cfg, at);
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return clusters >= 1;
}

void cluster_1d_config(const Cluster1D& c, cudaStream_t st, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)c.ranks;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg->gridDim = dim3((unsigned)c.ranks);
  cfg->blockDim = dim3((unsigned)c.threads);
  cfg->dynamicSmemBytes = c.smem;
  cfg->stream = st;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

}  // namespace gh
