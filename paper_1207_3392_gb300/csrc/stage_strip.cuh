// stage_strip.cuh -- RK stages on independent warps.
//
// 1D and 2D (StripKernel): a warp takes a strip of 28 columns (lane l holds
// column x0 + l - 2: two neighbours on each side) and marches along y.  The
// march axis lives in a register ring, as in stage_kernel.cuh; along x the
// warp's own shuffles move what neighbouring columns need: W of the two
// neighbours for the slope, the upper face value of the lower neighbour, and
// the flux of the upper face.  Each slope and each face flux is computed once
// per lane, nothing goes through shared memory, and no warp waits for another.
//
// 3D: two launches a stage.  The strips march along y in every plane and leave
// minus the x and y parts of the divergence in the stage's output array; then
// every thread takes one (x, y) column and marches along z (ZMarch): it adds
// the z part and finishes the cell (source, output, CFL speed, totals).
//
// What bounds it, and why this split.  2D: the row tiles it replaced (one row
// of a CTA per plane, two barriers a row, every x slope formed twice) ran about
// 640 instructions a cell at 47-67% of the issue slots, their warps waiting at
// the barriers.  Stages 1 and 2 of the row tiles and of the strips, HLLC with
// totals: 40.0 and 36.9 -> 28.2 and 26.6 us at 1024^2, 22.7 and 18.4 -> 13.2
// and 12.3 us at 256 x 768.  565 and 523 instructions a cell at 1024^2 (of them
// 54 and 0 for the compensated totals), 78% of the issue slots at 4096^2.
// 3D, FP32 HLLC at 256^3: the 32 x 8 tiles ran 981 and 894 instructions a cell at
// 64% of the issue slots, held back by two barriers a plane, 24 warps and 160
// halo cells recovered for 256 own ones: stages 1 and 2 685 and 660 us.  Here
// the strips run 485 and 512 (of 32 lanes 25.6 own a column at nx = 256) at 77%,
// and ZMarch 440 and 324 at 79% and 66%: 493 and 490 us together.  The price is
// memory traffic, 100 and 140 algorithmic bytes a cell for 40 and 60, half of
// what the launches' times could move.  Double word at 128^3: 558 and 549 ->
// 430 and 451 us (464 and 530 before its shorter multiply-add).  With the shock switch (bits read beside U, HLLC and HLL both
// compiled at every face), 203 x 91 x 61: 176 -> 148 us a step, 24^3 61 -> 39.
#pragma once

#include <type_traits>

#include "stage_kernel.cuh"

namespace gh {

// The march loops take two rows an iteration in FP32, so that half of the
// register ring's moves go (256^3: stages 1 and 2 508 and 502 -> 493 and 490
// us; three rows: 505 and 506).  The double-word body is too large for that.
template <class T>
constexpr int march_unroll() { return sizeof(T) == 4 ? 2 : 1; }
constexpr int STRIP_OWN = 28;  // columns a warp owns

__device__ __forceinline__ float lane_up(float x) { return __shfl_up_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ float lane_down(float x) { return __shfl_down_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ dw lane_up(dw x) { return dw(lane_up(x.hi), lane_up(x.lo)); }
__device__ __forceinline__ dw lane_down(dw x) { return dw(lane_down(x.hi), lane_down(x.lo)); }

// A lane's share of the conserved totals: its column sums and the FP64 product of
// the other axes' widths they are to be multiplied by.
template <int NV>
struct Shares {
  dw c[NV];
  double area = 0.0;
  __device__ __forceinline__ Shares() {
#pragma unroll
    for (int v = 0; v < NV; ++v) c[v] = dw(0.0f, 0.0f);
  }
};
__device__ __forceinline__ dw pair_of(const ColumnSum<float>& t) {
  dw c;
  fast_two_sum(t.hi, t.lo, c.hi, c.lo);
  return c;
}
__device__ __forceinline__ dw pair_of(const ColumnSum<dw>& t) { return t.s; }

// x 2^k exactly: on the integer pipe unless x is zero, not finite or subnormal,
// or the result leaves the normal range
__device__ __forceinline__ double times_pow2(double x, int k) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  if (ex > 0 && ex < 2047 && ex + k > 0 && ex + k < 2047) return __longlong_as_double(b + ((long long)k << 52));
  return scalbn(x, k);
}

// Brings the warp's largest area, and the largest column sum of each variable,
// to [1, 2) by powers of two; scale[v] is what the sum of variable v is then to
// be multiplied by.
template <int NV>
__device__ __forceinline__ void scale_shares(Shares<NV>& t, int (&scale)[NV]) {
  const long long ab = __double_as_longlong(t.area);  // areas are positive
  const int ea = (int)(ab >> 52);
  const int ea_max = (int)__reduce_max_sync(0xffffffffu, (unsigned)ea), up = 1023 - ea_max;
  t.area = ea > 0 && ea + up > 0 ? __longlong_as_double(ab + ((long long)up << 52)) : 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(t.c[v].hi) & 0x7fffffffu) >> 23;
    const int e = (int)min(max(m, 1u), 253u);
    const float f = __uint_as_float((unsigned)(254 - e) << 23);  // 2^(127 - e)
    t.c[v] = dw(mul_rn(t.c[v].hi, f), mul_rn(t.c[v].lo, f));
    scale[v] = e - 127 - up;
  }
}

// Sums of the NV shares over the warp into red[0 .. NV - 1], in double word on
// the FP32 pipes (as FP64 additions this tail took 2-5 us of a stage on a mesh of
// 0.2 to 1 million cells).  Where areas or column sums are so large or small that
// a share or its low word could leave FP32's range (an area above 2^128 gave NaN,
// a share below 2^-102 lost its low word), all are scaled first and the scales
// return with the FP64 result (a step of 256 x 768 takes 0.5% longer for it, of
// 1024^2 0.3%; scaled always 0.8% and 0.5%).
// The area enters as three floats: the pair alone would leave 2^-49 of it out.
// Halving the first four variables with the lanes takes six additions instead of
// twenty.
template <int NV>
__device__ __forceinline__ void warp_totals(Shares<NV> t, double* red) {
  static_assert(NV == 4 || NV == 5, "2D or 3D");
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, q = lane & 8;
  int scale[NV];
  unsigned most = 0, least = 0xffffffffu;  // |column sums|; least: bits - 1, so that zeros are left out
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    scale[v] = 0;
    const unsigned m = __float_as_uint(t.c[v].hi) & 0x7fffffffu;
    most = max(most, m);
    least = min(least, m - 1u);
  }
  // column sums in 2^-46 .. 2^60 or 0, areas in 2^-30 .. 2^30 or 0
  const unsigned ea = (unsigned)(__double_as_longlong(t.area) >> 52);
  const bool usual = most < (127u + 60u) << 23 && least >= (127u - 46u) << 23 && (ea - (1023u - 30u) < 60u || ea == 0u);
  if (!__all_sync(0xffffffffu, usual)) scale_shares<NV>(t, scale);
  const float a1 = (float)t.area;
  const double r1 = t.area - (double)a1;
  const float a2 = (float)r1, a3 = (float)(r1 - (double)a2);
  dw s[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const dw r = t.c[v] * dw(a1, a2);
    fast_two_sum(r.hi, fma_rn(t.c[v].hi, a3, r.lo), s[v].hi, s[v].lo);
  }
  auto across = [](dw x, int o) {
    return dw(__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o));
  };
  // lanes 0..15 keep variables 0, 1; lanes 16..31 keep 2, 3
  const dw a = (h ? s[2] : s[0]) + across(h ? s[0] : s[2], 16);
  const dw b = (h ? s[3] : s[1]) + across(h ? s[1] : s[3], 16);
  dw r = (q ? b : a) + across(q ? a : b, 8);
  for (int o = 4; o > 0; o >>= 1) r += across(r, o);
  const int k = h ? (q ? scale[3] : scale[2]) : (q ? scale[1] : scale[0]);
  if ((lane & 7) == 0) red[lane >> 3] = k ? times_pow2((double)r, k) : (double)r;  // lane 8 v holds variable v
  if constexpr (NV == 5) {
    dw x = s[4];
    for (int o = 16; o > 0; o >>= 1) x += across(x, o);
    if (lane == 0) red[4] = scale[4] ? times_pow2((double)x, scale[4]) : (double)x;
  }
}

// Loads of the state and of K in the marches.  WIDE: 64-bit cell offsets, for
// meshes of more than 2^30 cells.
// FP32: the loads are not ordered against the march's own stores (nothing that a
// march reads is written by it), so that a row's can be issued before the last
// row's stores; held() makes the address depend on a point after chain_wait(), which
// keeps them behind the predecessor's writes.  With plain loads a step of 1024^2
// takes 1687 us for 32 instead of 1668.  Double word has no registers left for the
// pointers (128^3, 6 steps: 5824 us with them) and takes plain loads (5627).
template <class T, bool WIDE>
struct CellAccess {
  using Off = typename std::conditional<WIDE, size_t, unsigned>::type;
  static __device__ __forceinline__ const T* held(const T* p) { return p; }
  static __device__ __forceinline__ T at(const T* p, Off c) { return p[c]; }
};
template <bool WIDE>
struct CellAccess<float, WIDE> {
  using Off = typename std::conditional<WIDE, size_t, unsigned>::type;
  static __device__ __forceinline__ const float* held(const float* p) {
    asm volatile("" : "+l"(p) : : "memory");
    return p;
  }
  static __device__ __forceinline__ float at(const float* p, Off c) {
    float x;
    asm("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(__cvta_generic_to_global(p + c)));
    return x;
  }
};

// The march-axis step shared by the strips (along y) and ZMarch (along z):
// limited slope and lower face value of the cell above from W of three
// neighbours and the scaled difference dlo across the face below it, which
// moves on to the face above (a cell's upper scaled difference and its upper
// neighbour's lower one are the same number).
template <int NV, class T>
__device__ __forceinline__ void march_slope(const T (&wm)[NV], const T (&wc)[NV], const T (&wp)[NV], const Geo<T>& g,
                                            T (&dlo)[NV], T (&s)[NV], T (&wr)[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const T dhi = mul_rn(sub_rn(wp[v], wc[v]), g.tipc);
    s[v] = minmod3(dlo[v], mul_rn(sub_rn(wp[v], wm[v]), g.ipm), dhi);
    wr[v] = face_lo(s[v], g.h, wc[v]);
    dlo[v] = dhi;
  }
}

template <int NDIM, class T, int SOLVER, int STAGE, bool WIDE>
struct StripKernel {
  using Base = StageKernel<NDIM, T, SOLVER, STAGE, 32, 1, false>;
  using Acc = CellAccess<T, WIDE>;
  using Off = typename Acc::Off;
  static constexpr int NV = NDIM + 2;
  static constexpr bool SW = Base::SW;  // per-face HLLC/HLL choice from shock bits

  // minus the x part of the flux divergence of the lanes' cells of one row
  // (valid on the owned lanes), from W of the row
  static __device__ __forceinline__ void x_part(const StageArgs<T>& A, const T (&w)[NV], const Geo<T>& g, T iwx,
                                                unsigned fl, T (&d)[NV]) {
    T wl[NV], wr[NV], f[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T hi;
      face_pair(limited_slope(lane_up(w[v]), w[v], lane_down(w[v]), g), g.h, w[v], wr[v], hi);
      wl[v] = lane_up(hi);
    }
    if constexpr (SW) fl |= __shfl_up_sync(0xffffffffu, fl, 1);
    Base::template flux<0>(A, wl, wr, fl, f);  // the face below each column
#pragma unroll
    for (int v = 0; v < NV; ++v) d[v] = mul_rn(sub_rn(f[v], lane_down(f[v])), iwx);
  }

  // Strip of columns x0 .. x0 + 27, rows m0 .. m1 - 1 (1D: the one row; 3D: of
  // plane k, and only minus the x and y parts of the divergence go to A.out).
  // Accumulates the lane's CFL speed and, with totals, its share of them
  // (stage 1), and the non-physical flag.  The whole warp calls it.
  static __device__ __forceinline__ void strip(const StageArgs<T>& A, int x0, int m0, int m1, int k, T& speed_out,
                                               Shares<NV>& tot, bool& bad) {
    const int lane = threadIdx.x & 31;
    const T* const un = Acc::held(A.un);
    const T* const k1 = STAGE == 2 ? Acc::held(A.k1) : nullptr;
    const int nx = A.n[0], ny = NDIM >= 2 ? A.n[1] : 1;
    const size_t vs = NDIM == 3 ? (size_t)nx * ny * A.n[2] : (size_t)nx * ny;
    const T dt = STAGE == 2 ? (T)(*A.dt) : T(0);
    const int col = x0 + lane - 2;
    const bool own = lane >= 2 && lane < 2 + STRIP_OWN && col < nx;
    bool fa;
    Off off = (Off)bc_map(col, nx, A.bc_lo[0], A.bc_hi[0], fa);
    if constexpr (NDIM == 3) off += (Off)k * ((Off)nx * (Off)ny);
    const Geo<T> gx = Base::geo(A, 0, col);
    const T iwx = A.iw[0][min(col, nx + 1) + 2];
    ColumnSum<T> tcol[NV];
    T speed_max = T(0);

    // state of the cell at offset c (stage 2: U^n + dt K), x mirrored
    auto load = [&](Off c, T (&u)[NV]) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        u[v] = Acc::at(un + v * vs, c);
        if (STAGE == 2) u[v] = fma_rn(dt, Acc::at(k1 + v * vs, c), u[v]);
      }
    };
    // Epilogue of the own cell at offset c: L = minus the divergence, source,
    // output, and in stage 1 the CFL speed.
    auto finish = [&](Off c, T (&L)[NV], const T (&w)[NV], T iwm) {
      if constexpr (NDIM == 3) {
        if (own) {
#pragma unroll
          for (int v = 0; v < NV; ++v) A.out[v * vs + c] = L[v];
        }
        return;
      }
      if (A.has_source) Base::add_source(A, w, L);
      bad |= own && Base::nonphysical(w, A.gm1);
      if (STAGE == 1) {
        const T cs = sound_speed(A.gamma, mul_rn(A.gm1, w[NV - 1]), w[0]);
        T s = mul_rn(add_rn(fabs(w[1]), cs), iwx);
        if constexpr (NDIM == 2) s = fmax(s, mul_rn(add_rn(fabs(w[NDIM]), cs), iwm));
        speed_max = fmax(speed_max, s);
        if (own) {
#pragma unroll
          for (int v = 0; v < NV; ++v) A.out[v * vs + c] = L[v];
        }
      } else {
        const T hdt = half_of(dt);
        T r[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v)
          r[v] = fma_rn(hdt, add_rn(Acc::at(k1 + v * vs, c), L[v]), Acc::at(un + v * vs, c));
        if (own) {
#pragma unroll
          for (int v = 0; v < NV; ++v) A.out[v * vs + c] = r[v];
        }
      }
    };

    if constexpr (NDIM == 1) {
      T u[NV], w[NV], L[NV];
      load(off, u);
      if (fa) u[1] = -u[1];
      recover<NDIM>(u, w);
      x_part(A, w, gx, iwx, 0u, L);
      finish(off, L, w, T(0));
    } else {
      // W of row m (boundary-mapped); with totals also the row's share of the
      // column sums when it is one of the strip's own
      // (AHEAD: m >= 0, so that only the upper end needs the boundary rule)
      auto row = [&](int m, T (&u)[NV], unsigned& fl, auto ahead) {
        bool fm = false;
        int sm = m;
        if (!decltype(ahead)::value || m >= ny) sm = bc_map(m, ny, A.bc_lo[1], A.bc_hi[1], fm);
        load(off + (Off)sm * (Off)nx, u);
        if constexpr (SW) fl = A.flags[off + (Off)sm * (Off)nx];
        if (NDIM == 2 && STAGE == 1 && A.want_totals && m >= m0 && m < m1) {
          const T hi = A.wdh[1][m], lo = A.wdl[1][m];
#pragma unroll
          for (int v = 0; v < NV; ++v) tcol[v].add_product(u[v], hi, lo);
        }
        if (fa) u[1] = -u[1];
        if (fm) u[2] = -u[2];
      };
      // At the top of iteration m: wk = W(m), wk1 = W(m + 1), dlo = the scaled
      // difference across face m + 1/2, hi = the upper face value of cell m,
      // flo = the flux through face m - 1/2.
      T wk[NV], wk1[NV], w2[NV], dlo[NV], hi[NV], flo[NV], u[NV], s[NV], wr[NV];
      unsigned fk = 0, fk1 = 0, fk2 = 0;  // shock bits of rows m, m + 1, m + 2
      row(m0 - 2, u, fk, std::false_type());
      recover<NDIM>(u, wk);
      row(m0 - 1, u, fk, std::false_type());
      recover<NDIM>(u, wk1);
      row(m0, u, fk1, std::false_type());
      recover<NDIM>(u, w2);
      {
        const T t = Base::geo(A, 1, m0 - 2).tipc;
#pragma unroll
        for (int v = 0; v < NV; ++v) dlo[v] = mul_rn(sub_rn(wk1[v], wk[v]), t);
        const Geo<T> g = Base::geo(A, 1, m0 - 1);
        march_slope<NV, T>(wk, wk1, w2, g, dlo, s, wr);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          hi[v] = face_hi(s[v], g.h, wk1[v]);
          wk[v] = wk1[v];
          wk1[v] = w2[v];
        }
      }
      row(m0 + 1, u, fk2, std::false_type());
      recover<NDIM>(u, w2);
      {
        const Geo<T> g = Base::geo(A, 1, m0);
        march_slope<NV, T>(wk, wk1, w2, g, dlo, s, wr);
        Base::template flux<1>(A, hi, wr, fk | fk1, flo);
        fk = fk1;
        fk1 = fk2;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          hi[v] = face_hi(s[v], g.h, wk1[v]);
          wk[v] = wk1[v];
          wk1[v] = w2[v];
        }
      }
#pragma unroll march_unroll<T>()
      for (int m = m0; m < m1; ++m) {
        T L[NV], fhi[NV];
        row(m + 2, u, fk2, std::true_type());  // lands during the x part
        x_part(A, wk, gx, iwx, fk, L);
        recover<NDIM>(u, w2);
        const Geo<T> g = A.geo[1][m + 3];  // of row m + 1
        const T iwm = A.iw[1][m + 2];
        march_slope<NV, T>(wk, wk1, w2, g, dlo, s, wr);
        // face m + 1/2 between the upper value of m and the lower of m + 1
        Base::template flux<1>(A, hi, wr, fk | fk1, fhi);
        fk = fk1;
        fk1 = fk2;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          L[v] = fma_rn(sub_rn(flo[v], fhi[v]), iwm, L[v]);
          flo[v] = fhi[v];
        }
        finish(off + (Off)m * (Off)nx, L, wk, iwm);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          hi[v] = face_hi(s[v], g.h, wk1[v]);
          wk[v] = wk1[v];
          wk1[v] = w2[v];
        }
      }
    }
    if (NDIM < 3 && STAGE == 1 && own) {
      if (NDIM == 2 && A.want_totals) {
#pragma unroll
        for (int v = 0; v < NV; ++v) tot.c[v] = pair_of(tcol[v]);
        tot.area = A.wd[0][col];
      }
      speed_out = fmax(speed_out, speed_max);
    }
  }
};

// Fixed-order reduction of the warps' speeds and totals into CTA blk's partials.
template <int NV, int NW, class T>
__device__ __forceinline__ void write_warp_partials(const StageArgs<T>& A, size_t blk, int warp, T speed,
                                                    const Shares<NV>& tot, double (&red)[NW][NV + 1]) {
  double s;
  if constexpr (std::is_same<T, float>::value) s = (double)warp_max(speed);
  else s = warp_max((double)speed);
  if ((threadIdx.x & 31) == 0) red[warp][0] = s;
  if (A.want_totals) warp_totals<NV>(tot, &red[warp][1]);
  else if ((threadIdx.x & 31) < NV) red[warp][1 + (threadIdx.x & 31)] = 0.0;
  __syncthreads();
  const int t = threadIdx.x;
  if (t <= NV) {
    double acc = red[0][t];
    for (int w = 1; w < NW; ++w) acc = t == 0 ? fmax(acc, red[w][0]) : acc + red[w][t];
    if (t == 0) A.part_speed[blk] = acc;
    else A.part_tot[blk * NV + (t - 1)] = acc;
  }
}

// Registers: FP32 2D 64 (32 warps per SM), 3D 80 (24 warps); double word 128
// (16 warps).
template <class T, int NDIM>
constexpr int strip_warps() { return sizeof(T) == 8 ? 16 : NDIM == 3 ? 24 : 32; }

// 2D single mesh: CTA (x, chunk) of NW warps, each its own strip.
template <class T, int SOLVER, int STAGE, int NW, bool WIDE>
__global__ void __launch_bounds__(32 * NW, (strip_warps<T, 2>() / NW)) hydro_strip_kernel(const StageArgs<T> A) {
  using K = StripKernel<2, T, SOLVER, STAGE, WIDE>;
  constexpr int NV = 4;
  __shared__ double red[NW][NV + 1];
  chain_wait();
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int x0 = (blockIdx.x * NW + warp) * STRIP_OWN;
  const int m0 = blockIdx.z * A.kchunk, m1 = min(A.n[1], m0 + A.kchunk);
  T speed = T(0);
  Shares<NV> tot;
  bool bad = false;
  if (x0 < A.n[0]) K::strip(A, x0, m0, m1, 0, speed, tot, bad);
  if (bad) atomicOr(A.status, STATUS_NONPHYS);
  if (STAGE == 1)
    write_warp_partials<NV, NW>(A, (size_t)blockIdx.z * gridDim.x + blockIdx.x, warp, speed, tot, red);
}

// 3D, x and y parts: one warp per (strip, plane, chunk of ychunk rows); strips
// and planes are numbered along grid x, chunks along grid y.
template <class T, int SOLVER, int STAGE, int NW, bool WIDE>
__global__ void __launch_bounds__(32 * NW, (strip_warps<T, 3>() / NW))
    hydro_strip_xy_kernel(const StageArgs<T> A, int strips, int ychunk) {
  using K = StripKernel<3, T, SOLVER, STAGE, WIDE>;
  chain_wait();
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int id = blockIdx.x * NW + warp;
  const int k = id / strips;
  if (k >= A.n[2]) return;
  const int x0 = (id - k * strips) * STRIP_OWN;
  const int m0 = blockIdx.y * ychunk, m1 = min(A.n[1], m0 + ychunk);
  T speed = T(0);
  Shares<5> tot;
  bool bad = false;
  K::strip(A, x0, m0, m1, k, speed, tot, bad);
}

// 3D, z part and epilogue: one thread per (x, y) column and chunk of planes.
//
// ASYNC (FP32, planes of a multiple of 4 cells): every warp keeps its own ring
// of SLOTS planes in shared memory, filled ahead of the march by 16-byte
// cp.async copies (a lane moves a quarter of a row of a quarter of the arrays:
// 3 or 4 copies a plane for U, K and the strips' L), so that a plane's loads
// have 3 or 4 planes of arithmetic to land in, and the plane's second use (U and
// K of the stage combine) reads shared memory again.  Only __syncwarp separates
// filling from reading.
template <class T, int SOLVER, int STAGE, bool WIDE, bool ASYNC>
struct ZMarch {
  static_assert(!ASYNC || (std::is_same<T, float>::value && !WIDE), "the ring moves FP32 rows");
  using Base = StageKernel<3, T, SOLVER, STAGE, 32, 1, false>;
  using Acc = CellAccess<T, WIDE>;
  using Off = typename Acc::Off;
  static constexpr int NV = 5;
  static constexpr int NARR = STAGE == 1 ? 10 : 15;        // U, (K,) L
  static constexpr int SLOTS = STAGE == 1 ? 7 : 6;
  static constexpr int COPIES = (NARR * 8 + 31) / 32;      // 16-byte copies a lane and plane
  struct Ring {
    float a[SLOTS][NARR][32];
  };
  static constexpr size_t SMEM = ASYNC ? 4 * sizeof(Ring) : 0;  // four warps a CTA

  static __device__ __forceinline__ void march(const StageArgs<T>& A, Ring* ring, unsigned j, int m0, int m1,
                                               T& speed_max, Shares<NV>& tot, bool& bad) {
    const int lane = threadIdx.x & 31;
    const T* const un = Acc::held(A.un);
    const T* const k1 = STAGE == 2 ? Acc::held(A.k1) : nullptr;
    const int nx = A.n[0], ny = A.n[1], nz = A.n[2];
    const unsigned plane = (unsigned)nx * (unsigned)ny;
    const size_t vs = (size_t)plane * nz;
    const bool own = j < plane;
    const unsigned jc = own ? j : plane - 1;
    const int x = (int)(jc % (unsigned)nx), y = (int)(jc / (unsigned)nx);
    const T dt = STAGE == 2 ? (T)(*A.dt) : T(0);
    const T iwx = A.iw[0][x + 2], iwy = A.iw[1][y + 2];
    ColumnSum<T> tcol[NV];

    // ring: source (array, quarter row) and destination of the lane's copies
    const char* src[ASYNC ? COPIES : 1];
    unsigned dst = 0;
    bool quarter = false;  // the lane's quarter rows lie inside the mesh
    if constexpr (ASYNC) {
      const unsigned j0 = j - lane;
      quarter = j0 + 4u * (lane & 7) < plane;
      dst = (unsigned)__cvta_generic_to_shared(&ring->a[0][0][0]) + 16u * lane;
#pragma unroll
      for (int i = 0; i < COPIES; ++i) {
        const int idx = i * 32 + lane, arr = idx >> 3;
        // lanes past the plane repeat its last four columns of U and K (L: left as it
        // is); nothing of theirs leaves the march
        const unsigned col = min(j0 + 4u * (lane & 7), plane - 4u);
        const T* base = arr < 5 ? A.un + arr * vs
                        : STAGE == 2 && arr < 10 ? A.k1 + (arr - 5) * vs
                                                 : A.out + (size_t)min(arr - (NARR - 5), 4) * vs;
        src[i] = reinterpret_cast<const char*>(base + col);
      }
    }
    // Fill slot `slot` with plane m (boundary-mapped; L only for the chunk's own
    // planes); planes past the march leave an empty group.
    auto fill = [&](int m, int slot) {
      if constexpr (ASYNC) {
        if (m < m1 + 2) {
          bool fm;
          int sm = m;
          if (m < 0 || m >= nz) sm = bc_map(m, nz, A.bc_lo[2], A.bc_hi[2], fm);
          const size_t off = (size_t)sm * plane * sizeof(T);
          const bool inner = m >= m0 && m < m1 && quarter;
#pragma unroll
          for (int i = 0; i < COPIES; ++i) {
            const int arr = (i * 32 + lane) >> 3;
            if (arr < NARR - 5 || (inner && arr < NARR))
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + slot * (unsigned)sizeof(ring->a[0]) +
                                                                            i * 512u),
                           "l"(src[i] + off)
                           : "memory");
          }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    };
    auto row = [&](int m, int slot, T (&u)[NV], unsigned& fl, auto ahead) {
      bool fm = false;
      int sm = m;
      if (!decltype(ahead)::value || m >= nz) sm = bc_map(m, nz, A.bc_lo[2], A.bc_hi[2], fm);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        if constexpr (ASYNC) {
          u[v] = ring->a[slot][v][lane];
          if (STAGE == 2) u[v] = fma_rn(dt, ring->a[slot][5 + v][lane], u[v]);
        } else {
          const Off c = (Off)sm * (Off)plane + (Off)jc;
          u[v] = Acc::at(un + v * vs, c);
          if (STAGE == 2) u[v] = fma_rn(dt, Acc::at(k1 + v * vs, c), u[v]);
        }
      }
      if constexpr (Base::SW) fl = A.flags[(Off)sm * (Off)plane + (Off)jc];
      if (STAGE == 1 && A.want_totals && m >= m0 && m < m1) {
        const T hi = A.wdh[2][m], lo = A.wdl[2][m];
#pragma unroll
        for (int v = 0; v < NV; ++v) tcol[v].add_product(u[v], hi, lo);
      }
      if (fm) u[3] = -u[3];
    };
    T wk[NV], wk1[NV], w2[NV], dlo[NV], hi[NV], flo[NV], u[NV], s[NV], wr[NV];
    unsigned fk = 0, fk1 = 0, fk2 = 0;  // shock bits of planes m, m + 1, m + 2
    // the first SLOTS planes; the four below are consumed before the march
    if constexpr (ASYNC) {
      for (int i = 0; i < SLOTS; ++i) fill(m0 - 2 + i, i);
      asm volatile("cp.async.wait_group %0;" ::"n"(SLOTS - 4) : "memory");
      __syncwarp();
    }
    row(m0 - 2, 0, u, fk, std::false_type());
    recover<3>(u, wk);
    row(m0 - 1, 1, u, fk, std::false_type());
    recover<3>(u, wk1);
    row(m0, 2, u, fk1, std::false_type());
    recover<3>(u, w2);
    {
      const T t = Base::geo(A, 2, m0 - 2).tipc;
#pragma unroll
      for (int v = 0; v < NV; ++v) dlo[v] = mul_rn(sub_rn(wk1[v], wk[v]), t);
      const Geo<T> g = Base::geo(A, 2, m0 - 1);
      march_slope<NV, T>(wk, wk1, w2, g, dlo, s, wr);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        hi[v] = face_hi(s[v], g.h, wk1[v]);
        wk[v] = wk1[v];
        wk1[v] = w2[v];
      }
    }
    row(m0 + 1, 3, u, fk2, std::false_type());
    recover<3>(u, w2);
    {
      const Geo<T> g = Base::geo(A, 2, m0);
      march_slope<NV, T>(wk, wk1, w2, g, dlo, s, wr);
      Base::template flux<2>(A, hi, wr, fk | fk1, flo);
      fk = fk1;
      fk1 = fk2;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        hi[v] = face_hi(s[v], g.h, wk1[v]);
        wk[v] = wk1[v];
        wk1[v] = w2[v];
      }
    }
    if constexpr (ASYNC) {
      __syncwarp();
      fill(m0 - 2 + SLOTS, 0);
    }
    // slots of planes m - 1 (free in iteration m), m, m + 1 and m + 2
    int slf = 1, sl0 = 2, sl1 = 3, sl2 = 4;
#pragma unroll march_unroll<T>()
    for (int m = m0; m < m1; ++m) {
      const Off c = (Off)m * (Off)plane + (Off)jc;
      T L[NV], fhi[NV];
      if constexpr (ASYNC) {
        asm volatile("cp.async.wait_group %0;" ::"n"(SLOTS - 4) : "memory");  // plane m + 2 has landed
        __syncwarp();  // for every lane, and every lane is done with plane m - 1
        fill(m - 1 + SLOTS, slf);
      }
      row(m + 2, sl2, u, fk2, std::true_type());
#pragma unroll
      for (int v = 0; v < NV; ++v) {  // the strips' x and y parts
        if constexpr (ASYNC) L[v] = ring->a[sl0][NARR - 5 + v][lane];
        else L[v] = own ? A.out[v * vs + c] : T(0);
      }
      recover<3>(u, w2);
      const Geo<T> g = A.geo[2][m + 3];  // of plane m + 1
      const T iwm = A.iw[2][m + 2];
      march_slope<NV, T>(wk, wk1, w2, g, dlo, s, wr);
      Base::template flux<2>(A, hi, wr, fk | fk1, fhi);
      fk = fk1;
      fk1 = fk2;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        L[v] = fma_rn(sub_rn(flo[v], fhi[v]), iwm, L[v]);
        flo[v] = fhi[v];
      }
      if (A.has_source) Base::add_source(A, wk, L);
      bad |= own && Base::nonphysical(wk, A.gm1);
      if (STAGE == 1) {
        const T cs = sound_speed(A.gamma, mul_rn(A.gm1, wk[4]), wk[0]);
        T sp = mul_rn(add_rn(fabs(wk[1]), cs), iwx);
        sp = fmax(sp, mul_rn(add_rn(fabs(wk[2]), cs), iwy));
        sp = fmax(sp, mul_rn(add_rn(fabs(wk[3]), cs), iwm));
        speed_max = fmax(speed_max, sp);
      } else {
        const T hdt = half_of(dt);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          T u0, k;
          if constexpr (ASYNC) {
            u0 = ring->a[sl0][v][lane];
            k = ring->a[sl0][5 + v][lane];
          } else {
            u0 = Acc::at(un + v * vs, c);
            k = Acc::at(k1 + v * vs, c);
          }
          L[v] = fma_rn(hdt, add_rn(k, L[v]), u0);
        }
      }
      if (own) {
#pragma unroll
        for (int v = 0; v < NV; ++v) A.out[v * vs + c] = L[v];
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        hi[v] = face_hi(s[v], g.h, wk1[v]);
        wk[v] = wk1[v];
        wk1[v] = w2[v];
      }
      slf = sl0;
      sl0 = sl1;
      sl1 = sl2;
      sl2 = sl2 + 1 == SLOTS ? 0 : sl2 + 1;
    }
    if constexpr (ASYNC) asm volatile("cp.async.wait_group 0;" ::: "memory");
    // a lane past the plane has W of one cell and the widths of another
    if (!own) speed_max = T(0);
    if (STAGE == 1 && A.want_totals && own) {
#pragma unroll
      for (int v = 0; v < NV; ++v) tot.c[v] = pair_of(tcol[v]);
      tot.area = A.wd[0][x] * A.wd[1][y];
    }
  }
};

template <class T, int SOLVER, int STAGE, bool WIDE, bool ASYNC>
__global__ void __launch_bounds__(128, (sizeof(T) == 8 ? 4 : ASYNC && STAGE == 2 ? 4 : 6))
    hydro_march_z_kernel(const StageArgs<T> A) {
  using K = ZMarch<T, SOLVER, STAGE, WIDE, ASYNC>;
  constexpr int NV = 5, NW = 4;
  extern __shared__ __align__(16) unsigned char smem_z[];
  __shared__ double red[NW][NV + 1];
  chain_wait();
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  // chunks in descending order: the strips' last planes are still in L2
  const int chunk = gridDim.z - 1 - blockIdx.z;
  const int m0 = chunk * A.kchunk, m1 = min(A.n[2], m0 + A.kchunk);
  T speed = T(0);
  Shares<NV> tot;
  bool bad = false;
  K::march(A, reinterpret_cast<typename K::Ring*>(smem_z) + warp, blockIdx.x * 128u + threadIdx.x, m0, m1, speed, tot,
           bad);
  if (bad) atomicOr(A.status, STATUS_NONPHYS);
  if (STAGE == 1) write_warp_partials<NV, NW>(A, (size_t)chunk * gridDim.x + blockIdx.x, warp, speed, tot, red);
}

}  // namespace gh
