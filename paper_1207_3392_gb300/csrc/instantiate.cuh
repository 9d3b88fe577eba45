// instantiate.cuh -- helpers that register explicit instantiations of the stage
// kernel in the variant table (one translation unit per dimensionality and
// precision so that they compile in parallel).
#pragma once

#include "registry.h"
#include "stage_kernel.cuh"
#include "stage_strip.cuh"

namespace gh {

template <int NDIM, class T, int SOLVER, int STAGE, int TX, int TY, int MINB, bool PRE>
inline void fill_variant(StageVariant* out) {
  using K = StageKernel<NDIM, T, SOLVER, STAGE, TX, TY, PRE>;
  out->fn = reinterpret_cast<const void*>(&hydro_stage_kernel<NDIM, T, SOLVER, STAGE, TX, TY, MINB, PRE>);
  out->smem = sizeof(typename K::Smem);
  out->tx = K::OWN;  // columns of cells per tile (TX - 1 in 1D/2D)
  out->ty = TY;
  out->threads = TX * TY;
  out->chain = NDIM == 1;
}

// PRE: in-plane face states formed once per cell (see stage_kernel.cuh).
template <int NDIM, class T, int TX, int TY, int MINB = 1, bool PRE = (NDIM == 3)>
inline bool pick_variant(int solver, int stage, StageVariant* out) {
  if (solver == SOLVER_HLL && stage == 1) fill_variant<NDIM, T, SOLVER_HLL, 1, TX, TY, MINB, PRE>(out);
  else if (solver == SOLVER_HLL && stage == 2) fill_variant<NDIM, T, SOLVER_HLL, 2, TX, TY, MINB, PRE>(out);
  else if (solver == SOLVER_HLLC && stage == 1) fill_variant<NDIM, T, SOLVER_HLLC, 1, TX, TY, MINB, PRE>(out);
  else if (solver == SOLVER_HLLC && stage == 2) fill_variant<NDIM, T, SOLVER_HLLC, 2, TX, TY, MINB, PRE>(out);
  else return false;
  return true;
}

// HLLC with the shock switch (compiled for one tile per dimensionality).
template <int NDIM, class T, int TX, int TY, int MINB = 1, bool PRE = (NDIM == 3)>
inline bool pick_switch(int stage, StageVariant* out) {
  if (stage == 1) fill_variant<NDIM, T, SOLVER_HLLC_SW, 1, TX, TY, MINB, PRE>(out);
  else if (stage == 2) fill_variant<NDIM, T, SOLVER_HLLC_SW, 2, TX, TY, MINB, PRE>(out);
  else return false;
  return true;
}

// 2D on independent warps (stage_strip.cuh), NW strips per CTA.
template <class T, int SOLVER, int STAGE, int NW>
inline void fill_strip(StageVariant* out) {
  out->fn = reinterpret_cast<const void*>(&hydro_strip_kernel<T, SOLVER, STAGE, NW, false>);
  out->fn_wide = reinterpret_cast<const void*>(&hydro_strip_kernel<T, SOLVER, STAGE, NW, true>);
  out->smem = 0;
  out->tx = STRIP_OWN * NW;
  out->ty = 1;
  out->threads = 32 * NW;
  out->strips = 1;
  out->chain = 1;
}
template <class T, int NW>
inline bool pick_strip_switch(int stage, StageVariant* out) {
  if (stage == 1) fill_strip<T, SOLVER_HLLC_SW, 1, NW>(out);
  else if (stage == 2) fill_strip<T, SOLVER_HLLC_SW, 2, NW>(out);
  else return false;
  return true;
}
template <class T, int NW>
inline bool pick_strip(int solver, int stage, StageVariant* out) {
  if (solver == SOLVER_HLL && stage == 1) fill_strip<T, SOLVER_HLL, 1, NW>(out);
  else if (solver == SOLVER_HLL && stage == 2) fill_strip<T, SOLVER_HLL, 2, NW>(out);
  else if (solver == SOLVER_HLLC && stage == 1) fill_strip<T, SOLVER_HLLC, 1, NW>(out);
  else if (solver == SOLVER_HLLC && stage == 2) fill_strip<T, SOLVER_HLLC, 2, NW>(out);
  else return false;
  return true;
}

// 3D on independent warps: the strips' launch (x and y parts), then ZMarch's.
template <class T, int SOLVER, int STAGE>
inline void fill_split(StageVariant* out) {
  constexpr int NW = 4;
  out->xy_fn = reinterpret_cast<const void*>(&hydro_strip_xy_kernel<T, SOLVER, STAGE, NW, false>);
  out->xy_fn_wide = reinterpret_cast<const void*>(&hydro_strip_xy_kernel<T, SOLVER, STAGE, NW, true>);
  out->xy_warps = NW;
  constexpr bool RING = std::is_same<T, float>::value;
  out->fn = reinterpret_cast<const void*>(&hydro_march_z_kernel<T, SOLVER, STAGE, false, RING>);
  out->smem = ZMarch<T, SOLVER, STAGE, false, RING>::SMEM;
  if (RING) out->fn_odd = reinterpret_cast<const void*>(&hydro_march_z_kernel<T, SOLVER, STAGE, false, false>);
  out->fn_wide = reinterpret_cast<const void*>(&hydro_march_z_kernel<T, SOLVER, STAGE, true, false>);
  out->tx = 128;
  out->ty = 1;
  out->threads = 128;
  out->chain = 1;
}
template <class T>
inline bool pick_split_switch(int stage, StageVariant* out) {
  if (stage == 1) fill_split<T, SOLVER_HLLC_SW, 1>(out);
  else if (stage == 2) fill_split<T, SOLVER_HLLC_SW, 2>(out);
  else return false;
  return true;
}
template <class T>
inline bool pick_split(int solver, int stage, StageVariant* out) {
  if (solver == SOLVER_HLL && stage == 1) fill_split<T, SOLVER_HLL, 1>(out);
  else if (solver == SOLVER_HLL && stage == 2) fill_split<T, SOLVER_HLL, 2>(out);
  else if (solver == SOLVER_HLLC && stage == 1) fill_split<T, SOLVER_HLLC, 1>(out);
  else if (solver == SOLVER_HLLC && stage == 2) fill_split<T, SOLVER_HLLC, 2>(out);
  else return false;
  return true;
}

}  // namespace gh
