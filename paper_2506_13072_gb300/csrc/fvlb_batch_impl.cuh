// fvlb_batch_impl.cuh -- templated host launchers of the batched step, one
// translation unit per storage type (k_batch_<storage>.cu).
#pragma once

#include "fvlb_batch.h"
#include "fvlb_launch.cuh"

namespace fvlb {

// Threads per node and resident blocks per SM (registers and stage buffers
// are budgeted for them).  FP16, 96 grids, us per step: 12 / GX blocks 198,
// 8 / GX 205, 16 / GX 199, 20 / GX 212; FP32: 8 / GX 216, 4 / GX 263,
// 12 / GX 219.
template <class S, int GX>
struct BatchMinB {
  static constexpr int KG = sizeof(S) == 8 ? 3 : 1;
  static constexpr int value = (sizeof(S) == 8 ? 4 : (sizeof(S) == 2 ? 12 : 8)) / GX;
};
template <class S, int GX>
using BatchCfg = TileCfg<D2Q9, S, GX, BatchMinB<S, GX>::KG, BatchMinB<S, GX>::value, true, false>;

template <class S, int GX>
cudaError_t batch_launch_gx(const BatchLaunch& d) {
  constexpr int NT = FusedShape<D2Q9, S, GX, BatchMinB<S, GX>::KG>::NT;
  constexpr size_t dyn = sizeof(typename BatchCfg<S, GX>::Smem);
  using X = typename Store<S>::X;
  auto kern = k_step_batched<D2Q9, S, GX, BatchMinB<S, GX>::KG, BatchMinB<S, GX>::value>;
  const cudaError_t e = allow_dynamic_smem(kern, dyn);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(d.ntiles), NT, dyn, d.stream, static_cast<const BatchInst<S>*>(d.inst),
                    static_cast<const BatchTile*>(d.tiles), static_cast<S*>(d.fA),
                    static_cast<S*>(d.fB), static_cast<S*>(d.hA), static_cast<S*>(d.hB),
                    static_cast<X*>(d.chi), d.parity, d.first, d.tstep, d.mchunk,
                    static_cast<const StageMaps*>(d.maps));
}

template <class S>
cudaError_t batch_step_impl(const BatchLaunch& d) {
  switch (d.gx) {
    case 1: return batch_launch_gx<S, 1>(d);
    case 2: return batch_launch_gx<S, 2>(d);
    case 4: return batch_launch_gx<S, 4>(d);
    default: return cudaErrorInvalidValue;
  }
}

template <class S>
void batch_maps_impl(StageMaps* m, int gx, const void* f, const void* h, const void* chi,
                     long long pitch) {
  const int BX = gx == 1 ? BatchCfg<S, 1>::BX : (gx == 2 ? BatchCfg<S, 2>::BX : BatchCfg<S, 4>::BX);
  *m = stage_maps<D2Q9, S>(f, h, chi, pitch, BX);
}

template <class S>
void batch_inst_fill_impl(void* dst, int nx, int ny, int walls, long long pitch, double tau_f,
                          double tau_h, double eta_p, double lambda, int force_kind,
                          const double* F0, double omega, const void* tables, long long f_off,
                          long long h_off, long long chi_off, unsigned* err) {
  using R = RT<S>;
  BatchInst<S> I{};
  I.g = Grid{nx, ny, 1, walls, pitch};
  StepDesc sd{};
  sd.nx = nx;
  sd.ny = ny;
  sd.nz = 1;
  sd.tau_f = tau_f;
  sd.tau_h = tau_h;
  sd.eta_p = eta_p;
  sd.lambda = lambda;
  sd.four_roll = force_kind == 2;
  sd.amp = F0[0];
  sd.tables = tables;
  sd.err = err;
  for (int a = 0; a < 3; ++a) sd.Fv[a] = force_kind == 1 ? F0[a] : 0.0;
  I.ph = make_phys<R>(sd);
  I.f_off = f_off;
  I.h_off = h_off;
  I.chi_off = chi_off;
  I.cosine = force_kind == 3;
  for (int a = 0; a < 3; ++a) I.F0[a] = F0[a];
  I.omega = omega;
  *static_cast<BatchInst<S>*>(dst) = I;
}

}  // namespace fvlb
