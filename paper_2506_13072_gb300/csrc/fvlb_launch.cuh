// fvlb_launch.cuh -- host-side launch logic, templated on the lattice; each
// lattice's translation unit instantiates it once.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "fvlb_internal.h"
#include "fvlb_kernels.cuh"

namespace fvlb {

// An integer from the environment.
inline int tune_int(const char* name, int dflt) {
  const char* v = std::getenv(name);
  return v && *v ? std::atoi(v) : dflt;
}

template <class R>
Phys<R> make_phys(const StepDesc& d) {
  Phys<R> p;
  p.tau_f = R(d.tau_f);
  p.inv_tau_f = R(1.0 / d.tau_f);
  p.inv_tau_h = R(1.0 / d.tau_h);
  p.kh = R(1.0 - 0.5 / d.tau_h);
  p.kf = R(1.0 - 0.5 / d.tau_f);
  p.eta_over_lam = R(d.eta_p / d.lambda);
  p.inv_lam = R(1.0 / d.lambda);
  p.four_roll = d.four_roll;
  p.Fv[0] = R(d.Fv[0]);
  p.Fv[1] = R(d.Fv[1]);
  p.Fv[2] = R(d.Fv[2]);
  p.amp = R(d.amp);
  const R* t = static_cast<const R*>(d.tables);
  p.sx = t;
  p.cxs = t ? t + d.nx : nullptr;
  p.sy = t ? t + 2 * d.nx : nullptr;
  p.cys = t ? t + 2 * d.nx + d.ny : nullptr;
  p.first = d.first;
  p.step = (uint32_t)d.step;
  p.lam = R(d.lambda);
  p.mlp = d.mlp;
  p.cl_tol2 = float(d.cl_tol * d.cl_tol);
  p.cl_count = d.cl_count;
  p.model = d.model;
  p.mpar = R(d.mpar);
  p.fdiv = nullptr;
  p.err = d.err;
  return p;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (the
// library does not link the driver API); null when it is unavailable
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    cudaGetLastError();
  });
  return fn;
}

// One tiled map without swizzle or interleave; dims[0] runs over the nodes
// of a population array, strides are the byte strides of dims 1 ...
inline bool encode_map(CUtensorMap* m, CUtensorMapDataType t, int rank, const void* base,
                       const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
  const auto enc = tensor_map_encoder();
  if (!enc) return false;
  const cuuint32_t es[3] = {1, 1, 1};
  return enc(m, t, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
             CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tensor maps of a fused launch whose stage holds BX nodes of every
// array (StageMaps in fvlb_kernels.cuh); `on` = 0 (each lane copies its own
// node) when a buffer is not 16-byte aligned, an encoding fails, or
// FVLB_STAGE_TMA=0.
template <class L, class S>
StageMaps stage_maps(const void* f, const void* h, const void* chi, long long pitch, int BX) {
  StageMaps m;
  std::memset(&m, 0, sizeof m);
  constexpr int Q = L::Q, C = L::C, D = L::D;
  constexpr cuuint64_t es = sizeof(S), xs = sizeof(typename Store<S>::X);
  if (tune_int("FVLB_STAGE_TMA", 1) == 0) return m;
  auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (!aligned(f) || !aligned(h) || !aligned(chi)) return m;
  const CUtensorMapDataType tf = CU_TENSOR_MAP_DATA_TYPE_FLOAT32, td = CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
  const CUtensorMapDataType t = es == 8 ? td : (es == 4 ? tf : CU_TENSOR_MAP_DATA_TYPE_UINT16);
  const cuuint64_t P = (cuuint64_t)pitch;
  const cuuint32_t bx = (cuuint32_t)BX;
  bool ok = true;
  auto rows = [&](CUtensorMap* mp, CUtensorMapDataType ty, cuuint64_t sz, const void* base, int n) {
    const cuuint64_t dims[2] = {P, (cuuint64_t)n}, st[1] = {P * sz};
    const cuuint32_t box[2] = {bx, (cuuint32_t)n};
    ok = ok && encode_map(mp, ty, 2, base, dims, st, box);
  };
  rows(&m.f, t, es, f, Q);
  rows(&m.x, xs == 8 ? td : tf, xs, chi, C);
  if constexpr (Store<S>::V2) {
    const char* h0 = static_cast<const char*>(h) + es * C * Q * P;
    const char* U = static_cast<const char*>(f) + es * Q * P;
    if (!aligned(h0) || !aligned(U)) return m;
    rows(&m.e0, tf, 4, h0, C);
    rows(&m.u, tf, 4, U, D);
    // (the i = 0 slots are unused: directions 1 .. Q - 1 of every component)
    const cuuint64_t dims[3] = {P, (cuuint64_t)Q, (cuuint64_t)C}, st[2] = {P * es, Q * P * es};
    const cuuint32_t box[3] = {bx, (cuuint32_t)(Q - 1), (cuuint32_t)C};
    ok = ok && encode_map(&m.h, t, 3, h, dims, st, box);
  } else {
    rows(&m.h, t, es, h, C * Q);
  }
  m.on = ok ? 1 : 0;
  return m;
}

inline int grid_stride_blocks(long long N, int threads, int sms) {
  const long long want = (N + threads - 1) / threads;
  const long long cap = (long long)std::max(sms, 1) * 16;
  return (int)std::max<long long>(1, std::min(want, cap));
}

// Let kernel `kern` take `bytes` of dynamic shared memory on the current
// device: set once per device and kernel (before its first launch, so also
// before a stream capture that contains one).
template <class K>
cudaError_t allow_dynamic_smem(K* kern, size_t bytes) {
  static std::mutex mu;
  static std::vector<std::pair<const void*, int>> done;  // (kernel, device) set
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const std::pair<const void*, int> key{reinterpret_cast<const void*>(kern), dev};
  std::lock_guard<std::mutex> lock(mu);
  for (const auto& d : done)
    if (d == key) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) done.push_back(key);
  return e;
}

// Tile shapes of the fused step: 32 GX nodes along x, KG threads per node,
// MINB resident blocks per SM (registers and stage buffers are budgeted for
// them).  Measured on GB300, MLUPS (the 256^3 / 2048^2 periodic flows; in
// brackets the kernel with one thread per stress component):
//   D3Q19 FP32 2,2,2: 5795 (5244); KG 1: 5480, KG 3: 5680
//   D3Q19 FP16 2,2,3: 7110 (4803); KG 1: 5080, KG 3: 6240, MINB 2: 7130 (128^3
//     6540 against 7120)
//   D3Q19 FP64 (96^3) 1,2,2: 577 (343); KG 1: 366, KG 3: 550
//   D2Q9 FP32 4,1,2: 20270 (18102); KG 3: 18223, GX 2: 19012
//   D2Q9 FP16 4,1,4: 28200 (14835); MINB 3: 27000, 5: 23800, GX 2: 23520
//   D2Q9 FP64 (512^2) 2,1,3: 2110 (948); KG 3: 1463, GX 4: 1968
// With stochastic rounding 2,2,3 and 4,1,4 as well (us a step, the kernel with
// one thread per stress component and now: 128^3 FP16 625 / 510, BF16
// 556 / 424; 1024^2 FP16 94 / 57, BF16 90 / 52).
// Spills that these budgets cost (bytes stored / loaded per thread): D3Q19
// 16-bit 24 / 24 to 28 / 28 at 80 registers, 24 / 24 to 44 / 44 with
// stochastic rounding (MINB 2 leaves 128 registers and is slower at 128^3, see
// above); D2Q9 FP64 up to 92 / 80 at 128 registers, 160 / 104 in the original
// scheme; D2Q9 16-bit with stochastic rounding 8 / 8.
// SMALL: one warp's nodes per tile, for grids that leave the chip idle
// otherwise (the larger KG spreads FP64 over the four quarters of an SM; 32^3
// FP32 1,2,4 6.9 us a step, 1,2,3 8.2, the wide tile 11.7; 48^3 FP16 1,2,5
// 23.2, 1,2,4 25.8).
template <class L, class S, bool SMALL>
struct StepShape {
  static constexpr int B = sizeof(S);
  static constexpr int GX = L::D == 3 ? (SMALL || B == 8 ? 1 : 2) : (SMALL ? 1 : (B == 8 ? 2 : 4));
  static constexpr int KG = L::D == 3 ? 2 : (SMALL && B == 8 ? 3 : 1);
  static constexpr int MINB = L::D == 3 ? (B == 8 ? 2 : (SMALL ? (B == 2 ? 5 : 4) : (B == 2 ? 3 : 2)))
                                        : (SMALL ? (B == 8 ? 3 : 4) : (B == 2 ? 4 : (B == 8 ? 3 : 2)));
};

// Planes per block along the march axis, from a model of the launch, fitted
// on GB300 to chunks of 1 to 24 planes of 16 grids.  With k blocks on an SM a
// plane takes slope k + lat (in units of one block's share of a busy SM): more
// blocks share its throughput, one alone leaves part of it idle.
//  - One wave (every block resident): the fullest SM's blocks and a prologue
//    of 1.5 planes.
//  - More: all planes and the prologues' work (`pro` planes a block) at the
//    full SM's rate, and a share of one block's time for the uneven end.
// us per step, this rule and the one before it (the fewest planes that still
// fill the last wave, 2.5 planes a prologue), both with the present kernels:
// 64^2 FP64 6.1 / 10.2, 8x128 FP32 2.2 / 2.6, 100^3 FP32 208 / 216, 161x97x65
// 226 / 245, 64^3 FP64 467 / 501, 128^3 FP16 297 / 298.
struct ChunkModel {
  double slope, lat, pro, tail;
};
template <class L, class S, bool SMALL>
constexpr ChunkModel chunk_model() {
  constexpr bool f64 = L::D == 3 && sizeof(S) == 8;
  return {SMALL ? 0.6 : 1.0, L::D == 3 && !f64 ? 2.0 : 1.0,
          f64 ? 0.3 : (L::D == 3 && sizeof(S) == 2 ? 1.2 : 0.6),
          f64 ? 0.8 : (sizeof(S) == 2 ? 0.25 : 0.5)};
}
inline int pick_chunk(long long tiles, int nm, int sms, int minb, const ChunkModel& cm,
                      double* cost_out = nullptr) {
  constexpr double kPrologue = 1.5;
  constexpr int kMost = 32;
  const int least = (nm + 65534) / 65535;   // the chunks are the grid's z extent
  int best = least;
  double cost = 1e300;
  for (int c = least; c <= std::max(least, std::min(nm, kMost)); ++c) {
    const long long blocks = tiles * ((nm + c - 1) / c);
    const double full = cm.slope * minb + cm.lat;
    double t;
    if (blocks <= (long long)sms * minb)
      t = (c + kPrologue) * (cm.slope * (double)((blocks + sms - 1) / sms) + cm.lat);
    else
      t = ((double)tiles * nm + (double)blocks * cm.pro) / sms * full / minb +
          cm.tail * (c + kPrologue) * full;
    if (t <= cost) {
      cost = t;
      best = c;
    }
  }
  if (cost_out) *cost_out = cost;
  return best;
}

// Launch with a programmatic edge to the previous kernel of the stream: the
// blocks may start while it drains, and wait for its end themselves (pdl_wait).
template <class... P, class... A>
cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                       const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <class L, class S, bool SMALL, int GX, int KG, int MINB, bool WALLS, bool PADDED, bool CL,
          bool ORIG>
cudaError_t launch_kernel(const StepDesc& d, const Grid& g, const Phys<RT<S>>& ph,
                          const Bufs<S>& b) {
  using Sh = FusedShape<L, S, GX, KG, CL>;
  using Cfg = TileCfg<L, S, GX, KG, MINB, PADDED, CL>;
  auto kern = k_step_fused<L, S, GX, KG, MINB, WALLS, PADDED, CL, ORIG>;
  const int bx = (d.nx + Sh::TXS - 1) / Sh::TXS;
  const int by = L::D == 3 ? d.ny : 1;
  const int nm = L::D == 3 ? g.nz : d.ny;
  static_assert(sizeof(StageMaps) <= sizeof(StepPlan::maps[0]), "room for the tensor maps");
  StepPlan once;
  StepPlan& pl = d.plan ? *d.plan : once;
  if (pl.kern != reinterpret_cast<const void*>(kern)) {
    const cudaError_t e = allow_dynamic_smem(kern, sizeof(typename Cfg::Smem));
    if (e != cudaSuccess) return e;
    pl.mchunk = pick_chunk((long long)bx * by, nm, std::max(d.sms, 1), blocks_of(MINB),
                           chunk_model<L, S, SMALL>());
    pl.mapped[0] = pl.mapped[1] = -1;
    pl.kern = reinterpret_cast<const void*>(kern);
  }
  StageMaps& tm = *reinterpret_cast<StageMaps*>(pl.maps[d.parity & 1]);
  if (pl.mapped[d.parity & 1] < 0) {
    tm = stage_maps<L, S>(b.f_in, b.h_in, b.chi, d.pitch, Cfg::BX);
    pl.mapped[d.parity & 1] = tm.on;
  }
  return launch_pdl(kern, dim3(bx, by, (nm + pl.mchunk - 1) / pl.mchunk), Sh::NT,
                    sizeof(typename Cfg::Smem), d.stream, g, ph, b, pl.mchunk, tm);
}

// The kernel variant of a grid: row starts on 16-byte boundaries need no
// padded stage; padded tiles serve walled and periodic grids alike.
template <class L, class S, bool SMALL, int GX, int KG, int MINB, bool CL, bool ORIG>
cudaError_t launch_fused(const StepDesc& d, const Grid& g, const Phys<RT<S>>& ph,
                         const Bufs<S>& b) {
  if (d.nx % (16 / (int)sizeof(S)))
    return launch_kernel<L, S, SMALL, GX, KG, MINB, true, true, CL, ORIG>(d, g, ph, b);
  if (d.walls) return launch_kernel<L, S, SMALL, GX, KG, MINB, true, false, CL, ORIG>(d, g, ph, b);
  return launch_kernel<L, S, SMALL, GX, KG, MINB, false, false, CL, ORIG>(d, g, ph, b);
}

// The fused step.  ORIG: the original scheme's step (div tau_p from ph.fdiv in
// the body force, f^B off).
template <class L, class S, bool ORIG>
cudaError_t fused_step(const StepDesc& d, const Grid& g, const Phys<RT<S>>& ph,
                       const Bufs<S>& b) {
  using Big = StepShape<L, S, false>;
  using Small = StepShape<L, S, true>;
  if constexpr (std::is_same<S, float>::value && !ORIG) {
    if (d.mlp) return launch_fused<L, S, false, Big::GX, (L::D == 3 ? 2 : 1), 2, true, false>(d, g, ph, b);
  }
  if constexpr (Big::GX != Small::GX) {
    const int by = L::D == 3 ? d.ny : 1, nm = L::D == 3 ? g.nz : d.ny;
    int small = d.plan ? d.plan->small : -1;
    if (small < 0) {
      auto tiles = [&](int gx) { return (long long)((d.nx + 32 * gx - 1) / (32 * gx)) * by; };
      double cs, cb;
      const int sms = std::max(d.sms, 1);
      pick_chunk(tiles(Small::GX), nm, sms, Small::MINB, chunk_model<L, S, true>(), &cs);
      pick_chunk(tiles(Big::GX), nm, sms, Big::MINB, chunk_model<L, S, false>(), &cb);
      small = cs < cb;
      if (d.plan) d.plan->small = small;
    }
    if (small)
      return launch_fused<L, S, true, Small::GX, Small::KG, Small::MINB, false, ORIG>(d, g, ph, b);
  }
  // D2Q9 FP32 with more than one wave of 32-row chunks (1.25 M nodes): a fourth
  // stage buffer.  us a step with four and three, constant force: 512^2 11.2
  // and 10.9, 1024^2 53.3 and 53.1, 1120^2 68.2 and 69.6, 1280^2 83.7 and 86.2,
  // 1536^2 118.7 and 121.9, 1733x1337 121.5 and 122.9, 2048^2 201.8 and 210.0
  // (a fifth costs 1 % there; with 16-bit storage the fourth costs 5 %)
  if constexpr (L::D == 2 && std::is_same<S, float>::value && !ORIG) {
    if ((long long)d.nx * d.ny > (long long)d.sms * Big::MINB * 32 * 32 * Big::GX)
      return launch_fused<L, S, false, Big::GX, Big::KG, 400 + Big::MINB, false, ORIG>(d, g, ph, b);
  }
  return launch_fused<L, S, false, Big::GX, Big::KG, Big::MINB, false, ORIG>(d, g, ph, b);
}

template <class L, class S>
cudaError_t step_impl(const StepDesc& d) {
  using R = RT<S>;
  using X = typename Store<S>::X;
  Grid g{d.nx, d.ny, L::D == 3 ? d.nz : 1, d.walls, d.pitch};
  Phys<R> ph = make_phys<R>(d);
  Bufs<S> b{static_cast<const S*>(d.f_in), static_cast<S*>(d.f_out),
            static_cast<const S*>(d.h_in), static_cast<S*>(d.h_out),
            static_cast<X*>(d.chi)};
  if (d.scheme == 1) {
    // the original scheme: the polymer stress of every node, then either its
    // divergence per node and the fused step with it as part of the body
    // force and f^B off (three launches), or the split velocity and
    // collision kernels, which take the divergence themselves
    const int threads = 128;
    const int blocks = grid_stride_blocks(d.N, threads, d.sms);
    R* taup = static_cast<R*>(d.taup);
    k_taup<L, S><<<blocks, threads, 0, d.stream>>>(g, ph, b.h_in, taup, d.N);
    if constexpr (sizeof(S) >= 4) {  // fused form for FP32 and FP64 storage
      if (d.variant == 0 && !d.mlp) {
        R* fdiv = static_cast<R*>(d.fdiv);
        k_fdiv<L, S><<<blocks, threads, 0, d.stream>>>(g, taup, fdiv, d.N);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ph.fdiv = fdiv;
        return fused_step<L, S, true>(d, g, ph, b);
      }
    }
    R* ubuf = static_cast<R*>(d.ubuf);
    k_velocity<L, S, true><<<blocks, threads, 0, d.stream>>>(g, ph, b.f_in, ubuf, taup, d.N);
    k_collide_split<L, S, true, true><<<blocks, threads, 0, d.stream>>>(g, ph, b, ubuf, taup, d.N);
    return cudaGetLastError();
  }
  if (d.variant == 0) {
    return fused_step<L, S, false>(d, g, ph, b);
  } else {
    const int threads = 128;
    const int blocks = grid_stride_blocks(d.N, threads, d.sms);
    R* ubuf = static_cast<R*>(d.ubuf);
    k_velocity<L, S><<<blocks, threads, 0, d.stream>>>(g, ph, b.f_in, ubuf, nullptr, d.N);
    k_collide_split<L, S, true><<<blocks, threads, 0, d.stream>>>(g, ph, b, ubuf, nullptr, d.N);
  }
  return cudaGetLastError();
}

template <class L, class S>
cudaError_t init_impl(const InitDesc& d) {
  Grid g{d.nx, d.ny, L::D == 3 ? d.nz : 1, 0, d.pitch};
  const int threads = 256;
  const int blocks = grid_stride_blocks(d.N, threads, d.sms);
  k_init<L, S><<<blocks, threads, 0, d.stream>>>(
      g, static_cast<S*>(d.f), static_cast<S*>(d.h),
      static_cast<typename Store<S>::X*>(d.chi), d.u0, d.p0, d.A0, d.N);
  return cudaGetLastError();
}

template <class L, class S, bool ORIG>
cudaError_t launch_fields(const StepDesc& d, const Grid& g, const Phys<RT<S>>& ph, int which,
                          double* out, const RT<S>* taup) {
  const int threads = 128;
  const int blocks = grid_stride_blocks(d.N, threads, d.sms);
  const S* f = static_cast<const S*>(d.f_in);
  const S* h = static_cast<const S*>(d.h_in);
  switch (which) {
    case 0: k_fields<L, S, 0, ORIG><<<blocks, threads, 0, d.stream>>>(g, ph, f, h, out, taup, d.N); break;
    case 1: k_fields<L, S, 1, ORIG><<<blocks, threads, 0, d.stream>>>(g, ph, f, h, out, taup, d.N); break;
    case 2: k_fields<L, S, 2><<<blocks, threads, 0, d.stream>>>(g, ph, f, h, out, taup, d.N); break;
    default: k_fields<L, S, 3><<<blocks, threads, 0, d.stream>>>(g, ph, f, h, out, taup, d.N); break;
  }
  return cudaGetLastError();
}

template <class L, class S>
cudaError_t fields_impl(const StepDesc& d, int which, double* out) {
  using R = RT<S>;
  Grid g{d.nx, d.ny, L::D == 3 ? d.nz : 1, d.walls, d.pitch};
  Phys<R> ph = make_phys<R>(d);
  if (d.scheme == 1) {
    R* taup = static_cast<R*>(d.taup);
    k_taup<L, S><<<grid_stride_blocks(d.N, 256, d.sms), 256, 0, d.stream>>>(
        g, ph, static_cast<const S*>(d.h_in), taup, d.N);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_fields<L, S, true>(d, g, ph, which, out, taup);
  }
  return launch_fields<L, S, false>(d, g, ph, which, out, nullptr);
}

template <class L, class S>
cudaError_t reduce_impl(const StepDesc& d, double* part, double* out) {
  using R = RT<S>;
  Grid g{d.nx, d.ny, L::D == 3 ? d.nz : 1, d.walls, d.pitch};
  Phys<R> ph = make_phys<R>(d);
  const int nparts = reduce_parts(d.N);
  const S* f = static_cast<const S*>(d.f_in);
  const S* h = static_cast<const S*>(d.h_in);
  if (d.scheme == 1) {
    R* taup = static_cast<R*>(d.taup);
    k_taup<L, S><<<grid_stride_blocks(d.N, 256, d.sms), 256, 0, d.stream>>>(g, ph, h, taup, d.N);
    k_reduce_partial<L, S, true><<<nparts, kReduceThreads, 0, d.stream>>>(g, ph, f, h, part, d.N,
                                                                          taup);
  } else {
    k_reduce_partial<L, S><<<nparts, kReduceThreads, 0, d.stream>>>(g, ph, f, h, part, d.N);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return reduce_finalize(part, nparts, d.N, out, d.stream);
}

template <class L, class S>
cudaError_t conf_impl(const StepDesc& d, double* part, double* out) {
  Grid g{d.nx, d.ny, L::D == 3 ? d.nz : 1, d.walls, d.pitch};
  const int nparts = reduce_parts(d.N);
  k_conf_partial<L, S><<<nparts, kReduceThreads, 0, d.stream>>>(
      g, static_cast<const S*>(d.h_in), part, d.N);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_conf_final<<<1, kReduceThreads, 0, d.stream>>>(part, nparts, out);
  return cudaGetLastError();
}

template <class L, class S>
cudaError_t repair_impl(const StepDesc& d, double eps, unsigned long long* count) {
  Grid g{d.nx, d.ny, L::D == 3 ? d.nz : 1, d.walls, d.pitch};
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), d.stream);
  if (e != cudaSuccess) return e;
  k_repair<L, S><<<grid_stride_blocks(d.N, kReduceThreads, d.sms), kReduceThreads, 0, d.stream>>>(
      g, static_cast<S*>(const_cast<void*>(d.h_in)), eps, count, d.N);
  return cudaGetLastError();
}

// step_impl is instantiated per (lattice, storage) in its own translation
// unit (k_step_<lattice>_<storage>.cu) so that the library builds in parallel.
#define FVLB_EXTERN_STEP(L)                                                   \
  extern template cudaError_t step_impl<L, double>(const StepDesc&);        \
  extern template cudaError_t step_impl<L, float>(const StepDesc&);         \
  extern template cudaError_t step_impl<L, __half>(const StepDesc&);        \
  extern template cudaError_t step_impl<L, __nv_bfloat16>(const StepDesc&); \
  extern template cudaError_t step_impl<L, half_sr>(const StepDesc&);       \
  extern template cudaError_t step_impl<L, bf16_sr>(const StepDesc&);

#define FVLB_DISPATCH(storage, CALL)                              \
  switch (storage) {                                              \
    case kFP64: return CALL(double);                              \
    case kFP32: return CALL(float);                               \
    case kFP16Dev: return CALL(__half);                           \
    case kBF16Dev: return CALL(__nv_bfloat16);                    \
    case kFP16DevSR: return CALL(half_sr);                        \
    case kBF16DevSR: return CALL(bf16_sr);                        \
    default: return cudaErrorInvalidValue;                        \
  }

}  // namespace fvlb
