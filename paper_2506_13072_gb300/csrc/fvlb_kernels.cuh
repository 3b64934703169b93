// fvlb_kernels.cuh -- CUDA kernels of one fluctuating-LB time step
// (arXiv 2506.13072, Sec. 2.2 flow LB with f^B and Guo forcing, Sec. 2.3
// conformation LB), plus initialisation, field extraction and the FP64
// diagnostics reduction.
//
// Data layout in HBM (structure of arrays, x fastest, each array padded to
// `pitch` elements):  f[Q][pitch], h[C][Q][pitch], chi[C][pitch].  The state
// is double-buffered (f and h read from one buffer, written to the other);
// chi is read and rewritten in place by its own site only.
//
// A step is "collide, then push": the site reads its own populations
// (coalesced, unshifted), collides, and writes population i to the
// neighbour x + c_i of the other buffer (or, through a halfway-bounce-back
// wall, to its own node in the opposite direction).  The velocity gradient
// in chi needs the same-step velocity of the 2 (2D) or 6 (3D) nearest
// neighbours, which with push streaming are one node away, so a one-node
// velocity halo suffices.
#pragma once

#include <cuda.h>   // CUtensorMap (the type only; maps are encoded on the host)

#include <type_traits>

#include "fvlb_lattice.cuh"
#include "fvlb_mlp.cuh"

namespace fvlb {

template <class S>
using RT = typename Store<S>::R;

// Bulk tensor copies (TMA) into shared memory, completed on an mbarrier.
// One thread of the block arms the barrier with the byte count of a buffer's
// copies and issues them; every warp that reads the buffer waits for the
// barrier's phase.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// make initialised barriers visible to the copy engine
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
  return t;
}
// Wait for the phase of parity `parity` to complete, for at most about 2 s;
// on time-out record bit 0 in *err (when given) and return false.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, unsigned* err) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_ns() - t0 > 2000000000ull) {
      if (err) atomicOr(err, 1u);
      return false;
    }
  }
  return true;
}
// order this thread's earlier shared-memory accesses before later accesses
// of the copy engine to the same memory
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];\n" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(c0), "r"(c1), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(c0), "r"(c1), "r"(c2),
      "r"(smem_addr(bar))
      : "memory");
}

// Programmatic dependent launch: let the next kernel of the stream start its
// blocks while this one drains, and wait until the previous one has finished
// and its writes are visible.  Without a programmatic edge both do nothing.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Tensor maps of one launch's staged arrays (the fused step's copies of a
// tile's row of nodes into its stage), encoded on the host; `on` = 0: the
// lanes copy their own nodes instead.  Dimension 0 is the node index within
// a population array (x fastest, `pitch` long) and a box of BX nodes is one
// tile row; the arrays must start on 16-byte boundaries, and so must the
// first node of a box (which the kernel rounds down where nx does not give it).
struct StageMaps {
  CUtensorMap h;    // h as [C Q][pitch]; box BX x C Q (16-bit forms: [C][Q][pitch], box BX x Q-1 x C)
  CUtensorMap f;    // f[Q][pitch]; box BX x Q
  CUtensorMap x;    // chi[C][pitch]; box BX x C
  CUtensorMap e0;   // 16-bit forms: FP32 rest stress populations h0[C][pitch]; box BX x C
  CUtensorMap u;    // 16-bit forms: FP32 velocities U[D][pitch]; box BX x D
  int on;
};

// Maps in global memory: order the host's writes of them before this
// block's copies through them.
__device__ __forceinline__ void fence_tensor_maps(const StageMaps* m) {
  const CUtensorMap* p[5] = {&m->h, &m->f, &m->x, &m->e0, &m->u};
#pragma unroll
  for (int q = 0; q < 5; ++q)
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;\n" ::"l"(
                     reinterpret_cast<unsigned long long>(p[q]))
                 : "memory");
}

// Make a pointer opaque to the compiler at this point of the program.  Used
// to stop the 114 population addresses of a D3Q19 site from being computed
// once and kept live (in registers) between the two reads of the stress
// populations, which would cap the number of resident warps.
template <class T>
__device__ __forceinline__ T* opaque(T* p) {
  asm volatile("" : "+l"(p));
  return p;
}

// load f_i(s) (16-bit forms: s_i / KF + e_i(U) with the node's stored U).
// BITS: 16-bit values by the builtin load of their bits.  (The headers' __ldg
// of the 16-bit types are inline assembly, which the compiler keeps in place:
// better or worse from kernel to kernel, see k_fields.)
template <class L, class S, bool BITS = false>
__device__ __forceinline__ void load_f(const S* __restrict__ f, long long pitch,
                                       long long s, RT<S> (&fv)[L::Q]) {
  using R = RT<S>;
  if constexpr (Store<S>::V2) {
    const float* U = f_ext<L>(f, pitch);
    R u[L::D];
#pragma unroll
    for (int a = 0; a < L::D; ++a) u[a] = U[a * pitch + s];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      R v;
      if constexpr (BITS)
        v = Store<S>::cvtb(__ldg(reinterpret_cast<const unsigned short*>(f + i * pitch + s)));
      else
        v = Store<S>::ld(f + i * pitch + s);
      fv[i] = v * R(1.0f / Store<S>::KF) + feq_u<L, R>(i, u);
    }
  } else {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) fv[i] = Store<S>::ld(f + i * pitch + s);
  }
}

// Stress populations are held as deviations from the rest equilibrium,
// h'_{k,i} = h_{k,i} - w_i delta_k (delta_k = 1 on diagonal components), in
// every storage precision: the conformation then enters as A - I = sum_i h'
// without the cancellation of summing h ~ w_i A and subtracting I.
// (16-bit forms: the rest population from its FP32 array)
template <class L, class S>
__device__ __forceinline__ RT<S> load_h(const S* __restrict__ h, long long pitch,
                                        long long s, int k, int i) {
  if constexpr (Store<S>::V2) {
    if (i == 0) return h_ext<L>(h, pitch)[k * pitch + s];
  }
  return Store<S>::ld(h + (long long)(k * L::Q + i) * pitch + s);
}

// second read of a stress population within one site update (served by L2);
// hs points at the site's first population
template <class L, class S>
__device__ __forceinline__ RT<S> reload_h(const S* hs, long long pitch, int k, int i) {
  return Store<S>::ld_l2(hs + (long long)(k * L::Q + i) * pitch);
}

template <class L, class S>
__device__ __forceinline__ void store_h(S* __restrict__ h, long long pitch,
                                        long long s, int k, int i, RT<S> v, uint32_t r) {
  Store<S>::st(h + (long long)(k * L::Q + i) * pitch + s, v, r);
}

template <class L>
__host__ __device__ constexpr bool diag(int k) {
  return L::ca(k) == L::cb(k);
}

// Streaming destination of population i leaving (x, y, z) (node s):
// periodic wrap, or halfway bounce-back to the same node, opposite direction.
template <class L>
__device__ __forceinline__ long long push_dest(const Grid& g, int i, int x, int y,
                                               int z, long long s, int& j) {
  int xd = x + L::cx(i), yd = y + L::cy(i), zd = z + L::cz(i);
  bool bb = false;
  if (L::cx(i) != 0 && (xd < 0 || xd >= g.nx)) {
    if (g.walls & 1) bb = true;
    else xd = xd < 0 ? xd + g.nx : xd - g.nx;
  }
  if (L::cy(i) != 0 && (yd < 0 || yd >= g.ny)) {
    if (g.walls & 2) bb = true;
    else yd = yd < 0 ? yd + g.ny : yd - g.ny;
  }
  if (L::D == 3 && L::cz(i) != 0 && (zd < 0 || zd >= g.nz)) {
    if (g.walls & 4) bb = true;
    else zd = zd < 0 ? zd + g.nz : zd - g.nz;
  }
  if (bb) {
    j = L::opp(i);
    return s;
  }
  j = i;
  return ((long long)zd * g.ny + yd) * g.nx + xd;
}

// p = c_s^2 / (1 - w_0) [sum_{i!=0} f_i + s_0(u) + tau_f F_0 + tau_f f^B_0]
// (Sec. 2.2, Appendix B) with F_0 = -3 w_0 (1 - 1/(2 tau_f)) F.u and
// s_0 = -1.5 w_0 |u|^2; returned as the pressure variable of p_part (p in
// FP64, p / (3 w_1) in FP32).
template <class L, class R>
__device__ __forceinline__ R pressure(const Phys<R>& ph, const R (&f)[L::Q],
                                      const R (&u)[L::D], const R F[3], R fB0) {
  R sum = R(0);
#pragma unroll
  for (int i = 1; i < L::Q; ++i) sum += f[i];
  R uu = R(0), Fu = R(0);
#pragma unroll
  for (int a = 0; a < L::D; ++a) {
    uu += u[a] * u[a];
    Fu += F[a] * u[a];
  }
  constexpr double w0 = L::w(0);
  const R s0 = R(-1.5 * w0) * uu;
  const R F0 = R(-3.0 * w0) * ph.kf * Fu;
  return p_part<L, R>(sum + s0 + ph.tau_f * F0 + ph.tau_f * fB0);
}

// ---------------------------------------------------------------------------
// Collide one site and push its populations.  u and gr (d_a u_b) are the
// site's velocity and velocity gradient of this step; f its populations.
// HOLD_H keeps all C*Q stress populations in registers (2D); otherwise the
// conformation is summed in a first pass and each component re-read for its
// collision (3D, where C*Q = 114).
// ORIG: the original scheme the paper compares with (Sec. 1, Tables 1-2):
// no fluctuation term f^B; the caller's F already holds the stress
// divergence, so it enters u, the pressure and the Guo term as a body force.
// ---------------------------------------------------------------------------
template <class L, class S, bool HOLD_H, bool ORIG = false>
__device__ __forceinline__ void collide_site(const Grid& g, const Phys<RT<S>>& ph,
                                             const Bufs<S>& b, long long s, int x,
                                             int y, int z, const RT<S> (&u)[L::D],
                                             const RT<S> (&gr)[L::D][L::D],
                                             const RT<S> (&f)[L::Q], const RT<S> F[3],
                                             const RT<S>* __restrict__ ubuf = nullptr) {
  using R = RT<S>;
  using X = typename Store<S>::X;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  const long long P = g.pitch;
  // stochastic-rounding stream of this site and step (unused otherwise)
  uint32_t rng = Store<S>::sr ? hash32((uint32_t)s * 0x9e3779b9u ^ hash32(ph.step)) : 0u;

  // --- conformation A = I + sum_i h' (Sec. 2.3) --------------------------
  R Ad[C];  // A - I
  R hv[HOLD_H ? C : 1][HOLD_H ? Q : 1];
#pragma unroll
  for (int k = 0; k < C; ++k) {
    // Q loads in flight per component: keeps the register footprint (and so
    // the number of resident warps) bounded when the populations are re-read
    // below instead of held.
    const S* hk = HOLD_H ? b.h_in + s : opaque(b.h_in + s);
    R a = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const R v = (Store<S>::V2 && i == 0) ? R(h_ext<L>(b.h_in, P)[k * P + s])
                                           : Store<S>::ld(hk + (long long)(k * Q + i) * P);
      if (HOLD_H) hv[HOLD_H ? k : 0][HOLD_H ? i : 0] = v;
      a += v;
    }
    Ad[k] = a;
  }
  // --- flow collision inputs (Sec. 2.2) ------------------------------------
  // f^B is linear in tau_p = (eta_p/lambda)(A - I): evaluate it on A - I with
  // the factor eta_p / (lambda tau_f) folded in.
  const R kB = ph.eta_over_lam * ph.inv_tau_f;
  R uu = R(0), Fu = R(0);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    uu += u[a] * u[a];
    Fu += F[a] * u[a];
  }
  const R fB0 = ORIG ? R(0) : fB_dir<L, R>(0, Ad, kB);
  const R p = pressure<L, R>(ph, f, u, F, fB0);

  // --- stress source (Sec. 2.3) ---------------------------------------------
  R src[C];
  {
    R A[C], chi[C];
#pragma unroll
    for (int k = 0; k < C; ++k) A[k] = Ad[k] + (diag<L>(k) ? R(1) : R(0));
    chi_tensor<L, R>(A, Ad, gr, ph, chi);
#pragma unroll
    for (int k = 0; k < C; ++k) {
      R old = R(b.chi[k * P + s]);
      if (ph.first) old = chi[k];
      b.chi[k * P + s] = X(chi[k]);
      // chi_i + 0.5 (chi_i^n - chi_i^{n-1}) = phi_i (1.5 chi - 0.5 chi_old)
      src[k] = R(1.5) * chi[k] - R(0.5) * old;
    }
  }

  // --- collide and push, one direction at a time ----------------------------
  // The destination of direction i is computed once and shared by f_i and
  // the C stress populations h_{k,i}.
  const S* hs = b.h_in + s;
  // 16-bit forms: the rest stress populations (stored last, in FP32, with
  // the rounding residuals of the component's other populations) and this
  // node's velocity for the flow populations it receives next step
  // The rest stress population keeps the node's populations summing to the
  // post-collision zeroth moment (as in the fused step): FP32 storage takes
  // it as that moment minus the other populations' sum; the 16-bit forms
  // take the rounding residuals less the rounded weights' excess
  constexpr bool RS = std::is_same<S, float>::value;
  constexpr double kWx = weight_sum_excess<L, R>();
  R h0post[Store<S>::V2 ? C : 1], hres[(Store<S>::V2 || RS) ? C : 1];
  if constexpr (RS) {
#pragma unroll
    for (int k = 0; k < C; ++k) hres[k] = R(0);
  }
  if constexpr (Store<S>::V2) {
#pragma unroll
    for (int k = 0; k < C; ++k) hres[k] = R(0);
    float* Uo = f_ext<L>(b.f_out, P);
#pragma unroll
    for (int a = 0; a < D; ++a) Uo[a * P + s] = float(u[a]);
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (!HOLD_H && i % 3 == 0) hs = opaque(hs);
    R cu = R(0), cF = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int c = cc<L>(i, a);
      if (c == 1) { cu += u[a]; cF += F[a]; }
      if (c == -1) { cu -= u[a]; cF -= F[a]; }
    }
    int j;
    const long long d = push_dest<L>(g, i, x, y, z, s, j);
    const R wi = R(L::w(i));

    // flow: f* = f - (f - f^eq)/tau_f + f^B + F_i (Sec. 2.2)
    const R lam_i = R(p_coef<L, R>(i));
    const R w3i = R(w3<L, R>(i));
    const R feq = lam_i * p + (w3i * cu + wi * (R(4.5) * cu * cu - R(1.5) * uu));
    const R Fi = ph.kf * (w3i * cF + wi * (R(9) * cF * cu - R(3) * Fu));
    const R fBi = ORIG ? R(0) : fB_dir<L, R>(i, Ad, kB);
    const R fpost = f[i] - (f[i] - feq) * ph.inv_tau_f + fBi + Fi;
    if constexpr (Store<S>::V2) {
      // deviation from e_j(u) of the receiving node (velocity of this step)
      R ud[D];
#pragma unroll
      for (int a = 0; a < D; ++a) ud[a] = ubuf[a * P + d];
      Store<S>::st(b.f_out + j * P + d, R(Store<S>::KF) * (fpost - feq_u<L, R>(j, ud)),
                   Store<S>::sr ? lcg_next(rng) : 0u);
    } else {
      Store<S>::st(b.f_out + j * P + d, fpost, Store<S>::sr ? lcg_next(rng) : 0u);
    }

    // stress: h* = h - (h - h^eq)/tau_h + phi_i src, phi_i = w_i [1 + (1 - 1/(2 tau_h)) c.u/c_s^2]
    const R phi = wi * (R(1) + ph.kh * R(3) * cu);
#pragma unroll
    for (int k = 0; k < C; ++k) {
      R hi;
      if (HOLD_H) hi = hv[HOLD_H ? k : 0][HOLD_H ? i : 0];
      else if (Store<S>::V2 && i == 0) hi = R(h_ext<L>(b.h_in, P)[k * P + s]);
      else hi = reload_h<L, S>(hs, P, k, i);
      // h^eq - w_i delta_k = w_i [(A - I)_k + A_k c_i.u / c_s^2]
      const R heq = wi * (Ad[k] + (Ad[k] + (diag<L>(k) ? R(1) : R(0))) * (R(3) * cu));
      const R post = hi - (hi - heq) * ph.inv_tau_h + phi * src[k];
      if constexpr (Store<S>::V2) {
        if (i == 0) {
          // less the weights' excess times the weight-proportional part
          h0post[k] = post - R(kWx) * (ph.inv_tau_h * Ad[k] + src[k]);
        } else {
          S* q = b.h_out + (long long)(k * Q + j) * P + d;
          hres[k] -= Store<S>::st_d(q, post, Store<S>::sr ? lcg_next(rng) : 0u);
        }
      } else if constexpr (RS) {
        if (i != 0) {
          hres[k] += post;
          store_h<L, S>(b.h_out, P, d, k, j, post, 0u);
        }
      } else {
        store_h<L, S>(b.h_out, P, d, k, j, post, Store<S>::sr ? lcg_next(rng) : 0u);
      }
    }
  }
  if constexpr (RS) {
#pragma unroll
    for (int k = 0; k < C; ++k) store_h<L, S>(b.h_out, P, s, k, 0, (Ad[k] + src[k]) - hres[k], 0u);
  }
  if constexpr (Store<S>::V2) {
    float* h0o = h_ext<L>(b.h_out, P);
#pragma unroll
    for (int k = 0; k < C; ++k) h0o[k * P + s] = float(h0post[k] + hres[k]);
  }
}

}  // namespace fvlb

#include "fvlb_fused.cuh"

namespace fvlb {

// ---------------------------------------------------------------------------
// Original scheme (Sec. 1, Tables 1-2): the polymer stress of every node in
// a working array tau_p[C][pitch], then its divergence by finite
// differences: central (periodic wrap), and next to a wall the one-sided
// second-order difference (-3 t0 + 4 t1 - t2) / 2 through the two nodes
// inside (sign mirrored at the upper wall), since no stress is known at the
// wall.  Needs 3 nodes across a walled axis.
// ---------------------------------------------------------------------------
template <class L, class S>
__global__ void k_taup(Grid g, Phys<RT<S>> ph, const S* __restrict__ h,
                       RT<S>* __restrict__ taup, long long N) {
  using R = RT<S>;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int k = 0; k < L::C; ++k) {
      R a = R(0);  // (A - I)_k from the deviations h'
#pragma unroll
      for (int i = 0; i < L::Q; ++i) a += load_h<L, S>(h, g.pitch, s, k, i);
      taup[k * g.pitch + s] = ph.eta_over_lam * a;
    }
  }
}

// dv_b = sum_a d_a tau_ab at node (x, y, z) = s
template <class L, class R>
__device__ __forceinline__ void div_taup(const Grid& g, const R* __restrict__ tp, int x, int y,
                                         int z, long long s, R (&dv)[3]) {
  const int p[3] = {x, y, z};
  const int n[3] = {g.nx, g.ny, g.nz};
  const long long st[3] = {1, g.nx, (long long)g.nx * g.ny};
  dv[0] = dv[1] = dv[2] = R(0);
#pragma unroll
  for (int a = 0; a < L::D; ++a) {
    if (n[a] == 1) continue;
    const bool wall = (g.walls >> a) & 1;
    const bool edge = wall && (p[a] == 0 || p[a] == n[a] - 1);
    const long long e = p[a] == 0 ? st[a] : -st[a];
    const long long sp = p[a] + 1 < n[a] ? s + st[a] : s - (long long)(n[a] - 1) * st[a];
    const long long sm = p[a] > 0 ? s - st[a] : s + (long long)(n[a] - 1) * st[a];
#pragma unroll
    for (int b = 0; b < L::D; ++b) {
      const R* t = tp + (long long)sym<L>(a, b) * g.pitch;
      R d;
      if (edge) {
        d = R(0.5) * (R(-3) * t[s] + R(4) * t[s + e] - t[s + 2 * e]);
        if (p[a] != 0) d = -d;
      } else {
        d = R(0.5) * (t[sp] - t[sm]);
      }
      dv[b] += d;
    }
  }
}

// The original scheme ahead of the fused step: div tau_p of every node into
// fdiv[a * pitch + s] (read by the fused step as part of the body force).
template <class L, class S>
__global__ void k_fdiv(Grid g, const RT<S>* __restrict__ taup, RT<S>* __restrict__ fdiv,
                       long long N) {
  using R = RT<S>;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(s % g.nx);
    const int y = (int)((s / g.nx) % g.ny);
    const int z = (int)(s / ((long long)g.nx * g.ny));
    R dv[3];
    div_taup<L, R>(g, taup, x, y, z, s, dv);
#pragma unroll
    for (int a = 0; a < L::D; ++a) fdiv[a * g.pitch + s] = dv[a];
  }
}

// ---------------------------------------------------------------------------
// Split step: velocity field to a device buffer, then collide-and-push with
// the gradient read from that buffer.  One thread per site.  ORIG: the
// original scheme, the stress divergence added to the body force.
// ---------------------------------------------------------------------------
template <class L, class S, bool ORIG = false>
__global__ void k_velocity(Grid g, Phys<RT<S>> ph, const S* __restrict__ f,
                           RT<S>* __restrict__ ubuf, const RT<S>* __restrict__ taup,
                           long long N) {
  using R = RT<S>;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(s % g.nx);
    const int y = (int)((s / g.nx) % g.ny);
    R fv[L::Q];
    load_f<L, S>(f, g.pitch, s, fv);
    R F[3];
    body_force<L, R>(ph, x, y, F);
    if constexpr (ORIG) {
      R dv[3];
      div_taup<L, R>(g, taup, x, y, (int)(s / ((long long)g.nx * g.ny)), s, dv);
      F[0] += dv[0];
      F[1] += dv[1];
      F[2] += dv[2];
    }
    R u[L::D];
    velocity<L, R>(fv, F, u);
#pragma unroll
    for (int a = 0; a < L::D; ++a) ubuf[a * g.pitch + s] = u[a];
  }
}

template <class L, class S, bool HOLD_H, bool ORIG = false>
__global__ void k_collide_split(Grid g, Phys<RT<S>> ph, Bufs<S> b,
                                const RT<S>* __restrict__ ubuf, const RT<S>* __restrict__ taup,
                                long long N) {
  using R = RT<S>;
  constexpr int D = L::D;
  const long long P = g.pitch;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(s % g.nx);
    const int y = (int)((s / g.nx) % g.ny);
    const int z = (int)(s / ((long long)g.nx * g.ny));
    const int p[3] = {x, y, z};
    const int n[3] = {g.nx, g.ny, g.nz};
    const long long stride[3] = {1, g.nx, (long long)g.nx * g.ny};
    R u[D], gr[D][D];
#pragma unroll
    for (int a = 0; a < D; ++a) u[a] = ubuf[a * P + s];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const bool wall = (g.walls >> a) & 1;
      const long long sp = p[a] + 1 < n[a] ? s + stride[a] : s - (long long)(n[a] - 1) * stride[a];
      const long long sm = p[a] > 0 ? s - stride[a] : s + (long long)(n[a] - 1) * stride[a];
#pragma unroll
      for (int bq = 0; bq < D; ++bq) {
        const R up = ubuf[bq * P + sp], um = ubuf[bq * P + sm];
        R d = R(0.5) * (up - um);
        if (wall && p[a] == 0) d = u[bq] + up * R(1.0 / 3.0);
        if (wall && p[a] == n[a] - 1) d = -(u[bq] + um * R(1.0 / 3.0));
        gr[a][bq] = d;
      }
    }
    R fv[L::Q];
    load_f<L, S>(b.f_in, P, s, fv);
    R F[3];
    body_force<L, R>(ph, x, y, F);
    if constexpr (ORIG) {
      R dv[3];
      div_taup<L, R>(g, taup, x, y, z, s, dv);
      F[0] += dv[0];
      F[1] += dv[1];
      F[2] += dv[2];
    }
    collide_site<L, S, HOLD_H, ORIG>(g, ph, b, s, x, y, z, u, gr, fv, F, ubuf);
  }
}

// ---------------------------------------------------------------------------
// Initial state: f = f^eq(p0, u0), h = w_i A0 (1 + c_i.u0 / c_s^2), chi = 0.
// u0 [N][D], p0 [N], A0 [N][C] in FP64 (each may be null: 0, 0, I).
// ---------------------------------------------------------------------------
template <class L, class S>
__global__ void k_init(Grid g, S* __restrict__ f, S* __restrict__ h,
                       typename Store<S>::X* __restrict__ chi,
                       const double* __restrict__ u0, const double* __restrict__ p0,
                       const double* __restrict__ A0, long long N) {
  using R = RT<S>;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  const long long P = g.pitch;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    R u[D], A[C];
    R uu = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
      u[a] = u0 ? R(u0[s * D + a]) : R(0);
      uu += u[a] * u[a];
    }
#pragma unroll
    for (int k = 0; k < C; ++k)
      A[k] = A0 ? R(A0[s * C + k]) : (L::ca(k) == L::cb(k) ? R(1) : R(0));
    const R p = p_part_of_p<L, R>(p0 ? R(p0[s]) : R(0));
    R hres[C];
#pragma unroll
    for (int k = 0; k < C; ++k) hres[k] = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      R cu = R(0);
#pragma unroll
      for (int a = 0; a < D; ++a) cu += R(cc<L>(i, a)) * u[a];
      const R wi = R(L::w(i));
      const R lam_i = R(p_coef<L, R>(i));
      if constexpr (Store<S>::V2) {
        // f^eq(p, u) - e_i(u) = lam_i p, scaled; U = u
        Store<S>::st(f + i * P + s, R(Store<S>::KF) * (lam_i * p), 0x80000000u);
      } else {
        Store<S>::st(f + i * P + s,
                     lam_i * p + (R(w3<L, R>(i)) * cu + wi * (R(4.5) * cu * cu - R(1.5) * uu)),
                     0x80000000u);
      }
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const R v = wi * ((A[k] - (diag<L>(k) ? R(1) : R(0))) + A[k] * (R(3) * cu));
        if constexpr (Store<S>::V2) {
          if (i > 0) hres[k] += v - Store<S>::st_r(h + (long long)(k * Q + i) * P + s, v, 0x80000000u);
        } else {
          store_h<L, S>(h, P, s, k, i, v, 0x80000000u);
        }
      }
    }
    if constexpr (Store<S>::V2) {
      float* U = f_ext<L>(f, P);
      float* h0 = h_ext<L>(h, P);
#pragma unroll
      for (int a = 0; a < D; ++a) U[a * P + s] = float(u[a]);
#pragma unroll
      for (int k = 0; k < C; ++k) {
        R cu0 = R(0);
        const R v0 = R(L::w(0)) * ((A[k] - (diag<L>(k) ? R(1) : R(0))) + A[k] * (R(3) * cu0));
        h0[k * P + s] = float(v0 + hres[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) chi[k * P + s] = 0;
  }
}

// ---------------------------------------------------------------------------
// Macroscopic fields of the current state into a device FP64 buffer.
// WHICH: 0 u [N][D], 1 p [N], 2 A [N][C], 3 tau_p [N][C].  Bound by the reads
// of the populations; one instance per field, so that each reads only what
// its field needs and keeps its registers for loads in flight (256^3 FP32, p
// 4.2 / 1.0 ms and A 4.4 / 1.4 ms).  16-bit u reads the bits of its values
// (FP16, us per call: 32^3 43 without, 35 with, 128^3 401 and 339); p, A and
// the original scheme's u do not (128^3 p 203 without, 287 with, A 691 and
// 737, the original scheme's u 638 and 649).
// ---------------------------------------------------------------------------
// a product that is not contracted into a following sum
__device__ __forceinline__ float mul_rounded(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rounded(double a, double b) { return __dmul_rn(a, b); }

template <class L, class S, int WHICH, bool ORIG = false>
__global__ void __launch_bounds__(128)
    k_fields(Grid g, Phys<RT<S>> ph, const S* __restrict__ f, const S* __restrict__ h,
             double* __restrict__ out, const RT<S>* __restrict__ taup, long long N) {
  using R = RT<S>;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  const long long P = g.pitch;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    R a[C];
    if constexpr (WHICH != 0) {
#pragma unroll
      for (int k = 0; k < C; ++k) {
        a[k] = R(0);
#pragma unroll
        for (int i = 0; i < Q; ++i) a[k] += load_h<L, S>(h, P, s, k, i);
      }
    }
    if constexpr (WHICH == 2) {
#pragma unroll
      for (int k = 0; k < C; ++k) out[s * C + k] = double(a[k] + (diag<L>(k) ? R(1) : R(0)));
      continue;
    }
    if constexpr (WHICH == 3) {
#pragma unroll
      for (int k = 0; k < C; ++k) out[s * C + k] = double(ph.eta_over_lam * a[k]);
      continue;
    }
    if constexpr (WHICH < 2) {
      const int x = (int)(s % g.nx);
      const int y = (int)((s / g.nx) % g.ny);
      R fv[Q];
      load_f<L, S, WHICH == 0 && !ORIG>(f, P, s, fv);
      R F[3];
      body_force<L, R>(ph, x, y, F);
      if constexpr (ORIG) {  // the original scheme: stress divergence in the force
        R dv[3];
        div_taup<L, R>(g, taup, x, y, (int)(s / ((long long)g.nx * g.ny)), s, dv);
        F[0] += dv[0];
        F[1] += dv[1];
        F[2] += dv[2];
      }
      R u[D];
      velocity<L, R>(fv, F, u);
      if constexpr (WHICH == 0) {
#pragma unroll
        for (int q = 0; q < D; ++q) out[s * D + q] = double(u[q]);
      } else {
        R tp[C];
#pragma unroll
        for (int k = 0; k < C; ++k) tp[k] = mul_rounded(ph.eta_over_lam, a[k]);
        const R fB0 = ORIG ? R(0) : fB_dir<L, R>(0, tp, ph.inv_tau_f);
        out[s] = p_of_part<L, R>(pressure<L, R>(ph, fv, u, F, fB0));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 diagnostics: per-block partial sums (fixed thread-to-site mapping and
// a fixed shuffle tree), then one block reduces the partials in index order.
// Deterministic for a given launch shape.
// part: [gridDim.x][8] = {mass, Px, Py, Pz, sum |u|^2/2, sum tr(tau_p)/2,
// non-finite count, max |u|}.
// ---------------------------------------------------------------------------
constexpr int kReduceThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  return v;
}

template <class L, class S, bool ORIG = false>
__global__ void __launch_bounds__(kReduceThreads)
    k_reduce_partial(Grid g, Phys<RT<S>> ph, const S* __restrict__ f,
                     const S* __restrict__ h, double* __restrict__ part, long long N,
                     const RT<S>* __restrict__ taup = nullptr) {
  using R = RT<S>;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  const long long P = g.pitch;
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(s % g.nx);
    const int y = (int)((s / g.nx) % g.ny);
    R fv[Q];
    load_f<L, S>(f, P, s, fv);
    bool bad = false;
    double m = 0.0, mom[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const double v = double(fv[i]);
      bad |= !isfinite(v);
      m += v;
#pragma unroll
      for (int a = 0; a < D; ++a) mom[a] += double(cc<L>(i, a)) * v;
    }
    R F[3];
    body_force<L, R>(ph, x, y, F);
    if constexpr (ORIG) {  // the original scheme: stress divergence in the force
      R dv[3];
      div_taup<L, R>(g, taup, x, y, (int)(s / ((long long)g.nx * g.ny)), s, dv);
      F[0] += dv[0];
      F[1] += dv[1];
      F[2] += dv[2];
    }
    R u[D];
    velocity<L, R>(fv, F, u);
    double uu = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) uu += double(u[a]) * double(u[a]);
    double tr = 0.0;
#pragma unroll
    for (int k = 0; k < C; ++k) {
      if (L::ca(k) != L::cb(k)) {
        // off-diagonal components only enter the finiteness check
#pragma unroll
        for (int i = 0; i < Q; ++i) bad |= !isfinite(double(load_h<L, S>(h, P, s, k, i)));
        continue;
      }
      double a = 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) a += double(load_h<L, S>(h, P, s, k, i));
      bad |= !isfinite(a);
      tr += double(ph.eta_over_lam) * a;
    }
    bad |= !isfinite(uu);
    acc[0] += m;
    acc[1] += mom[0];
    acc[2] += mom[1];
    acc[3] += mom[2];
    acc[4] += 0.5 * uu;
    acc[5] += 0.5 * tr;
    acc[6] += bad ? 1.0 : 0.0;
    acc[7] = fmax(acc[7], isfinite(uu) ? sqrt(uu) : 0.0);
  }
  __shared__ double sm[kReduceThreads / 32][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double v = q == 7 ? warp_max(acc[q]) : warp_sum(acc[q]);
    if (lane == 0) sm[wid][q] = v;
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    const int q = threadIdx.x;
    double v = sm[0][q];
    for (int w = 1; w < kReduceThreads / 32; ++w) v = q == 7 ? fmax(v, sm[w][q]) : v + sm[w][q];
    part[blockIdx.x * 8 + q] = v;
  }
}

// One block of kReduceThreads threads reduces the partials in index order;
// out[8] as documented for fvlb_reduce in fvlb.h.  (static: each translation
// unit that launches it has its own copy.)
static __global__ void __launch_bounds__(kReduceThreads)
    k_reduce_final(const double* __restrict__ part, int nparts, long long nsites,
                   double* __restrict__ out) {
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int p = threadIdx.x; p < nparts; p += blockDim.x) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const double v = part[p * 8 + q];
      acc[q] = q == 7 ? fmax(acc[q], v) : acc[q] + v;
    }
  }
  __shared__ double sm[kReduceThreads / 32][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double v = q == 7 ? warp_max(acc[q]) : warp_sum(acc[q]);
    if (lane == 0) sm[wid][q] = v;
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    const int q = threadIdx.x;
    double v = sm[0][q];
    for (int w = 1; w < kReduceThreads / 32; ++w) v = q == 7 ? fmax(v, sm[w][q]) : v + sm[w][q];
    if (q == 4 || q == 5) v /= (double)nsites;
    out[q] = v;
  }
}

// ---------------------------------------------------------------------------
// Conformation check.  A = I + M must stay symmetric positive definite in
// every model; losing it is how a run at high Wi fails (the four-roll mill
// of Sec. 3.1 goes up to Wi = 5).  Per node the smallest eigenvalue of A:
// in 2D the closed form of a symmetric 2 x 2 matrix, in 3D the Jacobi
// eigenvalue method (plane rotations; accurate to rounding relative to |A|
// also for nearly repeated eigenvalues, where roots of the characteristic
// cubic lose half the digits).  Per block: number of
// nodes whose smallest eigenvalue is not > 0 (non-finite included), the
// smallest eigenvalue, the largest tr A.
// ---------------------------------------------------------------------------
template <class L>
__device__ __forceinline__ double min_eigenvalue(const double (&M)[L::C]) {
  constexpr int D = L::D;
  if constexpr (D == 2) {
    const double a = 1.0 + M[sym<L>(0, 0)], c = 1.0 + M[sym<L>(1, 1)], b = M[sym<L>(0, 1)];
    const double h = 0.5 * (a - c);
    return 0.5 * (a + c) - sqrt(h * h + b * b);
  } else {
    // cyclic Jacobi rotations: each zeroes one off-diagonal entry; six
    // sweeps of the three pairs take a 3 x 3 matrix to diagonal in double
    double a[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) a[r][c] = M[sym<L>(r, c)] + (r == c ? 1.0 : 0.0);
#pragma unroll 1
    for (int sweep = 0; sweep < 6; ++sweep) {
#pragma unroll
      for (int pr = 0; pr < 3; ++pr) {
        const int p = pr == 2 ? 1 : 0, q = pr == 0 ? 1 : 2, o = 3 - p - q;
        const double apq = a[p][q];
        if (apq == 0.0) continue;
        const double th = (a[q][q] - a[p][p]) / (2.0 * apq);
        const double t = copysign(1.0, th) / (fabs(th) + hypot(th, 1.0));
        const double c = 1.0 / sqrt(t * t + 1.0), sn = t * c;
        a[p][p] -= t * apq;
        a[q][q] += t * apq;
        a[p][q] = a[q][p] = 0.0;
        const double aop = a[o][p], aoq = a[o][q];
        a[o][p] = a[p][o] = c * aop - sn * aoq;
        a[o][q] = a[q][o] = sn * aop + c * aoq;
      }
    }
    return fmin(a[0][0], fmin(a[1][1], a[2][2]));
  }
}

template <class L, class S>
__global__ void __launch_bounds__(kReduceThreads)
    k_conf_partial(Grid g, const S* __restrict__ h, double* __restrict__ part, long long N) {
  constexpr int Q = L::Q, C = L::C;
  const long long P = g.pitch;
  double cnt = 0.0, emin = INFINITY, trmax = -INFINITY;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    double M[C];
    double tr = 0.0;
    bool fin = true;
#pragma unroll
    for (int k = 0; k < C; ++k) {
      double a = 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) a += double(load_h<L, S>(h, P, s, k, i));
      M[k] = a;
      fin &= isfinite(a);
      if (L::ca(k) == L::cb(k)) tr += 1.0 + a;
    }
    if (!fin) {             // (fmin in the eigenvalue routine would drop a NaN)
      cnt += 1.0;
      continue;
    }
    const double e = min_eigenvalue<L>(M);
    cnt += (e > 0.0) ? 0.0 : 1.0;
    emin = fmin(emin, e);
    trmax = fmax(trmax, tr);
  }
  __shared__ double sm[kReduceThreads / 32][3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const double v0 = warp_sum(cnt), v1 = -warp_max(-emin), v2 = warp_max(trmax);
  if (lane == 0) {
    sm[wid][0] = v0;
    sm[wid][1] = v1;
    sm[wid][2] = v2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double c = sm[0][0], mn = sm[0][1], mx = sm[0][2];
    for (int w = 1; w < kReduceThreads / 32; ++w) {
      c += sm[w][0];
      mn = fmin(mn, sm[w][1]);
      mx = fmax(mx, sm[w][2]);
    }
    part[blockIdx.x * 3 + 0] = c;
    part[blockIdx.x * 3 + 1] = mn;
    part[blockIdx.x * 3 + 2] = mx;
  }
}

// (static: each translation unit that launches it has its own copy.)
static __global__ void __launch_bounds__(kReduceThreads)
    k_conf_final(const double* __restrict__ part, int nparts, double* __restrict__ out) {
  double c = 0.0, mn = INFINITY, mx = -INFINITY;
  for (int p = threadIdx.x; p < nparts; p += blockDim.x) {
    c += part[p * 3 + 0];
    mn = fmin(mn, part[p * 3 + 1]);
    mx = fmax(mx, part[p * 3 + 2]);
  }
  __shared__ double sm[kReduceThreads / 32][3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const double v0 = warp_sum(c), v1 = -warp_max(-mn), v2 = warp_max(mx);
  if (lane == 0) {
    sm[wid][0] = v0;
    sm[wid][1] = v1;
    sm[wid][2] = v2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kReduceThreads / 32; ++w) {
      sm[0][0] += sm[w][0];
      sm[0][1] = fmin(sm[0][1], sm[w][1]);
      sm[0][2] = fmax(sm[0][2], sm[w][2]);
    }
    out[0] = sm[0][0];
    out[1] = sm[0][1];
    out[2] = sm[0][2];
  }
}

// ---------------------------------------------------------------------------
// High-Wi repair of the conformation (fvlb_repair_conformation).  Per node,
// in FP64: A from the stress populations, its eigen-decomposition by cyclic
// Jacobi rotations with the rotations accumulated into the eigenvectors
// (ten sweeps), and where the smallest eigenvalue is below eps,
// A' = V max(Lambda, eps) V^T, applied as h'_{k,i} += w_i (A' - A)_k, which
// moves the zeroth moment of h only (sum_i w_i c_i = 0).  16-bit forms: the
// 16-bit populations are re-rounded and their rounding residual goes to the
// FP32 rest population, as in the step.  count[0] += nodes changed (a node
// with a non-finite A is counted and left as it is).
// ---------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ void jacobi_eig(double (&a)[3][3], double (&v)[3][3]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) v[r][c] = r == c ? 1.0 : 0.0;
#pragma unroll 1
  for (int sweep = 0; sweep < 10; ++sweep) {
#pragma unroll
    for (int pr = 0; pr < (D == 3 ? 3 : 1); ++pr) {
      const int p = pr == 2 ? 1 : 0, q = pr == 0 ? 1 : 2;
      const double apq = a[p][q];
      if (apq == 0.0) continue;
      const double th = (a[q][q] - a[p][p]) / (2.0 * apq);
      const double t = copysign(1.0, th) / (fabs(th) + hypot(th, 1.0));
      const double c = 1.0 / sqrt(t * t + 1.0), sn = t * c;
      // a <- J^T a J and v <- v J for the rotation J in the (p, q) plane
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const double akp = a[k][p], akq = a[k][q];
        a[k][p] = c * akp - sn * akq;
        a[k][q] = sn * akp + c * akq;
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const double apk = a[p][k], aqk = a[q][k];
        a[p][k] = c * apk - sn * aqk;
        a[q][k] = sn * apk + c * aqk;
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const double vkp = v[k][p], vkq = v[k][q];
        v[k][p] = c * vkp - sn * vkq;
        v[k][q] = sn * vkp + c * vkq;
      }
    }
  }
}

template <class L, class S>
__global__ void __launch_bounds__(kReduceThreads)
    k_repair(Grid g, S* __restrict__ h, double eps, unsigned long long* __restrict__ count,
             long long N) {
  using R = RT<S>;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  const long long P = g.pitch;
  unsigned long long mine = 0;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    double M[C];
    bool fin = true;
#pragma unroll
    for (int k = 0; k < C; ++k) {
      double acc = 0.0;
#pragma unroll
      for (int i = 0; i < Q; ++i) acc += double(load_h<L, S>(h, P, s, k, i));
      M[k] = acc;
      fin &= isfinite(acc);
    }
    if (!fin) {
      ++mine;
      continue;
    }
    double a[3][3], v[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        a[r][c] = (r < D && c < D) ? M[sym<L>(r, c)] + (r == c ? 1.0 : 0.0) : 0.0;
    jacobi_eig<D>(a, v);
    double lmin = a[0][0];
#pragma unroll
    for (int k = 1; k < D; ++k) lmin = fmin(lmin, a[k][k]);
    if (!(lmin < eps)) continue;
    ++mine;
    double dA[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const int ra = L::ca(k), rb = L::cb(k);
      double An = 0.0;
#pragma unroll
      for (int j = 0; j < D; ++j) An += v[ra][j] * fmax(a[j][j], eps) * v[rb][j];
      dA[k] = An - (M[k] + (ra == rb ? 1.0 : 0.0));
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
      R res = R(0);
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        S* q = h + (long long)(k * Q + i) * P + s;
        const R nv = R(double(Store<S>::cvt(*q)) + L::w(i) * dA[k]);
        if constexpr (Store<S>::V2) res += nv - Store<S>::st_r(q, nv, 0x80000000u);
        else Store<S>::st(q, nv, 0u);
      }
      if constexpr (Store<S>::V2) {
        float* h0 = h_ext<L>(h, P) + k * P + s;
        *h0 = float(double(*h0) + L::w(0) * dA[k] + double(res));
      } else {
        S* q = h + (long long)(k * Q) * P + s;
        Store<S>::st(q, R(double(Store<S>::cvt(*q)) + L::w(0) * dA[k]), 0u);
      }
    }
  }
  // block total, then one atomic per block (an integer sum: order-free)
  __shared__ unsigned long long sm[kReduceThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kReduceThreads / 32; ++w) t += sm[w];
    if (t) atomicAdd(count, t);
  }
}

}  // namespace fvlb
