// mlp.cu -- the learned stress closure: training-pair collection from the
// plain method's state, GPU training of the network (hand-written forward,
// backward and Adam kernels), FP16 packing, tensor-core inference, and the
// fvlb_mlp_* C ABI.  Applying the network inside the step is in
// k_step_fused (fvlb_set_closure).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "fvlb.h"
#include "fvlb_internal.h"
#include "fvlb_launch.cuh"
#include "fvlb_mlp.cuh"

namespace fvlb {

// ---------------------------------------------------------------------------
// Training pairs from the current state of a grid (the plain method).
// For every stride-th node s: x = (lambda grad u, A - I, [dt/lambda]) and
// target y = lambda chi, with grad u and chi exactly as the step forms them.
// ---------------------------------------------------------------------------
template <class L, class S>
__device__ void node_velocity(const Grid& g, const Phys<RT<S>>& ph, const S* __restrict__ f,
                              int x, int y, int z, RT<S> (&u)[L::D]) {
  using R = RT<S>;
  const long long s = ((long long)z * g.ny + y) * g.nx + x;
  R fv[L::Q];
  load_f<L, S>(f, g.pitch, s, fv);
  R F[3];
  body_force<L, R>(ph, x, y, F);
  velocity<L, R>(fv, F, u);
}

template <class L, class S>
__global__ void k_closure_pairs(Grid g, Phys<RT<S>> ph, const S* __restrict__ f,
                                const S* __restrict__ h, long long N, long long stride,
                                long long npairs, float* __restrict__ X, float* __restrict__ T,
                                double lam) {
  using R = RT<S>;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  constexpr int IN = MlpDims<D>::IN, OUT = MlpDims<D>::OUT;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < npairs;
       j += (long long)gridDim.x * blockDim.x) {
    const long long s = (j * stride) % N;
    const int p[3] = {(int)(s % g.nx), (int)((s / g.nx) % g.ny), (int)(s / ((long long)g.nx * g.ny))};
    const int n[3] = {g.nx, g.ny, g.nz};
    R u[D];
    node_velocity<L, S>(g, ph, f, p[0], p[1], p[2], u);
    R gr[D][D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      int qp[3] = {p[0], p[1], p[2]}, qm[3] = {p[0], p[1], p[2]};
      qp[a] = (p[a] + 1) % n[a];
      qm[a] = (p[a] - 1 + n[a]) % n[a];
      R up[D], um[D];
      node_velocity<L, S>(g, ph, f, qp[0], qp[1], qp[2], up);
      node_velocity<L, S>(g, ph, f, qm[0], qm[1], qm[2], um);
      const bool wall = (g.walls >> a) & 1;
#pragma unroll
      for (int b = 0; b < D; ++b) {
        R d = R(0.5) * (up[b] - um[b]);
        if (wall && p[a] == 0) d = u[b] + up[b] * R(1.0 / 3.0);
        if (wall && p[a] == n[a] - 1) d = -(u[b] + um[b] * R(1.0 / 3.0));
        gr[a][b] = d;
      }
    }
    R Ad[C], A[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      R a = R(0);
#pragma unroll
      for (int i = 0; i < Q; ++i) a += load_h<L, S>(h, g.pitch, s, k, i);
      Ad[k] = a;
      A[k] = a + (diag<L>(k) ? R(1) : R(0));
    }
    R chi[C];
    chi_tensor<L, R>(A, Ad, gr, ph, chi);
    float* xr = X + j * IN;
    int q = 0;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int b = 0; b < D; ++b) xr[q++] = float(lam * double(gr[a][b]));
#pragma unroll
    for (int k = 0; k < C; ++k) xr[q++] = float(Ad[k]);
    if (D == 2) xr[q++] = float(1.0 / lam);
    float* tr = T + j * OUT;
#pragma unroll
    for (int k = 0; k < C; ++k) tr[k] = float(lam * double(chi[k]));
  }
}

// ---------------------------------------------------------------------------
// Training: forward, backward and weight gradients of tiles of 32 samples.
//
// What bounds it: FP32 fused multiply-adds (16.3 k a sample in 3D; the
// operands are FP32 and stay FP32, so no tensor cores).  A block of 128
// threads takes every kGradBlocks-th tile; each layer is a small matrix
// product of which a thread holds a 4 x 4 (activations) or 8 x 4 (weight
// gradient) piece, so one 16-byte shared-memory load feeds 8 to 11 FMAs.
// The weight gradients stay in registers over all tiles of a block and are
// written once, as one partial per block.  Every sum has a fixed order and
// the assignment of tiles does not depend on the device: deterministic.
// Activations lie unit-major ([unit][sample], rows of 32 + 4 floats), so
// that a thread's four samples are one 16-byte load and neighbouring rows
// start in different banks.
// 32768 samples in 3D, a call of fvlb_mlp_grad from host arrays: 310 us with
// one thread per sample, 125 us now; of these this kernel 50 us (10.7 TFMA/s,
// 27 % of the FMA pipe's 40.3: shared-memory latency at 12 warps an SM, and 2.25
// tiles a block on average where some have 3) and the sum of the partials 10.
// ---------------------------------------------------------------------------

// GELU in its tanh form, 0.5 z (1 + tanh(u)) = z / (1 + exp(-2 u)), and its
// derivative.
__device__ __forceinline__ float gelu_acc(float z, float& dz) {
  const float c = 0.7978845608028654f;
  const float z2 = z * z;
  const float u = c * (z + 0.044715f * z2 * z);
  const float sg = 1.0f / (1.0f + expf(-2.0f * u));
  dz = sg + 2.0f * z * sg * (1.0f - sg) * (c * (1.0f + 3.0f * 0.044715f * z2));
  return z * sg;
}

__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  return hash32(x);
}

constexpr int kTB = 64;          // a training batch is a multiple of this ...
constexpr int kMaxBatches = 4096; // ... and at most so many of it
constexpr int kTS = 32;          // samples per tile
constexpr int kGT = 128;         // threads of a gradient block
constexpr int kGradBlocks = 456; // most blocks (three per SM of a 152-SM device)

template <int IN, int OUT>
struct GradSmem {
  static constexpr int LD = kTS + 4;
  float W1[16][kMlpH];           // [k][j], k < IN
  float W2[kMlpH][kMlpH];        // [j][k]
  float W3[8][kMlpH];            // [o][k], o < OUT
  float b1[kMlpH], b2[kMlpH], b3[8];
  float x[16][LD];               // inputs, [k][sample]
  float h1[kMlpH][LD], d1[kMlpH][LD];   // activations; GELU derivatives, then dz
  float h2[kMlpH][LD], d2[kMlpH][LD];
  float dy[8][LD];
  double loss[kGT / 32];
};

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// dot product of four samples of two rows, added to a in sample order
__device__ __forceinline__ float dot4(float a, const float4& p, const float4& q) {
  a += p.x * q.x;
  a += p.y * q.y;
  a += p.z * q.z;
  a += p.w * q.w;
  return a;
}

template <int IN, int OUT>
__global__ void __launch_bounds__(kGT, 3)
    k_mlp_grad(const float* __restrict__ prm, const float* __restrict__ X,
               const float* __restrict__ T, long long count, long long n, int sample_seed,
               float delta2, float* __restrict__ part, double* __restrict__ part_loss) {
  using PP = MlpParams<IN, OUT>;
  constexpr int H = kMlpH;
  extern __shared__ __align__(16) unsigned char grad_smem[];
  auto& sm = *reinterpret_cast<GradSmem<IN, OUT>*>(grad_smem);
  const int tid = threadIdx.x;
  for (int e = tid; e < 16 * H; e += kGT) {
    const int k = e / H, j = e % H;
    sm.W1[k][j] = k < IN ? prm[PP::W1 + j * IN + k] : 0.f;
  }
  for (int e = tid; e < H * H; e += kGT) sm.W2[e / H][e % H] = prm[PP::W2 + e];
  for (int e = tid; e < 8 * H; e += kGT) sm.W3[e / H][e % H] = e < OUT * H ? prm[PP::W3 + e] : 0.f;
  for (int e = tid; e < H; e += kGT) {
    sm.b1[e] = prm[PP::B1 + e];
    sm.b2[e] = prm[PP::B2 + e];
  }
  if (tid < 8) sm.b3[tid] = tid < OUT ? prm[PP::B3 + tid] : 0.f;

  // pieces of the products: samples 4 s4 .. + 3 and units 4 j4 .. + 3;
  // weight gradients rows ti + 8 r and columns tk + 16 c
  const int s4 = tid & 7, j4 = tid >> 3;
  const int ti = tid >> 4, tk = tid & 15;
  float gw2[8][4] = {}, gw1[8] = {}, gw3[4] = {}, gb = 0.f, gb3 = 0.f;
  // FP64 from tile to tile: a block has up to 18 tiles (576 samples of the
  // largest call), and beside a large residual of one a sum in FP32 loses the
  // small ones of the others
  double loss = 0.0;

  const long long ntiles = (n + kTS - 1) / kTS;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    // inputs and weights of the tile's samples; thread tid < 32: its sample
    __syncthreads();
    long long src = -1;
    if (tid < kTS) {
      const long long off = tile * kTS + tid;
      if (off < n) {
        src = sample_seed >= 0
                  ? (long long)(((uint64_t)mix32((uint32_t)off * 0x9e3779b9u ^ mix32((uint32_t)sample_seed)) *
                                 (uint64_t)count) >> 32)
                  : off;
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) sm.x[k][tid] = src >= 0 && k < IN ? X[src * IN + k] : 0.f;
    }
    __syncthreads();
    // layer 1
    {
      float a[4][4];   // [unit][sample]
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[j][q] = sm.b1[4 * j4 + j];
#pragma unroll
      for (int k = 0; k < IN; ++k) {
        const float4 xs = lds4(&sm.x[k][4 * s4]), ws = lds4(&sm.W1[k][4 * j4]);
        const float xv[4] = {xs.x, xs.y, xs.z, xs.w}, wv[4] = {ws.x, ws.y, ws.z, ws.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) a[j][q] += wv[j] * xv[q];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float hv[4], dv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hv[q] = gelu_acc(a[j][q], dv[q]);
        *reinterpret_cast<float4*>(&sm.h1[4 * j4 + j][4 * s4]) = make_float4(hv[0], hv[1], hv[2], hv[3]);
        *reinterpret_cast<float4*>(&sm.d1[4 * j4 + j][4 * s4]) = make_float4(dv[0], dv[1], dv[2], dv[3]);
      }
    }
    __syncthreads();
    // layer 2
    {
      float a[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[j][q] = sm.b2[4 * j4 + j];
#pragma unroll 4
      for (int k = 0; k < H; k += 4) {
        float4 hs[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hs[q] = lds4(&sm.h1[k + q][4 * s4]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 ws = lds4(&sm.W2[4 * j4 + j][k]);
          const float wv[4] = {ws.x, ws.y, ws.z, ws.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            a[j][0] += wv[q] * hs[q].x;
            a[j][1] += wv[q] * hs[q].y;
            a[j][2] += wv[q] * hs[q].z;
            a[j][3] += wv[q] * hs[q].w;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float hv[4], dv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) hv[q] = gelu_acc(a[j][q], dv[q]);
        *reinterpret_cast<float4*>(&sm.h2[4 * j4 + j][4 * s4]) = make_float4(hv[0], hv[1], hv[2], hv[3]);
        *reinterpret_cast<float4*>(&sm.d2[4 * j4 + j][4 * s4]) = make_float4(dv[0], dv[1], dv[2], dv[3]);
      }
    }
    __syncthreads();
    // layer 3, loss and dy: thread (sample tid % 32, outputs tid / 32 and + 4)
    {
      const int sp = tid & 31, o0 = tid >> 5;
      // the sample of this thread, for its targets
      const long long off = tile * kTS + sp;
      long long sr = -1;
      if (off < n) {
        sr = sample_seed >= 0
                 ? (long long)(((uint64_t)mix32((uint32_t)off * 0x9e3779b9u ^ mix32((uint32_t)sample_seed)) *
                                (uint64_t)count) >> 32)
                 : off;
      }
      // sample weight: 1, or 1 / (mean_o t_o^2 + delta^2) for the relative loss
      float wgt = 1.f;
      if (delta2 > 0.f && sr >= 0) {
        float tt = 0.f;
        for (int o = 0; o < OUT; ++o) tt += T[sr * OUT + o] * T[sr * OUT + o];
        wgt = 1.f / (tt / float(OUT) + delta2);
      }
      const float scale = 2.0f * wgt / (float(n) * float(OUT));
      float tl = 0.f;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int o = o0 + 4 * p;
        float y = sm.b3[o];
#pragma unroll 8
        for (int k = 0; k < H; ++k) y += sm.W3[o][k] * sm.h2[k][sp];
        const float r = sr >= 0 && o < OUT ? y - T[sr * OUT + (o < OUT ? o : 0)] : 0.f;
        tl += wgt * r * r;
        sm.dy[o][sp] = scale * r;
      }
      loss += (double)tl;
    }
    __syncthreads();
    // backward through layer 3 and GELU: dz2 over d2
    {
      float a[4][4] = {};
#pragma unroll
      for (int o = 0; o < OUT; ++o) {
        const float4 ds = lds4(&sm.dy[o][4 * s4]), ws = lds4(&sm.W3[o][4 * j4]);
        const float dv[4] = {ds.x, ds.y, ds.z, ds.w}, wv[4] = {ws.x, ws.y, ws.z, ws.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) a[j][q] += wv[j] * dv[q];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float4* d = reinterpret_cast<float4*>(&sm.d2[4 * j4 + j][4 * s4]);
        const float4 g = *d;
        *d = make_float4(a[j][0] * g.x, a[j][1] * g.y, a[j][2] * g.z, a[j][3] * g.w);
      }
    }
    __syncthreads();
    // through layer 2: dz1 over d1
    {
      float a[4][4] = {};
#pragma unroll 8
      for (int i = 0; i < H; ++i) {
        const float4 ds = lds4(&sm.d2[i][4 * s4]), ws = lds4(&sm.W2[i][4 * j4]);
        const float dv[4] = {ds.x, ds.y, ds.z, ds.w}, wv[4] = {ws.x, ws.y, ws.z, ws.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) a[j][q] += wv[j] * dv[q];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float4* d = reinterpret_cast<float4*>(&sm.d1[4 * j4 + j][4 * s4]);
        const float4 g = *d;
        *d = make_float4(a[j][0] * g.x, a[j][1] * g.y, a[j][2] * g.z, a[j][3] * g.w);
      }
    }
    __syncthreads();
    // weight gradients, in sample order
#pragma unroll 1
    for (int q = 0; q < kTS; q += 4) {
      float4 hv[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) hv[c] = lds4(&sm.h1[tk + 16 * c][q]);
      const float4 xv = lds4(&sm.x[tk][q]);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float4 d = lds4(&sm.d2[ti + 8 * r][q]);
#pragma unroll
        for (int c = 0; c < 4; ++c) gw2[r][c] = dot4(gw2[r][c], d, hv[c]);
        gw1[r] = dot4(gw1[r], lds4(&sm.d1[ti + 8 * r][q]), xv);
      }
      const float4 yv = lds4(&sm.dy[ti][q]);
#pragma unroll
      for (int c = 0; c < 4; ++c) gw3[c] = dot4(gw3[c], yv, lds4(&sm.h2[tk + 16 * c][q]));
      const float4 one = make_float4(1.f, 1.f, 1.f, 1.f);
      gb = dot4(gb, lds4(tid < H ? &sm.d1[tid & (H - 1)][q] : &sm.d2[tid & (H - 1)][q]), one);
      if (tid < 8) gb3 = dot4(gb3, lds4(&sm.dy[tid][q]), one);
    }
  }
  // the block's partial
  float* out = part + (long long)blockIdx.x * PP::N;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = ti + 8 * r;
#pragma unroll
    for (int c = 0; c < 4; ++c) out[PP::W2 + i * H + tk + 16 * c] = gw2[r][c];
    if (tk < IN) out[PP::W1 + i * IN + tk] = gw1[r];
  }
  if (ti < OUT) {
#pragma unroll
    for (int c = 0; c < 4; ++c) out[PP::W3 + ti * H + tk + 16 * c] = gw3[c];
  }
  out[(tid < H ? PP::B1 : PP::B2) + (tid & (H - 1))] = gb;
  if (tid < OUT) out[PP::B3 + tid] = gb3;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, o);
  if ((tid & 31) == 0) sm.loss[tid >> 5] = loss;
  __syncthreads();
  if (tid == 0) {
    double a = sm.loss[0];
#pragma unroll
    for (int q = 1; q < kGT / 32; ++q) a += sm.loss[q];
    part_loss[blockIdx.x] = a;
  }
}

// Sum the block partials (fixed order) into grad[] (and the loss); if adam,
// apply one Adam step to the FP32 master parameters.  A block takes 32
// parameters, each of its 8 warps every 8th partial.
constexpr int kUpdT = 256;
__global__ void __launch_bounds__(kUpdT)
    k_mlp_update(float* __restrict__ prm, float* __restrict__ mo, float* __restrict__ ve,
                 const float* __restrict__ part, const double* __restrict__ part_loss, int nblocks,
                 int nparam, float* __restrict__ grad, double* __restrict__ loss,
                 double loss_scale, int adam, float lr, float bc1, float bc2) {
  __shared__ float sum[kUpdT / 32][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float g = 0.f;
  if (p < nparam) {
#pragma unroll 8
    for (int b = w; b < nblocks; b += kUpdT / 32) g += part[(long long)b * nparam + p];
  }
  sum[w][lane] = g;
  if (blockIdx.x == 0 && w == kUpdT / 32 - 1) {
    double a = 0.0;
    for (int b = lane; b < nblocks; b += 32) a += part_loss[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) *loss = a * loss_scale;
  }
  __syncthreads();
  if (w != 0 || p >= nparam) return;
  g = sum[0][lane];
#pragma unroll
  for (int q = 1; q < kUpdT / 32; ++q) g += sum[q][lane];
  if (grad) grad[p] = g;
  if (adam) {
    const float b1 = 0.9f, b2 = 0.999f;
    const float m = b1 * mo[p] + (1.f - b1) * g;
    const float v = b2 * ve[p] + (1.f - b2) * g * g;
    mo[p] = m;
    ve[p] = v;
    prm[p] -= lr * (m / bc1) / (sqrtf(v / bc2) + 1e-8f);
  }
}

// FP32 master parameters -> packed FP16 inference weights
template <int IN, int OUT>
__global__ void k_mlp_pack(const float* __restrict__ prm, MlpPacked* __restrict__ P) {
  using PP = MlpParams<IN, OUT>;
  constexpr int H = kMlpH;
  // (see MlpPacked) e = lane * 4 + register within each 128-register piece
  for (int e = threadIdx.x; e < 4 * 128; e += blockDim.x) {
    const int nt = e >> 7, lane = (e >> 2) & 31, q = e & 3;
    P->W1[nt][lane][q] = mlp_b_register(lane, q & 1, [&](int g, int k) {
      return k < IN ? prm[PP::W1 + (16 * nt + 8 * (q >> 1) + g) * IN + k] : 0.f;
    });
  }
  for (int e = threadIdx.x; e < 16 * 128; e += blockDim.x) {
    const int nt = e >> 9, kt = (e >> 7) & 3, lane = (e >> 2) & 31, q = e & 3;
    P->W2[nt][kt][lane][q] = mlp_b_register(lane, q & 1, [&](int g, int k) {
      return prm[PP::W2 + (16 * nt + 8 * (q >> 1) + g) * H + 16 * kt + k];
    });
  }
  for (int e = threadIdx.x; e < 2 * 128; e += blockDim.x) {
    const int kp = e >> 7, lane = (e >> 2) & 31, q = e & 3;
    P->W3[kp][lane][q] = mlp_b_register(lane, q & 1, [&](int g, int k) {
      return g < OUT ? prm[PP::W3 + g * H + 32 * kp + 16 * (q >> 1) + k] : 0.f;
    });
  }
  for (int e = threadIdx.x; e < H; e += blockDim.x) {
    P->b1[e] = prm[PP::B1 + e];
    P->b2[e] = prm[PP::B2 + e];
  }
  for (int e = threadIdx.x; e < 8; e += blockDim.x) P->b3[e] = e < OUT ? prm[PP::B3 + e] : 0.f;
}

// Tensor-core inference of n samples (32 per warp).
template <int IN, int OUT>
__global__ void __launch_bounds__(128) k_mlp_infer(const MlpPacked* __restrict__ Pg,
                                                   const float* __restrict__ X, long long n,
                                                   float* __restrict__ Y) {
  __shared__ MlpPacked P;
  __shared__ __half xs[4][32][24];
  __shared__ float ys[4][32][8];
  mlp_load(P, Pg);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long base = (blockIdx.x * 4LL + w) * 32; base < n; base += gridDim.x * 128LL) {
    const long long r = base + lane;
    for (int k = 0; k < 24; ++k)
      xs[w][lane][k] = __float2half_rn(r < n && k < IN ? X[r * IN + k] : 0.f);
    __syncwarp();
    mlp_warp(P, xs[w], ys[w]);
    __syncwarp();
    if (r < n)
      for (int o = 0; o < OUT; ++o) Y[r * OUT + o] = ys[w][lane][o];
    __syncwarp();
  }
}

}  // namespace fvlb

// ===========================================================================
// C ABI
// ===========================================================================
using namespace fvlb;

struct fvlb_mlp_s {
  int lattice = 9, D = 2, IN = 8, OUT = 3, NP = 0;
  long long cap = 0, count = 0;
  float *prm = nullptr, *mo = nullptr, *ve = nullptr, *grad = nullptr;
  float *X = nullptr, *T = nullptr;
  float* part = nullptr;
  double* part_loss = nullptr;
  double* loss = nullptr;
  MlpPacked* packed = nullptr;
  long long adam_t = 0;
  double delta = 0.0;       // relative-loss floor (0: plain mean squared error)
  cudaStream_t stream = nullptr;
  fvlb_alloc_fn alloc = nullptr;
  fvlb_free_fn free_ = nullptr;
  void* actx = nullptr;
  // samples of fvlb_mlp_grad / _infer on the device, kept from call to call:
  // grown to the largest one within keep_floats, given back with the network
  float* stage = nullptr;
  size_t stage_floats = 0;
  std::vector<void*> owned;
  std::string err;
};

namespace {

int mfail(fvlb_mlp_t m, int code, const std::string& msg) {
  if (m) m->err = msg;
  else set_global_error(code, msg.c_str());
  return code;
}

void* malloc_dev(fvlb_mlp_t m, size_t bytes) {
  bytes = (bytes + 255) & ~size_t(255);
  void* p = nullptr;
  if (m->alloc) p = m->alloc(bytes, m->actx);
  else if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  if (p) m->owned.push_back(p);
  return p;
}

void free_dev(fvlb_mlp_t m, void* p) {
  m->owned.erase(std::find(m->owned.begin(), m->owned.end(), p));
  if (m->free_) m->free_(p, m->actx);
  else cudaFree(p);
}

// Samples a network may keep between calls: those of the largest gradient
// (22 MB in 3D).  Inference takes any number.
size_t keep_floats(fvlb_mlp_t m) { return (size_t)(m->IN + m->OUT) * kMaxBatches * kTB; }

// The device buffer for a call's samples, and its return at the call's end
// (the stream is idle): a larger one than may be kept is freed.
float* stage_take(fvlb_mlp_t m, size_t floats) {
  if (floats > keep_floats(m)) return static_cast<float*>(malloc_dev(m, sizeof(float) * floats));
  if (floats > m->stage_floats) {
    if (m->stage) free_dev(m, m->stage);
    m->stage = static_cast<float*>(malloc_dev(m, sizeof(float) * floats));
    m->stage_floats = m->stage ? floats : 0;
  }
  return m->stage;
}
void stage_give(fvlb_mlp_t m, float* p) {
  if (p != m->stage) free_dev(m, p);
}

// blocks of a gradient over n samples
int grad_blocks(long long n) {
  return (int)std::min<long long>((n + kTS - 1) / kTS, kGradBlocks);
}

template <int IN, int OUT>
cudaError_t launch_grad_of(fvlb_mlp_t m, const float* X, const float* T, long long count,
                           long long n, int seed, float d2) {
  constexpr size_t sm = sizeof(GradSmem<IN, OUT>);
  auto kern = k_mlp_grad<IN, OUT>;
  const cudaError_t e = allow_dynamic_smem(kern, sm);
  if (e != cudaSuccess) return e;
  kern<<<grad_blocks(n), kGT, sm, m->stream>>>(m->prm, X, T, count, n, seed, d2, m->part,
                                               m->part_loss);
  return cudaGetLastError();
}

cudaError_t launch_grad(fvlb_mlp_t m, const float* X, const float* T, long long count,
                        long long n, int seed) {
  const float d2 = float(m->delta * m->delta);
  return m->D == 2 ? launch_grad_of<8, 3>(m, X, T, count, n, seed, d2)
                   : launch_grad_of<15, 6>(m, X, T, count, n, seed, d2);
}

cudaError_t repack(fvlb_mlp_t m) {
  if (m->D == 2) k_mlp_pack<8, 3><<<1, 256, 0, m->stream>>>(m->prm, m->packed);
  else k_mlp_pack<15, 6><<<1, 256, 0, m->stream>>>(m->prm, m->packed);
  return cudaGetLastError();
}

uint32_t host_hash(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

}  // namespace

namespace fvlb {
const void* mlp_packed(fvlb_mlp_t m) { return m ? m->packed : nullptr; }
int mlp_lattice(fvlb_mlp_t m) { return m ? m->lattice : 0; }
}  // namespace fvlb

extern "C" {

int fvlb_mlp_create(fvlb_mlp_t* out, int lattice, long capacity, unsigned seed) {
  if (!out) return set_global_error(FVLB_EINVAL, "fvlb_mlp_create: out is NULL");
  *out = nullptr;
  if (lattice != FVLB_D2Q9 && lattice != FVLB_D3Q19)
    return set_global_error(FVLB_EINVAL, "fvlb_mlp_create: unknown lattice");
  if (capacity < 1) return set_global_error(FVLB_EINVAL, "fvlb_mlp_create: capacity must be >= 1");
  fvlb_mlp_s* m = new (std::nothrow) fvlb_mlp_s();
  if (!m) return set_global_error(FVLB_ENOMEM, "fvlb_mlp_create: out of host memory");
  m->lattice = lattice;
  m->D = lattice == FVLB_D2Q9 ? 2 : 3;
  m->IN = m->D == 2 ? 8 : 15;
  m->OUT = m->D == 2 ? 3 : 6;
  m->NP = m->D == 2 ? MlpParams<8, 3>::N : MlpParams<15, 6>::N;
  m->cap = capacity;
  current_allocator(&m->alloc, &m->free_, &m->actx);
  cudaError_t e = cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    delete m;
    return set_global_error(FVLB_ECUDA, "fvlb_mlp_create: stream creation failed");
  }
  m->prm = static_cast<float*>(malloc_dev(m, sizeof(float) * m->NP));
  m->mo = static_cast<float*>(malloc_dev(m, sizeof(float) * m->NP));
  m->ve = static_cast<float*>(malloc_dev(m, sizeof(float) * m->NP));
  m->grad = static_cast<float*>(malloc_dev(m, sizeof(float) * m->NP));
  m->X = static_cast<float*>(malloc_dev(m, sizeof(float) * m->IN * capacity));
  m->T = static_cast<float*>(malloc_dev(m, sizeof(float) * m->OUT * capacity));
  m->part = static_cast<float*>(malloc_dev(m, sizeof(float) * m->NP * (size_t)kGradBlocks));
  m->part_loss = static_cast<double*>(malloc_dev(m, sizeof(double) * kGradBlocks));
  m->loss = static_cast<double*>(malloc_dev(m, sizeof(double)));
  m->packed = static_cast<MlpPacked*>(malloc_dev(m, sizeof(MlpPacked)));
  if (!m->prm || !m->mo || !m->ve || !m->grad || !m->X || !m->T || !m->part || !m->part_loss ||
      !m->loss || !m->packed) {
    fvlb_mlp_destroy(m);
    return set_global_error(FVLB_ENOMEM, "fvlb_mlp_create: device allocation failed");
  }
  // He initialisation from a counter-based hash (Box-Muller), biases zero
  std::vector<float> p(m->NP, 0.f);
  const int H = kMlpH;
  auto normal = [&](uint32_t i) {
    const uint32_t a = host_hash(seed * 0x9e3779b9u ^ (2 * i + 1));
    const uint32_t b = host_hash(seed * 0x85ebca6bu ^ (2 * i + 2));
    const double u1 = (a + 1.0) / 4294967297.0, u2 = b / 4294967296.0;
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
  };
  const int w1 = 0, w2 = H * m->IN + H, w3 = w2 + H * H + H;
  for (int i = 0; i < H * m->IN; ++i) p[w1 + i] = float(normal(i) * std::sqrt(2.0 / m->IN));
  for (int i = 0; i < H * H; ++i) p[w2 + i] = float(normal(100000 + i) * std::sqrt(2.0 / H));
  for (int i = 0; i < m->OUT * H; ++i) p[w3 + i] = float(normal(200000 + i) * std::sqrt(1.0 / H));
  e = cudaMemcpy(m->prm, p.data(), sizeof(float) * m->NP, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(m->mo, 0, sizeof(float) * m->NP);
  if (e == cudaSuccess) e = cudaMemset(m->ve, 0, sizeof(float) * m->NP);
  if (e == cudaSuccess) e = repack(m);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) {
    fvlb_mlp_destroy(m);
    return set_global_error(FVLB_ECUDA, "fvlb_mlp_create: initialisation failed");
  }
  *out = m;
  return FVLB_OK;
}

int fvlb_mlp_num_params(fvlb_mlp_t m, size_t* n) {
  if (!m || !n) return mfail(m, FVLB_EINVAL, "fvlb_mlp_num_params: NULL argument");
  *n = (size_t)m->NP;
  return FVLB_OK;
}

int fvlb_mlp_get_params(fvlb_mlp_t m, float* host, size_t count) {
  if (!m || !host || count < (size_t)m->NP) return mfail(m, FVLB_EINVAL, "fvlb_mlp_get_params: bad buffer");
  cudaError_t e = cudaMemcpyAsync(host, m->prm, sizeof(float) * m->NP, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, cudaGetErrorString(e));
  return FVLB_OK;
}

int fvlb_mlp_set_params(fvlb_mlp_t m, const float* host, size_t count) {
  if (!m || !host || count != (size_t)m->NP) return mfail(m, FVLB_EINVAL, "fvlb_mlp_set_params: bad buffer");
  cudaError_t e = cudaMemcpyAsync(m->prm, host, sizeof(float) * m->NP, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = repack(m);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, cudaGetErrorString(e));
  return FVLB_OK;
}

int fvlb_mlp_collect(fvlb_mlp_t m, fvlb_t h, long stride) {
  if (!m || !h) return mfail(m, FVLB_EINVAL, "fvlb_mlp_collect: NULL argument");
  if (stride < 1) return mfail(m, FVLB_EINVAL, "fvlb_mlp_collect: stride must be >= 1");
  StateView v;
  int r = state_view(h, &v);
  if (r != FVLB_OK) return mfail(m, r, "fvlb_mlp_collect: no state");
  if (v.lattice != m->lattice) return mfail(m, FVLB_EINVAL, "fvlb_mlp_collect: lattice mismatch");
  const long long want = (v.N + stride - 1) / stride;
  const long long n = std::min<long long>(want, m->cap - m->count);
  if (n <= 0) return FVLB_OK;
  StepDesc d = v.desc;
  const int threads = 128;
  const int blocks = (int)std::min<long long>((n + threads - 1) / threads, 4096);
  float* X = m->X + m->count * m->IN;
  float* T = m->T + m->count * m->OUT;
  Grid g{d.nx, d.ny, m->D == 3 ? d.nz : 1, d.walls, d.pitch};
  cudaError_t e = cudaSuccess;
#define PAIRS(L, S)                                                                          \
  {                                                                                          \
    using R = RT<S>;                                                                         \
    Phys<R> ph = make_phys<R>(d);                                                            \
    k_closure_pairs<L, S><<<blocks, threads, 0, d.stream>>>(                                 \
        g, ph, static_cast<const S*>(d.f_in), static_cast<const S*>(d.h_in), d.N, stride, n, X, \
        T, d.lambda);                                                                        \
    e = cudaGetLastError();                                                                  \
  }
  if (d.storage == kFP64) {
    if (m->D == 2) PAIRS(D2Q9, double) else PAIRS(D3Q19, double)
  } else if (d.storage == kFP32) {
    if (m->D == 2) PAIRS(D2Q9, float) else PAIRS(D3Q19, float)
  } else {
    return mfail(m, FVLB_EINVAL, "fvlb_mlp_collect: collect from an FP64 or FP32 state");
  }
#undef PAIRS
  if (e == cudaSuccess) e = cudaStreamSynchronize(d.stream);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, std::string("fvlb_mlp_collect: ") + cudaGetErrorString(e));
  m->count += n;
  return FVLB_OK;
}

int fvlb_mlp_set_loss(fvlb_mlp_t m, double delta) {
  if (!m) return set_global_error(FVLB_EINVAL, "NULL mlp");
  if (!(delta >= 0.0) || !std::isfinite(delta)) return mfail(m, FVLB_EINVAL, "fvlb_mlp_set_loss: delta must be >= 0");
  m->delta = delta;
  return FVLB_OK;
}

int fvlb_mlp_count(fvlb_mlp_t m, long* count) {
  if (!m || !count) return mfail(m, FVLB_EINVAL, "fvlb_mlp_count: NULL argument");
  *count = (long)m->count;
  return FVLB_OK;
}

int fvlb_mlp_get_pairs(fvlb_mlp_t m, float* x, float* t, long n) {
  if (!m || !x || !t || n < 0 || n > m->count) return mfail(m, FVLB_EINVAL, "fvlb_mlp_get_pairs: bad arguments");
  cudaError_t e = cudaMemcpyAsync(x, m->X, sizeof(float) * m->IN * n, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(t, m->T, sizeof(float) * m->OUT * n, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, cudaGetErrorString(e));
  return FVLB_OK;
}

int fvlb_mlp_train(fvlb_mlp_t m, long steps, int batch, double lr, double* last_loss) {
  if (!m) return set_global_error(FVLB_EINVAL, "NULL mlp");
  if (steps < 0 || batch < kTB || batch % kTB || batch / kTB > kMaxBatches || !(lr > 0))
    return mfail(m, FVLB_EINVAL, "fvlb_mlp_train: batch must be a multiple of 64 (<= 262144), lr > 0");
  if (m->count < 1) return mfail(m, FVLB_ESTATE, "fvlb_mlp_train: no training pairs");
  const int nblocks = grad_blocks(batch);
  cudaError_t e = cudaSuccess;
  for (long s = 0; s < steps && e == cudaSuccess; ++s) {
    m->adam_t += 1;
    e = launch_grad(m, m->X, m->T, m->count, batch, (int)(m->adam_t & 0x7fffffff));
    if (e != cudaSuccess) break;
    const float bc1 = 1.f - std::pow(0.9f, (float)m->adam_t), bc2 = 1.f - std::pow(0.999f, (float)m->adam_t);
    k_mlp_update<<<(m->NP + 31) / 32, kUpdT, 0, m->stream>>>(
        m->prm, m->mo, m->ve, m->part, m->part_loss, nblocks, m->NP, nullptr, m->loss,
        1.0 / ((double)batch * m->OUT), 1, (float)lr, bc1, bc2);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = repack(m);
  if (e == cudaSuccess && last_loss)
    e = cudaMemcpyAsync(last_loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, std::string("fvlb_mlp_train: ") + cudaGetErrorString(e));
  return FVLB_OK;
}

int fvlb_mlp_grad(fvlb_mlp_t m, const float* x, const float* t, long n, float* grad, double* loss) {
  if (!m || !x || !t || !grad || n < 1) return mfail(m, FVLB_EINVAL, "fvlb_mlp_grad: bad arguments");
  if ((n + kTB - 1) / kTB > kMaxBatches) return mfail(m, FVLB_EINVAL, "fvlb_mlp_grad: too many samples");
  float* dx = stage_take(m, (size_t)(m->IN + m->OUT) * (size_t)n);
  if (!dx) return mfail(m, FVLB_ENOMEM, "fvlb_mlp_grad: device allocation failed");
  float* dt = dx + (size_t)m->IN * n;
  cudaError_t e = cudaMemcpyAsync(dx, x, sizeof(float) * m->IN * n, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dt, t, sizeof(float) * m->OUT * n, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = launch_grad(m, dx, dt, n, n, -1);
  if (e == cudaSuccess) {
    k_mlp_update<<<(m->NP + 31) / 32, kUpdT, 0, m->stream>>>(
        m->prm, m->mo, m->ve, m->part, m->part_loss, grad_blocks(n), m->NP, m->grad, m->loss,
        1.0 / ((double)n * m->OUT), 0, 0.f, 1.f, 1.f);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(grad, m->grad, sizeof(float) * m->NP, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  else cudaStreamSynchronize(m->stream);
  stage_give(m, dx);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, std::string("fvlb_mlp_grad: ") + cudaGetErrorString(e));
  return FVLB_OK;
}

int fvlb_mlp_infer(fvlb_mlp_t m, const float* x, long n, float* y) {
  if (!m || !x || !y || n < 1) return mfail(m, FVLB_EINVAL, "fvlb_mlp_infer: bad arguments");
  float* dx = stage_take(m, (size_t)(m->IN + m->OUT) * (size_t)n);
  if (!dx) return mfail(m, FVLB_ENOMEM, "fvlb_mlp_infer: device allocation failed");
  float* dy = dx + (size_t)m->IN * n;
  cudaError_t e = cudaMemcpyAsync(dx, x, sizeof(float) * m->IN * n, cudaMemcpyHostToDevice, m->stream);
  const int blocks = (int)std::min<long long>((n + 127) / 128, 4096);
  if (e == cudaSuccess) {
    if (m->D == 2) k_mlp_infer<8, 3><<<blocks, 128, 0, m->stream>>>(m->packed, dx, n, dy);
    else k_mlp_infer<15, 6><<<blocks, 128, 0, m->stream>>>(m->packed, dx, n, dy);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(y, dy, sizeof(float) * m->OUT * n, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  else cudaStreamSynchronize(m->stream);
  stage_give(m, dx);
  if (e != cudaSuccess) return mfail(m, FVLB_ECUDA, std::string("fvlb_mlp_infer: ") + cudaGetErrorString(e));
  return FVLB_OK;
}

const char* fvlb_mlp_last_error(fvlb_mlp_t m) {
  if (!m) return fvlb_last_error(nullptr);
  return m->err.c_str();
}

int fvlb_mlp_destroy(fvlb_mlp_t m) {
  if (!m) return FVLB_OK;
  if (m->stream) cudaStreamSynchronize(m->stream);
  for (void* p : m->owned) {
    if (m->free_) m->free_(p, m->actx);
    else cudaFree(p);
  }
  m->owned.clear();
  if (m->stream) cudaStreamDestroy(m->stream);
  delete m;
  return FVLB_OK;
}

}  // extern "C"
