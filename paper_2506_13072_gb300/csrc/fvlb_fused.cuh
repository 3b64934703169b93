// fvlb_fused.cuh -- the fused step: one launch per time step (arXiv
// 2506.13072, Sec. 2.2-2.3), and the batched step built on the
// same tile routine.  Included by fvlb_kernels.cuh.
#pragma once

#include <type_traits>

namespace fvlb {

// ---------------------------------------------------------------------------
// Fused step.
//
// Tile: a block owns 32 GX consecutive x-nodes of one row (3D: of one y) and
// marches along the slowest axis (2D: y, 3D: z) over a chunk of `mchunk`
// planes.  KG threads in KG warps update a node: thread kg collides and
// pushes the KC = C / KG stress components kg KC ... and its share of the
// flow populations.  With KG = 1 everything that components share (velocity
// gradient, pressure, c_i.u, destinations) is formed once per node and A - I
// stays in registers; KG > 1 repeats that part, exchanges A - I and the
// pressure sums through shared memory, and has KG times the warps, each with
// 1 / KG of the serial work.  NFW fill warps keep the velocity ring and issue
// the copies.
//
// What bounds it: HBM in D3Q19 and D2Q9 FP32 (each population read and
// written once); instruction issue with 16-bit storage; the FP64 pipe in
// FP64, where the operation count matters, and that all four quarters of an
// SM (each with its own share of the pipe) have collision warps.
//
// Stage: the populations, chi (and the 16-bit forms' FP32 arrays) of the
// next planes, NST buffers deep, copied by bulk tensor copies (TMA) of whole
// array groups: one box for all stress rows, one for the flow rows, one for
// chi (two more for the 16-bit forms), completed on one mbarrier per buffer.
// A copy must start on a 16-byte boundary; PADDED tiles (row starts at any
// node) round the start down and copy 16 bytes more per row.
//
// Velocity gradient: the same-step velocity of the tile and a one-node halo
// sits in a four-plane shared-memory ring (planes m-1 .. m+2).  The fill
// warps compute plane m+2 from its populations (loaded one plane ahead, held
// in registers across the barrier) while the collision warps update plane m;
// halo velocities are recomputed through L2, so blocks never wait on each
// other.  One barrier per plane:
//   A(m)  plane m+1 of the ring is written and every warp is done with plane
//         m-1, so between A(m) and A(m+1) the fill warps may overwrite the
//         ring slot of plane m-2 (with plane m+2) and refill the stage buffer
//         of plane m-1.
// ---------------------------------------------------------------------------

// Velocity of a ring slot: the D components in one 16-byte (FP32) or
// 32-byte (FP64) record (3D: and |u|^2), so a slot is read and written with
// vector shared-memory accesses.
template <class R, int D>
struct alignas(sizeof(R) * (D == 3 ? 4 : 2)) Vel {
  R v[D == 3 ? 4 : 2];
};

// A kernel's MINB: the resident blocks per SM its registers and stage buffers
// are budgeted for, plus 100 times the most stage buffers where that is not
// three.
__host__ __device__ constexpr int blocks_of(int minb) { return minb % 100; }
__host__ __device__ constexpr int stages_of(int minb) { return minb >= 100 ? minb / 100 : 3; }

template <class L, class S, int GX, int KG, bool CL = false>
struct FusedShape {
  static_assert(L::C % KG == 0, "whole components per thread");
  static constexpr int NCW = GX * KG;             // collision warps
  static constexpr int TXS = GX * 32;             // tile extent along x
  static constexpr int EX = TXS + 2;
  static constexpr int EY = (L::D == 3) ? 3 : 1;
  static constexpr int NE = EX * EY;              // ring slots per plane
  // 16-bit storage: a fill thread takes two x-neighbouring nodes (one 4-byte
  // load per population) where nx is even; otherwise one slot per thread
  static constexpr bool PAIRS = sizeof(S) == 2;
  static constexpr int PX = (EX + 2) / 2;         // pairs of a ring row
  static constexpr int NPR = EY * PX;
  // Fill warps: one slot (or pair) per thread.  The learned closure in 3D
  // has four with two slots each: its planes take longer, and 256 threads at
  // two blocks per SM leave 128 registers, without which the network spills
  // (128^3, us per step: four 488, five 504, seven at 80 registers 521).
  static constexpr int NFW = CL && L::D == 3 ? 4 : ((PAIRS ? NPR : NE) + 31) / 32;
  static constexpr int SPF = (NE + NFW * 32 - 1) / (NFW * 32);  // slots per fill thread
  static constexpr int NT = (NCW + NFW) * 32;     // threads
};

// Shared memory of the learned closure in a tile: the packed network, and
// the FP16 input rows, FP32 output rows and chosen chi of each group of 32
// nodes.
template <int GX, int C>
struct ClosureSmem {
  MlpPacked P;
  __half X[GX][32][24];
  float Y[GX][32][8];
  float chi[C][GX * 32];
};
struct NoClosureSmem {
  int unused;
};

template <class L, class S, int GX, int KG, int MINB, bool PADDED, bool CL>
struct TileCfg {
  using R = RT<S>;
  using X = typename Store<S>::X;
  using Sh = FusedShape<L, S, GX, KG, CL>;
  static constexpr int D = L::D, Q = L::Q, C = L::C;
  static constexpr bool V2 = Store<S>::V2;
  static constexpr int H0 = V2 ? 1 : 0;           // first staged stress direction
  static constexpr int EPC = 16 / (int)sizeof(S); // elements per 16 bytes
  static constexpr int BX = Sh::TXS + (PADDED ? EPC : 0);  // stage columns
  // every part starts on a 128-byte boundary, as a bulk tensor copy requires
  struct Stage0 {
    alignas(128) S h[C][Q - H0][BX];
    alignas(128) S f[Q][BX];
    alignas(128) X chi[C][BX];
  };
  struct StageV2 : Stage0 {
    alignas(128) float h0[C][BX];                 // FP32 rest stress populations
    alignas(128) float U[D][BX];                  // stored velocity
  };
  using Stage = typename std::conditional<V2, StageV2, Stage0>::type;
  static constexpr unsigned kBytes =              // of one buffer's copies
      (unsigned)(BX * ((C * (Q - H0) + Q) * (int)sizeof(S) + C * (int)sizeof(X) +
                       (V2 ? (C + D) * 4 : 0)));
  using CLS = typename std::conditional<CL, ClosureSmem<GX, C>, NoClosureSmem>::type;
  // Exchange of a node's A - I and partial pressure sums between its threads:
  // thread kg's KC of each.  A record of 2 C values (FP32 3D: 48 bytes) puts
  // eight neighbouring nodes' 16-byte pieces in different banks; the records
  // of 16 values that this replaces cost 28 % of a 16-bit step's shared-memory
  // wavefronts (us per step: 128^3 FP16 353 / 296, 256^3 FP32 2943 / 2901)
  struct alignas(16) Exchange {
    R v[KG][2 * (C / KG)];
  };
  static constexpr int NEX = KG > 1 ? Sh::TXS : 1;
  // MINB blocks per SM share 227 KB (1 KB per block is the system's)
  static constexpr size_t kLimit = (size_t)(227 / blocks_of(MINB) - 1) * 1024;
  static constexpr size_t kOther = sizeof(Vel<R, D>) * 4 * Sh::NE +
                                   sizeof(Exchange) * NEX + sizeof(CLS) + 256;
  // stage buffers: what fits, up to stages_of(MINB)
  static constexpr int NST =
      stages_of(MINB) > 3 && kOther + 4 * sizeof(Stage) <= kLimit
          ? 4
          : (kOther + 3 * sizeof(Stage) <= kLimit ? 3 : 2);
  struct Smem {
    alignas(16) Vel<R, D> ring[4][Sh::NE];        // velocity of planes m-1 .. m+2
    Exchange ex[NEX];
    alignas(16) CLS cls;                          // learned closure (CL only)
    uint64_t bar[NST];                            // bulk-copy barriers of the stage buffers
    alignas(128) Stage stage[NST];
  };
  static_assert(sizeof(Smem) <= kLimit, "MINB blocks must fit an SM");
};

// Where a warp stands in the cycle of stage buffers.
struct StagePos {
  int st = 0;
  unsigned par = 0;
  template <int NST>
  __device__ __forceinline__ void next() {
    if (++st == NST) {
      st = 0;
      par ^= 1u;
    }
  }
};

// One tile of the fused step: tile (bx, by) of the plane, chunk bz of the
// march axis.  Called by k_step_fused and by the batched kernel, once per
// block.  `tma`:
// the stage is filled by bulk tensor copies through *tm (the barriers are
// initialised), otherwise each lane copies its own node.  FENCE_MAPS: *tm is
// in global memory.
template <class L, class S, int GX, int KG, int MINB, bool WALLS, bool PADDED, bool CL, bool ORIG,
          bool FENCE_MAPS = false>
__device__ __forceinline__ void fused_tile(
    typename TileCfg<L, S, GX, KG, MINB, PADDED, CL>::Smem& sm, const Grid& g, const Phys<RT<S>>& ph,
    const Bufs<S>& b, int mchunk, int bx, int by, int bz, const StageMaps* tm, bool tma,
    StagePos& pos) {
  using R = RT<S>;
  using X = typename Store<S>::X;
  using Sh = FusedShape<L, S, GX, KG, CL>;
  using Cfg = TileCfg<L, S, GX, KG, MINB, PADDED, CL>;
  constexpr int D = L::D, Q = L::Q, C = L::C;
  constexpr int NCW = Sh::NCW, TXS = Sh::TXS, EX = Sh::EX, NE = Sh::NE;
  constexpr int NFW = Sh::NFW, SPF = Sh::SPF, NST = Cfg::NST, H0 = Cfg::H0;
  constexpr bool V2 = Cfg::V2;
  constexpr bool F64 = std::is_same<R, double>::value;
  // FP32 storage: the rest stress population from the post-collision zeroth
  // moment (see the collision)
  constexpr bool RS = std::is_same<S, float>::value;
  static_assert(!CL || std::is_same<R, float>::value, "the learned closure runs in FP32");
  auto& ring = sm.ring;

  const int nx = g.nx, ny = g.ny;
  const int nm = (D == 3) ? g.nz : g.ny;
  const bool wall_x = WALLS && (g.walls & 1);
  const bool wall_y = WALLS && (D == 3) && ((g.walls >> 1) & 1);
  const bool wall_m = WALLS && ((g.walls >> (D - 1)) & 1);
  const int x0 = bx * TXS;
  const int y = (D == 3) ? by : 0;
  const int m0 = bz * mchunk;
  const int m1 = min(m0 + mchunk, nm);
  const long long P = g.pitch;
  const uint32_t P32 = (uint32_t)P;   // offsets within the arrays are 32-bit (Q * pitch < 2^32)

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  auto slot = [&](int q) { return (q - m0 + 1) & 3; };
  auto plane_of = [&](int q) -> int {  // -1: beyond a wall
    // (planes -1 .. nm are used: one wrap at most)
    if (q < 0) return wall_m ? -1 : q + nm;
    if (q >= nm) return wall_m ? -1 : q - nm;
    return q;
  };
  // ring slot (ex, ey)'s node, one node outside the tile on each side: none
  // beyond a wall, and none past the slot after the row's last node
  auto ring_node = [&](int ex, int ey, int& gx, int& gy) -> bool {
    gx = x0 + ex - 1;
    gy = (D == 3) ? y + ey - 1 : 0;
    bool has = gx <= nx;
    if (gx < 0 || gx == nx) {
      if (wall_x) has = false;
      gx = gx < 0 ? nx - 1 : 0;
    }
    if (D == 3 && (gy < 0 || gy == ny)) {
      if (wall_y) has = false;
      gy = gy < 0 ? ny - 1 : 0;
    }
    return has;
  };
  auto node_of = [&](int mm, int gx, int gy) -> uint32_t {
    return (D == 3) ? ((uint32_t)mm * (uint32_t)ny + (uint32_t)gy) * (uint32_t)nx + (uint32_t)gx
                    : (uint32_t)mm * (uint32_t)nx + (uint32_t)gx;
  };

  // Velocity of ring slot e of plane q from its momentum sums `mo` (when
  // `ok`), into the ring.
  auto ring_store = [&](int e, bool ok, int mm, int gx, int gy, const R (&mo)[D],
                        const R (&Ub)[D], int q) {
    R u[D];
#pragma unroll
    for (int a = 0; a < D; ++a) u[a] = R(0);
    if (ok) {
      R F[3];
      body_force<L, R>(ph, gx, D == 3 ? gy : mm, F);
      if constexpr (ORIG) {  // the original scheme: + div tau_p of this node
        const uint32_t sf = node_of(mm, gx, gy);
#pragma unroll
        for (int a = 0; a < D; ++a) F[a] += ph.fdiv[(uint32_t)a * P32 + sf];
      }
#pragma unroll
      for (int a = 0; a < D; ++a) {
        // 16-bit forms: u = U + sum_i c_i s_i / KF + F/2 (the velocity part
        // e_i(U) of the stored deviations carries momentum U and no other
        // first moment)
        if constexpr (V2) u[a] = mo[a] * R(1.0f / Store<S>::KF) + Ub[a] + R(0.5) * F[a];
        else u[a] = mo[a] + R(0.5) * F[a];
      }
    }
    Vel<R, D> t;
#pragma unroll
    for (int a = 0; a < D; ++a) t.v[a] = u[a];
    if constexpr (D == 3) {
      // |u|^2, which the 16-bit forms ask for at 18 neighbours
      if constexpr (V2) t.v[3] = __fmaf_rn(u[2], u[2], __fmaf_rn(u[0], u[0], __fmul_rn(u[1], u[1])));
      else t.v[3] = R(0);
    }
    ring[slot(q)][e] = t;
  };
  // the same from raw 16-bit populations: each enters the momentum sums
  // with one mixed-precision add or subtract, the accumulator's sign
  // tracked at compile time (f - v = -(v - f) exactly)
  auto bits_store = [&](int e, bool ok, int mm, int gx, int gy, const unsigned short (&sb)[Q],
                        const R (&Ub)[D], int q) {
    if constexpr (V2) {
      R mo[D];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        R v = R(0);
        bool neg = false;   // v = -(momentum sum) while set
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const int c = cc<L>(i, a);
          if (c == 0) continue;
          if ((c == 1) != neg) {
            v = Store<S>::accb(v, sb[i]);
          } else {
            v = Store<S>::subb(sb[i], v);
            neg = !neg;
          }
        }
        mo[a] = neg ? -v : v;
      }
      ring_store(e, ok, mm, gx, gy, mo, Ub, q);
    }
  };

  // one ring slot's populations: loaded, then turned into its velocity
  struct Held {
    S f[Q];
    R u[D];
  };
  auto slot_load = [&](bool has, int mm, int gx, int gy, Held& v) {
    if (has && mm >= 0) {
      const uint32_t s = node_of(mm, gx, gy);
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        if constexpr (V2) v.f[i] = ld_state(b.f_in + ((uint32_t)i * P32 + s));
        else v.f[i] = b.f_in[(uint32_t)i * P32 + s];
      }
      if constexpr (V2) {
        const float* U = f_ext<L>(b.f_in, P);
#pragma unroll
        for (int a = 0; a < D; ++a) v.u[a] = ld_state(U + ((uint32_t)a * P32 + s));
      }
    }
  };
  auto slot_store = [&](int e, bool has, int mm, int gx, int gy, int q, const Held& v) {
    const bool ok = has && mm >= 0;
    if constexpr (V2) {
      unsigned short hb[Q];
      hb[0] = 0;
#pragma unroll
      for (int i = 1; i < Q; ++i) hb[i] = *reinterpret_cast<const unsigned short*>(&v.f[i]);
      bits_store(e, ok, mm, gx, gy, hb, v.u, q);
    } else {
      R mo[D];
      momentum<L, R>(v.f, mo);
      ring_store(e, ok, mm, gx, gy, mo, mo, q);
    }
  };
  // The first three planes of the ring, by all warps, their loads in flight
  // together (a chunk of one plane spends more on them than on its own plane).
  auto prologue = [&]() {
    constexpr int NPRO = (3 * NE + Sh::NT - 1) / Sh::NT;
    Held v[NPRO];
    int gx[NPRO], gy[NPRO], mm[NPRO];
    bool has[NPRO];
#pragma unroll
    for (int t = 0; t < NPRO; ++t) {
      const int n = tid + t * Sh::NT;
      const int e = n % NE, pq = n / NE;
      has[t] = ring_node(e % EX, e / EX, gx[t], gy[t]) && n < 3 * NE;
      mm[t] = plane_of(m0 - 1 + pq);
      slot_load(has[t], mm[t], gx[t], gy[t], v[t]);
    }
#pragma unroll
    for (int t = 0; t < NPRO; ++t) {
      const int n = tid + t * Sh::NT;
      if (n < 3 * NE) slot_store(n % NE, has[t], mm[t], gx[t], gy[t], m0 - 1 + n / NE, v[t]);
    }
  };

  // The first fill thread issues the stage copies of the block.
  StagePos pst = pos;
  if (FENCE_MAPS && tma && tid == NCW * 32) fence_tensor_maps(tm);
  auto produce = [&](int q) {
    if (!tma || tid != NCW * 32 || q >= m1) return;
    auto& W = sm.stage[pst.st];
    uint64_t* bar = &sm.bar[pst.st];
    pst.template next<NST>();
    int s0 = (int)node_of(q, x0, y);
    if constexpr (PADDED) s0 &= ~(Cfg::EPC - 1);
    fence_proxy_async();   // the collision warps' reads of this buffer (ordered by A) first
    mbar_arrive_expect_tx(bar, Cfg::kBytes);
    tma_load_2d(&W.f[0][0], &tm->f, s0, 0, bar);
    if constexpr (V2) {
      tma_load_2d(&W.U[0][0], &tm->u, s0, 0, bar);
      tma_load_2d(&W.h0[0][0], &tm->e0, s0, 0, bar);
      tma_load_3d(&W.h[0][0][0], &tm->h, s0, 1, 0, bar);
    } else {
      tma_load_2d(&W.h[0][0][0], &tm->h, s0, 0, bar);
    }
    tma_load_2d(&W.chi[0][0], &tm->x, s0, 0, bar);
  };
  produce(m0);
#pragma unroll
  for (int q = 1; q < NST - 1; ++q) produce(m0 + q);
  prologue();

  if (warp >= NCW) {
    // ---------------- fill warps ---------------------------------------------
    if constexpr (Sh::PAIRS) {
      // Even nx and no walls across x: thread pp takes the node pair (x even,
      // x + 1) px of ring row ey, ring slots 2 px - 1 and 2 px (those in the
      // row): half the loads and held registers of one slot per load.
      if ((nx & 1) == 0 && !wall_x) {
        const int pp = tid - NCW * 32;
        const int ey = pp / Sh::PX, px = pp - ey * Sh::PX;
        const bool pact = pp < Sh::NPR;
        int gx0 = x0 + 2 * px - 2, gy;              // even
        bool has = pact && gx0 <= nx;
        if (gx0 < 0) gx0 += nx;                     // periodic in x (nx even: stays even)
        if (gx0 == nx) gx0 = 0;
        int gxn;
        has = ring_node(1, ey, gxn, gy) && has;     // (the row's gy)
        const int ea = ey * EX + 2 * px - 1;        // slot of node gx0 (px > 0)
        const bool sa = pact && px > 0, sb = pact && 2 * px < EX;
        struct Pair {
          uint32_t f[Q];
          float2 u[D];
        };
        auto pload = [&](int mm, Pair& v) {
          if (has && mm >= 0) {
            const uint32_t s0 = node_of(mm, gx0, gy);
            const uint32_t* fw = reinterpret_cast<const uint32_t*>(b.f_in);
            const float* U = f_ext<L>(b.f_in, P);
#pragma unroll
            for (int i = 1; i < Q; ++i) v.f[i] = ld_state(fw + (((uint32_t)i * P32 + s0) >> 1));
#pragma unroll
            for (int a = 0; a < D; ++a)
              v.u[a] = ld_state(reinterpret_cast<const float2*>(U + ((uint32_t)a * P32 + s0)));
          }
        };
        auto pstore = [&](int mm, int q, const Pair& v) {
          const bool ok = has && mm >= 0;
#pragma unroll
          for (int n = 0; n < 2; ++n) {
            if (n == 0 ? !sa : !sb) continue;
            unsigned short hb[Q];
            R Ub[D];
            hb[0] = 0;
#pragma unroll
            for (int i = 1; i < Q; ++i) hb[i] = (unsigned short)(n ? v.f[i] >> 16 : v.f[i] & 0xffffu);
#pragma unroll
            for (int a = 0; a < D; ++a) Ub[a] = n ? v.u[a].y : v.u[a].x;
            bits_store(ea + n, ok, mm, gx0 + n, gy, hb, Ub, q);
          }
        };
        Pair v;
        int mq = plane_of(m0 + 2);
        if (m0 + 2 <= m1) pload(mq, v);
        for (int m = m0; m < m1; ++m) {
          __syncthreads();               // A(m)
          produce(m + NST - 1);
          if (m + 2 <= m1) {             // overlaps the collision of plane m
            pstore(mq, m + 2, v);
            mq = plane_of(m + 3);
            if (m + 3 <= m1) pload(mq, v);
          }
        }
        pos = pst;
        return;
      }
    }
    // One ring slot per load: thread t of the fill warps takes the slots
    // t + j 32 NFW, j < SPF, whose nodes are fixed for the whole tile.
    const int e0 = tid - NCW * 32;
    int sgx[SPF], sgy[SPF];
    bool shas[SPF];
#pragma unroll
    for (int t = 0; t < SPF; ++t) {
      const int e = e0 + t * NFW * 32;
      shas[t] = ring_node(e % EX, e / EX, sgx[t], sgy[t]) && e < NE;
    }
    auto fload = [&](int t, int mm, Held& v) { slot_load(shas[t], mm, sgx[t], sgy[t], v); };
    auto fstore = [&](int t, int mm, int q, const Held& v) {
      const int e = e0 + t * NFW * 32;
      if (e < NE) slot_store(e, shas[t], mm, sgx[t], sgy[t], q, v);
    };
    Held v[SPF];
    int mq = plane_of(m0 + 2);
    if (m0 + 2 <= m1) {
#pragma unroll
      for (int t = 0; t < SPF; ++t) fload(t, mq, v[t]);
    }
    for (int m = m0; m < m1; ++m) {
      __syncthreads();               // A(m)
      produce(m + NST - 1);
      if (m + 2 <= m1) {             // overlaps the collision of plane m
#pragma unroll
        for (int t = 0; t < SPF; ++t) fstore(t, mq, m + 2, v[t]);
        mq = plane_of(m + 3);
        if (m + 3 <= m1) {
#pragma unroll
          for (int t = 0; t < SPF; ++t) fload(t, mq, v[t]);
        }
      }
    }
    pos = pst;
    return;
  }

  // ---------------- collision warps ------------------------------------------
  constexpr int KC = C / KG;            // components of a thread
  const int grp = warp / KG;
  const int kg = KG > 1 ? warp - grp * KG : 0;
  const int tx = grp * 32 + lane;       // node of the tile
  const int x = x0 + tx;
  const bool active = x < nx;
  const int eo = (D == 3) ? EX + tx + 1 : tx + 1;   // own ring slot
  // neighbour offsets: x and y are constant over the march
  const int strm = (D == 3) ? nx * ny : nx;
  int sp[3], sn[3];                     // offset of the neighbour at +1 / -1 along an axis
  sp[0] = (x == nx - 1) ? -(nx - 1) : 1;
  sn[0] = (x == 0) ? nx - 1 : -1;
  sp[1] = (D == 3) ? ((y == ny - 1) ? -(ny - 1) * nx : nx) : 0;
  sn[1] = (D == 3) ? ((y == 0) ? (ny - 1) * nx : -nx) : 0;
  // at a wall on the upper / lower side of an axis
  bool hi[3] = {wall_x && x == nx - 1, wall_y && y == ny - 1, false};
  bool lo[3] = {wall_x && x == 0, wall_y && y == 0, false};
  constexpr int AM = D - 1;             // march axis
  // the group's KG warps
  auto group_sync = [&]() {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(KG * 32) : "memory");
  };
  // FP32 arithmetic fixes the order and the fused multiply-adds of the
  // collision that its long-run accuracy was established with, whatever the
  // compiler would contract: another rounding of a slow flow's pressure
  // differs by as much as its error, and with 16-bit storage one flipped
  // rounding changes all later ones.  FP64 shares more between directions and
  // leaves the contraction to the compiler.
  constexpr bool ORD = !F64;

  const R om = ph.inv_tau_h;
  const R keep = R(1) - om;

  int cl_used = 0;                      // learned closure: this warp's nodes on the network
#pragma unroll 1
  for (int m = m0; m < m1; ++m) {
    const int st = pos.st;
    const unsigned par = pos.par;
    if (tma) pos.template next<NST>();
    __syncthreads();                    // A(m)
    if (KG == 1 && !CL && !active) continue;
    auto& W = sm.stage[st];
    const uint32_t s = node_of(m, x, y);
    int col = tx;
    if (tma) {
      if constexpr (PADDED) col += (int)(node_of(m, 0, y) & (uint32_t)(Cfg::EPC - 1));
      mbar_wait(&sm.bar[st], par, ph.err);
    } else {
      // no bulk copies: the lanes copy their own nodes into their columns
      if (active && kg == 0) {
#pragma unroll 1
        for (int q = 0; q < C; ++q) {
#pragma unroll 1
          for (int i = H0; i < Q; ++i) W.h[q][i - H0][tx] = b.h_in[(long long)(q * Q + i) * P + s];
          W.chi[q][tx] = b.chi[(uint32_t)q * P32 + s];
          if constexpr (V2) W.h0[q][tx] = h_ext<L>(b.h_in, P)[(uint32_t)q * P32 + s];
        }
#pragma unroll 1
        for (int i = 0; i < Q; ++i) W.f[i][tx] = b.f_in[(uint32_t)i * P32 + s];
        if constexpr (V2) {
#pragma unroll 1
          for (int a = 0; a < D; ++a) W.U[a][tx] = f_ext<L>(b.f_in, P)[(uint32_t)a * P32 + s];
        }
      }
      if constexpr (KG > 1) group_sync();
    }
    if (WALLS) {
      hi[AM] = wall_m && m == nm - 1;
      lo[AM] = wall_m && m == 0;
    }
    sp[AM] = (m == nm - 1) ? -(nm - 1) * strm : strm;
    sn[AM] = (m == 0) ? (nm - 1) * strm : -strm;
    const int rm = slot(m - 1), rc = slot(m), rp = slot(m + 1);
    // component q of this thread: k = kg KC + q
    const auto& Wh = W.h;
    const int k0 = kg * KC;

    R Ad[C];                            // A - I = sum_i h' (Sec. 2.3)
    R own[KC];                          // of this thread's components
    R sumf = R(0);                      // sum of f_i, i != 0
    if (active || KG == 1) {
#pragma unroll
      for (int q = 0; q < KC; ++q) {
        if constexpr (V2) own[q] = W.h0[k0 + q][col];
        else own[q] = Store<S>::cvt(Wh[k0 + q][0][col]);
      }
#pragma unroll
      for (int i = 1; i < Q; ++i) {
#pragma unroll
        for (int q = 0; q < KC; ++q) own[q] = Store<S>::acc(own[q], Wh[k0 + q][i - H0][col]);
      }
      // partial pressure sums: f_i with i = k (mod C), i != 0
      R pf[KC];
#pragma unroll
      for (int q = 0; q < KC; ++q) {
        pf[q] = R(0);
#pragma unroll
        for (int j = 0; j < (Q + C - 1) / C; ++j) {
          if (KG == 1) {
            const int i = q + j * C;
            if (i == 0 || i >= Q) continue;
            pf[q] = Store<S>::acc(pf[q], W.f[i][col]);
          } else {
            const int i = k0 + q + j * C;
            if (i != 0 && i < Q) pf[q] = Store<S>::acc(pf[q], W.f[i][col]);
          }
        }
        if constexpr (V2) pf[q] *= R(1.0f / Store<S>::KF);
      }
      if constexpr (KG == 1) {
#pragma unroll
        for (int k = 0; k < C; ++k) {
          Ad[k] = own[k];
          sumf += pf[k];
        }
      } else {
        auto& ex = sm.ex[tx].v[kg];
#pragma unroll
        for (int q = 0; q < KC; ++q) {
          ex[q] = own[q];
          ex[KC + q] = pf[q];
        }
      }
    }
    if constexpr (KG > 1) {
      group_sync();
      if (!CL && !active) continue;
      const auto& ex = sm.ex[tx];
#pragma unroll
      for (int k = 0; k < C; ++k) {
        Ad[k] = ex.v[k / KC][k % KC];
        sumf += ex.v[k / KC][KC + k % KC];
      }
    }

    // --- velocity and its gradient: G_rb = 2 d_r u_b, central, or through the
    // wall point half a node away (u = 0 there): d = u0 + u1 / 3 ---------------
    R u[D], G[D][D];
    {
      const Vel<R, D> t = ring[rc][eo];
#pragma unroll
      for (int a = 0; a < D; ++a) u[a] = t.v[a];
    }
    R uu = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) uu += u[a] * u[a];
#pragma unroll
    for (int r = 0; r < D; ++r) {
      const int ep = r == AM ? eo : (r == 0 ? eo + 1 : eo + EX);
      const int em = r == AM ? eo : (r == 0 ? eo - 1 : eo - EX);
      const Vel<R, D> vp = ring[r == AM ? rp : rc][ep], vm = ring[r == AM ? rm : rc][em];
#pragma unroll
      for (int a = 0; a < D; ++a) G[r][a] = vp.v[a] - vm.v[a];
      if (WALLS && (lo[r] || hi[r])) {
#pragma unroll
        for (int a = 0; a < D; ++a)
          G[r][a] = lo[r] ? R(2) * (u[a] + vp.v[a] * R(1.0 / 3.0))
                          : R(-2) * (u[a] + vm.v[a] * R(1.0 / 3.0));
      }
    }
    // --- stress source (Sec. 2.3): chi_ab = -P_ab / lambda
    //     + sum_r (A_ar d_r u_b + d_r u_a A_rb), component k ---------------------
    auto source = [&](auto KI) -> R {
      constexpr int k = decltype(KI)::value;
      constexpr int a = L::ca(k), bb = L::cb(k);
      if constexpr (ORD) {
        R v = -(ph.model ? relax_part<L, R>(k, Ad, ph.model, ph.mpar) : Ad[k]) * ph.inv_lam;
#pragma unroll
        for (int r = 0; r < D; ++r) {
          const R dua = R(0.5) * G[r][a], dub = R(0.5) * G[r][bb];
          const R Aar = Ad[sym<L>(a, r)] + (a == r ? R(1) : R(0));
          const R Arb = Ad[sym<L>(r, bb)] + (r == bb ? R(1) : R(0));
          v += Aar * dub + dua * Arb;
        }
        return v;
      } else {
        R v = R(0);
#pragma unroll
        for (int r = 0; r < D; ++r) {
          const R Aar = Ad[sym<L>(a, r)] + (a == r ? R(1) : R(0));
          v = r == 0 ? Aar * G[r][bb] : v + Aar * G[r][bb];
          if (a != bb) v += G[r][a] * (Ad[sym<L>(r, bb)] + (r == bb ? R(1) : R(0)));
        }
        if (a != bb) v *= R(0.5);
        return v - (ph.model ? relax_part<L, R>(k, Ad, ph.model, ph.mpar) : Ad[k]) * ph.inv_lam;
      }
    };
    R chi[KC];                          // of this thread's components
    auto sources = [&](auto K0) {
      constexpr int kb = decltype(K0)::value;
      chi[0] = source(std::integral_constant<int, kb>{});
      if constexpr (KC > 1) chi[1] = source(std::integral_constant<int, kb + (KC > 1 ? 1 : 0)>{});
      if constexpr (KC > 2) chi[2] = source(std::integral_constant<int, kb + (KC > 2 ? 2 : 0)>{});
      if constexpr (KC > 3) {
        chi[3] = source(std::integral_constant<int, kb + (KC > 3 ? 3 : 0)>{});
        chi[4] = source(std::integral_constant<int, kb + (KC > 3 ? 4 : 0)>{});
        chi[5] = source(std::integral_constant<int, kb + (KC > 3 ? 5 : 0)>{});
      }
    };
    static_assert(KC == 1 || KC == 2 || KC == 3 || KC == 6, "components of a thread");

    // ---- learned closure: the group's warps evaluate the network, each for
    // its share of the two 16-node tiles; a node keeps the analytic source
    // where the network is off -----------------------------------------------
    if constexpr (CL) {
      auto& cls = sm.cls;
      static_assert(KG <= 2, "two m16 tiles per group");
      const bool mine = KG == 1 || (lane >> 4) == kg;
      if (mine) {
        float xin[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) xin[q] = 0.f;
        if (active) {
          int q = 0;
#pragma unroll
          for (int a = 0; a < D; ++a)
#pragma unroll
            for (int bq = 0; bq < D; ++bq) xin[q++] = float(ph.lam * (R(0.5) * G[a][bq]));
#pragma unroll
          for (int c = 0; c < C; ++c) xin[q++] = float(Ad[c]);
          if (D == 2) xin[q++] = float(ph.inv_lam);
        }
#pragma unroll
        for (int q = 0; q < 16; q += 2)
          *reinterpret_cast<uint32_t*>(&cls.X[grp][lane][q]) = pack_f16x2(xin[q], xin[q + 1]);
      }
      __syncwarp();
      if constexpr (KG == 1) mlp_warp(cls.P, cls.X[grp], cls.Y[grp]);
      else mlp_tile(cls.P, cls.X[grp], cls.Y[grp], kg);
      __syncwarp();
      bool used = false;
      if (active && mine) {
        float num = 0.f, den = 0.f, an[C], nn[C];
        auto term = [&](auto KI) {
          constexpr int c = decltype(KI)::value;
          an[c] = float(source(KI));
          nn[c] = cls.Y[grp][lane][c] * float(ph.inv_lam);
          const float dd = nn[c] - an[c];
          num += dd * dd;
          den += an[c] * an[c];
        };
        term(std::integral_constant<int, 0>{});
        term(std::integral_constant<int, 1>{});
        term(std::integral_constant<int, 2>{});
        if constexpr (C > 3) {
          term(std::integral_constant<int, (C > 3 ? 3 : 0)>{});
          term(std::integral_constant<int, (C > 3 ? 4 : 0)>{});
          term(std::integral_constant<int, (C > 3 ? 5 : 0)>{});
        }
        // per-node residual check: fall back to the analytic source
        used = num <= ph.cl_tol2 * den;
#pragma unroll
        for (int c = 0; c < C; ++c) cls.chi[c][tx] = used ? nn[c] : an[c];
      }
      cl_used += __popc(__ballot_sync(0xffffffffu, used));
      if constexpr (KG > 1) group_sync();
      else __syncwarp();
      if (!active) continue;
#pragma unroll
      for (int q = 0; q < KC; ++q) chi[q] = R(cls.chi[k0 + q][tx]);
    } else {
      if constexpr (KG == 1) {
        sources(std::integral_constant<int, 0>{});
      } else {
        if (kg == 0) sources(std::integral_constant<int, 0>{});
        else if (KG == 2 || kg == 1) sources(std::integral_constant<int, KC>{});
        else sources(std::integral_constant<int, (KG > 2 ? 2 * KC : 0)>{});
      }
    }

    // The collision reads the stress populations again from the stage: held
    // in registers across the source they would spill.
    if constexpr (D == 3 || V2) asm volatile("" ::: "memory");

    // --- stress collision: h* = (1 - 1/tau_h) h + w_i [alpha + c_i.u beta] with
    // alpha = (A-I)_k / tau_h + src and beta = 3 (A_k / tau_h + kh src);
    // src = chi + 0.5 (chi^n - chi^{n-1}) -------------------------------------
    R wax[KC], wdg[KC];                 // w_i alpha of the axis and the diagonal directions
    R bax[KC], bdg[ORD ? KC : 1];       // w_i beta (not ORD: beta)
    R alf[ORD && D == 2 ? KC : 1];      // alpha
    R rest[KC];                         // towards the rest population
    R h0p[V2 ? KC : 1];                 // 16-bit forms: it, before the rounding residuals
    constexpr double kWx = weight_sum_excess<L, R>();
#pragma unroll
    for (int q = 0; q < KC; ++q) {
      const int k = k0 + q;
      const bool dg = D == 2 ? k != 1 : k < 3;     // a diagonal component
      const R old = ph.first ? chi[q] : R(W.chi[k][col]);
      b.chi[(uint32_t)k * P32 + s] = X(chi[q]);
      const R src = R(1.5) * chi[q] - R(0.5) * old;
      R alpha;
      if constexpr (ORD) alpha = __fmaf_rn(om, own[q], src);
      else alpha = om * own[q] + src;
      const R A_k = own[q] + (dg ? R(1) : R(0));
      wax[q] = R(L::w(1)) * alpha;
      wdg[q] = R(L::w(Q - 1)) * alpha;
      if constexpr (ORD) {
        const R beta = R(3) * __fmaf_rn(om, A_k, __fmul_rn(ph.kh, src));
        if constexpr (D == 2) alf[q] = alpha;
        bax[q] = R(L::w(1)) * beta;
        bdg[q] = R(L::w(Q - 1)) * beta;
      } else {
        bax[q] = (R(3) * om) * A_k + (R(3) * ph.kh) * src;
      }
      // The rest population (which stays at this node) keeps the node's
      // stored populations summing to the post-collision zeroth moment
      // (A - I)_k + src (sum_i w_i = 1, sum_i w_i c_i = 0):
      //  - FP32: it is that moment minus the other populations' sum, so
      //    neither the rounded weights (whose sum exceeds one by 7e-9 in
      //    2D, 1.5e-8 in 3D) nor the rounding of the collision moves A;
      //  - 16-bit forms: it takes the rounding residuals of the 16-bit
      //    stores, less the weights' excess times alpha.
      if constexpr (RS) {
        rest[q] = R(0);
        own[q] += src;                             // the zeroth moment, for the end
      } else if constexpr (V2) {
        rest[q] = R(0);
        h0p[q] = __fmaf_rn(-R(kWx), alpha,
                           __fmaf_rn(keep, W.h0[k][col], __fmul_rn(R(L::w(0)), alpha)));
      } else {
        rest[q] = keep * Store<S>::cvt(Wh[k][0][col]) + R(L::w(0)) * alpha;
      }
    }

    // --- flow collision inputs (Sec. 2.2) -------------------------------------
    R F[3];
    body_force<L, R>(ph, x, D == 3 ? y : m, F);
    if constexpr (ORIG) {  // the original scheme: + div tau_p of this node, no f^B
#pragma unroll
      for (int a = 0; a < D; ++a) F[a] += ph.fdiv[(uint32_t)a * P32 + s];
    }
    R Fu = R(0);
#pragma unroll
    for (int a = 0; a < D; ++a) Fu += F[a] * u[a];
    // 16-bit forms: the node's stored velocity U is the reference of its
    // flow populations; sum_{i != 0} e_i(U) = 1.5 w_0 |U|^2
    R Us[D] = {};
    R UU = R(0);
    if constexpr (V2) {
#pragma unroll
      for (int a = 0; a < D; ++a) {
        Us[a] = W.U[a][col];
        UU += Us[a] * Us[a];
      }
      sumf = __fmaf_rn(R(1.5 * L::w(0)), UU, sumf);
    }
    const R kB = ORIG ? R(0) : ph.eta_over_lam * ph.inv_tau_f;
    FBTerms<L, R> fb = {};
    if constexpr (!ORD && !ORIG) fb.set(Ad, kB);
    // pressure (Sec. 2.2, Appendix B)
    constexpr double w0 = L::w(0);
    R psum;
    if constexpr (ORD) {
      psum = __fmaf_rn(R(-1.5 * w0), uu, sumf);
      psum = __fmaf_rn(ph.tau_f, __fmul_rn(__fmul_rn(R(-3.0 * w0), ph.kf), Fu), psum);
      psum = __fmaf_rn(ph.tau_f, __fmul_rn(fB_ordered<L>(0, Ad), kB), psum);
    } else {
      psum = sumf + R(-1.5 * w0) * uu + ph.tau_f * (R(-3.0 * w0) * ph.kf * Fu) + ph.tau_f * fb.q0;
    }
    const R p = p_part<L, R>(psum);
    const R itf = ph.inv_tau_f, kf = ph.kf;
    R Fd[D];                              // F (FP64: kf F)
#pragma unroll
    for (int a = 0; a < D; ++a) Fd[a] = F64 ? kf * F[a] : F[a];
    const R kFu = kf * Fu;

    // stochastic rounding: one stream per node and component k, whose draw i is
    // for h_{k,i} and draw Q + j for f_{k + j C}
    const uint32_t hs = Store<S>::sr ? hash32(ph.step) : 0u;
    auto rnd = [&](int k, int n) -> uint32_t {
      return Store<S>::sr ? lcg_at(hash32((s * 8u + (uint32_t)k) * 0x9e3779b9u ^ hs), n) : 0u;
    };
    auto rnd_f = [&](int i) -> uint32_t { return Store<S>::sr ? rnd(i % C, Q + i / C) : 0u; };

    if constexpr (V2) {
      // this node's velocity: the reference of the flow populations it
      // receives for the next step
      if (kg == KG - 1) {
        float* Uo = f_ext<L>(b.f_out, P);
#pragma unroll
        for (int a = 0; a < D; ++a) Uo[(uint32_t)a * P32 + s] = float(u[a]);
      }
    }

    // --- collide and push, a pair (i, j) of opposite directions at a time: the
    // parts even and odd in c_i are shared, and one destination serves f_i and
    // the stress populations of a direction.  cu, cF, cU: c_i.u, c_i.F (FP64:
    // kf c_i.F), c_i.U; fbv: f^B_i; di, dj: destination nodes, through a wall
    // where bi, bj: the own node, direction reversed; ri, rj: ring records of
    // the receiving nodes, from the own one; mine: whether this thread has the
    // pair's flow populations. -----------------------------------------------
    const Vel<R, D>* rown = &ring[rc][eo];
    // 16-bit forms: where a deviation is rounded in the other order (see dev
    // below), in walled grids only: a batch's periodic grids have the bits of
    // the same grid in a handle of its own.  In 2D the two forms say the same;
    // which one compiles better (us a step, first / second): padded rows, 96
    // FP16 grids 200.5 / 207, 517x333 FP16 12.07 / 12.14; aligned rows, 512^2
    // FP16 13.44 / 13.33.
    const bool edge = D == 2 && PADDED
                          ? wall_x || lo[AM] || hi[AM]
                          : g.walls && (wall_x || (D == 3 && (y == 0 || y == ny - 1)) || m == 0 ||
                                        m == nm - 1);
    S* hout = b.h_out + (long long)k0 * Q * P;
    R held[ORD && D == 2 ? KC : 1][2];    // D2Q9: summed in direction order
    auto pair = [&](auto AX, int i, int j, bool mine, R cu, R cF, R cU, R fbv, int di, int dj,
                    bool bi, bool bj, int ri, int rj, auto cdot, auto PH) {
      constexpr bool axis = decltype(AX)::value;
      constexpr int half = decltype(PH)::value;
      constexpr int I0 = axis ? 1 : Q - 1;         // a direction of this class
      const R wi = R(L::w(I0)), lam_i = R(p_coef<L, R>(I0)), w3i = R(w3<L, R>(I0));
      uint32_t oi = (uint32_t)i * P32 + (uint32_t)di, oj = (uint32_t)j * P32 + (uint32_t)dj;
      if (WALLS) {
        oi = bi ? (uint32_t)j * P32 + s : oi;
        oj = bj ? (uint32_t)i * P32 + s : oj;
      }
      const R wcu = wi * cu;
#pragma unroll
      for (int q = 0; q < KC; ++q) {
        const R wa = axis ? wax[q] : wdg[q];
        const R hvi = Store<S>::cvt(Wh[k0 + q][i - H0][col]);
        const R hvj = Store<S>::cvt(Wh[k0 + q][j - H0][col]);
        R pi, pj;
        if constexpr (ORD) {
          const R wb = axis ? bax[q] : bdg[q];
          R xi, xj;
          if constexpr (D == 3) {
            xi = __fmaf_rn(cu, wb, wa);
            xj = __fmaf_rn(-cu, wb, wa);
          } else {
            const R t = __fmul_rn(cu, wb);
            xi = __fmaf_rn(wi, alf[q], t);
            xj = __fmaf_rn(wi, alf[q], -t);
          }
          pi = __fmaf_rn(keep, hvi, xi);
          pj = __fmaf_rn(keep, hvj, xj);
        } else {
          pi = keep * hvi + (wa + wcu * bax[q]);
          pj = keep * hvj + (wa - wcu * bax[q]);
        }
        S* out = hout + (long long)q * Q * P;
        if constexpr (V2) {
          // what the rest population makes up for: the rounding residuals
          pi = -Store<S>::st_d(out + oi, pi, rnd(k0 + q, i));
          pj = -Store<S>::st_d(out + oj, pj, rnd(k0 + q, j));
        } else {
          Store<S>::st(out + oi, pi, 0u);
          Store<S>::st(out + oj, pj, 0u);
        }
        if constexpr (ORD && (D == 3 || half == 1)) {
          // (2D: pairs (1, 3) (2, 4), then (5, 7) (6, 8))
          if constexpr (D == 2) rest[q] += held[q][0];
          rest[q] += pi;
          if constexpr (D == 2) rest[q] += held[q][1];
          rest[q] += pj;
        } else if constexpr (ORD) {
          held[q][0] = pi;
          held[q][1] = pj;
        }
      }
      if (KG > 1 && !mine) return;
      // f* = f - (f - f^eq)/tau_f + f^B + F_i (Sec. 2.2)
      if constexpr (F64) {
        R ev = itf * (lam_i * p - (R(1.5) * wi) * uu) - (R(3) * wi) * kFu;
        if constexpr (!ORIG) ev += fbv;
        ev += cu * ((R(4.5) * wi * itf) * cu + (R(9) * wi) * cF);
        const R od = w3i * (itf * cu + cF);
        const R kp = R(1) - itf;
        Store<S>::st(b.f_out + oi, kp * Store<S>::cvt(W.f[i][col]) + (ev + od), 0u);
        Store<S>::st(b.f_out + oj, kp * Store<S>::cvt(W.f[j][col]) + (ev - od), 0u);
      } else {
        // (f^B and q, Y are even in c_i)
        const R fbi = fB_ordered<L>(i, Ad);
        const R q = __fmaf_rn(__fmul_rn(R(4.5), cu), cu, -__fmul_rn(R(1.5), uu));
        const R Y = __fmaf_rn(__fmul_rn(R(9), cF), cu, -__fmul_rn(R(3), Fu));
        const R lin = __fmul_rn(w3i, cu), linF = __fmul_rn(w3i, cF);
        auto post = [&](R f, R l, R lF) -> R {
          const R feq = __fmaf_rn(lam_i, p, __fmaf_rn(wi, q, l));
          const R r = __fmaf_rn(-(f - feq), itf, f);
          return __fmaf_rn(kf, __fmaf_rn(wi, Y, lF), __fmaf_rn(fbi, kB, r));
        };
        if constexpr (V2) {
          // velocity part of the equilibrium in direction +-c, from c.v, v.v
          auto evel = [&](R c, R vv, bool plus) -> R {
            const R qv = __fmul_rn(wi, __fmaf_rn(__fmul_rn(R(4.5), c), c, -__fmul_rn(R(1.5), vv)));
            return __fmaf_rn(w3i, plus ? c : -c, qv);
          };
          const R pi = post(Store<S>::dev_add(W.f[i][col], evel(cU, UU, true)), lin, linF);
          const R pj = post(Store<S>::dev_add(W.f[j][col], evel(cU, UU, false)), -lin, -linF);
          // scaled deviation from e(u) of the receiving node (through a wall:
          // of this node, in the reversed direction)
          auto dev = [&](bool fwd, bool bounced, int r, R post) -> R {
            const Vel<R, D> t = rown[WALLS && bounced ? 0 : r];
            R ud2;
            if constexpr (D == 3) ud2 = t.v[3];
            else ud2 = __fmaf_rn(t.v[0], t.v[0], __fmul_rn(t.v[1], t.v[1]));
            const R c = cdot(t);
            const bool plus = fwd != (WALLS && bounced);
            if (WALLS && edge) {
              // The sum of the two parts rounded the other way round.  It is
              // as exact as evel (errors against FP64 over 26 flows within
              // 1 % of each other on average), and kept because the states
              // of walled grids have its bits.  Its price: evel alone
              // takes 190.0 us a step of 96 FP16 grids (this 200.5), 208 of
              // the 161x97x65 FP16 duct (230).
              const R qv = __fmaf_rn(__fmul_rn(R(4.5), c), c, -__fmul_rn(R(1.5), ud2));
              return R(Store<S>::KF) * (post - __fmaf_rn(wi, qv, __fmul_rn(w3i, plus ? c : -c)));
            }
            return R(Store<S>::KF) * (post - evel(c, ud2, plus));
          };
          Store<S>::st(b.f_out + oi, dev(true, bi, ri, pi), rnd_f(i));
          Store<S>::st(b.f_out + oj, dev(false, bj, rj, pj), rnd_f(j));
        } else {
          Store<S>::st(b.f_out + oi, post(W.f[i][col], lin, linF), 0u);
          Store<S>::st(b.f_out + oj, post(W.f[j][col], -lin, -linF), 0u);
        }
      }
    };
    using Axis = std::true_type;
    using Diag = std::false_type;
    using First = std::integral_constant<int, 0>;
    using Second = std::integral_constant<int, 1>;
    // ring records of the neighbours along each axis
    int np[D], nn[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      np[a] = a == AM ? (rp - rc) * NE : (a == 0 ? 1 : EX);
      nn[a] = a == AM ? (rm - rc) * NE : (a == 0 ? -1 : -EX);
    }
    // the pair along axis a, and the two of the plane (a, b)
    auto on_axis = [&](int a, int i, int j, bool mine, R fbv, auto PH) {
      pair(Axis{}, i, j, mine, u[a], Fd[a], Us[a], fbv, (int)s + sp[a], (int)s + sn[a], hi[a], lo[a],
           np[a], nn[a], [&](const Vel<R, D>& t) { return t.v[a]; }, PH);
    };
    auto on_plus = [&](int a, int b2, int pp, int mm, bool mine, R fbv, auto PH) {
      pair(Diag{}, pp, mm, mine, u[a] + u[b2], Fd[a] + Fd[b2], Us[a] + Us[b2], fbv,
           (int)s + sp[a] + sp[b2], (int)s + sn[a] + sn[b2], hi[a] || hi[b2], lo[a] || lo[b2],
           np[a] + np[b2], nn[a] + nn[b2], [&](const Vel<R, D>& t) { return t.v[a] + t.v[b2]; }, PH);
    };
    auto on_minus = [&](int a, int b2, int pm, int mp, bool mine, R fbv, auto PH) {
      pair(Diag{}, pm, mp, mine, u[a] - u[b2], Fd[a] - Fd[b2], Us[a] - Us[b2], fbv,
           (int)s + sp[a] + sn[b2], (int)s + sn[a] + sp[b2], hi[a] || lo[b2], lo[a] || hi[b2],
           np[a] + nn[b2], nn[a] + np[b2], [&](const Vel<R, D>& t) { return t.v[a] - t.v[b2]; }, PH);
    };
    if constexpr (D == 2) {
      const int k1 = KG == 3 ? 1 : 0, k2 = KG - 1;   // owners of the flow pairs
      on_axis(0, 1, 3, kg == 0, fb.q1 - fb.T[0], First{});
      on_axis(1, 2, 4, kg == 0, fb.q1 - fb.T[1], Second{});
      on_plus(0, 1, 5, 7, kg == k1, fb.q2 - fb.s[0], First{});
      on_minus(1, 0, 6, 8, kg == k2, fb.q2 + fb.s[0], Second{});
    } else if constexpr (F64) {
      // FP64: one pass of a rolled loop per axis, the per-axis values rotated
      // by one place after each (unrolled, the nine pairs spill)
      auto turn = [](auto& v) {
        const auto t = v[0];
        v[0] = v[1];
        v[1] = v[2];
        v[2] = t;
      };
#pragma unroll 1
      for (int q = 0; q < 3; ++q) {
        const int ia = 1 + 2 * q, id = q == 0 ? 7 : (q == 1 ? 15 : 11);
        const int ipm = q == 2 ? id + 3 : id + 2, imp = q == 2 ? id + 2 : id + 3;
        const int o0 = q % KG, o1 = (q + 1) % KG, o2 = (q + 2) % KG;
        on_axis(0, ia, ia + 1, kg == o0, fb.q1 - fb.T[0], First{});
        on_plus(0, 1, id, id + 1, kg == o1, fb.q2 + fb.T[2] - fb.s[2], First{});
        on_minus(0, 1, ipm, imp, kg == o2, fb.q2 + fb.T[2] + fb.s[2], First{});
        turn(u);
        turn(Fd);
        turn(fb.T);
        turn(fb.s);
        turn(sp);
        turn(sn);
        turn(hi);
        turn(lo);
      }
    } else {
      // (in the order of the directions)
      auto own_pair = [&](int n) { return n * KG / 9 == kg; };
      on_axis(0, 1, 2, own_pair(0), fb.q1 - fb.T[0], First{});
      on_axis(1, 3, 4, own_pair(1), fb.q1 - fb.T[1], First{});
      on_axis(2, 5, 6, own_pair(2), fb.q1 - fb.T[2], First{});
      on_plus(0, 1, 7, 8, own_pair(3), fb.q2 + fb.T[2] - fb.s[2], First{});
      on_minus(0, 1, 9, 10, own_pair(4), fb.q2 + fb.T[2] + fb.s[2], First{});
      on_plus(0, 2, 11, 12, own_pair(5), fb.q2 + fb.T[1] - fb.s[1], First{});
      on_minus(0, 2, 13, 14, own_pair(6), fb.q2 + fb.T[1] + fb.s[1], First{});
      on_plus(1, 2, 15, 16, own_pair(7), fb.q2 + fb.T[0] - fb.s[0], First{});
      on_minus(1, 2, 17, 18, own_pair(8), fb.q2 + fb.T[0] + fb.s[0], First{});
    }
    // the rest populations
    if (KG == 1 || kg == KG - 1) {
      const R lam0 = R(p_coef<L, R>(0));
      R f0;
      if constexpr (V2) f0 = Store<S>::dev_add(W.f[0][col], R(w0) * -(R(1.5) * UU));
      else f0 = Store<S>::cvt(W.f[0][col]);
      R post;
      const R e0 = R(w0) * -(R(1.5) * uu);
      if constexpr (ORD) {
        const R feq = __fmaf_rn(lam0, p, e0);
        const R r = __fmaf_rn(-(f0 - feq), itf, f0);
        post = __fmaf_rn(kf, __fmul_rn(R(w0), -__fmul_rn(R(3), Fu)),
                         __fmaf_rn(fB_ordered<L>(0, Ad), kB, r));
        if constexpr (V2) post = R(Store<S>::KF) * (post - e0);
      } else {
        post = f0 - (f0 - (lam0 * p + e0)) * itf + (kf * (R(-3.0 * w0) * Fu) + fb.q0);
      }
      Store<S>::st(b.f_out + s, post, rnd_f(0));
    }
#pragma unroll
    for (int q = 0; q < KC; ++q) {
      if constexpr (V2) h_ext<L>(b.h_out, P)[(uint32_t)(k0 + q) * P32 + s] = h0p[q] + rest[q];
      else if constexpr (RS) Store<S>::st(hout + (long long)q * Q * P + s, own[q] - rest[q], 0u);
      else Store<S>::st(hout + (long long)q * Q * P + s, rest[q], 0u);
    }
  }
  // The closure's counts, once per warp and tile: two additions per warp and
  // plane to the same two words kept a 128^3 step 23 us longer.
  if constexpr (CL) {
    const unsigned act = __ballot_sync(0xffffffffu, active && (KG == 1 || (lane >> 4) == kg));
    if (lane == 0 && ph.cl_count && act) {
      atomicAdd(ph.cl_count, (unsigned long long)cl_used);
      atomicAdd(ph.cl_count + 1, (unsigned long long)(__popc(act) * (m1 - m0) - cl_used));
    }
  }
}

// Initialise a block's stage barriers (one thread; the first copies are
// issued by the same thread, and the other warps first meet a barrier).
template <int NST>
__device__ __forceinline__ void stage_barriers_init(uint64_t (&bar)[NST]) {
#pragma unroll
  for (int q = 0; q < NST; ++q) mbar_init(&bar[q], 1);
  mbar_init_fence();
}

template <class L, class S, int GX, int KG, int MINB, bool WALLS, bool PADDED, bool CL, bool ORIG>
__global__ void __launch_bounds__(FusedShape<L, S, GX, KG, CL>::NT, blocks_of(MINB))
    k_step_fused(Grid g, Phys<RT<S>> ph, Bufs<S> b, int mchunk,
                 const __grid_constant__ StageMaps tm) {
  using Cfg = TileCfg<L, S, GX, KG, MINB, PADDED, CL>;
  extern __shared__ __align__(128) unsigned char fvlb_tile_smem[];
  auto& sm = *reinterpret_cast<typename Cfg::Smem*>(fvlb_tile_smem);
  if (threadIdx.x == FusedShape<L, S, GX, KG, CL>::NCW * 32) stage_barriers_init(sm.bar);
  pdl_wait();   // nothing above reads or writes global memory
  if constexpr (CL) mlp_load(sm.cls.P, static_cast<const MlpPacked*>(ph.mlp));
  StagePos pos;
  fused_tile<L, S, GX, KG, MINB, WALLS, PADDED, CL, ORIG>(sm, g, ph, b, mchunk, blockIdx.x,
                                                      blockIdx.y, blockIdx.z, &tm, tm.on != 0, pos);
  // The next step's blocks may come in when every block's collision warps are
  // through (an exit counts as well: without the call the times are the same).
  // Earlier, they take the free slots of SMs that are busy with this step: 64^2
  // FP64 12.6 us a step with the trigger at the start, 6.3 at the last plane,
  // 6.1 here, 8.2 without the programmatic edge; 128^2 FP32 3.25, 2.96, 2.57
  // and 4.10; 517 x 333 FP32 10.6, 10.3, 10.05 and 12.3; 128^3 FP32 360.6 to
  // 362.0 and 363.8.
  if (threadIdx.x < FusedShape<L, S, GX, KG, CL>::NCW * 32) pdl_trigger();
}

// ---------------------------------------------------------------------------
// Batched step: many independent grids (instances) of one lattice in one
// launch, one block per tile.  The host lists the tiles of every instance
// (instance, x tile, march chunk), largest instances first, so the blocks
// that start last are the small ones.  Per-instance geometry, physics and
// array offsets come from `inst`; the double buffers of all instances live in
// two arenas and `parity` says which one holds the current state.  The step
// count is in device memory so that a captured CUDA graph can replay steps:
// tstep[parity] is read, and the first block leaves the next step's count in
// the other place.
// 96 grids of 33^2 to 455^2 (3.6 M nodes), us per step: FP16 198, FP32 216.
// (Resident blocks that walk the list with a stride: 261 and 230, with the
// loop's state in registers or in shared memory; the uneven ends of their
// shares, and the registers, were what it cost.)
// ---------------------------------------------------------------------------
template <class S>
struct BatchInst {
  Grid g;
  Phys<RT<S>> ph;          // first / step / Fv filled in per launch
  long long f_off, h_off, chi_off;  // element offsets into the arenas
  int cosine;              // F = F0 cos(omega t)
  double F0[3];
  double omega;
};

struct BatchTile {
  int inst;
  int bx;
  int bz;
};

template <class L, class S, int GX, int KG, int MINB>
__global__ void __launch_bounds__(FusedShape<L, S, GX, KG>::NT, blocks_of(MINB))
    k_step_batched(const BatchInst<S>* __restrict__ inst, const BatchTile* __restrict__ tiles,
                   S* fA, S* fB, S* hA, S* hB, typename Store<S>::X* chi, int parity, int first,
                   long long* __restrict__ tstep, int mchunk, const StageMaps* maps) {
  using R = RT<S>;
  extern __shared__ __align__(128) unsigned char fvlb_tile_smem[];
  auto& sm = *reinterpret_cast<typename TileCfg<L, S, GX, KG, MINB, true, false>::Smem*>(fvlb_tile_smem);
  if (threadIdx.x == FusedShape<L, S, GX, KG>::NCW * 32) stage_barriers_init(sm.bar);
  // (the lists were uploaded before any step: not written by a kernel)
  const BatchTile tl = tiles[blockIdx.x];
  const BatchInst<S>& I = inst[tl.inst];
  StagePos pos;
  const Grid g = I.g;
  Phys<R> ph = I.ph;
  Bufs<S> b;
  pdl_wait();
  const long long t = tstep[parity];
  if (blockIdx.x == 0 && threadIdx.x == 0) tstep[1 - parity] = t + 1;
  ph.first = first;
  ph.step = (uint32_t)t;
  if (I.cosine) {
    const double c = cos(I.omega * (double)t);
    ph.Fv[0] = R(I.F0[0] * c);
    ph.Fv[1] = R(I.F0[1] * c);
    ph.Fv[2] = R(I.F0[2] * c);
  }
  b.f_in = (parity ? fB : fA) + I.f_off;
  b.f_out = (parity ? fA : fB) + I.f_off;
  b.h_in = (parity ? hB : hA) + I.h_off;
  b.h_out = (parity ? hA : hB) + I.h_off;
  b.chi = chi + I.chi_off;
  const StageMaps* tm = maps ? maps + tl.inst : nullptr;
  fused_tile<L, S, GX, KG, MINB, true, true, false, false, true>(sm, g, ph, b, mchunk, tl.bx, 0,
                                                                 tl.bz, tm, tm && tm->on, pos);
  if (threadIdx.x < FusedShape<L, S, GX, KG>::NCW * 32) pdl_trigger();
}

}  // namespace fvlb
