// Tensor-core RK stage with the operator streamed from L2 and FP32-class
// accumulation (orders 8 and 9, whose operator fits neither shared nor tensor
// memory).
//
// The contraction is that of tc_stage.cuh: with X = [g^r g^s g^t flux] (one row
// per field c and element e, g^mu_c = sign_c (r_mu,a U_a - r_mu,b U_b)) and
// Op = [Dr Ds Dt LIFT],  rhs[(c,e), i] = sum_k X[(c,e), k] Op[i, k]  (Eq.
// semidiscrete-dg with the chain rule of Eq. dg-reference-matrices applied
// before differentiating), as three FP16 products hi.hi + hi.lo + lo.hi of
// power-of-two scaled rows with FP32 accumulation.
//
// K runs in steps of 16 columns, ordered so that one pass over the fields serves
// the three derivative blocks: node block jb of g^r, g^s, g^t (3 steps), then the
// next node block, then the face nodes.
//   * The operator is stored step by step ([step][hi, lo][2 x 8 columns][node]) and
//     streams through a ring of NB shared-memory slots (one bulk copy a step; 495 KB
//     per tile of 20 tetrahedra at N = 8, 803 KB per 16 at N = 9, all from L2).
//   * Four producer warps build X in registers, split it and write it to a ring of NA
//     tensor-memory slots (FL steps each).
//   * D annihilates constants, so g is formed from U less its value at a node near
//     the centroid: the rounding of g, of its FP16 pieces and of the accumulation then
//     scale with the field's variation within the element instead of its magnitude.
//   * The tensor cores add into FP32 with truncation, and 3 x 45 truncated additions
//     into one accumulator lose ten times what the FP32 CUDA-core stage does.  So
//     every FL steps start a fresh accumulator, two taking turns, and the epilogue
//     warps add the finished one to FP32 registers, rounded to nearest.
// Relative L2 error of one right-hand side against FP64, streamed / FP32 stage:
// smooth fields 2.0e-7 / 2.6e-7 (N = 8), 1.4e-7 / 2.9e-7 (N = 9), random fields
// 2.5e-7 / 3.3e-7 and 2.0e-7 / 3.9e-7.
// Per tile: all worker warps form the fluxes and the row bounds together, the
// producers build X while the epilogue warps collect the accumulators, then all of
// them apply the LSERK4 update (rhs staged through the flux buffer, u from shared
// memory, res straight from and to global memory), every access coalesced.
//
// Measured, ~1.7e7 unknowns: N = 8 161 us a stage, N = 9 214 us, against 1014 and 1214
// us for the FP32 stage; K Np off the 16-byte grid (SH) 182 us.  A tile takes ~57 k
// cycles at N = 8: fields 4-7 k, gathers and fluxes 13 k (issue bound), bounds 3 k,
// MMAs 22 k (12.5 k of tensor-pipe time; the producers' chain sets the pace), update
// 8-13 k.  The CTAs run in step, so L2 sees each phase from all SMs at once.
//
// SH: fields whose chunks are not 16-byte aligned (K Np not a multiple of 4): each
// field lands in shared memory at its global address modulo 16, its aligned part by
// a bulk copy and at most three values at either end by plain loads.
#pragma once

#include <type_traits>

#include <cuda_runtime.h>

#include "device.h"
#include "launch.cuh"
#include "tc_stage.cuh"
#include "tcgen05.cuh"

namespace dgdev {

template <int N> struct TwDims {
  static constexpr int Np = (N + 1) * (N + 2) * (N + 3) / 6;
  static constexpr int Nfp = (N + 1) * (N + 2) / 2;
  static constexpr int NF = 4 * Nfp;
  static constexpr int E = tc_tile_elems(N);
  static constexpr int ROWS = 6 * E;
  static constexpr int JC = tc_central_node(N);
  static constexpr int JB = tw_jblocks(N);             // node blocks of 16
  static constexpr int FB = tw_fblocks(N);             // face-node blocks of 16
  static constexpr int KS = 3 * JB + FB;               // K steps of a tile
  static constexpr int NN = tw_nn(N);                  // MMA N
  static constexpr int FL = 512 - 2 * NN >= 96 ? 3 : 2;   // K steps per accumulator and X slot
  static constexpr int NG = (KS + FL - 1) / FL;        // accumulators of a tile
  static constexpr int NA = (512 - 2 * NN) / (16 * FL);   // X slots (16 columns a step)
  static constexpr int A0 = 2 * NN;                    // first X column
  // Epilogue warps: one per lane quarter and column group.  With at most 96 rows
  // the warps of lane quarter 3 hold no row: two of them issue the MMAs and the
  // copies, else two further warps do.
  static constexpr bool Q3 = ROWS > 96;
  static constexpr int QS = Q3 ? 4 : 3;                // lane quarters with rows
  static constexpr int CG = Q3 ? 2 : 4;                // column groups
  static constexpr int NC = NN / CG;                   // accumulator columns per thread
  static constexpr int EPI = 4 * CG;                   // first producer warp
  static constexpr int MMA_WARP = Q3 ? EPI + 4 : 3, LD_WARP = Q3 ? EPI + 5 : 7;
  static constexpr int WARPS = EPI + 4 + (Q3 ? 2 : 0);
  static constexpr int THREADS = 32 * WARPS;
  static constexpr int NWW = QS * CG + 4;              // worker warps
  static constexpr int NW = 32 * NWW;
  static constexpr int PARTS = NW / ROWS;              // threads per row of the bound pass
  static constexpr int ITEMS = (E * NF + NW - 1) / NW; // face nodes per worker
  static constexpr int FSTR = (NF / 4) % 2 ? NF : NF + 4;   // 16-byte reads of 8 rows conflict-free
  static constexpr int PIECE = NN * 32;                // bytes of one operator piece of a step
  static constexpr int SLOT = 2 * PIECE;
  // shared memory (bytes)
  static constexpr int UST = E * Np + 4;               // field stride (floats), shifted: room for it
  static constexpr int G_FLOATS = tc_geo_floats(N);
  static constexpr int F_FLOATS = ROWS * (FSTR > Np ? FSTR : Np);   // fluxes, then staged rhs
  static constexpr int U_BYTES = 6 * UST * 4, F_BYTES = F_FLOATS * 4, G_BYTES = G_FLOATS * 4;
  static constexpr int P_BYTES = 2 * PARTS * ROWS * 4;
  static constexpr int T_BYTES = (NF + 15) & ~15;
  static constexpr int REST = U_BYTES + F_BYTES + G_BYTES + P_BYTES + T_BYTES;
  static constexpr int NB_FIT = (226 * 1024 - REST) / SLOT;
  static constexpr int NB = NB_FIT > 4 ? 4 : NB_FIT;   // operator slots
  static constexpr int OFF_U = NB * SLOT;
  static constexpr int OFF_F = OFF_U + U_BYTES;
  static constexpr int OFF_G = OFF_F + F_BYTES;
  static constexpr int OFF_P = OFF_G + G_BYTES;
  static constexpr int OFF_T = OFF_P + P_BYTES;
  static constexpr int SMEM = OFF_T + T_BYTES;
  static_assert(NB >= 3 && NA >= 2 && SMEM <= 226 * 1024, "ring depths");
  static_assert(ROWS <= 128 && NN % 16 == 0 && NN <= 256 && NC % 4 == 0, "MMA shape");
  static_assert(SLOT % 128 == 0 && OFF_F % 16 == 0 && OFF_G % 16 == 0 && UST % 4 == 0, "alignment");
  static_assert((E * Np) % 4 == 0 && G_BYTES % 16 == 0 && NF % 4 == 0, "bulk-copy sizes");
};

static_assert(tw_b_bytes(8) == TwDims<8>::KS * TwDims<8>::SLOT, "operator stream size");

// Accumulator columns [0, NC) of this thread's group: acc += tensor memory.
template <int NC>
__device__ __forceinline__ void tw_add_cols(uint32_t taddr, float* acc) {
  if constexpr (NC > 0) {
    constexpr int CH = NC >= 16 ? 16 : NC >= 8 ? 8 : 4;
    uint32_t v[CH];
    tc::tmem_ld<CH>(taddr, v);
    tc::tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < CH; i += 2) {
      const float2 s = __fadd2_rn(make_float2(acc[i], acc[i + 1]),
                                  make_float2(__uint_as_float(v[i]), __uint_as_float(v[i + 1])));
      acc[i] = s.x;
      acc[i + 1] = s.y;
    }
    tw_add_cols<NC - CH>(taddr + CH, acc + CH);
  }
}

// As wait_or_flag, each lane of a converged warp watching its own barrier.  The loop
// ends for all lanes at once: lanes leaving it one by one would stay apart, and every
// elect.sync of the MMAs that follow would have to gather them (~480 cycles an MMA
// instead of ~15).
__device__ __forceinline__ void wait_lanes_or_flag(uint64_t* bar, uint32_t parity, int* status) {
  bool ok = false;
  for (uint32_t i = 0; i < kWaitLimit; ++i) {
    ok = ok || tc::mbar_try_wait(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return;
  }
  if (status) atomicExch(status, 1);
}

template <int N, bool RK, bool EXT, bool SH>
__global__ void __launch_bounds__(TwDims<N>::THREADS, 1)
tw_stage_kernel(const __grid_constant__ StageArgs A) {
  using D = TwDims<N>;
  constexpr int E = D::E, Np = D::Np, Nfp = D::Nfp, NF = D::NF, ROWS = D::ROWS, FSTR = D::FSTR;
  constexpr int UST = SH ? D::UST : E * Np, NB = D::NB, NA = D::NA, KS = D::KS, NG = D::NG;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint32_t s_tmem;
  // s_done: the MMAs of X slot i are complete (X slot free, accumulator full)
  __shared__ __align__(8) uint64_t s_b_full[NB], s_b_free[NB], s_a_full[NA], s_done[NA];
  __shared__ __align__(8) uint64_t s_acc_free[2], s_u_full, s_u_free;

  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int K = A.K, ncta = int(gridDim.x), cta = int(blockIdx.x);
  const int ntiles = (A.num_tiles - cta + ncta - 1) / ncta;
  const int base = A.tile0 + cta;

  float* sU = reinterpret_cast<float*>(smem + D::OFF_U);
  float* sF = reinterpret_cast<float*>(smem + D::OFF_F);
  const float* sG = reinterpret_cast<const float*>(smem + D::OFF_G);
  float* sP = reinterpret_cast<float*>(smem + D::OFF_P);          // [fields, fluxes][PARTS][ROWS]
  unsigned char* sFmask = smem + D::OFF_T;

  for (int i = tid; i < NF; i += D::THREADS) sFmask[i] = __ldg(A.fmask + i);
  if (warp == 0) tc::tmem_alloc(&s_tmem, 512);
  if (tid == 0) {
    for (int i = 0; i < NB; ++i) {
      tc::mbar_init(&s_b_full[i], 1);
      tc::mbar_init(&s_b_free[i], 1);
    }
    for (int i = 0; i < NA; ++i) {
      tc::mbar_init(&s_a_full[i], D::QS);            // one arrival per producer warp with rows
      tc::mbar_init(&s_done[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&s_acc_free[i], D::QS * D::CG);  // one arrival per epilogue warp
    }
    tc::mbar_init(&s_u_full, 1);
    tc::mbar_init(&s_u_free, D::NWW);                // one arrival per worker warp
    tc::fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = s_tmem;
  // field c of a tile starts at sU + c * UST + shift(c): with SH its global
  // address modulo 16 bytes (a tile's offset k0 * Np is a multiple of 4)
  const int sh0 = SH ? int(reinterpret_cast<uintptr_t>(A.u_in) >> 2) & 3 : 0;
  const int shk = SH ? (K * Np) & 3 : 0;
  auto ubase = [&](int c) { return c * UST + (SH ? (sh0 + c * shk) & 3 : 0); };

  if (warp == D::MMA_WARP) {
    // ============================== MMA issue ================================
    constexpr uint32_t IDESC = tc::idesc_f16(128, D::NN);
    const uint64_t b0 = tc::smem_desc(tc::smem_u32(smem), D::NN * 16, 128);
    int as = 0, bs = 0, ap = 0, bp = 0, g = 0;       // X and operator slot and phase, unit
    for (int t = 0; t < ntiles; ++t) {
#pragma unroll 1
      for (int st = 0; st < KS; st += D::FL, ++g) {
        const int n = min(D::FL, KS - st);
        const uint32_t d = tbase + (g & 1) * D::NN;
        const uint32_t a0 = tbase + D::A0 + as * (16 * D::FL);
#pragma unroll
        for (int q = 0; q < D::FL; ++q) {
          if (KS % D::FL && q >= n) break;
          // one poll watches everything these MMAs need (a poll of a ready barrier costs
          // ~100 cycles here): lane 0 the operator step; before the first step of an
          // accumulator also lane 1 the accumulator and the others the X slot
          uint64_t* bar = &s_b_full[bs];
          int parity = bp;
          if (q == 0 && lane >= 1) {
            bar = &s_a_full[as];
            parity = ap;
            if (lane == 1 && g >= 2) {
              bar = &s_acc_free[g & 1];
              parity = ((g >> 1) - 1) & 1;
            }
          }
          wait_lanes_or_flag(bar, parity, A.status);
          tc::fence_after_sync();
          const uint32_t a = a0 + q * 16;
          const uint64_t b = b0 + uint64_t((bs * D::SLOT) >> 4);
          const uint64_t bl = b + uint64_t(D::PIECE >> 4);
          tc::mma_f16_ts_warp(d, a + 8, b, IDESC, q ? 1u : 0u);    // lo.hi
          tc::mma_f16_ts_warp(d, a, bl, IDESC, 1u);                // hi.lo
          tc::mma_f16_ts_warp(d, a, b, IDESC, 1u);                 // hi.hi
          tc::mma_commit_warp(&s_b_free[bs]);
          if (++bs == NB) { bs = 0; bp ^= 1; }
        }
        tc::mma_commit_warp(&s_done[as]);
        if (++as == NA) { as = 0; ap ^= 1; }
      }
    }
  } else if (warp == D::LD_WARP) {
    // ============================ bulk copies ================================
    const unsigned char* op = static_cast<const unsigned char*>(A.twB);
    int bs = 0, bp = 0, step = 0;                    // operator slot, phase; steps issued
    auto load_steps = [&](int upto) {                // operator steps until `upto` are issued
      for (; step < upto; ++step) {
        if (step >= NB) wait_or_flag(&s_b_free[bs], bp ^ 1, A.status);
        if (tc::elect_one()) {
          tc::mbar_expect_tx(&s_b_full[bs], D::SLOT);
          tc::bulk_g2s(smem + bs * D::SLOT, op + size_t(step % KS) * D::SLOT, D::SLOT,
                       &s_b_full[bs]);
        }
        __syncwarp();
        if (++bs == NB) { bs = 0; bp ^= 1; }
      }
    };
    auto load_fields = [&](int t) {
      const int tile = base + t * ncta, k0 = tile * E, n = min(E, K - k0) * Np;
      if (t >= 1) wait_or_flag(&s_u_free, (t - 1) & 1, A.status);
      tc::fence_proxy_async_smem();
      uint32_t bytes = D::G_BYTES;
      if constexpr (SH) {
        // values before and after the 16-byte aligned part of each field, three
        // candidates at either end: lane l < 18 the heads, 18 <= l < 36 the tails
        for (int l = lane; l < 36; l += 32) {
          const int c = (l % 18) / 3, j = l % 3, sh = ubase(c) & 3;
          const int head = min(n, (4 - sh) & 3), mid = (n - head) & ~3;
          const int i = l < 18 ? j : head + mid + j;
          if (l < 18 ? j < head : i < n)
            sU[ubase(c) + i] = __ldg(A.u_in + (size_t(c) * K + k0) * Np + i);
        }
        for (int c = 0; c < 6; ++c) bytes += uint32_t((n - min(n, (4 - (ubase(c) & 3)) & 3)) & ~3) * 4;
      } else {
        bytes += uint32_t(6 * n) * 4;
      }
      __syncwarp();
      if (tc::elect_one()) {
        tc::mbar_expect_tx(&s_u_full, bytes);
        for (int c = 0; c < 6; ++c) {
          const int head = SH ? min(n, (4 - (ubase(c) & 3)) & 3) : 0, mid = (n - head) & ~3;
          if (mid)
            tc::bulk_g2s(sU + ubase(c) + head, A.u_in + (size_t(c) * K + k0) * Np + head,
                         uint32_t(mid) * 4, &s_u_full);
        }
        tc::bulk_g2s(smem + D::OFF_G, A.tcgeo + size_t(tile) * A.tc_geo_stride, D::G_BYTES,
                     &s_u_full);
      }
      __syncwarp();
    };
    // L2 prefetch of tile t's RK register and (t >= 1) fields, a tile ahead, so that
    // HBM works while the tensor cores do
    auto prefetch = [&](int t) {
      if (SH || t >= ntiles || !tc::elect_one()) return;
      const int k0 = (base + t * ncta) * E, n = min(E, K - k0) * Np;
      for (int c = 0; c < 6; ++c) {
        const size_t gi = (size_t(c) * K + k0) * Np;
        if (t >= 1) tc::bulk_prefetch_l2(A.u_in + gi, uint32_t(n) * 4);
        if (RK) tc::bulk_prefetch_l2(A.res + gi, uint32_t(n) * 4);
      }
    };
    // the operator is constant: its first steps may overlap the previous kernel
    load_steps(NB);
    pdl_wait();
    load_fields(0);
    prefetch(0);
    for (int t = 0; t < ntiles; ++t) {
      prefetch(t + 1);
      __syncwarp();
      load_steps((t + 1) * KS);
      if (t + 1 < ntiles) load_fields(t + 1);
    }
  } else if (warp >= D::EPI || (warp & 3) < D::QS) {
    // ============================= worker warps ==============================
    pdl_wait();
    const bool epi = warp < D::EPI;
    const int quarter = warp & 3, group = warp >> 2;
    // this thread among the workers
    const int w = (epi ? (warp >> 2) * D::QS + quarter : D::QS * D::CG + warp - D::EPI) * 32 + lane;
    // X row (c, e) of the tile, curl fields fa, fb of component c
    const int row = quarter * 32 + lane;
    const bool live = row < ROWS;
    const int rc = live ? row / E : 0, re = live ? row - rc * E : 0;
    const int o = rc % 3;
    const int fa = rc < 3 ? 3 + (o + 2) % 3 : (o + 2) % 3;
    const int fb = rc < 3 ? 3 + (o + 1) % 3 : (o + 1) % 3;
    const float sgn = rc < 3 ? 1.f : -1.f;
    const uint32_t lane_off = uint32_t(quarter * 32) << 16;
    const unsigned char* nodes = reinterpret_cast<const unsigned char*>(sG + kTcGeoWords * E);

    for (int t = 0; t < ntiles; ++t) {
      const int k0 = (base + t * ncta) * E, Ev = min(E, K - k0);
      wait_or_flag(&s_u_full, t & 1, A.status);
      // ---- fluxes (Alg. 3): item idx = w + q NW is face node m of element e, of kind
      // 0 none, 1 wall, 2 neighbour in the tile, 3 outside it.  First every gather of
      // kind 3 is started (the neighbour's values go into the words the item's flux will
      // overwrite), then the field bounds are formed while they fly, then the fluxes,
      // two items at a time; classifying twice is cheaper than keeping every item
      struct Item { int e, m, f, ofs, k2, i2; uint32_t kind; bool zero; };
      auto classify = [&](int q) {
        Item x;
        const int idx = w + q * D::NW;
        x.e = idx / NF;
        x.m = idx - x.e * NF;
        x.f = x.m / Nfp;
        const bool ok = idx < E * NF && x.e < Ev;
        if (!ok) x.e = 0;
        const unsigned code = (__float_as_uint(sG[9 * E + x.e]) >> (8 * x.f)) & 0xffu;
        x.k2 = __float_as_int(sG[(26 + x.f) * E + x.e]);
        x.i2 = nodes[x.e * NF + x.m];
        const int e2 = x.k2 - k0;
        x.zero = EXT && code == kAbsorbingCode;      // absorbing: u+ = 0
        x.kind = !ok ? 0u : (code == 0u || x.zero) ? 1u : unsigned(e2) < unsigned(Ev) ? 2u : 3u;
        x.ofs = x.kind == 2u ? e2 * Np + x.i2 : x.e * Np + int(sFmask[x.m]);
        return x;
      };
      auto flux = [&](const Item (&it)[2]) {
        float uM[2][6], up[2][6], nv[2][4];
        float4 cf[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const Item& x = it[h];
          const int iM = x.e * Np + int(sFmask[x.m]);
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            uM[h][c] = sU[ubase(c) + iM];
            up[h][c] = x.zero ? 0.f
                       : x.kind == 3u ? sF[(c * E + x.e) * FSTR + x.m] : sU[ubase(c) + x.ofs];
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) nv[h][k] = sG[(10 + 4 * x.f + k) * E + x.e];
          if constexpr (EXT)
            cf[h] = A.mat && x.kind ? __ldg(A.mat + size_t(k0 + x.e) * kMatVecs + 1 + x.f)
                                    : make_float4(1.f, 0.5f, 1.f, 0.5f);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const Item& x = it[h];
          const float nwe = x.kind == 1u ? 1.f : -1.f;  // E+ = -E- on conducting walls
          const float dEx = fmaf(nwe, up[h][0], uM[h][0]);
          const float dEy = fmaf(nwe, up[h][1], uM[h][1]);
          const float dEz = fmaf(nwe, up[h][2], uM[h][2]);
          const float dHx = uM[h][3] - up[h][3], dHy = uM[h][4] - up[h][4];
          const float dHz = uM[h][5] - up[h][5];
          const float nx = nv[h][0], ny = nv[h][1], nz = nv[h][2], sc = 0.5f * nv[h][3];
          const float al = A.alpha;
          const float aE = al * fmaf(nz, dEz, fmaf(ny, dEy, nx * dEx));
          const float aH = al * fmaf(nz, dHz, fmaf(ny, dHy, nx * dHx));
          // -n x dH + alpha (n (n.dE) - dE) and n x dE + alpha (n (n.dH) - dH); EXT:
          // B_E (Z+ (-n x dH) + ...), B_H (Y+ (n x dE) + ...) with Fscale
          float zp = 1.f, yp = 1.f, scE = sc, scH = sc;
          if constexpr (EXT) {
            zp = cf[h].x;
            yp = cf[h].z;
            scE = cf[h].y * nv[h][3];
            scH = cf[h].w * nv[h][3];
          }
          float fl[6];
          fl[0] = fmaf(-al, dEx, fmaf(nx, aE, zp * fmaf(-ny, dHz, nz * dHy)));
          fl[1] = fmaf(-al, dEy, fmaf(ny, aE, zp * fmaf(-nz, dHx, nx * dHz)));
          fl[2] = fmaf(-al, dEz, fmaf(nz, aE, zp * fmaf(-nx, dHy, ny * dHx)));
          fl[3] = fmaf(-al, dHx, fmaf(nx, aH, yp * fmaf(-nz, dEy, ny * dEz)));
          fl[4] = fmaf(-al, dHy, fmaf(ny, aH, yp * fmaf(-nx, dEz, nz * dEx)));
          fl[5] = fmaf(-al, dHz, fmaf(nz, aH, yp * fmaf(-ny, dEx, nx * dEy)));
          if (x.kind) {
#pragma unroll
            for (int c = 0; c < 6; ++c)
              sF[(c * E + x.e) * FSTR + x.m] = (c < 3 ? scE : scH) * fl[c];
          }
        }
      };
#pragma unroll 2
      for (int q = 0; q < D::ITEMS; ++q) {
        const Item x = classify(q);
        if (x.kind == 3u) {
          const float* src = A.u_in + size_t(x.k2) * Np + x.i2;
#pragma unroll
          for (int c = 0; c < 6; ++c)
            tc::cp_async4(sF + (c * E + x.e) * FSTR + x.m, src + size_t(c) * K * Np);
        }
      }
      tc::cp_async_commit();
      // bounds: part p of row r takes every PARTS-th value of field row r (less its
      // reference value) and, once they are formed, every PARTS-th 16 bytes of flux row r
      const int bp = w / ROWS, br = w - bp * ROWS, bc = br / E, be = br - bc * E;
      const bool bounds = bp < D::PARTS && be < Ev;
      if (bounds) {
        float um = 0.f;
        if constexpr (Np % 4 == 0) {
          const float4* ur = reinterpret_cast<const float4*>(sU + bc * UST + be * Np);
          const float u0 = sU[bc * UST + be * Np + D::JC];
#pragma unroll 4
          for (int j = bp; j < Np / 4; j += D::PARTS) {
            const float4 x = ur[j];
            um = fmaxf(fmaxf(um, fmaxf(fabsf(x.x - u0), fabsf(x.y - u0))),
                       fmaxf(fabsf(x.z - u0), fabsf(x.w - u0)));
          }
        } else {
          const float* ur = sU + ubase(bc) + be * Np;
          const float u0 = ur[D::JC];
#pragma unroll 8
          for (int j = bp; j < Np; j += D::PARTS) um = fmaxf(um, fabsf(ur[j] - u0));
        }
        sP[bp * ROWS + br] = um;
      }
      tc::cp_async_wait_all();
#pragma unroll 1
      for (int q = 0; q < D::ITEMS; q += 2) {
        const Item it[2] = {classify(q), classify(q + 1)};   // none past the last item
        flux(it);
      }
      named_sync(1, D::NW);                          // fluxes complete
      if (bounds) {
        float fm = 0.f;
        const float4* fr = reinterpret_cast<const float4*>(sF + br * FSTR);
#pragma unroll 5
        for (int j = bp; j < NF / 4; j += D::PARTS) {
          const float4 x = fr[j];
          fm = fmaxf(fmaxf(fm, fmaxf(fabsf(x.x), fabsf(x.y))), fmaxf(fabsf(x.z), fabsf(x.w)));
        }
        sP[(D::PARTS + bp) * ROWS + br] = fm;
      }
      named_sync(1, D::NW);                          // bounds published
      // ---- row scale: |g^mu| <= (|r_mu,a| + |r_mu,b|) max(max|U_a|, max|U_b|)
      const bool lv = live && re < Ev;
      float ca[3], cb[3], s = 1.f;
#pragma unroll
      for (int mu = 0; mu < 3; ++mu) ca[mu] = cb[mu] = 0.f;
      if (lv) {
        float um = 0.f, fm = 0.f, cm = 0.f;
#pragma unroll
        for (int p = 0; p < D::PARTS; ++p) {
          um = fmaxf(um, fmaxf(sP[p * ROWS + fa * E + re], sP[p * ROWS + fb * E + re]));
          fm = fmaxf(fm, sP[(D::PARTS + p) * ROWS + row]);
        }
#pragma unroll
        for (int mu = 0; mu < 3; ++mu) {
          ca[mu] = sgn * sG[(3 * mu + (o + 1) % 3) * E + re];
          cb[mu] = -sgn * sG[(3 * mu + (o + 2) % 3) * E + re];
          cm = fmaxf(cm, fabsf(ca[mu]) + fabsf(cb[mu]));
        }
        s = row_scale(fmaxf(cm * um, fm));
      }
      if (epi) {
        // ---- collect the units: FP32 registers, rounded to nearest
        float acc[D::NC];
#pragma unroll
        for (int i = 0; i < D::NC; ++i) acc[i] = 0.f;
#pragma unroll 1
        for (int u = 0; u < NG; ++u) {
          const int g = t * NG + u, buf = g & 1;
          wait_or_flag(&s_done[g % NA], (g / NA) & 1, A.status);
          tc::fence_after_sync();
          tw_add_cols<D::NC>(tbase + lane_off + buf * D::NN + group * D::NC, acc);
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&s_acc_free[buf]);
        }
        // ---- rhs (times the step) into the flux buffer, in the fields' own layout
        // (every flux has been read: the last unit's MMAs are complete)
        if (lv) {
          float f = A.tc_inv_bscale / s;
          if (EXT && A.mat) {                        // rhs_E / eps, rhs_H / mu
            const float4 mw = __ldg(A.mat + size_t(k0 + re) * kMatVecs);
            f *= rc < 3 ? mw.x : mw.y;
          }
          const float dte = RK ? (A.dt_elem ? __ldg(A.dt_elem + k0 + re) : A.dt) : 1.f;
          float* dst = sF + row * Np;
          const int c0 = group * D::NC;
          if constexpr (Np % 4 == 0) {
#pragma unroll
            for (int i = 0; i < D::NC; i += 4)
              if (c0 + i < Np)
                *reinterpret_cast<float4*>(dst + c0 + i) =
                    make_float4(dte * (acc[i] * f), dte * (acc[i + 1] * f), dte * (acc[i + 2] * f),
                                dte * (acc[i + 3] * f));
          } else {
#pragma unroll
            for (int i = 0; i < D::NC; ++i)
              if (c0 + i < Np) dst[c0 + i] = dte * (acc[i] * f);
          }
        }
      } else {
        // ---- X(t), step by step; a slot is signalled after the next step's values
        // are formed, when its stores have long completed
        const float* ua = sU + ubase(fa) + re * Np;
        const float* ub = sU + ubase(fb) + re * Np;
        const float* fr = sF + (live ? row : 0) * FSTR;
        const float a0 = -ua[D::JC], b0 = -ub[D::JC];
        int pend = -1;
        auto signal = [&]() {
          tc::tmem_st_wait();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&s_a_full[pend]);
        };
        auto put = [&](const float2 (&v)[8], int st) {   // step st of the tile
          const int g = t * NG + st / D::FL, slot = g % NA, q = st % D::FL;
          uint32_t hi[8], lo[8];
#pragma unroll
          for (int p = 0; p < 8; ++p) tc::split2<true>(v[p].x, v[p].y, hi[p], lo[p]);
          if (q == 0) {
            if (pend >= 0) signal();
            if (g >= NA) wait_or_flag(&s_done[slot], (g / NA - 1) & 1, A.status);
            tc::fence_after_sync();
            pend = slot;
          }
          tc::tmem_st<8>(tbase + lane_off + D::A0 + (slot * D::FL + q) * 16, hi);
          tc::tmem_st<8>(tbase + lane_off + D::A0 + (slot * D::FL + q) * 16 + 8, lo);
          if (q == D::FL - 1) {
            signal();
            pend = -1;
          }
        };
        // rows past the tile's elements hold whatever is there: no other row sees it
        auto load_nodes = [&](const float* p, int j0, float pad, float2 (&x)[8], auto part) {
          if constexpr (Np % 4 == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 y = !part.value || 4 * i < Np % 16
                                   ? *reinterpret_cast<const float4*>(p + j0 + 4 * i)
                                   : make_float4(pad, pad, pad, pad);
              x[2 * i] = make_float2(y.x, y.y);
              x[2 * i + 1] = make_float2(y.z, y.w);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              x[i] = make_float2(!part.value || 2 * i < Np % 16 ? p[j0 + 2 * i] : pad,
                                 !part.value || 2 * i + 1 < Np % 16 ? p[j0 + 2 * i + 1] : pad);
          }
        };
        // the three steps of node block u from its values (a, b), which then take the
        // next block's
        auto put_nodes = [&](float2 (&a)[8], float2 (&b)[8], int u, auto next) {
          // the scale goes on the fields: s may reach 2^127 for a row of tiny values,
          // while |U s| < 2^15 / (|r_a| + |r_b|)
          float2 x[8], y[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            x[i] = __fmul2_rn(__fadd2_rn(a[i], f2(a0)), f2(s));
            y[i] = __fmul2_rn(__fadd2_rn(b[i], f2(b0)), f2(s));
          }
          next();
#pragma unroll
          for (int mu = 0; mu < 3; ++mu) {
            float2 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
              v[i] = __ffma2_rn(f2(ca[mu]), x[i], __fmul2_rn(f2(cb[mu]), y[i]));
            put(v, 3 * u + mu);
          }
        };
        if (D::Q3 || quarter < D::QS) {
          using Part = std::integral_constant<bool, Np % 16 != 0>;
          float2 a[8], b[8];
          load_nodes(ua, 0, 0.f, a, std::false_type{});
          load_nodes(ub, 0, 0.f, b, std::false_type{});
#pragma unroll 1
          for (int u = 0; u < D::JB - 2; ++u)
            put_nodes(a, b, u, [&] {
              load_nodes(ua, 16 * (u + 1), 0.f, a, std::false_type{});
              load_nodes(ub, 16 * (u + 1), 0.f, b, std::false_type{});
            });
          put_nodes(a, b, D::JB - 2, [&] {
            load_nodes(ua, 16 * (D::JB - 1), -a0, a, Part{});
            load_nodes(ub, 16 * (D::JB - 1), -b0, b, Part{});
          });
          put_nodes(a, b, D::JB - 1, [] {});
        }
        if (D::Q3 || quarter < D::QS) {
#pragma unroll 1
          for (int q = 0; q < D::FB; ++q) {
            float2 v[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 x = 16 * q + 4 * i < NF
                                   ? *reinterpret_cast<const float4*>(fr + 16 * q + 4 * i)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
              v[2 * i] = __fmul2_rn(make_float2(x.x, x.y), f2(s));
              v[2 * i + 1] = __fmul2_rn(make_float2(x.z, x.w), f2(s));
            }
            put(v, 3 * D::JB + q);
          }
          if (pend >= 0) signal();
        }
      }
      // ---- LSERK4 update res <- a res + dt rhs, u <- u + b res (or the bare rhs),
      // chunk w + q NW of the tile's [6][Ev][Np] values (16 bytes, single values where
      // shifted); every chunk's res is under way before the staged rhs is complete, so
      // the update costs one trip to memory
      if constexpr (SH) {
        named_sync(1, D::NW);                        // rhs staged
        for (int i = w; i < Ev * Np; i += D::NW) {
          float rv[6];
          if (RK) {
#pragma unroll
            for (int c = 0; c < 6; ++c) rv[c] = A.res[(size_t(c) * K + k0) * Np + i];
          }
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            const size_t gi = (size_t(c) * K + k0) * Np + i;
            const float r = sF[c * E * Np + i];
            if (RK) {
              const float rn = fmaf(A.a, rv[c], r);
              A.res[gi] = rn;
              A.u_out[gi] = fmaf(A.b, rn, sU[ubase(c) + i]);
            } else {
              A.rhs[gi] = r;
            }
          }
        }
      } else {
        constexpr int C4 = E * Np / 4, QN = (6 * C4 + D::NW - 1) / D::NW;
        // chunk x is chunk i of field c, at off(x) 16-byte words (a ragged tile has
        // fewer than C4 a field)
        const int n4 = Ev * Np / 4, S4 = K * Np / 4;
        const uint32_t at = uint32_t(size_t(k0) * Np / 4);
        auto valid = [&](int x) { return x < 6 * C4 && x - x / C4 * C4 < n4; };
        auto off = [&](int x) { return at + uint32_t(x) + uint32_t(x / C4) * uint32_t(S4 - C4); };
        float4* res4 = reinterpret_cast<float4*>(A.res);
        constexpr int QH = (QN + 1) / 2;             // (all at once would not fit the registers)
        float4 rv[QH];
        auto load_res = [&](int q0) {
#pragma unroll
          for (int q = 0; q < QH; ++q)
            if (RK && q0 + q < QN && valid(w + (q0 + q) * D::NW))
              rv[q] = res4[off(w + (q0 + q) * D::NW)];
        };
        auto update = [&](int q0) {
#pragma unroll
          for (int q = 0; q < QH; ++q) {
            const int x = w + (q0 + q) * D::NW;
            if (q0 + q < QN && valid(x)) {
              const float4 r = reinterpret_cast<const float4*>(sF)[x];
              if (RK) {
                const float4 u = reinterpret_cast<const float4*>(sU)[x];
                float4 rn, un;
                rn.x = fmaf(A.a, rv[q].x, r.x);
                rn.y = fmaf(A.a, rv[q].y, r.y);
                rn.z = fmaf(A.a, rv[q].z, r.z);
                rn.w = fmaf(A.a, rv[q].w, r.w);
                un.x = fmaf(A.b, rn.x, u.x);
                un.y = fmaf(A.b, rn.y, u.y);
                un.z = fmaf(A.b, rn.z, u.z);
                un.w = fmaf(A.b, rn.w, u.w);
                res4[off(x)] = rn;
                reinterpret_cast<float4*>(A.u_out)[off(x)] = un;
              } else {
                reinterpret_cast<float4*>(A.rhs)[off(x)] = r;
              }
            }
          }
        };
        load_res(0);
        named_sync(1, D::NW);                        // rhs staged
        update(0);
        load_res(QH);
        update(QH);
      }
      __syncwarp();                                  // the fields have been read
      if (lane == 0) tc::mbar_arrive(&s_u_free);
      named_sync(1, D::NW);                          // the flux buffer is free again
    }
  }
  __syncwarp();
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, 512);
}

template <int N>
cudaError_t launch_tw_stage_n(bool rk, bool shifted, const StageArgs& a, int num_sms,
                              cudaStream_t s) {
  using D = TwDims<N>;
  static bool attr[8][16] = {};         // [rk, ext, shifted][device]: attribute set
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  const bool ext = a.mat || a.absorbing;
  void (*kern)(const StageArgs) = nullptr;
  if constexpr (D::Np % 4 != 0) {       // a shift arises only where K Np can be off by it
    if (shifted)
      kern = rk ? (ext ? tw_stage_kernel<N, true, true, true> : tw_stage_kernel<N, true, false, true>)
                : (ext ? tw_stage_kernel<N, false, true, true>
                       : tw_stage_kernel<N, false, false, true>);
  } else if (shifted) {
    return cudaErrorInvalidValue;
  }
  if (!kern)
    kern = rk ? (ext ? tw_stage_kernel<N, true, true, false> : tw_stage_kernel<N, true, false, false>)
              : (ext ? tw_stage_kernel<N, false, true, false>
                     : tw_stage_kernel<N, false, false, false>);
  // at least 120 KB of shared memory: never two CTAs (each takes all 512
  // tensor-memory columns) on one SM
  constexpr int smem = D::SMEM > 120 * 1024 ? D::SMEM : 120 * 1024;
  bool& done = attr[(rk ? 4 : 0) + (ext ? 2 : 0) + (shifted ? 1 : 0)][dev & 15];
  if (!done) {
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err != cudaSuccess) return err;
    done = true;
  }
  const int grid = a.num_tiles < num_sms ? a.num_tiles : num_sms;
  if (grid <= 0) return cudaSuccess;
  return launch_pdl(kern, grid, D::THREADS, smem, s, a);
}

}  // namespace dgdev

#define DG_INSTANTIATE_TW_STAGE(NN)                                                              \
  namespace dgdev {                                                                               \
  template cudaError_t launch_tw_stage_n<NN>(bool, bool, const StageArgs&, int, cudaStream_t);    \
  }
