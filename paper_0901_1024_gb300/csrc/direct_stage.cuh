// FP32 RK stage with one thread per tetrahedron, everything in registers.
//
// At the lowest order an element is 6 x 4 values: the tiled FP32 stage
// (stage_kernel.cuh) spends its time staging them through shared memory by 4-byte
// copies and on five barriers a tile, at a quarter of the HBM bandwidth.  Here a
// thread reads its element's rows as 16-byte words (consecutive lanes, consecutive
// elements: coalesced), the four neighbours' rows the same way (the neighbours of
// consecutive elements lie close together: L1 and L2), and the operators come as
// constant-bank operands of the multiply-adds (they are a kernel parameter).  The
// geometry is read from the tiled word-major copy of the tensor-core stages, whose
// runs of tc_tile_elems elements are nearly coalesced too.
// Arithmetic as in stage_kernel.cuh: differentiate, chain rule and curl, flux, lifting.
// 128 registers a thread, 16 warps an SM; the latency of the first loads bounds it.
// 705 894 tetrahedra: 83-86 us a stage (64 % of the HBM roofline) against 196 us for the
// tiles; without the L2 prefetch of the RK register 98 us; blocks capped at 96 or 80
// registers 100-103 us, 64-thread blocks 97 us.
#pragma once

#include <cuda_runtime.h>

#include "device.h"
#include "launch.cuh"

namespace dgdev {

// Node index (first reference coordinate fastest) of face node j of face f at order N:
// faces t = -1, s = -1, r + s + t = -1, r = -1, their nodes ascending.
__host__ __device__ constexpr int direct_face_node(int N, int f, int j) {
  int n = 0, hit = 0;
  for (int c = 0; c <= N; ++c)
    for (int b = 0; b + c <= N; ++b)
      for (int a = 0; a + b + c <= N; ++a, ++n) {
        const bool on = f == 0 ? c == 0 : f == 1 ? b == 0 : f == 2 ? a + b + c == N : a == 0;
        if (on && hit++ == j) return n;
      }
  return -1;
}

constexpr int kDirectThreads = 128;

// What a mesh has beside vacuum and conducting walls: nothing, absorbing faces, materials
// (and absorbing faces, maybe), or either as the arguments say.  The last is the fastest on
// large meshes (705 894 tetrahedra: absorbing 86 us a stage, materials 92; told apart at
// compile time 92 and 104, by more registers in flight and spills), but its branches keep a
// face's loads behind the face before, which small meshes wait for.
enum class Ext { none, absorbing, materials, any };
// Told apart where at most every other SM has a CTA (1 296 tetrahedra: absorbing 6.6 -> 5.6 us a
// stage, materials 6.7 -> 6.2, tiles 6.0 and 6.2; 6 000: 6.9 -> 5.9, 7.2 -> 6.5, tiles 10.1 and 10.4;
// 10 368, 81 CTAs: 8.2 and 8.6, told apart 8.6 and 9.1).
inline Ext direct_ext(bool materials, bool absorbing, int grid, int num_sms) {
  if (!materials && !absorbing) return Ext::none;
  if (2 * grid > num_sms) return Ext::any;
  return materials ? Ext::materials : Ext::absorbing;
}

template <int N, bool RK, Ext EXT>
__global__ void __launch_bounds__(kDirectThreads, 4)
direct_stage_kernel(const __grid_constant__ StageArgs A, const __grid_constant__ DirectOps<N> O) {
  constexpr int Np = DirectOps<N>::Np, Nfp = DirectOps<N>::Nfp, NF = 4 * Nfp;
  constexpr int TE = tc_tile_elems(N);
  const bool mat = EXT == Ext::materials || (EXT == Ext::any && A.mat);
  static_assert(Np == 4, "a row is one 16-byte word");
  pdl_launch_dependents();
  const int k = A.tile0 + int(blockIdx.x) * kDirectThreads + int(threadIdx.x);   // first element: tile0
  const int K = A.K;
  // geometry: constant data, read before the previous stage's fields are complete
  const bool live = k < A.tile0 + A.num_tiles;
  const int kk = live ? k : A.tile0, tile = kk / TE, ke = kk - tile * TE;
  const float* g = A.tcgeo + size_t(tile) * A.tc_geo_stride + ke;
  float met[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) met[a] = __ldg(g + a * TE);
  const unsigned codes = __float_as_uint(__ldg(g + 9 * TE));
  const unsigned* nodes = reinterpret_cast<const unsigned*>(
      A.tcgeo + size_t(tile) * A.tc_geo_stride + kTcGeoWords * TE) + ke * (NF / 4);
  unsigned nb[NF / 4];                             // matching node of face node m: byte m
#pragma unroll
  for (int q = 0; q < NF / 4; ++q) nb[q] = __ldg(nodes + q);
  int k2[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) k2[f] = __float_as_int(__ldg(g + (26 + f) * TE));
  pdl_wait();
  if (!live) return;
  if (RK) {                                        // on its way from HBM until the update reads it
#pragma unroll
    for (int c = 0; c < 6; ++c)
      asm volatile("prefetch.global.L2 [%0];"
                   :: "l"(reinterpret_cast<const float4*>(A.res) + size_t(c) * K + k));
  }

  const float4* U = reinterpret_cast<const float4*>(A.u_in);
  float wE = 1.f, wH = 1.f;                        // rhs_E / eps, rhs_H / mu
  if constexpr (EXT == Ext::materials) {
    const float4 w = __ldg(A.mat + size_t(k) * kMatVecs);
    wE = w.x;
    wH = w.y;
  }
  float u[6][Np];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const float4 x = __ldg(U + size_t(c) * K + k);
    u[c][0] = x.x; u[c][1] = x.y; u[c][2] = x.z; u[c][3] = x.w;
  }
  float rhs[6][Np];
  // local differentiation and curl, H fields first (dE/dt = curl H), then E
  const float rx = met[0], ry = met[1], rz = met[2];
  const float sx = met[3], sy = met[4], sz = met[5];
  const float tx = met[6], ty = met[7], tz = met[8];
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    const int fb = pass == 0 ? 3 : 0;
#pragma unroll
    for (int i = 0; i < Np; ++i) {
      float acc[3][3];                             // [field][r, s, t]
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          acc[c][m] = 0.f;
#pragma unroll
          for (int j = 0; j < Np; ++j) acc[c][m] = fmaf(O.D[m][i][j], u[fb + c][j], acc[c][m]);
        }
      float dx[3], dy[3], dz[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        dx[c] = rx * acc[c][0] + sx * acc[c][1] + tx * acc[c][2];
        dy[c] = ry * acc[c][0] + sy * acc[c][1] + ty * acc[c][2];
        dz[c] = rz * acc[c][0] + sz * acc[c][1] + tz * acc[c][2];
      }
      const float cx = dy[2] - dz[1], cy = dz[0] - dx[2], cz = dx[1] - dy[0];
      if (pass == 0) {
        rhs[0][i] = cx; rhs[1][i] = cy; rhs[2][i] = cz;
      } else {
        rhs[3][i] = -cx; rhs[4][i] = -cy; rhs[5][i] = -cz;
      }
    }
  }
  // face by face: neighbour rows, upwind flux of its nodes, lifting
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const unsigned code = (codes >> (8 * f)) & 0xffu;
    const bool absorbing = EXT != Ext::none && code == kAbsorbingCode, wall = code == 0u || absorbing;
    float n[6][Np];                                // neighbour rows (walls: the element's own)
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float4 x = __ldg(U + size_t(c) * K + (wall ? k : k2[f]));
      n[c][0] = x.x; n[c][1] = x.y; n[c][2] = x.z; n[c][3] = x.w;
    }
    const float nx = __ldg(g + (10 + 4 * f) * TE), ny = __ldg(g + (11 + 4 * f) * TE);
    const float nz = __ldg(g + (12 + 4 * f) * TE), sc = 0.5f * __ldg(g + (13 + 4 * f) * TE);
    float4 cf = make_float4(1.f, 0.5f, 1.f, 0.5f);
    if (mat) cf = __ldg(A.mat + size_t(k) * kMatVecs + 1 + f);
    const float al = A.alpha;
#pragma unroll
    for (int j = 0; j < Nfp; ++j) {
      constexpr int FN[4][3] = {
          {direct_face_node(1, 0, 0), direct_face_node(1, 0, 1), direct_face_node(1, 0, 2)},
          {direct_face_node(1, 1, 0), direct_face_node(1, 1, 1), direct_face_node(1, 1, 2)},
          {direct_face_node(1, 2, 0), direct_face_node(1, 2, 1), direct_face_node(1, 2, 2)},
          {direct_face_node(1, 3, 0), direct_face_node(1, 3, 1), direct_face_node(1, 3, 2)}};
      const int iM = FN[f][j], m = f * Nfp + j;
      const unsigned i2 = wall ? unsigned(iM) : (nb[m / 4] >> (8 * (m % 4))) & 3u;
      const bool hi = i2 & 2u, lo = i2 & 1u;
      float up[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const float a = lo ? n[c][1] : n[c][0], b = lo ? n[c][3] : n[c][2];
        up[c] = hi ? b : a;
        if (absorbing) up[c] = 0.f;                // absorbing: exterior state zero
      }
      if (wall && !absorbing) {                    // conductor: E+ = -E-
#pragma unroll
        for (int c = 0; c < 3; ++c) up[c] = -up[c];
      }
      const float dEx = u[0][iM] - up[0], dEy = u[1][iM] - up[1], dEz = u[2][iM] - up[2];
      const float dHx = u[3][iM] - up[3], dHy = u[4][iM] - up[4], dHz = u[5][iM] - up[5];
      const float ndE = nx * dEx + ny * dEy + nz * dEz;
      const float ndH = nx * dHx + ny * dHy + nz * dHz;
      // E: -n x dH + alpha (n (n.dE) - dE);  H: n x dE + alpha (n (n.dH) - dH), with
      // impedances as in stage_kernel.cuh (the same expressions: the same rounding)
      float fl[6];
      if (!mat) {
        const float v[6] = {
            -(ny * dHz - nz * dHy) + al * (nx * ndE - dEx),
            -(nz * dHx - nx * dHz) + al * (ny * ndE - dEy),
            -(nx * dHy - ny * dHx) + al * (nz * ndE - dEz),
            (ny * dEz - nz * dEy) + al * (nx * ndH - dHx),
            (nz * dEx - nx * dEz) + al * (ny * ndH - dHy),
            (nx * dEy - ny * dEx) + al * (nz * ndH - dHz)};
#pragma unroll
        for (int c = 0; c < 6; ++c) fl[c] = sc * v[c];
      } else {
        const float fs = 2.f * sc, sE = fs * cf.y, sH = fs * cf.w;
        const float v[6] = {
            fmaf(al, nx * ndE - dEx, cf.x * -(ny * dHz - nz * dHy)),
            fmaf(al, ny * ndE - dEy, cf.x * -(nz * dHx - nx * dHz)),
            fmaf(al, nz * ndE - dEz, cf.x * -(nx * dHy - ny * dHx)),
            fmaf(al, nx * ndH - dHx, cf.z * (ny * dEz - nz * dEy)),
            fmaf(al, ny * ndH - dHy, cf.z * (nz * dEx - nx * dEz)),
            fmaf(al, nz * ndH - dHz, cf.z * (nx * dEy - ny * dEx))};
#pragma unroll
        for (int c = 0; c < 6; ++c) fl[c] = (c < 3 ? sE : sH) * v[c];
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
#pragma unroll
        for (int i = 0; i < Np; ++i) rhs[c][i] = fmaf(O.L[i][m], fl[c], rhs[c][i]);
      }
    }
  }
  if constexpr (EXT == Ext::any) {
    if (mat) {
      const float4 w = __ldg(A.mat + size_t(k) * kMatVecs);
      wE = w.x;
      wH = w.y;
    }
  }
  const float dt = RK ? (A.dt_elem ? __ldg(A.dt_elem + k) : A.dt) : 1.f;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    float r[Np];
#pragma unroll
    for (int i = 0; i < Np; ++i) r[i] = EXT != Ext::none ? rhs[c][i] * (c < 3 ? wE : wH) : rhs[c][i];
    const size_t at = size_t(c) * K + k;
    if (RK) {
      const float4 o = reinterpret_cast<const float4*>(A.res)[at];
      const float4 rn = make_float4(fmaf(A.a, o.x, dt * r[0]), fmaf(A.a, o.y, dt * r[1]),
                                    fmaf(A.a, o.z, dt * r[2]), fmaf(A.a, o.w, dt * r[3]));
      reinterpret_cast<float4*>(A.res)[at] = rn;
      reinterpret_cast<float4*>(A.u_out)[at] =
          make_float4(fmaf(A.b, rn.x, u[c][0]), fmaf(A.b, rn.y, u[c][1]),
                      fmaf(A.b, rn.z, u[c][2]), fmaf(A.b, rn.w, u[c][3]));
    } else {
      reinterpret_cast<float4*>(A.rhs)[at] = make_float4(r[0], r[1], r[2], r[3]);
    }
  }
}

}  // namespace dgdev
