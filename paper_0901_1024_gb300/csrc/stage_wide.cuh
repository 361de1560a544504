// FP32 RK stage of orders 8 and 9 (CUDA cores), register tiled.
//
// The arithmetic is that of stage_kernel.cuh, value for value and in the same order:
// results are the same bit for bit.  The multiply-adds bound it (N = 8: 11.0 G on 16 464
// tetrahedra, 273 us at the FP32 peak).  The tiled stage gives a thread 3 or 4 matrix
// rows of one element and reads 4 floats of Dr, Ds, Dt (one of them padding) per row and
// column for 9 multiply-adds, twice a tile (27 % of the peak).  Here
//   * a thread holds 7 rows of one element for all six fields at once, 126
//     accumulators, so that every Dr, Ds, Dt value read serves six multiply-adds, and two
//     columns cost 21 + 6 8-byte loads for 252 multiply-adds;
//   * the operator comes packed ([chunk of JC columns][row][column][r, s, t]) through two
//     shared-memory buffers, one bulk copy a chunk, the next chunk's under way while one
//     is multiplied; LIFT follows through the same buffers.
// Measured (~1.7e7 unknowns, before and after): N = 8 1014 -> 720-730 us, N = 9 1214 -> 940-950
// us; 37 and 40 % of the FP32 peak.  Half of the cycles issue nothing (N = 8: issue 52 %, FMA
// pipe 43 %): first for the global loads of staging, fluxes and update, which no multiply-add
// of the CTA runs beside (long scoreboard 1.29 per issued instruction), then for register
// banks in the loop (dispatch 0.86).  Two CTAs an SM with half the tile 732 / 965 us, packed
// FP32x2 multiply-adds with 8 rows a thread 747 / 957 us.
#pragma once

#include <algorithm>

#include <cuda_runtime.h>

#include "device.h"
#include "launch.cuh"
#include "tc_stage.cuh"
#include "tcgen05.cuh"

namespace dgdev {

template <int N> struct WideDims {
  static constexpr int Np = (N + 1) * (N + 2) * (N + 3) / 6;
  static constexpr int Nfp = (N + 1) * (N + 2) / 2;
  static constexpr int NF = 4 * Nfp;
  static constexpr int E = N == 8 ? 16 : 8, R = 7;             // elements of a tile; rows of a thread
  static constexpr int TE = stage_tile_elems(N);               // unit of StageArgs' tile0, num_tiles
  static constexpr int G = (Np + R - 1) / R, T = E * G;       // row groups; threads
  static constexpr int JC = wide_jc(N), NCH = wide_chunks(N), JP = JC * NCH;
  static constexpr int MC = wide_mc(N), NLC = NF / 4 / MC;
  static constexpr int CHB = wide_chunk_bytes(N);              // bytes of a chunk slot
  static constexpr int US = (JP / 2) % 2 ? JP : JP + 2;        // 8-byte reads of 16 rows: no conflicts
  static constexpr int FS = (NF / 4) % 2 ? NF : NF + 4;        // 16-byte reads of 8 rows: none
  static constexpr int UT = 6 * E * US, FT = 6 * E * (FS > US ? FS : US), GT = E * kGeoWords;
  static constexpr int OFF_C = 0, OFF_U = 2 * CHB, OFF_F = OFF_U + UT * 4, OFF_G = OFF_F + FT * 4;
  static constexpr int SMEM = OFF_G + GT * 4;
  static_assert(T % 32 == 0 && T <= 512 && JC % 2 == 0 && JP >= Np && NF / 4 % MC == 0, "tiling");
  static_assert(CHB % 128 == 0 && Np * JC * 12 <= CHB && Np * MC * 16 <= CHB, "chunk slot");
  static_assert((UT * 4) % 16 == 0 && (FT * 4) % 16 == 0 && US % 2 == 0 && SMEM <= 227 * 1024 - 64,
                "shared memory");
};

template <int N, bool RK, bool EXT>
__global__ void __launch_bounds__(WideDims<N>::T, 1) stage_wide_kernel(const __grid_constant__ StageArgs A) {
  using D = WideDims<N>;
  constexpr int E = D::E, G = D::G, Np = D::Np, Nfp = D::Nfp, NF = D::NF, R = D::R;
  constexpr int US = D::US, FS = D::FS, JC = D::JC, MC = D::MC, NCH = D::NCH;
  constexpr int CHUNKS = D::NCH + D::NLC;            // chunks of a tile
  extern __shared__ __align__(1024) unsigned char smem[];
  float* su = reinterpret_cast<float*>(smem + D::OFF_U);
  float* sf = reinterpret_cast<float*>(smem + D::OFF_F);
  float* sg = reinterpret_cast<float*>(smem + D::OFF_G);
  __shared__ __align__(8) uint64_t s_full[2];
  pdl_launch_dependents();
  const int tid = threadIdx.x, e = tid % E, g = tid / E, K = A.K;
  const int first = A.tile0 * D::TE, last = min(K, (A.tile0 + A.num_tiles) * D::TE);   // elements
  const int ntiles = ((last - first + E - 1) / E - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x);
  const int total = ntiles * CHUNKS;
  // chunk n of this CTA (its tiles' chunks in a row) into buffer n & 1; the buffer's
  // last readers have passed a barrier
  auto issue = [&](int n) {
    if (n < total) {
      const int c = n % CHUNKS;
      const uint32_t bytes = c < NCH ? (Np * JC * 12 + 15) & ~15 : Np * MC * 16;
      tc::fence_proxy_async_smem();
      tc::mbar_expect_tx(&s_full[n & 1], bytes);
      tc::bulk_g2s(smem + D::OFF_C + (n & 1) * D::CHB,
                   static_cast<const unsigned char*>(A.wide) + size_t(c) * D::CHB, bytes,
                   &s_full[n & 1]);
    }
  };
  if (tid == 0) {
    tc::mbar_init(&s_full[0], 1);
    tc::mbar_init(&s_full[1], 1);
    tc::fence_mbar_init();
    issue(0);                                        // constant data: may overlap the previous kernel
    issue(1);
  }
  // columns past the last node multiply zeros of the packed operator: keep them finite
  for (int i = tid; i < 6 * E * (US - Np); i += D::T)
    su[i / (US - Np) * US + Np + i % (US - Np)] = 0.f;
  __syncthreads();
  pdl_wait();

  int n = 0;                                         // chunk being multiplied
  for (int t = 0; t < ntiles; ++t) {
    const int k0 = first + (int(blockIdx.x) + t * int(gridDim.x)) * E, Ev = min(E, last - k0);
    // ---- stage geometry and fields (asynchronous copies, all in flight) --------
    for (int idx = tid; idx < Ev * (kGeoWords / 4); idx += D::T)
      tc::cp_async16(reinterpret_cast<float4*>(sg) + idx, &A.geo[size_t(k0) * (kGeoWords / 4) + idx]);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float* src = A.u_in + (size_t(c) * K + k0) * Np;
      for (int idx = tid; idx < Ev * Np; idx += D::T) {
        const int ee = idx / Np, i = idx - ee * Np;
        tc::cp_async4(su + (c * E + ee) * US + i, src + idx);
      }
    }
    tc::cp_async_commit();
    tc::cp_async_wait_all();
    __syncthreads();

    // ---- flux extraction ---------------------------------------------------------
    if (e < Ev) {
      const float* ge = sg + e * kGeoWords;
      const unsigned codes = __float_as_uint(ge[10]);
#pragma unroll 2
      for (int m = g; m < NF; m += G) {
        const int f = m / Nfp, j = m - f * Nfp;
        const int idM = __ldg(A.fmask + m);
        float uM[6], uP[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) uM[c] = su[(c * E + e) * US + idM];
        const unsigned code = (codes >> (8 * f)) & 0xffu;
        if (code == 0u) {                       // perfectly conducting wall
#pragma unroll
          for (int c = 0; c < 3; ++c) { uP[c] = -uM[c]; uP[c + 3] = uM[c + 3]; }
        } else if (EXT && code == kAbsorbingCode) {   // characteristic absorbing: no incoming wave
#pragma unroll
          for (int c = 0; c < 6; ++c) uP[c] = 0.f;
        } else {
          const int k2 = __float_as_int(ge[28 + f]);
          const int i2 = __ldg(A.perm + (f * 24 + int(code) - 1) * Nfp + j);
          const int e2 = k2 - k0;
          if (e2 >= 0 && e2 < Ev) {
#pragma unroll
            for (int c = 0; c < 6; ++c) uP[c] = su[(c * E + e2) * US + i2];
          } else {
#pragma unroll
            for (int c = 0; c < 6; ++c) uP[c] = __ldg(A.u_in + (size_t(c) * K + k2) * Np + i2);
          }
        }
        const float nx = ge[12 + 4 * f], ny = ge[13 + 4 * f], nz = ge[14 + 4 * f];
        const float sc = 0.5f * ge[15 + 4 * f];
        const float dEx = uM[0] - uP[0], dEy = uM[1] - uP[1], dEz = uM[2] - uP[2];
        const float dHx = uM[3] - uP[3], dHy = uM[4] - uP[4], dHz = uM[5] - uP[5];
        const float ndE = nx * dEx + ny * dEy + nz * dEz;
        const float ndH = nx * dHx + ny * dHy + nz * dHz;
        const float al = A.alpha;
        if (!EXT || !A.mat) {
          const float fl[6] = {
              -(ny * dHz - nz * dHy) + al * (nx * ndE - dEx),
              -(nz * dHx - nx * dHz) + al * (ny * ndE - dEy),
              -(nx * dHy - ny * dHx) + al * (nz * ndE - dEz),
              (ny * dEz - nz * dEy) + al * (nx * ndH - dHx),
              (nz * dEx - nx * dEz) + al * (ny * ndH - dHy),
              (nx * dEy - ny * dEx) + al * (nz * ndH - dHz)};
#pragma unroll
          for (int c = 0; c < 6; ++c) sf[(c * E + e) * FS + m] = sc * fl[c];
        } else {
          const float4 cf = __ldg(A.mat + size_t(k0 + e) * kMatVecs + 1 + f);
          const float fs = 2.f * sc, sE = fs * cf.y, sH = fs * cf.w;
          const float fl[6] = {
              cf.x * -(ny * dHz - nz * dHy) + al * (nx * ndE - dEx),
              cf.x * -(nz * dHx - nx * dHz) + al * (ny * ndE - dEy),
              cf.x * -(nx * dHy - ny * dHx) + al * (nz * ndE - dEz),
              cf.z * (ny * dEz - nz * dEy) + al * (nx * ndH - dHx),
              cf.z * (nz * dEx - nx * dEz) + al * (ny * ndH - dHy),
              cf.z * (nx * dEy - ny * dEx) + al * (nz * ndH - dHz)};
#pragma unroll
          for (int c = 0; c < 6; ++c) sf[(c * E + e) * FS + m] = (c < 3 ? sE : sH) * fl[c];
        }
      }
    }
    // (the first operator chunk's barriers come after every flux is stored: LIFT follows)

    // ---- local differentiation of all six fields ------------------------------------
    int row[R];
#pragma unroll
    for (int q = 0; q < R; ++q) row[q] = min(g + G * q, Np - 1);
    float acc[6][3][R];
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int q = 0; q < R; ++q) acc[c][d][q] = 0.f;
    const float* ue = su + e * US;
#pragma unroll 1
    for (int c0 = 0; c0 < NCH; ++c0, ++n) {
      wait_or_flag(&s_full[n & 1], (n >> 1) & 1, A.status);
      const float* cb = reinterpret_cast<const float*>(smem + D::OFF_C + (n & 1) * D::CHB);
#pragma unroll 1
      for (int jj = 0; jj < JC; jj += 2) {
        float2 v[6];
#pragma unroll
        for (int c = 0; c < 6; ++c)
          v[c] = *reinterpret_cast<const float2*>(ue + c * E * US + c0 * JC + jj);
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float2* d = reinterpret_cast<const float2*>(cb + (row[q] * JC + jj) * 3);
          const float2 x = d[0], y = d[1], z = d[2];   // r s, t r', s' t'
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            acc[c][0][q] = fmaf(x.x, v[c].x, acc[c][0][q]);
            acc[c][1][q] = fmaf(x.y, v[c].x, acc[c][1][q]);
            acc[c][2][q] = fmaf(y.x, v[c].x, acc[c][2][q]);
            acc[c][0][q] = fmaf(y.y, v[c].y, acc[c][0][q]);
            acc[c][1][q] = fmaf(z.x, v[c].y, acc[c][1][q]);
            acc[c][2][q] = fmaf(z.y, v[c].y, acc[c][2][q]);
          }
        }
      }
      __syncthreads();                               // buffer n & 1 may be refilled
      if (tid == 0) issue(n + 2);
    }
    // ---- chain rule and curl ---------------------------------------------------------
    float rhs[6][R];
    {
      const float* ge = sg + e * kGeoWords;
      const float rx = ge[0], ry = ge[1], rz = ge[2];
      const float sx = ge[3], sy = ge[4], sz = ge[5];
      const float tx = ge[6], ty = ge[7], tz = ge[8];
#pragma unroll
      for (int pass = 0; pass < 2; ++pass) {
        const int fb = pass == 0 ? 3 : 0;            // H fields first (curl H), then E
#pragma unroll
        for (int q = 0; q < R; ++q) {
          float dx[3], dy[3], dz[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            dx[c] = rx * acc[fb + c][0][q] + sx * acc[fb + c][1][q] + tx * acc[fb + c][2][q];
            dy[c] = ry * acc[fb + c][0][q] + sy * acc[fb + c][1][q] + ty * acc[fb + c][2][q];
            dz[c] = rz * acc[fb + c][0][q] + sz * acc[fb + c][1][q] + tz * acc[fb + c][2][q];
          }
          const float cx = dy[2] - dz[1], cy = dz[0] - dx[2], cz = dx[1] - dy[0];
          if (pass == 0) {        // dE/dt = curl H
            rhs[0][q] = cx; rhs[1][q] = cy; rhs[2][q] = cz;
          } else {                // dH/dt = -curl E
            rhs[3][q] = -cx; rhs[4][q] = -cy; rhs[5][q] = -cz;
          }
        }
      }
    }
    // ---- lifting -----------------------------------------------------------------------
    const float4* f4[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) f4[c] = reinterpret_cast<const float4*>(sf + (c * E + e) * FS);
#pragma unroll 1
    for (int lc = 0; lc < D::NLC; ++lc, ++n) {
      wait_or_flag(&s_full[n & 1], (n >> 1) & 1, A.status);
      const float4* cb = reinterpret_cast<const float4*>(smem + D::OFF_C + (n & 1) * D::CHB);
#pragma unroll 1
      for (int mm = 0; mm < MC; ++mm) {
        float4 fv[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) fv[c] = f4[c][lc * MC + mm];
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float4 L = cb[row[q] * MC + mm];
#pragma unroll
          for (int c = 0; c < 6; ++c) {
            float s = rhs[c][q];
            s = fmaf(L.x, fv[c].x, s);
            s = fmaf(L.y, fv[c].y, s);
            s = fmaf(L.z, fv[c].z, s);
            s = fmaf(L.w, fv[c].w, s);
            rhs[c][q] = s;
          }
        }
      }
      __syncthreads();                               // buffer free; after the last: the fluxes too
      if (tid == 0) issue(n + 2);
    }
    // ---- update through a staged copy of rhs, coalesced ----------------------------------
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = g + G * q;
      if (i < Np && e < Ev) {
#pragma unroll
        for (int c = 0; c < 6; ++c) sf[(c * E + e) * US + i] = rhs[c][q];
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const size_t base = (size_t(c) * K + k0) * Np;
#pragma unroll 4
      for (int idx = tid; idx < Ev * Np; idx += D::T) {
        const int ee = idx / Np, i = idx - ee * Np;
        float r = sf[(c * E + ee) * US + i];
        if (EXT && A.mat) {                          // rhs_E / eps, rhs_H / mu
          const float4 w = __ldg(A.mat + size_t(k0 + ee) * kMatVecs);
          r *= c < 3 ? w.x : w.y;
        }
        if (RK) {
          const float dtk = A.dt_elem ? __ldg(A.dt_elem + k0 + ee) : A.dt;
          const float rn = fmaf(A.a, A.res[base + idx], dtk * r);
          A.res[base + idx] = rn;
          A.u_out[base + idx] = fmaf(A.b, rn, su[(c * E + ee) * US + i]);
        } else {
          A.rhs[base + idx] = r;
        }
      }
    }
    __syncthreads();
  }
  // every chunk has been waited for; after a wait that ran out, once more (as bounded) for
  // the last copy into each buffer before the shared memory is given up
  if (tid == 0)
    for (int i = max(n - 2, 0); i < n; ++i) wait_or_flag(&s_full[i & 1], (i >> 1) & 1, A.status);
}

template <int N>
cudaError_t launch_stage_wide(bool rk, const StageArgs& a, int num_sms, cudaStream_t s) {
  using D = WideDims<N>;
  static bool attr[2][2][16] = {};      // [rk][ext][device]: attribute set
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  const bool ext = a.mat || a.absorbing;
  auto kern = rk ? (ext ? stage_wide_kernel<N, true, true> : stage_wide_kernel<N, true, false>)
                 : (ext ? stage_wide_kernel<N, false, true> : stage_wide_kernel<N, false, false>);
  bool& done = attr[rk ? 1 : 0][ext ? 1 : 0][dev & 15];
  if (!done) {
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, D::SMEM);
    if (err != cudaSuccess) return err;
    done = true;
  }
  const int tiles = (std::min(a.K - a.tile0 * D::TE, a.num_tiles * D::TE) + D::E - 1) / D::E;
  const int grid = tiles < num_sms ? tiles : num_sms;
  if (grid <= 0) return cudaSuccess;
  return launch_pdl(kern, grid, D::T, D::SMEM, s, a);
}

}  // namespace dgdev
