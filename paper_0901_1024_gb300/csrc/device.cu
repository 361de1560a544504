// Device buffers of a mesh, kernel dispatch, the energy reduction and the
// host-facing device operations behind the C ABI.
#include <algorithm>
#include <cstdint>
#include <initializer_list>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <map>
#include <mutex>
#include <vector>

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "device.h"
#include "dg_internal.h"
#include "tcgen05.cuh"

namespace dgdev {

template <int N>
cudaError_t launch_stage_n(bool rk, const StageArgs& a, int num_sms, cudaStream_t s, int shape);

template <int N>
cudaError_t launch_tc_stage_n(bool rk, const StageArgs& a, int num_sms, cudaStream_t s);
template <int N>
cudaError_t launch_tt_stage_n(bool rk, const StageArgs& a, int num_sms, cudaStream_t s);

cudaError_t launch_tc_stage(int N, bool rk, const StageArgs& a, int num_sms, cudaStream_t s) {
  switch (N) {
    case 1: return launch_tc_stage_n<1>(rk, a, num_sms, s);
    case 2: return launch_tc_stage_n<2>(rk, a, num_sms, s);
    case 3: return launch_tc_stage_n<3>(rk, a, num_sms, s);
    case 4: return launch_tc_stage_n<4>(rk, a, num_sms, s);
    case 5: return launch_tt_stage_n<5>(rk, a, num_sms, s);
    case 6: return launch_tt_stage_n<6>(rk, a, num_sms, s);
    case 7: return launch_tt_stage_n<7>(rk, a, num_sms, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_stage(int N, bool rk, const StageArgs& a, int num_sms, cudaStream_t s,
                         int shape) {
  switch (N) {
    case 1: return launch_stage_n<1>(rk, a, num_sms, s, shape);
    case 2: return launch_stage_n<2>(rk, a, num_sms, s, shape);
    case 3: return launch_stage_n<3>(rk, a, num_sms, s, shape);
    case 4: return launch_stage_n<4>(rk, a, num_sms, s, shape);
    case 5: return launch_stage_n<5>(rk, a, num_sms, s, shape);
    case 6: return launch_stage_n<6>(rk, a, num_sms, s, shape);
    case 7: return launch_stage_n<7>(rk, a, num_sms, s, shape);
    case 8: return launch_stage_n<8>(rk, a, num_sms, s, shape);
    case 9: return launch_stage_n<9>(rk, a, num_sms, s, shape);
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------- energy -----
// E = 1/2 sum_k J_k sum_c u_kc^T M u_kc.  Each block writes one FP64 partial
// (its threads' sums, added in a fixed order) and a one-warp kernel adds the
// partials in a fixed order, so the result is deterministic.
//
// With T_ji = M_ii, 2 M_ij for j > i, 0 for j < i (M symmetric), u^T M u =
// sum_i u_i s_i, s_i = sum_{j >= i} T_ji u_j: a small triangular matrix product over
// all rows (c, k).  It is bound by FP32 arithmetic from N = 6 on (N = 9: 3.8 GFLOP on
// 1.7e7 unknowns, 48 us at the FP32 peak, against 10 us to read the fields) and by
// reading them below.  So it runs as a register-tiled product: blocks of 32 outputs i
// (the triangle is skipped at that grain), a warp forms 32 rows x 32 outputs of one
// block, a lane 8 rows x 4 outputs, and 4 columns j cost it 12 16-byte shared loads for
// 128 multiply-adds (the row-per-thread kernels before it loaded 32 bytes of M for 8 or
// 16, with one to eight warps an SM).  T and a pass of rows sit in shared memory; the
// (row set, output block) tasks go to the warps longest first, every second round in
// reverse, which balances the triangle.  FP32 products and row sums, FP64 sums of the
// weighted rows.  A whole dg_energy call on ~1.7e7 unknowns (35 us of it launches, copy
// and synchronisation), before and after: N = 9 1184 -> 160 us, N = 8 515 -> 127, N = 7
// 207 -> 98, N = 6 122 -> 86, N = 5 110 -> 76, N = 4 83 -> 76, N = 3 84 -> 64.  The
// Jacobians are read from an array of their own: from the 128-byte element records each
// row would fetch a whole sector for one word.
template <int N> struct EnergyShape {
  static constexpr int NP = (N + 1) * (N + 2) * (N + 3) / 6;
  static constexpr int NP4 = (NP + 3) & ~3;            // row stride: 4 rows of a warp never share banks
  static constexpr int NB = (NP + 31) / 32;            // output blocks
  static constexpr int RSETS = N == 8 ? 2 : 4;         // row sets of 32 per pass
  static constexpr int ROWS = 32 * RSETS;
  static constexpr int WARPS = N == 9 ? 14 : N == 8 ? 6 : N >= 6 ? 8 : 4;
  static constexpr int THREADS = 32 * WARPS, MIN_BLOCKS = N == 9 ? 1 : N >= 6 ? 2 : 4;
  __host__ __device__ static constexpr int t_off(int ob) {   // first float of output block ob
    int o = 0;
    for (int b = 0; b < ob; ++b) o += (NP4 - 32 * b) * 32;
    return o;
  }
  static constexpr int T_FLOATS = t_off(NB);           // [block][j - 32 block][32 outputs]
  static constexpr int BYTES = (T_FLOATS + ROWS * NP4) * 4 + ROWS * 12;
  static_assert(NP4 % 32 % 16 != 0, "bank-conflict-free row reads");
  static_assert(BYTES <= 227 * 1024, "shared memory");
};

template <int N, bool VEC, class Index>
__global__ void __launch_bounds__(EnergyShape<N>::THREADS, EnergyShape<N>::MIN_BLOCKS)
energy_tile_kernel(const EnergyArgs A) {
  using S = EnergyShape<N>;
  constexpr int NP = S::NP, NP4 = S::NP4, NB = S::NB, ROWS = S::ROWS, TH = S::THREADS;
  extern __shared__ __align__(16) float esm[];
  float* sT = esm;
  float* sU = esm + S::T_FLOATS;                       // [ROWS][NP4]
  int64_t* sRow = reinterpret_cast<int64_t*>(sU + ROWS * NP4);
  float* sW = reinterpret_cast<float*>(sRow + ROWS);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rg = lane >> 3, og = lane & 7;
  for (int i = tid; i < S::T_FLOATS / 4; i += TH)
    tc::cp_async16(reinterpret_cast<float4*>(sT) + i, reinterpret_cast<const float4*>(A.T) + i);
  if constexpr (NP4 != NP)                             // padding columns stay zero
    for (int i = tid; i < ROWS * (NP4 - NP); i += TH)
      sU[i / (NP4 - NP) * NP4 + NP + i % (NP4 - NP)] = 0.f;
  const Index rows = Index(energy_rows(A.k0, A.k1)), step = Index(gridDim.x) * ROWS;
  double acc = 0.0;
  for (Index r0 = Index(blockIdx.x) * ROWS; r0 < rows; r0 += step) {
    const int nr = int(min(rows - r0, Index(ROWS)));
    __syncthreads();                                   // the previous pass is consumed
    for (int i = tid; i < nr; i += TH) {
      const auto [c, kr] = energy_row<Index>(r0 + i, A.k0, A.k1);
      const int64_t k = A.k0 + kr;
      sRow[i] = (int64_t(c) * A.K + k) * NP;
      float wgt = __ldg(A.J + k);
      if (A.mat) {
        const float4 m = __ldg(A.mat + k * kMatVecs);
        wgt *= c < 3 ? m.z : m.w;
      }
      sW[i] = wgt;                                     // J_k (times eps_k or mu_k)
    }
    __syncthreads();
    if constexpr (VEC) {                               // whole 16-byte words
      for (int i = tid; i < nr * (NP / 4); i += TH) {
        const int r = i / (NP / 4), q = i - r * (NP / 4);
        tc::cp_async16(reinterpret_cast<float4*>(sU + r * NP4) + q,
                       reinterpret_cast<const float4*>(A.u + sRow[r]) + q);
      }
    } else {
      for (int i = tid; i < nr * NP; i += TH) {
        const int r = i / NP, j = i - r * NP;
        tc::cp_async4(sU + r * NP4 + j, A.u + sRow[r] + j);
      }
    }
    tc::cp_async_commit();
    tc::cp_async_wait_all();
    __syncthreads();
#pragma unroll 1
    for (int round = 0; round * S::WARPS < NB * S::RSETS; ++round) {
      const int task = round * S::WARPS + (round & 1 ? S::WARPS - 1 - warp : warp);
      if (task >= NB * S::RSETS) continue;
      const int ob = task / S::RSETS, row0 = (task - ob * S::RSETS) * 32 + rg;   // rows row0 + 4 i
      if (row0 - rg >= nr) continue;
      const float* u0 = sU + row0 * NP4;
      const float* t0 = sT + 16 * ob * (2 * NP4 - 32 * (ob - 1)) + og * 4;       // t_off(ob)
      float s[8][4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int x = 0; x < 4; ++x) s[i][x] = 0.f;
#pragma unroll 1
      for (int j = 32 * ob; j < NP4; j += 4) {
        float4 t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) t[q] = *reinterpret_cast<const float4*>(t0 + (j - 32 * ob + q) * 32);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 u = *reinterpret_cast<const float4*>(u0 + 4 * i * NP4 + j);
          const float v[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            s[i][0] = fmaf(t[q].x, v[q], s[i][0]);
            s[i][1] = fmaf(t[q].y, v[q], s[i][1]);
            s[i][2] = fmaf(t[q].z, v[q], s[i][2]);
            s[i][3] = fmaf(t[q].w, v[q], s[i][3]);
          }
        }
      }
      // e_i = sum of u s over this lane's outputs, then over the 8 lanes of the row
      // group: lane og ends with row row0 + 4 og (the same tree for every row)
      float e[8];
      const int i0 = 32 * ob + og * 4;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 u = i0 < NP4 ? *reinterpret_cast<const float4*>(u0 + 4 * i * NP4 + i0)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        e[i] = fmaf(u.w, s[i][3], fmaf(u.z, s[i][2], fmaf(u.y, s[i][1], u.x * s[i][0])));
      }
#pragma unroll
      for (int h = 4; h; h >>= 1) {
        const bool high = og & h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
          const float keep = high ? e[i + h] : e[i], send = high ? e[i] : e[i + h];
          e[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
      }
      const int row = row0 + 4 * og;
      if (row < nr) acc += double(sW[row]) * double(e[0]);
    }
  }
  tc::cp_async_wait_all();
  __shared__ double sw[S::WARPS];
#pragma unroll
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) sw[warp] = acc;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < S::WARPS; ++w) t += sw[w];
    A.partials[blockIdx.x] = t;
  }
}

// One warp: lane l adds partials l, l + 32, ... in order, then a fixed
// butterfly adds the lanes.
__global__ void energy_finalize(const double* partials, int n, double* result) {
  double t = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) t += partials[i];
#pragma unroll
  for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (threadIdx.x == 0) result[0] = 0.5 * t;
}

// Orders 1 and 2 (4 and 10 nodes): a row per thread straight from global memory, the
// packed triangle in shared memory.  Reading the fields bounds it; staging rows for a
// product this small cost more than it saved (a dg_energy call, staged before and now:
// N = 1, 705 894 tets 121 -> 64 us; N = 2, 279 936 tets 83 -> 50 us).  A row sum is one
// chain of multiply-adds at N = 1 and two at N = 2, whichever is the nearer to 64 bits (rms
// over random rows, one chain and two: N = 1 6.57e-8 and 6.71e-8, N = 2 8.38e-8 and 8.06e-8).
template <int NP, bool VEC, class Index>
__global__ void __launch_bounds__(256) energy_row_kernel(const EnergyArgs A) {
  constexpr int NT = NP * (NP + 1) / 2, NT4 = (NT + 3) & ~3;
  __shared__ __align__(16) float sT[NT4];              // rows i: T_ii, T_i+1,i, ...
  for (int x = threadIdx.x; x < NT; x += 256) {
    int i = 0, o = x;
    while (o >= NP - i) o -= NP - i++;
    sT[x] = __ldg(A.T + (i + o) * 32 + i);
  }
  __syncthreads();
  const Index rows = Index(energy_rows(A.k0, A.k1)), step = Index(gridDim.x) * 256;
  double acc = 0.0;
#pragma unroll 2
  for (Index g = Index(blockIdx.x) * 256 + threadIdx.x; g < rows; g += step) {
    const auto [c, kr] = energy_row<Index>(g, A.k0, A.k1);
    const int64_t k = A.k0 + kr;
    const float* row = A.u + (int64_t(c) * A.K + k) * NP;
    float u[NP];
    if constexpr (VEC) {
#pragma unroll
      for (int q = 0; q < NP / 4; ++q) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(row) + q);
        u[4 * q] = x.x; u[4 * q + 1] = x.y; u[4 * q + 2] = x.z; u[4 * q + 3] = x.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NP; ++j) u[j] = __ldg(row + j);
    }
    float wgt = __ldg(A.J + k);
    if (A.mat) {
      const float4 m = __ldg(A.mat + k * kMatVecs);
      wgt *= c < 3 ? m.z : m.w;
    }
    float e = 0.f;
    int x = 0;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      float s[2] = {0.f, 0.f};                         // order 2: every other column apart
#pragma unroll
      for (int j = i; j < NP; ++j) {
        float& t = s[NP > 4 ? (j - i) & 1 : 0];
        t = fmaf(sT[x++], u[j], t);
      }
      e = fmaf(u[i], NP > 4 ? s[0] + s[1] : s[0], e);
    }
    acc += double(wgt) * double(e);
  }
  __shared__ double sw[8];
#pragma unroll
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += sw[w];
    A.partials[blockIdx.x] = t;
  }
}

// Partial sums kept per mesh; a launch uses as many as it has blocks.
int energy_grid(int num_sms) { return 8 * num_sms; }

template <int NP, bool VEC>
static cudaError_t launch_energy_row(const EnergyArgs& a, int num_sms, int* grid, cudaStream_t s) {
  const int64_t blocks = (energy_rows(a.k0, a.k1) + 255) / 256;
  *grid = int(std::min<int64_t>(blocks, energy_grid(num_sms)));
  if (energy_index32(energy_rows(a.k0, a.k1), int64_t(*grid) * 256))
    energy_row_kernel<NP, VEC, unsigned><<<*grid, 256, 0, s>>>(a);
  else
    energy_row_kernel<NP, VEC, int64_t><<<*grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

template <int N>
static cudaError_t launch_energy_n(const EnergyArgs& a, int num_sms, int* grid, cudaStream_t s) {
  using S = EnergyShape<N>;
  // 16-byte copies where every row starts on a 16-byte boundary
  const bool vec = S::NP % 4 == 0 && reinterpret_cast<uintptr_t>(a.u) % 16 == 0;
  // (the row numbers of meshes past 32 bits: 4-byte copies serve)
  const bool i32 = energy_index32(energy_rows(a.k0, a.k1), int64_t(energy_grid(num_sms)) * S::ROWS);
  auto kern = i32 ? energy_tile_kernel<N, false, unsigned> : energy_tile_kernel<N, false, int64_t>;
  if constexpr (S::NP % 4 == 0)
    if (vec && i32) kern = energy_tile_kernel<N, true, unsigned>;
  static int occ[3][16] = {};                          // [form][device]: blocks per SM
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  int& o = occ[!i32 ? 2 : vec ? 1 : 0][dev & 15];
  if (o == 0) {
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::BYTES);
    if (err != cudaSuccess) return err;
    int n = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, S::THREADS, S::BYTES);
    if (err != cudaSuccess) return err;
    o = n < 1 ? 1 : n > 8 ? 8 : n;
  }
  const int64_t passes = (energy_rows(a.k0, a.k1) + S::ROWS - 1) / S::ROWS;
  *grid = int(std::min<int64_t>(passes, int64_t(num_sms) * o));
  kern<<<*grid, S::THREADS, S::BYTES, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_energy_partials(int N, const EnergyArgs& a, int num_sms, int* grid,
                                   cudaStream_t s) {
  switch (N) {
    case 1: return reinterpret_cast<uintptr_t>(a.u) % 16 == 0
                       ? launch_energy_row<4, true>(a, num_sms, grid, s)
                       : launch_energy_row<4, false>(a, num_sms, grid, s);
    case 2: return launch_energy_row<10, false>(a, num_sms, grid, s);
    case 3: return launch_energy_n<3>(a, num_sms, grid, s);
    case 4: return launch_energy_n<4>(a, num_sms, grid, s);
    case 5: return launch_energy_n<5>(a, num_sms, grid, s);
    case 6: return launch_energy_n<6>(a, num_sms, grid, s);
    case 7: return launch_energy_n<7>(a, num_sms, grid, s);
    case 8: return launch_energy_n<8>(a, num_sms, grid, s);
    case 9: return launch_energy_n<9>(a, num_sms, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_energy_final(const EnergyArgs& a, int grid, cudaStream_t s) {
  energy_finalize<<<1, 32, 0, s>>>(a.partials, grid, a.result);
  return cudaGetLastError();
}

// ------------------------------------------------------- device state -----
struct DeviceState {
  int device = -1;
  int N = 0;
  int64_t K = 0;
  int Np = 0, Nfp = 0;
  int num_sms = 0;
  float4* geo = nullptr;
  float* J = nullptr;           // Jacobians alone (energy)
  float4* D4 = nullptr;
  float4* LIFT4 = nullptr;
  float* M = nullptr;
  float* T = nullptr;
  unsigned char* fmask = nullptr;
  unsigned char* perm = nullptr;
  float* u_work = nullptr;      // second state buffer for the stage ping-pong
  float* h_u = nullptr;         // device copies for dg_step_host
  float* h_res = nullptr;
  cudaStream_t copies = nullptr;   // dg_step_host: copies beside the caller's stream
  cudaEvent_t ready[5] = {};       // and the events between the two
  double* partials = nullptr;   // energy partials, one per block
  double* result = nullptr;
  int egrid = 0;
  void* wide = nullptr;         // packed operator chunks (orders 8, 9)
  void* tcB = nullptr;          // tensor-core B pieces (orders <= kTcMaxOrder)
  float4* mat = nullptr;        // material records (meshes with materials), in the arena
  bool absorbing = false;       // some boundary face is absorbing
  bool scattered = false;       // most faces' neighbours lie far off (order 3: tc_paired)
  float* tcgeo = nullptr;       // word-major geometry for the tensor-core stage
  int tc_geo_stride = 0;
  float tc_inv_bscale = 1.f;
  int* status = nullptr;        // pipeline status word (0 = ok)
  void* arena = nullptr;        // one allocation: geo, tcgeo, status, partials, result
  // D4, LIFT4, M, fmask, perm and tcB belong to the per-(device, order) cache
  // per-launch tracing: event pair 2i, 2i+1 around launch i
  std::vector<cudaEvent_t> ev;
  std::vector<int> kind;
  size_t nrec = 0;
};

void destroy_device_state(DeviceState* d) {
  if (!d) return;
  int cur = -1;
  cudaGetDevice(&cur);
  if (d->device >= 0) cudaSetDevice(d->device);
  cudaFree(d->arena); cudaFree(d->u_work); cudaFree(d->h_u); cudaFree(d->h_res);
  for (cudaEvent_t e : d->ev) cudaEventDestroy(e);
  for (cudaEvent_t e : d->ready)
    if (e) cudaEventDestroy(e);
  if (d->copies) cudaStreamDestroy(d->copies);
  if (cur >= 0) cudaSetDevice(cur);
  delete d;
}

}  // namespace dgdev

namespace dg {
using dgdev::DeviceState;

static int cuda_fail(cudaError_t e, const char* what, std::string& err) {
  err = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? DG_ERR_OOM : DG_ERR_CUDA;
}

#define DG_CUDA(call, what)                                        \
  do {                                                             \
    cudaError_t e_ = (call);                                       \
    if (e_ != cudaSuccess) return cuda_fail(e_, what, err);        \
  } while (0)

template <class T>
static int upload(T** dst, const std::vector<T>& src, std::string& err) {
  DG_CUDA(cudaMalloc(reinterpret_cast<void**>(dst), src.size() * sizeof(T)), "cudaMalloc");
  DG_CUDA(cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice),
          "cudaMemcpy H2D");
  return DG_OK;
}

// Launches `fn` (returning cudaError_t) and, when tracing, brackets it with a
// pair of events on stream s.
template <class F>
static cudaError_t traced(dg_mesh* m, cudaStream_t s, int kind, F&& fn) {
  DeviceState* d = m->dev;
  if (!m->trace) return fn();
  const size_t i = d->nrec;
  while (d->ev.size() < 2 * i + 2) {
    cudaEvent_t e;
    cudaError_t c = cudaEventCreate(&e);
    if (c != cudaSuccess) return c;
    d->ev.push_back(e);
  }
  if (d->kind.size() < i + 1) d->kind.resize(i + 1);
  cudaError_t c = cudaEventRecord(d->ev[2 * i], s);
  if (c != cudaSuccess) return c;
  if ((c = fn()) != cudaSuccess) return c;
  if ((c = cudaEventRecord(d->ev[2 * i + 1], s)) != cudaSuccess) return c;
  d->kind[i] = kind;
  d->nrec = i + 1;
  return cudaSuccess;
}

int ensure_device(dg_mesh* m, std::string& err);

int trace_launch(dg_mesh* m, void* stream, int kind, int (*launch)(void*), void* ctx) {
  return static_cast<int>(traced(m, static_cast<cudaStream_t>(stream), kind,
                                 [&] { return static_cast<cudaError_t>(launch(ctx)); }));
}

int device_trace_reset(dg_mesh* m, int reserve, std::string& err) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  DeviceState* d = m->dev;
  d->nrec = 0;
  while (d->ev.size() < 2 * static_cast<size_t>(reserve)) {
    cudaEvent_t e;
    DG_CUDA(cudaEventCreate(&e), "cudaEventCreate");
    d->ev.push_back(e);
  }
  d->kind.resize(std::max(d->kind.size(), static_cast<size_t>(reserve)));
  return DG_OK;
}

int device_trace_read(dg_mesh* m, double* ms, int32_t* kind, int64_t cap, int64_t* count,
                      std::string& err) {
  DeviceState* d = m->dev;
  if (!d || d->nrec == 0) { err = "no traced launches recorded"; return DG_ERR_STATE; }
  DG_CUDA(cudaEventSynchronize(d->ev[2 * d->nrec - 1]), "cudaEventSynchronize");
  *count = static_cast<int64_t>(d->nrec);
  for (size_t i = 0; i < d->nrec && static_cast<int64_t>(i) < cap; ++i) {
    float t = 0.f;
    DG_CUDA(cudaEventElapsedTime(&t, d->ev[2 * i], d->ev[2 * i + 1]), "cudaEventElapsedTime");
    ms[i] = t;
    if (kind) kind[i] = d->kind[i];
  }
  return DG_OK;
}

// Order-dependent device operators, shared by every mesh of that order on a
// device (built once, kept for the life of the process): Dr/Ds/Dt as float4
// rows, LIFT, M, the face-node tables and the tensor-core B pieces.
struct OrderOps {
  float4* D4 = nullptr;
  float4* LIFT4 = nullptr;
  float* M = nullptr;
  float* T = nullptr;           // weighted triangle of M, energy kernel layout
  unsigned char* fmask = nullptr;
  unsigned char* perm = nullptr;
  void* tcB = nullptr;
  void* wide = nullptr;
  float tc_inv_bscale = 1.f;
};

static std::mutex g_ops_mutex;
static std::map<std::pair<int, int>, OrderOps> g_ops;

static int order_ops(const dg_mesh* m, int dev, OrderOps& out, std::string& err) {
  std::lock_guard<std::mutex> lock(g_ops_mutex);
  auto it = g_ops.find({dev, m->N});
  if (it != g_ops.end()) {
    out = it->second;
    return DG_OK;
  }
  OrderOps o;
  const int Np = m->ops.Np, NF = 4 * m->ops.Nfp;
  std::vector<float4> D4(static_cast<size_t>(Np) * Np);
  for (int i = 0; i < Np; ++i)
    for (int j = 0; j < Np; ++j)
      D4[i * Np + j] = make_float4(static_cast<float>(m->ops.Dr[i * Np + j]),
                                   static_cast<float>(m->ops.Ds[i * Np + j]),
                                   static_cast<float>(m->ops.Dt[i * Np + j]), 0.f);
  int rc;
  if ((rc = upload(&o.D4, D4, err))) return rc;
  std::vector<float4> L4(static_cast<size_t>(Np) * NF / 4);
  for (int i = 0; i < Np; ++i)
    for (int q = 0; q < NF / 4; ++q)
      L4[i * (NF / 4) + q] = make_float4(static_cast<float>(m->ops.LIFT[i * NF + 4 * q + 0]),
                                         static_cast<float>(m->ops.LIFT[i * NF + 4 * q + 1]),
                                         static_cast<float>(m->ops.LIFT[i * NF + 4 * q + 2]),
                                         static_cast<float>(m->ops.LIFT[i * NF + 4 * q + 3]));
  if ((rc = upload(&o.LIFT4, L4, err))) return rc;
  std::vector<float> Mf(m->ops.M.begin(), m->ops.M.end());
  if ((rc = upload(&o.M, Mf, err))) return rc;
  // T_ji = M_ii, 2 M_ij (j > i): [output block of 32][j from the block's first][output]
  {
    const int NP4 = (Np + 3) & ~3;
    std::vector<float> T;
    for (int i0 = 0; i0 < Np; i0 += 32)
      for (int j = i0; j < NP4; ++j)
        for (int i = i0; i < i0 + 32; ++i)
          T.push_back(i >= Np || j >= Np || j < i
                          ? 0.f
                          : (j > i ? 2.f : 1.f) * static_cast<float>(m->ops.M[i * Np + j]));
    if ((rc = upload(&o.T, T, err))) return rc;
  }
  std::vector<unsigned char> fm(m->ops.Fmask.begin(), m->ops.Fmask.end());
  if ((rc = upload(&o.fmask, fm, err))) return rc;
  std::vector<unsigned char> pm(m->ops.perm.begin(), m->ops.perm.end());
  if ((rc = upload(&o.perm, pm, err))) return rc;
  if (m->N > 4 && m->N <= dgdev::kTcMaxOrder) {
    // Orders 5..7: Op = [Dr Ds Dt LIFT] (Np x KT, each derivative block padded
    // to KB columns, zero padded), scaled by 2^p, split into FP16 hi + lo, as
    // tensor-memory rows: [piece][lane = node, 128][KT / 2] words, word p of a
    // row holding columns 2p (low half) and 2p + 1.
    const int KB = dgdev::tt_kb(m->N), KT = dgdev::tt_kt(m->N), AC = dgdev::tt_acols(m->N);
    std::vector<double> Op(static_cast<size_t>(Np) * KT, 0.0);
    double mx = 0.0;
    for (int n = 0; n < Np; ++n)
      for (int k = 0; k < KT; ++k) {
        double v = 0.0;
        if (k < 3 * KB) {
          const int mu = k / KB, j = k % KB;
          const std::vector<double>& Dm = mu == 0 ? m->ops.Dr : mu == 1 ? m->ops.Ds : m->ops.Dt;
          if (j < Np) v = Dm[n * Np + j];
        } else if (k < 3 * KB + NF) {
          v = m->ops.LIFT[n * NF + (k - 3 * KB)];
        }
        Op[n * KT + k] = v;
        mx = std::max(mx, std::fabs(v));
      }
    const double sB = std::ldexp(1.0, static_cast<int>(std::floor(std::log2(16384.0 / mx))));
    o.tc_inv_bscale = static_cast<float>(1.0 / sB);
    const size_t piece = static_cast<size_t>(128) * AC * 2;      // halves
    std::vector<__half> P(2 * piece, __float2half_rn(0.f));
    for (int n = 0; n < Np; ++n)
      for (int k = 0; k < KT; ++k) {
        const float x = static_cast<float>(Op[n * KT + k] * sB);
        const __half hi = __float2half_rn(x);
        const __half lo = __float2half_rn(x - __half2float(hi));
        const size_t off = static_cast<size_t>(n) * AC * 2 + k;   // word k / 2, half k % 2
        P[off] = hi;
        P[piece + off] = lo;
      }
    if ((rc = upload(reinterpret_cast<__half**>(&o.tcB), P, err))) return rc;
  } else if (m->N <= 4) {
    // B = [Dr Ds Dt LIFT] (Np x KT, zero padded), scaled by 2^p, split into FP16
    // hi + lo, stored in the canonical K-major core-matrix layout.
    const int KB = (Np + 1) & ~1, KT = (3 * KB + NF + 15) & ~15, NN = (Np + 15) & ~15;
    std::vector<double> B(static_cast<size_t>(NN) * KT, 0.0);
    double mx = 0.0;
    for (int n = 0; n < Np; ++n)
      for (int k = 0; k < KT; ++k) {
        double v = 0.0;
        if (k < 3 * KB) {
          const int mu = k / KB, j = k % KB;
          const std::vector<double>& Dm = mu == 0 ? m->ops.Dr : mu == 1 ? m->ops.Ds : m->ops.Dt;
          if (j < Np) v = Dm[n * Np + j];
        } else if (k < 3 * KB + NF) {
          v = m->ops.LIFT[n * NF + (k - 3 * KB)];
        }
        B[n * KT + k] = v;
        mx = std::max(mx, std::fabs(v));
      }
    const double sB = std::ldexp(1.0, static_cast<int>(std::floor(std::log2(16384.0 / mx))));
    o.tc_inv_bscale = static_cast<float>(1.0 / sB);
    const size_t piece = static_cast<size_t>(NN) * KT;
    std::vector<__half> P(2 * piece);
    for (int n = 0; n < NN; ++n)
      for (int k = 0; k < KT; ++k) {
        const float x = static_cast<float>(B[n * KT + k] * sB);
        const __half hi = __float2half_rn(x);
        const __half lo = __float2half_rn(x - __half2float(hi));
        const size_t off = ((k / 8) * (NN / 8) + n / 8) * 64 + (n % 8) * 8 + (k % 8);
        P[off] = hi;
        P[piece + off] = lo;
      }
    if ((rc = upload(reinterpret_cast<__half**>(&o.tcB), P, err))) return rc;
  }
  if (m->N >= 8) {
    // the register-tiled FP32 stage's operator, chunk by chunk (device.h)
    const int JC = dgdev::wide_jc(m->N), NCH = dgdev::wide_chunks(m->N), MC = dgdev::wide_mc(m->N);
    const int slot = dgdev::wide_chunk_bytes(m->N) / 4, NLC = NF / 4 / MC;
    std::vector<float> W(static_cast<size_t>(NCH + NLC) * slot, 0.f);
    for (int c = 0; c < NCH; ++c)
      for (int i = 0; i < Np; ++i)
        for (int jj = 0; jj < JC && c * JC + jj < Np; ++jj) {
          const float4 d = D4[i * Np + c * JC + jj];
          float* w = &W[static_cast<size_t>(c) * slot + (i * JC + jj) * 3];
          w[0] = d.x;
          w[1] = d.y;
          w[2] = d.z;
        }
    for (int c = 0; c < NLC; ++c)
      for (int i = 0; i < Np; ++i)
        std::memcpy(&W[static_cast<size_t>(NCH + c) * slot + i * MC * 4], &L4[i * (NF / 4) + c * MC],
                    sizeof(float4) * MC);
    float* dw = nullptr;
    if ((rc = upload(&dw, W, err))) return rc;
    o.wide = dw;
  }
  g_ops[{dev, m->N}] = o;
  out = o;
  return DG_OK;
}

// Creates (or re-creates after an order change) the device copy of the mesh:
// the shared order operators plus one arena holding this mesh's geometry
// records, its tiled tensor-core geometry, the status word and the energy
// partial sums (one allocation, one copy).
int ensure_device(dg_mesh* m, std::string& err) {
  if (m->N == 0) { err = "dg_set_order() has not been called"; return DG_ERR_STATE; }
  int cur = 0;
  DG_CUDA(cudaGetDevice(&cur), "cudaGetDevice");
  if (m->dev && m->dev->N == m->N && m->dev->device == cur) return DG_OK;
  if (m->dev) { dgdev::destroy_device_state(m->dev); m->dev = nullptr; }
  auto* d = new DeviceState();
  m->dev = d;
  d->device = cur;
  d->N = m->N;
  d->K = m->K;
  d->Np = m->ops.Np;
  d->Nfp = m->ops.Nfp;
  DG_CUDA(cudaDeviceGetAttribute(&d->num_sms, cudaDevAttrMultiProcessorCount, cur),
          "cudaDeviceGetAttribute");
  OrderOps ops;
  int rc = order_ops(m, cur, ops, err);
  if (rc) return rc;
  d->D4 = ops.D4;
  d->LIFT4 = ops.LIFT4;
  d->M = ops.M;
  d->T = ops.T;
  d->fmask = ops.fmask;
  d->perm = ops.perm;
  d->tcB = ops.tcB;
  d->wide = ops.wide;
  d->tc_inv_bscale = ops.tc_inv_bscale;
  const int64_t K = m->K;
  const int Nfp = d->Nfp, NF = 4 * Nfp;
  const bool tc = d->N <= dgdev::kTcMaxOrder;
  const int E = dgdev::tc_tile_elems(d->N);
  const int64_t ntiles = (K + E - 1) / E;
  d->tc_geo_stride = tc ? dgdev::tc_geo_floats(d->N) : 0;
  d->egrid = dgdev::energy_grid(d->num_sms);
  // arena layout (bytes, each part 256-byte aligned)
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  const size_t geo_b = static_cast<size_t>(K) * dgdev::kGeoWords * 4;
  const size_t mat_b = m->eps.empty() ? 0 : static_cast<size_t>(K) * dgdev::kMatVecs * 16;
  const size_t tcg_b = tc ? static_cast<size_t>(ntiles) * d->tc_geo_stride * 4 : 0;
  const size_t o_mat = up(geo_b), o_tcg = o_mat + up(mat_b), o_J = o_tcg + up(tcg_b);
  const size_t o_part = o_J + up(static_cast<size_t>(K) * 4);
  // the energy and the status word share 16 bytes: one copy reads both
  const size_t o_res = o_part + up(sizeof(double) * d->egrid), o_stat = o_res + 8;
  const size_t total = o_res + 256;
  std::vector<unsigned char> host(o_part, 0);

  // geometry records
  float* geo = reinterpret_cast<float*>(host.data());
  for (int64_t k = 0; k < K; ++k) {
    float* g = &geo[k * dgdev::kGeoWords];
    for (int a = 0; a < 9; ++a) g[a] = static_cast<float>(m->metric[a * K + k]);
    g[9] = static_cast<float>(m->J[k]);
    reinterpret_cast<float*>(host.data() + o_J)[k] = g[9];
    uint32_t codes = 0;
    for (int f = 0; f < 4; ++f) {
      const int c = m->nbr_code[4 * k + f];
      const bool absorbing = c < 0 && !m->bc.empty() && m->bc[4 * k + f] == DG_BC_ABSORBING;
      d->absorbing = d->absorbing || absorbing;
      codes |= (absorbing ? dgdev::kAbsorbingCode : static_cast<uint32_t>(c + 1)) << (8 * f);
      for (int dd = 0; dd < 3; ++dd)
        g[12 + 4 * f + dd] = static_cast<float>(m->normals[(dd * K + k) * 4 + f]);
      g[15 + 4 * f] = static_cast<float>(m->Fscale[4 * k + f]);
      const int32_t nb = m->nbr_elem[4 * k + f];
      std::memcpy(&g[28 + f], &nb, 4);
    }
    std::memcpy(&g[10], &codes, 4);
  }
  d->scattered = m->N == 3 && dgdev::scattered_mesh(m->nbr_elem.data(), m->nbr_code.data(), K);
  if (mat_b) {
    // material records: 1/eps, 1/mu, eps, mu, then the flux coefficients of each
    // face from the impedances of both sides (the element's own on boundaries)
    float4* mr = reinterpret_cast<float4*>(host.data() + o_mat);
    for (int64_t k = 0; k < K; ++k) {
      const double e = m->eps[k], u = m->mu[k], zm = std::sqrt(u / e);
      mr[k * dgdev::kMatVecs] = make_float4(static_cast<float>(1.0 / e), static_cast<float>(1.0 / u),
                                            static_cast<float>(e), static_cast<float>(u));
      for (int f = 0; f < 4; ++f) {
        const int64_t k2 = m->nbr_code[4 * k + f] < 0 ? k : m->nbr_elem[4 * k + f];
        const double zp = std::sqrt(m->mu[k2] / m->eps[k2]), ym = 1.0 / zm, yp = 1.0 / zp;
        mr[k * dgdev::kMatVecs + 1 + f] =
            make_float4(static_cast<float>(zp), static_cast<float>(1.0 / (zm + zp)),
                        static_cast<float>(yp), static_cast<float>(1.0 / (ym + yp)));
      }
    }
  }
  if (tc) {
    // tiled geometry, one contiguous block per tile: word-major [kTcGeoWords][E]
    // (record words {0..8 metric, 10 codes, 12..27 faces, 28..31 neighbours} ->
    // words {0..8, 9, 10..25, 26..29}), then one byte per face node (e, m):
    // the node of the neighbour across face m / Nfp that matches it (0 on walls)
    float* tg = reinterpret_cast<float*>(host.data() + o_tcg);
    for (int64_t k = 0; k < K; ++k) {
      float* blk = &tg[(k / E) * d->tc_geo_stride];
      for (int w = 0; w < dgdev::kTcGeoWords; ++w) {
        const int src = w < 9 ? w : (w == 9 ? 10 : w + 2);
        blk[w * E + k % E] = geo[k * dgdev::kGeoWords + src];
      }
      unsigned char* nodes = reinterpret_cast<unsigned char*>(blk + dgdev::kTcGeoWords * E);
      for (int f = 0; f < 4; ++f) {
        const int c = m->nbr_code[4 * k + f];
        for (int j = 0; j < Nfp; ++j)
          nodes[(k % E) * NF + f * Nfp + j] =
              c < 0 ? 0 : static_cast<unsigned char>(m->ops.perm[(f * 24 + c) * Nfp + j]);
      }
    }
  }
  DG_CUDA(cudaMalloc(&d->arena, total), "cudaMalloc");
  unsigned char* base = static_cast<unsigned char*>(d->arena);
  DG_CUDA(cudaMemcpy(base, host.data(), host.size(), cudaMemcpyHostToDevice), "cudaMemcpy H2D");
  DG_CUDA(cudaMemset(base + o_res, 0, 256), "cudaMemset");
  d->geo = reinterpret_cast<float4*>(base);
  d->J = reinterpret_cast<float*>(base + o_J);
  d->mat = mat_b ? reinterpret_cast<float4*>(base + o_mat) : nullptr;
  d->tcgeo = tc ? reinterpret_cast<float*>(base + o_tcg) : nullptr;
  d->partials = reinterpret_cast<double*>(base + o_part);
  d->result = reinterpret_cast<double*>(base + o_res);
  d->status = reinterpret_cast<int*>(base + o_stat);
  return DG_OK;
}

// The kernel family of a stage call.
enum class Path { fp32, direct, tc };

// DG_STAGE_TC and orders 2..7 of DG_STAGE_AUTO: the tensor-core stages of
// tc_stage.cuh and tc_stage_t.cuh, which move whole tiles with bulk copies and need
// every field chunk 16-byte aligned ((K * Np) % 4 == 0 and 16-byte aligned buffers).
// Everything else: FP32 CUDA cores, at order 1 (faster there than on the tensor cores,
// Np = 4) one thread per element for 16-byte aligned buffers and the default tile shape,
// else tiles.
static Path stage_path(const dg_mesh* m, std::initializer_list<const void*> bufs) {
  bool aligned = (m->K * m->ops.Np) % 4 == 0;
  for (const void* p : bufs) aligned = aligned && reinterpret_cast<uintptr_t>(p) % 16 == 0;
  const Path cuda_cores = m->N == 1 && aligned && m->stage_shape == 0 ? Path::direct : Path::fp32;
  if (m->stage_impl == DG_STAGE_FP32 || (m->stage_impl == DG_STAGE_AUTO && m->N == 1))
    return cuda_cores;
  return m->N <= dgdev::kTcMaxOrder && aligned ? Path::tc : Path::fp32;
}

static bool on_cuda_cores(Path p) { return p == Path::fp32 || p == Path::direct; }

static int stage_tile(const dg_mesh* m, Path p) {
  return on_cuda_cores(p) ? dgdev::stage_tile_elems(m->N, m->stage_shape)
                         : dgdev::tc_tile_elems(m->N);
}

static dgdev::StageArgs stage_args(dg_mesh* m, Path p) {
  DeviceState* d = m->dev;
  dgdev::StageArgs a{};
  a.tcB = d->tcB;
  a.wide = d->wide;
  a.tcgeo = d->tcgeo;
  a.tc_geo_stride = d->tc_geo_stride;
  a.tc_inv_bscale = d->tc_inv_bscale;
  a.status = d->status;
  a.geo = d->geo;
  a.mat = d->mat;
  a.absorbing = d->absorbing ? 1 : 0;
  a.scattered = d->scattered ? 1 : 0;
  a.D4 = d->D4;
  a.LIFT4 = d->LIFT4;
  a.fmask = d->fmask;
  a.perm = d->perm;
  a.K = static_cast<int>(d->K);
  a.alpha = static_cast<float>(m->alpha);
  const int E = stage_tile(m, p);
  a.num_tiles = static_cast<int>((d->K + E - 1) / E);
  return a;
}

static cudaError_t launch_path(const dg_mesh* m, Path p, bool rk, const dgdev::StageArgs& a,
                               cudaStream_t s) {
  const int sms = m->dev->num_sms;
  switch (p) {
    case Path::direct: {
      dgdev::StageArgs e = a;                        // tiles -> elements
      const int E = stage_tile(m, p);
      e.tile0 = a.tile0 * E;
      e.num_tiles = std::min(a.num_tiles * E, a.K - e.tile0);
      dgdev::DirectOps<1> o;
      for (int i = 0; i < o.Np; ++i) {
        for (int j = 0; j < o.Np; ++j) {
          o.D[0][i][j] = static_cast<float>(m->ops.Dr[i * o.Np + j]);
          o.D[1][i][j] = static_cast<float>(m->ops.Ds[i * o.Np + j]);
          o.D[2][i][j] = static_cast<float>(m->ops.Dt[i * o.Np + j]);
        }
        for (int f = 0; f < 4 * o.Nfp; ++f)
          o.L[i][f] = static_cast<float>(m->ops.LIFT[i * 4 * o.Nfp + f]);
      }
      return dgdev::launch_direct_stage(rk, e, o, sms, s);
    }
    case Path::tc: return dgdev::launch_tc_stage(m->N, rk, a, sms, s);
    default: return dgdev::launch_stage(m->N, rk, a, sms, s, m->stage_shape);
  }
}

int device_rhs(dg_mesh* m, const float* u, float* rhs, void* stream, std::string& err) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = ensure_device(m, err);
  if (rc) return rc;
  const Path p = stage_path(m, {u, rhs});
  dgdev::StageArgs a = stage_args(m, p);
  a.u_in = u;
  a.rhs = rhs;
  DG_CUDA(traced(m, s, on_cuda_cores(p) ? 1 : 5, [&] { return launch_path(m, p, false, a, s); }),
          "stage kernel launch");
  m->last_launches = 1;
  return DG_OK;
}

// LSERK4 coefficients (Carpenter & Kennedy 1994, five stages, two registers).
static const double kRkA[5] = {0.0, -567301805773.0 / 1357537059087.0,
                               -2404267990393.0 / 2016746695238.0,
                               -3550918686646.0 / 2091501179385.0,
                               -1275806237668.0 / 842570457699.0};
static const double kRkB[5] = {1432997174477.0 / 9575080441755.0,
                               5161836677717.0 / 13612068292357.0,
                               1720146321549.0 / 2090206949498.0,
                               3134564353537.0 / 4481467310338.0,
                               2277821191437.0 / 14882151754819.0};

// The stages of nsteps steps, u and the work buffer taking turns; *at receives the buffer
// that holds the state.  parts > 1: the last stage as that many ranges of whole tiles,
// part i ending before element cut[i], ready[i] recorded after it.
static int run_stages(dg_mesh* m, float* u, float* res, double dt, int nsteps, cudaStream_t s,
                      std::string& err, float** at, int parts = 1, const int64_t* cut = nullptr,
                      cudaEvent_t* ready = nullptr) {
  DeviceState* d = m->dev;
  const size_t n = static_cast<size_t>(6) * d->K * d->Np;
  if (!d->u_work) DG_CUDA(cudaMalloc(&d->u_work, n * sizeof(float)), "cudaMalloc work state");
  const Path p = stage_path(m, {u, res, d->u_work});
  dgdev::StageArgs a = stage_args(m, p);
  const int E = stage_tile(m, p), all = a.num_tiles;
  a.res = res;
  a.dt = static_cast<float>(dt);
  float* src = u;
  float* dst = d->u_work;
  int64_t launches = 0;
  for (int st = 0; st < nsteps; ++st)
    for (int i = 0; i < 5; ++i) {
      a.u_in = src;
      a.u_out = dst;
      a.a = static_cast<float>(kRkA[i]);
      a.b = static_cast<float>(kRkB[i]);
      const int np = st == nsteps - 1 && i == 4 ? parts : 1;
      for (int q = 0; q < np; ++q) {
        if (np > 1) {
          a.tile0 = q ? static_cast<int>(cut[q - 1] / E) : 0;
          a.num_tiles = (q == np - 1 ? all : static_cast<int>(cut[q] / E)) - a.tile0;
        }
        DG_CUDA(traced(m, s, on_cuda_cores(p) ? 0 : 4,
                       [&] { return launch_path(m, p, true, a, s); }), "stage kernel launch");
        ++launches;
        if (np > 1) DG_CUDA(cudaEventRecord(ready[q], s), "cudaEventRecord");
      }
      std::swap(src, dst);
    }
  *at = src;
  m->last_launches = launches;
  return DG_OK;
}

static int step_impl(dg_mesh* m, float* u, float* res, double dt, int nsteps, cudaStream_t s,
                     std::string& err) {
  float* at = nullptr;
  if (int rc = run_stages(m, u, res, dt, nsteps, s, err, &at)) return rc;
  if (at != u)  // odd number of stages: the state sits in the work buffer
    DG_CUDA(cudaMemcpyAsync(u, at, static_cast<size_t>(6) * m->dev->K * m->dev->Np * sizeof(float),
                            cudaMemcpyDeviceToDevice, s), "cudaMemcpyAsync D2D");
  return DG_OK;
}

int device_stage_tile(dg_mesh* m, const float* u_in, const float* u_out, const float* res,
                      int* tile, std::string& err) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  *tile = stage_tile(m, stage_path(m, {u_in, u_out, res}));
  return DG_OK;
}

int device_stage(dg_mesh* m, const float* u_in, float* u_out, float* res, int stage, double dt,
                 const float* dt_elem, void* stream, std::string& err, int64_t k0, int64_t k1) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Path p = stage_path(m, {u_in, u_out, res});
  dgdev::StageArgs a = stage_args(m, p);
  if (k1 >= 0) {                        // elements [k0, k1): whole tiles of the kernel that runs
    const int E = stage_tile(m, p);
    if (k0 < 0 || k1 <= k0 || k1 > m->K || k0 % E != 0 || (k1 % E != 0 && k1 != m->K)) {
      err = "the element range must be [k0, k1) with k0 and k1 multiples of the stage's tile of " +
            std::to_string(E) + " tetrahedra (or k1 = K), 0 <= k0 < k1 <= K";
      return DG_ERR_ARG;
    }
    a.tile0 = static_cast<int>(k0 / E);
    a.num_tiles = static_cast<int>((k1 + E - 1) / E - k0 / E);
  }
  a.u_in = u_in;
  a.u_out = u_out;
  a.res = res;
  a.dt = static_cast<float>(dt);
  a.dt_elem = dt_elem;
  a.a = static_cast<float>(kRkA[stage]);
  a.b = static_cast<float>(kRkB[stage]);
  DG_CUDA(traced(m, s, on_cuda_cores(p) ? 0 : 4, [&] { return launch_path(m, p, true, a, s); }),
          "stage kernel launch");
  m->last_launches = 1;
  return DG_OK;
}

// Default cost of one tile on one SM in microseconds, orders 1..6 on the
// tensor cores in the one-CTA form that a mixed launch runs (GB300: stage time x
// SMs / tiles at ~1.7e7 unknowns), used to split a mixed launch's CTAs when the
// caller gives no costs.
static double default_tile_cost(int N) {
  static const double c[7] = {1.0, 1.6, 1.9, 2.7, 3.6, 3.1, 3.9};
  return N >= 1 && N <= 6 ? c[N] : 1.0;
}

// CTAs of a mixed launch: one per group at least, `total` in all, each further
// CTA to the group whose span ceil(tiles / ctas) x cost is then the longest
// (so the groups of one launch finish together).
static std::vector<int> split_ctas(const std::vector<int64_t>& tiles,
                                   const std::vector<double>& cost, int total) {
  const size_t n = tiles.size();
  std::vector<int> c(n, 1);
  int used = static_cast<int>(n);
  auto span = [&](size_t g) {
    return static_cast<double>((tiles[g] + c[g] - 1) / c[g]) * cost[g];
  };
  while (used < total) {
    size_t best = n;
    for (size_t g = 0; g < n; ++g)
      if (c[g] < tiles[g] && (best == n || span(g) > span(best))) best = g;
    if (best == n) break;
    ++c[best];
    ++used;
  }
  return c;
}

int device_stage_multi(dg_mesh* const* ms, int n, const float* const* u_in, float* const* u_out,
                       float* const* res, const float* const* dt_elem, int stage, double dt,
                       const double* tile_cost, void* stream, std::string& err) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int64_t launches = 0;
  std::vector<int> fam(n, 0);        // 0: its own launch (order 7, FP32), 1: orders 1..4, 2: orders 5, 6
  for (int i = 0; i < n; ++i) {
    if (int rc = ensure_device(ms[i], err)) return rc;
    if (ms[i]->dev->device != ms[0]->dev->device) {
      err = "every mesh of one call must be on the same device";
      return DG_ERR_ARG;
    }
    if (stage_path(ms[i], {u_in[i], u_out[i], res[i]}) == Path::tc) fam[i] = ms[i]->N <= 4 ? 1 : ms[i]->N <= 6 ? 2 : 0;
  }
  for (int i = 0; i < n; ++i)
    if (fam[i] == 0) {
      if (int rc = device_stage(ms[i], u_in[i], u_out[i], res[i], stage, dt,
                                dt_elem ? dt_elem[i] : nullptr, stream, err))
        return rc;
      ++launches;
    }
  const int sms = ms[0]->dev->num_sms;
  for (int f = 1; f <= 2; ++f) {
    std::vector<int> idx;
    for (int i = 0; i < n; ++i)
      if (fam[i] == f) idx.push_back(i);
    for (size_t c0 = 0; c0 < idx.size(); c0 += dgdev::kMaxMixedGroups) {
      const size_t ng = std::min(idx.size() - c0, static_cast<size_t>(dgdev::kMaxMixedGroups));
      std::vector<int64_t> tiles(ng);
      std::vector<double> cost(ng);
      dgdev::MixedArgs M{};
      M.ngroups = static_cast<int>(ng);
      int64_t all = 0;
      for (size_t g = 0; g < ng; ++g) {
        const int i = idx[c0 + g];
        dgdev::StageArgs a = stage_args(ms[i], Path::tc);
        a.u_in = u_in[i];
        a.u_out = u_out[i];
        a.res = res[i];
        a.dt = static_cast<float>(dt);
        a.dt_elem = dt_elem ? dt_elem[i] : nullptr;
        a.a = static_cast<float>(kRkA[stage]);
        a.b = static_cast<float>(kRkB[stage]);
        M.g[g].a = a;
        M.g[g].N = ms[i]->N;
        M.g[g].ext = (a.mat || a.absorbing) ? 1 : 0;
        tiles[g] = a.num_tiles;
        cost[g] = tile_cost && tile_cost[i] > 0.0 ? tile_cost[i] : default_tile_cost(ms[i]->N);
        all += a.num_tiles;
      }
      const int total = static_cast<int>(std::min<int64_t>(sms, all));
      const std::vector<int> c = split_ctas(tiles, cost, total);
      int grid = 0;
      for (size_t g = 0; g < ng; ++g) {
        M.g[g].first = grid;
        M.g[g].count = c[g];
        grid += c[g];
      }
      DG_CUDA(traced(ms[0], s, 6, [&] {
                return f == 1 ? dgdev::launch_tc_mixed(M, grid, s)
                              : dgdev::launch_tt_mixed(M, grid, s);
              }), "mixed stage kernel launch");
      ++launches;
    }
  }
  for (int i = 0; i < n; ++i) ms[i]->last_launches = 0;
  ms[0]->last_launches = launches;
  return DG_OK;
}

int device_step(dg_mesh* m, float* u, float* res, double dt, int nsteps, void* stream,
                std::string& err) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  return step_impl(m, u, res, dt, nsteps, static_cast<cudaStream_t>(stream), err);
}

// Clears a set status word and reports it.
static int report_status(dg_mesh* m, int st, std::string& err) {
  if (st != 0) {
    DG_CUDA(cudaMemset(m->dev->status, 0, sizeof(int)), "cudaMemset");
    err = "stage kernel: a wait for a copy or for tensor-core results timed out (results invalid)";
    return DG_ERR_CUDA;
  }
  return DG_OK;
}

// Reads (and clears) the pipeline status word; only after a synchronisation.
static int check_status(dg_mesh* m, std::string& err) {
  int st = 0;
  DG_CUDA(cudaMemcpy(&st, m->dev->status, sizeof(int), cudaMemcpyDeviceToHost), "cudaMemcpy D2H");
  return report_status(m, st, err);
}

int device_wait_selftest(dg_mesh* m, uint32_t polls, double* seconds, std::string& err) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  DeviceState* d = m->dev;
  auto* ns = reinterpret_cast<unsigned long long*>(d->result);   // 8-byte scratch word
  DG_CUDA(dgdev::launch_wait_selftest(d->status, polls, ns, nullptr), "self-test launch");
  unsigned long long h = 0;
  DG_CUDA(cudaMemcpy(&h, ns, sizeof(h), cudaMemcpyDeviceToHost), "cudaMemcpy D2H");
  if (seconds) *seconds = static_cast<double>(h) * 1e-9;
  return check_status(m, err);
}

static int energy_impl(dg_mesh* m, const float* u, double* out, cudaStream_t s,
                       std::string& err, int64_t k0 = 0, int64_t k1 = -1) {
  DeviceState* d = m->dev;
  dgdev::EnergyArgs a{u, d->T, d->J, static_cast<int>(d->K), d->partials, d->result,
                      static_cast<int>(k0), static_cast<int>(k1 < 0 ? d->K : k1), d->mat};
  int grid = 0;
  DG_CUDA(traced(m, s, 2, [&] {
            return dgdev::launch_energy_partials(m->N, a, d->num_sms, &grid, s);
          }), "energy kernel launch");
  DG_CUDA(traced(m, s, 3, [&] { return dgdev::launch_energy_final(a, grid, s); }),
          "energy kernel launch");
  // the energy and, beside it, the status word of the stages before it
  struct { double energy; int status, unused; } r = {0.0, 0, 0};
  static_assert(sizeof(r) == 16, "layout");
  DG_CUDA(cudaMemcpyAsync(&r, d->result, sizeof(r), cudaMemcpyDeviceToHost, s),
          "cudaMemcpyAsync D2H");
  DG_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  if (int rc = report_status(m, r.status, err)) return rc;
  const double h = r.energy;
  *out = h;
  m->last_launches = 2;
  if (!std::isfinite(h)) { err = "energy is not finite (unstable run)"; return DG_ERR_UNSTABLE; }
  return DG_OK;
}

int device_resident(const dg_mesh* m, const float** M, const void** geo, const void** mat,
                    int64_t* K, int* Np, std::string& err) {
  int cur = -1;
  DG_CUDA(cudaGetDevice(&cur), "cudaGetDevice");
  const DeviceState* d = m->dev;
  if (!d || d->N != m->N || d->device != cur) {
    err = "mesh data is not on the current device yet (make one dg_rhs, dg_step or "
          "dg_energy call on this device first)";
    return DG_ERR_STATE;
  }
  *M = d->M;
  *geo = d->geo;
  *mat = d->mat;
  *K = d->K;
  *Np = d->Np;
  return DG_OK;
}

int device_energy_range(dg_mesh* m, const float* u, int64_t k0, int64_t k1, double* out,
                        void* stream, std::string& err) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  return energy_impl(m, u, out, static_cast<cudaStream_t>(stream), err, k0, k1);
}

int device_energy(dg_mesh* m, const float* u, double* out, void* stream, std::string& err) {
  int rc = ensure_device(m, err);
  if (rc) return rc;
  return energy_impl(m, u, out, static_cast<cudaStream_t>(stream), err);
}

// Host buffers cross the bus at ~200 GB/s (146 334 order-3 tetrahedra: 0.34 ms in, 0.37
// ms out, against 0.12 ms a stage), so whatever needs not wait for a copy runs beside it:
// the RK register is cleared while the fields come in, the last stage runs as up to four
// ranges of tiles whose fields leave while the next range is computed, straight from the
// buffer the last stage wrote, and the energy is formed while they leave.
int device_step_host(dg_mesh* m, float* u, float* res, double dt, int nsteps, double* energy,
                     void* stream, std::string& err) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int rc = ensure_device(m, err);
  if (rc) return rc;
  DeviceState* d = m->dev;
  const size_t pitch = static_cast<size_t>(d->K) * d->Np * sizeof(float), bytes = 6 * pitch;
  if (!d->h_u) DG_CUDA(cudaMalloc(&d->h_u, bytes), "cudaMalloc");
  if (!d->h_res) DG_CUDA(cudaMalloc(&d->h_res, bytes), "cudaMalloc");
  if (!d->copies)
    DG_CUDA(cudaStreamCreateWithFlags(&d->copies, cudaStreamNonBlocking), "cudaStreamCreate");
  for (cudaEvent_t& e : d->ready)
    if (!e) DG_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "cudaEventCreate");
  cudaEvent_t* const ready = d->ready;
  cudaEvent_t other = d->ready[4];
  // the copy stream's work of this call ends before the call does, whatever its outcome
  struct Drain {
    cudaStream_t a, b;
    ~Drain() {
      cudaStreamSynchronize(a);
      cudaStreamSynchronize(b);
    }
  } drain{d->copies, s};
  // without a host RK register the device one starts from zero (the first
  // LSERK4 stage has a = 0, so a step's result does not depend on it)
  if (!res) {
    DG_CUDA(cudaMemsetAsync(d->h_res, 0, bytes, d->copies), "cudaMemsetAsync");
    DG_CUDA(cudaEventRecord(other, d->copies), "cudaEventRecord");
  }
  DG_CUDA(cudaMemcpyAsync(d->h_u, u, bytes, cudaMemcpyHostToDevice, s), "cudaMemcpyAsync H2D");
  if (res) DG_CUDA(cudaMemcpyAsync(d->h_res, res, bytes, cudaMemcpyHostToDevice, s), "cudaMemcpyAsync H2D");
  else DG_CUDA(cudaStreamWaitEvent(s, other, 0), "cudaStreamWaitEvent");
  // energy-growth check (opt-in): the energy of the incoming state first
  const bool check = m->energy_check >= 0.0;
  double e_in = 0.0;
  int64_t launches = 0;
  if (check) {
    if ((rc = energy_impl(m, d->h_u, &e_in, s, err))) return rc;
    launches += 2;
  }
  // ranges of the last stage: whole waves of tiles, none below 8 MB of fields
  int parts = 1;
  int64_t cut[4] = {d->K, d->K, d->K, d->K};
  if (nsteps > 0) {
    if (!d->u_work) DG_CUDA(cudaMalloc(&d->u_work, bytes), "cudaMalloc work state");
    const int E = stage_tile(m, stage_path(m, {d->h_u, d->h_res, d->u_work}));
    const int64_t wave = int64_t(2) * d->num_sms * E, waves = d->K / wave;
    const int64_t most = std::min<int64_t>(std::min<int64_t>(4, waves), bytes / (8 << 20));
    if (most > 1 && pitch <= 0x7fffffff) {           // (a 2D copy's largest pitch)
      parts = static_cast<int>(most);
      for (int q = 0; q + 1 < parts; ++q) cut[q] = waves * (q + 1) / parts * wave;
    }
  }
  float* at = d->h_u;
  if (nsteps > 0) {
    if ((rc = run_stages(m, d->h_u, d->h_res, dt, nsteps, s, err, &at, parts, cut, ready)))
      return rc;
    launches += m->last_launches;
  }
  if (parts == 1) DG_CUDA(cudaEventRecord(ready[0], s), "cudaEventRecord");
  for (int q = 0; q < parts; ++q) {
    DG_CUDA(cudaStreamWaitEvent(d->copies, ready[q], 0), "cudaStreamWaitEvent");
    const int64_t k0 = q ? cut[q - 1] : 0, k1 = q == parts - 1 ? d->K : cut[q];
    const size_t first = static_cast<size_t>(k0) * d->Np;
    if (parts == 1)
      DG_CUDA(cudaMemcpyAsync(u, at, bytes, cudaMemcpyDeviceToHost, d->copies),
              "cudaMemcpyAsync D2H");
    else
      DG_CUDA(cudaMemcpy2DAsync(u + first, pitch, at + first, pitch,
                                static_cast<size_t>(k1 - k0) * d->Np * sizeof(float), 6,
                                cudaMemcpyDeviceToHost, d->copies), "cudaMemcpy2DAsync D2H");
  }
  if (res) DG_CUDA(cudaMemcpyAsync(res, d->h_res, bytes, cudaMemcpyDeviceToHost, d->copies), "cudaMemcpyAsync D2H");
  m->last_launches = launches;
  if (energy || check) {
    double e_out = 0.0;
    rc = energy_impl(m, at, &e_out, s, err);
    launches += 2;
    m->last_launches = launches;
    if (energy) *energy = e_out;
    if (rc) return rc;                       // includes a non-finite energy (DG_ERR_UNSTABLE)
    DG_CUDA(cudaStreamSynchronize(d->copies), "cudaStreamSynchronize");
    if (check && e_out > e_in * (1.0 + m->energy_check)) {
      char buf[160];
      std::snprintf(buf, sizeof buf, "energy grew from %.9g to %.9g over %d steps "
                    "(allowed factor 1 + %g): unstable run", e_in, e_out, nsteps, m->energy_check);
      err = buf;
      return DG_ERR_UNSTABLE;
    }
  } else {
    DG_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
    DG_CUDA(cudaStreamSynchronize(d->copies), "cudaStreamSynchronize");
    if ((rc = check_status(m, err))) return rc;
  }
  return DG_OK;
}

}  // namespace dg
