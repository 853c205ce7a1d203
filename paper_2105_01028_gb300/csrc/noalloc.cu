// Source iteration on caller-owned device buffers, with no device allocation at all.
//
// Some callers cannot call cudaMalloc at the point where they need a solve: code that
// runs inside a region where the device allocator must not be touched (for example a
// framework's own memory pool that owns every byte of the device, or a real-time loop
// that forbids allocation), or callers that hand out their own preallocated buffers and
// expect a library call to add nothing to the device footprint.  This file gives them
// one entry point that uses no allocator: the kernel's scratch memory (per-voxel
// contraction bounds, a max-reduction cell and iteration counters) lives in a
// file-scope static device array of fixed size, which every GPU that loads the library
// holds until the process exits.  Inputs and outputs are still the caller's.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <mutex>

#include "device.cuh"
#include "trinity.h"

namespace trinity {
namespace {

constexpr int kNoAllocMaxVoxels = 1 << 20;  // 1,048,576 voxels: 4 MiB of bounds
constexpr int kNaTile = 32;                   // voxels per CTA (as in the FP32 kernel)

struct NoAllocScratch {
  unsigned smax;       // max |S_prev| as float bits (the stop rule's floor scale)
  int iters_max;       // largest iteration count of the call
  int nonconv;         // voxels that reached max_iters
  int error;           // device error word (a bounded wait ran out)
  float rho[kNoAllocMaxVoxels];  // per-voxel contraction bound (1 - eps) max_d b1
  // the caller's P, split for the tensor cores (48 and 192 directions; see scatter_split.cu)
  alignas(128) uint16_t ph[3 * 192 * 64];
  alignas(128) uint16_t pl[2 * 3 * 192 * 64];  // Pm, then Pl
  float diag[3 * 192];
  float cw[64];
  float dyn[4];        // unit, Chebyshev interval
};

static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

NoAllocScratch* g_scratch_ptr[kMaxDevices] = {};
std::mutex g_scratch_mu;

// Device address of the scratch array for the current device (looked up once per
// device; in host code the symbol's name is only a host-side stand-in).
int scratch_for_current_device(NoAllocScratch** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return TRINITY_E_CUDA;
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return TRINITY_E_CUDA;
    g_scratch_ptr[dev] = static_cast<NoAllocScratch*>(p);
  }
  *out = g_scratch_ptr[dev];
  return TRINITY_OK;
}

// Max |S_prev| over everything and (b1 given: 12 directions) per voxel rho = (1 - eps) max_d b1.
__global__ void noalloc_prepass(int na, int nvox, const float* __restrict__ b1, const float* __restrict__ eps,
                                const float* __restrict__ S_prev, NoAllocScratch* sc) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  float sm = 0.0f;
  if (v < nvox) {
    float bmax = 0.0f;
#pragma unroll 8
    for (int d = 0; d < na; ++d) {
      if (b1) bmax = fmaxf(bmax, b1[static_cast<size_t>(d) * nvox + v]);
      sm = fmaxf(sm, fabsf(S_prev[static_cast<size_t>(d) * nvox + v]));
    }
    if (b1) sc->rho[v] = (1.0f - eps[v]) * bmax;
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) sm = fmaxf(sm, __shfl_xor_sync(0xffffffffu, sm, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&sc->smax, __float_as_uint(sm));
}

// Split of the caller's P on the device (the host form is scatter_split_image): blocks
// 1 .. NA / 8 build eight rows each (every block takes the largest entry and row weight for
// itself: 147 KB from L2), block 0 estimates the spectrum of P without the constant vector
// by power iteration, its matrix in registers (the context path knows the spectrum from g).
// The estimate sets the interval of the Chebyshev weights only; an eigenvalue above it is
// still damped, as in the plain iteration.  One block doing all of it in turn took 520 us,
// a third of a 110592-voxel call.
template <int NA>
__global__ void __launch_bounds__(1024) noalloc_split_prep(const float* __restrict__ P, NoAllocScratch* sc) {
  constexpr int kW = 32;                    // warps
  constexpr int kC = (NA + 31) / 32;        // columns per lane
  constexpr int kR = (NA + kW - 1) / kW;    // rows per warp
  constexpr int kKb = (NA + 63) / 64;       // K blocks of the operand images
  __shared__ float x_s[kC * 32], y_s[kC * 32];
  __shared__ float red_s[kW], red2_s[kW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // every block: the whole matrix, row i = warp + 32 r, column j = lane + 32 c, with the
  // indices exchanged (P is symmetric; a column of the caller's array is a row here)
  float p[kR][kC];
#pragma unroll
  for (int r = 0; r < kR; ++r)
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      const int i = warp + kW * r, j = lane + 32 * c;
      p[r][c] = (i < NA && j < NA) ? __ldg(P + static_cast<size_t>(i) * NA + j) : 0.0f;
    }
  if (blockIdx.x > 0) {
    float pm = 0.0f, rm = 0.0f;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      float s = 0.0f;
#pragma unroll
      for (int c = 0; c < kC; ++c)
        if (lane + 32 * c != warp + kW * r) {
          pm = fmaxf(pm, fabsf(p[r][c]));
          s += fabsf(p[r][c]);
        }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      rm = fmaxf(rm, s);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
    if (lane == 0) {
      red_s[warp] = pm;
      red2_s[warp] = rm;
    }
    __syncthreads();
    pm = red_s[lane];
    rm = red2_s[lane];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
      rm = fmaxf(rm, __shfl_xor_sync(0xffffffffu, rm, o));
    }
    int t = 0;
    while (t < 20 && ldexpf(pm, t + 1) <= 2046.0f && ldexpf(rm, t + 1) + NA / 2 <= 16128.0f) ++t;
    const float whole = floorf(ldexpf(pm, t));
    const float unit = (whole >= 1.0f ? pm / whole : ldexpf(1.0f, -t)) * 0.0625f;
    const double inv = 1.0 / static_cast<double>(unit);
    if (warp < 8) {
      const int i = (blockIdx.x - 1) * 8 + warp;
      double sh = 0.0, sum = 0.0;
#pragma unroll
      for (int c = 0; c < kC; ++c) {
        const int j = lane + 32 * c;
        if (j >= NA) break;
        const double u = j != i ? __ldg(P + static_cast<size_t>(j) * NA + i) : 0.0f;
        const double uu = u * inv, h = 16.0 * rint(uu * 0.0625);
        const __half l = __double2half(uu - h);
        const __half m = __double2half(uu - h - static_cast<double>(__half2float(l)));
        sh += h;
        sum += u;
        const int k = j >> 6, ch = (j & 63) >> 3;
        const int in_row = ((ch ^ (i & 7)) << 3) + (j & 7);
        const int prow = NA >= 192 ? (k * (NA / 96) + i / 96) * 96 + i % 96 : k * NA + i;
        sc->ph[(k * NA + i) * 64 + in_row] = __half_as_ushort(__double2half(h));
        sc->pl[prow * 64 + in_row] = __half_as_ushort(m);
        sc->pl[(kKb * NA + prow) * 64 + in_row] = __half_as_ushort(l);
      }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        sh += __shfl_xor_sync(0xffffffffu, sh, o);
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
      }
      if (lane == 0) {
        const double d = 1.0 - sum;
        sc->diag[i] = static_cast<float>(d);
        sc->diag[NA + i] = static_cast<float>(d - static_cast<double>(static_cast<float>(d)));
        sc->diag[2 * NA + i] = static_cast<float>(1.0 - sh * unit);
      }
    }
    if (blockIdx.x == 1 && tid == 0) sc->dyn[0] = unit;
    return;
  }
  // block 0: the largest |eigenvalue| besides the constant vector's, then the largest of
  // (that - eigenvalue), which tells how far the spectrum reaches below zero
  float lam = 0.0f, low = 0.0f;
#pragma unroll 1
  for (int stage = 0; stage < 2; ++stage) {
    if (tid < kC * 32) {
      unsigned h = (tid + 1) * 2654435761u;
      h ^= h >> 15;
      x_s[tid] = tid < NA ? static_cast<float>(h & 0xffffu) / 65536.0f - 0.5f : 0.0f;
    }
    __syncthreads();
    float norm = 0.0f;
#pragma unroll 1
    for (int it = 0; it < (stage == 0 ? 40 : 24); ++it) {
      float xv[kC];
#pragma unroll
      for (int c = 0; c < kC; ++c) xv[c] = x_s[lane + 32 * c];
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        float s = 0.0f;
#pragma unroll
        for (int c = 0; c < kC; ++c) s = fmaf(p[r][c], xv[c], s);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const int i = warp + kW * r;
        if (lane == 0 && i < NA) y_s[i] = stage == 0 ? s : fmaf(lam, x_s[i], -s);
      }
      __syncthreads();
      if (warp == 0) {  // without the mean, to unit length
        float yv[kC], m = 0.0f, q = 0.0f;
#pragma unroll
        for (int c = 0; c < kC; ++c) {
          yv[c] = lane + 32 * c < NA ? y_s[lane + 32 * c] : 0.0f;
          m += yv[c];
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
        m /= NA;
#pragma unroll
        for (int c = 0; c < kC; ++c) {
          yv[c] = lane + 32 * c < NA ? yv[c] - m : 0.0f;
          q = fmaf(yv[c], yv[c], q);
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        norm = sqrtf(q);
        const float iv = norm > 1e-30f ? 1.0f / norm : 0.0f;
#pragma unroll
        for (int c = 0; c < kC; ++c) x_s[lane + 32 * c] = yv[c] * iv;
        if (lane == 0) red_s[0] = norm;
      }
      __syncthreads();
    }
    norm = red_s[0];
    if (stage == 0)
      lam = norm;
    else
      low = lam - norm;
    __syncthreads();
  }
  if (tid == 0) {
    sc->dyn[1] = fminf(fmaxf(lam, 0.0f) * 1.01f + 0.01f, 0.5f * (fminf(lam, 0.999f) + 1.0f));
    sc->dyn[2] = low < -0.02f ? -1.0f : 0.0f;
    const int root[8] = {15, 1, 9, 7, 13, 3, 11, 5};  // as scatter_split_image orders them
    for (int k = 0; k < 64; ++k) sc->cw[k] = k < 8 ? cospif(root[k] / 16.0f) : 0.0f;
  }
}

__device__ __forceinline__ float noalloc_transpose_max(float (&vals)[32], int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const bool upper = (lane & s) != 0;
#pragma unroll
    for (int k = 0; k < s; ++k) {
      const float send = upper ? vals[k] : vals[k + s];
      const float keep = upper ? vals[k + s] : vals[k];
      const float recv = __shfl_xor_sync(0xffffffffu, send, s);
      vals[k] = fmaxf(keep, recv);
    }
  }
  return vals[0];
}

// The FP32 source iteration (same arithmetic and stop rule as the context path), with b1
// given per (direction, voxel) instead of derived from the optics, and its scratch in the
// static array.
template <int NA>
__global__ void __launch_bounds__(((NA + 31) / 32) * 32)
    noalloc_iteration(int nvox, const float* __restrict__ P, const float* __restrict__ Q,
                      const float* __restrict__ b1g, const float* __restrict__ eps,
                      const float* __restrict__ S_prev, float* __restrict__ S_out, float* __restrict__ I_out,
                      float tol, int max_iters, NoAllocScratch* sc) {
  constexpr int W = ((NA + 31) / 32);
  constexpr int kBlk = 4;
  __shared__ __align__(16) float Xs[2][NA][kNaTile + 4];
  __shared__ float red_d[W][kNaTile], red_s[W][kNaTile];
  __shared__ float e_s[kNaTile], rho_s[kNaTile], best_s[kNaTile];
  __shared__ int iters_s[kNaTile], stall_s[kNaTile];
  __shared__ unsigned act_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i = tid;
  const bool live = i < NA;
  const int v0 = blockIdx.x * kNaTile;
  const size_t plane = static_cast<size_t>(nvox);
  const float s_glob = __uint_as_float(sc->smax);
  if (tid < kNaTile) {
    const int v = v0 + tid;
    e_s[tid] = v < nvox ? eps[v] : 1.0f;
    rho_s[tid] = v < nvox ? sc->rho[v] : 0.0f;
    best_s[tid] = 3.0e38f;
    stall_s[tid] = 0;
    iters_s[tid] = 0;
  }
  if (tid == 0) act_s = (nvox - v0 >= kNaTile) ? 0xffffffffu : ((1u << (nvox - v0)) - 1u);
  // row-sum correction of this P (FP64 sum): P + diag(r) has unit row sums
  float ri = 0.0f;
  if (live) {
    double rs = 0.0;
    for (int j = 0; j < NA; ++j) rs += static_cast<double>(P[static_cast<size_t>(i) * NA + j]);
    ri = static_cast<float>(1.0 - rs);
  }
  __syncthreads();
  float q[kNaTile], b1[kNaTile], so[kNaTile], acc[kNaTile];
#pragma unroll
  for (int v = 0; v < kNaTile; ++v) {
    const int vv = v0 + v;
    const bool ok = live && vv < nvox;
    q[v] = ok ? Q[static_cast<size_t>(i) * plane + vv] : 0.0f;
    b1[v] = ok ? b1g[static_cast<size_t>(i) * plane + vv] : 0.0f;
    so[v] = ok ? S_prev[static_cast<size_t>(i) * plane + vv] : 0.0f;
  }
  if (live) {
#pragma unroll
    for (int v = 0; v < kNaTile; v += 4)
      *reinterpret_cast<float4*>(&Xs[0][i][v]) =
          make_float4(q[v] + b1[v] * so[v], q[v + 1] + b1[v + 1] * so[v + 1], q[v + 2] + b1[v + 2] * so[v + 2],
                      q[v + 3] + b1[v + 3] * so[v + 3]);
  }
  unsigned act = act_s;
  int cur = 0, k = 0;
  while (act != 0u && k < max_iters) {
    ++k;
    __syncthreads();
#pragma unroll
    for (int v = 0; v < kNaTile; ++v) acc[v] = 0.0f;
    if (live) {
#pragma unroll 1
      for (int j0 = 0; j0 < NA; j0 += kBlk) {
        float t[kNaTile];
#pragma unroll
        for (int v = 0; v < kNaTile; ++v) t[v] = 0.0f;
#pragma unroll
        for (int j = j0; j < j0 + kBlk; ++j) {
          const float p = __ldg(P + static_cast<size_t>(j) * NA + i);  // P symmetric
          const float4* xr = reinterpret_cast<const float4*>(&Xs[cur][j][0]);
#pragma unroll
          for (int v4 = 0; v4 < kNaTile / 4; ++v4) {
            const float4 x4 = xr[v4];
            t[4 * v4 + 0] = fmaf(p, x4.x, t[4 * v4 + 0]);
            t[4 * v4 + 1] = fmaf(p, x4.y, t[4 * v4 + 1]);
            t[4 * v4 + 2] = fmaf(p, x4.z, t[4 * v4 + 2]);
            t[4 * v4 + 3] = fmaf(p, x4.w, t[4 * v4 + 3]);
          }
        }
#pragma unroll
        for (int v = 0; v < kNaTile; ++v) acc[v] += t[v];
      }
    }
    float dsv[kNaTile], smv[kNaTile];
#pragma unroll
    for (int v = 0; v < kNaTile; ++v) {
      const bool on = live && ((act >> v) & 1u);
      const float y = fmaf(ri, fmaf(b1[v], so[v], q[v]), acc[v]);
      const float sn = fmaf(-e_s[v], y, y);
      dsv[v] = on ? fabsf(sn - so[v]) : 0.0f;
      smv[v] = on ? fabsf(sn) : 0.0f;
      so[v] = on ? sn : so[v];
    }
    const int nxt = cur ^ 1;
    if (live) {
#pragma unroll
      for (int v = 0; v < kNaTile; v += 4)
        *reinterpret_cast<float4*>(&Xs[nxt][i][v]) =
            make_float4(q[v] + b1[v] * so[v], q[v + 1] + b1[v + 1] * so[v + 1], q[v + 2] + b1[v + 2] * so[v + 2],
                        q[v + 3] + b1[v + 3] * so[v + 3]);
    }
    red_d[warp][lane] = noalloc_transpose_max(dsv, lane);
    red_s[warp][lane] = noalloc_transpose_max(smv, lane);
    __syncthreads();
    if (tid < kNaTile) {
      const int v = tid;
      unsigned done = 0u;
      if ((act >> v) & 1u) {
        float D = 0.0f, Sm = 0.0f;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          D = fmaxf(D, red_d[w][v]);
          Sm = fmaxf(Sm, red_s[w][v]);
        }
        const float r = rho_s[v];
        const float scale = fmaxf(Sm, 1e-6f * s_glob);
        if (D < best_s[v]) {
          best_s[v] = D;
          stall_s[v] = 0;
        } else {
          stall_s[v] += 1;
        }
        if ((r / (1.0f - r)) * D <= tol * scale || stall_s[v] >= 3) {
          done = 1u;
          iters_s[v] = k;
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, done);
      if (tid == 0) act_s = act & ~mask;
    }
    __syncthreads();
    act = act_s;
    cur = nxt;
  }
  if (tid < kNaTile && ((act >> tid) & 1u)) {
    iters_s[tid] = k;
    atomicAdd(&sc->nonconv, 1);
  }
  if (live) {
#pragma unroll
    for (int v = 0; v < kNaTile; ++v) {
      const int vv = v0 + v;
      if (vv < nvox) {
        S_out[static_cast<size_t>(i) * plane + vv] = so[v];
        I_out[static_cast<size_t>(i) * plane + vv] = fmaf(b1[v], so[v], q[v]);
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    int im = 0;
    for (int v = 0; v < kNaTile && v0 + v < nvox; ++v) im = max(im, iters_s[v]);
    atomicMax(&sc->iters_max, im);
  }
}

}  // namespace
}  // namespace trinity

using namespace trinity;

extern "C" int trinity_source_iteration_noalloc(int na, int nvox, const float* P, const float* Q, const float* b1,
                                                const float* eps, const float* S_prev, float* S_out, float* I_out,
                                                double tol, int max_iters, int* iters_max, void* stream) {
  if (na != 12 && na != 48 && na != 192) return TRINITY_E_INVALID;
  if (nvox < 1 || nvox > kNoAllocMaxVoxels) return TRINITY_E_INVALID;  // beyond the static scratch
  if (!P || !Q || !b1 || !eps || !S_prev || !S_out || !I_out || !(tol > 0.0) || max_iters < 1)
    return TRINITY_E_INVALID;
  NoAllocScratch* sc = nullptr;
  int rc = scratch_for_current_device(&sc);
  if (rc != TRINITY_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the counters and the max cell start at zero on every call; rho is overwritten below
  if (cudaMemsetAsync(sc, 0, offsetof(NoAllocScratch, rho), st) != cudaSuccess) return TRINITY_E_CUDA;
  noalloc_prepass<<<(nvox + 255) / 256, 256, 0, st>>>(na, nvox, na == 12 ? b1 : nullptr, eps, S_prev, sc);
  const float ftol = static_cast<float>(tol);
  if (na == 12) {
    const int tiles = (nvox + kNaTile - 1) / kNaTile;
    noalloc_iteration<12><<<tiles, 32, 0, st>>>(nvox, P, Q, b1, eps, S_prev, S_out, I_out, ftol, max_iters, sc);
  } else {
    if (!scatter_split_supported(na, 0)) return TRINITY_E_CUDA;
    if (na == 48)
      noalloc_split_prep<48><<<1 + 48 / 8, 1024, 0, st>>>(P, sc);
    else
      noalloc_split_prep<192><<<1 + 192 / 8, 1024, 0, st>>>(P, sc);
    SplitTables sp{};
    sp.ph = reinterpret_cast<const uint8_t*>(sc->ph);
    sp.pl = reinterpret_cast<const uint8_t*>(sc->pl);
    sp.diag = sc->diag;
    sp.cw = sc->cw;
    sp.dyn = sc->dyn;
    sp.cycle = 8;
    sp.max_inner = 256;
    SplitIo io{};
    io.q = Q;
    io.s1 = S_prev;
    io.eps = eps;
    io.b1 = b1;
    io.s_glob = &sc->smax;
    io.I = I_out;
    io.S = S_out;
    if (launch_scatter_split_buffers(na, nvox, sp, io, ftol, max_iters, &sc->iters_max, &sc->nonconv, &sc->error, st) !=
        cudaSuccess)
      return TRINITY_E_CUDA;
  }
  if (cudaGetLastError() != cudaSuccess) return TRINITY_E_CUDA;
  int counters[3] = {0, 0, 0};
  if (cudaMemcpyAsync(counters, &sc->iters_max, sizeof(counters), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return TRINITY_E_CUDA;
  if (counters[2] != 0) return TRINITY_E_TIMEOUT;
  if (iters_max) *iters_max = counters[0];
  return counters[1] > 0 ? TRINITY_W_NOT_CONVERGED : TRINITY_OK;
}
