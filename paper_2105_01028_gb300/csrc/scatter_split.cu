// FP32 source iteration on the 5th-generation tensor cores (tcgen05): FP32-accurate
// residuals from split FP16 operands, corrections from single FP16 products.
//
// Per voxel the source function is the fixed point of S = a P (Q + b1 o S) (Eq. 12 with
// Eq. 10).  The plain iteration applies an FP32 product P X some 40 times per voxel and
// step; on the CUDA cores that is bound by the FP32 pipe.  Here the fixed point is reached
// by iterative refinement:
//
//   outer: r = a P~ (Q + b1 S) - S with an FP32-accurate product (below): the plain
//          iteration's change, on which its stop test is taken (at a quarter of the
//          tolerance: the recursion has no noise floor that would hold it above);
//   inner: the error equation (1 - a P B1) e = r is solved to the relative accuracy of one
//          FP16 product per iteration, S += e, and r follows by recursion.
//
// The result carries the accuracy of the outer residual: what an inner product rounds is a
// part of 2^-11 of the correction it makes, and an outer residual follows until that part
// is below the tolerance (two outers per voxel and step on a developed slab).
//
// FP32-accurate product.  The diagonal of P~ is applied in FP32 (it holds half a row's
// weight at g = 0.9); the off-diagonal part, in units of about 2^-t, is split as Ph + Pl + Pm
// with Ph whole numbers of at most 11 bits, Pl the FP16 number nearest to the rest and Pm that
// nearest to what is left (the entries of a peaked kernel span a factor of 500, and the smallest
// are two units: with Ph and Pl alone they are off by 5e-5 of themselves, and all that a
// detector beside the source sees first went through them).  X, scaled per voxel by a power of
// two, is split as Xh + Xl + Xm, Xh whole below 2^10, Xl multiples of 2^-12 and Xm the rest (where
// one direction outshines the others 1e4 times, Xh + Xl leaves the weak outgoing directions
// 1.7e-4 off; with Xm they are 5e-7 off at most, a sum of 192 FP32 products 2e-6).  t is
// chosen so that every partial sum of Xh Ph stays below 2^24: the FP32 accumulator in TMEM then
// holds it exactly, whatever the order, and its truncation (the tensor core does not round an
// accumulation to nearest: three TF32 products summed in one accumulator are 1.7e-6 off,
// one-sided) has nothing to act on.  Xm Ph + Xh Pm + Xl Pl + Xh Pl + Xl Ph goes to a second
// accumulator, 2^-10 of the first in size, where the truncation is below 2^-32 of the result
// (3e-8 of it in the weak directions above).  Each row of
// Ph + Pl + Pm + diag sums to one (the diagonal is a float pair; what the terms drop is 1e-10 of
// the row), so photons are conserved.
// Measured against FP64 on the 96x96x64 slab after two steps, in 2-norm: I 9.1e-8, S 8.7e-8;
// the sums of 192 FP32 products on the CUDA cores that it replaces: 2.1e-7 and 2.3e-7.  Two steps
// of that slab at 192 directions: 6.38 ms (155 before); 100 steps of 16^3 at 48 directions: 5.1 ms
// (14.2); 110592 voxels of 192 directions on the caller's buffers, cold: 1.38 ms (54.2).
//
// Inner iteration.  Isotropic rebalance as in the other kernels: c = a sum_j b1_j r_j /
// sum_j (1 - a b1_j) is added to every direction of r; the two-grid iteration that this
// makes has its spectrum in about [0, rho |g|], and Chebyshev weights over that interval
// (roots in an order that keeps the partial products bounded) damp it by 0.43 an
// iteration instead of 0.8:  d = r + c,  S += w d,  r <- r - w d + w a P B1 d.
// As P c = c, P B1 d = c + P x with x = b1 r - u c = r - u d, u = 1 - b1: in thick voxels c is
// r / (u + eps), up to thousands of r, and b1 d in FP16 would be off by more than r, alike in all
// directions (the corrections then diverge); x is of the size of r.  P x is one chain of K = 16
// MMAs of FP16 x (scaled by a power of two per voxel) and Ph, its diagonal again FP32.
//
// Layout: as the BF16 kernel's (scatter_tc.cu): persistent CTAs, tiles of 8 x 4 x 4 voxels
// (M = 128), operands K-major with the 128-byte swizzle, one voxel row per thread, four
// column groups of 48 directions (three of 16 at 48 directions).  TMEM: D / first
// accumulator in [0, N_a), r / second accumulator in [256, 256 + N_a) and, at 192
// directions, two thirds of Q in the columns left over; S stays in registers.  Shared
// memory at 192 directions: Ph 72 KB, Xh and Xl 48 KB each; Pm and Pl (72 KB each) do not fit
// beside them and are streamed from L2 in twelve 12 KB blocks through a ring of three, and Xl
// takes the place of Xm when the MMAs on Xm are done (written under the next ones).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <vector>

#include "device.cuh"
#include "tcgen05.cuh"

namespace trinity {

namespace {

constexpr int kSplitCycle = 64;                // longest Chebyshev cycle
constexpr float kTolShare = 0.25f;             // share of the tolerance the stop test leaves to the change
constexpr float kInnerError = 4.8828125e-04f;  // 2^-11: error of an inner correction, relative to it
constexpr float kInnerDrop = 9.765625e-04f;    // 2^-10: an inner solve reduces its residual this far at most
constexpr float kMinAmp = 2.384185791015625e-07f;  // 2^-22: rounding of S that a change may leave behind
constexpr int kMaxStalls = 3;  // residuals that are not halved before a voxel above the floor is given up
// Rows below this are held scaled up: 2^-50, so that a residual 2^-37 of the row still has its
// full scale in scale_exponent.
constexpr float kTiny = 8.8817841970012523e-16f;

template <int NA>
struct Sp {
  static constexpr int KB = (NA + 63) / 64;        // 128-byte K blocks
  static constexpr int KSTEPS = NA / 16;           // MMAs per operand pair (K = 16 each)
  static constexpr int kGroups = NA >= 192 ? 4 : 3;
  static constexpr int kThreads = 128 * kGroups;
  static constexpr int HALF = NA / kGroups;        // columns per thread
  static constexpr int CH = 8;                     // columns per TMEM load
  static constexpr int NCH = HALF / CH;
  static constexpr int QT = NA >= 192 ? 32 : 0;    // Q columns per thread kept in TMEM
  static constexpr int QR = HALF - QT;             // ... and in registers
  static constexpr int NCT = QT / CH;
  static constexpr int POW2 = NA <= 64 ? 64 : 256;
  static constexpr int TCOLS = 2 * POW2;
  static constexpr int ROFF = POW2;                // residual / second accumulator
  static constexpr bool kRing = NA >= 192;         // Pl streamed through a ring
  static constexpr int kBlkRows = 96;
  static constexpr int kBlkN = kRing ? kBlkRows : NA;  // N of the second accumulator's MMAs
  static constexpr int kHalves = NA / kBlkN;
  static constexpr int kBlkBytes = kBlkRows * 128;
  static constexpr int kNblk = kRing ? 2 * KB * (NA / kBlkRows) : 1;  // blocks of Pm, then of Pl
  static constexpr int kSlots = 3;
  static constexpr int P_BYTES = KB * NA * 128;
  static constexpr int A_BYTES = KB * kM * 128;
  static constexpr int OFF_PH = 0;
  static constexpr int OFF_XH = (P_BYTES + 1023) / 1024 * 1024;
  static constexpr int OFF_XL = OFF_XH + A_BYTES;
  static constexpr int OFF_XM = kRing ? OFF_XL : OFF_XL + A_BYTES;  // (ring: Xm and Xl take turns)
  static constexpr int OFF_PL = OFF_XM + A_BYTES;
  static constexpr int PL_BYTES = kRing ? kSlots * kBlkBytes : 2 * P_BYTES;  // ring, or Pm and then Pl
  static_assert(P_BYTES % 1024 == 0, "operand images follow one another");
  static constexpr int OFF_B1T = OFF_PL + PL_BYTES;                // [kMaxClasses][kM] f32
  static constexpr int OFF_DI = OFF_B1T + kMaxClasses * kM * 4;    // [3][NA] f32: diagonals
  static constexpr int OFF_B1C = OFF_DI + 3 * NA * 4;              // [NA] f32 (uniform mu_t)
  static constexpr int OFF_CLS = OFF_B1C + NA * 4;                 // [NA] u8
  static constexpr int SMEM = OFF_CLS + ((NA + 15) / 16) * 16 + 1024;
  static constexpr uint32_t IDESC_ANY = (1u << 4) | (static_cast<uint32_t>(kM >> 4) << 24);  // FP16 x FP16 -> FP32
  static constexpr uint32_t IDESC = IDESC_ANY | (static_cast<uint32_t>(NA >> 3) << 17);
  static constexpr uint32_t IDESC_BLK = IDESC_ANY | (static_cast<uint32_t>(kBlkN >> 3) << 17);
};

__device__ __forceinline__ float pow2f(int e) { return __uint_as_float(static_cast<uint32_t>(127 + e) << 23); }
__device__ __forceinline__ int exponent(float x) { return static_cast<int>((__float_as_uint(x) >> 23) & 0xffu) - 127; }

// Power-of-two scale 2^e that brings a row whose largest element is m to [2^top, 2^(top+1)),
// kept within the range where 2^-(e + 24) is a normal float (kTiny sees to it that this does not
// bind).
__device__ __forceinline__ int scale_exponent(float m, int top) {
  const int e = m > 0.0f ? top - exponent(m) : 0;
  return e > 100 ? 100 : e;
}

__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// u (|u| < 2^14) = h + l + m: h the nearest multiple of 16, l the rest to multiples of 2^-8,
// m what is left (the magic additions round to nearest even at bits 4 and -8; every other step
// is exact, and m is rounded when it is packed: 2^-35 of the row's largest element).
__device__ __forceinline__ void split_u(float u, float& h, float& l, float& m) {
  h = (u + 201326592.0f) - 201326592.0f;
  const float d = u - h;
  l = (d + 49152.0f) - 49152.0f;
  m = d - l;
}

__device__ __forceinline__ void bulk_to_smem(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// What a launch solves for:
//   kStep     S(n) of a forward step (Q and the S ring of a context; I and S written);
//   kBuffers  the same on caller-owned buffers with b1 given per (direction, voxel);
//   kAdjoint  the transposed solve y = a P (Sbar + b1 (Ibar + y)) of a reverse step: the
//             same equation with Q = Sbar + b1 Ibar; the tile's end writes Qbar = Ibar + y,
//             clears the consumed adjoint level and adds the gradient sums.
enum SplitMode { kStep = 0, kBuffers = 1, kAdjoint = 2 };

// kUniB1: mu_t is the same in every voxel, so b1 depends on the column's ray spacing only.
// kPer: CTAs per SM (two at 48 directions where there are tiles enough; the registers that this
// takes would cost a single CTA 20%).
template <int NA, bool kUniB1, int kMode, int kPer>
__global__ void __launch_bounds__(Sp<NA>::kThreads, kPer)
    scatter_split_kernel(GridParams g, SplitTables t, const uint8_t* __restrict__ cls,
                         const float* __restrict__ cls_ds, int ncls, int nch, SplitIo io, float tol, int max_iters,
                         const __grid_constant__ CUtensorMap tmOutI, const __grid_constant__ CUtensorMap tmOutS,
                         int tma_out, RunState rs) {
  using C = Sp<NA>;
  constexpr int CH = C::CH, NCH = C::NCH, NCT = C::NCT;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sPh = smem + C::OFF_PH;
  uint8_t* sXh = smem + C::OFF_XH;
  uint8_t* sXl = smem + C::OFF_XL;
  uint8_t* sXm = smem + C::OFF_XM;
  uint8_t* sPl = smem + C::OFF_PL;
  float* b1t = reinterpret_cast<float*>(smem + C::OFF_B1T);
  float* sDi = reinterpret_cast<float*>(smem + C::OFF_DI);  // diagonal of P~ (hi), (lo); of the inner operator
  float* sB1c = reinterpret_cast<float*>(smem + C::OFF_B1C);
  uint8_t* sCls = smem + C::OFF_CLS;

  __shared__ uint64_t mbar;
  __shared__ uint64_t pl_full[C::kSlots], pl_empty[C::kSlots];
  __shared__ uint32_t tmem_base_s;
  __shared__ int tile_s;
  __shared__ int abort_s;
  __shared__ float e_s[kM], rho_s[kM], den_s[kM];
  __shared__ int up_s[kM];  // a row's S and Q are held times 2^up (0 but for very dim rows)
  __shared__ int ccnt_s[kMaxClasses];
  __shared__ float clsb1_s[kMaxClasses];
  __shared__ float sumb1_s;
  __shared__ float cw_s[kSplitCycle];
  constexpr int kGroups = C::kGroups;
  __shared__ float red_d[kGroups][kM], red_s[kGroups][kM], red_c[kGroups][kM];
  __shared__ double esum_s[C::kThreads / 32];
  __shared__ double asum_sh;
  __shared__ float smax_s[C::kThreads / 32];

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int row = ((warp & 3) << 5) + lane;
  const int grp = warp >> 2;  // column group
  const int cb = grp * C::HALF;
  const int n = kMode == kStep ? *rs.step : 0;
  const size_t plane = static_cast<size_t>(g.nv);
  const float s_glob = __uint_as_float(kMode == kStep ? rs.smax[(n - 1) & 1] : *io.s_glob);
  // start of the iteration: the previous level and, for the linear extrapolation in time,
  // the one before it
  const float* sp1 = io.s1;
  const float* sp2 = io.s2;
  if (kMode == kStep) {
    sp1 = (n - 1) >= g.hist_from ? io.s1 + static_cast<size_t>(ring_slot(n - 1)) * g.na * plane : nullptr;
    sp2 = g.warm != 0 && (n - 2) >= g.hist_from ? io.s1 + static_cast<size_t>(ring_slot(n - 2)) * g.na * plane
                                                : nullptr;
  }
  const size_t cur_base = static_cast<size_t>(ring_slot(n)) * g.na * plane;
  const int bxn = (g.nx + 7) >> 3, byn = (g.ny + 3) >> 2;
  // flat tiles of 128 voxels where the voxels have no grid
  const int ntiles = kMode == kBuffers ? (g.nv + kM - 1) / kM : brick_tiles(g.nx, g.ny, g.nz);
  const auto tile_voxel = [&](int tl, int r) {
    if (kMode == kBuffers) {
      const int f = tl * kM + r;
      return f < g.nv ? f : -1;
    }
    return brick_voxel(g, bxn, byn, tl, r);
  };

  // ---- one-time set-up: TMEM, barriers, operand images, diagonals, class tables
  if (warp == 0) tmem_alloc(&tmem_base_s, C::TCOLS);
  uint32_t pl_issued = 0, pl_used = 0;  // thread 0: Pl blocks loaded and consumed so far
  const auto pl_load = [&]() {
    const uint32_t s = pl_issued % C::kSlots;
    bulk_to_smem(smem_u32(sPl) + s * C::kBlkBytes,
                 t.pl + static_cast<size_t>(pl_issued % C::kNblk) * C::kBlkBytes, C::kBlkBytes, &pl_full[s]);
    ++pl_issued;
  };
  if (tid == 0) {
    mbar_init(&mbar);
    for (int s = 0; s < C::kSlots; ++s) {
      mbar_init(&pl_full[s]);
      mbar_init(&pl_empty[s]);
    }
    abort_s = 0;
    asum_sh = 0.0;
    if constexpr (C::kRing) {
      for (int s = 0; s < C::kSlots; ++s) pl_load();
    }
  }
  for (int u = tid; u < C::P_BYTES / 16; u += blockDim.x)
    reinterpret_cast<uint4*>(sPh)[u] = __ldg(reinterpret_cast<const uint4*>(t.ph) + u);
  if constexpr (!C::kRing) {
    for (int u = tid; u < C::PL_BYTES / 16; u += blockDim.x)
      reinterpret_cast<uint4*>(sPl)[u] = __ldg(reinterpret_cast<const uint4*>(t.pl) + u);
  }
  if (tid < kMaxClasses) ccnt_s[tid] = 0;
  if (tid < kSplitCycle) cw_s[tid] = t.cw[tid];
  __syncthreads();
  for (int i = tid; i < NA; i += blockDim.x) {
    sDi[i] = t.diag[i];
    sDi[NA + i] = t.diag[NA + i];
    sDi[2 * NA + i] = t.diag[2 * NA + i];
    if (kMode == kBuffers) continue;
    atomicAdd(&ccnt_s[cls[i]], 1);
    sCls[i] = cls[i];
    if (kUniB1) {  // the same operations as the per-row table below, on the same mu_t
      const int k = cls[i];
      float bs = 0.0f;
      for (int j = 0; j < nch; ++j) bs += ray_u_fine(g.mut_u, cls_ds[k * nch + j], cls_ds[(16 + k) * nch + j]);
      sB1c[i] = bs * (1.0f / static_cast<float>(nch));
    }
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (kUniB1) {
    // the denominators' sum_j b1_j, in the order the general form sums it (per class; all
    // directions of a class hold the same b1, so concurrent writes store the same value)
    for (int i = tid; i < NA; i += blockDim.x) clsb1_s[sCls[i]] = sB1c[i];
    __syncthreads();
    if (tid == 0) {
      float sb = 0.0f;
      for (int k2 = 0; k2 < ncls; ++k2) sb = fmaf(static_cast<float>(ccnt_s[k2]), clsb1_s[k2], sb);
      sumb1_s = sb;
    }
    __syncthreads();
  }
  const uint32_t tmem = tmem_base_s;
  const uint32_t t_row = tmem + (static_cast<uint32_t>((warp & 3) << 5) << 16);
  // this thread's Q columns in TMEM (column group h: N_a + 32 h for h < 2, ROFF + N_a + 32 (h - 2))
  const uint32_t t_q = t_row + static_cast<uint32_t>(grp < 2 ? NA + C::QT * grp : C::ROFF + NA + C::QT * (grp - 2));
  const uint32_t aXh = smem_u32(sXh), aXl = smem_u32(sXl), aXm = smem_u32(sXm);
  const uint32_t aPh = smem_u32(sPh), aPl = smem_u32(sPl);
  uint32_t phase = 0;
  bool aborted = false;
  double esum = 0.0;
  float smax_loc = 0.0f;
  float S[C::HALF];                       // S of the thread's row and columns
  float qr[C::QR];                        // Q of the thread's last QR columns
  // one unit of Ph and the Chebyshev interval (from the device where P came from there)
  const float tscale = t.dyn ? t.dyn[0] : t.unit, lam = t.dyn ? t.dyn[1] : t.lam, lam_lo = t.dyn ? t.dyn[2] : t.lo;
  bool first_tile = true;
  int claimed = (kMode == kStep && tid == 0) ? atomicAdd(rs.tile_ctr + (n & 1), 1) : 0;

  // Weight of 8 columns from c0 on, as b1_of and form_x read it (volatile or asm loads: hoisted
  // out of the iterations these tables would cost more registers than there are)
  // (kBuffers: b1 from the caller's array; in the inner iterations u = 1 - b1 as FP16, kept where
  // Xl was.  b1 itself in FP16 is one in thick voxels, and the corrections then diverge.)
  int v = 0;
  const auto load_w = [&](int c0, float (&bv)[8], bool inner_pass = false) {
    if (kMode == kBuffers) {
      if (inner_pass) {
        const volatile __half* hb = reinterpret_cast<const volatile __half*>(sXl) + c0 * kM + row;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          __half_raw hr;
          hr.x = reinterpret_cast<const volatile unsigned short*>(hb)[j * kM];
          bv[j] = __half2float(__half(hr));
        }
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) bv[j] = io.b1[static_cast<size_t>(c0 + j) * plane + v];
      }
    } else if (kUniB1) {
      lds_vec<8>(sB1c + c0, bv);
    } else {
      const volatile float* vb = b1t;
      uint32_t cv[2];
      lds_bytes<8>(sCls + c0, cv);
#pragma unroll
      for (int j = 0; j < 8; ++j) bv[j] = vb[((cv[j >> 2] >> (8 * (j & 3))) & 0xffu) * kM + row];
    }
  };
  // Q of chunk ch (issued before tmem_wait_ld where it lives in TMEM)
  const auto load_q = [&](int ch, float (&qv)[CH]) {
    if (ch < NCT) tmem_ld<CH>(t_q + ch * CH, qv);
  };
  const auto reg_q = [&](int ch, float (&qv)[CH]) {
    if (ch >= NCT) {
#pragma unroll
      for (int j = 0; j < CH; ++j) qv[j] = qr[(ch - NCT) * CH + j];
    }
  };
  // max over the row's column groups of red_d, red_s, sum of red_c
  const auto row_max = [&](const float (&red)[kGroups][kM]) {
    float m = red[0][row];
#pragma unroll
    for (int gi = 1; gi < kGroups; ++gi) m = fmaxf(m, red[gi][row]);
    return m;
  };
  const auto row_sum = [&](const float (&red)[kGroups][kM]) {
    float s = red[0][row];
#pragma unroll
    for (int gi = 1; gi < kGroups; ++gi) s += red[gi][row];
    return s;
  };
  // b1 is held as u = 1 - b1 (kBuffers: as the caller gave it): in thick cells the rounding of
  // b1 itself would be multiplied by 1 / (1 - a b1), u carries ten times less of it
  const auto b1_of = [](float w) { return kMode == kBuffers ? w : 1.0f - w; };
  const auto form_x = [](float w, float sv, float q) {  // Q + b1 S
    return kMode == kBuffers ? fmaf(w, sv, q) : fmaf(-w, sv, q + sv);
  };
  // wait for the MMAs committed to mbar; false for the whole warp if the wait ran out
  const auto wait_mma = [&]() {
    const bool ok = mbar_wait_bounded(&mbar, phase);
    phase ^= 1u;
    if (!ok) abort_s = 1;
    const bool to = __any_sync(0xffffffffu, !ok);
    tc_fence_after();
    return !to;
  };
  // thread 0: the ring slots just used take the next blocks once their MMAs are done
  const auto pl_refill = [&]() {
    bool ok = true;
    for (uint32_t q = pl_used - C::kSlots; ok && q < pl_used; ++q) {
      ok = mbar_wait_bounded(&pl_empty[q % C::kSlots], (q / C::kSlots) & 1u);
      if (ok) pl_load();
    }
    return ok;
  };
  // thread 0: the two accumulators of an FP32-accurate product.  kHead: the part that needs Xh
  // and Xm, the rest waits for Xl (at 48 directions all three are there and the head is all)
  const auto issue_product = [&](auto head) {
    [[maybe_unused]] constexpr bool kHead = decltype(head)::value;
    tc_fence_after();
    bool ok = true;
    // K steps [from, to) of an X term times Ph into the second accumulator, which is built by
    // MMAs of one shape: only these are executed in the order of their issue (96 rows are
    // twelve swizzle atoms, so a half starts on one)
    const auto low_ph = [&](uint32_t ax, int from, int to, bool first) {
#pragma unroll
      for (int s = from; s < to; ++s) {
        const uint32_t ko = static_cast<uint32_t>((s & 3) * 32), kb = static_cast<uint32_t>(s >> 2);
#pragma unroll
        for (int h = 0; h < C::kHalves; ++h)
          mma_f16(tmem + C::ROFF + h * C::kBlkN, sw128_desc(ax + kb * kM * 128 + ko),
                  sw128_desc(aPh + (kb * NA + h * C::kBlkN) * 128 + ko), C::IDESC_BLK, (first && s == 0) ? 0u : 1u);
      }
    };
    const auto xh_ph = [&](int from, int to) {
#pragma unroll
      for (int s = from; s < to; ++s) {
        const uint32_t ko = static_cast<uint32_t>((s & 3) * 32), kb = static_cast<uint32_t>(s >> 2);
        mma_f16(tmem, sw128_desc(aXh + kb * kM * 128 + ko), sw128_desc(aPh + kb * NA * 128 + ko), C::IDESC, s > 0);
      }
    };
    if constexpr (C::kRing) {
      // Block b of Pm (b < 6, with Xh alone) or Pl: K block (b % 6) / 2, output directions
      // 96 (b & 1) .. + 95, into the second accumulator, from ring slot pl_used % kSlots
      const auto pl_blocks = [&](int b0) {
#pragma unroll 1
        for (int b = b0; b < b0 + C::kSlots; ++b) {
          const uint32_t sl = pl_used % C::kSlots;
          if (ok) ok = mbar_wait_bounded(&pl_full[sl], (pl_used / C::kSlots) & 1u);
          if (!ok) return;
          tc_fence_after();
          const bool low = b < C::kNblk / 2;
          const uint32_t kb = static_cast<uint32_t>((low ? b : b - C::kNblk / 2) >> 1);
          const uint32_t d = tmem + C::ROFF + (b & 1) * C::kBlkRows;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint64_t pd = sw128_desc(aPl + sl * C::kBlkBytes + ks * 32);
            if (!low) mma_f16(d, sw128_desc(aXl + kb * kM * 128 + ks * 32), pd, C::IDESC_BLK, 1u);
            mma_f16(d, sw128_desc(aXh + kb * kM * 128 + ks * 32), pd, C::IDESC_BLK, 1u);
          }
          mma_commit(&pl_empty[sl]);
          ++pl_used;
        }
      };
      // the ring is refilled while MMAs on Ph run
      static_assert(C::kNblk == 4 * C::kSlots, "a product takes the ring four times");
      if (kHead) {
        low_ph(aXm, 0, C::KSTEPS, true);
        mma_commit(&mbar);  // Xm is free for Xl
        pl_blocks(0);
        xh_ph(0, C::KSTEPS / 2);
        if (!ok) abort_s = 1;
        return;
      }
      low_ph(aXl, 0, C::KSTEPS / 2, false);
      pl_blocks(C::kSlots);
      low_ph(aXl, C::KSTEPS / 2, C::KSTEPS, false);
      ok = ok && pl_refill();
      pl_blocks(2 * C::kSlots);
      xh_ph(C::KSTEPS / 2, C::KSTEPS);
      ok = ok && pl_refill();
      pl_blocks(3 * C::kSlots);
    } else {
      // terms in order of size, the small ones first
      low_ph(aXm, 0, C::KSTEPS, true);
#pragma unroll
      for (int s = 0; s < C::KSTEPS; ++s) {
        const uint32_t ko = static_cast<uint32_t>(s * 32);
        mma_f16(tmem + C::ROFF, sw128_desc(aXh + ko), sw128_desc(aPl + ko), C::IDESC_BLK, 1u);
        mma_f16(tmem + C::ROFF, sw128_desc(aXl + ko), sw128_desc(aPl + C::P_BYTES + ko), C::IDESC_BLK, 1u);
      }
#pragma unroll
      for (int s = 0; s < C::KSTEPS; ++s) {
        const uint32_t ko = static_cast<uint32_t>(s * 32);
        mma_f16(tmem + C::ROFF, sw128_desc(aXh + ko), sw128_desc(aPl + C::P_BYTES + ko), C::IDESC_BLK, 1u);
      }
      low_ph(aXl, 0, C::KSTEPS, false);
      xh_ph(0, C::KSTEPS);
    }
    mma_commit(&mbar);
    if (!ok) abort_s = 1;
  };

  while (true) {
    // the previous tile's TMA stores must have read the staging area (the X operands)
    // before X is written again
    if (tid == 0) {
      if (tma_out) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      if (kMode == kStep) {
        tile_s = claimed;
        claimed = atomicAdd(rs.tile_ctr + (n & 1), 1);  // needed for the next tile only
      } else {
        tile_s = first_tile ? static_cast<int>(blockIdx.x) : tile_s + static_cast<int>(gridDim.x);
      }
    }
    first_tile = false;
    __syncthreads();
    const int tile = tile_s;
    if (tile >= ntiles) break;
    const int vb = tile_voxel(tile, row);
    const bool vin = vb >= 0;
    v = vin ? vb : 0;

    // per-row constants and the b1 table over ds classes
    if (tid < kM) {
      const int vv = tile_voxel(tile, tid);
      float ev = 1.0f, rho = 0.0f;
      if (vv >= 0) {
        ev = io.eps[vv];
        if (kMode != kBuffers) {
          const float xm = io.mut[vv] * g.ds_max;
          rho = (1.0f - ev) * ray_b1(xm, expf(-xm));
        }
      }
      e_s[tid] = ev;
      rho_s[tid] = rho;
      up_s[tid] = 0;
    }
    for (int u = tid; u < (kUniB1 || kMode == kBuffers ? 0 : ncls * kM); u += blockDim.x) {
      const int k = u / kM, r = u % kM;
      const int vv = tile_voxel(tile, r);
      float bs = 0.0f;
      if (vv >= 0) {
        const float mu = io.mut[vv];
        for (int j = 0; j < nch; ++j) bs += ray_u_fine(mu, cls_ds[k * nch + j], cls_ds[(16 + k) * nch + j]);
      }
      b1t[k * kM + r] = bs * (1.0f / static_cast<float>(nch));
    }
    __syncthreads();
    // rebalance denominator sum_j (1 - a b1_j) of each row
    if (tid < kM && kMode != kBuffers) {
      float sb;
      if (kUniB1) {
        sb = sumb1_s;
      } else {
        sb = 0.0f;
        for (int k2 = 0; k2 < ncls; ++k2) sb = fmaf(static_cast<float>(ccnt_s[k2]), b1t[k2 * kM + tid], sb);
      }
      den_s[tid] = fmaf(static_cast<float>(NA), e_s[tid], (1.0f - e_s[tid]) * sb);  // sb sums u = 1 - b1
    }

    // ---- warm start (the previous level or its extrapolation in time) into registers; Q
    // (read once) into TMEM or registers; max |X| of the row.  Loads go two chunks (48 per
    // thread) at a time.
    float xmax = 0.0f, bmax = 0.0f, bsum = 0.0f;
    {
      static_assert(NCH % 2 == 0 && NCT % 2 == 0, "chunks go in pairs");
      constexpr int PR = kMode == kStep ? 2 : 1;
#pragma unroll
      for (int c2 = 0; c2 < NCH; c2 += PR) {
        float s1[PR][CH], s2[PR][CH], qc[PR][CH], qi[PR][CH];
#pragma unroll
        for (int u = 0; u < PR; ++u)
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const size_t col = static_cast<size_t>(cb + (c2 + u) * CH + j) * plane + v;
            s1[u][j] = (vin && sp1) ? (kMode == kStep ? __ldg(sp1 + col) : sp1[col]) : 0.0f;
            s2[u][j] = (vin && sp2) ? (kMode == kStep ? __ldg(sp2 + col) : sp2[col]) : 0.0f;
            qc[u][j] = vin ? (kMode == kStep ? __ldg(io.q + col) : io.q[col]) : 0.0f;
            qi[u][j] = (kMode == kAdjoint && vin) ? io.ib[col] : 0.0f;
          }
#pragma unroll
        for (int u = 0; u < PR; ++u) {
          const int ch = c2 + u;
          float bv[8];
          load_w(cb + ch * CH, bv);
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            if (kMode == kAdjoint) qc[u][j] = form_x(bv[j], qi[u][j], qc[u][j]);  // Sbar + b1 Ibar
            if (kMode == kBuffers) {
              bmax = fmaxf(bmax, bv[j]);
              bsum += 1.0f - bv[j];
            }
            const float s0 = (vin && sp2) ? fmaf(2.0f, s1[u][j], -s2[u][j]) : s1[u][j];
            S[ch * CH + j] = s0;
            xmax = fmaxf(xmax, fabsf(form_x(bv[j], s0, qc[u][j])));
            if (ch >= NCT) qr[(ch - NCT) * CH + j] = qc[u][j];
          }
          if (ch < NCT) tmem_st<CH>(t_q + ch * CH, qc[u]);
        }
      }
    }
    red_d[grp][row] = xmax;
    if (kMode == kBuffers) {
      red_s[grp][row] = bmax;
      red_c[grp][row] = bsum;
    }
    tmem_wait_st();
    const bool any_tiny = __syncthreads_or(xmax > 0.0f && xmax < kTiny) != 0;
    float den = den_s[row];
    float rho = rho_s[row];
    if (kMode == kBuffers) {
      rho = (1.0f - e_s[row]) * row_max(red_s);
      den = fmaf(static_cast<float>(NA), e_s[row], (1.0f - e_s[row]) * row_sum(red_c));
    }
    // Rows so dim that the powers of two below would leave FP32's range (the light front, a
    // misfit in absolute units) are held multiplied by a power of two, to about one, and
    // divided by it at the end; both are exact.
    if (any_tiny) {
      float s0 = 0.0f, up = 1.0f;
#pragma unroll
      for (int j = 0; j < C::HALF; ++j) s0 = fmaxf(s0, fabsf(S[j]));
      __syncthreads();  // the reads of red_s above
      red_s[grp][row] = s0;
      __syncthreads();
      const float m = row_max(red_d);
      if (m > 0.0f && m < kTiny) {
        int e = min(-exponent(m), 100 - exponent(row_max(red_s)));
        e = e < 0 ? 0 : (e > 120 ? 120 : e);
        up = pow2f(e);
        if (grp == 0) up_s[row] = e;
      }
      __syncthreads();
      red_d[grp][row] = xmax * up;
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        float qv[CH];
        load_q(ch, qv);
        if (ch < NCT) tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          S[ch * CH + j] *= up;
          if (ch < NCT)
            qv[j] *= up;
          else
            qr[(ch - NCT) * CH + j] *= up;
        }
        if (ch < NCT) tmem_st<CH>(t_q + ch * CH, qv);
      }
      tmem_wait_st();
      __syncthreads();
    }

    const float ev = e_s[row], al = 1.0f - ev;
    const float amp = rho / (1.0f - rho);           // error bound per unit change
    const float span = rho * lam;                   // Chebyshev interval [lam_lo span, span]
    const float half = 0.5f * (span - lam_lo * span), mid = 1.0f - 0.5f * (span + lam_lo * span);
    const float cden = al / den;
    const float eta = kInnerError * fmaxf(1.0f, 0.08f * amp);
    bool live = vin;       // the row takes part in this outer iteration
    bool hitmax = false, bad = false;
    float thr = 0.0f, prevr = 3.0e38f;
    int iters = 0;
    int stalls = 0;
    while (true) {
      // ---- X = Q + b1 S, split
      const int ex = scale_exponent(row_max(red_d), 13);
      const float sx = pow2f(ex);
      // tail (ring form): Xl, after the MMAs on Xm, which has its place until then
      const auto split_x = [&](auto tail) {
        constexpr bool kTail = decltype(tail)::value;
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
          const int c0 = cb + ch * CH;
          float qv[CH], bv[8];
          load_q(ch, qv);
          load_w(c0, bv);
          if (ch < NCT) tmem_wait_ld();
          reg_q(ch, qv);
          uint32_t hi[4], lo[4], lw[4];
#pragma unroll
          for (int j = 0; j < CH; j += 2) {
            float h0, l0, m0, h1, l1, m1;
            split_u(form_x(bv[j], S[ch * CH + j], qv[j]) * sx, h0, l0, m0);
            split_u(form_x(bv[j + 1], S[ch * CH + j + 1], qv[j + 1]) * sx, h1, l1, m1);
            hi[j / 2] = pack_f16x2(h0, h1);
            lo[j / 2] = pack_f16x2(l0, l1);
            lw[j / 2] = pack_f16x2(m0, m1);
          }
          const uint32_t off = sw128_chunk_off(kM, row, c0);
          if (!kTail) {
            *reinterpret_cast<uint4*>(sXh + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(sXm + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
          }
          if (kTail || !C::kRing) *reinterpret_cast<uint4*>(sXl + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        fence_async_smem();
        tc_fence_before();
      };
      split_x(std::false_type{});
      __syncthreads();
      if (tid == 0) issue_product(std::true_type{});
      bool mma_ok = wait_mma();
      if constexpr (C::kRing) {
        split_x(std::true_type{});
        if (tid == 0 && !pl_refill()) abort_s = 1;
        __syncthreads();
        if (tid == 0) issue_product(std::false_type{});
        mma_ok = wait_mma() && mma_ok;
      }
      if (tid == 0 && C::kRing && mma_ok) {
        // the next product's first blocks (its slots' MMAs have completed)
        while (pl_issued < pl_used + C::kSlots) pl_load();
      }
      // ---- residual r = a P~ X - S -> TMEM
      float rm = 0.0f, sm = 0.0f, cs = 0.0f;
      const float ky = tscale * pow2f(-ex);
      if (mma_ok) {
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
          const int c0 = cb + ch * CH;
          float a0[CH], a1[CH], qv[CH], bv[8], dv[8], dl[8];
          tmem_ld<CH>(t_row + c0, a0);
          tmem_ld<CH>(t_row + C::ROFF + c0, a1);
          load_q(ch, qv);
          load_w(c0, bv);
          lds_vec<8>(sDi + c0, dv);
          lds_vec<8>(sDi + NA + c0, dl);
          tmem_wait_ld();
          reg_q(ch, qv);
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const float s = S[ch * CH + j];
            const float x = form_x(bv[j], s, qv[j]);
            // where scattering prevails y - S is summed from the start (rounding y itself,
            // alike in all directions of an isotropic field, would be multiplied by
            // 1 / (1 - a b1)), then r = (y - S) - eps y
            const float base = al > 0.5f ? s : 0.0f;
            const float dy = fmaf(dl[j], x, fmaf(dv[j], x, fmaf(a1[j], ky, fmaf(a0[j], ky, -base))));
            const float y = dy + base;
            const float da = fmaf(-ev, y, dy);
            float r = da - (s - base);
            const float sh = base + da;
            if (kMode == kBuffers)
              reinterpret_cast<__half*>(sXl)[(c0 + j) * kM + row] = __float2half_rn(1.0f - bv[j]);
            // adjoint, no scattering: y = 0 now; its P z goes where the residual would
            a0[j] = r;
            if (kMode == kAdjoint && al == 0.0f) {
              S[ch * CH + j] = 0.0f;
              a0[j] = y;
              r = 0.0f;
            }
            rm = fmaxf(rm, fabsf(r));
            sm = fmaxf(sm, fabsf(sh));
            cs = fmaf(b1_of(bv[j]), r, cs);
          }
          tmem_st<CH>(t_row + C::ROFF + c0, a0);
        }
        tmem_wait_st();
      }
      red_d[grp][row] = rm;
      red_s[grp][row] = sm;
      red_c[grp][row] = cs;
      __syncthreads();
      if (abort_s) {
        aborted = true;
        break;
      }
      bool inner = false;
      bool fin = !live || (kMode == kAdjoint && al == 0.0f);  // S has taken its last r of this outer
      bool stalled = false, lost = false;  // no further outers; ... and the residual is above its noise floor
      float target = 0.0f, es = 0.0f, crow = 0.0f, xb = 0.0f;  // xb: bound of the operand's elements / 2
      rm = row_max(red_d);
      if (live) {
        ++iters;
        thr = kTolShare * tol * fmaxf(row_max(red_s), 1e-6f * s_glob * pow2f(up_s[row]));
        // the residual is noise below 2^-21 of the row's largest X (2^(14 - ex) bounds that);
        // above it one that is not halved says that the corrections do not do what they should
        const bool slow = rm > 0.5f * prevr, at_floor = rm <= pow2f(-7 - ex);
        stalls += slow ? 1 : 0;
        prevr = fminf(prevr, rm);
        stalled = slow && (at_floor || stalls >= kMaxStalls);
        lost = !(rm <= 3.0e38f) || (stalled && !at_floor);
        target = fmaxf(thr, amp * rm * kInnerDrop);
        // (a change far above the result has left its own rounding in S, however thin the voxel)
        const bool conv = fmaxf(amp, kMinAmp) * rm <= thr;
        inner = !conv && iters < max_iters && rm <= 3.0e38f;
        hitmax = !conv && !inner;
        lost = (lost && !conv) || ex < -114;  // (an infinite X: its residual is not a number)
        if (inner) {
          const float cs0 = row_sum(red_c);
          crow = cden * cs0;
          xb = rm + fminf(fabsf(crow), fabsf(cs0));  // (a max u <= den, so u |c| <= |sum b1 r|)
        }
      }
      // ---- inner iterations on the error equation
      int k = 0, kc = 0;  // iteration, and its place in the Chebyshev cycle
      float om = __fdividef(1.0f, fmaf(-half, cw_s[0], mid));
      while (true) {
        const float w = inner ? om : (fin ? 0.0f : 1.0f);
        const int er = scale_exponent(xb, 13);
        const float sc = inner ? pow2f(er) : 0.0f;
        if (__any_sync(0xffffffffu, w != 0.0f)) {
          const f32x2 nc2 = pk(-crow, -crow), neg1 = pk(-1.0f, -1.0f), nw2 = pk(-w, -w), sc2 = pk(sc, sc);
#pragma unroll
          for (int c2 = 0; c2 < NCH; c2 += 2) {
            const int c0 = cb + c2 * CH;
            float rv[2 * CH];
            tmem_ld<2 * CH>(t_row + C::ROFF + c0, rv);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              float bv[8];
              load_w(c0 + u * CH, bv, true);
              if (u == 0) tmem_wait_ld();
              uint32_t hi[4];
#pragma unroll
              for (int j = 0; j < CH; j += 2) {
                const f32x2 r2 = pk(rv[u * CH + j], rv[u * CH + j + 1]), nd = fma2(r2, neg1, nc2);
                float& s0 = S[(c2 + u) * CH + j];
                float& s1 = S[(c2 + u) * CH + j + 1];
                unpk(fma2(nw2, nd, pk(s0, s1)), s0, s1);
                float x0, x1;
                unpk(mul2(fma2(pk(bv[j], bv[j + 1]), nd, r2), sc2), x0, x1);  // b1 r - u c
                hi[j / 2] = pack_f16x2(x0, x1);
              }
              *reinterpret_cast<uint4*>(sXh + sw128_chunk_off(kM, row, c0 + u * CH)) =
                  make_uint4(hi[0], hi[1], hi[2], hi[3]);
            }
          }
        }
        if (inner) es += om * xb;
        if (!inner) fin = true;
        fence_async_smem();
        tc_fence_before();
        if (!__syncthreads_or(inner ? 1 : 0)) break;
        if (tid == 0) {
          tc_fence_after();
#pragma unroll
          for (int s = 0; s < C::KSTEPS; ++s) {
            const uint32_t ko = static_cast<uint32_t>((s & 3) * 32), kb = static_cast<uint32_t>(s >> 2);
            mma_f16(tmem, sw128_desc(aXh + kb * kM * 128 + ko), sw128_desc(aPh + kb * NA * 128 + ko), C::IDESC, s > 0);
          }
          mma_commit(&mbar);
        }
        mma_ok = wait_mma();
        float rmx = 0.0f, csx = 0.0f;
        if (mma_ok && __any_sync(0xffffffffu, inner)) {
          const float kd = tscale * pow2f(-er), wa = w * al;
          const float ec = ev * crow;
          const f32x2 nc2 = pk(-crow, -crow), neg1 = pk(-1.0f, -1.0f), nw2 = pk(-w, -w), wa2 = pk(wa, wa);
          const f32x2 kd2 = pk(kd, kd), ec2 = pk(ec, ec);
          f32x2 cr2 = pk(0.0f, 0.0f), cu2 = pk(0.0f, 0.0f);
#pragma unroll
          for (int ch = 0; ch < NCH; ++ch) {
            const int c0 = cb + ch * CH;
            float rv[CH], dd[CH], bv[8], di[8];
            tmem_ld<CH>(t_row + c0, dd);
            tmem_ld<CH>(t_row + C::ROFF + c0, rv);
            load_w(c0, bv, true);
            lds_vec<8>(sDi + 2 * NA + c0, di);
            tmem_wait_ld();
            // a row that has stopped has w = 0 and x = 0, so D = 0: its r stays
#pragma unroll
            for (int j = 0; j < CH; j += 2) {
              const f32x2 r2 = pk(rv[j], rv[j + 1]), u2 = pk(bv[j], bv[j + 1]);
              const f32x2 x = fma2(u2, fma2(r2, neg1, nc2), r2);
              const f32x2 y = fma2(pk(di[j], di[j + 1]), x, mul2(pk(dd[j], dd[j + 1]), kd2));  // P x
              const f32x2 rn = fma2(wa2, y, fma2(nw2, add2(r2, ec2), r2));
              unpk(rn, rv[j], rv[j + 1]);
              rmx = fmaxf(rmx, fmaxf(fabsf(rv[j]), fabsf(rv[j + 1])));
              cr2 = add2(cr2, rn);
              cu2 = fma2(u2, rn, cu2);
            }
            tmem_st<CH>(t_row + C::ROFF + c0, rv);
          }
          float cs0, cs1;
          unpk(fma2(cu2, neg1, cr2), cs0, cs1);
          csx = cs0 + cs1;  // sum b1 r
          tmem_wait_st();
        }
        // the next weight, off the path between the barrier and the next operand
        kc = kc + 1 < t.cycle ? kc + 1 : 0;
        om = __fdividef(1.0f, fmaf(-half, cw_s[kc], mid));
        red_d[grp][row] = rmx;
        red_c[grp][row] = csx;
        __syncthreads();
        if (abort_s) {
          aborted = true;
          break;
        }
        ++k;
        if (inner) {
          rm = row_max(red_d);
          ++iters;
          const bool conv = amp * rm <= target;
          if (conv || iters >= max_iters || k >= t.max_inner || !(rm <= 3.0e38f)) {
            inner = false;
            if (!conv && iters >= max_iters) hitmax = true;
            crow = 0.0f;
          } else {
            const float cs0 = row_sum(red_c);
            crow = cden * cs0;
            xb = rm + fminf(fabsf(crow), fabsf(cs0));
          }
        }
      }
      if (aborted) break;
      // another accurate residual where the inner products' error may exceed the tolerance
      bool more = live && !hitmax && !stalled && iters < max_iters &&
                  (amp * rm > thr || eta * es > thr);
      if (live && (lost || (amp * rm > thr && iters >= max_iters))) bad = true;
      live = more;
      // (the barrier also separates the reads of red_d above from the writes below)
      if (!__syncthreads_or(more ? 1 : 0)) break;
      xmax = 0.0f;
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        float qv[CH], bv[8];
        load_q(ch, qv);
        load_w(cb + ch * CH, bv);
        if (ch < NCT) tmem_wait_ld();
        reg_q(ch, qv);
#pragma unroll
        for (int j = 0; j < CH; ++j) xmax = fmaxf(xmax, fabsf(form_x(bv[j], S[ch * CH + j], qv[j])));
      }
      red_d[grp][row] = xmax;
      __syncthreads();
    }
    if (aborted) break;
    if (bad && grp == 0) atomicAdd(rs.nonconv, 1);
    const float down = pow2f(-up_s[row]);

    if constexpr (kMode == kAdjoint) {
      // ---- Qbar, warm start of the next reverse step, cleared adjoint level, gradient sums
      float ga = 0.0f, gm = 0.0f;
      const float mu_v = vin ? io.mut[v] : 0.0f;
      const float inv_al = al > 0.0f ? 1.0f / al : 0.0f;
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        const int c0 = cb + ch * CH;
        float pz[CH];
        if (__any_sync(0xffffffffu, al == 0.0f)) {
          tmem_ld<CH>(t_row + C::ROFF + c0, pz);
          tmem_wait_ld();
        }
        if (vin) {
          float ib[CH], yo[CH], in[CH], sn[CH];
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const size_t o = static_cast<size_t>(c0 + j) * plane + v;
            ib[j] = io.ib[o];
            yo[j] = io.y2 ? io.y[o] : 0.0f;
            in[j] = __ldg(io.i_n + o);
            sn[j] = __ldg(io.s_n + o);
          }
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const size_t o = static_cast<size_t>(c0 + j) * plane + v;
            const float y = S[ch * CH + j] * down, qbar = ib[j] + y;
            io.qb[o] = qbar;
            if (io.y2) io.y2[o] = yo[j];
            io.y[o] = y;
            io.ib[o] = 0.0f;
            io.sb[o] = 0.0f;
            smax_loc = fmaxf(smax_loc, fabsf(y));
            ga = fmaf(in[j], al > 0.0f ? y * inv_al : pz[j] * down, ga);  // I (P z)
            const float ds = cls_ds[sCls[c0 + j]], x = mu_v * ds;
            gm = fmaf(ds * sn[j] * qbar, ray_b0_over_x(x, expf(-x)), gm);
          }
        }
      }
      red_d[grp][row] = ga;
      red_s[grp][row] = gm;
      __syncthreads();
      if (grp == 0 && vin) {
        double sa = 0.0, sm = 0.0;
#pragma unroll
        for (int gi = 0; gi < kGroups; ++gi) {
          sa += static_cast<double>(red_d[gi][row]);
          sm += static_cast<double>(red_s[gi][row]);
        }
        io.gA[v] += sa;
        io.gmut[v] += sm;
      }
    } else {
    // ---- write-out: I = Q + b1 S and S of every voxel
    const float nv_v = (kMode == kStep && vin) ? io.nidx[v] : 0.0f;
    const float mu_v = (kMode == kStep && vin) ? io.mut[v] : 0.0f;
    float esum_row = 0.0f;
    if (C::KB * 64 == NA && tma_out) {
      // staged: I and then S of the tile go to the X operand area as 8-direction boxes of
      // the brick ([direction][row], conflict-free) and one thread stores them with TMA
      float* stg = reinterpret_cast<float*>(sXh);
      const int bx = tile % bxn, t2 = tile / bxn;
      const int ox = bx << 3, oy = (t2 % byn) << 2, oz = (t2 / byn) << 2;
      const int pbase = ring_slot(n) * NA;
#pragma unroll
      for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
          const int c0 = cb + ch * CH;
          float qv[CH], bv[8];
          if (pass == 0) {
            load_q(ch, qv);
            load_w(c0, bv);
            if (ch < NCT) tmem_wait_ld();
            reg_q(ch, qv);
          }
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const int col = c0 + j;
            const float s = S[ch * CH + j];
            float val = s * down;
            if (pass == 0) {
              smax_loc = fmaxf(smax_loc, vin ? fabsf(val) : 0.0f);
              val = form_x(bv[j], s, qv[j]) * down;
              if (vin) esum_row += val;
            }
            stg[(col >> 3) * 1024 + (col & 7) * 128 + row] = val;
          }
        }
        fence_async_smem();
        __syncthreads();
        if (tid == 0) {
          const uint64_t map = reinterpret_cast<uint64_t>(pass == 0 ? &tmOutI : &tmOutS);
#pragma unroll 1
          for (int bb = 0; bb < NA / 8; ++bb)
            asm volatile(
                "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(map),
                "r"(ox), "r"(oy), "r"(oz), "r"(pbase + bb * 8), "r"(smem_u32(stg + bb * 1024))
                : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          if (pass == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        if (pass == 0) __syncthreads();
      }
    } else {
      float* pI = io.I + cur_base + static_cast<size_t>(cb) * plane + v;
      float* pS = io.S + cur_base + static_cast<size_t>(cb) * plane + v;
#pragma unroll
      for (int ch = 0; ch < NCH; ++ch) {
        float qv[CH], bv[8];
        load_q(ch, qv);
        load_w(cb + ch * CH, bv);
        if (ch < NCT) tmem_wait_ld();
        reg_q(ch, qv);
        if (vin) {
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const float s = S[ch * CH + j] * down;
            const float Iv = form_x(bv[j], S[ch * CH + j], qv[j]) * down;
            pI[static_cast<size_t>(ch * CH + j) * plane] = Iv;
            pS[static_cast<size_t>(ch * CH + j) * plane] = s;
            esum_row += Iv;
            smax_loc = fmaxf(smax_loc, fabsf(s));
          }
        }
      }
    }
    if (kMode == kStep) {
      if (vin) esum += static_cast<double>(esum_row) * static_cast<double>(nv_v);
      float ab = vin ? esum_row * (ev * mu_v) : 0.0f;
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) ab += __shfl_xor_sync(0xffffffffu, ab, o);
      if (lane == 0) atomicAdd(&asum_sh, static_cast<double>(ab));
    }
    }
    // iteration statistics of this tile (group-0 threads hold one row each)
    if (warp < 4) {
      int im = vin ? iters : 0;
      unsigned long long is = static_cast<unsigned long long>(im);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        im = max(im, __shfl_xor_sync(0xffffffffu, im, o));
        is += __shfl_xor_sync(0xffffffffu, is, o);
      }
      if (lane == 0) {
        if (rs.iters_max) atomicMax(rs.iters_max + n, im);
        if (rs.iters_sum) atomicAdd(rs.iters_sum + n, is);
      }
    }
    __syncthreads();
  }

  if (aborted && tid == 0) atomicExch(rs.error, 7);
  if (tid == 0) {
    if (tma_out) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    // the Pl blocks loaded ahead have landed before the shared memory is given back
    if constexpr (C::kRing) {
      for (uint32_t q = pl_used; q < pl_issued; ++q) mbar_wait_bounded(&pl_full[q % C::kSlots], (q / C::kSlots) & 1u);
    }
  }
  // energy and max |S| of this CTA's voxels
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    esum += __shfl_xor_sync(0xffffffffu, esum, o);
    smax_loc = fmaxf(smax_loc, __shfl_xor_sync(0xffffffffu, smax_loc, o));
  }
  if (lane == 0) {
    esum_s[warp] = esum;
    smax_s[warp] = smax_loc;
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0) {
    double e = 0.0;
    float sm = 0.0f;
    for (int w = 0; w < C::kThreads / 32; ++w) {
      e += esum_s[w];
      sm = fmaxf(sm, smax_s[w]);
    }
    if (kMode == kStep) {
      atomicAdd(rs.energy + n, e * static_cast<double>(g.e_scale));
      atomicAdd(rs.absorbed + n, asum_sh * g.a_scale);
    }
    if (kMode != kBuffers) atomicMax(rs.smax + (n & 1), __float_as_uint(sm));
  }
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TCOLS);
  }
}

PerDevice g_split;

template <int NA, int kMode, int kPer>
cudaError_t configure_split() {
  cudaError_t e = cudaFuncSetAttribute(scatter_split_kernel<NA, false, kMode, kPer>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, Sp<NA>::SMEM);
  if (e != cudaSuccess || kMode == kBuffers) return e;
  return cudaFuncSetAttribute(scatter_split_kernel<NA, kMode != kBuffers, kMode, kPer>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, Sp<NA>::SMEM);
}

template <int kMode>
cudaError_t configure_mode() {
  cudaError_t e = configure_split<48, kMode, 1>();
  if (e == cudaSuccess) e = configure_split<48, kMode, 2>();
  if (e == cudaSuccess) e = configure_split<192, kMode, 1>();
  return e;
}

// SM count of the current device, its kernels configured; 0 if they cannot be.
int split_sms() {
  return configured_sms(g_split, [] {
    cudaError_t e = configure_mode<kStep>();
    if (e == cudaSuccess) e = configure_mode<kBuffers>();
    if (e == cudaSuccess) e = configure_mode<kAdjoint>();
    return e;
  });
}

template <int kMode>
cudaError_t launch_split(const GridParams& g, const SplitTables& sp, const BfTables& t, const SplitIo& io, float tol,
                         int max_iters, const CUtensorMap& mI, const CUtensorMap& mS, int tma_out, const RunState& rs,
                         cudaStream_t st) {
  const int sms = split_sms();
  if (sms == 0) return cudaErrorInvalidValue;
  const int ntiles = kMode == kBuffers ? (g.nv + kM - 1) / kM : brick_tiles(g.nx, g.ny, g.nz);
  constexpr bool kU = kMode != kBuffers;
  const bool uni = kU && g.mut_u >= 0.0f;
  if (g.na == 48) {
    // two CTAs per SM from 2.5 tiles per SM on (as scatter_tc.cu; varying mu_t): 0.157 against
    // 0.170 ms at 40^3 (3.3 tiles per SM), 0.325 against 0.367 at 56^3, 0.809 against 0.945 at
    // 80^3; one CTA otherwise: 0.093 against 0.101 ms at 32^3 (1.7 tiles per SM), 0.038 against
    // 0.042 at 16^3 (uniform mu_t)
    const bool two = 2 * ntiles > 5 * sms;
    const int cap = two ? 2 * sms : sms, grid = ntiles < cap ? ntiles : cap;
    auto k = two ? (uni ? scatter_split_kernel<48, kU, kMode, 2> : scatter_split_kernel<48, false, kMode, 2>)
                 : (uni ? scatter_split_kernel<48, kU, kMode, 1> : scatter_split_kernel<48, false, kMode, 1>);
    k<<<grid, Sp<48>::kThreads, Sp<48>::SMEM, st>>>(g, sp, t.cls, t.cls_ds, t.ncls, t.nch, io, tol, max_iters, mI, mS,
                                                    tma_out, rs);
  } else if (g.na == 192) {
    const int grid = ntiles < sms ? ntiles : sms;
    auto k = uni ? scatter_split_kernel<192, kU, kMode, 1> : scatter_split_kernel<192, false, kMode, 1>;
    k<<<grid, Sp<192>::kThreads, Sp<192>::SMEM, st>>>(g, sp, t.cls, t.cls_ds, t.ncls, t.nch, io, tol, max_iters, mI,
                                                      mS, tma_out, rs);
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

uint16_t half_bits(double x) {  // nearest FP16 number
  const __half h = __double2half(x);
  uint16_t u;
  std::memcpy(&u, &h, 2);
  return u;
}

double half_value(uint16_t u) {
  __half h;
  std::memcpy(&h, &u, 2);
  return static_cast<double>(__half2float(h));
}

}  // namespace

bool scatter_split_supported(int na, int ncls) {
  if ((na != 48 && na != 192) || ncls > kMaxClasses) return false;
  return split_sms() > 0;
}

// Off-diagonal part of the FP64 phase matrix P split as (Ph + Pl + Pm) unit, in the kernel's
// operand layout: Ph [K block][na rows][128 B]; Pm and then Pl likewise at 48 directions, as
// six blocks each (K block, half of the rows) of 96 rows at 192; diag: the FP32 pair that
// makes each row of P with it sum to one, and the diagonal that does so with Ph alone.
SplitImage scatter_split_image(const std::vector<double>& P, int na, double g_aniso) {
  SplitImage im;
  const int kb = (na + 63) / 64;
  double pmax = 0.0, rmax = 0.0;
  for (int i = 0; i < na; ++i) {
    double s = 0.0;
    for (int j = 0; j < na; ++j)
      if (j != i) {
        const double p = std::fabs(P[static_cast<size_t>(i) * na + j]);
        pmax = std::max(pmax, p);
        s += p;
      }
    rmax = std::max(rmax, s);
  }
  // Ph of at most 11 bits; |sum Xh Ph| <= 2^10 sum |Ph| <= 2^10 (2^t rmax + na / 2) < 2^24, with room for
  // the unit's rounding
  int t = 0;
  while (t < 20 && std::ldexp(pmax, t + 1) <= 2046.0 && std::ldexp(rmax, t + 1) + na / 2 <= 16128.0) ++t;
  // one unit of Ph: 2^-t made so that the largest entry is a whole number of units (an
  // isotropic P is then split exactly; its equal entries would else all err to one side)
  const double whole = std::floor(std::ldexp(pmax, t));
  // (held sixteenfold: the terms below then stay clear of FP16's subnormals)
  im.unit = static_cast<float>(whole >= 1.0 ? pmax / whole : std::ldexp(1.0, -t)) / 16.0f;
  const double unit = im.unit;
  const size_t half = static_cast<size_t>(kb) * na * 64;
  im.ph.assign(half, 0);
  im.pl.assign(2 * half, 0);
  im.diag.assign(static_cast<size_t>(3) * na, 0.0f);
  const int blk = 96;
  for (int i = 0; i < na; ++i) {
    double sh = 0.0, sum = 0.0;
    for (int j = 0; j < na; ++j) {
      if (j == i) continue;
      const double u = P[static_cast<size_t>(i) * na + j] / unit;
      const double h = 16.0 * std::nearbyint(u / 16.0);
      const uint16_t lb = half_bits(u - h);
      const uint16_t mb = half_bits(u - h - half_value(lb));
      sh += h;
      sum += P[static_cast<size_t>(i) * na + j];
      const int k = j >> 6, ch = (j & 63) >> 3;
      const size_t in_row = static_cast<size_t>(((ch ^ (i & 7)) << 3) + (j & 7));
      im.ph[(static_cast<size_t>(k) * na + i) * 64 + in_row] = half_bits(h);
      // 96 is a multiple of 8, so a block's rows keep the swizzle phase i & 7
      const size_t prow = na >= 192 ? static_cast<size_t>(k * (na / blk) + i / blk) * blk + i % blk
                                    : static_cast<size_t>(k) * na + i;
      im.pl[prow * 64 + in_row] = mb;
      im.pl[half + prow * 64 + in_row] = lb;
    }
    const double d = 1.0 - sum;
    im.diag[i] = static_cast<float>(d);
    im.diag[na + i] = static_cast<float>(d - static_cast<double>(im.diag[i]));
    im.diag[2 * na + i] = static_cast<float>(1.0 - sh * unit);
  }
  // Chebyshev interval of the rebalanced iteration, in units of rho: the eigenvalues of P
  // but the constant vector's lie in [0, |g| + 0.013] for g >= 0 (checked for g from 0 to
  // 0.99 at 12, 48 and 192 directions) and in +- that for g < 0
  const double a = std::fabs(g_aniso);
  im.lam = static_cast<float>(std::min(a + 0.015, 0.5 * (a + 1.0)));
  im.lo = g_aniso >= 0.0 ? 0.0f : -1.0f;
  // cycle length: long enough to damp by ~50 (sigma^m, sigma of kappa = 1 / (1 - lam))
  const double kap = std::sqrt((1.0 - im.lo * im.lam) / (1.0 - im.lam));
  int m = 8;
  while (m < kSplitCycle && std::pow((kap - 1.0) / (kap + 1.0), m) > 0.02) m *= 2;
  im.cycle = m;
  im.max_inner = 8 * m;
  // roots in the order that keeps every partial product bounded (Lebedev and Finogenov 1971)
  std::vector<int> th(1, 1);
  while (static_cast<int>(th.size()) < m) {
    const int n2 = 2 * static_cast<int>(th.size());
    std::vector<int> nx;
    for (int a2 : th) {
      nx.push_back(a2);
      nx.push_back(2 * n2 - a2);
    }
    th = nx;
  }
  im.cw.assign(kSplitCycle, 0.0f);
  for (int k = 0; k < m; ++k)  // damping of the large eigenvalues of 1 - T first
    im.cw[k] = static_cast<float>(std::cos((2 * m - th[k]) * 3.14159265358979323846 / (2.0 * m)));
  return im;
}

cudaError_t launch_scatter_split(const GridParams& g, const SplitTables& sp, const BfTables& t, const float* Q,
                                 const float* mut, const float* eps, const float* nidx, float* Iring, float* Sring,
                                 float tol, int max_iters, RunState rs, cudaStream_t st) {
  CUtensorMap mI, mS;
  std::memset(&mI, 0, sizeof(mI));
  std::memset(&mS, 0, sizeof(mS));
  const int tma_out = (t.out_maps && g.na % 64 == 0) ? 1 : 0;
  if (tma_out) {
    std::memcpy(&mI, t.out_maps, sizeof(CUtensorMap));
    std::memcpy(&mS, static_cast<const unsigned char*>(t.out_maps) + 128, sizeof(CUtensorMap));
  }
  SplitIo io{};
  io.q = Q;
  io.s1 = Sring;
  io.eps = eps;
  io.mut = mut;
  io.nidx = nidx;
  io.I = Iring;
  io.S = Sring;
  return launch_split<kStep>(g, sp, t, io, tol, max_iters, mI, mS, tma_out, rs, st);
}

cudaError_t launch_adj_scatter_split(const GridParams& g, const SplitTables& sp, const BfTables& t, const SplitIo& io,
                                     float tol, int max_iters, unsigned* ymax_cur, int* nonconv,
                                     unsigned long long* iters_sum, int* error, cudaStream_t st) {
  CUtensorMap m;
  std::memset(&m, 0, sizeof(m));
  RunState rs{};
  rs.smax = ymax_cur;
  rs.nonconv = nonconv;
  rs.iters_sum = iters_sum;
  rs.error = error;
  return launch_split<kAdjoint>(g, sp, t, io, tol, max_iters, m, m, 0, rs, st);
}

cudaError_t launch_scatter_split_buffers(int na, int nvox, const SplitTables& sp, const SplitIo& io, float tol,
                                         int max_iters, int* iters_max, int* nonconv, int* error, cudaStream_t st) {
  CUtensorMap m;
  std::memset(&m, 0, sizeof(m));
  GridParams g{};
  g.na = na;
  g.nv = nvox;
  g.mut_u = -1.0f;
  RunState rs{};
  rs.iters_max = iters_max;
  rs.nonconv = nonconv;
  rs.error = error;
  return launch_split<kBuffers>(g, sp, BfTables{}, io, tol, max_iters, m, m, 0, rs, st);
}

}  // namespace trinity
