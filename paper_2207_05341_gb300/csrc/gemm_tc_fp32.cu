// FP32 complex products on the tensor cores (tcgen05) with no loss against FP32 arithmetic:
//   X = T T, Y = G T        (Chol_H, Sec. 3.2 eq. unified_DP and its backward)
//   X = T^dag T, Z = T G    (Chol_Delta, Sec. 2.2.1 eq. T_matrix)
// for d >= 128, as C = A B from the planes of A and of B^dag (row-major, K-major operands).
//
// Each FP32 entry x (scaled by the power of two that brings the matrix's largest entry into [1, 2)) is the
// exact sum of three BF16 terms x = h + m + l (8 + 8 + 8 significant bits), so the operands carry all 24 bits
// of FP32, whatever the spread of the entries.  The product keeps the six term pairs down to 2^-18,
//   l h + h l + m m + m h + h m + h h,
// and drops m l, l m and l l: |m| reaches 2^-8 and |l| 2^-17 of |x| (both just above a power of two), so at most
// 2^-24 of |a b|, half an FP32 ulp, and 2^-27.5 in the mean square over all mantissas.  An infinite entry gives NaN
// (x - h), where FP32 arithmetic would also give infinities.
//
// Accumulation.  The tensor core truncates its FP32 sums: over a K = 2d chain that bias reaches 1.3e-5 at
// d = 1024 (the mixed path).  Here every block of 32 K elements is a chain of its own, issued from the
// smallest term pair to h h, so that only its two h h steps truncate at full size; the block's sum is then
// added to an FP32 register accumulator, round to nearest, as an FP32 FMA chain would be.  Measured against
// 64 bits: X at N = 7..10 is off by 0.9..1.6e-7 of its norm off the diagonal and 0.5..1.1e-7 on it (CUDA-core
// products: 2.9..8.1e-7 and 2.4..5.9e-7), with no bias above 5e-8 on either.
//
// A complex product is one real product with the K axis doubled, A' = [A_re | A_im], and the N axis doubled:
// with the planes P_re, P_im, P_nim = -P_im of B^dag, Re C uses [P_re | P_im] and Im C uses [P_nim | P_re].
//
// Kernel: one CTA, or below d = 2048 a cluster of ks CTAs that share the K blocks, per 128 x 128 complex tile
// (N = 256 real columns), 10 warps.  Warp 8 streams K blocks with TMA into a ring (A: 3 terms x 128 rows, B:
// 3 terms x 256 rows of 64 bytes, 64-byte swizzle: 47 bytes per clock; a 128 x 64 tile needs 62, at the limit of
// what an SM takes from L2, and was twice as slow per product), warp 9 issues
// the block's 12 MMAs into one of two TMEM accumulators, and warps 0-7 drain the other one into registers
// (TMEM to FP32 adds), so the promotion runs beside the MMAs: 12 MMAs of N = 256 take about 1540 cycles, the
// drain of 128 x 256 sums about 500.  Bound by the tensor pipe: at N = 11 X = T T takes 129 us and Y = G T 253 us
// (206 and 412 GFLOP of BF16 products, 1.6 PFLOP/s; 914 and 1778 us on the CUDA cores), at N = 9 27 and 26 us
// (231 and 232), there mostly fixed costs.  Every mbarrier wait is bounded; on timeout the kernel raises *err,
// drains its copies, frees TMEM and returns.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>

#include "impl.h"
#include "tc.cuh"

namespace qst {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 32;                       // K elements per block: rows of 64 bytes
constexpr int kRow = kBK * 2;
constexpr int kEpiWarps = 8;
constexpr int kThreads32 = (kEpiWarps + 2) * 32;

constexpr int kBN = 128;                      // complex columns of a tile
constexpr int kA = kBM * kRow;                // bytes of one term of A in a stage
constexpr int kB = kBN * kRow;                // bytes of one term of one half of B
constexpr int kStage = 3 * kA + 6 * kB;
constexpr int kStages = 3;
constexpr int kSmem = kStages * kStage + 1024 + 256;
constexpr int kTmem = 4 * kBN;                // two accumulators of 256 columns
constexpr int kMaxSplit = 4;                  // CTAs that share a tile, at most
static_assert(kBM * kBN * 8 <= kStages * kStage, "a partial tile fits in the ring");

struct Maps32 {
  CUtensorMap a;  // 6 planes: re h, m, l; im h, m, l (box 32 x 128 x 3)
  CUtensorMap b;  // 9 planes: re, im, -im, each h, m, l (box 32 x 128 x 1)
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// K-major shared-memory descriptor, 64-byte swizzled rows (8-row atoms of 512 bytes)
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)((8 * kRow) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// kind::f16, FP32 accumulators, BF16 operands, both K-major, M = 128, N = 256
constexpr uint32_t kIdesc32 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * kBN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);

// krange: 0 all of K; 1 only k >= the tile's first row (A and B^dag upper triangular, tiles I >= J);
// 2 only k <= the tile's last row (A lower triangular).  What is left out is multiplied by zeros.
// ks: CTAs of a cluster that share a tile (rank r takes the r-th part of the K blocks); their partial tiles meet in
// distributed shared memory, rank r summing its rows over the ranks in order.
// tab: a batched launch (grid z = tomography); row z holds the tensor maps' device copy, C, sA, sB, err, clear.
__global__ void __launch_bounds__(kThreads32, 1)
    k_tc_cgemm32(const __grid_constant__ Maps32 maps, float2* __restrict__ C, int d, int lower, int krange, int ks,
                 const double* sA, const double* sB, unsigned int* err, unsigned int* clear, int no_loads,
                 const void* const* tab) {
  const Maps32* mp = &maps;
  rebind(tab, mp, C, sA, sB, err, clear);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = smem_u32(bars + kStages);
  const uint32_t accf0 = smem_u32(bars + 2 * kStages);      // accumulator b complete
  const uint32_t acce0 = smem_u32(bars + 2 * kStages + 2);  // accumulator b drained
  const uint32_t done = smem_u32(bars + 2 * kStages + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5);
  __shared__ int s_fail;  // a drain warp gave up: this CTA's partial tile is not whole

  int I, J;  // the tile: rows 128 I .., columns 128 J ..
  const int rank = (int)blockIdx.x % ks;
  if (lower) {
    tri_decode(blockIdx.x / ks, I, J);
  } else {
    I = blockIdx.y;
    J = (int)blockIdx.x / ks;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // barriers, TMEM and descriptors before the wait for the kernel that makes the planes
  if (threadIdx.x == 0) {
    if (!tab) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mp->a)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mp->b)) : "memory");
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf0 + 8 * b, 1);
      mbar_init(acce0 + 8 * b, kEpiWarps);
    }
    mbar_init(done, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  grid_dep_wait();
  after_wait(mp, C, sA, sB, err, clear);
  if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0u;
  const int kbeg = krange == 1 ? I * kBM : 0, kend = krange == 2 ? (I + 1) * kBM : d;
  const int half = (kend - kbeg) / kBK;                       // K blocks of the real part, and of the imaginary part
  const int kb0 = 2 * half * rank / ks, nkb = 2 * half * (rank + 1) / ks - kb0;  // this CTA's

  if (warp == kEpiWarps) {
    if (lane == 0) {  // ---------------- TMA producer
      if (tab) {      // the maps are this tomography's copies in global memory
        tensormap_acquire(&mp->a);
        tensormap_acquire(&mp->b);
      }
      int issued = 0;
      for (int kb = 0; kb < (no_loads ? 0 : nkb); ++kb) {
        const int s = kb % kStages, it = kb / kStages;
        if (kb >= kStages && !mbar_wait(empty0 + 8 * s, (uint32_t)((it - 1) & 1))) {
          atomicOr(err, 1u);
          break;
        }
        const uint32_t fb = full0 + 8 * s;
        mbar_expect_tx(fb, kStage);
        const int part = kb0 + kb < half ? 0 : 1;
        const int col = kbeg + (kb0 + kb - part * half) * kBK;
        const uint32_t base = smem_u32(smem + s * kStage), bb = base + 3 * kA;
        tma_load_3d(base, &mp->a, col, I * kBM, 3 * part, fb);
        const int z1 = part == 0 ? 0 : 3, z2 = part == 0 ? 6 : 0;  // Re: re | im; Im: -im | re
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          tma_load_3d(bb + (2 * t) * kB, &mp->b, col, J * kBN, z1 + t, fb);
          tma_load_3d(bb + (2 * t + 1) * kB, &mp->b, col, J * kBN, z2 + t, fb);
        }
        ++issued;
      }
      // every stage issued must have landed before the CTA may exit
      for (int kb = (issued > kStages ? issued - kStages : 0); kb < issued; ++kb) {
        if (!mbar_wait(full0 + 8 * (kb % kStages), (uint32_t)((kb / kStages) & 1))) {
          atomicOr(err, 1u);
          break;
        }
      }
    }
    __syncwarp();
  } else if (warp == kEpiWarps + 1) {
    if (lane == 0) {  // ---------------- MMA issuer
      bool ok = true;
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % kStages, b = kb & 1;
        if (!mbar_wait(full0 + 8 * s, (uint32_t)((kb / kStages) & 1))) { ok = false; break; }
        if (kb >= 2 && !mbar_wait(acce0 + 8 * b, (uint32_t)(((kb >> 1) - 1) & 1))) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t base = smem_u32(smem + s * kStage), bb = base + 3 * kA;
        const uint32_t acc = tmem + (uint32_t)(b * 2 * kBN);
        constexpr int ta[6] = {2, 0, 1, 1, 0, 0}, tb[6] = {0, 2, 1, 0, 1, 0};  // lh hl mm mh hm hh
#pragma unroll
        for (int p = 0; p < 6; ++p) {
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            mma_f16(acc, desc64(base + ta[p] * kA + kk * 32), desc64(bb + 2 * tb[p] * kB + kk * 32),
                    kIdesc32, p > 0 || kk > 0 ? 1u : 0u);
        }
        mma_commit(empty0 + 8 * s);
        mma_commit(accf0 + 8 * b);
      }
      if (!ok) atomicOr(err, 2u);
      mma_commit(done);  // arrives once all MMAs issued so far have completed
    }
    __syncwarp();
  } else {
    // ---------------- promotion: warp w drains TMEM lanes 32 (w % 4) .. and half w / 4 of the columns
    constexpr int CH = kBN / 2;  // complex columns of this warp
    const int q = warp & 3, hf = warp >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hf * CH);
    float re[CH], im[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) re[c] = im[c] = 0.f;
    bool ok = true;
    for (int kb = 0; kb < nkb; ++kb) {
      const int b = kb & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(accf0 + 8 * b, (uint32_t)((kb >> 1) & 1)));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t src = lane_base + (uint32_t)(b * 2 * kBN);
#pragma unroll
      for (int c = 0; c < CH; c += 16) {
        uint32_t r[16], i[16];
        tmem_ld16(src + (uint32_t)c, r);
        tmem_ld16(src + (uint32_t)(kBN + c), i);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          re[c + u] += __uint_as_float(r[u]);
          im[c + u] += __uint_as_float(i[u]);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acce0 + 8 * b);
    }
    if (ok && ks > 1) {  // the partial tile to shared memory (every operand has been used), 16-byte chunks swizzled
      const int row = q * 32 + lane;
      float4* part = reinterpret_cast<float4*>(smem) + row * (kBN / 2);
#pragma unroll
      for (int c = 0; c < CH; c += 2)
        part[(hf * (CH / 2) + c / 2) ^ (row & (kBN / 2 - 1))] = make_float4(re[c], im[c], re[c + 1], im[c + 1]);
    } else if (ok) {
      // C = acc / (sA sB), both powers of two; the smaller factor first (no overflow on the way)
      const float ua = pow2f(-exponent_of(*sA)), ub = pow2f(-exponent_of(*sB));
      const float u1 = fminf(ua, ub), u2 = fmaxf(ua, ub);
      float2* out = C + (long long)(I * kBM + q * 32 + lane) * d + (long long)J * kBN + hf * CH;
#pragma unroll
      for (int c = 0; c < CH; c += 2)
        *reinterpret_cast<float4*>(out + c) = make_float4(re[c] * u1 * u2, im[c] * u1 * u2, re[c + 1] * u1 * u2,
                                                          im[c + 1] * u1 * u2);
    } else if (lane == 0) {
      s_fail = 1;
      atomicOr(err, 1u);
    }
  }
  if (ks > 1) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __syncwarp();
    cl.sync();
    const float ua = pow2f(-exponent_of(*sA)), ub = pow2f(-exponent_of(*sB));
    const float u1 = fminf(ua, ub), u2 = fmaxf(ua, ub);
    const int rows = kBM / ks;
    int fail[kMaxSplit];  // a rank without its partial tile: no rank stores (the flags are read along with the sums)
#pragma unroll
    for (int r = 0; r < kMaxSplit; ++r) fail[r] = r < ks ? *cl.map_shared_rank(&s_fail, r) : 0;
    constexpr int kChunks = kBN / 2, kFly = 4;  // a thread's chunks in flight together
    for (int e0 = threadIdx.x; e0 < rows * kChunks; e0 += kFly * kThreads32) {
      float4 v[kFly];
      for (int r = 0; r < ks; ++r) {
        float4 w[kFly];
#pragma unroll
        for (int u = 0; u < kFly; ++u) {
          const int e = e0 + u * kThreads32;
          if (e < rows * kChunks) {
            const int row = rank * rows + e / kChunks, ch = e % kChunks;
            w[u] = *cl.map_shared_rank(reinterpret_cast<float4*>(smem) + row * kChunks + (ch ^ (row & (kChunks - 1))), r);
          }
        }
#pragma unroll
        for (int u = 0; u < kFly; ++u) {
          if (r == 0) { v[u] = w[u]; continue; }
          v[u].x += w[u].x; v[u].y += w[u].y; v[u].z += w[u].z; v[u].w += w[u].w;
        }
      }
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const int e = e0 + u * kThreads32;
        if (e >= rows * kChunks || (fail[0] | fail[1] | fail[2] | fail[3])) continue;
        const int row = rank * rows + e / kChunks, ch = e % kChunks;
        *reinterpret_cast<float4*>(C + (long long)(I * kBM + row) * d + (long long)J * kBN + 2 * ch) =
            make_float4(v[u].x * u1 * u2, v[u].y * u1 * u2, v[u].z * u1 * u2, v[u].w * u1 * u2);
      }
    }
    cl.sync();  // no CTA leaves while its part may still be read
  }
  if (warp == 0) mbar_wait(done, 0u);  // no MMA in flight when TMEM is freed
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem) : "memory");
  }
}

// x = h + m + l, each BF16 (exact for 24 significant bits away from the subnormal range)
struct Terms {
  __nv_bfloat16 v[3];
};
__device__ __forceinline__ Terms split3(float x) {
  Terms t;
  t.v[0] = __float2bfloat16_rn(x);
  const float r = x - __bfloat162float(t.v[0]);
  t.v[1] = __float2bfloat16_rn(r);
  t.v[2] = __float2bfloat16_rn(r - __bfloat162float(t.v[1]));
  return t;
}
__device__ __forceinline__ __nv_bfloat16 neg(__nv_bfloat16 x) { return __hneg(x); }

union Pack8 {
  uint4 v;
  __nv_bfloat16 h[8];
};

// Planes of a complex matrix, 8 consecutive entries per thread: re, im (and, with nine, -im), each h, m, l.
// *s_slot: the scale, 2^split_exponent(amax), written here; with keep, the scale already there.
// X (may be NULL; A is then G = dL/dX of Chol_H): X's lower 128 x 128 tiles.  L does not change with the scale
// of T, so Tr(G X) = 0; rounding of G's identity component (one scalar of about 2^-25 of sum f / Tr X) breaks
// that, and its product with T is most of the gradient's error (2.4e-6 of its norm at N = 9, 3.5e-7 without).
// The last block leaves scal[kGauge] = -Tr(G X) / Tr X, the multiple of T that k_symmetrize adds to Y; 0 when
// likelihood terms were clamped since the last time (flags[0] against flags[4]): L then does change with scale.
__global__ void __launch_bounds__(256) k_split3(const float2* __restrict__ A, __nv_bfloat16* __restrict__ P,
                                                 long long nn, int nine, int keep, const unsigned int* amax,
                                                 double* s_slot, const float2* __restrict__ X, int logd, double* scal,
                                                 double* partials, unsigned int* counter, unsigned int* flags,
                                                 const void* const* tab) {
  rebind(tab, A, P, amax, s_slot, X, scal, partials, counter, flags);
  grid_dep_wait();
  after_wait(A, P, amax, s_slot, X, scal, partials, counter, flags);
  asm volatile("griddepcontrol.launch_dependents;");  // the product's prologue may start
  const int se = keep ? exponent_of(*s_slot) : split_exponent(amax);
  const float sc = pow2f(se);
  if (!keep && blockIdx.x == 0 && threadIdx.x == 0) *s_slot = pow2d(se);
  const long long n8 = nn / 8;
  PairSum dsum;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n8; q += (long long)gridDim.x * blockDim.x) {
    const float4* src = reinterpret_cast<const float4*>(A + 8 * q);
    Pack8 r[3], i[3];
    float4 av[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) av[u] = src[u];
    if (X) {
      const int ti = (int)((8 * q) >> (logd + 7)), tj = (int)((8 * q) & ((1LL << logd) - 1)) >> 7;
      if (ti >= tj) {
        const float4* xs = reinterpret_cast<const float4*>(X + 8 * q);
        float p = 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 x = xs[u];
          p = fmaf(av[u].x, x.x, fmaf(av[u].y, x.y, fmaf(av[u].z, x.z, fmaf(av[u].w, x.w, p))));
        }
        dsum.add(ti > tj ? 2.f * p : p);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 a = av[u];
      const Terms x0 = split3(sc * a.x), y0 = split3(sc * a.y), x1 = split3(sc * a.z), y1 = split3(sc * a.w);
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        r[t].h[2 * u] = x0.v[t];
        i[t].h[2 * u] = y0.v[t];
        r[t].h[2 * u + 1] = x1.v[t];
        i[t].h[2 * u + 1] = y1.v[t];
      }
    }
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      *reinterpret_cast<uint4*>(P + t * nn + 8 * q) = r[t].v;
      *reinterpret_cast<uint4*>(P + (3 + t) * nn + 8 * q) = i[t].v;
      if (nine) {
        Pack8 m;
#pragma unroll
        for (int u = 0; u < 8; ++u) m.h[u] = neg(i[t].h[u]);
        *reinterpret_cast<uint4*>(P + (6 + t) * nn + 8 * q) = m.v;
      }
    }
  }
  if (!X) return;
  __shared__ double red[8];
  const double dot = warp_sum(dsum.value());
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dot;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    partials[blockIdx.x] = s;
  }
  if (last_block_arrived(counter)) {
    if (threadIdx.x < 32) {
      double v = 0.0;
      for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) v += partials[b];
      v = warp_sum(v);
      if (threadIdx.x == 0) {
        scal[kGauge] = flags[0] == flags[4] ? -v / scal[0] : 0.0;
        flags[4] = flags[0];
        *counter = 0u;
      }
    }
  }
}

// The nine planes of the Hermitian T of t (R = t as d x d row-major; T_ii = R_ii, T_ij = R_ij + i R_ji for
// i > j, T_ji = conj T_ij), straight from t: 64 x 64 tile pairs, as k_hermitian_planes64 in gemm_tc.cu.
__global__ void __launch_bounds__(256) k_hermitian_planes3(const float* __restrict__ t, int d,
                                                            __nv_bfloat16* __restrict__ P, const unsigned int* amax,
                                                            double* s_slot, const void* const* tab) {
  rebind(tab, t, P, amax, s_slot);
  grid_dep_wait();
  after_wait(t, P, amax, s_slot);
  asm volatile("griddepcontrol.launch_dependents;");  // the product's prologue may start
  __shared__ float Ra[64][65];
  __shared__ float Rb[64][65];
  const int se = split_exponent(amax);
  const float sc = pow2f(se);
  if (blockIdx.x == 0 && threadIdx.x == 0) *s_slot = pow2d(se);
  const long long nn = (long long)d * d;
  int I, J;
  tri_decode(blockIdx.x, I, J);
  const int tid = threadIdx.x;
  {
    float4 a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // 1024 float4 per tile: row q >> 4, columns 4 (q & 15) ..
      const int q = tid + 256 * k, row = q >> 4, col = (q & 15) * 4;
      a[k] = *reinterpret_cast<const float4*>(t + (long long)(I * 64 + row) * d + J * 64 + col);
      b[k] = I != J ? *reinterpret_cast<const float4*>(t + (long long)(J * 64 + row) * d + I * 64 + col)
                    : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = tid + 256 * k, row = q >> 4, col = (q & 15) * 4;
      Ra[row][col] = a[k].x; Ra[row][col + 1] = a[k].y; Ra[row][col + 2] = a[k].z; Ra[row][col + 3] = a[k].w;
      Rb[row][col] = b[k].x; Rb[row][col + 1] = b[k].y; Rb[row][col + 2] = b[k].z; Rb[row][col + 3] = b[k].w;
    }
  }
  __syncthreads();
  const bool upper = tid >= 128;
  if (upper && I == J) return;
  const int c = (tid & 7) * 8;
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    const int r = ((tid & 127) >> 3) + 16 * k;
    Pack8 pr[3], pi[3], pm[3];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int cc = c + u;
      float re, im;
      if (upper) { re = Ra[cc][r]; im = -Rb[r][cc]; }  // T[J 64 + r][I 64 + cc] = conj T[I 64 + cc][J 64 + r]
      else if (I != J) { re = Ra[r][cc]; im = Rb[cc][r]; }
      else if (r > cc) { re = Ra[r][cc]; im = Ra[cc][r]; }
      else if (r < cc) { re = Ra[cc][r]; im = -Ra[r][cc]; }
      else { re = Ra[r][r]; im = 0.f; }
      const Terms x = split3(sc * re), y = split3(sc * im);
#pragma unroll
      for (int t3 = 0; t3 < 3; ++t3) {
        pr[t3].h[u] = x.v[t3];
        pi[t3].h[u] = y.v[t3];
        pm[t3].h[u] = neg(y.v[t3]);
      }
    }
    const long long idx = upper ? (long long)(J * 64 + r) * d + I * 64 + c : (long long)(I * 64 + r) * d + J * 64 + c;
#pragma unroll
    for (int t3 = 0; t3 < 3; ++t3) {
      *reinterpret_cast<uint4*>(P + t3 * nn + idx) = pr[t3].v;
      *reinterpret_cast<uint4*>(P + (3 + t3) * nn + idx) = pi[t3].v;
      *reinterpret_cast<uint4*>(P + (6 + t3) * nn + idx) = pm[t3].v;
    }
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 3-D map over `planes` d x d BF16 planes, box 32 columns x rows x depth, rows swizzled over 64 bytes.
bool planes_map(CUtensorMap* m, const void* base, int d, int planes, int rows, int depth) {
  EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(tma_encoder());
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)d, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)d * d * 2};
  cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)rows, (cuuint32_t)depth};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool tc32_ok(int d) { return d >= 128 && d % 128 == 0 && tc_available(); }

cudaError_t tc32_planes_T(int d, const float* t, void* P, const unsigned int* amax, double* s_slot, cudaStream_t s) {
  if (d % 64) return cudaErrorInvalidValue;
  BatchArgs ba;
  if (batch_take(ba, {t, P, amax, s_slot})) return cudaSuccess;
  const int n64 = d / 64;
  return launch_dep(k_hermitian_planes3, dim3((unsigned)(n64 * (n64 + 1) / 2), 1, ba.nz), dim3(256), 0, s, t, d,
                    (__nv_bfloat16*)P, amax, s_slot, ba.tab);
}

cudaError_t tc32_split(int d, const float2* A, void* P, int planes, bool keep_scale, const unsigned int* amax,
                       double* s_slot, cudaStream_t s, const float2* X, double* scal, double* partials,
                       unsigned int* counter, unsigned int* flags) {
  const long long nn = (long long)d * d;
  if (nn % 1024 || (planes != 6 && planes != 9)) return cudaErrorInvalidValue;
  long long blocks = (nn / 8 + 255) / 256;
  if (blocks > (X ? 608 : 2048)) blocks = X ? 608 : 2048;  // with X: four per SM, fewer FP64 sums
  BatchArgs ba;
  if (batch_take(ba, {A, P, amax, s_slot, X, scal, partials, counter, flags})) return cudaSuccess;
  return launch_dep(k_split3, dim3((unsigned)blocks, 1, ba.nz), dim3(256), 0, s, A, (__nv_bfloat16*)P, nn,
                    planes == 9 ? 1 : 0, keep_scale ? 1 : 0, amax, s_slot, X, __builtin_ctz((unsigned)d), scal,
                    partials, counter, flags, ba.tab);
}

// CTAs per tile: one from d = 2048 on (136 and 256 tiles on 152 SMs); below, K shared so that a single product
// reaches more SMs (the order of the sums depends on d alone, so a batch has the bits of its members).
static int k_split(int d) { return d >= 2048 ? 1 : d >= 512 ? 2 : kMaxSplit; }

cudaError_t tc32_product(int d, const void* Ap, const void* Bp, const double* sA, const double* sB, float2* C,
                         bool lower, int krange, unsigned int* err, unsigned int* clear, cudaStream_t s) {
  if (d < kBM || d % kBM) return cudaErrorInvalidValue;
  cudaError_t e = ensure_dynamic_smem((const void*)k_tc_cgemm32, kSmem);
  if (e != cudaSuccess) return e;
  Maps32 M;
  if (!planes_map(&M.a, Ap, d, 6, kBM, 3) || !planes_map(&M.b, Bp, d, 9, kBN, 1)) return cudaErrorInvalidValue;
  BatchArgs ba;
  if (batch_take(ba, {C, sA, sB, err, clear}, &M, sizeof(Maps32))) return cudaSuccess;
  const int no_loads = inject_take(INJ_TC_LOADS) ? 1 : 0;
  const int nt = d / kBM, ks = k_split(d);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = lower ? dim3((unsigned)(nt * (nt + 1) / 2 * ks), 1, ba.nz) : dim3(nt * ks, nt, ba.nz);
  cfg.blockDim = dim3(kThreads32);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)ks;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_tc_cgemm32, M, C, d, lower ? 1 : 0, krange, ks, sA, sB, err, clear, no_loads,
                            ba.tab);
}

}  // namespace qst
