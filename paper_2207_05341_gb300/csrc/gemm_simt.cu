// Complex d x d products on the CUDA cores (FP64, and FP32 where gemm_tc_fp32.cu does not run them):
//   X = T T   (Sec. 3.2 eq. unified_DP, Hermitian: only tiles I >= J are computed)
//   Y = G T   (backward of X = T T)
// Row-major complex operands.
//
// FP32 (k_cgemm): packed FMAs and 16-byte shared loads only in the inner loop: A is staged as (x, x, -y, y) and B
// as (x, y, y, x), the operand pairs of the two FMAs of a complex product (packing them in registers cost more than
// the shorter loads saved: 63 against 54 us at d = 512), and a thread's 4 x 4 entries take 32 FMAs from 8 loads.
// What bounds it below d = 1024 is latency, two warps to a tile and one or two tiles to an SM (8 x 4 entries a
// thread, half the warps: 101 us).  The next K slice is loaded into registers meanwhile.  Every entry is the sum
// over k in order, re: a.x b.x then -a.y b.y, im: a.x b.y then a.y b.x, whatever the tile.
//
// FP64 has its own kernel (k_cgemm_f64): this part does 2 FP64 FMAs per clock and SM, a fortieth of its FP32
// rate, so what counts is that every SM gets the same share of them, not the operand traffic.
#include <cooperative_groups.h>

#include "impl.h"

namespace qst {

// BM x BM tile by (BM / 4)^2 threads: thread (ty, tx) the rows ty + BM / 4 i and columns tx + BM / 4 j.
template <int BM, int BK>
__global__ void __launch_bounds__((BM / 4) * (BM / 4)) k_cgemm(int d, const float2* __restrict__ A,
                                                               const float2* __restrict__ B, float2* __restrict__ C,
                                                               int lower, const void* const* tab) {
  rebind(tab, A, B, C);
  constexpr int TX = BM / 4, NT = TX * TX, L = BM * BK / NT;
  __shared__ float4 As[2][BK][BM + 1];
  __shared__ float4 Bs[2][BK][BM];
  int I, J;
  if (lower) tri_decode(blockIdx.x, I, J);
  else { I = blockIdx.y; J = blockIdx.x; }
  const int m0 = I * BM, n0 = J * BM, tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  float2 ra[L], rb[L];
  auto gload = [&](int k0) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const int e = tid + l * NT;
      ra[l] = A[(long long)(m0 + e / BK) * d + k0 + e % BK];
      rb[l] = B[(long long)(k0 + e / BM) * d + n0 + e % BM];
    }
  };
  auto sstore = [&](int buf) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const int e = tid + l * NT;
      As[buf][e % BK][e / BK] = make_float4(ra[l].x, ra[l].x, -ra[l].y, ra[l].y);
      Bs[buf][e / BM][e % BM] = make_float4(rb[l].x, rb[l].y, rb[l].y, rb[l].x);
    }
  };
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int nk = d / BK;
  gload(0);
  sstore(0);
  __syncthreads();
  for (int kt = 0; kt < nk; ++kt) {
    const int buf = kt & 1;
    if (kt + 1 < nk) gload((kt + 1) * BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float4 a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[buf][k][ty + TX * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[buf][k][tx + TX * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          acc[i][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), make_float2(b[j].z, b[j].w),
                                 __ffma2_rn(make_float2(a[i].x, a[i].y), make_float2(b[j].x, b[j].y), acc[i][j]));
    }
    if (kt + 1 < nk) {
      sstore(buf ^ 1);
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) C[(long long)(m0 + ty + TX * i) * d + n0 + tx + TX * j] = acc[i][j];
}

// d >= 2048, where tiles abound: 128 x 128 tiles, 8 x 8 entries a thread (half the shared loads per FMA; X = T T at
// d = 2048 in 914 us against 1035 with k_cgemm's 64 x 64 tiles, Y = G T in 1778 against 1838).  Same order of sums.
__global__ void __launch_bounds__(256) k_cgemm_large(int d, const float2* __restrict__ A, const float2* __restrict__ B,
                                                     float2* __restrict__ C, int lower, const void* const* tab) {
  using V = float2;
  using R = float;
  constexpr int BM = 128, BN = 128, BK = 8, TM = 8, TN = 8;
  rebind(tab, A, B, C);
  constexpr int NTX = BN / TN, NTY = BM / TM, NT = NTX * NTY;
  constexpr int LA = BM * BK / NT, LB = BK * BN / NT;
  constexpr int PAD = 4;
  constexpr int CW = 16 / (int)sizeof(V);  // complex entries per 16-byte chunk
  static_assert(TN % CW == 0, "a thread's columns are whole 16-byte chunks");
  static_assert(LA >= 1 && LB >= 1, "tile too small for the thread count");
  __shared__ __align__(16) V As[2][BK][BM + PAD];
  __shared__ __align__(16) V Bs[2][BK][BN + PAD];

  int I, J;
  if (lower) tri_decode(blockIdx.x, I, J);
  else { I = blockIdx.y; J = blockIdx.x; }
  const int m0 = I * BM, n0 = J * BN;
  const int tid = threadIdx.x;
  const int tx = tid % NTX, ty = tid / NTX;

  V ra[LA], rb[LB];
  auto gload = [&](int k0) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = tid + l * NT;
      const int m = e / BK, kk = e % BK;
      ra[l] = A[(long long)(m0 + m) * d + k0 + kk];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = tid + l * NT;
      const int kk = e / BN, nn = e % BN;
      rb[l] = B[(long long)(k0 + kk) * d + n0 + nn];
    }
  };
  auto sstore = [&](int buf) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = tid + l * NT;
      As[buf][e % BK][e / BK] = ra[l];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = tid + l * NT;
      Bs[buf][e / BN][e % BN] = rb[l];
    }
  };

  R accr[TM][TN], acci[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) { accr[i][j] = R(0); acci[i][j] = R(0); }

  const int nk = d / BK;
  gload(0);
  sstore(0);
  __syncthreads();
  for (int kt = 0; kt < nk; ++kt) {
    const int buf = kt & 1;
    if (kt + 1 < nk) gload((kt + 1) * BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      V a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM / 2; ++i) {
        a[i] = As[buf][k][ty * (TM / 2) + i];
        a[TM / 2 + i] = As[buf][k][BM / 2 + ty * (TM / 2) + i];
      }
#pragma unroll
      for (int g = 0; g < TN / CW; ++g)
#pragma unroll
        for (int j = 0; j < CW; ++j) b[g * CW + j] = Bs[buf][k][g * (NTX * CW) + tx * CW + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          accr[i][j] = fma(a[i].x, b[j].x, accr[i][j]);
          accr[i][j] = fma(-a[i].y, b[j].y, accr[i][j]);
          acci[i][j] = fma(a[i].x, b[j].y, acci[i][j]);
          acci[i][j] = fma(a[i].y, b[j].x, acci[i][j]);
        }
    }
    if (kt + 1 < nk) {
      sstore(buf ^ 1);
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + (i < TM / 2 ? ty * (TM / 2) + i : BM / 2 + ty * (TM / 2) + (i - TM / 2));
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int nn = n0 + (j / CW) * (NTX * CW) + tx * CW + j % CW;
      C[(long long)m * d + nn] = cmake<V>(accr[i][j], acci[i][j]);
    }
  }
}

// FP64, d >= 32: 16 x 16 output tiles, each the work of a cluster of gridDim.x / tiles CTAs that split K between
// them (CTA r of a cluster takes d / ks consecutive k), so that the small sizes reach all SMs: at d = 128 the
// 64 x 64 tiles it replaces were 3 and 4 CTAs on 152 SMs (521 us each; the FMAs alone are 7 and 13 us spread
// over the chip, and 14 and 21 us is what this kernel takes).  A thread holds one row and two columns (8 FMAs per k from 3 entries).  The partial tiles
// meet in distributed shared memory: CTA r sums rows r 16 / ks .. of all ranks, in the order of the ranks.
constexpr int kT64 = 16;

__global__ void __launch_bounds__(128) k_cgemm_f64(int d, const double2* __restrict__ A,
                                                    const double2* __restrict__ B, double2* __restrict__ C, int lower,
                                                    int ks) {
  namespace cg = cooperative_groups;
  __shared__ double2 As[2][kT64][kT64 + 1];
  __shared__ double2 Bs[2][kT64][kT64];
  __shared__ double2 part[kT64][kT64];
  const int tile = (int)blockIdx.x / ks, rank = (int)blockIdx.x % ks, nt = d / kT64;
  int I, J;
  if (lower) tri_decode((uint32_t)tile, I, J);
  else { I = tile / nt; J = tile % nt; }
  const int tid = threadIdx.x, row = tid >> 3, col = tid & 7;
  const int k0 = rank * (d / ks), steps = d / ks / kT64;
  double2 ra[2], rb[2];
  auto gload = [&](int k) {
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const int e = tid + 128 * l, r = e >> 4, c = e & 15;
      ra[l] = A[(long long)(I * kT64 + r) * d + k + c];
      rb[l] = B[(long long)(k + r) * d + J * kT64 + c];
    }
  };
  double re[2] = {0.0, 0.0}, im[2] = {0.0, 0.0};
  gload(k0);
  for (int s = 0; s < steps; ++s) {
    const int buf = s & 1;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const int e = tid + 128 * l;
      As[buf][e >> 4][e & 15] = ra[l];
      Bs[buf][e >> 4][e & 15] = rb[l];
    }
    __syncthreads();
    if (s + 1 < steps) gload(k0 + (s + 1) * kT64);
#pragma unroll
    for (int k = 0; k < kT64; ++k) {
      const double2 a = As[buf][row][k];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const double2 b = Bs[buf][k][col + 8 * j];
        re[j] = fma(a.x, b.x, re[j]);
        im[j] = fma(a.x, b.y, im[j]);
        re[j] = fma(-a.y, b.y, re[j]);
        im[j] = fma(a.y, b.x, im[j]);
      }
    }
  }
  double2* out = C + (long long)(I * kT64) * d + J * kT64;
  if (ks == 1) {
#pragma unroll
    for (int j = 0; j < 2; ++j) out[(long long)row * d + col + 8 * j] = make_double2(re[j], im[j]);
    return;
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) part[row][col + 8 * j] = make_double2(re[j], im[j]);
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  const int rows = kT64 / ks;
  for (int e = tid; e < rows * kT64; e += 128) {
    const int r = rank * rows + (e >> 4), c = e & 15;
    double2 s = make_double2(0.0, 0.0);
    for (int q = 0; q < ks; ++q) {
      const double2 v = *cl.map_shared_rank(&part[r][c], q);
      s.x += v.x;
      s.y += v.y;
    }
    out[(long long)r * d + c] = s;
  }
  cl.sync();  // no CTA leaves while its part may still be read
}

// Small matrices (d <= 16): one thread per output element.
template <class R>
__global__ void k_cgemm_small(int d, const cx_t<R>* A, const cx_t<R>* B, cx_t<R>* C, int lower) {
  using V = cx_t<R>;
  for (int e = threadIdx.x + blockIdx.x * blockDim.x; e < d * d; e += blockDim.x * gridDim.x) {
    const int m = e / d, nn = e % d;
    R sr = R(0), si = R(0);
    for (int k = 0; k < d; ++k) {
      const V a = A[m * d + k], b = B[k * d + nn];
      sr = fma(a.x, b.x, sr); sr = fma(-a.y, b.y, sr);
      si = fma(a.x, b.y, si); si = fma(a.y, b.x, si);
    }
    C[e] = cmake<V>(sr, si);
  }
}

template <int BM, int BK>
static cudaError_t run_tiled(int d, const float2* A, const float2* B, float2* C, bool lower, cudaStream_t s) {
  constexpr int NT = (BM / 4) * (BM / 4);
  const int nt = d / BM;
  BatchArgs ba;
  if (batch_take(ba, {A, B, C})) return cudaSuccess;
  const dim3 grid = lower ? dim3((unsigned)(nt * (nt + 1) / 2), 1, ba.nz) : dim3(nt, nt, ba.nz);
  k_cgemm<BM, BK><<<grid, NT, 0, s>>>(d, A, B, C, lower ? 1 : 0, ba.tab);
  return cudaGetLastError();
}

// 64 x 64 tiles at d = 1024 (136 and 256 of them on 152 SMs); 32 x 32 tiles of two warps below, where 64-wide ones
// would be 64 CTAs at most (d = 512: 54 us, 231 with 128 x 128 tiles).  A lower result covers the diagonal tiles
// whole; its readers take entries on or below the diagonal only.
template <>
cudaError_t cgemm_simt<float>(int d, const float2* A, const float2* B, float2* C, bool lower, cudaStream_t s) {
  if (d >= 2048) {
    const int nt = d / 128;
    BatchArgs ba;
    if (batch_take(ba, {A, B, C})) return cudaSuccess;
    k_cgemm_large<<<lower ? dim3((unsigned)(nt * (nt + 1) / 2), 1, ba.nz) : dim3(nt, nt, ba.nz), 256, 0, s>>>(
        d, A, B, C, lower ? 1 : 0, ba.tab);
    return cudaGetLastError();
  }
  if (d == 1024) return run_tiled<64, 8>(d, A, B, C, lower, s);
  if (d >= 32) return run_tiled<32, 16>(d, A, B, C, lower, s);
  k_cgemm_small<float><<<1, 256, 0, s>>>(d, A, B, C, lower ? 1 : 0);
  return cudaGetLastError();
}

// At least four CTAs per SM where K can be split that far (16 elements of K per CTA, clusters of up to 8).
template <>
cudaError_t cgemm_simt<double>(int d, const double2* A, const double2* B, double2* C, bool lower, cudaStream_t s) {
  if (d <= kT64) {
    k_cgemm_small<double><<<1, 256, 0, s>>>(d, A, B, C, lower ? 1 : 0);
    return cudaGetLastError();
  }
  if (d % kT64) return cudaErrorInvalidValue;
  const int nt = d / kT64, tiles = lower ? nt * (nt + 1) / 2 : nt * nt;
  int ks = 1;
  while (ks < 8 && tiles * ks < 4 * 152 && d / (2 * ks) >= kT64) ks *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * ks));
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ks;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_cgemm_f64, d, A, B, C, lower ? 1 : 0, ks);
}

}  // namespace qst
