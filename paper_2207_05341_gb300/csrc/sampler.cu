// Synthetic measurement data on the GPU (Sec. 4): the test states of the paper's sweeps and seeded
// multinomial counts of a probability vector (Sec. 4.5.1: "a certain number of samples from sampling a
// multinomial distribution of measurement probabilities").
//
// States: rho = w |psi><psi| + (1 - w) I / d for the product state ((|0> + |1>)/sqrt 2)^N, the GHZi state
// (|0..0> + i |1..1>)/sqrt 2 and the W state (equal superposition of the N one-excitation states); white
// noise uses w = p, the depolarising channel w = 1 - lambda.
//
// Counts: each probability becomes an integer weight w_k = floor(max(P_k, 0) 2^52) (P_k <= 1), so the
// running sums C_k are exact whatever the order of the scan.  Shot s takes z_s = splitmix64(seed, s)
// (SplitMix64, Steele, Lea and Flood, OOPSLA 2014: x = seed + (s + 1) 0x9E3779B97F4A7C15, then its
// published mix), t_s = floor((z_s >> 11) W / 2^53) with W = C_{n-1} (exact 128-bit product), and the
// outcome k_s = the smallest k with C_k > t_s; counts[k_s] += 1 (integer atomics: the counts do not depend
// on the order).  Every decision is integer arithmetic, so the counts are bit-exact and reproducible.
#include "../../include/qst.h"
#include "impl.h"
#include "rng.cuh"

namespace qst {

namespace {

constexpr int kPer = 8;
constexpr int kBlockElems = 256 * kPer;

template <class R>
__global__ void __launch_bounds__(256) k_test_state(cx_t<R>* __restrict__ rho, int N, int kind, double w) {
  const int d = 1 << N;
  const long long nn = (long long)d * d;
  const R s2 = (R)0.70710678118654752440;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nn; e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / d), j = (int)(e % d);
    auto amp = [&](int k, R& re, R& im) {  // psi_k
      re = R(0);
      im = R(0);
      if (kind == QST_STATE_PRODUCT) {
        re = (R)(1.0 / sqrt((double)d));
      } else if (kind == QST_STATE_GHZI) {
        if (k == 0) re = s2;
        if (k == d - 1) im = s2;
      } else if (__popc(k) == 1) {  // W
        re = (R)(1.0 / sqrt((double)N));
      }
    };
    R ar, ai, br, bi;
    amp(i, ar, ai);
    amp(j, br, bi);
    // w psi_i conj(psi_j) + (1 - w) delta_ij / d
    R re = (R)w * (ar * br + ai * bi), im = (R)w * (ai * br - ar * bi);
    if (i == j) re += (R)((1.0 - w) / d);
    rho[e] = cmake<cx_t<R>>(re, im);
  }
}

// floor(max(p, 0) 2^52) from the bits of p (FP64 arithmetic is two operations per clock and SM here); a bad
// probability (not finite, or above 1) raises *bad.
__device__ __forceinline__ unsigned long long weight_of(double p, unsigned int* bad) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(p), mag = b & 0x7FFFFFFFFFFFFFFFull;
  if (mag >= 0x7FF0000000000000ull || (b == mag && mag > 0x3FF0000000000000ull)) {
    atomicOr(bad, 1u);
    return 0;
  }
  if (b != mag) return 0;  // negative (or -0)
  const int sh = 1023 - (int)(mag >> 52);  // p = m 2^(-52 - sh), m in [2^52, 2^53): the weight is m >> sh
  return sh > 52 ? 0 : ((mag & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) >> sh;
}

// The weights of a block's kBlockElems outcomes, summed (SCAN false: their total to tops[block]) or as running
// sums on top of tops[block] (SCAN true: C, and counts cleared).  Two passes over P instead of a pass over P and
// one over C: nothing is written before it is final (10 and 16 us at N = 11, 46 and 14 before).
template <bool SCAN>
__global__ void __launch_bounds__(256) k_weights(const double* __restrict__ P, long long n,
                                                  unsigned long long* __restrict__ C,
                                                  unsigned long long* __restrict__ tops,
                                                  long long* __restrict__ counts, unsigned int* bad) {
  __shared__ unsigned long long wsum[8];
  // thread t takes the pairs t, t + 256, ... of the block: whole lines per warp and load
  const long long base = (long long)blockIdx.x * kBlockElems;
  const bool vec = ((reinterpret_cast<uintptr_t>(P) | reinterpret_cast<uintptr_t>(SCAN ? counts : nullptr)) & 15u) == 0 &&
                   base + kBlockElems <= n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long before = SCAN ? tops[blockIdx.x] : 0;
  unsigned long long total = 0;
  double2 pv[kPer / 2];
#pragma unroll
  for (int k = 0; k < kPer / 2; ++k) {
    const long long i = base + 2 * (threadIdx.x + 256 * k);
    if (vec) pv[k] = *reinterpret_cast<const double2*>(P + i);
    else pv[k] = make_double2(i < n ? P[i] : 0.0, i + 1 < n ? P[i + 1] : 0.0);
  }
#pragma unroll
  for (int k = 0; k < kPer / 2; ++k) {
    if (base + 512LL * k >= n) break;  // the whole slice is past the end
    const unsigned long long w0 = weight_of(pv[k].x, bad), w1 = weight_of(pv[k].y, bad);
    if (!SCAN) {
      total += w0 + w1;
      continue;
    }
    unsigned long long x = w0 + w1;  // inclusive scan of the pairs over the block
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    __syncthreads();  // the slice before has read wsum
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    unsigned long long off = before, all = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      off += w < warp ? wsum[w] : 0;
      all += wsum[w];
    }
    before += all;
    const long long i = base + 2 * (threadIdx.x + 256 * k);
    const unsigned long long c1 = off + x, c0 = c1 - w1;
    if (vec) {
      *reinterpret_cast<ulonglong2*>(C + i) = make_ulonglong2(c0, c1);
      *reinterpret_cast<longlong2*>(counts + i) = make_longlong2(0, 0);
    } else {
      if (i < n) { C[i] = c0; counts[i] = 0; }
      if (i + 1 < n) { C[i + 1] = c1; counts[i + 1] = 0; }
    }
  }
  if (!SCAN) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (lane == 0) wsum[warp] = total;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long t = 0;
      for (int w = 0; w < 8; ++w) t += wsum[w];
      tops[blockIdx.x] = t;
    }
  }
}

__global__ void __launch_bounds__(1024) k_tops_scan(unsigned long long* tops, int nb) {
  __shared__ unsigned long long wsum[32];
  const int per = (nb + 1023) / 1024;
  const int b0 = threadIdx.x * per;
  unsigned long long run = 0;
  for (int b = b0; b < b0 + per && b < nb; ++b) run += tops[b];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long x = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  unsigned long long off = x - run;
  for (int w = 0; w < warp; ++w) off += wsum[w];
  for (int b = b0; b < b0 + per && b < nb; ++b) {
    const unsigned long long t = tops[b];
    tops[b] = off;
    off += t;
  }
}

// smallest k in [lo, hi] with C[k] > t (C[hi] > t, or hi = n - 1)
__device__ __forceinline__ long long first_above(const unsigned long long* __restrict__ C, unsigned long long t,
                                                 long long lo, long long hi) {
  while (lo < hi) {
    const long long m = (lo + hi) >> 1;
    if (C[m] > t) hi = m;
    else lo = m + 1;
  }
  return lo;
}

// start[b] = the outcome of the draw t = b 2^sh, b = 0 .. M - 1, and start[M] = n - 1 (M 2^sh is at least the total
// weight, and 2^64 where that has 64 bits): a draw t then lies between start[t >> sh] and the entry after it.
// Neighbouring buckets search neighbouring places, so this costs far less than as many draws.
__global__ void __launch_bounds__(256) k_guide(const unsigned long long* __restrict__ C, long long n, int M, int sh,
                                                int* __restrict__ start) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= M; b += gridDim.x * blockDim.x)
    start[b] = b < M ? (int)first_above(C, (unsigned long long)b << sh, 0, n - 1) : (int)(n - 1);
}

// One draw: a bucket of the guide table and, within it, a search over the few outcomes that share it (about four at
// n = 4 M; without the table every draw was 22 dependent loads over 33 MB, 600 us for 10^7 shots at N = 11; now 148 us, the
// table 29, bound by the random sectors of C and the atomics on counts).
__global__ void __launch_bounds__(256) k_draw(const unsigned long long* __restrict__ C, long long n, long long shots,
                                               unsigned long long seed, const int* __restrict__ start, int sh,
                                               long long* __restrict__ counts) {
  const unsigned long long W = C[n - 1];
  for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < shots; s += (long long)gridDim.x * blockDim.x) {
    const unsigned long long a = splitmix64(seed, (unsigned long long)s) >> 11;  // < 2^53
    const unsigned long long hi = __umul64hi(a, W), lo = a * W;
    const unsigned long long t = (hi << 11) | (lo >> 53);                         // floor(a W / 2^53) < W
    const int b = (int)(t >> sh);
    const long long l = start ? first_above(C, t, start[b], start[b + 1]) : first_above(C, t, 0, n - 1);
    atomicAdd(reinterpret_cast<unsigned long long*>(counts + l), 1ull);
  }
}

// f = counts / shots, correctly rounded as on the host.  Nearly all counts are small and share few quotients, so a
// block makes those once (one FP64 division per entry was 169 us at N = 11; this is 20).
constexpr int kQuot = 256;
template <class R>
__global__ void __launch_bounds__(256) k_freq(const long long* __restrict__ counts, long long n, long long shots,
                                               R* __restrict__ f) {
  __shared__ R quot[kQuot];
  for (int c = threadIdx.x; c < kQuot; c += blockDim.x) quot[c] = (R)((double)c / (double)shots);
  __syncthreads();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long c = counts[i];
    f[i] = c >= 0 && c < kQuot ? quot[c] : (R)((double)c / (double)shots);
  }
}

int grid_of(long long work, int sms_mult = 8) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long g = (work + 255) / 256;
  const long long cap = (long long)sms * sms_mult;
  if (g > cap) g = cap;
  return g < 1 ? 1 : (int)g;
}

}  // namespace

long long sampler_scratch_words(long long n) { return n + (n + kBlockElems - 1) / kBlockElems; }

template <class R> cudaError_t make_test_state(int N, int kind, double w, cx_t<R>* rho, cudaStream_t s) {
  const long long nn = 1LL << (2 * N);
  k_test_state<R><<<grid_of(nn), 256, 0, s>>>(rho, N, kind, w);
  return cudaGetLastError();
}

cudaError_t multinomial_prepare(long long n, const double* P, unsigned long long* scratch, long long* counts,
                                unsigned int* bad, cudaStream_t s) {
  const int nb = (int)((n + kBlockElems - 1) / kBlockElems);
  unsigned long long* C = scratch;
  unsigned long long* tops = scratch + n;
  k_weights<false><<<nb, 256, 0, s>>>(P, n, C, tops, counts, bad);
  k_tops_scan<<<1, 1024, 0, s>>>(tops, nb);
  k_weights<true><<<nb, 256, 0, s>>>(P, n, C, tops, counts, bad);
  return cudaGetLastError();
}

// The guide table has a bucket for every four outcomes, or every four shots where those are fewer (building it is then
// a fraction of the draws).  None below 2^19 shots or 4096 outcomes: its launch costs 4 us, more than it saves on
// 10^5 draws (N = 6: 39.7 us without, 43.7 with; N = 9 and 10^4 draws 45.7 and 50.8; 10^7 draws at N = 6 277 and 203),
// and below 4096 outcomes the atomics on the counts are what a draw waits for (N = 5, 10^7 draws: 544 and 545).
cudaError_t multinomial_draw(long long n, long long shots, unsigned long long seed, unsigned long long W,
                             const unsigned long long* scratch, int* guide, long long* counts, int* kernels,
                             cudaStream_t s) {
  *kernels = 0;
  if (shots <= 0) return cudaSuccess;
  int lm = 0, bits = 64;
  while (lm < 30 && (1LL << (lm + 1)) <= shots / 4 && (1LL << (lm + 1)) <= n / 4) ++lm;
  while (bits > 0 && !((W - 1) >> (bits - 1) & 1ull)) --bits;  // (W - 1) >> (bits - lm) < 2^lm
  const int M = 1 << lm, sh = bits > lm ? bits - lm : 0;
  const bool table = guide && shots >= (1LL << 19) && n >= 4096 && sh < 64;
  if (table) k_guide<<<grid_of(M + 1), 256, 0, s>>>(scratch, n, M, sh, guide);
  k_draw<<<grid_of(shots), 256, 0, s>>>(scratch, n, shots, seed, table ? guide : nullptr, table ? sh : 0, counts);
  *kernels = table ? 2 : 1;
  return cudaGetLastError();
}

template <class R> cudaError_t counts_to_frequencies(long long n, const long long* counts, long long shots, R* f,
                                                     cudaStream_t s) {
  k_freq<R><<<grid_of(n, 4), 256, 0, s>>>(counts, n, shots, f);
  return cudaGetLastError();
}

template cudaError_t make_test_state<float>(int, int, double, cx_t<float>*, cudaStream_t);
template cudaError_t make_test_state<double>(int, int, double, cx_t<double>*, cudaStream_t);
template cudaError_t counts_to_frequencies<float>(long long, const long long*, long long, float*, cudaStream_t);
template cudaError_t counts_to_frequencies<double>(long long, const long long*, long long, double*, cudaStream_t);

}  // namespace qst
