// The single-qubit mode maps over a whole tile in shared memory (povm.cu, tomo_fused.cu).
#pragma once

#include "common.cuh"

namespace qst {

// The mode maps of all g qubits of an S x S tile (S = 2^g), two qubits per sweep: a thread takes
// the 4 x 4 elements that bits (b, b+1) of the row and column index span, applies qubit b and
// then qubit b + 1 in registers and stores them back (each element sees the same operations in
// the same order as with one qubit per sweep, so the result is bit-identical, with half the
// shared-memory traffic and barriers).
template <class R, bool ADJ>
__device__ void apply_modes_tile(cx_t<R>* Z, int g, int pitch, const PovmB<R>& B) {
  using V = cx_t<R>;
  int b = 0;
  // FP64: one qubit per sweep, so that a 16 x 16 tile keeps two warps on two FP64 pipes instead of half a warp
  for (; sizeof(R) == 4 && b + 1 < g; b += 2) {
    const int gh = g - 2;
    const int groups = 1 << (2 * gh);
    const int low = (1 << b) - 1;
    for (int t = threadIdx.x; t < groups; t += blockDim.x) {
      const int rr = t >> gh, cc = t & ((1 << gh) - 1);
      const int r0 = ((rr & ~low) << 2) | (rr & low);
      const int c0 = ((cc & ~low) << 2) | (cc & low);
      V x[4][4];  // [k][l]: row offset (k >> 1) << (b + 1) | (k & 1) << b, column offset likewise
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int l = 0; l < 4; ++l)
          x[k][l] = Z[(r0 + (((k >> 1) << (b + 1)) | ((k & 1) << b))) * pitch + c0 + (((l >> 1) << (b + 1)) | ((l & 1) << b))];
#pragma unroll
      for (int hk = 0; hk < 2; ++hk)
#pragma unroll
        for (int hl = 0; hl < 2; ++hl) {  // qubit b: row bit k & 1, column bit l & 1
          if (ADJ) mode_adj(B, x[2 * hk][2 * hl], x[2 * hk][2 * hl + 1], x[2 * hk + 1][2 * hl], x[2 * hk + 1][2 * hl + 1]);
          else mode_fwd(B, x[2 * hk][2 * hl], x[2 * hk][2 * hl + 1], x[2 * hk + 1][2 * hl], x[2 * hk + 1][2 * hl + 1]);
        }
#pragma unroll
      for (int lk = 0; lk < 2; ++lk)
#pragma unroll
        for (int ll = 0; ll < 2; ++ll) {  // qubit b + 1: row bit k >> 1, column bit l >> 1
          if (ADJ) mode_adj(B, x[lk][ll], x[lk][2 + ll], x[2 + lk][ll], x[2 + lk][2 + ll]);
          else mode_fwd(B, x[lk][ll], x[lk][2 + ll], x[2 + lk][ll], x[2 + lk][2 + ll]);
        }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int l = 0; l < 4; ++l)
          Z[(r0 + (((k >> 1) << (b + 1)) | ((k & 1) << b))) * pitch + c0 + (((l >> 1) << (b + 1)) | ((l & 1) << b))] = x[k][l];
    }
    __syncthreads();
  }
  for (; b < g; ++b) {  // odd g: the last qubit alone
    const int half = g - 1;
    const int groups = 1 << (2 * half);
    const int bit = 1 << b, low = bit - 1;
    for (int t = threadIdx.x; t < groups; t += blockDim.x) {
      const int rr = t >> half, cc = t & ((1 << half) - 1);
      const int r0 = ((rr & ~low) << 1) | (rr & low);
      const int c0 = ((cc & ~low) << 1) | (cc & low);
      V* p00 = Z + r0 * pitch + c0;
      V x00 = p00[0], x01 = p00[bit], x10 = p00[bit * pitch], x11 = p00[bit * pitch + bit];
      if (ADJ) mode_adj(B, x00, x01, x10, x11);
      else mode_fwd(B, x00, x01, x10, x11);
      p00[0] = x00; p00[bit] = x01; p00[bit * pitch] = x10; p00[bit * pitch + bit] = x11;
    }
    __syncthreads();
  }
}

}  // namespace qst
