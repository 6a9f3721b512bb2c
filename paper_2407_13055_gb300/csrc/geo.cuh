// Launch geometry of the row/column kernels for each supported ring degree.
#pragma once
#include "ntt.cuh"

namespace ckks {

// EC, ER: values per thread in the column and row phases; H = EC^2 rows of
// W = ER^2 words. Supported: N = 2^8 (4, 4), 2^12 (8, 8), 2^16 (8, 32).
template <int EC_, int ER_>
struct Geo {
  static constexpr int EC = EC_, ER = ER_;
  static constexpr int H = EC * EC, W = ER * ER, N = H * W;
  static constexpr int RPC = (128 / ER < H) ? 128 / ER : H;  // rows per row-kernel block
  static constexpr int RT = RPC * ER;                         // row-kernel threads
  static constexpr int TC = 16;                               // columns per column-kernel block
  static constexpr int CT = TC * EC;                          // column-kernel threads
  static constexpr int ROWBUF = W + ER;                       // words per row transpose buffer
  static constexpr int COLBUF = (H + EC) * TC;                // words per column transpose buffer
};

#define CKKS_DISPATCH_LOGN(log_n, ...)                    \
  do {                                                    \
    switch (log_n) {                                      \
      case 8: {                                           \
        using G = ::ckks::Geo<4, 4>;                      \
        __VA_ARGS__;                                      \
      } break;                                            \
      case 12: {                                          \
        using G = ::ckks::Geo<8, 8>;                      \
        __VA_ARGS__;                                      \
      } break;                                            \
      case 16: {                                          \
        using G = ::ckks::Geo<8, 32>;                     \
        __VA_ARGS__;                                      \
      } break;                                            \
      default:                                            \
        break;                                            \
    }                                                     \
  } while (0)

__device__ __forceinline__ uint32_t brev_n(uint32_t v, int log_n) { return __brev(v) >> (32 - log_n); }

// Source position (internal bit-reversed layout) of destination position p
// under the NTT-domain automorphism out[j] = in[((2j+1)k mod 2N - 1)/2] (Eq. 4).
__device__ __forceinline__ uint32_t auto_src(uint32_t p, uint32_t k, int log_n) {
  uint32_t j = brev_n(p, log_n);
  uint32_t mask = (2u << log_n) - 1;
  uint32_t jp = (((2 * j + 1) * k) & mask) >> 1;
  return brev_n(jp, log_n);
}

// The automorphism's sources of four consecutive positions p0 .. p0 + 3 (p0 a
// multiple of 4). Their indices j differ in the top two bits only, and an odd
// multiple of that difference stays there, so the sources are one aligned quad
// in another order: one 16-byte load (s 16-byte aligned) and two rounds of
// swaps instead of four index computations and 4-byte loads. The swaps wait
// for the load, so a kernel with several quads issues every load first.
struct AutoQuad {
  uint32_t at, a, b;  // the quad's first word; its order
  __device__ __forceinline__ AutoQuad(uint32_t p0, uint32_t k, int log_n) {
    const uint32_t mask = (2u << log_n) - 1, jp = (((2 * brev_n(p0, log_n) + 1) * k) & mask) >> 1;
    at = brev_n(jp, log_n) & ~3u;
    a = jp >> (log_n - 2);
    b = a + k;
  }
  __device__ __forceinline__ uint4 load(const uint32_t* __restrict__ s) const {
    return __ldg(reinterpret_cast<const uint4*>(s + at));
  }
  __device__ __forceinline__ void order(const uint4& w, uint32_t (&v)[4]) const {
    const bool hi = a & 1, s0 = a & 2, s1 = b & 2;
    const uint32_t l0 = hi ? w.z : w.x, l1 = hi ? w.w : w.y, u0 = hi ? w.x : w.z, u1 = hi ? w.y : w.w;
    v[0] = s0 ? l1 : l0;
    v[1] = s0 ? l0 : l1;
    v[2] = s1 ? u1 : u0;
    v[3] = s1 ? u0 : u1;
  }
};

}  // namespace ckks
