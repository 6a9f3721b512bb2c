// Row phase of the NTT / iNTT as standalone kernels over a list of limbs.
//
// Each warp-group of ER threads owns one row of W = ER^2 words. All global
// loads a thread needs (its row elements and the twiddles of its second
// register pass, which are specific to the thread) are issued before the
// first butterfly, so a warp waits for memory once instead of once per stage.
#pragma once
#include <type_traits>

#include "geo.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace ckks {

// Limb list of a row launch: launch index y -> (data limb index, prime id).
// Rule (no table): y = u * pl + r selects limb first + r of polynomial u,
// whose limbs start at data limb u * ps; that limb's extended index
// t = (first + r) % per is q_(base + t) for t < n, else p_(t - n) (base: the
// first prime of the level's window).
struct LimbMap {
  const int2* tab;  // explicit table, or null for the rule
  int first;
  int per, n, L;
  int pl = 1 << 30, ps = 0;
  int fixed = -1;   // >= 0: every limb uses this prime id
  int base = 0;
  int tail = 1 << 30, tail_prime = 0;  // launch limbs y >= tail: (y, tail_prime)
  // > 0: the launch's limbs are two polynomials of this many, taken limb by limb, so that what
  // both outputs of a limb read comes from memory once (HMult + rescale, level 39: 138.9 -> 137.2
  // us; without such operands it costs: HRot 119.1 -> 119.6, hoisted rotations 383 -> 389)
  int pairs = 0;
  // Launch limb of grid row b.
  __device__ __forceinline__ int limb(int b) const { return pairs ? (b & 1) * pairs + (b >> 1) : b; }
  __device__ __forceinline__ int2 operator()(int y) const {
    if (y >= tail) return make_int2(y, tail_prime);
    if (tab) return tab[y];
    const int u = y / pl, r = y % pl;
    const int t = (first + r) % per;
    return make_int2(u * ps + first + r, fixed >= 0 ? fixed : (t < n ? base + t : L + (t - n)));
  }
};

// Epilogues that read operands after the transform may name them up front
// (a method prefetch(dp, y, pos0)): the row kernel asks for them to be moved
// into L2 before it starts its passes, so the epilogue's loads find them there.
template <class Epi, class = void>
struct HasPrefetch : std::false_type {};
template <class Epi>
struct HasPrefetch<Epi, std::void_t<decltype(&Epi::prefetch)>> : std::true_type {};

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Register-resident twiddles of one pass: tw[(1 << s) - 1 + b] for local
// stage s and block b (2^s blocks).
template <int E, bool LAZY>
__device__ __forceinline__ void ct_pass_reg(uint32_t (&x)[E], const uint2 (&tw)[E - 1], uint32_t q) {
  constexpr int e = Log2<E>::v;
#pragma unroll
  for (int s = 0; s < e; ++s) {
    const int half = E >> (s + 1);
#pragma unroll
    for (int b = 0; b < (1 << s); ++b) {
      const uint2 w = tw[(1 << s) - 1 + b];
#pragma unroll
      for (int r = 0; r < half; ++r) {
        const int i0 = b * 2 * half + r;
        ct_bfly<LAZY>(x[i0], x[i0 + half], w.x, w.y, q);
      }
    }
  }
}

template <int E, bool LAZY>
__device__ __forceinline__ void gs_pass_reg(uint32_t (&x)[E], const uint2 (&tw)[E - 1], uint32_t q) {
  constexpr int e = Log2<E>::v;
#pragma unroll
  for (int s = e - 1; s >= 0; --s) {
    const int half = E >> (s + 1);
#pragma unroll
    for (int b = 0; b < (1 << s); ++b) {
      const uint2 w = tw[(1 << s) - 1 + b];
#pragma unroll
      for (int r = 0; r < half; ++r) {
        const int i0 = b * 2 * half + r;
        gs_bfly<LAZY>(x[i0], x[i0 + half], w.x, w.y, q);
      }
    }
  }
}

// First-pass twiddles of row h (the same for every thread of the row):
// local stage s, block b uses index (H + h) 2^s + b; the row's ER threads
// stage them in the row's own shared slice at (2^s - 1) + b and sync with a
// warp barrier (a row never spans two warps).
template <int E, int H>
__device__ __forceinline__ void stage_row_twiddles(uint2* sm, const uint2* __restrict__ t, int h, int jj) {
  for (int idx = jj; idx < E - 1; idx += E) {
    const int s = 31 - __clz(idx + 1);
    const int b = idx + 1 - (1 << s);
    sm[idx] = __ldg(t + ((uint32_t)(H + h) << s) + b);
  }
  __syncwarp();
}

template <int E, bool LAZY>
__device__ __forceinline__ void ct_pass_sm(uint32_t (&x)[E], const uint2* sm, uint32_t q) {
  constexpr int e = Log2<E>::v;
#pragma unroll
  for (int s = 0; s < e; ++s) {
    const int half = E >> (s + 1);
#pragma unroll
    for (int b = 0; b < (1 << s); ++b) {
      const uint2 w = sm[(1 << s) - 1 + b];
#pragma unroll
      for (int k = 0; k < half; ++k) {
        const int i0 = b * 2 * half + k;
        ct_bfly<LAZY>(x[i0], x[i0 + half], w.x, w.y, q);
      }
    }
  }
}

template <int E, bool LAZY>
__device__ __forceinline__ void gs_pass_sm(uint32_t (&x)[E], const uint2* sm, uint32_t q) {
  constexpr int e = Log2<E>::v;
#pragma unroll
  for (int s = e - 1; s >= 0; --s) {
    const int half = E >> (s + 1);
#pragma unroll
    for (int b = 0; b < (1 << s); ++b) {
      const uint2 w = sm[(1 << s) - 1 + b];
#pragma unroll
      for (int k = 0; k < half; ++k) {
        const int i0 = b * 2 * half + k;
        gs_bfly<LAZY>(x[i0], x[i0 + half], w.x, w.y, q);
      }
    }
  }
}

// Second-pass twiddles of thread jj in row h: indices ((H + h) E + jj) 2^s + b,
// contiguous for each stage, so stages s >= 1 load with 16-byte vectors.
template <int E, int H>
__device__ __forceinline__ void load_pass_b_twiddles(uint2 (&tw)[E - 1], const uint2* __restrict__ t, int h,
                                                     int jj) {
  constexpr int e = Log2<E>::v;
  const uint32_t base = (uint32_t)(H + h) * E + jj;
  tw[0] = __ldg(t + base);
#pragma unroll
  for (int s = 1; s < e; ++s) {
    const uint4* p = reinterpret_cast<const uint4*>(t + (base << s));
#pragma unroll
    for (int b2 = 0; b2 < (1 << (s - 1)); ++b2) {
      const uint4 v = __ldg(p + b2);
      tw[(1 << s) - 1 + 2 * b2] = make_uint2(v.x, v.y);
      tw[(1 << s) + 2 * b2] = make_uint2(v.z, v.w);
    }
  }
}

// Where a forward row phase puts its results, and where an inverse row phase
// gets its inputs. A thread holds E device positions of its row of launch
// limb y, whose data limb and prime are lm = map(y): E / 4 runs of four
// consecutive words, run c at pos0 + CS c. CS = 4 is the B layout (E
// consecutive words from pos0 = h W + E jj); CS = 128 is the warp's 512 words
// dealt out in 16-byte units, lane after lane, so that each access of a warp
// covers 512 consecutive bytes. The plain forms store to
// / load from a limb array; the key-switch kernels supply fused ones (input
// preparation before the iNTT, ModDown and rescale epilogues after the NTT).
// An epilogue's early() loads its first operand; the three-pass kernel calls it
// before the last pass, so that the load's latency passes behind it.
struct RowStore {
  uint32_t* dst;
  int compact;  // write launch limb y at dst + y N instead of at data limb lm.x
  template <int E, int CS>
  __device__ __forceinline__ void early(const DevParams&, uint32_t (&)[E], int, uint32_t) const {}
  template <int E, int CS>
  __device__ __forceinline__ void apply(const DevParams& dp, uint32_t (&x)[E], const uint32_t (&)[E], int y, int2 lm,
                                        uint32_t pos0) const {
    const size_t dl = compact ? (size_t)y : (size_t)lm.x;
    store_runs<E, CS>(dst + (dl << dp.log_n) + pos0, x);
  }
};

struct RowLoad {
  const uint32_t* src;
  template <int E, int CS>
  __device__ __forceinline__ void apply(const DevParams& dp, uint32_t (&x)[E], int, int2 lm, uint32_t pos0) const {
    load_runs<E, CS>(x, src + ((size_t)lm.x << dp.log_n) + pos0);
  }
};

// Forward row phase: src in A layout (column-phase output, natural
// positions); the epilogue receives the B-layout results normalized to
// [0, q). Launched with programmatic dependent launch: the twiddles are
// loaded before waiting for the previous kernel.
template <class G, class Epi>
__global__ void __launch_bounds__(G::RT) k_rows_fwd_t(DevParams dp, const uint32_t* src, Epi epi, LimbMap map) {
  __shared__ uint32_t buf[G::RPC * G::ROWBUF];
  __shared__ uint2 twa[G::RPC * (G::ER - 1)];
  const int r = threadIdx.x / G::ER, jj = threadIdx.x % G::ER;
  const int h = blockIdx.x * G::RPC + r;
  const int y = map.limb(blockIdx.y);
  const int2 lm = map(y);
  const uint32_t q = dp.pc[lm.y].q;
  const uint2* tw = dp.tw + ((size_t)lm.y << dp.log_n);
  uint2 twb[G::ER - 1];
  load_pass_b_twiddles<G::ER, G::H>(twb, tw, h, jj);
  uint2* tr = twa + r * (G::ER - 1);
  stage_row_twiddles<G::ER, G::H>(tr, tw, h, jj);
  pdl_wait();
  pdl_trigger();
  const uint32_t* s = src + ((size_t)lm.x << dp.log_n) + (size_t)h * G::W;
  uint32_t x[G::ER];
#pragma unroll
  for (int i = 0; i < G::ER; ++i) x[i] = s[jj + G::ER * i];
  uint32_t* b = buf + r * G::ROWBUF;
  if (q < (1u << 30)) {
    ct_pass_sm<G::ER, true>(x, tr, q);
    row_a_to_b<G::ER>(x, b, jj);
    ct_pass_reg<G::ER, true>(x, twb, q);
#pragma unroll
    for (int i = 0; i < G::ER; ++i) x[i] = normalize<true>(x[i], q);
  } else {
    ct_pass_sm<G::ER, false>(x, tr, q);
    row_a_to_b<G::ER>(x, b, jj);
    ct_pass_reg<G::ER, false>(x, twb, q);
#pragma unroll
    for (int i = 0; i < G::ER; ++i) x[i] = normalize<false>(x[i], q);
  }
  uint32_t op[G::ER];
  epi.template early<G::ER, 4>(dp, op, y, (uint32_t)(h * G::W + G::ER * jj));
  epi.template apply<G::ER, 4>(dp, x, op, y, lm, (uint32_t)(h * G::W + G::ER * jj));
}

// Inverse row phase: the source gives B-layout values in [0, q) (NTT domain);
// dst in A layout, lazy range [0, 2q) (the column phase that follows accepts
// it). dst_compact: write limb y at dst + y N instead of at data limb lm.x.
template <class G, class Src>
__global__ void __launch_bounds__(G::RT) k_rows_inv_t(DevParams dp, Src src, uint32_t* dst, LimbMap map,
                                                      int dst_compact) {
  __shared__ uint32_t buf[G::RPC * G::ROWBUF];
  __shared__ uint2 twa[G::RPC * (G::ER - 1)];
  const int r = threadIdx.x / G::ER, jj = threadIdx.x % G::ER;
  const int h = blockIdx.x * G::RPC + r;
  const int2 lm = map(blockIdx.y);
  const uint32_t q = dp.pc[lm.y].q;
  const uint2* itw = dp.itw + ((size_t)lm.y << dp.log_n);
  uint2 twb[G::ER - 1];
  load_pass_b_twiddles<G::ER, G::H>(twb, itw, h, jj);
  uint2* tr = twa + r * (G::ER - 1);
  stage_row_twiddles<G::ER, G::H>(tr, itw, h, jj);
  pdl_wait();
  pdl_trigger();
  uint32_t x[G::ER];
  src.template apply<G::ER, 4>(dp, x, (int)blockIdx.y, lm, (uint32_t)(h * G::W + G::ER * jj));
  uint32_t* b = buf + r * G::ROWBUF;
  if (q < (1u << 30)) {
    gs_pass_reg<G::ER, true>(x, twb, q);
    row_b_to_a<G::ER>(x, b, jj);
    gs_pass_sm<G::ER, true>(x, tr, q);
  } else {
    gs_pass_reg<G::ER, false>(x, twb, q);
    row_b_to_a<G::ER>(x, b, jj);
    gs_pass_sm<G::ER, false>(x, tr, q);
  }
  const size_t dl = dst_compact ? (size_t)blockIdx.y : (size_t)lm.x;
  uint32_t* o = dst + (dl << dp.log_n) + (size_t)h * G::W;
#pragma unroll
  for (int i = 0; i < G::ER; ++i) o[jj + G::ER * i] = x[i];
}

// ---------------------------------------------------------------------------
// Rows of W = 1024 words (N = 2^16) in three register passes of 4, 3 and 3
// stages on 64 threads per row, 16 values per thread, so that a thread keeps
// 16 values and 21 twiddle pairs (7 shared by its pass-B groups, 14 for its
// two pass-C groups) instead of 32 values and 31 pairs: twice the resident
// warps of the two-pass form. Element e of the row (0 .. 1023) sits at
//   A layout (pass A):  thread t, value i < 16:         e = t + 64 i
//   B layout (pass B):  thread t, group g < 2, i < 8:   e = 64 (t >> 2) + 8 i + 2 (t & 3) + g
//   C layout (pass C):  thread t, group g < 2, i < 8:   e = 16 t + 8 g + i
//   dealt-out layout:   thread t, run c < 4, k < 4:     e = 512 (t >> 5) + 128 c + 4 (t & 31) + k
// Forward stage k (0 .. 9 of the row) uses twiddle (H + h) 2^k + (e >> (10 - k));
// pass A's 15 depend on the row only and are staged in shared memory, pass B's
// on o = t >> 2 (base (H + h) 16 + o), pass C's on the group (base (H + h) 128
// + 2 t + g; read from a copy of the table in the order the threads take them).
//
// Transposes go through one padded buffer per row, element e at word e + 8
// (e >> 6) + 4 ((e >> 5) & 1): 32-bit accesses in A, 64-bit in B, 128-bit in C
// and dealt out are all conflict-free, and a thread's accesses of a layout
// differ by constants (no address arithmetic; an XOR swizzle with 32-bit
// accesses took one operation per element and 64 accesses instead of 44).
// Global memory is read and written in A or dealt out, whole 128- and 512-byte
// runs per access of a warp: with the C layout's 16 consecutive words per
// thread each 16-byte access touched 32 sectors and used half of each.
//
// Launch bounds, forward: 12 blocks of 2 warps per SM (80 registers), 24 resident
// warps, against 16 for the two-pass form at 128 registers (14 blocks: 17.6 us
// for the ModUp rows of two-row blocks, 10: 18.6; HRot level 39 118.8 us at 12,
// 121.0 at 10). Inverse: 10 blocks (96 registers), whose sources keep more loads
// in flight (HMult + rescale level 39 136.5 us at 12, 134.9 at 10, 9 and 8; level 20
// 78.3, 76.8; the 25-30 system's level 6 57.9, 56.6).
//
// Bound and figures (ModUp rows at the top level, 40 primes, dnum = 3, 122
// limbs, launched back to back): 24.4 us with the XOR swizzle, table-order
// twiddles and strided stores (21.2 with the shorter butterflies and whole-run
// stores) -> 16.5; 32 MB in, 32 MB out and 62 MB of twiddles, all in L2. A warp
// issues in half the cycles; loads from L2 are the largest stall, the multiply
// pipe is half busy. Whole operations: HRot 133.3 -> 122.0 us, HMult + rescale
// 153.1 -> 140.1.
// ---------------------------------------------------------------------------

constexpr int kRow3Words = 1152;
__device__ __forceinline__ int row3_a(int t) { return t + 4 * (t >> 5); }                  // + 72 i
__device__ __forceinline__ int row3_b(int t) { return 72 * (t >> 2) + 2 * (t & 3); }      // + 8 i + 4 (i >> 2) + g
__device__ __forceinline__ int row3_c(int t) { return 72 * (t >> 2) + 16 * (t & 3) + 4 * ((t >> 1) & 1); }  // + 8 g + i
__device__ __forceinline__ int row3_dealt(int t) { return 512 * (t >> 5) + 4 * (t & 31); }  // element of run 0
__device__ __forceinline__ int row3_d(int t) {                                            // + 144 c
  const int e = row3_dealt(t);
  return e + 8 * (e >> 6) + 4 * ((e >> 5) & 1);
}

__device__ __forceinline__ void row3_put_a(uint32_t* b, int t, const uint32_t (&x)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) b[row3_a(t) + 72 * i] = x[i];
}
__device__ __forceinline__ void row3_get_a(const uint32_t* b, int t, uint32_t (&x)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) x[i] = b[row3_a(t) + 72 * i];
}
__device__ __forceinline__ void row3_put_b(uint32_t* b, int t, const uint32_t (&y0)[8], const uint32_t (&y1)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<uint2*>(b + row3_b(t) + 8 * i + 4 * (i >> 2)) = make_uint2(y0[i], y1[i]);
}
__device__ __forceinline__ void row3_get_b(const uint32_t* b, int t, uint32_t (&y0)[8], uint32_t (&y1)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint2 v = *reinterpret_cast<const uint2*>(b + row3_b(t) + 8 * i + 4 * (i >> 2));
    y0[i] = v.x;
    y1[i] = v.y;
  }
}
// Four 16-byte units from word `at`, STEP words apart.
template <int STEP>
__device__ __forceinline__ void row3_put4(uint32_t* at, const uint32_t (&x)[16]) {
#pragma unroll
  for (int c = 0; c < 4; ++c)
    *reinterpret_cast<uint4*>(at + STEP * c) = make_uint4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
}
template <int STEP>
__device__ __forceinline__ void row3_get4(const uint32_t* at, uint32_t (&x)[16]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint4 v = *reinterpret_cast<const uint4*>(at + STEP * c);
    x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
  }
}
__device__ __forceinline__ void row3_split(const uint32_t (&x)[16], uint32_t (&y0)[8], uint32_t (&y1)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    y0[i] = x[i];
    y1[i] = x[8 + i];
  }
}

// Pass-B twiddles of thread t in row h: local stage s, block b at entry
// (2^s - 1) + b, global index base 2^s + b.
template <int H>
__device__ __forceinline__ void row3_twiddles_b(uint2 (&tb)[7], const uint2* __restrict__ t, int h, int tid) {
  const uint32_t bb = (uint32_t)(H + h) * 16 + (tid >> 2);
  tb[0] = __ldg(t + bb);
  {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(t + 2 * bb));
    tb[1] = make_uint2(v.x, v.y);
    tb[2] = make_uint2(v.z, v.w);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(t + 4 * bb) + k);
    tb[3 + 2 * k] = make_uint2(v.x, v.y);
    tb[4 + 2 * k] = make_uint2(v.z, v.w);
  }
}

// Pass-C twiddles of thread t in row h, from the table in thread order
// (DevParams::twc / itwc): unit k of thread t at (h 7 + k) 64 + t, unit 0 =
// stage 0 of groups 0 and 1, 1 + g = stage 1 of group g, 3 + 2g and 4 + 2g =
// stage 2 of group g. Whole 512-byte runs per access; in table order the
// accesses of stages 1 and 2 were 32 and 64 bytes apart (84 instead of 28
// 128-byte lines per warp).
__device__ __forceinline__ void row3_twiddles_c(uint2 (&tc)[2][7], const uint4* __restrict__ t, int h, int tid) {
  uint4 v[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) v[k] = __ldg(t + (h * 7 + k) * 64 + tid);
  tc[0][0] = make_uint2(v[0].x, v[0].y);
  tc[1][0] = make_uint2(v[0].z, v[0].w);
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    tc[g][1] = make_uint2(v[1 + g].x, v[1 + g].y);
    tc[g][2] = make_uint2(v[1 + g].z, v[1 + g].w);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      tc[g][3 + 2 * k] = make_uint2(v[3 + 2 * g + k].x, v[3 + 2 * g + k].y);
      tc[g][4 + 2 * k] = make_uint2(v[3 + 2 * g + k].z, v[3 + 2 * g + k].w);
    }
  }
}

// Pass-A twiddles of row h (15 entries, shared by its 64 threads).
template <int H>
__device__ __forceinline__ void row3_stage_a(uint2* sm, const uint2* __restrict__ t, int h, int tid) {
  if (tid < 15) {
    const int s = 31 - __clz(tid + 1);
    const int b = tid + 1 - (1 << s);
    sm[tid] = __ldg(t + ((uint32_t)(H + h) << s) + b);
  }
}

constexpr int kRow3Rows = 1;  // rows per block (two: ModUp rows 17.4 us, one: 16.5; the barriers join fewer warps)

template <class G, class Epi>
__global__ void __launch_bounds__(64 * kRow3Rows, 12 / kRow3Rows)
    k_rows3_fwd_t(DevParams dp, const uint32_t* src, Epi epi, LimbMap map) {
  static_assert(G::W == 1024, "three-pass rows are for W = 1024");
  __shared__ __align__(16) uint32_t buf[kRow3Rows][kRow3Words];
  __shared__ uint2 twa[kRow3Rows][15];
  const int r = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int h = blockIdx.x * kRow3Rows + r;
  const int y = map.limb(blockIdx.y);
  const int2 lm = map(y);
  const uint32_t q = dp.pc[lm.y].q;
  const uint2* tw = dp.tw + ((size_t)lm.y << dp.log_n);
  uint2 tb[7], tc[2][7];
  row3_twiddles_b<G::H>(tb, tw, h, t);
  row3_twiddles_c(tc, dp.twc + (size_t)lm.y * (G::H * 448), h, t);
  row3_stage_a<G::H>(twa[r], tw, h, t);
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const uint32_t pos = (uint32_t)(h * 1024 + row3_dealt(t));
  if constexpr (HasPrefetch<Epi>::value) epi.prefetch(dp, y, (uint32_t)(h * 1024 + 16 * t));
  const uint32_t* s = src + ((size_t)lm.x << dp.log_n) + (size_t)h * 1024;
  uint32_t x[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) x[i] = s[t + 64 * i];
  uint32_t* b = buf[r];
  uint32_t y0[8], y1[8];
  const bool lazy = q < (1u << 30);
  if (lazy) ct_pass_sm<16, true>(x, twa[r], q);
  else ct_pass_sm<16, false>(x, twa[r], q);
  row3_put_a(b, t, x);
  __syncthreads();
  row3_get_b(b, t, y0, y1);
  if (lazy) {
    ct_pass_reg<8, true>(y0, tb, q);
    ct_pass_reg<8, true>(y1, tb, q);
  } else {
    ct_pass_reg<8, false>(y0, tb, q);
    ct_pass_reg<8, false>(y1, tb, q);
  }
  row3_put_b(b, t, y0, y1);  // where the thread read them
  uint32_t op[16];
  epi.template early<16, 128>(dp, op, y, pos);
  __syncthreads();
  row3_get4<4>(b + row3_c(t), x);
  row3_split(x, y0, y1);
  if (lazy) {
    ct_pass_reg<8, true>(y0, tc[0], q);
    ct_pass_reg<8, true>(y1, tc[1], q);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = normalize<true>(y0[i], q);
      x[8 + i] = normalize<true>(y1[i], q);
    }
  } else {
    ct_pass_reg<8, false>(y0, tc[0], q);
    ct_pass_reg<8, false>(y1, tc[1], q);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = normalize<false>(y0[i], q);
      x[8 + i] = normalize<false>(y1[i], q);
    }
  }
  // deal out: C layout and dealt-out runs stay in the warp's half of the row
  row3_put4<4>(b + row3_c(t), x);
  __syncwarp();
  row3_get4<144>(b + row3_d(t), x);
  epi.template apply<16, 128>(dp, x, op, y, lm, pos);
}

template <class G, class Src>
__global__ void __launch_bounds__(64 * kRow3Rows, 10 / kRow3Rows)
    k_rows3_inv_t(DevParams dp, Src src, uint32_t* dst, LimbMap map, int dst_compact) {
  static_assert(G::W == 1024, "three-pass rows are for W = 1024");
  __shared__ __align__(16) uint32_t buf[kRow3Rows][kRow3Words];
  __shared__ uint2 twa[kRow3Rows][15];
  const int r = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int h = blockIdx.x * kRow3Rows + r;
  const int2 lm = map(blockIdx.y);
  const uint32_t q = dp.pc[lm.y].q;
  const uint2* itw = dp.itw + ((size_t)lm.y << dp.log_n);
  uint2 tb[7], tc[2][7];
  row3_twiddles_c(tc, dp.itwc + (size_t)lm.y * (G::H * 448), h, t);
  row3_stage_a<G::H>(twa[r], itw, h, t);
  pdl_wait();
  pdl_trigger();
  uint32_t x[16];
  src.template apply<16, 128>(dp, x, (int)blockIdx.y, lm, (uint32_t)(h * 1024 + row3_dealt(t)));
  uint32_t* b = buf[r];
  row3_put4<144>(b + row3_d(t), x);
  row3_twiddles_b<G::H>(tb, itw, h, t);  // not before the sources' loads: registers
  __syncwarp();
  row3_get4<4>(b + row3_c(t), x);
  uint32_t y0[8], y1[8];
  row3_split(x, y0, y1);
  const bool lazy = q < (1u << 30);
  if (lazy) {
    gs_pass_reg<8, true>(y0, tc[0], q);
    gs_pass_reg<8, true>(y1, tc[1], q);
  } else {
    gs_pass_reg<8, false>(y0, tc[0], q);
    gs_pass_reg<8, false>(y1, tc[1], q);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    x[i] = y0[i];
    x[8 + i] = y1[i];
  }
  row3_put4<4>(b + row3_c(t), x);  // where the thread read them
  __syncthreads();
  row3_get_b(b, t, y0, y1);
  if (lazy) {
    gs_pass_reg<8, true>(y0, tb, q);
    gs_pass_reg<8, true>(y1, tb, q);
  } else {
    gs_pass_reg<8, false>(y0, tb, q);
    gs_pass_reg<8, false>(y1, tb, q);
  }
  row3_put_b(b, t, y0, y1);
  __syncthreads();
  row3_get_a(b, t, x);
  if (lazy) gs_pass_sm<16, true>(x, twa[r], q);
  else gs_pass_sm<16, false>(x, twa[r], q);
  const size_t dl = dst_compact ? (size_t)blockIdx.y : (size_t)lm.x;
  uint32_t* o = dst + (dl << dp.log_n) + (size_t)h * 1024;
#pragma unroll
  for (int i = 0; i < 16; ++i) o[t + 64 * i] = x[i];
}

// At N = 2^16 rows_passes = 2 selects the two-pass kernels, anything else the
// three-pass ones.
template <class G, class Epi>
inline void launch_rows_fwd(const DevParams& dp, const uint32_t* src, const Epi& epi, int limbs, LimbMap map,
                            cudaStream_t st) {
  if (limbs <= 0) return;
  count_launch(1);
  if constexpr (G::W == 1024) {
    if (dp.rows_passes != 2) {
      launch_pdl(dp.pdl, k_rows3_fwd_t<G, Epi>, dim3(G::H / kRow3Rows, limbs), dim3(64 * kRow3Rows), 0, st, dp, src,
                 epi, map);
      return;
    }
  }
  launch_pdl(dp.pdl, k_rows_fwd_t<G, Epi>, dim3(G::H / G::RPC, limbs), dim3(G::RT), 0, st, dp, src, epi, map);
}

template <class G, class Src>
inline void launch_rows_inv(const DevParams& dp, const Src& srcf, uint32_t* dst, int limbs, LimbMap map,
                            bool dst_compact, cudaStream_t st) {
  if (limbs <= 0) return;
  count_launch(1);
  if constexpr (G::W == 1024) {
    if (dp.rows_passes != 2) {
      launch_pdl(dp.pdl, k_rows3_inv_t<G, Src>, dim3(G::H / kRow3Rows, limbs), dim3(64 * kRow3Rows), 0, st, dp, srcf,
                 dst, map, dst_compact ? 1 : 0);
      return;
    }
  }
  launch_pdl(dp.pdl, k_rows_inv_t<G, Src>, dim3(G::H / G::RPC, limbs), dim3(G::RT), 0, st, dp, srcf, dst, map,
             dst_compact ? 1 : 0);
}

template <class G>
inline void launch_rows_g(const DevParams& dp, bool inverse, const uint32_t* src, uint32_t* dst, int limbs,
                          LimbMap map, bool dst_compact, cudaStream_t st) {
  if (inverse) launch_rows_inv<G>(dp, RowLoad{src}, dst, limbs, map, dst_compact, st);
  else launch_rows_fwd<G>(dp, src, RowStore{dst, dst_compact ? 1 : 0}, limbs, map, st);
}

}  // namespace ckks
