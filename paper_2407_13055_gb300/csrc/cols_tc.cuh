// Column kernels with the BConv on the tensor cores (tcgen05, kind::f16).
//
// The column phase of a ModSwitch (iNTT columns -> BConv, Eq. 2 -> NTT
// columns, Alg. 1) on tiles of 16 columns x 64 rows = 1024 coefficients. On
// CUDA cores the BConv costs K multiply-adds of 32 x 32 + 64 bits per output
// (5 issue cycles each, 70 for K = 14); here the conversion of a tile to four
// targets is one exact matrix product (tc.cuh) of the sources' byte digits
// (A, M = coefficients, K = 4 digits per source) with the matrix's byte planes
// (B, N = 4 planes per target), whose four plane sums become a residue in 10
// to 15 instructions.
//
// Layout. Thread p of a warpgroup is TMEM lane p: a pair of warps holds 8
// columns c and the 8 row offsets jj; M tile i (of 8) holds the rows jj + 8 i. That is the
// register layout between a column's two radix-8 passes, so a thread moves its
// 8 coefficients between registers and tensor memory without any exchange:
// the iNTT columns end with tcgen05.st of the digits into A (tensor memory
// columns 0-255: 32 per M tile), and a target's plane sums arrive with
// tcgen05.ld as the input of its first NTT pass. Shared memory holds only the
// transposes between the passes, the matrix planes and the column twiddles.
//
// Roles. Five warpgroups split the sources and then the targets (products come
// in groups of four targets); four more warps issue the products, two groups
// of targets ahead (two D buffers of 128 tensor-memory columns), and one of
// them brings in the planes and twiddles of the next segment with bulk copies. The warpgroups never meet at a block barrier; mbarriers order
// A (written by all), D full (products done) and D empty (sums read).
//
// Work. One block per SM (a block takes all 512 tensor-memory columns). The
// (tile, conversion) items are cut so that every block has the same work, an
// item's second part costing its sources once more (tc_plan in host.cu, made
// once per level): whole items would leave SMs idle at most levels (192 items
// on 152 SMs at 40 limbs, three digits).
//
// Bound and figures (N = 2^16, 40 primes, dnum = 3, top level; one kernel after
// another, GB300): ModUp columns 44.7 us on CUDA cores in their best shape ->
// 29.3, ModDown 32 -> 19.2, fused rescale 32.4 -> 21.2. A ModUp block issues in
// 62% of its cycles; half of that is the butterflies, a quarter the sources'
// digits and the plane sums' residues. The tensor pipe is active in 6%. Five
// warpgroups at 80 registers measured as four at 96 and seven at 64 (29.3 -
// 31.3 us): the instruction rate bounds it, and per block its start (about
// 3000 cycles) and the first product of each segment.
//
// Every mbarrier wait is bounded. When one expires the block records the
// timeout in dp.status, skips all further waits and starts no further copy (a
// segment buffer's barrier takes one copy group at a time): its results are
// undefined but no address depends on them, and it ends after its own products
// and copies (bounded again); the host reports CKKS_ETIMEOUT at the next
// synchronizing call.
#pragma once
#include "tc.cuh"

namespace ckks {

// Largest source count of the tensor-core kernels (K extent 64).
constexpr int kTcMaxSources = 16;
// Targets per segment (shared-memory room for their planes and twiddles).
constexpr int kTcCap = 56;
// Cycles any wait on a block's own copies and products may take at least
// (about 8 ms) where the shape was not set by hand: they end in microseconds,
// whatever dp.wait_limit asks for waits on the host.
constexpr long long kTcWaitFloor = 1ll << 24;
constexpr long long kTcDrainLimit = 1ll << 32;

constexpr int kTcColumns = 16;
constexpr int kTcMaxGroups = 8;  // conversions of a launch (ModUp digits)
constexpr int kTcMmaWarps = 4;   // one per scheduler
constexpr int kTcThreads = (kTcWarpgroups * 4 + kTcMmaWarps) * 32;
constexpr uint32_t kTcTrWords = 72 * 8;  // transpose buffer of two warps
constexpr uint32_t kTcRecBytes = 544;
static_assert(sizeof(TcSrcRec) == kTcRecBytes && sizeof(TcTgtRec) == kTcRecBytes && offsetof(TcSrcRec, prime) == 512 &&
                  offsetof(TcTgtRec, tw) == 32,
              "records");

// K extent of the product for K sources: four digits each, in steps of 16
// (one kind::f16 instruction).
__host__ __device__ inline int tc_kr(int K) { return 16 * ((K + 3) / 4); }

// One conversion (a ModUp digit, or a polynomial of a ModDown or rescaling):
// K sources (limb k step of src) with primes id0 + k (or idtab[k].y) and input
// constants cin[k], to M targets. Target m is limb t = m, or m + skip from m =
// lo on (a digit's own limbs are left out): limb t at dst + t N, prime base + t
// for t < n, else L + t - n. img is the matrix's plane image. With top (ModDown
// fused with rescaling, TOP below) source K - 1 is made inside the tile: the
// top limb's ModDown output, from the P limbs' conversion to q_l (the image's
// first group of targets) and E at top; its prime is id M
// (top_limb_sources in cols.cuh has the algebra).
struct TcGroup {
  const uint32_t* src;
  const uint2* cin;
  const uint8_t* img;
  const int2* idtab;
  const uint32_t* top;
  uint32_t* dst;
  int K, M, id0, lo, skip;
  int step = 1;  // source k's limb is k step limbs behind src
  __device__ __forceinline__ int id(int k) const { return idtab ? idtab[k].y : id0 + k; }
};
// Block boundaries of a launch (kTcMaxBlocks blocks at most).
struct TcPlan {
  uint32_t at[kTcMaxBlocks + 1];
};
struct TcJob {
  int n, base;
  TcGroup g[kTcMaxGroups];
  __device__ __forceinline__ int limb(const TcGroup& u, int m) const { return m < u.lo ? m : m + u.skip; }
  __device__ __forceinline__ int prime(const DevParams& dp, int t) const { return t < n ? base + t : dp.L + t - n; }
};

// A piece of work: targets m0 .. m1 - 1 of tile `tile` in conversion g (m1 may
// pass the last target: groups of four are padded).
struct TcSeg {
  int g, tile, m0, m1;
};

// Segments of one block: plan[b] .. plan[b + 1] are positions item * 256 + m / 4
// (tc_plan in host.cu), item = g * tiles + tile; at most cap targets each.
struct TcIter {
  uint32_t pos, end;
  __device__ __forceinline__ TcIter(const TcPlan& plan, int b) : pos(plan.at[b]), end(plan.at[b + 1]) {}
  template <class Job>
  __device__ __forceinline__ bool next(const Job& job, int tiles, int cap, TcSeg& sg) {
    if (pos >= end) return false;
    const int item = pos >> 8;
    sg.g = item / tiles;
    sg.tile = item % tiles;
    sg.m0 = 4 * (int)(pos & 255u);
    sg.m1 = (end >> 8) == (uint32_t)item ? 4 * (int)(end & 255u) : (job.g[sg.g].M + 3) & ~3;
    if (sg.m1 - sg.m0 > cap) sg.m1 = sg.m0 + cap;
    pos = sg.m1 >= job.g[sg.g].M ? (uint32_t)(item + 1) << 8 : (uint32_t)item << 8 | (uint32_t)(sg.m1 / 4);
    return true;
  }
};

// Shared-memory layout (byte offsets): transposes, two segment buffers
// (planes, source twiddles, target twiddles), barriers.
struct TcLayout {
  uint32_t seg, seg_bytes, srec, trec, bar, total;
};
inline TcLayout tc_layout(int cap, int kr) {
  TcLayout s;
  s.seg = kTcWarpgroups * 2 * 2 * kTcTrWords * 4;
  s.srec = (uint32_t)(cap + 4) * 4u * kr * 2u;
  s.trec = s.srec + kTcMaxSources * kTcRecBytes;
  s.seg_bytes = s.trec + (uint32_t)cap * kTcRecBytes;
  s.bar = s.seg + 2 * s.seg_bytes;
  s.total = s.bar + 8 * 8 + 8;
  return s;
}

// Radix-8 pass with the twiddles of its block o in shared memory (the prime's
// table from entry 0): stage s, block b at entry (o << s) + b.
struct Tw8 {
  uint2 w[7];
  __device__ __forceinline__ Tw8(const uint2* tw, int o) {
    w[0] = tw[o];
    const uint4 a = *reinterpret_cast<const uint4*>(tw + 2 * o);
    const uint4 b = *reinterpret_cast<const uint4*>(tw + 4 * o);
    const uint4 c = *reinterpret_cast<const uint4*>(tw + 4 * o + 2);
    w[1] = make_uint2(a.x, a.y);
    w[2] = make_uint2(a.z, a.w);
    w[3] = make_uint2(b.x, b.y);
    w[4] = make_uint2(b.z, b.w);
    w[5] = make_uint2(c.x, c.y);
    w[6] = make_uint2(c.z, c.w);
  }
};
template <bool LAZY>
__device__ __forceinline__ void ct8(uint32_t (&x)[8], const uint2* tw, int o, uint32_t q) {
  const Tw8 t(tw, o);
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int half = 4 >> s;
#pragma unroll
    for (int b = 0; b < (1 << s); ++b)
#pragma unroll
      for (int r = 0; r < half; ++r)
        ct_bfly<LAZY>(x[2 * half * b + r], x[2 * half * b + r + half], t.w[(1 << s) - 1 + b].x, t.w[(1 << s) - 1 + b].y, q);
  }
}
template <bool LAZY>
__device__ __forceinline__ void gs8(uint32_t (&x)[8], const uint2* tw, int o, uint32_t q) {
  const Tw8 t(tw, o);
#pragma unroll
  for (int s = 2; s >= 0; --s) {
    const int half = 4 >> s;
#pragma unroll
    for (int b = 0; b < (1 << s); ++b)
#pragma unroll
      for (int r = 0; r < half; ++r)
        gs_bfly<LAZY>(x[2 * half * b + r], x[2 * half * b + r + half], t.w[(1 << s) - 1 + b].x, t.w[(1 << s) - 1 + b].y, q);
  }
}

// Transpose of the 8 columns of two warps between rows jj + 8 i and 8 jj + i.
// Two buffers in turn: one barrier (of 64 threads) per transpose; a buffer is
// written again two transposes later, after a barrier that every thread
// reaches with its reads done.
struct TcTranspose {
  uint32_t* buf;
  int bar, flip = 0;
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory"); }
  __device__ __forceinline__ void a_to_b(uint32_t (&x)[8], int jj, int c) {
    uint32_t* b = buf + flip * kTcTrWords + c;
    flip ^= 1;
#pragma unroll
    for (int i = 0; i < 8; ++i) b[(jj + 9 * i) * 8] = x[i];
    sync();
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = b[(9 * jj + i) * 8];
  }
  __device__ __forceinline__ void b_to_a(uint32_t (&x)[8], int jj, int c) {
    uint32_t* b = buf + flip * kTcTrWords + c;
    flip ^= 1;
#pragma unroll
    for (int i = 0; i < 8; ++i) b[(9 * jj + i) * 8] = x[i];
    sync();
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = b[(jj + 9 * i) * 8];
  }
};

__device__ __forceinline__ TcPrime load_tc_prime(const uint8_t* p) {
  const uint4 a = *reinterpret_cast<const uint4*>(p), b = *reinterpret_cast<const uint4*>(p + 16);
  return TcPrime{a.x, a.y, a.z, a.w, b.x, b.y, 0u, 0u};
}

// Residue of one output from its four plane sums, in the range the forward
// butterflies take ([0, 4q) for q < 2^30, [0, 2q) above). Adding 1.5 2^23
// puts P + 0x4B400000 in the float's bit pattern; A = P_0 + 2^8 P_1 and B =
// P_2 + 2^8 P_3 fit 32 bits (|A|, |B| < 2^28) and the value is A + 2^16 B mod
// q: Shoup's product of B (made positive) by 2^16, with the constants that
// undo the biases folded into ea and eb (host.cu).
template <int MODE>
__device__ __forceinline__ uint32_t tc_residue(const uint32_t* f, const TcPrime& P) {
  const float kMagic = 12582912.0f;
  uint32_t v[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) v[b] = __float_as_uint(__fadd_rn(__uint_as_float(f[b]), kMagic));
  uint32_t A = v[0] + (v[1] << 8) + P.ea, B = v[2] + (v[3] << 8);
  if (MODE == 0) return A + B * P.c - __umulhi(B, P.csh) * P.q;  // 2^29 <= q < 2^30
  B += P.eb;
  const uint32_t t = B * P.c - __umulhi(B, P.csh) * P.q;
  if (MODE == 1) return csub(t, P.q) + min(A, A + P.q);  // q > 2^30: |A| < q / 4
  return t + A - __umulhi(A, P.inv) * P.q;  // q < 2^29: A reduced as well
}

// A group of four targets, two M tiles: KS steps of 16 along K.
template <int KS>
__device__ __forceinline__ void tc_product(uint32_t d, uint32_t a, uint64_t b) {
  constexpr uint32_t idesc = tc::idesc_f16(128, 16);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    tc::mma_f16_ts<false>(d + i * 16, a + i * 32, b, idesc);
#pragma unroll
    for (int s = 1; s < KS; ++s) tc::mma_f16_ts<true>(d + i * 16, a + i * 32 + s * 8, b + 16 * s, idesc);
  }
}

template <class G, bool TOP>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_cols_tc(const __grid_constant__ DevParams dp, const __grid_constant__ TcJob job,
              const __grid_constant__ TcPlan plan, int cap, TcLayout lay) {
  static_assert(G::EC == 8 && G::H == 64, "column tiles are two radix-8 passes");
  extern __shared__ __align__(1024) uint8_t sm[];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t bars = tc::smem_u32(sm + lay.bar);
  auto b_ld = [&](int i) { return bars + 8u * i; };
  auto b_full = [&](int i) { return bars + 16u + 8u * i; };
  auto b_empty = [&](int i) { return bars + 32u + 8u * i; };
  const uint32_t b_a = bars + 48u, b_done = bars + 56u;
  volatile uint32_t* slot = reinterpret_cast<volatile uint32_t*>(sm + lay.bar + 64);
  volatile uint32_t* flag = reinterpret_cast<volatile uint32_t*>(sm + lay.bar + 68);
  const long long limit = dp.wait_limit;
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (!tc::mbar_try(bar, parity) && !*flag && !tc::mbar_wait(bar, parity, limit)) {
      *flag = 1;
      tc::report_timeout(dp.status);
    }
  };
  // The products' wait for the sources, which takes a block's longest: a limit
  // below kPollLimit expires here, before the blocking try.
  auto wait_sources = [&](uint32_t parity) {
    if (!*flag && !tc::mbar_wait(b_a, parity, limit)) {
      *flag = 1;
      tc::report_timeout(dp.status);
    }
  };

  constexpr int tiles = G::W / kTcColumns;
  TcIter iter(plan, blockIdx.x);
  TcSeg seg;
  bool have = iter.next(job, tiles, cap, seg);

  if (warp >= kTcWarpgroups * 4) {
    // ---- the warps of copies and products: each issues the products of two M
    // tiles, so that a group's 32 products do not wait for one warp's share of
    // its scheduler (1400 cycles a group beside five busy warps); the first
    // also brings in the segments' tables
    const int mw = warp - kTcWarpgroups * 4;
    if (mw == 0) {
      tc::tmem_alloc(tc::smem_u32(const_cast<uint32_t*>(slot)), 512);
      if (lane == 0) {
        for (int i = 0; i < 2; ++i) {
          tc::mbar_init(b_ld(i), 1);
          tc::mbar_init(b_full(i), kTcMmaWarps);
          tc::mbar_init(b_empty(i), 16);  // the warps of four targets
        }
        tc::mbar_init(b_a, kTcWarpgroups * 4);
        tc::mbar_init(b_done, kTcMmaWarps);
        tc::mbar_init_fence();
        *flag = 0;
      }
      __syncwarp();
    }
    auto load = [&](const TcSeg& sg, int bf) {
      const TcGroup& it = job.g[sg.g];
      const int kr = tc_kr(it.K), m1 = min(sg.m1, it.M);
      const uint32_t dst = tc::smem_u32(sm + lay.seg + bf * lay.seg_bytes);
      // image groups of four targets: [top group,] then the segment's
      const uint32_t gb = (uint32_t)kr * 32u, top = TOP ? gb : 0u;
      const uint32_t pb = (uint32_t)((m1 - sg.m0 + 3) / 4) * gb;
      tc::mbar_expect_tx(b_ld(bf), top + pb + (uint32_t)(it.K + m1 - sg.m0) * kTcRecBytes);
      // sources: one run of primes, or one by one; the top limb is prime n - 1 = M
      const int Kp = it.K - (TOP ? 1 : 0);
      if (it.idtab)
        for (int k = 0; k < Kp; ++k)
          tc::bulk_g2s(dst + lay.srec + k * kTcRecBytes, dp.ks.tc_src + it.id(k), kTcRecBytes, b_ld(bf));
      else
        tc::bulk_g2s(dst + lay.srec, dp.ks.tc_src + it.id0, Kp * kTcRecBytes, b_ld(bf));
      if (TOP) {
        tc::bulk_g2s(dst + lay.srec + Kp * kTcRecBytes, dp.ks.tc_src + it.M, kTcRecBytes, b_ld(bf));
        tc::bulk_g2s(dst, it.img, gb, b_ld(bf));
      }
      tc::bulk_g2s(dst + top, it.img + top + (size_t)(sg.m0 / 4) * gb, pb, b_ld(bf));
      // targets: runs of consecutive primes (broken at the digit's own limbs
      // and where the auxiliary primes begin)
      for (int m = sg.m0; m < m1;) {
        const int t = job.limb(it, m);
        int run = m1 - m;
        if (m < it.lo) run = min(run, it.lo - m);
        if (t < job.n) run = min(run, job.n - t);
        tc::bulk_g2s(dst + lay.trec + (m - sg.m0) * kTcRecBytes, dp.ks.tc_tgt + job.prime(dp, t), run * kTcRecBytes,
                     b_ld(bf));
        m += run;
      }
    };
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    int loads = 0;  // of the lane that loads
    if (have && mw == 0 && lane == 0) {
      load(seg, 0);
      ++loads;
    }
    __syncwarp();
    const uint32_t tmem = *slot;
    int it_no = 0, gc = 0, a_no = 0;
    while (have) {
      TcSeg nx;
      const bool more = iter.next(job, tiles, cap, nx);
      const TcGroup& it = job.g[seg.g];
      const int kr = tc_kr(it.K);
      const uint32_t sbo = (uint32_t)kr * 16u, gb = (uint32_t)kr * 32u;
      uint32_t b0 = tc::smem_u32(sm + lay.seg + (it_no & 1) * lay.seg_bytes);
      wait(b_ld(it_no & 1), (it_no >> 1) & 1);
      wait_sources(a_no & 1);
      ++a_no;
      tc::fence_after_sync();
      // every warpgroup is past the previous segment: its buffer is free (with
      // the flag down, the waits so far, that for the buffer's last copies
      // among them, ended by completion)
      if (more && mw == 0 && lane == 0 && !*flag) {
        load(nx, (it_no + 1) & 1);
        ++loads;
      }
      __syncwarp();
      auto product = [&]() {
        if (gc >= 2) {
          wait(b_empty(gc & 1), ((gc >> 1) - 1) & 1);
          tc::fence_after_sync();
        }
        const uint32_t d = tmem + 256 + (gc & 1) * 128 + mw * 32, a = tmem + mw * 64;
        const uint64_t bd = tc::sdesc(b0, 128, sbo);
        switch (kr) {
          case 16: tc_product<1>(d, a, bd); break;
          case 32: tc_product<2>(d, a, bd); break;
          case 48: tc_product<3>(d, a, bd); break;
          default: tc_product<4>(d, a, bd); break;
        }
        tc::commit(b_full(gc & 1));
        b0 += gb;
        ++gc;
      };
      if constexpr (TOP) {
        product();
        wait_sources(a_no & 1);
        ++a_no;
        tc::fence_after_sync();
      }
      const int ng = (min(seg.m1, it.M) - seg.m0 + 3) / 4;
      for (int g = 0; g < ng; ++g) product();
      ++it_no;
      seg = nx;
      have = more;
    }
    // the block ends after all its products and copies, after a timeout too
    tc::commit(b_done);
    if (lane == 0) {
      tc::mbar_wait(b_done, 0, kTcDrainLimit);
      for (int u = loads < 2 ? 0 : loads - 2; u < loads; ++u) tc::mbar_wait(b_ld(u & 1), (u >> 1) & 1, kTcDrainLimit);
    }
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (mw == 0) tc::tmem_dealloc(tmem, 512);
    return;
  }

  // ---- the warpgroups
  const int wg = warp >> 2, jj = (lane >> 3) + 4 * (warp & 1), ct = lane & 7, c = ct + 8 * ((warp >> 1) & 1);
  TcTranspose tr{reinterpret_cast<uint32_t*>(sm) + (warp >> 1) * 2 * kTcTrWords, (warp >> 1) + 1};
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *slot;
  const uint32_t lanes = tmem + ((uint32_t)(warp & 3) << 21);  // this warp's lane quadrant
  pdl_wait();
  pdl_trigger();
  auto arrive = [&](uint32_t bar) {
    tc::fence_before_sync();
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(bar);
  };
  int it_no = 0, gc = 0;
  uint32_t nx[8];  // the next source's coefficients, loaded one source ahead
  uint2 nw;        // and its input constant
  auto fetch_source = [&](const TcSeg& sg, int k) {
    const TcGroup& t = job.g[sg.g];
    if (k >= t.K) return;
    const bool top = TOP && k == t.K - 1;
    const uint32_t* s = (top ? t.top : t.src + ((size_t)(k * t.step) << dp.log_n)) + 8 * jj * G::W + sg.tile * kTcColumns + c;
#pragma unroll
    for (int i = 0; i < 8; ++i) nx[i] = s[i * G::W];
    nw = top ? make_uint2(dp.pc[t.M].ninv, dp.pc[t.M].ninv_sh) : __ldg(t.cin + k);
  };
  if (have) fetch_source(seg, wg);
  while (have) {
    const TcGroup& it = job.g[seg.g];
    const uint8_t* srec = sm + lay.seg + (it_no & 1) * lay.seg_bytes + lay.srec;
    const uint8_t* trec = sm + lay.seg + (it_no & 1) * lay.seg_bytes + lay.trec;
    TcSeg nseg;
    const bool more = iter.next(job, tiles, cap, nseg);
    auto put = [&](int k, int i, uint32_t z) {
      const uint2 d = tc::digits_f16(z);
      tc::tmem_st2(lanes + i * 32 + 2 * k, d.x, d.y);
    };
    wait(b_ld(it_no & 1), (it_no >> 1) & 1);
    uint32_t e[8];  // TOP: the top limb's E, in the warpgroup of source K - 1
    for (int k = wg; k < it.K; k += kTcWarpgroups) {
      uint32_t x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = nx[i];
      const uint2 w = nw;
      fetch_source(seg, k + kTcWarpgroups);
      // iNTT columns: rows 8 jj + i in, jj + 8 i out
      const uint2* t = reinterpret_cast<const uint2*>(srec + k * kTcRecBytes);
      const uint32_t q = *reinterpret_cast<const uint32_t*>(srec + k * kTcRecBytes + 512);
      if (q < (1u << 30)) {
        gs8<true>(x, t, 8 + jj, q);
        tr.b_to_a(x, jj, ct);
        gs8<true>(x, t, 1, q);
      } else {
        gs8<false>(x, t, 8 + jj, q);
        tr.b_to_a(x, jj, ct);
        gs8<false>(x, t, 1, q);
      }
      if (TOP && k == it.K - 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          e[i] = csub(shoup(x[i], w.x, w.y, q), q);
          tc::tmem_st2(lanes + i * 32 + 2 * k, 0u, 0u);  // until V replaces it
        }
      } else {
        // times cin, then the centered representative: v + h reduced to
        // [0, q), less h (h = (q - 1) / 2), and with it the digits' bias
        const uint32_t h = q >> 1, bias = 0x80808080u - h;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint32_t v;
          if (q < (1u << 30)) {
            v = x[i] * w.x + h - __umulhi(x[i], w.y) * q;  // below 2q + h < 2^32
            v = csub(csub(v, q), q);
          } else {
            v = csub(csub(shoup(x[i], w.x, w.y, q), q) + h, q);
          }
          put(k, i, v + bias);
        }
      }
    }
    // digits of the unused source slots
    for (int k = wg; k < tc_kr(it.K) / 4; k += kTcWarpgroups) {
      if (k < it.K) continue;
#pragma unroll
      for (int i = 0; i < 8; ++i) tc::tmem_st2(lanes + i * 32 + 2 * k, 0u, 0u);
    }
    tc::tmem_wait_st();
    arrive(b_a);
    if (more) fetch_source(nseg, wg);
    // Targets are dealt out to the warpgroups one by one; the plane sums of a
    // warpgroup's next target are asked for before the current one is stored.
    uint32_t f[32];
    auto ask = [&](int t) {  // target t of the segment (group gc + t / 4, place t % 4)
      const int u = gc + (t >> 2);
      wait(b_full(u & 1), (u >> 1) & 1);
      tc::fence_after_sync();
#pragma unroll
      for (int i = 0; i < 8; ++i)
        tc::tmem_ld4(lanes + 256 + (u & 1) * 128 + i * 16 + (t & 3) * 4, f[4 * i], f[4 * i + 1], f[4 * i + 2], f[4 * i + 3]);
    };
    auto take = [&](int t) {
      tc::tmem_wait_ld32(f);
      arrive(b_empty((gc + (t >> 2)) & 1));
    };
    auto residues = [&](uint32_t (&x)[8], const TcPrime& P) {
      if (P.q > (1u << 30)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = tc_residue<1>(f + 4 * i, P);
      } else if (P.q > (1u << 29)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = tc_residue<0>(f + 4 * i, P);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = tc_residue<2>(f + 4 * i, P);
      }
    };

    const int m1 = min(seg.m1, it.M), np = (m1 - seg.m0 + 3) & ~3;
    if constexpr (TOP) {
      // z = BConv(P -> q_l), the image's first group; V = E - z P^-1, centered,
      // is source K - 1
      const int own = (it.K - 1) % kTcWarpgroups;
      ask(0);
      if (wg == own) {
        const TcPrime P = load_tc_prime(srec + (it.K - 1) * kTcRecBytes + 512);
        take(0);
        uint32_t x[8];
        residues(x, P);
        const uint2 pinv = dp.ks.dn_pinv[it.M];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          put(it.K - 1, i,
              (uint32_t)centered(csub(e[i] + P.q - csub(shoup(x[i], pinv.x, pinv.y, P.q), P.q), P.q), P.q) + 0x80808080u);
      } else {
        tc::tmem_wait_ld32(f);
        if ((wg + kTcWarpgroups - own) % kTcWarpgroups < 4) arrive(b_empty(gc & 1));
      }
      ++gc;
      tc::tmem_wait_st();
      arrive(b_a);
    }
    if (wg < np) ask(wg);
    for (int t = wg; t < np; t += kTcWarpgroups) {
      const int m = seg.m0 + t;
      const bool on = m < m1;
      const uint8_t* rec = trec + (on ? t : 0) * kTcRecBytes;
      const uint2* tw = reinterpret_cast<const uint2*>(rec + 32);
      const TcPrime P = load_tc_prime(rec);
      take(t);
      uint32_t x[8];
      residues(x, P);
      if (on) {
        if (P.q > (1u << 30)) {
          ct8<false>(x, tw, 1, P.q);
          tr.a_to_b(x, jj, ct);
          ct8<false>(x, tw, 8 + jj, P.q);
        } else {
          ct8<true>(x, tw, 1, P.q);
          tr.a_to_b(x, jj, ct);
          ct8<true>(x, tw, 8 + jj, P.q);
        }
      }
      if (t + kTcWarpgroups < np) ask(t + kTcWarpgroups);
      if (!on) continue;
      uint32_t* dst = it.dst + ((size_t)job.limb(it, m) << dp.log_n) + 8 * jj * G::W + seg.tile * kTcColumns + c;
#pragma unroll
      for (int i = 0; i < 8; ++i) dst[i * G::W] = x[i];
    }
    // every product is done before A is written again
    gc += np / 4;
    wait(b_full((gc - 1) & 1), ((gc - 1) >> 1) & 1);
    tc::fence_after_sync();  // a warpgroup without a target in the last group has not ordered itself behind it
    ++it_no;
    seg = nseg;
    have = more;
  }
  tc::fence_before_sync();
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Launch
// ---------------------------------------------------------------------------

// exact_limit: dp.wait_limit as it is, without the floor (a shape set by hand).
template <class G, bool TOP>
void launch_cols_tc(const DevParams& dp0, const TcJob& job, int groups, int2 plan, bool exact_limit, cudaStream_t st) {
  if constexpr (G::H == 64) {
    DevParams dp = dp0;
    if (!exact_limit) dp.wait_limit = std::max(dp.wait_limit, kTcWaitFloor);
    int kr = 16, cap = 4;
    for (int g = 0; g < groups; ++g) {
      kr = std::max(kr, tc_kr(job.g[g].K));
      cap = std::max(cap, (job.g[g].M + 3) & ~3);
    }
    cap = std::min(cap, kTcCap);
    const TcLayout lay = tc_layout(cap, kr);
    set_col_smem((const void*)k_cols_tc<G, TOP>, lay.total);
    TcPlan pl;
    std::copy(dp.ks.h->plan + plan.x, dp.ks.h->plan + plan.x + plan.y + 1, pl.at);
    launch_pdl(dp.pdl, k_cols_tc<G, TOP>, dim3(plan.y), dim3(kTcThreads), lay.total, st, dp, job, pl, cap, lay);
    count_launch(1);
  }
}

// Compiled once, in k_cols_tc.cu.
extern template void launch_cols_tc<Geo<8, 32>, false>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);
extern template void launch_cols_tc<Geo<8, 32>, true>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);
extern template void launch_cols_tc<Geo<8, 8>, false>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);
extern template void launch_cols_tc<Geo<8, 8>, true>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);

// ModUp of the level's digits: each to every other prime of the extended basis.
template <class G>
static void launch_modup_tc(const DevParams& dp, int n, int base, int tix, int digits, const Scratch& sc,
                            const ColShape& s, cudaStream_t st) {
  TcJob job{n, base, {}};
  for (int j = 0; j < digits; ++j) {
    const int g = base / dp.alpha + j;
    const int lo = std::max(0, g * dp.alpha - base), hi = std::min(n, (g + 1) * dp.alpha - base);
    const size_t at = (size_t)tix * dp.dnum + j;
    job.g[j] = TcGroup{sc.S + ((size_t)lo << dp.log_n), dp.ks.up_cin + dp.ks.h->up_off[at].x,
                       dp.ks.tc_img + dp.ks.h->up_img[at].x, nullptr, nullptr,
                       sc.T + ((size_t)j * (n + dp.alpha) << dp.log_n), hi - lo, n + dp.alpha - (hi - lo), base + lo, lo,
                       hi - lo};
  }
  launch_cols_tc<G, false>(dp, job, digits, dp.ks.h->up_plan[tix], s.by_hand, st);
}

// ModDown of both polynomials to the window.
template <class G>
static void launch_moddown_tc(const DevParams& dp, int n, int base, int tix, const Scratch& sc, const ColShape& s,
                              cudaStream_t st) {
  TcJob job{n, base, {}};
  for (int u = 0; u < 2; ++u)
    job.g[u] = TcGroup{sc.S + ((size_t)u * dp.alpha << dp.log_n), dp.ks.dn_cin, dp.ks.tc_img + dp.ks.h->dn_img[tix].x,
                       nullptr, nullptr, sc.T + ((size_t)u * n << dp.log_n), dp.alpha, n, dp.L, n, 0};
  launch_cols_tc<G, false>(dp, job, 2, dp.ks.h->dn_plan[tix], s.by_hand, st);
}

// ModDown fused with rescaling by the top prime.
template <class G>
static void launch_rs_fused_tc(const DevParams& dp, int n, const Scratch& sc, uint32_t* T3, const ColShape& s,
                               cudaStream_t st) {
  TcJob job{n - 1, 0, {}};
  for (int u = 0; u < 2; ++u)
    job.g[u] = TcGroup{sc.S + ((size_t)u * dp.alpha << dp.log_n), dp.ks.dn_cin, dp.ks.tc_img + dp.ks.h->rs_img[n].x,
                       nullptr, sc.S + ((size_t)(2 * dp.alpha + u) << dp.log_n),
                       T3 + ((size_t)u * (n - 1) << dp.log_n), dp.alpha + 1, n - 1, dp.L, n, 0};
  launch_cols_tc<G, true>(dp, job, 2, dp.ks.h->rs_plan[n], s.by_hand, st);
}

// ModDown merged into the rescaling (Sec. 6).
template <class G>
static void launch_mm_tc(const DevParams& dp, const MmArgs& m, const Scratch& sc, const ColShape& s, cudaStream_t st) {
  TcJob job{m.n1, m.s1, {}};
  for (int u = 0; u < 2; ++u)
    job.g[u] = TcGroup{sc.S + ((size_t)u * m.K << dp.log_n), m.cin, dp.ks.tc_img + m.img, m.rows, nullptr,
                       sc.T + ((size_t)u * m.n1 << dp.log_n), m.K, m.n1, 0, m.n1, 0};
  launch_cols_tc<G, false>(dp, job, 2, m.plan, s.by_hand, st);
}

// Rescaling by the top prime q_(n-1): its limb of both polynomials (S = [2])
// reduced, centered, into every lower prime: a conversion with one source.
template <class G>
static void launch_rescale_tc(const DevParams& dp, int n, const Scratch& sc, cudaStream_t st) {
  TcJob job{n - 1, 0, {}};
  for (int u = 0; u < 2; ++u)
    job.g[u] = TcGroup{sc.S + ((size_t)u << dp.log_n), reinterpret_cast<const uint2*>(&dp.pc[n - 1].ninv),
                       dp.ks.tc_img + dp.ks.one_img, nullptr, nullptr, sc.T + ((size_t)u * (n - 1) << dp.log_n), 1,
                       n - 1, n - 1, n, 0};
  launch_cols_tc<G, false>(dp, job, 2, dp.ks.h->one_plan[n], false, st);
}

// Rational rescaling: the dropped limbs (S = [K][2]) to the new window.
template <class G>
static void launch_rr_tc(const DevParams& dp, const RrArgs& r, const Scratch& sc, cudaStream_t st) {
  TcJob job{r.n1, r.s1, {}};
  for (int u = 0; u < 2; ++u)
    job.g[u] = TcGroup{sc.S + ((size_t)u << dp.log_n), r.cin, dp.ks.tc_img + r.img, r.drop, nullptr,
                       sc.T + ((size_t)u * r.n1 << dp.log_n), r.K, r.n1, 0, r.n1, 0, 2};
  launch_cols_tc<G, false>(dp, job, 2, r.plan, false, st);
}

// Tensor-core launch shapes: tp = 8 or 16 with the (tc, sl) pairs below and
// z = 1. All of them run the one tensor-core kernel, whose division of the
// work follows from the level.
inline bool is_tc_shape(const ColShape& s) { return s.tp == 8 || s.tp == 16; }

template <class G>
static bool tc_shape_ok(const ColShape& s) {
  return G::H == 64 && s.z == 1 && is_tc_shape(s) &&
         ((s.tc == 8 && (s.sl == 2 || s.sl == 4)) || (s.tc == 4 && (s.sl == 4 || s.sl == 8)));
}

}  // namespace ckks
