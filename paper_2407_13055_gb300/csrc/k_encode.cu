// Encoding and decoding (CKKS canonical embedding) on the device in binary64:
// slot j of a plaintext is its polynomial's value at zeta^(5^j mod 2N), zeta =
// exp(i pi / N), and the conjugate at the inverse, so both directions are a
// length-N complex FFT with a twist by powers of zeta.
//
//   encode: slots -> values at zeta^(2i + 1), bit-reversed -> FFT (sign -) ->
//           times zeta^-k / N * scale, rounded half away from zero
//   decode: residues -> mixed-radix digits -> centered value (Horner from the
//           top digit) times zeta^k, bit-reversed -> FFT (sign +) -> slots
//
// The FFT is radix 2, decimation in time: the first eight stages on runs of
// 256 values, the others on columns of stride 256, each set in shared memory
// in one kernel. The twiddles are a table of zeta^k in the host library's
// cosines and sines, and the fused multiply-adds are written out, so the
// rounded coefficients do not depend on a compiler's contraction.
//
// Bound by launches, copies and the plaintext's allocation: N = 2^16 takes 1 M
// complex multiply-adds and moves a few MB between L2 and the SMs. On the host
// (a cosine and a sine per butterfly, a division per Garner step) encode +
// decode took 20.07 ms at six limbs and 383 ms at forty; here 0.476 and 0.55.
// At N = 2^8 an encode takes 42 us (46), a decode 45 (55).
#include "internal.h"

namespace ckks {

namespace {

constexpr int kLogRun = 8, kRun = 1 << kLogRun;

__device__ __forceinline__ uint32_t brev_log(uint32_t v, int log_n) { return __brev(v) >> (32 - log_n); }

// a w whose plain form came out as NaN in both parts: infinite operands and
// overflowed products keep an infinity (C99, Annex G.5.1).
__device__ __noinline__ double2 cmul_special(double2 a, double2 w, double2 r) {
  const double ac = __dmul_rn(a.x, w.x), bd = __dmul_rn(a.y, w.y), ad = __dmul_rn(a.x, w.y), bc = __dmul_rn(a.y, w.x);
  const bool over = isinf(ac) || isinf(bd) || isinf(ad) || isinf(bc);
  bool redo = false;
  if (isinf(a.x) || isinf(a.y)) {
    a = make_double2(copysign(isinf(a.x) ? 1.0 : 0.0, a.x), copysign(isinf(a.y) ? 1.0 : 0.0, a.y));
    redo = true;
  }
  if (!redo && over) {
    if (isnan(a.x)) a.x = copysign(0.0, a.x);
    if (isnan(a.y)) a.y = copysign(0.0, a.y);
    redo = true;
  }
  if (!redo) return r;
  const double inf = __longlong_as_double(0x7ff0000000000000ll);
  return make_double2(inf * (a.x * w.x - a.y * w.y), inf * (a.x * w.y + a.y * w.x));
}

__device__ __forceinline__ double2 cmul(double2 a, double2 w) {
  const double2 r = make_double2(__fma_rn(a.x, w.x, -__dmul_rn(a.y, w.y)), __fma_rn(a.x, w.y, __dmul_rn(a.y, w.x)));
  if ((__double2hiint(r.x) & __double2hiint(r.y) & 0x7ff00000) == 0x7ff00000 && isnan(r.x) && isnan(r.y))
    return cmul_special(a, w, r);
  return r;
}

template <int SIGN>
__device__ __forceinline__ double2 twiddle(const double2* __restrict__ tw, uint32_t k) {
  double2 w = tw[k];
  if (SIGN < 0) w.y = -w.y;
  return w;
}

__device__ __forceinline__ void bfly(double2& a, double2& b, double2 w) {
  const double2 v = cmul(b, w), u = a;
  a = make_double2(__dadd_rn(u.x, v.x), __dadd_rn(u.y, v.y));
  b = make_double2(__dsub_rn(u.x, v.x), __dsub_rn(u.y, v.y));
}

// The j with 5^j = e mod 2^(log_n + 1), for e = 1 mod 4: 5^(2^b) = 1 + 2^(b + 2)
// mod 2^(b + 3), so the lowest bits of e divided by the powers found so far
// give j's bits one after the other.
__device__ __forceinline__ uint32_t log5(uint32_t e, int log_n) {
  uint32_t j = 0, inv = 0xCCCCCCCDu;  // 5^-(2^b) mod 2^32
  for (int b = 0; b < log_n - 1; ++b, inv *= inv)
    if ((e >> (b + 2)) & 1) {
      e *= inv;
      j |= 1u << b;
    }
  return j;
}

// Where the FFT's kernels read value i of their input and put value i of their
// output: the complex array itself, the slots (input of the encoding, whose
// value i belongs to zeta^(2 brev(i) + 1); output of the decoding), or the
// rounded coefficients (output of the encoding).
struct AtArray {
  double2* z;
  __device__ __forceinline__ double2 get(uint32_t i) const { return z[i]; }
  __device__ __forceinline__ void put(uint32_t i, double2 v) const { z[i] = v; }
};
struct FromSlots {
  const double2* slots;
  int log_n;
  __device__ __forceinline__ double2 get(uint32_t i) const {
    const uint32_t e = 2 * brev_log(i, log_n) + 1;
    double2 v = slots[log5((e & 3) == 1 ? e : 0u - e, log_n)];
    if ((e & 3) != 1) v.y = -v.y;
    return v;
  }
};
struct ToSlots {
  double2* slots;
  double scale;
  int log_n;
  __device__ __forceinline__ void put(uint32_t i, double2 v) const {
    if (i % 2 == 0) slots[log5(2 * i + 1, log_n)] = make_double2(__ddiv_rn(v.x, scale), __ddiv_rn(v.y, scale));
  }
};
struct ToCoeffs {
  int64_t* coeffs;
  const double2* tw;
  double scale;
  int log_n;
  __device__ __forceinline__ void put(uint32_t k, double2 z) const {
    const double x = cmul(z, twiddle<-1>(tw, k)).x;
    const double v = __dmul_rn(__ddiv_rn(x, (double)(1u << log_n)), scale);
    const double r = v < 0 ? -floor(__dadd_rn(-v, 0.5)) : floor(__dadd_rn(v, 0.5));
    coeffs[k] = isnan(r) ? 0 : __double2ll_rz(r);  // saturates
  }
};

// Stages 0 .. 7 on 256 consecutive values, 128 threads; the stages' twiddles
// are loaded before the first. (N = 256, one block: the output may overwrite
// the input.)
template <int SIGN, class In, class Out>
__global__ void __launch_bounds__(kRun / 2) k_fft_runs(In in, Out out, const double2* tw, int log_n) {
  __shared__ double2 s[kRun];
  const int t = threadIdx.x;
  const uint32_t run = blockIdx.x * kRun;
  double2 w[kLogRun];
#pragma unroll
  for (int st = 0; st < kLogRun; ++st) w[st] = twiddle<SIGN>(tw, (uint32_t)(t & ((1 << st) - 1)) << (log_n - st));
  s[t] = in.get(run + t);
  s[t + kRun / 2] = in.get(run + t + kRun / 2);
#pragma unroll
  for (int st = 0; st < kLogRun; ++st) {
    __syncthreads();
    const int i = ((t >> st) << (st + 1)) | (t & ((1 << st) - 1));
    bfly(s[i], s[i + (1 << st)], w[st]);
  }
  __syncthreads();
  out.put(run + t, s[t]);
  out.put(run + t + kRun / 2, s[t + kRun / 2]);
}

// Stages 8 .. 8 + LR - 1 (N = 2^(8 + LR)) on 2^LR rows of 512 / 2^LR columns.
template <int SIGN, int LR, class Out>
__global__ void __launch_bounds__(256) k_fft_cols(const double2* z, Out out, const double2* tw) {
  constexpr int R = 1 << LR, C = 512 >> LR;
  __shared__ double2 s[R * C];
  const int c = threadIdx.x % C, m = threadIdx.x / C, col = blockIdx.x * C + c;
  double2 w[LR];
#pragma unroll
  for (int st = 0; st < LR; ++st)
    w[st] = twiddle<SIGN>(tw, (uint32_t)((m & ((1 << st) - 1)) * kRun + col) << (LR - st));
  s[m * C + c] = z[m * kRun + col];
  s[(m + R / 2) * C + c] = z[(m + R / 2) * kRun + col];
#pragma unroll
  for (int st = 0; st < LR; ++st) {
    __syncthreads();
    const int i = ((m >> st) << (st + 1)) | (m & ((1 << st) - 1));
    bfly(s[i * C + c], s[(i + (1 << st)) * C + c], w[st]);
  }
  __syncthreads();
  out.put(m * kRun + col, s[m * C + c]);
  out.put((m + R / 2) * kRun + col, s[(m + R / 2) * C + c]);
}

template <int SIGN, class In, class Out>
void fft(In in, double2* z, Out out, const double2* tw, int log_n, cudaStream_t st) {
  if (log_n == kLogRun) {
    k_fft_runs<SIGN><<<1, kRun / 2, 0, st>>>(in, out, tw, log_n);
    count_launch(1);
    return;
  }
  k_fft_runs<SIGN><<<1 << (log_n - kLogRun), kRun / 2, 0, st>>>(in, AtArray{z}, tw, log_n);
  if (log_n == 12) k_fft_cols<SIGN, 4><<<kRun / 32, 256, 0, st>>>(z, out, tw);
  else k_fft_cols<SIGN, 8><<<kRun / 2, 256, 0, st>>>(z, out, tw);
  count_launch(2);
}

// Coefficient k: mixed-radix (Garner) digits v_i of its residues, one below
// the other in shared memory, v_i = ((r_i - v_0) / q_0 - v_1) / q_1 ... mod q_i;
// half: the digits of (Q - 1) / 2, above which the value is negative. The
// value is d_0 + q_0 (d_1 + q_1 (d_2 + ...)) from the top digit: the leading
// digits of a small value are 0 (or q_i - 1 for a negative one), so nothing
// overflows however many limbs there are.
__global__ void k_dec_value(DevParams dp, EncTables et, const uint32_t* res, int nl, int base, const uint32_t* half,
                            double2* z) {
  extern __shared__ uint32_t digits[];
  const int log_n = dp.log_n, T = blockDim.x;
  const uint32_t k = blockIdx.x * T + threadIdx.x;
  uint32_t* v = digits + threadIdx.x;
  const PrimeConst* pc = dp.pc + base;
  for (int i = 0; i < nl; ++i) {
    const uint32_t q = pc[i].q, up = ((1u << 31) - 1) / q * q + q;  // a multiple of q, 2^31 <= up < 2^31 + q
    const uint2* inv = et.inv + (size_t)(base + i) * dp.L + base;
    uint32_t t = res[((size_t)i << log_n) + k];
    for (int j = 0; j < i; ++j) {
      const uint32_t d = v[j * T];
      const uint2 w = inv[j];
      t = csub(shoup(t - d + (t < d ? up : 0u), w.x, w.y, q), q);
    }
    v[i * T] = t;
  }
  bool neg = false;
  for (int i = nl - 1; i >= 0; --i) {
    const uint32_t d = v[i * T], h = half[i];
    if (d != h) {
      neg = d > h;
      break;
    }
  }
  double x = 0;
  for (int i = nl - 1; i >= 0; --i) {
    const uint32_t q = pc[i].q, d = v[i * T];
    x = __fma_rn(x, (double)q, (double)(neg ? q - 1 - d : d));
  }
  if (neg) x = -(x + 1);
  const double2 w = et.tw[k];
  z[brev_log(k, log_n)] = make_double2(__dmul_rn(x, w.x), __dmul_rn(x, w.y));
}

}  // namespace

void launch_encode(const DevParams& dp, const EncTables& et, double2* slots, double2* z, double scale,
                   cudaStream_t st) {
  fft<-1>(FromSlots{slots, dp.log_n}, z, ToCoeffs{reinterpret_cast<int64_t*>(slots), et.tw, scale, dp.log_n}, et.tw,
          dp.log_n, st);
}

void launch_decode(const DevParams& dp, const EncTables& et, const uint32_t* res, int nl, int base,
                   const uint32_t* half, double scale, double2* z, double2* slots, cudaStream_t st) {
  int th = 64;  // digits in 48 KB of shared memory: 192 limbs at 64 threads
  while (th > 1 && (size_t)th * nl * 4 > 48 * 1024) th >>= 1;
  k_dec_value<<<(1 << dp.log_n) / th, th, (size_t)th * nl * 4, st>>>(dp, et, res, nl, base, half, z);
  count_launch(1);
  fft<1>(AtArray{z}, z, ToSlots{slots, scale, dp.log_n}, et.tw, dp.log_n, st);
}

}  // namespace ckks
