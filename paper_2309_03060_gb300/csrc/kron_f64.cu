// FP64 Kronecker mode products on the tcgen05 tensor cores (sm_103a).
//
// One FP64 mode step  Y[r][m][i] = alpha sum_j F[i][j] X[r][j][m] + beta Y
// (Sec. 3.2, Table 3) by an error-free split into integer digits, the scheme
// of Ozaki, Ogita, Oishi & Rump (Numer. Algorithms 59, 2012; on tensor cores
// Mukunoki et al. 2020): over a k chunk of at most 128 entries every factor
// row and every vector gets a power-of-two scale from its largest exponent,
//   f_ij = 2^(Ef_i - 55) sum_t a_t 256^(6-t),   x_jm = 2^(Ex_m - 54) sum_t b_t 256^(6-t),
// with signed base-256 digits (|a_0| <= 256, |b_0| <= 128, the others in
// [-128, 127]) that are exact in FP16.  The sums D_d = sum_{s+t=d} sum_j a_s b_t
// of the 28 digit pairs with s + t <= 6 stay within 2^22 + d 2^21 <= 2^24 for 128
// terms, so the FP32 accumulators hold them exactly; they are combined in 64-bit
// integers (in units of D_5) and rounded to FP64 once.  What is lost: what lies below
// 2^-56 of a row's and 2^-55 of a vector's largest binade, and the pairs s + t >= 7;
// together at most 1.14 2^-52 K 2^(Ef + Ex) of an output with K entries.
//
// That is a bound by row and vector.  An output is to be as accurate as FP64 products
// make it by its own sum |f| |x|, however small that is beside the row's and the
// vector's largest entries (graded vectors, columns of a covariance, block factors).  So
// one more product runs on the tensor cores: the sum of leading magnitudes |a_0| |b_0|,
// truncated to E5M2 (8-bit MMAs, 4 instead of 8 per 128 k).  Where it is at least
// kLeadMin, sum |f| |x| is at least 2^-3.7 2^(Ef + Ex) and the loss of the order of FP64
// roundings.  A factor row with a single entry takes twice that: the vector's entry is
// then within a binade of its largest and exact in units of D_5 (an identity factor
// returns its input).  The other outputs, and those of rows and vectors without digits
// (non-finite, far exponents), are listed and computed with FP64 multiply-adds once the
// CTA's tiles are done.
// Largest error over sum |f| |x|, in units of 2^-53, measured on RBF factors with sides
// 32 .. 200: 0.6 .. 5.4, against 3.3 .. 9.9 in FP64 multiply-adds; graded vectors 20
// against 20, identity 0 against 0, unit vectors 1.6 against 0.  What it costs: nothing
// where no output is low, the rate of the FP64 units where most are (identity 128^3 x 4:
// 5.8 ms for the three steps, 5.25 ms in 32 x 32 tiles there; columns of a 128 x 128 RBF
// product, 64 of them: 0.30 against 0.47 ms), and on short RBF factors of a small
// lengthscale, some of whose points have no neighbour, part of the gain: sides 32, 48,
// lengthscale 0.05, 16 vectors 123, 184 us against 87, 140 without it and 123, 625 on the
// FP64 units.
//
// Why: this GPU's FP64 units do 2 multiply-adds per clock and SM (1.2 TFLOP/s),
// its tensor cores ~1900 TFLOP/s in FP16, so 28 products are still ~50 times
// cheaper.  Every FP64 pipe use in the inner path is avoided: exponents and
// digits come from integer operations, and so do the combination and its
// conversion; of the outputs only alpha, beta other than 1, 0 take FP64 instructions.
//
// Kernel layout (persistent, one 576-thread CTA per SM), tile = 64 vectors m x
// 128 outputs i, step = tile x k chunk:
//   warps 0-7   converters: load the 64 x 128 FP64 block into registers, find each
//               vector's exponent and write the 7 digit images of the B operand
//               (vectors x k, K-major, 128-byte swizzle, 112 KB) and its leading
//               magnitudes (8 KB)
//   warps 8-15  drainers: note the outputs with too small a sum of magnitudes, add
//               the accumulators up in 64-bit integers, scale, store
//   warp 16     copies the factor's leading magnitudes (16 KB) and digit images
//               (32 KB each; three buffers, cp.async.bulk from the prepared image, L2
//               resident)
//   warp 17     issues the MMAs: the magnitudes', then factor digit s = 0 .. 6
//               outermost, so that group s is the last to use B digit 6 - s and completes
//               accumulator D_s;
//               D_s is drained and digit 6 - s refilled for the next step while
//               the later groups run, and only D_6 and digit 0 are left when the
//               MMAs of a step end
// Measured (128^3 x 16, one mode step, 268 MB in and out): 270 us against 6.97 ms
// on the FP64 units.  What bounds it: the chain of conversion, MMAs and drain of a
// step, each waiting for the one before with 18 warps on the SM: the integer pipe (8192
// entries converted, 8192 outputs combined per step) is active 0.58 of the time, the
// tensor-core pipe (224 MMAs of 128 x 64 x 16 per step) 0.61, issue slots 0.50;
// converting and draining in separate warps, both beside the MMAs, took it from 395 us,
// no FP64 conversion per output from 450 us, and issuing from a converged warp (uniform
// descriptors) from 520 us.  18 warps hold a thread to 96 registers (72 bytes of spills;
// 280 in the variant with a table of problems).
// Accumulators: D_0 .. D_6 and the magnitudes', 64 FP32 columns each of tensor memory
// (all 512).  Every mbarrier wait gives up after ~2 s and raises the error flag.
#include <cuda_fp16.h>

#include <algorithm>
#include <string>
#include <vector>

#include "internal.h"
#include "tc_ptx.cuh"

namespace cola {

namespace {

constexpr int kDg = 7;             // digits per operand
constexpr int kVec = 64;           // vectors per tile (N of the MMA)
constexpr int kOut = 128;          // outputs per tile (M of the MMA)
constexpr int kKc = 128;           // k chunk
constexpr int kConvWarps = 8, kDrainWarps = 8;
constexpr int kLoadWarp = kConvWarps + kDrainWarps, kMmaWarp = kLoadWarp + 1;
constexpr int kThreadsF64 = 32 * (kMmaWarp + 1);
constexpr uint32_t kBDig = kVec * kKc * 2;   // 16 KB per B digit
constexpr uint32_t kADig = kOut * kKc * 2;   // 32 KB per A digit
constexpr uint32_t kBLead = kVec * kKc;      // 8 KB of leading magnitudes of B
constexpr uint32_t kALead = kOut * kKc;      // 16 KB of A
constexpr uint32_t kABlk = kDg * kADig + kALead;  // image of one 128 x 128 factor block
constexpr int kABufs = 3;
constexpr size_t kSmemF64 = 1024 + kDg * kBDig + kBLead + kABufs * kADig + 6144;
// Outputs whose sum of leading magnitudes is below this take plain products.  For rows
// with one entry: 128 (|a_0| of a power of two) times 40, the smallest E5M2 number above
// 32 = |b_0| of an entry a binade below its vector's largest.
constexpr float kLeadMin = 2560.0f, kLeadMinOne = 5120.0f;
// Magnitude (E5M2, 2^8) that stands for every entry of a zero row or vector, whose outputs
// are exact (0, or without digits on the other side).
constexpr uint32_t kLeadZero = 0x5c;
constexpr int kPlain = 1 << 20;  // exponent mark of a factor row that takes plain products

struct F64Params {
  const double* X;
  double* Y;
  const double* F;      // the factor itself (plain products)
  const uint16_t* img;  // [nchunks][kchunks][digit][k block][128][64], swizzled rows
  const int* fexp;      // [nchunks][kchunks][128]: 2 Ef, + 1 for a row with one entry
  int64_t f_i, f_j;     // element strides of F
  int64_t size_in, size_out;
  int rest, tiles_m, ntiles, n_in, n_out, nchunks, kchunks;
  double alpha, beta;
  int has_alpha, has_beta;  // alpha != 1, beta != 0 (a compare is an FP64-pipe instruction)
};

// Launch-wide settings.
struct F64Launch {
  int* err;
  uint64_t stall_ns;
  // Outputs left to plain products: per CTA low_cap entries, each one thread's of one
  // step (thread of the drainers + 256 times the CTA's tile; k chunk; the mask of its
  // 32 outputs).
  uint32_t* low;
  int64_t low_cap;
  int kmax;  // most k chunks of a problem
};

// Where a tile's parameters come from: one problem by value, or a device table
// of problems (tile -> problem, first tile of each).
struct F64One {
  F64Params p;
  __device__ __forceinline__ int count() const { return p.ntiles; }
  __device__ __forceinline__ const F64Params& get(int t, int& lt) const {
    lt = t;
    return p;
  }
};
struct F64Tab {
  const F64Params* probs;
  const int* tile_prob;
  const int* first;
  int ntiles;
  __device__ __forceinline__ int count() const { return ntiles; }
  __device__ __forceinline__ const F64Params& get(int t, int& lt) const {
    const int i = __ldg(tile_prob + t);
    lt = t - __ldg(first + i);
    return probs[i];
  }
};

// Magnitude key of FP64 entries: the largest high word without the sign, or 1
// when only low words are not zero, so that it is 0 only for +-0.
__device__ __forceinline__ void mag_key(unsigned long long x, uint32_t& hi, uint32_t& lo) {
  hi = max(hi, (uint32_t)(x >> 32) & 0x7fffffffu);
  lo |= (uint32_t)x;
}

// A row or vector whose largest key is `key` has digits when it is zero or its
// largest entry is finite and at least 2^-959 (below that a denormal entry
// could still reach the digits, which fixed_digits does not expect); others
// take plain FP64 products.
__device__ __forceinline__ bool has_digits(int key) {
  const int f = key >> 20;
  return key == 0 || (f > 63 && f < 0x7ff);
}

constexpr unsigned long long kZeroDigits = 0x0100808080808080ull;

// The digits of x, |x| < 2^(emax - 1022), scaled by 2^(52 + UP - (emax - 1023)) and rounded to
// an integer v: v plus 128 in each byte 0 .. 5 and 256 at bit 48, so that bytes
// 0 .. 5 are digits 6 .. 1 plus 128 and the bits from 48 on digit 0 plus 256.
// emax > 63 (any value when x = 0): a zero or denormal entry shifts out
// completely.
template <int UP>
__device__ __forceinline__ unsigned long long fixed_digits(unsigned long long x, int emax) {
  const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
  const int sh = min(63, emax - (int)((hi >> 20) & 0x7ffu));
  const unsigned long long m =
      (((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << (UP + 1);
  const unsigned long long w = m >> sh;  // twice |v|, one bit below it
  const long long sg = (int)hi >> 31;    // 0 or -1
  constexpr long long bias = (long long)kZeroDigits;
  // x >= 0: floor((w + 1) / 2); x < 0: floor(-w / 2), as ~w + 1 = -w; plus the bias
  return (unsigned long long)(((long long)(w ^ (unsigned long long)sg) + (2 * bias + 1)) >> 1);
}
// Digit t of two values as an FP16 pair: 0x6400 | b is 1024 + b for b < 1024,
// the bias comes off exactly.
template <int t>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long a, unsigned long long b) {
  constexpr int byte = 6 - t;  // byte position in the 64-bit word
  const uint32_t aw = byte < 4 ? (uint32_t)a : (uint32_t)(a >> 32);
  const uint32_t bw = byte < 4 ? (uint32_t)b : (uint32_t)(b >> 32);
  constexpr uint32_t p = byte & 3;
  uint32_t w, bias;
  if constexpr (t == 0) {
    w = __byte_perm(aw, bw, 0x7632) | 0x64006400u;
    bias = 0x65006500u;  // 1024 + 256
  } else {
    w = (__byte_perm(aw, bw, p | (p << 4) | ((4 + p) << 8) | ((4 + p) << 12)) & 0x00ff00ffu) |
        0x64006400u;
    bias = 0x64806480u;  // 1024 + 128
  }
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&w),
                            *reinterpret_cast<const __half2*>(&bias));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// a 2^e rounded to FP64 for 1023 + 62 + |e| within the exponent range, by
// integer operations (an FP64 conversion is two instructions of 16 clocks each
// on the SM's FP64 units): the leading bit of |a| goes to bit 63, bits 63 .. 11
// rounded are the significand with its hidden bit, which adds 1 to the exponent.
__device__ __forceinline__ double scaled_double(long long a, int e) {
  const uint32_t sg = (uint32_t)(a >> 63);
  const unsigned long long m = ((unsigned long long)a ^ (unsigned long long)(long long)(int)sg) -
                               (unsigned long long)(long long)(int)sg;
  const int lz = __clzll((long long)m);  // 64 for 0: the shift below leaves 0
  const unsigned long long n = lz < 64 ? m << lz : 0ull;
  const unsigned long long r = (n + 0x400ull) >> 11;
  const bool carry = n + 0x400ull < n;  // rounded up to 2^64
  uint32_t hi = (uint32_t)(r >> 32) + ((uint32_t)(1023 + 62 - lz + e) << 20);
  if (carry) hi = (uint32_t)(1023 + 64 - lz + e) << 20;
  if (m == 0) hi = 0;
  return __hiloint2double((int)(hi | (sg & 0x80000000u)), (int)(uint32_t)r);
}
constexpr int kFarExp = 450;  // |exponent| of a row or vector up to which it does
constexpr int kHidden = 4;    // see the drain
__device__ __forceinline__ bool far_key(int key) {
  return key != 0 && (!has_digits(key) || abs((key >> 20) - 1023) > kFarExp);
}

// y += alpha f . x (y = of a single step without old values) over the k chunk [k0, k1)
// for the columns (vectors) of one mask: column c at x + c and y + c n_out.  Four columns
// at a time share the loads of f and are a chain each.
__device__ __forceinline__ void plain_columns(const F64Params& p, uint32_t mask, int k0, int k1,
                                              const double* f, const double* x, double* y) {
  while (mask != 0) {
    int c[4];
    const int nc = min(4, __popc(mask));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      c[q] = q < nc ? __ffs(mask) - 1 : c[0];
      if (q < nc) mask &= mask - 1;
    }
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int k = k0;
    for (; k + 4 <= k1; k += 4) {
      double fv[4], xv[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        fv[u] = f[(k + u) * p.f_j];
#pragma unroll
        for (int q = 0; q < 4; ++q) xv[u][q] = x[(int64_t)(k + u) * p.rest + c[q]];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = fma(fv[u], xv[u][q], a[q]);
    }
    for (; k < k1; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] = fma(f[k * p.f_j], x[(int64_t)k * p.rest + c[q]], a[q]);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < nc) {
        double* o = y + (int64_t)c[q] * p.n_out;
        *o = p.kchunks == 1 && !p.has_beta ? p.alpha * a[q] : fma(p.alpha, a[q], *o);
      }
  }
}

// The digit images and exponents of one factor (chunk): block (row of the
// padded 128-row output chunk, output chunk, k chunk), one thread per k.
__global__ void __launch_bounds__(kKc) k_f64_digits(const double* F, int64_t f_i, int64_t f_j,
                                                    int n_out, int n_in, int kchunks,
                                                    uint16_t* img, int* fexp) {
  const int row = blockIdx.x, nc = blockIdx.y, kc = blockIdx.z, k = threadIdx.x;
  const int i = nc * kOut + row, j = kc * kKc + k;
  __shared__ int smax[kKc / 32];
  const double x = (i < n_out && j < n_in) ? F[i * f_i + j * f_j] : 0.0;
  uint32_t xh = 0, xl = 0;
  mag_key((unsigned long long)__double_as_longlong(x), xh, xl);
  int mx = xh | (xh == 0 && xl != 0 ? 1 : 0);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((k & 31) == 0) smax[k >> 5] = mx;
  __syncthreads();
  mx = max(max(smax[0], smax[1]), max(smax[2], smax[3]));
  const int emax = mx >> 20;
  const bool dig = has_digits(mx);
  const int64_t blk = (int64_t)nc * kchunks + kc;
  const unsigned long long u =
      dig && mx ? fixed_digits<3>((unsigned long long)__double_as_longlong(x), emax) : kZeroDigits;
  // digit t: k block (k / 64), row, 16-byte chunk (k / 8) mod 8 swizzled by the row
  uint16_t* p = img + blk * (kABlk / 2) + (size_t)(k >> 6) * (kOut * 64) + row * 64 +
                ((((k >> 3) & 7) ^ (row & 7)) << 3) + (k & 7);
  constexpr size_t st = kADig / 2;
  const uint32_t lead = digit_pair<0>(u, u);
  // entries of the row with a leading magnitude: one alone takes the strict threshold
  int cnt = __popc(__ballot_sync(0xffffffffu, (lead & 0x7fffu) != 0));
  __syncthreads();  // smax is no longer read
  if ((k & 31) == 0) smax[k >> 5] = cnt;
  __syncthreads();
  if (k == 0) {
    cnt = smax[0] + smax[1] + smax[2] + smax[3];
    fexp[blk * kOut + row] = (dig ? (mx ? emax - 1023 : 0) : kPlain) * 2 + (cnt <= 1);
  }
  p[0 * st] = (uint16_t)lead;
  // the leading magnitude: 16-byte chunk k / 16 of the row, swizzled likewise
  reinterpret_cast<unsigned char*>(img + blk * (kABlk / 2))[kDg * kADig + row * kKc +
                                                            (((k >> 4) ^ (row & 7)) << 4) +
                                                            (k & 15)] =
      (unsigned char)(mx ? (lead >> 8) & 0x7fu : (j < n_in ? kLeadZero : 0u));
  p[1 * st] = (uint16_t)digit_pair<1>(u, u);
  p[2 * st] = (uint16_t)digit_pair<2>(u, u);
  p[3 * st] = (uint16_t)digit_pair<3>(u, u);
  p[4 * st] = (uint16_t)digit_pair<4>(u, u);
  p[5 * st] = (uint16_t)digit_pair<5>(u, u);
  p[6 * st] = (uint16_t)digit_pair<6>(u, u);
}

// One (tile, k chunk) step.
struct F64Step {
  int r, m0, nc, kc;
};
__device__ __forceinline__ F64Step step_of(const F64Params& p, int tile, int kc) {
  F64Step s;
  s.nc = tile % p.nchunks;
  const int t = tile / p.nchunks;
  s.r = t / p.tiles_m;
  s.m0 = (t - s.r * p.tiles_m) * kVec;
  s.kc = kc;
  return s;
}

__device__ __forceinline__ void mad_wide(long long& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// Folds accumulator D_T's 32 columns into the integer sums (units of D_5).
template <int T>
__device__ __forceinline__ void fold(uint32_t taddr, long long (&acc)[32]) {
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    uint32_t v[8];
    tmem_ld8(taddr + T * kVec + h * 8, v);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int c = h * 8 + e;
      const int d = __float2int_rn(__uint_as_float(v[e]));
      if constexpr (T == 0) {
        acc[c] = (long long)((unsigned long long)((uint32_t)d << 8) << 32);
      } else if constexpr (T == 1) {
        acc[c] += (long long)((unsigned long long)(uint32_t)d << 32);
      } else if constexpr (T == 6) {
        mad_wide(acc[c], (d + 128) >> 8, 1);
      } else {
        mad_wide(acc[c], d, 1 << (8 * (5 - T)));
      }
    }
  }
}

// Writes digit T of this thread's four 8-entry k runs (run h at k = 8 oct + 32 h:
// k block h / 2, 16-byte chunk (oct + 4 h) mod 8).
template <int T>
__device__ __forceinline__ void put_digit(unsigned char* bdig, const unsigned long long (&u)[32],
                                          int n, int oct, int kpad) {
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    if (oct * 8 + h * 32 >= kpad) continue;
    uint4 w;
    w.x = digit_pair<T>(u[8 * h + 0], u[8 * h + 1]);
    w.y = digit_pair<T>(u[8 * h + 2], u[8 * h + 3]);
    w.z = digit_pair<T>(u[8 * h + 4], u[8 * h + 5]);
    w.w = digit_pair<T>(u[8 * h + 6], u[8 * h + 7]);
    const int ch = (oct + 4 * (h & 1)) ^ (n & 7);
    *reinterpret_cast<uint4*>(bdig + T * kBDig + (h >> 1) * (kBDig / 2) + n * 128 + ch * 16) = w;
  }
}

// put_digit<0> and this thread's leading magnitudes, |digit 0| truncated to E5M2 (the
// upper byte of its FP16 form), up to kpad rounded to the 32 k of an 8-bit MMA
// (entries past n_in are zeros); keys: the four magnitude keys of the vector.
__device__ __forceinline__ void put_lead(unsigned char* bdig, unsigned char* blead,
                                         const unsigned long long (&u)[32], int n, int oct,
                                         int kpad, const int* keys) {
  const bool zero = (keys[0] | keys[kVec] | keys[2 * kVec] | keys[3 * kVec]) == 0;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    if (oct * 8 + h * 32 >= (kpad + 31) / 32 * 32) continue;
    uint4 w;
    w.x = digit_pair<0>(u[8 * h + 0], u[8 * h + 1]);
    w.y = digit_pair<0>(u[8 * h + 2], u[8 * h + 3]);
    w.z = digit_pair<0>(u[8 * h + 4], u[8 * h + 5]);
    w.w = digit_pair<0>(u[8 * h + 6], u[8 * h + 7]);
    const int ch = (oct + 4 * (h & 1)) ^ (n & 7);
    *reinterpret_cast<uint4*>(bdig + (h >> 1) * (kBDig / 2) + n * 128 + ch * 16) = w;
    uint2 m = make_uint2(__byte_perm(w.x, w.y, 0x7531) & 0x7f7f7f7fu,
                         __byte_perm(w.z, w.w, 0x7531) & 0x7f7f7f7fu);
    if (zero) m = make_uint2(kLeadZero * 0x01010101u, kLeadZero * 0x01010101u);
    *reinterpret_cast<uint2*>(blead + n * kKc + ((((oct >> 1) + 2 * h) ^ (n & 7)) << 4) +
                              (oct & 1) * 8) = m;
  }
}

// Which of this thread's 32 outputs have too small a sum of leading magnitudes.
__device__ __forceinline__ uint32_t low_outputs(uint32_t taddr, bool one) {
  const float least = one ? kLeadMinOne : kLeadMin;
  uint32_t v[32];
  tmem_ld32(taddr + kDg * kVec, v);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  float mn = __uint_as_float(v[0]);
#pragma unroll
  for (int e = 1; e < 32; ++e) mn = fminf(mn, __uint_as_float(v[e]));
  uint32_t low = 0;
  if (__any_sync(0xffffffffu, mn < least)) {
#pragma unroll
    for (int e = 0; e < 32; ++e) low |= (__uint_as_float(v[e]) < least ? 1u : 0u) << e;
  }
  return low;
}

// The MMAs of factor digit a with every B digit t <= 6 - a (t downwards: digit
// 0 is refilled last).  One warp issues 224 MMAs per step, so the k loop is
// unrolled with constant descriptor offsets.
template <bool FULL>
__device__ __forceinline__ void issue_group(uint32_t tmem, uint64_t ad, uint64_t bdesc,
                                            uint32_t idesc, int a, int ksteps,
                                            uint32_t elect) {
#pragma unroll 1
  for (int t = kDg - 1 - a; t >= 0; --t) {
    const uint32_t d = tmem + (uint32_t)(a + t) * kVec;
    const uint64_t bd = bdesc + (uint64_t)((uint32_t)t * (kBDig >> 4));
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (!FULL && k >= ksteps) break;
      const uint64_t ko = (uint64_t)(k & 3) * 2;
      mma_one(d, ad + (uint64_t)(k >> 2) * (kADig >> 5) + ko,
                   bd + (uint64_t)(k >> 2) * (kBDig >> 5) + ko, idesc,
                   k == 0 ? (a == 0 ? 0u : 1u) : 1u, elect);
    }
  }
}

template <class Src>
__global__ void __launch_bounds__(kThreadsF64, 1)
    k_kron_f64_tc(const __grid_constant__ Src src, const F64Launch L) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* bdig = base;
  unsigned char* blead = base + kDg * kBDig;
  unsigned char* adig = blead + kBLead;
  uint64_t* afull = (uint64_t*)(adig + kABufs * kADig);
  uint64_t* aempty = afull + kABufs;
  uint64_t* ready = aempty + kABufs;  // B digits written, D of the step before drained
  uint64_t* dfull = ready + 1;        // [7] D_s complete, B digit 6 - s no longer read
  uint64_t* kfull = dfull + kDg;      // [2] keys of an even / odd step written
  uint64_t* kfree = kfull + 2;        // [2] and no longer read
  uint64_t* drain = kfree + 2;
  uint64_t* stall = drain + 1;  // never completed (time-out test)
  uint32_t* tmem_slot = (uint32_t*)(stall + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  // per (step parity, converter k group, vector): largest magnitude key; then
  // per (parity, vector): the key, and per (parity, warp) whether any vector of
  // the step needs more than the exponent addition
  int* cmax = (int*)(tmem_slot + 2);     // [2][4][64]
  int* ckey = cmax + 8 * kVec;           // [2][64]
  volatile int* cfar = ckey + 2 * kVec;  // [2][2]
  // per drainer thread: the outputs of its step with too small a sum of leading
  // magnitudes; entries of L.low so far
  volatile uint32_t* clow = (volatile uint32_t*)(cfar + 4);  // [32 kDrainWarps]
  int* nlow = (int*)(clow + 32 * kDrainWarps);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kABufs; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
    }
    mbar_init(ready, kConvWarps + kDrainWarps);
    for (int t = 0; t < kDg; ++t) mbar_init(&dfull[t], 1);
    for (int q = 0; q < 2; ++q) {
      mbar_init(&kfull[q], kConvWarps);
      mbar_init(&kfree[q], kDrainWarps);
    }
    mbar_init(drain, 1);
    mbar_init(stall, 1);
    *abort_flag = 0;
    *nlow = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int ntiles = src.count();

  if (warp == kLoadWarp) {
    // -------------------------------------------------- factor digit copies
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0, issued = 0, issued_ph = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        int lt;
        const F64Params& p = src.get(tile, lt);
        const int kchunks = p.kchunks, nc = lt % p.nchunks;
        const int kb_last = (p.n_in - (kchunks - 1) * kKc + 63) / 64;  // k blocks, last chunk
        const unsigned char* img =
            (const unsigned char*)p.img + (int64_t)nc * kchunks * (int64_t)kABlk;
        for (int kc = 0; kc < kchunks && ok; ++kc, img += kABlk) {
          // the leading magnitudes (after the digits in the image), then the digits
          for (int a = -1; a < kDg; ++a) {
            const uint32_t bytes = a < 0 ? kALead : (kc == kchunks - 1 ? kb_last : 2) * (kADig / 2);
            if (!mbar_wait(&aempty[s], ph ^ 1u, abort_flag, L.err)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&afull[s], bytes);
            bulk_g2s(adig + s * kADig, img + (a < 0 ? kDg : a) * kADig, bytes, &afull[s]);
            issued |= 1u << s;
            issued_ph = (issued_ph & ~(1u << s)) | (ph << s);
            if (++s == kABufs) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
      }
      // the latest copy into each buffer is the only one that can be in flight
      for (int b = 0; b < kABufs; ++b)
        if (issued & (1u << b)) mbar_wait_own(&afull[b], (issued_ph >> b) & 1u, L.err);
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA
    // the whole warp runs the loop, one elected lane issues
    const uint32_t elect = elect_one();
    constexpr uint32_t idesc = idesc_f16(kOut, kVec);
    bool ok = true;
    if (L.stall_ns)
      ok = __all_sync(0xffffffffu, mbar_wait_slow(stall, 0, abort_flag, L.err, L.stall_ns));
    const uint64_t adesc = sw128_desc(smem_u32(adig)), bdesc = sw128_desc(smem_u32(bdig));
    const uint64_t ldesc = sw128_desc(smem_u32(blead));
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);
    int s = 0;
    uint32_t ph = 0, sph = 0;
    for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      int lt;
      const F64Params& p = src.get(tile, lt);
      const int kchunks = p.kchunks, n_in = p.n_in;
      for (int kc = 0; kc < kchunks && ok; ++kc, sph ^= 1u) {
        const int kleft = n_in - kc * kKc;
        const int ksteps = kleft >= kKc ? 8 : (kleft + 15) / 16;
        ok = mbar_wait_warp(ready, sph, abort_flag, L.err);
        if (!ok) break;
        tc_fence_after();
        // the sums of leading magnitudes (complete and its operands free with group 0)
        ok = mbar_wait_warp(&afull[s], ph, abort_flag, L.err);
        if (!ok) break;
        tc_fence_after();
        {
          const uint64_t ad = adesc + (uint64_t)((uint32_t)s * (kADig >> 4));
          const int lsteps = (min(kleft, kKc) + 31) / 32;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (k >= lsteps) break;
            mma_one_f8(tmem + kDg * kVec, ad + (uint64_t)k * 2, ldesc + (uint64_t)k * 2,
                       idesc_e5m2(kOut, kVec), k ? 1u : 0u, elect);
          }
          mma_commit_one(&aempty[s], elect);
          if (++s == kABufs) {
            s = 0;
            ph ^= 1u;
          }
        }
        for (int a = 0; a < kDg; ++a) {
          ok = mbar_wait_warp(&afull[s], ph, abort_flag, L.err);
          if (!ok) break;
          tc_fence_after();
          // descriptors advance by address / 16: 2 per 16-wide k step
          const uint64_t ad = adesc + (uint64_t)((uint32_t)s * (kADig >> 4));
          if (ksteps == 8)
            issue_group<true>(tmem, ad, bdesc, idesc, a, 8, elect);
          else
            issue_group<false>(tmem, ad, bdesc, idesc, a, ksteps, elect);
          mma_commit_one(&dfull[a], elect);
          mma_commit_one(&aempty[s], elect);
          if (++s == kABufs) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
    }
    // the elected lane's commit covers every MMA it issued
    mma_commit_one(drain, elect);
    if (elect) mbar_wait_own(drain, 0, L.err);
    __syncwarp();
  } else if (warp < kConvWarps) {
    // ----------------------------------------------------------- converters
    // vector n of the tile, 8-entry k runs at k = 8 oct + 32 h, h < 4
    const int n = (warp & 1) * 32 + lane, oct = warp >> 1;
    unsigned long long u[32];
    auto load = [&](const F64Params& p, const F64Step& s) {
      const int m = s.m0 + n;
      const double* x = p.X + s.r * p.size_in + m;
      const int k0 = s.kc * kKc + oct * 8;
      if (m < p.rest && k0 + 104 <= p.n_in) {
        x += (int64_t)k0 * p.rest;
#pragma unroll
        for (int e = 0; e < 32; ++e)
          u[e] = (unsigned long long)__double_as_longlong(
              __ldg(x + ((e & 7) + (e >> 3) * 32) * p.rest));
        return;
      }
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        const int k = k0 + (e & 7) + (e >> 3) * 32;
        u[e] = (m < p.rest && k < p.n_in)
                   ? (unsigned long long)__double_as_longlong(x[k * p.rest])
                   : 0ull;
      }
    };
    int tile = blockIdx.x, kc = 0;
    if (tile < ntiles) {
      int lt;
      const F64Params& p = src.get(tile, lt);
      load(p, step_of(p, lt, 0));
    }
    bool ok = true;
    for (int st = 0; tile < ntiles; ++st) {
      int lt;
      const F64Params& p = src.get(tile, lt);
      const int par = st & 1;
      uint32_t xh = 0, xl = 0;
#pragma unroll
      for (int e = 0; e < 32; ++e) mag_key(u[e], xh, xl);
      cmax[(par * 4 + oct) * kVec + n] = (int)(xh | (xh == 0 && xl != 0 ? 1u : 0u));
      asm volatile("bar.sync 1, 256;" ::: "memory");
      int key = 0;
#pragma unroll
      for (int o = 0; o < 4; ++o) key = max(key, cmax[(par * 4 + o) * kVec + n]);
      const int emax = key >> 20;
      const bool dig = key != 0 && has_digits(key);
      if (st > 1) {  // the drainers are done with the keys of step st - 2
        if (ok) ok = mbar_wait(&kfree[par], (uint32_t)((st >> 1) + 1) & 1u, abort_flag, L.err);
        ok = __all_sync(0xffffffffu, ok);
      }
      if (oct == 0) {
        ckey[par * kVec + n] = key;
        const bool any = __any_sync(0xffffffffu, far_key(key));
        if (lane == 0) cfar[par * 2 + warp] = any;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&kfull[par]);
#pragma unroll
      for (int e = 0; e < 32; ++e) u[e] = dig ? fixed_digits<2>(u[e], emax) : kZeroDigits;
        // keep the conversion ahead of the waits below, beside the MMAs
#pragma unroll
      for (int e = 0; e < 32; ++e) asm volatile("" : "+l"(u[e]));
      const int kpad = (min(p.n_in - kc * kKc, kKc) + 15) / 16 * 16;
      // digit 6 - S is free once MMA group S of the step before is done
      const uint32_t dph = (uint32_t)((st + 1) & 1);
#define COLA_DIGIT(S)                                                      \
  if (st > 0) {                                                            \
    if (ok) ok = mbar_wait(&dfull[S], dph, abort_flag, L.err);             \
    ok = __all_sync(0xffffffffu, ok);                                      \
  }                                                                        \
  if constexpr (S < 6)                                                     \
    put_digit<6 - S>(bdig, u, n, oct, kpad);                               \
  else                                                                     \
    put_lead(bdig, blead, u, n, oct, kpad, cmax + par * 4 * kVec + n);
      COLA_DIGIT(0)
      COLA_DIGIT(1)
      COLA_DIGIT(2)
      COLA_DIGIT(3)
      COLA_DIGIT(4)
      COLA_DIGIT(5)
      COLA_DIGIT(6)
#undef COLA_DIGIT
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(ready);
      const bool wrap = kc + 1 == p.kchunks;
      tile = wrap ? tile + (int)gridDim.x : tile;
      kc = wrap ? 0 : kc + 1;
      if (tile < ntiles) {
        int nlt;
        const F64Params& q = src.get(tile, nlt);
        load(q, step_of(q, nlt, kc));
        // the block after it: DRAM to L2, two 128-byte lines a thread
        const bool wrap2 = kc + 1 == q.kchunks;
        const int t2 = wrap2 ? tile + (int)gridDim.x : tile;
        if (t2 < ntiles) {
          int lt2;
          const F64Params& n2 = src.get(t2, lt2);
          const F64Step f = step_of(n2, lt2, wrap2 ? 0 : kc + 1);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int k = f.kc * kKc + (tid >> 2) + 64 * h, m = f.m0 + (tid & 3) * 16;
            if (k < n2.n_in && m < n2.rest)
              asm volatile("prefetch.global.L2 [%0];" ::"l"(n2.X + f.r * n2.size_in +
                                                             (int64_t)k * n2.rest + m));
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------- drainers
    // output lane 32 (warp mod 4) + lane, 32 vectors from oc0
    const int orow = (warp & 3) * 32 + lane, oc0 = ((warp - kConvWarps) >> 2) * 32;
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)oc0;
    long long acc[32];
    int tile = blockIdx.x, kc = 0;
    bool ok = true;
    if (tile < ntiles && lane == 0) mbar_arrive(ready);  // nothing to drain before step 0
    for (int st = 0; tile < ntiles; ++st) {
      int lt;
      const F64Params& p = src.get(tile, lt);
      const int par = st & 1;
      const int nc = lt % p.nchunks;
      // the factor row's exponent, ahead of its use in the store
      const int ef2 = __ldg(&p.fexp[((int64_t)nc * p.kchunks + kc) * kOut + orow]);
#define COLA_DIGIT(S)                                                      \
  if (ok) ok = mbar_wait(&dfull[S], (uint32_t)par, abort_flag, L.err);     \
  ok = __all_sync(0xffffffffu, ok);                                        \
  tc_fence_after();                                                        \
  if (ok) {                                                                \
    if constexpr (S == 0) clow[tid - 32 * kConvWarps] = low_outputs(taddr, ef2 & 1); \
    fold<S>(taddr, acc);                                                   \
  }
      COLA_DIGIT(0)
      COLA_DIGIT(1)
      COLA_DIGIT(2)
      COLA_DIGIT(3)
      COLA_DIGIT(4)
      COLA_DIGIT(5)
      COLA_DIGIT(6)
#undef COLA_DIGIT
      tc_fence_before();
      __syncwarp();
      const bool more = kc + 1 < p.kchunks || tile + (int)gridDim.x < ntiles;
      if (lane == 0 && more) mbar_arrive(ready);
      if (ok) ok = mbar_wait(&kfull[par], (uint32_t)(st >> 1) & 1u, abort_flag, L.err);
      ok = __all_sync(0xffffffffu, ok);
      const F64Step cur = step_of(p, lt, kc);
      const int i = nc * kOut + orow;
      const int cnt = min(32, p.rest - cur.m0 - oc0);
      if (ok && i < p.n_out && cnt > 0) {
        double* y = p.Y + cur.r * p.size_out + (int64_t)(cur.m0 + oc0) * p.n_out + i;
        const int* keys = ckey + par * kVec + oc0;
        uint32_t low = clow[tid - 32 * kConvWarps];  // outputs that take plain products
        const int ef = ef2 >> 1;
        const bool near = abs(ef) <= kFarExp && !(cfar[par * 2] | cfar[par * 2 + 1]);
        const int e0 = ef - 53 - 1023;
        // Y's old values join with beta (first k chunk) or 1 (later chunks)
        const bool old = kc > 0 || p.has_beta;
        const double bo = kc > 0 ? 1.0 : p.beta;
        auto leave_out = [&](uint32_t mask) {
          uint32_t* e = L.low + 3 * ((int64_t)blockIdx.x * L.low_cap + atomicAdd(nlow, 1));
          e[0] = (uint32_t)((tile - (int)blockIdx.x) / (int)gridDim.x * (32 * kDrainWarps) +
                            tid - 32 * kConvWarps);
          e[1] = (uint32_t)kc;
          e[2] = mask;
        };
        // where nothing is added to, the plain products write over their outputs
        const bool over = p.kchunks == 1 && !p.has_beta;
        if (near && (low == 0 || over) && cnt == 32) {  // no branch per output
#pragma unroll
          for (int g = 0; g < 32; g += 4) {
            double v[4];
            if (old) {
#pragma unroll
              for (int c = 0; c < 4; ++c) v[c] = y[(g + c) * p.n_out];
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              double w = scaled_double(acc[g + c], e0 + (keys[g + c] >> 20));
              if (p.has_alpha) w *= p.alpha;
              if (old) w = fma(bo, v[c], w);
              y[(g + c) * p.n_out] = w;
            }
          }
          if (low != 0) leave_out(low);
        } else {
          if (cnt < 32) low &= (1u << cnt) - 1;
#pragma unroll 1
          for (int c = 0; c < cnt; ++c) {
            long long ac = 0;
#pragma unroll
            for (int q = 0; q < 32; ++q)
              if (q == c) ac = acc[q];
            const int key = keys[c], e = e0 + (key >> 20);
            const double yo = old ? *y : 0.0;
            if (abs(ef) > kFarExp || far_key(key)) {  // out of scaled_double's range
              low |= 1u << c;
            } else if (low >> c & 1u) {
              // too small a sum of leading magnitudes, except where the digits' error, below
              // 2^-51 K 2^(Ef + Ex), is hidden by the rounding of a sum so far of at least
              // 2^kHidden of that binade
              if (kc > 0 && fabs(yo) >= fabs(p.alpha) *
                                            __hiloint2double((1023 + 53 + kHidden + e) << 20, 0))
                low ^= 1u << c;
            }
            double v = scaled_double(low >> c & 1u ? 0ll : ac, e);
            if (p.has_alpha) v *= p.alpha;
            if (old) v = fma(bo, yo, v);
            *y = v;
            y += p.n_out;
          }
          if (low != 0) leave_out(low);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&kfree[par]);
      if (++kc == p.kchunks) {
        kc = 0;
        tile += gridDim.x;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(512)
                 : "memory");
  }
  // The outputs left out above, on the FP64 units (their rate bounds it: 300 us a
  // tile whose outputs are all plain).  Y is this CTA's own.
  // One k chunk after the other, as an output may be left out of several; eight columns
  // of an entry to a thread, so that a few entries still reach every warp.
  const int entries = *abort_flag ? 0 : *nlow;
  for (int kc = 0; kc < (entries ? L.kmax : 0); ++kc) {
    for (int64_t u = tid; u < 4 * (int64_t)entries; u += kThreadsF64) {
      const int n = (int)(u % entries);
      const uint32_t* e = L.low + 3 * ((int64_t)blockIdx.x * L.low_cap + n);
      const uint32_t mask = e[2] & 0xffu << (8 * (int)(u / entries));
      if (e[1] != (uint32_t)kc || mask == 0) continue;
      const int thr = e[0] % (32 * kDrainWarps);
      int lt;
      const F64Params& p = src.get(
          (int)blockIdx.x + (int)(e[0] / (32 * kDrainWarps)) * (int)gridDim.x, lt);
      const F64Step cur = step_of(p, lt, kc);
      const int i = cur.nc * kOut + thr % kOut, m = cur.m0 + thr / kOut * 32;
      plain_columns(p, mask, kc * kKc, min(p.n_in, (kc + 1) * kKc), p.F + i * p.f_i,
                    p.X + cur.r * p.size_in + m,
                    p.Y + cur.r * p.size_out + (int64_t)m * p.n_out + i);
    }
    __syncthreads();
  }
}

}  // namespace

// The list of outputs left to plain products, for `ntiles` tiles of at most
// kchunks k chunks (5 % of Y's bytes per chunk); false when it does not fit.  One buffer
// per power of two of bytes, which never moves (see f64_tc_mode_step).
static bool f64_low_list(Ctx* c, int ntiles, int kchunks, F64Launch* L) {
  const int grid = std::min(ntiles, c->num_sms), per = (ntiles + grid - 1) / grid;
  if (per >= 1 << 24) return false;
  L->low_cap = (int64_t)per * kchunks * (32 * kDrainWarps);
  L->kmax = kchunks;
  const size_t bytes = 12 * (size_t)grid * L->low_cap;
  int lg = 16;
  while (((size_t)1 << lg) < bytes) ++lg;
  L->low = (uint32_t*)c->optional_ws("f64.low" + std::to_string(lg), (size_t)1 << lg);
  return L->low != nullptr;
}

template <class Src>
static void f64_launch(Ctx* c, const Src& src, int ntiles, F64Launch L) {
  L.err = tc_errflag(c);
  if (c->tc_stall_ns > 0 && !c->capturing) {
    L.stall_ns = (uint64_t)c->tc_stall_ns;  // armed once by cola_test_stall_next_launch
    c->tc_stall_ns = 0;
  }
  COLA_CUDA(cudaFuncSetAttribute(k_kron_f64_tc<Src>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmemF64));
  k_kron_f64_tc<Src><<<std::min(ntiles, c->num_sms), kThreadsF64, kSmemF64, c->s>>>(src, L);
  c->count_launch();
  c->f64_tc_used = true;
  COLA_CUDA(cudaGetLastError());
}

size_t f64_image_bytes(int64_t n_out, int64_t n_in) {
  return (size_t)((n_out + kOut - 1) / kOut) * (size_t)((n_in + kKc - 1) / kKc) *
         (kABlk + kOut * 4);
}

void f64_factor_image(Ctx* c, const double* F, int64_t f_i, int64_t f_j, int n_out, int n_in,
                      void* mem) {
  const int nch = (n_out + kOut - 1) / kOut, kch = (n_in + kKc - 1) / kKc;
  k_f64_digits<<<dim3(kOut, (unsigned)nch, (unsigned)kch), kKc, 0, c->s>>>(
      F, f_i, f_j, n_out, n_in, kch, (uint16_t*)mem,
      (int*)((char*)mem + (size_t)nch * kch * kABlk));
  c->count_launch();
  COLA_CUDA(cudaGetLastError());
}

bool f64_tc_batch(Ctx* c, const std::vector<F64Batch>& probs, const char* tag) {
  std::vector<F64Params> hp(probs.size());
  std::vector<int> first(probs.size()), tile_prob;
  for (size_t i = 0; i < probs.size(); ++i) {
    const F64Batch& b = probs[i];
    F64Params& p = hp[i];
    p = F64Params{};
    p.nchunks = (b.n_out + kOut - 1) / kOut;
    p.kchunks = (b.n_in + kKc - 1) / kKc;
    p.tiles_m = (b.rest + kVec - 1) / kVec;
    p.ntiles = (int)(b.R * p.tiles_m * p.nchunks);
    p.X = b.X;
    p.Y = b.Y;
    p.F = b.F;
    p.f_i = b.n_in;
    p.f_j = 1;
    p.img = (const uint16_t*)b.image;
    p.fexp = (const int*)((const char*)b.image + (size_t)p.nchunks * p.kchunks * kABlk);
    p.rest = b.rest;
    p.n_in = b.n_in;
    p.n_out = b.n_out;
    p.size_in = b.size_in;
    p.size_out = b.size_out;
    p.alpha = b.alpha;
    p.beta = b.beta;
    p.has_alpha = b.alpha != 1.0;
    p.has_beta = b.beta != 0.0;
    first[i] = (int)tile_prob.size();
    tile_prob.insert(tile_prob.end(), (size_t)p.ntiles, (int)i);
  }
  const int nt = (int)tile_prob.size(), np = (int)probs.size();
  if (nt == 0) return true;
  int kmax = 1;
  for (const F64Params& p : hp) kmax = std::max(kmax, p.kchunks);
  F64Launch L{};
  if (!f64_low_list(c, nt, kmax, &L)) return false;
  const std::string t = tag;
  F64Tab src{};
  src.probs = (const F64Params*)c->ws.get(t + ".p", sizeof(F64Params) * np);
  src.tile_prob = (const int*)c->ws.get(t + ".t", 4 * (size_t)nt);
  src.first = (const int*)c->ws.get(t + ".f", 4 * (size_t)np);
  src.ntiles = nt;
  COLA_CUDA(cudaMemcpyAsync((void*)src.probs, hp.data(), sizeof(F64Params) * np,
                            cudaMemcpyHostToDevice, c->s));
  COLA_CUDA(cudaMemcpyAsync((void*)src.tile_prob, tile_prob.data(), 4 * (size_t)nt,
                            cudaMemcpyHostToDevice, c->s));
  COLA_CUDA(cudaMemcpyAsync((void*)src.first, first.data(), 4 * (size_t)np,
                            cudaMemcpyHostToDevice, c->s));
  f64_launch(c, src, nt, L);
  COLA_CUDA(cudaStreamSynchronize(c->s));  // the host tables go out of scope
  return true;
}

bool f64_tc_mode_step(Ctx* c, int64_t rest, int n_out, int n_in, double alpha, const double* X,
                      int64_t size_in, const double* F, int64_t f_i, int64_t f_j, double beta,
                      double* Y, int64_t size_out, int64_t R) {
  F64Params p{};
  p.nchunks = (n_out + kOut - 1) / kOut;
  p.kchunks = (n_in + kKc - 1) / kKc;
  const int64_t tiles_m = (rest + kVec - 1) / kVec;
  // indices within one vector block and tile numbers are 32-bit
  if (rest * std::max(n_in, n_out) >= ((int64_t)1 << 31) - 1024 ||
      R * tiles_m * p.nchunks * p.kchunks >= ((int64_t)1 << 31) - 1024)
    return false;
  p.tiles_m = (int)tiles_m;
  p.ntiles = (int)(R * tiles_m * p.nchunks);
  const size_t blocks = (size_t)p.nchunks * p.kchunks;
  if (p.nchunks > 65535 || p.kchunks > 65535 || blocks > 1024) return false;
  // One buffer per power of two of blocks, which never grows (0.5 GB for all of
  // them): a graph that a caller captured around a product keeps its image when a
  // later product has a larger factor.
  size_t cap = 1;
  while (cap < blocks) cap *= 2;
  const std::string cls = std::to_string(cap);
  uint16_t* img = (uint16_t*)c->optional_ws("f64.img" + cls, cap * kABlk);
  int* fexp = (int*)c->optional_ws("f64.exp" + cls, cap * kOut * 4);
  F64Launch L{};
  if (!img || !fexp || !f64_low_list(c, p.ntiles, p.kchunks, &L)) return false;
  k_f64_digits<<<dim3(kOut, (unsigned)p.nchunks, (unsigned)p.kchunks), kKc, 0, c->s>>>(
      F, f_i, f_j, n_out, n_in, p.kchunks, img, fexp);
  c->count_launch();
  p.X = X;
  p.Y = Y;
  p.F = F;
  p.img = img;
  p.fexp = fexp;
  p.f_i = f_i;
  p.f_j = f_j;
  p.rest = (int)rest;
  p.size_in = size_in;
  p.size_out = size_out;
  p.n_in = n_in;
  p.n_out = n_out;
  p.alpha = alpha;
  p.beta = beta;
  p.has_alpha = alpha != 1.0;
  p.has_beta = beta != 0.0;
  f64_launch(c, F64One{p}, p.ntiles, L);
  return true;
}

}  // namespace cola
