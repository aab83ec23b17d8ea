// Spectral derivative along one axis (Sec. 2.2: the derivatives are taken
// with FFTs) as a dense contraction on the 5th-generation tensor cores, for
// the FP64 form.
//
// Along axis j the FFT derivative d_j f = IFFT_j[i (k + theta/L) FFT_j[f]] is
// one linear map applied to every line of n points: the circulant n x n
// complex matrix
//     D[m][q] = d[(m - q) mod n],  d[r] = (i / n) sum_a kappa_a e^{2 pi i a r / n},
// kappa_a = (2 pi a' + theta) / L with a' = a or a - n (FFT order; the Nyquist
// wavenumber kept, as in the line passes).  On the interleaved (re, im)
// storage it is the real 2n x 2n matrix
//     Dr[2m + c'][2q + c] = [[Re D, -Im D], [Im D, Re D]][c'][c],
// so one pass over nb arrays is OUT = LINES Dr^T with one row per line
// (nb G / n rows, K = N = 2n, padded to NC = a multiple of 16).  Both
// operands are cut into six base-256 digits (oz_digits.cuh), each line scaled
// by its own exponent and each row of Dr by its own; digit s is kept as the bf16
// number alpha_s 2^{-8(s+1)} (exact), so that digit products carry their own
// weight.  The 21 products of weight g = s + t <= 5 are summed in FP32 in TMEM:
// weights 0-3 exactly, one accumulator each (per K value |G_g| <= (g + 3) 2^14
// units, K <= 64, so every sum stays an integer below 2^24 units), weights 4 and
// 5 together in a fifth; its FP32 rounding, at most K 2^-24 of a sum below 2^23
// at weight 2^-32, is about 2^-49 of the largest term.  The accumulators lie
// side by side and the operator's digits one below the other, so digit p of the
// lines times digits 0 .. 4 - p of the operator is one MMA of (5 - p) NC columns
// into the accumulators p .. 4 (two for NC = 64, p = 0): 11 MMAs per 16 values
// of K instead of 21 (24^3, 280 states: 116 us per pass with 21 issued by one
// lane of a diverged warp, 100 us; 84 us with pairs out).  The sums are combined exactly in a 64-bit
// integer, rounded once to FP64 and scaled by the two exponents, or, for arrays
// that stay inside h psi, into a pair of floats by error-free additions.  The
// error is that rounding plus the truncated digit expansion, about 2^-48 of the
// line's and the row's largest values.
//
// Arrays between the passes of h psi hold float pairs (re hi, re lo, im hi, im
// lo in the 16 bytes of a complex double): the digits of a pair and the sum of
// the accumulators into a pair are FP32 operations (about 26 and 30 per real),
// where doubles take integer work at half the FP32 rate (about 35 and 50
// instructions).  All of h psi, 24^3, 280 states: 1393 us with doubles between
// the passes, 845 us; what is left is issue (60% of the slots) and the latency of
// the loads ahead of each block.
//
// Persistent kernel, one CTA per SM, 128 lines per tile:
//   warps 0-7   producers: warp w takes lines 16 w .. 16 w + 15 of the tile,
//               lanes 0-15 the first half of each line's points and lanes
//               16-31 the second; a thread loads its half line at once, the
//               pair agrees on the line's exponent by one shuffle, and each
//               writes its digits into a ring stage in the canonical
//               no-swizzle K-major layout (8-row x 16-byte core matrices),
//               fences the writes for the tensor core's proxy and arrives;
//   warp 8      owns TMEM (two accumulator sets of 5 x NC fp32 columns, so
//               the MMAs of one tile run while the epilogue drains the
//               previous one; one set when 5 NC > 256); it stays converged and
//               one elected lane executes tcgen05.mma (M = 128, K = 16);
//   warps 9-16  epilogue: two warps per TMEM lane quadrant, half the columns
//               each, in blocks of 8 columns; they combine the groups into
//               64-bit integers, round, scale and store the (re, im) pairs at
//               the line's points (in place is allowed: tiles own disjoint
//               lines), then hand the accumulator set back.
// The operator's digits, computed once per context on the host in long
// double, stay in shared memory for the whole launch.  Every mbarrier wait is
// bounded; a timeout sets SKY_ETIMEOUT, the kernel waits (bounded) for the
// MMAs it issued, frees TMEM and returns.
#include <cmath>
#include <cstring>
#include <vector>

#include <type_traits>

#include "dd.cuh"
#include "oz_digits.cuh"
#include "oz_gemm.cuh"

namespace sky {
namespace ozd {

using namespace ozdig;
using tc::fence_after;
using tc::fence_before;
using tc::idesc_bf16;
using tc::mbar_init;
using tc::mbar_wait;
using oz::elect_one;
using oz::mbar_wait_warp;
using oz::mma_bf16_elect;
using oz::mma_commit_elect;
using tc::smem_u32;

constexpr int S = 6;               // digits per operand (FP64 inputs)
constexpr int BM = 128;            // lines per tile (MMA M)
constexpr int kProd = 8, kEpi = 8;   // producer warps: two threads per line
constexpr int THREADS = 32 * (kProd + 1 + kEpi);
constexpr int kSmemMax = 232448;   // dynamic shared memory opt-in limit per CTA
constexpr int kBars = 24;
constexpr int NG = 5;              // TMEM groups: weights 0, 1, 2, 3 and {4, 5}

__host__ __device__ constexpr int nc_of(int n) { return ((2 * n + 15) / 16) * 16; }

// Operators of an axis: the derivative, the forward and the inverse DFT.
constexpr int kOpDeriv = 0, kOpFwd = 1, kOpInv = 2;
// Producer input: the lines of src, the residual src - eps psi (src = h psi), or
// lines of float pairs.
constexpr int kInPlain = 0, kInResidual = 1, kInPair = 2;
// Epilogue output: the product; times P[point] scale; psi - w[point] times it; as
// pairs; added to the pairs in dst; the sum of that addition as FP64.
constexpr int kOutPlain = 0, kOutScaleP = 1, kOutUpdate = 2, kOutPair = 3, kOutAddPair = 4,
              kOutAddF64 = 5;

template <int N>
struct Shape {
  static constexpr int NC = nc_of(N);          // K and output columns (reals), padded
  static constexpr int TILE_A = BM * NC * 2;   // one digit of a tile of lines
  static constexpr int STAGE = S * TILE_A;
  static constexpr int TILE_B = NC * NC * 2;   // one digit of the operator
  static constexpr int OPB = S * TILE_B;       // its digits
  static constexpr int NBUF = NG * NC <= 256 ? 2 : 1;   // TMEM accumulator sets
  static constexpr int AUX = NC * 4 + 2 * BM * 4 + kBars * 8 + 16;
  static constexpr int H0 = ((N / 2 + 3) / 4) * 4;             // points of a line's first half
  // staging of the next tile's lines when it fits beside one ring stage: one
  // 16-byte slot per point of each producer thread's half line, or, along x, the
  // warp's 16 lines as they lie in memory, padded by a point each
  static constexpr int STG_Y = H0 * kProd * 32 * 16, STG_X = kProd * 16 * (N + 1) * 16;
  static constexpr int STG_BYTES = STG_Y > STG_X ? STG_Y : STG_X;
  static constexpr bool PREFETCH = STAGE + OPB + AUX + STG_BYTES + 1024 <= kSmemMax;
  static constexpr int STG = PREFETCH ? STG_BYTES : 0;
  static constexpr int STAGES = (2 * STAGE + OPB + AUX + STG + 1024 <= kSmemMax) ? 2 : 1;
  static constexpr int SMEM = STAGES * STAGE + OPB + AUX + STG + 1024;
  static constexpr int HALF = NC / 2;          // columns per epilogue warp
  static_assert(NG * NC <= 512, "TMEM columns");
  static_assert(SMEM <= kSmemMax, "shared memory");
  static_assert(HALF % 8 == 0, "TMEM load blocks of 8 columns");
  static_assert(NC <= 64, "int32 bounds of the group combination");
};

// Byte offset of element (r, k) of a K-major bf16 tile with nc columns in the
// canonical no-swizzle layout: 8 x 8 core matrices of 128 contiguous bytes,
// 128 bytes apart along K, 16 nc bytes apart along the rows.
__host__ __device__ constexpr int cm_off(int r, int k, int nc) {
  return (r >> 3) * (nc * 16) + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}
// Shared-memory matrix descriptor of that layout: leading byte offset 128
// (core matrices along K), stride byte offset 16 nc (8-row groups), version 1,
// layout type 0 (no swizzle); low word by address, high word fixed.
__device__ __forceinline__ uint32_t ns_lo(uint32_t saddr) {
  return ((saddr >> 4) & 0x3FFFu) | ((128u >> 4) << 16);
}
__host__ __device__ constexpr uint32_t ns_hi(int nc) { return (uint32_t)((nc * 16) >> 4) | (1u << 14); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// 16-byte asynchronous copy global -> shared (zero fill when !valid).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// 2^k as a float, k in [-150, 128] (subnormal below -126, 0 at -150, infinity at 128).
__device__ __forceinline__ float pow2f(int k) {
  return __int_as_float(k >= -126 ? (k + 127) << 23 : 0x00400000 >> (-127 - k));
}
// The six balanced base-256 digits of the signed integer Y = +-round(|x|
// 2^{48 - E}) (|Y| <= 2^48), digit s as the float alpha_s 2^{-8(s+1)}: adding 128
// to each of the five lower byte positions (0x8080808080) turns every lower
// byte, minus 128, into a digit in [-128, 127], with the carries propagated by
// the addition; the top digit is the rest, an arithmetic shift (|digit 0| <=
// 256).  A byte placed below the bits of 2^23 u (u the digit's unit) is that
// float plus byte u; subtracting (2^23 + 128) u leaves the digit, exactly.
__device__ __forceinline__ void digits6f(double x, int E, float* d) {
  long long Y = (long long)fixed_of<6>(x, E);
  if (sign_of(x)) Y = -Y;
  const long long Z = Y + 0x8080808080LL;
  const unsigned lo = (unsigned)Z, hi = (unsigned)((unsigned long long)Z >> 32);
  constexpr unsigned kOne = 0x4B000000u, kU = 8u << 23;     // 2^23; one unit step
  auto f = [](unsigned word, unsigned sel, unsigned steps) {
    const unsigned m = kOne - steps * kU;
    return __uint_as_float(__byte_perm(word, m, sel)) - (__uint_as_float(m) + 128.0f * __uint_as_float(0x3F800000u - steps * kU));
  };
  d[5] = f(lo, 0x7650, 6);
  d[4] = f(lo, 0x7651, 5);
  d[3] = f(lo, 0x7652, 4);
  d[2] = f(lo, 0x7653, 3);
  d[1] = f(hi, 0x7650, 2);
  d[0] = __int_as_float((int)(0x4B400000u - kU) + (int)(Z >> 40)) - __uint_as_float(0x4B400000u - kU);
}
// The same digits of a float pair scaled to |h + l| <= 1 (h = fl(h + l)): each
// digit is the part of the remainder above half a unit, cut off by adding and
// subtracting 1.5 2^23 units; three digits take h's 24 bits, then l joins the
// remainder (its rounding there is below 2^-49).
__device__ __forceinline__ void digits6p(float h, float l, float* d) {
  auto cut = [](float r, int s) {
    const float m = 12582912.0f * __uint_as_float(0x3F800000u - (unsigned)(s + 1) * (8u << 23));
    return __fsub_rn(__fadd_rn(r, m), m);
  };
  float r = h;
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    d[s] = cut(r, s);
    r = __fsub_rn(r, d[s]);
    if (s == 2) r = __fadd_rn(r, l);
  }
  d[5] = cut(r, 5);
}
// The accumulators g0 .. g4 (decreasing weight) as a float pair.
__device__ __forceinline__ dd pair_of_groups(float g0, float g1, float g2, float g3, float g4) {
  const dd a = two_sum(g0, g1), b = two_sum(g2, g3);
  const dd u = two_sum(a.lo, b.hi);
  const dd t = two_sum(a.hi, u.hi);
  return fast_two_sum(t.hi, __fadd_rn(t.lo, __fadd_rn(u.lo, __fadd_rn(b.lo, g4))));
}
// An exponent whose power of two pow2f forms: what is beyond the floats becomes 0 or
// infinity.
__device__ __forceinline__ int clamp_exp(int k) { return k < -150 ? -150 : k > 128 ? 128 : k; }
// exp_of for the lines of pairs, whose smallest values may be subnormal.
__device__ __forceinline__ int exp_of_pair(float x) { return x == 0.0f ? INT_MIN : max(exp_of(x), -126); }
__device__ __forceinline__ unsigned bf16x2(float lo, float hi) {   // lo in the low half
  unsigned r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// v 2^sc rounded to the nearest double (halfway cases away from zero), by
// integer operations on the bit pattern; results outside the normal range go
// through ldexp.
__device__ __forceinline__ double scaled_double(long long v, int sc) {
  if (v == 0) return 0.0;
  const unsigned long long neg = v < 0 ? (1ull << 63) : 0ull;
  const unsigned long long u = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int pb = 63 - __clzll((long long)u);   // position of the leading bit
  const int be = pb + sc + 1023;               // biased exponent of the result
  if (be < 1 || be > 2045) return ldexp((double)v, sc);
  unsigned long long r;
  if (pb > 52) {
    const int sh = pb - 52;
    r = ((u >> (sh - 1)) + 1ull) >> 1;           // 53 bits, rounded; 2^53 on carry
  } else {
    r = u << (52 - pb);
  }
  // r in [2^52, 2^53]: adding it to (be - 1) << 52 sets the implicit bit's
  // exponent and carries a rounding overflow into the exponent.
  return __longlong_as_double((long long)(neg | ((((unsigned long long)(be - 1)) << 52) + r)));
}

// n / d for 0 <= n < 2^31 by an invariant multiplier (Granlund and Montgomery,
// PLDI 1994): with L = ceil(log2 d) and p = 31 + L, m = ceil(2^p / d) < 2^32
// and floor(n / d) = floor(n m / 2^p), because n m / 2^p exceeds n / d by
// less than n / 2^p < 2^-L <= 1 / d; d = 1 is the identity.
struct FastDiv {
  unsigned d, m;
  int sh;   // p - 32
};
inline FastDiv make_fastdiv(unsigned d) {
  FastDiv f{d, 0u, 0};
  if (d > 1) {
    int L = 0;
    while ((1ull << L) < d) ++L;
    const int p = 31 + L;
    f.m = (unsigned)(((1ull << p) + d - 1) / d);
    f.sh = p - 32;
  }
  return f;
}
__device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv& f) {
  return f.d == 1 ? n : (__umulhi(n, f.m) >> f.sh);
}

// 4 x 4 transpose over the lanes of a quad: afterwards z[k] of lane j is what
// z[j] of lane k was.
__device__ __forceinline__ float4 shfl4(float4 v, int mask) {
  return make_float4(__shfl_xor_sync(0xffffffffu, v.x, mask), __shfl_xor_sync(0xffffffffu, v.y, mask),
                     __shfl_xor_sync(0xffffffffu, v.z, mask), __shfl_xor_sync(0xffffffffu, v.w, mask));
}
__device__ __forceinline__ void quad_transpose(float4 (&z)[4], int lane) {
#pragma unroll
  for (int h = 1; h <= 2; h <<= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i & h) continue;
      const float4 recv = shfl4(up ? z[i] : z[i + h], h);
      if (up) z[i] = recv;
      else z[i + h] = recv;
    }
  }
}

struct DerivArgs {
  const double2* src;   // nb arrays of G complex points (may equal dst)
  double2* dst;
  const uint4* op;      // operator digits, S * TILE_B bytes in the canonical layout
  const int* ope;       // operator row exponents [NC]
  int nx, ny, nz;
  long long G;
  long long nlines;   // < 2^31
  int ntiles;
  FastDiv div1, div2;   // by nx, then by nz (lines along y) or ny (lines along z)
  FastDiv div0;         // by ny nz (lines along x: the array of a line)
  const double2* psi;   // kInResidual: psi (src is h psi); kOutUpdate: psi of the update
  const double* eps;    // kInResidual: eps per state (array b is state b / 2)
  const double* P;      // kOutScaleP: factor per point, times scale
  double scale;
  const float* w;       // kOutUpdate: weight per point, or null for 1
  int* status;
};

// First point and stride of line l (lines of one axis, x fastest, then the
// remaining axes in storage order, then the array).
template <int N, int AXIS>
__device__ __forceinline__ long long line_base(const DerivArgs& a, long long l, long long& stride) {
  if constexpr (AXIS == 0) {
    stride = 1;
    return l * N;
  } else {
    const unsigned lu = (unsigned)l;
    const unsigned t = fdiv(lu, a.div1), x = lu - t * (unsigned)a.nx;
    const unsigned b = fdiv(t, a.div2);
    if constexpr (AXIS == 1) {
      const unsigned z = t - b * (unsigned)a.nz;
      stride = a.nx;
      return (long long)b * a.G + (long long)(z * (unsigned)(a.ny * a.nx) + x);
    } else {
      const unsigned y = t - b * (unsigned)a.ny;
      stride = (long long)a.nx * a.ny;
      return (long long)b * a.G + (long long)(y * (unsigned)a.nx + x);
    }
  }
}

// Index b of the array that line l belongs to.
template <int N, int AXIS>
__device__ __forceinline__ unsigned line_array(const DerivArgs& a, long long l) {
  const unsigned lu = (unsigned)l;
  if constexpr (AXIS == 0) return fdiv(lu, a.div0);
  else return fdiv(fdiv(lu, a.div1), a.div2);
}

template <int N, int AXIS, int IN, int OUT>
__global__ void __launch_bounds__(THREADS, 1) k_oz_deriv(const DerivArgs a) {
  using Sh = Shape<N>;
  constexpr int NC = Sh::NC, STAGES = Sh::STAGES, HALF = Sh::HALF;
  constexpr int TILE_A = Sh::TILE_A, TILE_B = Sh::TILE_B, STAGE = Sh::STAGE;
  constexpr uint32_t TMEM_COLS = 512;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((unsigned long long)smem_raw + 1023ull) & ~1023ull);
  unsigned char* opb = base;                                  // operator digits
  unsigned char* ring = base + Sh::OPB;                       // STAGES x STAGE
  unsigned char* stg = ring + STAGES * STAGE;                 // [H0][producer thread] 16 B
  int* s_eb = (int*)(stg + Sh::STG);                          // [NC]
  int* s_ea = s_eb + NC;                                      // [2][BM]
  unsigned long long* bars = (unsigned long long*)(s_ea + 2 * BM);
  uint32_t* tmem_slot = (uint32_t*)(bars + kBars);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (2 + s); };
  auto acc_full = [&](int b) { return bar0 + 8u * (4 + b); };
  auto acc_empty = [&](int b) { return bar0 + 8u * (4 + S + b); };
  auto ea_full = [&](int j) { return bar0 + 8u * (4 + 2 * S + j); };
  auto ea_empty = [&](int j) { return bar0 + 8u * (6 + 2 * S + j); };
  const uint32_t drain = bar0 + 8u * (8 + 2 * S);

  // the operator's digits and row exponents, for the whole launch
  for (int i = threadIdx.x; i < Sh::OPB / 16; i += blockDim.x) ((uint4*)opb)[i] = a.op[i];
  // row exponents; as factors where the output is pairs
  for (int i = threadIdx.x; i < NC; i += blockDim.x)
    s_eb[i] = OUT >= kOutPair ? __float_as_int(pow2f(clamp_exp(a.ope[i]))) : a.ope[i];
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full(s), kProd * 32);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), kEpi);
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(ea_full(j), kProd * 32);
      mbar_init(ea_empty(j), kEpi * 32);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kProd) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp < kProd) {
    // ---------------------------------------------------------------- producers
    // half 0 takes points [0, H0), half 1 [H0, N): H0 a multiple of 4, so each
    // half covers whole 16-byte chunks (8 reals) of the digit rows.  With
    // PREFETCH a thread copies its half line of the next tile into its own
    // staging slots (cp.async) while it splits the current one: no other
    // thread takes part in the hand-over.
    constexpr int H0 = Sh::H0, H1 = N - H0;
    static_assert(H1 > 0 && H1 <= H0 && H1 % 4 == 0, "line halves");
    constexpr int PT = kProd * 32;            // producer threads
    const int r = warp * 16 + (lane & 15);    // row (line) of the tile
    const int hh = lane >> 4;                 // which half of the line
    const int np = hh ? H1 : H0;              // points of this half
    const int p0 = hh ? H0 : 0;               // first point
    const uint32_t my_stg = smem_u32(stg) + (uint32_t)threadIdx.x * 16u;
    // lines along x are consecutive in memory: the warp copies its 16 lines in
    // order (whole sectors; a lane per half line had fetched every sector twice)
    constexpr bool XW = AXIS == 0;
    const uint32_t warp_stg = smem_u32(stg) + (uint32_t)(warp * 16 * (N + 1) * 16);
    auto prefetch = [&](int t, bool go) {     // go: a data dependency on the caller's reads
      if constexpr (XW) {
        __syncwarp();                         // every lane has read its slots
        const long long l0 = (long long)t * BM + warp * 16;   // nlines is a multiple of 16
        const bool valid = go && l0 < a.nlines;
        const double2* src = a.src + (valid ? l0 * N : 0);
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
          const int e = k * 32 + lane, rr = e / N;
          cp_async16(warp_stg + (uint32_t)((e + rr) * 16), src + (valid ? e : 0), valid);
        }
        cp_async_commit();
        return;
      }
      const long long l = (long long)t * BM + r;
      const bool valid = go && l < a.nlines;
      long long stride = 0;
      const long long lb = valid ? line_base<N, AXIS>(a, l, stride) : 0;
#pragma unroll
      for (int j = 0; j < H0; ++j)
        if (j < np)
          cp_async16(my_stg + (uint32_t)(j * PT * 16),
                     valid ? (const void*)(a.src + lb + (long long)(p0 + j) * stride)
                           : (const void*)a.src,
                     valid);
      cp_async_commit();
    };
    constexpr bool PF = Sh::PREFETCH && IN != kInResidual;
    if constexpr (PF)
      if (blockIdx.x < a.ntiles) prefetch(blockIdx.x, true);
    int it = 0;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x, ++it) {
      const int s = it % STAGES, u = it / STAGES, slot = it & 1;
      using V = std::conditional_t<IN == kInPair, float4, double2>;
      V v[H0];
      if constexpr (PF) {
        cp_async_wait_all();
        if constexpr (XW) __syncwarp();       // the other lanes' copies too
#pragma unroll
        for (int j = 0; j < H0; ++j)
          v[j] = j < np ? (XW ? *(const V*)(stg + (warp * 16 * (N + 1) + (lane & 15) * (N + 1) + p0 + j) * 16)
                              : *(const V*)(stg + (j * PT + threadIdx.x) * 16))
                        : V{};
      } else {
        const long long l = (long long)t * BM + r;
        const bool valid = l < a.nlines;
        long long stride = 0;
        const long long lb = valid ? line_base<N, AXIS>(a, l, stride) : 0;
#pragma unroll
        for (int j = 0; j < H0; ++j)
          v[j] = (valid && j < np) ? ((const V*)a.src)[lb + (long long)(p0 + j) * stride] : V{};
        if constexpr (IN == kInResidual) {    // src - eps psi (src = h psi)
          const double e = valid ? a.eps[line_array<N, AXIS>(a, l) >> 1] : 0.0;
#pragma unroll
          for (int j = 0; j < H0; ++j)
            if (valid && j < np) {
              const double2 ps = a.psi[lb + (long long)(p0 + j) * stride];
              v[j] = make_double2(fma(-e, ps.x, v[j].x), fma(-e, ps.y, v[j].y));
            }
        }
      }
      int E = INT_MIN;
#pragma unroll
      for (int j = 0; j < H0; ++j) {
        if constexpr (IN == kInPair) E = max(E, max(exp_of_pair(v[j].x), exp_of_pair(v[j].z)));
        else E = max(E, max(exp_of(v[j].x), exp_of(v[j].y)));
      }
      if constexpr (PF) {
        // the next copy overwrites the slots just read: it is issued after E,
        // which depends on every value read
        if (t + (int)gridDim.x < a.ntiles) prefetch(t + gridDim.x, E != INT_MAX);
      }
      E = max(E, __shfl_xor_sync(0xffffffffu, E, 16));
      if (E == INT_MIN) E = 0;
      if (u > 0 && !mbar_wait(empty(s), (uint32_t)((u - 1) & 1))) {
        flag_status(a.status, SKY_ETIMEOUT);
        break;
      }
      if (it >= 2 && !mbar_wait(ea_empty(slot), (uint32_t)(((it >> 1) - 1) & 1))) {
        flag_status(a.status, SKY_ETIMEOUT);
        break;
      }
      if (hh == 0) s_ea[slot * BM + r] = E;
      const float sc = IN == kInPair ? pow2f(-E) : 1.0f;   // pairs: -126 <= E <= 129
      unsigned char* ta = ring + s * STAGE;
#pragma unroll
      for (int c = 0; c < H0 / 4; ++c) {
        if (c < np / 4) {
          unsigned w[S][4];   // digit p of the chunk's 8 reals, as 4 bf16 pairs
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float dr[S], di[S];
            if constexpr (IN == kInPair) {
              const float4 z = v[4 * c + j];
              digits6p(z.x * sc, z.y * sc, dr);
              digits6p(z.z * sc, z.w * sc, di);
            } else {
              digits6f(v[4 * c + j].x, E, dr);
              digits6f(v[4 * c + j].y, E, di);
            }
#pragma unroll
            for (int p = 0; p < S; ++p) w[p][j] = bf16x2(dr[p], di[p]);
          }
          const int k0 = 2 * p0 + 8 * c;
#pragma unroll
          for (int p = 0; p < S; ++p)
            *(uint4*)(ta + p * TILE_A + cm_off(r, k0, NC)) =
                make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
        }
      }
      // columns 2N .. NC - 1 (padding): zeros, from the second half
      if (hh == 1) {
#pragma unroll
        for (int k = 2 * N; k < NC; k += 8)
#pragma unroll
          for (int p = 0; p < S; ++p)
            *(uint4*)(ta + p * TILE_A + cm_off(r, k, NC)) = make_uint4(0u, 0u, 0u, 0u);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(full(s));
      mbar_arrive(ea_full(slot));
    }
    if constexpr (PF) cp_async_wait_all();   // no copy outlives the launch
  } else if (warp == kProd) {
    // ---------------------------------------------------------------- MMA issue
    const uint32_t el = elect_one();
    const uint32_t lb = ns_lo(smem_u32(opb));
    constexpr uint32_t dhi = ns_hi(NC);
    constexpr int NBUF = Sh::NBUF;
    int it = 0;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x, ++it) {
      const int s = it % STAGES, u = it / STAGES;
      if (!mbar_wait_warp(full(s), (uint32_t)(u & 1))) {
        if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
        break;
      }
      fence_after();
      const uint32_t la = ns_lo(smem_u32(ring + s * STAGE));
      const int b = it % NBUF, use = it / NBUF;
      if (use > 0) {
        // the epilogue must have drained this accumulator set
        if (!mbar_wait_warp(acc_empty(b), (uint32_t)((use - 1) & 1))) {
          if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
          break;
        }
        fence_after();
      }
      const uint32_t acc = tmem + (uint32_t)(b * 256);
#pragma unroll
      for (int ks = 0; ks < NC / 16; ++ks) {   // 16 values of K = two core matrices
        const uint32_t ka = la + (uint32_t)((ks * 256) >> 4), kb = lb + (uint32_t)((ks * 256) >> 4);
        // weights up to 4: digit p of the lines with digits 0 .. 4 - p; the first
        // MMA of the tile writes every accumulator
#pragma unroll
        for (int p = 0; p < NG; ++p) {
          constexpr int most = 256 / NC;       // digits per MMA
          const int n = NG - p, n0 = n < most ? n : most;
          mma_bf16_elect(acc + (uint32_t)(p * NC), ka + (uint32_t)(p * (TILE_A >> 4)), kb, dhi,
                         idesc_bf16(BM, n0 * NC), (p == 0 && ks == 0) ? 0u : 1u, el);
          if (n > n0)
            mma_bf16_elect(acc + (uint32_t)((p + n0) * NC), ka + (uint32_t)(p * (TILE_A >> 4)),
                           kb + (uint32_t)(n0 * (TILE_B >> 4)), dhi, idesc_bf16(BM, (n - n0) * NC),
                           (p == 0 && ks == 0) ? 0u : 1u, el);
        }
        // weight 5 into the last accumulator
#pragma unroll
        for (int p = 0; p < S; ++p)
          mma_bf16_elect(acc + (uint32_t)((NG - 1) * NC), ka + (uint32_t)(p * (TILE_A >> 4)),
                         kb + (uint32_t)((S - 1 - p) * (TILE_B >> 4)), dhi, idesc_bf16(BM, NC), 1u, el);
      }
      mma_commit_elect(acc_full(b), el);   // arrives when this tile's MMAs have completed
      mma_commit_elect(empty(s), el);
    }
    // every MMA issued by this warp completes before TMEM is freed
    mma_commit_elect(drain, el);
    if (!mbar_wait_warp(drain, 0) && lane == 0) flag_status(a.status, SKY_ETIMEOUT);
  } else {
    // ---------------------------------------------------------------- epilogue
    const int w = warp - kProd - 1;            // 0 .. kEpi - 1
    const int q = warp & 3, half = w >> 2;     // TMEM lane quadrant = warp id mod 4
    const int row = q * 32 + lane;
    bool ok = true;
    int it = 0;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x, ++it) {
      const int slot = it & 1;
      if (!mbar_wait(ea_full(slot), (uint32_t)((it >> 1) & 1))) {
        if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
        break;
      }
      const int E = s_ea[slot * BM + row];
      mbar_arrive(ea_empty(slot));
      const long long l = (long long)t * BM + row;
      long long stride = 0;
      const long long lb = l < a.nlines ? line_base<N, AXIS>(a, l, stride) : 0;
      long long bG = 0;
      if constexpr (OUT == kOutUpdate) bG = l < a.nlines ? (long long)line_array<N, AXIS>(a, l) * a.G : 0;
      const int sc = E - 16 - 8 * (S - 1);
      constexpr int NBUF = Sh::NBUF;
      const int b = it % NBUF, use = it / NBUF;
      // A thread's four outputs of a block of 8 columns (4 points from m0): its own
      // line's points, or, along x, where points are consecutive in memory, point
      // m0 + lane % 4 of the four lines of its lane quad (the quad transposes its
      // 4 x 4 results, so that a quad stores 64 consecutive bytes).
      const long long lq = (long long)t * BM + q * 32 + (lane & 28);
      auto at_of = [&](int m0, int c, bool& on) -> long long {
        if constexpr (AXIS == 0) {
          on = lq + c < a.nlines;
          return (lq + c) * N + m0 + (lane & 3);
        } else {
          on = l < a.nlines;
          return lb + (long long)(m0 + c) * stride;
        }
      };
      // the epilogue's own operands (psi and w, P, or the pairs to add to) are
      // loaded before the block's sums are read and combined, the first before the
      // wait: behind the stores they would be a chain of round trips (24^3, 280
      // states: the step with its two such passes 905 us with the loads behind the
      // stores, 840 us ahead of them)
      constexpr bool ADD = OUT == kOutAddPair || OUT == kOutAddF64;
      constexpr bool PAIR = ADD || OUT == kOutPair;
      constexpr bool AHEAD = ADD || OUT == kOutScaleP || OUT == kOutUpdate;
      const float fE = pow2f(clamp_exp(E));
      double2 xp[4];
      double xf[4];
      float xw[4];
      float4 xh[4];
      auto ahead = [&](int m0) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          bool on;
          const long long at = at_of(m0, c, on);
          if constexpr (OUT == kOutUpdate) {
            xp[c] = on ? __ldg(a.psi + at) : make_double2(0.0, 0.0);
            xw[c] = on && a.w ? __ldg(a.w + (at - bG)) : 1.0f;
          } else if constexpr (OUT == kOutScaleP) {   // lines along x
            xf[c] = on ? __ldg(a.P + (at - (long long)line_array<N, AXIS>(a, lq + c) * a.G)) : 0.0;
          } else if constexpr (ADD) {
            xh[c] = on ? ((const float4*)a.dst)[at] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          }
        }
      };
      if constexpr (AHEAD) ahead(half * HALF / 2);
      if (!mbar_wait(acc_full(b), (uint32_t)(use & 1))) {
        if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
        break;
      }
      fence_after();
      // columns in blocks of 8 (4 points).  FP64 out: the exact group sums
      // (integers G_g of units 2^{-8(g+2)}, |G_g| < 2^24) fold into int32: u = G0
      // 2^8 + G1, w = G2 2^8 + G3, and x = round(2^8 G45) from the weight-{4,5}
      // group (|x| < 2^31 for K <= 64); the total sum_g G_g 2^{8(5-g)} = u 2^32 +
      // w 2^16 + x.
#pragma unroll 1
      for (int cb = 0; cb < HALF; cb += 8) {
        const int o = half * HALF + cb, m0 = o >> 1;
        if (m0 >= N) break;                    // padding (N is a multiple of 4)
        if constexpr (AHEAD)
          if (cb > 0) ahead(m0);
        uint32_t v[NG][8];
#pragma unroll
        for (int g = 0; g < NG; ++g)
          oz::tmem_ld<8>(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * 256 + g * NC + o), v[g]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float4 z[4];                           // four results: pairs, or the bits of two doubles
        if constexpr (PAIR) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float r[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int k = 2 * c + h;
              const dd p = pair_of_groups(__uint_as_float(v[0][k]), __uint_as_float(v[1][k]),
                                          __uint_as_float(v[2][k]), __uint_as_float(v[3][k]),
                                          __uint_as_float(v[4][k]));
              const float f = fE * __int_as_float(s_eb[o + k]);
              r[2 * h] = p.hi * f;
              r[2 * h + 1] = p.lo * f;
            }
            z[c] = make_float4(r[0], r[1], r[2], r[3]);
          }
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            double r[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int k = 2 * c + h;
              const int fu = __float2int_rn(__uint_as_float(v[0][k]) * 0x1p16f) * 256 +
                             __float2int_rn(__uint_as_float(v[1][k]) * 0x1p24f);
              const int fw = __float2int_rn(__uint_as_float(v[2][k]) * 0x1p32f) * 256 +
                             __float2int_rn(__uint_as_float(v[3][k]) * 0x1p40f);
              const int fx = __float2int_rn(__uint_as_float(v[4][k]) * 0x1p56f);
              r[h] = scaled_double(((long long)fu << 32) + ((long long)fw << 16) + (long long)fx,
                                   sc + s_eb[o + k]);
            }
            z[c] = make_float4(__int_as_float(__double2loint(r[0])), __int_as_float(__double2hiint(r[0])),
                               __int_as_float(__double2loint(r[1])), __int_as_float(__double2hiint(r[1])));
          }
        }
        if constexpr (AXIS == 0) quad_transpose(z, lane);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          bool on;
          const long long at = at_of(m0, c, on);
          if (!on) continue;
          if constexpr (PAIR) {
            if constexpr (ADD) {
              const float4 h = xh[c];
              const ddc r = ddc{dd(h.x, h.y), dd(h.z, h.w)} + ddc{dd(z[c].x, z[c].y), dd(z[c].z, z[c].w)};
              if constexpr (OUT == kOutAddF64) a.dst[at] = make_double2(dbl_of_near(r.x), dbl_of_near(r.y));
              else ((float4*)a.dst)[at] = make_float4(r.x.hi, r.x.lo, r.y.hi, r.y.lo);
            } else {
              ((float4*)a.dst)[at] = z[c];
            }
          } else {
            double2 res = make_double2(__hiloint2double(__float_as_int(z[c].y), __float_as_int(z[c].x)),
                                       __hiloint2double(__float_as_int(z[c].w), __float_as_int(z[c].z)));
            if constexpr (OUT == kOutScaleP) {
              const double f = xf[c] * a.scale;
              res = make_double2(res.x * f, res.y * f);
            } else if constexpr (OUT == kOutUpdate) {
              const double2 ps = xp[c];
              if (a.w) {
                const double f = (double)xw[c];
                res = make_double2(fma(-f, res.x, ps.x), fma(-f, res.y, ps.y));
              } else {
                res = make_double2(ps.x - res.x, ps.y - res.y);
              }
            }
            a.dst[at] = res;
          }
        }
      }
      // this warp's lanes of the accumulator set are read: hand it back
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty(b));
    }
  }
  fence_before();
  __syncthreads();
  if (warp == kProd) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

// ------------------------------------------------------------ host side
bool supported(int n) { return n == 8 || n == 12 || n == 16 || n == 20 || n == 24 || n == 32; }

// Digits [S][NC][NC] (canonical layout, bf16 bit patterns of alpha_s 2^{-8(s+1)})
// and row exponents [NC] of the real operator
// of one axis, built in long double.  kind: kOpDeriv the derivative, the
// circulant D[m][q] = d[(m - q) mod n], d[r] = (i/n) sum_a kappa_a
// e^{2 pi i a r / n}; kOpFwd / kOpInv the unnormalised DFT, D[m][q] =
// e^{-+2 pi i (m q mod n) / n}.
void build_operator(int n, double L, double theta, int kind, std::vector<unsigned short>& dig,
                    std::vector<int>& ex) {
  const int NC = nc_of(n);
  const long double two_pi = 6.283185307179586476925286766559005768L;
  std::vector<long double> dre(n), dim(n);
  if (kind == kOpDeriv) {
    for (int r = 0; r < n; ++r) {
      long double sr = 0.0L, si = 0.0L;
      for (int a = 0; a < n; ++a) {
        const int mm = a < (n + 1) / 2 ? a : a - n;
        const long double kap = (two_pi * mm + (long double)theta) / (long double)L;
        const long double ang = two_pi * (long double)(((long long)a * r) % n) / (long double)n;
        sr -= kap * sinl(ang);   // Re of i kappa e^{i ang}
        si += kap * cosl(ang);   // Im
      }
      dre[r] = sr / n;
      dim[r] = si / n;
    }
  }
  auto entry = [&](int m, int q, double& re, double& im) {
    if (kind == kOpDeriv) {
      const int r = ((m - q) % n + n) % n;
      re = (double)dre[r];
      im = (double)dim[r];
    } else {
      const long double ang = two_pi * (long double)(((long long)m * q) % n) / (long double)n;
      re = (double)cosl(ang);
      im = (double)(kind == kOpFwd ? -sinl(ang) : sinl(ang));
    }
  };
  std::vector<double> B((size_t)NC * NC, 0.0);
  for (int m = 0; m < n; ++m)
    for (int q = 0; q < n; ++q) {
      double re, im;
      entry(m, q, re, im);
      B[(size_t)(2 * m) * NC + 2 * q] = re;
      B[(size_t)(2 * m) * NC + 2 * q + 1] = -im;
      B[(size_t)(2 * m + 1) * NC + 2 * q] = im;
      B[(size_t)(2 * m + 1) * NC + 2 * q + 1] = re;
    }
  dig.assign((size_t)S * NC * NC, 0);
  ex.assign(NC, 0);
  for (int o = 0; o < NC; ++o) {
    int F = INT_MIN;
    for (int k = 0; k < NC; ++k) {
      const double x = B[(size_t)o * NC + k];
      if (x != 0.0) {
        int e;
        std::frexp(x, &e);   // |x| < 2^e
        F = e > F ? e : F;
      }
    }
    if (F == INT_MIN) F = 0;
    ex[o] = F;
    for (int k = 0; k < NC; ++k) {
      const double x = B[(size_t)o * NC + k];
      // X = round(|x| 2^{8S - F}) < 2^48 + 1, exact (power-of-two scaling, then +0.5)
      long long X = (long long)std::floor(std::ldexp(std::fabs(x), 8 * S - F) + 0.5);
      int d[S];
      for (int s = S - 1; s >= 1; --s) {
        int v = (int)(X & 255);
        X >>= 8;
        if (v >= 128) { v -= 256; ++X; }
        d[s] = v;
      }
      d[0] = (int)X;
      for (int p = 0; p < S; ++p) {
        const float f = std::ldexp((float)(x < 0.0 ? -d[p] : d[p]), -8 * (p + 1));   // |d| <= 256: exact in bf16
        unsigned u;
        std::memcpy(&u, &f, 4);
        dig[((size_t)p * NC * NC * 2 + cm_off(o, k, NC)) / 2] = (unsigned short)(u >> 16);
      }
    }
  }
}

template <int N, int AXIS, int IN, int OUT>
cudaError_t launch(const DerivArgs& a, const Ctx* c) {
  using Sh = Shape<N>;
  static bool set[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!set[dev]) {
    e = cudaFuncSetAttribute(k_oz_deriv<N, AXIS, IN, OUT>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
    if (e != cudaSuccess) return e;
    set[dev] = true;
  }
  const int grid = a.ntiles < c->num_sms ? a.ntiles : c->num_sms;
  k_oz_deriv<N, AXIS, IN, OUT><<<grid, THREADS, Sh::SMEM, c->stream>>>(a);
  note_launch();
  return cudaGetLastError();
}

}  // namespace ozd

static sky_status upload_operator(Ctx* c, int n, double L, double theta, int kind, void** dig_out,
                                  int** ex_out) {
  std::vector<unsigned short> dig;
  std::vector<int> ex;
  ozd::build_operator(n, L, theta, kind, dig, ex);
  cudaError_t e = cudaMalloc(dig_out, dig.size() * sizeof(unsigned short));
  if (e == cudaSuccess) e = cudaMalloc(ex_out, ex.size() * sizeof(int));
  if (e == cudaSuccess)
    e = cudaMemcpy(*dig_out, dig.data(), dig.size() * sizeof(unsigned short), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(*ex_out, ex.data(), ex.size() * sizeof(int), cudaMemcpyHostToDevice);
  return cuda_check(c, e, "operator upload");
}

sky_status deriv_tc_init(Ctx* c) {
  for (int j = 0; j < 3; ++j) {
    c->d_dop[j] = nullptr;
    c->d_dope[j] = nullptr;
    for (int k = 0; k < 2; ++k) {
      c->d_dft[j][k] = nullptr;
      c->d_dfte[j][k] = nullptr;
    }
  }
  if (c->prec != SKY_F64) return SKY_OK;
  for (int j = 0; j < 3; ++j) {
    if (!ozd::supported(c->n[j])) continue;
    sky_status s = upload_operator(c, c->n[j], c->L[j], c->theta[j], ozd::kOpDeriv, &c->d_dop[j],
                                   &c->d_dope[j]);
    for (int k = 0; k < 2 && s == SKY_OK; ++k)
      s = upload_operator(c, c->n[j], c->L[j], c->theta[j], k == 0 ? ozd::kOpFwd : ozd::kOpInv,
                          &c->d_dft[j][k], &c->d_dfte[j][k]);
    if (s != SKY_OK) return s;
  }
  return SKY_OK;
}

namespace {

ozd::DerivArgs op_args(const Ctx* c, int ax, const double2* src, double2* dst, long long nb,
                       const void* op, const int* ope) {
  ozd::DerivArgs a{};
  a.src = src;
  a.dst = dst;
  a.op = (const uint4*)op;
  a.ope = ope;
  a.nx = c->n[0];
  a.ny = c->n[1];
  a.nz = c->n[2];
  a.G = c->G;
  a.nlines = nb * (c->G / c->n[ax]);
  a.div1 = ozd::make_fastdiv((unsigned)c->n[0]);
  a.div2 = ozd::make_fastdiv((unsigned)(ax == 1 ? c->n[2] : c->n[1]));
  a.div0 = ozd::make_fastdiv((unsigned)(c->n[1] * c->n[2]));
  const long long nt = (a.nlines + ozd::BM - 1) / ozd::BM;
  a.ntiles = nt > INT_MAX ? INT_MAX : (int)nt;
  a.status = c->d_status;
  return a;
}

// One operator pass along ax with the given modes (only the combinations
// the library uses are instantiated).
template <int IN, int OUT>
cudaError_t op_pass(const Ctx* c, int ax, const ozd::DerivArgs& a) {
  if (a.nlines == 0) return cudaSuccess;
  if (a.nlines >= (1LL << 31)) return cudaErrorInvalidValue;
  auto go = [&](auto NC) -> cudaError_t {
    constexpr int N = decltype(NC)::value;
    if constexpr (IN == ozd::kInResidual) {
      return ax == 2 ? ozd::launch<N, 2, IN, OUT>(a, c) : cudaErrorInvalidValue;
    } else if constexpr (OUT == ozd::kOutScaleP) {
      return ax == 0 ? ozd::launch<N, 0, IN, OUT>(a, c) : cudaErrorInvalidValue;
    } else if constexpr (OUT == ozd::kOutUpdate || OUT == ozd::kOutAddF64) {
      return ax == 2 ? ozd::launch<N, 2, IN, OUT>(a, c) : cudaErrorInvalidValue;
    } else if constexpr (OUT == ozd::kOutAddPair) {
      if (ax == 0) return ozd::launch<N, 0, IN, OUT>(a, c);
      return ax == 1 ? ozd::launch<N, 1, IN, OUT>(a, c) : cudaErrorInvalidValue;
    } else {
      if (ax == 0) return ozd::launch<N, 0, IN, OUT>(a, c);
      if (ax == 1) return ozd::launch<N, 1, IN, OUT>(a, c);
      return ozd::launch<N, 2, IN, OUT>(a, c);
    }
  };
  switch (c->n[ax]) {
    case 8: return go(std::integral_constant<int, 8>{});
    case 12: return go(std::integral_constant<int, 12>{});
    case 16: return go(std::integral_constant<int, 16>{});
    case 20: return go(std::integral_constant<int, 20>{});
    case 24: return go(std::integral_constant<int, 24>{});
    case 32: return go(std::integral_constant<int, 32>{});
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

// dst = d_ax src over nb arrays of G complex doubles (dst may equal src).
cudaError_t deriv_tc(Ctx* c, int ax, const double2* src, double2* dst, long long nb) {
  if (!c->d_dop[ax]) return cudaErrorInvalidValue;
  return op_pass<ozd::kInPlain, ozd::kOutPlain>(
      c, ax, op_args(c, ax, src, dst, nb, c->d_dop[ax], c->d_dope[ax]));
}

// The passes of h psi on pairs (hamiltonian.cu): G = d_ax psi as pairs; h += d_ax F
// along x and y (pairs), along z with FP64 out.
cudaError_t deriv_tc_pair(Ctx* c, int ax, const double2* psi, void* g, long long nb) {
  return op_pass<ozd::kInPlain, ozd::kOutPair>(
      c, ax, op_args(c, ax, psi, (double2*)g, nb, c->d_dop[ax], c->d_dope[ax]));
}
cudaError_t deriv_tc_add(Ctx* c, int ax, const void* f, void* h, long long nb) {
  const ozd::DerivArgs a = op_args(c, ax, (const double2*)f, (double2*)h, nb, c->d_dop[ax], c->d_dope[ax]);
  return ax < 2 ? op_pass<ozd::kInPair, ozd::kOutAddPair>(c, ax, a)
                : op_pass<ozd::kInPair, ozd::kOutAddF64>(c, ax, a);
}

bool damp_tc_available(const Ctx* c) {
  for (int j = 0; j < 3; ++j)
    if (!c->d_dft[j][0] || !c->d_dft[j][1]) return false;
  return true;
}

// The damped step's 3D transform pair as six operator passes over the 2I
// arrays (the damping table P must be current): phi = F_z F_y F_x of
// (h psi - eps psi), times P x0 / G in the last forward pass, the inverse
// passes, phi = psi - w (result) in the last.
cudaError_t damp_tc(Ctx* c, int q, const double2* psi, const double2* hpsi, const double* eps,
                    double2* phi, int I, double x0, const float* w) {
  const long long nb = 2LL * I;
  auto args = [&](int ax, int k, const double2* src) {
    return op_args(c, ax, src, phi, nb, c->d_dft[ax][k], c->d_dfte[ax][k]);
  };
  ozd::DerivArgs a = args(2, 0, hpsi);
  a.psi = psi;
  a.eps = eps;
  cudaError_t e = op_pass<ozd::kInResidual, ozd::kOutPlain>(c, 2, a);
  if (e == cudaSuccess) e = op_pass<ozd::kInPlain, ozd::kOutPlain>(c, 1, args(1, 0, phi));
  if (e == cudaSuccess) {
    ozd::DerivArgs b = args(0, 0, phi);
    b.P = c->d_damp[q];
    b.scale = x0 / (double)c->G;
    e = op_pass<ozd::kInPlain, ozd::kOutScaleP>(c, 0, b);
  }
  if (e == cudaSuccess) e = op_pass<ozd::kInPlain, ozd::kOutPlain>(c, 0, args(0, 1, phi));
  if (e == cudaSuccess) e = op_pass<ozd::kInPlain, ozd::kOutPlain>(c, 1, args(1, 1, phi));
  if (e == cudaSuccess) {
    ozd::DerivArgs d = args(2, 1, phi);
    d.psi = psi;
    d.w = w;
    e = op_pass<ozd::kInPlain, ozd::kOutUpdate>(c, 2, d);
  }
  return e;
}

}  // namespace sky
