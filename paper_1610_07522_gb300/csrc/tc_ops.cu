// Split-BF16 tensor-core forms of the overlap / Hamiltonian matrix (Eqs.
// normmatrix, hammatrix) and of the recombination (Sec. 3.3.3) for FP32
// spinors.  Each FP32 value x is split into bf16 pieces x = x_0 + x_1 (+ x_2)
// with x_0 = bf16(x), x_1 = bf16(x - x_0), x_2 = bf16(x - x_0 - x_1); the
// products kept are those of total weight <= nsplit - 1 (3 products for a
// 2-way split, 6 for a 3-way split), accumulated in FP32 in TMEM.
//
// Complex contractions become single real GEMMs over the interleaved (re, im)
// storage:
//   <a|b>:  Re = sum_k a_r[k] b_r[k],  Im = sum_k a_r[k] b'_r[k],
//           b' = (Im b, -Re b) per entry, so D = a_r [b_r; b'_r]^T holds Re | Im;
//   psi_a = sum_b M[b][a] phi_b:  P = M_re^T phi_r, Q = M_im^T phi_r over phi's
//           own layout, psi = (P_re - Q_im, P_im + Q_re) per entry.
#include <cuda_bf16.h>

#include <cfloat>

#include "dd.cuh"
#include "tc_gemm.cuh"

namespace sky {

__device__ __forceinline__ void split3(float x, int n, __nv_bfloat16* out) {
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  out[0] = h;
  if (n > 1) {
    const float r = x - __bfloat162float(h);
    const __nv_bfloat16 m = __float2bfloat16_rn(r);
    out[1] = m;
    if (n > 2) out[2] = __float2bfloat16_rn(r - __bfloat162float(m));
  }
}

// Row operands of <a|b>: dst[i][row][k] for the real view of src ([rows][K]);
// with prime != 0, rows [rows, 2 rows) receive (Im, -Re) of each entry.
__global__ void k_split_rows(const float* __restrict__ src, long long rows, long long K, int n,
                             int prime, __nv_bfloat16* d0, __nv_bfloat16* d1, __nv_bfloat16* d2) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // complex entry
  const long long nc = rows * (K / 2);
  if (e >= nc) return;
  const long long r = e / (K / 2), c = e % (K / 2);
  __nv_bfloat16 sr[3], si[3];
  split3(src[2 * e], n, sr);
  split3(src[2 * e + 1], n, si);
  __nv_bfloat16* d[3] = {d0, d1, d2};
  for (int i = 0; i < n; ++i) {
    __nv_bfloat162 v;
    v.x = sr[i]; v.y = si[i];
    *reinterpret_cast<__nv_bfloat162*>(d[i] + r * K + 2 * c) = v;
    if (prime) {
      __nv_bfloat162 w;
      w.x = si[i]; w.y = __hneg(sr[i]);
      *reinterpret_cast<__nv_bfloat162*>(d[i] + (rows + r) * K + 2 * c) = w;
    }
  }
}

// Operand of the recombination: the n bf16 pieces of every real of phi, in
// phi's own layout [I][2 V] (the product reads it MN-major).  Eight reals per
// thread: two 16-byte loads, one 16-byte store per piece.  HBM-bound: 32^3, 700
// states, x3: 734 MB in 104 us (7.1 TB/s); the transposed [V][2 I] operand that held every
// value twice (phi and i phi) took 482 us.
__global__ void __launch_bounds__(256) k_split_flat(const float4* __restrict__ phi, long long n8,
                                                    int n, uint4* d0, uint4* d1, uint4* d2) {
  const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
  if (e >= n8) return;
  const float4 a = phi[2 * e], b = phi[2 * e + 1];
  const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  __nv_bfloat16 s[8][3];
#pragma unroll
  for (int k = 0; k < 8; ++k) split3(x[k], n, s[k]);
  uint4* d[3] = {d0, d1, d2};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i >= n) break;
    unsigned w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __nv_bfloat162 v;
      v.x = s[2 * k][i];
      v.y = s[2 * k + 1][i];
      w[k] = *reinterpret_cast<unsigned*>(&v);
    }
    d[i][e] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Coefficient operand of the recombination: rows 2a and 2a + 1 of A hold
// M_re[beta][a] and M_im[beta][a] over beta (row stride ld, ld - I zeros),
// split into bf16 pieces.
__global__ void k_split_rot_a(const double2* __restrict__ M, int I, long long ld, int n,
                              __nv_bfloat16* d0, __nv_bfloat16* d1, __nv_bfloat16* d2) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 2 * I * ld) return;
  const int r = (int)(e / ld), beta = (int)(e % ld);
  double xd = 0.0;
  if (beta < I) {
    const double2 m = M[(long long)beta * I + (r >> 1)];
    xd = (r & 1) ? m.y : m.x;   // the FP64 value keeps its residual in the lower pieces
  }
  __nv_bfloat16 s[3];
  const __nv_bfloat16 h = __double2bfloat16(xd);
  s[0] = h;
  if (n > 1) {
    const double r1 = xd - (double)__bfloat162float(h);
    const __nv_bfloat16 mm = __double2bfloat16(r1);
    s[1] = mm;
    if (n > 2) s[2] = __double2bfloat16(r1 - (double)__bfloat162float(mm));
  }
  __nv_bfloat16* d[3] = {d0, d1, d2};
  for (int i = 0; i < n; ++i) d[i][e] = s[i];
}

// A sum of floats to 72 bits: TwoSum into hi, its errors by TwoSum into mid, theirs
// into lo.
struct SumF3 {
  float hi = 0.0f, mid = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float x) {
    const dd s = two_sum(hi, x);
    hi = s.hi;
    const dd m = two_sum(mid, s.lo);
    mid = m.hi;
    lo = __fadd_rn(lo, m.lo);
  }
  __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};

// X[a][b] (+)= dV sum_z (D_z[a][b] + i D_z[a][I + b]) for a >= b, mirrored.  In
// FP64 the conversions and additions bound it (32^3, 700 states: 200 us with 64
// partials, 395 us with 128); with triples of floats, which lose nothing against
// FP64, the partials' bytes and latency do (33 and 68 us; 83 and 172 us without the
// loads ahead of the sums).  A sum beyond the floats' range is formed again in FP64.
constexpr int kRedLoads = 8;            // partials of a thread in flight
__global__ void __launch_bounds__(128) k_tc_overlap_reduce(const float* __restrict__ D, int nz,
                                                           long long sstride, long long ldd, int I,
                                                           double dV, double2* X, int add) {
  const int a = blockIdx.x, b = blockIdx.y * 128 + threadIdx.x;
  if (b > a) return;
  const float* Da = D + (long long)a * ldd + b;
  SumF3 r, i;
  for (int z0 = 0; z0 < nz; z0 += kRedLoads) {
    float x[kRedLoads], y[kRedLoads];
#pragma unroll
    for (int k = 0; k < kRedLoads; ++k) {
      const bool on = z0 + k < nz;
      x[k] = on ? Da[(z0 + k) * sstride] : 0.0f;
      y[k] = on ? Da[(z0 + k) * sstride + I] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kRedLoads; ++k) {
      r.add(x[k]);
      i.add(y[k]);
    }
  }
  double re = r.value(), im = i.value();
  if (!(fabsf(r.hi) <= FLT_MAX && fabsf(i.hi) <= FLT_MAX)) {
    re = im = 0.0;
    for (int z = 0; z < nz; ++z) {
      re += (double)Da[z * sstride];
      im += (double)Da[z * sstride + I];
    }
  }
  double2 s = make_double2(dV * re, dV * im);
  if (add) s = X[(long long)a * I + b] + s;
  X[(long long)a * I + b] = s;
  if (a != b) X[(long long)b * I + a] = conjx(s);
}

static inline long long round8(long long x) { return (x + 7) / 8 * 8; }   // 16-byte rows of bf16

int tc_nsplit(sky_prec p) { return p == SKY_F32_BF16X6 ? 3 : 2; }

// FP32 accumulation in TMEM loses accuracy over long K (its rounding error
// grows with the length of the sum): every split-K partial of the overlap
// covers at most kMaxAccK values of K, and the partials are summed to FP64 by
// the reduce.  Where the partials of half that length are small enough to stay
// in L2 (kSmallPartials), they are half as long: it costs nothing there (small
// boxes have too few tiles to fill the GPU otherwise) and halves the error (12^3,
// 43 states: the energy 5e-5 MeV per nucleon from that of 64-value partials
// with 2048, 2e-5 with 1024).  The six products of the x6 form, which is there for
// its accuracy, always take half-length partials: the diagonal's truncation is
// 1.1e-5 with 2048 values in either form (32^3, 700 states), 7e-6 with 1024, which
// the recombination's own (3.9e-6) does not hide.  Where they do not fit the buffer
// at once (kMostPartials), they are formed and summed in several rounds over K.
constexpr long long kMaxAccK = 2048;
constexpr long long kSmallPartials = 4LL << 20;    // fp32 values: 16 MB
constexpr long long kMostPartials = 64LL << 20;    // 256 MB: 32^3, 700 states in two rounds (1284 us of
                                                   // products with 16 to 64 M values, 1277 in one round)
static long long half_splits(long long K) { return (K + kMaxAccK / 2 - 1) / (kMaxAccK / 2); }
static int tc_min_splits(long long K, int I, int nsplit) {
  const long long z = half_splits(K);
  const long long ldd = (2LL * I + 3) / 4 * 4;
  return (int)(nsplit == 3 || z * I * ldd <= kSmallPartials ? z : (K + kMaxAccK - 1) / kMaxAccK);
}

// Scratch (bf16 elements per piece / fp32 partials) for I states of V complex.
void tc_scratch_sizes(int I, long long V, int num_sms, int nsplit, size_t* piece_a, size_t* piece_b,
                      size_t* piece_rot_a, size_t* partial) {
  const long long K = 2 * V;
  *piece_a = (size_t)I * K;              // also the states' pieces of the recombination
  *piece_b = (size_t)2 * I * K;
  *piece_rot_a = (size_t)2 * I * round8(I);
  const long long ldd = (2LL * I + 3) / 4 * 4;
  const int tiles = ((I + tc::BM - 1) / tc::BM) * ((2 * I + tc::BN - 1) / tc::BN);
  int z = kMaxTcWaves * num_sms / (tiles > 0 ? tiles : 1);
  const int zacc = (int)((K + kMaxAccK - 1) / kMaxAccK);
  if (z < zacc) z = zacc;
  if (z < 1) z = 1;
  *partial = (size_t)z * I * ldd;
  // half-length partials of these states, or of fewer
  const long long half = half_splits(K) * I * ldd, most = nsplit == 3 ? kMostPartials : kSmallPartials;
  const size_t need = (size_t)(half < most ? half : most);
  if (*partial < need) *partial = need;
}

sky_status tc_overlap(Ctx* c, const void* a, const void* b, int I, double2* X) {
  const long long V = 2LL * c->G, K = 2 * V;
  const int n = tc_nsplit(c->prec);
  __nv_bfloat16* A[3] = {(__nv_bfloat16*)c->d_tcA[0], (__nv_bfloat16*)c->d_tcA[1],
                         (__nv_bfloat16*)c->d_tcA[2]};
  __nv_bfloat16* Bp[3] = {(__nv_bfloat16*)c->d_tcB[0], (__nv_bfloat16*)c->d_tcB[1],
                          (__nv_bfloat16*)c->d_tcB[2]};
  const long long nc = (long long)I * V;
  k_split_rows<<<div_up(nc, 256), 256, 0, c->stream>>>((const float*)a, I, K, n, 0, A[0], A[1],
                                                       A[2]);
  k_split_rows<<<div_up(nc, 256), 256, 0, c->stream>>>((const float*)b, I, K, n, 1, Bp[0], Bp[1],
                                                       Bp[2]);
  note_launch(2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_check(c, e, "tc split");
  const long long ldd = (2LL * I + 3) / 4 * 4;
  const int tiles = ((I + tc::BM - 1) / tc::BM) * ((2 * I + tc::BN - 1) / tc::BN);
  // tc_waves 0: the fewest splits the accumulation bound allows (for boxes
  // that share the GPU with others), else about that many waves of SMs
  const long long sstride = (long long)I * ldd;
  const long long fit = (long long)(c->tc_partial_elems / sstride);   // partials at once
  if (fit < 1) return set_err(c, SKY_EINVAL, "tc overlap: partial buffer too small for I=%d", I);
  long long z = c->tc_waves * c->num_sms / tiles;
  if (z > fit) z = fit;
  if (z < tc_min_splits(K, I, n)) z = tc_min_splits(K, I, n);   // bounded FP32 accumulation length
  if (z < 1) z = 1;
  const long long nkb = (K + tc::BK - 1) / tc::BK, per = (nkb + z - 1) / z;   // K blocks of a partial
  const long long step = fit * per * tc::BK;
  for (long long k0 = 0; k0 < K; k0 += step) {
    const long long k = K - k0 < step ? K - k0 : step;
    const void *pa[3] = {nullptr}, *pb[3] = {nullptr};
    for (int i = 0; i < n; ++i) {
      pa[i] = A[i] + k0;
      pb[i] = Bp[i] + k0;
    }
    int zk = (int)((k + per * tc::BK - 1) / (per * tc::BK));
    e = tc::gemm_bf16<false>(pa, K, pb, K, n, I, 2 * I, (int)k, &zk, c->d_tcPart, ldd, sstride,
                             c->d_status, c->stream, c->tc_tile_n);
    if (e != cudaSuccess) return cuda_check(c, e, "tc overlap gemm");
    k_tc_overlap_reduce<<<dim3(I, div_up(I, 128)), 128, 0, c->stream>>>(
        c->d_tcPart, zk, sstride, ldd, I, c->dV, X, k0 > 0);
    note_launch();
  }
  return cuda_check(c, cudaGetLastError(), "tc overlap reduce");
}

// psi_a = sum_b M[b][a] phi_b as one real product over the states' own layout:
// [P; Q] = [M_re^T; M_im^T] phi (2 I rows, K = I, N = 2 V reals), combined in
// the epilogue.
sky_status tc_rotate(Ctx* c, const void* phi, const double2* M, int I, void* out) {
  const long long V = 2LL * c->G, K2V = 2 * V;
  const int n = tc_nsplit(c->prec);
  const long long lda = round8(I);
  __nv_bfloat16* Ra[3] = {(__nv_bfloat16*)c->d_tcRotA[0], (__nv_bfloat16*)c->d_tcRotA[1],
                          (__nv_bfloat16*)c->d_tcRotA[2]};
  __nv_bfloat16* Bp[3] = {(__nv_bfloat16*)c->d_tcA[0], (__nv_bfloat16*)c->d_tcA[1],
                          (__nv_bfloat16*)c->d_tcA[2]};
  k_split_rot_a<<<div_up(2 * I * lda, 256), 256, 0, c->stream>>>(M, I, lda, n, Ra[0], Ra[1], Ra[2]);
  const long long n8 = I * K2V / 8;      // K2V = 4 G, every axis a multiple of 4
  if (((uintptr_t)phi & 15) == 0)
    k_split_flat<<<div_up(n8, 256), 256, 0, c->stream>>>((const float4*)phi, n8, n, (uint4*)Bp[0],
                                                         (uint4*)Bp[1], (uint4*)Bp[2]);
  else                                   // states at an 8-byte boundary: scalar loads
    k_split_rows<<<div_up((long long)I * V, 256), 256, 0, c->stream>>>((const float*)phi, I, K2V, n, 0,
                                                                       Bp[0], Bp[1], Bp[2]);
  note_launch(2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_check(c, e, "tc rotate split");
  int z = 1;
  const void* pa[3] = {Ra[0], Ra[1], Ra[2]};
  const void* pb[3] = {Bp[0], Bp[1], Bp[2]};
  e = tc::gemm_bf16<true>(pa, lda, pb, K2V, n, 2 * I, (int)K2V, I, &z, (float*)out, K2V, 0,
                          c->d_status, c->stream, c->tc_tile_n);
  return cuda_check(c, e, "tc rotate gemm");
}

}  // namespace sky
