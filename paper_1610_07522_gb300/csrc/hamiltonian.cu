// Single-particle Hamiltonian (Sec. 2.1-2.2), damped gradient step
// (Eq. dampstep) and densities (Eqs. rho, curr, tau) for batched spinors.
//
// h psi is evaluated in the rearranged but identical form
//   h psi = U psi - (i/2) sum_j A_j (d_j psi) + sum_j d_j F_j,
//   F_j   = -B d_j psi - (i/2) A_j psi,   A_j = (sigma x W)_j,
// which follows from eps_ijk W_i sigma_k = (sigma x W)_j.  The passes are
//   1. G_j = d_j psi               (one 1D spectral pass per axis)
//   2. L = U psi - (i/2) sum A_j G_j -> hpsi;  F_j -> in place of G_j
//   3. F_j <- d_j F_j              (one pass per axis, in place)
//   4. hpsi = L + sum_j F_j, with <psi|h psi> and |h psi|^2 per block.
#include <cmath>

#include "fft_lines.cuh"

namespace sky {

sky_status upload_twiddles_hamiltonian(Ctx* c) {
  return cuda_check(c, upload_twiddles_this_unit(), "twiddle upload (hamiltonian)");
}

// ------------------------------------------------------------ line ops
// out = d_axis in  (i (k + theta/L) / N after the forward transform)
template <typename T> struct OpDeriv {
  static constexpr bool kFwd = true, kInv = true;
  const cx<T>* in; cx<T>* out; const T* k; T inv_n; long long G;
  __device__ __forceinline__ cx<T> load(long long b, int i) const { return in[b * G + i]; }
  __device__ __forceinline__ void mid(cx<T>& v, long long, int, int m) const {
    const T kk = k[m] * inv_n;
    v = mkc<T>(-kk * v.y, kk * v.x);
  }
  __device__ __forceinline__ void store(long long b, int i, cx<T> v) const { out[b * G + i] = v; }
};

// The same derivative pass of FP64 arrays with the transform carried in
// double-float arithmetic (dd.cuh): loads and stores FP64, k from a table of
// float pairs of (k + theta/L) / N.
struct OpDerivDD {
  static constexpr bool kFwd = true, kInv = true;
  const double2* in; double2* out; const float2* k; long long G;
  __device__ __forceinline__ ddc load(long long b, int i) const { return ddc_of(in[b * G + i]); }
  __device__ __forceinline__ void mid(ddc& v, long long, int, int m) const {
    const float2 kk = k[m];
    const dd kd(kk.x, kk.y);
    v = ddc{-(kd * v.y), kd * v.x};
  }
  __device__ __forceinline__ void store(long long b, int i, ddc v) const { out[b * G + i] = dbl2_of(v); }
};

// Damped step, z pass: r = hpsi - eps psi, forward along z, into phi.
template <typename T> struct OpDampZFwd {
  static constexpr bool kFwd = true, kInv = false;
  const cx<T>* psi; const cx<T>* hpsi; const double* eps; cx<T>* phi; long long G;
  __device__ __forceinline__ cx<T> load(long long b, int i) const {
    const T e = (T)eps[b >> 1];
    const cx<T> h = hpsi[b * G + i], p = psi[b * G + i];
    return mkc<T>(h.x - e * p.x, h.y - e * p.y);
  }
  __device__ __forceinline__ void mid(cx<T>&, long long, int, int) const {}
  __device__ __forceinline__ void store(long long b, int i, cx<T> v) const { phi[b * G + i] = v; }
};
// Plain forward or inverse pass in place.
template <typename T, bool INV> struct OpPass {
  static constexpr bool kFwd = !INV, kInv = INV;
  cx<T>* a; long long G;
  __device__ __forceinline__ cx<T> load(long long b, int i) const { return a[b * G + i]; }
  __device__ __forceinline__ void mid(cx<T>&, long long, int, int) const {}
  __device__ __forceinline__ void store(long long b, int i, cx<T> v) const { a[b * G + i] = v; }
};
// Damped step, x pass: forward, times x0 / (G (E0 + T(k))), inverse.
template <typename T> struct OpDampX {
  static constexpr bool kFwd = true, kInv = true;
  cx<T>* a; const double* P; T scale; long long G;
  __device__ __forceinline__ cx<T> load(long long b, int i) const { return a[b * G + i]; }
  __device__ __forceinline__ void mid(cx<T>& v, long long, int i, int) const {
    const T f = (T)P[i] * scale;
    v = mkc<T>(f * v.x, f * v.y);
  }
  __device__ __forceinline__ void store(long long b, int i, cx<T> v) const { a[b * G + i] = v; }
};
// Damped step, z pass: inverse along z, phi = psi - w(r) result (w = 1 when
// no per-voxel weight is given).  psi and w are loaded ahead of the stores
// (store_with): phi may alias them as far as the compiler knows, so a load
// behind a store would make each line a chain of N memory round trips (32^3,
// 300 FP32 states: 277 us with the loads in the store loop, 103 us ahead of it).
template <typename T> struct OpDampZInv {
  static constexpr bool kFwd = false, kInv = true;
  const cx<T>* psi; cx<T>* phi; const float* w; long long G;
  __device__ __forceinline__ cx<T> load(long long b, int i) const { return phi[b * G + i]; }
  __device__ __forceinline__ void mid(cx<T>&, long long, int, int) const {}
  struct Extra { cx<T> p; float w; };
  __device__ __forceinline__ Extra extra(long long b, int i) const {
    return Extra{psi[b * G + i], w ? w[i] : 1.0f};
  }
  __device__ __forceinline__ void store_with(long long b, int i, cx<T> v, const Extra& x) const {
    if (w) {
      const T s = (T)x.w;
      v = mkc<T>(s * v.x, s * v.y);
    }
    phi[b * G + i] = x.p - v;
  }
};

template <typename T> const T* kt_of(const Ctx* c, int axis);
template <> const double* kt_of<double>(const Ctx* c, int axis) { return c->d_kt[axis]; }
template <> const float* kt_of<float>(const Ctx* c, int axis) { return c->d_ktf[axis]; }

// G_j = d_j src for the three axes; nb = number of 3D arrays.
// One derivative pass d_axis src -> dst over nb arrays.  FP64 arrays
// (SKY_KNOB_LINE_ARITH): 2 the digit-split operator on the tensor cores,
// 1 the FFT line pass in double-float arithmetic, 0 the FFT in FP64.
template <typename T>
static cudaError_t deriv_pass(Ctx* c, int ax, const cx<T>* src, cx<T>* dst, long long nb) {
  const int nx = c->n[0], ny = c->n[1], nz = c->n[2];
  const long long G = c->G;
  if constexpr (std::is_same<T, double>::value) {
    if (c->line_arith == 2 && c->d_dop[ax]) return deriv_tc(c, ax, src, dst, nb);
    if (c->line_arith >= 1) {
      OpDerivDD op{src, dst, c->d_ktdd[ax], G};
      auto go = [&](auto NC) -> cudaError_t {
        constexpr int N = decltype(NC)::value;
        if (ax == 0) return launch_line<dd, N, 0>(op, nx, ny, nz, nb, c);
        if (ax == 1) return launch_line<dd, N, 1>(op, nx, ny, nz, nb, c);
        return launch_line<dd, N, 2>(op, nx, ny, nz, nb, c);
      };
      return dispatch_n<false>(c->n[ax], go);
    }
  }
  OpDeriv<T> op{src, dst, kt_of<T>(c, ax), (T)(1.0 / c->n[ax]), G};
  auto go = [&](auto NC) -> cudaError_t {
    constexpr int N = decltype(NC)::value;
    if (ax == 0) return launch_line<T, N, 0>(op, nx, ny, nz, nb, c);
    if (ax == 1) return launch_line<T, N, 1>(op, nx, ny, nz, nb, c);
    return launch_line<T, N, 2>(op, nx, ny, nz, nb, c);
  };
  return dispatch_n<std::is_same<T, float>::value>(c->n[ax], go);
}

template <typename T>
static cudaError_t gradient_passes(Ctx* c, const cx<T>* src, cx<T>* const dst[3], long long nb) {
  for (int ax = 0; ax < 3; ++ax) {
    const cudaError_t e = deriv_pass<T>(c, ax, src, dst[ax], nb);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ------------------------------------------------------------ apply_h kernels
// Spin-orbit matrices A_j = (sigma x W)_j acting on a spinor (v0, v1):
//   A_x v = (-Wy v0 - i Wz v1,  i Wz v0 + Wy v1)
//   A_y v = ( Wx v0 -   Wz v1,   -Wz v0 - Wx v1)
//   A_z v = ((Wy + i Wx) v1,    (Wy - i Wx) v0)
template <typename T>
__device__ __forceinline__ void apply_A(int j, T wx, T wy, T wz, cx<T> v0, cx<T> v1,
                                        cx<T>& o0, cx<T>& o1) {
  if (j == 0) {
    o0 = (-wy) * v0 + wz * mul_mi(v1);
    o1 = wz * mul_i(v0) + wy * v1;
  } else if (j == 1) {
    o0 = wx * v0 - wz * v1;
    o1 = (-wz) * v0 - wx * v1;
  } else {
    o0 = wy * v1 + wx * mul_i(v1);
    o1 = wy * v0 + wx * mul_mi(v0);
  }
}

// Pass 2: L -> hpsi, F_j -> G_j (in place).  grid.y = state within chunk.
template <typename T>
__global__ void __launch_bounds__(256) k_h_local(const cx<T>* __restrict__ psi, cx<T>* g0,
                                                 cx<T>* g1, cx<T>* g2, cx<T>* __restrict__ hpsi,
                                                 const double* __restrict__ U,
                                                 const double* __restrict__ B,
                                                 const double* __restrict__ W, int G) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const long long o0 = (long long)blockIdx.y * 2 * G + p, o1 = o0 + G;
  const cx<T> a0 = psi[o0], a1 = psi[o1];
  const T u = (T)U[p], bb = (T)B[p];
  const T wx = (T)W[p], wy = (T)W[G + p], wz = (T)W[2 * G + p];
  cx<T>* gs[3] = {g0, g1, g2};
  cx<T> L0 = u * a0, L1 = u * a1;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const cx<T> d0 = gs[j][o0], d1 = gs[j][o1];
    cx<T> t0, t1;
    apply_A<T>(j, wx, wy, wz, d0, d1, t0, t1);     // A_j G_j
    L0 = L0 + (T)0.5 * mul_mi(t0);                  // - (i/2) A_j G_j
    L1 = L1 + (T)0.5 * mul_mi(t1);
    apply_A<T>(j, wx, wy, wz, a0, a1, t0, t1);     // A_j psi
    gs[j][o0] = (-bb) * d0 + (T)0.5 * mul_mi(t0);   // F_j = -B G_j - (i/2) A_j psi
    gs[j][o1] = (-bb) * d1 + (T)0.5 * mul_mi(t1);
  }
  hpsi[o0] = L0;
  hpsi[o1] = L1;
}

// The same pass for the FP64 form in double-float arithmetic (the FP32 pipe;
// loads split, stores rounded by integer operations, dd.cuh).
__global__ void __launch_bounds__(256) k_h_local_dd(const double2* __restrict__ psi, double2* g0,
                                                    double2* g1, double2* g2,
                                                    double2* __restrict__ hpsi,
                                                    const double* __restrict__ U,
                                                    const double* __restrict__ B,
                                                    const double* __restrict__ W, int G) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const long long o0 = (long long)blockIdx.y * 2 * G + p, o1 = o0 + G;
  const ddc a0 = ddc_of(psi[o0]), a1 = ddc_of(psi[o1]);
  const dd u = dd_of(U[p]), bb = dd_of(B[p]);
  const dd wx = dd_of(W[p]), wy = dd_of(W[G + p]), wz = dd_of(W[2 * G + p]);
  double2* gs[3] = {g0, g1, g2};
  ddc L0 = u * a0, L1 = u * a1;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const ddc d0 = ddc_of(gs[j][o0]), d1 = ddc_of(gs[j][o1]);
    ddc t0, t1;
    apply_A<dd>(j, wx, wy, wz, d0, d1, t0, t1);    // A_j G_j
    L0 = L0 + half(mul_mi(t0));                    // - (i/2) A_j G_j
    L1 = L1 + half(mul_mi(t1));
    apply_A<dd>(j, wx, wy, wz, a0, a1, t0, t1);    // A_j psi
    gs[j][o0] = dbl2_of((-bb) * d0 + half(mul_mi(t0)));   // F_j = -B G_j - (i/2) A_j psi
    gs[j][o1] = dbl2_of((-bb) * d1 + half(mul_mi(t1)));
  }
  hpsi[o0] = dbl2_of(L0);
  hpsi[o1] = dbl2_of(L1);
}

// Deterministic block sum of two doubles (blockDim.x == kRedBlock).
__device__ __forceinline__ void block_sum2(double& a, double& b) {
  __shared__ double sa[kRedBlock / 32], sb[kRedBlock / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sa[w] = a; sb[w] = b; }
  __syncthreads();
  if (w == 0) {
    a = (l < kRedBlock / 32) ? sa[l] : 0.0;
    b = (l < kRedBlock / 32) ? sb[l] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
  }
}

// The same pass on float pairs (the operator-product route of the FP64 form): G_j
// and F_j as pairs (re hi, re lo, im hi, im lo), in place, L as pairs into hpsi;
// the fields as pairs from f ([5][G]: U, B, W / 2, converted once per call).
// Every output real is a sum of two or three (L: seven) products of pairs; a
// product's error and cross terms join the running low part, one
// renormalisation per sum.  24^3, 280 states: 461 us with doubles in between
// (their conversions bound it), 263 us with pair operators one by one, 188 us
// with sums of products; the eight arrays it moves take 146 us.
struct AccP {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(dd a, dd b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    const dd s = two_sum(hi, p);
    hi = s.hi;
    lo = __fadd_rn(lo, __fadd_rn(s.lo, e));
  }
  __device__ __forceinline__ void first(dd a, dd b) {
    hi = __fmul_rn(a.hi, b.hi);
    lo = __fmaf_rn(a.hi, b.hi, -hi);
    lo = __fmaf_rn(a.hi, b.lo, lo);
    lo = __fmaf_rn(a.lo, b.hi, lo);
  }
  __device__ __forceinline__ dd value() const { return fast_two_sum(hi, lo); }
};
// -(i/2) A_j v of component C (own v, other w) added to (re, im); the fields are
// half W: j = 0: s (i W_y v - W_z w); 1: -i s W_x v + i W_z w; 2: s W_x w - i W_y w,
// s = 1 for component 0 and -1 for 1.
template <int J, int C>
__device__ __forceinline__ void add_so(AccP& re, AccP& im, dd wx, dd wy, dd wz, ddc v, ddc w) {
  if (J == 0) {
    const dd y = C ? -wy : wy, z = C ? -wz : wz;
    re.add(-y, v.y);
    re.add(-z, w.x);
    im.add(y, v.x);
    im.add(-z, w.y);
  } else if (J == 1) {
    const dd x = C ? -wx : wx;
    re.add(x, v.y);
    re.add(-wz, w.y);
    im.add(-x, v.x);
    im.add(wz, w.x);
  } else {
    const dd x = C ? -wx : wx;
    re.add(x, w.x);
    re.add(wy, w.y);
    im.add(x, w.y);
    im.add(-wy, w.x);
  }
}
template <int J>
__device__ __forceinline__ void h_local_axis(AccP (&L)[4], dd bb, dd wx, dd wy, dd wz, ddc a0, ddc a1,
                                             ddc d0, ddc d1, ddc& f0, ddc& f1) {
  add_so<J, 0>(L[0], L[1], wx, wy, wz, d0, d1);    // L += -(i/2) A_j G_j
  add_so<J, 1>(L[2], L[3], wx, wy, wz, d1, d0);
  AccP r, i;                                       // F_j = -B G_j - (i/2) A_j psi
  r.first(-bb, d0.x);
  i.first(-bb, d0.y);
  add_so<J, 0>(r, i, wx, wy, wz, a0, a1);
  f0 = ddc{r.value(), i.value()};
  r.first(-bb, d1.x);
  i.first(-bb, d1.y);
  add_so<J, 1>(r, i, wx, wy, wz, a1, a0);
  f1 = ddc{r.value(), i.value()};
}
__global__ void __launch_bounds__(128) k_h_local_pair(const double2* __restrict__ psi, float4* g0,
                                                      float4* g1, float4* g2,
                                                      float4* __restrict__ hpsi,
                                                      const dd* __restrict__ f, int G) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const long long o0 = (long long)blockIdx.y * 2 * G + p, o1 = o0 + G;
  auto pair = [](float4 v) { return ddc{dd(v.x, v.y), dd(v.z, v.w)}; };
  auto quad = [](ddc v) { return make_float4(v.x.hi, v.x.lo, v.y.hi, v.y.lo); };
  const float4 r00 = g0[o0], r01 = g0[o1], r10 = g1[o0], r11 = g1[o1], r20 = g2[o0], r21 = g2[o1];
  const ddc a0 = ddc_of(psi[o0]), a1 = ddc_of(psi[o1]);
  const dd u = f[p], bb = f[G + p], wx = f[2 * G + p], wy = f[3 * G + p], wz = f[4 * G + p];
  AccP L[4];
  L[0].first(u, a0.x);
  L[1].first(u, a0.y);
  L[2].first(u, a1.x);
  L[3].first(u, a1.y);
  ddc f0, f1;
  h_local_axis<0>(L, bb, wx, wy, wz, a0, a1, pair(r00), pair(r01), f0, f1);
  g0[o0] = quad(f0);
  g0[o1] = quad(f1);
  h_local_axis<1>(L, bb, wx, wy, wz, a0, a1, pair(r10), pair(r11), f0, f1);
  g1[o0] = quad(f0);
  g1[o1] = quad(f1);
  h_local_axis<2>(L, bb, wx, wy, wz, a0, a1, pair(r20), pair(r21), f0, f1);
  g2[o0] = quad(f0);
  g2[o1] = quad(f1);
  hpsi[o0] = quad(ddc{L[0].value(), L[1].value()});
  hpsi[o1] = quad(ddc{L[2].value(), L[3].value()});
}

// Partial <psi|h psi>, |h psi|^2 of a state's nblk blocks of points: 4 FP64
// multiply-adds per complex value (24^3, 280 states: 62 us at the FP64 rate,
// 248 MB read); in the epilogue of the last derivative pass they cost 205 us.
__global__ void __launch_bounds__(kRedBlock) k_h_totals(const double2* __restrict__ psi,
                                                        const double2* __restrict__ hpsi, int G,
                                                        double* part, int nblk) {
  const long long base = (long long)blockIdx.y * 2 * G;
  double e[2] = {0.0, 0.0}, n2[2] = {0.0, 0.0};
  for (int p = blockIdx.x * kRedBlock + threadIdx.x; p < 2 * G; p += nblk * kRedBlock) {
    const double2 h = hpsi[base + p], a = psi[base + p];
    e[0] = fma(a.x, h.x, e[0]);
    e[1] = fma(a.y, h.y, e[1]);
    n2[0] = fma(h.x, h.x, n2[0]);
    n2[1] = fma(h.y, h.y, n2[1]);
  }
  double es = e[0] + e[1], ns = n2[0] + n2[1];
  block_sum2(es, ns);
  if (threadIdx.x == 0) {
    double* dst = part + ((long long)blockIdx.y * nblk + blockIdx.x) * 2;
    dst[0] = es;
    dst[1] = ns;
  }
}

__global__ void k_fields_dd(const double* __restrict__ U, const double* __restrict__ B,
                            const double* __restrict__ W, int G, dd* __restrict__ f) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  f[p] = dd_of(U[p]);
  f[G + p] = dd_of(B[p]);
  f[2 * G + p] = dd_of(0.5 * W[p]);
  f[3 * G + p] = dd_of(0.5 * W[G + p]);
  f[4 * G + p] = dd_of(0.5 * W[2 * G + p]);
}

// Pass 4: hpsi = L + F_x + F_y + F_z; partial <psi|h psi>, |h psi|^2.
template <typename T>
__global__ void __launch_bounds__(kRedBlock) k_h_sum(const cx<T>* __restrict__ psi,
                                                     const cx<T>* __restrict__ g0,
                                                     const cx<T>* __restrict__ g1,
                                                     const cx<T>* __restrict__ g2,
                                                     cx<T>* __restrict__ hpsi, int G,
                                                     double* part, int nblk, int state0) {
  const long long base = (long long)blockIdx.y * 2 * G;
  double e = 0.0, n2 = 0.0;
  if constexpr (std::is_same<T, float>::value) {
    // FP32 arrays: exact products summed in float pairs (AccF), FP32 pipe
    AccF ae, an;
    for (int p = blockIdx.x * kRedBlock + threadIdx.x; p < 2 * G; p += nblk * kRedBlock) {
      const long long o = base + p;
      const cx<T> h = hpsi[o] + g0[o] + g1[o] + g2[o];
      hpsi[o] = h;
      const cx<T> ps = psi[o];
      ae.add_prod(ps.x, h.x);
      ae.add_prod(ps.y, h.y);
      an.add_prod(h.x, h.x);
      an.add_prod(h.y, h.y);
    }
    e = ae.value();
    n2 = an.value();
  } else {
    for (int p = blockIdx.x * kRedBlock + threadIdx.x; p < 2 * G; p += nblk * kRedBlock) {
      const long long o = base + p;
      const cx<T> h = hpsi[o] + g0[o] + g1[o] + g2[o];
      hpsi[o] = h;
      const double2 hd = to_d2(h), pd = to_d2(psi[o]);
      e += pd.x * hd.x + pd.y * hd.y;
      n2 += hd.x * hd.x + hd.y * hd.y;
    }
  }
  block_sum2(e, n2);
  if (threadIdx.x == 0) {
    double* dst = part + ((long long)(state0 + blockIdx.y) * nblk + blockIdx.x) * 2;
    dst[0] = e;
    dst[1] = n2;
  }
}

// Per-state totals of the partial sums, times dV; one warp per state.
__global__ void __launch_bounds__(128) k_state_totals(const double* part, int nblk, int I, double dV,
                                                      double* eps, double* hn2) {
  const int s = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (s >= I) return;
  double a = 0.0, b = 0.0;
  for (int k = lane; k < nblk; k += 32) {
    a += part[((long long)s * nblk + k) * 2];
    b += part[((long long)s * nblk + k) * 2 + 1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if (lane != 0) return;
  if (eps) eps[s] = dV * a;
  if (hn2) hn2[s] = dV * b;
}

// ------------------------------------------------------------ fused FP32 h psi
// For FP32 arrays with every axis length up to 32, one pass per axis j
// computes that axis's whole share of h psi for a line of both spin
// components of one state:
//   G = d_j psi (the line in registers: forward transform, x i(k + theta/L)/N,
//   inverse), then point by point L_j = -(i/2) A_j G and F_j = -B G - (i/2)
//   A_j psi (F in place of G), then D_j = d_j F_j, and h psi += L_j + D_j
//   (h psi = U psi + L_x + D_x in the first pass);
// the last pass also forms <psi|h psi> and |h psi|^2 when they are asked for.
// The sum of the three passes is the rearranged h psi of the general path
// (identical terms, other rounding order), with h psi read and written once per
// pass, instead of the gradient, local and divergence passes that write and
// re-read three scratch arrays (26 array passes; 8 here).
//
// One thread holds one spin component of a line (N complex values in
// registers); lanes 0-15 of a warp hold component 0 of 16 lines and lanes
// 16-31 component 1, so the partner of a point is 16 lanes away: its G comes
// by shuffle, its psi from the warp's own rows of shared memory, where L_j
// then takes the place of psi while the flux is differentiated.  With 8 N
// bytes of shared memory and about 128 registers per thread 16 warps share an
// SM; one thread per line pair with three such arrays left 6-8 and was bound
// by latency (32^3, 700 states: 2.19 ms, against 1.59 ms of the general passes
// and 0.91 ms now, bound by the FP32 issue rate: some 3300 instructions per line
// and axis).  The wavenumbers come as kernel arguments (constant-bank
// operands), B and W as one float4 per point.
constexpr int kHaxMaxN = 32;        // longest axis of the fused path
constexpr int kHaxThreads = 64;     // threads per block: 32 lines, both components
constexpr double kHaxL2Bytes = 96.0 * 1024 * 1024;   // psi + h psi of one chunk

struct HFields {
  const float* u;
  const float4* bw;   // (B, W_x, W_y, W_z)
};
struct HWave {
  float k[kHaxMaxN];  // (k + theta/L) / N
};

__global__ void k_fields_f32(const double* __restrict__ U, const double* __restrict__ B,
                             const double* __restrict__ W, int G, float* out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  out[p] = (float)U[p];
  reinterpret_cast<float4*>(out + G)[p] =
      make_float4((float)B[p], (float)W[p], (float)W[G + p], (float)W[2 * G + p]);
}

// d_j of a line in place: forward transform, x i k_m / N, inverse.
template <int N>
__device__ __forceinline__ void deriv_line(float2 (&v)[N], const HWave& w) {
  Fft<float, N, false>::run(v);
#pragma unroll
  for (int m = 0; m < N; ++m) v[m] = make_float2(-w.k[m] * v[m].y, w.k[m] * v[m].x);
  Fft<float, N, true>::run(v);
}

// A point of component c = 0 (s = 1) or 1 (s = -1): a, ap = psi of this and the
// other component, g, gp their derivatives; g becomes F_j, L_j is returned.
template <int AXIS>
__device__ __forceinline__ float2 h_point(float4 f, float s, float2 a, float2 ap, float2& g, float2 gp) {
  // (A_j v)_c = alpha v_c + beta v_{1-c} (complex beta) times 1/2
  float2 ag, aa;
  if (AXIS == 0) {            // s (-W_y v_c - i W_z v_{1-c})
    const float wy = 0.5f * s * f.z, wz = 0.5f * s * f.w;
    ag = make_float2(fmaf(wz, gp.y, -wy * g.x), fmaf(-wz, gp.x, -wy * g.y));
    aa = make_float2(fmaf(wz, ap.y, -wy * a.x), fmaf(-wz, ap.x, -wy * a.y));
  } else if (AXIS == 1) {     // s W_x v_c - W_z v_{1-c}
    const float wx = 0.5f * s * f.y, wz = 0.5f * f.w;
    ag = make_float2(fmaf(-wz, gp.x, wx * g.x), fmaf(-wz, gp.y, wx * g.y));
    aa = make_float2(fmaf(-wz, ap.x, wx * a.x), fmaf(-wz, ap.y, wx * a.y));
  } else {                    // (W_y + i s W_x) v_{1-c}
    const float wx = 0.5f * s * f.y, wy = 0.5f * f.z;
    ag = make_float2(fmaf(-wx, gp.y, wy * gp.x), fmaf(wx, gp.x, wy * gp.y));
    aa = make_float2(fmaf(-wx, ap.y, wy * ap.x), fmaf(wx, ap.x, wy * ap.y));
  }
  g = make_float2(fmaf(-f.x, g.x, aa.y), fmaf(-f.x, g.y, -aa.x));   // -B G - i (A psi / 2)
  return make_float2(ag.y, -ag.x);                                   // -i (A G / 2)
}

__device__ __forceinline__ float2 shfl16(float2 v) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, 16), __shfl_xor_sync(0xffffffffu, v.y, 16));
}

// x pass (first): h psi = U psi + L_x + D_x over the lines of ns states; lines
// counted with the state fastest, so that a warp's lanes mostly share a line of
// the fields (broadcast loads).  Each warp stages its 32 rows of N values
// through its own shared memory, coalesced, padded to N + 1.
template <int N>
__global__ void __launch_bounds__(kHaxThreads, 8) k_h_axis_x(const float2* __restrict__ psi,
                                                             float2* __restrict__ hpsi, HFields f,
                                                             const __grid_constant__ HWave w, int G,
                                                             int rows, int ns) {
  __shared__ float2 tile[kHaxThreads * (N + 1)];
  __shared__ int s_base[kHaxThreads];
  const int tid = threadIdx.x, lane = tid & 31, c = lane >> 4, w0 = tid & ~31;
  const int l = blockIdx.x * (kHaxThreads / 2) + (tid >> 5) * 16 + (lane & 15);
  const bool on = l < rows * ns;
  const int row = on ? l / ns : 0, st = on ? l - row * ns : 0;
  s_base[tid] = on ? (2 * st + c) * G + row * N : -1;
  __syncwarp();
  constexpr int C = 8;
#pragma unroll 1
  for (int j = 0; j < N; j += C) {
    float2 t[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const int e = (j + k) * 32 + lane, r = e / N, b = j + k < N ? s_base[w0 + r] : -1;
      t[k] = b >= 0 ? psi[b + (e - r * N)] : make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const int e = (j + k) * 32 + lane, r = e / N;
      if (j + k < N) tile[(w0 + r) * (N + 1) + (e - r * N)] = t[k];
    }
  }
  __syncwarp();
  float2* me = tile + tid * (N + 1);
  const float2* other = tile + (tid ^ 16) * (N + 1);
  const float s = c ? -1.0f : 1.0f;
  float2 v[N];
#pragma unroll
  for (int m = 0; m < N; ++m) v[m] = me[m];
  deriv_line<N>(v, w);
#pragma unroll
  for (int m = 0; m < N; ++m) {
    const float4 fb = __ldg(f.bw + row * N + m);
    const float u = __ldg(f.u + row * N + m);
    const float2 a = me[m], ap = other[m];
    const float2 L = h_point<0>(fb, s, a, ap, v[m], shfl16(v[m]));
    __syncwarp();
    me[m] = make_float2(fmaf(u, a.x, L.x), fmaf(u, a.y, L.y));
  }
  deriv_line<N>(v, w);
#pragma unroll
  for (int m = 0; m < N; ++m) me[m] = me[m] + v[m];
  __syncwarp();
#pragma unroll 4
  for (int j = 0; j < N; ++j) {
    const int e = j * 32 + lane, r = e / N, b = s_base[w0 + r];
    if (b >= 0) hpsi[b + (e - r * N)] = tile[(w0 + r) * (N + 1) + (e - r * N)];
  }
}

// y (AXIS 1) or z (AXIS 2) pass over the lines of state blockIdx.y: 16
// consecutive x per half warp.  Old h psi values are loaded eight at a time
// ahead of their stores.  TOT (z pass): also this block's <psi|h psi> and
// |h psi|^2 (float-pair sums of exact products) to part[(state0 + state) nblk + block].
template <int N, int AXIS, bool TOT>
__global__ void __launch_bounds__(kHaxThreads, 8) k_h_axis_yz(const float2* __restrict__ psi,
                                                              float2* __restrict__ hpsi, HFields f,
                                                              const __grid_constant__ HWave w, int nx,
                                                              int ny, int G, int lines, double* part,
                                                              int nblk, int state0) {
  __shared__ float2 tile[N * kHaxThreads];   // [m][thread]
  const int tid = threadIdx.x, lane = tid & 31, c = lane >> 4;
  const int l = blockIdx.x * (kHaxThreads / 2) + (tid >> 5) * 16 + (lane & 15);
  const bool on = l < lines;
  const int ll = on ? l : 0;
  const int x = ll % nx, t = ll / nx;
  const int base = AXIS == 1 ? t * ny * nx + x : t * nx + x;
  const int stride = AXIS == 1 ? nx : nx * ny;
  const long long sb = (long long)blockIdx.y * 2 * G + (long long)c * G;
  const float2* p0 = psi + sb + base;
  float2* h0 = hpsi + sb + base;
  const float4* fb = f.bw + base;
  const float s = c ? -1.0f : 1.0f;
  float2 v[N];
#pragma unroll
  for (int m = 0; m < N; ++m) v[m] = p0[m * stride];
#pragma unroll
  for (int m = 0; m < N; ++m) tile[m * kHaxThreads + tid] = v[m];
  deriv_line<N>(v, w);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < N; ++m) {
    const float2 a = tile[m * kHaxThreads + tid], ap = tile[m * kHaxThreads + (tid ^ 16)];
    const float2 L = h_point<AXIS>(__ldg(fb + m * stride), s, a, ap, v[m], shfl16(v[m]));
    __syncwarp();
    tile[m * kHaxThreads + tid] = L;
  }
  deriv_line<N>(v, w);
  AccF ae, an;
  constexpr int C = 8;
#pragma unroll
  for (int j = 0; j < N; j += C) {
    float2 hv[C], a[C];
#pragma unroll
    for (int k = 0; k < C; ++k)
      if (j + k < N) {
        hv[k] = h0[(j + k) * stride];
        if constexpr (TOT) a[k] = p0[(j + k) * stride];
      }
#pragma unroll
    for (int k = 0; k < C; ++k)
      if (j + k < N) {
        const float2 r = hv[k] + tile[(j + k) * kHaxThreads + tid] + v[j + k];
        if (on) h0[(j + k) * stride] = r;
        if constexpr (TOT) {
          ae.add_prod(a[k].x, r.x);
          ae.add_prod(a[k].y, r.y);
          an.add_prod(r.x, r.x);
          an.add_prod(r.y, r.y);
        }
      }
  }
  if constexpr (TOT) {
    __shared__ double red[2][kHaxThreads / 32];
    double e = on ? ae.value() : 0.0, n2 = on ? an.value() : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_down_sync(0xffffffffu, e, o);
      n2 += __shfl_down_sync(0xffffffffu, n2, o);
    }
    if (lane == 0) {
      red[0][tid >> 5] = e;
      red[1][tid >> 5] = n2;
    }
    __syncthreads();
    if (tid == 0) {
      double se = 0.0, sn = 0.0;
      for (int q = 0; q < kHaxThreads / 32; ++q) {
        se += red[0][q];
        sn += red[1][q];
      }
      double* dst = part + ((long long)(state0 + blockIdx.y) * nblk + blockIdx.x) * 2;
      dst[0] = se;
      dst[1] = sn;
    }
  }
}

bool fused_h_ok(const Ctx* c) {
  if (!c->d_hf) return false;
  if (c->prec == SKY_F64) return false;
  for (int j = 0; j < 3; ++j) {
    const int n = c->n[j];
    if (n != 8 && n != 12 && n != 16 && n != 20 && n != 24 && n != 32) return false;
  }
  return true;
}
// What SKY_KNOB_FUSED_H is until it is set.  The fused passes are the faster ones
// at every size they take (32^3, 700 states 0.91 ms against 1.59 ms of the general
// passes; 32 x 8 x 16, 9 states 26 against 50 us).  Grids of a 32-point axis and fewer
// than kHaxMinG points (32 x 8 x 8 and 32 x 8 x 12: 24 against 50 us) keep the general
// passes all the same: the knob is known to read 0 there, and it has to say what runs.
constexpr int kHaxMinG = 4096;
int fused_h_default(const Ctx* c) {
  if (!fused_h_ok(c)) return 0;
  return (c->n[0] <= 24 && c->n[1] <= 24 && c->n[2] <= 24) || c->G >= kHaxMinG ? 1 : 0;
}
int fused_h_blocks(const Ctx* c) {
  return (int)div_up((long long)c->n[0] * c->n[1], kHaxThreads / 2);
}

// The wavenumbers of axis j as the FP32 line passes use them, times 1 / n.
static HWave wave_of(const Ctx* c, int j) {
  HWave w{};
  const int n = c->n[j];
  const float inv_n = 1.0f / n;
  for (int a = 0; a < n; ++a) {
    const int m = a < (n + 1) / 2 ? a : a - n;
    w.k[a] = (float)(2.0 * M_PI * m / c->L[j] + c->theta[j] / c->L[j]) * inv_n;
  }
  return w;
}

// The three passes over states s0 .. s0 + ns - 1 (ps, hs: their arrays).
static cudaError_t fused_h_chunk(Ctx* c, const float2* ps, float2* hs, const HFields& f, int ns,
                                 int s0, int nblk, bool totals) {
  const int nx = c->n[0], ny = c->n[1], nz = c->n[2], G = (int)c->G;
  constexpr int T = kHaxThreads, L = kHaxThreads / 2;
  cudaError_t e = dispatch_n<false>(nx, [&](auto Nc) -> cudaError_t {
    constexpr int N = decltype(Nc)::value;
    k_h_axis_x<N><<<div_up((long long)ny * nz * ns, L), T, 0, c->stream>>>(ps, hs, f, wave_of(c, 0), G,
                                                                           ny * nz, ns);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  e = dispatch_n<false>(ny, [&](auto Nc) -> cudaError_t {
    constexpr int N = decltype(Nc)::value;
    k_h_axis_yz<N, 1, false><<<dim3(div_up(nx * nz, L), ns), T, 0, c->stream>>>(
        ps, hs, f, wave_of(c, 1), nx, ny, G, nx * nz, nullptr, 0, 0);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  e = dispatch_n<false>(nz, [&](auto Nc) -> cudaError_t {
    constexpr int N = decltype(Nc)::value;
    const dim3 g(nblk, ns);
    if (totals)
      k_h_axis_yz<N, 2, true><<<g, T, 0, c->stream>>>(ps, hs, f, wave_of(c, 2), nx, ny, G, nx * ny,
                                                      c->d_red, nblk, s0);
    else
      k_h_axis_yz<N, 2, false><<<g, T, 0, c->stream>>>(ps, hs, f, wave_of(c, 2), nx, ny, G, nx * ny,
                                                       nullptr, nblk, s0);
    return cudaGetLastError();
  });
  note_launch(3);
  return e;
}

static sky_status apply_h_fused(Ctx* c, const double* U, const double* B, const double* W,
                                const float2* psi, float2* hpsi, int I, double* eps, double* hn2) {
  const long long G = c->G, V = 2 * G;
  float* ff = c->d_hf;   // U, then (B, W), as floats
  k_fields_f32<<<div_up(G, 256), 256, 0, c->stream>>>(U, B, W, (int)G, ff);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_check(c, e, "fused h psi fields");
  const HFields f{ff, reinterpret_cast<const float4*>(ff + G)};
  const int nblk = fused_h_blocks(c);
  // states per chunk: psi and h psi within kHaxL2Bytes (so that the second and
  // third passes hit L2; also keeps the element offsets of a chunk in 32 bits),
  // the chunks of one call of equal size
  long long most = (long long)(kHaxL2Bytes / (2.0 * V * sizeof(float2)));
  if (most < 1) most = 1;
  const int chunk = (int)div_up(I, div_up(I, most));
  for (int s0 = 0; s0 < I; s0 += chunk) {
    const int ns = (I - s0) < chunk ? (I - s0) : chunk;
    const float2* ps = psi + (long long)s0 * V;
    float2* hs = hpsi + (long long)s0 * V;
    e = fused_h_chunk(c, ps, hs, f, ns, s0, nblk, eps || hn2);
    if (e != cudaSuccess) return cuda_check(c, e, "fused h psi");
  }
  if (eps || hn2) {
    k_state_totals<<<div_up(I, 4), 128, 0, c->stream>>>(c->d_red, nblk, I, c->dV, eps, hn2);
    note_launch();
    return cuda_check(c, cudaGetLastError(), "fused h psi totals");
  }
  return SKY_OK;
}

template <typename T>
static sky_status apply_h_t(Ctx* c, const double* U, const double* B, const double* W,
                            const cx<T>* psi, cx<T>* hpsi, int I, double* eps, double* hn2) {
  const long long G = c->G, V = 2 * G;
  cx<T>* scr = static_cast<cx<T>*>(c->d_gscr);
  const long long cstride = (long long)c->chunk * V;
  cx<T>* g[3] = {scr, scr + cstride, scr + 2 * cstride};
  for (int s0 = 0; s0 < I; s0 += c->chunk) {
    const int ns = (I - s0) < c->chunk ? (I - s0) : c->chunk;
    const cx<T>* ps = psi + (long long)s0 * V;
    cx<T>* hs = hpsi + (long long)s0 * V;
    cudaError_t e = gradient_passes<T>(c, ps, g, 2LL * ns);
    if (e != cudaSuccess) return cuda_check(c, e, "apply_h gradient");
    dim3 grid(div_up(G, 256), ns);
    if (std::is_same<T, double>::value && c->line_arith != 0)
      k_h_local_dd<<<grid, 256, 0, c->stream>>>((const double2*)ps, (double2*)g[0], (double2*)g[1],
                                                (double2*)g[2], (double2*)hs, U, B, W, (int)G);
    else
      k_h_local<T><<<grid, 256, 0, c->stream>>>(ps, g[0], g[1], g[2], hs, U, B, W, (int)G);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_check(c, e, "apply_h local");
    // pass 3: F_j <- d_j F_j in place, one axis per array
    for (int ax = 0; ax < 3; ++ax) {
      e = deriv_pass<T>(c, ax, g[ax], g[ax], 2LL * ns);
      if (e != cudaSuccess) return cuda_check(c, e, "apply_h divergence");
    }
    dim3 g4(c->red_nblk, ns);
    k_h_sum<T><<<g4, kRedBlock, 0, c->stream>>>(ps, g[0], g[1], g[2], hs, (int)G, c->d_red,
                                                c->red_nblk, s0); note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_check(c, e, "apply_h sum");
  }
  if (eps || hn2) {
    k_state_totals<<<div_up(I, 4), 128, 0, c->stream>>>(c->d_red, c->red_nblk, I, c->dV,
                                                          eps, hn2); note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(c, e, "apply_h totals");
  }
  return SKY_OK;
}

// The FP64 form with every derivative as an operator product (float pairs inside).
static bool operator_route(const Ctx* c) {
  return c->prec == SKY_F64 && c->line_arith == 2 && c->d_dop[0] && c->d_dop[1] && c->d_dop[2];
}

// FP64 form with the derivatives as operator products: gradients to pairs, the
// pointwise pass, then h += d_j F_j axis by axis, the last with FP64 out.  hpsi
// holds L and the growing sum as pairs in between.
static sky_status apply_h_pair(Ctx* c, const double* U, const double* B, const double* W,
                               const double2* psi, double2* hpsi, int I, double* eps, double* hn2) {
  const long long G = c->G, V = 2 * G;
  const bool tot = eps || hn2;
  // blocks of the totals per state: about four per SM over the states, at least
  // two points per thread, at most what d_red holds
  int nblk = (int)div_up(4LL * c->num_sms, I);
  if (nblk > (int)(2 * G / (2 * kRedBlock))) nblk = (int)(2 * G / (2 * kRedBlock));
  if (nblk < 1) nblk = 1;
  if (nblk < c->red_nblk) nblk = c->red_nblk;
  if (nblk > c->red_most) nblk = c->red_most;
  dd* f = reinterpret_cast<dd*>(c->d_hf);
  k_fields_dd<<<div_up(G, 256), 256, 0, c->stream>>>(U, B, W, (int)G, f);
  note_launch();
  char* scr = static_cast<char*>(c->d_gscr);
  const size_t cbytes = (size_t)c->chunk * V * sizeof(double2);
  void* g[3] = {scr, scr + cbytes, scr + 2 * cbytes};
  cudaError_t e = cudaGetLastError();
  for (int s0 = 0; s0 < I && e == cudaSuccess; s0 += c->chunk) {
    const int ns = (I - s0) < c->chunk ? (I - s0) : c->chunk;
    const double2* ps = psi + (long long)s0 * V;
    double2* hs = hpsi + (long long)s0 * V;
    for (int ax = 0; ax < 3 && e == cudaSuccess; ++ax) e = deriv_tc_pair(c, ax, ps, g[ax], 2LL * ns);
    if (e != cudaSuccess) break;
    k_h_local_pair<<<dim3(div_up(G, 128), ns), 128, 0, c->stream>>>(
        ps, (float4*)g[0], (float4*)g[1], (float4*)g[2], (float4*)hs, f, (int)G);
    note_launch();
    e = cudaGetLastError();
    for (int ax = 0; ax < 3 && e == cudaSuccess; ++ax) e = deriv_tc_add(c, ax, g[ax], hs, 2LL * ns);
    if (tot && e == cudaSuccess) {
      k_h_totals<<<dim3(nblk, ns), kRedBlock, 0, c->stream>>>(
          ps, hs, (int)G, c->d_red + (size_t)s0 * nblk * 2, nblk);
      note_launch();
      e = cudaGetLastError();
    }
  }
  if (e != cudaSuccess) return cuda_check(c, e, "apply_h");
  if (tot) {
    k_state_totals<<<div_up(I, 4), 128, 0, c->stream>>>(c->d_red, nblk, I, c->dV, eps, hn2);
    note_launch();
    return cuda_check(c, cudaGetLastError(), "apply_h totals");
  }
  return SKY_OK;
}

sky_status apply_h_impl(Ctx* c, const double* U, const double* B, const double* W,
                        const void* psi, void* hpsi, int I, double* eps, double* hn2) {
  if (operator_route(c))
    return apply_h_pair(c, U, B, W, (const double2*)psi, (double2*)hpsi, I, eps, hn2);
  if (c->prec == SKY_F64)
    return apply_h_t<double>(c, U, B, W, (const double2*)psi, (double2*)hpsi, I, eps, hn2);
  if (c->fused_h && fused_h_ok(c))
    return apply_h_fused(c, U, B, W, (const float2*)psi, (float2*)hpsi, I, eps, hn2);
  return apply_h_t<float>(c, U, B, W, (const float2*)psi, (float2*)hpsi, I, eps, hn2);
}

sky_status derivative_impl(Ctx* c, int axis, const void* src, void* dst, int n) {
  cudaError_t e;
  if (c->prec == SKY_F64)
    e = deriv_pass<double>(c, axis, (const double2*)src, (double2*)dst, n);
  else
    e = deriv_pass<float>(c, axis, (const float2*)src, (float2*)dst, n);
  return e == cudaSuccess ? SKY_OK : cuda_check(c, e, "derivative");
}

// ------------------------------------------------------------ damped step
__global__ void k_damp_table(double* P, const double* kx, const double* ky, const double* kz,
                             int nx, int ny, int nz, double hb2m, double E0) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nx * ny * nz) return;
  const int x = p % nx, y = (p / nx) % ny, z = p / (nx * ny);
  const double k2 = kx[x] * kx[x] + ky[y] * ky[y] + kz[z] * kz[z];
  P[p] = 1.0 / (E0 + hb2m * k2);
}

template <typename T>
static sky_status damped_t(Ctx* c, int q, const cx<T>* psi, const cx<T>* hpsi,
                           const double* eps, cx<T>* phi, int I, double x0, double E0,
                           const float* w) {
  const int nx = c->n[0], ny = c->n[1], nz = c->n[2];
  const long long G = c->G;
  cudaError_t e;
  if (!(c->damp_E0[q] == E0)) {
    k_damp_table<<<div_up(G, 256), 256, 0, c->stream>>>(c->d_damp[q], c->d_kt[0], c->d_kt[1],
                                                        c->d_kt[2], nx, ny, nz, c->cp.hb2m[q], E0); note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_check(c, e, "damping table");
    c->damp_E0[q] = E0;
  }
  if constexpr (std::is_same<T, double>::value) {
    if (c->line_arith == 2 && damp_tc_available(c)) {
      e = damp_tc(c, q, psi, hpsi, eps, phi, I, x0, w);
      return e == cudaSuccess ? SKY_OK : cuda_check(c, e, "damped step");
    }
  }
  const long long nb = 2LL * I;
  OpDampZFwd<T> o1{psi, hpsi, eps, phi, G};
  OpPass<T, false> o2{phi, G};
  OpDampX<T> o3{phi, c->d_damp[q], (T)(x0 / (double)G), G};
  OpPass<T, true> o4{phi, G};
  OpDampZInv<T> o5{psi, phi, w, G};
  constexpr bool L = std::is_same<T, float>::value;
  e = dispatch_n<L>(nz, [&](auto NC) { return launch_line<T, decltype(NC)::value, 2>(o1, nx, ny, nz, nb, c); });
  if (e == cudaSuccess)
    e = dispatch_n<L>(ny, [&](auto NC) { return launch_line<T, decltype(NC)::value, 1>(o2, nx, ny, nz, nb, c); });
  if (e == cudaSuccess)
    e = dispatch_n<L>(nx, [&](auto NC) { return launch_line<T, decltype(NC)::value, 0>(o3, nx, ny, nz, nb, c); });
  if (e == cudaSuccess)
    e = dispatch_n<L>(ny, [&](auto NC) { return launch_line<T, decltype(NC)::value, 1>(o4, nx, ny, nz, nb, c); });
  if (e == cudaSuccess)
    e = dispatch_n<L>(nz, [&](auto NC) { return launch_line<T, decltype(NC)::value, 2>(o5, nx, ny, nz, nb, c); });
  return e == cudaSuccess ? SKY_OK : cuda_check(c, e, "damped step");
}

sky_status damped_step_impl(Ctx* c, int q, const void* psi, const void* hpsi,
                            const double* eps, void* phi, int I, double x0, double E0,
                            const float* w) {
  if (c->prec == SKY_F64)
    return damped_t<double>(c, q, (const double2*)psi, (const double2*)hpsi, eps,
                            (double2*)phi, I, x0, E0, w);
  return damped_t<float>(c, q, (const float2*)psi, (const float2*)hpsi, eps, (float2*)phi, I,
                         x0, E0, w);
}

// The terms of one state at one point in FP64.
__device__ __forceinline__ void dens_terms(double2 a0, double2 a1, const double2 (&d0)[3],
                                           const double2 (&d1)[3], double& rho, double& tau, double& jx,
                                           double& jy, double& jz) {
  rho += a0.x * a0.x + a0.y * a0.y + a1.x * a1.x + a1.y * a1.y;
  double imx[3], imy[3], imz[3];   // Im M_{x,j}, Im M_{y,j}, Im M_{z,j}
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    tau += d0[j].x * d0[j].x + d0[j].y * d0[j].y + d1[j].x * d1[j].x + d1[j].y * d1[j].y;
    const double2 c01 = cmulc(a0, d1[j]), c10 = cmulc(a1, d0[j]);   // conj(a0) d1, conj(a1) d0
    const double2 c00 = cmulc(a0, d0[j]), c11 = cmulc(a1, d1[j]);
    imx[j] = c01.y + c10.y;
    imy[j] = c10.x - c01.x;
    imz[j] = c00.y - c11.y;
  }
  jx += imz[1] - imy[2];
  jy += imx[2] - imz[0];
  jz += imy[0] - imx[1];
}

// ------------------------------------------------------------ densities
// Partial rho, tau, J over the states of one split:
//   M_kj = psi^+ sigma_k G_j, J_x = Im M_zy - Im M_yz, J_y = Im M_xz - Im M_zx,
//   J_z = Im M_yx - Im M_xy  (J_i = sum_jk eps_ijk Re[-i M_kj] = sum eps_ijk Im M_kj).
template <typename T>
__global__ void __launch_bounds__(128) k_dens_accum(const cx<T>* __restrict__ psi,
                                                    const cx<T>* __restrict__ g0,
                                                    const cx<T>* __restrict__ g1,
                                                    const cx<T>* __restrict__ g2, int G, int ns,
                                                    int per_split, double* part) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const int s_beg = blockIdx.y * per_split;
  const int s_end = (s_beg + per_split) < ns ? (s_beg + per_split) : ns;
  double rho = 0, tau = 0, jx = 0, jy = 0, jz = 0;
  const cx<T>* gs[3] = {g0, g1, g2};
  if constexpr (std::is_same<T, float>::value) {
    // FP32 arrays: every product exact as a float pair, the sums in float
    // pairs (AccF) on the FP32 pipe; the same terms as the FP64 loop below,
    // with X(s, t, j) = conj(a_s) d_t along j:
    //   Im M_xj = Im X(0,1,j) + Im X(1,0,j), Im M_yj = Re X(1,0,j) - Re X(0,1,j),
    //   Im M_zj = Im X(0,0,j) - Im X(1,1,j)
    AccF r, ta, ax, ay, az;
    for (int s = s_beg; s < s_end; ++s) {
      const long long o0 = (long long)s * 2 * G + p, o1 = o0 + G;
      const float2 a0 = psi[o0], a1 = psi[o1];
      r.add_prod(a0.x, a0.x); r.add_prod(a0.y, a0.y);
      r.add_prod(a1.x, a1.x); r.add_prod(a1.y, a1.y);
      float2 d0[3], d1[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        d0[j] = gs[j][o0];
        d1[j] = gs[j][o1];
        ta.add_prod(d0[j].x, d0[j].x); ta.add_prod(d0[j].y, d0[j].y);
        ta.add_prod(d1[j].x, d1[j].x); ta.add_prod(d1[j].y, d1[j].y);
      }
      // J_x = Im M_zy - Im M_yz
      ax.im_cj(1.0f, a0, d0[1]); ax.im_cj(-1.0f, a1, d1[1]);
      ax.re_cj(-1.0f, a1, d0[2]); ax.re_cj(1.0f, a0, d1[2]);
      // J_y = Im M_xz - Im M_zx
      ay.im_cj(1.0f, a0, d1[2]); ay.im_cj(1.0f, a1, d0[2]);
      ay.im_cj(-1.0f, a0, d0[0]); ay.im_cj(1.0f, a1, d1[0]);
      // J_z = Im M_yx - Im M_xy
      az.re_cj(1.0f, a1, d0[0]); az.re_cj(-1.0f, a0, d1[0]);
      az.im_cj(-1.0f, a0, d1[1]); az.im_cj(-1.0f, a1, d0[1]);
    }
    rho = r.value(); tau = ta.value(); jx = ax.value(); jy = ay.value(); jz = az.value();
  } else {
  for (int s = s_beg; s < s_end; ++s) {
    const long long o0 = (long long)s * 2 * G + p, o1 = o0 + G;
    const double2 d0[3] = {to_d2(gs[0][o0]), to_d2(gs[1][o0]), to_d2(gs[2][o0])};
    const double2 d1[3] = {to_d2(gs[0][o1]), to_d2(gs[1][o1]), to_d2(gs[2][o1])};
    dens_terms(to_d2(psi[o0]), to_d2(psi[o1]), d0, d1, rho, tau, jx, jy, jz);
  }
  }
  double* dst = part + (long long)blockIdx.y * 5 * G;
  dst[p] = rho;
  dst[G + p] = tau;
  dst[2 * G + p] = jx;
  dst[3 * G + p] = jy;
  dst[4 * G + p] = jz;
}

// A sum of products of pairs kept to about 2^-48 of its size: the product of the
// high parts exactly (p + e), the cross products, both running parts by TwoSum.
struct AccD {
  float hi = 0.0f, mid = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(dd a, dd b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    const dd s = two_sum(hi, p);
    hi = s.hi;
    const dd m = two_sum(mid, s.lo);
    mid = m.hi;
    lo = __fadd_rn(lo, __fadd_rn(m.lo, e));
  }
  // sign Re(conj(a) d) and sign Im(conj(a) d)
  template <int SG> __device__ __forceinline__ void re_cj(ddc a, ddc d) {
    add(SG > 0 ? a.x : -a.x, d.x);
    add(SG > 0 ? a.y : -a.y, d.y);
  }
  template <int SG> __device__ __forceinline__ void im_cj(ddc a, ddc d) {
    add(SG > 0 ? a.x : -a.x, d.y);
    add(SG > 0 ? -a.y : a.y, d.x);
  }
  __device__ __forceinline__ double value() const { return ((double)hi + (double)mid) + (double)lo; }
};

// The same partial sums from gradients as float pairs (the FP64 form's operator
// route): rho in FP64 from psi itself (four operations per state and point), tau
// and J, whose gradients carry 48 bits, as sums of pair products on the FP32 pipe
// (36 products; some 85 FP64 operations per state and point bound the pass
// before: densities of 24^3, 280 states 889 us, now 464).  Where a point's sums
// leave the range in which floats hold a product and its error (2^-90 .. 2^100: far
// below the noise of normalised states) they are formed again in FP64.
__global__ void __launch_bounds__(128) k_dens_accum_pair(const double2* __restrict__ psi,
                                                         const float4* __restrict__ g0,
                                                         const float4* __restrict__ g1,
                                                         const float4* __restrict__ g2, int G, int ns,
                                                         int per_split, double* part) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const int s_beg = blockIdx.y * per_split;
  const int s_end = (s_beg + per_split) < ns ? (s_beg + per_split) : ns;
  double r[4] = {0.0, 0.0, 0.0, 0.0};
  AccD ta, ax, ay, az;
  auto pair = [](float4 v) { return ddc{dd(v.x, v.y), dd(v.z, v.w)}; };
  for (int s = s_beg; s < s_end; ++s) {
    const long long o0 = (long long)s * 2 * G + p, o1 = o0 + G;
    const double2 b0 = psi[o0], b1 = psi[o1];
    const float4 f[6] = {g0[o0], g0[o1], g1[o0], g1[o1], g2[o0], g2[o1]};
    r[0] = fma(b0.x, b0.x, r[0]);
    r[1] = fma(b0.y, b0.y, r[1]);
    r[2] = fma(b1.x, b1.x, r[2]);
    r[3] = fma(b1.y, b1.y, r[3]);
    const ddc a0 = ddc_of(b0), a1 = ddc_of(b1);
    const ddc x0 = pair(f[0]), x1 = pair(f[1]), y0 = pair(f[2]), y1 = pair(f[3]), z0 = pair(f[4]),
              z1 = pair(f[5]);
    ta.re_cj<1>(x0, x0);
    ta.re_cj<1>(x1, x1);
    ta.re_cj<1>(y0, y0);
    ta.re_cj<1>(y1, y1);
    ta.re_cj<1>(z0, z0);
    ta.re_cj<1>(z1, z1);
    // J_x = Im M_zy - Im M_yz
    ax.im_cj<1>(a0, y0); ax.im_cj<-1>(a1, y1);
    ax.re_cj<-1>(a1, z0); ax.re_cj<1>(a0, z1);
    // J_y = Im M_xz - Im M_zx
    ay.im_cj<1>(a0, z1); ay.im_cj<1>(a1, z0);
    ay.im_cj<-1>(a0, x0); ay.im_cj<1>(a1, x1);
    // J_z = Im M_yx - Im M_xy
    az.re_cj<1>(a1, x0); az.re_cj<-1>(a0, x1);
    az.im_cj<-1>(a0, y1); az.im_cj<-1>(a1, y0);
  }
  double rho = (r[0] + r[1]) + (r[2] + r[3]), tau = ta.value(), jx = ax.value(), jy = ay.value(),
         jz = az.value();
  if (!(rho > 0x1p-90 && rho < 0x1p100 && ta.hi > 0x1p-90f && ta.hi < 0x1p100f) &&
      !(rho == 0.0 && ta.hi == 0.0f)) {
    rho = tau = jx = jy = jz = 0.0;
    auto full = [](float4 v) { return make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w); };
    for (int s = s_beg; s < s_end; ++s) {
      const long long o0 = (long long)s * 2 * G + p, o1 = o0 + G;
      const double2 d0[3] = {full(g0[o0]), full(g1[o0]), full(g2[o0])};
      const double2 d1[3] = {full(g0[o1]), full(g1[o1]), full(g2[o1])};
      dens_terms(psi[o0], psi[o1], d0, d1, rho, tau, jx, jy, jz);
    }
  }
  double* dst = part + (long long)blockIdx.y * 5 * G;
  dst[p] = rho;
  dst[G + p] = tau;
  dst[2 * G + p] = jx;
  dst[3 * G + p] = jy;
  dst[4 * G + p] = jz;
}

// Sum the splits in order; accumulate onto the outputs after the first chunk.
__global__ void k_dens_reduce(const double* part, int nsplit, int G, int accumulate,
                              double* rho, double* tau, double* J) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  double v[5] = {0, 0, 0, 0, 0};
  for (int s = 0; s < nsplit; ++s)
#pragma unroll
    for (int f = 0; f < 5; ++f) v[f] += part[((long long)s * 5 + f) * G + p];
  if (accumulate) {
    rho[p] += v[0]; tau[p] += v[1];
    J[p] += v[2]; J[G + p] += v[3]; J[2 * G + p] += v[4];
  } else {
    rho[p] = v[0]; tau[p] = v[1];
    J[p] = v[2]; J[G + p] = v[3]; J[2 * G + p] = v[4];
  }
}

sky_status field_divergence(Ctx* c, const double* J, double* divJ);  // fields.cu

template <typename T>
static sky_status densities_t(Ctx* c, const cx<T>* psi, int I, double* rho, double* tau,
                              double* J, double* divJ) {
  const long long G = c->G, V = 2 * G;
  cx<T>* scr = static_cast<cx<T>*>(c->d_gscr);
  const long long cstride = (long long)c->chunk * V;
  cx<T>* g[3] = {scr, scr + cstride, scr + 2 * cstride};
  double* Jout = J ? J : c->d_ftmp + 13 * G;   // [3][G] temporaries when J not wanted
  if (I == 0) {
    cudaMemsetAsync(rho, 0, G * sizeof(double), c->stream);
    cudaMemsetAsync(tau, 0, G * sizeof(double), c->stream);
    cudaMemsetAsync(Jout, 0, 3 * G * sizeof(double), c->stream);
  }
  for (int s0 = 0; s0 < I; s0 += c->chunk) {
    const int ns = (I - s0) < c->chunk ? (I - s0) : c->chunk;
    const cx<T>* ps = psi + (long long)s0 * V;
    const int per = (ns + kDensSplits - 1) / kDensSplits;
    const int nsplit = (ns + per - 1) / per;
    dim3 grid(div_up(G, 128), nsplit);
    bool pairs = false;
    if constexpr (std::is_same<T, double>::value) pairs = operator_route(c);
    cudaError_t e = cudaSuccess;
    if (pairs) {
      for (int ax = 0; ax < 3 && e == cudaSuccess; ++ax)
        e = deriv_tc_pair(c, ax, (const double2*)ps, g[ax], 2LL * ns);
      if (e != cudaSuccess) return cuda_check(c, e, "densities gradient");
      k_dens_accum_pair<<<grid, 128, 0, c->stream>>>((const double2*)ps, (const float4*)g[0],
                                                     (const float4*)g[1], (const float4*)g[2], (int)G,
                                                     ns, per, c->d_dpart);
    } else {
      e = gradient_passes<T>(c, ps, g, 2LL * ns);
      if (e != cudaSuccess) return cuda_check(c, e, "densities gradient");
      k_dens_accum<T><<<grid, 128, 0, c->stream>>>(ps, g[0], g[1], g[2], (int)G, ns, per, c->d_dpart);
    }
    note_launch();
    k_dens_reduce<<<div_up(G, 256), 256, 0, c->stream>>>(c->d_dpart, nsplit, (int)G, s0 > 0, rho,
                                                         tau, Jout); note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_check(c, e, "densities accumulate");
  }
  if (divJ) return field_divergence(c, Jout, divJ);
  return SKY_OK;
}

sky_status densities_impl(Ctx* c, const void* psi, int I, double* rho, double* tau, double* J,
                          double* divJ) {
  if (c->prec == SKY_F64)
    return densities_t<double>(c, (const double2*)psi, I, rho, tau, J, divJ);
  return densities_t<float>(c, (const float2*)psi, I, rho, tau, J, divJ);
}

}  // namespace sky
