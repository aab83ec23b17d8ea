// Mean fields, Coulomb potential, energy and the convergence measure
// (Eq. Skyrme, Sec. 2.2, Eq. convergence).  Fields are FP64 for every
// spinor precision; real-field derivatives are spectral with the plain
// wavenumbers, real part kept.
#include <cmath>

#include "sky_internal.cuh"

namespace sky {

// ------------------------------------------------------------ real-field operators
// A spectral derivative of a real field along one axis is a real circulant
// operator on its lines, Re IFFT[i k FFT[f]]_m = sum_q D1[(m - q) mod n] f_q,
// and so is the second derivative:
//   D1[r] = -(1/n) sum_a k_a sin(2 pi a r / n),  D2[r] = -(1/n) sum_a k_a^2 cos(2 pi a r / n).
// The fields are small (8 kB to 2 MB, all in L2) and FP64, and on this chip a
// dependent FP64 operation takes ~67 cycles, so an FFT with one thread per
// line (400 lines at 20^3) was bound by that latency: 22-27 us for each axis
// and derivative, 9 to 12 of them per call.  Here one thread per point sums
// its 3 n terms directly, every derivative of both species in one launch,
// with independent accumulators; the FP64 rate (2 per clock and SM) bounds it:
// 12 n multiply-adds per point.  20^3: the nine passes of a mean field 215 us,
// now 15; the three of a divergence 72 us, now 7.  Tables built once per
// context in long double.
// d_fop[axis]: [4][n] = D1, D2, cos(2 pi r / n), sin(2 pi r / n).
constexpr int kFieldThreads = 64;    // small blocks: an 8^3 .. 24^3 field covers more SMs
constexpr int kFieldMaxN = 64;

sky_status build_field_tables(Ctx* c) {
  const long double two_pi = 6.283185307179586476925286766559005768L;
  for (int j = 0; j < 3; ++j) {
    const int n = c->n[j];
    double t[4 * kFieldMaxN];
    long double cs[kFieldMaxN], sn[kFieldMaxN];
    for (int r = 0; r < n; ++r) {
      cs[r] = cosl(two_pi * r / (long double)n);
      sn[r] = sinl(two_pi * r / (long double)n);
    }
    for (int r = 0; r < n; ++r) {
      long double d1 = 0.0L, d2 = 0.0L;
      for (int a = 0; a < n; ++a) {
        const int m = a < (n + 1) / 2 ? a : a - n;
        const long double k = two_pi * m / (long double)c->L[j];
        d1 -= k * sn[(a * r) % n];
        d2 -= k * k * cs[(a * r) % n];
      }
      t[r] = (double)(d1 / n);
      t[n + r] = (double)(d2 / n);
      t[2 * n + r] = (double)cs[r];
      t[3 * n + r] = (double)sn[r];
    }
    const cudaError_t e = cudaMemcpy(c->d_fop[j], t, 4 * n * sizeof(double), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_check(c, e, "field tables");
  }
  return SKY_OK;
}

struct FieldGeom {
  int n[3];
  int G;
  const double* op[3];
};
static FieldGeom field_geom(const Ctx* c) {
  FieldGeom g;
  for (int j = 0; j < 3; ++j) {
    g.n[j] = c->n[j];
    g.op[j] = c->d_fop[j];
  }
  g.G = c->G;
  return g;
}

// The point's position m along axis j, the line's first point and its stride.
__device__ __forceinline__ void field_line(const FieldGeom& g, int p, int j, int& m, int& base, int& stride) {
  const int nx = g.n[0], ny = g.n[1];
  const int x = p % nx, t = p / nx, y = t % ny, z = t / ny;
  stride = j == 0 ? 1 : j == 1 ? nx : nx * ny;
  m = j == 0 ? x : j == 1 ? y : z;
  base = p - m * stride;
}

// rho_T, Delta rho_T and (GRAD) d_j rho_T of both isospins T (the layout of
// d_ftmp below).  The sums run over the two species (even and odd q apart:
// eight independent chains with GRAD, four without) and combine at the end.
template <bool GRAD>
__global__ void __launch_bounds__(kFieldThreads) k_field_derivs(const double* __restrict__ rho,
                                                                FieldGeom g, double* __restrict__ f) {
  __shared__ double tab[3][2][kFieldMaxN];
#pragma unroll
  for (int j = 0; j < 3; ++j)
    for (int i = threadIdx.x; i < 2 * g.n[j]; i += kFieldThreads)
      tab[j][i >= g.n[j]][i >= g.n[j] ? i - g.n[j] : i] = g.op[j][i];
  __syncthreads();
  const int p = blockIdx.x * kFieldThreads + threadIdx.x, G = g.G;
  if (p >= G) return;
  double ln[2] = {0.0, 0.0}, lp[2] = {0.0, 0.0};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    int m, base, stride;
    field_line(g, p, j, m, base, stride);
    const int n = g.n[j];
    double gn[2] = {0.0, 0.0}, gp[2] = {0.0, 0.0};
    int r = m;                              // (m - q) mod n
#pragma unroll 2
    for (int q = 0; q < n; q += 2) {        // n is even
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double a = rho[base + (q + h) * stride], b = rho[G + base + (q + h) * stride];
        const double d2 = tab[j][1][r];
        ln[h] = fma(d2, a, ln[h]);
        lp[h] = fma(d2, b, lp[h]);
        if constexpr (GRAD) {
          const double d1 = tab[j][0][r];
          gn[h] = fma(d1, a, gn[h]);
          gp[h] = fma(d1, b, gp[h]);
        }
        r = r == 0 ? n - 1 : r - 1;
      }
    }
    if constexpr (GRAD) {
      const double a = gn[0] + gn[1], b = gp[0] + gp[1];
      f[(4 + 2 * j) * (long long)G + p] = a + b;
      f[(5 + 2 * j) * (long long)G + p] = a - b;
    }
  }
  const double a = ln[0] + ln[1], b = lp[0] + lp[1];
  const double rn = rho[p], rp = rho[G + p];
  f[p] = rn + rp;
  f[G + p] = rn - rp;
  f[2LL * G + p] = a + b;
  f[3LL * G + p] = a - b;
}

// divJ = sum_j d_j J_j for one [3][G] vector field.
__global__ void __launch_bounds__(kFieldThreads) k_field_div(const double* __restrict__ J, FieldGeom g,
                                                             double* __restrict__ out) {
  __shared__ double tab[3][kFieldMaxN];
#pragma unroll
  for (int j = 0; j < 3; ++j)
    for (int i = threadIdx.x; i < g.n[j]; i += kFieldThreads) tab[j][i] = g.op[j][i];
  __syncthreads();
  const int p = blockIdx.x * kFieldThreads + threadIdx.x, G = g.G;
  if (p >= G) return;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    int m, base, stride;
    field_line(g, p, j, m, base, stride);
    const int n = g.n[j];
    const double* src = J + (long long)j * G;
    int r = m;
    for (int q = 0; q < n; q += 4) {        // n is a multiple of 4
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        acc[h] = fma(tab[j][r], src[base + (q + h) * stride], acc[h]);
        r = r == 0 ? n - 1 : r - 1;
      }
    }
  }
  out[p] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

sky_status field_divergence(Ctx* c, const double* J, double* divJ) {
  k_field_div<<<div_up(c->G, kFieldThreads), kFieldThreads, 0, c->stream>>>(J, field_geom(c), divJ);
  note_launch();
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess)
    return set_err(c, SKY_ECUDA, "divergence (%d x %d x %d): %s", c->n[0], c->n[1], c->n[2],
                   cudaGetErrorString(e));
  return SKY_OK;
}

// Coulomb potential by the half spectrum of the real proton density: the DFT
// along z for k_z = 0 .. n_z / 2 only (the rest are complex conjugates), then
// y, x, times 4 pi e^2 / (G |k|^2), and back; the inverse along z takes k_z = 0
// and n_z / 2 once and the others twice.  Direct sums with one thread per
// output, for the same reason as above.
// z forward (FWD: rho -> half spectrum) and inverse (half spectrum -> V).
template <bool FWD>
__global__ void __launch_bounds__(kFieldThreads) k_coul_z(const double* __restrict__ rho,
                                                          double2* __restrict__ a,
                                                          double* __restrict__ V, FieldGeom g) {
  __shared__ double tc[kFieldMaxN], ts[kFieldMaxN];
  const int n = g.n[2], np = g.n[0] * g.n[1];
  for (int i = threadIdx.x; i < n; i += kFieldThreads) {
    tc[i] = g.op[2][2 * n + i];
    ts[i] = g.op[2][3 * n + i];
  }
  __syncthreads();
  const int p = blockIdx.x * kFieldThreads + threadIdx.x;
  const int h = n / 2 + 1;
  if (p >= (FWD ? h : n) * np) return;
  const int k = p / np, xy = p - k * np;
  double s0[2] = {0.0, 0.0}, s1[2] = {0.0, 0.0};
  int r = 0;                                // k q mod n
  if constexpr (FWD) {
    for (int q = 0; q < n; q += 2) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const double v = rho[(q + u) * np + xy];
        s0[u] = fma(v, tc[r], s0[u]);
        s1[u] = fma(-v, ts[r], s1[u]);
        r += k;
        if (r >= n) r -= n;
      }
    }
    a[p] = make_double2(s0[0] + s0[1], s1[0] + s1[1]);
  } else {
    for (int q = 0; q < h; ++q) {
      const double2 v = a[q * np + xy];
      const double w = q == 0 || 2 * q == n ? 1.0 : 2.0;
      s0[q & 1] = fma(w * v.x, tc[r], s0[q & 1]);
      s1[q & 1] = fma(-w * v.y, ts[r], s1[q & 1]);
      r += k;
      if (r >= n) r -= n;
    }
    V[p] = (s0[0] + s0[1]) + (s1[0] + s1[1]);
  }
}
// DFT along x or y of the half spectrum, out of place; SCALE multiplies the
// output by Pc scale (Pc of the full grid: its first n_z / 2 + 1 planes).
template <bool INV, bool SCALE>
__global__ void __launch_bounds__(kFieldThreads) k_coul_xy(const double2* __restrict__ in,
                                                           double2* __restrict__ out, FieldGeom g,
                                                           int axis, const double* __restrict__ Pc,
                                                           double scale) {
  __shared__ double tc[kFieldMaxN], ts[kFieldMaxN];
  const int n = g.n[axis];
  for (int i = threadIdx.x; i < n; i += kFieldThreads) {
    tc[i] = g.op[axis][2 * n + i];
    ts[i] = INV ? g.op[axis][3 * n + i] : -g.op[axis][3 * n + i];
  }
  __syncthreads();
  const int p = blockIdx.x * kFieldThreads + threadIdx.x;
  if (p >= (g.n[2] / 2 + 1) * g.n[0] * g.n[1]) return;
  int k, base, stride;
  field_line(g, p, axis, k, base, stride);
  double rc = 0.0, rs = 0.0, ic = 0.0, is = 0.0;
  int r = 0;
#pragma unroll 4
  for (int q = 0; q < n; ++q) {
    const double2 v = in[base + q * stride];
    rc = fma(v.x, tc[r], rc);
    rs = fma(v.x, ts[r], rs);
    ic = fma(v.y, tc[r], ic);
    is = fma(v.y, ts[r], is);
    r += k;
    if (r >= n) r -= n;
  }
  double2 o = make_double2(rc - is, ic + rs);
  if constexpr (SCALE) {
    const double s = Pc[p] * scale;
    o = make_double2(o.x * s, o.y * s);
  }
  out[p] = o;
}

// Temporaries in d_ftmp ([16][G]): 0-1 rho_T, 2-3 Delta rho_T,
// 4-9 d_j rho_T at 4 + 2j + T, 10 V_C, 11-12 reduction partials,
// 13-15 spin-orbit density when the caller does not want it.
__global__ void k_coul_table(double* Pc, const double* kx, const double* ky, const double* kz,
                             int nx, int ny, int nz, double e2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nx * ny * nz) return;
  const int x = p % nx, y = (p / nx) % ny, z = p / (nx * ny);
  const double k2 = kx[x] * kx[x] + ky[y] * ky[y] + kz[z] * kz[z];
  Pc[p] = k2 > 0.0 ? 4.0 * 3.14159265358979323846 * e2 / k2 : 0.0;
}

sky_status build_coulomb_table(Ctx* c) {
  k_coul_table<<<div_up(c->G, 256), 256, 0, c->stream>>>(c->d_coul, c->d_kp[0], c->d_kp[1],
                                                         c->d_kp[2], c->n[0], c->n[1], c->n[2],
                                                         c->cp.e2); note_launch();
  return cuda_check(c, cudaGetLastError(), "coulomb table");
}

// Shared first part of mean fields and energy: rho_T, Delta rho_T, grad rho_T, V_C.
static sky_status field_prep(Ctx* c, const double* rho, bool need_grad) {
  const int G = c->G, T = kFieldThreads;
  double* f = c->d_ftmp;
  const FieldGeom g = field_geom(c);
  if (need_grad)
    k_field_derivs<true><<<div_up(G, T), T, 0, c->stream>>>(rho, g, f);
  else
    k_field_derivs<false><<<div_up(G, T), T, 0, c->stream>>>(rho, g, f);
  note_launch();
  if (c->cp.coulomb) {
    const int gh = (c->n[2] / 2 + 1) * c->n[0] * c->n[1];
    double2 *a = c->d_fcx, *b = c->d_fcx + gh;
    const unsigned nb = div_up(gh, T);
    k_coul_z<true><<<nb, T, 0, c->stream>>>(rho + G, a, nullptr, g);
    k_coul_xy<false, false><<<nb, T, 0, c->stream>>>(a, b, g, 1, nullptr, 0.0);
    k_coul_xy<false, true><<<nb, T, 0, c->stream>>>(b, a, g, 0, c->d_coul, 1.0 / (double)G);
    k_coul_xy<true, false><<<nb, T, 0, c->stream>>>(a, b, g, 0, nullptr, 0.0);
    k_coul_xy<true, false><<<nb, T, 0, c->stream>>>(b, a, g, 1, nullptr, 0.0);
    k_coul_z<false><<<div_up(G, T), T, 0, c->stream>>>(nullptr, a, f + 10LL * G, g);
    note_launch(6);
  }
  return cuda_check(c, cudaGetLastError(), "field derivatives");
}

__device__ __forceinline__ void rho0_powers(double r0, double alpha, double& r0a, double& r0am1) {
  if (r0 > 1e-30) {
    r0a = pow(r0, alpha);
    r0am1 = r0a / r0;
  } else {
    r0a = 0.0;
    r0am1 = 0.0;
  }
}

__global__ void k_mean_fields(Couplings cp, const double* tau, const double* divJ,
                              const double* f, int G, double* U, double* B, double* W) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const double r[2] = {f[p], f[G + p]};
  const double l[2] = {f[2 * G + p], f[3 * G + p]};
  const double t[2] = {tau[p] + tau[G + p], tau[p] - tau[G + p]};
  const double d[2] = {divJ[p] + divJ[G + p], divJ[p] - divJ[G + p]};
  double r0a, r0am1;
  rho0_powers(r[0], cp.alpha, r0a, r0am1);
  const double dd = cp.alpha * r0am1 * (cp.rhoa[0] * r[0] * r[0] + cp.rhoa[1] * r[1] * r[1]);
  double uT[2];
#pragma unroll
  for (int T = 0; T < 2; ++T)
    uT[T] = 2.0 * (cp.rho[T] + cp.rhoa[T] * r0a) * r[T] + cp.tau[T] * t[T] +
            2.0 * cp.drho[T] * l[T] + cp.nJ[T] * d[T];
  const double vc = cp.coulomb ? f[10 * G + p] : 0.0;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double s1 = q == 0 ? 1.0 : -1.0;
    U[q * G + p] = uT[0] + s1 * uT[1] + dd + (q == 1 ? vc : 0.0);
    B[q * G + p] = cp.hb2m[q] + cp.tau[0] * r[0] + s1 * cp.tau[1] * r[1];
#pragma unroll
    for (int j = 0; j < 3; ++j)
      W[(q * 3 + j) * G + p] = -(cp.nJ[0] * f[(4 + 2 * j) * G + p] +
                                 s1 * cp.nJ[1] * f[(5 + 2 * j) * G + p]);
  }
}

sky_status mean_fields_impl(Ctx* c, const double* rho, const double* tau, const double* divJ,
                            double* U, double* B, double* W) {
  sky_status s = field_prep(c, rho, true);
  if (s != SKY_OK) return s;
  k_mean_fields<<<div_up(c->G, 256), 256, 0, c->stream>>>(c->cp, tau, divJ, c->d_ftmp, c->G, U,
                                                          B, W); note_launch();
  return cuda_check(c, cudaGetLastError(), "mean fields");
}

// ------------------------------------------------------------ energy
constexpr int kEnBlock = 256;
constexpr int kEnParts = 7;   // kin, rho, tau, drho, nJ, coul, A

__global__ void __launch_bounds__(kEnBlock) k_energy_parts(Couplings cp, const double* rho,
                                                           const double* tau,
                                                           const double* divJ,
                                                           const double* f, int G,
                                                           double* part) {
  double acc[kEnParts] = {0, 0, 0, 0, 0, 0, 0};
  for (int p = blockIdx.x * kEnBlock + threadIdx.x; p < G; p += gridDim.x * kEnBlock) {
    const double r[2] = {f[p], f[G + p]};
    const double l[2] = {f[2 * G + p], f[3 * G + p]};
    const double t[2] = {tau[p] + tau[G + p], tau[p] - tau[G + p]};
    const double d[2] = {divJ[p] + divJ[G + p], divJ[p] - divJ[G + p]};
    double r0a, r0am1;
    rho0_powers(r[0], cp.alpha, r0a, r0am1);
    acc[0] += cp.hb2m[0] * tau[p] + cp.hb2m[1] * tau[G + p];
#pragma unroll
    for (int T = 0; T < 2; ++T) {
      acc[1] += (cp.rho[T] + cp.rhoa[T] * r0a) * r[T] * r[T];
      acc[2] += cp.tau[T] * r[T] * t[T];
      acc[3] += cp.drho[T] * r[T] * l[T];
      acc[4] += cp.nJ[T] * r[T] * d[T];
    }
    if (cp.coulomb) acc[5] += 0.5 * rho[G + p] * f[10 * G + p];
    acc[6] += rho[p] + rho[G + p];
  }
  __shared__ double sh[kEnBlock / 32][kEnParts];
#pragma unroll
  for (int k = 0; k < kEnParts; ++k) {
    double v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kEnParts) {
    double v = 0.0;
    for (int w = 0; w < kEnBlock / 32; ++w) v += sh[w][threadIdx.x];
    part[blockIdx.x * kEnParts + threadIdx.x] = v;
  }
}

// One warp per part (a single thread walking the 64 x 7 partial sums: 22 us
// of dependent FP64 additions).
__global__ void __launch_bounds__(32 * kEnParts) k_energy_final(const double* part, int nblk, double dV,
                                                                double* out, int* status) {
  __shared__ double s[kEnParts];
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double v = 0.0;
  for (int b = lane; b < nblk; b += 32) v += part[b * kEnParts + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) s[k] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  double tot = 0.0;
  for (int q = 0; q < 6; ++q) {
    out[1 + q] = dV * s[q];
    tot += dV * s[q];
  }
  out[0] = tot;
  out[7] = dV * s[6];
  if (!isfinite(tot)) flag_status(status, SKY_ENAN);
}

sky_status energy_impl(Ctx* c, const double* rho, const double* tau, const double* divJ,
                       double* out) {
  sky_status s = field_prep(c, rho, false);
  if (s != SKY_OK) return s;
  const int nblk = 64;
  double* part = c->d_ftmp + 11 * (long long)c->G;
  k_energy_parts<<<nblk, kEnBlock, 0, c->stream>>>(c->cp, rho, tau, divJ, c->d_ftmp, c->G, part); note_launch();
  k_energy_final<<<1, 32 * kEnParts, 0, c->stream>>>(part, nblk, c->dV, out, c->d_status); note_launch();
  return cuda_check(c, cudaGetLastError(), "energy");
}

// ------------------------------------------------------------ convergence
__global__ void k_sp_spread(const double* eps, const double* hn2, int A, double* out) {
  __shared__ double sa[32], sb[32];
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < A; i += blockDim.x) {
    a += hn2[i] - eps[i] * eps[i];
    b += eps[i];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) { sa[threadIdx.x >> 5] = a; sb[threadIdx.x >> 5] = b; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double x = 0.0, y = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { x += sa[w]; y += sb[w]; }
    out[0] = A > 0 ? sqrt(fmax(x, 0.0) / A) : 0.0;
    out[1] = y;
  }
}

sky_status sp_spread_impl(Ctx* c, const double* eps, const double* hn2, int A, double* out) {
  k_sp_spread<<<1, 1024, 0, c->stream>>>(eps, hn2, A, out); note_launch();
  return cuda_check(c, cudaGetLastError(), "sp spread");
}

}  // namespace sky
