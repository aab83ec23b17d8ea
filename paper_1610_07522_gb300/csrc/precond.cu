// Learned damping weight of the damped gradient step (an extension of
// Sec. 2.2, Eq. dampstep): a periodic 3x3x3 convolutional network
//   x = (U/50, B/hb2m - 1, |W|/5) -> tanh conv 16 -> tanh conv 16 -> conv 1
//   w = WMAX sigmoid(z)
// with its training kernels: the per-voxel statistics of the one-step loss,
// the backward pass through the three layers, and Adam.
//
// Layout: every activation is channel-planar [C][nz][ny][nx] float, x
// fastest, so neighbouring threads read neighbouring voxels.  The layers are
// small (27 x 16 x 16 multiply-adds per voxel, 8^3 .. 64^3 voxels): what bounds
// them is loads per multiply-add and warps in flight.  A thread computes eight
// output channels of one voxel from weights in shared memory, eight per two
// 16-byte broadcasts; a weight-gradient thread keeps four output channels x 27
// taps, 108 multiply-adds per 31 loads.  Weight gradients are summed over a
// voxel range by one block, then over the ranges in a fixed order, so every
// result is deterministic.
#include "sky_internal.cuh"

namespace sky {

constexpr int kH = SKY_NET_HIDDEN;
constexpr int kConvThreads = 128;
constexpr int kWgThreads = 128;
constexpr int kTaps = 27;
// parameter offsets (the order of the flat vector)
constexpr int oW1 = 0, ob1 = oW1 + kH * 3 * kTaps, oW2 = ob1 + kH, ob2 = oW2 + kH * kH * kTaps,
              oW3 = ob2 + kH, ob3 = oW3 + kH * kTaps, kNParam = ob3 + 1;
static_assert(kNParam == SKY_NET_NPARAM, "parameter count");
// workspace offsets in units of G floats
constexpr int wsX = 0, wsH1 = 3, wsH2 = wsH1 + kH, wsW = wsH2 + kH, wsDZ = wsW + 1,
              wsD2 = wsDZ + 1, wsD1 = wsD2 + kH, wsEnd = wsD1 + kH;
static_assert(wsEnd <= SKY_NET_WS_PER_POINT, "workspace per grid point");

// Partial sums of a backward pass: 28 per (output, input) pair and voxel range
// of each layer (at most kSplits1 .. kSplits3 ranges), then the loss blocks.
constexpr int kSplits1 = 24, kSplits2 = 8, kSplits3 = 64;
constexpr size_t kPart2 = 0, kPart3 = kPart2 + (size_t)kH * kH * kSplits2 * 28,
                 kPart1 = kPart3 + (size_t)kH * kSplits3 * 28,
                 kPartLoss = kPart1 + (size_t)kH * 3 * kSplits1 * 28;

size_t net_partial_elems(int G) { return kPartLoss + (size_t)div_up(G, kConvThreads) + 8; }

// Offsets of the 27 periodic neighbours of voxel p, tap 9 (dz+1) + 3 (dy+1) + (dx+1).
__device__ __forceinline__ void neighbours(int p, int nx, int ny, int nz, int (&q)[kTaps]) {
  const int x = p % nx, y = (p / nx) % ny, z = p / (nx * ny), s = nx * ny;
  const int xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
  const int ys[3] = {(y == 0 ? ny - 1 : y - 1) * nx, y * nx, (y == ny - 1 ? 0 : y + 1) * nx};
  const int zs[3] = {(z == 0 ? nz - 1 : z - 1) * s, z * s, (z == nz - 1 ? 0 : z + 1) * s};
#pragma unroll
  for (int t = 0; t < kTaps; ++t) q[t] = zs[t / 9] + ys[(t / 3) % 3] + xs[t % 3];
}

__global__ void k_net_features(const double* __restrict__ U, const double* __restrict__ B,
                               const double* __restrict__ W, int G, double hb2m, float* __restrict__ x) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= G) return;
  const double wx = W[p], wy = W[G + p], wz = W[2 * G + p];
  x[p] = (float)(U[p] / SKY_NET_USCALE);
  x[G + p] = (float)(B[p] / hb2m - 1.0);
  x[2 * G + p] = (float)(sqrt(wx * wx + wy * wy + wz * wz) / SKY_NET_WSCALE);
}

// One layer, forward or backward:
//   FWD: out_o(r) = b_o + sum_{i,t} W[o][i][t] in_i(r + d_t), then
//        EPI 0: tanh; EPI 1: the weight, out = WMAX sigmoid (the network's own
//        output) and wout = 1 + scale (out - 1) (the weight the step uses);
//   !FWD (EPI 2): out_o(r) = (1 - h_o(r)^2) sum_{i,t} W[i][o][t] in_i(r - d_t),
//        the gradient of the layer's input (in = the gradient of its output, h
//        its input activation).
// A block serves kConvVox voxels; its warps split the NO output channels into
// groups of OG and the NI input channels into IS parts (added up through
// shared memory): the single-output layer is split by inputs.  The weights lie
// in shared memory as rows (input, tap) of NO values, padded to stay
// 16-byte aligned and nearly free of bank conflicts while they are stored.
// 24^3: 16 -> 16 forward 33 us with one thread per voxel and scalar weight
// loads, 18 us; its weight gradient 55 -> 24 us.
constexpr int kConvVox = 64;
template <int NI, int NO, int OG, int IS, bool FWD, int EPI>
__global__ void __launch_bounds__(kConvVox * (NO / OG) * IS)
    k_conv(const float* __restrict__ in, const float* __restrict__ Wt, const float* __restrict__ bias,
           const float* __restrict__ hin, float* __restrict__ out, int nx, int ny, int nz,
           float* __restrict__ wout, float scale) {
  constexpr int S = NO >= 4 ? NO + 4 : 1, T = kConvVox * (NO / OG) * IS, NIS = NI / IS;
  static_assert(NI % IS == 0 && NO % OG == 0, "channel groups");
  __shared__ __align__(16) float sw[NI * kTaps * S];
  __shared__ float sacc[IS > 1 ? (IS - 1) * OG * kConvVox : 1];
  const int tid = threadIdx.x, v = tid % kConvVox, grp = tid / kConvVox;
  const int og = (grp % (NO / OG)) * OG, is = grp / (NO / OG);
  for (int e = tid; e < NI * NO * kTaps; e += T) {
    const int first = e / kTaps, t = e - first * kTaps;   // FWD: first = o NI + i; else i NO + o
    const int o = FWD ? first / NI : first % NO, i = FWD ? first % NI : first / NO;
    sw[(i * kTaps + (FWD ? t : kTaps - 1 - t)) * S + o] = Wt[e];   // r - d_t is tap 26 - t
  }
  __syncthreads();
  const int G = nx * ny * nz;
  const int p = blockIdx.x * kConvVox + v;
  int q[kTaps];
  neighbours(p < G ? p : 0, nx, ny, nz, q);
  float acc[OG];
#pragma unroll
  for (int o = 0; o < OG; ++o) acc[o] = FWD && is == 0 ? bias[og + o] : 0.0f;
#pragma unroll 1
  for (int i = is * NIS; i < (is + 1) * NIS; ++i) {
    const float* src = in + (size_t)i * G;
    float x[kTaps];
#pragma unroll
    for (int t = 0; t < kTaps; ++t) x[t] = __ldg(src + q[t]);
    const float* w = sw + i * kTaps * S + og;
#pragma unroll
    for (int t = 0; t < kTaps; ++t) {
      if constexpr (OG % 4 == 0) {
#pragma unroll
        for (int o = 0; o < OG; o += 4) {
          const float4 k = *reinterpret_cast<const float4*>(w + t * S + o);
          acc[o] = fmaf(k.x, x[t], acc[o]);
          acc[o + 1] = fmaf(k.y, x[t], acc[o + 1]);
          acc[o + 2] = fmaf(k.z, x[t], acc[o + 2]);
          acc[o + 3] = fmaf(k.w, x[t], acc[o + 3]);
        }
      } else {
#pragma unroll
        for (int o = 0; o < OG; ++o) acc[o] = fmaf(w[t * S + o], x[t], acc[o]);
      }
    }
  }
  if constexpr (IS > 1) {
    static_assert(NO == OG, "input parts of one output group");
#pragma unroll
    for (int o = 0; o < OG; ++o)
      if (is > 0) sacc[((is - 1) * OG + o) * kConvVox + v] = acc[o];
    __syncthreads();
    if (is > 0) return;
#pragma unroll
    for (int k = 0; k < IS - 1; ++k)
#pragma unroll
      for (int o = 0; o < OG; ++o) acc[o] += sacc[(k * OG + o) * kConvVox + v];
  }
  if (p >= G) return;
#pragma unroll
  for (int o = 0; o < OG; ++o) {
    const size_t at = (size_t)(og + o) * G + p;
    if constexpr (EPI == 0) {
      out[at] = tanhf(acc[o]);
    } else if constexpr (EPI == 1) {
      const float w = (float)SKY_NET_WMAX / (1.0f + expf(-acc[o]));
      out[at] = w;
      wout[p] = 1.0f + scale * (w - 1.0f);
    } else {
      const float h = hin[at];
      out[at] = acc[o] * (1.0f - h * h);
    }
  }
}

// Sums of 32 values over the warp at once: a[k] in, lane k gets the total of
// value k; 31 shuffles instead of 160.
__device__ __forceinline__ float warp_sums32(float (&a)[32], int lane) {
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const float keep = up ? a[k + h] : a[k], send = up ? a[k] : a[k + h];
      a[k] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  return a[0];
}

// part[((o CIN + i) nsplit + split) 28 + t] = sum over the split's voxels of
// dout_o(r) in_i(r + d_t) (t < 27) and dout_o(r) (t = 27), for OG outputs o and
// one input i per block.
template <int CIN, int OG>
__global__ void __launch_bounds__(kWgThreads) k_conv_wgrad(const float* __restrict__ dout,
                                                           const float* __restrict__ in, int nx,
                                                           int ny, int nz, int chunk,
                                                           double* __restrict__ part) {
  const int o0 = (blockIdx.x / CIN) * OG, i = blockIdx.x % CIN;
  const int G = nx * ny * nz;
  const int p0 = blockIdx.y * chunk, p1 = min(G, p0 + chunk);
  float acc[OG][28];
#pragma unroll
  for (int o = 0; o < OG; ++o)
#pragma unroll
    for (int t = 0; t < 28; ++t) acc[o][t] = 0.0f;
  const float* xi = in + (size_t)i * G;
  for (int p = p0 + threadIdx.x; p < p1; p += kWgThreads) {
    float d[OG];
#pragma unroll
    for (int o = 0; o < OG; ++o) d[o] = __ldg(dout + (size_t)(o0 + o) * G + p);
    int q[kTaps];
    neighbours(p, nx, ny, nz, q);
#pragma unroll
    for (int t = 0; t < kTaps; ++t) {
      const float x = __ldg(xi + q[t]);
#pragma unroll
      for (int o = 0; o < OG; ++o) acc[o][t] = fmaf(d[o], x, acc[o][t]);
    }
#pragma unroll
    for (int o = 0; o < OG; ++o) acc[o][27] += d[o];
  }
  __shared__ float sred[kWgThreads / 32][OG][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 0; o < OG; ++o) {
    float a[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) a[t] = t < 28 ? acc[o][t] : 0.0f;
    sred[warp][o][lane] = warp_sums32(a, lane);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < OG * 32; e += kWgThreads) {
    const int o = e >> 5, t = e & 31;
    if (t >= 28) continue;
    double s = 0.0;
    for (int w = 0; w < kWgThreads / 32; ++w) s += (double)sred[w][o][t];
    part[((size_t)((o0 + o) * CIN + i) * gridDim.y + blockIdx.y) * 28 + t] = s;
  }
}

// All layers' gradients from the partial sums, and the loss:
// grad[oW + pair * 27 + t] += sum_split part; grad[ob + o] += bias part of pair
// (o, 0).  Blocks: the pairs of layer 2, 3, 1, then one for the loss.
struct WgradSums {
  int pairs[3], cin[3], nsplit[3], ow[3], ob[3];
  size_t part[3];
  int nblk;
};
__global__ void __launch_bounds__(128) k_wgrad_reduce(const double* __restrict__ part, WgradSums a,
                                                      const double* __restrict__ norm,
                                                      double* __restrict__ grad,
                                                      double* __restrict__ loss) {
  __shared__ double red[4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int pair = blockIdx.x, l = 0;
  while (l < 3 && pair >= a.pairs[l]) pair -= a.pairs[l++];
  double s = 0.0;
  if (l < 3) {
    const double* src = part + a.part[l] + (size_t)pair * a.nsplit[l] * 28;
    if (lane < 28)
      for (int k = warp; k < a.nsplit[l]; k += 4) s += src[k * 28 + lane];
  } else {
    for (int k = threadIdx.x; k < a.nblk; k += 128) s += part[kPartLoss + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp != 0) return;
  s = (red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane]);
  if (l == 3) {
    if (lane == 0) loss[0] += s / norm[0];
  } else if (lane < kTaps) {
    grad[a.ow[l] + (size_t)pair * kTaps + lane] += s;
  } else if (lane == kTaps && pair % a.cin[l] == 0) {
    grad[a.ob[l] + pair / a.cin[l]] += s;
  }
}

template <int NT>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double red[NT / 32];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < NT / 32; ++k) s += red[k];
  return s;
}

// dz(r) = d L / d z(r) with L = sum (a w^2 - 2 b w + c) / norm and
// w = WMAX sigmoid(z); block partials of the unnormalised loss.
__global__ void __launch_bounds__(kConvThreads) k_net_head(const float* __restrict__ w,
                                                           const double* __restrict__ abc,
                                                           const double* __restrict__ norm, int G,
                                                           float* __restrict__ dz,
                                                           double* __restrict__ lpart) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  double l = 0.0;
  if (p < G) {
    const double a = abc[p], b = abc[G + p], c = abc[2 * G + p], ww = w[p];
    const double dw = 2.0 * (a * ww - b) / norm[0];
    dz[p] = (float)(dw * ww * (1.0 - ww / SKY_NET_WMAX));
    l = a * ww * ww - 2.0 * b * ww + c;
  }
  l = block_sum<kConvThreads>(l);
  if (threadIdx.x == 0) lpart[blockIdx.x] = l;
}

__global__ void k_adam(float* __restrict__ theta, double* __restrict__ grad,
                       double* __restrict__ m, double* __restrict__ v, int n, double lr,
                       double b1, double b2, double eps, double c1, double c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double g = grad[i];
  const double mi = b1 * m[i] + (1.0 - b1) * g;
  const double vi = b2 * v[i] + (1.0 - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  theta[i] = (float)((double)theta[i] - lr * (mi / c1) / (sqrt(vi / c2) + eps));
  grad[i] = 0.0;
}

// a = sum |psi - phi|^2, b = sum Re(conj(psi - phi)(psi - ppsi)),
// c = sum |psi - ppsi|^2 over states and spin, per voxel; block partials of c.
template <typename T>
__global__ void __launch_bounds__(kConvThreads) k_precond_stats(const cx<T>* __restrict__ psi,
                                                                const cx<T>* __restrict__ phi,
                                                                const cx<T>* __restrict__ pp,
                                                                int I, int G,
                                                                double* __restrict__ abc,
                                                                double* __restrict__ cpart) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  double a = 0.0, b = 0.0, c = 0.0;
  if (p < G) {
    for (long long k = 0; k < 2LL * I; ++k) {
      const long long o = k * G + p;
      const double2 s = to_d2(psi[o]), f = to_d2(phi[o]), r = to_d2(pp[o]);
      const double gx = s.x - f.x, gy = s.y - f.y, dx = s.x - r.x, dy = s.y - r.y;
      a += gx * gx + gy * gy;
      b += gx * dx + gy * dy;
      c += dx * dx + dy * dy;
    }
    abc[p] = a;
    abc[G + p] = b;
    abc[2 * G + p] = c;
  }
  c = block_sum<kConvThreads>(c);
  if (threadIdx.x == 0) cpart[blockIdx.x] = c;
}

__global__ void k_norm_total(const double* __restrict__ cpart, int nblk, double* __restrict__ norm) {
  double s = 0.0;
  for (int k = threadIdx.x; k < nblk; k += blockDim.x) s += cpart[k];
  s = block_sum<256>(s);
  if (threadIdx.x == 0) norm[0] = s;
}

// ------------------------------------------------------------ host side
sky_status net_forward_impl(Ctx* c, int q, const float* theta, const double* U, const double* B,
                            const double* W, double scale, float* ws, float* w) {
  const int G = c->G, nx = c->n[0], ny = c->n[1], nz = c->n[2];
  const unsigned nb = div_up(G, kConvThreads);
  float* x = ws + (size_t)wsX * G;
  float* h1 = ws + (size_t)wsH1 * G;
  float* h2 = ws + (size_t)wsH2 * G;
  k_net_features<<<nb, kConvThreads, 0, c->stream>>>(U, B, W, G, c->cp.hb2m[q], x);
  const unsigned cb = div_up(G, kConvVox);
  k_conv<3, kH, 8, 1, true, 0><<<cb, 2 * kConvVox, 0, c->stream>>>(x, theta + oW1, theta + ob1, nullptr, h1,
                                                                   nx, ny, nz, nullptr, 0.0f);
  k_conv<kH, kH, 8, 1, true, 0><<<cb, 2 * kConvVox, 0, c->stream>>>(h1, theta + oW2, theta + ob2, nullptr,
                                                                    h2, nx, ny, nz, nullptr, 0.0f);
  k_conv<kH, 1, 1, 4, true, 1><<<cb, 4 * kConvVox, 0, c->stream>>>(
      h2, theta + oW3, theta + ob3, nullptr, ws + (size_t)wsW * G, nx, ny, nz, w, (float)scale);
  note_launch(4);
  return cuda_check(c, cudaGetLastError(), "net forward");
}

// Weight-gradient partials of one layer; *ns returns the voxel ranges used:
// enough blocks for about three per SM, at least two voxels per thread.
template <int CIN, int OG>
static void wgrad(Ctx* c, int cout, const float* dout, const float* in, int max_splits, size_t part,
                  int* ns_out) {
  const int G = c->G, groups = cout / OG * CIN;
  int ns = (int)div_up(3LL * c->num_sms, groups);
  const int most = (int)div_up(G, 2 * kWgThreads);
  if (ns > max_splits) ns = max_splits;
  if (ns > most) ns = most;
  const int chunk = (int)div_up(G, ns);
  ns = (int)div_up(G, chunk);
  k_conv_wgrad<CIN, OG><<<dim3(groups, ns), kWgThreads, 0, c->stream>>>(
      dout, in, c->n[0], c->n[1], c->n[2], chunk, c->d_netpart + part);
  note_launch();
  *ns_out = ns;
}

sky_status net_backward_impl(Ctx* c, const float* theta, float* ws, const double* abc,
                             const double* norm, double* grad, double* loss) {
  const int G = c->G, nx = c->n[0], ny = c->n[1], nz = c->n[2];
  const unsigned nb = div_up(G, kConvThreads);
  float* x = ws + (size_t)wsX * G;
  float* h1 = ws + (size_t)wsH1 * G;
  float* h2 = ws + (size_t)wsH2 * G;
  const float* w = ws + (size_t)wsW * G;
  float* dz = ws + (size_t)wsDZ * G;
  float* d2 = ws + (size_t)wsD2 * G;
  float* d1 = ws + (size_t)wsD1 * G;
  WgradSums r{{kH * kH, kH, 3 * kH}, {kH, kH, 3}, {0, 0, 0}, {oW2, oW3, oW1}, {ob2, ob3, ob1},
              {kPart2, kPart3, kPart1}, (int)nb};
  const unsigned cb = div_up(G, kConvVox);
  k_net_head<<<nb, kConvThreads, 0, c->stream>>>(w, abc, norm, G, dz, c->d_netpart + kPartLoss);
  wgrad<kH, 1>(c, 1, dz, h2, kSplits3, kPart3, &r.nsplit[1]);
  k_conv<1, kH, 8, 1, false, 2><<<cb, 2 * kConvVox, 0, c->stream>>>(dz, theta + oW3, nullptr, h2, d2, nx, ny,
                                                                    nz, nullptr, 0.0f);
  wgrad<kH, 4>(c, kH, d2, h1, kSplits2, kPart2, &r.nsplit[0]);
  k_conv<kH, kH, 8, 1, false, 2><<<cb, 2 * kConvVox, 0, c->stream>>>(d2, theta + oW2, nullptr, h1, d1, nx,
                                                                     ny, nz, nullptr, 0.0f);
  wgrad<3, 4>(c, kH, d1, x, kSplits1, kPart1, &r.nsplit[2]);
  k_wgrad_reduce<<<kH * kH + kH + 3 * kH + 1, 128, 0, c->stream>>>(c->d_netpart, r, norm, grad, loss);
  note_launch(4);
  const cudaError_t e = cudaGetLastError();
  return cuda_check(c, e, "net backward");
}

sky_status net_adam_impl(Ctx* c, float* theta, double* grad, double* m, double* v, int step,
                         double lr, double beta1, double beta2, double eps) {
  const double c1 = 1.0 - pow(beta1, (double)step), c2 = 1.0 - pow(beta2, (double)step);
  k_adam<<<div_up(kNParam, 256), 256, 0, c->stream>>>(theta, grad, m, v, kNParam, lr, beta1, beta2,
                                                      eps, c1, c2);
  note_launch();
  return cuda_check(c, cudaGetLastError(), "net adam");
}

sky_status precond_stats_impl(Ctx* c, const void* psi, const void* phi, const void* ppsi, int I,
                              double* abc, double* norm) {
  const int G = c->G;
  const unsigned nb = div_up(G, kConvThreads);
  if (c->prec == SKY_F64)
    k_precond_stats<double><<<nb, kConvThreads, 0, c->stream>>>(
        (const double2*)psi, (const double2*)phi, (const double2*)ppsi, I, G, abc, c->d_netpart);
  else
    k_precond_stats<float><<<nb, kConvThreads, 0, c->stream>>>(
        (const float2*)psi, (const float2*)phi, (const float2*)ppsi, I, G, abc, c->d_netpart);
  k_norm_total<<<1, 256, 0, c->stream>>>(c->d_netpart, (int)nb, norm);
  note_launch(2);
  return cuda_check(c, cudaGetLastError(), "precond stats");
}

}  // namespace sky
