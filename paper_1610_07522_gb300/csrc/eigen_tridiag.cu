// FP64 Hermitian eigensolver by reduction to real tridiagonal form, for the
// diagonalisations of steps 3b-3c (Sec. 3.3.2) at the sizes where the cyclic
// Jacobi method's O(I^3) work per sweep dominates an iteration.
//
// The paper hands these to ScaLAPACK's Hermitian tridiagonal reduction with
// the MRRR tridiagonal solver.  Here the same three stages are GPU kernels:
//
//  1. k_hh_tridiag: A = Q T Q^H with Q = H_0 H_1 ... H_{n-2}, each reflector
//     H_t = I - tau_t v_t v_t^H chosen so that H_t^H maps column t below the
//     diagonal onto beta_t e_1 with beta_t real (T is real symmetric).  One
//     cooperative kernel: the blocks keep the columns of the (full, Hermitian)
//     trailing matrix cyclically in shared memory.  The update by H_t is
//     A <- A - u w^H - w u^H with u the reflector's unscaled vector, p = A u and
//     w = tau p - (|tau|^2 u^H p / 2) u (tau for u).  Each owner forms p_j =
//     col_j^H u_t for its own columns, fused with that column's update by the
//     previous reflector, and publishes p, the next column and its block's
//     partial of u^H p; once these are there every block recomputes the next
//     column itself (the same arithmetic in every block), so each step costs one
//     exchange.  The heads of up to four problems run side by side on separate
//     warp groups.
//  2. k_tri_bisect: eigenvalues of T by multisection on the count of
//     negative LDL^T pivots of T - x I, one warp (kBisLanes points) per
//     eigenvalue and round: FP32 counts first, then double-float ones (the
//     chip's FP64 latency makes an FP64 count ~10 times slower).
//  3. k_tri_vectors: eigenvectors of T by inverse iteration (Gaussian
//     elimination with partial pivoting of T - lambda I, factored once, then
//     kInvIters solves from a counter-based random start); eigenvalues closer
//     than kTightRel ||T|| are handled by one thread in order, each new vector
//     orthogonalised against the cluster's earlier ones after every solve (as
//     LAPACK's dstein does).  k_tri_window then applies first-order Loewdin
//     steps Y <- Y (3 I - Y^T Y) / 2, with Y^T Y formed only between
//     eigenvalues within kWinRel ||T|| of each other (the inverse-iteration
//     vectors' mutual overlaps fall off like eps ||T|| / gap).  Z = Q Y is
//     formed from Q's compact WY form by tensor-core products (wy_back), or, for
//     small or device-gated batches, by k_hh_back, one warp per column, the
//     reflectors applied in reverse order.
//
// Eigenvalues come out ascending, eigenvectors as the columns of Z.
#include <algorithm>
#include <cmath>

#include "dd.cuh"
#include "eig_common.cuh"

namespace sky {

constexpr int kTriThreads = 512;
constexpr int kTriWarps = kTriThreads / 32;
constexpr int kBisLanes = 32;           // bisection points per eigenvalue and round: one warp,
                                        // so every eigenvalue has its own warp (one wave)
constexpr int kBisMaxRounds = 96;       // ample for 2 eps ||T|| at 33x per round
constexpr int kInvIters = 3;            // inverse-iteration solves per vector
constexpr int kVecThreads = 8;          // eigenvectors per block of k_tri_vectors
constexpr double kTightRel = 1e-9;      // cluster threshold relative to ||T||
constexpr double kWinRel = 0.05;        // Loewdin window relative to ||T||
constexpr int kWinMax = 128;            // neighbours per side in the window at most
constexpr int kWinThreads = 128;
constexpr int kWinChunks = (2 * kWinMax + 1 + 31) / 32;
constexpr int kBackWarps = 16;
constexpr size_t kTriSmemMax = 200 * 1024;   // dynamic shared memory of k_hh_tridiag / k_hh_back
constexpr double kEps = 2.220446049250313e-16;
constexpr int kTriBufs = 8;             // buffers of the published vectors (see unset)
constexpr int kTeamBarStride = 32;     // unsigned between team barrier counters (128 bytes)

struct TriBatch {
  const double2* A[kMaxBatch];   // input matrices, row-major n x n
  double* w[kMaxBatch];          // eigenvalues out (ascending)
  double2* Z[kMaxBatch];         // eigenvectors out, Z[i * n + k] = component i of vector k
  int n[kMaxBatch];
  int rot[kMaxBatch];            // column j of problem b lives in block (j + rot) mod G
  int soff[kMaxBatch];           // own columns' offset in dynamic shared memory, -1: global
  int voff[kMaxBatch];           // offset of the block's three work vectors, -1: global
  double2* gvec;                 // per (problem slot, block) work vectors when voff = -1
  size_t gvec_stride;            // double2 per (problem slot, block) in gvec
  int coff;                      // offset of the per-column partials (doubles) in shared memory
  int off[kMaxBatch + 1];        // prefix sums of n: eigenvalue / column items
  int sid[kMaxBatch];            // workspace slot of each problem
  int np;
  double2* S0;                   // per problem: own columns (global home), later U0
  double2* S1;                   // per problem: reflectors V[t * n + i]
  double2* S2;                   // per problem: Y and its Loewdin ping-pong buffer
  size_t slot;                   // double2 per problem in S0, S1, S2
  double* T;                     // per problem: U2, published vectors, tau, d, e, e^2, lambda
  size_t tslot;                  // doubles per problem in T
  int m;                         // stride of the vectors in T (even, >= every n)
  const int* run;                // problem b runs iff run == null or run[b * run_stride] != 0
  int run_stride;
  double* sp;                    // per problem slot: [2][gridDim.x] partials of Re(v^H p)
  size_t sp_stride;
  int* status;
  long long spins;
  long long* stats;
  // Teams (stage 1): the blocks tg0[k] .. tg0[k+1]-1 reduce the problems
  // tmem[tp0[k]] .. tmem[tp0[k+1]-1] by themselves, with their own barrier
  // counter tbar[kTeamBarStride k]; one team of all blocks when nteam = 1.
  int nteam;
  int tmem[kMaxBatch];
  int tp0[kMaxBatch + 1];
  int tg0[kMaxBatch + 1];
  unsigned* tbar;
};

// This block's team: its size G, the block's rank gb in it, its problems
// (positions p0 .. p1-1 of tmem) and its barrier counter.
struct TeamView {
  int G, gb, p0, p1;
  unsigned* bar;
};

struct TriPtrs {
  double2* cols;                 // own columns, global home: column j at cols + j * n
  double2* V;
  double *Y, *Y2, *U0, *U2;      // U0: pairs (1 / pivot, first superdiagonal)
  double2 *P, *C, *tau;          // published p and columns, kTriBufs of m each
  double *d, *e, *e2, *lam;
  float *df, *e2f;               // d and e^2 rounded to float (coarse bisection rounds)
  dd *ddd, *e2dd;                // d and e^2 as float pairs (fine bisection rounds)
};

__device__ __forceinline__ TriPtrs tri_ptrs(const TriBatch& a, int b) {
  TriPtrs p;
  const size_t n = (size_t)a.n[b], m = (size_t)a.m, k = (size_t)a.sid[b];
  p.cols = a.S0 + k * a.slot;
  p.U0 = reinterpret_cast<double*>(p.cols);
  p.V = a.S1 + k * a.slot;
  p.Y = reinterpret_cast<double*>(a.S2 + k * a.slot);
  p.Y2 = p.Y + n * n;
  double* t = a.T + k * a.tslot;
  p.U2 = t;
  double2* vecs = reinterpret_cast<double2*>(t + m * m);   // m even: 16-byte aligned
  p.P = vecs; p.C = vecs + kTriBufs * m; p.tau = vecs + 2 * kTriBufs * m;
  double* s = reinterpret_cast<double*>(vecs + (2 * kTriBufs + 1) * m);
  p.d = s; p.e = s + m; p.e2 = s + 2 * m; p.lam = s + 3 * m;
  p.ddd = reinterpret_cast<dd*>(s + 4 * m); p.e2dd = p.ddd + m;        // m doubles each
  p.df = reinterpret_cast<float*>(s + 6 * m); p.e2f = p.df + m;        // m / 2 doubles each
  return p;
}

// The block's three work vectors of problem b (v_t, v_{t-1}, w): in shared
// memory, or, for problems too large for it, a private copy per block in
// global memory (every block computes the same vectors itself, so the copies
// must not be shared between blocks).
__device__ __forceinline__ double2* vec_base(const TriBatch& a, int b, double2* dsm) {
  return a.voff[b] >= 0
             ? dsm + a.voff[b]
             : a.gvec + ((size_t)a.sid[b] * gridDim.x + blockIdx.x) * a.gvec_stride;
}

__device__ __forceinline__ bool tri_run(const TriBatch& a, int b) {
  return a.n[b] > 0 && (!a.run || a.run[b * a.run_stride] != 0);
}

// Warp sum by butterfly: every lane ends with the same total.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Warp sums of two values, in lane 0 (five additions for both).
__device__ __forceinline__ void warp_sum2(double& x, double& y) {
  const int lane = threadIdx.x & 31;
  double v = lane < 16 ? x : y;
  v += __shfl_xor_sync(0xffffffffu, lane < 16 ? y : x, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  x = v;
  y = __shfl_sync(0xffffffffu, v, 16);
}

// ---- stage 1: Householder reduction ------------------------------------------
// What a step takes is FP64 instructions (a warp's takes the SM's unit 16 cycles
// whatever lanes are active) and the latency of what stands in a row (67 cycles
// each, an exchange between the blocks some thousands).  So:
//  - scalars are formed by one warp and passed on in shared memory, sums over a
//    block's threads go through shared memory to one warp;
//  - w is not formed (column j <- column j - u a_j - p b_j with a_j = conj(w_j) -
//    c conj(u_j), b_j = tau conj(u_j), c = |tau|^2 u^H p / 2), u stays unscaled
//    until k_hh_scale;
//  - norm, beta and tau are formed while the other warps update their columns:
//    these need only row t + 1 of u from it, whose term is added at the end;
//  - a block's columns are split over its warps by rows.
// With the published values as flags (kUnset) 700 + 300 states take 8.9 ms instead
// of 12.0 ms, 280 + 120 states 2.4 instead of 3.3 ms.
// The per-step vectors of a problem are short (n - t entries): its head work
// runs on a group of 16, 8 or 4 warps for one, two or more problems left, and the
// heads of up to kHeadGroups problems run side by side (one set of __syncthreads
// for all of them).
constexpr int kHeadGroups = 4;
constexpr int kHeadSums = 5;            // per-block partials a lane loads at once
constexpr int kHeadLoad = 4;            // elements per thread loaded ahead of the sums
constexpr int kTabProbs = 4;            // problems of a team whose a_j, b_j are tabulated
constexpr int kTabCols = 31;            // own columns of them
constexpr int kBodyItems = 64;          // column shares per pass of tri_body
constexpr int kMaxParts = 8;            // row shares of a column at most
constexpr int kPartWarps = 4;           // warps that share the block's columns, if fewer (each
                                        // costs a sum over its lanes; 700 states: 8.42 ms
                                        // with 4, 8.45 with 6, 8.56 with 9, 8.75 with 15 shares)

__device__ __forceinline__ TeamView team_view(const TriBatch& a) {
  const int k = find_prob(a.tg0, a.nteam, (int)blockIdx.x);
  TeamView v;
  v.G = a.tg0[k + 1] - a.tg0[k];
  v.gb = (int)blockIdx.x - a.tg0[k];
  v.p0 = a.tp0[k];
  v.p1 = a.tp0[k + 1];
  v.bar = a.tbar + (size_t)kTeamBarStride * k;
  return v;
}

// First own column of this block for problem b and the number of own columns
// (columns are dealt cyclically over the team's blocks).
__device__ __forceinline__ void own_range(const TriBatch& a, const TeamView& tv, int b, int& j0,
                                          int& ns) {
  const int G = tv.G, n = a.n[b];
  j0 = ((tv.gb - a.rot[b]) % G + G) % G;
  ns = j0 < n ? (n - 1 - j0) / G + 1 : 0;
}

__device__ __forceinline__ double2* own_col(const TriBatch& a, int b, double2* dsm, int j, int s) {
  const int n = a.n[b];
  return a.soff[b] >= 0 ? dsm + a.soff[b] + (size_t)s * n
                        : a.S0 + (size_t)a.sid[b] * a.slot + (size_t)j * n;
}

// Per-block partials of Re(u_t^H p_t) of problem b.
__device__ __forceinline__ double* sp_row(const TriBatch& a, int b, int t) {
  return a.sp + (size_t)a.sid[b] * a.sp_stride + (size_t)(t & (kTriBufs - 1)) * gridDim.x;
}

// The published values of step t (p, column t + 1, the partials of u^H p) are
// their own flags: a reader takes a word once it no longer holds kUnset, a
// signalling NaN that no arithmetic returns.  That is one trip through L2 per
// step, where a barrier costs the writers' fence, its counter, the poll and then
// the loads: 7.9 -> 7.4 us a step at 120 states, 13.2 -> 12.5 us at 700 when it came.
// The values of step t are in buffer t mod kTriBufs; while step t is under way its
// owners unset their words of the buffer of step t + 4, which held those of step t - 4.
// Two fences a step order that, both where their warps would only wait: (F) the warp
// that publishes the partials (the last one) before its shares, (A) the warps that
// read the partials (the heads' first ones) behind the shares.
//  - Everyone has read step t - 4: each block did in the head of step t - 3, its F and
//    its partial of that step follow; that partial was read here in the head of step
//    t - 2; A and a barrier of that step precede the unsetting.
//  - Nobody takes an old word for one of step t + 4: the unsetting, a barrier, F and
//    the partial of step t + 1; the others read that in the head of step t + 2, then A
//    and a barrier, and look for the words of step t + 4 in the head of step t + 5.
// (One fence between the heads and the shares, in the heads' first warps, with four
// buffers: it stands behind the reflector's scalars and costs 1 to 5 % of the
// reduction.)  Every wait is bounded.
constexpr unsigned long long kUnset = 0x7FF4000000C0FFEEull;
__device__ __forceinline__ double unset() { return __longlong_as_double((long long)kUnset); }
__device__ __forceinline__ bool is_unset(double x) {
  return (unsigned long long)__double_as_longlong(x) == kUnset;
}
__device__ __forceinline__ void put_word(double* p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ void put_word(double2* p, double2 v) {
  asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ double get_word(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double2 get_word(const double2* p) {
  double2 v;
  asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool is_unset(double2 v) { return is_unset(v.x) || is_unset(v.y); }
// Another try at a word that was not there: false when the wait is over.
struct TriWait {
  int* status;
  long long left;
  bool ok;
};
__device__ __forceinline__ bool wait_more(TriWait& w) {
  --w.left;
  if (w.left <= 0 || ((w.left & 63) == 0 && (*(volatile int*)w.status & SKY_STATUS_BIT(SKY_ETIMEOUT)))) {
    flag_status(w.status, SKY_ETIMEOUT);
    w.ok = false;
  }
  return w.ok;
}
template <typename T>
__device__ __forceinline__ T await_word(const T* p, T v, TriWait& w) {
  while (is_unset(v)) {
    if (!wait_more(w)) break;
    v = get_word(p);
  }
  return v;
}

struct HeadShared {
  double sg[kTriWarps][16];                 // the threads' |column|^2, pairs of lanes added
  double2 at[kHeadGroups][2];               // a_t, b_t
  double2 tab[kTabProbs][kTabCols][2];      // a_j, b_j of the own columns from slot smin on
  double2 acc[kBodyItems];                  // column shares' col^H u but for row t + 1
  double2 x1[kBodyItems];                   // row t + 1 of the columns
  int rescaled[2];                          // a reflector of step t (parity) has scl != 1
  int timeout[2];                           // a wait before the first, second barrier ran out
};
// Reflector t of a problem, the same in every block; entry b + kMaxBatch (t & 1).
struct TriStep {
  double2 tau;                              // for the unscaled u: H = I - tau u u^H
  double kap;                               // |tau|^2 / 2
  double c;                                 // of the reflector before: kap u^H p
  double scl;                               // power of two u was scaled by
  double beta, den;                         // den = |u_{t+1}|^2
};
// A problem of the team (by position): its size (0: not to be run), this block's
// own columns j0 + s G, s < ns, and the first s with j >= t + 1.
struct TriOwn {
  int n, j0, ns, smin;
};

// The r-th problem (position) still at work at step t, or -1; how many there are.
__device__ __forceinline__ int nth_active(const TriOwn* own, int np, int t, int r) {
  for (int k = 0; k < np; ++k)
    if (t < own[k].n && r-- == 0) return k;
  return -1;
}
__device__ __forceinline__ int count_active(const TriOwn* own, int np, int t) {
  int c = 0;
  for (int k = 0; k < np; ++k) c += t < own[k].n;
  return c;
}
// A warp group's problem in tri_heads (k < 0: none), found again only when the
// number of problems at work changes: the walk to it and its pointers took 1000
// cycles of each step.
struct TriHead {
  int k, b, n;
  double2* vb;                              // work vectors
  double2 *P, *C;
  double* sp;
};
__device__ __forceinline__ TriHead head_of(const TriBatch& a, const TeamView& tv, const TriOwn* own,
                                           int t, int r, double2* dsm) {
  TriHead h;
  h.k = nth_active(own, tv.p1 - tv.p0, t, r);
  h.b = h.k >= 0 ? a.tmem[tv.p0 + h.k] : 0;
  h.n = h.k >= 0 ? own[h.k].n : 0;
  const TriPtrs p = tri_ptrs(a, h.b);
  h.vb = h.k >= 0 ? vec_base(a, h.b, dsm) : dsm;
  h.P = p.P;
  h.C = p.C;
  h.sp = sp_row(a, h.b, 0);
  return h;
}
// Active own columns of a problem at step t (none at its last).
__device__ __forceinline__ int active_cols(const TriOwn& o, int t) {
  return t < o.n - 1 ? o.ns - o.smin : 0;
}
// a_j, b_j of column j from p_j, u_j.
__device__ __forceinline__ void column_factors(const TriStep& st, double2 pj, double2 uj, double2& fa,
                                               double2& fb) {
  const double c2 = 2.0 * st.c;
  fa = make_double2(fma(-c2, uj.x, fma(st.tau.x, pj.x, -st.tau.y * pj.y)),
                    fma(c2, uj.y, -fma(st.tau.x, pj.y, st.tau.y * pj.x)));
  fb = make_double2(fma(st.tau.x, uj.x, st.tau.y * uj.y), fma(st.tau.y, uj.x, -st.tau.x * uj.y));
}
// w = tau p - c u; with it the update of column j is x - u conj(w_j) - w conj(u_j).
__device__ __forceinline__ double2 w_entry(const TriStep& st, double2 p, double2 u) {
  return make_double2(fma(-st.c, u.x, fma(st.tau.x, p.x, -st.tau.y * p.y)),
                      fma(-st.c, u.y, fma(st.tau.x, p.y, st.tau.y * p.x)));
}
// x - u a - p b.
__device__ __forceinline__ double2 column_update(double2 x, double2 u, double2 p, double2 fa,
                                                 double2 fb) {
  return make_double2(
      fma(-u.x, fa.x, fma(u.y, fa.y, fma(-p.x, fb.x, fma(p.y, fb.y, x.x)))),
      fma(-u.x, fa.y, fma(-u.y, fa.x, fma(-p.x, fb.y, fma(-p.y, fb.x, x.y)))));
}

// The heads of a round's problems (h: this warp group's; 2^lg warps each), step t,
// every block of the team alike: column t of the trailing matrix
// (updated by reflector t-1 from the published copy) into vn, the published p
// into w, and reflector t.  vo = u_{t-1}.  u_{t-1}^H p_{t-1} is the sum of the
// owners' published per-block partials (the same order in every block).  The
// published p and column are loaded in one pass (one L2 round trip per step).
// The group's first warp ends with reflector t after the last barrier here: its
// results, u_{t+1} among them, are there after the next one.  False (in every
// thread) when a wait ran out.
template <bool ONE>
__device__ bool tri_heads(const TriBatch& a, const TeamView& tv, const TriHead& h, bool first, int lg,
                          int t, HeadShared& hs, TriStep* s_st, const TriOwn* own) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int q = wid >> lg, hwarp = wid & ((1 << lg) - 1), HT = 32 << lg, ht = hwarp * 32 + lane;
  const int k = h.k, b = h.b, n = h.n;
  const bool on = k >= 0;
  double2* vn = h.vb + (size_t)(t & 1) * n;
  const double2* vo = h.vb + (size_t)((t + 1) & 1) * n;
  double2* w = h.vb + 2 * (size_t)n;
  double sg = 0.0;                           // |column|^2 below the subdiagonal
  TriWait wt{a.status, a.spins, true};
  if (t == 0) {
    const double2* A = on ? a.A[b] : nullptr;
    for (int i = ht; i < n; i += HT) {
      double2 x = A[i];
      x.y = i == 0 ? 0.0 : -x.y;             // column 0 = conj(row 0)
      vn[i] = x;
      if (i >= 2) sg = fma(x.x, x.x, fma(x.y, x.y, sg));
    }
    if (first && threadIdx.x == 0) hs.rescaled[t & 1] = 0;
  } else {
    double2 xp[kHeadLoad], xc[kHeadLoad];
    const double2* Pp = h.P + (size_t)((t - 1) & (kTriBufs - 1)) * a.m;
    const double2* Cp = h.C + (size_t)((t - 1) & (kTriBufs - 1)) * a.m;
    if (on) {
#pragma unroll
      for (int r = 0; r < kHeadLoad; ++r) {
        const int i = t + ht + r * HT;
        if (i < n) {
          xp[r] = get_word(Pp + i);
          xc[r] = get_word(Cp + i);          // the column after step t-2's update
        }
      }
      if (hwarp == 0) {
        // lanes 0 .. 30: own columns; lane 31: column t
        const double* ps = h.sp + (size_t)((t - 1) & (kTriBufs - 1)) * gridDim.x;
        const int cb = active_cols(own[k], t);
        const int j = lane == 31 ? t : lane < cb ? own[k].j0 + (own[k].smin + lane) * tv.G : -1;
        double2 pj = j >= 0 ? get_word(Pp + j) : make_double2(0.0, 0.0);
        double S0 = 0.0, S1 = 0.0;
        for (int g = lane; g < tv.G; g += 32 * kHeadSums) {
          double x[kHeadSums];
#pragma unroll
          for (int r = 0; r < kHeadSums; ++r) x[r] = g + 32 * r < tv.G ? get_word(ps + g + 32 * r) : 0.0;
          for (;;) {                         // (all words that are missing at once)
            bool miss = false;
#pragma unroll
            for (int r = 0; r < kHeadSums; ++r) miss |= is_unset(x[r]);
            if (!miss || !wait_more(wt)) break;
#pragma unroll
            for (int r = 0; r < kHeadSums; ++r)
              if (is_unset(x[r])) x[r] = get_word(ps + g + 32 * r);
          }
#pragma unroll
          for (int r = 0; r < kHeadSums; ++r) (r & 1 ? S1 : S0) += x[r];
        }
        if (j >= 0) pj = await_word(Pp + j, pj, wt);
        const double2 uj = j >= 0 ? vo[j] : make_double2(0.0, 0.0);
        __syncwarp();
        TriStep& prev = s_st[b + (size_t)((t + 1) & 1) * kMaxBatch];
        TriStep st = prev;
        st.c = st.kap * warp_sum(S0 + S1);
        double2 fa, fb;
        if constexpr (!ONE) {
          column_factors(st, pj, uj, fa, fb);
        } else {
          fa = conjx(w_entry(st, pj, uj));
          fb = conjx(uj);
        }
        if (lane == 31) {
          hs.at[q][0] = fa;
          hs.at[q][1] = fb;
          prev.c = st.c;
        } else if (!ONE && lane < cb && k < kTabProbs) {
          hs.tab[k][lane][0] = fa;
          hs.tab[k][lane][1] = fb;
        }
      }
      for (;;) {
        bool miss = false;
#pragma unroll
        for (int r = 0; r < kHeadLoad; ++r)
          if (t + ht + r * HT < n) miss |= is_unset(xp[r]) || is_unset(xc[r]);
        if (!miss || !wait_more(wt)) break;
#pragma unroll
        for (int r = 0; r < kHeadLoad; ++r) {
          const int i = t + ht + r * HT;
          if (i < n) {
            if (is_unset(xp[r])) xp[r] = get_word(Pp + i);
            if (is_unset(xc[r])) xc[r] = get_word(Cp + i);
          }
        }
      }
      __syncwarp();
    }
    if (first && threadIdx.x == 0) hs.rescaled[t & 1] = 0;
    if (!wt.ok) hs.timeout[0] = 1;
    __syncthreads();
    if (hs.timeout[0]) return false;
    if (on) {
      const double2 fa = hs.at[q][0], fb = hs.at[q][1];
      const TriStep& prev = s_st[b + (size_t)((t + 1) & 1) * kMaxBatch];
      auto row = [&](int i, double2 pi, double2 ci) {
        if constexpr (ONE) pi = w_entry(prev, pi, vo[i]);
        const double2 y = column_update(ci, vo[i], pi, fa, fb);
        w[i] = pi;
        vn[i] = y;
        if (i >= t + 2) sg = fma(y.x, y.x, fma(y.y, y.y, sg));
      };
#pragma unroll
      for (int r = 0; r < kHeadLoad; ++r) {
        const int i = t + ht + r * HT;
        if (i < n) row(i, xp[r], xc[r]);
      }
      for (int i = t + ht + kHeadLoad * HT; i < n; i += HT)
        row(i, await_word(Pp + i, get_word(Pp + i), wt), await_word(Cp + i, get_word(Cp + i), wt));
      if (!wt.ok) hs.timeout[1] = 1;
      __syncwarp();
    }
  }
  if (t + hwarp * 32 < n || t == 0) sg += __shfl_xor_sync(0xffffffffu, sg, 16);
  if (lane < 16) hs.sg[wid][lane] = sg;
  __syncthreads();
  if (hs.timeout[1]) return false;
  if (hwarp != 0 || !on || t > n - 2) return true;
  double sig = 0.0;
  {
    double s2[8];                            // 16 gw values, half as many per lane
    const int half = lane >> 4;
#pragma unroll
    for (int r = 0; r < 8; ++r) s2[r] = r < (1 << lg) / 2 ? hs.sg[wid + 2 * r + half][lane & 15] : 0.0;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1)
      if (o < (1 << lg) / 2)
#pragma unroll
        for (int r = 0; r + o < 8; r += 2 * o) s2[r] += s2[r + o];
    sig = warp_sum(s2[0]);
  }
  if (lane != 0) return true;
  double2 al = vn[t + 1];
  TriStep st;
  st.c = 0.0;
  st.scl = 1.0;
  st.tau = make_double2(0.0, 0.0);
  st.kap = 0.0;
  st.den = 1.0;
  double2 u1 = make_double2(1.0, 0.0);
  if (sig == 0.0 && al.y == 0.0) {
    st.beta = al.x;                          // already real: H_t = I
  } else {
    double s2 = fma(al.x, al.x, fma(al.y, al.y, sig));
    double unscl = 1.0;
    if (!(s2 > 0x1p-60 && s2 < 0x1p+60) && s2 > 0.0 && s2 < 1.7e308) {
      // far from 1: u times a power of two, so that tau stays in range, as does what
      // the reciprocals below start from
      const int ex = (int)((__double_as_longlong(s2) >> 52) & 0x7FF);
      const int h = ex == 0 ? -537 : (ex - 1023) >> 1;
      st.scl = __longlong_as_double((long long)(1023 - h) << 52);
      unscl = __longlong_as_double((long long)(1023 + h) << 52);
      s2 = (s2 * st.scl) * st.scl;
      al.x *= st.scl;
      al.y *= st.scl;
      hs.rescaled[t & 1] = 1;
    }
    // |column|, by one step of Heron's rule from the refined reciprocal root
    const double rs = rsqrt_refined(s2);
    double nr = s2 * rs;
    nr = fma(0.5 * rs, fma(-nr, nr, s2), nr);
    const double beta = al.x >= 0.0 ? -nr : nr;
    st.beta = beta * unscl;
    const double dx = al.x - beta;           // |Re alpha| + nr: no cancellation
    st.den = fma(dx, dx, al.y * al.y);
    const double r = rcp_refined(beta * st.den);
    st.tau = make_double2(-dx * r, -al.y * r);
    st.kap = 0.5 * fma(st.tau.x, st.tau.x, st.tau.y * st.tau.y);
    u1 = make_double2(dx, al.y);             // alpha - beta
  }
  vn[t + 1] = u1;
  s_st[b + (size_t)(t & 1) * kMaxBatch] = st;
  return true;
}

// d_t, beta_t, the unscaled reflector t and its tau and |u_{t+1}|^2 (in e2) of the
// team's problems, by one block, a different one each step, while the arrivals
// are under way (k_hh_scale makes of them what is kept).
__device__ void tri_store(const TriBatch& a, const TeamView& tv, int t, double2* dsm,
                          const TriStep* s_st, const TriOwn* own) {
  for (int k = 0; k < tv.p1 - tv.p0; ++k) {
    const int b = a.tmem[tv.p0 + k], n = own[k].n;
    if (t >= n) continue;
    const double2* vn = vec_base(a, b, dsm) + (size_t)(t & 1) * n;
    const TriPtrs p = tri_ptrs(a, b);
    if (threadIdx.x == 0) p.d[t] = vn[t].x;
    if (t > n - 2) continue;
    if (threadIdx.x == 32) {
      const TriStep& st = s_st[b + (size_t)(t & 1) * kMaxBatch];
      p.e[t] = st.beta;
      p.e2[t] = st.den;
      p.tau[t] = st.tau;
    }
    double2* Vt = p.V + (size_t)t * n;
    for (int i = t + 1 + (int)threadIdx.x; i < n; i += kTriThreads) Vt[i] = vn[i];
  }
}

// This block's words of the buffer of step t + 4, by the warps other than the last:
// p of its columns, its partials, and as the owner of column t + 5 that.
__device__ __forceinline__ void tri_unset(const TriBatch& a, const TeamView& tv, int t,
                                          const TriOwn* own) {
  const int tid = (int)threadIdx.x;
  for (int k = 0; k < tv.p1 - tv.p0; ++k) {
    const int b = a.tmem[tv.p0 + k], n = own[k].n;
    if (t + 4 > n - 2) continue;             // step t + 4 publishes nothing
    const TriPtrs p = tri_ptrs(a, b);
    const size_t o = (size_t)((t + 4) & (kTriBufs - 1)) * a.m;
    const double2 no = make_double2(unset(), unset());
    for (int s = tid; s < own[k].ns; s += kTriThreads - 32)
      put_word(p.P + o + own[k].j0 + s * tv.G, no);
    if (tid == kTriThreads - 33) put_word(sp_row(a, b, t + 4) + tv.gb, unset());
    if ((t + 5 + a.rot[b]) % tv.G == tv.gb)
      for (int i = t + 5 + tid; i < n; i += kTriThreads - 32) put_word(p.C + o + i, no);
  }
}

// Own columns j >= t+1: update by reflector t-1 (rows > t), p_j = col_j^H u_t,
// publication of p_j and of column t+1, and the block's partial of Re(u_t^H p_t)
// per problem (over its own columns, in column order), for the team's problems.
// A column's rows go to `parts` warps in turn.  The first shares are begun while
// the first warps of the last ng groups of heads are at reflector t (so those get
// theirs last), and row t + 1 of u is added after the barrier.
template <bool ONE>
__device__ void tri_body(const TriBatch& a, const TeamView& tv, int t, int lg, int ng, double2* dsm,
                         double* contrib, HeadShared& hs, const TriStep* s_st, TriOwn* own) {
  const int G = tv.G, np = tv.p1 - tv.p0, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int grp = wid >> lg;
  const int rank = grp >= ng ? wid - ng
                             : (wid & ((1 << lg) - 1)) == 0 ? kTriWarps - ng + grp : wid - grp - 1;
  // F of kUnset (a team of one block reads its words behind its own barrier)
  constexpr int kLast = kTriWarps - 1;
  if (!ONE && wid == kLast) __threadfence();
  int C = 0, mmax = 0;
  for (int k = 0; k < np; ++k) {
    C += active_cols(own[k], t);
    mmax = own[k].n - t > mmax ? own[k].n - t : mmax;
  }
  // at least two rows per lane and share
  int parts = C > 0 ? (kPartWarps + C - 1) / C : 1;
  const int most = (mmax + 63) >> 6;
  parts = parts > most ? most : parts;
  parts = parts < 1 ? 1 : parts > kMaxParts ? kMaxParts : parts;
  const TriStep* cur = s_st + (size_t)(t & 1) * kMaxBatch;
  const TriStep* before = s_st + (size_t)((t + 1) & 1) * kMaxBatch;
  // column ci -> position k of its problem, its place among the active ones
  auto find = [&](int ci, int& k, int& rest) {
    rest = ci;
    for (k = 0; k < np; ++k) {
      const int cb = active_cols(own[k], t);
      if (rest < cb) return;
      rest -= cb;
    }
  };
  for (int c0 = 0; c0 < C || c0 == 0; c0 += kBodyItems) {
    const int cols = C - c0 < kBodyItems ? C - c0 : kBodyItems;
    for (int it = rank; it < cols * parts; it += kTriWarps) {
      const int part = parts == 1 ? 0 : it / cols, cj = it - part * cols;
      int k, rest;
      find(c0 + cj, k, rest);
      const int b = a.tmem[tv.p0 + k], n = own[k].n, s = own[k].smin + rest, j = own[k].j0 + s * G;
      double2* col = own_col(a, b, dsm, j, s);
      const double2* vb = vec_base(a, b, dsm);
      const double2* vn = vb + (size_t)(t & 1) * n;
      const double2* vo = vb + (size_t)((t + 1) & 1) * n;
      const double2* w = vb + 2 * (size_t)n;
      const bool upd = t >= 1, pub = (j == t + 1);
      double2* Cb = nullptr;
      if (pub) {
        const TriPtrs p = tri_ptrs(a, b);
        Cb = p.C + (size_t)(t & (kTriBufs - 1)) * a.m;
      }
      double2 fa = make_double2(0.0, 0.0), fb = fa;
      if (upd) {
        if constexpr (ONE) {
          fa = conjx(w[j]);
          fb = conjx(vo[j]);
        } else if (k < kTabProbs && rest < kTabCols) {
          fa = hs.tab[k][rest][0];
          fb = hs.tab[k][rest][1];
        } else {
          column_factors(before[b], w[j], vo[j], fa, fb);
        }
      }
      double ax = 0.0, ay = 0.0, bx = 0.0, by = 0.0;
      double2 x1 = make_double2(0.0, 0.0);
      const int step = 32 * parts;
      // two rows at a time, loads first
      for (int i = t + 1 + part * 32 + lane; i < n; i += 2 * step) {
        const int i2 = i + step;
        const bool two = i2 < n;
        double2 xa = col[i], xb = make_double2(0.0, 0.0), v2 = xb, va = xb;
        if (two) {
          xb = col[i2];
          v2 = vn[i2];
        }
        if (i > t + 1) va = vn[i];
        if (upd) {
          xa = column_update(xa, vo[i], w[i], fa, fb);
          if (two) xb = column_update(xb, vo[i2], w[i2], fa, fb);
          col[i] = xa;
          if (two) col[i2] = xb;
        }
        if (i == t + 1) x1 = xa;
        if (pub) {
          put_word(Cb + i, xa);
          if (two) put_word(Cb + i2, xb);
        }
        ax = fma(xa.x, va.x, fma(xa.y, va.y, ax));      // conj(x) u
        ay = fma(xa.x, va.y, fma(-xa.y, va.x, ay));
        bx = fma(xb.x, v2.x, fma(xb.y, v2.y, bx));
        by = fma(xb.x, v2.y, fma(-xb.y, v2.x, by));
      }
      ax += bx;
      ay += by;
      warp_sum2(ax, ay);
      if (lane == 0) {
        hs.acc[part * cols + cj] = make_double2(ax, ay);
        if (part == 0) hs.x1[cj] = x1;
      }
    }
    __syncthreads();                         // reflector t; the shares
    if (c0 == 0 && hs.rescaled[t & 1]) {
      for (int k = 0; k < np; ++k) {
        const int b = a.tmem[tv.p0 + k], n = own[k].n;
        if (t > n - 2 || cur[b].scl == 1.0) continue;
        double2* v = vec_base(a, b, dsm) + (size_t)(t & 1) * n;
        const double sc = cur[b].scl;
        for (int i = t + 2 + (int)threadIdx.x; i < n; i += kTriThreads)
          v[i] = make_double2(v[i].x * sc, v[i].y * sc);
      }
      __syncthreads();
    }
    if (!ONE && c0 == 0 && wid != kLast) {
      if ((wid & ((1 << lg) - 1)) == 0) __threadfence();   // A of kUnset
      tri_unset(a, tv, t, own);
    }
    if (ONE || wid == kLast)
      for (int cj = ONE ? (int)threadIdx.x : lane; cj < cols; cj += ONE ? kTriThreads : 32) {
        int k, rest;
        find(c0 + cj, k, rest);
        const int b = a.tmem[tv.p0 + k], n = own[k].n, j = own[k].j0 + (own[k].smin + rest) * G;
        const double2* vn = vec_base(a, b, dsm) + (size_t)(t & 1) * n;
        double2 z[kMaxParts];
#pragma unroll
        for (int q = 0; q < kMaxParts; ++q)
          z[q] = q < parts ? hs.acc[q * cols + cj] : make_double2(0.0, 0.0);
#pragma unroll
        for (int o = 1; o < kMaxParts; o <<= 1)
          if (o < parts)
#pragma unroll
            for (int q = 0; q + o < kMaxParts; q += 2 * o) z[q] = z[q] + z[q + o];
        const double2 u1 = vn[t + 1], x1 = hs.x1[cj], uj = vn[j];
        const double sc = cur[b].scl;        // (the shares are of u before its scaling)
        const double ax = fma(x1.x, u1.x, fma(x1.y, u1.y, sc * z[0].x));
        const double ay = fma(x1.x, u1.y, fma(-x1.y, u1.x, sc * z[0].y));
        const TriPtrs p = tri_ptrs(a, b);
        put_word(p.P + (size_t)(t & (kTriBufs - 1)) * a.m + j, make_double2(ax, ay));
        contrib[c0 + cj] = fma(uj.x, ax, uj.y * ay);   // Re(conj(u_t[j]) p_j)
      }
    if (c0 + kBodyItems < C) __syncthreads();
  }
  // per-problem partials, one lane per problem, own columns in order (one block has
  // all columns: one warp per problem); the next step's first own columns
  if constexpr (ONE) {
    __syncthreads();
    for (int k = wid; k < np; k += kTriWarps) {
      if (t > own[k].n - 2) continue;
      int first = 0;
      for (int kq = 0; kq < k; ++kq) first += active_cols(own[kq], t);
      const int cb = active_cols(own[k], t);
      double acc = 0.0;
      for (int i = lane; i < cb; i += 32) acc += contrib[first + i];
      acc = warp_sum(acc);
      if (lane == 0) put_word(sp_row(a, a.tmem[tv.p0 + k], t) + tv.gb, acc);
    }
    __syncthreads();                         // smin is read above
  }
  if (wid != kLast) return;
  __syncwarp();
  for (int k = lane; k < np && !ONE; k += 32) {
    TriOwn& o = own[k];
    if (t > o.n - 2) continue;
    int first = 0;
    for (int kq = 0; kq < k; ++kq) first += active_cols(own[kq], t);
    const int cb = active_cols(o, t);
    double acc = 0.0;
    for (int i = 0; i < cb; ++i) acc += contrib[first + i];
    put_word(sp_row(a, a.tmem[tv.p0 + k], t) + tv.gb, acc);
  }
  __syncwarp();
  for (int k = lane; k < np; k += 32)
    if (own[k].smin < own[k].ns && own[k].j0 + own[k].smin * G < t + 2) ++own[k].smin;
}

// All steps of a team.  False when a wait ran out.  ONE: a team of one block, which
// has every column.  It reads its own words behind its barrier (nothing to unset, no
// fence), takes w instead of p (one entry per row; factors per column cost 10 FP64
// instructions for each of up to hundreds of columns), and all its warps finish
// the columns and sum the partials (one warp did, column after column: 8400 cycles of
// a step at 125 columns).  One 100-state problem per block: 3.09 ms as the
// teams of several blocks do it, 2.70 ms; 128 problems of 37 to 290 states: 17.4 and
// 14.8 ms.
template <bool ONE>
__device__ bool tri_steps(const TriBatch& a, const TeamView& tv, int nrun, double2* dsm, double* contrib,
                          HeadShared& hs, TriStep* s_st, TriOwn* own) {
  const int tid = threadIdx.x, np = tv.p1 - tv.p0;
  TriHead h{};
  int seen = -1;
  for (int t = 0; t < nrun; ++t) {
    const int nact = count_active(own, np, t);
    const int lg = nact == 1 ? 4 : nact == 2 ? 3 : 2;
    const int per = kTriWarps >> lg;
    int last = 0;                            // problems of the last round of heads
    for (int r0 = 0; r0 < nact; r0 += per) {
      if (r0 > 0) __syncthreads();
      if (nact != seen || nact > per) h = head_of(a, tv, own, t, r0 + (tid >> (5 + lg)), dsm);
      seen = nact;
      if (!tri_heads<ONE>(a, tv, h, r0 == 0, lg, t, hs, s_st, own)) return false;
      last = nact - r0 < per ? nact - r0 : per;
    }
    tri_body<ONE>(a, tv, t, lg, last, dsm, contrib, hs, s_st, own);
    // (the next step's first loads wait for this one's values of every block)
    __syncthreads();
    if (tv.gb == t % tv.G) tri_store(a, tv, t, dsm, s_st, own);
  }
  return true;
}

__global__ void __launch_bounds__(kTriThreads, 1) k_hh_tridiag(TriBatch a) {
  extern __shared__ double2 dsm[];
  __shared__ HeadShared hs;
  __shared__ TriStep s_st[2 * kMaxBatch];
  __shared__ TriOwn own[kMaxBatch];
  const int tid = threadIdx.x, nt = blockDim.x;
  double* contrib = reinterpret_cast<double*>(dsm + a.coff);
  const TeamView tv = team_view(a);
  const int np = tv.p1 - tv.p0;
  unsigned epoch = 0;
  int nrun = 0;
  for (int k = 0; k < np; ++k) {
    const int b = a.tmem[tv.p0 + k];
    const bool r = tri_run(a, b);
    if (tid == 0) {
      TriOwn o;
      own_range(a, tv, b, o.j0, o.ns);
      o.n = r ? a.n[b] : 0;
      o.smin = o.j0 < 1 ? 1 : 0;             // the first column >= 1
      own[k] = o;
    }
    if (r && a.n[b] > nrun) nrun = a.n[b];
  }
  __syncthreads();
  // own columns: column j = conj(row j) of the Hermitian input
  for (int k = 0; k < np; ++k) {
    const int b = a.tmem[tv.p0 + k], n = own[k].n;
    if (n == 0) continue;
    const double2* A = a.A[b];
    for (int s = 0; s < own[k].ns; ++s) {
      const int j = own[k].j0 + s * tv.G;
      double2* col = own_col(a, b, dsm, j, s);
      for (int i = tid; i < n; i += nt) {
        double2 x = A[(size_t)j * n + i];
        // (step 0 publishes column 1 as it came: no input may look unset)
        if (is_unset(x.x)) x.x = NAN;
        x.y = i == j ? 0.0 : is_unset(x.y) ? NAN : -x.y;
        col[i] = x;
      }
    }
    // nothing published yet
    const TriPtrs p = tri_ptrs(a, b);
    const double2 no = make_double2(unset(), unset());
    for (int e = tid; e < own[k].ns * kTriBufs; e += nt) {
      const size_t o = (size_t)(e % kTriBufs) * a.m + own[k].j0 + (e / kTriBufs) * tv.G;
      put_word(p.P + o, no);
      put_word(p.C + o, no);
    }
    if (tid < kTriBufs) put_word(sp_row(a, b, tid) + tv.gb, unset());
  }
  if (tid == 0) hs.timeout[0] = hs.timeout[1] = 0;
  if (tv.G == 1) {
    __syncthreads();
  } else if (!blocks_barrier(tv.bar, epoch, (unsigned)tv.G, a.status, a.spins)) {
    return;
  }
  if (!(tv.G == 1 ? tri_steps<true>(a, tv, nrun, dsm, contrib, hs, s_st, own)
                  : tri_steps<false>(a, tv, nrun, dsm, contrib, hs, s_st, own)))
    return;
  if (tv.gb == 0 && tid == 0) {
    long long k = 0;
    for (int q = 0; q < np; ++q) k += own[q].n > 0;
    atomicAdd(reinterpret_cast<unsigned long long*>(a.stats + 6), (unsigned long long)k);
  }
}

// What is kept of reflector t (blockIdx.x) and of T: v = u / u_{t+1} and its tau, d
// and e in the forms the bisection reads.
__global__ void __launch_bounds__(128) k_hh_scale(TriBatch a) {
  const int b = blockIdx.y, t = blockIdx.x, n = a.n[b];
  if (t >= n || !tri_run(a, b)) return;
  const TriPtrs p = tri_ptrs(a, b);
  if (threadIdx.x == 0) {
    const double d = p.d[t];
    p.ddd[t] = dd_of(d);
    p.df[t] = __double2float_rn(d);
  }
  if (t > n - 2) return;
  double2* Vt = p.V + (size_t)t * n;
  const double2 u1 = Vt[t + 1];
  const double den = p.e2[t], r = 1.0 / den;
  const double2 sc = make_double2(u1.x * r, -u1.y * r);
  __syncthreads();
  if (threadIdx.x == 0) {
    const double e = p.e[t];
    const double2 tau = p.tau[t];
    p.e2[t] = e * e;
    p.e2dd[t] = dd_of(e) * dd_of(e);
    p.e2f[t] = __double2float_rn(e * e);
    p.tau[t] = make_double2(tau.x * den, tau.y * den);
    Vt[t + 1] = make_double2(1.0, 0.0);
  }
  for (int i = t + 2 + (int)threadIdx.x; i < n; i += 128) {
    const double2 x = Vt[i];
    Vt[i] = make_double2(fma(x.x, sc.x, -x.y * sc.y), fma(x.x, sc.y, x.y * sc.x));
  }
}

// ---- stage 2: eigenvalues of T -------------------------------------------------
// Number of eigenvalues of T below x: the number of negative pivots of the
// LDL^T factorisation of T - x I, q_0 = d_0 - x, q_k = (d_k - x) -
// e_{k-1}^2 / q_{k-1} (Sylvester's law of inertia); a pivot of modulus below
// pivmin is replaced by -pivmin.  The computed count is exact for T with
// every d_k - x and e_k^2 perturbed by a few units of the arithmetic's last
// place (Kahan; LAPACK's dstebz), so x is located to within that perturbation
// of ||T||.  On this chip a dependent FP64 operation takes ~67 cycles and an
// FP64 division ~670 (measured), FP32 ones ~5, so the count runs in FP32 to
// about 2^-16 ||T|| and then in double-float arithmetic (about 2^-46 per
// operation) to 2^-43 ||T||, no FP64 operation in the loops.
constexpr float kPivMin32 = 0x1p-100f;
constexpr double kBisF32Rel = 0x1p-16;   // FP32 rounds down to this width / ||T||
constexpr double kBisF32Pad = 0x1p-17;   // then widened by this much / ||T|| on each side
constexpr double kBisDDRel = 0x1p-43;    // double-float rounds down to this width / ||T||

__device__ __forceinline__ int sturm_count32(const float* __restrict__ d,
                                             const float* __restrict__ e2, int n, float x) {
  float q = __ldg(d) - x;
  int cnt = 0;
  for (int i = 1;; ++i) {
    if (fabsf(q) < kPivMin32) q = -kPivMin32;
    cnt += q < 0.0f;
    if (i >= n) break;
    q = (__ldg(d + i) - x) - __fdividef(__ldg(e2 + i - 1), q);
  }
  return cnt;
}
__device__ __forceinline__ int sturm_count_dd(const dd* __restrict__ d, const dd* __restrict__ e2,
                                              int n, dd x) {
  dd q = d[0] - x;
  int cnt = 0;
  for (int i = 1;; ++i) {
    if (fabsf(q.hi) < kPivMin32) q = dd(-kPivMin32, 0.0f);
    cnt += q.hi < 0.0f;
    if (i >= n) break;
    q = (d[i] - x) - ddiv(e2[i - 1], q);
  }
  return cnt;
}

// One warp per eigenvalue (every eigenvalue its own warp: one wave).  The
// lanes count at L points per round, so a round narrows the bracket L + 1
// times; the bracket invariant is count(lo) <= j < count(hi).
__global__ void __launch_bounds__(32) k_tri_bisect(TriBatch a) {
  constexpr int L = kBisLanes;
  static_assert(L == 32, "one warp per eigenvalue");
  const int l = threadIdx.x;
  const unsigned mask = 0xffffffffu;
  const int item = blockIdx.x;
  if (item >= a.off[a.np]) return;
  const int b = find_prob(a.off, a.np, item);
  if (!tri_run(a, b)) return;
  const int n = a.n[b], j = item - a.off[b];
  const TriPtrs p = tri_ptrs(a, b);
  // Gershgorin interval
  double glo = INFINITY, ghi = -INFINITY;
  for (int i = l; i < n; i += L) {
    const double r = (i > 0 ? fabs(p.e[i - 1]) : 0.0) + (i < n - 1 ? fabs(p.e[i]) : 0.0);
    glo = fmin(glo, p.d[i] - r);
    ghi = fmax(ghi, p.d[i] + r);
  }
#pragma unroll
  for (int o = 1; o < L; o <<= 1) {
    glo = fmin(glo, __shfl_xor_sync(mask, glo, o));
    ghi = fmax(ghi, __shfl_xor_sync(mask, ghi, o));
  }
  const double nrm = fmax(fmax(fabs(glo), fabs(ghi)), 1e-290);
  const double pad = 2.0 * kEps * nrm + 1e-290;
  glo -= pad;
  ghi += pad;
  // a round: counts at L interior points (or, with ends, at L points from lo
  // to hi inclusive); returns false when the ends do not bracket j
  auto narrow = [&](double& lo, double& hi, int cnt, double x) {
    double nlo = lo, nhi = hi;
    bool above = false;
#pragma unroll 4
    for (int k = 0; k < L; ++k) {
      const double xk = __shfl_sync(mask, x, k);
      const int ck = __shfl_sync(mask, cnt, k);
      if (!above) {
        if (ck <= j) nlo = xk;
        else { nhi = xk; above = true; }
      }
    }
    lo = nlo;
    hi = nhi;
  };
  // FP32 rounds
  double lo = glo, hi = ghi;
  {
    float lo32 = __double2float_rd(lo), hi32 = __double2float_ru(hi);
    const float w32 = (float)(kBisF32Rel * nrm);
    for (int round = 0; round < 12 && hi32 - lo32 > w32; ++round) {
      const float x = lo32 + (hi32 - lo32) * ((float)(l + 1) / (float)(L + 1));
      const int cnt = sturm_count32(p.df, p.e2f, n, x);
      double dlo = lo32, dhi = hi32;
      narrow(dlo, dhi, cnt, (double)x);
      lo32 = (float)dlo;
      hi32 = (float)dhi;
    }
    lo = fmax((double)lo32 - kBisF32Pad * nrm, glo);
    hi = fmin((double)hi32 + kBisF32Pad * nrm, ghi);
  }
  // double-float rounds; the first one includes both ends as a check
  {
    const double x = lo + (hi - lo) * ((double)l / (double)(L - 1));
    const int cnt = sturm_count_dd(p.ddd, p.e2dd, n, dd_of(x));
    const int c0 = __shfl_sync(mask, cnt, 0), cL = __shfl_sync(mask, cnt, L - 1);
    if (c0 <= j && cL > j) {
      narrow(lo, hi, cnt, x);
    } else {
      lo = glo;                              // the FP32 bracket missed: start over
      hi = ghi;
    }
  }
  const double tol = kBisDDRel * nrm;
  for (int round = 0; round < kBisMaxRounds && hi - lo > tol; ++round) {
    const double x = lo + (hi - lo) * ((double)(l + 1) / (double)(L + 1));
    const int cnt = sturm_count_dd(p.ddd, p.e2dd, n, dd_of(x));
    narrow(lo, hi, cnt, x);
  }
  if (l == 0) {
    const double lam = 0.5 * (lo + hi);
    p.lam[j] = lam;
    a.w[b][j] = lam;
  }
}

// ---- stage 3: eigenvectors of T ---------------------------------------------------
// Uniform in [-1, 1) from (k, i): the splitmix64 finaliser of a Weyl sequence.
__device__ __forceinline__ double start_entry(unsigned long long k, unsigned long long i) {
  unsigned long long x = k * 0x9E3779B97F4A7C15ull + (i + 1) * 0xD1B54A32D192ED03ull;
  x ^= x >> 30; x *= 0xBF58476D1CE4E5B9ull;
  x ^= x >> 27; x *= 0x94D049BB133111EBull;
  x ^= x >> 31;
  return (double)(x >> 11) * (1.0 / 4503599627370496.0) - 1.0;
}

// The solver's columns of vector k, row stride n: U = (1 / pivot, first
// superdiagonal of U), L = the multiplier of the row operation, its lowest mantissa
// bit set when rows i and i+1 were swapped (then U's second superdiagonal is
// e_{i+1}, else 0), Y = the vector.
//
// A thread works one vector off row by row, one warp per SM: what it takes is
// instructions (eight cycles each with nothing to overlap them) and, where a load
// waits behind a store that may alias it, memory round trips.  So the
// factorisation carries the forward sweep of the first solve with it, the sweeps
// walk pointers in unpredicated chunks whose loads are issued a chunk ahead, and
// the norm is formed in the backward sweep and applied by the next solve (700 +
// 300 states: 1.84 ms with a pass each for start, norm and scaling, 1.10 ms).
struct TriCol {
  double2* U;
  double* L;
  double* Y;
};
__device__ __forceinline__ double pack_piv(double l, bool piv) {
  return __longlong_as_double((__double_as_longlong(l) & ~1ll) | (long long)piv);
}
__device__ __forceinline__ bool piv_of(double l) { return (__double2loint(l) & 1) != 0; }

// LU factors with partial pivoting of T - lam I (one reciprocal per row; a zero
// pivot is replaced by pert), and y <- L^{-1} P (start vector k).
__device__ __forceinline__ void tri_factor(const double* __restrict__ d, const double* __restrict__ e,
                                           TriCol c, int n, int k, double lam, double pert) {
  const size_t sn = (size_t)n;
  double cur0 = __ldg(d) - lam, cur1 = n > 1 ? __ldg(e) : 0.0;
  double rc = start_entry((unsigned long long)k, 0);
  double sub = cur1;
#pragma unroll 2
  for (int i = 0; i < n - 1; ++i) {
    const double nd = __ldg(d + i + 1) - lam;
    const double nsup = i + 1 < n - 1 ? __ldg(e + i + 1) : 0.0;
    const bool piv = fabs(sub) > fabs(cur0);
    const double c0 = cur0 == 0.0 ? pert : cur0;
    const double r = 1.0 / (piv ? sub : c0);
    const double l = (piv ? cur0 : sub) * r;
    const double lv = pack_piv(l, piv);
    const double rn = start_entry((unsigned long long)k, (unsigned long long)(i + 1));
    *c.U = make_double2(r, piv ? nd : cur1);
    *c.L = lv;
    *c.Y = piv ? rn : rc;
    rc = piv ? fma(-lv, rn, rc) : fma(-lv, rc, rn);
    c.U += sn;
    c.L += sn;
    c.Y += sn;
    cur0 = piv ? fma(-l, nd, cur1) : fma(-l, cur1, nd);
    cur1 = piv ? -l * nsup : nsup;
    sub = nsup;
  }
  c.U->x = 1.0 / (cur0 == 0.0 ? pert : cur0);
  *c.Y = rc;
}

constexpr int kSolveRows = 8;
// y <- L^{-1} P (scale y).
__device__ __forceinline__ void tri_forward(const TriCol& c, int n, double scale) {
  constexpr int C = kSolveRows;
  const size_t sn = (size_t)n;
  double rc = scale * *c.Y;
  const double* __restrict__ L = c.L;
  const double* R = c.Y + sn;   // row i + 1
  double* W = c.Y;
  auto row = [&](double lv, double r0) {
    const double rn = scale * r0;
    const bool piv = piv_of(lv);
    *W = piv ? rn : rc;
    rc = piv ? fma(-lv, rn, rc) : fma(-lv, rc, rn);
    W += sn;
  };
  int left = n - 1;
  double lv[C], rn[C];
  auto load = [&]() {
#pragma unroll
    for (int q = 0; q < C; ++q) {
      lv[q] = *L;
      rn[q] = *R;
      L += sn;
      R += sn;
    }
  };
  if (left >= C) load();
  while (left >= C) {
    double l2[C], r2[C];
#pragma unroll
    for (int q = 0; q < C; ++q) {
      l2[q] = lv[q];
      r2[q] = rn[q];
    }
    if (left >= 2 * C) load();
#pragma unroll
    for (int q = 0; q < C; ++q) row(l2[q], r2[q]);
    left -= C;
  }
  for (; left > 0; --left, L += sn, R += sn) row(*L, *R);
  *W = rc;
}
// y <- U^{-1} y; returns the sum of squares of the result.
__device__ __forceinline__ double tri_backward(const TriCol& c, const double* __restrict__ e, int n) {
  constexpr int C = kSolveRows;
  const size_t sn = (size_t)n;
  const double2* __restrict__ U = c.U + (size_t)(n - 1) * sn;
  const double* __restrict__ L = c.L + (size_t)(n - 1) * sn;
  const double* R = c.Y + (size_t)(n - 1) * sn;
  double* W = c.Y + (size_t)(n - 1) * sn;
  double y1 = 0.0, y2 = 0.0, s0 = 0.0, s1 = 0.0;   // y[i+1], y[i+2]
  auto row = [&](double y, double r, double u1, double u2) {
    const double yi = fma(-u1, y1, fma(-u2, y2, y)) * r;
    *W = yi;
    W -= sn;
    y2 = y1;
    y1 = yi;
  };
  // the last two rows have no second, the last no first superdiagonal (those
  // entries are never formed)
  row(*R, U->x, 0.0, 0.0);
  s0 = y1 * y1;
  if (n == 1) return s0;
  U -= sn;
  L -= sn;
  R -= sn;
  row(*R, U->x, U->y, 0.0);
  s1 = y1 * y1;
  U -= sn;
  L -= sn;
  R -= sn;
  int i = n - 3;
  double yy[C], u2[C];
  double2 u[C];
  auto load = [&](int top) {
#pragma unroll
    for (int q = 0; q < C; ++q) {
      yy[q] = *R;
      u[q] = *U;
      u2[q] = piv_of(*L) ? __ldg(e + top - q + 1) : 0.0;
      R -= sn;
      U -= sn;
      L -= sn;
    }
  };
  if (i + 1 >= C) load(i);
  while (i + 1 >= C) {
    double ya[C], ua[C];
    double2 va[C];
#pragma unroll
    for (int q = 0; q < C; ++q) {
      ya[q] = yy[q];
      ua[q] = u2[q];
      va[q] = u[q];
    }
    if (i + 1 >= 2 * C) load(i - C);
#pragma unroll
    for (int q = 0; q < C; ++q) {
      row(ya[q], va[q].x, va[q].y, ua[q]);
      if (q & 1) s1 = fma(y1, y1, s1);
      else s0 = fma(y1, y1, s0);
    }
    i -= C;
  }
  for (; i >= 0; --i, R -= sn, U -= sn, L -= sn) {
    row(*R, U->x, U->y, piv_of(*L) ? __ldg(e + i + 1) : 0.0);
    s0 = fma(y1, y1, s0);
  }
  return s0 + s1;
}

// One thread per eigenvalue; the first of a cluster does the whole cluster.
// Blocks of kVecThreads spread the serial work over the SMs.
__global__ void __launch_bounds__(kVecThreads, 1) k_tri_vectors(TriBatch a) {
  const int item = blockIdx.x * kVecThreads + threadIdx.x;
  if (item >= a.off[a.np]) return;
  const int b = find_prob(a.off, a.np, item);
  if (!tri_run(a, b)) return;
  const int n = a.n[b], j = item - a.off[b];
  const TriPtrs p = tri_ptrs(a, b);
  const double* lam = p.lam;
  const double nrm = fmax(fmax(fabs(lam[0]), fabs(lam[n - 1])), 1e-300);
  const double tight = kTightRel * nrm;
  if (j > 0 && lam[j] - lam[j - 1] <= tight) return;   // not the first of its cluster
  int end = j + 1;
  while (end < n && lam[end] - lam[end - 1] <= tight) ++end;
  const double pert = kEps * nrm;
  const size_t sn = (size_t)n;
  double* Y = p.Y;
  for (int k = j; k < end; ++k) {
    const TriCol col{reinterpret_cast<double2*>(p.U0) + k, p.U2 + k, Y + k};
    tri_factor(p.d, p.e, col, n, k, lam[k], pert);
    double r = 1.0;                          // scale of the next solve's right-hand side
    for (int it = 0; it < kInvIters; ++it) {
      if (it > 0) tri_forward(col, n, r);
      double sq = tri_backward(col, p.e, n);
      for (int c = j; c < k; ++c) {          // against the cluster's earlier vectors
        double dot = 0.0;
        for (int i = 0; i < n; ++i) dot = fma(Y[(size_t)i * sn + c], Y[(size_t)i * sn + k], dot);
        for (int i = 0; i < n; ++i) Y[(size_t)i * sn + k] = fma(-dot, Y[(size_t)i * sn + c], Y[(size_t)i * sn + k]);
      }
      if (k > j) {
        sq = 0.0;
        for (int i = 0; i < n; ++i) sq = fma(Y[(size_t)i * sn + k], Y[(size_t)i * sn + k], sq);
      }
      double s = sqrt(sq);
      if (!(s > 0.0) || !isfinite(s)) {
        flag_status(a.status, SKY_ENOCONV);
        s = 1.0;
      }
      r = 1.0 / s;
    }
    for (int i0 = 0; i0 < n; i0 += 16) {     // the unit vector
      double y[16];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (i0 + c < n) y[c] = Y[(size_t)(i0 + c) * sn + k];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if (i0 + c < n) Y[(size_t)(i0 + c) * sn + k] = y[c] * r;
    }
  }
}

// One first-order Loewdin step on the columns of Y within each eigenvalue's
// window: Yout[:, j] = Yin[:, j] (3 - G_jj)/2 - sum_{k != j} G_kj Yin[:, k] / 2.
__global__ void __launch_bounds__(kWinThreads) k_tri_window(TriBatch a, int pass) {
  __shared__ double gpart[kWinThreads / 32][2 * kWinMax + 1];
  __shared__ double coef[2 * kWinMax + 1];
  const int item = blockIdx.x;
  const int b = find_prob(a.off, a.np, item);
  if (!tri_run(a, b)) return;
  const int n = a.n[b], j = item - a.off[b];
  const TriPtrs p = tri_ptrs(a, b);
  const double* Yin = pass ? p.Y2 : p.Y;
  double* Yout = pass ? p.Y : p.Y2;
  const double* lam = p.lam;
  const double gw = kWinRel * fmax(fabs(lam[0]), fabs(lam[n - 1]));
  int lo = j, hi = j;
  while (lo > 0 && j - lo < kWinMax && lam[j] - lam[lo - 1] <= gw) --lo;
  while (hi < n - 1 && hi - j < kWinMax && lam[hi + 1] - lam[j] <= gw) ++hi;
  const int K = hi - lo + 1;
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const size_t sn = (size_t)n;
  double acc[kWinChunks];
#pragma unroll
  for (int c = 0; c < kWinChunks; ++c) acc[c] = 0.0;
  for (int i = wq; i < n; i += kWinThreads / 32) {
    const double* row = Yin + (size_t)i * sn;
    const double yj = row[j];
#pragma unroll
    for (int c = 0; c < kWinChunks; ++c) {
      const int t = lane + 32 * c;
      if (t < K) acc[c] = fma(row[lo + t], yj, acc[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < kWinChunks; ++c) {
    const int t = lane + 32 * c;
    if (t < K) gpart[wq][t] = acc[c];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < K; t += kWinThreads) {
    double g = gpart[0][t];
    for (int q = 1; q < kWinThreads / 32; ++q) g += gpart[q][t];
    coef[t] = (lo + t == j) ? 1.5 - 0.5 * g : -0.5 * g;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kWinThreads) {
    const double* row = Yin + (size_t)i * sn + lo;
    double s = 0.0;
    for (int t = 0; t < K; ++t) s = fma(coef[t], row[t], s);
    Yout[(size_t)i * sn + j] = s;
  }
}

// ---- back-transformation: Z = H_0 H_1 ... H_{n-2} Y, one warp per column ----------
__global__ void __launch_bounds__(kBackWarps * 32) k_hh_back(TriBatch a, int zstride) {
  extern __shared__ double2 dsm[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double2* z = dsm + (size_t)wid * zstride;
  const int nw = gridDim.x * (blockDim.x >> 5);
  const int total = a.off[a.np];
  for (int it = wid * gridDim.x + blockIdx.x; it < total; it += nw) {
    const int b = find_prob(a.off, a.np, it);
    if (!tri_run(a, b)) continue;
    const int n = a.n[b], col = it - a.off[b];
    const TriPtrs p = tri_ptrs(a, b);
    for (int i = lane; i < n; i += 32) z[i] = make_double2(p.Y[(size_t)i * n + col], 0.0);
    for (int k = n - 2; k >= 0; --k) {
      const double2 tau = p.tau[k];
      if (tau.x == 0.0 && tau.y == 0.0) continue;
      const double2* v = p.V + (size_t)k * n;
      const int i0 = ((k + 1) >> 5) * 32 + lane;
      double sx = 0.0, sy = 0.0;
      for (int i = i0; i < n; i += 32) {
        if (i <= k) continue;
        const double2 vi = v[i], zi = z[i];
        sx = fma(vi.x, zi.x, fma(vi.y, zi.y, sx));     // conj(v) z
        sy = fma(vi.x, zi.y, fma(-vi.y, zi.x, sy));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
      }
      const double2 f = cmul(tau, make_double2(sx, sy));
      for (int i = i0; i < n; i += 32) {
        if (i <= k) continue;
        const double2 vi = v[i];
        double2 zi = z[i];
        zi.x = fma(-vi.x, f.x, fma(vi.y, f.y, zi.x));     // z -= v f
        zi.y = fma(-vi.x, f.y, fma(-vi.y, f.x, zi.y));
        z[i] = zi;
      }
    }
    double2* Z = a.Z[b];
    for (int i = lane; i < n; i += 32) Z[(size_t)i * n + col] = z[i];
    __syncwarp();
  }
}

// ---- back-transformation by the compact WY form ----------------------------------
// Q = H_0 ... H_{n-2} = I - V T V^H with V's columns v_t and T upper triangular,
// T^{-1} = striu(V^H V) + diag(1 / tau_t) (Puglisi 1992; a reflector with tau_t = 0
// enters as v_t = 0).  With P = V^H:  G = P P^H; T's diagonal blocks of kWyBlock by
// back substitution; then T's blocks doubled in size level by level, the upper
// right block of a pair being -T_11 G_12 T_22, which the full products (T G) T
// hold in that place because T is block diagonal so far; Z = Y - P^H (T (P Y)).
// All products are digit-split tensor-core ones with seven digits (4 + 2 log2(n /
// kWyBlock) of them); applying the reflectors one by one costs 4 n^3 FP64 multiply-adds,
// which bound k_hh_back (72% of the FP64 pipe): 700 + 300 states 4.1 ms, here
// 1.4 ms; 280 + 120 states 0.93 ms, here 0.55 ms.  The eigenvectors' orthogonality
// and residuals stay what they were (128 to 1000 states, dense and nearly diagonal
// matrices: 6e-15 to 6e-14 sqrt(n), both ways).
constexpr int kWyBlock = 64;
// It is used from kWyMin states on (one diagonalisation, reflectors one by one and
// compact WY: 160 states 2.13 and 2.17 ms, 192 2.60 and 2.58, 256 3.51 and 3.21), and
// from kWyManyMin states on in batches of kWyMany states in all (6 of 128: 2.79 and
// 2.82 ms, 12 of 128: 2.32 and 2.26 ms).
constexpr int kWyMin = 192, kWyManyMin = 128, kWyMany = 1536;

struct WyJobs {
  double2* P[kMaxBatch];               // in: row t = v_t; out: row t = v_t^H
  const double2* tau[kMaxBatch];
  const double* Y[kMaxBatch];
  double2* Z[kMaxBatch];               // Y as a complex matrix, later the result
  const double2* G[kMaxBatch];
  double2* T[kMaxBatch];
  const double2* N[kMaxBatch];         // (T G) T of a level, or P^H X at the end
  int n[kMaxBatch];
};
// Row t (blockIdx.x) of P and of Y as complex values.
__global__ void __launch_bounds__(256) k_wy_prep(const __grid_constant__ WyJobs j) {
  const int b = blockIdx.y, n = j.n[b], t = blockIdx.x;
  if (t >= n) return;
  double2 tau = make_double2(0.0, 0.0);
  if (t < n - 1) tau = j.tau[b][t];
  const bool on = tau.x != 0.0 || tau.y != 0.0;
  const long long r = (long long)t * n;
  for (int i = threadIdx.x; i < n; i += 256) {
    // entries up to t are not part of the reflector (never written)
    j.P[b][r + i] = on && i > t ? conjx(j.P[b][r + i]) : make_double2(0.0, 0.0);
    j.Z[b][r + i] = make_double2(j.Y[b][r + i], 0.0);
  }
}
// Diagonal block blockIdx.x of T, columns kWyCols blockIdx.z .. of it: the inverse
// of the block of striu(G) + diag(1 / tau) by back substitution, and zeros in the
// rest of its rows (its share of them).  A warp per column, lane l with rows l and
// l + 32: as x_k is known every row above takes its term, so a step is one shuffle
// and one multiply-add deep; with the rows scaled by -tau_i beforehand the sum of
// row i is x_i.  FP64 instructions bound it (127 us at 700 + 300 states with the row
// sums split over 16 threads and added up row by row).
constexpr int kWyCols = 8, kWyThreads = 32 * kWyCols;
static_assert(kWyBlock == 64, "two rows per lane");
__global__ void __launch_bounds__(kWyThreads) k_wy_diag(const __grid_constant__ WyJobs j) {
  extern __shared__ double2 wsm[];
  constexpr int B = kWyBlock, LD = kWyBlock + 1;
  double2* m = wsm;                     // [B][LD] -tau_i G_ik
  double2* dg = wsm + B * LD;           // [B] tau (1 / the diagonal)
  const int b = blockIdx.y, n = j.n[b], k0 = blockIdx.x * B;
  if (k0 >= n) return;
  const int nb = n - k0 < B ? n - k0 : B;
  for (int i = threadIdx.x; i < B; i += kWyThreads) {
    double2 t = make_double2(1.0, 0.0);
    if (k0 + i < n - 1) {
      const double2 u = j.tau[b][k0 + i];
      if (u.x != 0.0 || u.y != 0.0) t = u;
    }
    dg[i] = t;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < B * B; e += kWyThreads) {
    const int i = e / B, c = e % B;
    const bool on = i < c && c < nb;
    m[i * LD + c] = on ? -cmul(dg[i], j.G[b][(long long)(k0 + i) * n + k0 + c]) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, c = blockIdx.z * kWyCols + (threadIdx.x >> 5);
  if (c < nb) {
    // x0, x1: rows lane and lane + 32 of column c (rows beyond c stay zero)
    double2 x0 = make_double2(0.0, 0.0), x1 = x0;
    if (lane == (c & 31)) (c < 32 ? x0 : x1) = dg[c];
    for (int k = c; k > 0; --k) {
      const double2 s = k < 32 ? x0 : x1;
      const double2 v = make_double2(__shfl_sync(0xffffffffu, s.x, k & 31), __shfl_sync(0xffffffffu, s.y, k & 31));
      const double2 a0 = m[lane * LD + k];
      x0.x = fma(a0.x, v.x, x0.x);
      x0.y = fma(a0.x, v.y, x0.y);
      x0.x = fma(-a0.y, v.y, x0.x);
      x0.y = fma(a0.y, v.x, x0.y);
      if (k > 32) {
        const double2 a1 = m[(lane + 32) * LD + k];
        x1.x = fma(a1.x, v.x, x1.x);
        x1.y = fma(a1.x, v.y, x1.y);
        x1.x = fma(-a1.y, v.y, x1.x);
        x1.y = fma(a1.y, v.x, x1.y);
      }
    }
    double2* t = j.T[b] + (long long)k0 * n + k0 + c;
    if (lane < nb) t[(long long)lane * n] = x0;
    if (lane + 32 < nb) t[(long long)(lane + 32) * n] = x1;
  }
  // every gridDim.z-th row outside the diagonal block
  for (int i = blockIdx.z; i < nb; i += gridDim.z)
    for (int e = threadIdx.x; e < n; e += kWyThreads)
      if (e < k0 || e >= k0 + nb) j.T[b][(long long)(k0 + i) * n + e] = make_double2(0.0, 0.0);
}
constexpr size_t kWySmem = ((size_t)kWyBlock * (kWyBlock + 1) + kWyBlock) * sizeof(double2);
// T's upper right blocks of the pairs of blocks of s rows: -(T G) T there.
__global__ void __launch_bounds__(256) k_wy_level(const __grid_constant__ WyJobs j, int s) {
  const int b = blockIdx.y, n = j.n[b], i = blockIdx.x;
  if (i >= n || ((i / s) & 1)) return;
  const int c0 = (i / s + 1) * s, c1 = c0 + s < n ? c0 + s : n;
  const long long r = (long long)i * n;
  for (int c = c0 + threadIdx.x; c < c1; c += 256) j.T[b][r + c] = -j.N[b][r + c];
}
// Z = Y - P^H X.
__global__ void __launch_bounds__(256) k_wy_final(const __grid_constant__ WyJobs j) {
  const int b = blockIdx.y, n = j.n[b], i = blockIdx.x;
  if (i >= n) return;
  const long long r = (long long)i * n;
  for (int c = threadIdx.x; c < n; c += 256) j.Z[b][r + c] = j.Z[b][r + c] - j.N[b][r + c];
}

// Z = Q Y for the problems idx[0..np) of a batch.  Workspace: the tridiagonal
// solver's three slots (own columns and LU rows: done; reflectors: P in place; Y:
// done once it is copied) and two of the callers' I x I temporaries (4 and 5,
// which no caller holds across an eigensolve).
static sky_status wy_back(Ctx* c, int np, const int* idx, const int* n, double2* const* Z,
                          const TriBatch& a) {
  WyJobs j;
  double2 *S0[kMaxBatch], *S2[kMaxBatch], *U[kMaxBatch], *T[kMaxBatch], *P[kMaxBatch], *Zb[kMaxBatch];
  int nn[kMaxBatch], nmax = 1;
  for (int q = 0; q < np; ++q) {
    const int b = idx[q];
    nn[q] = n[b];
    nmax = n[b] > nmax ? n[b] : nmax;
    S0[q] = c->d_eigA[0] + (size_t)b * c->eig_slot;
    P[q] = c->d_eigA[1] + (size_t)b * c->eig_slot;
    S2[q] = c->d_eigV + (size_t)b * c->eig_slot;
    U[q] = c->d_small[4] + (size_t)b * c->small_slot;
    T[q] = c->d_small[5] + (size_t)b * c->small_slot;
    Zb[q] = Z[b];
    j.P[q] = P[q];
    j.tau[q] = reinterpret_cast<const double2*>(a.T + (size_t)b * a.tslot + (size_t)a.m * a.m) + 2 * kTriBufs * (size_t)a.m;
    j.Y[q] = reinterpret_cast<const double*>(S2[q]);
    j.Z[q] = Zb[q];
    j.G[q] = S0[q];
    j.T[q] = T[q];
    j.N[q] = S2[q];
    j.n[q] = n[b];
  }
  const int* none[kMaxBatch] = {nullptr};
  const dim3 rows(nmax, np);
  auto mul = [&](bool ah, bool bh, double2* const* A, double2* const* B, double2* const* C) {
    return zgemm_batch(c, zjobs(np, ah, bh, (const double2* const*)A, (const double2* const*)B, C, nn, none, none, 7));
  };
  k_wy_prep<<<rows, 256, 0, c->stream>>>(j);
  sky_status s = mul(false, true, P, P, S0);                       // G = P P^H
  if (s != SKY_OK) return s;
  k_wy_diag<<<dim3(div_up(nmax, kWyBlock), np, kWyBlock / kWyCols), kWyThreads, kWySmem, c->stream>>>(j);
  note_launch(2);
  for (int w = kWyBlock; w < nmax; w *= 2) {
    if ((s = mul(false, false, T, S0, U)) != SKY_OK) return s;     // T G
    if ((s = mul(false, false, U, T, S2)) != SKY_OK) return s;     // (T G) T
    k_wy_level<<<rows, 256, 0, c->stream>>>(j, w);
    note_launch();
  }
  if ((s = mul(false, false, P, Zb, U)) != SKY_OK) return s;       // P Y
  if ((s = mul(false, false, T, U, S2)) != SKY_OK) return s;       // T (P Y)
  if ((s = mul(true, false, P, S2, S0)) != SKY_OK) return s;       // P^H X
  for (int q = 0; q < np; ++q) j.N[q] = S0[q];
  k_wy_final<<<rows, 256, 0, c->stream>>>(j);
  note_launch();
  return cuda_check(c, cudaGetLastError(), "back-transformation");
}

__global__ void k_tri_reset(unsigned* bar) { bar[(size_t)kTeamBarStride * threadIdx.x] = 0u; }

// A problem of n states keeps its work vectors in global memory when they
// alone (with the per-column partials) exceed the shared-memory budget.
bool tri_vectors_global(int n) {
  return (3 * (size_t)n + (n + 1) / 2 + 1) * sizeof(double2) > kTriSmemMax;
}

// double2 elements of the global work vectors for the problems of a batch
// of nb problems of up to m states on nsm blocks: needed when one problem,
// or the tridiagonal route's largest batch (8 problems) of them, does not fit
// in shared memory (0 otherwise).
size_t tri_vec_elems(int m, int nb, int nsm) {
  const int k = nb < 8 ? nb : 8;
  const size_t one = (3 * (size_t)m + (m + 1) / 2 + 1) * sizeof(double2);
  return (tri_vectors_global(m) || k * one > kTriSmemMax) ? (size_t)k * nsm * 3 * (size_t)m : 0;
}

// Shared-memory opt-in of the two kernels that take more than 48 KB (once per
// context, outside any stream capture).
sky_status tri_init(Ctx* c) {
  cudaError_t e = cudaFuncSetAttribute(k_hh_tridiag, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kTriSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hh_back, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTriSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wy_diag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWySmem);
  return cuda_check(c, e, "tridiagonal solver attributes");
}

// ---- teams of blocks for batches of many problems ----------------------------------
// With one team, every block takes part in every problem's steps and the
// slowest problem sets the pace of all: n_max steps, each with the head work
// of every problem.  A batch of more than kTeamMin problems (the many boxes of
// twist-averaged runs) is split instead: a problem whose work needs several
// blocks gets a team of its own, smaller ones share one-block teams (no
// barrier at all), each team stepping at its own pace.  The split minimises
// the largest estimated team time
//   steps x (per-step latency) + sum over its problems of 4 n^3 FMAs / rate,
// by bisection on the time target: problems are taken largest first, teams
// of several blocks sized to the target, the rest packed first-fit into
// one-block teams whose work vectors fit in shared memory.
constexpr int kTeamMin = 8;
constexpr double kTeamFma = 3.4e9;      // FP64 FMAs per second of one block (one per SM)
constexpr double kTeamStep1 = 1.5e-6;   // seconds per step of a one-block team
constexpr double kTeamStepG = 5.0e-6;   // seconds per step of a team with a barrier
constexpr double kTeamHead = 1.0e-6;    // per step and further group of kHeadGroups problems
constexpr int kTeamMinCols = 4;         // own columns per block of a team at least

struct TeamPlan {
  int nteam;
  int mem[kMaxBatch];
  int p0[kMaxBatch + 1];
  int g0[kMaxBatch + 1];
};

static double team_work(int n) { return 4.0 * (double)n * n * n / kTeamFma; }
static size_t team_vec(int n) { return 3 * (size_t)n + (size_t)(n + 1) / 2 + 1; }   // double2

// Estimated time of a team of g blocks for problems mem[k0 .. k1).
static double team_time(const int* n, const int* mem, int k0, int k1, int g) {
  int nmax = 0;
  double w = 0.0;
  for (int k = k0; k < k1; ++k) {
    nmax = n[mem[k]] > nmax ? n[mem[k]] : nmax;
    w += team_work(n[mem[k]]);
  }
  const int groups = (k1 - k0 + kHeadGroups - 1) / kHeadGroups;
  const double step = (g > 1 ? kTeamStepG : kTeamStep1) + kTeamHead * (groups - 1);
  return nmax * step + w / g;
}

// Teams for the target time T (problems in `order`, largest first); returns
// the blocks used, or a number above `blocks` when T cannot be met.
static int plan_at(int np, const int* n, const int* order, double T, size_t budget, TeamPlan& p) {
  int used = 0, k = 0;
  p.nteam = 0;
  bool packed[kMaxBatch];
  for (int i = 0; i < np; ++i) {
    const int b = order[i];
    packed[b] = team_work(n[b]) + n[b] * kTeamStep1 <= T;
    if (packed[b]) continue;
    const double room = T - n[b] * kTeamStepG;
    const int gmax = n[b] / kTeamMinCols > 2 ? n[b] / kTeamMinCols : 2;
    if (room <= 0.0) return 1 << 30;
    const double gf = team_work(n[b]) / room;
    if (gf > gmax) return 1 << 30;
    int g = (int)std::ceil(gf);
    g = g < 2 ? 2 : g;
    p.p0[p.nteam] = k;
    p.g0[p.nteam] = used;
    p.mem[k++] = b;
    used += g;
    ++p.nteam;
  }
  // first fit, largest first, into one-block teams
  int bin_of[kMaxBatch], nbin = 0;
  double bw[kMaxBatch];
  int bn[kMaxBatch], bk[kMaxBatch];
  size_t bv[kMaxBatch];
  for (int i = 0; i < np; ++i) {
    const int b = order[i];
    if (!packed[b]) continue;
    int f = -1;
    for (int q = 0; q < nbin && f < 0; ++q) {
      const int groups = (bk[q] + 1 + kHeadGroups - 1) / kHeadGroups;
      const double t = bn[q] * (kTeamStep1 + kTeamHead * (groups - 1)) + bw[q] + team_work(n[b]);
      if (t <= T && bv[q] + team_vec(n[b]) <= budget) f = q;
    }
    if (f < 0) {
      if (team_vec(n[b]) > budget) return 1 << 30;
      f = nbin++;
      bw[f] = 0.0; bn[f] = n[b]; bk[f] = 0; bv[f] = 0;
    }
    bw[f] += team_work(n[b]);
    bk[f] += 1;
    bv[f] += team_vec(n[b]);
    bin_of[b] = f;
  }
  for (int q = 0; q < nbin; ++q) {
    p.p0[p.nteam] = k;
    p.g0[p.nteam] = used++;
    for (int i = 0; i < np; ++i)
      if (packed[order[i]] && bin_of[order[i]] == q) p.mem[k++] = order[i];
    ++p.nteam;
  }
  p.p0[p.nteam] = k;
  p.g0[p.nteam] = used;
  return used;
}

// The team split of np problems over `blocks` blocks (false if none fits).
static bool plan_teams(int np, const int* n, int blocks, size_t budget, TeamPlan& p) {
  int order[kMaxBatch];
  for (int b = 0; b < np; ++b) order[b] = b;
  std::sort(order, order + np, [&](int x, int y) { return n[x] != n[y] ? n[x] > n[y] : x < y; });
  // an upper time bound that fits (1 s covers the usual batches on a full GPU;
  // larger batches on fewer blocks need longer), then bisection
  double hi = 1.0, lo = 0.0;
  while (plan_at(np, n, order, hi, budget, p) > blocks) {
    lo = hi;
    hi *= 2.0;
    if (hi > 1e7) return false;   // no split fits (shared memory bounds the packing)
  }
  for (int it = 0; it < 48; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (plan_at(np, n, order, mid, budget, p) <= blocks) hi = mid; else lo = mid;
  }
  int used = plan_at(np, n, order, hi, budget, p);
  // spare blocks to the slowest single-problem teams
  while (used < blocks) {
    int best = -1;
    double bt = 0.0;
    for (int t = 0; t < p.nteam; ++t) {
      const int g = p.g0[t + 1] - p.g0[t];
      if (p.p0[t + 1] - p.p0[t] != 1 || g + 1 > n[p.mem[p.p0[t]]] / kTeamMinCols) continue;
      const double tt = team_time(n, p.mem, p.p0[t], p.p0[t + 1], g);
      if (tt > bt) { bt = tt; best = t; }
    }
    if (best < 0) break;
    for (int t = best + 1; t <= p.nteam; ++t) p.g0[t] += 1;
    ++used;
  }
  return true;
}

// The team split of a batch on `blocks` blocks for callers (sky_tri_team_plan):
// the number of teams, 0 if it cannot be split.
int tri_team_plan(int np, const int* n, int blocks, int* team, int* first, int* count) {
  if (np < 1 || np > kMaxBatch || blocks < 1 || !n || !team || !first || !count) return 0;
  for (int b = 0; b < np; ++b)
    if (n[b] < 1 || tri_vectors_global(n[b])) return 0;
  TeamPlan tp;
  if (!plan_teams(np, n, blocks, kTriSmemMax / sizeof(double2) - 64, tp)) return 0;
  for (int t = 0; t < tp.nteam; ++t) {
    first[t] = tp.g0[t];
    count[t] = tp.g0[t + 1] - tp.g0[t];
    for (int k = tp.p0[t]; k < tp.p0[t + 1]; ++k) team[tp.mem[k]] = t;
  }
  return tp.nteam;
}

// One launch sequence for the problems idx[0..np) of a batch (their vectors fit).
static sky_status tri_group(Ctx* c, int np, const int* idx, const double2* const* A, const int* n,
                            double* const* w, double2* const* Z, const int* run, int run_stride,
                            const bool* gvec) {
  TriBatch a;
  a.np = np;
  a.off[0] = 0;
  long long ntot = 0;
  int nmax = 1;
  for (int q = 0; q < np; ++q) {
    const int b = idx[q];
    a.A[q] = A[b]; a.w[q] = w[b]; a.Z[q] = Z[b]; a.n[q] = n[b]; a.sid[q] = b;
    a.off[q + 1] = a.off[q] + n[b];
    ntot += n[b];
    if (n[b] > nmax) nmax = n[b];
  }
  if (ntot == 0) return SKY_OK;
  int G = (int)(ntot < c->num_sms ? ntot : c->num_sms);
  size_t used = 0;
  a.gvec = c->d_trivec;
  a.gvec_stride = 3 * (size_t)c->tri_m;
  if (np > kTeamMin) {
    // teams: the per-column partials first (one region for every team), then
    // each team's work vectors and own columns while they fit
    TeamPlan tp;
    const size_t budget = kTriSmemMax / sizeof(double2);
    G = c->num_sms;
    if (!plan_teams(np, a.n, G, budget - 64, tp)) return SKY_EUNSUPPORTED;
    G = tp.g0[tp.nteam];
    a.nteam = tp.nteam;
    size_t cmax = 0;
    for (int t = 0; t <= tp.nteam; ++t) {
      a.tp0[t] = tp.p0[t];
      a.tg0[t] = tp.g0[t];
    }
    for (int k = 0; k < np; ++k) a.tmem[k] = tp.mem[k];
    for (int t = 0; t < tp.nteam; ++t) {
      const int g = tp.g0[t + 1] - tp.g0[t];
      size_t own = 0;
      for (int k = tp.p0[t]; k < tp.p0[t + 1]; ++k) own += (a.n[tp.mem[k]] + g - 1) / g;
      cmax = own > cmax ? own : cmax;
    }
    a.coff = 0;
    const size_t base = (cmax + 1) / 2 + 1;
    used = base;
    for (int t = 0; t < tp.nteam; ++t) {
      const int g = tp.g0[t + 1] - tp.g0[t];
      size_t u = base;
      for (int k = tp.p0[t]; k < tp.p0[t + 1]; ++k) {
        const int q = tp.mem[k];
        if (gvec[idx[q]]) return SKY_EUNSUPPORTED;
        a.voff[q] = (int)u;
        u += 3 * (size_t)a.n[q];
        a.rot[q] = 0;
      }
      if (u > budget) return SKY_EUNSUPPORTED;
      for (int k = tp.p0[t]; k < tp.p0[t + 1]; ++k) {
        const int q = tp.mem[k];
        const size_t need = (size_t)((a.n[q] + g - 1) / g) * a.n[q];
        if (u + need <= budget) {
          a.soff[q] = (int)u;
          u += need;
        } else {
          a.soff[q] = -1;
        }
      }
      used = u > used ? u : used;
    }
    a.tbar = c->d_tbar;
  } else {
    // one team of all blocks.  Shared memory: three work vectors per problem
    // (in global memory for a problem whose vectors alone exceed it), then own
    // columns while they fit
    int maxown = 0;
    for (int q = 0; q < np; ++q) {
      if (gvec[idx[q]]) {
        a.voff[q] = -1;
      } else {
        a.voff[q] = (int)used;
        used += 3 * (size_t)a.n[q];
      }
      maxown += (a.n[q] + G - 1) / G;
    }
    a.coff = (int)used;
    used += (size_t)(maxown + 1) / 2;
    int rot = 0;
    for (int q = 0; q < np; ++q) {
      const size_t need = (size_t)((a.n[q] + G - 1) / G) * a.n[q];
      if ((used + need) * sizeof(double2) <= kTriSmemMax) {
        a.soff[q] = (int)used;
        used += need;
      } else {
        a.soff[q] = -1;
      }
      a.rot[q] = rot;
      rot = (rot + a.n[q]) % G;
    }
    a.nteam = 1;
    a.tp0[0] = 0; a.tp0[1] = np;
    a.tg0[0] = 0; a.tg0[1] = G;
    for (int q = 0; q < np; ++q) a.tmem[q] = q;
    a.tbar = c->d_bar;
  }
  const int zstride = nmax + (nmax & 1);
  int back_warps = kBackWarps;
  while (back_warps > 1 && (size_t)back_warps * zstride * sizeof(double2) > kTriSmemMax) back_warps >>= 1;
  a.S0 = c->d_eigA[0]; a.S1 = c->d_eigA[1]; a.S2 = c->d_eigV; a.slot = c->eig_slot;
  a.T = c->d_trid; a.tslot = c->tri_slot; a.m = c->tri_m;
  a.sp = c->d_eigpart; a.sp_stride = (size_t)kTriBufs * c->eig_grid_max;
  a.run = run; a.run_stride = run_stride;
  a.status = c->d_status; a.spins = c->wait_spins; a.stats = c->d_stats;
  // run flags are indexed by the batch position of each problem
  if (run) {
    bool ident = true;
    for (int q = 0; q < np; ++q) ident = ident && idx[q] == q;
    if (!ident) return SKY_EUNSUPPORTED;
  }
  cudaError_t e;
  k_tri_reset<<<1, a.nteam, 0, c->stream>>>(a.tbar);
  note_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_check(c, e, "tridiagonal reset");
  void* args[] = {&a};
  note_launch();
  e = cudaLaunchCooperativeKernel((const void*)k_hh_tridiag, dim3(G), dim3(kTriThreads), args,
                                  used * sizeof(double2), c->stream);
  if (e != cudaSuccess) return cuda_check(c, e, "householder tridiagonalisation");
  k_hh_scale<<<dim3(nmax, np), 128, 0, c->stream>>>(a);
  k_tri_bisect<<<(unsigned)ntot, 32, 0, c->stream>>>(a);
  k_tri_vectors<<<div_up(ntot, kVecThreads), kVecThreads, 0, c->stream>>>(a);
  k_tri_window<<<(unsigned)ntot, kWinThreads, 0, c->stream>>>(a, 0);
  k_tri_window<<<(unsigned)ntot, kWinThreads, 0, c->stream>>>(a, 1);
  note_launch(5);
  // the products by tensor cores, unless the batch is gated (skipped products
  // still cost their launches) or its problems are small
  if (!run && (nmax >= kWyMin || (nmax >= kWyManyMin && ntot >= kWyMany))) {
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_check(c, e, "tridiagonal eigensolver");
    return wy_back(c, np, idx, n, Z, a);
  }
  // columns spread over all SMs first (consecutive items go to different blocks)
  const int back_blocks = (int)(ntot < c->num_sms ? ntot : c->num_sms);
  const int need_warps = (int)div_up(ntot, back_blocks);
  if (need_warps < back_warps) back_warps = need_warps;
  k_hh_back<<<back_blocks, back_warps * 32, (size_t)back_warps * zstride * sizeof(double2),
              c->stream>>>(a, zstride);
  note_launch();
  return cuda_check(c, cudaGetLastError(), "tridiagonal eigensolver");
}

// Eigendecomposition of np Hermitian matrices by the tridiagonal route, in
// groups whose work vectors fit in shared memory (problems of one group share
// every launch).  Returns SKY_EUNSUPPORTED, with nothing enqueued, when a
// single problem's vectors do not fit (or a device-gated batch would need more
// than one group); the caller then uses the Jacobi solver.
sky_status eigh_batch_tri(Ctx* c, int np, const double2* const* A, const int* n,
                          double* const* w, double2* const* Z, const int* run, int run_stride) {
  int groups[kMaxBatch + 1], order[kMaxBatch];
  bool gvec[kMaxBatch];
  int ng = 0;
  size_t used = 0;
  groups[0] = 0;
  if (np > kTeamMin) {
    // one launch sequence, the blocks split into teams (tri_group)
    for (int b = 0; b < np; ++b) {
      gvec[b] = false;
      order[b] = b;
      if (tri_vectors_global(n[b]) || n[b] > c->tri_m) return SKY_EUNSUPPORTED;
    }
    return tri_group(c, np, order, A, n, w, Z, run, run_stride, gvec);
  }
  // work vectors in global memory for problems too large for shared memory,
  // and, when the global buffer has room, for the largest problems until the
  // whole batch fits one launch sequence (a device-gated batch must: it
  // cannot be split)
  const bool room = c->d_trivec && np <= c->tri_vec_slots;
  size_t total = 0;
  for (int b = 0; b < np; ++b) {
    gvec[b] = tri_vectors_global(n[b]);
    total += ((gvec[b] ? 0 : 3 * (size_t)n[b]) + (n[b] + 1) / 2 + 1) * sizeof(double2);
  }
  while (room && total > kTriSmemMax) {
    int big = -1;
    for (int b = 0; b < np; ++b)
      if (!gvec[b] && (big < 0 || n[b] > n[big])) big = b;
    if (big < 0) break;
    gvec[big] = true;
    total -= 3 * (size_t)n[big] * sizeof(double2);
  }
  for (int b = 0; b < np; ++b) {
    const bool gv = gvec[b];
    if (gv && (!room || n[b] > c->tri_m)) return SKY_EUNSUPPORTED;
    const size_t need = ((gv ? 0 : 3 * (size_t)n[b]) + (n[b] + 1) / 2 + 1) * sizeof(double2);
    const size_t zneed = (size_t)(n[b] + (n[b] & 1)) * sizeof(double2);
    if (need > kTriSmemMax || zneed > kTriSmemMax) return SKY_EUNSUPPORTED;
    if (used + need > kTriSmemMax) {
      groups[++ng] = b;
      used = 0;
    }
    used += need;
    order[b] = b;
  }
  groups[++ng] = np;
  if (run && ng > 1) return SKY_EUNSUPPORTED;
  for (int g = 0; g < ng; ++g) {
    const sky_status s = tri_group(c, groups[g + 1] - groups[g], order + groups[g], A, n, w, Z,
                                   run, run_stride, gvec);
    if (s != SKY_OK) return s;
  }
  return SKY_OK;
}

}  // namespace sky
