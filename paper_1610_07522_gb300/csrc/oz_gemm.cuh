// Exact-integer split GEMM on the 5th-generation tensor cores (sm_103a) for the
// FP64 and FP32 forms of the overlap / Hamiltonian matrices (Eqs. normmatrix,
// hammatrix) and of the recombination (Sec. 3.3.3).
//
// Each row r of an operand is scaled by a power of two 2^e[r] (|x| < 2^e[r])
// and written as S signed base-256 digits,
//     x = 2^e[r] sum_{s<S} alpha_s 2^{-8(s+1)}   (+ a remainder below 2^{-8S}),
// |alpha_0| <= 256, |alpha_s| <= 128 (s >= 1): small integers that bf16
// holds exactly ("slices", Ozaki, Ogita, Oishi and Rump 2012).  The product
// keeps the slice pairs of total weight g = s + t <= S - 1:
//     sum_k A[m][k] B[n][k] = 2^{e_m + f_n - 16} sum_g 2^{-8g} G_g[m][n],
//     G_g = sum_{s + t = g} alpha_s beta_t^T.
// Every G_g is a sum of integer products, so its FP32 accumulation in TMEM is
// exact as long as it stays below 2^24: per K value |G_g| <= (g + 3) 2^14
// (g >= 1) or 2^16 (g = 0), so a segment of 128 values of K (4 K blocks of
// 32) is exact for every g <= 5.  One TMEM accumulator of BNT columns per
// group, the groups side by side, and the slices of B one below the other in
// shared memory: the products of slice s of A with consecutive slices t .. t'
// of B are one MMA of N = (t' - t + 1) BNT columns into the groups s + t ..
// s + t'.  The groups form two sets, L = {g < S/2} and H = the rest, and no MMA
// crosses them: 9 MMAs of up to 240 columns per 16 values of K instead of 21
// of 80 (each reads its 128 x 16 of A from shared memory once).  A set is
// drained ("flushed") after each of its segments, L after K blocks 1 mod 4 and
// H after 3 mod 4; a K block issues first the set whose segment ends, commits
// it, then the other, and the next block starts with that other set, so a
// drain has the products of two half blocks to hide behind.  The drained exact
// sums are added, scaled by 2^{-8g}, into an unevaluated FP32 pair (hi, lo)
// per output element (about 48 significant bits): groups 0 .. 3 by error-free
// TwoSum, groups 4 and 5, which lie below hi's last bit, straight into lo.  With
// seven slices a third sum takes what lo drops, and the partial results keep all
// three (a pair's own rounding, 2^-49, is 16 times that of FP64).
// What bounds it: shared memory.  Per 16 values of K the MMAs read 9 x 4 + 21 x
// 2.5 KiB of operands against 840 cycles on the tensor pipe, and the copies write
// 39 KiB: about 1000 cycles at 128 bytes per clock.  24^3, 280 states, one
// overlap: 560 us with one MMA per slice pair issued by one lane of a diverged
// warp (about 117 cycles from one to the next), 310 us now (1360 cycles).
//
// Persistent kernel, one CTA per SM; work items are (128 x BNT output tile,
// K range).  Warp roles:
//   warp 0     producer: bulk copies of one 32-wide K block of every slice of A
//              (128 rows) and B (BNT rows) into a ring of stages;
//   warp 1     owns TMEM (S accumulators of BNT fp32 columns) and issues
//              tcgen05.mma (M = 128, K = 16) as a converged warp, one elected
//              lane executing them;
//   warps 2-9  epilogue: two warps per TMEM lane quadrant, each half of the
//              columns; drain a group when its segment ends, accumulate
//              (hi, lo); write the item's result at its end.
// Operand layout in global memory (dig_off): the shared-memory image itself,
// blocks of BNT rows x 32 values of K x S slices, K block outermost, then the
// row tile, then the slice, each slice BNT rows of 64 bytes with the 16-byte
// chunks of a row in the 64-byte swizzle's order.  A tile of B is one contiguous
// 30 kB copy and 128 rows of A are two or three runs per slice; against tensor
// maps over row-major digits the product itself stays the same (310-315 us), the
// split kernels write whole blocks (103 -> 86 us per operand) and the small
// I x I products start sooner (17 -> 15 us; no maps to encode and fetch).
// Rows beyond an operand's last are never read as far as results go: whatever
// they hold reaches only outputs that are not stored; K beyond the operand's
// last value holds zeros.
// Every mbarrier wait is bounded; a timeout sets SKY_ETIMEOUT in the status
// word, the kernel waits (bounded) for the MMAs it issued, frees TMEM and
// returns.
#pragma once

#include <type_traits>

#include "tc_gemm.cuh"

namespace sky {
namespace oz {

using tc::fence_after;
using tc::fence_before;
using tc::idesc_bf16;
using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::mbar_wait;
using tc::smem_u32;

constexpr int BM = 128;
constexpr int BK = 32;                    // bf16 K block: one 64-byte swizzle row
// K blocks per exact segment: 128 values for S <= 6; with seven slices group 6
// reaches 9 x 2^14 per value, so 96
__host__ __device__ constexpr int seg_kb(int S) { return S <= 6 ? 4 : 3; }
constexpr int kEpiWarps = 8;
constexpr int THREADS = 64 + 32 * kEpiWarps;
constexpr int kMaxS = 7;
constexpr int kMaxStages = 4;
constexpr int kSmemMax = 232448;          // dynamic shared memory opt-in limit per CTA
constexpr int kSmemExtra = 1024 + 256;    // alignment slack + barriers
constexpr int TILE_A = BM * BK * 2;       // 8 KiB per A slice tile

// Slices of the FP64 and FP32 forms and their tile widths (S groups x BNT
// columns of TMEM <= 512).
constexpr int kS64 = 6, kBN64 = 80;
constexpr int kS32 = 4, kBN32 = 96;
// Seven slices hold a double's 53 bits whole; with them the products of weight 7
// count too (the last of two sets of four groups).  For the back-transformation of
// the eigensolver, whose reflectors' entries spread far below their largest one:
// the orthogonality it leaves at 700 states (Frobenius norm over sqrt(n)) is 1e-12
// with six slices, 3e-14 with seven and float-pair sums, 7.1e-15 as it is and
// 7.1e-15 with the reflectors applied in FP64.
constexpr int kS7 = 7, kBN7 = 64;
__host__ __device__ constexpr int num_groups(int S) { return S == kMaxS ? S + 1 : S; }
// Float pairs of a partial result: (hi, lo), with seven slices (hi, lo), (tail, 0).
__host__ __device__ constexpr int part_width(int S) { return S == kMaxS ? 2 : 1; }
template <int S>
__device__ __forceinline__ double part_value(const float2* row, int c) {
  if constexpr (S == kMaxS) {
    const float4 r = reinterpret_cast<const float4*>(row)[c];
    return (double)r.x + ((double)r.y + (double)r.z);
  } else {
    const float2 r = row[c];
    return (double)r.x + (double)r.y;
  }
}

// Element (row, k) of slice s of an operand of nt row tiles of BNT rows (2-byte
// elements); eight consecutive k from a multiple of 8 are consecutive.
template <int S, int BNT>
__host__ __device__ __forceinline__ long long dig_off(int row, int k, int s, int nt) {
  const int t = row / BNT, r = row - t * BNT;
  return (((long long)(k >> 5) * nt + t) * S + s) * (BNT * BK) + r * BK +
         ((((k >> 3) & 3) ^ ((r >> 1) & 3)) << 3) + (k & 7);
}
__host__ __device__ constexpr long long dig_tiles(long long rows, int bnt) { return (rows + bnt - 1) / bnt; }
__host__ __device__ constexpr long long dig_elems(long long rows, long long K, int S, int bnt) {
  return (K + BK - 1) / BK * dig_tiles(rows, bnt) * S * bnt * BK;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
// Shared-memory matrix descriptor: K-major tile with 64-byte swizzle, rows of
// 64 bytes, 8-row groups 512 bytes apart (stride byte offset), descriptor
// version 1, layout type 4 (64B swizzle).  Low word by address, high word fixed.
__device__ __forceinline__ uint32_t sw64_lo(uint32_t saddr) {
  return ((saddr >> 4) & 0x3FFFu) | (1u << 16);
}
constexpr uint32_t kSw64Hi = 32u | (1u << 14) | (4u << 29);
// NC consecutive fp32 columns (NC = 8, 16 or 32) of this warp's 32 TMEM lanes.
template <int NC>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r);
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
}
// Columns [0, NC) of a warp's share, NC = 32, 40 or 48, as 32, 32 + 8 or 32 + 16
// (complete after tmem_wait).
template <int NC>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t* r) {
  static_assert(NC == 32 || NC == 40 || NC == 48, "column share");
  tmem_ld<32>(taddr, r);
  if constexpr (NC > 32) tmem_ld<NC - 32>(taddr + 32, r + 32);
}
__device__ __forceinline__ void tmem_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The segment of set h (0: L, 1: H) ends after K block j (of nkb in the item):
// every SEG blocks, L after the second and H after the last of them, and at the
// item's last block.
template <int SEG>
__device__ __forceinline__ bool flush_at(int j, int h, int nkb) {
  return j == nkb - 1 || j % SEG == (h ? SEG - 1 : 1);
}

// One lane of a converged warp, as a flag (the same lane at every use of it).
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e;
}
// tcgen05.mma and its commit by the elected lane only, the warp converged
// around them; descriptors as low words with one common high word.
__device__ __forceinline__ void mma_bf16_elect(uint32_t tmem_d, uint32_t da, uint32_t db, uint32_t dhi,
                                               uint32_t idesc, uint32_t accumulate, uint32_t el) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 p, %5, 0;\n setp.ne.b32 q, %6, 0;\n"
      " mov.b64 a, {%1, %3};\n mov.b64 b, {%2, %3};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n}\n" ::"r"(tmem_d),
      "r"(da), "r"(db), "r"(dhi), "r"(idesc), "r"(accumulate), "r"(el)
      : "memory");
}
__device__ __forceinline__ void mma_commit_elect(uint32_t bar, uint32_t el) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
      "r"(el)
      : "memory");
}
// The bounded wait by a whole converged warp.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}

struct OzArgs {
  const unsigned short* A;  // operands in the blocked layout, nta and ntb row tiles
  const unsigned short* B;
  int nta, ntb;
  int M, N, K;              // rows of A, rows of B, K
  int kb_per_split;         // K blocks per split
  int nsplit;               // K splits
  int tri;                  // overlap lower-triangle pruning: B = [b; b'] with I rows each
  int I;
  int ntiles;               // output tiles in use (pruned when tri)
  int mode;                 // 0: (hi, lo) partials; 1: scaled final output
  float2* P;                // mode 0: P[z][m][n], row stride ldp, split stride sp (float2s)
  long long ldp, sp;
  void* out;                // mode 1: out[m][n] (double, or float when out_f32), row stride ldo
  long long ldo;
  int out_f32;
  const int* ea;            // mode 1: row exponents of A [M]
  const int* eb;            // mode 1: row exponents of B, eb[n >> eb_shift]
  int eb_shift;
  int* status;
  const int* run;           // device gate: the launch does nothing when *run == 0 or *stop != 0
  const int* stop;
};

// First 128-row tile a column tile of the [b; b'] overlap layout needs
// (rows a >= the smallest state index b its columns hold).
__host__ __device__ inline int tri_mi_min(int nj, int bnt, int N, int I) {
  const int n0 = nj * bnt;
  int n1 = n0 + bnt;
  if (n1 > N) n1 = N;
  --n1;
  const int bmin = (n0 < I && n1 >= I) ? 0 : (n0 < I ? n0 : n0 - I);
  return bmin / BM;
}

__host__ __device__ inline void item_of(const OzArgs& a, int bnt, int t, int& m0, int& n0, int& kb0,
                                        int& nkb) {
  const int mt = (a.M + BM - 1) / BM, nt = (a.N + bnt - 1) / bnt;
  const int z = t / a.ntiles;
  int tt = t - z * a.ntiles;
  int mi, nj;
  if (!a.tri) {
    mi = tt % mt;
    nj = tt / mt;
  } else {
    nj = 0;
    for (; nj < nt; ++nj) {
      int lo = tri_mi_min(nj, bnt, a.N, a.I);
      if (lo > mt) lo = mt;
      const int cnt = mt - lo;
      if (tt < cnt) break;
      tt -= cnt;
    }
    int lo = tri_mi_min(nj, bnt, a.N, a.I);
    if (lo > mt) lo = mt;
    mi = lo + tt;
  }
  m0 = mi * BM;
  n0 = nj * bnt;
  const int nkb_total = (a.K + BK - 1) / BK;
  kb0 = z * a.kb_per_split;
  nkb = nkb_total - kb0;
  if (nkb > a.kb_per_split) nkb = a.kb_per_split;
  if (nkb < 0) nkb = 0;
}

// Grouped products: np independent n x n complex products in one launch
// (the many small problems of a batched eigensolve).  Problem b's operands lie
// in the blocked layout from a.A + ao[b] (n rows) and a.B + bo[b] (2n rows), K =
// 2n, their row exponents from ra[b] and rb[b]; its items are the output tiles
// tile0[b] .. tile0[b+1] - 1 (one K range each); its partials go to P + po[b],
// rows of 2n.
struct OzGroup {
  int np;
  int tile0[kMaxBatch + 1];
  int n[kMaxBatch];
  int ra[kMaxBatch];
  int rb[kMaxBatch];
  long long ao[kMaxBatch];
  long long bo[kMaxBatch];
  long long po[kMaxBatch];
  const double2* A[kMaxBatch];
  const double2* B[kMaxBatch];
  double2* C[kMaxBatch];
  const int* run[kMaxBatch];
  const int* stop[kMaxBatch];
};

__host__ __device__ inline bool group_gated(const OzGroup& G, int b) {
  return (G.run[b] && *G.run[b] == 0) || (G.stop[b] && *G.stop[b] != 0);
}

// One work item: rows from m0 (A) and n0 (B), K blocks kb0 .. kb0 + nkb - 1 of
// the operands A, B (nta, ntb row tiles), of an M x N result (of problem b in a
// grouped launch).
struct OzItem {
  const unsigned short *A, *B;
  int nta, ntb;
  int m0, n0, kb0, nkb, b, M, N;
};

template <bool GROUP>
__device__ __forceinline__ bool item_at(const OzArgs& a, const OzGroup* G, int bnt, int t,
                                        OzItem& it) {
  if constexpr (GROUP) {
    int lo = 0, hi = G->np - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (G->tile0[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const int b = lo, n = G->n[b];
    if (group_gated(*G, b)) return false;
    const int mt = (n + BM - 1) / BM, tt = t - G->tile0[b];
    const int mi = tt % mt, nj = tt / mt;
    it.b = b;
    it.m0 = mi * BM;
    it.n0 = nj * bnt;
    it.A = a.A + G->ao[b];
    it.B = a.B + G->bo[b];
    it.nta = (n + bnt - 1) / bnt;
    it.ntb = (2 * n + bnt - 1) / bnt;
    it.kb0 = 0;
    it.nkb = (2 * n + BK - 1) / BK;
    it.M = n;
    it.N = 2 * n;
  } else {
    item_of(a, bnt, t, it.m0, it.n0, it.kb0, it.nkb);
    it.b = t / a.ntiles;   // the K split
    it.A = a.A;
    it.B = a.B;
    it.nta = a.nta;
    it.ntb = a.ntb;
    it.M = a.M;
    it.N = a.N;
  }
  return true;
}

__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float y) {
  const float s = hi + y;
  const float bp = s - hi;
  const float e = (hi - (s - bp)) + (y - bp);
  hi = s;
  lo += e;
}

// 2^k as a double (k in the normal range).
__device__ __forceinline__ double pow2d(int k) {
  return __longlong_as_double((long long)(1023 + k) << 52);
}

template <int S, int BNT, bool GROUP>
__device__ __forceinline__ void oz_gemm_body(const OzArgs& a, const OzGroup* grp) {
  if ((a.run && *a.run == 0) || (a.stop && *a.stop != 0)) return;   // uniform in the CTA
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((unsigned long long)smem_raw + 1023ull) & ~1023ull);
  constexpr int TILE_B = BNT * BK * 2;
  constexpr int STAGE = S * (TILE_A + TILE_B);
  constexpr int STAGES = (kSmemMax - kSmemExtra) / STAGE < kMaxStages
                             ? (kSmemMax - kSmemExtra) / STAGE
                             : kMaxStages;
  static_assert(STAGES >= 2, "ring");
  constexpr int NG = num_groups(S);
  static_assert(NG * BNT <= 512, "TMEM");
  static_assert(TILE_B % 1024 == 0, "swizzle alignment");
  constexpr uint32_t TMEM_COLS = 512;
  constexpr int HALF = BNT / 2;
  unsigned long long* bars = (unsigned long long*)(base + STAGES * STAGE);
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * kMaxStages + 2 * kMaxS + 1);
  constexpr int HS = NG / 2;                // groups of set L; H has the rest
  constexpr int SEG = seg_kb(S);
  static_assert((NG - HS) * BNT <= 256 && HS >= 2 && NG - HS <= 4, "sets of groups");
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int nitems = GROUP ? grp->tile0[grp->np] : a.ntiles * a.nsplit;
  // items of this CTA: every second round in reverse, so that the CTAs whose last
  // item was a short one (the later problems of a group) take the next first;
  // -1 at the end
  auto item_index = [&](int w) {
    const int g = (int)gridDim.x, b = (int)blockIdx.x;
    const long long first = (long long)w * g;
    if (first >= nitems) return -1;
    const int t = (int)first + ((w & 1) ? g - 1 - b : b);
    return t < nitems ? t : -1;
  };
  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
  auto acc_full = [&](int h) { return bar0 + 8u * (2 * kMaxStages + h); };
  auto acc_empty = [&](int h) { return bar0 + 8u * (2 * kMaxStages + kMaxS + h); };
  const uint32_t drain = bar0 + 8u * (2 * kMaxStages + 2 * kMaxS);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(acc_full(h), 1);
      mbar_init(acc_empty(h), kEpiWarps);   // one arrival per epilogue warp
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
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

  if (warp == 0) {
    // stage layout: A slices 0..S-1, then B slices 0..S-1.  Lane 0 arms the
    // stage's barrier and copies B (a partly filled tile of B: lane i slice i of
    // it); lane i copies run i % 3 (a row tile of A) of slice i / 3.
    static_assert(3 * S <= 32 && 2 * BNT >= BM, "runs of A");
    long long g = 0;
    bool ok = true;
    for (int w = 0, t; (t = item_index(w)) >= 0 && ok; ++w) {
      OzItem it;
      if (!item_at<GROUP>(a, grp, BNT, t, it)) continue;
      // rows that hold an operand's, in whole groups of 8 (the padding of a tile
      // is not fetched: 32^3, 5 FP32 states, whose tiles of B are 9/10 padding, one
      // overlap 160 us with it, 127 us)
      const int ma = (it.M + 7) & ~7, mb = (it.N - it.n0 + 7) & ~7;
      const int end = it.m0 + BM < ma ? it.m0 + BM : ma;
      const int rows_b = mb < BNT ? mb : BNT;
      const int p = lane / 3, ta = it.m0 / BNT + lane % 3;
      const int lo = ta * BNT > it.m0 ? ta * BNT : it.m0;
      const int hi = (ta + 1) * BNT < end ? (ta + 1) * BNT : end;
      const bool mine = lane < 3 * S && hi > lo;
      const long long ka = (long long)it.nta * S * (BNT * BK), kb = (long long)it.ntb * S * (BNT * BK);
      const unsigned short* srcA =
          it.A + it.kb0 * ka + ((long long)ta * S + p) * (BNT * BK) + (long long)(lo - ta * BNT) * BK;
      const bool whole_b = rows_b == BNT;
      const unsigned short* srcB = it.B + it.kb0 * kb + (long long)(it.n0 / BNT) * S * (BNT * BK) +
                                   (whole_b ? 0 : lane * (BNT * BK));
      const uint32_t dstB = (uint32_t)(S * TILE_A + (whole_b ? 0 : lane * TILE_B));
      const uint32_t bytes_b = whole_b ? (lane == 0 ? S * TILE_B : 0) : (lane < S ? rows_b * (BK * 2) : 0);
      const uint32_t bytes_a = mine ? (hi - lo) * (BK * 2) : 0;
      const uint32_t bytes = S * (end - it.m0 + rows_b) * (BK * 2);
      const uint32_t dstA = (uint32_t)(p * TILE_A + (lo - it.m0) * (BK * 2));
      for (int j = 0; j < it.nkb; ++j, ++g, srcA += ka, srcB += kb) {
        const int s = (int)(g % STAGES);
        const long long u = g / STAGES;
        if (u > 0 && !mbar_wait_warp(empty(s), (uint32_t)((u - 1) & 1))) {
          if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
          ok = false;
          break;
        }
        const uint32_t sa = smem_u32(base + s * STAGE);
        if (lane == 0) mbar_expect_tx(full(s), bytes);
        __syncwarp();
        if (bytes_b) bulk_load(sa + dstB, srcB, bytes_b, full(s));
        if (bytes_a) bulk_load(sa + dstA, srcA, bytes_a, full(s));
      }
    }
  } else if (warp == 1) {
    // the whole warp runs the loop, converged; the elected lane issues
    const uint32_t el = elect_one();
    uint32_t nfl[2] = {0u, 0u};
    long long gpos = 0;
    bool ok = true;
    for (int w = 0, t; (t = item_index(w)) >= 0 && ok; ++w) {
      OzItem it;
      if (!item_at<GROUP>(a, grp, BNT, t, it)) continue;
      const int nkb = it.nkb;
      for (int j = 0; j < nkb && ok; ++j, ++gpos) {
        const int s = (int)(gpos % STAGES);
        const long long u = gpos / STAGES;
        if (!mbar_wait_warp(full(s), (uint32_t)(u & 1))) {
          if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
          ok = false;
          break;
        }
        fence_after();
        const uint32_t la = sw64_lo(smem_u32(base + s * STAGE));
        const uint32_t lb = sw64_lo(smem_u32(base + s * STAGE + S * TILE_A));
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          const int h = j % SEG >= 2 ? 1 - o : o;     // the set whose segment may end here first
          const bool start = j == 0 || flush_at<SEG>(j - 1, h, nkb);
          if (start && nfl[h] > 0) {
            // the epilogue must have drained this set's previous segment
            if (!mbar_wait_warp(acc_empty(h), (nfl[h] - 1) & 1)) {
              if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
              ok = false;
              break;
            }
            fence_after();
          }
          auto issue = [&](auto hc) {
            constexpr int H = decltype(hc)::value;
#pragma unroll
            for (int i = 0; i < (H ? S : HS); ++i) {
              // the first MMA of a segment sets every group of its set, so with a
              // group beyond S slice 1 of A goes first
              const int p = H && NG > S && i < 2 ? 1 - i : i;
              const int top = !H ? HS : p + S < NG ? p + S : NG;
              const int g0 = H && p < HS ? HS : p;         // first group
              const int q0 = g0 - p;                        // first slice of B
              const uint32_t idesc = idesc_bf16(BM, (top - g0) * BNT);
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)   // +32 bytes along K = +2 in the encoded address
                mma_bf16_elect(tmem + (uint32_t)(g0 * BNT), la + (uint32_t)(p * (TILE_A >> 4) + 2 * k),
                               lb + (uint32_t)(q0 * (TILE_B >> 4) + 2 * k), kSw64Hi, idesc,
                               (start && i == 0 && k == 0) ? 0u : 1u, el);
            }
          };
          if (h) issue(std::integral_constant<int, 1>{});
          else issue(std::integral_constant<int, 0>{});
          if (flush_at<SEG>(j, h, nkb)) {
            mma_commit_elect(acc_full(h), el);   // arrives when this set's MMAs have completed
            ++nfl[h];
          }
        }
        if (!ok) break;
        mma_commit_elect(empty(s), el);
      }
    }
    // every MMA issued by this warp completes before TMEM is freed
    mma_commit_elect(drain, el);
    if (!mbar_wait_warp(drain, 0) && lane == 0) flag_status(a.status, SKY_ETIMEOUT);
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, columns half * HALF ..
    const int q = warp & 3, half = (warp - 2) >> 2;
    uint32_t efl[2] = {0u, 0u};
    auto hand_back = [&](int h) {            // this warp's lanes of the set are read
      fence_before();
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty(h)) : "memory");
    };
    bool ok = true;
    for (int w = 0, t; (t = item_index(w)) >= 0 && ok; ++w) {
      OzItem it;
      if (!item_at<GROUP>(a, grp, BNT, t, it)) continue;
      const int nkb = it.nkb;
      float hi[HALF], lo[HALF];
#pragma unroll
      for (int c = 0; c < HALF; ++c) hi[c] = lo[c] = 0.0f;
      float tail[S == kMaxS ? HALF : 1];     // seven slices: what lies below lo
      if constexpr (S == kMaxS) {
#pragma unroll
        for (int c = 0; c < HALF; ++c) tail[c] = 0.0f;
      }
      for (int j = 0; j < nkb && ok; ++j) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!flush_at<SEG>(j, h, nkb)) continue;
          if (!mbar_wait_warp(acc_full(h), efl[h] & 1)) {
            if (lane == 0) flag_status(a.status, SKY_ETIMEOUT);
            ok = false;
            break;
          }
          fence_after();
          const uint32_t col = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * HS * BNT + half * HALF);
          auto add = [&](const uint32_t* v, int g) {
            const float sc = __int_as_float((127 - 8 * g) << 23);   // 2^{-8g}, exact
#pragma unroll
            for (int c = 0; c < HALF; ++c) {
              const float y = __uint_as_float(v[c]);
              if (g < 4) two_sum_acc(hi[c], lo[c], y * sc);
              else lo[c] = fmaf(y, sc, lo[c]);
            }
          };
          if constexpr (S == kMaxS) {
            // 16 columns at a time, so that the set's four groups are at hand: the
            // rounding errors of groups 0 .. 2 (whole numbers below 2^4 times 2^-16)
            // add up exactly, and lo takes them and groups 3 and 4 by TwoSum, with
            // what it drops and groups 5 .. 7 in tail
            static_assert(NG == 8 && HS == 4 && HALF % 16 == 0, "two sets of four groups");
#pragma unroll
            for (int cc = 0; cc < HALF; cc += 16) {
              uint32_t v[4][16];
#pragma unroll
              for (int g = 0; g < 4; ++g) tmem_ld<16>(col + (uint32_t)(g * BNT + cc), v[g]);
              tmem_wait();
              if (cc + 16 == HALF) hand_back(h);
#pragma unroll
              for (int c = 0; c < 16; ++c) {
                auto y = [&](int g) {
                  return __uint_as_float(v[g][c]) * __int_as_float((127 - 8 * (g + 4 * h)) << 23);
                };
                if (h == 0) {
                  float e = 0.0f;
                  two_sum_acc(hi[cc + c], e, y(0));
                  two_sum_acc(hi[cc + c], e, y(1));
                  two_sum_acc(hi[cc + c], e, y(2));
                  two_sum_acc(lo[cc + c], tail[cc + c], e);
                  two_sum_acc(lo[cc + c], tail[cc + c], y(3));
                } else {
                  two_sum_acc(lo[cc + c], tail[cc + c], y(0));
                  tail[cc + c] += y(1) + (y(2) + y(3));
                }
              }
            }
            ++efl[h];
            continue;
          }
          // hand the set back as early as the registers allow: with narrow shares
          // two groups at once, the next ones read as the first are added
          uint32_t v0[HALF];
          tmem_ld_cols<HALF>(col, v0);
          if constexpr (HALF <= 40) {
            uint32_t v1[HALF];
            const int g = h * HS;
            tmem_ld_cols<HALF>(col + BNT, v1);
            tmem_wait();
            add(v0, g);
            tmem_ld_cols<HALF>(col + 2 * BNT, v0);
            tmem_wait();
            hand_back(h);
            add(v1, g + 1);
            add(v0, g + 2);
          } else {
            tmem_wait();
            add(v0, h * HS);
            tmem_ld_cols<HALF>(col + BNT, v0);
            tmem_wait();
            hand_back(h);
            add(v0, h * HS + 1);
          }
          ++efl[h];
        }
      }
      if (!ok) break;
      const int row = it.m0 + q * 32 + lane;
      const int col0 = it.n0 + half * HALF;
      if (row < it.M) {
        if (GROUP || a.mode == 0) {
          float2* prow = GROUP ? a.P + part_width(S) * (grp->po[it.b] + (long long)row * it.N)
                               : a.P + (long long)it.b * a.sp + (long long)row * a.ldp;
#pragma unroll
          for (int c = 0; c < HALF; ++c)
            if (col0 + c < it.N) {
              if constexpr (S == kMaxS)
                reinterpret_cast<float4*>(prow)[col0 + c] = make_float4(hi[c], lo[c], tail[c], 0.0f);
              else
                prow[col0 + c] = make_float2(hi[c], lo[c]);
            }
        } else if constexpr (S < kMaxS) {      // seven slices: partials only
          const int er = a.ea[row] - 16;
          if (a.out_f32) {
            float* orow = (float*)a.out + (long long)row * a.ldo;
#pragma unroll
            for (int c = 0; c < HALF; ++c)
              if (col0 + c < a.N) {
                const double sc = pow2d(er + a.eb[(col0 + c) >> a.eb_shift]);
                orow[col0 + c] = (float)(((double)hi[c] + (double)lo[c]) * sc);
              }
          } else {
            double* orow = (double*)a.out + (long long)row * a.ldo;
#pragma unroll
            for (int c = 0; c < HALF; ++c)
              if (col0 + c < a.N) {
                const double sc = pow2d(er + a.eb[(col0 + c) >> a.eb_shift]);
                orow[col0 + c] = ((double)hi[c] + (double)lo[c]) * sc;
              }
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

template <int S, int BNT>
__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const __grid_constant__ OzArgs a) {
  oz_gemm_body<S, BNT, false>(a, nullptr);
}

template <int S, int BNT>
__global__ void __launch_bounds__(THREADS, 1)
    k_oz_gemm_group(const __grid_constant__ OzArgs a, const __grid_constant__ OzGroup grp) {
  oz_gemm_body<S, BNT, true>(a, &grp);
}

template <int S, int BNT>
constexpr int smem_bytes() {
  constexpr int stage = S * (TILE_A + BNT * BK * 2);
  constexpr int st = (kSmemMax - kSmemExtra) / stage < kMaxStages ? (kSmemMax - kSmemExtra) / stage
                                                                    : kMaxStages;
  return st * stage + kSmemExtra;
}

// Number of output tiles of an M x N product (pruned to the tiles that hold
// an element a >= b of the [b; b'] overlap layout when tri).
inline int count_tiles(int M, int N, int bnt, bool tri, int I) {
  const int mt = (M + BM - 1) / BM, nt = (N + bnt - 1) / bnt;
  if (!tri) return mt * nt;
  int n = 0;
  for (int nj = 0; nj < nt; ++nj) {
    int lo = tri_mi_min(nj, bnt, N, I);
    if (lo > mt) lo = mt;
    n += mt - lo;
  }
  return n;
}

// Launch k_oz_gemm<S, BNT> on A (M rows) and B (N rows) in the blocked layout,
// 16-byte aligned, nta and ntb row tiles.  *splits in: the K splits wanted; out:
// the splits used (mode 0 writes P[z] for z < *splits).
template <int S, int BNT>
inline cudaError_t oz_gemm(const void* A, int nta, int M, const void* B, int ntb, int N, int K, bool tri,
                           int I, OzArgs g, int* splits, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0) { *splits = 0; return cudaSuccess; }
  if (dig_tiles(M, BNT) > nta || dig_tiles(N, BNT) > ntb) return cudaErrorInvalidValue;
  cudaError_t e;
  static bool smem_set[64] = {false};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!smem_set[dev]) {
    e = cudaFuncSetAttribute(k_oz_gemm<S, BNT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_bytes<S, BNT>());
    if (e != cudaSuccess) return e;
    smem_set[dev] = true;
  }
  const int nkb = (K + BK - 1) / BK;
  int z = *splits < 1 ? 1 : *splits;
  if (z > nkb) z = nkb;
  g.A = (const unsigned short*)A;
  g.B = (const unsigned short*)B;
  g.nta = nta; g.ntb = ntb;
  g.M = M; g.N = N; g.K = K;
  g.kb_per_split = (nkb + z - 1) / z;
  z = (nkb + g.kb_per_split - 1) / g.kb_per_split;
  g.nsplit = z;
  g.tri = tri ? 1 : 0;
  g.I = I;
  g.ntiles = count_tiles(M, N, BNT, tri, I);
  const long long items = (long long)g.ntiles * z;
  int nsm = 0;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int grid = (int)(items < nsm ? items : nsm);
  k_oz_gemm<S, BNT><<<grid, THREADS, smem_bytes<S, BNT>(), s>>>(g);
  note_launch();
  *splits = z;
  return cudaGetLastError();
}

// Launch the grouped form over grp's problems (operands from A + ao[b], B + bo[b]).
template <int S, int BNT>
inline cudaError_t oz_gemm_group(const void* A, const void* B, const OzGroup& grp, OzArgs g, cudaStream_t s) {
  if (grp.np <= 0 || grp.tile0[grp.np] == 0) return cudaSuccess;
  cudaError_t e;
  static bool smem_set[64] = {false};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!smem_set[dev]) {
    e = cudaFuncSetAttribute(k_oz_gemm_group<S, BNT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_bytes<S, BNT>());
    if (e != cudaSuccess) return e;
    smem_set[dev] = true;
  }
  int nsm = 0;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int items = grp.tile0[grp.np];
  const int grid = items < nsm ? items : nsm;
  g.A = (const unsigned short*)A;
  g.B = (const unsigned short*)B;
  g.mode = 0;
  g.run = g.stop = nullptr;
  k_oz_gemm_group<S, BNT><<<grid, THREADS, smem_bytes<S, BNT>(), s>>>(g, grp);
  note_launch();
  return cudaGetLastError();
}

}  // namespace oz
}  // namespace sky
