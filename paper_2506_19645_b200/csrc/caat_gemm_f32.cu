// fp32 GEMMs on the bf16 tensor cores, with errors that on ordinary data are below those of chains of fp32 FMAs.
//
// Every fp32 operand is split exactly into three bf16 parts, x = h + m + l (8 + 8 + 8 bits of significand, each rounded
// to nearest; Henry, Tang, Heinecke, "Leveraging the bfloat16 Artificial Intelligence Datatype For Higher-Precision
// Computations", 2019), and a product is six products of parts: h h, h m, m h, m m, h l, l h.  What is left out (m l, l m,
// l l) is at most 2^-24 of the product (x = 1.0038986 = 1 + 2^-8 - 2^-17 squared), as much as one fp32 rounding, and above 2^-26 for
// 2.8 % of random pairs.  The tensor core truncates when it adds to its fp32 accumulator (measured: 16 products 2.5e-8 of the
// result, 64 products 6.5e-8, 1024 products 4.7e-7, a bias towards zero), so an accumulator takes 64 elements of the
// contraction, smallest parts first, and the epilogue adds those partial sums in fp32 registers, rounded to nearest: results are
// 4e-8 to 6e-8 too small on average, where chains of FMAs have no bias.  Relative error (2-norm) against 64 bits, chains of FMAs
// on the CUDA cores / here: 4 x 768, 2000 tokens, layer output 2.1e-7 / 1.2e-7, data gradient 3.5e-7 / 1.1e-7, weight gradient
// 5.7e-7 / 1.4e-7; 8 x 5120, 60 tokens, the worst of the three 6.4e-7 / 1.9e-7; a weight gradient over 16, 64, 256 and 4096
// tokens 6.0e-8 / 4.8e-8, 1.1e-7 / 7.8e-8, 2.1e-7 / 8.8e-8, 2.9e-7 / 1.2e-7.  Operands made of that x and powers of two, where an FMA
// chain hardly rounds: 7.7e-8 / 1.3e-7 over 4096.
//
// A layer's training step at 4 x 768, 2000 tokens (28 GFLOP of products): 811 -> 270 us (three ring stages per pair instead of two,
// which leave the first-level cache too little: products 211 -> 230 us).  What bounds a
// stage (2.4 to 4 k cycles where its 24 products take 1.5 k) is the way round: loads, split, stores, barrier, products, barrier.
//
// Operands are multiplied by 2^16 on their way into parts and the accumulators' sums by 2^-32 where they are added up, both
// exact: an operand below 2^-110 would lose the last part's bits under bf16's smallest number (2^-133); so every fp32 number
// keeps all of them.  A result that is not finite is computed again from the operands with FMAs: sums of 2^96 and more,
// which overflow in the accumulator, and infinities and NaN, which come out as chains of FMAs give them (an infinity times a
// part that is zero would turn into NaN).  The epilogue only marks such a tile; a CTA goes over its marked tiles when its
// products are complete and no role waits for another (redo_tile).
//
// Persistent CTAs, one per SM:
//   warps 8..23  load fp32 operands (eight warps each; any of the two majors, 16-byte or element-wise), split them in
//                registers and store the parts into a two-stage ring in the layout that the tensor core reads;
//   warp 24      issues 24 tcgen05.mma of 128 x N x 16 per stage into one of four accumulators;
//   warps 0..7   add the accumulators to 64 columns each in registers and store the tile.
// A tile's contraction may be dealt over the CTAs of a cluster; the partial tiles are then summed in order through
// distributed shared memory.  Either operand may be the 128-row side (a few tokens: the weights).
#include <algorithm>
#include <cfloat>
#include <cstdlib>
#include <mutex>
#include <utility>

#include "caat_tc_ptx.cuh"

namespace caat {
namespace {

using namespace tc;

constexpr int XM = 128, XN = 128, XK = 64;
// CG = 1: a CTA's tile is 128 x 128 (few rows).  CG = 2: a pair of CTAs (tcgen05 cta_group::2) works on 256 x 128; each CTA stages its
// 128 rows of A and half of the columns of B, so it splits a quarter less, and the tensor cores read a quarter less of its
// shared memory per product, which is what bounds CG = 1: 24 products of a stage read 192 KB where 1536 cycles deliver 196,
// and the producers store 96 KB beside them.
constexpr int kPartA = 128 * XK * 2;              // one part of one operand of a stage
template <int CG> constexpr int kPartB = kPartA / CG;
constexpr int kOperandA = 3 * kPartA;
template <int CG> constexpr int kStageBytes = kOperandA + 3 * kPartB<CG>;
constexpr int kStages = 2;
constexpr int kAccs = 4;                          // accumulators of 128 columns: all of tensor memory
constexpr int kEpiWarps = 8, kProdWarp0 = 8, kProdWarps = 16, kMmaWarp = 24;
// Seven warpgroups at 72 registers; B's producers and the last group (the issuing warp and three idle ones) give up what
// the epilogue's two take: 2 x 96 + 2 x 72 + 2 x 64 + 40 = 7 x 72.
constexpr int kThreads = 896;
// behind the ring: barriers, the tensor-memory address and the abort flag; then a bit per item (or group of items)
constexpr int kBarBytes = 256, kMarkWords = 64;
constexpr int kBars = 2 * kStages + 2 * kAccs + 3;
template <int CG> constexpr int kSmem = kStages * kStageBytes<CG> + 1024 + kBarBytes + 4 * kMarkWords;
constexpr uint32_t kSpinCap = 1u << 22;

struct XSeg {                 // one segment of the contraction: A(b, q, row, k) and B(b, q, col, k)
  const float *A, *B;
  long long sAb, sAq, sAl, sBb, sBq, sBl;     // sAl, sBl: the stride that is not 1 (of rows if k is contiguous, else of k)
  int Q, Kd;
};
struct XProblem {
  int nseg;
  XSeg seg[2];
  float* C;
  long long sCb, sCi, sCj;    // sCi or sCj is 1
  int M, N, batch;
  int ntm, ntn, tiles, chunks, split;
};
struct XParams {
  XProblem p[2];
  int nprob;
  int csize;                  // tiles side by side in a cluster: CTAs, or pairs of CTAs
  int items0, items;          // cluster items of problem 0, of both
  unsigned int* status;
  uint32_t spin_cap;
  int stall;                  // the time-out test: stages are filled but never announced
};

// ------------------------------------------------------------------ schedule
struct Item { int prob, b, i0, j0, c0, c1, cols; bool split, valid; };

// crank: the CTA's (pair's) place among the csize of its cluster
template <int CG>
__device__ __forceinline__ Item item_at(const XParams& p, int n, int crank) {
  Item t;
  t.prob = n >= p.items0 ? 1 : 0;
  const XProblem& g = p.p[t.prob];
  const int local = n - (t.prob ? p.items0 : 0);
  t.split = g.split != 0;
  int tile = t.split ? local : local * p.csize + crank;
  t.valid = tile < g.tiles;
  t.c0 = 0; t.c1 = g.chunks;
  if (t.split) {
    t.c0 = g.chunks * crank / p.csize;
    t.c1 = g.chunks * (crank + 1) / p.csize;
  }
  t.j0 = tile % g.ntn * XN; tile /= g.ntn;
  t.i0 = tile % g.ntm * (XM * CG);
  t.b = tile / g.ntm;
  const int left = g.N - t.j0;
  t.cols = left >= XN ? XN : (left + 16 * CG - 1) / (16 * CG) * (16 * CG);
  return t;
}

// position in the contraction of a problem: the chunks of all segments and ranks form one sequence
struct KPos { int seg, q, k0; };
__device__ __forceinline__ KPos kpos_at(const XProblem& g, int n) {
  KPos p{0, 0, 0};
  const int n0 = g.seg[0].Q * ((g.seg[0].Kd + XK - 1) / XK);
  if (n >= n0) { p.seg = 1; n -= n0; }
  const int per = (g.seg[p.seg].Kd + XK - 1) / XK;
  p.q = n / per;
  p.k0 = (n - p.q * per) * XK;
  return p;
}

// ------------------------------------------------------------------ operands
// A thread owns four pieces of eight elements along the contiguous axis of a 128 x 64 operand tile:
//   k contiguous     rows r, r + 32, r + 64, r + 96 (r = tid / 8), elements 8 (tid % 8) of k
//   rows contiguous  k, k + 16, k + 32, k + 48 (k = tid / 16), rows 8 (tid % 16)
// Both ways eight neighbouring lanes write one 128-byte line of the swizzled tile, and a warp's loads are whole sectors.
template <bool VEC>
__device__ __forceinline__ void load8(float (&v)[8], const float* p, int left) {
  if (VEC && left >= 8) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = e < left ? p[e] : 0.f;
  }
}

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&b);
}
constexpr float kScale = 65536.f;
// the three parts of eight elements, stored at the same place of the three part tiles
__device__ __forceinline__ float2 less(float2 x, uint32_t part) {      // x minus a pair of parts: exact
  return __ffma2_rn(make_float2(__uint_as_float(part << 16), __uint_as_float(part & 0xffff0000u)), make_float2(-1.f, -1.f), x);
}
__device__ __forceinline__ uint32_t scaled(uint32_t h) {      // a pair of first parts: exact, and one instruction for both
  const __nv_bfloat162 b = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&h), __float2bfloat162_rn(kScale));
  return *reinterpret_cast<const uint32_t*>(&b);
}
template <int PART>
__device__ __forceinline__ void split_store(const float (&v)[8], uint32_t dst) {
  uint32_t h[4], m[4], l[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float2 x = make_float2(v[2 * q], v[2 * q + 1]);
    h[q] = scaled(bf16x2(x.x, x.y));
    x = make_float2(fmaf(x.x, kScale, -__uint_as_float(h[q] << 16)), fmaf(x.y, kScale, -__uint_as_float(h[q] & 0xffff0000u)));
    m[q] = bf16x2(x.x, x.y);
    x = less(x, m[q]);
    l[q] = bf16x2(x.x, x.y);
  }
  sts128(dst, h[0], h[1], h[2], h[3]);
  sts128(dst + PART, m[0], m[1], m[2], m[3]);
  sts128(dst + 2 * PART, l[0], l[1], l[2], l[3]);
}
template <bool KM, int ROWS>
__device__ __forceinline__ uint32_t piece_offset(int tid, int u) {
  if (KM) {
    const int r = (tid >> 3) + 32 * u;
    return (uint32_t)(r * 128 + (((tid & 7) ^ (r & 7)) << 4));
  }
  constexpr int W = ROWS / 8;                     // pieces of a k
  const int k = tid / W + 256 / W * u, c = tid % W;
  return (uint32_t)((c >> 3) * (64 * XK * 2) + k * 128 + (((c & 7) ^ (k & 7)) << 4));
}

__device__ __forceinline__ bool not_finite(float x) { return !(fabsf(x) <= FLT_MAX); }

__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag, uint32_t cap) {
  for (uint32_t it = 0; it < cap; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if ((it & 1023u) == 1023u && *abort_flag) return false;
  }
  return false;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory"); }
__device__ __forceinline__ bool epi_all(bool ok) {       // barrier with a vote
  int r;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n barrier.red.and.pred q, 1, %2, p;\n selp.s32 %0, 1, 0, q;\n}"
               : "=r"(r) : "r"((int)ok), "n"(kEpiWarps * 32) : "memory");
  return r != 0;
}

// ------------------------------------------------------------------ results that are not finite
// the mark of a CTA's item: its number among the CTA's, several to a mark where there are more items than marks
__device__ __forceinline__ int mark_of(int items, int n, int worker, int nworkers) {
  int shift = 0;
  while (items / nworkers >> shift >= 32 * kMarkWords) ++shift;
  return (n - worker) / nworkers >> shift;
}
// ROWS x 64 elements of an operand into [k][row] by 256 threads.  k contiguous: a warp takes 8 k of 4 rows at a time, whole sectors
// into 32 banks (LD is 4 more than a multiple of 32).  Through registers: with one cp.async anywhere in the kernel, executed or not,
// the producers' fences above wait longer (three products of a step at 4 x 768, 2000 tokens: 217 -> 225 us).
template <bool KM, int ROWS, int LD>
__device__ __forceinline__ void redo_load(float* dst, const float* p, long long ld, int rows, int k_left, int tid) {
  constexpr int STEP = KM ? 4 : 256 / ROWS, N = KM ? ROWS / 4 : XK / STEP, B = 8;       // B loads in flight
  const int k = KM ? (tid >> 5) * 8 + (tid & 7) : tid / ROWS, r = KM ? tid >> 3 & 3 : tid % ROWS;
  const int slow = KM ? r : k, slow_end = (KM ? k < k_left : r < rows) ? (KM ? rows : k_left) : 0;
  const float* src = p + slow * ld + (KM ? k : r);
  dst += k * LD + r;
#pragma unroll 1
  for (int u = 0; u < N; u += B, src += B * STEP * ld, dst += B * STEP * (KM ? 1 : LD)) {
    float v[B];
#pragma unroll
    for (int b = 0; b < B; ++b) v[b] = slow + (u + b) * STEP < slow_end ? src[b * STEP * ld] : 0.f;
#pragma unroll
    for (int b = 0; b < B; ++b) dst[b * STEP * (KM ? 1 : LD)] = v[b];
  }
}
// The results of 128 rows from i0 and the columns [j0, j1) that are not finite, from the operands by chains of 64 FMAs, added up in
// fp32.  The epilogue's 256 threads, 32 columns at a time, 4 x 4 results per thread, both operands two chunks deep in `stage`
// (the ring).  A warp whose 16 rows need nothing (finite, or NaN by now) only helps to load.  Two warps per scheduler bound it,
// and the few CTAs that hold marked tiles.  A training step of one layer, CUDA cores (any data) / here with one infinite token / one
// infinite value / all infinite, us: 4 x 768, 2000 tokens 827 / 610 / 824 / 1134; 2 x 1024, 300 tokens 296 / 316 / 603 / 709;
// 8 x 5120, 100 tokens 1585 / 2021 / 3412 / 3999.
constexpr int kRedoCols = 32, kRedoLdA = XM + 4, kRedoLdB = kRedoCols + 4, kRedoStage = XK * (kRedoLdA + kRedoLdB);
static_assert(2 * kRedoStage * 4 <= kStages * kStageBytes<2> && XM * kRedoCols == 16 * 256, "");

template <bool AK, bool BKM>
__device__ __forceinline__ void redo_tile(const XProblem& g, int b, int i0, int j0, int j1, float* stage, int tid) {
  const int r4 = (tid >> 3) * 4, c4 = (tid & 7) * 4;
  if (j1 > g.N) j1 = g.N;
  for (int jc = j0; jc < j1; jc += kRedoCols) {
    float* out = g.C + b * g.sCb + (i0 + r4) * g.sCi + (jc + c4) * g.sCj;
    uint32_t todo = 0;                               // results of this thread that are not finite
#pragma unroll 4
    for (int e = 0; e < 16; ++e)
      if (i0 + r4 + (e >> 2) < g.M && jc + c4 + (e & 3) < j1 && not_finite(out[(e >> 2) * g.sCi + (e & 3) * g.sCj])) todo |= 1u << e;
    bool idle = __all_sync(0xffffffffu, todo == 0);
    if (epi_all(idle)) continue;
    auto load = [&](int n) {
      const KPos pos = kpos_at(g, n);
      const XSeg& s = g.seg[pos.seg];
      const float* A = s.A + b * s.sAb + pos.q * s.sAq + (AK ? i0 * s.sAl + pos.k0 : pos.k0 * s.sAl + i0);
      const float* B = s.B + b * s.sBb + pos.q * s.sBq + (BKM ? jc * s.sBl + pos.k0 : pos.k0 * s.sBl + jc);
      float* dst = stage + (n & 1) * kRedoStage;
      redo_load<AK, XM, kRedoLdA>(dst, A, s.sAl, g.M - i0, s.Kd - pos.k0, tid);
      redo_load<BKM, kRedoCols, kRedoLdB>(dst + XK * kRedoLdA, B, s.sBl, g.N - jc, s.Kd - pos.k0, tid);
    };
    float sum[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) sum[e] = 0.f;
    load(0);
#pragma unroll 1
    for (int n = 0; n < g.chunks; ++n) {
      if (n + 1 < g.chunks) load(n + 1);
      epi_sync();
      if (!idle) {
        const float* A = stage + (n & 1) * kRedoStage + r4;
        const float* B = stage + (n & 1) * kRedoStage + XK * kRedoLdA + c4;
        float acc[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.f;
#pragma unroll 2
        for (int k = 0; k < XK; ++k, A += kRedoLdA, B += kRedoLdB) {
          const float4 a = *reinterpret_cast<const float4*>(A), v = *reinterpret_cast<const float4*>(B);
          const float x[4] = {a.x, a.y, a.z, a.w}, y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 16; ++e) acc[e] = fmaf(x[e >> 2], y[e & 3], acc[e]);
        }
        uint32_t open = 0;                           // a sum that is NaN stays NaN
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          sum[e] += acc[e];
          open |= sum[e] == sum[e] ? 1u << e : 0u;
        }
        idle = __all_sync(0xffffffffu, (todo & open) == 0);
      }
      if (epi_all(idle)) break;
    }
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (todo >> e & 1u) out[(e >> 2) * g.sCi + (e & 3) * g.sCj] = sum[e];
  }
}

// The epilogue's last step, when every product of the CTA is complete: its ring is idle, and nobody waits for these warps but
// barriers without a limit.  Reads its place anew, so that the loop before it keeps no registers for it.
__device__ __forceinline__ uint8_t* ring_base() {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
}
template <int CG, bool AK, bool BKM>
__device__ __forceinline__ void redo_marked(const XParams& p) {
  uint32_t tid, block, blocks;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(block));
  asm volatile("mov.u32 %0, %%nctaid.x;" : "=r"(blocks));
  uint8_t* base = ring_base();
  const unsigned int* marks = reinterpret_cast<const unsigned int*>(base + kStages * kStageBytes<CG> + kBarBytes);
  const volatile int* aborted = reinterpret_cast<const volatile int*>(base + kStages * kStageBytes<CG> + 8 * kBars + 4);
  epi_sync();                                        // the marks are complete; a wait that ran out has raised the flag
  if (epi_all(tid >= kMarkWords || marks[tid % kMarkWords] == 0 || *aborted)) return;
  const int ctas = p.csize * CG, cta = ctas > 1 ? (int)cluster_ctarank() : 0, crank = cta / CG;
  const int worker = block / ctas, nworkers = blocks / ctas;
  for (int n = worker; n < p.items; n += nworkers) {
    const int m = mark_of(p.items, n, worker, nworkers);
    const Item it = item_at<CG>(p, n, crank);
    if (!(marks[m >> 5] >> (m & 31) & 1u) || !it.valid) continue;
    const int cw = XN / p.csize, j0 = it.split ? it.j0 + crank * cw : it.j0;      // the columns that this CTA stored
    redo_tile<AK, BKM>(p.p[it.prob], it.b, it.i0 + cta % CG * XM, j0, it.split ? j0 + cw : j0 + XN, reinterpret_cast<float*>(base), tid);
  }
}

// ------------------------------------------------------------------ producers
// Eight warps fill one operand's half of the ring's stages.  A chunk's registers are loaded while the one before it is split.
// half: this CTA's place in its pair.  full0: the barriers of the pair's leader.
template <int CG, bool IS_A, bool KM, bool VEC>
__device__ __forceinline__ void produce(const XParams& p, int tid, int worker, int nworkers, int crank, int half, uint32_t ring,
                                        uint32_t full0, uint32_t empty0, uint32_t done, volatile int* abort_flag) {
  constexpr int ROWS = IS_A ? XM : XN / CG, W = ROWS / 8, U = ROWS * XK / 8 / 256;      // rows of the operand here, pieces of a thread
  constexpr int kStep = KM ? 32 : 256 / W;
  const int fast0 = KM ? (tid & 7) * 8 : tid % W * 8, slow0 = KM ? tid >> 3 : tid / W;
  int stage = 0; uint32_t phase = 0, done_phase = 0;
  int n = worker - nworkers;
  int prob = 0, seg = 0, q = 0;
  int chunks = 0, k_left = 0, rows = 0, cols = 0;   // chunks of the item left, k left in the segment, rows of the matrix from the tile's first
  bool split = false, behind_split = false;         // behind_split: the ring holds partial tiles until `done`
  const float* src = nullptr;                       // this thread's first piece
  long long ld = 0;
  float v[U][8];
  // the next chunk of the schedule; false at the end
  auto advance = [&]() {
    if (--chunks > 0 && k_left > XK) {
      k_left -= XK;
      src += KM ? (long long)XK : XK * ld;
      return true;
    }
    int b, r0, k0 = 0;
    if (chunks > 0) {                               // the next rank or segment of the same tile
      const Item it = item_at<CG>(p, n, crank);
      b = it.b; r0 = IS_A ? it.i0 + half * XM : it.j0 + half * (cols / CG);
      if (++q >= p.p[prob].seg[seg].Q) { q = 0; seg = 1; }
    } else {
      behind_split = split;
      for (;;) {
        if ((n += nworkers) >= p.items) return false;
        const Item it = item_at<CG>(p, n, crank);
        if (!it.valid || it.c0 >= it.c1) continue;
        const KPos pos = kpos_at(p.p[it.prob], it.c0);
        prob = it.prob; seg = pos.seg; q = pos.q; k0 = pos.k0;
        chunks = it.c1 - it.c0; split = it.split; cols = it.cols;
        b = it.b; r0 = IS_A ? it.i0 + half * XM : it.j0 + half * (cols / CG);
        break;
      }
    }
    const XProblem& g = p.p[prob];
    const XSeg& s = g.seg[seg];
    ld = IS_A ? s.sAl : s.sBl;
    rows = (IS_A ? g.M : g.N) - r0;
    k_left = s.Kd - k0;
    src = (IS_A ? s.A + b * s.sAb + q * s.sAq : s.B + b * s.sBb + q * s.sBq) +
          (KM ? (r0 + slow0) * ld + k0 + fast0 : (k0 + slow0) * ld + r0 + fast0);
    return true;
  };
  auto load = [&](int u) {
    const int slow_left = (KM ? rows : k_left) - slow0, left = (KM ? k_left : rows) - fast0;
    load8<VEC>(v[u], src + kStep * u * ld, kStep * u < slow_left ? left : 0);
  };
  chunks = 1;
  bool more = advance(), ok = true;
  behind_split = false;
  if (more) {
#pragma unroll
    for (int u = 0; u < U; ++u) load(u);
  }
  while (more) {
    const int now_cols = cols;
    const bool wait_done = behind_split;
    behind_split = false;
    more = advance();             // where the chunk after this one comes from
    if (wait_done) {
      ok = mbar_wait_warp(done, done_phase, abort_flag, p.spin_cap);
      done_phase ^= 1u;
    }
    if (!ok || !mbar_wait_warp(empty0 + 8 * stage, phase ^ 1u, abort_flag, p.spin_cap)) { ok = false; break; }
    const uint32_t dst = ring + (uint32_t)stage * kStageBytes<CG>;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      // rows that a narrow tile's products do not read are left as they are
      if (IS_A || !KM || 32 * CG * u < now_cols) split_store<IS_A ? kPartA : kPartB<CG>>(v[u], dst + piece_offset<KM, ROWS>(tid, u));
      if (more) load(u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if ((tid & 31) == 0 && !p.stall) {
      if (CG == 2) mbar_arrive_shared(full0 + 8 * stage); else mbar_arrive(full0 + 8 * stage);
    }
    if (++stage == kStages) { stage = 0; phase ^= 1u; }
  }
  if (!ok && (tid & 31) == 0) { *abort_flag = 1; atomicExch(p.status, 1u); }
}

// ------------------------------------------------------------------ kernel
// AK / BKM: k is the contiguous axis of A / B (else its rows are)
template <int CG, bool AK, bool BKM, bool VEC>
__global__ void __launch_bounds__(kThreads, 1) gemm_f32_kernel(const __grid_constant__ XParams p) {
  uint8_t* base = ring_base();
  const uint32_t ring = smem_u32(base);
  // behind the ring: full, empty (a stage each), tfull[4], tempty[4], ready, data, done, tensor-memory address, abort flag
  const uint32_t full0 = ring + kStages * kStageBytes<CG>, empty0 = full0 + 8 * kStages, tfull0 = empty0 + 8 * kStages;
  const uint32_t tempty0 = tfull0 + 8 * kAccs, ready = tempty0 + 8 * kAccs, data = ready + 8, done = data + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + kStages * kStageBytes<CG> + 8 * kBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  unsigned int* marks = reinterpret_cast<unsigned int*>(base + kStages * kStageBytes<CG> + kBarBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int csize = p.csize, ctas = csize * CG, cta = ctas > 1 ? (int)cluster_ctarank() : 0;      // of the cluster
  const int crank = cta / CG, pair_half = cta % CG, leader = cta - pair_half;
  const int worker = blockIdx.x / ctas, nworkers = gridDim.x / ctas;

  if (threadIdx.x < kMarkWords) marks[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full0 + 8 * s, kProdWarps * CG); mbar_init(empty0 + 8 * s, 1); }
    for (int a = 0; a < kAccs; ++a) { mbar_init(tfull0 + 8 * a, 1); mbar_init(tempty0 + 8 * a, kEpiWarps * CG); }
    mbar_init(ready, csize); mbar_init(data, csize); mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    if (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kAccs * XN) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kAccs * XN) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (ctas > 1) cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();

  if (warp >= kProdWarp0 && warp < kMmaWarp) {
    // ------------------------------------------------------------ producers
    const uint32_t full = CG == 2 ? mapa_rank(full0, leader) : full0;
    if (threadIdx.x < (kProdWarp0 + kProdWarps / 2) * 32)
      produce<CG, true, AK, VEC>(p, threadIdx.x - kProdWarp0 * 32, worker, nworkers, crank, pair_half, ring, full, empty0, done, abort_flag);
    else {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
      produce<CG, false, BKM, VEC>(p, threadIdx.x - (kProdWarp0 + kProdWarps / 2) * 32, worker, nworkers, crank, pair_half,
                                   ring + kOperandA, full, empty0, done, abort_flag);
    }
  } else if (warp >= kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == kMmaWarp && pair_half == 0) {
      const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)!AK << 15) | ((uint32_t)!BKM << 16) |
                              ((uint32_t)((XM * CG) >> 4) << 24);
      const uint64_t ac = AK ? make_desc(0, 16, 1024) : make_desc(0, 64 * XK * 2, 1024);
      const uint64_t bc = BKM ? make_desc(0, 16, 1024) : make_desc(0, 64 * XK * 2, 1024);
      constexpr uint32_t ak16 = (AK ? 32 : 2048) >> 4, bk16 = (BKM ? 32 : 2048) >> 4, pa16 = kPartA >> 4, pb16 = kPartB<CG> >> 4;
      int stage = 0, acc = 0; uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (int n = worker; n < p.items && ok; n += nworkers) {
        const Item it = item_at<CG>(p, n, crank);
        if (!it.valid) continue;
        const uint32_t idesc = idesc0 | ((uint32_t)(it.cols >> 3) << 17);
        for (int c = it.c0; c < it.c1; ++c) {
          const bool landed = CG == 2 ? __all_sync(0xffffffffu, mbar_wait_cluster(full0 + 8 * stage, phase, abort_flag, p.spin_cap))
                                      : mbar_wait_warp(full0 + 8 * stage, phase, abort_flag, p.spin_cap);
          if (!landed || !mbar_wait_warp(tempty0 + 8 * acc, acc_phase ^ 1u, abort_flag, p.spin_cap)) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
            const uint32_t sa = (ring & 0x3FFFFu) + (uint32_t)stage * kStageBytes<CG>;      // without the rank bits of a cluster's address
            const uint32_t a0 = (uint32_t)ac + (sa >> 4), b0 = (uint32_t)bc + ((sa + kOperandA) >> 4);
            const uint32_t d = tmem + (uint32_t)(acc * XN);
            // parts of A, of B (two bits each, first product lowest): h l, l h, m m, h m, m h, h h
            uint32_t parts_a = 0x118u, parts_b = 0x052u;
#pragma unroll 1
            for (int q = 0; q < 6; ++q, parts_a >>= 2, parts_b >>= 2) {
              uint32_t al = a0 + (parts_a & 3u) * pa16, bl = b0 + (parts_b & 3u) * pb16;
#pragma unroll
              for (int k = 0; k < XK / 16; ++k) {
                const uint64_t ad = (ac & 0xffffffff00000000ull) | (al + k * ak16), bd = (bc & 0xffffffff00000000ull) | (bl + k * bk16);
                if (CG == 2) umma_bf16_pair(d, ad, bd, idesc, q + k > 0 ? 1u : 0u); else umma_bf16(d, ad, bd, idesc, q + k > 0 ? 1u : 0u);
              }
            }
            if (CG == 2) {
              umma_commit_ctas(empty0 + 8 * stage, 3u << leader);
              umma_commit_ctas(tfull0 + 8 * acc, 3u << leader);
            } else {
              umma_commit(empty0 + 8 * stage);
              umma_commit(tfull0 + 8 * acc);
            }
          }
          __syncwarp();
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
          if (++acc == kAccs) { acc = 0; acc_phase ^= 1u; }
        }
      }
      if (!ok && lane == 0) { *abort_flag = 1; atomicExch(p.status, 2u); }
    }
  } else {
    // ------------------------------------------------------------ epilogue: 32 rows x 64 columns per warp
    asm volatile("setmaxnreg.inc.sync.aligned.u32 96;");
    const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
    int acc = 0; uint32_t acc_phase = 0, red_phase = 0;
    bool ok = true;        // a warp whose wait ran out goes on to the next vote, so that no barrier misses it
    for (int n = worker; n < p.items; n += nworkers) {
      const Item it = item_at<CG>(p, n, crank);
      if (!it.valid) continue;
      const XProblem& g = p.p[it.prob];
      float sum[64];
#pragma unroll
      for (int e = 0; e < 64; ++e) sum[e] = 0.f;
      for (int c = it.c0; c < it.c1 && ok; ++c) {
        if (!mbar_wait_warp(tfull0 + 8 * acc, acc_phase, abort_flag, p.spin_cap)) { ok = false; break; }
        tc_fence_after();
        const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * XN + half * 64);
#pragma unroll
        for (int e = 0; e < 64; e += 16) {
          if (half * 64 + e >= it.cols) break;
          uint32_t v[32];
          tmem_ld16(ta + e, v);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 16; ++k) sum[e + k] = fmaf(__uint_as_float(v[k]), 1 / (kScale * kScale), sum[e + k]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (CG == 2) mbar_arrive_remote(mapa_rank(tempty0 + 8 * acc, leader)); else mbar_arrive(tempty0 + 8 * acc);
        }
        if (++acc == kAccs) { acc = 0; acc_phase ^= 1u; }
      }
      const int i = it.i0 + pair_half * XM + row;
      float* crow = g.C + it.b * g.sCb + i * g.sCi;
      float poison = 0.f;         // becomes NaN with the first value that is not finite
      // four neighbouring columns of this thread's row
      auto store4 = [&](float* dst, int j, float a, float b, float c, float d) {
        if (i >= g.M || j >= g.N) return;
        poison = fmaf(a, 0.f, poison);
        if (j + 3 < g.N) {
          poison = fmaf(b, 0.f, fmaf(c, 0.f, fmaf(d, 0.f, poison)));
          if (VEC && g.sCj == 1) {
            *reinterpret_cast<float4*>(dst) = make_float4(a, b, c, d);
            return;
          }
          dst[0] = a; dst += g.sCj;
          dst[0] = b; dst += g.sCj;
          dst[0] = c; dst += g.sCj;
          dst[0] = d;
          return;
        }
        dst[0] = a;
        if (j + 1 < g.N) { dst[g.sCj] = b; poison = fmaf(b, 0.f, poison); }
        if (j + 2 < g.N) { dst[2 * g.sCj] = c; poison = fmaf(c, 0.f, poison); }
      };
      if (!it.split) {
        if (!ok) continue;
        const int jb = it.j0 + half * 64;
        float* dst = crow + jb * g.sCj;
#pragma unroll
        for (int e = 0; e < 64; e += 4, dst += 4 * g.sCj) store4(dst, jb + e, sum[e], sum[e + 1], sum[e + 2], sum[e + 3]);
      } else {
        // place r of the cluster finishes columns r * cw .. of the tile: it gets them from every place (pairs: from the CTA
        // with the same rows), [source][column][row] in its ring, which is free once its own products are complete
        const int cw = XN / csize;
        if (!epi_all(ok)) { ok = false; break; }
        if (threadIdx.x < csize) mbar_arrive_release(mapa_rank(ready, threadIdx.x * CG + pair_half));
        ok = mbar_wait_cluster(ready, red_phase, abort_flag, p.spin_cap);
        if (!epi_all(ok)) { ok = false; break; }
#pragma unroll
        for (int e0 = 0; e0 < 64; e0 += 16) {            // cw is a multiple of 16
          const int col = half * 64 + e0, dest = col / cw;
          const uint32_t a = mapa_rank(ring + (uint32_t)(((crank * cw + col - dest * cw) * 128 + row) * 4), dest * CG + pair_half);
#pragma unroll
          for (int e = 0; e < 16; ++e)
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a + e * 512), "f"(sum[e0 + e]) : "memory");
        }
        epi_sync();
        if (threadIdx.x < csize) mbar_arrive_release(mapa_rank(data, threadIdx.x * CG + pair_half));
        ok = mbar_wait_cluster(data, red_phase, abort_flag, p.spin_cap);
        red_phase ^= 1u;
        if (!epi_all(ok)) { ok = false; break; }
        const float* part = reinterpret_cast<const float*>(base) + row;
        const int c0 = half * (cw / 2);
        for (int c = c0; c < c0 + cw / 2; c += 4) {
          float s[4] = {0.f, 0.f, 0.f, 0.f};
          for (int src = 0; src < csize; ++src)
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] += part[(src * cw + c + e) * 128];
          store4(crow + (it.j0 + crank * cw + c) * g.sCj, it.j0 + crank * cw + c, s[0], s[1], s[2], s[3]);
        }
        epi_sync();
        if (threadIdx.x == 0) mbar_arrive(done);
      }
      if (poison != poison) {
        const int m = mark_of(p.items, n, worker, nworkers);
        atomicOr(&marks[m >> 5], 1u << (m & 31));
      }
    }
    if (!ok && lane == 0) { *abort_flag = 1; atomicExch(p.status, 3u); }
    redo_marked<CG, AK, BKM>(p);
  }

  tc_fence_before();
  __syncthreads();
  if (ctas > 1) cluster_sync();      // peers write into this CTA's ring: leave together
  if (warp == kMmaWarp) {
    tc_fence_after();
    if (CG == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAccs * XN) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAccs * XN) : "memory");
  }
}

// ------------------------------------------------------------------ host side
XProblem convert(const GemmProblem& g, bool ak, bool bk, bool swap, int cg) {
  XProblem x{};
  x.nseg = 0;
  for (int s = 0; s < g.nseg; ++s) {
    const GemmSeg& q = g.seg[s];
    if (q.Q <= 0 || q.Kd <= 0) continue;
    XSeg& d = x.seg[x.nseg++];
    d = XSeg{static_cast<const float*>(q.A), static_cast<const float*>(q.B), q.sAb, q.sAq, ak ? q.sAi : q.sAk,
             q.sBb, q.sBq, bk ? q.sBj : q.sBk, q.Q, q.Kd};
    if (swap) {
      std::swap(d.A, d.B); std::swap(d.sAb, d.sBb); std::swap(d.sAq, d.sBq); std::swap(d.sAl, d.sBl);
    }
    x.chunks += q.Q * ((q.Kd + XK - 1) / XK);
  }
  x.C = static_cast<float*>(g.C);
  x.sCb = g.sCb; x.sCi = g.sCi; x.sCj = 1;
  x.M = g.M; x.N = g.N; x.batch = g.batch;
  if (swap) { std::swap(x.sCi, x.sCj); std::swap(x.M, x.N); }
  x.ntm = (x.M + XM * cg - 1) / (XM * cg); x.ntn = (x.N + XN - 1) / XN;
  x.tiles = x.ntm * x.ntn * x.batch;
  return x;
}

// microseconds, fitted to the sizes above: a chunk of 64 of the contraction of a CTA's (a pair's) tile, what a tile costs beside
// its chunks, and a tile summed over a cluster on top
// a tile that is stored element by element with the results' contiguous axis along a thread's columns, not along the lanes (backward at
// p = 0.9, CUDA cores / without regard to it / here: 8 x 2048, 5632, 16 tokens 169 / 148 / 83, 64 tokens 218 / 166 / 93; 8 x 4096,
// 11008, 16 tokens 597 / 472 / 240; long contractions choose as before: 4 x 1536, 333 tokens 163 / 163)
constexpr double kChunkUs[2] = {2.2, 1.7}, kTileUs = 1.0, kReduceUs = 4.0, kScatterUs = 3.0;

double chunk_us(const XProblem& g, int cg) {      // narrow tiles: the A parts cost what they cost
  const int last = g.N % XN, w = last ? (last + 15) / 16 * 16 : XN;
  const double full = g.ntn - (last ? 1 : 0), c = fmax(w / 128.0, 0.5);
  return kChunkUs[cg - 1] * (full + (last ? c : 0.0)) / g.ntn;
}

// time of the busiest cluster, items dealt round-robin, problem after problem
double plan_cost(const XProblem* g, int n, int cg, int csize, const int* split, int workers, bool vec) {
  double load_all = 0, worst = 0, len[2];
  long long items[2] = {0, 0};
  for (int i = 0; i < n; ++i) {
    const double c = split[i] ? (double)((g[i].chunks + csize - 1) / csize) : (double)g[i].chunks;
    len[i] = c * chunk_us(g[i], cg) + kTileUs + (split[i] ? kReduceUs : 0.0) + (!vec && g[i].sCj == 1 ? kScatterUs / (split[i] ? csize : 1) : 0.0);
    items[i] = split[i] ? g[i].tiles : (g[i].tiles + csize - 1) / csize;
    load_all += items[i] * len[i];
  }
  const long long first = items[0] % workers, total = items[0] + (n > 1 ? items[1] : 0);
  for (long long w : {0LL, first, first > 0 ? first - 1 : 0LL, total % workers, total % workers > 0 ? total % workers - 1 : 0LL}) {
    const long long a = items[0] / workers + (w < first), all = total / workers + (w < total % workers);
    worst = fmax(worst, a * len[0] + (n > 1 ? (all - a) * len[1] : 0.0));
  }
  return worst;
}

void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int cg, int ctas, int cluster) {
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = cg == 2 ? kSmem<2> : kSmem<1>;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
}

// Clusters that the device holds at once (1: no answer).  A schedule for more would leave whole clusters for a second round.
template <int CG>
int resident_clusters(int cluster) {
  static int cache[64][4] = {};
  const int slot = cluster == 2 ? 1 : (cluster == 4 ? 2 : 3);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  std::lock_guard<std::mutex> lock(host_cache_mutex());
  int& n = cache[dev][slot];
  if (n == 0) {
    n = 1;
    auto kernel = gemm_f32_kernel<CG, true, true, true>;       // the shared memory and the threads decide: the same for all forms
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem<CG>) == cudaSuccess) {
      cudaLaunchConfig_t cfg{};
      cudaLaunchAttribute attr{};
      cluster_config(cfg, &attr, CG, cluster * 64, cluster);
      int got = 0;
      if (cudaOccupancyMaxActiveClusters(&got, kernel, &cfg) == cudaSuccess && got > 0) n = got;
    }
    (void)cudaGetLastError();
  }
  return n;
}

template <int CG, bool AK, bool BKM, bool VEC>
cudaError_t launch_kernel(const XParams& p, int ctas, int kind, cudaStream_t st) {
  auto kernel = gemm_f32_kernel<CG, AK, BKM, VEC>;
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (std::lock_guard<std::mutex> lock(host_cache_mutex()); !attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem<CG>);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2] = {};
  cluster_config(cfg, attr, CG, ctas, p.csize * CG);
  cfg.stream = st;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  if (pdl_enabled()) cfg.numAttrs = 2;
  LaunchScope scope(kind, st);
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <int CG, bool VEC>
cudaError_t launch_layout(bool ak, bool bk, const XParams& p, int ctas, int kind, cudaStream_t st) {
  if (ak && bk) return launch_kernel<CG, true, true, VEC>(p, ctas, kind, st);
  if (ak) return launch_kernel<CG, true, false, VEC>(p, ctas, kind, st);
  if (bk) return launch_kernel<CG, false, true, VEC>(p, ctas, kind, st);
  return launch_kernel<CG, false, false, VEC>(p, ctas, kind, st);
}

}  // namespace

// Products of fewer operations than this stay on the CUDA cores, whose 32 x 32 tiles are spread over more SMs.  Either side of
// the lines (layer, CUDA cores / here, us): forward, 0.07 GFLOP 12.1 / 16.0, 0.21 GFLOP 27.2 / 20.4, 0.30 GFLOP 19.5 / 17.2;
// backward, 0.13 GFLOP a product 25.8 / 28.5 (2 x 256) but 44.2 / 26.3 (2 x 512), 0.15 GFLOP 40.6 / 34.4.
// Above them forward products of few tiles and a long contraction stay there, which the plan below puts behind the CUDA cores'
// (simt_forward_us): layer forward, 64 tokens of h 128, K 16384 23.5 / 60.7; 256 tokens 39.8 / 75.9; 100 tokens of 256,
// 8192 23.7 / 42.5; 512 tokens of 64, 4096 15.5 / 23.7 - but 1024 tokens of 128, 16384 138 / 77; 64 tokens of 8 x 2048, 5632 at
// p = 0.9 153 / 67.  (720 shapes of 0.02 to 5 GFLOP, timed from graphs: 85 were slower here than on the CUDA cores, up to 2.6 times;
// now 22, by 22 % and less, most by 1 to 2 us.)
constexpr double kMinForward = 2.0e8, kMinGradient = 1.45e8;

bool launch_gemm_f32(const GemmProblem* problems, int n, bool ak, bool bk, bool vec, cudaStream_t st, cudaError_t* err) {
  double work = 0;
  for (int i = 0; i < n; ++i)
    for (int k = 0; k < problems[i].nseg; ++k) {
      const GemmSeg& e = problems[i].seg[k];
      if (e.Q > 0 && e.Kd > 0) work += 2.0 * problems[i].batch * problems[i].M * problems[i].N * e.Q * e.Kd;
    }
  if (work < (ak && bk ? kMinForward : kMinGradient)) return false;
  double best = -1;
  XParams p{};
  bool best_swap = false;
  int ctas = 0;
  const int sms = sm_count();
  int cg = 1;
  for (int form = 0; form < 4; ++form) {
    const int swap = form & 1, pair = 1 + (form >> 1);
    XProblem g[2];
    for (int i = 0; i < n; ++i) g[i] = convert(problems[i], ak, bk, swap != 0, pair);
    if (n > 1 && g[1].chunks > g[0].chunks) std::swap(g[0], g[1]);         // longest contraction first
    for (int c = 1; c * pair <= 8; c *= 2) {
      const int workers = c * pair == 1 ? sms : (pair == 2 ? resident_clusters<2>(2 * c) : resident_clusters<1>(c));
      for (int m = c == 1 ? 0 : 1; m < (c == 1 ? 1 : 1 << n); ++m) {
        const int split[2] = {m & 1, m >> 1 & 1};
        bool can = true;
        for (int i = 0; i < n; ++i) can &= !split[i] || g[i].chunks >= c;
        if (!can) continue;
        const double cost = plan_cost(g, n, pair, c, split, workers, vec);
        if (best >= 0 && cost >= best) continue;
        best = cost; best_swap = swap != 0; cg = pair;
        p.nprob = n; p.csize = c;
        p.items = 0;
        for (int i = 0; i < n; ++i) {
          p.p[i] = g[i];
          p.p[i].split = split[i];
          p.items += split[i] ? g[i].tiles : (g[i].tiles + c - 1) / c;
          if (i == 0) p.items0 = p.items;
        }
        ctas = (p.items < workers ? p.items : workers) * c * pair;
      }
    }
  }
  if (ak && bk && best >= simt_forward_us(problems, n)) return false;
  p.status = device_status_word();
  if (!p.status) { *err = cudaErrorUnknown; return true; }
  static const uint32_t cap_env = [] { const char* e = getenv("CAAT_TC_SPINCAP"); return e ? (uint32_t)atoi(e) : 0u; }();
  p.spin_cap = cap_env >= 1024 ? cap_env : kSpinCap;
  static const int stall = [] { const char* e = getenv("CAAT_TC_DEBUG"); return e ? atoi(e) & 1024 : 0; }();
  p.stall = stall;
  const int kind = ak && bk ? CAAT_K_TC_FORWARD : (ak ? CAAT_K_TC_DGRAD : CAAT_K_TC_WGRAD);
  const bool a = best_swap ? bk : ak, b = best_swap ? ak : bk;
  if (cg == 2) *err = vec ? launch_layout<2, true>(a, b, p, ctas, kind, st) : launch_layout<2, false>(a, b, p, ctas, kind, st);
  else *err = vec ? launch_layout<1, true>(a, b, p, ctas, kind, st) : launch_layout<1, false>(a, b, p, ctas, kind, st);
  return true;
}

}  // namespace caat
