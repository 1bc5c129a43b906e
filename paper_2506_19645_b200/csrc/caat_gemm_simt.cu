// Generic strided batched GEMM on CUDA cores with fp32 accumulation.
//
// It serves small fp32 products (large ones run on the tensor cores in three bf16 parts per operand, caat_gemm_f32.cu, unless
// the CUDA cores are asked for) and bf16 shapes the tensor-core kernels do not take (K_r not a multiple of 8).  Every operand is addressed through element strides, one
// of which is 1, so the same kernels run the forward product, the data gradient and the weight gradient; the "two
// segment" form covers the [shared | private] split of the contraction axis, and the products of a call that do not
// depend on each other (shared and private columns) share one launch.
//
// Arithmetic is packed fp32 (two IEEE FMAs per instruction): a loop of register-only FMAs runs at 63 TFLOP/s packed and
// 54 scalar on this part.  Two kernels:
//  * warp tiles: 32 x 32 outputs per CTA, the contraction dealt over its eight warps and over the CTAs of a cluster,
//    every warp with k-tiles of its own (no CTA barrier until the partial tiles are summed, warps in order, then CTAs in
//    order through distributed shared memory: deterministic).  Both operands [row][k] in shared memory, an FMA pair is
//    two k of one output.  Every forward product (its operands lie that way in memory), and small gradients.
//  * CTA tiles: 128 x 64 outputs, 256 threads, k-tiles of 16 in a three-stage ring, two CTAs per SM, an FMA pair is two
//    neighbouring columns.  The gradients of problems that fill the GPU.
#include <cooperative_groups.h>

#include "caat_rows_common.cuh"

namespace caat {
namespace {

namespace cgx = cooperative_groups;
using rows::fma2;

constexpr int kMaxProblems = 2;
struct GemmList {
  int n;
  GemmProblem p[kMaxProblems];
  int tile_end[kMaxProblems];   // tiles of problems 0..i
  int ntn[kMaxProblems], ntm[kMaxProblems];
  int ksplit[kMaxProblems];     // CTA tiles: 1, or the cluster size: a tile's contraction is split over a cluster
  int cta_end[kMaxProblems];    // CTA tiles: CTAs of problems 0..i
};
struct Tile { int b, i0, j0; };

__device__ __forceinline__ Tile decode(const GemmList& L, int prob, int tile, int BM, int BN) {
  Tile t;
  int rem = prob ? tile - L.tile_end[0] : tile;
  const int ntn = L.ntn[prob], ntm = L.ntm[prob];
  t.j0 = rem % ntn * BN; rem /= ntn;
  t.i0 = rem % ntm * BM;
  t.b = rem / ntm;
  return t;
}

template <typename T_>
__device__ __forceinline__ float ldf(const void* p, long long off);
template <>
__device__ __forceinline__ float ldf<float>(const void* p, long long off) {
  return static_cast<const float*>(p)[off];
}
template <>
__device__ __forceinline__ float ldf<__nv_bfloat16>(const void* p, long long off) {
  return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[off]);
}

// Four consecutive elements along the operand's unit stride, `left` of them inside the matrix (may be <= 0 or > 4).
template <typename T_>
__device__ __forceinline__ float4 ld4(const void* p, long long off, int left) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (left > 0) v.x = ldf<T_>(p, off);
  if (left > 1) v.y = ldf<T_>(p, off + 1);
  if (left > 2) v.z = ldf<T_>(p, off + 2);
  if (left > 3) v.w = ldf<T_>(p, off + 3);
  return v;
}
// 16 bytes into shared memory, the last 16 - `bytes` of them zero (bytes = 0: the source is not read)
__device__ __forceinline__ void cp_async16z(float* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
// A run of four-element pieces, `step` elements apart in memory and `dstep` floats apart in shared memory: piece u is
// inside the matrix while first + inc * u < limit, and then holds `left` elements.  One address per run: with the 64-bit index
// arithmetic of a piece at a time the packed FMAs were 40 % of the forward kernel's instructions (9.4 GFLOP forward of
// 4 x 2000 tokens, h = 768: 300 us, now 266).
template <typename T_, bool VEC, int NU>
__device__ __forceinline__ void put_run(float* dst, int dstep, const void* src, long long off, long long step, int first, int inc,
                                        int limit, int left) {
  if (VEC) {
    const int n = left >= 4 ? 16 : (left > 0 ? 4 * left : 0);
    const float* p = static_cast<const float*>(src) + off;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      cp_async16z(dst + u * dstep, p, first + inc * u < limit ? n : 0);     // 0 bytes: the source is not read
      p += step;
    }
  } else {
#pragma unroll
    for (int u = 0; u < NU; ++u)
      *reinterpret_cast<float4*>(dst + u * dstep) = ld4<T_>(src, off + u * step, first + inc * u < limit ? left : 0);
  }
}

// Position in the contraction: segment, rank q of the segment, k offset.  The k-tiles of all segments and ranks form
// one sequence.
struct KPos { int seg, q, k0; };

template <int BK>
__host__ __device__ __forceinline__ int seg_tiles(const GemmSeg& s) {
  return s.Q > 0 && s.Kd > 0 ? s.Q * ((s.Kd + BK - 1) / BK) : 0;
}
template <int BK>
__host__ __device__ __forceinline__ int ktiles_of(const GemmProblem& g) {
  int n = seg_tiles<BK>(g.seg[0]);
  if (g.nseg > 1) n += seg_tiles<BK>(g.seg[1]);
  return n;
}
template <int BK>
__device__ __forceinline__ KPos kpos_at(const GemmProblem& g, int n) {    // the n-th k-tile
  KPos p{0, 0, 0};
  const int n0 = seg_tiles<BK>(g.seg[0]);
  if (n >= n0) { p.seg = 1; n -= n0; }
  const int per = (g.seg[p.seg].Kd + BK - 1) / BK;
  p.q = n / per;
  p.k0 = (n - p.q * per) * BK;
  return p;
}
template <int BK>
__device__ __forceinline__ void kpos_next(const GemmProblem& g, KPos& p) {   // callers count the tiles
  p.k0 += BK;
  if (p.k0 >= g.seg[p.seg].Kd) {
    p.k0 = 0;
    if (++p.q >= g.seg[p.seg].Q) { p.q = 0; p.seg = 1; }
  }
}

__device__ __forceinline__ void store_out(const GemmProblem& g, int b, int i, int j, float v, bool f32) {
  const long long off = (long long)b * g.sCb + (long long)i * g.sCi + j;
  if (f32) static_cast<float*>(g.C)[off] = v;
  else static_cast<__nv_bfloat16*>(g.C)[off] = __float2bfloat16_rn(v);
}

// ------------------------------------------------------------------ CTA tiles
constexpr int TBM = 128, TBN = 64, TBK = 16, kTStages = 3, kTThreads = 256;
constexpr int LDA = TBM + 4, LDB = TBN + 4;            // row pitch of the [k][row] tiles (16-byte multiples)
constexpr int kTA = TBK * LDA, kTB = TBK * LDB;        // floats per stage

// AK: A's unit stride is along k (data gradient), else along i (weight gradient); B's is along j.
// Both tiles are [k][row] in shared memory.  An operand that lies so in memory is copied by cp.async; an A that lies
// [row][k] passes through registers (loaded before a k-tile's products, stored after them).  A warp's 128-bit shared load
// costs four cycles of the SM's return path however many lanes share an address, so the thread tile decides: 8 x 8
// outputs need four such loads per k for 32 packed FMAs.  Warps 0-3 and 4-7 cover the tile once each and take every
// other group of four k; the two halves exchange half of their sums at the end, which leaves 32 finished outputs per
// thread.  4 x (2000 x 768) gradient against 768 x 3072 weights (9.4 GFLOP): data gradient 437 -> 297 us, weight
// gradient 738 -> 219 us (43 TFLOP/s) over the former 64 x 64 tiles with 4 x 4 outputs per thread.
template <typename T_, bool AK, bool VEC>
__global__ void __launch_bounds__(kTThreads, 2) gemm_simt_tiled(const __grid_constant__ GemmList L, int csize) {
  constexpr int kSm = kTStages * (kTA + kTB) > 32 * kTThreads ? kTStages * (kTA + kTB) : 32 * kTThreads;
  __shared__ __align__(16) float sm[kSm];
  pdl_wait();
  cgx::cluster_group cluster = cgx::this_cluster();
  // the CTAs of a cluster share a tile of a split problem (a slice of its k-tiles each) or have a tile of their own
  const int crank = csize > 1 ? (int)cluster.block_rank() : 0;
  const int prob = (L.n > 1 && (int)blockIdx.x >= L.cta_end[0]) ? 1 : 0;
  const bool split = L.ksplit[prob] > 1;
  const int first = (int)blockIdx.x - (prob ? L.cta_end[0] : 0), tile0 = prob ? L.tile_end[0] : 0;
  const int tile = tile0 + (split ? first / csize : first);
  if (tile >= L.tile_end[prob]) return;            // padding to whole clusters (never in a split problem)
  const Tile tl = decode(L, prob, tile, TBM, TBN);
  const GemmProblem& g = L.p[prob];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int khalf = warp >> 2;
  const int r0 = (warp & 1) * 64 + (lane & 7) * 4, c0 = ((warp >> 1) & 1) * 32 + (lane >> 3) * 4;
  auto row_of = [&](int x) { return r0 + (x & 3) + (x >> 2) * 32; };
  auto col_of = [&](int y) { return c0 + (y & 3) + (y >> 2) * 16; };
  float2 acc[8][4];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = make_float2(0.f, 0.f);

  float4 ra[2];                    // A on its way through registers
  auto ldv = [&](const void* src, long long off, int left) {
    return VEC && left >= 4 ? *reinterpret_cast<const float4*>(static_cast<const float*>(src) + off) : ld4<T_>(src, off, left);
  };
  auto fetch = [&](const KPos& p, float* As) {
    const GemmSeg& s = g.seg[p.seg];
    float* Bs = As + kTA;
    const long long a0 = (long long)tl.b * s.sAb + (long long)p.q * s.sAq;
    const long long b0 = (long long)tl.b * s.sBb + (long long)p.q * s.sBq;
    if (AK) {
      const int i = tl.i0 + (tid >> 2), k = p.k0 + (tid & 3) * 4, left = s.Kd - k;
      const long long off = a0 + (long long)i * s.sAi + k;
#pragma unroll
      for (int r = 0; r < 2; ++r) ra[r] = ldv(s.A, off + r * (kTThreads / 4) * s.sAi, i + r * (kTThreads / 4) < g.M ? left : 0);
    } else {
      const int kk = tid >> 5, row = (tid & 31) * 4, i = tl.i0 + row, k = p.k0 + kk;
      put_run<T_, VEC, 2>(As + kk * LDA + row, 8 * LDA, s.A, a0 + (long long)k * s.sAk + i, 8 * s.sAk, k, 8, s.Kd, g.M - i);
    }
    const int kk = tid >> 4, col = (tid & 15) * 4, j = tl.j0 + col, k = p.k0 + kk;
    put_run<T_, VEC, 1>(Bs + kk * LDB + col, 0, s.B, b0 + (long long)k * s.sBk + j, 0, k, 1, s.Kd, g.N - j);
  };
  auto park = [&](float* As) {
    if (AK) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float* d = As + ((tid & 3) * 4) * LDA + ((tid + r * kTThreads) >> 2);
        d[0] = ra[r].x; d[LDA] = ra[r].y; d[2 * LDA] = ra[r].z; d[3 * LDA] = ra[r].w;
      }
    }
  };

  int begin = 0, left = ktiles_of<TBK>(g);     // k-tiles still to fetch
  if (split) {
    begin = (int)((long long)left * crank / csize);
    left = (int)((long long)left * (crank + 1) / csize) - begin;
  }
  KPos ahead = kpos_at<TBK>(g, begin);
  const int ntiles = left;
  float* const ring_end = sm + kTStages * (kTA + kTB);
  float* fill = sm;
#pragma unroll
  for (int q = 0; q < kTStages - 1; ++q) {     // one commit group per k-tile, empty past the end
    if (left > 0) { fetch(ahead, fill); kpos_next<TBK>(g, ahead); --left; park(fill); }
    asm volatile("cp.async.commit_group;" ::: "memory");
    fill += kTA + kTB;
  }
  const float* As = sm;
  for (int done = 0; done < ntiles; ++done) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kTStages - 2) : "memory");
    __syncthreads();               // this stage has landed for every thread, and the one refilled below is read
    const bool more = left > 0;
    if (more) { fetch(ahead, fill); kpos_next<TBK>(g, ahead); --left; }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* Bs = As + kTA;
#pragma unroll
    for (int kk = 0; kk < TBK; kk += 8) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = kk + 4 * khalf + e;
        const float4 a0 = *reinterpret_cast<const float4*>(As + k * LDA + r0);
        const float4 a1 = *reinterpret_cast<const float4*>(As + k * LDA + r0 + 32);
        const float4 b0 = *reinterpret_cast<const float4*>(Bs + k * LDB + c0);
        const float4 b1 = *reinterpret_cast<const float4*>(Bs + k * LDB + c0 + 16);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
        for (int x = 0; x < 8; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) acc[x][y] = fma2(rows::f2(av[x]), bv[y], acc[x][y]);
      }
    }
    if (more) park(fill);
    fill = fill + (kTA + kTB) == ring_end ? sm : fill + (kTA + kTB);
    As = As + (kTA + kTB) == ring_end ? sm : As + (kTA + kTB);
  }
  // this thread's 32 outputs: four of its eight rows x eight columns
  float out[32];
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int o = 0; o < 32; ++o) {   // the rows the other half keeps
    const float2 lo = acc[o >> 3][(o & 7) >> 1], hi = acc[4 + (o >> 3)][(o & 7) >> 1];
    const float2 v = khalf ? lo : hi;
    sm[o * kTThreads + tid] = (o & 1) ? v.y : v.x;
  }
  __syncthreads();
#pragma unroll
  for (int o = 0; o < 32; ++o) {
    const float2 lo = acc[o >> 3][(o & 7) >> 1], hi = acc[4 + (o >> 3)][(o & 7) >> 1];
    const float2 v = khalf ? hi : lo;
    out[o] = ((o & 1) ? v.y : v.x) + sm[o * kTThreads + (tid ^ 128)];
  }
  auto out_row = [&](int o) { return tl.i0 + row_of((khalf ? 4 : 0) + (o >> 3)); };
  auto out_col = [&](int o) { return tl.j0 + col_of(o & 7); };
  const bool f32 = g.c_f32 || sizeof(T_) == 4;
  if (split) {
    // the CTAs of the cluster in order; every CTA finishes its slice of the 32 outputs of each thread
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 32; ++o) sm[o * kTThreads + tid] = out[o];
    cluster.sync();
    const int per = 32 / csize;
    for (int o = crank * per; o < (crank + 1) * per; ++o) {
      float v = 0.f;
      for (int c = 0; c < csize; ++c) v += cluster.map_shared_rank(sm, c)[o * kTThreads + tid];
      if (out_row(o) < g.M && out_col(o) < g.N) store_out(g, tl.b, out_row(o), out_col(o), v, f32);
    }
    cluster.sync();                // a peer may still be reading this CTA's sums
    return;
  }
#pragma unroll
  for (int o = 0; o < 32; o += 4) {
    if (out_row(o) >= g.M) continue;
    if (VEC && out_col(o) + 3 < g.N) {     // VEC: the output rows are 16-byte aligned as well
      *reinterpret_cast<float4*>(static_cast<float*>(g.C) + (long long)tl.b * g.sCb + (long long)out_row(o) * g.sCi + out_col(o)) =
          make_float4(out[o], out[o + 1], out[o + 2], out[o + 3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (out_col(o + e) < g.N) store_out(g, tl.b, out_row(o), out_col(o + e), out[o + e], f32);
    }
  }
}

// ------------------------------------------------------------------ warp tiles
constexpr int SB = 32;                         // tile edge and k-tile
constexpr int kSPitch = SB + 4;                // row pitch of a warp's [row][k] tile: 8 rows cover all banks
constexpr int kWarpTile = 2 * SB * kSPitch;    // floats: A tile, B tile
constexpr int kSmallWarps = 8;

template <typename T_, bool AK, bool BKF, bool VEC>
__global__ void __launch_bounds__(256, 2) gemm_simt_small(const __grid_constant__ GemmList L, int csize, int nbuf) {
  extern __shared__ __align__(16) float dsm[];
  pdl_wait();
  cgx::cluster_group cluster = cgx::this_cluster();
  const int crank = csize > 1 ? (int)cluster.block_rank() : 0;
  const int tile = (int)blockIdx.x / csize, prob = (L.n > 1 && tile >= L.tile_end[0]) ? 1 : 0;
  const Tile tl = decode(L, prob, tile, SB, SB);
  const GemmProblem& g = L.p[prob];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lm = lane & 7, ln = lane >> 3;     // rows lm + 8 x, columns ln + 4 y
  float* mine = dsm + (size_t)warp * nbuf * kWarpTile;

  // one k-tile of this warp into its own buffer: [row][k]
  auto fetch = [&](const KPos& p, float* dst) {
    const GemmSeg& s = g.seg[p.seg];
    const long long a0 = (long long)tl.b * s.sAb + (long long)p.q * s.sAq;
    const long long b0 = (long long)tl.b * s.sBb + (long long)p.q * s.sBq;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const bool kf = half == 0 ? AK : BKF;
      const void* src = half == 0 ? s.A : s.B;
      const long long base = half == 0 ? a0 : b0, row_ld = half == 0 ? s.sAi : s.sBj, k_ld = half == 0 ? s.sAk : s.sBk;
      const int r0 = half == 0 ? tl.i0 : tl.j0, rmax = half == 0 ? g.M : g.N;
      float* d = dst + half * (SB * kSPitch);
      const int fast = (lane & 7) * 4, slow = lane >> 3;
      if (kf) {
        const int row = r0 + slow, k = p.k0 + fast;
        put_run<T_, VEC, 8>(d + slow * kSPitch + fast, 4 * kSPitch, src, base + (long long)row * row_ld + k, 4 * row_ld, row, 4, rmax,
                            s.Kd - k);
      } else {
        const int row = r0 + fast, k = p.k0 + slow;
        long long off = base + (long long)k * k_ld + row;
#pragma unroll
        for (int u = 0; u < 8; ++u, off += 4 * k_ld) {
          const int left = k + 4 * u < s.Kd ? rmax - row : 0;
          const float4 v = VEC && left >= 4 ? *reinterpret_cast<const float4*>(static_cast<const float*>(src) + off)
                                            : ld4<T_>(src, off, left);
          float* t = d + fast * kSPitch + slow + 4 * u;
          t[0] = v.x; t[kSPitch] = v.y; t[2 * kSPitch] = v.z; t[3 * kSPitch] = v.w;
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  float2 acc[4][8];                            // a pair: even and odd k of one output
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) acc[x][y] = make_float2(0.f, 0.f);
  // the k-tiles are dealt round-robin over the cluster's warps
  const int total = ktiles_of<SB>(g), stride = csize * kSmallWarps;
  int n = crank * kSmallWarps + warp, buf = 0;
  if (n < total) fetch(kpos_at<SB>(g, n), mine);
  for (; n < total; n += stride) {
    const bool more = n + stride < total;
    if (more && nbuf > 1) {
      fetch(kpos_at<SB>(g, n + stride), mine + (buf ^ 1) * kWarpTile);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    const float* A = mine + buf * kWarpTile;
    const float* B = A + SB * kSPitch;
#pragma unroll 4
    for (int k = 0; k < SB; k += 4) {
      float4 av[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) av[x] = *reinterpret_cast<const float4*>(A + (lm + 8 * x) * kSPitch + k);
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        const float4 bv = *reinterpret_cast<const float4*>(B + (ln + 4 * y) * kSPitch + k);
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x][y] = fma2(make_float2(av[x].x, av[x].y), make_float2(bv.x, bv.y), acc[x][y]);
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x][y] = fma2(make_float2(av[x].z, av[x].w), make_float2(bv.z, bv.w), acc[x][y]);
      }
    }
    __syncwarp();                       // the buffer may be refilled
    if (more && nbuf == 1) fetch(kpos_at<SB>(g, n + stride), mine);
    if (nbuf > 1) buf ^= 1;
  }
  // warps in order, then CTAs of the cluster in order
  float* part = mine;                   // this warp's partial tile, [row][SB + 1]
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) part[(lm + 8 * x) * (SB + 1) + ln + 4 * y] = acc[x][y].x + acc[x][y].y;
  __syncthreads();
  float out[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kSmallWarps; ++w) v += dsm[(size_t)w * nbuf * kWarpTile + (warp + 8 * u) * (SB + 1) + lane];
    out[u] = v;
  }
  const bool f32 = g.c_f32 || sizeof(T_) == 4;
  if (csize == 1) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = tl.i0 + warp + 8 * u, j = tl.j0 + lane;
      if (i < g.M && j < g.N) store_out(g, tl.b, i, j, out[u], f32);
    }
    return;
  }
  float* sum = dsm + (size_t)kSmallWarps * nbuf * kWarpTile;    // [SB][SB], read by the peers
#pragma unroll
  for (int u = 0; u < 4; ++u) sum[(warp + 8 * u) * SB + lane] = out[u];
  cluster.sync();
  const int rows = SB / csize;
  for (int q = threadIdx.x; q < rows * SB; q += 256) {
    const int row = crank * rows + q / SB, col = q % SB;
    float v = 0.f;
    for (int c = 0; c < csize; ++c) v += cluster.map_shared_rank(sum, c)[row * SB + col];
    const int i = tl.i0 + row, j = tl.j0 + col;
    if (i < g.M && j < g.N) store_out(g, tl.b, i, j, v, f32);
  }
  cluster.sync();                       // a peer may still be reading this CTA's tile
}

// ------------------------------------------------------------------ host side
void set_tiles(GemmList& L, int BM, int BN) {
  int end = 0;
  for (int i = 0; i < L.n; ++i) {
    L.ntn[i] = (L.p[i].N + BN - 1) / BN;
    L.ntm[i] = (L.p[i].M + BM - 1) / BM;
    end += L.ntn[i] * L.ntm[i] * L.p[i].batch;
    L.tile_end[i] = end;
  }
}

void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int ctas, int threads, int csize, size_t smem,
                    cudaStream_t st) {
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
}

// cluster size of the warp-tile kernel (tiles set): a power of two up to the portable size, while every warp has a k-tile
int small_cluster(const GemmList& L, int* ktiles_out) {
  const int slots = 2 * sm_count(), tiles = L.tile_end[L.n - 1];
  int ktiles = 1, csize = 1;            // of the longest contraction
  for (int i = 0; i < L.n; ++i) {
    const int k = ktiles_of<SB>(L.p[i]);
    if (k > ktiles) ktiles = k;
  }
  while (csize < 8 && 2 * csize * kSmallWarps <= ktiles && 2 * tiles * csize <= slots) csize *= 2;
  *ktiles_out = ktiles;
  return csize;
}

// Gradients of at least this much work per SM, in k-tiles of the CTA-tile kernel (0.26 MFLOP), run on it.  Measured
// (whole backward of a layer, warp tiles / CTA tiles): 5.4 per SM 39 / 46 us, 13.8 67 / 57 us, 31 132 / 97 us.  Forward
// products stay on the warp tiles at any size: 61 per SM 86 us against 119 on CTA tiles with the operands transposed on
// the way, 243 per SM 321 against 390 us, 486 per SM 624 against 710 us.
constexpr double kCtaTileWork = 10;

template <typename T_, bool AK, bool BKF, bool VEC>
cudaError_t launch_layout(GemmList& L, cudaStream_t st) {
  cudaLaunchAttribute attr[2] = {};
  cudaLaunchConfig_t cfg{};
  const int slots = 2 * sm_count();     // resident CTAs of either kernel
  if constexpr (!BKF) {
    set_tiles(L, TBM, TBN);
    double work = 0;
    int longest = 0;
    for (int i = 0; i < L.n; ++i) {
      const int k = ktiles_of<TBK>(L.p[i]);
      work += (double)(L.tile_end[i] - (i ? L.tile_end[i - 1] : 0)) * k;
      if (k > longest) longest = k;
    }
    if (work >= kCtaTileWork * sm_count()) {
      // A tile whose contraction is longer than a CTA slot's fair share would finish alone: split it over a cluster.
      const double share = work / slots > 8 ? work / slots : 8;
      int csize = 1;
      while (csize < 8 && longest > 1.1 * share * csize) csize *= 2;
      int ctas = 0;
      for (int i = 0; i < L.n; ++i) {
        const int tiles = L.tile_end[i] - (i ? L.tile_end[i - 1] : 0);
        L.ksplit[i] = csize > 1 && ktiles_of<TBK>(L.p[i]) > 1.1 * share ? csize : 1;
        ctas += L.ksplit[i] > 1 ? tiles * csize : round_up(tiles, csize);
        L.cta_end[i] = ctas;
      }
      cluster_config(cfg, attr, ctas, kTThreads, csize, 0, st);
      LaunchScope scope(CAAT_K_GEMM_CUDA_CORE, st);
      return cudaLaunchKernelEx(&cfg, gemm_simt_tiled<T_, AK, VEC>, (const GemmList&)L, csize);
    }
  }
  set_tiles(L, SB, SB);
  const int tiles = L.tile_end[L.n - 1];
  int ktiles;
  const int csize = small_cluster(L, &ktiles);
  const int nbuf = ktiles > csize * kSmallWarps && tiles * csize <= sm_count() ? 2 : 1;
  const size_t smem = ((size_t)kSmallWarps * nbuf * kWarpTile + SB * SB) * sizeof(float);
  auto kernel = gemm_simt_small<T_, AK, BKF, VEC>;
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (std::lock_guard<std::mutex> lock(host_cache_mutex()); !attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  cluster_config(cfg, attr, tiles * csize, 256, csize, smem, st);
  LaunchScope scope(CAAT_K_GEMM_CUDA_CORE, st);
  return cudaLaunchKernelEx(&cfg, kernel, (const GemmList&)L, csize, nbuf);
}

template <typename T_, bool VEC>
cudaError_t launch_typed(GemmList& L, bool ak, bool bk, cudaStream_t st) {
  if (ak && bk) return launch_layout<T_, true, true, VEC>(L, st);       // forward
  if (ak) return launch_layout<T_, true, false, VEC>(L, st);            // data gradient
  return launch_layout<T_, false, false, VEC>(L, st);                   // weight gradient
}

}  // namespace

// A forward product's time on the warp-tile kernel on the scale of the tensor-core kernel's plan (caat_gemm_f32.cu), in us: the
// serial k-tiles of a warp and the k-tiles per SM.  Where no product is wider than a tile on its narrow side the
// tensor-core kernel's tiles are at their emptiest, which its plan does not see.
double simt_forward_us(const GemmProblem* problems, int n) {
  GemmList L{};
  bool narrow = true;
  for (int i = 0; i < n; ++i) {
    L.p[L.n++] = problems[i];
    narrow &= problems[i].M <= SB || problems[i].N <= SB;
  }
  set_tiles(L, SB, SB);
  int ktiles;
  const int csize = small_cluster(L, &ktiles);
  double work = 0;
  for (int i = 0; i < L.n; ++i) work += (double)(L.tile_end[i] - (i ? L.tile_end[i - 1] : 0)) * ktiles_of<SB>(L.p[i]);
  const int serial = (ktiles + csize * kSmallWarps - 1) / (csize * kSmallWarps);
  return (2.25 * serial + 0.20 * work / sm_count()) * (narrow ? 0.8 : 1.0);
}

cudaError_t launch_gemm_simt(const GemmProblem* problems, int n, caat_dtype dtype, int force_simt, cudaStream_t st) {
  GemmList L{};
  for (int i = 0; i < n; ++i) {
    if (problems[i].M <= 0 || problems[i].N <= 0 || problems[i].batch <= 0) continue;
    if (L.n == kMaxProblems) return cudaErrorInvalidValue;
    L.p[L.n++] = problems[i];
  }
  if (L.n == 0) return cudaSuccess;
  // one launch takes one operand layout (a stride of 1 on both axes fits either); 16-byte accesses need every address
  // along the unit stride on that grid
  bool can_ak = true, can_ai = true, can_bk = true, can_bj = true;
  for (int i = 0; i < L.n; ++i) {
    if ((long long)L.p[i].M * L.p[i].N * L.p[i].batch / 1024 > 200000000LL) return cudaErrorInvalidConfiguration;
    for (int s = 0; s < L.p[i].nseg; ++s) {
      const GemmSeg& q = L.p[i].seg[s];
      if (q.Q <= 0 || q.Kd <= 0) continue;
      can_ak &= q.sAk == 1; can_ai &= q.sAi == 1;
      can_bk &= q.sBk == 1; can_bj &= q.sBj == 1;
    }
  }
  bool ak, bk;
  if (can_ak && can_bk) ak = bk = true;                   // forward
  else if (can_ak && can_bj) { ak = true; bk = false; }   // data gradient
  else if (can_ai && can_bj) ak = bk = false;             // weight gradient
  else return cudaErrorInvalidValue;
  bool vec = dtype == CAAT_F32;
  for (int i = 0; i < L.n; ++i) {
    const GemmProblem& g = L.p[i];
    if (reinterpret_cast<uintptr_t>(g.C) % 16 || g.sCb % 4 || g.sCi % 4) vec = false;
    for (int s = 0; s < g.nseg; ++s) {
      const GemmSeg& q = g.seg[s];
      if (q.Q <= 0 || q.Kd <= 0) continue;
      if (reinterpret_cast<uintptr_t>(q.A) % 16 || reinterpret_cast<uintptr_t>(q.B) % 16 || (ak ? q.sAi : q.sAk) % 4 ||
          (bk ? q.sBj : q.sBk) % 4 || q.sAb % 4 || q.sAq % 4 || q.sBb % 4 || q.sBq % 4)
        vec = false;
    }
  }
  if (dtype == CAAT_BF16) return launch_typed<__nv_bfloat16, false>(L, ak, bk, st);
  cudaError_t err;
  if (!force_simt && launch_gemm_f32(L.p, L.n, ak, bk, vec, st, &err)) return err;
  return vec ? launch_typed<float, true>(L, ak, bk, st) : launch_typed<float, false>(L, ak, bk, st);
}

}  // namespace caat
