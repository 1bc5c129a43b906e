// bf16 tensor-core GEMMs for sm_100a: TMA -> shared-memory ring -> tcgen05.mma with the
// fp32 accumulator in tensor memory -> tcgen05.ld epilogue.
//
// One persistent, warp-specialised kernel serves the three contractions of the layer:
//   forward   Zt = Y W^T        A = Y  (K-major),  B = W (K-major)
//   dgrad     dY = dZt W        A = dZt (K-major), B = W (N-major: K_r contiguous)
//   wgrad     dW = dZt^T Y      A = dZt (M-major: channels contiguous), B = Y (N-major)
// where dZt / Zt live in the split scratch layout [shared once | private per rank].
// Shared output columns of the forward accumulate over ALL ranks in one accumulator (the
// partial channel-reduce of Eq. A3 becomes a longer contraction), so rank partials of the
// shared channels never exist in memory.
//
// Roles per CTA (224 threads): warp 0 issues the TMA loads of the A operand and warp 6 those
// of the B operand (one thread issuing every box of a stage was the limiter when a stage is
// four boxes; two instruction streams walk the same schedule independently), warp 1 issues
// MMAs and owns the tensor-memory allocation, warps 2-5 drain accumulators (tcgen05.ld) and
// store.  Two
// accumulators of up to 256 columns alternate so a tile's epilogue overlaps the next
// tile's MMAs.  Every mbarrier wait is bounded; on a timeout the kernel records a status
// word, drains its own copies in flight, frees tensor memory and returns.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <utility>

#include "caat_tc_ptx.cuh"

namespace caat {
namespace {

using namespace tc;

constexpr int BM = 128;           // rows of an output tile (UMMA M, cta_group::1)
constexpr int BK = 64;            // contraction elements per pipeline stage (128 bytes of bf16)
constexpr int UMMA_K = 16;        // contraction elements per tcgen05.mma (kind::f16)
constexpr int kThreads = 224;     // warps: 0 = A producer, 1 = MMA issuer, 2..5 = epilogue, 6 = B producer
constexpr int kProducerB = 6;
constexpr int kAccCols = 256;     // column stride between the two accumulators
constexpr int kTmemCols = 512;
constexpr uint32_t kSpinCap = 1u << 22;
constexpr int kMaxStages = 8;
constexpr int kSlabBytes = 128;   // an epilogue warp drains slabs of 32 rows x 128 bytes (64 bf16 / 32 fp32 columns)
constexpr int kCBuf = 32 * kSlabBytes;            // one output staging buffer of one epilogue warp
constexpr int kCStage = 4 * 2 * kCBuf;            // four warps, two buffers each
// Measurement aids that make results wrong (phase ablation: skipped loads, stores, barriers) and the
// tile-shape overrides exist only in builds compiled with -DCAAT_MEASUREMENT_AIDS; the library as
// built by build.py honours none of them.  Bit 1024 (a stage wait made to run out, for the time-out
// test) stays: it changes no result of a call that returns CAAT_OK.
#ifdef CAAT_MEASUREMENT_AIDS
constexpr int kAidMask = ~0;
#else
constexpr int kAidMask = 1024;
#endif

constexpr int kMaxRegions = 6;      // four, but for the launch of a block's four gradient products

struct Unit {            // one contraction segment of a tile
  int mapA, mapB;        // indices into the tensor-map array
  int ak0, am0;          // offsets added to A's K / M coordinate
  int bk0, bn0;          // offsets added to B's K / N coordinate
  int a_zb, a_zq;        // A's z coordinate = b * a_zb + q * a_zq
  int b_zb, b_zq;
  int Q;                 // rank loop (forward shared columns: all ranks, else 1)
  int ksteps;            // stages per q = ceil(extent / BK)
};

struct Region {          // a family of output tiles with the same operand wiring
  int nunits;
  Unit u[2];
  int M, N, batch;       // valid output extents per batch
  int mtiles, ntiles;    // the output goes through the region's own tensor map (TMA store);
                         // its z coordinate is split * batch + b
  float* out_t;          // transposed direct-store output (few tokens): [z][N][out_ld] fp32, else unused
  long long out_ld;
  // Weight gradient with a partition off the 8-channel grid: the private rows start at S_lo (TMA reads channels in
  // 16-byte units), and the first `skip` = S - S_lo rows, which belong to the shared region, are not stored.  Only the
  // region's first row tile has such rows; it stores fp32 straight from registers to skip_out (plane z of skip_plane
  // elements, rows of N).
  int skip;
  float* skip_out;
  long long skip_plane;
  int splits;            // split-K factor of this region's tiles (set by finish_tiles from Params::splits when 0)
  int qper;              // > 0: the splits divide the rank loop, qper ranks each, instead of the k-steps
  int out_f32;
  int b_slowest;         // tile order: 1 = rank index slowest (a rank's weights / activations stay
                         // hot in L2 while its row tiles stream), 0 = row tile slowest
  float scale = 1.f;     // outputs are multiplied by it in the epilogue
  int a_mn;              // MIXED launches: as Params::a_mn, per region
};

struct Params {
  int nregions;
  Region r[kMaxRegions];
  int BN;                // tile width (UMMA N): multiple of 16 (of 64 when B is N-major)
  int nstages;
  int a_mn, b_mn;        // 1: operand is MN-major in global memory
  int cg;                // CTAs per tile: 1, or 2 (tcgen05 cta_group::2, clusters of two)
  int splits;            // split-K factor (only with a single unit and Q == 1)
  int push_slice;        // > 0: tiles of region 0 (the shared columns) are stored into the peer GPUs' receive slots, the
                         // owner of a tile being its first row / push_slice (a multiple of the tile's rows)
  int tile_end[kMaxRegions];   // tiles of regions 0..i (including splits)
  int tiles_total;
  unsigned int* status;
  uint32_t spin_cap;     // polls of one mbarrier wait before the role gives up (kSpinCap; CAAT_TC_SPINCAP for the timeout test)
  int debug;             // measurement aid (env CAAT_TC_DEBUG, masked by kAidMask; results are then wrong): 1 = no operand loads,
                         // 2 = no epilogue work at all, 4 = no A loads, 8 = no B loads; epilogue stops after the
                         // tensor-memory load (32) / after the staging stores (16);
                         // 128 = no TMA store; 512 = producer lanes take no second k-step; 1024 = the A boxes are
                         // announced to the stage barrier but never issued, so the consumers' waits run out
                         // (the timeout test: the kernel must flag it, drain and return)
};

// Output maps of the peers' receive slots (the exchange of the shared-channel slab over peer memory).
struct PeerMaps { CUtensorMap m[CAAT_MAX_PEERS]; };

// Operand maps (A and B of up to two layers or units) and output maps, one per region.
template <bool MIXED> struct MapsT { CUtensorMap ab[4], c[4]; };
template <> struct MapsT<true> { CUtensorMap ab[14], c[kMaxRegions]; };
using Maps = MapsT<false>;

// The swapped variant's tiles dealt to CTAs by their length (longest first, each to the least loaded CTA): CTA w works
// item[first[w]] .. item[first[w + 1] - 1].  dealt == 0: round-robin by tile number.
constexpr int kMaxDealWorkers = 160, kMaxDealItems = 1024;
struct Deal {
  int dealt;
  uint16_t first[kMaxDealWorkers + 1];
  uint16_t item[kMaxDealItems];
};
template <int SWAP> struct ExtraArg { using type = Deal; };
template <> struct ExtraArg<0> { using type = PeerMaps; };

// the tiles of one worker, in order
template <int SWAP>
struct TileIter {
  const typename ExtraArg<SWAP>::type& x;
  int pos, end, step;
  __device__ __forceinline__ TileIter(const typename ExtraArg<SWAP>::type& x_, int worker, int nworkers, int total) : x(x_) {
    pos = worker; end = total; step = nworkers;
    if constexpr (SWAP) {
      if (x.dealt) { pos = x.first[worker]; end = x.first[worker + 1]; step = 1; }
    }
  }
  __device__ __forceinline__ bool valid() const { return pos < end; }
  __device__ __forceinline__ int tile() const {
    if constexpr (SWAP) return x.dealt ? x.item[pos] : pos;
    return pos;
  }
  __device__ __forceinline__ void next() { pos += step; }
};

struct TileCoord {
  int region, b, mt, nt, split;
};

template <int NREGIONS>
__device__ __forceinline__ TileCoord decode_tile(const Params& p, int tile) {
  TileCoord c;
  c.region = 0;
#pragma unroll
  for (int g = 0; g + 1 < NREGIONS; ++g)
    if (tile >= p.tile_end[g]) c.region = g + 1;       // unused regions end where the last used one does: never reached
  int rem = tile - (c.region ? p.tile_end[c.region - 1] : 0);
  const Region& r = p.r[c.region];
  c.nt = rem % r.ntiles; rem /= r.ntiles;
  c.split = rem % r.splits; rem /= r.splits;
  if (r.b_slowest) {
    c.mt = rem % r.mtiles; rem /= r.mtiles;
    c.b = rem;
  } else {
    c.b = rem % r.batch; rem /= r.batch;
    c.mt = rem;
  }
  return c;
}

// Columns of B a tile really needs: the last tile of a ragged N (N-major B only) is narrowed to
// whole 64-column chunks per CTA, so no padded columns are loaded or multiplied.
__device__ __forceinline__ int tile_cols(const Params& p, const Region& r, int nt, int cg) {
  if (!p.b_mn) return p.BN;
  const int left = r.N - nt * p.BN;
  if (left >= p.BN) return p.BN;
  const int q = 64 * cg;
  return (left + q - 1) / q * q;
}

// rank and k-step range of a unit for a split
__device__ __forceinline__ void split_range(const Region& r, const Unit& u, int split, int& q_begin, int& q_end, int& k_begin,
                                            int& k_end) {
  q_begin = 0; q_end = u.Q; k_begin = 0; k_end = u.ksteps;
  if (r.splits == 1) return;
  if (r.qper > 0) {
    q_begin = split * r.qper;
    q_end = q_begin + r.qper < u.Q ? q_begin + r.qper : u.Q;
    return;
  }
  const int per = (u.ksteps + r.splits - 1) / r.splits;
  k_begin = split * per;
  k_end = k_begin + per < u.ksteps ? k_begin + per : u.ksteps;
  if (k_begin > k_end) k_begin = k_end;
}

// ---- CG == 2: a CTA pair works on one 256-row tile -------------------------------------------
// TMA load whose completion may be signalled on the peer CTA's mbarrier (the data lands in the issuing CTA only)
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// CG = 1: one CTA per 128-row tile.  CG = 2: a cluster of two CTAs per 256-row tile
// (tcgen05 cta_group::2): each CTA stages its own 128 rows of A and HALF of the B tile, the
// leader (cluster rank 0) issues the MMAs for both and the tensor cores read B from both CTAs'
// shared memory, so the operand bytes a CTA pulls from L2 per flop drop by a third.
// SWAP: the operands are swapped (weights on the 128-row side) and the sums are stored straight from registers: 1 = few tokens,
// fp32 planes, an accumulator per rank; 2 = some hundreds of tokens, one accumulator per tile, in the run's type or fp32 planes.
template <int CG, int SWAP, bool MIXED>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_kernel(const __grid_constant__ MapsT<MIXED> mp, const __grid_constant__ typename ExtraArg<SWAP>::type extra,
               const __grid_constant__ Params p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int BMT = BM * CG;                     // rows of a tile (of the pair's tile)
  const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
  const int worker = blockIdx.x / CG, nworkers = gridDim.x / CG;
  // carve: [stages x (A tile | this CTA's part of the B tile)], output staging, barriers
  const uint32_t bn_cta = (uint32_t)p.BN / CG;
  const uint32_t a_bytes = BM * BK * 2;
  const uint32_t b_bytes = bn_cta * BK * 2;
  const uint32_t stage_bytes = a_bytes + b_bytes;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t tiles_sa = smem_u32(base);
  uint8_t* cstage = base + (size_t)p.nstages * stage_bytes;   // output staging, kCStage bytes
  uint64_t* bars = reinterpret_cast<uint64_t*>(cstage + kCStage);
  // bars: full[nstages], empty[nstages], tfull[2], tempty[2]
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8u * p.nstages;
  const uint32_t tfull0 = empty0 + 8u * p.nstages;
  const uint32_t tempty0 = tfull0 + 16u;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * p.nstages + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.nstages; ++s) { mbar_init(full0 + 8u * s, 1); mbar_init(empty0 + 8u * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull0 + 8u * a, 1); mbar_init(tempty0 + 8u * a, 4 * CG); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();      // the peer's barriers are initialised before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();   // set-up done; operands and outputs may still be in use by the previous kernel until here

  if (warp == 0 || warp == kProducerB) {
    // ------------------------------------------------------------ TMA producers
    // Two producer warps run the same schedule: warp 0 issues the A boxes (and, in the leader CTA, posts
    // the stage's expected bytes), warp kProducerB the B boxes.
    const bool isA = warp == 0;
    // Lanes of the producer warp share the issue work: lane = (k-step of a group of kKI consecutive k-steps,
    // box of the stage).  A K-major operand is one box per stage, an M-/N-major one a box per 64 rows or
    // columns.  All active lanes run the same instructions on different stages / boxes, so the group is
    // issued in the time of one k-step: a single lane needs ~575 cycles per k-step (240 for the wait on a
    // barrier that is already free, 250 for the announcement and one box, 85 of loop), more than the 384-512
    // cycles the tensor cores take for it.
    constexpr int kKI = 2;
    const bool multi = MIXED || (isA ? p.a_mn : p.b_mn) != 0;       // MIXED: some regions' A, every region's B
    const int nbmax = multi ? (isA ? BM / 64 : (int)(p.BN / CG) / 64) : 1;      // boxes per stage, at most
    // measured: pays for multi-box operands (dgrad / wgrad -5...-8 %) and the weight stream of the decode
    // path (-5 %); a K-major operand of the large GEMMs gains nothing (its tiles wait for L2, not for the
    // issue) and a ring shorter than six stages loses more to pairwise refills than it gains
    const int nki = ((multi || SWAP) && p.nstages >= 6 && !(p.debug & kAidMask & 512)) ? kKI : 1;
    const int jk = lane / nbmax, box = lane - jk * nbmax;                         // this lane's k-step slot and box
    if (jk < nki) {
      int stage = 0; uint32_t phase = 0;
      long long issued = 0;
      bool ok = true;
      for (TileIter<SWAP> it(extra, worker, nworkers, p.tiles_total); it.valid() && ok; it.next()) {
        const TileCoord c = decode_tile<MIXED ? kMaxRegions : 4>(p, it.tile());
        const Region& r = p.r[c.region];
        const uint32_t cols_cta = (uint32_t)tile_cols(p, r, c.nt, CG) / CG;    // B columns this CTA stages
        const uint32_t b_tile_bytes = cols_cta * BK * 2;
        const int m0 = c.mt * BMT + (int)rank * BM, n0 = c.nt * p.BN + (int)(rank * cols_cta);
        const uint32_t tx = (uint32_t)CG * (((p.debug & kAidMask & 4) ? 0u : a_bytes) + ((p.debug & kAidMask & 8) ? 0u : b_tile_bytes));
        const bool skip = isA ? (p.debug & kAidMask & (4 | 1024)) != 0 : (p.debug & kAidMask & 8) != 0;
        const int a_mn = MIXED ? r.a_mn : p.a_mn;
        const int nb = isA ? (a_mn ? BM / 64 : 1) : (multi ? (int)cols_cta / 64 : 1);         // boxes of this tile's stages
        for (int ui = 0; ui < r.nunits && ok; ++ui) {
          const Unit& u = r.u[ui];
          const CUtensorMap* map = &mp.ab[isA ? u.mapA : u.mapB];
          int q0, q1, kb, ke;
          split_range(r, u, c.split, q0, q1, kb, ke);
          for (int q = q0; q < q1 && ok; ++q) {
            const int z = isA ? c.b * u.a_zb + q * u.a_zq : c.b * u.b_zb + q * u.b_zq;
            for (int k0 = kb; k0 < ke; k0 += nki) {
              const int ngrp = ke - k0 < nki ? ke - k0 : nki;      // k-steps of this group
              if (jk < ngrp) {
                const int kk = k0 + jk;
                int st = stage + jk; uint32_t ph = phase;
                if (st >= p.nstages) { st -= p.nstages; ph ^= 1u; }
                if (!mbar_wait(empty0 + 8u * st, ph ^ 1u, abort_flag, p.spin_cap)) { ok = false; break; }
                const uint32_t fb_local = full0 + 8u * st;
                // completion is signalled on the LEADER's barrier; the leader expects both CTAs' bytes
                const uint32_t fb = CG == 2 ? mapa_rank(fb_local, 0) : fb_local;
                const uint32_t sa = tiles_sa + (uint32_t)st * stage_bytes, sb = sa + a_bytes;
                if (isA && rank == 0 && box == 0) {
                  if (p.debug & kAidMask & 1) mbar_arrive(fb_local); else mbar_expect_tx(fb_local, tx);
                }
                if (!(p.debug & kAidMask & 1) && !skip && box < nb) {
                  auto load = [&](uint32_t dst, int x, int y) {
                    if (CG == 2) tma_load_3d_pair(dst, map, x, y, z, fb); else tma_load_3d(dst, map, x, y, z, fb);
                  };
                  if (isA) {
                    if (!a_mn) load(sa, u.ak0 + kk * BK, u.am0 + m0);
                    else load(sa + box * (64 * BK * 2), u.am0 + m0 + box * 64, u.ak0 + kk * BK);
                  } else {
                    if (!p.b_mn) load(sb, u.bk0 + kk * BK, u.bn0 + n0);
                    else load(sb + box * (64 * BK * 2), u.bn0 + n0 + box * 64, u.bk0 + kk * BK);
                  }
                }
              }
              issued += ngrp;
              stage += ngrp;
              if (stage >= p.nstages) { stage -= p.nstages; phase ^= 1u; }
            }
          }
        }
      }
      if (!ok && lane == 0) {
        // gave up: flag it, then wait (bounded) for the copies still in flight
        // (the pair's copies complete on the leader's barriers; the peer just gives them time)
        *abort_flag = 1;
        atomicExch(p.status, 1u);
        const int pending = issued < p.nstages ? (int)issued : p.nstages;
        int s = stage; uint32_t ph = phase;
        for (int k = 0; k < pending; ++k) {
          if (--s < 0) { s = p.nstages - 1; ph ^= 1u; }
          for (uint32_t it = 0; it < (p.spin_cap < (1u << 20) ? p.spin_cap : (1u << 20)); ++it)
            if (rank == 0 && mbar_try(full0 + 8u * s, ph)) break;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader CTA only when CG == 2)
    if (rank == 0) {                              // the whole warp walks the schedule, one elected lane issues
      const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(MIXED ? 0 : p.a_mn) << 15) | ((uint32_t)p.b_mn << 16) |
                              ((uint32_t)(BMT >> 4) << 24);
      int stage = 0; uint32_t phase = 0;
      int acc = 0; uint32_t acc_phase = 0;
      bool ok = true;
      // Descriptors differ from stage to stage and from MMA to MMA only in their 14-bit address field:
      // the constant part is built once and the loop adds 16-byte units to the low word.  The issuing
      // thread's instruction count per k-step is what bounds short contractions.
      const uint64_t a_const = p.a_mn && !MIXED ? make_desc(0, 64 * BK * 2, 1024) : make_desc(0, 16, 1024);
      const uint32_t a_mn_lo = (uint32_t)make_desc(0, 64 * BK * 2, 1024) - (uint32_t)make_desc(0, 16, 1024);
      const uint64_t b_const = p.b_mn ? make_desc(0, 64 * BK * 2, 1024) : make_desc(0, 16, 1024);
      const uint32_t a_hi = (uint32_t)(a_const >> 32), b_hi = (uint32_t)(b_const >> 32);
      uint32_t a_k16 = (p.a_mn && !MIXED ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      const uint32_t b_k16 = (p.b_mn ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      const uint32_t stage16 = stage_bytes >> 4;
      uint32_t a_lo0 = (uint32_t)a_const + (tiles_sa >> 4);
      const uint32_t b_lo0 = (uint32_t)b_const + ((tiles_sa + a_bytes) >> 4);
      uint32_t a_lo = a_lo0, b_lo = b_lo0;
      uint32_t full_bar = full0, empty_bar = empty0;
      for (TileIter<SWAP> it(extra, worker, nworkers, p.tiles_total); it.valid() && ok; it.next()) {
        const TileCoord c = decode_tile<MIXED ? kMaxRegions : 4>(p, it.tile());
        const Region& r = p.r[c.region];
        uint32_t d_tmem = 0, accumulate = 0;
        auto begin = [&]() {                        // the next free accumulator
          if (!mbar_wait_warp(tempty0 + 8u * acc, acc_phase ^ 1u, abort_flag, p.spin_cap)) return false;
          tc_fence_after();
          d_tmem = tmem_base + (uint32_t)(acc * kAccCols);
          accumulate = 0;
          return true;
        };
        auto finish = [&]() {                       // accumulator complete (in both CTAs)
          if (elect_one()) {
            if (CG == 2) umma_commit_pair(tfull0 + 8u * acc); else umma_commit(tfull0 + 8u * acc);
          }
          acc ^= 1;
          if (acc == 0) acc_phase ^= 1u;
        };
        if (SWAP != 1 && !begin()) { ok = false; break; }
        uint32_t idesc = idesc0 | ((uint32_t)(tile_cols(p, r, c.nt, CG) >> 3) << 17);
        if constexpr (MIXED) {
          idesc |= (uint32_t)r.a_mn << 15;
          a_k16 = (r.a_mn ? UMMA_K * 128 : UMMA_K * 2) >> 4;
          a_lo0 = (uint32_t)a_const + (tiles_sa >> 4) + (r.a_mn ? a_mn_lo : 0u);
          a_lo = a_lo0 + (uint32_t)stage * stage16;
        }
        for (int ui = 0; ui < r.nunits && ok; ++ui) {
          const Unit& u = r.u[ui];
          int q0, q1, kb, ke;
          split_range(r, u, c.split, q0, q1, kb, ke);
          for (int q = q0; q < q1 && ok; ++q) {
            if (SWAP == 1 && !begin()) { ok = false; break; }      // an accumulator per rank, see the epilogue
            for (int kk = kb; kk < ke; ++kk) {
              if (!mbar_wait_warp(full_bar, phase, abort_flag, p.spin_cap)) { ok = false; break; }
              tc_fence_after();
              if (elect_one()) {
#pragma unroll
                for (int k = 0; k < BK / UMMA_K; ++k) {
                  const uint64_t ad = ((uint64_t)a_hi << 32) | (a_lo + (uint32_t)k * a_k16);
                  const uint64_t bd = ((uint64_t)b_hi << 32) | (b_lo + (uint32_t)k * b_k16);
                  if (CG == 2) umma_bf16_pair(d_tmem, ad, bd, idesc, k == 0 ? accumulate : 1u);
                  else umma_bf16(d_tmem, ad, bd, idesc, k == 0 ? accumulate : 1u);
                }
                // frees the stage (in both CTAs) once these MMAs have read it
                if (CG == 2) umma_commit_pair(empty_bar); else umma_commit(empty_bar);
              }
              accumulate = 1;
              a_lo += stage16; b_lo += stage16; full_bar += 8u; empty_bar += 8u;
              if (++stage == p.nstages) {
                stage = 0; phase ^= 1u;
                a_lo = a_lo0; b_lo = b_lo0; full_bar = full0; empty_bar = empty0;
              }
            }
            if (SWAP == 1 && ok) finish();
          }
        }
        if (SWAP != 1 && ok) finish();
      }
      if (!ok && lane == 0) { *abort_flag = 1; atomicExch(p.status, 2u); }
    }
  } else if (warp <= 5) {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int quarter = warp & 3;                 // TMEM lanes [32*quarter, 32*quarter+32)
    int acc = 0; uint32_t acc_phase = 0;
    uint32_t slab = 0;
    bool ok = true;
    for (TileIter<SWAP> it(extra, worker, nworkers, p.tiles_total); it.valid() && ok; it.next()) {
      const TileCoord c = decode_tile<MIXED ? kMaxRegions : 4>(p, it.tile());
      const Region& r = p.r[c.region];
      // a tile whose contraction range is empty leaves the accumulator undefined: its value is 0
      int total_k = 0, nq = 0;
      for (int ui = 0; ui < r.nunits; ++ui) {
        int q0, q1, kb, ke;
        split_range(r, r.u[ui], c.split, q0, q1, kb, ke);
        total_k += (ke - kb) * (q1 - q0);
        nq += q1 - q0;
      }
      const int n0 = c.nt * p.BN;
      const int m0 = c.mt * BMT + (int)rank * BM;
      const int zc = c.split * r.batch + c.b;
      const int rr = quarter * 32 + lane;                 // row of the tile this thread holds
      // this warp's part of the accumulator is drained: tell the MMA issuer
      auto release = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (CG == 2) mbar_arrive_remote(mapa_rank(tempty0 + 8u * acc, 0)); else mbar_arrive(tempty0 + 8u * acc);
        }
      };
      if constexpr (SWAP == 1) {
        // swap-AB (decode): TMEM lane = output channel, column = token.  Every rank of the tile's group comes in an
        // accumulator of its own and the ranks are added here, as the row kernel adds the planes: one accumulator over all
        // ranks rounds every k-step's partial sum in the tensor core, which cost the row statistics a factor of three in
        // accuracy (7B shapes, 1 and 61 tokens: 2.5e-7 against 7.0e-7 from the exact ones).
        const long long chan = (long long)m0 + rr;
        // for a fixed token the 32 lanes of a warp hold 32 consecutive channels: plain 128-byte coalesced stores
        auto store = [&](int cc, const auto& value) {
          if (chan >= r.M) return;
          float* dst = r.out_t + ((long long)zc * r.N + cc) * r.out_ld + chan;
          const int ntok = r.N - cc;                      // tokens left from this column on (>= 1)
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            if (e < ntok) *dst = total_k == 0 ? 0.f : value(e);
            dst += r.out_ld;
          }
        };
        auto next = [&]() {
          if (!mbar_wait_warp(tfull0 + 8u * acc, acc_phase, abort_flag, p.spin_cap)) return false;
          tc_fence_after();
          return true;
        };
        auto done = [&]() {
          release();
          acc ^= 1;
          if (acc == 0) acc_phase ^= 1u;
        };
        const uint32_t tlane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        if (nq == 1) {          // short code of its own: it runs once or twice a launch (0.4 us of 11 at 57 tokens of 4 x 768)
          if (!next()) { ok = false; break; }
          for (int cc = 0; cc < r.N; cc += 32) {
            uint32_t v[32];
            tmem_ld32(tlane + (uint32_t)(acc * kAccCols + cc), v);
            tmem_ld_wait();
            store(cc, [&](int e) { return __uint_as_float(v[e]); });
          }
          done();
          continue;
        }
        float sum[kDecodeMaxTokens / 32][32] = {};
        for (int q = 0; q < nq; ++q) {
          if (!next()) { ok = false; break; }
#pragma unroll
          for (int j = 0; j < kDecodeMaxTokens / 32; ++j) {
            if (32 * j >= r.N) break;
            uint32_t v[32];
            tmem_ld32(tlane + (uint32_t)(acc * kAccCols + 32 * j), v);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e) sum[j][e] += __uint_as_float(v[e]);
          }
          done();
        }
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < kDecodeMaxTokens / 32; ++j)
          if (32 * j < r.N) store(32 * j, [&](int e) { return sum[j][e]; });
        continue;
      }
      if constexpr (SWAP == 2) {
        // TMEM lane = output channel, column = token: for a token the 32 lanes of a warp hold 32 consecutive channels, stored
        // as one run of 64 (128) bytes
        if (!mbar_wait_warp(tfull0 + 8u * acc, acc_phase, abort_flag, p.spin_cap)) { ok = false; break; }
        tc_fence_after();
        const long long chan = (long long)m0 + rr;
        const int ntok = r.N - n0 < p.BN ? r.N - n0 : p.BN;
        const long long at = ((long long)zc * r.N + n0) * r.out_ld + chan;
        float* f32 = r.out_t + at;
        __nv_bfloat16* b16 = reinterpret_cast<__nv_bfloat16*>(r.out_t) + at;
        const bool mine = chan < r.M;
        for (int cc = 0; cc < ntok; cc += 32) {
          uint32_t v[32];
          __syncwarp();
          tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * kAccCols + cc), v);
          tmem_ld_wait();
          if (cc + 32 >= ntok) release();
          if (total_k == 0) {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = 0u;
          }
          const int left = mine ? ntok - cc : 0;
          if (r.out_f32) {
#pragma unroll
            for (int e = 0; e < 32; ++e, f32 += r.out_ld)
              if (e < left) *f32 = __uint_as_float(v[e]);
          } else {
#pragma unroll
            for (int e = 0; e < 32; ++e, b16 += r.out_ld)
              if (e < left) *b16 = __float2bfloat16_rn(__uint_as_float(v[e]));
          }
        }
        acc ^= 1;
        if (acc == 0) acc_phase ^= 1u;
        continue;
      }
      // one verdict for the warp: the tensor-memory loads below are instructions of all its lanes
      if (!mbar_wait_warp(tfull0 + 8u * acc, acc_phase, abort_flag, p.spin_cap)) { ok = false; break; }
      tc_fence_after();
      // Every warp drains its 32 rows by itself in slabs of 128 bytes: TMEM -> registers -> swizzled staging buffer ->
      // TMA store (whole 128-byte lines; rows and columns outside the region's extents are clipped by the tensor map).
      // Two buffers per warp, no barrier across warps.  Short contractions are bound by this drain: the forward GEMM at
      // t = 8, K_r = 256, h = 2048, 8192 tokens took 79.3 us with slabs of 64 bytes x 128 rows and a barrier per slab
      // (54.5 without any epilogue), 71.5 like this; at p = 0.25 89.7 -> 78.8.
      //
      // where this tile's rows go: the region's own output, or - shared columns of a multi-GPU forward - the
      // receive slot of the GPU that owns these token rows, through its own map (row 0 = the owner's first token)
      const CUtensorMap* omap = &mp.c[c.region];
      int om0 = m0;
      if constexpr (!SWAP) {
        if (p.push_slice > 0 && c.region == 0) {
          const int owner = m0 / p.push_slice;
          omap = &extra.m[owner];
          om0 = m0 - owner * p.push_slice;
        }
      }
      const uint32_t sw = (uint32_t)(lane & 7);           // 128-byte swizzle: 16-byte chunk ^= row % 8
      if (r.skip > 0 && c.mt == 0) {
        const int row = m0 + rr;
        float* dst = r.skip_out + (long long)zc * r.skip_plane + (long long)row * r.N + n0;
        for (int cc = 0; cc < p.BN && n0 + cc < r.N; cc += 16) {
          uint32_t v[32];
          tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * kAccCols + cc), v);
          tmem_ld_wait();
          if (row >= r.skip && row < r.M) {
#pragma unroll
            for (int e = 0; e < 16; e += 4)
              if (n0 + cc + e < r.N)            // N is a multiple of 8
                *reinterpret_cast<float4*>(dst + cc + e) =
                    total_k == 0 ? make_float4(0.f, 0.f, 0.f, 0.f)
                                 : make_float4(__uint_as_float(v[e]) * r.scale, __uint_as_float(v[e + 1]) * r.scale,
                                               __uint_as_float(v[e + 2]) * r.scale, __uint_as_float(v[e + 3]) * r.scale);
          }
        }
        release();
      } else {
        const bool out_f32 = r.out_f32 != 0;
        const int sub = out_f32 ? 32 : 64;
        const int cols = (p.debug & kAidMask & 2) ? 0 : (r.N - n0 < p.BN ? r.N - n0 : p.BN);
        const bool scaled = r.scale != 1.f;
        if (cols <= 0) release();
        for (int cc = 0; cc < cols; cc += sub) {
          uint32_t v[32], w[32];
          const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * kAccCols + cc);
          tmem_ld32(taddr, v);
          if (!out_f32) tmem_ld32(taddr + 32, w);
          tmem_ld_wait();
          if (cc + sub >= cols) release();
          if (total_k == 0) {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = w[e] = 0u;
          }
          if (p.debug & kAidMask & 32) { ++slab; continue; }
          // the store that last used this buffer (two slabs ago) has finished reading it
          if (lane == 0) bulk_wait_read1();
          __syncwarp();
          const uint32_t buf = smem_u32(cstage + (size_t)((quarter * 2 + (slab & 1)) * kCBuf));
          const uint32_t rowaddr = buf + (uint32_t)lane * kSlabBytes;
          if (out_f32) {
            if (scaled) {
#pragma unroll
              for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * r.scale);
            }
#pragma unroll
            for (int q4 = 0; q4 < 8; ++q4)
              sts128(rowaddr + (((uint32_t)q4 ^ sw) << 4), v[4 * q4], v[4 * q4 + 1], v[4 * q4 + 2], v[4 * q4 + 3]);
          } else {
            if (scaled) {
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                v[e] = __float_as_uint(__uint_as_float(v[e]) * r.scale);
                w[e] = __float_as_uint(__uint_as_float(w[e]) * r.scale);
              }
            }
            auto pack = [](uint32_t lo, uint32_t hi) {
              __nv_bfloat162 bb = __floats2bfloat162_rn(__uint_as_float(lo), __uint_as_float(hi));
              return *reinterpret_cast<uint32_t*>(&bb);
            };
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4)
              sts128(rowaddr + (((uint32_t)q4 ^ sw) << 4), pack(v[8 * q4], v[8 * q4 + 1]), pack(v[8 * q4 + 2], v[8 * q4 + 3]),
                     pack(v[8 * q4 + 4], v[8 * q4 + 5]), pack(v[8 * q4 + 6], v[8 * q4 + 7]));
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4)
              sts128(rowaddr + (((uint32_t)(q4 + 4) ^ sw) << 4), pack(w[8 * q4], w[8 * q4 + 1]), pack(w[8 * q4 + 2], w[8 * q4 + 3]),
                     pack(w[8 * q4 + 4], w[8 * q4 + 5]), pack(w[8 * q4 + 6], w[8 * q4 + 7]));
          }
          if (p.debug & kAidMask & 16) { ++slab; continue; }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0 && !(p.debug & kAidMask & 128)) {
            tma_store_3d(omap, n0 + cc, om0 + quarter * 32, zc, buf);
            bulk_commit();
          }
          ++slab;
        }
      }
      acc ^= 1;
      if (acc == 0) acc_phase ^= 1u;
    }
    if (lane == 0) bulk_wait_all();   // all output stores of this warp are complete
    if (!ok && lane == 0) { *abort_flag = 1; atomicExch(p.status, 3u); }
  }

  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();   // the leader's MMAs read the peer's shared memory: leave together
  if (warp == 1) {
    tc_fence_after();
    if (CG == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// out[i] = sum_s part[s][i], s ascending (deterministic split-K reduction)
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float4* __restrict__ part, float4* __restrict__ out,
                                                            long long n4, int splits) {
  pdl_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (long long)gridDim.x * blockDim.x) {
    float4 s = part[i];
    for (int k = 1; k < splits; ++k) {
      const float4 v = part[(long long)k * n4 + i];
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    out[i] = s;
  }
}

// zs[i] = round(sum_g planes[g][i]), g ascending: the rank groups of a split shared region, 8 elements per thread.  With
// slice > 0 row i of the sum goes to slot `rank` of GPU i / slice instead (the exchange over peer memory).
struct SlotTarget { uint4* recv[CAAT_MAX_PEERS]; int slice, rank; };

__global__ void __launch_bounds__(256) sum_groups_kernel(const float4* __restrict__ planes, uint4* __restrict__ zs, int T, int row8,
                                                         int groups, const __grid_constant__ SlotTarget slots) {
  pdl_wait();
  const long long n8 = (long long)T * row8;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += (long long)gridDim.x * blockDim.x) {
    float4 a = planes[2 * i], b = planes[2 * i + 1];
    for (int g = 1; g < groups; ++g) {
      const float4 x = planes[2 * (g * n8 + i)], y = planes[2 * (g * n8 + i) + 1];
      a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
      b.x += y.x; b.y += y.y; b.z += y.z; b.w += y.w;
    }
    __nv_bfloat162 o[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w), __floats2bfloat162_rn(b.x, b.y),
                           __floats2bfloat162_rn(b.z, b.w)};
    uint4* dst = zs + i;
    if (slots.slice > 0) {
      const int row = (int)(i / row8), q = row / slots.slice;
      dst = slots.recv[q] + ((long long)slots.rank * slots.slice + (row - q * slots.slice)) * row8 + (i - (long long)row * row8);
    }
    *dst = *reinterpret_cast<uint4*>(o);
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(f);
  });
  return fn;
}

// Tensor [d2][d1][d0] (d0 contiguous) with row pitch ld1 and plane pitch ld2 (elements);
// box = (b0, b1, 1); out-of-range elements read as zero and are not written.
bool make_map(CUtensorMap* m, const void* base, long long d0, long long d1, long long d2, long long ld1, long long ld2,
              int b0, int b1, bool f32 = false, CUtensorMapSwizzle swz = CU_TENSOR_MAP_SWIZZLE_128B) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  if (d0 < 1 || d1 < 1 || d2 < 1) return false;
  const cuuint64_t es_bytes = f32 ? 4 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)d0, (cuuint64_t)d1, (cuuint64_t)d2};
  cuuint64_t strides[2] = {(cuuint64_t)ld1 * es_bytes, (cuuint64_t)ld2 * es_bytes};
  cuuint32_t box[3] = {(cuuint32_t)b0, (cuuint32_t)b1, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                  const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Output map: slabs of 128 bytes x 32 rows, 128-byte swizzle (matches the epilogue's staging layout).
bool make_cmap(CUtensorMap* m, const void* base, long long d0, long long d1, long long d2, long long ld1,
               long long ld2, bool f32) {
  return make_map(m, base, d0, d1, d2, ld1, ld2, kSlabBytes / (f32 ? 4 : 2), 32, f32);
}

// ---- tile configuration ------------------------------------------------------------------
// A small cost model picks the tile width BN, the CTA-pair mode cg and (weight gradient) the
// split-K factor.  Unit of time: one 128 x 256 x 64 MMA step at full tensor rate (~0.2 us).
//  * a k-step of a 128 x BN (x cg) tile costs BN/256, stretched when the operand bytes a CTA
//    pulls from L2 per flop, proportional to (128 + BN/cg) / BN, exceed what L2 delivers
//    (measured: 128 x 256 tiles with cg = 1 run at ~0.73 of the tensor rate);
//  * the epilogue of a tile (~10 units at BN = 256) overlaps the next tile's main loop, so a
//    tile costs max(main loop, epilogue) plus a fixed hand-off (larger across a CTA pair);
//  * tiles are dealt round-robin to 148 / cg workers: few tiles cost whole waves;
//  * split-K partials are written and read back once (fp32).
// Regions are dealt one after the other (the first one's tiles are the longest); a worker's load is the sum of its tiles.
struct RegionShape { int M, N, batch, ksteps; };
struct TileCfg { int bn, cg, splits; double cost; };

// The busiest worker's load when the regions' tiles, n[i] of length len[i], are dealt round-robin one region after the other.
double makespan(const long long* n, const double* len, int nr, long long W) {
  double worst = 0;
  long long start = 0;
  for (int q = 0; q <= nr; ++q) {            // loads change only where a region's last round ends
    const long long w = start % W;
    double load = 0;
    long long e = 0, before = 0;
    for (int i = 0; i < nr; ++i) {
      e += n[i];
      const long long upto = e / W + (w < e % W);
      load += (double)(upto - before) * len[i];
      before = upto;
    }
    worst = fmax(worst, load);
    if (q < nr) start += n[q];
  }
  return worst;
}

double estimate_cost(const RegionShape* r, int nr, int bn, int cg, int splits, double out_bytes, bool b_n_major) {
  const double workers = 148.0 / cg;
  const double step = (bn / 256.0) * fmax(1.0, 0.92 * (128.0 + (double)bn / cg) / bn);
  const double epi = 10.0 * bn / 256.0;
  const double handoff = cg == 2 ? 3.5 : 2.0;
  double total = 0, len[kMaxRegions] = {};
  long long n[kMaxRegions] = {}, tiles = 0;
  for (int i = 0; i < nr; ++i) {
    if (r[i].M <= 0 || r[i].N <= 0) continue;
    const long long rows = (long long)((r[i].M + 128 * cg - 1) / (128 * cg)) * r[i].batch * splits;
    const double ks = (double)((r[i].ksteps + splits - 1) / splits);
    const int full = r[i].N / bn, rest = r[i].N % bn;
    double region = rows * full * (fmax(ks * step, epi) + handoff);
    n[i] = rows * full;
    if (rest) {   // the last, ragged tile: an N-major B operand is narrowed to whole 64-column chunks
      const double w = b_n_major ? (double)((rest + 64 * cg - 1) / (64 * cg) * (64 * cg)) / bn : 1.0;
      region += rows * (fmax(ks * step * w, epi * w) + handoff);
      n[i] += rows;
    }
    total += region;
    tiles += n[i];
    if (n[i]) len[i] = region / n[i];
  }
  if (tiles == 0) return 0;
  double t = fmax(total / workers, makespan(n, len, nr, (long long)workers));
  if (splits > 1) t += 2.0 * splits * out_bytes / 6.4e12 / 0.2e-6;
  return t;
}

TileCfg pick_tile(const RegionShape* r, int nr, bool b_n_major, int max_splits, double out_bytes) {
#ifdef CAAT_MEASUREMENT_AIDS
  static const int max_cg = [] { const char* e = getenv("CAAT_TC_CG"); return e && atoi(e) == 1 ? 1 : 2; }();
  // CAAT_TC_BN / CAAT_TC_CGF pin the tile width / the pair mode instead of the model's choice
  static const int force_bn = [] { const char* e = getenv("CAAT_TC_BN"); return e ? atoi(e) : 0; }();
  static const int force_cg = [] { const char* e = getenv("CAAT_TC_CGF"); return e ? atoi(e) : 0; }();
#else
  constexpr int max_cg = 2, force_bn = 0, force_cg = 0;
#endif
  TileCfg best{256, 1, 1, -1.0};
  int min_ksteps = 1 << 30;
  for (int i = 0; i < nr; ++i)
    if (r[i].M > 0 && r[i].N > 0 && r[i].ksteps < min_ksteps) min_ksteps = r[i].ksteps;
  for (int cg = 1; cg <= max_cg; ++cg) {
    bool ok = true;
    int nmin = 1 << 30;
    for (int i = 0; i < nr; ++i) {
      if (r[i].M <= 0 || r[i].N <= 0) continue;
      if (cg == 2 && r[i].M < 256) ok = false;          // a pair needs two row blocks
      if (r[i].N < nmin) nmin = r[i].N;
    }
    if (!ok) continue;
    if (force_cg && cg != force_cg && !(force_cg == 2 && cg == 1 && max_cg == 2)) continue;
    const int step = b_n_major ? 64 * cg : 64;    // whole output slabs; N-major B: whole 64-column chunks per CTA
    for (int bn = 256; bn >= 64 * cg; bn -= step) {
      if (force_bn && bn != force_bn && force_bn % step == 0 && force_bn >= 64 * cg) continue;
      for (int splits = 1; splits <= max_splits; ++splits) {
        if (splits > 1 && min_ksteps / splits < 8) break;
        const double c = estimate_cost(r, nr, bn, cg, splits, out_bytes, b_n_major);
        if (best.cost < 0 || c < best.cost * 0.995) best = TileCfg{bn, cg, splits, c};
      }
    }
  }
  return best;
}

template <bool MIXED = false>
cudaError_t launch(const MapsT<MIXED>& maps, Params& p, int kind, cudaStream_t st, const PeerMaps* peer_maps = nullptr,
                   const Deal* deal = nullptr) {
  const LaunchLimits lim = effective_limits();
  const int stage_bytes = BM * BK * 2 + (p.BN / p.cg) * BK * 2;
  const int budget = lim.gemm_smem > 0 && lim.gemm_smem < 227 * 1024 ? lim.gemm_smem : 227 * 1024;
  int nst = (budget - 2048 - kCStage) / stage_bytes;
  if (nst > kMaxStages) nst = kMaxStages;
  if (nst < 2) return cudaErrorInvalidConfiguration;
  p.nstages = nst;
  const size_t smem = (size_t)nst * stage_bytes + kCStage + 1024 /*alignment slack*/ + (2 * nst + 4) * 8 + 16;
  static bool attr_set[64] = {};      // the attribute belongs to the device's copy of the kernel: once per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (std::lock_guard<std::mutex> lock(host_cache_mutex()); !attr_set[dev]) {
    auto allow = [](auto k) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024); };
    cudaError_t e = allow(tc_gemm_kernel<1, 0, MIXED>);
    if (e == cudaSuccess) e = allow(tc_gemm_kernel<2, 0, MIXED>);
    if constexpr (!MIXED) {
      if (e == cudaSuccess) e = allow(tc_gemm_kernel<1, 1, false>);
      if (e == cudaSuccess) e = allow(tc_gemm_kernel<2, 2, false>);
    }
    if (e != cudaSuccess) return e;
    attr_set[dev] = true;
  }
  p.status = device_status_word();
  if (!p.status) return cudaErrorUnknown;
  static const int dbg = [] { const char* e = getenv("CAAT_TC_DEBUG"); return e ? atoi(e) : 0; }();
  p.debug = dbg & kAidMask;
  static const uint32_t cap_env = [] { const char* e = getenv("CAAT_TC_SPINCAP"); return e ? (uint32_t)atoi(e) : 0u; }();
  p.spin_cap = cap_env >= 1024 ? cap_env : kSpinCap;
  static const bool verbose = getenv("CAAT_TC_VERBOSE") != nullptr;
  if (verbose)
    fprintf(stderr, "[caat tc] kind=%d BN=%d cg=%d splits=%d stages=%d tiles=%d (r0 M=%d N=%d b=%d)\n", kind, p.BN, p.cg,
            p.splits, nst, p.tiles_total, p.r[0].M, p.r[0].N, p.r[0].batch);
  int workers_max = sm_count() / p.cg;
  if (lim.gemm_workers > 0 && lim.gemm_workers / p.cg < workers_max) workers_max = lim.gemm_workers / p.cg;
  if (deal && workers_max > kMaxDealWorkers) workers_max = kMaxDealWorkers;
  const int workers = p.tiles_total < workers_max ? p.tiles_total : workers_max;
  if (workers < 1) return cudaSuccess;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(workers * p.cg));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.cg;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  LaunchScope scope(kind, st);
  if constexpr (!MIXED) {
    if (deal) {
      // a deal to more CTAs than this launch has would leave tiles out: those go round by number instead
      static const Deal by_number{};
      const Deal& d = deal->dealt && deal->first[workers] != p.tiles_total ? by_number : *deal;
      if (p.cg == 2) return cudaLaunchKernelEx(&cfg, tc_gemm_kernel<2, 2, false>, maps, d, (const Params&)p);
      return cudaLaunchKernelEx(&cfg, tc_gemm_kernel<1, 1, false>, maps, d, (const Params&)p);
    }
  }
  static const PeerMaps no_peers{};
  const PeerMaps& pm = peer_maps ? *peer_maps : no_peers;
  if (p.cg == 2) return cudaLaunchKernelEx(&cfg, tc_gemm_kernel<2, 0, MIXED>, maps, pm, (const Params&)p);
  return cudaLaunchKernelEx(&cfg, tc_gemm_kernel<1, 0, MIXED>, maps, pm, (const Params&)p);
}

void finish_tiles(Params& p) {
  for (int g = 0; g < p.nregions; ++g) {
    Region& r = p.r[g];
    r.mtiles = (r.M + BM * p.cg - 1) / (BM * p.cg);
    r.ntiles = (r.N + p.BN - 1) / p.BN;
    if (r.splits < 1) r.splits = p.splits < 1 ? 1 : p.splits;
  }
  p.tiles_total = 0;
  for (int g = 0; g < kMaxRegions; ++g) {
    if (g < p.nregions) p.tiles_total += p.r[g].mtiles * p.r[g].ntiles * p.r[g].batch * p.r[g].splits;
    p.tile_end[g] = p.tiles_total;
  }
}

}  // namespace

bool tc_gemm_usable(const caat_ctx* ctx, int K_r) {
  return ctx->dtype == CAAT_BF16 && !ctx->force_simt && K_r % 8 == 0 && ctx->h % 8 == 0;
}

// ---- forward: zs[T,S] = sum_m Y[m] W[m][:S]^T ; zp[m][T,h-S_lo] = Y[m] W[m][S_lo:]^T
// Any partition S: TMA wants 16-byte coordinates along a row's channels, so the private products start at S_lo; their
// S - S_lo extra columns land in the scratch columns that no row kernel reads.  (Partitions off the 8-channel grid ran on
// the CUDA-core GEMM before: a training step of a block at h = 2048, 2999 tokens, p = 0.7 took 17.5 ms, now 0.52 ms.)
// A shared tile's contraction is t times a private one's, and with few tokens there are only a handful of them: the
// GEMM then waits for its longest tiles (T = 300 at the 7B MLP shapes: 16 tiles of 176 k-steps where the even share of a
// worker is 76).  Given `planes` ([max_groups][T][S_hi] fp32 scratch), the rank loop may be split into groups of ranks:
// every group's partial sum is a tile of its own, and the row kernel adds the planes where it would read the sum (alone,
// GEMM of that layer alone, 300 tokens: 67 -> 41 us; 80 tokens: 54 -> 21).  The cost model
// decides.
struct ForwardPlan { TileCfg tile; int groups, qper; };

static double plane_cost(const RowparShapes& s, int groups) {      // the planes' round trip through L2
  return groups > 1 ? (8.0 * groups * s.T * s.S_hi / 10e12 + 1e-6) / 0.2e-6 : 0;
}

static ForwardPlan forward_plan(const RowparShapes& s, int max_groups) {
  const int n_sh = s.S, n_pr = s.S < s.h ? s.h - s.S_lo : 0, ksteps = (s.K_r + BK - 1) / BK;
  ForwardPlan f{};
  for (int per = s.t; per >= 1; per = per > 1 ? (per + 1) / 2 : 0) {
    const int g = (s.t + per - 1) / per;
    if (g > 1 && (n_sh == 0 || g > max_groups)) break;
    const RegionShape rs[2] = {{s.T, n_sh, g, ksteps * per}, {s.T, n_pr, s.t, ksteps}};
    TileCfg c = pick_tile(rs, 2, false, 1, 0.0);
    c.cost += plane_cost(s, g);
    if (g == 1 || c.cost < f.tile.cost) { f = ForwardPlan{c, g, per}; }
  }
  return f;
}

// operand maps of one layer's forward product: mp.ab[2 l] = Y, mp.ab[2 l + 1] = W
static bool forward_maps(Maps& mp, int l, const RowparShapes& s, const void* Y, const void* W, const Params& p) {
  return make_map(&mp.ab[2 * l], Y, s.K_r, s.T, s.t, s.K_r, (long long)s.T * s.K_r, BK, BM) &&
         make_map(&mp.ab[2 * l + 1], W, s.K_r, s.h, s.t, s.K_r, (long long)s.h * s.K_r, BK, p.BN / p.cg);
}
// the next region of the launch: the shared columns, all ranks in the contraction (or groups of qper ranks)
static bool forward_shared(Maps& mp, Params& p, int l, const RowparShapes& s, void* zs, void* planes, int groups, int qper) {
  const int g = p.nregions++;
  Region& r = p.r[g];
  r.nunits = 1;
  r.u[0] = Unit{2 * l, 2 * l + 1, 0, 0, 0, 0, /*a_zb*/ 0, /*a_zq*/ 1, /*b_zb*/ 0, /*b_zq*/ 1, s.t, (s.K_r + BK - 1) / BK};
  r.M = s.T; r.N = s.S; r.batch = 1; r.b_slowest = 0;
  if (groups > 1) { r.splits = groups; r.qper = qper; r.out_f32 = 1; }
  return make_cmap(&mp.c[g], groups > 1 ? planes : zs, s.S, s.T, groups, s.S_hi, (long long)s.T * s.S_hi, groups > 1);
}
// the next region: the private columns, per rank
static bool forward_private(Maps& mp, Params& p, int l, const RowparShapes& s, void* zp) {
  const int g = p.nregions++;
  Region& r = p.r[g];
  r.nunits = 1;
  r.u[0] = Unit{2 * l, 2 * l + 1, 0, 0, 0, s.S_lo, 1, 0, 1, 0, 1, (s.K_r + BK - 1) / BK};
  r.M = s.T; r.N = s.h - s.S_lo; r.batch = s.t; r.b_slowest = 1;
  return make_cmap(&mp.c[g], zp, s.h - s.S_lo, s.T, s.t, s.P, (long long)s.T * s.P, false);
}

// ---- few tokens: the operands are swapped (weights on the 128-row side, tokens on the narrow side), so that a tile streams
// 128 weight rows however few tokens there are, and the sums leave as fp32 planes for the row kernel:
//   zs[g][i][l]  l < S     sum over the g-th group of qper ranks (qper = 0: one plane per rank and k-split)
//   zp[k][m][i][l - S_lo]  l >= S, the k-th part of the contraction
// A tile is (plane, 128 channels).  Both layers of a block go in one launch.  Tiles differ in length (qper ranks of k-steps
// against one), so they are dealt longest first to the least loaded CTA.  Fewer, longer tiles mean fewer planes for the
// row kernel - with many tokens every rank's CTA reads every shared plane - but a coarser deal; few_token_plan weighs them.
namespace {
struct FewPlan { FewSplit l[2]; Deal deal; };

constexpr double kItemOverhead = 1.5;     // of a tile, in k-steps: refill of the pipeline and the epilogue
constexpr double kStepUs = 0.38;          // a k-step of 16 KB of weights on one of 148 SMs at 6.4 TB/s
// Where the tiles leave SMs idle a k-step is bound by the CTA's own round trips (4 x 768: every k-step less on 48 tiles takes
// 0.25 us off), and a split of the contraction costs more than its planes' bytes (0.3 us beside them).  A block of 4 x 768, split
// in four by the bytes alone / as now: 64 tokens 12.7 / 10.0 us, 57 tokens of nothing shared 11.1 / 9.5, 16 tokens 9.7 / 8.7.
constexpr double kLoneStepUs = 0.27, kSplitUs = 0.3;

// The tiles of a plan by their length: at most full, last and empty ones of the shared and of the private part of either layer.
// first, step, run: the tiles first + i * step + j, j < run, in the kernel's numbering (decode_tile with one column tile:
// region, then split fastest, then mt, then b).
struct FewRun { float len; int first, step, run, n; };
struct FewTiles { int nruns, tiles; FewRun r[12]; };

FewTiles few_tiles(int t, int h, int S, const int* K_r, int n, const FewSplit* sp, int rows = BM, int ncols = 1, double overhead = kItemOverhead) {
  FewTiles f{};
  const int S_lo = round_down(S, kLayoutVec);
  for (int g = 0; g < n; ++g) {
    const int ks = (K_r[g] + BK - 1) / BK;
    for (int part = 0; part < 2; ++part) {
      const int M = part == 0 ? S : (S < h ? h - S_lo : 0);
      if (M <= 0) continue;
      const bool grouped = part == 0 && sp[g].qper > 0;
      const int splits = grouped ? (t + sp[g].qper - 1) / sp[g].qper : sp[g].ksplits;
      const int outer = (M + rows - 1) / rows * (grouped ? 1 : t);
      // a split is `per` pieces of `unit` k-steps long; the last one may be shorter, and those of a k-split past it are empty
      const int pieces = grouped ? t : ks, unit = grouped ? ks : 1, per = grouped ? sp[g].qper : (ks + splits - 1) / splits;
      const int full = pieces / per, rest = pieces - full * per, used = full + (rest > 0);
      auto add = [&](int split, int count, int length) {
        if (count > 0) f.r[f.nruns++] = FewRun{(float)(length * unit + overhead), f.tiles + split * ncols, splits * ncols, count * ncols, outer};
      };
      add(0, full, per);
      add(full, used - full, rest);
      add(used, splits - used, 0);
      f.tiles += outer * splits * ncols;
    }
  }
  std::sort(f.r, f.r + f.nruns, [](const FewRun& x, const FewRun& y) { return x.len > y.len || (x.len == y.len && x.first < y.first); });
  return f;
}

// Longest first, each to the least loaded worker: the busiest worker's load.  Workers of equal load are one group and take
// their next tiles together, so a deal costs a few dozen steps however many tiles there are.
double few_makespan(const FewTiles& f, int workers) {
  struct Group { float load; int count; } g[kMaxDealWorkers];
  int ng = 1;
  g[0] = Group{0.f, workers};
  for (int i = 0; i < f.nruns; ++i)
    for (int left = f.r[i].n * f.r[i].run; left > 0;) {
      const int take = left < g[0].count ? left : g[0].count;
      const float load = g[0].load + f.r[i].len;
      left -= take;
      int at = 0;
      if ((g[0].count -= take) == 0) {           // the group is gone: the others move down past its new place
        for (; at + 1 < ng && g[at + 1].load < load; ++at) g[at] = g[at + 1];
        if (at + 1 < ng && g[at + 1].load == load) {
          g[at] = g[at + 1];
          g[at].count += take;
          for (int k = at + 1; k + 1 < ng; ++k) g[k] = g[k + 1];
          --ng;
        } else {
          g[at] = Group{load, take};
        }
      } else {
        for (at = 1; at < ng && g[at].load < load;) ++at;
        if (at < ng && g[at].load == load) {
          g[at].count += take;
        } else {
          for (int k = ng++; k > at; --k) g[k] = g[k - 1];
          g[at] = Group{load, take};
        }
      }
    }
  return g[ng - 1].load;
}

// the same deal, tile by tile
void few_deal(const FewTiles& f, int workers, Deal* deal) {
  struct Worker { float load; int id; bool operator<(const Worker& o) const { return load < o.load || (load == o.load && id < o.id); } };
  Worker w[kMaxDealWorkers], merged[kMaxDealWorkers];       // ascending
  uint16_t tile[kMaxDealItems];          // longest first
  uint8_t owner[kMaxDealItems];
  int count[kMaxDealWorkers] = {};
  for (int i = 0; i < workers; ++i) w[i] = Worker{0.f, i};
  int n = 0;
  for (int i = 0; i < f.nruns; ++i) {
    const int begin = n;
    for (int o = 0; o < f.r[i].n; ++o)
      for (int k = 0; k < f.r[i].run; ++k) tile[n++] = (uint16_t)(f.r[i].first + o * f.r[i].step + k);
    for (int j = begin; j < n;) {
      int take = 1;
      while (take < workers && take < n - j && w[take].load == w[0].load) ++take;
      for (int k = 0; k < take; ++k) {
        owner[j++] = (uint8_t)w[k].id;
        ++count[w[k].id];
        w[k].load += f.r[i].len;
      }
      std::merge(w, w + take, w + take, w + workers, merged);
      std::copy(merged, merged + workers, w);
    }
  }
  int at[kMaxDealWorkers], pos = 0;
  for (int i = 0; i < workers; ++i) { deal->first[i] = (uint16_t)pos; at[i] = pos; pos += count[i]; }
  deal->first[workers] = (uint16_t)pos;
  for (int j = 0; j < n; ++j) deal->item[at[owner[j]]++] = tile[j];
  deal->dealt = 1;
}

// Chooses the splits of one or two layers.  The row kernel's share: a plane of the shared part is written once and read
// by every rank's CTA (once per token when the ranks share it through a cluster), a private plane is read once.
void few_token_plan(int t, int T, int h, int S, const int* K_r, int n, int sms, FewPlan* best) {
  const int workers = sms < kMaxDealWorkers ? sms : kMaxDealWorkers;
  double best_cost = -1;
  const bool clustered = (long long)T * t <= (long long)sms * 3 / 4;
  FewSplit cand[2][16];
  int nc[2] = {0, 0};
  for (int g = 0; g < n; ++g) {
    const int ks = (K_r[g] + BK - 1) / BK;
    for (int q = t; q >= 1; q = q > 1 ? (q + 1) / 2 : 0)
      if (nc[g] < 12) cand[g][nc[g]++] = FewSplit{q, 1};
    for (int k = 2; k <= kDecodeMaxSplits && 2 * k <= ks; ++k) cand[g][nc[g]++] = FewSplit{0, k};
  }
  if (n == 1) { cand[1][0] = FewSplit{t, 1}; nc[1] = 1; }
  best->l[0] = best->l[1] = FewSplit{1, 1};
  // a deal is computed only where its lower bound (even share, longest tile, planes) can still win
  struct Cand { double bound, rest; FewSplit l[2]; };
  Cand all[256];
  int na = 0;
  for (int i = 0; i < nc[0]; ++i)
    for (int j = 0; j < nc[1]; ++j) {
      Cand c{0, 0, {cand[0][i], cand[1][j]}};
      double total = 0, longest = 0;
      for (int g = 0; g < n; ++g) {
        const int ks = (K_r[g] + BK - 1) / BK, ns = few_shared_planes(c.l[g], t);
        const int ms = (S + BM - 1) / BM, mp = S < h ? (h - round_down(S, kLayoutVec) + BM - 1) / BM : 0;
        total += (double)(ms + mp) * t * ks + kItemOverhead * ((double)ms * ns + (double)mp * t * c.l[g].ksplits);
        const double len = c.l[g].qper > 0 ? (S > 0 ? c.l[g].qper : 1) * ks : (ks + c.l[g].ksplits - 1) / c.l[g].ksplits;
        if (len > longest) longest = len;
        const double bytes = 4.0 * T * ((double)ns * S * (clustered ? 2 : 1 + t) + 2.0 * c.l[g].ksplits * t * (h - S));
        c.rest += bytes / 8e12 * 1e6 + kSplitUs * (c.l[g].ksplits - 1);
      }
      c.bound = fmax(total / workers * kStepUs, (longest + kItemOverhead) * kLoneStepUs) + c.rest;
      all[na++] = c;
    }
  std::sort(all, all + na, [](const Cand& a, const Cand& b) { return a.bound < b.bound; });
  for (int i = 0; i < na && (best_cost < 0 || all[i].bound < best_cost); ++i) {
    const FewTiles f = few_tiles(t, h, S, K_r, n, all[i].l);
    if (f.tiles > kMaxDealItems) continue;
    const double share = kStepUs * (f.tiles < workers ? f.tiles : workers) / workers;
    const double cost = few_makespan(f, workers) * fmax(share, kLoneStepUs) + all[i].rest;
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best->l[0] = all[i].l[0]; best->l[1] = all[i].l[1]; }
  }
  const FewTiles f = few_tiles(t, h, S, K_r, n, best->l);
  best->deal.dealt = 0;
  if (f.tiles > workers && f.tiles <= kMaxDealItems) few_deal(f, workers, &best->deal);     // else a tile each, or by number
}

// Plans depend on the shapes (and the device's SMs) alone.  Making one takes 4 us (7B shapes, on the host of the measurements); the
// 64 used last are kept.  They are made outside the lock, so that one thread's new shape holds up no other thread's call.
template <typename Plan, int N>
struct PlanCache {
  struct Key { int v[N]; bool operator==(const Key& o) const { return !memcmp(v, o.v, sizeof(v)); } };
  static constexpr int kPlans = 64;
  Key keys[kPlans];
  unsigned long long used[kPlans] = {}, clock = 0;      // used == 0: an empty slot
  Plan plans[kPlans];
  std::mutex m;

  int find(const Key& key) const {
    for (int i = 0; i < kPlans; ++i)
      if (used[i] && keys[i] == key) return i;
    return -1;
  }
  template <typename Make>
  void get(const Key& key, Plan* out, Make make) {
    {
      std::lock_guard<std::mutex> lock(m);
      const int i = find(key);
      if (i >= 0) {
        used[i] = ++clock;
        *out = plans[i];
        return;
      }
    }
    make(out);
    std::lock_guard<std::mutex> lock(m);
    int i = find(key);                  // another thread may have made it meanwhile
    if (i < 0) {
      i = (int)(std::min_element(used, used + kPlans) - used);
      keys[i] = key;
      plans[i] = *out;
    }
    used[i] = ++clock;
  }
};

void few_plan_cached(int t, int T, int h, int S, const int* K_r, int n, FewPlan* out) {
  static PlanCache<FewPlan, 7> cache;
  const int sms = sm_count();
  cache.get({{t, T, h, S, K_r[0], n > 1 ? K_r[1] : 0, sms}}, out,
            [&](FewPlan* p) { few_token_plan(t, T, h, S, K_r, n, sms, p); });
}
}  // namespace

// ---- a block's products with some hundreds of tokens: weights on the row side of a CTA pair's 256-row tiles, up to 256 tokens on
// the column side, both layers in one launch, tiles dealt by length.  With tokens on the row side a tile is at least 128
// tokens high and every one of them streams the weights again; what bounds these calls is the operand bytes from L2 (300
// tokens of 8 x 4096: 550 MB, here 390 MB).  Outputs as in the normal forward: zs and zp, or fp32 planes of the shared part over
// groups of ranks.  The groups are the normal forward's and every output's products are added in the same order, so the sums are
// the same bits either way.
// The rule: cheaper than the two layers' tiles by 5 % of the models' figures, and not so short that the launch alone decides.
// Of 280 sizes (seven models from 2 x 1024 to 8 x 5120, p = 0, 0.25, 0.5, 0.75, 1, eight token counts from 65 to 512; replayed from
// graphs) 113 are taken, at 0.72 to 1.01 of the time with tokens on the rows.  The models underrate the gain elsewhere, and
// sizes are refused that would be faster here: 8 x 4096, 65 / 100 / 128 tokens 48.8 / 41.3, 54.0 / 46.8, 57.6 / 50.0; 2 x 3072,
// 400 / 512 tokens 53.7 / 43.0, 57.2 / 47.3; 8 x 5120, 256 / 512 tokens 95.8 / 89.1, 171.7 / 145.7; 4 x 1536, 512 tokens 29.1 / 26.9.
// Block forward on either side of the line, tokens on the rows / here, us: taken - 8 x 4096, 200 tokens 72.5 / 59.6, 300 tokens
// 88.1 / 74.7, 400 tokens 93.6 / 88.0, nothing shared 78.3 / 69.9; 8 x 5120, 200 tokens 99.3 / 80.2, 300 tokens 118 / 106; 2 x 3072,
// 300 tokens 50.6 / 37.6; 8 x 2048, 65 tokens 17.9 / 17.9, 300 tokens 37.6 / 34.2; 4 x 1536, 400 tokens 29.4 / 25.2; not taken and rightly so -
// 4 x 768, 65 tokens 15.5 / 16.8, 300 tokens 14.6 / 15.0 (short); 2 x 3072, 256 tokens 33.6 / 37.2 (a whole row tile pair);
// 8 x 2048, 100 tokens 21.1 / 21.9; 8 x 4096, everything shared, 300 tokens 77.0 / 78.5.
struct MidPlan { ForwardPlan one[2]; bool use; int bn, ncols; double us; Deal deal; };      // one: the layers' own plans

constexpr int kMidMaxTokens = 512;
constexpr double kMidItem = 3.0;                    // of a tile beside its k-steps, in k-steps
constexpr double kMidMargin = 1.05, kMidShortest = 6.0;
static double mid_step_us(int bn) { return 0.09 + 0.10 * bn / 160.0; }

static int mid_workers() { return sm_count() / 2 < kMaxDealWorkers ? sm_count() / 2 : kMaxDealWorkers; }

// max_groups: 1 where the layer has no planes
static void mid_plan(const RowparShapes* s, const int* max_groups, MidPlan* out) {
  constexpr int n = 2;
  MidPlan& m = *out;
  const ForwardPlan* f = m.one;
  for (int l = 0; l < n; ++l) m.one[l] = forward_plan(s[l], max_groups[l]);
  m.use = false;
  m.deal.dealt = 0;
  if (s[0].T <= kDecodeMaxTokens || s[0].T > kMidMaxTokens) return;
  m.ncols = (s[0].T + 255) / 256;
  m.bn = round_up((s[0].T + m.ncols - 1) / m.ncols, 32);
  FewSplit sp[2];
  int K[2];
  double us = 0;
  for (int l = 0; l < n; ++l) {
    sp[l] = FewSplit{f[l].qper, 1};
    K[l] = s[l].K_r;
    us += 0.2 * plane_cost(s[l], f[l].groups);
  }
  const FewTiles t = few_tiles(s[0].t, s[0].h, s[0].S, K, n, sp, 2 * BM, m.ncols, kMidItem);
  m.us = us + few_makespan(t, mid_workers()) * mid_step_us(m.bn);
  m.use = t.tiles <= kMaxDealItems && m.us >= kMidShortest && m.us * kMidMargin < 0.2 * (f[0].tile.cost + f[1].tile.cost);
  if (m.use && t.tiles > mid_workers()) few_deal(t, mid_workers(), &m.deal);
}

// the plans of up to kMidMaxTokens tokens are kept; for more there is only forward_plan, once a call as ever
static void mid_plan_cached(const RowparShapes* s, const int* max_groups, MidPlan* out) {
  static PlanCache<MidPlan, 9> cache;
  if (s[0].T > kMidMaxTokens) return mid_plan(s, max_groups, out);
  cache.get({{s[0].t, s[0].T, s[0].h, s[0].S, s[0].K_r, s[1].K_r, max_groups[0], max_groups[1], sm_count()}}, out,
            [&](MidPlan* p) { mid_plan(s, max_groups, p); });
}

static cudaError_t launch_mid(const RowparShapes* s, const MidPlan& m, const void* const* Y, const void* const* W,
                              void* const* zs, void* const* zp, void* const* planes, cudaStream_t st) {
  const ForwardPlan* fp = m.one;
  Maps mp;
  Params p{};
  p.BN = m.bn; p.cg = 2; p.splits = 1;
  for (int l = 0; l < 2; ++l) {
    const int ks = (s[l].K_r + BK - 1) / BK;
    if (!make_map(&mp.ab[2 * l], W[l], s[l].K_r, s[l].h, s[l].t, s[l].K_r, (long long)s[l].h * s[l].K_r, BK, BM) ||
        !make_map(&mp.ab[2 * l + 1], Y[l], s[l].K_r, s[l].T, s[l].t, s[l].K_r, (long long)s[l].T * s[l].K_r, BK, p.BN / 2))
      return cudaErrorInvalidValue;
    if (s[l].S > 0) {
      Region& r = p.r[p.nregions++];
      r.nunits = 1;
      r.u[0] = Unit{2 * l, 2 * l + 1, 0, 0, 0, 0, 0, 1, 0, 1, s[l].t, ks};
      r.M = s[l].S; r.N = s[l].T; r.batch = 1; r.b_slowest = 1;
      r.splits = fp[l].groups; r.qper = fp[l].groups > 1 ? fp[l].qper : 0;
      r.out_f32 = fp[l].groups > 1;
      r.out_t = static_cast<float*>(r.out_f32 ? planes[l] : zs[l]); r.out_ld = s[l].S_hi;
    }
    if (s[l].S < s[l].h) {
      Region& r = p.r[p.nregions++];
      r.nunits = 1;
      r.u[0] = Unit{2 * l, 2 * l + 1, 0, s[l].S_lo, 0, 0, 1, 0, 1, 0, 1, ks};
      r.M = s[l].P; r.N = s[l].T; r.batch = s[l].t; r.b_slowest = 1;
      r.splits = 1;
      r.out_t = static_cast<float*>(zp[l]); r.out_ld = s[l].P;
    }
  }
  for (CUtensorMap& c : mp.c) c = mp.ab[0];          // unused: the epilogue stores directly
  finish_tiles(p);
  return launch(mp, p, CAAT_K_TC_FORWARD, st, nullptr, &m.deal);
}

// When the products of a block's two layers share a launch (units of 0.2 us): a launch of its own is worth kLaunchGap, the
// shared one has to win by kMargin, and it has to be shorter than kLongest.
constexpr double kLaunchGap = 12, kMargin = 1.05, kLongest = 1200;

// Both layers' forward products of a block (they do not depend on each other): one launch where the cost model sees a
// gain - one ramp, one tail and a finer deal where a layer's tiles do not fill the GPU - else one after the other.  Each
// layer keeps the rank groups that it would have alone, so its sums do not depend on the schedule.
// The rule: a launch of its own costs 2.4 us; against that, one launch has to be cheaper than the two by 5 % of its own
// time, which is what it loses to the model when both layers' operands go through L2 and only one tile width is left to
// choose.  Block forward on either side of the line (apart / merged, us): taken - h 768, 300 tokens 21.9 / 14.9; h 2048,
// 300 tokens 44.0 / 38.8, 2000 tokens 147 / 143; h 4096, 600 tokens 153 / 147, 3000 tokens 571 / 539; not taken - h 4096,
// 1400 tokens 273 / 285; h 5120, 1000 tokens 306 / 312; h 4096, p = 0.75 on 2 ranks, 300 tokens 75 / 87; long launches (see
// the backward's) - h 4096, 8192 tokens 1389 / 1394, whole step 3810 / 3832, 65536 tokens of 4 x 768 2309 / 2337.
cudaError_t launch_tc_forward_block(const RowparShapes* s, const void* const* Y, const void* const* W, void* const* zs,
                                    void* const* zp, void* const* planes, const int* max_groups, int* groups, cudaStream_t st) {
  static thread_local MidPlan mid;
  const int room[2] = {planes[0] ? max_groups[0] : 1, planes[1] ? max_groups[1] : 1};
  mid_plan_cached(s, room, &mid);
  const ForwardPlan* one = mid.one;
  if (mid.use) {
    for (int l = 0; l < 2; ++l) groups[l] = one[l].groups;
    return launch_mid(s, mid, Y, W, zs, zp, planes, st);
  }
  const int ks[2] = {(s[0].K_r + BK - 1) / BK, (s[1].K_r + BK - 1) / BK};
  const int lead = ks[1] * one[1].qper >= ks[0] * one[0].qper ? 1 : 0;        // the layer with the longer shared tiles
  RegionShape rs[4];
  for (int i = 0; i < 2; ++i) {
    const int l = i == 0 ? lead : 1 - lead;
    rs[i] = RegionShape{s[l].T, s[l].S, one[l].groups, ks[l] * one[l].qper};
    rs[2 + i] = RegionShape{s[l].T, s[l].S < s[l].h ? s[l].h - s[l].S_lo : 0, s[l].t, ks[l]};
  }
  TileCfg both = pick_tile(rs, 4, false, 1, 0.0);
  for (int l = 0; l < 2; ++l) both.cost += plane_cost(s[l], one[l].groups);
  if (both.cost * kMargin >= one[0].tile.cost + one[1].tile.cost + kLaunchGap || both.cost >= kLongest) {
    for (int l = 0; l < 2; ++l) {
      const cudaError_t e = launch_tc_forward(s[l], Y[l], W[l], zs[l], zp[l], st, nullptr, planes[l], max_groups[l], &groups[l]);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  Maps mp;
  Params p{};
  p.BN = both.bn; p.cg = both.cg; p.splits = 1;
  for (int l = 0; l < 2; ++l) {
    groups[l] = one[l].groups;
    if (!forward_maps(mp, l, s[l], Y[l], W[l], p)) return cudaErrorInvalidValue;
  }
  for (int i = 0; i < 2; ++i) {
    const int l = i == 0 ? lead : 1 - lead;
    if (s[l].S > 0 && !forward_shared(mp, p, l, s[l], zs[l], planes[l], one[l].groups, one[l].qper)) return cudaErrorInvalidValue;
  }
  for (int i = 0; i < 2; ++i) {
    const int l = i == 0 ? lead : 1 - lead;
    if (s[l].S < s[l].h && !forward_private(mp, p, l, s[l], zp[l])) return cudaErrorInvalidValue;
  }
  finish_tiles(p);
  return launch(mp, p, CAAT_K_TC_FORWARD, st);
}

int tc_forward_groups(const RowparShapes& s, int max_groups) { return forward_plan(s, max_groups).groups; }

cudaError_t launch_tc_forward(const RowparShapes& s, const void* Y, const void* W, void* zs, void* zp,
                              cudaStream_t st, const PushTarget* push, void* planes, int max_groups, int* groups_out) {
  Maps mp;
  CUtensorMap *maps = mp.ab, *cmaps = mp.c;
  PeerMaps pmaps{};
  Params p{};
  const int n_sh = s.S, n_pr = s.S < s.h ? s.h - s.S_lo : 0;
  const ForwardPlan plan = forward_plan(s, planes ? max_groups : 1);
  const int groups = plan.groups, qper = plan.qper;
  p.BN = plan.tile.bn; p.cg = plan.tile.cg;
  if (groups_out) *groups_out = groups;
  p.a_mn = 0; p.b_mn = 0; p.splits = 1;
  if (!forward_maps(mp, 0, s, Y, W, p)) return cudaErrorInvalidValue;
  maps[2] = maps[0];
  maps[3] = maps[1];
  if (n_sh > 0 && !forward_shared(mp, p, 0, s, zs, planes, groups, qper)) return cudaErrorInvalidValue;
  if (n_pr > 0 && !forward_private(mp, p, 0, s, zp)) return cudaErrorInvalidValue;
  if (push && n_sh > 0 && groups == 1) {
    // shared tiles go to the owners' receive slots: slot `rank` of GPU q is [slice, S] 16-bit elements; the map of
    // owner q covers only the tokens q really owns, so rows past the end of a ragged last slice are clipped
    if (push->world < 1 || push->world > CAAT_MAX_PEERS || push->slice % (BM * p.cg) != 0) return cudaErrorInvalidValue;
    for (int q = 0; q < push->world; ++q) {
      long long rows = (long long)s.T - (long long)q * push->slice;
      if (rows > push->slice) rows = push->slice;
      if (rows < 1) { pmaps.m[q] = cmaps[0]; continue; }     // owns no token: never addressed
      __nv_bfloat16* slot = static_cast<__nv_bfloat16*>(push->recv[q]) + (size_t)push->rank * push->slice * n_sh;
      if (!make_cmap(&pmaps.m[q], slot, n_sh, rows, 1, n_sh, (long long)push->slice * n_sh, false)) return cudaErrorInvalidValue;
    }
    p.push_slice = push->slice;
  }
  finish_tiles(p);
  const cudaError_t e = launch(mp, p, CAAT_K_TC_FORWARD, st, push && n_sh > 0 && groups == 1 ? &pmaps : nullptr);
  if (e != cudaSuccess || groups == 1 || groups_out) return e;
  const long long n8 = (long long)s.T * s.S_hi / 8;
  const int blocks = (int)((n8 + 255) / 256 < 8 * sm_count() ? (n8 + 255) / 256 : 8 * sm_count());
  LaunchScope scope(CAAT_K_SPLITK_REDUCE, st);
  SlotTarget slots{};
  if (push) {
    slots.slice = push->slice; slots.rank = push->rank;
    for (int q = 0; q < push->world; ++q) slots.recv[q] = static_cast<uint4*>(push->recv[q]);
  }
  return launch_pdl(sum_groups_kernel, dim3(blocks), dim3(256), 0, st, static_cast<const float4*>(planes), static_cast<uint4*>(zs),
                    s.T, s.S_hi / 8, groups, slots);
}

cudaError_t launch_tc_forward_decode(int t, int T, int h, int S, DecodeProblem* pr, int n, cudaStream_t st) {
  if (n < 1 || n > 2) return cudaErrorInvalidValue;
  static thread_local FewPlan plan;
  {
    const int K[2] = {pr[0].K_r, n > 1 ? pr[1].K_r : 0};
    few_plan_cached(t, T, h, S, K, n, &plan);
  }
  Maps mp;
  Params p{};
  p.BN = (T + 31) / 32 * 32;
  if (p.BN > kDecodeMaxTokens) return cudaErrorInvalidValue;
  p.cg = 1;
  p.splits = 1;
  const int S_lo = round_down(S, kLayoutVec), S_hi = round_up(S, kLayoutVec), P = h - S_lo;
  int g = 0;
  for (int l = 0; l < n; ++l) {
    DecodeProblem& q = pr[l];
    const FewSplit sp = plan.l[l];
    const int ks = (q.K_r + BK - 1) / BK;
    q.ns = S > 0 ? few_shared_planes(sp, t) : 0;
    q.np = S < h ? sp.ksplits : 0;
    q.zp = q.zs + (size_t)q.ns * T * S_hi;
    if (!make_map(&mp.ab[2 * l], q.W, q.K_r, h, t, q.K_r, (long long)h * q.K_r, BK, BM)) return cudaErrorInvalidValue;
    if (!make_map(&mp.ab[2 * l + 1], q.Y, q.K_r, T, t, q.K_r, (long long)T * q.K_r, BK, p.BN)) return cudaErrorInvalidValue;
    if (S > 0) {
      Region& r = p.r[g++];
      const bool grouped = sp.qper > 0;
      r.nunits = 1;
      r.u[0] = Unit{2 * l, 2 * l + 1, 0, 0, 0, 0, !grouped, grouped, !grouped, grouped, grouped ? t : 1, ks};
      r.M = S; r.N = T; r.batch = grouped ? 1 : t; r.b_slowest = 1;
      r.splits = grouped ? q.ns : sp.ksplits;
      r.qper = sp.qper;
      r.out_t = q.zs; r.out_ld = S_hi;
    }
    if (S < h) {
      Region& r = p.r[g++];
      r.nunits = 1;
      r.u[0] = Unit{2 * l, 2 * l + 1, 0, S_lo, 0, 0, 1, 0, 1, 0, 1, ks};
      r.M = P; r.N = T; r.batch = t; r.b_slowest = 1;
      r.splits = sp.ksplits;
      r.out_t = q.zp; r.out_ld = P;
    }
  }
  if (n == 1) { mp.ab[2] = mp.ab[0]; mp.ab[3] = mp.ab[1]; }
  for (CUtensorMap& c : mp.c) c = mp.ab[0];          // unused: the epilogue stores directly
  p.nregions = g;
  finish_tiles(p);
  return launch(mp, p, CAAT_K_TC_FORWARD, st, nullptr, &plan.deal);
}

// ---- dgrad: dY[m] = gs W[m][:S] + (alpha gp[m]) W[m][S:]
// pv describes where the private gradient lives and what still multiplies it (see PrivOperand); when
// pv.alpha != 1, w_scaled ([t, h, K_r], only rows >= S are used) must hold alpha times the private rows of W.
// Any partition S: the private gradient is read from column S_lo on, and the weights' map starts at row S with the
// coordinate -(S - S_lo), so the shared columns among them meet rows that TMA fills with zeros.
static RegionShape dgrad_shape(const RowparShapes& s) {
  return RegionShape{s.T, s.K_r, s.t, (s.S + BK - 1) / BK + (s.h - s.S_lo + BK - 1) / BK};
}

// the next region of the launch: one layer's data gradient, its operand maps ab[b] .. ab[b + 3]
template <typename M>
static bool dgrad_region(M& mp, Params& p, int b, const RowparShapes& s, const void* gs, const PrivOperand& pv, const void* W,
                         void* dY, const void* w_scaled) {
  CUtensorMap* maps = mp.ab + b;
  const int n_sh = s.S, n_pr = s.S < s.h ? s.h - s.S_lo : 0;
  // B = W[m] as [h rows (contraction)][K_r contiguous (N)]: N-major, boxes of 64 (N) x 64 (K)
  if (!make_map(&maps[1], W, s.K_r, s.h, s.t, s.K_r, (long long)s.h * s.K_r, 64, BK)) return false;
  maps[3] = maps[1];
  if (n_pr > 0) {
    const void* wp = W;
    if (pv.alpha != 1.0f && !pv.gs_over_alpha) {
      // sum_l (alpha g[l]) W[l][k] = sum_l g[l] (alpha W[l][k]): the private gradient is read as stored in dR,
      // the weights' private rows (the small operand) carry alpha; they were scaled by the launch before this one
      if (!w_scaled) return false;
      wp = w_scaled;
    }
    if (!make_map(&maps[3], static_cast<const __nv_bfloat16*>(wp) + (long long)s.S * s.K_r, s.K_r, s.h - s.S, s.t, s.K_r,
                  (long long)s.h * s.K_r, 64, BK))
      return false;
  }
  if (n_sh > 0 && !make_map(&maps[0], gs, n_sh, s.T, 1, s.S_hi, (long long)s.T * s.S_hi, BK, BM)) return false;
  if (n_pr > 0 && !make_map(&maps[2], pv.ptr, pv.ld, s.T, s.t, pv.ld, (long long)s.T * pv.ld, BK, BM)) return false;
  if (n_sh == 0) maps[0] = maps[2];
  if (n_pr == 0) maps[2] = maps[0];
  Region& r = p.r[p.nregions];
  int nu = 0;
  if (n_sh > 0) r.u[nu++] = Unit{b, b + 1, 0, 0, 0, 0, 0, 0, 1, 0, 1, (n_sh + BK - 1) / BK};
  if (n_pr > 0) r.u[nu++] = Unit{b + 2, b + 3, pv.col0, 0, s.S_lo - s.S, 0, 1, 0, 1, 0, 1, (n_pr + BK - 1) / BK};
  r.nunits = nu;
  r.M = s.T; r.N = s.K_r; r.batch = s.t; r.b_slowest = 1; r.scale = pv.gs_over_alpha ? pv.alpha : 1.0f;
  return make_cmap(&mp.c[p.nregions++], dY, s.K_r, s.T, s.t, s.K_r, (long long)s.T * s.K_r, false);
}

cudaError_t launch_tc_dgrad(const RowparShapes& s, const void* gs, const PrivOperand& pv, const void* W, void* dY,
                            void* w_scaled, bool w_scaled_ready, cudaStream_t st) {
  Maps mp;
  Params p{};
  const RegionShape rs = dgrad_shape(s);
  const TileCfg c = pick_tile(&rs, 1, true, 1, 0.0);
  p.BN = c.bn; p.cg = c.cg;
  p.a_mn = 0; p.b_mn = 1;  p.splits = 1;
  if (!dgrad_region(mp, p, 0, s, gs, pv, W, dY, w_scaled_ready ? w_scaled : nullptr)) return cudaErrorInvalidValue;
  finish_tiles(p);
  return launch(mp, p, CAAT_K_TC_DGRAD, st);
}

static TileCfg wgrad_cfg(const RowparShapes& s) {
  const int ksteps = (s.T + BK - 1) / BK;
  const RegionShape rs[2] = {{s.S, s.K_r, s.t, ksteps}, {s.S < s.h ? s.h - s.S_lo : 0, s.K_r, s.t, ksteps}};
  return pick_tile(rs, 2, true, 16, (double)s.t * s.h * s.K_r * sizeof(float));
}

size_t tc_wgrad_splitk_bytes(const RowparShapes& s) {
  const int splits = wgrad_cfg(s).splits;
  return splits > 1 ? (size_t)splits * s.t * s.h * s.K_r * sizeof(float) : 0;
}

// ---- wgrad: dW[m][:S] = gs^T Y[m] ; dW[m][S:] = alpha gp[m]^T Y[m]      (fp32 out; alpha in the epilogue)
// operand maps of one layer: ab[b] the shared gradient, ab[b + 1] the activations, ab[b + 2] the private gradient
template <typename M>
static bool wgrad_maps(M& mp, int b, const RowparShapes& s, const void* gs, const PrivOperand& pv, const void* Y) {
  CUtensorMap* maps = mp.ab + b;
  const int n_sh = s.S, n_pr = s.S < s.h ? s.h - s.S_lo : 0;
  // A = dZt as [T rows (contraction)][channels contiguous (M)]: M-major, boxes of 64 (M) x 64 (K)
  if (n_sh > 0 && !make_map(&maps[0], gs, n_sh, s.T, 1, s.S_hi, (long long)s.T * s.S_hi, 64, BK)) return false;
  if (n_pr > 0 && !make_map(&maps[2], pv.ptr, pv.ld, s.T, s.t, pv.ld, (long long)s.T * pv.ld, 64, BK)) return false;
  // B = Y[m] as [T rows (contraction)][K_r contiguous (N)]: N-major
  if (!make_map(&maps[1], Y, s.K_r, s.T, s.t, s.K_r, (long long)s.T * s.K_r, 64, BK)) return false;
  if (n_sh == 0) maps[0] = maps[2];
  if (n_pr == 0) maps[2] = maps[0];
  return true;
}
// the next region or regions of the launch; out: dW, or the split-K planes
template <typename M>
static bool wgrad_regions(M& mp, Params& p, int b, const RowparShapes& s, const PrivOperand& pv, float* out, int splits) {
  const int n_sh = s.S, n_pr = s.S < s.h ? s.h - s.S_lo : 0, ksteps = (s.T + BK - 1) / BK;
  if (n_sh > 0) {
    Region& r = p.r[p.nregions];
    r.nunits = 1;
    r.u[0] = Unit{b, b + 1, 0, 0, 0, 0, 0, 0, 1, 0, 1, ksteps};
    r.out_f32 = 1;
    r.a_mn = 1;
    r.M = n_sh; r.N = s.K_r; r.batch = s.t; r.b_slowest = 0;   // the shared gradient panel serves all ranks at once
    r.scale = pv.gs_over_alpha ? pv.alpha : 1.0f;
    if (!make_cmap(&mp.c[p.nregions++], out, s.K_r, n_sh, (long long)s.t * splits, s.K_r, (long long)s.h * s.K_r, true)) return false;
  }
  if (n_pr > 0) {
    Region& r = p.r[p.nregions];
    r.nunits = 1;
    r.u[0] = Unit{b + 2, b + 1, 0, pv.col0, 0, 0, 1, 0, 1, 0, 1, ksteps};
    r.out_f32 = 1;
    r.a_mn = 1;
    r.M = n_pr; r.N = s.K_r; r.batch = s.t; r.b_slowest = 1;
    r.scale = pv.alpha;
    r.skip = s.S - s.S_lo;
    r.skip_out = out + (long long)s.S_lo * s.K_r;
    r.skip_plane = (long long)s.h * s.K_r;
    if (!make_cmap(&mp.c[p.nregions++], out + (long long)s.S_lo * s.K_r, s.K_r, n_pr, (long long)s.t * splits, s.K_r,
                   (long long)s.h * s.K_r, true))
      return false;
  }
  return true;
}

cudaError_t launch_tc_wgrad(const RowparShapes& s, const void* gs, const PrivOperand& pv, const void* Y, float* dW,
                            void* splitk, size_t splitk_bytes, cudaStream_t st) {
  Maps mp;
  Params p{};
  const TileCfg wc = wgrad_cfg(s);
  p.BN = wc.bn; p.cg = wc.cg;
  const int splits = wc.splits;
  const long long dw_elems = (long long)s.t * s.h * s.K_r;
  if (splits > 1 && splitk_bytes < (size_t)splits * dw_elems * sizeof(float)) return cudaErrorInvalidValue;
  p.a_mn = 1; p.b_mn = 1;  p.splits = splits;
  if (!wgrad_maps(mp, 0, s, gs, pv, Y) || !wgrad_regions(mp, p, 0, s, pv, splits > 1 ? static_cast<float*>(splitk) : dW, splits))
    return cudaErrorInvalidValue;
  finish_tiles(p);
  cudaError_t e = launch(mp, p, CAAT_K_TC_WGRAD, st);
  if (e != cudaSuccess) return e;
  if (splits > 1) {
    const long long n4 = dw_elems / 4;   // K_r is a multiple of 8
    int blocks = (int)((n4 + 255) / 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    LaunchScope scope(CAAT_K_SPLITK_REDUCE, st);
    e = launch_pdl(splitk_reduce_kernel, dim3(blocks), dim3(256), 0, st, static_cast<const float4*>(splitk),
                   reinterpret_cast<float4*>(dW), n4, splits);
  }
  return e;
}

// ---- a block's four gradient products, independent of one another once both layers' row work is done: one launch,
// longest contractions first, so that the short tiles of the data gradients fill the last rounds of the weight gradients
// and three ramps and tails go away.  A launch of its own is worth 2.4 us and one launch has to win by 5 % of its time, as
// in the forward; and it has to be short: the CTAs of a long launch drift apart and stop sharing operands in L2, which costs
// more than the tails.  Training step of a block, four launches / one (us): taken - 4 x 768, 300 tokens 56.9 / 39.8, 3000
// tokens 148 / 131, 16384 tokens 606 / 596; 8 x 2048, 600 tokens 166 / 150, 2999 tokens (p = 0.7) 549 / 537, 8192 tokens
// 1360 / 1340; 8 x 4096, 300 tokens 289 / 281, 1000 tokens 572 / 554; not taken - 3000 tokens 1500 / 1503, 16384 tokens
// 7730 / 8250.
BwdBlockPlan tc_backward_block_plan(const RowparShapes* shapes) {
  RegionShape rs[kMaxRegions] = {};
  BwdBlockPlan b{};
  int n = 0;
  b.wgrad_first = (shapes[0].T + BK - 1) / BK >= dgrad_shape(shapes[0]).ksteps;
  double apart = 3 * kLaunchGap;
  for (int pass = 0; pass < 2; ++pass)
    for (int l = 1; l >= 0; --l) {
      const RowparShapes& s = shapes[l];
      if ((pass == 0) == b.wgrad_first) {
        const int ksteps = (s.T + BK - 1) / BK;
        apart += wgrad_cfg(s).cost;
        rs[n++] = RegionShape{s.S, s.K_r, s.t, ksteps};
        rs[n++] = RegionShape{s.S < s.h ? s.h - s.S_lo : 0, s.K_r, s.t, ksteps};
      } else {
        rs[n] = dgrad_shape(s);
        apart += pick_tile(rs + n, 1, true, 1, 0.0).cost;
        ++n;
      }
    }
  const TileCfg c = pick_tile(rs, n, true, 1, 0.0);
  b.bn = c.bn; b.cg = c.cg;
  b.merged = c.cost * kMargin < apart && c.cost < kLongest;
  return b;
}

cudaError_t launch_tc_backward_block(const BwdBlockPlan& b, const BwdGemm* L, cudaStream_t st) {
  MapsT<true> mp;
  Params p{};
  p.BN = b.bn; p.cg = b.cg; p.b_mn = 1; p.splits = 1;
  for (int l = 0; l < 2; ++l)
    if (!wgrad_maps(mp, 8 + 3 * l, L[l].s, L[l].gs, L[l].pv, L[l].Y)) return cudaErrorInvalidValue;
  for (int pass = 0; pass < 2; ++pass)
    for (int l = 1; l >= 0; --l) {
      const BwdGemm& g = L[l];
      const bool ok = (pass == 0) == b.wgrad_first ? wgrad_regions(mp, p, 8 + 3 * l, g.s, g.pv, g.dW, 1)
                                                   : dgrad_region(mp, p, 4 * l, g.s, g.gs, g.pv, g.W, g.dY, g.w_scaled);
      if (!ok) return cudaErrorInvalidValue;
    }
  finish_tiles(p);
  return launch<true>(mp, p, CAAT_K_TC_WGRAD, st);
}

}  // namespace caat
