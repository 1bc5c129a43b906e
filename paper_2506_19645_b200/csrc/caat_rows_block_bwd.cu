// Row work of BOTH layers of a block backward in one pass (bulk-copy staged).
//
// The second layer's residual gradient is the first one's stream gradient, so a pass per layer writes it and reads it
// back: one of the eight row-sized transfers of the two passes (dX, Hn, dHn, dR each).  Neither layer's row sums need the
// other layer's result - the stream gradient is only added at the end - so a CTA reduces both rows with one barrier
// instead of one per layer.  Bound by HBM (seven transfers of a row), with the instruction issue close behind.
//
// Training step of a block, a pass per layer -> one pass: 4 x 768 (h), 500 tokens 78.7 -> 68.7 us, 16384 tokens 605 -> 589;
// 4 x 1024, 3000 tokens 227 -> 193, LayerNorm 274 -> 207; 8 x 2048, 600 tokens 179.6 -> 166.6, 2999 tokens (p = 0.7)
// 568 -> 540, 8192 tokens on the compact stream 1378 -> 1340, p = 0.25 1408 -> 1395; 8 x 3072, 500 tokens 241 -> 236;
// 8 x 4096, 1000 tokens 591 -> 577, 8192 tokens 3800 -> 3779 (the whole step is bound by the GEMMs' power there).
//
// Ring, bounded waits and time-outs are the staged kernel's (caat_rows_staged.cu).
#include "caat_rows_bulk.cuh"

namespace caat {
namespace {

using namespace rows;
using bf16 = __nv_bfloat16;

constexpr int V = 8, H2 = 4, ES = 2;

struct BwdBlockGeom {
  int nstages;
  // per layer (0: first, 1: second): dX rows, rows of the new stream; compact: shared rows of the stream.  The gradient on
  // the outgoing stream belongs to the second layer.
  uint32_t off_x[2], off_h[2], off_hs[2], off_dh, off_dhs, zero_off, stage_bytes;
  uint32_t bar_off, red_off, ring_off;
  size_t smem;
  uint32_t spin_cap, stall_bytes;
};

// sums of NV values over each token row's warps with one CTA barrier, which also ORs `failed` over the CTA
template <int NV>
__device__ __forceinline__ int row_sums(float (&v)[NV], float* red, int& par, int warps_x, int wx, int lane, int failed) {
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = warp_sum(v[q]);
  float* buf = red + ((par * blockDim.y + threadIdx.y) * NV) * 16;
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) buf[q * 16 + wx] = v[q];
  }
  const int bad = __syncthreads_or(failed);
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const float* b = buf + q * 16;      // entries past the row's warps stay zero
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < 16; w += 4) {
      if (w >= warps_x) break;
      const float4 x = *reinterpret_cast<const float4*>(b + w);
      s += (x.x + x.y) + (x.z + x.w);
    }
    v[q] = s;
  }
  par ^= 1;
  return bad;
}

template <int CPT, bool LN, int MAXT, int MINB, bool CL, bool DH>
__global__ void __launch_bounds__(MAXT, MINB)
rows_backward_block(const RowBlockBwdArgs a, const BwdBlockGeom sg, int ngroups, unsigned int* status) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t ring32 = smem_u32(smem + sg.ring_off);
  const uint32_t bar0 = smem_u32(smem + sg.bar_off);
  float* red = reinterpret_cast<float*>(smem + sg.red_off);
  const int TX = blockDim.x, TY = blockDim.y;
  const int tid = threadIdx.y * TX + threadIdx.x, nthr = TX * TY;
  const int lane = tid & 31;
  const int wid = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int wx = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const int warps_x = TX >> 5, nwarps = nthr >> 5;
  const int NS = sg.nstages, t = a.t;
  const float inv_h = 1.0f / (float)a.h;
  const int my_groups = (int)blockIdx.x < ngroups ? (ngroups - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
  const long long total = (long long)my_groups * t;

  // Producer: the next (token group, rank) to fetch.  The copies of a stage - five; compact, rank 0: eight - are dealt to
  // the warps (at least three); warp 0 posts the expected bytes.
  int pn = 0, pm = 0;
  auto fetch = [&](uint32_t stage, uint32_t bar) {
    if (pn >= my_groups) return;
    const int n = pn, m = pm;
    if (++pm == t) { pm = 0; ++pn; }
    const long long i0 = ((long long)blockIdx.x + (long long)n * gridDim.x) * TY;
    const int rowsN = (int)((a.T - i0) < TY ? (a.T - i0) : TY);
    const long long row = (long long)m * a.T + i0;
    const uint32_t b = (uint32_t)rowsN * a.h * ES;
    const uint32_t bH = CL ? (uint32_t)rowsN * a.P * ES : b;          // 0 when there is no private part
    const uint32_t bS = CL && m == 0 ? (uint32_t)rowsN * a.S_hi * ES : 0u;
    const long long offx = row * a.h * ES, offh = CL ? row * a.P * ES : offx, offs = i0 * a.S_hi * ES;
    if (!elect_one()) return;
    if (wid == 0) mbar_expect_tx(bar, 2 * b + (DH ? 3 : 2) * (bH + bS) + sg.stall_bytes);
    auto mine = [&](int c) { return c == wid || c - nwarps == wid || c - 2 * nwarps == wid; };
    if (mine(0)) bulk_g2s(stage + sg.off_x[1], static_cast<const char*>(a.dX[1]) + offx, b, bar);
    if (mine(1) && bH) bulk_g2s(stage + sg.off_h[1], static_cast<const char*>(a.Hn[1]) + offh, bH, bar);
    if (mine(2)) bulk_g2s(stage + sg.off_x[0], static_cast<const char*>(a.dX[0]) + offx, b, bar);
    if (mine(3) && bH) bulk_g2s(stage + sg.off_h[0], static_cast<const char*>(a.Hn[0]) + offh, bH, bar);
    if (DH && mine(4) && bH) bulk_g2s(stage + sg.off_dh, static_cast<const char*>(a.dHn) + offh, bH, bar);
    if constexpr (CL) {
      if (mine(5) && bS) bulk_g2s(stage + sg.off_hs[1], static_cast<const char*>(a.Hns[1]) + offs, bS, bar);
      if (mine(6) && bS) bulk_g2s(stage + sg.off_hs[0], static_cast<const char*>(a.Hns[0]) + offs, bS, bar);
      if (DH && mine(7) && bS) bulk_g2s(stage + sg.off_dhs, static_cast<const char*>(a.dHns) + offs, bS, bar);
    }
  };

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(bar0 + 8u * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < NS)   // the zero slot of every stage (no copy ever lands there)
    *reinterpret_cast<uint4*>(smem + sg.ring_off + (size_t)tid * sg.stage_bytes + sg.zero_off) = make_uint4(0u, 0u, 0u, 0u);
  constexpr int NV = LN ? 4 : 2;
  for (int q = tid; q < 2 * TY * NV * 16; q += nthr) red[q] = 0.f;
  __syncthreads();
  pdl_wait();   // from here on global memory is touched
  if (wid < 8)
    for (int q = 0; q < NS; ++q) fetch(ring32 + (uint32_t)q * sg.stage_bytes, bar0 + 8u * q);

  int col[CPT], cls[CPT];
  bool colok[CPT], kept[CPT];                  // kept - compact: this chunk of the stream exists once
  uint4 gam[2][CPT];
  float2 dg[2][CPT][H2], db[LN ? 2 : 1][CPT][H2];
  uint32_t oX[CPT], oH[CPT];
#pragma unroll
  for (int j = 0; j < CPT; ++j) {
    col[j] = (threadIdx.x + j * TX) * V;
    colok[j] = col[j] < a.h;
    cls[j] = colok[j] ? chunk_class(col[j], V, a.S) : 1;
    kept[j] = CL && cls[j] == 0;
    oX[j] = ((uint32_t)threadIdx.y * a.h + col[j]) * ES;
    oH[j] = CL ? ((uint32_t)threadIdx.y * a.P + (uint32_t)(col[j] - a.S_lo)) * ES : oX[j];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      gam[l][j] = colok[j] ? ldg<uint4>(static_cast<const char*>(a.gamma[l]) + (long long)col[j] * ES) : zero_raw<uint4>();
#pragma unroll
      for (int q = 0; q < H2; ++q) { dg[l][j][q] = f2(0.f); if constexpr (LN) db[l][j][q] = f2(0.f); }
    }
  }
  const long long rank_dr = (long long)a.T * (CL ? a.P : a.h) * ES;

  long long k = 0;
  bool dead = false;
  uint32_t sb = ring32, cph = 0;
  int cs = 0, par = 0;
  // row statistics, loaded one unit ahead
  float rs_n[2] = {0.f, 0.f}, mu_n[2] = {0.f, 0.f};
  auto load_stats = [&](uint32_t q) {
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      rs_n[l] = a.rstd[l][q];
      if (LN) mu_n[l] = a.mean[l][q];
    }
  };
  if (my_groups > 0) load_stats(min((int)(blockIdx.x * TY + threadIdx.y), a.T - 1));
  for (int n = 0; n < my_groups && !dead; ++n) {
    const long long i = ((long long)blockIdx.x + (long long)n * gridDim.x) * TY + threadIdx.y;
    uint32_t q0 = (uint32_t)min((int)i, a.T - 1);      // of this unit's row statistics (rows past T: of the last token)
    bool act[CPT];
    // stage-relative addresses of the chunk in the dX and stream rows of either layer and in the stream's gradient; the
    // zero slot when inactive: chunks past the row end or past T add exact zeros
    uint32_t aX[2][CPT], aH[2][CPT], aD[CPT], off[CPT];      // off: of the chunk inside one rank's plane of dR
    float2 gs[2][CPT][H2];
    uint4 hsh[CL ? 2 : 1][CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      act[j] = i < a.T && colok[j];
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        aX[l][j] = act[j] ? sg.off_x[l] + oX[j] : sg.zero_off;
        aH[l][j] = act[j] ? sg.off_h[l] + oH[j] : sg.zero_off;
      }
      aD[j] = act[j] && !kept[j] ? sg.off_dh + oH[j] : sg.zero_off;
      off[j] = (uint32_t)(CL ? (i * a.P + (col[j] - a.S_lo)) * ES : (i * a.h + col[j]) * ES);
#pragma unroll
      for (int q = 0; q < H2; ++q) gs[0][j][q] = gs[1][j][q] = f2(0.f);
    }

    char* dr[2] = {static_cast<char*>(a.dR[0]), static_cast<char*>(a.dR[1])};
    for (int m = 0; m < t; ++m, ++k) {
      const int failed = mbar_wait(bar0 + 8u * cs, cph, sg.spin_cap) ? 0 : 1;
      const float rs[2] = {rs_n[0], rs_n[1]}, mu[2] = {mu_n[0], mu_n[1]};
      float2 xh[2][CPT][H2], dxh[2][CPT][H2];
      uint4 rdh[CPT];
      float2 s1[2], s2[2];
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        s1[l] = s2[l] = f2(0.f);
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
          const uint4 rx = lds32<uint4>(sb + aX[l][j]);
          uint4 rh;
          if (CL && kept[j]) {
            if (m == 0) {
              const uint32_t oS = ((uint32_t)threadIdx.y * a.S_hi + col[j]) * ES;
              hsh[CL ? l : 0][j] = lds32<uint4>(sb + (act[j] ? sg.off_hs[l] + oS : sg.zero_off));
              if (DH && l == 1) unpack2(lds32<uint4>(sb + (act[j] ? sg.off_dhs + oS : sg.zero_off)), gs[1][j]);   // once
            }
            rh = hsh[CL ? l : 0][j];
          } else {
            rh = lds32<uint4>(sb + aH[l][j]);
          }
          if (l == 1) rdh[j] = DH ? lds32<uint4>(sb + aD[j]) : zero_raw<uint4>();
          float2 dx[H2], hn[H2], g[H2];
          unpack2(rx, dx);
          unpack2(rh, hn);
          unpack2(gam[l][j], g);
#pragma unroll
          for (int q = 0; q < H2; ++q) {
            xh[l][j][q] = LN ? mul2(add2(hn[q], f2(-mu[l])), f2(rs[l])) : mul2(hn[q], f2(rs[l]));
            dxh[l][j][q] = mul2(dx[q], g[q]);
            if (LN) s1[l] = add2(s1[l], dxh[l][j][q]);
            s2[l] = fma2(dxh[l][j][q], xh[l][j][q], s2[l]);
            dg[l][j][q] = fma2(dx[q], xh[l][j][q], dg[l][j][q]);
            if constexpr (LN) db[l][j][q] = add2(db[l][j][q], dx[q]);
          }
        }
      }
      float sum[NV];
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        sum[l] = s2[l].x + s2[l].y;
        if constexpr (LN) sum[2 + l] = s1[l].x + s1[l].y;
      }
      if (row_sums<NV>(sum, red, par, warps_x, wx, lane, failed)) { dead = true; break; }   // barrier: stage fully read
      if (wid < 8) fetch(sb, bar0 + 8u * cs);
      sb += sg.stage_bytes;
      if (++cs == NS) { cs = 0; cph ^= 1u; sb = ring32; }
      if (m + 1 < t) load_stats(q0 += a.T);
      else if (n + 1 < my_groups) load_stats(min((int)i + (int)gridDim.x * TY, a.T - 1));

      float2 nc1[2], nc2[2];
#pragma unroll
      for (int l = 0; l < 2; ++l) { nc2[l] = f2(-sum[l] * inv_h); nc1[l] = f2(LN ? -sum[LN ? 2 + l : 0] * inv_h : 0.f); }
#pragma unroll
      for (int j = 0; j < CPT; ++j) {
        float2 dh[H2];
        unpack2(rdh[j], dh);
#pragma unroll
        for (int l = 1; l >= 0; --l) {        // the second layer's residual gradient is the first one's stream gradient
          float2 gg[H2];
#pragma unroll
          for (int q = 0; q < H2; ++q) {
            float2 tt = fma2(xh[l][j][q], nc2[l], dxh[l][j][q]);
            if (LN) tt = add2(tt, nc1[l]);
            gg[q] = fma2(f2(rs[l]), tt, dh[q]);
          }
          const uint4 p = pack2(gg);
          if (act[j] && !kept[j]) stg<uint4>(dr[l] + off[j], p);
          if (l == 1 && !kept[j]) unpack2(p, dh);         // as stored
          if (cls[j] == 0) {
#pragma unroll
            for (int q = 0; q < H2; ++q) gs[l][j][q] = add2(gs[l][j][q], gg[q]);   // fp32 rank sum, m ascending
          } else if (!CL && cls[j] == 2) {                // the one chunk that straddles the partition
#pragma unroll
            for (int q = 0; q < H2; ++q) {
              gs[l][j][q].x += col[j] + 2 * q < a.S ? gg[q].x : 0.f;
              gs[l][j][q].y += col[j] + 2 * q + 1 < a.S ? gg[q].y : 0.f;
            }
          }
        }
      }
      dr[0] += rank_dr; dr[1] += rank_dr;
    }
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      if (dead || !act[j] || cls[j] == 1) continue;
      const long long os = (i * a.S_hi + col[j]) * ES;
      const uint4 p = pack2_scaled(gs[1][j], a.gs_scale);
      stg<uint4>(static_cast<char*>(a.gs[1]) + os, p);
      if constexpr (CL) {                            // the single shared stream: its gradient joins the first layer's sum
        float2 d[H2];
        unpack2(p, d);
#pragma unroll
        for (int q = 0; q < H2; ++q) gs[0][j][q] = add2(gs[0][j][q], d[q]);
      }
      stg<uint4>(static_cast<char*>(a.gs[0]) + os, pack2_scaled(gs[0][j], a.gs_scale));
    }
  }
  if (dead) {
    if (tid == 0) {
      atomicExch(status, 11u);
      const long long issued = (k + NS) < total ? (k + NS) : total;
      for (long long q = k + 1; q < issued; ++q)
        for (uint32_t it = 0; it < (1u << 10); ++it)   // each poll sleeps up to the suspend hint: ~20 ms per stage at most
          if (mbar_try(bar0 + 8u * (uint32_t)(q % NS), (uint32_t)((q / NS) & 1))) break;
    }
    return;
  }

  // Partial norm-parameter gradients of this CTA: one row of [h] per CTA, its token rows summed in order through shared
  // memory (over the ring, which nothing reads any more).
  float* acc = reinterpret_cast<float*>(smem + sg.ring_off);   // [TY][TX * V]
  const int per_row = TX * CPT * V;
#pragma unroll
  for (int which = 0; which < (LN ? 4 : 2); ++which) {
    const int l = which & 1;
    float* out = which < 2 ? a.dgpart[l] : a.dbpart[l];
    if (TY > 1) __syncthreads();
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      const float2* src = which < 2 ? dg[l][j] : db[LN ? l : 0][j];
      if (TY > 1) {
#pragma unroll
        for (int q = 0; q < H2; ++q) *reinterpret_cast<float2*>(acc + threadIdx.y * per_row + col[j] + 2 * q) = src[q];
      } else if (colok[j]) {
#pragma unroll
        for (int q = 0; q < H2; q += 2)
          *reinterpret_cast<float4*>(out + (size_t)blockIdx.x * a.h + col[j] + 2 * q) =
              make_float4(src[q].x, src[q].y, src[q + 1].x, src[q + 1].y);
      }
    }
    if (TY > 1) {
      __syncthreads();
      for (int c = tid * 4; c < a.h; c += nthr * 4) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int y = 0; y < TY; ++y) {
          const float4 v = *reinterpret_cast<const float4*>(acc + y * per_row + c);
          s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *reinterpret_cast<float4*>(out + (size_t)blockIdx.x * a.h + c) = s;
      }
    }
  }
}

// The norm-gradient and rank sums of two layers in fp32 take most of a thread's registers: one chunk per thread fits 168 (at
// 128 it costs 5 % at h = 2048, and 3000 tokens of 4 x 768 take 174 us instead of 148).  That is twelve warps per SM for
// rows of up to 192 and of 257 to 384 chunks; the other lengths take two chunks per thread at 256 registers, eight warps
// (h = 2048, 8192 tokens: 1395 us; one chunk at 128 registers 1450).
RowGeom bwd_block_rows(int h) {
  RowGeom g{};
  const int chunks = h / V;
  g.CPT = chunks <= 192 || (chunks > 256 && chunks <= 384) ? 1 : 2;
  g.TX = round_up((chunks + g.CPT - 1) / g.CPT, 32);
  g.TY = g.TX >= 96 ? 1 : 128 / g.TX;
  return g;
}
// LayerNorm: at most three CTAs (4 x 768, 16384 tokens: 684 us with three, 728 with four; RMSNorm 624 and 589).
int bwd_block_ctas(const RowGeom& g, int norm) {
  const int n = 65536 / (g.TX * g.TY * (g.CPT == 1 ? 168 : 256));
  return norm == 1 && n > 3 ? 3 : n;
}

BwdBlockGeom bwd_block_geometry(const RowGeom& g, int h, int P, int S_hi, bool compact, bool has_dh, int norm, size_t budget) {
  BwdBlockGeom b{};
  const uint32_t rowH = (uint32_t)g.TY * h * ES, rowP = (uint32_t)g.TY * P * ES, rowS = (uint32_t)g.TY * S_hi * ES;
  uint32_t o = 0;
  auto put = [&](uint32_t bytes) { const uint32_t at = o; o += bytes; return at; };
  for (int l = 0; l < 2; ++l) b.off_x[l] = put(rowH);
  for (int l = 0; l < 2; ++l) b.off_h[l] = put(compact ? rowP : rowH);
  if (has_dh) b.off_dh = put(compact ? rowP : rowH);
  if (compact) {
    for (int l = 0; l < 2; ++l) b.off_hs[l] = put(rowS);
    if (has_dh) b.off_dhs = put(rowS);
  }
  b.zero_off = o;
  b.stage_bytes = (o + 16u + 127u) & ~127u;
  size_t off = 8 * kMaxStages;
  b.red_off = (uint32_t)off; off += (size_t)2 * g.TY * 16 * (norm == 1 ? 4 : 2) * sizeof(float);
  off = align_up(off, 128);
  b.ring_off = (uint32_t)off;
  int ns = budget > off ? (int)((budget - off) / b.stage_bytes) : 0;
  b.nstages = ns > kMaxStages ? kMaxStages : ns;
  const size_t ring = (size_t)b.nstages * b.stage_bytes, acc = g.TY > 1 ? (size_t)g.TY * g.TX * g.CPT * V * sizeof(float) : 0;
  b.smem = off + (ring > acc ? ring : acc);
  const RowsHooks hooks = rows_hooks();
  b.spin_cap = hooks.spin_cap;
  b.stall_bytes = hooks.stall ? 16u : 0u;
  return b;
}

template <bool LN, bool CL>
cudaError_t launch_t(const RowBlockBwdArgs& a, const RowGeom& g, const BwdBlockGeom& sg, int grid, int ngroups,
                     unsigned int* status, cudaStream_t st) {
  const dim3 block(g.TX, g.TY);
  LaunchScope scope(CAAT_K_ROWS_BACKWARD, st);
  auto go = [&](auto k) {
    const cudaError_t e = set_smem(k, sg.smem);
    return e != cudaSuccess ? e : launch_pdl(k, dim3(grid), block, sg.smem, st, a, sg, ngroups, status);
  };
  const bool dh = a.dHn || a.dHns;
  cudaError_t e;
#define CAAT_GO(C, T, M) e = dh ? go(rows_backward_block<C, LN, T, M, CL, true>) : go(rows_backward_block<C, LN, T, M, CL, false>)
  const int n = g.TX * g.TY;
  if (g.CPT == 1 && n <= 128) CAAT_GO(1, 128, 3);
  else if (g.CPT == 1 && n <= 192) CAAT_GO(1, 192, 2);
  else if (g.CPT == 1) CAAT_GO(1, 384, 1);
  else if constexpr (!LN) {
    if (n <= 128) CAAT_GO(2, 128, 2);
    else CAAT_GO(2, 256, 1);
  } else {
    return cudaErrorInvalidValue;
  }
#undef CAAT_GO
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

bool rows_block_bwd_usable(int h, int T, int P, int S_hi, caat_dtype dtype, int compact, int norm) {
  if (dtype != CAAT_BF16 || h / V > 512 || (long long)T * h * ES >= (1LL << 32)) return false;     // 32-bit offsets in a plane
  const RowGeom g = bwd_block_rows(h);
  // a pass per layer is the faster one for: LayerNorm with two chunks per thread, whose sums spill (8 x 2048, 2000 tokens:
  // 437 us apart, 452 in one pass; 300 tokens 154 both), and many tokens of short compact rows, which the warp-per-token
  // kernels read without barriers (4 x 768, 1500 tokens: 110 and 104; 4000 tokens: 198 and 205)
  if (g.CPT == 2 && norm == 1) return false;
  if (compact && h / V <= 96 && T > 2000) return false;
  return bwd_block_geometry(g, h, P, S_hi, compact != 0, true, norm, kSmemPerSm / bwd_block_ctas(g, norm) - 1024).nstages >= 3;
}

cudaError_t launch_rows_backward_block(const RowBlockBwdArgs& a, cudaStream_t st) {
  const RowGeom g = bwd_block_rows(a.h);
  const int ngroups = (a.T + g.TY - 1) / g.TY;
  // a token's ranks are a serial chain in one CTA: before a nearly empty last round a CTA less per SM is faster (3000 tokens
  // of 4 x 768: 161 us with four, 148 with three)
  int per_sm = bwd_block_ctas(g, a.norm);
  auto used = [&](int n) { const int grid = sm_count() * n; return (double)ngroups / ((double)((ngroups + grid - 1) / grid) * grid); };
  if (per_sm > 2 && used(per_sm - 1) > 1.1 * used(per_sm)) --per_sm;
  const BwdBlockGeom sg = bwd_block_geometry(g, a.h, a.P, a.S_hi, a.compact != 0, a.dHn || a.dHns, a.norm, kSmemPerSm / per_sm - 1024);
  if (sg.nstages < 2) return cudaErrorInvalidConfiguration;
  int grid = sm_count() * per_sm;
  const int cap = rows_backward_partial_rows(a.h, a.T, CAAT_BF16);      // rows of norm-gradient partials in the scratch
  if (grid > ngroups) grid = ngroups;
  if (grid > cap) grid = cap;
  unsigned int* status = device_status_word();
  if (!status) return cudaErrorUnknown;
  cudaError_t e;
  if (a.compact) e = a.norm == 1 ? launch_t<true, true>(a, g, sg, grid, ngroups, status, st) : launch_t<false, true>(a, g, sg, grid, ngroups, status, st);
  else e = a.norm == 1 ? launch_t<true, false>(a, g, sg, grid, ngroups, status, st) : launch_t<false, false>(a, g, sg, grid, ngroups, status, st);
  if (e != cudaSuccess) return e;
  NormGradReduce r{};
  r.rows = grid;
  r.h = a.h;
  for (int l = 0; l < 2; ++l) {
    r.part[r.n] = a.dgpart[l]; r.out[r.n++] = a.dgamma[l];
    if (a.norm == 1) { r.part[r.n] = a.dbpart[l]; r.out[r.n++] = a.dbeta[l]; }
    if (a.w_dst[l]) r.scale[l] = ScaleJob{a.w_src[l], a.w_dst[l], a.t, a.h, a.w_Kr[l], a.S, a.alpha};
  }
  return launch_norm_grad_reduce(r, st);
}

}  // namespace caat
