// Row work of BOTH layers of a block forward in one pass (bulk-copy staged).
//
// The second layer's residual is the first one's new stream, so a pass per layer writes that stream and reads it back:
// one of the nine row-sized transfers of the two passes (R, Hn1, X1; Hn1, Hn2, X2 and the partial sums).  Here a CTA
// walks (token, rank) units as the staged kernel does, forms both new streams before the first reduction - the
// second stream needs the first one's values, not its norm - and reduces both rows' statistics in one CTA barrier
// (LayerNorm: two) instead of one per layer.  Bound by HBM, with the instruction issue close behind.  Block forward, a pass
// per layer -> one pass: 8 x 4096 (h), 8192 tokens 1492 -> 1424 us, 300 tokens 98.9 -> 95.3; 2 x 1024, 4000 tokens
// 87.0 -> 78.4; 4 x 768, 16384 tokens 236.4 (side by side with a GEMM) -> 227.4.  Training steps: 8 x 2048, 8192 tokens,
// p = 0.25 1439 -> 1412, compact stream 1401 -> 1374; 8 x 4096, 8192 tokens 4087 -> 3986.
//
// Layout of a stage, mapping of threads to 16-byte chunks, unit ranges and time-outs are the staged kernel's
// (caat_rows_staged.cu); what a thread keeps per token (shared sums, norm gains) stays packed in bf16, because two
// layers of it in fp32 would not fit 128 registers.
#include "caat_rows_bulk.cuh"

namespace caat {
namespace {

using namespace rows;
using bf16 = __nv_bfloat16;

constexpr int V = 8, H2 = 4, ES = 2;

struct BlockGeom {
  int nstages;
  uint32_t off_r, off_p[2], off_s[2], off_rs, zero_off, stage_bytes;   // residual, partial sums per layer, compact: shared residual
  uint32_t bar_off, red_off, ring_off;
  size_t smem;
  uint32_t spin_cap, stall_bytes;
};

// rounds a packed row of pairs to bf16 and gives the rounded values back
__device__ __forceinline__ uint4 round_pack(float2 (&f)[H2]) {
  const uint4 p = pack2(f);
  unpack2(p, f);
  return p;
}

template <int CPT, bool LN, int MAXT, bool CL, bool FEW>
__global__ void __launch_bounds__(MAXT, MAXT == 128 ? 3 : MinBlocks<CPT, MAXT>::value)
rows_forward_block(const RowBlockArgs a, const BlockGeom sg, int ngroups, unsigned int* status) {
  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t* ring = smem + sg.ring_off;
  const uint32_t bar0 = smem_u32(smem + sg.bar_off);
  float* red = reinterpret_cast<float*>(smem + sg.red_off);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + sg.bar_off + 8 * kMaxStages);
  int par = 0;
  const int TX = blockDim.x, TY = blockDim.y;
  const int tid = threadIdx.y * TX + threadIdx.x;
  const float inv_h = 1.0f / (float)a.h;
  const int NS = sg.nstages;
  const UnitRange ur = unit_range(FEW && a.flat, ngroups, a.t);
  const long long total = ur.total;

  // Fetch the next unit into stage ss.  Every thread keeps the counters; the copies of a stage are issued by elected
  // lanes of different warps, warp 0 posts the expected bytes.
  int nn = ur.n0, mm = ur.m0, ss = 0;
  long long to_issue = total;
  const int issuer = __shfl_sync(0xffffffffu, tid >> 5, 0), nwarps = TX * TY / 32;
  auto issue = [&]() {
    if (to_issue == 0) return;
    const bool first = mm == 0 || (FEW && to_issue == total);
    --to_issue;
    const int n = nn, m = mm, s = ss;
    if (++mm == a.t) { mm = 0; nn += ur.nstep; }
    if (++ss == NS) ss = 0;
    if (issuer > 5) return;
    const long long i0 = (long long)n * TY;
    const int rowsN = (int)((a.T - i0) < TY ? (a.T - i0) : TY);
    const uint32_t bar = bar0 + 8u * s;
    const uint32_t dst = smem_u32(ring + (size_t)s * sg.stage_bytes);
    const uint32_t bP = a.S < a.h ? (uint32_t)rowsN * a.P * ES : 0u;
    const uint32_t bR = CL ? bP : (uint32_t)rowsN * a.h * ES;
    const uint32_t bS = first && a.S > 0 ? (uint32_t)rowsN * a.S_hi * ES : 0u;
    const uint32_t b0 = FEW && a.zgroups[0] > 1 ? 0u : bS, b1 = FEW && a.zgroups[1] > 1 ? 0u : bS, bRs = CL ? bS : 0u;
    const long long row = (long long)m * a.T + i0;
    if (!elect_one()) return;
    if (issuer == 0) mbar_expect_tx(bar, bR + 2 * bP + b0 + b1 + bRs + sg.stall_bytes);
    auto mine = [&](int c) { return c == issuer || c - nwarps == issuer; };     // at least three warps
    if (mine(0) && bR) bulk_g2s(dst + sg.off_r, static_cast<const char*>(a.R) + row * (CL ? a.P : a.h) * ES, bR, bar);
    if (mine(1) && bP) bulk_g2s(dst + sg.off_p[0], static_cast<const char*>(a.zp[0]) + row * a.P * ES, bP, bar);
    if (mine(2) && bP) bulk_g2s(dst + sg.off_p[1], static_cast<const char*>(a.zp[1]) + row * a.P * ES, bP, bar);
    if (mine(3) && b0) bulk_g2s(dst + sg.off_s[0], static_cast<const char*>(a.zs[0]) + i0 * a.S_hi * ES, b0, bar);
    if (mine(4) && b1) bulk_g2s(dst + sg.off_s[1], static_cast<const char*>(a.zs[1]) + i0 * a.S_hi * ES, b1, bar);
    if (mine(5) && bRs) bulk_g2s(dst + sg.off_rs, static_cast<const char*>(a.Rs) + i0 * a.S_hi * ES, bRs, bar);
  };

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(bar0 + 8u * s, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < NS)   // the zero slot of every stage (no copy ever lands there)
    *reinterpret_cast<uint4*>(ring + (size_t)tid * sg.stage_bytes + sg.zero_off) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  pdl_wait();   // from here on global memory is touched
  for (int q = 0; q < NS; ++q) issue();

  const uint32_t ring32 = smem_u32(ring);
  int col[CPT], cls[CPT];
  bool colok[CPT];
  uint32_t oR[CPT], oP[CPT];      // byte offsets of the chunk inside the residual's and the private sums' rows of a stage
  uint4 gam[2][CPT], bet[LN ? 2 : 1][CPT];
#pragma unroll
  for (int j = 0; j < CPT; ++j) {
    col[j] = (threadIdx.x + j * TX) * V;
    colok[j] = col[j] < a.h;
    cls[j] = chunk_class(col[j], V, a.S);
    const uint32_t priv = ((uint32_t)threadIdx.y * a.P + (uint32_t)(col[j] - a.S_lo)) * ES;
    const uint32_t full = ((uint32_t)threadIdx.y * a.h + col[j]) * ES;
    oP[j] = priv;
    oR[j] = sg.zero_off;
    if (colok[j] && !(CL && cls[j] == 0)) oR[j] = sg.off_r + (CL ? priv : full);
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      gam[l][j] = colok[j] ? ldg<uint4>(static_cast<const char*>(a.gamma[l]) + (long long)col[j] * ES) : zero_raw<uint4>();
      if constexpr (LN)
        bet[l][j] = colok[j] && a.beta[l] ? ldg<uint4>(static_cast<const char*>(a.beta[l]) + (long long)col[j] * ES) : zero_raw<uint4>();
    }
  }
  const float2 alpha2 = f2(a.alpha);
  const long long rank_h = (long long)a.T * a.h * ES;
  const long long rank_hn = CL ? (long long)a.T * a.P * ES : rank_h;

  long long k = 0;
  uint32_t sb = ring32;
  int cs = 0;
  uint32_t cph = 0;
  bool dead = false;
  int m_first = ur.m0;
  for (int n = ur.n0; k < total && !dead; n += ur.nstep, m_first = 0) {
    const long long i = (long long)n * TY + threadIdx.y;
    const int m_end = FEW && total - k < a.t - m_first ? m_first + (int)(total - k) : a.t;
    const bool valid = i < a.T;
    uint4 zs[2][CPT], rsh[CL ? CPT : 1];     // this token's shared sums; compact: its shared residual
    long long qH[CPT], qX[CPT];              // byte offsets of the chunk in the new streams and in the normalised rows
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      zs[0][j] = zs[1][j] = zero_raw<uint4>();
      if constexpr (CL) rsh[j] = zero_raw<uint4>();
      qX[j] = (i * a.h + col[j]) * ES + m_first * rank_h;
      qH[j] = CL ? (i * a.P + (col[j] - a.S_lo)) * ES + m_first * rank_hn : qX[j];
    }
    long long stat = i + (long long)m_first * a.T;

    for (int m = m_first; m < m_end; ++m, ++k) {
      if (!mbar_wait(bar0 + 8u * cs, cph, sg.spin_cap)) *abort_flag = 1;
      float2 h1[CPT][H2], h2[CPT][H2];
      float2 acc1 = f2(0.f), acc2 = f2(0.f);
#pragma unroll
      for (int j = 0; j < CPT; ++j) {
        if (m == m_first && cls[j] != 1 && colok[j]) {
          const uint32_t os = ((uint32_t)threadIdx.y * a.S_hi + col[j]) * ES;
#pragma unroll
          for (int l = 0; l < 2; ++l) {
            if (FEW && a.zgroups[l] > 1)
              zs[l][j] = valid ? sum_planes<bf16>(a.zplanes[l] + i * a.S_hi + col[j], (long long)a.T * a.S_hi, a.zgroups[l])
                               : zero_raw<uint4>();
            else
              zs[l][j] = lds32<uint4>(sb + sg.off_s[l] + os);
          }
          if constexpr (CL) rsh[j] = lds32<uint4>(sb + sg.off_rs + os);
        }
        float2 r[H2], z1[H2], z2[H2];
        if (CL && cls[j] == 0) unpack2(rsh[CL ? j : 0], r);
        else unpack2(lds32<uint4>(sb + oR[j]), r);
        uint4 p1;
        if (cls[j] == 0) {
          unpack2(zs[0][j], z1);
          unpack2(zs[1][j], z2);
#pragma unroll
          for (int q = 0; q < H2; ++q) { h1[j][q] = add2(z1[q], r[q]); r[q] = h1[j][q]; }
          p1 = round_pack(r);
#pragma unroll
          for (int q = 0; q < H2; ++q) h2[j][q] = add2(z2[q], r[q]);
        } else {
          unpack2(lds32<uint4>(colok[j] ? sb + sg.off_p[0] + oP[j] : sb + sg.zero_off), z1);
          unpack2(lds32<uint4>(colok[j] ? sb + sg.off_p[1] + oP[j] : sb + sg.zero_off), z2);
          if (cls[j] == 2) {       // the one chunk that straddles the partition
            float2 s1[H2], s2[H2];
            unpack2(zs[0][j], s1);
            unpack2(zs[1][j], s2);
#pragma unroll
            for (int q = 0; q < H2; ++q) {
              const bool sx = col[j] + 2 * q < a.S, sy = col[j] + 2 * q + 1 < a.S;
              h1[j][q].x = (sx ? s1[q].x : a.alpha * z1[q].x) + r[q].x;
              h1[j][q].y = (sy ? s1[q].y : a.alpha * z1[q].y) + r[q].y;
              r[q] = h1[j][q];
            }
            p1 = round_pack(r);
#pragma unroll
            for (int q = 0; q < H2; ++q) {
              const bool sx = col[j] + 2 * q < a.S, sy = col[j] + 2 * q + 1 < a.S;
              h2[j][q].x = (sx ? s2[q].x : a.alpha * z2[q].x) + r[q].x;
              h2[j][q].y = (sy ? s2[q].y : a.alpha * z2[q].y) + r[q].y;
            }
          } else {
#pragma unroll
            for (int q = 0; q < H2; ++q) { h1[j][q] = fma2(alpha2, z1[q], r[q]); r[q] = h1[j][q]; }
            p1 = round_pack(r);
#pragma unroll
            for (int q = 0; q < H2; ++q) h2[j][q] = fma2(alpha2, z2[q], r[q]);
          }
        }
        if (valid && colok[j]) {
          if (CL && cls[j] == 0) {
            if (m == 0) {
              const long long os = (i * a.S_hi + col[j]) * ES;
              stg<uint4>(static_cast<char*>(a.Hns[0]) + os, p1);
              stg<uint4>(static_cast<char*>(a.Hns[1]) + os, pack2(h2[j]));
            }
          } else {
            stg<uint4>(static_cast<char*>(a.Hn[0]) + qH[j], p1);
            stg<uint4>(static_cast<char*>(a.Hn[1]) + qH[j], pack2(h2[j]));
          }
        }
        qH[j] += rank_hn;
#pragma unroll
        for (int q = 0; q < H2; ++q) {
          acc1 = LN ? add2(acc1, h1[j][q]) : fma2(h1[j][q], h1[j][q], acc1);
          acc2 = LN ? add2(acc2, h2[j][q]) : fma2(h2[j][q], h2[j][q], acc2);
        }
      }
      float st[2] = {acc1.x + acc1.y, acc2.x + acc2.y};
      row_reduce_sync<2>(st, red, par);      // CTA barrier: every thread is done reading this stage
      if (*abort_flag) { dead = true; break; }
      issue();
      sb += sg.stage_bytes;
      if (++cs == NS) { cs = 0; cph ^= 1u; sb = ring32; }
      float mu[2] = {0.f, 0.f}, rs[2];
      if (LN) {
        mu[0] = st[0] * inv_h;
        mu[1] = st[1] * inv_h;
        float2 v1 = f2(0.f), v2 = f2(0.f);
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
          if (!colok[j]) continue;
#pragma unroll
          for (int q = 0; q < H2; ++q) {
            const float2 d1 = add2(h1[j][q], f2(-mu[0])), d2 = add2(h2[j][q], f2(-mu[1]));
            v1 = fma2(d1, d1, v1);
            v2 = fma2(d2, d2, v2);
          }
        }
        float sq[2] = {v1.x + v1.y, v2.x + v2.y};
        row_reduce_sync<2>(sq, red, par);
        rs[0] = rsqrtf(fmaf(sq[0], inv_h, a.eps));
        rs[1] = rsqrtf(fmaf(sq[1], inv_h, a.eps));
      } else {
        rs[0] = rsqrtf(fmaf(st[0], inv_h, a.eps));
        rs[1] = rsqrtf(fmaf(st[1], inv_h, a.eps));
      }
#pragma unroll
      for (int j = 0; j < CPT; ++j) {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          float2 g[H2], x[H2];
          unpack2(gam[l][j], g);
          if constexpr (LN) {
            float2 b[H2];
            unpack2(bet[l][j], b);
#pragma unroll
            for (int q = 0; q < H2; ++q) x[q] = fma2(add2(l ? h2[j][q] : h1[j][q], f2(-mu[l])), mul2(f2(rs[l]), g[q]), b[q]);
          } else {
#pragma unroll
            for (int q = 0; q < H2; ++q) x[q] = mul2(l ? h2[j][q] : h1[j][q], mul2(f2(rs[l]), g[q]));
          }
          if (valid && colok[j]) stg<uint4>(static_cast<char*>(a.X[l]) + qX[j], pack2(x));
        }
        qX[j] += rank_h;
      }
      if (valid && threadIdx.x == 0) {
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          a.rstd[l][stat] = rs[l];
          if (LN && a.mean[l]) a.mean[l][stat] = mu[l];
        }
      }
      stat += a.T;
    }
  }
  if (dead && tid == 0) {
    atomicExch(status, 10u);
    // wait (bounded) for this CTA's copies still in flight before its shared memory goes away
    const long long issued = (k + NS) < total ? (k + NS) : total;
    for (long long q = k + 1; q < issued; ++q)
      for (uint32_t it = 0; it < (1u << 10); ++it)   // each poll sleeps up to the suspend hint: ~20 ms per stage at most
        if (mbar_try(bar0 + 8u * (uint32_t)(q % NS), (uint32_t)((q / NS) & 1))) break;
  }
}

BlockGeom block_geometry(const RowGeom& g, int h, int P, int S_hi, bool compact, size_t budget) {
  BlockGeom b{};
  const uint32_t rowH = (uint32_t)g.TY * h * ES, rowP = (uint32_t)g.TY * P * ES, rowS = (uint32_t)g.TY * S_hi * ES;
  uint32_t o = compact ? rowP : rowH;
  b.off_p[0] = o; o += rowP;
  b.off_p[1] = o; o += rowP;
  b.off_s[0] = o; o += rowS;
  b.off_s[1] = o; o += rowS;
  b.off_rs = o; if (compact) o += rowS;
  b.zero_off = o;
  b.stage_bytes = (o + 16u + 127u) & ~127u;
  size_t off = 8 * kMaxStages + 16;
  off = align_up(off, 16);
  b.red_off = (uint32_t)off; off += (size_t)2 * g.TY * 16 * 2 * sizeof(float);
  off = align_up(off, 128);
  b.ring_off = (uint32_t)off;
  int ns = budget > off ? (int)((budget - off) / b.stage_bytes) : 0;
  b.nstages = ns > kMaxStages ? kMaxStages : ns;
  b.smem = off + (size_t)b.nstages * b.stage_bytes;
  const RowsHooks hooks = rows_hooks();
  b.spin_cap = hooks.spin_cap;
  b.stall_bytes = hooks.stall ? 16u : 0u;
  return b;
}

template <bool LN, bool CL>
cudaError_t launch_t(const RowBlockArgs& a, const RowGeom& g, const BlockGeom& sg, int grid, int ngroups, unsigned int* status,
                     cudaStream_t st) {
  const dim3 block(g.TX, g.TY);
  const int threads = g.TX * g.TY;
  const bool few = a.flat || a.zgroups[0] > 1 || a.zgroups[1] > 1;
  cudaError_t e = cudaSuccess;
  LaunchScope scope(CAAT_K_ROWS_FORWARD, st);
#define CAAT_LAUNCH(CPT_, MAXT_)                                                                                     \
  do {                                                                                                               \
    auto k = few ? rows_forward_block<CPT_, LN, MAXT_, CL, true> : rows_forward_block<CPT_, LN, MAXT_, CL, false>;   \
    e = set_smem(k, sg.smem);                                                                                        \
    if (e == cudaSuccess) e = launch_pdl(k, dim3(grid), block, sg.smem, st, a, sg, ngroups, status);                 \
  } while (0)
  if (g.CPT == 3) CAAT_LAUNCH(3, 128);
  else if (g.CPT == 1) CAAT_LAUNCH(1, 256);
  else if constexpr (!LN) {
    if (threads <= 256) CAAT_LAUNCH(2, 256);
    else CAAT_LAUNCH(2, 512);
  } else {
    return cudaErrorInvalidValue;       // rows_block_usable leaves these to a pass per layer
  }
#undef CAAT_LAUNCH
  return e != cudaSuccess ? e : cudaGetLastError();
}

int block_ctas_per_sm(const RowGeom& g) {
  const int threads = g.TX * g.TY;
  return g.CPT == 3 ? 3 : threads <= 256 ? (g.CPT == 1 ? 3 : 2) : 1;
}

// Rows of 65 to 96 chunks (h = 768): a warp per token, three chunks per lane, four tokens per CTA (a block forward of
// 16384 tokens of 4 x 768: 228 us; one chunk per thread, two tokens per CTA: 259; four CTAs per SM with spills: 239).
RowGeom block_rows(int h) {
  RowGeom g = row_geometry(h, CAAT_BF16);
  const int chunks = h / V;
  if (chunks > 64 && chunks <= 96) { g.TX = 32; g.TY = 4; g.CPT = 3; }
  return g;
}

}  // namespace

// Rows of up to 8192 bf16 channels and a ring of at least three stages.  LayerNorm with two chunks per thread stays with a
// pass per layer: norm gains and biases of two layers do not fit the registers beside two streams (8192 tokens of
// 8 x 2048, whole step: 1567 us apart, 1577 in one pass; with spills avoided by half the threads 1551 both).
bool rows_block_usable(int h, int P, int S_hi, caat_dtype dtype, int compact, int norm) {
  if (dtype != CAAT_BF16) return false;
  const RowGeom g = block_rows(h);
  if (norm == 1 && g.CPT == 2) return false;
  if (g.CPT > 3 || (g.CPT == 1 && g.TX * g.TY > 256)) return false;
  return block_geometry(g, h, P, S_hi, compact != 0, kSmemPerSm / block_ctas_per_sm(g) - 1024).nstages >= 3;
}

cudaError_t launch_rows_forward_block(const RowBlockArgs& args, cudaStream_t st) {
  RowBlockArgs a = args;
  const RowGeom g = block_rows(a.h);
  const int per_sm = block_ctas_per_sm(g);
  const BlockGeom sg = block_geometry(g, a.h, a.P, a.S_hi, a.compact != 0, kSmemPerSm / per_sm - 1024);
  if (sg.nstages < 2) return cudaErrorInvalidConfiguration;
  const int ngroups = (a.T + g.TY - 1) / g.TY;
  int grid = sm_count() * per_sm;
  a.flat = flat_units(a.t, a.compact && (a.Rs == a.Hns[0] || a.Rs == a.Hns[1]), ngroups, grid);
  unsigned int* status = device_status_word();
  if (!status) return cudaErrorUnknown;
  if (a.compact) return a.norm == 1 ? launch_t<true, true>(a, g, sg, grid, ngroups, status, st) : launch_t<false, true>(a, g, sg, grid, ngroups, status, st);
  return a.norm == 1 ? launch_t<true, false>(a, g, sg, grid, ngroups, status, st) : launch_t<false, false>(a, g, sg, grid, ngroups, status, st);
}

}  // namespace caat
