// Prefill projections: Y[tok][f] = sum_k B[tok][k] W[f][k] for a whole
// prompt pass (hundreds to thousands of token rows), where the work is a
// dense contraction and the tensor pipe, not HBM, bounds it.
//
// The decode kernel (proj.cu) puts the weights on the MMA's M side and the
// few token rows on N, so each weight tile is read once per launch.  With a
// long pass that layout would re-read every weight once per 128 tokens of
// the pass; here the roles swap.  A CTA owns a tile of 128 token rows (the
// tcgen05 M dimension) by 256 output features (N):
//
//   A = activation rows, a bf16 pair hi + lo per value (two planes of the
//       activation buffer): two MMAs per K step, D += A_hi W + A_lo W, into
//       one accumulator -- the product carries the rounding of the weights
//       only, and the weight tile serves both halves of the pair;
//   B = 256 weight rows (two 128-row TMA boxes: q/k/v sections, or 128 gate
//       rows followed by the same 128 up rows).
//
// Per 64-wide K block a stage holds A_hi, A_lo (16 KB each) and B (32 KB):
// 64 KB for 2 x 128 x 256 x 64 multiply-adds.  Three stages fill the shared
// memory of one CTA per SM.  CTAs are persistent: CTA c takes tiles c,
// c + grid, ... (token tile fastest, so the CTAs running at one time share
// their weight tiles through L2 and HBM sees each weight about once per
// pass).  The 512 TMEM columns hold two 256-column accumulators, so the
// epilogue of one tile overlaps the MMAs of the next.
//
// Roles (320 threads): warp 8 issues the TMA loads, warp 9 the MMAs, warps
// 0-7 run the epilogue, one token row and half of the tile's columns per
// thread (TMEM lane = token row):
// the row's 1/rms of the RMSNorm feeding the projection (its gain is folded
// into the activation rows), then the fused epilogue of the decode kernel's
// flavours: RoPE + q rows + K/V cache rows (QKV), residual add + next
// norm's activation rows + per-128-feature sums of squares (O, down),
// SiLU(gate) * up (gate/up).  Every wait is bounded (flag, then wind down).
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace dvi {

namespace {

constexpr int kPfM = 128;                         // token rows per tile (MMA M)
constexpr int kPfN = 256;                         // output features per tile (MMA N)
constexpr int kPfStages = 3;
constexpr int kPfEpi = 8;                         // epilogue warps
constexpr int kPfThreads = 32 * (kPfEpi + 2);     // and the TMA and MMA warps
constexpr int kPfA = kPfM * 128;                  // one plane of the activation tile: 16 KB
constexpr int kPfB = kPfN * 128;                  // weight tile: 32 KB
constexpr int kPfStage = 2 * kPfA + kPfB;         // 64 KB
constexpr int kPfSmem = kPfStages * kPfStage + 1024 /*align*/ + 256 /*barriers, TMEM slot*/;
constexpr uint32_t kPfCols = 2 * kPfN;            // two accumulators

// Weight rows of half h (0, 1) of feature tile nt: which map, which row.
// QKV: the 256 features of the tile run over [q; k; v] (each section a
// multiple of 128 rows); gate/up: half 0 = gate rows, half 1 = the same up
// rows; other flavours: rows nt*256 + h*128 of the one weight.
__device__ __forceinline__ int pf_half_row(const ProjArgs& p, int nt, int h, int& map) {
  if (p.flavor == EPI_GATEUP) {
    map = h;
    return nt * kTileRows;
  }
  const int f = nt * kPfN + h * kTileRows;
  if (p.flavor == EPI_QKV) {
    if (f < p.rows_q) { map = 0; return f; }
    if (f < p.rows_q + p.rows_k) { map = 1; return f - p.rows_q; }
    map = 2;
    return f - p.rows_q - p.rows_k;   // past rows_v: zero fill
  }
  map = 0;
  return f;
}

// Sixteen f32 values as hi and lo bf16 planes (8 values per 16-byte store).
__device__ __forceinline__ void st_act16(__nv_bfloat16* dst, size_t plane, const float (&v)[16]) {
  uint32_t hi[8], lo[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) split_bf16x2(v[2 * e], v[2 * e + 1], hi[e], lo[e]);
  uint4* h4 = reinterpret_cast<uint4*>(dst);
  uint4* l4 = reinterpret_cast<uint4*>(dst + plane);
  h4[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  h4[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
  l4[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  l4[1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
}

// Sequence and cache position of pass row n.
__device__ __forceinline__ void pf_row_pos(const ProjArgs& p, int n, int& seq, int& pos) {
  seq = p.seq0 + n / p.rows_per_seq;
  pos = p.lens[seq] + p.pos_off + n % p.rows_per_seq;
}

// A row's values read ahead of the accumulator: the residual's first steps
// (O, down) or the rotations of the first 16 dims (QKV).
constexpr int kResAhead = 4;
using Ahead = float4[kResAhead][4];

// 1/rms of row n for the norm feeding the projection (1 without one); the
// sums are read eight at a time and added in tile order.
__device__ __forceinline__ float pf_rstd(const ProjArgs& p, int n) {
  if (!p.ss) return 1.f;
  float sq = 0.f;
  for (int q = 0; q < p.ss_tiles; q += 8) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      x[u] = q + u < p.ss_tiles ? __ldcg(p.ss + static_cast<size_t>(q + u) * p.ss_ld + n) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) sq += x[u];
  }
  return rsqrtf(sq / static_cast<float>(p.d_norm) + p.eps);
}

// QKV: RoPE (rotate-half pairs dim and dim + hd/2 of one head, both in the
// tile since sections and heads are 128-aligned), q rows in f32, k and v
// rows into the cache at the row's position.  16 dims at a time over every
// head of the tile, so a rotation is read once, one step ahead of its use.
__device__ __forceinline__ void pf_load_rope(const ProjArgs& p, int pos, int j, Ahead& ahead) {
  const float4* r = reinterpret_cast<const float4*>(p.rope + static_cast<size_t>(pos) * (p.head_dim >> 1) + j);
#pragma unroll
  for (int e = 0; e < 8; ++e) ahead[e >> 2][e & 3] = __ldg(r + e);
}
// Section (0 q, 1 k, 2 v) and head of the tile's feature column c0 (a
// multiple of the head dim); false past the last section.
__device__ __forceinline__ bool pf_section(const ProjArgs& p, int f0, int& sec, int& head) {
  int fl;
  if (f0 < p.rows_q) { sec = 0; fl = f0; }
  else if (f0 < p.rows_q + p.rows_k) { sec = 1; fl = f0 - p.rows_q; }
  else if (f0 < p.rows_q + p.rows_k + p.rows_v) { sec = 2; fl = f0 - p.rows_q - p.rows_k; }
  else return false;
  head = fl / p.head_dim;
  return true;
}
// Dims j .. j + 15 (a) and their rotation partners (b) of one head of row n.
__device__ __forceinline__ void pf_put_qkv(const ProjArgs& p, int sec, int head, int n, int seq, int pos, int j,
                                           float rstd, const float4 (&rot)[8], float (&a)[16], float (&b)[16]) {
  const int hd = p.head_dim, half = hd >> 1;
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    a[e] *= rstd;
    b[e] *= rstd;
  }
  if (sec < 2) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float rx = e & 1 ? rot[e >> 1].z : rot[e >> 1].x, ry = e & 1 ? rot[e >> 1].w : rot[e >> 1].y;
      // (fused as in the one-tile kernel: the two agree bit for bit)
      const float x1 = fmaf(a[e], rx, -(b[e] * ry));
      const float x2 = fmaf(b[e], rx, a[e] * ry);
      a[e] = x1;
      b[e] = x2;
    }
  }
  if (sec == 0) {
    float4* q0 = reinterpret_cast<float4*>(p.q_out + static_cast<size_t>(n) * p.ld_q + head * hd + j);
    float4* q1 = reinterpret_cast<float4*>(p.q_out + static_cast<size_t>(n) * p.ld_q + head * hd + half + j);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      q0[e] = make_float4(a[4 * e], a[4 * e + 1], a[4 * e + 2], a[4 * e + 3]);
      q1[e] = make_float4(b[4 * e], b[4 * e + 1], b[4 * e + 2], b[4 * e + 3]);
    }
  } else {
    __nv_bfloat16* c = static_cast<__nv_bfloat16*>(sec == 1 ? p.kc : p.vc) +
                       ((static_cast<size_t>(seq) * p.n_kv_heads + head) * p.max_len + pos) * hd;
    uint32_t pa[8], pb[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      pa[e] = pack_bf16x2(a[2 * e], a[2 * e + 1]);
      pb[e] = pack_bf16x2(b[2 * e], b[2 * e + 1]);
    }
    uint4* c0p = reinterpret_cast<uint4*>(c + j);
    uint4* c1p = reinterpret_cast<uint4*>(c + half + j);
    c0p[0] = make_uint4(pa[0], pa[1], pa[2], pa[3]);
    c0p[1] = make_uint4(pa[4], pa[5], pa[6], pa[7]);
    c1p[0] = make_uint4(pb[0], pb[1], pb[2], pb[3]);
    c1p[1] = make_uint4(pb[4], pb[5], pb[6], pb[7]);
  }
}
__device__ __forceinline__ void pf_epi_qkv(const ProjArgs& p, uint32_t acc, int nt, int h, int n, int seq, int pos,
                                           bool st, float rstd, Ahead& ahead) {
  const int hd = p.head_dim, half = hd >> 1;
  for (int j = 0; j < half; j += 16) {
    float4 rot[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) rot[e] = ahead[e >> 2][e & 3];
    if (st && j + 16 < half) pf_load_rope(p, pos, j + 16, ahead);
    for (int c0 = h * kTileRows; c0 < (h + 1) * kTileRows; c0 += hd) {
      int sec, head;
      if (!pf_section(p, nt * kPfN + c0, sec, head)) break;
      float a[16], b[16];
      tmem_ld16(acc + static_cast<uint32_t>(c0 + j), a);
      tmem_ld16(acc + static_cast<uint32_t>(c0 + half + j), b);
      if (st) pf_put_qkv(p, sec, head, n, seq, pos, j, rstd, rot, a, b);
    }
  }
}

// A row's sum of squares over 128 features, added in one order everywhere:
// four features at a time, then the tree of a warp that holds four a lane.
__device__ __forceinline__ float sq4(float4 x) { return fmaf(x.w, x.w, fmaf(x.z, x.z, fmaf(x.y, x.y, x.x * x.x))); }

// Features f .. f + 15 of row n: x (the residual) += v, x * g for the next
// projection; the sums of squares of each four in q4.
__device__ __forceinline__ void pf_put_resid(const ProjArgs& p, int n, int f, const float4 (&res)[4],
                                             const float (&v)[16], float (&q4)[4]) {
  float x[16];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    x[4 * e] = res[e].x + v[4 * e];
    x[4 * e + 1] = res[e].y + v[4 * e + 1];
    x[4 * e + 2] = res[e].z + v[4 * e + 2];
    x[4 * e + 3] = res[e].w + v[4 * e + 3];
  }
  float4* xp = reinterpret_cast<float4*>(p.x_res + static_cast<size_t>(n) * p.ld_res + f);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    xp[e] = make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
    q4[e] = sq4(make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]));
  }
  if (p.xg_out) {
    const float4* g4 = reinterpret_cast<const float4*>(p.g_next + f);
    float y[16];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 g = g4[e];
      y[4 * e] = x[4 * e] * g.x;
      y[4 * e + 1] = x[4 * e + 1] * g.y;
      y[4 * e + 2] = x[4 * e + 2] * g.z;
      y[4 * e + 3] = x[4 * e + 3] * g.w;
    }
    st_act16(static_cast<__nv_bfloat16*>(p.xg_out) + static_cast<size_t>(n) * p.ld_xg + f, p.xg_plane, y);
  }
}
// O and down: x += y, the next norm's activation rows x * g (hi/lo), and
// the sums of squares of the new x per 128 features (in feature order).
// The tile's residual row is read kResAhead steps of 16 features ahead of
// its use (a step's four loads take about a microsecond, with one thread a
// row and nothing else in flight: 16 of them in turn were a tail of 12 us).
__device__ __forceinline__ void pf_epi_resid(const ProjArgs& p, uint32_t acc, int nt, int h, int n, bool live,
                                             Ahead& ahead) {
  const int f0 = nt * kPfN + h * kTileRows;
  if (f0 >= p.n_out) return;
  float* xrow = p.x_res + static_cast<size_t>(live ? n : 0) * p.ld_res + f0;
  constexpr int kSteps = kTileRows / 16;
  float q[16];   // sums of four features: lanes l and l + 16 of the tree added
#pragma unroll
  for (int st = 0; st < kSteps; ++st) {
    float v[16];
    tmem_ld16(acc + static_cast<uint32_t>(h * kTileRows + st * 16), v);
    if (!live) continue;
    const int u = st % kResAhead;
    float4 res[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) res[e] = ahead[u][e];
    if (st + kResAhead < kSteps) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        ahead[u][e] = __ldcg(reinterpret_cast<const float4*>(xrow + (st + kResAhead) * 16) + e);
    }
    float q4[4];
    pf_put_resid(p, n, f0 + st * 16, res, v, q4);
#pragma unroll
    for (int e = 0; e < 4; ++e) q[4 * u + e] = st < kResAhead ? q4[e] : q[4 * u + e] + q4[e];
  }
  if (!live) return;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int e = 0; e < o; ++e) q[e] += q[e + o];
  p.ss_out[static_cast<size_t>(f0 / kTileRows) * p.ss_out_ld + n] = q[0];
}

// gate/up: columns [0, 128) are the gate rows, [128, 256) the up rows of the
// same 128 features; h = SiLU(gate) * up.
__device__ __forceinline__ void pf_put_gateup(const ProjArgs& p, int n, int f, float rstd, const float (&g)[16],
                                              const float (&u)[16]) {
  if (f >= p.n_out) return;
  float hv[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const float gt = g[e] * rstd;
    hv[e] = gt / (1.f + expf(-gt)) * (u[e] * rstd);
  }
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.h_out) + static_cast<size_t>(n) * p.ld_h + f;
  if (f + 16 <= p.n_out) {
    st_act16(dst, p.h_plane, hv);
  } else {
    for (int e = 0; f + e < p.n_out; ++e) Act<__nv_bfloat16>::st(dst + e, p.h_plane, hv[e]);
  }
}
__device__ __forceinline__ void pf_epi_gateup(const ProjArgs& p, uint32_t acc, int nt, int h, int n, bool live,
                                              float rstd) {
  for (int j = h * 64; j < h * 64 + 64; j += 16) {
    float g[16], u[16];
    tmem_ld16(acc + static_cast<uint32_t>(j), g);
    tmem_ld16(acc + static_cast<uint32_t>(kTileRows + j), u);
    if (live) pf_put_gateup(p, n, nt * kTileRows + j, rstd, g, u);
  }
}

}  // namespace

__global__ void __launch_bounds__(kPfThreads, 1)
    proj_pf_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mw0,
                   const __grid_constant__ CUtensorMap mw1, const __grid_constant__ CUtensorMap mw2,
                   const ProjArgs p, int n_mtiles, int n_ntiles) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* ring = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + kPfStages * kPfStage);
  uint64_t* empty = full + kPfStages;
  uint64_t* accf = empty + kPfStages;   // [2] accumulator b holds a finished tile
  uint64_t* acce = accf + 2;            // [2] accumulator b has been read
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(acce + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tiles = n_mtiles * n_ntiles;
  const int nkb = p.kb_total;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPfStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], kPfEpi);
    }
    mbar_fence_init();
  }
  if (warp == 0) tmem_alloc(tmem_holder, kPfCols);
  if (warp == kPfEpi && lane == 0) {
    tma_prefetch_desc(&ma);
    tma_prefetch_desc(&mw0);
    if (p.flavor == EPI_GATEUP || p.flavor == EPI_QKV) tma_prefetch_desc(&mw1);
    if (p.flavor == EPI_QKV) tma_prefetch_desc(&mw2);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == kPfEpi) {
    // ---------------- TMA producer
    if (lane == 0) {
      const uint64_t pol = 0ull;   // default L2 policy: weights are re-read by the other token tiles
      auto wmap = [&](int m) { return m == 0 ? &mw0 : (m == 1 ? &mw1 : &mw2); };
      auto load_w = [&](int nt, int kb, int s) {
        for (int h = 0; h < 2; ++h) {
          int m = 0;
          const int y = pf_half_row(p, nt, h, m);
          tma_load_2d(ring + s * kPfStage + 2 * kPfA + h * (kPfB / 2), wmap(m), kb * kKBlock, y, &full[s], pol);
        }
      };
      auto load_a = [&](int mt, int kb, int s) {
        tma_load_3d(ring + s * kPfStage, &ma, kb * kKBlock, p.act_row0 + mt * kPfM, 0, &full[s], 0ull);
        tma_load_3d(ring + s * kPfStage + kPfA, &ma, kb * kKBlock, p.act_row0 + mt * kPfM, 1, &full[s], 0ull);
      };
      // The first tile's first weight blocks do not depend on earlier kernels.
      int it = 0, issued = 0;
      bool ok = true;
      const int t0 = blockIdx.x;
      const int pre = t0 < n_tiles ? min(kPfStages, nkb) : 0;
      for (int i = 0; i < pre; ++i) {
        mbar_arrive_expect_tx(&full[i], kPfStage);
        load_w(t0 / n_mtiles, i, i);
      }
      griddep_wait();
      for (int i = 0; i < pre; ++i) load_a(t0 % n_mtiles, i, i);
      it = issued = pre;
      for (int t = t0; t < n_tiles && ok; t += gridDim.x) {
        const int mt = t % n_mtiles, nt = t / n_mtiles;
        for (int kb = (t == t0 ? pre : 0); kb < nkb; ++kb, ++it) {
          const int s = it % kPfStages;
          if (!mbar_wait(&empty[s], ((it / kPfStages) & 1) ^ 1, p.status)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[s], kPfStage);
          load_w(nt, kb, s);
          load_a(mt, kb, s);
          issued = it + 1;
        }
      }
      // every issued copy has landed before the CTA moves on
      for (int i = max(0, issued - kPfStages); i < issued; ++i)
        mbar_wait(&full[i % kPfStages], (i / kPfStages) & 1, p.status);
    }
    __syncwarp();
  } else if (warp == kPfEpi + 1) {
    // ---------------- MMA issuer: D += A_hi W + A_lo W per K step
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_m128(kPfN);
      int it = 0, j = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++j) {
        const int b = j & 1;
        if (!mbar_wait(&acce[b], ((j >> 1) & 1) ^ 1, p.status)) break;
        tc_fence_after();
        const uint32_t d = tmem + static_cast<uint32_t>(b * kPfN);
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % kPfStages;
          if (!mbar_wait(&full[s], (it / kPfStages) & 1, p.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t ahi = smem_u32(ring + s * kPfStage);
          const uint32_t alo = ahi + kPfA;
          const uint32_t bw = ahi + 2 * kPfA;
#pragma unroll
          for (int kk = 0; kk < kKBlock / 16; ++kk) {
            const uint64_t bd = smem_desc_sw128(bw + kk * 32);
            tc_mma_bf16(d, smem_desc_sw128(ahi + kk * 32), bd, idesc, (kb | kk) != 0);
            tc_mma_bf16(d, smem_desc_sw128(alo + kk * 32), bd, idesc, 1u);
          }
          tc_commit(&empty[s]);
        }
        // The next kernel's CTAs may take their places once every CTA's last
        // tile is issued: its epilogue covers their launch.  From the start
        // they would hold SMs (this kernel's 200 KB each) while they wait.
        if (t + static_cast<int>(gridDim.x) >= n_tiles) griddep_launch();
        // also after a failed wait, so the epilogue's wait ends and every
        // MMA issued has completed before the TMEM is freed
        tc_commit(&accf[b]);
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: warp w reads TMEM lanes (token rows) 32 (w mod 4) ..,
    // half w / 4 of the tile's columns
    griddep_wait();
    const int row = (warp & 3) * 32 + lane, h = warp >> 2;
    int j = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++j) {
      const int b = j & 1;
      const int mt = t % n_mtiles, nt = t / n_mtiles;
      const int n = mt * kPfM + row;
      const bool live = n < p.M;
      // the row's 1/rms (before the wait: it reads only earlier kernels' output)
      const float rstd = live ? pf_rstd(p, n) : 1.f;
      // and what its epilogue reads first: the residual row's first steps (nt * 256
      // + 64 <= n_out: n_out is a multiple of 128), or the row's first rotations
      Ahead ahead;
      int seq = 0, pos = 0;
      bool st = live;
      if (p.flavor == EPI_QKV && live) {
        pf_row_pos(p, n, seq, pos);
        st = pos >= 0 && pos < p.max_len;
        if (!st) flag_status(p.status, DVI_DEV_KV_FULL);
        else pf_load_rope(p, pos, 0, ahead);
      }
      const int f0 = nt * kPfN + h * kTileRows;
      if (p.flavor == EPI_RESID && live && f0 < p.n_out) {
        const float4* x4 = reinterpret_cast<const float4*>(p.x_res + static_cast<size_t>(n) * p.ld_res + f0);
#pragma unroll
        for (int u = 0; u < kResAhead; ++u)
#pragma unroll
          for (int e = 0; e < 4; ++e) ahead[u][e] = __ldcg(x4 + 4 * u + e);
      }
      if (!mbar_wait(&accf[b], (j >> 1) & 1, p.status)) break;
      tc_fence_after();
      const uint32_t acc = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(b * kPfN);
      if (p.flavor == EPI_QKV) pf_epi_qkv(p, acc, nt, h, n, seq, pos, st, rstd, ahead);
      else if (p.flavor == EPI_GATEUP) pf_epi_gateup(p, acc, nt, h, n, live, rstd);
      else pf_epi_resid(p, acc, nt, h, n, live, ahead);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[b]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kPfCols);
  }
}


// ------------------------------------------------------------------ one tile per CTA
// Passes whose tiles fit the SMs at once.  A CTA (or, for short prompts, a
// cluster of S CTAs that split the tile's K) computes one tile with the stages
// and MMAs of the kernel above; then the ring is free, so the tile goes
// through shared memory, [128 rows][256] f32, and the epilogue runs with a
// warp per row and four columns a lane: every global access is a whole
// 128- to 512-byte run of a row, where a thread per TMEM lane touches 32 rows
// per instruction.  Split over K, rank r of the cluster finishes the tile's rows
// [r R, (r + 1) R), R = 128 / S, each value summed over the ranks in rank
// order through distributed shared memory.  An unsplit tile has the same
// result in both kernels.
//
// Eighteen warps: 0-15 the epilogue (four per TMEM lane quarter), 16 the TMA
// loads, 17 the MMAs; the epilogue is latency-bound and its time falls with
// its warps (4, 8, 16: the unsplit O projection of the 1B shape at 512 tokens
// 35, 28.6, 26 us, of which 17.6 are MMAs).  Per launch at the 1B shape, 23 /
// 301 / 512 tokens, against the kernel above with four epilogue warps: QKV 23 /
// 27 / 27 -> 11 / 17 / 26 us, O 30 / 37 / 37 -> 10 / 12 / 17, down 61 / 67 / 68
// -> 14 / 21 / 33; 7B shape at 1024 tokens: O 64 -> 47, down 123 -> 108 us.
constexpr int kPsMaxSplits = 8;
constexpr int kPsEpi = 16;                 // epilogue warps
constexpr int kPsThreads = 32 * (kPsEpi + 2);

namespace {
constexpr int kPsLd = kPfN + 4;                     // floats per row: 16-byte accesses of 8 rows meet no bank twice
constexpr int kPsPart = kPfM * kPsLd * 4;
static_assert(kPsPart + 2 * kPfM * 4 <= kPfStages * kPfStage, "the tile and its rows' scalars lie in the ring");

__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
// Columns col .. col + 3 of tile row `row`, summed over the ranks in order.
template <int S>
__device__ __forceinline__ float4 ps_gather(uint32_t part, int row, int col) {
  const uint32_t at = part + static_cast<uint32_t>((row * kPsLd + col) * 4);
  float4 t[S];
#pragma unroll
  for (int r = 0; r < S; ++r) t[r] = ld_cluster_f32x4(S == 1 ? at : mapa_shared(at, r));
#pragma unroll
  for (int r = 1; r < S; ++r) {
    t[0].x += t[r].x;
    t[0].y += t[r].y;
    t[0].z += t[r].z;
    t[0].w += t[r].w;
  }
  return t[0];
}
__device__ __forceinline__ void st_act4(__nv_bfloat16* dst, size_t plane, float4 v) {
  uint2 hi, lo;
  split_bf16x2(v.x, v.y, hi.x, lo.x);
  split_bf16x2(v.z, v.w, hi.y, lo.y);
  *reinterpret_cast<uint2*>(dst) = hi;
  *reinterpret_cast<uint2*>(dst + plane) = lo;
}
}  // namespace

template <int S>
__global__ void __launch_bounds__(kPsThreads, 1)
    proj_ps_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mw0,
                   const __grid_constant__ CUtensorMap mw1, const __grid_constant__ CUtensorMap mw2,
                   const ProjArgs p, int n_mtiles) {
  constexpr int R = kPfM / S;                                   // rows this rank finishes
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* ring = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + kPfStages * kPfStage);
  uint64_t* empty = full + kPfStages;
  uint64_t* done = empty + kPfStages;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(done + 1);
  float* part = reinterpret_cast<float*>(ring);                 // [128][kPsLd] once the MMAs are done
  float* rstd_s = reinterpret_cast<float*>(ring + kPsPart);     // [R] 1/rms, then
  int* pos_s = reinterpret_cast<int*>(rstd_s + kPfM);           // [R] position of each row (-1: past the cache)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x / S, split = blockIdx.x % S;
  const int mt = tile % n_mtiles, nt = tile / n_mtiles;
  const int kb0 = split * p.kb_per_split;
  const int nkb = max(0, min(p.kb_per_split, p.kb_total - kb0));

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPfStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    mbar_fence_init();
  }
  if (warp == 0) tmem_alloc(tmem_holder, kPfN);
  if (warp == kPsEpi && lane == 0) {
    tma_prefetch_desc(&ma);
    tma_prefetch_desc(&mw0);
    if (p.flavor == EPI_GATEUP || p.flavor == EPI_QKV) tma_prefetch_desc(&mw1);
    if (p.flavor == EPI_QKV) tma_prefetch_desc(&mw2);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  const int n0 = mt * kPfM + split * R;                         // first pass row of the rank
  bool ok = true;

  if (warp == kPsEpi) {
    // ---------------- TMA producer
    if (lane == 0) {
      auto wmap = [&](int m) { return m == 0 ? &mw0 : (m == 1 ? &mw1 : &mw2); };
      auto load_w = [&](int i, int s) {
        for (int h = 0; h < 2; ++h) {
          int m = 0;
          const int y = pf_half_row(p, nt, h, m);
          tma_load_2d(ring + s * kPfStage + 2 * kPfA + h * (kPfB / 2), wmap(m), (kb0 + i) * kKBlock, y, &full[s], 0ull);
        }
      };
      auto load_a = [&](int i, int s) {
        const int x = (kb0 + i) * kKBlock, y = p.act_row0 + mt * kPfM;
        tma_load_3d(ring + s * kPfStage, &ma, x, y, 0, &full[s], 0ull);
        tma_load_3d(ring + s * kPfStage + kPfA, &ma, x, y, 1, &full[s], 0ull);
      };
      const int pre = min(kPfStages, nkb);
      for (int i = 0; i < pre; ++i) {
        mbar_arrive_expect_tx(&full[i], kPfStage);
        load_w(i, i);
      }
      griddep_wait();
      for (int i = 0; i < pre; ++i) load_a(i, i);
      int issued = pre;
      for (int i = pre; i < nkb; ++i) {
        const int s = i % kPfStages;
        if (!mbar_wait(&empty[s], ((i / kPfStages) & 1) ^ 1, p.status)) break;
        mbar_arrive_expect_tx(&full[s], kPfStage);
        load_w(i, s);
        load_a(i, s);
        issued = i + 1;
      }
      // every issued copy has landed before the CTA moves on
      for (int i = max(0, issued - kPfStages); i < issued; ++i)
        mbar_wait(&full[i % kPfStages], (i / kPfStages) & 1, p.status);
    }
    __syncwarp();
  } else if (warp == kPsEpi + 1) {
    // ---------------- MMA issuer: D += A_hi W + A_lo W per K step
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_m128(kPfN);
      for (int i = 0; i < nkb; ++i) {
        const int s = i % kPfStages;
        if (!mbar_wait(&full[s], (i / kPfStages) & 1, p.status)) break;
        tc_fence_after();
        const uint32_t ahi = smem_u32(ring + s * kPfStage);
        const uint32_t alo = ahi + kPfA;
        const uint32_t bw = ahi + 2 * kPfA;
#pragma unroll
        for (int kk = 0; kk < kKBlock / 16; ++kk) {
          const uint64_t bd = smem_desc_sw128(bw + kk * 32);
          tc_mma_bf16(tmem, smem_desc_sw128(ahi + kk * 32), bd, idesc, (i | kk) != 0);
          tc_mma_bf16(tmem, smem_desc_sw128(alo + kk * 32), bd, idesc, 1u);
        }
        tc_commit(&empty[s]);
      }
      griddep_launch();   // the next kernel's launch overlaps the epilogue
      tc_commit(done);
    }
    __syncwarp();
  } else {
    // ---------------- the rows' 1/rms and positions, then the tile into shared memory
    griddep_wait();
    const int tid = threadIdx.x;
    float rstd = 1.f;
    int pos = -1;
    if (tid < R && n0 + tid < p.M) {
      rstd = pf_rstd(p, n0 + tid);
      if (p.flavor == EPI_QKV) {
        int seq;
        pf_row_pos(p, n0 + tid, seq, pos);
        if (pos < 0 || pos >= p.max_len) {
          pos = -1;
          flag_status(p.status, DVI_DEV_KV_FULL);
        }
      }
    }
    ok = mbar_wait(done, 0, p.status);
    tc_fence_after();
    if (tid < R) {
      rstd_s[tid] = rstd;
      pos_s[tid] = pos;
    }
    const uint32_t acc = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    float4* row4 = reinterpret_cast<float4*>(part + (tid & (kPfM - 1)) * kPsLd);
    constexpr int kCols = kPfN / (kPsEpi / 4);   // of a warp
    const int col0 = (warp >> 2) * kCols;
#pragma unroll 1
    for (int c = col0; c < col0 + kCols; c += 32) {
      float v[32];
      tmem_ld32_async(acc + static_cast<uint32_t>(c), v);
      tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 8; ++e)   // a rank without K blocks (nkb 0) adds zeros
        row4[c / 4 + e] = nkb > 0 ? make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3])
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    tc_fence_before();
    named_bar(1, 32 * kPsEpi);
    if (warp == 0) {
      tc_fence_after();
      tmem_dealloc(tmem, kPfN);
    }
  }
  if constexpr (S > 1) {
    cluster_arrive_release();
    cluster_wait_acquire();
  }
  if (warp < kPsEpi && ok) {
    // ---------------- epilogue: row i of the rank by warp i mod kPsEpi
    const uint32_t mine = smem_u32(part);
    const int rows = min(R, p.M - n0);
    if (p.flavor == EPI_QKV) {
      const int hd = p.head_dim, half = hd >> 1;
      const int dim = (4 * lane) & (hd - 1);   // the lane's first dim, in either half of the tile
      const float sg = dim < half ? -1.f : 1.f;
      constexpr int U = 4;                     // rows whose rotations are in flight
      for (int i0 = warp; i0 < rows; i0 += kPsEpi * U) {
        float4 ra[U], rb[U];                   // (cos, sin) of the four dims
        int pos[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          pos[u] = i0 + kPsEpi * u < rows ? pos_s[i0 + kPsEpi * u] : -1;
          const float4* r4 = reinterpret_cast<const float4*>(p.rope + static_cast<size_t>(max(pos[u], 0)) * half +
                                                             (dim & (half - 1)));
          ra[u] = __ldg(r4);
          rb[u] = __ldg(r4 + 1);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int col = h * kTileRows + 4 * lane;
          int sec, head;
          if (!pf_section(p, nt * kPfN + col - dim, sec, head)) continue;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int i = i0 + kPsEpi * u;
            if (i >= rows) break;
            const int n = n0 + i;
            const float rstd = rstd_s[i];
            float4 v = ps_gather<S>(mine, split * R + i, col);
            v.x *= rstd;
            v.y *= rstd;
            v.z *= rstd;
            v.w *= rstd;
            if (sec < 2) {   // (uniform: a section is a multiple of 128 rows)
              // the partner dims (dim +- hd / 2) are hd / 8 lanes away
              float4 w;
              w.x = __shfl_xor_sync(0xffffffffu, v.x, hd / 8);
              w.y = __shfl_xor_sync(0xffffffffu, v.y, hd / 8);
              w.z = __shfl_xor_sync(0xffffffffu, v.z, hd / 8);
              w.w = __shfl_xor_sync(0xffffffffu, v.w, hd / 8);
              v.x = fmaf(v.x, ra[u].x, sg * (w.x * ra[u].y));
              v.y = fmaf(v.y, ra[u].z, sg * (w.y * ra[u].w));
              v.z = fmaf(v.z, rb[u].x, sg * (w.z * rb[u].y));
              v.w = fmaf(v.w, rb[u].z, sg * (w.w * rb[u].w));
            }
            if (pos[u] < 0) continue;
            if (sec == 0) {
              *reinterpret_cast<float4*>(p.q_out + static_cast<size_t>(n) * p.ld_q + head * hd + dim) = v;
            } else {
              const int seq = p.seq0 + n / p.rows_per_seq;
              __nv_bfloat16* c = static_cast<__nv_bfloat16*>(sec == 1 ? p.kc : p.vc) +
                                 ((static_cast<size_t>(seq) * p.n_kv_heads + head) * p.max_len + pos[u]) * hd + dim;
              *reinterpret_cast<uint2*>(c) = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
            }
          }
        }
      }
    } else if (p.flavor == EPI_GATEUP) {
      const int f = nt * kTileRows + 4 * lane;
#pragma unroll 2
      for (int i = warp; i < rows; i += kPsEpi) {
        const float rstd = rstd_s[i];
        const float4 g = ps_gather<S>(mine, split * R + i, 4 * lane);
        const float4 u = ps_gather<S>(mine, split * R + i, kTileRows + 4 * lane);
        auto swiglu = [rstd](float a, float b) {
          const float t = a * rstd;
          return t / (1.f + expf(-t)) * (b * rstd);
        };
        if (f < p.n_out)   // n_out is a multiple of 8: four columns are in or out together
          st_act4(static_cast<__nv_bfloat16*>(p.h_out) + static_cast<size_t>(n0 + i) * p.ld_h + f, p.h_plane,
                  make_float4(swiglu(g.x, u.x), swiglu(g.y, u.y), swiglu(g.z, u.z), swiglu(g.w, u.w)));
      }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int f = nt * kPfN + h * kTileRows + 4 * lane;
        if (nt * kPfN + h * kTileRows >= p.n_out) break;
        const float4 g = __ldg(reinterpret_cast<const float4*>(p.g_next + f));
        constexpr int U = S >= 4 ? 2 : 4;   // rows in flight
        for (int i0 = warp; i0 < rows; i0 += kPsEpi * U) {
          float4 x[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (i0 + kPsEpi * u < rows)
              x[u] = __ldcg(reinterpret_cast<const float4*>(p.x_res + static_cast<size_t>(n0 + i0 + kPsEpi * u) * p.ld_res + f));
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int i = i0 + kPsEpi * u, n = n0 + i;
            if (i >= rows) break;
            const float4 v = ps_gather<S>(mine, split * R + i, h * kTileRows + 4 * lane);
            const float4 y = make_float4(x[u].x + v.x, x[u].y + v.y, x[u].z + v.z, x[u].w + v.w);
            *reinterpret_cast<float4*>(p.x_res + static_cast<size_t>(n) * p.ld_res + f) = y;
            if (p.xg_out)
              st_act4(static_cast<__nv_bfloat16*>(p.xg_out) + static_cast<size_t>(n) * p.ld_xg + f, p.xg_plane,
                      make_float4(y.x * g.x, y.y * g.y, y.z * g.z, y.w * g.w));
            const float ssq = warp_sum(sq4(y));
            if (lane == 0) p.ss_out[static_cast<size_t>(nt * 2 + h) * p.ss_out_ld + n] = ssq;
          }
        }
      }
    }
  }
  if constexpr (S > 1) {
    // every rank keeps its shared memory until all have read it
    cluster_arrive_release();
    cluster_wait_acquire();
  }
}

// Feature tiles of a projection.
static int pf_ntiles(const ProjArgs& a) {
  if (a.flavor == EPI_QKV) return (a.rows_q + a.rows_k + a.rows_v + kPfN - 1) / kPfN;
  if (a.flavor == EPI_GATEUP) return (a.n_out + kTileRows - 1) / kTileRows;
  if (a.flavor == EPI_RESID) return (a.n_out + kPfN - 1) / kPfN;
  return 0;
}

// K ranges of a tile's cluster for a prompt of n_tokens: the most of 8, 4, 2
// that fill at most two thirds of the SMs with at least four K blocks each
// (four take 2 us of MMAs, the exchange about as long); 1 = unsplit.  With
// the SMs filled further (136 of 152) a 512-token prompt of the 1B shape alone
// took 2.2 ms instead of 2.7 but 1.62 instead of 1.45 with two other streams
// beside it; with at most half, eight prompts of 23 to 301 tokens 13.9 ms
// instead of 12.5 alone.  A function of the prompt and the weight only, never
// of the pass's rows, so the chunk size does not change a row's result.
static int pf_splits(const ProjArgs& a, int n_tokens, int n_sms) {
  const long tiles = static_cast<long>((n_tokens + kPfM - 1) / kPfM) * pf_ntiles(a);
  const int nkb = (a.K + kKBlock - 1) / kKBlock;
  for (int s = kPsMaxSplits; s > 1; s /= 2)
    if (tiles * s <= 2 * n_sms / 3 && nkb / s >= 4) return s;
  return 1;
}

template <int S>
static cudaError_t launch_ps(const ProjArgs& a, const PfMaps& m, int n_mtiles, int n_tiles, cudaStream_t s) {
  static PerDevice attr;
  attr.once([] { cudaFuncSetAttribute(proj_ps_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPfSmem); });
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_tiles * S);
  cfg.blockDim = dim3(kPsThreads);
  cfg.dynamicSmemBytes = kPfSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = S;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = S > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, proj_ps_kernel<S>, m.act, m.w0, m.w1, m.w2, a, n_mtiles);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_proj_pf(const ProjArgs& a0, const PfMaps& m, int n_tokens, int n_sms, cudaStream_t s) {
  static PerDevice attr;
  attr.once([] {
    cudaFuncSetAttribute(proj_pf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPfSmem);
  });
  ProjArgs a = a0;
  a.kb_total = (a.K + kKBlock - 1) / kKBlock;
  const int n_ntiles = pf_ntiles(a);
  if (n_ntiles == 0) return cudaErrorInvalidValue;
  const int n_mtiles = (a.M + kPfM - 1) / kPfM;
  const int n_tiles = n_mtiles * n_ntiles;
  a.n_splits = pf_splits(a, n_tokens, n_sms);
  a.kb_per_split = (a.kb_total + a.n_splits - 1) / a.n_splits;
  switch (a.n_splits) {
    case 8: return launch_ps<8>(a, m, n_mtiles, n_tiles, s);
    case 4: return launch_ps<4>(a, m, n_mtiles, n_tiles, s);
    case 2: return launch_ps<2>(a, m, n_mtiles, n_tiles, s);
  }
  if (n_tiles <= n_sms) return launch_ps<1>(a, m, n_mtiles, n_tiles, s);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::max(1, std::min(n_tiles, n_sms)));
  cfg.blockDim = dim3(kPfThreads);
  cfg.dynamicSmemBytes = kPfSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, proj_pf_kernel, m.act, m.w0, m.w1, m.w2, a, n_mtiles, n_ntiles);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace dvi
