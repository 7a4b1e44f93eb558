// Prompt-pass attention (bf16, GQA groups of at most 8): block-causal softmax
// attention of many query rows over the KV cache on tcgen05 / TMEM.
//
// A CTA owns one KV head and one or two tiles of 128 query vectors (tile row
// v: pass row v / G, query head v % G of the KV head's G) and walks the
// 128-position chunks of the cache that its rows can see.  Both tiles share
// every chunk, so the cache crosses L2 once per 256 query vectors.  Per chunk
// and tile:
//   S = Q K^T      M = 128 vectors, N = 128 positions, K = hd; the query
//                  (pre-scaled by log2(e) / sqrt(hd)) as a bf16 pair hi + lo:
//                  two chains of MMAs into one TMEM accumulator;
//   softmax        one thread per vector (TMEM lane): the causal limit, the
//                  running maximum, p = 2^(s - m), the sum, and p as a bf16
//                  pair hi + lo back into the TMEM columns of S;
//   O += P V       A = P from TMEM, B = the V chunk as it lies in the cache
//                  (positions are the K index, so B is MN-major).
// The queries, probabilities and sums carry the rounding of f32 / bf16 pairs
// only, as in the decode kernels.  The accumulator is rescaled only when a
// row's maximum has grown by more than 2^kLazy since the reference it uses
// (a multiplication by 1 for the other rows of the warp): p stays below
// 2^kLazy and the final division by the sum removes the reference again.  A
// row's result is its own softmax over chunks 0 .. p / 128 in order, whatever
// rows share its CTA or its pass.
//
// Roles (384 threads): warps 0-3 and 4-7 are the softmax of tile 0 and 1 (one
// TMEM lane quarter per warp), warp 8 issues the TMA loads, warp 9 the MMAs
// (warps 10-11 complete the warpgroup whose registers the softmax warps
// take).  While one tile is in its softmax the tensor pipe works on the
// other.  Shared memory: the queries (hi and lo of both tiles, 128 KB at hd
// 128) and three 128-position K or V stages of 32 KB.
//
// What bounds it: the MMAs at M = N = 128.  At hd 128 a chunk's S takes 1280
// cycles and its P V 1700 (16 MMAs of 128 x 128 x 16 each, 80 to 105 cycles
// apiece; 64, so 1024 for the 16, at the pipe's nominal rate), a softmax 1700.
// Two tiles take 6200 cycles a chunk: an MMA is in flight in 96 % of them, but
// by the nominal rate the pipe is two thirds busy (4096 cycles).  1024 rows
// over 32 heads: 38.5 us (62 on warp MMAs, 64 vectors per CTA and chunks of 64
// positions), over a cached prefix of 8192 positions on average 230 us (834).
//
// Every wait is bounded (flag, then wind down).
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace dvi {

namespace {

constexpr int kAfThreads = 384;
constexpr int kAfSoftRegs = 224, kAfOtherRegs = 56;
static_assert(256 * kAfSoftRegs + 128 * kAfOtherRegs <= kAfThreads * 168, "the launch's registers");
constexpr int kAfQ = 128;       // query vectors per tile
constexpr int kAfPos = 128;     // positions per chunk
constexpr int kAfStages = 3;
constexpr float kLazy = 8.f;    // growth of a row's maximum (base 2) that rescales the accumulator
constexpr float kAfLog2e = 1.4426950408889634f;

template <int HD>
struct AfSmem {
  static constexpr int kBoxes = HD / 64;                  // 64-dim boxes per row
  static constexpr int kBox = kAfPos * 128;               // 128 rows x 64 dims: 16 KB
  static constexpr int kStage = kBoxes * kBox;            // one chunk's K or V
  static constexpr int kQ = 2 * kBoxes * kBox;            // hi boxes, then lo boxes, of one tile
  static constexpr int kRing = 2 * kQ;
  static constexpr int kBars = kRing + kAfStages * kStage;
  static constexpr int kTotal = kBars + 256 + 1024 /*align*/;
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace

template <int HD>
__global__ void __launch_bounds__(kAfThreads, 1)
    attn_pf_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                   const __grid_constant__ AttnArgs a, int n_tiles) {
  using SM = AfSmem<HD>;
  extern __shared__ uint8_t dsm_raw[];
  const uint32_t raw = smem_u32(dsm_raw);
  uint8_t* sm = dsm_raw + (((raw + 1023u) & ~1023u) - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + SM::kBars);
  uint64_t* empty = full + kAfStages;
  uint64_t* q_ready = empty + kAfStages;   // the queries are in shared memory
  uint64_t* s_full = q_ready + 1;          // [2] the tile's scores are in TMEM
  uint64_t* p_ready = s_full + 2;          // [2] its probabilities are
  uint64_t* pv_done = p_ready + 2;         // [2] its accumulator holds the chunk
  uint64_t* fin = pv_done + 2;             // every MMA issued is done
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(fin + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = a.n_heads / a.n_kv_heads;
  const int RT = kAfQ / G;                             // pass rows per tile
  const int g = blockIdx.x;
  const int grp = static_cast<int>(gridDim.y) - 1 - static_cast<int>(blockIdx.y);   // longest prefixes first
  const int sl = blockIdx.z, seq = a.seq0 + sl;
  const int i0 = grp * n_tiles * RT;                   // first pass row

  if (tid == 0) {
    for (int s = 0; s < kAfStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(q_ready, 8);
    for (int t = 0; t < 2; ++t) {
      mbar_init(&s_full[t], 1);
      mbar_init(&p_ready[t], 4);
      mbar_init(&pv_done[t], 1);
    }
    mbar_init(fin, 1);
    mbar_fence_init();
  }
  if (warp == 9) tmem_alloc(tmem_holder, 512);
  if (warp == 8 && lane == 0) {
    tma_prefetch_desc(&mk);
    tma_prefetch_desc(&mv);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  // S / P of tile t: columns 128 t ..; O: 256 + 128 t ..
  griddep_wait();
  const int base = a.lens[seq] + a.pos_off;            // position of pass row 0
  // chunks of tile t (0: the tile has no row)
  auto chunks = [&](int t) {
    const int r0 = i0 + t * RT, nr = t < n_tiles ? min(RT, a.rows_per_seq - r0) : 0;
    if (nr <= 0) return 0;
    return max(0, min(base + r0 + nr - 1, a.max_len - 1)) / kAfPos + 1;
  };
  const int nch0 = chunks(0), nch1 = chunks(1);
  const int nch = max(nch0, nch1);
  // Rows of the last chunk from here on lie past every position that the CTA's
  // rows see: an earlier request's, another head's, or never written.  The
  // probability 0 of such a row leaves NaN in O if its value is not finite, so
  // the values there are cleared in shared memory.
  const int past = min(base + min(i0 + n_tiles * RT, a.rows_per_seq) - 1, a.max_len - 1) % kAfPos + 1;

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kAfOtherRegs));
    if (warp == 8 && lane == 0) {
      // ---------------- TMA producer: K chunk, V chunk, K chunk, ...
      const int row0 = static_cast<int>(a.kv_row0 + (static_cast<long long>(seq) * a.n_kv_heads + g) * a.max_len);
      int issued = 0;
      for (int it = 0; it < 2 * nch; ++it) {
        const int s = it % kAfStages;
        if (!mbar_wait(&empty[s], ((it / kAfStages) & 1) ^ 1, a.status)) break;
        const CUtensorMap* m = it & 1 ? &mv : &mk;
        uint8_t* dst = sm + SM::kRing + s * SM::kStage;
        const int y = row0 + (it >> 1) * kAfPos;
        mbar_arrive_expect_tx(&full[s], SM::kStage);
        for (int b = 0; b < SM::kBoxes; ++b)
          for (int h = 0; h < 2; ++h)
            tma_load_2d(dst + b * SM::kBox + h * (SM::kBox / 2), m, b * 64, y + 64 * h, &full[s], 0ull);
        issued = it + 1;
      }
      // every issued copy has landed before the CTA moves on
      for (int it = max(0, issued - kAfStages); it < issued; ++it)
        mbar_wait(&full[it % kAfStages], (it / kAfStages) & 1, a.status);
    } else if (warp == 9 && lane == 0) {
      // ---------------- MMA issuer
      const uint32_t id_s = idesc_bf16_m128(kAfPos);
      const uint32_t id_o = idesc_bf16_m128(HD) | kIdescBMn;
      auto scores = [&](int t, int s) {
        const uint32_t q = smem_u32(sm + t * SM::kQ), k = smem_u32(sm + SM::kRing + s * SM::kStage);
#pragma unroll
        for (int half = 0; half < 2; ++half)   // hi, then lo
#pragma unroll
          for (int kk = 0; kk < HD / 16; ++kk) {
            const uint32_t off = (kk / 4) * SM::kBox + (kk % 4) * 32;
            tc_mma_bf16(tmem + 128u * t, smem_desc_sw128(q + half * (SM::kQ / 2) + off), smem_desc_sw128(k + off),
                        id_s, (half | kk) != 0);
          }
        tc_commit(&s_full[t]);
      };
      auto values = [&](int t, int s, bool first) {
        const uint32_t v = smem_u32(sm + SM::kRing + s * SM::kStage);
#pragma unroll
        for (int half = 0; half < 2; ++half)
#pragma unroll
          for (int kk = 0; kk < kAfPos / 16; ++kk)
            tc_mma_bf16_ta(tmem + 256u + 128u * t, tmem + 128u * t + 64u * half + 8u * kk,
                           smem_desc_sw128_mn(v + kk * 2048, SM::kBox), id_o, !first || (half | kk) != 0);
        tc_commit(&pv_done[t]);
      };
      auto full_wait = [&](int it) { return mbar_wait(&full[it % kAfStages], (it / kAfStages) & 1, a.status); };
      bool ok = nch > 0 && mbar_wait(q_ready, 0, a.status) && full_wait(0);
      if (ok) {
        tc_fence_after();
        if (nch0 > 0) scores(0, 0);
        if (nch1 > 0) scores(1, 0);
        tc_commit(&empty[0]);
      }
      // P V of both tiles, then both next S: the pipe works on one tile while
      // the other is in its softmax (letting whichever tile is ready go first
      // put both softmaxes side by side: 261 us against 228)
      for (int i = 0; i < nch && ok; ++i) {
        const int iv = 2 * i + 1, sv = iv % kAfStages;
        ok = full_wait(iv);
        for (int t = 0; t < 2 && ok; ++t) {
          if (i >= (t ? nch1 : nch0)) continue;
          ok = mbar_wait(&p_ready[t], i & 1, a.status);
          if (!ok) break;
          tc_fence_after();
          values(t, sv, i == 0);
        }
        if (!ok) break;
        tc_commit(&empty[sv]);
        // the next kernel's CTAs take their places while the outputs are written
        if (i + 1 >= nch) {
          griddep_launch();
          break;
        }
        const int ik = 2 * i + 2, sk = ik % kAfStages;
        ok = full_wait(ik);
        for (int t = 0; t < 2 && ok; ++t) {
          if (i + 1 >= (t ? nch1 : nch0)) continue;
          // the chunk's P V has read the columns that the next scores overwrite
          ok = mbar_wait(&pv_done[t], i & 1, a.status);
          if (!ok) break;
          tc_fence_after();
          scores(t, sk);
        }
        if (ok) tc_commit(&empty[sk]);
      }
      // every MMA issued is done before the TMEM is freed
      tc_commit(fin);
      mbar_wait(fin, 0, a.status);
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kAfSoftRegs));
    const int t = warp >> 2, wq = warp & 3;
    const int r0 = i0 + t * RT;
    const int nrows = t < n_tiles ? max(0, min(RT, a.rows_per_seq - r0)) : 0;
    // ---------------- the tile's queries as hi / lo planes: a warp per vector,
    // four dims a lane
    {
      const float sc = a.scale * kAfLog2e;
      constexpr int kPer = HD == 128 ? 1 : 2;   // vectors per warp step
      const int sub = HD == 128 ? 0 : lane >> 4, c4 = HD == 128 ? lane : lane & 15;
      uint8_t* qs = sm + t * SM::kQ;
#pragma unroll 16
      for (int u = 0; u < 32; u += kPer) {
        const int v = wq * 32 + u + sub;
        const int ii = v / G, hh = v - ii * G;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ii < nrows)
          x = __ldcg(reinterpret_cast<const float4*>(a.q + static_cast<size_t>(sl * a.rows_per_seq + r0 + ii) * a.ld_q +
                                                     (g * G + hh) * HD) + c4);
        uint2 hi, lo;
        split_bf16x2(x.x * sc, x.y * sc, hi.x, lo.x);
        split_bf16x2(x.z * sc, x.w * sc, hi.y, lo.y);
        const int col = 4 * c4;
        const uint32_t off = (col / 64) * SM::kBox + sw128_offset(v, col % 64);
        *reinterpret_cast<uint2*>(qs + off) = hi;
        *reinterpret_cast<uint2*>(qs + SM::kQ / 2 + off) = lo;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(q_ready);
    }
    // ---------------- softmax: thread = TMEM lane = vector
    const int v = wq * 32 + lane, vi = v / G, vh = v - vi * G;
    const bool live = vi < nrows;
    const int lim = live ? base + r0 + vi : -1;        // the last position the row sees
    const uint32_t lanes = static_cast<uint32_t>(wq * 32) << 16;
    const uint32_t ts = tmem + 128u * t + lanes, to = tmem + 256u + 128u * t + lanes;
    const int my = t ? nch1 : nch0;
    float m = -INFINITY, l = 0.f;
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i < my; ++i) {
      // the first tile that has the last chunk clears its values past the end
      // before its probabilities let P V start.  (The stage's copy before this
      // one, K chunk i - 1, is complete: its scores were read; none follows.)
      if (i == nch - 1 && t == (nch0 == nch ? 0 : 1) && past < kAfPos) {
        const int iv = 2 * i + 1, sv = iv % kAfStages;
        if (!mbar_wait(&full[sv], (iv / kAfStages) & 1, a.status)) {
          ok = false;
          break;
        }
        uint8_t* vs = sm + SM::kRing + sv * SM::kStage;
        for (int e = wq * 32 + lane; e < (kAfPos - past) * (HD / 8); e += kAfQ) {
          const int row = past + e / (HD / 8), q = e % (HD / 8);
          *reinterpret_cast<uint4*>(vs + (q >> 3) * SM::kBox + sw128_offset(row, 8 * (q & 7))) =
              make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
      }
      if (!mbar_wait(&s_full[t], i & 1, a.status)) {
        ok = false;
        break;
      }
      tc_fence_after();
      float s[kAfPos];
#pragma unroll
      for (int c = 0; c < kAfPos; c += 32) tmem_ld32_async(ts + c, s + c);
      tmem_ld_wait();
      const int see = lim - i * kAfPos;                // positions 0 .. see of the chunk are visible
      if (see < kAfPos - 1) {
#pragma unroll
        for (int c = 0; c < kAfPos; ++c) s[c] = c <= see ? s[c] : -INFINITY;
      }
      float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
      for (int c = 4; c < kAfPos; ++c) mx[c & 3] = fmaxf(mx[c & 3], s[c]);
      const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
      // a new reference: the first chunk, or the maximum has outgrown the old one
      const bool move = top > m + kLazy || (m == -INFINITY && top > m);
      if (__any_sync(0xffffffffu, move)) {
        const float f = move ? (m == -INFINITY ? 0.f : ex2(m - top)) : 1.f;
        if (move) m = top;
        l *= f;
        if (i > 0) {
          if (!mbar_wait(&pv_done[t], (i - 1) & 1, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < HD; c += 16) {
            float o[16];
            tmem_ld16(to + c, o);
            uint32_t r[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(o[e] * f);
            tmem_st16(to + c, r);
          }
          tmem_st_wait();
        }
      }
      const float mu = m == -INFINITY ? 0.f : m;
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < kAfPos; c += 32) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float p0 = ex2(s[c + 2 * e] - mu), p1 = ex2(s[c + 2 * e + 1] - mu);
          sum[(2 * e) & 3] += p0;
          sum[(2 * e + 1) & 3] += p1;
          split_bf16x2(p0, p1, hi[e], lo[e]);
        }
        tmem_st16(ts + c / 2, hi);
        tmem_st16(ts + 64 + c / 2, lo);
      }
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_ready[t]);
    }
    // ---------------- O / l as hi / lo rows
    if (ok && my > 0 && mbar_wait(&pv_done[t], (my - 1) & 1, a.status)) {
      tc_fence_after();
      const float inv = 1.f / l;
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(a.o) +
                           static_cast<size_t>(sl * a.rows_per_seq + r0 + vi) * a.ld_o + (g * G + vh) * HD;
#pragma unroll 1
      for (int c = 0; c < HD; c += 16) {
        float o[16];
        tmem_ld16(to + c, o);
        if (!live) continue;
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) split_bf16x2(o[2 * e] * inv, o[2 * e + 1] * inv, hi[e], lo[e]);
        uint4* h4 = reinterpret_cast<uint4*>(out + c);
        uint4* l4 = reinterpret_cast<uint4*>(out + a.o_plane + c);
        h4[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        h4[1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
        l4[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        l4[1] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

namespace {
// Registers per thread that the kernel was compiled with.
template <int HD>
int af_regs() {
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, attn_pf_kernel<HD>) == cudaSuccess) return fa.numRegs;
  cudaGetLastError();
  return 0;
}

template <int HD>
cudaError_t launch_af(const AttnArgs& a, cudaStream_t s) {
  static PerDevice attr;
  attr.once([] {
    cudaFuncSetAttribute(attn_pf_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, AfSmem<HD>::kTotal);
  });
  // One tile per CTA while the waves allow it: a lone tile's chunk is S,
  // softmax and P V in turn (about 4700 cycles at hd 128), a pair's 6200.
  // At hd 64 the ratio serves too (32 heads, pairs against single tiles: 512
  // rows 23.1 / 21.1 us, 2048 rows 88.5 / 96.0, 8192 rows 909 / 1192; 16 heads
  // over 4 KV heads, always single here: 23.7 / 20.2, 95 / 77, 939 / 723) but
  // where a pair saves the second of two waves (700 rows 29.6 / 25.9, 1024 rows
  // 32.6 / 31.1: pairs are taken).
  const int rt = kAfQ / (a.n_heads / a.n_kv_heads);
  const int u1 = (a.rows_per_seq + rt - 1) / rt, u2 = (u1 + 1) / 2;
  const long heads = static_cast<long>(a.n_kv_heads) * a.n_seqs;
  const long w1 = (heads * u1 + a.n_sms - 1) / a.n_sms, w2 = (heads * u2 + a.n_sms - 1) / a.n_sms;
  const int n_tiles = w1 * 4700 <= w2 * 6200 ? 1 : 2;
  return launch_pdl(attn_pf_kernel<HD>, dim3(a.n_kv_heads, n_tiles == 1 ? u1 : u2, a.n_seqs), dim3(kAfThreads),
                    AfSmem<HD>::kTotal, s, *a.kmap, *a.vmap, a, n_tiles);
}
}  // namespace

// The softmax warps' register increase draws on what the block was launched
// with and waits for ever if that is less than the split needs.
bool attn_pf_ok(int head_dim) {
  const int regs = head_dim == 128 ? af_regs<128>() : af_regs<64>();
  return regs * kAfThreads >= 256 * kAfSoftRegs + 128 * kAfOtherRegs;
}

cudaError_t launch_attn_pf(const AttnArgs& a, cudaStream_t s) {
  return a.head_dim == 128 ? launch_af<128>(a, s) : launch_af<64>(a, s);
}

}  // namespace dvi
