// The finalize steps of the decode passes (Sec. 3.3) as device functions
// that any 128 threads of a CTA can run together: the standalone finalize
// kernels (one CTA of 128 threads) and the last CTA of a head projection,
// whose 128 epilogue threads run them once every head CTA has published its
// argmax (the fused head -> argmax -> accept -> commit path).  Their block
// barriers are a named barrier of those 128 threads (fin_sync).
//
// finalize_verify is the accept/commit/rollback step of Sec. 3.3: with
// y*_{n+i} the verifier's argmax at block row i-1 and t~_i the drafts,
// m = max{i <= K : t~_j = y*_{n+j} for all j <= i}; the step commits
// t~_1..t~_m and, when m < K, the correction y*_{n+m+1} -- min(m+1, K)
// tokens -- and the cache length advances by the same count, which discards
// the KV rows of rejected drafts (they are overwritten later; no data moves).
// With the bonus row (verify rows for t~_1..t~_K and one more for t~_K's
// successor) y*_{n+K+1} exists too, and every step commits m + 1 tokens.
// The replay-buffer tuples of rows 1..min(m+1, K) get r = 1 up to m and r = 0
// at the first reject (Sec. 3.3); later rows stay invalid (counterfactual).
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace dvi {

constexpr int kMaxTiles = 64;   // d <= 8192
constexpr int kFinThreads = 128;

// Barrier of the 128 threads running a finalize step (the whole CTA of a
// finalize kernel, the epilogue warps of a head projection).
__device__ __forceinline__ void fin_sync() { named_bar(2, kFinThreads); }

// Shared memory of a finalize step.
struct FinSmem {
  int tok_s[64];
  int m_s[64];                    // verify: accept lengths,
  int y_s[kMaxTokens];            // y* of every verify row,
  int dr_s[kMaxTokens + 64];      // and the block's tokens [B][K + 1]
  float red[kMaxTiles * 4];
  float rstd_s;
  int last;   // head projection: this CTA is the last to finish
};

// One residual row from the embedding table (128 threads): x, x * g and the
// per-tile sums of squares.  All of the row's loads are issued before any is
// used (one memory round trip), then a single block barrier.
template <typename T>
__device__ void embed_row_block(const T* table, int tok, int d, float* x, const float* g, T* xg, size_t plane,
                                float* ss, int ss_ld, int row, float* red) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NT = kMaxTiles;
  const int nt = d / kTileRows;
  const T* src = table + static_cast<size_t>(tok) * d;
  float v[NT], gv[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    if (t < nt) {
      v[t] = DT<T>::ld(src + t * kTileRows + tid);
      gv[t] = g[t * kTileRows + tid];
    }
  }
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    if (t < nt) {
      const int c = t * kTileRows + tid;
      x[c] = v[t];
      Act<T>::st(xg + c, plane, v[t] * gv[t]);
      const float s = warp_sum(v[t] * v[t]);
      if (lane == 0) red[t * 4 + warp] = s;
    }
  }
  fin_sync();
  for (int t = tid; t < nt; t += kFinThreads)
    ss[static_cast<size_t>(t) * ss_ld + row] = (red[t * 4] + red[t * 4 + 1]) + (red[t * 4 + 2] + red[t * 4 + 3]);
  fin_sync();
}


// One row of the drafter-head preparation (128 threads): x = h_k, its
// per-tile sums of squares and 1/rms, u = x * rstd * gain into `us` (when
// non-null), and, when `io` is set, u into the replay buffer and h_k handed
// to the verify rows (x, x * g_copy and the sums of squares).
template <typename T, int NT = kMaxTiles>
__device__ void prep_row(const HeadPrepArgs& a, int row, bool io, float* red, float* rstd_s, float* us) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* x = a.x + static_cast<size_t>(row) * a.ldx;
  const int nt = a.d / kTileRows;
  float xv[NT], gv[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (t < nt) {
      xv[t] = x[t * kTileRows + tid];
      gv[t] = a.gain[t * kTileRows + tid];
    }
  // per-tile sums of squares (also the hand-off's statistics), then 1/rms
#pragma unroll
  for (int t = 0; t < NT; ++t)
    if (t < nt) {
      const float s = warp_sum(xv[t] * xv[t]);
      if (lane == 0) red[t * 4 + warp] = s;
    }
  fin_sync();
  if (tid == 0) {
    float s = 0.f;
    for (int t = 0; t < nt; ++t) s += (red[t * 4] + red[t * 4 + 1]) + (red[t * 4 + 2] + red[t * 4 + 3]);
    *rstd_s = rsqrtf(s / static_cast<float>(a.d) + a.eps);
  }
  fin_sync();
  const float rstd = *rstd_s;
  if (us) {
#pragma unroll
    for (int t = 0; t < NT; ++t)
      if (t < nt) us[t * kTileRows + tid] = xv[t] * rstd * gv[t];
  }
  if (io) {
    T* lu = nullptr;
    if (a.log_u && a.log_enabled) {
      const int ls = *a.log_step;
      if (ls < a.log_cap_steps)
        lu = static_cast<T*>(a.log_u) +
             (static_cast<size_t>(ls) * a.log_rows_per_step + static_cast<size_t>(row) * a.log_row_stride +
              a.log_row_off) * a.d;
    }
    if (lu) {
#pragma unroll
      for (int t = 0; t < NT; ++t)
        if (t < nt) Act<T>::st(lu + t * kTileRows + tid, a.log_plane, xv[t] * rstd * gv[t]);
    }
    if (a.x_copy) {
      const int crow = row * a.copy_row_stride + a.copy_row_off;
      float* xc = a.x_copy + static_cast<size_t>(crow) * a.ld_copy;
      T* xgc = static_cast<T*>(a.xg_copy) + static_cast<size_t>(crow) * a.ld_copy;
      float gc[NT];
#pragma unroll
      for (int t = 0; t < NT; ++t)
        if (t < nt) gc[t] = a.g_copy[t * kTileRows + tid];
#pragma unroll
      for (int t = 0; t < NT; ++t)
        if (t < nt) {
          xc[t * kTileRows + tid] = xv[t];
          Act<T>::st(xgc + t * kTileRows + tid, a.xg_copy_plane, xv[t] * gc[t]);
        }
      for (int t = tid; t < nt; t += 128)
        a.ss_copy[static_cast<size_t>(t) * a.ss_copy_ld + crow] =
            (red[t * 4] + red[t * 4 + 1]) + (red[t * 4 + 2] + red[t * 4 + 3]);
    }
  }
}


__device__ __forceinline__ int take_argmax(unsigned long long* slot, int* status) {
  const unsigned long long k = __ldcg(slot);
  *slot = 0ull;
  if (k == 0ull) {
    flag_status(status, DVI_DEV_NONFINITE);
    return 0;
  }
  return argmax_idx(k);
}

// Four consecutive values (a column that is a multiple of 4); one vector load
// where the row's address allows it.
__device__ __forceinline__ float4 ld_row4(const __nv_bfloat16* p, bool vec) {
  if (!vec) return make_float4(__bfloat162float(p[0]), __bfloat162float(p[1]), __bfloat162float(p[2]),
                               __bfloat162float(p[3]));
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(bf16_lo(u.x), bf16_hi(u.x), bf16_lo(u.y), bf16_hi(u.y));
}
// The activation row's four values at p (hi and lo planes).
__device__ __forceinline__ void st_act_row4(__nv_bfloat16* p, size_t plane, float4 v) {
  uint2 hi, lo;
  split_bf16x2(v.x, v.y, hi.x, lo.x);
  split_bf16x2(v.z, v.w, hi.y, lo.y);
  *reinterpret_cast<uint2*>(p) = hi;
  *reinterpret_cast<uint2*>(p + plane) = lo;
}

// Embeds each sequence's next input token into the draft residual stream: x,
// x * g and the per-tile sums of squares.  A warp per eight 128-feature tiles
// of a row, four features of each a lane, its loads in flight together;
// `staged`: the rows in shared memory, else they come from the table.  f32
// rows keep the order of their sums (a warp's 32 features at a time).  (One row after
// another by all 128 threads took 14 us a row: 110 of a draft head's 162 us
// at batch 8.)
template <typename T>
__device__ void embed_rows(const StepState& st, const int* toks, const T* staged = nullptr) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d = st.d, nt = d / kTileRows;
  [[maybe_unused]] const bool svec = staged || (reinterpret_cast<uintptr_t>(st.embed) & 15u) == 0;
  const int parts = (nt + 7) / 8;
  for (int it = warp; it < st.B * parts; it += kFinThreads / 32) {
    const int b = it / parts, t0 = it % parts * 8;
    const T* src = (staged ? staged + static_cast<size_t>(b) * d
                           : static_cast<const T*>(st.embed) + static_cast<size_t>(toks[b]) * d);
    float* x = st.x_dr + static_cast<size_t>(b) * d;
    T* xg = static_cast<T*>(st.xg_dr) + static_cast<size_t>(b) * d;
    if constexpr (sizeof(T) == 4) {
      for (int t = t0; t < min(t0 + 8, nt); ++t) {
        float q[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int c = t * kTileRows + 32 * e + lane;
          const float f = src[c];
          x[c] = f;
          xg[c] = f * st.g0[c];
          q[e] = f * f;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) q[e] = warp_sum(q[e]);
        if (lane == 0) st.ss_dr[static_cast<size_t>(t) * st.ss_dr_ld + b] = (q[0] + q[1]) + (q[2] + q[3]);
      }
    } else {
      src += 4 * lane;
      x += 4 * lane;
      xg += 4 * lane;
      float4 v[8], g[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = min(t0 + u, nt - 1);
        v[u] = ld_row4(src + t * kTileRows, svec);
        const float* gp = st.g0 + t * kTileRows + 4 * lane;   // 16-byte aligned (bf16 models)
        g[u] = *reinterpret_cast<const float4*>(gp);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = t0 + u;
        if (t >= nt) break;
        *reinterpret_cast<float4*>(x + t * kTileRows) = v[u];
        st_act_row4(xg + t * kTileRows, st.xg_dr_plane,
                    make_float4(v[u].x * g[u].x, v[u].y * g[u].y, v[u].z * g[u].z, v[u].w * g[u].w));
        const float q = warp_sum((v[u].x * v[u].x + v[u].y * v[u].y) + (v[u].z * v[u].z + v[u].w * v[u].w));
        if (lane == 0) st.ss_dr[static_cast<size_t>(t) * st.ss_dr_ld + b] = q;
      }
    }
  }
}


// 16-byte asynchronous copy global -> shared (completes at cp_async_wait).
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_all;" ::: "memory");
}


// With `prep` set, the drafter-head preparation of the pass (the logged u
// and the hand-off of h_k to the verify rows; the head computed B u itself)
// runs here, for every row before its residual is overwritten by the next
// pass's embedding.  The drafted tokens are read first; with `emb_raw` set
// (B * d elements of shared memory) the next pass's embedding rows are
// copied into shared memory asynchronously while the preparation runs, so
// their load is off the critical path.
template <typename T, int NT = kMaxTiles>
__device__ void finalize_draft_body(const StepState& st, int j, const HeadPrepArgs& hp, int prep, FinSmem& fs,
                                    uint8_t* emb_raw) {
  for (int b = threadIdx.x; b < st.B; b += kFinThreads) {
    const int t = take_argmax(st.amax + b, st.status);
    st.draft_ids[b * (st.K + 1) + j + 1] = t;
    fs.tok_s[b] = t;
  }
  fin_sync();
  const bool next = j + 1 < st.Kv;   // the next pass's token (t~_K feeds the bonus row)
  if (next && emb_raw) {
    const int per_row = st.d * static_cast<int>(sizeof(T)) / 16;
    for (int i = threadIdx.x; i < st.B * per_row; i += kFinThreads) {
      const int b = i / per_row, c = i % per_row;
      int tok = fs.tok_s[b];
      if (tok < 0 || tok >= st.vocab) tok = 0;   // flagged by the embedding below
      cp_async16(emb_raw + static_cast<size_t>(i) * 16,
                 reinterpret_cast<const uint8_t*>(static_cast<const T*>(st.embed) + static_cast<size_t>(tok) * st.d) +
                     static_cast<size_t>(c) * 16);
    }
  }
  if (prep) {
    for (int b = 0; b < hp.rows; ++b) {
      prep_row<T, NT>(hp, b, true, fs.red, &fs.rstd_s, nullptr);
      fin_sync();
    }
  }
  if (!next) return;
  if (!emb_raw) {
    embed_rows<T>(st, fs.tok_s);
    return;
  }
  cp_async_wait();
  fin_sync();
  for (int b = threadIdx.x; b < st.B; b += kFinThreads)
    if (fs.tok_s[b] < 0 || fs.tok_s[b] >= st.vocab) flag_status(st.status, DVI_DEV_BAD_TOKEN);
  embed_rows<T>(st, fs.tok_s, reinterpret_cast<const T*>(emb_raw));
}

// Accept length, commit and rollback, the replay-buffer tuples' metadata,
// and the next pass's embedding (finalize_verify).
template <typename T>
__device__ void finalize_verify_body(const StepState& st, FinSmem& fs) {
  const int K = st.K, Kv = st.Kv;
  // one round trip: every row's argmax and every drafted token by a thread of
  // its own (a sequence's thread reading them in turn took 10 us)
  for (int t = threadIdx.x; t < st.B * Kv; t += kFinThreads) fs.y_s[t] = take_argmax(st.amax + t, st.status);
  for (int t = threadIdx.x; t < st.B * (K + 1); t += kFinThreads) fs.dr_s[t] = st.draft_ids[t];
  const int ls = *st.log_step;
  const bool log_ok = st.log_enabled && ls < st.log_cap_steps;
  fin_sync();
  for (int b = threadIdx.x; b < st.B; b += kFinThreads) {
    const int* y = fs.y_s + b * Kv;
    const int* dr = fs.dr_s + b * (K + 1);
    int m = 0;
    while (m < K && dr[m + 1] == y[m]) ++m;
    // the correction y*_{n+m+1} exists for m < K, and for m = K with the bonus row
    const int c = m < Kv ? m + 1 : K;
    const int newtok = m < Kv ? y[m] : dr[K];
    st.n_committed[b] = c;
    st.n_accepted[b] = m;
    st.lens[b] += c;
    st.pending[b] = newtok;
    st.draft_ids[b * (K + 1)] = newtok;
    fs.tok_s[b] = newtok;
    fs.m_s[b] = m;
    atomicAdd(reinterpret_cast<unsigned long long*>(st.counters + 2), static_cast<unsigned long long>(m));
    atomicAdd(reinterpret_cast<unsigned long long*>(st.counters + 3), static_cast<unsigned long long>(c));
  }
  fin_sync();
  for (int t = threadIdx.x; t < st.B * Kv; t += kFinThreads) {
    const int b = t / Kv, i = t % Kv, m = fs.m_s[b];
    const int* dr = fs.dr_s + b * (K + 1);
    st.out_ids[t] = i < m ? dr[i + 1] : (i == m ? fs.y_s[t] : -1);
    if (log_ok && i < K) {
      const int c = m < Kv ? m + 1 : K;
      int* meta = st.log_meta + (static_cast<size_t>(ls) * st.B * K + b * K + i) * 6;
      meta[0] = i < c;
      meta[1] = dr[i + 1];
      meta[2] = i < m ? 1 : 0;
      meta[3] = i + 1;
      meta[4] = dr[i];
      meta[5] = fs.y_s[t];
    }
  }
  if (threadIdx.x == 0) {
    st.counters[0] += 1;
    st.counters[1] += static_cast<long long>(st.B) * K;
    if (st.log_enabled) {
      if (ls < st.log_cap_steps) *st.log_step = ls + 1;
      else flag_status(st.status, DVI_DEV_LOG_FULL);
    }
  }
  embed_rows<T>(st, fs.tok_s);
}

// Greedy AR: the argmax is the next token of every sequence (finalize_ar).
template <typename T>
__device__ void finalize_ar_body(const StepState& st, FinSmem& fs) {
  for (int b = threadIdx.x; b < st.B; b += kFinThreads) {
    const int y = take_argmax(st.amax + b, st.status);
    st.out_ids[b] = y;
    st.lens[b] += 1;
    st.pending[b] = y;
    st.draft_ids[b * (st.K + 1)] = y;
    fs.tok_s[b] = y;
  }
  fin_sync();
  embed_rows<T>(st, fs.tok_s);
}

// The drafter-head preparation of a draft pass whose finalize step runs in
// the head: CTA b takes row b while the weights stream (only the finalize
// step, after every CTA, overwrites the rows).  In the last CTA, row after
// row, it and the embedding took 110 us of a 209 us head launch at batch 8.
template <int NT>
__device__ __forceinline__ void head_prepare(const FinArgs& f, float* red, float* rstd_s) {
  if (f.kind != FIN_DRAFT || !f.prep) return;
  for (int b = blockIdx.x; b < f.hp.rows; b += gridDim.x) {
    prep_row<__nv_bfloat16, NT>(f.hp, b, true, red, rstd_s, nullptr);
    fin_sync();
  }
}

// The finalize step after a head projection, in the head's last CTA: every
// head CTA's argmax keys are published before the count reaches the grid.
// `smem` is free shared memory of the CTA: the FinSmem, then (f.stage) the
// staged embedding rows.
// NT bounds d / 128 (the per-thread register arrays of the row steps).
template <int NT>
__device__ __forceinline__ void head_finalize(const FinArgs& f, uint8_t* smem, int tid) {
  FinSmem& fs = *reinterpret_cast<FinSmem*>(smem);
  __threadfence();
  fin_sync();
  if (tid == 0) fs.last = atomicAdd(f.ctr, 1) == static_cast<int>(gridDim.x) - 1;
  fin_sync();
  if (!fs.last) return;
  __threadfence();
  if (tid == 0) *f.ctr = 0;
  uint8_t* emb = f.stage ? smem + (sizeof(FinSmem) + 15) / 16 * 16 : nullptr;
  // (the preparation ran in the head's first CTAs)
  if (f.kind == FIN_DRAFT) finalize_draft_body<__nv_bfloat16, NT>(f.st, f.j, f.hp, 0, fs, emb);
  else if (f.kind == FIN_VERIFY) finalize_verify_body<__nv_bfloat16>(f.st, fs);
  else finalize_ar_body<__nv_bfloat16>(f.st, fs);
}

}  // namespace dvi
