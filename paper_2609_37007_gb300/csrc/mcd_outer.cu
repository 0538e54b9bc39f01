// Outer CodeDecoder and the full frame pipeline (arXiv 2609.37007, Sec. 1 and Fig. 1).
//
// Per 80 ms frame the CodeDecoder (28 pre-norm layers, the MultiCodeDecoder's block) runs
// one row over its utterance-long KV cache, its c0 head gives the frame's seed code c0 (top-k
// / temperature sampling, Philox counter of position 0), and its post-norm hidden state plus
// the c0 embedding start the MultiCodeDecoder's frame, which emits c1..c15.  The next
// frame's CodeDecoder input is the sum of the text row (if any) and the embeddings of the 16
// codes just emitted.  Before frame 0 the text prompt is prefilled: with the shapes the
// tcgen05 block kernels take, every row as one batch on the tensor cores (outer_tc_prefill, hi + lo
// operands like outer_kernel's), else up to 16 rows per outer_kernel launch; outer_kernel
// then runs the c0 head of the last row and samples frame 0's c0.
//
// outer_kernel is one cooperative launch of one CTA per SM, built on the same weight ring
// and unit GEMMs as the frame kernel (mcd_stage.cuh): per layer QKV -> attention -> Wo ->
// gate/up -> down, each stage ordered by a grid-wide arrival counter.  Attention over the
// long cache is split over key blocks (flash-decoding style): one task per (KV head, block
// of 32 keys) normalises and rotates its rows' queries and new keys, writes the new K / V
// to the cache (rounded to the cache dtype), and leaves per-row partial softmax sums
// (max, sum of exponentials, weighted values); the CTAs of the Wo stage merge the blocks of
// their head before multiplying.  The last CTA to finish the c0 head samples c0.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../../include/mcd_pipeline.h"
#include "mcd_host.cuh"
#include "mcd_internal.cuh"
#include "mcd_sampler.cuh"
#include "mcd_stage.cuh"
#include "mcd_tcops.cuh"

namespace mcd {

constexpr int kKeyBlock = 32;          // keys per attention task
constexpr int kMaxOuterTokens = 1024;  // KV capacity: at most 32 key blocks (one lane each)
constexpr int kMaxPrefillRows = 16;    // rows per prefill launch (bf16 hi/lo operand)
constexpr int kMaxQVec = 32;           // query vectors per attention task (rows x group)
constexpr int kPartLd = 132;           // floats per partial record: D (<= 128) values, max, sum

struct OuterStep {
  uint8_t* kcache;                 // [L][NKV][cap][D] in the weight dtype
  uint8_t* vcache;
  int cap;
  const float2* rope;              // [cap][D/2] (cos, sin)
  int pos0, nr, head;              // first new position, new rows, 1 = c0 head + sampling
  int l0;                          // first layer to run (L: the c0 head alone, on the row in p.x)
  const int* text_ids;             // prefill: ids of the rows (device), else null
  const int* prev_codes;           // frame step: c0..c_P of the previous frame (device)
  int text_id;                     // frame step: text row added to the sum, -1 = none
  const uint8_t* text_table;
  int text_vocab;
  const uint8_t* c0_table;
  int c0_vocab;
  const uint8_t* code_tables;      // inner table j (1 <= j < P) at code_tables + j * code_stride
  long long code_stride;
  int code_vocab, P;
  const uint8_t* last_table;       // table P (owned by the outer model)
  float* part;                     // [n_blocks][nr][NH][kPartLd]
  int* c0_out;
  int* c0_out2;                    // optional second destination of c0
  float* cond_out;                 // [H] post-norm hidden state of the last row
  float* c0emb_out;                // [H] c0 embedding (fp32)
  float* trace;                    // optional [C0V + 2H]: c0 logits, cond, c0 embedding
  unsigned stream_id, frame_id;
};

// ------------------------------------------------------------------------------------
// Producer: the CTA's units of every stage, in stage order.
// ------------------------------------------------------------------------------------
__device__ void outer_producer(const FrameParams& p, const OuterStep& o, Smem& sm) {
  const uint64_t pol = policy_evict_first();
  const volatile int* stop = sm.flags;
  const int heads[1] = {1};
  const int ns = 4 * p.L + (o.head ? 1 : 0);
  uint32_t issued = 0;
  int rot = 0;
  bool halt = false;
  for (int si = 4 * o.l0; si < ns && !halt; ++si) {
    const int n = stage_units(p, si, 1);
    const uint32_t bytes = (uint32_t)p.g[stage_kind(si, p.L)].unit_bytes;
    const UnitRange ur = unit_range(si, p.L, n, blockIdx.x, rot, p.n_cta);
    for (int u = ur.first; u < ur.end && !halt; u += ur.step)
      halt = !ring_issue(p, sm, issued, unit_src(p, si, u, heads), bytes, pol, stop);
    rot = (rot + n) % p.n_cta;
  }
  ring_drain(p, sm, issued);
}

// ------------------------------------------------------------------------------------
// Attention task (KV head g, key block b)
// ------------------------------------------------------------------------------------
// Keys j0..j1-1 of the block: cached positions (< pos0) come from the cache, new positions
// from this launch's QKV output.  Query vector qi is row n_lo + qi / group, query head
// g * group + qi % group; rows below n_lo see no key of the block.  Scratch (act + bfrag):
// q [32][D + 8], k [32][D + 8], v [32][D], scores [32][32], rope rows [16][D/2], gains.
template <int WT>
__device__ void outer_attention(Cons& c, const OuterStep& o, int layer, int g, int b) {
  const FrameParams& p = c.p;
  const int D = p.D, half = D >> 1, group = p.NH / p.NKV, nr = o.nr, pos0 = o.pos0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = b * kKeyBlock, j1 = min(j0 + kKeyBlock, pos0 + nr), nk = j1 - j0;
  const int jn = min(max(j0, pos0), j1);      // first new key of the block (j1: none)
  const int n_lo = max(0, j0 - pos0);         // first row that sees a key of the block
  const int nq = (nr - n_lo) * group;
  const int KS = D + 8;
  const int cpr = D >> 2;                     // 16-byte fp32 chunks per row
  float* qs = c.sm.act;
  float* ks = qs + kMaxQVec * 136;
  float* vs = ks + kKeyBlock * 136;
  float* sc = vs + kKeyBlock * 128;
  float2* cs = reinterpret_cast<float2*>(sc + kMaxQVec * kKeyBlock);
  float* gq = reinterpret_cast<float*>(cs + kMaxPrefillRows * 64);
  float* gk = gq + 128;
  const size_t es = WT == MCD_WEIGHT_BF16 ? 2 : 4;
  const size_t cache_off = (((size_t)layer * p.NKV + g) * o.cap) * D;   // elements
  const int qkv_dim = p.qkv_dim, koff = p.NH * D + g * D, voff = p.NH * D + p.NKV * D + g * D;
  // ---- (A) loads, 16-byte chunks, a batch of 8 per thread in flight -----------------------
  {
    const int e_q = nq * cpr;                         // queries
    const int e_new = e_q + 2 * (j1 - jn) * cpr;      // new keys then new values
    const int ccpr = WT == MCD_WEIGHT_BF16 ? (D >> 3) : cpr;   // chunks per cached row
    const int e_old = e_new + 2 * (jn - j0) * ccpr;   // cached keys then cached values
    const int e_cs = e_old + (nr - n_lo) * (half >> 1);
    const int e_all = e_cs + (p.qk_norm ? 2 * cpr : 0);
    for (int base = 0; base < e_all; base += 8 * kConsumerThreads) {
      float4 v[8];
      int kind[8];
      void* dst[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = base + tid + u * kConsumerThreads;
        kind[u] = -1;
        if (i >= e_all) continue;
        if (i < e_q) {
          const int qi = i / cpr, ch = i - qi * cpr, n = n_lo + qi / group, h = g * group + qi % group;
          v[u] = __ldcg(reinterpret_cast<const float4*>(p.qkv + (size_t)n * qkv_dim + h * D) + ch);
          dst[u] = reinterpret_cast<float4*>(qs + qi * KS) + ch;
          kind[u] = 0;
        } else if (i < e_new) {
          const int r = i - e_q, isv = r >= (j1 - jn) * cpr, rr = r - (isv ? (j1 - jn) * cpr : 0);
          const int jj = rr / cpr, ch = rr - jj * cpr, n = jn + jj - pos0;
          v[u] = __ldcg(reinterpret_cast<const float4*>(p.qkv + (size_t)n * qkv_dim + (isv ? voff : koff)) + ch);
          dst[u] = isv ? reinterpret_cast<float4*>(vs + (jn + jj - j0) * D) + ch
                       : reinterpret_cast<float4*>(ks + (jn + jj - j0) * KS) + ch;
          kind[u] = 0;
        } else if (i < e_old) {
          const int r = i - e_new, isv = r >= (jn - j0) * ccpr, rr = r - (isv ? (jn - j0) * ccpr : 0);
          const int jj = rr / ccpr, ch = rr - jj * ccpr;
          const uint8_t* src = (isv ? o.vcache : o.kcache) + (cache_off + (size_t)(j0 + jj) * D) * es;
          v[u] = __ldcg(reinterpret_cast<const float4*>(src) + ch);
          float* row = isv ? vs + jj * D : ks + jj * KS;
          dst[u] = row + ch * (WT == MCD_WEIGHT_BF16 ? 8 : 4);
          kind[u] = WT == MCD_WEIGHT_BF16 ? 1 : 0;
        } else if (i < e_cs) {
          const int r = i - e_old, n = n_lo + r / (half >> 1), ch = r % (half >> 1);
          v[u] = __ldg(reinterpret_cast<const float4*>(o.rope + (size_t)(pos0 + n) * half) + ch);
          dst[u] = reinterpret_cast<float4*>(cs + n * 64) + ch;
          kind[u] = 0;
        } else {
          const int r = i - e_cs, w = r / cpr, ch = r - w * cpr;
          v[u] = __ldg(reinterpret_cast<const float4*>((w == 0 ? p.q_norm : p.k_norm) + (size_t)layer * D) + ch);
          dst[u] = reinterpret_cast<float4*>(w == 0 ? gq : gk) + ch;
          kind[u] = 0;
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (kind[u] == 0) {
          *reinterpret_cast<float4*>(dst[u]) = v[u];
        } else if (kind[u] == 1) {   // 8 bf16 -> 8 floats
          const uint32_t w[4] = {__float_as_uint(v[u].x), __float_as_uint(v[u].y), __float_as_uint(v[u].z),
                                 __float_as_uint(v[u].w)};
          float4* d4 = reinterpret_cast<float4*>(dst[u]);
          d4[0] = make_float4(bf16_lo_f32(w[0]), bf16_hi_f32(w[0]), bf16_lo_f32(w[1]), bf16_hi_f32(w[1]));
          d4[1] = make_float4(bf16_lo_f32(w[2]), bf16_hi_f32(w[2]), bf16_lo_f32(w[3]), bf16_hi_f32(w[3]));
        }
      }
    }
  }
  consumer_sync();
  // ---- (B) QK-norm + RoPE of the queries and new keys; new K / V rounded and cached -------
  const int nd = D >> 5;   // dims per lane (lane + 32 i)
  const int n_new = j1 - jn;
  for (int vi = warp; vi < nq + 2 * n_new; vi += kConsumerWarps) {
    const int kind = vi < nq ? 0 : (vi < nq + n_new ? 1 : 2);   // query, new key, new value
    const int jj = kind == 0 ? 0 : (kind == 1 ? vi - nq : vi - nq - n_new);
    const int n = kind == 0 ? n_lo + vi / group : jn + jj - pos0;
    float* row = kind == 0 ? qs + vi * KS : (kind == 1 ? ks + (jn + jj - j0) * KS : vs + (jn + jj - j0) * D);
    float x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = i < nd ? row[lane + 32 * i] : 0.f;
    if (kind < 2) {
      if (p.qk_norm) {
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) ss += x[i] * x[i];
#pragma unroll
        for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
        const float scl = rsqrtf(ss / (float)D + p.eps);
        const float* gg = kind == 0 ? gq : gk;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < nd) x[i] = x[i] * scl * gg[lane + 32 * i];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i < nd / 2) {
          const float2 r = cs[n * 64 + lane + 32 * i];
          const float a = x[i], bb = x[i + nd / 2];
          x[i] = a * r.x - bb * r.y;
          x[i + nd / 2] = bb * r.x + a * r.y;
        }
      }
    }
    if (kind > 0) {   // cache dtype: the value every later read sees, this task's included
      uint8_t* dst = (kind == 1 ? o.kcache : o.vcache) + (cache_off + (size_t)(pos0 + n) * D) * es;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i < nd) {
          if (WT == MCD_WEIGHT_BF16) {
            const uint32_t bits = bf16_rn_bits(x[i]);
            reinterpret_cast<uint16_t*>(dst)[lane + 32 * i] = (uint16_t)bits;
            x[i] = bf16_bits_to_f32(bits);
          } else {
            reinterpret_cast<float*>(dst)[lane + 32 * i] = x[i];
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < nd) row[lane + 32 * i] = x[i];
  }
  consumer_sync();
  // ---- (C) scores: two threads per (query, key), interleaved 16-byte chunks ---------------
  const float scale = rsqrtf((float)D);
  for (int t = tid; t < nq * 2 * kKeyBlock; t += kConsumerThreads) {
    const int qi = t / (2 * kKeyBlock), kk = (t >> 1) & (kKeyBlock - 1), hf = t & 1;
    const int n = n_lo + qi / group;
    const bool live = kk < nk && j0 + kk <= pos0 + n;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    if (live) {
      const float4* q4 = reinterpret_cast<const float4*>(qs + qi * KS) + hf;
      const float4* k4 = reinterpret_cast<const float4*>(ks + kk * KS) + hf;
#pragma unroll 8
      for (int ch = 0; ch < (cpr >> 1); ++ch) {
        const float4 q = q4[2 * ch], k = k4[2 * ch];
        a0 += q.x * k.x;
        a1 += q.y * k.y;
        a2 += q.z * k.z;
        a3 += q.w * k.w;
      }
    }
    float acc = (a0 + a1) + (a2 + a3);
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
    if (hf == 0) sc[qi * kKeyBlock + kk] = live ? acc * scale : -INFINITY;
  }
  consumer_sync();
  // ---- (D) block softmax statistics: one warp per query (lane = key) ------------------------
  for (int qi = warp; qi < nq; qi += kConsumerWarps) {
    const int n = n_lo + qi / group, h = g * group + qi % group;
    const float s = sc[qi * kKeyBlock + lane];
    float m = s;
#pragma unroll
    for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
    const float e = s == -INFINITY ? 0.f : __expf(s - m);
    float l = e;
#pragma unroll
    for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, off);
    sc[qi * kKeyBlock + lane] = e;
    if (lane == 0) {
      float* rec = o.part + (((size_t)b * nr + n) * p.NH + h) * kPartLd;
      rec[D] = m;
      rec[D + 1] = l;
    }
  }
  consumer_sync();
  // ---- (E) weighted values: one thread per (query, dim pair) -------------------------------
  for (int t = tid; t < nq * half; t += kConsumerThreads) {
    const int qi = t / half, d = 2 * (t - qi * half);
    const int n = n_lo + qi / group, h = g * group + qi % group;
    const float* pr = sc + qi * kKeyBlock;
    float2 acc = make_float2(0.f, 0.f);
    for (int kk = 0; kk < nk; ++kk) {
      const float w = pr[kk];
      const float2 v = *reinterpret_cast<const float2*>(vs + kk * D + d);
      acc.x += w * v.x;
      acc.y += w * v.y;
    }
    *reinterpret_cast<float2*>(o.part + (((size_t)b * nr + n) * p.NH + h) * kPartLd + d) = acc;
  }
  consumer_sync();
}

// The same task for one row of the standard geometry (D = 128, two query heads per KV head, bf16
// cache).  Everything that does not depend on the row's QKV product is under way before the grid
// barrier in front of it: the block's cached K and V (cp.async, kept as bf16), the RoPE row and the
// gains.  After it warps 0 and 1 take a query head each, warps 2 and 3 the new key and value where
// the block holds the row's position; then four threads per (query, key) score, and each warp
// takes the softmax statistics of its query (redundantly) and 32 of the output's dims.
// A chain of L2 round trips and shuffles bounds it.  12 rows at 333 positions with their prompt:
// 10253 us with the general task and merge (9.1 k and 4.0 k of 48 k cycles per layer, stamped in an
// instrumented copy), 9016 with these; 8850 with the waits of every stage inline.
constexpr int kRowLd = 160;            // staged row (bf16): neighbouring keys 16 banks apart
struct RowAttn {
  uint16_t *kb, *vb;                   // [32][kRowLd]
  float *qs, *sc;                      // queries [2][128], scores [2][32]
  __device__ explicit RowAttn(float* act)
      : kb(reinterpret_cast<uint16_t*>(act)), vb(kb + kKeyBlock * kRowLd),
        qs(reinterpret_cast<float*>(vb + kKeyBlock * kRowLd)), sc(qs + 256) {}
};
static_assert(2 * kKeyBlock * kRowLd * 2 + (256 + 2 * kKeyBlock) * 4 <= kActBytes, "row attention scratch");
struct RowAhead {
  float gain[4];
  float2 rope[2];
};
__device__ __noinline__ RowAhead row_attention_ahead(const FrameParams& p, const OuterStep& o, float* act, int layer, int g, int b) {
  const RowAttn a(act);
  RowAhead ra{};
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = b * kKeyBlock, n_old = min(kKeyBlock, o.pos0 - j0);
  const size_t off = (((size_t)layer * p.NKV + g) * o.cap + j0) * 128;
  const uint16_t* kc = reinterpret_cast<const uint16_t*>(o.kcache) + off;
  const uint16_t* vc = reinterpret_cast<const uint16_t*>(o.vcache) + off;
  for (int i = tid; i < n_old * 16; i += kConsumerThreads) {
    const int jj = i >> 4, ch = 8 * (i & 15);
    cpa16(a.kb + jj * kRowLd + ch, kc + jj * 128 + ch);
    cpa16(a.vb + jj * kRowLd + ch, vc + jj * 128 + ch);
  }
  if (warp < 3) {
    const float* gg = (warp < 2 ? p.q_norm : p.k_norm) + (size_t)layer * 128;
#pragma unroll
    for (int i = 0; i < 4; ++i) ra.gain[i] = p.qk_norm ? __ldg(gg + lane + 32 * i) : 1.f;
#pragma unroll
    for (int i = 0; i < 2; ++i) ra.rope[i] = __ldg(o.rope + (size_t)o.pos0 * 64 + lane + 32 * i);
  }
  return ra;
}
__device__ __noinline__ void row_attention(const FrameParams& p, const OuterStep& o, float* act, int layer, int g, int b,
                                           RowAhead ra) {
  const RowAttn a(act);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, pos0 = o.pos0;
  const int j0 = b * kKeyBlock, nk = min(kKeyBlock, pos0 + 1 - j0);
  const bool has_new = pos0 - j0 < kKeyBlock;
  if (warp < (has_new ? 4 : 2)) {
    const int NH = p.NH, NKV = p.NKV;
    const float* src = p.qkv + (warp < 2 ? 2 * g + warp : warp == 2 ? NH + g : NH + NKV + g) * 128;
    float x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = __ldcg(src + lane + 32 * i);
    if (warp < 3) {
      if (p.qk_norm) {
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) ss += x[i] * x[i];
#pragma unroll
        for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
        const float scl = rsqrtf(ss / 128.f + p.eps);
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = x[i] * scl * ra.gain[i];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float e = x[i], f = x[i + 2];
        x[i] = e * ra.rope[i].x - f * ra.rope[i].y;
        x[i + 2] = f * ra.rope[i].x + e * ra.rope[i].y;
      }
    }
    if (warp < 2) {
#pragma unroll
      for (int i = 0; i < 4; ++i) a.qs[warp * 128 + lane + 32 * i] = x[i];
    } else {              // rounded to the cache's bf16: the value every later read sees, this one included
      uint16_t* row = (warp == 2 ? a.kb : a.vb) + (pos0 - j0) * kRowLd;
      uint16_t* dst = reinterpret_cast<uint16_t*>(warp == 2 ? o.kcache : o.vcache) +
                      (((size_t)layer * NKV + g) * o.cap + pos0) * 128;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint16_t bits = (uint16_t)bf16_rn_bits(x[i]);
        row[lane + 32 * i] = bits;
        dst[lane + 32 * i] = bits;
      }
    }
  }
  cpa_wait_all();
  consumer_sync();
  {
    const int qi = tid >> 7, kk = (tid >> 2) & 31, part = tid & 3;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    if (kk < nk) {
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const int d = 8 * (part + 4 * ch);
        const uint4 k = *reinterpret_cast<const uint4*>(a.kb + kk * kRowLd + d);
        const float4 q0 = *reinterpret_cast<const float4*>(a.qs + qi * 128 + d);
        const float4 q1 = *reinterpret_cast<const float4*>(a.qs + qi * 128 + d + 4);
        s0 += q0.x * bf16_lo_f32(k.x);
        s1 += q0.y * bf16_hi_f32(k.x);
        s2 += q0.z * bf16_lo_f32(k.y);
        s3 += q0.w * bf16_hi_f32(k.y);
        s0 += q1.x * bf16_lo_f32(k.z);
        s1 += q1.y * bf16_hi_f32(k.z);
        s2 += q1.z * bf16_lo_f32(k.w);
        s3 += q1.w * bf16_hi_f32(k.w);
      }
    }
    float sc = (s0 + s1) + (s2 + s3);
    sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 1);
    sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 2);
    if (part == 0) a.sc[qi * kKeyBlock + kk] = kk < nk ? sc * rsqrtf(128.f) : -INFINITY;
  }
  consumer_sync();
  const int qi = warp >> 2, d = 32 * (warp & 3) + 2 * (lane & 15), kh = lane >> 4;
  const float s = a.sc[qi * kKeyBlock + lane];
  uint32_t v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i)
    v[i] = 2 * i + kh < nk ? *reinterpret_cast<const uint32_t*>(a.vb + (2 * i + kh) * kRowLd + d) : 0u;
  float m = s;
#pragma unroll
  for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
  const float e = lane < nk ? __expf(s - m) : 0.f;
  float l = e;
#pragma unroll
  for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, off);
  float2 acc = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float w = __shfl_sync(0xFFFFFFFFu, e, 2 * i + kh);
    acc.x += w * bf16_lo_f32(v[i]);
    acc.y += w * bf16_hi_f32(v[i]);
  }
  acc.x += __shfl_xor_sync(0xFFFFFFFFu, acc.x, 16);
  acc.y += __shfl_xor_sync(0xFFFFFFFFu, acc.y, 16);
  float* rec = o.part + ((size_t)b * p.NH + 2 * g + qi) * kPartLd;
  if (kh == 0) *reinterpret_cast<float2*>(rec + d) = acc;
  if ((warp & 3) == 0 && lane == 0) {
    rec[128] = m;
    rec[129] = l;
  }
}

// The merge (below) for one row of 128 dims: each warp computes the blocks' weights for itself while
// its loads of the partial sums are in flight; threads d and d + 128 take alternate blocks.
__device__ __noinline__ void row_merge(const FrameParams& p, const OuterStep& o, int h, float* ao) {
  const int tid = threadIdx.x, lane = tid & 31, d = tid & 127, half = tid >> 7;
  const int nb = o.pos0 / kKeyBlock + 1;
  const float* rec = o.part + (size_t)h * kPartLd;
  const size_t ld = (size_t)p.NH * kPartLd;
  float m = -INFINITY, l = 0.f, v[16];
  if (lane < nb) {
    m = __ldcg(rec + lane * ld + 128);
    l = __ldcg(rec + lane * ld + 129);
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = half + 2 * i < nb ? __ldcg(rec + (half + 2 * i) * ld + d) : 0.f;
  float M = m;
#pragma unroll
  for (int off = 16; off; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, off));
  const float w = lane < nb ? __expf(m - M) : 0.f;
  float den = w * l;
#pragma unroll
  for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xFFFFFFFFu, den, off);
  const float wn = w / den;
  float acc = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) acc += __shfl_sync(0xFFFFFFFFu, wn, half + 2 * i) * v[i];
  if (half) ao[128 + d] = acc;
  consumer_sync();
  if (!half) ao[d] = acc + ao[128 + d];
  consumer_sync();
}
static_assert(kConsumerThreads == 256 && kMaxOuterTokens <= 32 * kKeyBlock, "row attention: threads, key blocks");

// Attention output of query head h for every row: the merge of the key blocks' partial sums
// (each block rescaled by e^{m_b - M}), written to ao [nr][D] in shared memory.
__device__ void outer_merge(Cons& c, const OuterStep& o, int h, float* ao) {
  const FrameParams& p = c.p;
  const int D = p.D, nr = o.nr, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* wts = ao + kMaxPrefillRows * 128;     // [nr][32] block weights / denominator
  for (int n = warp; n < nr; n += kConsumerWarps) {
    const int nb = (o.pos0 + n) / kKeyBlock + 1;
    float m = -INFINITY, l = 0.f;
    if (lane < nb) {
      const float* rec = o.part + (((size_t)lane * nr + n) * p.NH + h) * kPartLd;
      m = __ldcg(rec + D);
      l = __ldcg(rec + D + 1);
    }
    float M = m;
#pragma unroll
    for (int off = 16; off; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, off));
    const float w = lane < nb ? __expf(m - M) : 0.f;
    float den = w * l;
#pragma unroll
    for (int off = 16; off; off >>= 1) den += __shfl_xor_sync(0xFFFFFFFFu, den, off);
    wts[n * 32 + lane] = w / den;
  }
  consumer_sync();
  for (int i = tid; i < nr * D; i += kConsumerThreads) {
    const int n = i / D, d = i - n * D, nb = (o.pos0 + n) / kKeyBlock + 1;
    float acc = 0.f;
    for (int b = 0; b < nb; ++b)
      acc += wts[n * 32 + b] * __ldcg(o.part + (((size_t)b * nr + n) * p.NH + h) * kPartLd + d);
    ao[n * D + d] = acc;
  }
  consumer_sync();
}

// c0 of the frame (run by the CTA that finished the c0 head last): top-k / temperature
// distribution of the logits, one draw with counter (stream, frame, 0, 0, 0); then the
// inner model's inputs: cond = post-norm hidden state, the c0 embedding in fp32.
template <int WT>
__device__ void outer_sample(Cons& c, const OuterStep& o) {
  const FrameParams& p = c.p;
  Smem& sm = c.sm;
  TopkScratch& ts = *reinterpret_cast<TopkScratch*>(sm.act);
  TopkRec* rec = reinterpret_cast<TopkRec*>(sm.bfrag);
  __shared__ int s_c0;
  block_topk(p.logits, p.V, p.top_k, p.T, 0, ts, rec);
  consumer_sync();
  if (threadIdx.x < 32) {
    const unsigned long long U = uniform_U(p.seed, o.stream_id, o.frame_id, 0, 0, PURPOSE_TARGET);
    const int d = warp_draw(rec, U);
    if (threadIdx.x == 0) s_c0 = d;
  }
  consumer_sync();
  const int c0 = s_c0;
  if (threadIdx.x == 0) {
    *o.c0_out = c0;
    if (o.c0_out2) *o.c0_out2 = c0;
  }
  // 1/rms of the row (this CTA need not have had a unit of the head, so it sums the row itself)
  const float* xl = p.x + (size_t)(o.nr - 1) * p.H;
  float ss = 0.f;
  for (int k = threadIdx.x; k < p.H; k += kConsumerThreads) {
    const float v = __ldcg(xl + k);
    ss += v * v;
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
  if ((threadIdx.x & 31) == 0) sm.part[threadIdx.x >> 5] = ss;
  consumer_sync();
  ss = 0.f;
#pragma unroll
  for (int w = 0; w < kConsumerWarps; ++w) ss += sm.part[w];
  const float inv = rsqrtf(__fmul_rn(ss, __frcp_rn((float)p.H)) + p.eps);
  for (int k = threadIdx.x; k < p.H; k += kConsumerThreads) {
    const float h = __ldcg(xl + k) * inv * __ldg(p.final_norm + k);
    const float e = WT == MCD_WEIGHT_BF16
                        ? bf16_bits_to_f32(reinterpret_cast<const uint16_t*>(o.c0_table)[(size_t)c0 * p.H + k])
                        : reinterpret_cast<const float*>(o.c0_table)[(size_t)c0 * p.H + k];
    o.cond_out[k] = h;
    o.c0emb_out[k] = e;
    if (o.trace) {
      o.trace[p.V + k] = h;
      o.trace[p.V + p.H + k] = e;
    }
  }
  if (o.trace)
    for (int i = threadIdx.x; i < p.V; i += kConsumerThreads) o.trace[i] = __ldcg(p.logits + i);
}

// ------------------------------------------------------------------------------------
// One launch: prefill rows or one frame row
// ------------------------------------------------------------------------------------
template <int WT, bool WIDE, bool STD>
__device__ void run_outer(Cons& c, const OuterStep& o) {
  const FrameParams& p = c.p;
  Smem& sm = c.sm;
  const int L = p.L, H = STD ? 1024 : p.H, D = STD ? 128 : p.D, F = p.F, nr = o.nr;
  unsigned* ctr = p.ctr;
  const unsigned N = (unsigned)p.n_cta;
  const size_t rb = (size_t)H * (WT == MCD_WEIGHT_BF16 ? 2 : 4);   // bytes per table row
  int* ids = sm.ci->r_id;    // prefill: text id per row; frame: c0..c_P, then the text id
  if (threadIdx.x < kMaxCols) {
    const int t = threadIdx.x;
    int id = -1, lim = 0;
    if (o.text_ids) {
      if (t < nr) {
        id = o.text_ids[t];
        lim = o.text_vocab;
      }
    } else if (t <= o.P) {
      id = o.prev_codes[t];
      lim = t == 0 ? o.c0_vocab : o.code_vocab;
    } else if (t == o.P + 1 && o.text_id >= 0) {
      id = o.text_id;
      lim = o.text_vocab;
    }
    if (lim > 0 && (id < 0 || id >= lim)) {   // an id outside its table: fail the step
      atomicCAS(p.err, 0, (int)MCD_ERR_INVALID_ARG);
      id = 0;
    }
    ids[t] = id;
  }
  // layer-0 row n: a prompt row, or the frame input text + E_c0(c0) + sum_j E_j(c_j)
  auto ld0 = [&](int n, int k, auto w) {
    constexpr int W = decltype(w)::value;
    auto row_v = [&](const uint8_t* row) {
      if constexpr (WT == MCD_WEIGHT_BF16) return ldg_bf16_v<W>(row, k);
      else return ldg_f32_v<W>(row, k);
    };
    if (o.text_ids) return row_v(o.text_table + (size_t)ids[n] * rb);
    vecf<W> s{};
    if (ids[o.P + 1] >= 0) s = row_v(o.text_table + (size_t)ids[o.P + 1] * rb);
    add_v<W>(s, row_v(o.c0_table + (size_t)ids[0] * rb));
    for (int j = 1; j < o.P; ++j) add_v<W>(s, row_v(o.code_tables + (long long)j * o.code_stride + (size_t)ids[j] * rb));
    add_v<W>(s, row_v(o.last_table + (size_t)ids[o.P] * rb));
    return s;
  };
  auto from_x = [&](int n, int k, auto w) { return ld_global_v<decltype(w)::value>(p.x + (size_t)n * H + k); };
  auto no_key = [](int) { return 0; };
  auto no_prep = [](int, int, int) {};
  const int n_blocks = (o.pos0 + nr + kKeyBlock - 1) / kKeyBlock;
  const bool row = STD && nr == 1 && p.NH == 16 && p.NKV == 8;        // row_attention's heads

  // a unit's m-block and k-chunk (the standard shapes' m-block counts are powers of two)
  constexpr int lg_wo = ilog2_c(1024 / (16 * StdUnit<WT, MAT_WO>::Mu)), lg_wd = ilog2_c(1024 / (16 * StdUnit<WT, MAT_WD>::Mu));
  auto wo_key = [&](int u) { return STD ? u >> lg_wo : u / p.g[MAT_WO].n_mb; };
  auto wd_key = [&](int u) { return STD ? u >> lg_wd : u / p.g[MAT_WD].n_mb; };
  auto wo_mb = [&](int u) { return STD ? u & ((1 << lg_wo) - 1) : u % p.g[MAT_WO].n_mb; };
  auto wd_mb = [&](int u) { return STD ? u & ((1 << lg_wd) - 1) : u % p.g[MAT_WD].n_mb; };
  auto resid_epi = [&](int row, int n, float v) { atomicAdd(p.x + (size_t)n * H + row, v); };
  for (int l = o.l0; l < L; ++l) {
    // ---- RMSNorm -> QKV -----------------------------------------------------------------
    NarrowGain gain;
    fetch_gain<STD>(c, gain, p.attn_norm + (size_t)l * H, H);
    const auto sp_qkv = plan_of<WT, WIDE, STD, MAT_QKV>(c, 4 * l, p.g[MAT_QKV].n_units, nr, no_key);
    const bool seeds = STD ? first_unit(sp_qkv) == 0 : blockIdx.x == 0;      // the CTA that seeds x
    auto qkv_epi = [&](int u, int mi, int rr, int n, float v, float, float inv) {
      p.qkv[(size_t)n * p.qkv_dim + (u * (STD ? StdUnit<WT, MAT_QKV>::Mu : p.g[MAT_QKV].Mu) + mi) * 16 + rr] = v * inv;
    };
    if (l == 0) {
      consumer_sync();                       // gain and ids in shared memory
      norm_product<WT, WIDE, STD, MAT_QKV>(c, 0, 0, sp_qkv, nr, H, gain, ld0, seeds ? p.x : nullptr, no_prep, qkv_epi);
    } else {
      if (!cons_wait(c, ctr + ctr_stage(l - 1, 3), N)) return;
      norm_product<WT, WIDE, STD, MAT_QKV>(c, 0, 4 * l, sp_qkv, nr, H, gain, from_x, nullptr, no_prep, qkv_epi);
    }
    if (c.abort_) return;
    cons_signal(c, ctr + ctr_stage(l, 0), 0, 0);

    // ---- attention: (KV head, key block) tasks, then one grid barrier -------------------------
    if (row) {
      int t = blockIdx.x;
      const int n_tasks = 8 * n_blocks;
      RowAhead ra{};
      if (t < n_tasks) ra = row_attention_ahead(p, o, sm.act, l, t & 7, t >> 3);
      if (!cons_wait(c, ctr + ctr_stage(l, 0), N)) {
        cpa_wait_all();
        return;
      }
      while (t < n_tasks) {
        row_attention(p, o, sm.act, l, t & 7, t >> 3, ra);
        t += p.n_cta;
        if (t >= n_tasks) break;
        consumer_sync();                                   // the scratch is read to the end
        ra = row_attention_ahead(p, o, sm.act, l, t & 7, t >> 3);
      }
    } else {
      if (!cons_wait(c, ctr + ctr_stage(l, 0), N)) return;
      for (int t = blockIdx.x; t < p.NKV * n_blocks; t += p.n_cta) outer_attention<WT>(c, o, l, t % p.NKV, t / p.NKV);
    }
    cons_signal(c, ctr + ctr_att(L, l), 0, 0);

    // ---- Wo + residual: unit u multiplies the merged output of head wo_key(u) ----------------
    const auto sp_wo = plan_of<WT, WIDE, STD, MAT_WO>(c, 4 * l + 1, p.g[MAT_WO].n_units, nr, wo_key);
    if (!cons_wait(c, ctr + ctr_att(L, l), N)) return;
    float* ao = reinterpret_cast<float*>(sm.bfrag);
    keyed_product<WT, WIDE, STD, MAT_WO, false>(
        c, 0, 4 * l + 1, sp_wo, nr, D, wo_key, [&](int u0) {
          if (row) row_merge(p, o, wo_key(u0), ao);
          else outer_merge(c, o, wo_key(u0), ao);
        },
        [&](int, int n, int k, auto w) { return ld_shared_v<decltype(w)::value>(ao + n * D + k); },
        reinterpret_cast<uint8_t*>(sm.act), [&](int u, int mi, int rr, int n, float v) {
          resid_epi((wo_mb(u) * (STD ? StdUnit<WT, MAT_WO>::Mu : p.g[MAT_WO].Mu) + mi) * 16 + rr, n, v);
        });
    if (c.abort_) return;
    cons_signal(c, ctr + ctr_stage(l, 1), 0, 0);

    // ---- RMSNorm -> gate/up -> SwiGLU ---------------------------------------------------------
    fetch_gain<STD>(c, gain, p.ffn_norm + (size_t)l * H, H);
    const auto sp_gu = plan_of<WT, WIDE, STD, MAT_GU>(c, 4 * l + 2, p.g[MAT_GU].n_units, nr, no_key);
    if (!cons_wait(c, ctr + ctr_stage(l, 1), N)) return;
    norm_product<WT, WIDE, STD, MAT_GU>(c, 0, 4 * l + 2, sp_gu, nr, H, gain, from_x, nullptr, no_prep,
                                        [&](int u, int mi, int rr, int n, float gate, float up, float inv) {
                                          const int mt = u * (STD ? StdUnit<WT, MAT_GU>::Mu : p.g[MAT_GU].Mu) + mi;
                                          const float gt = gate * inv;
                                          p.mbuf[(size_t)n * F + mt * 8 + rr] = gt / (1.0f + __expf(-gt)) * (up * inv);
                                        });
    if (c.abort_) return;
    cons_signal(c, ctr + ctr_stage(l, 2), 0, 0);

    // ---- down + residual ------------------------------------------------------------------------
    const auto sp_wd = plan_of<WT, WIDE, STD, MAT_WD>(c, 4 * l + 3, p.g[MAT_WD].n_units, nr, wd_key);
    if (!cons_wait(c, ctr + ctr_stage(l, 2), N)) return;
    const int Kc = STD ? 1024 : p.g[MAT_WD].Ku * 16;
    keyed_product<WT, WIDE, STD, MAT_WD, false>(
        c, 0, 4 * l + 3, sp_wd, nr, Kc, wd_key, [](int) {},
        [&](int u0, int n, int k, auto w) {
          return ld_global_v<decltype(w)::value>(p.mbuf + (size_t)wd_key(u0) * Kc + (size_t)n * F + k);
        },
        reinterpret_cast<uint8_t*>(sm.act), [&](int u, int mi, int rr, int n, float v) {
          resid_epi((wd_mb(u) * (STD ? StdUnit<WT, MAT_WD>::Mu : p.g[MAT_WD].Mu) + mi) * 16 + rr, n, v);
        });
    if (c.abort_) return;
    cons_signal(c, ctr + ctr_stage(l, 3), 0, 0);
  }
  if (!o.head) return;

  // ---- final RMSNorm of the last row -> c0 head -------------------------------------------
  NarrowGain gain;
  fetch_gain<STD>(c, gain, p.final_norm, H);
  const auto sp_head = plan_of<WT, WIDE, STD, MAT_HEAD>(c, 4 * L, p.g[MAT_HEAD].n_units, 1, no_key);
  if (o.l0 < L) {
    if (!cons_wait(c, ctr + ctr_stage(L - 1, 3), N)) return;
  } else {
    consumer_sync();                         // the gain, where it is in shared memory
  }
  const float* xl = p.x + (size_t)(nr - 1) * H;
  norm_product<WT, WIDE, STD, MAT_HEAD>(
      c, 0, 4 * L, sp_head, 1, H, gain, [&](int, int k, auto w) { return ld_global_v<decltype(w)::value>(xl + k); }, nullptr,
      no_prep, [&](int u, int, int rr, int, float v, float, float inv) { p.logits[u * 16 + rr] = v * inv; });
  if (c.abort_) return;
  consumer_sync();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned old = atomicAdd(ctr + ctr_heads(L), 1u);
    sm.flags[2] = old == N - 1u ? 1 : 0;
    if (sm.flags[2]) __threadfence();
  }
  consumer_sync();
  if (sm.flags[2]) outer_sample<WT>(c, o);
}

template <int WT, bool WIDE, bool STD>
__global__ void __launch_bounds__(kThreads, 1)
    outer_kernel(const __grid_constant__ FrameParams p, const __grid_constant__ OuterStep o) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  Smem sm = smem_layout(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    for (int s = 0; s < kNumSlots; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], kConsumerWarps);
    }
    sm.flags[0] = 0;
    sm.flags[1] = 0;
    sm.flags[2] = 0;
    fence_barrier_init();
  }
  __syncthreads();
  if (warp == kConsumerWarps) {
    if ((tid & 31) == 0) outer_producer(p, o, sm);
  } else {
    Cons c(p, sm);
    run_outer<WT, WIDE, STD>(c, o);
    if (tid == 0) sm.flags[0] = 1;   // stop the producer
  }
  __syncthreads();
}

__global__ void outer_begin_kernel(unsigned* ctr, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) ctr[i] = 0u;
}

template <int WT, bool WIDE, bool STD>
static void* outer_entry() {
  return (void*)outer_kernel<WT, WIDE, STD>;
}

static void* outer_fn(int wdtype, bool wide, bool std_geom) {
  if (!wide && std_geom) return outer_entry<MCD_WEIGHT_BF16, false, true>();
  return wdtype == MCD_WEIGHT_BF16
             ? (wide ? outer_entry<MCD_WEIGHT_BF16, true, false>() : outer_entry<MCD_WEIGHT_BF16, false, false>())
             : (wide ? outer_entry<MCD_WEIGHT_F32, true, false>() : outer_entry<MCD_WEIGHT_F32, false, false>());
}

}  // namespace mcd

using namespace mcd;

// ------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------
// Prompt prefill on the tensor cores: the rows of a prompt of two or more tokens go through the
// layers as one batch (tcgen05 products with hi + lo operands, causal attention, K / V written
// to the cache); outer_kernel then runs the c0 head on the last row's residual and samples c0.
// With single bf16 operands outside QKV the last row had to run through outer_kernel's layers
// again: 2.30 ms for 256 tokens, 0.61 of them in that row, against 1.69 ms; and the prompt's
// outputs were 8.6e-5 off a 64-bit evaluation against 2.2e-5.
struct OuterTc {
  bool on = false;
  int Rtc = 0;                     // capacity in operand rows
  uint8_t* w = nullptr;            // per layer: SW128 copies of the weights
  TcLayerOffsets off;
  float* X = nullptr;              // [Rtc][H] residual stream
  float* qkv = nullptr;            // [Rtc][qkv_dim], up to kTcSmallRows rows kTcQkvSplit partial sums
  float* q = nullptr;              // [Rtc][NH * D] normalised, rotated queries
  float* part = nullptr;           // k-split partial sums of the residual products (tc_part_floats)
  uint8_t *xn_hi = nullptr, *xn_lo = nullptr, *att_t = nullptr, *att_lo = nullptr, *act_t = nullptr, *act_lo = nullptr;   // operands
  int* rows = nullptr;             // device: live rows
};

__global__ void pf_set_rows_kernel(int* rows, int n) { *rows = n; }

// Prompt rows: X = the rows' text embeddings (bf16 table) and layer 0's QKV operand.  One CTA per
// row, thread t owns elements 8t..8t+7.
__global__ void __launch_bounds__(128) pf_embed_kernel(const int* __restrict__ ids, const int* nrows,
                                                       const uint8_t* __restrict__ table, int vocab, int H, float* X,
                                                       const float* __restrict__ gain, float eps, int Rtc, uint8_t* hi,
                                                       uint8_t* lo, int* err) {
  tc::pdl_wait();
  tc::pdl_trigger();
  const int r = blockIdx.x;
  if (r >= *nrows) return;
  const int t = threadIdx.x;
  int id = ids[r];
  if (id < 0 || id >= vocab) {              // an id outside the text table fails the prefill
    if (t == 0) atomicCAS(err, 0, (int)MCD_ERR_INVALID_ARG);
    id = 0;
  }
  const bool live = t < H / 8;
  float v[8];
  float s2 = 0.f;
  if (live) {
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(table + ((size_t)id * H + 8 * t) * 2));
    v[0] = bf16_lo_f32(w.x); v[1] = bf16_hi_f32(w.x); v[2] = bf16_lo_f32(w.y); v[3] = bf16_hi_f32(w.y);
    v[4] = bf16_lo_f32(w.z); v[5] = bf16_hi_f32(w.z); v[6] = bf16_lo_f32(w.w); v[7] = bf16_hi_f32(w.w);
    float4* xr = reinterpret_cast<float4*>(X + (size_t)r * H + 8 * t);
    xr[0] = make_float4(v[0], v[1], v[2], v[3]);
    xr[1] = make_float4(v[4], v[5], v[6], v[7]);
#pragma unroll
    for (int i = 0; i < 8; ++i) s2 += v[i] * v[i];
  }
  const float tot = block_sum128(s2);
  if (!live) return;
  const NormChunk c = norm_chunk(v, rsqrtf(tot / (float)H + eps), gain, t);
  const size_t off = tc::sw128_offset(Rtc, r, t >> 3, t & 7);
  *reinterpret_cast<uint4*>(hi + off) = c.hi;
  *reinterpret_cast<uint4*>(lo + off) = c.lo;
}

// QK-norm + RoPE (position = row index) of every prompt row's query and key heads; K and V
// rounded to bf16 into layer l's cache ([NKV][cap][D]), the rotated queries (fp32) into q.
// One warp per (row, vector), lane holding dims lane + 32 i.
__global__ void __launch_bounds__(256) pf_rope_kv_kernel(const float* __restrict__ qkv, int nz, size_t zs, int qkv_dim,
                                                         const int* nrows,
                                                         int NH, int NKV, int D, int qk_norm, const float* qn,
                                                         const float* kn, float eps, const float2* __restrict__ rope,
                                                         uint16_t* kc, uint16_t* vc, int cap, float* q) {
  tc::pdl_wait();
  tc::pdl_trigger();
  const int vecs = NH + 2 * NKV, w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int r = w / vecs, vi = w - r * vecs;
  if (r >= *nrows) return;
  const int kind = vi < NH ? 0 : (vi < NH + NKV ? 1 : 2), h = kind == 0 ? vi : (kind == 1 ? vi - NH : vi - NH - NKV);
  const int nd = D >> 5, half = D >> 1;
  const float* src = qkv + (size_t)r * qkv_dim + (kind == 0 ? h * D : NH * D + (kind == 2 ? NKV * D : 0) + h * D);
  float x[4];
  qkv_row(x, src, nd, lane, nz, zs);
  if (kind < 2) {
    if (qk_norm) {
      float ssq = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) ssq += x[i] * x[i];
#pragma unroll
      for (int off = 16; off; off >>= 1) ssq += __shfl_xor_sync(0xFFFFFFFFu, ssq, off);
      const float scl = rsqrtf(ssq / (float)D + eps);
      const float* gg = kind == 0 ? qn : kn;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nd) x[i] = x[i] * scl * __ldg(gg + lane + 32 * i);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i < nd / 2) {
        const float2 cs = __ldg(rope + (size_t)r * half + lane + 32 * i);
        const float a = x[i], b = x[i + nd / 2];
        x[i] = a * cs.x - b * cs.y;
        x[i + nd / 2] = b * cs.x + a * cs.y;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (i < nd) {
      const int d = lane + 32 * i;
      if (kind == 0)
        q[(size_t)r * NH * D + h * D + d] = x[i];
      else
        (kind == 1 ? kc : vc)[((size_t)h * cap + r) * D + d] = (uint16_t)bf16_rn_bits(x[i]);
    }
  }
}

// Causal attention of the prompt rows over the bf16 cache on mma.sync tiles (the contraction is
// 16 queries x 32 keys x D: too small for a 128-row tcgen05 tile, and softmax sits between its
// two halves).  One CTA per (16 query rows, query head), the longest rows first; its four warps
// take the 32-key blocks in turn (warp w: blocks w, w + 4, ...) and merge at the end, so a
// 256-token prompt is 256 CTAs of at most two blocks per warp.  Each warp stages its K and V
// block with cp.async, the next K in flight during softmax and P.V, the next V during the next
// scores.  K and V are bf16 as cached; queries and probabilities stay 32-bit values, multiplied
// as three bf16 terms (8 + 8 + 8 mantissa bits) with fp32 accumulation.
//
// Measured on a 256-token prompt (28 layers, 16 / 8 heads x 128): 5.45 ms with one warp per
// (row, head) and scalar products, where every warp read all its K and V for a single row (126
// us per layer under the profiler); 2.86 ms with this kernel at the time, 1.69 ms now.  It left the
// prompt's error against a 64-bit evaluation where it was (8.1e-5, then 8.2e-5): the products' single
// bf16 operands set that, and with hi + lo operands it is 2.2e-5.
constexpr int kPfRows = 16, kPfKeys = 32, kPfWarps = 4;
template <int D>
struct PfAttn {
  static constexpr int kLd = D + 8;                               // staged row (bf16): conflict-free ldmatrix
  static constexpr int kBlockBytes = kPfKeys * kLd * 2;
  static constexpr int kQBytes = (D / 16) * 3 * 32 * 16;          // A fragments of the three query terms
  static constexpr int kStatOff = kQBytes + kPfWarps * 2 * kBlockBytes;   // [warp][row] max, sum
  static constexpr int kSmemBytes = kStatOff + kPfWarps * kPfRows * 2 * 4;
  static_assert(kPfRows * D * 4 <= kBlockBytes, "a warp's partial output reuses its K block");
};
__device__ __forceinline__ void pf_ldmatrix(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void pf_ldmatrix_t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
// Two fp32 values as three packed bf16 pairs whose sum is the value (24 mantissa bits).
__device__ __forceinline__ void pf_split3(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf16x2(a, b);
  const float a1 = a - bf16_lo_f32(h), b1 = b - bf16_hi_f32(h);
  m = pack_bf16x2(a1, b1);
  l = pack_bf16x2(a1 - bf16_lo_f32(m), b1 - bf16_hi_f32(m));
}
// One block of keys j0 .. j0 + 31 of a [cap][D] cache into a warp's staging rows (keys at or
// past n_keys as zeros).
template <int D>
__device__ __forceinline__ void pf_stage(uint16_t* dst, const uint16_t* src, int j0, int n_keys, int lane) {
  constexpr int kChunks = D / 8;
#pragma unroll
  for (int i = 0; i < kPfKeys * kChunks / 32; ++i) {
    const int c = lane + 32 * i, j = c / kChunks, ch = c % kChunks;
    const bool ok = j0 + j < n_keys;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst + j * PfAttn<D>::kLd + ch * 8)),
                 "l"(src + (size_t)(ok ? j0 + j : 0) * D + ch * 8), "r"(ok ? 16 : 0)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int D>
__global__ void __launch_bounds__(kPfWarps * 32) pf_attn_kernel(const float* __restrict__ q, const int* nrows, int NH,
                                                                int NKV, const uint16_t* __restrict__ kc,
                                                                const uint16_t* __restrict__ vc, int cap, int Rtc,
                                                                uint8_t* att_t, uint8_t* att_lo) {
  using S = PfAttn<D>;
  extern __shared__ __align__(16) uint8_t pf_smem[];
  tc::pdl_wait();
  tc::pdl_trigger();
  const int M = *nrows, r0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * kPfRows, h = blockIdx.y, g = h / (NH / NKV);
  if (r0 >= M) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gr = lane >> 2, t = lane & 3;
  uint4* qf = reinterpret_cast<uint4*>(pf_smem);                             // [D / 16][3][32]
  uint16_t* ks = reinterpret_cast<uint16_t*>(pf_smem + S::kQBytes + warp * 2 * S::kBlockBytes);
  uint16_t* vs = ks + kPfKeys * S::kLd;
  float* stat = reinterpret_cast<float*>(pf_smem + S::kStatOff);             // [warp][row][max, sum]
  const uint16_t* kb = kc + (size_t)g * cap * D;
  const uint16_t* vb = vc + (size_t)g * cap * D;
  const int n_keys = min(r0 + kPfRows, M), n_blocks = (n_keys + kPfKeys - 1) / kPfKeys;
  if (warp < n_blocks) {
    pf_stage<D>(ks, kb, warp * kPfKeys, n_keys, lane);
    pf_stage<D>(vs, vb, warp * kPfKeys, n_keys, lane);
  }
  // the query terms in A-fragment order: lane holds rows lane / 4 (+ 8), dims 2 (lane % 4) (+ 8)
  for (int kt = warp; kt < D / 16; kt += kPfWarps) {
    uint4 f[3];
    uint32_t* w0 = reinterpret_cast<uint32_t*>(&f[0]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = r0 + gr + 8 * (e & 1), d = kt * 16 + 2 * t + 8 * (e >> 1);
      const float2 v = r < M ? __ldcg(reinterpret_cast<const float2*>(q + ((size_t)r * NH + h) * D + d)) : make_float2(0.f, 0.f);
      pf_split3(v.x, v.y, w0[e], w0[4 + e], w0[8 + e]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) qf[(kt * 3 + c) * 32 + lane] = f[c];
  }
  __syncthreads();
  const float scale = rsqrtf((float)D);
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};                     // rows gr, gr + 8
  float o[D / 8][4];
#pragma unroll
  for (int i = 0; i < D / 8; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
  for (int b = warp; b < n_blocks; b += kPfWarps) {
    const int j0 = b * kPfKeys, nx = b + kPfWarps;
    asm volatile("cp.async.wait_group 1;" ::: "memory");                       // this block's K
    __syncwarp();
    float sc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) sc[i][e] = 0.f;
#pragma unroll
    for (int kt = 0; kt < D / 16; ++kt) {
      uint32_t kf[2][4];
#pragma unroll
      for (int p2 = 0; p2 < 2; ++p2)
        pf_ldmatrix(kf[p2], ks + (p2 * 16 + (lane >> 4) * 8 + (lane & 7)) * S::kLd + kt * 16 + ((lane >> 3) & 1) * 8);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const uint4 a = qf[(kt * 3 + c) * 32 + lane];
#pragma unroll
        for (int i = 0; i < 4; ++i) mma_bf16_16816(sc[i], a, kf[i >> 1][2 * (i & 1)], kf[i >> 1][2 * (i & 1) + 1]);
      }
    }
    __syncwarp();
    if (nx < n_blocks) pf_stage<D>(ks, kb, nx * kPfKeys, n_keys, lane);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    // scale, causal mask, running maximum (every row sees at least key j0: j0 <= r0)
    float mb[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = j0 + 8 * i + 2 * t + (e & 1), r = r0 + gr + 8 * (e >> 1);
        sc[i][e] = j <= r ? sc[i][e] * scale : -INFINITY;
        mb[e >> 1] = fmaxf(mb[e >> 1], sc[i][e]);
      }
    float corr[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      mb[x] = fmaxf(mb[x], __shfl_xor_sync(0xFFFFFFFFu, mb[x], 1));
      mb[x] = fmaxf(mb[x], __shfl_xor_sync(0xFFFFFFFFu, mb[x], 2));
      const float mn = fmaxf(m[x], mb[x]);
      corr[x] = __expf(m[x] - mn);
      m[x] = mn;
    }
    float ps[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        sc[i][e] = __expf(sc[i][e] - m[e >> 1]);                             // masked: exp(-inf) = 0
        ps[e >> 1] += sc[i][e];
      }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      ps[x] += __shfl_xor_sync(0xFFFFFFFFu, ps[x], 1);
      ps[x] += __shfl_xor_sync(0xFFFFFFFFu, ps[x], 2);
      l[x] = l[x] * corr[x] + ps[x];
    }
#pragma unroll
    for (int i = 0; i < D / 8; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[i][e] *= corr[e >> 1];
    asm volatile("cp.async.wait_group 1;" ::: "memory");                       // this block's V
    __syncwarp();
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      uint4 pf[3];
      uint32_t* w0 = reinterpret_cast<uint32_t*>(&pf[0]);
      pf_split3(sc[2 * kk][0], sc[2 * kk][1], w0[0], w0[4], w0[8]);
      pf_split3(sc[2 * kk][2], sc[2 * kk][3], w0[1], w0[5], w0[9]);
      pf_split3(sc[2 * kk + 1][0], sc[2 * kk + 1][1], w0[2], w0[6], w0[10]);
      pf_split3(sc[2 * kk + 1][2], sc[2 * kk + 1][3], w0[3], w0[7], w0[11]);
#pragma unroll
      for (int n2 = 0; n2 < D / 16; ++n2) {
        uint32_t vf[4];
        pf_ldmatrix_t(vf, vs + (kk * 16 + ((lane >> 3) & 1) * 8 + (lane & 7)) * S::kLd + n2 * 16 + (lane >> 4) * 8);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          mma_bf16_16816(o[2 * n2], pf[c], vf[0], vf[1]);
          mma_bf16_16816(o[2 * n2 + 1], pf[c], vf[2], vf[3]);
        }
      }
    }
    __syncwarp();
    if (nx < n_blocks) pf_stage<D>(vs, vb, nx * kPfKeys, n_keys, lane);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  // merge of the four warps' partial sums, each rescaled by e^{m_w - max}
  float* po = reinterpret_cast<float*>(ks);                                     // [16][D]
#pragma unroll
  for (int i = 0; i < D / 8; ++i)
#pragma unroll
    for (int x = 0; x < 2; ++x)
      *reinterpret_cast<float2*>(po + (gr + 8 * x) * D + 8 * i + 2 * t) = make_float2(o[i][2 * x], o[i][2 * x + 1]);
  if (t == 0) {
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      stat[(warp * kPfRows + gr + 8 * x) * 2] = m[x];
      stat[(warp * kPfRows + gr + 8 * x) * 2 + 1] = l[x];
    }
  }
  __syncthreads();
  const int row = tid >> 3, r = r0 + row;
  if (r >= M) return;
  float mx = -INFINITY, den = 0.f, wt[kPfWarps];
#pragma unroll
  for (int w = 0; w < kPfWarps; ++w) mx = fmaxf(mx, stat[(w * kPfRows + row) * 2]);
#pragma unroll
  for (int w = 0; w < kPfWarps; ++w) {
    wt[w] = __expf(stat[(w * kPfRows + row) * 2] - mx);                        // a warp without blocks: e^-inf = 0
    den += wt[w] * stat[(w * kPfRows + row) * 2 + 1];
  }
  const float inv = 1.0f / den;
#pragma unroll
  for (int c = 0; c < D / 64; ++c) {
    const int d = (tid & 7) * 8 + 64 * c;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = 0.f;
#pragma unroll
    for (int w = 0; w < kPfWarps; ++w) {
      const float4* pr = reinterpret_cast<const float4*>(
          reinterpret_cast<const float*>(pf_smem + S::kQBytes + w * 2 * S::kBlockBytes) + row * D + d);
      const float4 a = pr[0], b = pr[1];
      v[0] += wt[w] * a.x; v[1] += wt[w] * a.y; v[2] += wt[w] * a.z; v[3] += wt[w] * a.w;
      v[4] += wt[w] * b.x; v[5] += wt[w] * b.y; v[6] += wt[w] * b.z; v[7] += wt[w] * b.w;
    }
    const int f = h * D + d;
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float a = v[2 * e] * inv, b = v[2 * e + 1] * inv;
      hi[e] = pack_bf16x2(a, b);
      lo[e] = pack_bf16x2(a - bf16_lo_f32(hi[e]), b - bf16_hi_f32(hi[e]));
    }
    const size_t off = tc::sw128_offset(Rtc, r, f >> 6, (f & 63) >> 3);
    *reinterpret_cast<uint4*>(att_t + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(att_lo + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}
static cudaError_t pf_attn_set_smem() {
  cudaError_t e = cudaFuncSetAttribute(pf_attn_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, PfAttn<64>::kSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pf_attn_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, PfAttn<128>::kSmemBytes);
  return e;
}
static void launch_pf_attn(const float* q, const int* nrows, int n, int NH, int NKV, int D, const uint16_t* kc,
                           const uint16_t* vc, int cap, int Rtc, uint8_t* att_t, uint8_t* att_lo, cudaStream_t s) {
  const dim3 grid((n + kPfRows - 1) / kPfRows, NH);
  auto go = [&](auto kernel, int smem) {
    tc::launch(true, kernel, grid, dim3(kPfWarps * 32), smem, s, q, nrows, NH, NKV, kc, vc, cap, Rtc, att_t, att_lo);
  };
  if (D == 128) go(pf_attn_kernel<128>, PfAttn<128>::kSmemBytes);
  else go(pf_attn_kernel<64>, PfAttn<64>::kSmemBytes);
}

struct mcd_outer {
  mcd_outer_config cfg;
  OuterTc tc;
  mcd_ctx* inner = nullptr;
  cudaStream_t stream = nullptr;
  FrameParams fp;
  OuterStep st;
  std::vector<void*> allocs;
  int P = 0;                    // codes per frame after c0 (the inner model's positions)
  int n_tok = 0;                // KV positions filled
  int frame = -1;               // frame whose c0 the last launch produced
  bool ready = false;           // that c0 has not yet started an inner frame
  bool weights_loaded = false;
  uint32_t stream_id = 0;
  int* c0_buf = nullptr;
  float* cond = nullptr;
  float* c0emb = nullptr;
  int* last_codes = nullptr;    // c0..c_P of the last frame a pipeline call decoded
  float* trace = nullptr;
  int trace_frames = 0;
};

template <class T>
static cudaError_t outer_alloc(mcd_outer* o, T** p, size_t bytes) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, bytes < 256 ? 256 : bytes);
  if (e != cudaSuccess) return e;
  o->allocs.push_back(q);
  *p = static_cast<T*>(q);
  return cudaSuccess;
}

static mcd_status validate_outer(const mcd_outer_config& c, const FrameParams& ip) {
  if (c.n_layers < 1 || c.hidden != ip.H) return MCD_ERR_UNSUPPORTED;
  if (!(c.head_dim == 64 || c.head_dim == 128)) return MCD_ERR_UNSUPPORTED;
  if (c.n_q_heads < 1 || c.n_kv_heads < 1 || c.n_q_heads % c.n_kv_heads) return MCD_ERR_INVALID_ARG;
  if (c.n_q_heads / c.n_kv_heads > 8) return MCD_ERR_UNSUPPORTED;
  if (c.ffn < 128 || c.ffn % 128) return MCD_ERR_UNSUPPORTED;
  if ((long long)c.n_q_heads * c.head_dim + 2LL * c.n_kv_heads * c.head_dim > 8192) return MCD_ERR_UNSUPPORTED;
  if (c.c0_vocab < 16 || c.c0_vocab % 16 || c.c0_vocab > kMaxVocab) return MCD_ERR_UNSUPPORTED;
  if (c.text_vocab < 1) return MCD_ERR_INVALID_ARG;
  if (c.max_tokens < 1 || c.max_tokens > kMaxOuterTokens) return MCD_ERR_UNSUPPORTED;
  if (c.top_k < 1 || c.top_k > kMaxTopK || c.top_k > c.c0_vocab) return MCD_ERR_UNSUPPORTED;
  if (!(c.temperature > 0.f) || !(c.rms_eps > 0.f) || !(c.rope_base > 1.f)) return MCD_ERR_INVALID_ARG;
  if (c.weight_dtype != ip.wdtype) return MCD_ERR_INVALID_ARG;   // the frame sum reads the inner tables
  if (c.weight_dtype == MCD_WEIGHT_INT8) return MCD_ERR_UNSUPPORTED;
  if (ip.C0V != 0) return MCD_ERR_INVALID_ARG;                   // the inner model takes the c0 vector
  return MCD_OK;
}

static int prefill_rows(const mcd_outer* o) {
  return std::min(kMaxPrefillRows, kMaxQVec / (o->fp.NH / o->fp.NKV));
}

// x: the residual row of a launch that runs the c0 head alone (null: the context's rows).
static mcd_status outer_launch(mcd_outer* o, const OuterStep& s, float* x = nullptr) {
  FrameParams p = o->fp;
  if (x) p.x = x;
  outer_begin_kernel<<<1, 256, 0, o->stream>>>(p.ctr, p.ctr_stride);
  MCD_CHECK(cudaGetLastError());
  void* args[] = {&p, const_cast<OuterStep*>(&s)};
  MCD_CHECK(cudaLaunchCooperativeKernel(outer_fn(p.wdtype, s.nr > kMaxRows, std_geometry(p)), dim3(p.n_cta), dim3(kThreads), args,
                                        (size_t)kSmemBytes, o->stream));
  return MCD_OK;
}

// One CodeDecoder row for frame o->frame + 1 from the previous frame's codes (device).
static mcd_status outer_step_launch(mcd_outer* o, const int32_t* prev_codes, int32_t text_id, int32_t* c0_out2) {
  if (o->n_tok < 1) return MCD_ERR_STATE;
  if (o->n_tok >= o->st.cap) return MCD_ERR_STATE;   // the KV cache is full
  if (!prev_codes) return MCD_ERR_INVALID_ARG;
  if (text_id >= o->cfg.text_vocab) return MCD_ERR_INVALID_ARG;
  OuterStep s = o->st;
  s.pos0 = o->n_tok;
  s.nr = 1;
  s.head = 1;
  s.text_ids = nullptr;
  s.prev_codes = prev_codes;
  s.text_id = text_id < 0 ? -1 : text_id;
  s.c0_out2 = c0_out2;
  s.frame_id = (unsigned)(o->frame + 1);
  s.trace = (o->trace && o->frame + 1 < o->trace_frames)
                ? o->trace + (size_t)(o->frame + 1) * (o->fp.V + 2 * o->fp.H)
                : nullptr;
  mcd_status r = outer_launch(o, s);
  if (r != MCD_OK) return r;
  o->n_tok += 1;
  o->frame += 1;
  o->ready = true;
  return MCD_OK;
}

extern "C" {

mcd_status mcd_outer_create(const mcd_outer_config* cfg, mcd_ctx* inner, mcd_outer** out) {
  if (!out) return MCD_ERR_INVALID_ARG;
  *out = nullptr;
  if (!cfg || !inner) return MCD_ERR_INVALID_ARG;
  const FrameParams& ip = ctx_params(inner);
  mcd_status vs = validate_outer(*cfg, ip);
  if (vs != MCD_OK) return vs;
  mcd_outer* o = new mcd_outer();
  o->cfg = *cfg;
  o->inner = inner;
  o->stream = ctx_stream(inner);
  o->P = ip.P;
  auto fail = [&](mcd_status s) {
    mcd_outer_destroy(o);
    return s;
  };
  for (void* fn : {outer_fn(MCD_WEIGHT_BF16, false, true), outer_fn(MCD_WEIGHT_BF16, false, false),
                   outer_fn(MCD_WEIGHT_BF16, true, false), outer_fn(MCD_WEIGHT_F32, false, false),
                   outer_fn(MCD_WEIGHT_F32, true, false)})
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess)
      return fail(MCD_ERR_CUDA);
  const mcd_outer_config& k = *cfg;
  FrameParams& p = o->fp;
  memset(&p, 0, sizeof(p));
  p.L = k.n_layers;
  p.H = k.hidden;
  p.NH = k.n_q_heads;
  p.NKV = k.n_kv_heads;
  p.D = k.head_dim;
  p.F = k.ffn;
  p.P = ip.P;
  p.V = k.c0_vocab;
  p.C0V = k.c0_vocab;
  p.K = 0;
  p.top_k = k.top_k;
  p.qk_norm = k.qk_norm;
  p.wdtype = k.weight_dtype;
  p.eps = k.rms_eps;
  p.T = k.temperature;
  p.seed = k.seed;
  p.qkv_dim = p.NH * p.D + 2 * p.NKV * p.D;
  p.n_cta = ip.n_cta;
  p.wait_ns = ip.wait_ns;
  p.S = 1;
  if (!backbone_geom(p, p.V)) return fail(MCD_ERR_UNSUPPORTED);
  p.ctr_stride = ctr_count(p.L);
  const size_t es = k.weight_dtype == MCD_WEIGHT_BF16 ? 2 : 4;
  cudaError_t e;
  uint8_t *wq, *wo, *wg, *wd, *wh;
#define OUTER_ALLOC(ptr, bytes)                                              \
  do {                                                                       \
    if ((e = outer_alloc(o, &(ptr), (bytes))) != cudaSuccess) return fail(cuda_status(e)); \
  } while (0)
  OUTER_ALLOC(wq, (size_t)p.g[MAT_QKV].stride * p.L);
  OUTER_ALLOC(wo, (size_t)p.g[MAT_WO].stride * p.L);
  OUTER_ALLOC(wg, (size_t)p.g[MAT_GU].stride * p.L);
  OUTER_ALLOC(wd, (size_t)p.g[MAT_WD].stride * p.L);
  OUTER_ALLOC(wh, (size_t)p.g[MAT_HEAD].stride);
  p.w_qkv = wq;
  p.w_wo = wo;
  p.w_gu = wg;
  p.w_wd = wd;
  p.w_head = wh;
  float* f32 = nullptr;
  OUTER_ALLOC(f32, sizeof(float) * ((size_t)p.L * p.H * 2 + (size_t)p.L * p.D * 2 + p.H));
  p.attn_norm = f32;
  p.ffn_norm = p.attn_norm + (size_t)p.L * p.H;
  p.q_norm = p.ffn_norm + (size_t)p.L * p.H;
  p.k_norm = p.q_norm + (size_t)p.L * p.D;
  p.final_norm = p.k_norm + (size_t)p.L * p.D;
  OUTER_ALLOC(p.x, sizeof(float) * kMaxCols * p.H);
  OUTER_ALLOC(p.qkv, sizeof(float) * kMaxCols * p.qkv_dim);
  OUTER_ALLOC(p.mbuf, sizeof(float) * kMaxCols * p.F);
  OUTER_ALLOC(p.logits, sizeof(float) * p.V);
  OUTER_ALLOC(p.ctr, sizeof(unsigned) * p.ctr_stride);
  OUTER_ALLOC(p.err, sizeof(int));
  OuterStep& s = o->st;
  memset(&s, 0, sizeof(s));
  s.cap = k.max_tokens;
  const size_t kv = (size_t)p.L * p.NKV * s.cap * p.D * es;
  OUTER_ALLOC(s.kcache, kv);
  OUTER_ALLOC(s.vcache, kv);
  float2* rope = nullptr;
  OUTER_ALLOC(rope, sizeof(float2) * (size_t)s.cap * (p.D / 2));
  s.rope = rope;
  uint8_t *tt, *ct, *lt;
  OUTER_ALLOC(tt, (size_t)k.text_vocab * p.H * es);
  OUTER_ALLOC(ct, (size_t)k.c0_vocab * p.H * es);
  OUTER_ALLOC(lt, (size_t)ip.V * p.H * es);
  s.text_table = tt;
  s.text_vocab = k.text_vocab;
  s.c0_table = ct;
  s.c0_vocab = k.c0_vocab;
  s.code_tables = ip.embed;
  s.code_stride = ip.embed_stride;
  s.code_vocab = ip.V;
  s.P = ip.P;
  s.last_table = lt;
  const int n_blocks = (s.cap + kKeyBlock - 1) / kKeyBlock;
  OUTER_ALLOC(s.part, sizeof(float) * (size_t)n_blocks * kMaxPrefillRows * p.NH * kPartLd);
  OUTER_ALLOC(o->c0_buf, sizeof(int) * 4);
  OUTER_ALLOC(o->cond, sizeof(float) * p.H);
  OUTER_ALLOC(o->c0emb, sizeof(float) * p.H);
  OUTER_ALLOC(o->last_codes, sizeof(int) * (o->P + 1));
  OuterTc& t = o->tc;
  t.on = tc_block_supported(p) && s.cap >= 2;
  if (t.on) {
    const int Rtc = (s.cap + tc::kBM - 1) / tc::kBM * tc::kBM;
    t.Rtc = Rtc;
    t.off = tc_layer_offsets(p);
    OUTER_ALLOC(t.w, t.off.layer * p.L);
    OUTER_ALLOC(t.X, sizeof(float) * (size_t)Rtc * p.H);
    OUTER_ALLOC(t.qkv, sizeof(float) * (size_t)std::max(Rtc, kTcQkvSplit * std::min(Rtc, kTcSmallRows)) * p.qkv_dim);
    OUTER_ALLOC(t.q, sizeof(float) * (size_t)Rtc * p.NH * p.D);
    OUTER_ALLOC(t.part, sizeof(float) * tc_part_floats(Rtc, p.H));
    OUTER_ALLOC(t.xn_hi, (size_t)Rtc * p.H * 2);
    OUTER_ALLOC(t.xn_lo, (size_t)Rtc * p.H * 2);
    OUTER_ALLOC(t.att_t, (size_t)Rtc * p.NH * p.D * 2);
    OUTER_ALLOC(t.att_lo, (size_t)Rtc * p.NH * p.D * 2);
    OUTER_ALLOC(t.act_t, (size_t)Rtc * p.F * 2);
    OUTER_ALLOC(t.act_lo, (size_t)Rtc * p.F * 2);
    OUTER_ALLOC(t.rows, sizeof(int));
    if (tc_block_set_smem<true>() != cudaSuccess || pf_attn_set_smem() != cudaSuccess) return fail(MCD_ERR_CUDA);
  }
#undef OUTER_ALLOC
  s.c0_out = o->c0_buf;
  s.cond_out = o->cond;
  s.c0emb_out = o->c0emb;
  if (cudaMemsetAsync(p.err, 0, sizeof(int), o->stream) != cudaSuccess) return fail(MCD_ERR_CUDA);
  if (cudaMemsetAsync(s.kcache, 0, kv, o->stream) != cudaSuccess) return fail(MCD_ERR_CUDA);
  if (cudaMemsetAsync(s.vcache, 0, kv, o->stream) != cudaSuccess) return fail(MCD_ERR_CUDA);
  rope_kernel<<<64, 256, 0, o->stream>>>(rope, p.D, (double)k.rope_base, s.cap);
  if (cudaGetLastError() != cudaSuccess) return fail(MCD_ERR_CUDA);
  if (cudaStreamSynchronize(o->stream) != cudaSuccess) return fail(MCD_ERR_CUDA);
  *out = o;
  return MCD_OK;
}

void mcd_outer_destroy(mcd_outer* o) {
  if (!o) return;
  cudaStreamSynchronize(o->stream);
  for (void* q : o->allocs) cudaFree(q);
  delete o;
}

mcd_status mcd_outer_load_weights(mcd_outer* o, int32_t n, const char* const* names, const void* const* host_ptrs,
                                  const int64_t* nbytes) {
  if (!o || n <= 0 || !names || !host_ptrs || !nbytes) return MCD_ERR_INVALID_ARG;
  FrameParams& p = o->fp;
  const int64_t es = p.wdtype == MCD_WEIGHT_BF16 ? 2 : 4;
  std::map<std::string, std::pair<const void*, int64_t>> given;
  for (int i = 0; i < n; ++i) {
    if (!names[i] || !host_ptrs[i]) return MCD_ERR_INVALID_ARG;
    if (given.count(names[i])) return MCD_ERR_WEIGHTS;
    given[names[i]] = {host_ptrs[i], nbytes[i]};
  }
  const int64_t H = p.H, D = p.D, qd = (int64_t)p.NH * D, kd = (int64_t)p.NKV * D, F = p.F;
  auto have = [&](const std::string& name, int64_t count) {
    auto it = given.find(name);
    const bool ok = it != given.end() && it->second.second == count * es;
    if (!ok && getenv("MCD_DEBUG")) fprintf(stderr, "mcd: outer weight %s missing or wrong size\n", name.c_str());
    return ok;
  };
  // check every tensor before copying anything
  for (int l = 0; l < p.L; ++l) {
    const std::string pre = "layers." + std::to_string(l) + ".";
    if (!have(pre + "attn_norm", H) || !have(pre + "wq", qd * H) || !have(pre + "wk", kd * H) ||
        !have(pre + "wv", kd * H) || !have(pre + "wo", H * qd) || !have(pre + "ffn_norm", H) ||
        !have(pre + "wg", F * H) || !have(pre + "wu", F * H) || !have(pre + "wd", H * F))
      return MCD_ERR_WEIGHTS;
    if (p.qk_norm && (!have(pre + "q_norm", D) || !have(pre + "k_norm", D))) return MCD_ERR_WEIGHTS;
  }
  const std::string last = "code_embed." + std::to_string(o->P);
  if (!have("final_norm", H) || !have("c0_head", (int64_t)p.V * H) || !have("c0_embed", (int64_t)p.V * H) ||
      !have("text_embed", (int64_t)o->cfg.text_vocab * H) || !have(last, (int64_t)o->st.code_vocab * H))
    return MCD_ERR_WEIGHTS;
  // one layer's tensors (or the c0 head / final norm) at a time through a staging buffer
  const size_t layer_bytes = (size_t)(2 * H + 2 * D + qd * H + 2 * kd * H + H * qd + 3 * F * H) * es + 16 * 256;
  const size_t stage_bytes = std::max(layer_bytes, (size_t)(p.V * H + H) * es + 512);
  uint8_t* stage = nullptr;
  MCD_CHECK(cudaMalloc(&stage, stage_bytes));
  auto cleanup = [&](mcd_status s) {
    cudaStreamSynchronize(o->stream);
    cudaFree(stage);
    return s;
  };
  size_t off = 0;
  std::map<std::string, const uint8_t*> at;
  auto put = [&](const std::string& name) -> bool {
    auto& gv = given[name];
    if (cudaMemcpyAsync(stage + off, gv.first, (size_t)gv.second, cudaMemcpyHostToDevice, o->stream) != cudaSuccess)
      return false;
    at[name] = stage + off;
    off += ((size_t)gv.second + 255) / 256 * 256;
    return true;
  };
  for (int l = 0; l < p.L; ++l) {
    const std::string pre = "layers." + std::to_string(l) + ".";
    off = 0;
    at.clear();
    // the previous layer's tiling kernels read the staging buffer: wait for them
    if (cudaStreamSynchronize(o->stream) != cudaSuccess) return cleanup(MCD_ERR_CUDA);
    for (const char* t : {"wq", "wk", "wv", "wo", "wg", "wu", "wd", "attn_norm", "ffn_norm"})
      if (!put(pre + t)) return cleanup(MCD_ERR_CUDA);
    if (p.qk_norm && (!put(pre + "q_norm") || !put(pre + "k_norm"))) return cleanup(MCD_ERR_CUDA);
    LayerSrc ls{at[pre + "wq"], at[pre + "wk"], at[pre + "wv"], at[pre + "wo"], at[pre + "wg"], at[pre + "wu"],
                at[pre + "wd"], at[pre + "attn_norm"], at[pre + "ffn_norm"],
                p.qk_norm ? at[pre + "q_norm"] : nullptr, p.qk_norm ? at[pre + "k_norm"] : nullptr};
    load_layer(p, o->stream, ls, l);
    if (o->tc.on)
      tc_tile_layer(p, o->stream, ls.wq, ls.wk, ls.wv, ls.wo, ls.wg, ls.wu, ls.wd,
                    o->tc.w + (size_t)l * o->tc.off.layer);
  }
  if (cudaStreamSynchronize(o->stream) != cudaSuccess) return cleanup(MCD_ERR_CUDA);
  off = 0;
  at.clear();
  if (!put("c0_head") || !put("final_norm")) return cleanup(MCD_ERR_CUDA);
  RowSrc rh{};
  rh.seg[0] = at["c0_head"];
  rh.seg_rows[0] = p.V;
  rh.nseg = 1;
  rh.src_cols = (int)H;
  tile_kernel<<<1024, 256, 0, o->stream>>>(rh, p.g[MAT_HEAD], p.wdtype, const_cast<uint8_t*>(p.w_head), nullptr);
  to_f32_kernel<<<64, 256, 0, o->stream>>>(at["final_norm"], p.wdtype, H, const_cast<float*>(p.final_norm));
  // row-major tables go straight to their arrays
  auto table = [&](const std::string& name, const uint8_t* dst) {
    auto& gv = given[name];
    return cudaMemcpyAsync(const_cast<uint8_t*>(dst), gv.first, (size_t)gv.second, cudaMemcpyHostToDevice,
                           o->stream) == cudaSuccess;
  };
  if (!table("c0_embed", o->st.c0_table) || !table("text_embed", o->st.text_table) || !table(last, o->st.last_table))
    return cleanup(MCD_ERR_CUDA);
  if (cudaGetLastError() != cudaSuccess) return cleanup(MCD_ERR_CUDA);
  mcd_status s = cleanup(MCD_OK);
  if (cudaGetLastError() != cudaSuccess) return MCD_ERR_CUDA;
  o->weights_loaded = true;
  return s;
}

// Rows 0..n-1 of the prompt (positions 0..n-1) through every layer on the tensor cores,
// leaving their K / V in the cache.
static mcd_status outer_tc_prefill(mcd_outer* o, const int32_t* text_ids, int n) {
  const FrameParams& p = o->fp;
  const OuterTc& t = o->tc;
  const OuterStep& st = o->st;
  cudaStream_t s = o->stream;
  // operand rows of this prompt, not of the capacity: the tiles are shared out over the SMs by
  // the rows there are (255 rows of 640: 144 CTAs instead of 64 to 96 per product)
  const int H = p.H, L = p.L, qd = p.NH * p.D, kvl = p.NKV * st.cap * p.D;
  const int Rtc = tc_operand_rows(n, p.qkv_dim, p.n_cta);
  // every kernel a dependent launch: 2333 us for a 256-token prompt, 2444 with the products alone
  const bool pdl = true;
  pf_set_rows_kernel<<<1, 1, 0, s>>>(t.rows, n);
  tc::launch(pdl, pf_embed_kernel, dim3(n), dim3(128), 0, s, text_ids, t.rows, st.text_table, st.text_vocab, H, t.X,
             p.attn_norm, p.eps, Rtc, t.xn_hi, t.xn_lo, p.err);
  for (int l = 0; l < L; ++l) {
    const uint8_t* wl = t.w + (size_t)l * t.off.layer;
    uint16_t* kc = reinterpret_cast<uint16_t*>(st.kcache) + (size_t)l * kvl;
    uint16_t* vc = reinterpret_cast<uint16_t*>(st.vcache) + (size_t)l * kvl;
    tc_launch_qkv(true, wl + t.off.qkv, t.xn_hi, t.xn_lo, t.qkv, p.qkv_dim, Rtc, H, t.rows, p.err, p.wait_ns, p.n_cta, pdl, s);
    const int vecs = p.NH + 2 * p.NKV;
    tc::launch(pdl, pf_rope_kv_kernel, dim3((n * vecs + 7) / 8), dim3(256), 0, s, t.qkv, tc_qkv_splits(p.qkv_dim, Rtc, H, p.n_cta, true),
               (size_t)Rtc * p.qkv_dim, p.qkv_dim, t.rows, p.NH, p.NKV, p.D, p.qk_norm,
                                                         p.q_norm + (size_t)l * p.D, p.k_norm + (size_t)l * p.D, p.eps,
                                                         st.rope, kc, vc, st.cap, t.q);
    launch_pf_attn(t.q, t.rows, n, p.NH, p.NKV, p.D, kc, vc, st.cap, Rtc, t.att_t, t.att_lo, s);
    tc_launch_resid<true>(wl + t.off.o, t.att_t, t.att_lo, t.part, H, Rtc, qd, t.rows, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid_norm(true, pdl, n, t.X, t.part, qd, Rtc, H, p.n_cta, t.rows, p.eps,
                         NormOut{p.ffn_norm + (size_t)l * H, t.xn_hi, t.xn_lo, nullptr, 0, nullptr}, s);
    tc_launch_gu<true>(wl + t.off.gu, t.xn_hi, t.xn_lo, t.act_t, t.act_lo, Rtc, t.rows, p.F, H, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid<true>(wl + t.off.d, t.act_t, t.act_lo, t.part, H, Rtc, p.F, t.rows, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid_norm(true, pdl, n, t.X, t.part, p.F, Rtc, H, p.n_cta, t.rows, p.eps,
                         NormOut{l + 1 < L ? p.attn_norm + (size_t)(l + 1) * H : nullptr, t.xn_hi, t.xn_lo, nullptr, 0, nullptr}, s);
  }
  MCD_CHECK(cudaGetLastError());
  return MCD_OK;
}

mcd_status mcd_outer_prefill(mcd_outer* o, uint32_t stream_id, int32_t n_tokens, const int32_t* text_ids,
                             int32_t* c0_out) {
  if (!o || !text_ids || n_tokens < 1) return MCD_ERR_INVALID_ARG;
  if (!o->weights_loaded) return MCD_ERR_STATE;
  if (n_tokens > o->st.cap) return MCD_ERR_UNSUPPORTED;
  const int R = prefill_rows(o);
  o->stream_id = stream_id;
  o->st.stream_id = stream_id;
  // every layer on the tensor cores (when the shapes allow), then outer_kernel for the c0 head
  // and the draw of the last row
  const bool batch = o->tc.on && n_tokens >= 2;
  if (batch) {
    mcd_status r = outer_tc_prefill(o, text_ids, n_tokens);
    if (r != MCD_OK) return r;
  }
  for (int s0 = batch ? n_tokens - 1 : 0; s0 < n_tokens; s0 += R) {
    OuterStep s = o->st;
    s.l0 = batch ? o->fp.L : 0;
    s.pos0 = s0;
    s.nr = std::min(R, n_tokens - s0);
    s.head = s0 + s.nr == n_tokens ? 1 : 0;
    s.text_ids = text_ids + s0;
    s.prev_codes = nullptr;
    s.text_id = -1;
    s.c0_out2 = s.head ? c0_out : nullptr;
    s.frame_id = 0;
    s.trace = (o->trace && o->trace_frames > 0) ? o->trace : nullptr;
    mcd_status r = outer_launch(o, s, batch ? o->tc.X + (size_t)(n_tokens - 1) * o->fp.H : nullptr);
    if (r != MCD_OK) return r;
  }
  o->n_tok = n_tokens;
  o->frame = 0;
  o->ready = true;
  return MCD_OK;
}

mcd_status mcd_outer_step(mcd_outer* o, const int32_t* prev_codes, int32_t text_id, int32_t* c0_out) {
  if (!o) return MCD_ERR_INVALID_ARG;
  if (!o->weights_loaded) return MCD_ERR_STATE;
  return outer_step_launch(o, prev_codes, text_id, c0_out);
}

mcd_status mcd_outer_frame_inputs(const mcd_outer* o, const float** cond, const float** c0_emb, const int32_t** c0,
                                  uint32_t* frame_idx) {
  if (!o) return MCD_ERR_INVALID_ARG;
  if (o->frame < 0) return MCD_ERR_STATE;
  if (cond) *cond = o->cond;
  if (c0_emb) *c0_emb = o->c0emb;
  if (c0) *c0 = o->c0_buf;
  if (frame_idx) *frame_idx = (uint32_t)o->frame;
  return MCD_OK;
}

mcd_status mcd_pipeline_frames(mcd_outer* o, int32_t n_frames, const int32_t* text_ids, int32_t* codes_out,
                               mcd_frame_stats* stats) {
  if (!o || n_frames < 0 || (!codes_out && n_frames > 0)) return MCD_ERR_INVALID_ARG;
  if (!o->weights_loaded || !ctx_weights_loaded(o->inner)) return MCD_ERR_STATE;
  if (o->frame < 0) return MCD_ERR_STATE;   // no prompt yet
  const int W = o->P + 1;
  for (int i = 0; i < n_frames; ++i) {
    int32_t* row = codes_out + (size_t)i * W;
    if (o->ready) {
      MCD_CHECK(cudaMemcpyAsync(row, o->c0_buf, sizeof(int32_t), cudaMemcpyDeviceToDevice, o->stream));
    } else {
      const int32_t* prev = i > 0 ? codes_out + (size_t)(i - 1) * W : o->last_codes;
      mcd_status r = outer_step_launch(o, prev, text_ids ? text_ids[i] : -1, row);
      if (r != MCD_OK) return r;
    }
    mcd_status r = mcd_decode_frame(o->inner, o->stream_id, (uint32_t)o->frame, o->cond, nullptr, o->c0emb, row + 1,
                                    stats ? stats + i : nullptr);
    if (r != MCD_OK) return r;
    o->ready = false;
  }
  if (n_frames > 0)
    MCD_CHECK(cudaMemcpyAsync(o->last_codes, codes_out + (size_t)(n_frames - 1) * W, sizeof(int32_t) * W,
                              cudaMemcpyDeviceToDevice, o->stream));
  return MCD_OK;
}

int64_t mcd_outer_trace_floats(const mcd_outer* o) { return o ? (int64_t)o->fp.V + 2LL * o->fp.H : 0; }

mcd_status mcd_outer_set_trace(mcd_outer* o, float* trace, int32_t n_frames) {
  if (!o || n_frames < 0 || (!trace && n_frames > 0)) return MCD_ERR_INVALID_ARG;
  o->trace = n_frames > 0 ? trace : nullptr;
  o->trace_frames = n_frames;
  return MCD_OK;
}

mcd_status mcd_outer_sync(mcd_outer* o) {
  if (!o) return MCD_ERR_INVALID_ARG;
  MCD_CHECK(cudaStreamSynchronize(o->stream));
  int err = 0;
  MCD_CHECK(cudaMemcpy(&err, o->fp.err, sizeof(int), cudaMemcpyDeviceToHost));
  return (mcd_status)err;
}

int64_t mcd_outer_step_weight_bytes(const mcd_outer* o) {
  if (!o) return 0;
  const FrameParams& p = o->fp;
  return (int64_t)p.L * (p.g[MAT_QKV].stride + p.g[MAT_WO].stride + p.g[MAT_GU].stride + p.g[MAT_WD].stride) +
         p.g[MAT_HEAD].stride;
}

}  // extern "C"
