// Batched decoding of many independent streams (up to 128 streams, 512 packed rows per
// call), and of one stream's larger sparse trees: the per-frame draft-and-verify loop of
// arXiv 2609.37007 (Sec. 2.2, Fig. 3) for every stream at once, with the rows of all unfinished
// streams re-packed every call.
//
// With hundreds of rows per call the weight matrices are multiplied as real GEMMs, so this
// path is a sequence of grid-wide kernels per call instead of the persistent frame kernel:
//
//   pack -> embed -> 5 x [QKV GEMM -> attention -> Wo GEMM (+residual) -> gate/up GEMM
//   (SwiGLU) -> down GEMM (+residual)] -> LM-head GEMM (grouped by head) -> top-k -> accept
//
// captured once per context as a CUDA graph: a while node whose body is one call, repeated
// until every stream's frame is complete (a call never emits fewer than one code, so n_pos
// calls always finish a frame).  A small kernel in front of the graph takes the frame's arguments by
// value.  Where the caller itself captures a graph, which cannot embed
// one that holds a conditional node, the n_pos bodies are enqueued one after another; bodies
// after the last active call find no rows and return at once.  Measured with frames of 5 calls of
// 15: 1725 us per frame of 8 streams and 2400 of 128 with the bodies enqueued, 1116 and 1758
// with the while node.  RMSNorm never gets its own pass.  With bf16
// weights whose widths are multiples of 128 (the MultiCodeDecoder's) every product runs on
// the tcgen05 GEMM (mcd_tcgemm.cuh, block kernels in mcd_tcops.cuh): weights and operand
// rows as 128-byte swizzled tiles, TMEM accumulators, the residual products split over k
// into partial sums that one per-row pass folds into the residual stream while it writes
// the next product's normalised operand.  Other shapes use the mma.sync GEMM below (the
// weights in the frame kernel's tiled unit layout, 128 weight rows x 64 packed rows per CTA
// through a 4-stage cp.async pipeline, the norm folded into the operand staging).  Sampling
// and acceptance use the same integer sampler as the frame kernel.
#include <algorithm>
#include <cstring>
#include <vector>

#include "mcd_host.cuh"
#include "mcd_internal.cuh"
#include "mcd_sampler.cuh"
#include "mcd_tcgemm.cuh"
#include "mcd_tcops.cuh"
#include "mcd_tree.cuh"

namespace mcd {

constexpr int kGM = 128;                 // weight rows per GEMM tile (8 m-tiles)
constexpr int kGN = 64;                  // packed rows per GEMM tile (8 n-tiles)
constexpr int kGK = 64;                  // k per pipeline stage (4 k-tiles)
constexpr int kGStages = 4;
constexpr int kGBStride = kGK + 8;       // bf16 per staged operand row (144 B: conflict-free ldmatrix)
constexpr int kGAStage = 32 * 512;       // 8 m-tiles x 4 k-tiles of 512 B
constexpr int kGBStage = kGN * kGBStride * 2;
constexpr int kGStagesHilo = 3;          // with the hi + lo operand: two CTAs per SM still fit
constexpr int kGemmSmem = kGStages * (kGAStage + kGBStage);
constexpr int kGemmSmemHilo = kGStagesHilo * (kGAStage + 2 * kGBStage);
constexpr int kRecSlots = kMaxDraft + 1;   // distributions per packed row (verify + drafts)
constexpr int kBatchQVec = 16;             // query vectors per attention CTA: rows x (q heads per KV head)
constexpr int kBatchKeys = 16;             // keys of a frame: positions 0..15 (c15 is never fed)

// Operand rows: fp32 rows normalised while staged (as one bf16, or as a bf16 hi + lo pair
// carrying about 16 mantissa bits, for the QKV and LM-head products whose errors the
// attention softmax and the sampler see directly), or rows already in bf16.
enum BSrc { BSRC_NORM = 0, BSRC_BF16 = 1, BSRC_NORM_HILO = 2 };
enum Epi { EPI_QKV = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_HEADS = 3 };

struct BatchRow {
  int s, n, pos, id;
  const uint8_t* src;     // layer-0 input row
  int f32;                // src is fp32 (else bf16)
};

struct BatchInfo {
  int M;                  // packed rows of the call
  int n_pairs;            // (row, j) distributions of the call
  int head_rows[16];      // rows reading LM head P (entries in head_list)
  int head_off[16];
  int call, next_call;    // index of the current call of the frame, and of the next one
  unsigned arrived;       // acceptance CTAs done (low half) and streams not complete (high half)
};

// The while node of the frame graph (valid = 0: the calls are enqueued one by one).
struct BatchLoop {
  cudaGraphConditionalHandle handle;
  int valid;
};

// Per-frame arguments, passed by value to batch_begin_kernel: a graph that the caller captures owns them.
struct BatchFrame {
  int S;
  unsigned stream_ids[kMaxBatchStreams];
  unsigned frame_ids[kMaxBatchStreams];
  const float* cond;
  const int* c0;
  const float* c0emb;
  int* codes_out;
  mcd_frame_stats* stats;
  uint8_t* trace;
  TreeDef tree;           // TREE mode (one stream)
};

struct BatchBufs {
  int R;                  // packed-row capacity
  BatchInfo* info;
  BatchFrame* frame;
  BatchRow* rows;         // [R]
  int* sbase;             // [kMaxBatchStreams] first packed row of each stream (-1: inactive)
  int* pairs;             // [R * kRecSlots] (row << 3) | j
  int* head_list;         // [R * kRecSlots] grouped by head
  int* head_slot;         // [R * kRecSlots] LM-head operand row of (row, j), -1: none
  float* X;               // [R][H] residual stream
  float* ss;              // [2L + 1][R] per-row sums of squares of X after each residual write
  float* qkv;             // [R][qkv_dim]; trees: qkv_nz partial sums, qkv_zs floats apart
  int qkv_nz;
  size_t qkv_zs;
  uint16_t* att;          // [R][NH * D] bf16 attention outputs
  uint16_t* act;          // [R][F] bf16 SwiGLU outputs
  float* logits;          // [R][kRecSlots][V]
  TopkRec* recs;          // [2][R][kRecSlots]
  // tensor-core GEMM operands (SW128 tiles of Rtc rows: tc_operand_rows)
  int Rtc;
  uint8_t* xn_hi;         // normalised rows, bf16 (and the low halves for the QKV product)
  uint8_t* xn_lo;
  uint8_t* att_t;         // attention outputs
  uint8_t* act_t;         // SwiGLU outputs
  uint8_t *att_lo, *act_lo;   // TREE mode: their low halves
  float* tree_q;          // TREE mode: [R][NH * D] normalised, rotated queries
  float* part;            // [splits][Rtc][H] k-split partial sums of the residual products
  int Qcap;               // LM-head operand rows: every (row, j) pair, groups padded per head
  uint8_t* hq_hi;         // LM-head operand (normalised rows of the pairs, grouped by head)
  uint8_t* hq_lo;
};

// Weights of the tensor-core GEMMs: per layer the row-major matrices as SW128 tiles.
struct TcWeights {
  uint8_t* arena = nullptr;
  TcLayerOffsets off;                                         // within a layer, layer stride
  uint8_t* heads = nullptr;                                   // [n_pos][V x H] SW128 tiles
};

// ------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ uint16_t f32_to_bf16(float x) { return (uint16_t)bf16_rn_bits(x); }

// Offset (bytes) of 16 x 16 tile (m-tile mt, k-tile kt) in a tiled bf16 matrix.
__device__ __forceinline__ size_t tile_byte_offset(const MatGeom& g, int mt, int kt) {
  const int kcu = kt / g.Ku, ktl = kt - kcu * g.Ku, mbu = mt / g.Mu, mi = mt - mbu * g.Mu;
  const long long u = (long long)kcu * g.n_mb + mbu;
  return (size_t)(((u * g.Mu + mi) * g.Ku) + ktl) * 512;
}

// ------------------------------------------------------------------------------------
// pack: the call's rows, distributions and head groups from every stream's state
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) batch_pack_kernel(FrameParams p, BatchBufs b) {
  __shared__ int s_cnt[16], s_pc[16], s_head[16], s_hcur[16], s_shift[16];
  const BatchFrame* fa = b.frame;
  const int S = fa->S, tid = threadIdx.x;
  if (tid < 16) s_head[tid] = 0;
  int nr = 0, np = 0;
  struct {
    int done, n_rows, pos0, a, code;
    const int* drafts;
  } st;
  if (tid < S) {
    const DevState* q = p.st + tid;
    st.done = q->done;
    st.n_rows = q->n_rows;
    st.pos0 = q->pos0;
    st.a = q->a;
    st.drafts = q->drafts;
    st.code = q->codes[st.a];          // the last code emitted (the first call: c0)
    if (!st.done) {
      nr = st.n_rows;
      for (int n = 0; n < nr; ++n) {
        const int pos = st.pos0 + n;
        if (pos >= 1) np += min(p.K, p.P - pos) + 1;
      }
    }
  }
  // inclusive scans of (rows, pairs) over the streams: within each warp by shuffles, then
  // over the 8 warp totals
  const int lane = tid & 31, warp = tid >> 5;
  int cr = nr, cp = np;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int a = __shfl_up_sync(0xFFFFFFFFu, cr, off), c = __shfl_up_sync(0xFFFFFFFFu, cp, off);
    if (lane >= off) {
      cr += a;
      cp += c;
    }
  }
  if (lane == 31) {
    s_cnt[warp] = cr;
    s_pc[warp] = cp;
  }
  __syncthreads();
  if (warp == 0) {
    int wr = lane < 8 ? s_cnt[lane] : 0, wp = lane < 8 ? s_pc[lane] : 0;
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
      const int a = __shfl_up_sync(0xFFFFFFFFu, wr, off), c = __shfl_up_sync(0xFFFFFFFFu, wp, off);
      if (lane >= off) {
        wr += a;
        wp += c;
      }
    }
    if (lane < 8) {
      s_cnt[8 + lane] = wr;             // inclusive totals through warp `lane`
      s_pc[8 + lane] = wp;
    }
  }
  __syncthreads();
  if (warp > 0) {
    cr += s_cnt[8 + warp - 1];
    cp += s_pc[8 + warp - 1];
  }
  const int base = cr - nr, pbase = cp - np;
  if (tid < S && nr > 0) {
    for (int n = 0; n < nr; ++n) {
      const int pos = st.pos0 + n, r = base + n;
      int id = st.pos0 == 0 ? (n == 0 ? -1 : st.code) : (n == 0 ? st.code : st.drafts[n - 1]);
      BatchRow row;
      row.s = tid;
      row.n = n;
      row.pos = pos;
      if (pos == 0 || (pos == 1 && p.C0V == 0)) {
        row.src = reinterpret_cast<const uint8_t*>((pos == 0 ? fa->cond : fa->c0emb) + (size_t)tid * p.H);
        row.f32 = 1;
      } else {
        const int table = pos - 1;
        if (id < 0 || id >= (table == 0 ? p.C0V : p.V)) {
          atomicCAS(p.err, 0, (int)MCD_ERR_INVALID_ARG);
          id = 0;
        }
        row.src = p.embed + (long long)table * p.embed_stride + (long long)id * p.H * 2;
        row.f32 = 0;
      }
      row.id = id;
      b.rows[r] = row;
      if (pos >= 1) {
        const int kn = min(p.K, p.P - pos);
        for (int j = 0; j <= kn; ++j) atomicAdd(&s_head[pos + j], 1);
      }
    }
  }
  if (tid < kMaxBatchStreams) b.sbase[tid] = (tid < S && nr > 0) ? base : -1;
  __syncthreads();
  if (tid == 0) {
    int off = 0, q = 0;
    for (int P = 0; P < 16; ++P) {
      b.info->head_rows[P] = s_head[P];
      b.info->head_off[P] = off;
      s_hcur[P] = off;
      s_shift[P] = q - off;              // operand rows: groups padded to 16
      off += s_head[P];
      q += (s_head[P] + 15) / 16 * 16;
    }
    b.info->M = s_cnt[8 + 7];
    b.info->n_pairs = s_pc[8 + 7];
    const int call = b.info->next_call;
    b.info->call = call;
    b.info->next_call = call + 1;
  }
  __syncthreads();
  if (tid < S && nr > 0) {
    int pi = pbase;
    for (int n = 0; n < nr; ++n) {
      const int pos = st.pos0 + n, r = base + n;
      const int kn = pos < 1 ? -1 : min(p.K, p.P - pos);
      for (int j = 0; j < kRecSlots; ++j) {
        int slot = -1;
        if (j <= kn) {
          b.pairs[pi++] = (r << 3) | j;
          const int at = atomicAdd(&s_hcur[pos + j], 1);
          b.head_list[at] = (r << 3) | j;
          slot = at + s_shift[pos + j];
        }
        b.head_slot[r * kRecSlots + j] = slot;
      }
    }
  }
}

// embed (tensor-core path): X[r] = the row's input vector, and layer 0's QKV operand.  The sum of
// squares takes the elements in batch_embed_kernel's order; then thread t owns elements 8t..8t+7.
__global__ void __launch_bounds__(256) batch_embed_tc_kernel(FrameParams p, BatchBufs b) {
  __shared__ __align__(16) float row_s[1024];
  __shared__ float sw[8];
  const int r = blockIdx.x, t = threadIdx.x;
  tc::pdl_wait();
  tc::pdl_trigger();
  if (r >= b.info->M) return;
  const BatchRow row = b.rows[r];
  float s = 0.f;
  for (int k = t; k < p.H; k += 256) {
    const float v = row.f32 ? __ldg(reinterpret_cast<const float*>(row.src) + k)
                            : bf16_bits_to_f32(__ldg(reinterpret_cast<const uint16_t*>(row.src) + k));
    b.X[(size_t)r * p.H + k] = v;
    row_s[k] = v;
    s += v * v;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if ((t & 31) == 0) sw[t >> 5] = s;
  __syncthreads();
  if (t >= p.H / 8) return;
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += sw[w];
  float v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = row_s[8 * t + i];
  const NormChunk c = norm_chunk(v, rsqrtf(tot / (float)p.H + p.eps), p.attn_norm, t);
  const size_t off = tc::sw128_offset(b.Rtc, r, t >> 3, t & 7);
  *reinterpret_cast<uint4*>(b.xn_hi + off) = c.hi;
  *reinterpret_cast<uint4*>(b.xn_lo + off) = c.lo;
}

// embed: X[r] = the row's input vector; ss[0][r] = sum of squares.
__global__ void __launch_bounds__(256) batch_embed_kernel(FrameParams p, BatchBufs b) {
  const int r = blockIdx.x;
  if (r >= b.info->M) return;
  const BatchRow row = b.rows[r];
  float s = 0.f;
  for (int k = threadIdx.x; k < p.H; k += blockDim.x) {
    const float v = row.f32 ? __ldg(reinterpret_cast<const float*>(row.src) + k)
                            : bf16_bits_to_f32(__ldg(reinterpret_cast<const uint16_t*>(row.src) + k));
    b.X[(size_t)r * p.H + k] = v;
    s += v * v;
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  __shared__ float sw[8];
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sw[w];
    b.ss[r] = t;
  }
}

// ------------------------------------------------------------------------------------
// GEMM: C[o][row] = sum_k W[o][k] X[row][k] over 128 weight rows x 64 packed rows per CTA
// ------------------------------------------------------------------------------------
struct GemmArgs {
  const uint8_t* W;       // tiled bf16 matrix (heads: head 1; head P at + (P-1) * g.stride)
  MatGeom g;
  // operand rows
  const float* X;         // BSRC_NORM: fp32 rows [R][ldx], scaled by gain[k] / rms(row)
  const float* gain;
  const float* ss;        // per-row sums of squares of X
  const uint16_t* Xb;     // BSRC_BF16: bf16 rows [R][ldx]
  int ldx;
  // outputs
  float* out;             // EPI_QKV: [R][ld]; EPI_RESID: the residual X [R][ld]
  uint16_t* act;          // EPI_SWIGLU: [R][ld]
  int ld;
  float* logits;          // EPI_HEADS: [R][kRecSlots][V]
  const float* head_bias; // EPI_HEADS: [n_pos][K][V]
  int K, V;
  const BatchInfo* info;
  const int* head_list;
  float eps;
};

template <int BSRC, int EPI>
__global__ void __launch_bounds__(256) batch_gemm_kernel(const __grid_constant__ GemmArgs a) {
  constexpr bool kNorm = BSRC != BSRC_BF16, kHilo = BSRC == BSRC_NORM_HILO;
  constexpr int kStages = kHilo ? kGStagesHilo : kGStages;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int s_row[kGN];
  __shared__ int s_j[kGN];
  __shared__ float s_inv[kGN];
  __shared__ float s_ss[kGN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const BatchInfo* info = a.info;
  int n_rows;
  const int* rlist = nullptr;
  const uint8_t* W = a.W;
  int P = 0;
  if (EPI == EPI_HEADS) {
    P = blockIdx.z + 1;
    n_rows = info->head_rows[P];
    rlist = a.head_list + info->head_off[P];
    W += (size_t)(P - 1) * a.g.stride;
  } else {
    n_rows = info->M;
  }
  const int r0 = blockIdx.y * kGN;
  if (r0 >= n_rows) return;
  const MatGeom& g = a.g;
  const int mt0 = blockIdx.x * (kGM / 16);                 // first m-tile of the CTA
  const int n_mt = g.M >> 4;
  const int Kdim = g.K;
  // k-chunks of this CTA: all of them, or (residual GEMMs) slice blockIdx.z of gridDim.z
  int kc0 = 0, kc1 = Kdim / kGK;
  if (EPI != EPI_HEADS && gridDim.z > 1) {
    const int per = (kc1 + gridDim.z - 1) / gridDim.z;
    kc0 = blockIdx.z * per;
    kc1 = min(kc1, kc0 + per);
    if (kc0 >= kc1) return;
  }
  const int n_kc = kc1 - kc0;
  if (tid < kGN) {
    const int i = r0 + tid;
    int r = -1, j = 0;
    if (i < n_rows) {
      if (rlist) {
        const int e = rlist[i];
        r = e >> 3;
        j = e & 7;
      } else {
        r = i;
      }
    }
    s_row[tid] = r;
    s_j[tid] = j;
    if (kNorm) s_inv[tid] = r >= 0 ? rsqrtf(a.ss[r] / (float)Kdim + a.eps) : 0.f;
    s_ss[tid] = 0.f;
  }
  __syncthreads();
  uint8_t* sA = smem;
  uint16_t* sB = reinterpret_cast<uint16_t*>(smem + kStages * kGAStage);
  uint16_t* sBl = sB + (size_t)kStages * kGN * kGBStride;   // lo parts (hi/lo operand)

  // ---- stage loaders ------------------------------------------------------------------------
  auto load_A = [&](int kc, int st) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = tid + 256 * i, t = c >> 5, part = c & 31;
      const int mt = mt0 + (t >> 2), kt = kc * 4 + (t & 3);
      uint8_t* dst = sA + st * kGAStage + t * 512 + part * 16;
      const bool ok = mt < n_mt;
      const uint8_t* src = W + (ok ? tile_byte_offset(g, mt, kt) : 0) + part * 16;
      cp_async16(dst, src, ok ? 16 : 0);
    }
  };
  float4 breg[4];
  auto fetch_B = [&](int kc) {           // BSRC_NORM: fp32 rows into registers
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = tid + 256 * i, rr = c >> 4, q = c & 15;
      const int r = s_row[rr];
      breg[i] = r >= 0 ? __ldcg(reinterpret_cast<const float4*>(a.X + (size_t)r * a.ldx + kc * kGK) + q)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto store_B = [&](int kc, int st) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = tid + 256 * i, rr = c >> 4, q = c & 15, k = kc * kGK + 4 * q;
      const float4 gg = __ldg(reinterpret_cast<const float4*>(a.gain + k));
      const float s = s_inv[rr];
      const float x0 = breg[i].x * gg.x * s, x1 = breg[i].y * gg.y * s, x2 = breg[i].z * gg.z * s,
                  x3 = breg[i].w * gg.w * s;
      const uint32_t h01 = pack_bf16x2(x0, x1), h23 = pack_bf16x2(x2, x3);
      const size_t off = (size_t)st * (kGN * kGBStride) + rr * kGBStride + 4 * q;
      *reinterpret_cast<uint2*>(sB + off) = make_uint2(h01, h23);
      if (kHilo) {
        const uint32_t l01 = pack_bf16x2(x0 - bf16_lo_f32(h01), x1 - bf16_hi_f32(h01));
        const uint32_t l23 = pack_bf16x2(x2 - bf16_lo_f32(h23), x3 - bf16_hi_f32(h23));
        *reinterpret_cast<uint2*>(sBl + off) = make_uint2(l01, l23);
      }
    }
  };
  auto load_B16 = [&](int kc, int st) {   // BSRC_BF16: cp.async
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int c = tid + 256 * i, rr = c >> 3, ch = c & 7;
      const int r = s_row[rr];
      const uint16_t* src = a.Xb + (size_t)(r >= 0 ? r : 0) * a.ldx + kc * kGK + ch * 8;
      cp_async16(sB + (size_t)st * (kGN * kGBStride) + rr * kGBStride + ch * 8, src, r >= 0 ? 16 : 0);
    }
  };

  // ---- main loop ------------------------------------------------------------------------------
  const int wm = (warp & 3) * 2;          // the warp's first m-tile within the CTA tile
  const int wn = (warp >> 2) * 4;         // its first n-tile
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;

#pragma unroll
  for (int st = 0; st < kStages - 1; ++st) {
    if (st < n_kc) {
      load_A(kc0 + st, st);
      if (!kNorm) {
        load_B16(kc0 + st, st);
      } else {
        fetch_B(kc0 + st);
        store_B(kc0 + st, st);
      }
    }
    cp_async_commit();
  }
  for (int it = 0; it < n_kc; ++it) {
    const int st = it % kStages;
    const int nk = it + kStages - 1;
    if (kNorm && nk < n_kc) fetch_B(kc0 + nk);
    cp_async_wait<kStages - 2>();
    __syncthreads();
    const uint8_t* A = sA + st * kGAStage;
    const uint16_t* B = sB + (size_t)st * (kGN * kGBStride);
    const uint16_t* Bl = sBl + (size_t)st * (kGN * kGBStride);
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) {
      const uint4 a0 = *reinterpret_cast<const uint4*>(A + ((wm + 0) * 4 + kt) * 512 + lane * 16);
      const uint4 a1 = *reinterpret_cast<const uint4*>(A + ((wm + 1) * 4 + kt) * 512 + lane * 16);
#pragma unroll
      for (int hp = 0; hp < 2; ++hp) {
        uint32_t bf[4];
        const int row = (wn + 2 * hp + (lane >> 4)) * 8 + (lane & 7);
        const int kk = kt * 16 + ((lane >> 3) & 1) * 8;
        ldmatrix_x4(bf, B + row * kGBStride + kk);
        mma_bf16_16816(acc[0][2 * hp], a0, bf[0], bf[1]);
        mma_bf16_16816(acc[0][2 * hp + 1], a0, bf[2], bf[3]);
        mma_bf16_16816(acc[1][2 * hp], a1, bf[0], bf[1]);
        mma_bf16_16816(acc[1][2 * hp + 1], a1, bf[2], bf[3]);
        if (kHilo) {
          ldmatrix_x4(bf, Bl + row * kGBStride + kk);
          mma_bf16_16816(acc[0][2 * hp], a0, bf[0], bf[1]);
          mma_bf16_16816(acc[0][2 * hp + 1], a0, bf[2], bf[3]);
          mma_bf16_16816(acc[1][2 * hp], a1, bf[0], bf[1]);
          mma_bf16_16816(acc[1][2 * hp + 1], a1, bf[2], bf[3]);
        }
      }
    }
    // stage nk % kStages was last read in iteration it - 1, which every warp has left
    if (nk < n_kc) {
      const int sn = nk % kStages;
      load_A(kc0 + nk, sn);
      if (!kNorm)
        load_B16(kc0 + nk, sn);
      else
        store_B(kc0 + nk, sn);
    }
    cp_async_commit();
  }
  cp_async_wait<0>();

  // ---- epilogue ----------------------------------------------------------------------------
  // acc[i][j]: m-tile wm + i, n-tile wn + j; c0/c1 -> weight row +lane/4, packed rows
  // 2(lane%4) + {0,1}; c2/c3 -> weight row +lane/4 + 8.
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int mt = mt0 + wm + i;
    if (mt >= n_mt) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {      // packed row 2(lane%4) + h
        const int rr = (wn + j) * 8 + 2 * (lane & 3) + h;
        const int r = s_row[rr];
        if (r < 0) continue;
        const float v_lo = acc[i][j][h], v_hi = acc[i][j][2 + h];   // weight rows +lane/4, +lane/4 + 8
        const int o = mt * 16 + (lane >> 2);
        if (EPI == EPI_QKV) {
          a.out[(size_t)r * a.ld + o] = v_lo;
          a.out[(size_t)r * a.ld + o + 8] = v_hi;
        } else if (EPI == EPI_RESID) {   // k-slices of several CTAs add into the residual
          float* xr = a.out + (size_t)r * a.ld;
          atomicAdd(xr + o, v_lo);
          atomicAdd(xr + o + 8, v_hi);
        } else if (EPI == EPI_SWIGLU) {
          const int jj = mt * 8 + (lane >> 2);       // gate row (tile row lane/4), up row (+8)
          const float gt = v_lo;
          a.act[(size_t)r * a.ld + jj] = f32_to_bf16(gt / (1.0f + __expf(-gt)) * v_hi);
        } else {
          const int jd = s_j[rr];
          float* lg = a.logits + ((size_t)r * kRecSlots + jd) * a.V;
          float b0 = 0.f, b1 = 0.f;
          if (jd >= 1) {
            const float* bias = a.head_bias + ((size_t)(P - 1) * a.K + (jd - 1)) * a.V;
            b0 = __ldg(bias + o);
            b1 = __ldg(bias + o + 8);
          }
          lg[o] = v_lo + b0;
          lg[o + 8] = v_hi + b1;
        }
      }
    }
  }
}

// LM heads.  The (row, j) pairs of the call are grouped by head (head_list); group P starts at
// operand row qoff(P) = the sum of the earlier groups rounded up to 16 rows, and its columns
// are split into n_t = ceil(rows / kHeadTileMax) tiles of equal width (a multiple of 16), so
// every tile of the product belongs to one head and is no wider than the group needs.
constexpr int kHeadTileMax = 176;      // three 60 KB ring stages with the hi + lo operand
__host__ __device__ __forceinline__ int tc_head_tiles(int rows) { return (rows + kHeadTileMax - 1) / kHeadTileMax; }
__host__ __device__ __forceinline__ int tc_head_width(int rows) {
  const int nt = tc_head_tiles(rows);
  return nt ? ((rows + nt - 1) / nt + 15) / 16 * 16 : 0;
}
// Grid bound over the tiles of every group: at most (K + 1) pairs per packed row.
inline int tc_head_grid_x(int R, int K, int n_pos) { return (R * (K + 1) + kHeadTileMax - 1) / kHeadTileMax + n_pos; }

// Logits of every pair: tile blockIdx.x (counted over the groups in head order) of head P's
// group times head P's weights (m-tile blockIdx.y), plus the draft-offset bias for j >= 1.
constexpr int kHeadsThreads = 256;     // eight warps: two per TMEM lane quarter in the epilogue
__global__ void __launch_bounds__(kHeadsThreads, 1) tc_heads_kernel(const tc::GemmArgs g, const uint8_t* w_heads,
                                                                    size_t head_bytes, float* logits,
                                                                    const float* head_bias, const BatchInfo* info,
                                                                    const int* head_list, int n_pos, int K, int V) {
  int P = 0, qoff = 0, c0 = 0, nw = 0, rows = 0;
  for (int i = 1, o = 0, t = blockIdx.x; i <= n_pos; ++i) {
    const int r = info->head_rows[i], nt = tc_head_tiles(r);
    if (P == 0 && t < nt) {
      const int w = tc_head_width(r);
      P = i;
      qoff = o;
      rows = r;
      c0 = t * w;
      nw = min(w, (r + 15) / 16 * 16 - c0);
    }
    t -= nt;
    o += (r + 15) / 16 * 16;
  }
  if (P == 0) return;                                   // past the last tile (uniform per CTA)
  const int off = info->head_off[P];
  // the tile's (row, j) entries in shared memory and this thread's bias of every offset j
  // (the epilogue's output row m is fixed per thread), loaded while the products run
  __shared__ int s_entry[kHeadTileMax];
  for (int i = threadIdx.x; i < nw; i += blockDim.x) s_entry[i] = c0 + i < rows ? head_list[off + c0 + i] : -1;
  const int m_t = blockIdx.y * tc::kBM + ((threadIdx.x >> 5) & 3) * 32 + (threadIdx.x & 31);
  float bias_j[kMaxDraft];
#pragma unroll
  for (int q = 0; q < kMaxDraft; ++q)
    bias_j[q] = q < K ? __ldg(head_bias + ((size_t)(P - 1) * K + q) * V + m_t) : 0.f;
  tc::GemmArgs ga = g;
  ga.a = w_heads + (size_t)(P - 1) * head_bytes;
  ga.n_active = nullptr;
  const int q0 = qoff + c0;
  tc::gemm_tile<kHeadTileMax, true>(
      ga,
      [&](int m, int n, float v) {
        const int e = s_entry[n - q0];
        if (e >= 0) {
          const int r = e >> 3, j = e & 7;
          float bias = 0.f;
#pragma unroll
          for (int q = 1; q <= kMaxDraft; ++q)
            if (j == q) bias = bias_j[q - 1];
          logits[((size_t)r * kRecSlots + j) * V + m] = v + bias;
        }
      },
      q0, nw);
}

// Per-row sums of squares of the residual stream after a residual GEMM (one warp per row):
// the next RMSNorm's 1/rms, applied while the next GEMM stages its operand.
__global__ void __launch_bounds__(256) batch_rowss_kernel(const float* X, int H, float* ss, const BatchInfo* info) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= info->M) return;
  const float4* x = reinterpret_cast<const float4*>(X + (size_t)r * H);
  float s = 0.f;
  for (int i = lane; i < (H >> 2); i += 32) {
    const float4 v = __ldcg(x + i);
    s += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if (lane == 0) ss[r] = s;
}

// ------------------------------------------------------------------------------------
// attention: one CTA per (stream, KV head).  At most 32 registers per thread, so that seven
// CTAs share an SM and the 1024 CTAs of 128 streams run as one wave.
// ------------------------------------------------------------------------------------
// Attention of the call's rows of stream s = blockIdx.x for KV head g = blockIdx.y and its
// `group` query heads (QK-norm, RoPE, causal softmax over the stream's cached positions and
// its new rows); outputs to the Wo product's operand.  Phases, with block barriers between
// them: (A) every input (the nr x group query vectors, cached and new K / V rows, RoPE rows
// of the new positions, QK-norm gains) copied into shared memory as 16-byte cp.async chunks,
// all in flight; (B) one warp per new q / k vector applies QK-norm and RoPE in registers and
// stores the new rows' K / V to the cache; (C) one warp per query vector: lanes 2j, 2j + 1
// score key j over interleaved chunks, softmax across the warp, then four output dims per
// lane summed over the keys.  Row and head of a query vector come from a table, not a
// division.
__global__ void __launch_bounds__(256, 7) batch_attn_kernel(FrameParams p, BatchBufs b, int layer) {
  tc::pdl_wait();
  tc::pdl_trigger();
  const int s = blockIdx.x, g = blockIdx.y;
  if (s >= b.frame->S) return;
  const int base = b.sbase[s];
  if (base < 0) return;
  const DevState* st = p.st + s;
  const int nr = st->n_rows, pos0 = st->pos0;
  const int D = p.D, half = D >> 1, group = p.NH / p.NKV, nq = nr * group;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lg4 = D == 128 ? 5 : 4, D4 = 1 << lg4;                // 16-byte chunks per row
  __shared__ __align__(16) float qs[kBatchQVec][132];
  __shared__ __align__(16) float ks[kBatchKeys][132];
  __shared__ __align__(16) float vs[kBatchKeys][128];
  __shared__ __align__(16) float2 cs[kMaxRows][64];               // RoPE (cos, sin) of the new rows
  __shared__ __align__(16) float gq[128], gk[128];
  __shared__ int q_row[kBatchQVec], q_head[kBatchQVec];
  const size_t cache_off = (size_t)s * p.kv_stride + ((size_t)layer * p.NKV + g) * p.kv_slots * D;
  const int nk = pos0 + nr;
  if (tid < nq) {
    q_row[tid] = tid / group;
    q_head[tid] = g * group + tid % group;
  }
  __syncthreads();
  // ---- (A) loads ----------------------------------------------------------------------
  {
    const int e_q = nq << lg4, e_k = e_q + (nk << lg4), e_v = e_k + (nk << lg4);
    const int e_cs = e_v + (nr << lg4), e_g = e_cs + (p.qk_norm ? 2 << lg4 : 0);
    for (int i = tid; i < e_g; i += 256) {
      const int ch = i & (D4 - 1);
      const float* src;
      float* dst;
      if (i < e_q) {
        const int qi = i >> lg4;
        src = b.qkv + (size_t)(base + q_row[qi]) * p.qkv_dim + q_head[qi] * D;
        dst = qs[qi];
      } else if (i < e_v) {
        const bool isv = i >= e_k;
        const int j = (i - (isv ? e_k : e_q)) >> lg4;
        if (j < pos0)
          src = (isv ? p.vcache : p.kcache) + cache_off + (size_t)j * D;
        else
          src = b.qkv + (size_t)(base + j - pos0) * p.qkv_dim + p.NH * D + (isv ? p.NKV * D : 0) + g * D;
        dst = isv ? vs[j] : ks[j];
      } else if (i < e_cs) {
        const int n = (i - e_v) >> lg4;
        src = reinterpret_cast<const float*>(p.rope + (size_t)(pos0 + n) * half);
        dst = reinterpret_cast<float*>(cs[n]);
      } else {
        const int w = (i - e_cs) >> lg4;
        src = (w == 0 ? p.q_norm : p.k_norm) + (size_t)layer * D;
        dst = w == 0 ? gq : gk;
      }
      cpa16(dst + 4 * ch, src + 4 * ch);
    }
    cpa_wait_all();
  }
  __syncthreads();
  // ---- (B) QK-norm + RoPE of the queries and the new keys; new K / V cached --------------
  const int nd = D >> 5;
  for (int vi = warp; vi < nq + nr; vi += 8) {
    const bool isq = vi < nq;
    const int n = isq ? q_row[vi] : vi - nq;
    float* row = isq ? qs[vi] : ks[pos0 + n];
    float x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = i < nd ? row[lane + 32 * i] : 0.f;
    if (p.qk_norm) {
      float ss = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) ss += x[i] * x[i];
#pragma unroll
      for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
      const float scl = rsqrtf(ss / (float)D + p.eps);
      const float* gg = isq ? gq : gk;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nd) x[i] = x[i] * scl * gg[lane + 32 * i];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i < nd / 2) {
        const float2 r = cs[n][lane + 32 * i];
        const float a0 = x[i], b0 = x[i + nd / 2];
        x[i] = a0 * r.x - b0 * r.y;
        x[i + nd / 2] = b0 * r.x + a0 * r.y;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < nd) row[lane + 32 * i] = x[i];
    if (!isq) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nd) {
          p.kcache[cache_off + (size_t)(pos0 + n) * D + lane + 32 * i] = x[i];
          p.vcache[cache_off + (size_t)(pos0 + n) * D + lane + 32 * i] = vs[pos0 + n][lane + 32 * i];
        }
    }
  }
  __syncthreads();
  // ---- (C) one warp per query vector: scores (lanes 2j, 2j+1), softmax, P.V ---------------
  const float scale = rsqrtf((float)D);
  for (int qi = warp; qi < nq; qi += 8) {
    const int n = q_row[qi], h = q_head[qi], npos = pos0 + n + 1;
    const int j = lane >> 1, hf = lane & 1;
    const bool live = j < npos;                      // causal: keys 0..pos0+n
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    if (live) {
      const float4* q4 = reinterpret_cast<const float4*>(qs[qi]) + hf;
      const float4* k4 = reinterpret_cast<const float4*>(ks[j]) + hf;
#pragma unroll 4
      for (int c2 = 0; c2 < (D4 >> 1); ++c2) {
        const float4 q = q4[2 * c2], k = k4[2 * c2];
        a0 += q.x * k.x;
        a1 += q.y * k.y;
        a2 += q.z * k.z;
        a3 += q.w * k.w;
      }
    }
    float sc = (a0 + a1) + (a2 + a3);
    sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 1);
    sc = live ? sc * scale : -INFINITY;
    float mx = sc;
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    const float e = live ? __expf(sc - mx) : 0.f;
    float sum = e;                                   // lanes of one parity hold every key once
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
    const float pj = e / sum;
    const int d0 = 4 * lane;                         // four dims per lane
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int jj = 0; jj < npos; ++jj) {
      const float w = __shfl_sync(0xFFFFFFFFu, pj, 2 * jj);
      if (d0 < D) {
        const float4 v = *reinterpret_cast<const float4*>(&vs[jj][d0]);
        acc.x += w * v.x;
        acc.y += w * v.y;
        acc.z += w * v.z;
        acc.w += w * v.w;
      }
    }
    if (d0 < D) {
      const int f = h * D + d0;
      const uint2 packed = make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
      if (b.att_t)        // the Wo product's operand, SW128 tiles (tensor-core path)
        *reinterpret_cast<uint2*>(b.att_t + tc::sw128_offset(b.Rtc, base + n, f >> 6, (f & 63) >> 3) + (f & 7) * 2) =
            packed;
      else
        *reinterpret_cast<uint2*>(b.att + (size_t)(base + n) * p.NH * D + f) = packed;
    }
  }
}

// ------------------------------------------------------------------------------------
// top-k of every (row, j) distribution of the call; then the acceptance per stream
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kConsumerThreads) batch_topk_kernel(FrameParams p, BatchBufs b) {
  __shared__ __align__(16) uint8_t smem_raw[sizeof(TopkScratch)];
  TopkScratch& ts = *reinterpret_cast<TopkScratch*>(smem_raw);
  const int call = b.info->call, n_pair_ctas = (int)gridDim.x - b.R;
  if ((int)blockIdx.x >= n_pair_ctas) {     // packed row r's verify logits into an optional trace
    const int r = (int)blockIdx.x - n_pair_ctas;
    if (!b.frame->trace || call >= kMaxCalls || r >= b.info->M || b.head_slot[r * kRecSlots] < 0) return;
    const BatchRow row = b.rows[r];
    uint8_t* tb = b.frame->trace + (size_t)row.s * p.trace_stride + sizeof(mcd_call_trace) * kMaxCalls;
    float* dst = reinterpret_cast<float*>(tb) + ((size_t)call * kMaxRows + row.n) * p.V;
    if (p.draft_mode == MCD_DRAFT_TREE)
      dst = reinterpret_cast<float*>(tb + (size_t)2 * kMaxCalls * kMaxRows * p.V * 4 + sizeof(mcd_tree_trace) * kMaxCalls) +
            ((size_t)call * kMaxTreeRows + row.n) * p.V;
    copy_logits(dst, b.logits + (size_t)r * kRecSlots * p.V, p.V);
    return;
  }
  if ((int)blockIdx.x >= b.info->n_pairs) return;
  const int e = b.pairs[blockIdx.x], r = e >> 3, j = e & 7;
  const int greedy = (j > 0 && p.draft_mode == MCD_DRAFT_GREEDY) ? 1 : 0;
  TopkRec* recs = b.recs + (size_t)(call & 1) * b.R * kRecSlots;
  block_topk(b.logits + ((size_t)r * kRecSlots + j) * p.V, p.V, p.top_k, p.T, greedy, ts,
             recs + (size_t)r * kRecSlots + j);
}

// End of a stream's acceptance (thread 0 of its CTA; `more`: its frame is not complete): the CTA
// that arrives last decides whether the while node runs another call.  The counter is back at
// zero for the next call.
__device__ __forceinline__ void batch_call_end(const FrameParams& p, const BatchBufs& b, const BatchLoop& loop, int call,
                                               bool more) {
  if (!loop.valid) return;
  const unsigned mine = 1u + (more ? 0x10000u : 0u);
  const unsigned all = atomicAdd(&b.info->arrived, mine) + mine;
  if ((all & 0xFFFFu) != gridDim.x) return;
  b.info->arrived = 0u;
  cudaGraphSetConditional(loop.handle, (all >> 16) != 0u && call + 1 < p.P ? 1u : 0u);
}

__global__ void __launch_bounds__(kConsumerThreads) batch_accept_kernel(FrameParams p, BatchBufs b, BatchLoop loop) {
  const int s = blockIdx.x, call = b.info->call;
  const BatchFrame* fa = b.frame;
  const int base = s < fa->S ? b.sbase[s] : -1;
  if (base < 0) {                       // no such stream, or its frame is complete
    if (threadIdx.x == 0) batch_call_end(p, b, loop, call, false);
    return;
  }
  DevState* st = p.st + s;
  __shared__ AcceptResult s_res;
  __shared__ int s_next[kMaxDraft], s_old[kMaxDraft + 1];
  const int a = st->a, n_d = st->n_d, pos0 = st->pos0, n_rows = st->n_rows, qrow = st->q_row;
  if (threadIdx.x <= kMaxDraft) s_old[threadIdx.x] = (int)threadIdx.x < n_d ? st->drafts[threadIdx.x] : -1;
  __syncthreads();
  const unsigned sid = fa->stream_ids[s], fid = fa->frame_ids[s];
  const TopkRec* cur = b.recs + (size_t)(call & 1) * b.R * kRecSlots;
  const TopkRec* prev = b.recs + (size_t)((call + 1) & 1) * b.R * kRecSlots;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // every record the acceptance reads, staged in shared memory first: p of positions
  // a+1 .. (the bonus row only when its position exists), then q of the drafts
  __shared__ __align__(16) TopkRec srec[2 * kMaxDraft + 1];
  const int n_p = a + 1 + n_d <= p.P ? n_d + 1 : n_d;
  stage_records(srec, n_p + n_d, p.top_k, [&](int r) {
    return r < n_p ? cur + (size_t)(base + a + 1 + r - pos0) * kRecSlots : prev + (size_t)qrow * kRecSlots + 1 + (r - n_p);
  });
  __syncthreads();
  // every draft's accept test and the residual draw it would take as the first rejection in
  // parallel (warp i for draft i), warp n_d the bonus draw; then the chain is read off in
  // order, taking the same decisions as testing the drafts one after another
  __shared__ int s_ok[kMaxDraft + 1], s_alt[kMaxDraft + 1];
  if (warp <= n_d) {
    const int i = warp, pos = a + 1 + i;
    if (i < n_d) {
      const TopkRec* pr = srec + i;
      const TopkRec* qr = srec + n_p + i;
      const int d = s_old[i];
      const unsigned long long wp = warp_weight(pr, d), wq = warp_weight(qr, d);
      const unsigned long long U = uniform_U(p.seed, sid, fid, call, pos, PURPOSE_ACCEPT);
      const bool ok = lt128(mul128x64(mul64(U, wq), pr->S), shl53(wp * qr->S));
      const int alt = ok ? -1 : warp_residual(pr, qr, uniform_U(p.seed, sid, fid, call, pos, PURPOSE_TARGET));
      if (lane == 0) {
        s_ok[i] = ok ? 1 : 0;
        s_alt[i] = alt;
      }
    } else if (pos <= p.P) {
      const int bonus = warp_draw(srec + n_d, uniform_U(p.seed, sid, fid, call, pos, PURPOSE_TARGET));
      if (lane == 0) s_alt[i] = bonus;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    AcceptResult r;
    r.n_acc = 0;
    r.n_emit = 0;
    bool rejected = false;
    for (int i = 0; i < n_d && !rejected; ++i) {
      if (s_ok[i]) {
        r.emitted[r.n_emit++] = s_old[i];
        ++r.n_acc;
      } else {
        r.emitted[r.n_emit++] = s_alt[i];
        rejected = true;
      }
    }
    if (!rejected && a + 1 + n_d <= p.P) r.emitted[r.n_emit++] = s_alt[n_d];
    s_res = r;
  }
  __syncthreads();
  const int n_emit = s_res.n_emit, n_acc = s_res.n_acc;
  const int a_new = a + n_emit, m = a_new - pos0, n_next = min(p.K, p.P - a_new);
  // next drafts from the draft distributions of row m, whose head emitted the last code
  stage_records(srec, n_next, p.top_k, [&](int r) { return cur + (size_t)(base + m) * kRecSlots + 1 + r; });
  __syncthreads();
  for (int j = 1 + warp; j <= n_next; j += kConsumerWarps) {
    const unsigned long long U = uniform_U(p.seed, sid, fid, call, a_new + j, PURPOSE_DRAFT);
    const int d = warp_draw(srec + (j - 1), U);
    if (lane == 0) s_next[j - 1] = d;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int* codes_out = fa->codes_out ? fa->codes_out + (size_t)s * p.P : nullptr;
    for (int t = 0; t < n_emit; ++t) {
      st->codes[a + 1 + t] = s_res.emitted[t];
      if (codes_out) codes_out[a + t] = s_res.emitted[t];
    }
    for (int j = 0; j < n_next; ++j) st->drafts[j] = s_next[j];
    for (int t = 0; t < n_emit; ++t) st->emitted_last[t] = s_res.emitted[t];
    const int p_lo = a + 1, p_hi = min(p.P, pos0 + n_rows - 1 + p.K);
    const int calls = st->calls + 1, heads = st->heads_read + p_hi - p_lo + 1;
    const int kvr = st->kv_rows + pos0 + n_rows, rf = st->rows_fed + n_rows;
    const int drafted = st->drafted + n_d, accepted = st->accepted + n_acc;
    st->n_emit_last = n_emit;
    st->n_acc_last = n_acc;
    st->a = a_new;
    st->n_d = n_next;
    st->pos0 = a_new + 1;
    st->n_rows = min(n_next + 1, p.P - a_new);
    st->top_pos = st->pos0 + st->n_rows - 1;
    st->round = call + 1;
    st->first_head_row = 0;
    st->calls = calls;
    st->heads_read = heads;
    st->kv_rows = kvr;
    st->rows_fed = rf;
    st->drafted = drafted;
    st->accepted = accepted;
    st->call = call + 1;
    st->done = a_new >= p.P ? 1 : 0;
    st->q_row = base + m;     // the next call's q: this call's records of packed row base + m
    if (a_new >= p.P && fa->stats) {
      mcd_frame_stats* fs = fa->stats + s;
      fs->calls = calls;
      fs->codes = a_new;
      fs->drafted = drafted;
      fs->accepted = accepted;
      fs->status = *(volatile int*)p.err;
      fs->heads_read = heads;
      fs->kv_rows = kvr;
      fs->rows_fed = rf;
    }
  }
  // optional trace, in the frame kernel's layout
  if (fa->trace && call < kMaxCalls) {
    uint8_t* tb = fa->trace + (size_t)s * p.trace_stride;
    mcd_call_trace* tr = reinterpret_cast<mcd_call_trace*>(tb) + call;
    if (threadIdx.x < kMaxRows) {
      const int t = threadIdx.x;
      tr->input_ids[t] = t < n_rows ? b.rows[base + t].id : -1;
      tr->drafts[t] = t < n_d ? s_old[t] : -1;
      tr->emitted[t] = t < n_emit ? s_res.emitted[t] : -1;
      tr->next_drafts[t] = t < n_next ? s_next[t] : -1;
      if (t == 0) {
        tr->a = a;
        tr->n_rows = n_rows;
        tr->pos0 = pos0;
        tr->n_drafts = n_d;
        tr->n_acc = n_acc;
        tr->n_emit = n_emit;
        tr->n_next = n_next;
        tr->draft_row = m;
      }
    }
    // the draft logits (the verify logits were copied beside the distributions)
    float* dlog = reinterpret_cast<float*>(tb + sizeof(mcd_call_trace) * kMaxCalls) + (size_t)kMaxCalls * kMaxRows * p.V +
                  (size_t)call * kMaxRows * p.V;
    const float* lg = b.logits + ((size_t)(base + m) * kRecSlots + 1) * p.V;
    copy_logits(dlog, lg, n_next * p.V);               // consecutive rows on both sides
  }
  if (threadIdx.x == 0) batch_call_end(p, b, loop, call, a_new < p.P);
}

// ------------------------------------------------------------------------------------
// tree calls: one stream, every row of the call (up to 65) in one pass
// ------------------------------------------------------------------------------------
// Row m >= 1 of a tree call is node m - 1 (the nodes whose candidates exist, a prefix of the
// breadth-first list), row 0 the last emitted code; the first call feeds [cond, c0].  K / V of
// the call's rows go to cache slots kMaxPos + m (row 0: its position) until the acceptance
// step moves the kept ones.  Every product takes hi + lo operands.
__device__ __forceinline__ int tree_row_slot(const DevState* st, int r) {
  return st->pos0 == 0 ? r : (r == 0 ? st->pos0 : kMaxPos + r);
}

// pack: one thread per row.
__global__ void __launch_bounds__(128) batch_tree_pack_kernel(FrameParams p, BatchBufs b) {
  __shared__ int s_head[16], s_hcur[16], s_shift[16], s_rows, s_pairs;
  const BatchFrame* fa = b.frame;
  const TreeDef& tree = fa->tree;
  const DevState* st = p.st;
  const int r = threadIdx.x;
  if (r < 16) s_head[r] = 0;
  if (r == 0) s_rows = s_pairs = 0;
  __syncthreads();
  const int a = st->a, pos0 = st->pos0;
  int pos = -1, id = -1;
  if (!st->done) {
    if (pos0 == 0) {
      if (r < 2) {
        pos = r;
        id = r == 0 ? -1 : st->codes[0];
      }
    } else if (r == 0) {
      pos = pos0;
      id = st->codes[a];
    } else if (r <= tree.n && tree.depth[r - 1] <= st->n_d && a + tree.depth[r - 1] < p.P) {
      const int d = tree.depth[r - 1];
      pos = pos0 + d;
      id = p.tree_cand[(d - 1) * kMaxTreeRank + tree.rank[r - 1]];
    }
  }
  const int kn = pos >= 1 ? min(p.K, p.P - pos) : -1;         // draft heads of the row (-1: none at all)
  if (pos >= 0) {
    atomicAdd(&s_rows, 1);
    BatchRow row;
    row.s = 0;
    row.n = r;
    row.pos = pos;
    if (pos == 0 || (pos == 1 && p.C0V == 0)) {
      row.src = reinterpret_cast<const uint8_t*>(pos == 0 ? fa->cond : fa->c0emb);
      row.f32 = 1;
    } else {
      const int table = pos - 1;
      if (id < 0 || id >= (table == 0 ? p.C0V : p.V)) {
        atomicCAS(p.err, 0, (int)MCD_ERR_INVALID_ARG);
        id = 0;
      }
      row.src = p.embed + (long long)table * p.embed_stride + (long long)id * p.H * 2;
      row.f32 = 0;
    }
    row.id = id;
    b.rows[r] = row;
    for (int j = 0; j <= kn; ++j) atomicAdd(&s_head[pos + j], 1);
  }
  __syncthreads();
  if (r == 0) {
    int off = 0, q = 0;
    for (int P = 0; P < 16; ++P) {
      b.info->head_rows[P] = s_head[P];
      b.info->head_off[P] = off;
      s_hcur[P] = off;
      s_shift[P] = q - off;              // operand rows: groups padded to 16
      off += s_head[P];
      q += (s_head[P] + 15) / 16 * 16;
    }
    b.info->M = s_rows;
    b.info->n_pairs = off;
    const int call = b.info->next_call;
    b.info->call = call;
    b.info->next_call = call + 1;
  }
  __syncthreads();
  for (int j = 0; j < kRecSlots && pos >= 0; ++j) {
    int slot = -1;
    if (j <= kn) {
      b.pairs[atomicAdd(&s_pairs, 1)] = (r << 3) | j;
      const int at = atomicAdd(&s_hcur[pos + j], 1);
      b.head_list[at] = (r << 3) | j;
      slot = at + s_shift[pos + j];
    }
    b.head_slot[r * kRecSlots + j] = slot;
  }
}

// QK-norm + RoPE of every row's query and key heads; K and V to the row's cache slot, the
// queries to tree_q.  One warp per (row, vector), lane holding dims lane + 32 i.
__global__ void __launch_bounds__(256) batch_tree_rope_kernel(FrameParams p, BatchBufs b, int layer) {
  const int vecs = p.NH + 2 * p.NKV, w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int r = w / vecs, vi = w - r * vecs;
  if (r >= b.info->M) return;
  const int NH = p.NH, D = p.D, nd = D >> 5;
  const int kind = vi < NH ? 0 : (vi < NH + p.NKV ? 1 : 2), h = kind == 0 ? vi : (kind == 1 ? vi - NH : vi - NH - p.NKV);
  const float* src = b.qkv + (size_t)r * p.qkv_dim + vi * D;
  float x[4];
  qkv_row(x, src, nd, lane, b.qkv_nz, b.qkv_zs);
  if (kind < 2) {
    if (p.qk_norm) {
      float ss = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) ss += x[i] * x[i];
#pragma unroll
      for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, off);
      const float scl = rsqrtf(ss / (float)D + p.eps);
      const float* gg = (kind == 0 ? p.q_norm : p.k_norm) + (size_t)layer * D;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nd) x[i] = x[i] * scl * __ldg(gg + lane + 32 * i);
    }
    const float2* rope = p.rope + (size_t)b.rows[r].pos * (D >> 1);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i < nd / 2) {
        const float2 cs = __ldg(rope + lane + 32 * i);
        const float e = x[i], f = x[i + nd / 2];
        x[i] = e * cs.x - f * cs.y;
        x[i + nd / 2] = f * cs.x + e * cs.y;
      }
    }
  }
  float* dst = kind == 0 ? b.tree_q + ((size_t)r * NH + h) * D
                         : (kind == 1 ? p.kcache : p.vcache) +
                               (((size_t)layer * p.NKV + h) * p.kv_slots + tree_row_slot(p.st, r)) * D;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (i < nd) dst[lane + 32 * i] = x[i];
}

// Attention of one (row, query head) per warp over the cache: the committed positions, row 0, the
// row's ancestors and itself (the sparse tree mask of Fig. 2); the first call is causal.  At
// most 15 + 1 + 7 keys: lane j holds key j's slot and score, four dims per lane of every K and V
// row, eight rows in flight.  Outputs as hi + lo halves to the Wo product's operand.
__global__ void __launch_bounds__(256) batch_tree_attn_kernel(FrameParams p, BatchBufs b, int layer) {
  tc::pdl_wait();
  tc::pdl_trigger();
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int NH = p.NH, D = p.D, r = w / NH, h = w - r * NH, g = h / (NH / p.NKV);
  if (r >= b.info->M) return;
  const DevState* st = p.st;
  const int pos0 = st->pos0;
  const unsigned long long anc = pos0 > 0 && r > 0 ? b.frame->tree.anc[r - 1] : 0ull;
  const int nk = pos0 == 0 ? r + 1 : pos0 + 1 + __popcll(anc);
  int slot = lane;                                   // committed positions, row 0's, the first call's rows
  if (pos0 > 0 && lane > pos0 && lane < nk) {        // ancestor number lane - pos0 - 1, in tree order
    unsigned long long m = anc;
    for (int i = pos0 + 1; i < lane; ++i) m &= m - 1ull;
    slot = kMaxPos + __ffsll((long long)m);          // node i is row i + 1
  }
  const size_t head_off = ((size_t)layer * p.NKV + g) * p.kv_slots * D;
  const int d0 = 4 * lane;
  const bool own = d0 < D;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 q = own ? __ldcg(reinterpret_cast<const float4*>(b.tree_q + ((size_t)r * NH + h) * D + d0)) : z;
  float score = -INFINITY;
  for (int jb = 0; jb < nk; jb += 8) {
    float4 kv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int sl = __shfl_sync(0xFFFFFFFFu, slot, (jb + i) & 31);
      kv[i] = jb + i < nk && own ? __ldcg(reinterpret_cast<const float4*>(p.kcache + head_off + (size_t)sl * D + d0)) : z;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float s = (q.x * kv[i].x + q.y * kv[i].y) + (q.z * kv[i].z + q.w * kv[i].w);
#pragma unroll
      for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      if (lane == jb + i && jb + i < nk) score = s * rsqrtf((float)D);
    }
  }
  float mx = score;
#pragma unroll
  for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
  const float e = lane < nk ? __expf(score - mx) : 0.f;
  float sum = e;
#pragma unroll
  for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
  const float pj = e / sum;
  float4 acc = z;
  for (int jb = 0; jb < nk; jb += 8) {
    float4 kv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int sl = __shfl_sync(0xFFFFFFFFu, slot, (jb + i) & 31);
      kv[i] = jb + i < nk && own ? __ldcg(reinterpret_cast<const float4*>(p.vcache + head_off + (size_t)sl * D + d0)) : z;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float wgt = __shfl_sync(0xFFFFFFFFu, pj, (jb + i) & 31);
      if (jb + i < nk) {
        acc.x += wgt * kv[i].x;
        acc.y += wgt * kv[i].y;
        acc.z += wgt * kv[i].z;
        acc.w += wgt * kv[i].w;
      }
    }
  }
  if (own) {
    const int f = h * D + d0;
    const size_t off = tc::sw128_offset(b.Rtc, r, f >> 6, (f & 63) >> 3) + (f & 7) * 2;
    const uint2 hi = make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
    *reinterpret_cast<uint2*>(b.att_t + off) = hi;
    *reinterpret_cast<uint2*>(b.att_lo + off) = make_uint2(
        pack_bf16x2(acc.x - bf16_lo_f32(hi.x), acc.y - bf16_hi_f32(hi.x)),
        pack_bf16x2(acc.z - bf16_lo_f32(hi.y), acc.w - bf16_hi_f32(hi.y)));
  }
}

// Acceptance of a tree call (mcd_tree.cuh) and the while node's condition.  The call is one pass;
// heads_read counts its heads once per 32 rows all the same, so that a frame's statistics do not
// depend on which kernels ran it.
__global__ void __launch_bounds__(kConsumerThreads) batch_tree_accept_kernel(FrameParams p, BatchBufs b, BatchLoop loop) {
  __shared__ DevState st;
  __shared__ int cand[kMaxDraft][kMaxTreeRank];
  const int call = b.info->call;
  for (int i = threadIdx.x; i < (int)(sizeof(DevState) / 4); i += kConsumerThreads)
    reinterpret_cast<int*>(&st)[i] = __ldcg(reinterpret_cast<const int*>(p.st) + i);
  for (int i = threadIdx.x; i < kMaxDraft * kMaxTreeRank; i += kConsumerThreads)
    cand[i / kMaxTreeRank][i % kMaxTreeRank] = __ldcg(p.tree_cand + i);
  __syncthreads();
  if (!st.done) {
    const BatchFrame* fa = b.frame;
    const int heads = (min(p.P, st.top_pos + p.K) - st.a) * ((st.n_rows + kMaxCols - 1) / kMaxCols);
    const TreeCall t{&fa->tree, &st, cand, b.recs + (size_t)(call & 1) * b.R * kRecSlots, b.logits, heads, 1,
                     fa->stream_ids[0], fa->frame_ids[0], fa->codes_out, fa->stats, fa->trace};
    const TreeDrafts d = accept_tree_call(p, t);
    if (fa->trace && st.round < kMaxCalls) {           // consecutive rows on both sides
      float* dlog = reinterpret_cast<float*>(fa->trace + sizeof(mcd_call_trace) * kMaxCalls) +
                    ((size_t)kMaxCalls + st.round) * kMaxRows * p.V;
      copy_logits(dlog, b.logits + ((size_t)d.row * (kMaxDraft + 1) + 1) * p.V, d.n * p.V);
    }
  }
  if (threadIdx.x == 0) batch_call_end(p, b, loop, call, !__ldcg(&p.st->done));
}

// Start of a frame: its arguments to *frame, every stream's state and the call counters reset.
__global__ void __launch_bounds__(256) batch_begin_kernel(const __grid_constant__ BatchFrame f, BatchFrame* frame,
                                                          BatchInfo* info, DevState* st, int c0_vocab) {
  static_assert(sizeof(BatchFrame) % 4 == 0, "copied in words");
  for (int i = threadIdx.x; i < (int)(sizeof(BatchFrame) / 4); i += blockDim.x)
    reinterpret_cast<int*>(frame)[i] = reinterpret_cast<const int*>(&f)[i];
  for (int s = threadIdx.x; s < f.S; s += blockDim.x) init_stream_state(st + s, c0_vocab > 0 ? f.c0[s] : -1);
  if (threadIdx.x == 0) {
    info->next_call = 0;
    info->arrived = 0u;
  }
}

}  // namespace mcd

// ------------------------------------------------------------------------------------
// Host side: buffers, the per-context graph, one launch per frame
// ------------------------------------------------------------------------------------
namespace mcd {

struct BatchState {
  BatchBufs b;
  int max_streams = 0;
  bool use_tc = false;        // QKV, Wo, gate/up and down on the tcgen05 GEMM
  bool tree = false;          // TREE mode: one stream's tree calls
  TcWeights tw;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaStream_t cap = nullptr;
  std::vector<void*> allocs;
};

template <class T>
static cudaError_t batch_alloc(BatchState* bs, T** p, size_t bytes) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, bytes < 256 ? 256 : bytes);
  if (e != cudaSuccess) return e;
  bs->allocs.push_back(q);
  *p = static_cast<T*>(q);
  return cudaSuccess;
}

void batch_destroy(BatchState* bs) {
  if (!bs) return;
  if (bs->exec) cudaGraphExecDestroy(bs->exec);
  if (bs->graph) cudaGraphDestroy(bs->graph);
  if (bs->cap) cudaStreamDestroy(bs->cap);
  for (void* q : bs->allocs) cudaFree(q);
  delete bs;
}

int batch_rows(const FrameParams& p, int max_streams) { return max_streams * std::max(p.K + 1, 2); }

// From 5 streams on, a launch the persistent frame kernel could take runs faster on the
// tensor-core batched path (measured on GB300: +10 % at 5 streams, +17 % at 8) when the
// shapes allow the tcgen05 GEMMs and one attention CTA holds a stream's query vectors.
bool batch_prefers(const FrameParams& p, int n_streams) {
  return n_streams >= kBatchMinStreams && tc_block_supported(p) &&
         std::max(p.K + 1, 2) * (p.NH / p.NKV) <= kBatchQVec && p.draft_mode != MCD_DRAFT_NOISY_TARGET &&
         p.draft_mode != MCD_DRAFT_TREE;
}

// A tree call of 1 + nodes rows is one pass here; the persistent frame kernel pays for every row and
// starts a new pass every 32.  Measured per call when the line was drawn, frame kernel / batched
// (us): 15 nodes 247 / 255,
// 16 nodes 280 / 255, 17 nodes 281 / 256, 31 nodes 330 / 262, 32 nodes 459 / 262, 64 nodes 737 / 273.
// Every operand is hi + lo here, at any row count (the frame kernel's are single bf16 values above
// 16 rows: 1.7e-3 off a 64-bit evaluation at 32 nodes against 3.6e-6).  A captured frame
// enqueues the bodies of all 15 calls, of which 5 to 7 did something in these frames, frame kernel /
// batched (us): 16 nodes 1848 / 2329, 24 nodes 1546 / 1942, 31 nodes 1627 / 1953, 32 nodes (two
// passes) 2302 / 1954, 64 nodes 3661 / 2014.
bool batch_tree_supported(const FrameParams& p) {
  return p.draft_mode == MCD_DRAFT_TREE && tc_block_supported(p) && p.V % tc::kBM == 0;
}
bool batch_tree_prefers(int nodes, bool captured) {
  return nodes >= (captured ? kBatchMinCapturedTreeNodes : kBatchMinTreeNodes);
}

mcd_status batch_create(const FrameParams& p, int max_streams, BatchState** out) {
  *out = nullptr;
  BatchState* bs = new BatchState();
  bs->max_streams = max_streams;
  bs->tree = p.draft_mode == MCD_DRAFT_TREE;
  auto fail = [&](mcd_status s) {
    batch_destroy(bs);
    return s;
  };
  BatchBufs& b = bs->b;
  memset(&b, 0, sizeof(b));
  const int rows = bs->tree ? kMaxTreeRows : batch_rows(p, max_streams);
  const int R = (rows + kGN - 1) / kGN * kGN;
  b.R = R;
  cudaError_t e;
#define BATCH_ALLOC(ptr, bytes)                                                        \
  do {                                                                                 \
    if ((e = batch_alloc(bs, &(ptr), (bytes))) != cudaSuccess) return fail(cuda_status(e)); \
  } while (0)
  BATCH_ALLOC(b.info, sizeof(BatchInfo));
  BATCH_ALLOC(b.frame, sizeof(BatchFrame));
  BATCH_ALLOC(b.rows, sizeof(BatchRow) * R);
  BATCH_ALLOC(b.sbase, sizeof(int) * kMaxBatchStreams);
  BATCH_ALLOC(b.pairs, sizeof(int) * R * kRecSlots);
  BATCH_ALLOC(b.head_list, sizeof(int) * R * kRecSlots);
  BATCH_ALLOC(b.head_slot, sizeof(int) * R * kRecSlots);
  BATCH_ALLOC(b.X, sizeof(float) * R * p.H);
  BATCH_ALLOC(b.ss, sizeof(float) * (2 * p.L + 1) * R);
  BATCH_ALLOC(b.att, sizeof(uint16_t) * R * p.NH * p.D);
  BATCH_ALLOC(b.act, sizeof(uint16_t) * R * p.F);
  BATCH_ALLOC(b.logits, sizeof(float) * R * kRecSlots * p.V);
  BATCH_ALLOC(b.recs, sizeof(TopkRec) * 2 * R * kRecSlots);
  bs->use_tc = tc_block_supported(p);
  if (bs->use_tc) {
    const int Rtc = tc_operand_rows(rows, p.qkv_dim, p.n_cta);
    b.Rtc = Rtc;
    b.qkv_nz = tc_qkv_splits(p.qkv_dim, Rtc, p.H, p.n_cta, bs->tree);
    b.qkv_zs = (size_t)Rtc * p.qkv_dim;
    BATCH_ALLOC(b.qkv, sizeof(float) * b.qkv_nz * b.qkv_zs);
    if (bs->tree) {
      BATCH_ALLOC(b.att_lo, (size_t)Rtc * p.NH * p.D * 2);
      BATCH_ALLOC(b.act_lo, (size_t)Rtc * p.F * 2);
      BATCH_ALLOC(b.tree_q, sizeof(float) * (size_t)R * p.NH * p.D);
    }
    BATCH_ALLOC(b.xn_hi, (size_t)Rtc * p.H * 2);
    BATCH_ALLOC(b.xn_lo, (size_t)Rtc * p.H * 2);
    BATCH_ALLOC(b.att_t, (size_t)Rtc * p.NH * p.D * 2);
    BATCH_ALLOC(b.act_t, (size_t)Rtc * p.F * 2);
    BATCH_ALLOC(b.part, sizeof(float) * tc_part_floats(Rtc, p.H));
    if (p.V % tc::kBM == 0) {
      b.Qcap = (R * kRecSlots + p.P * (kTcBN - 1) + kTcBN - 1) / kTcBN * kTcBN;
      BATCH_ALLOC(b.hq_hi, (size_t)b.Qcap * p.H * 2);
      BATCH_ALLOC(b.hq_lo, (size_t)b.Qcap * p.H * 2);
      BATCH_ALLOC(bs->tw.heads, (size_t)p.P * p.V * p.H * 2);
    }
    TcWeights& tw = bs->tw;
    tw.off = tc_layer_offsets(p);
    BATCH_ALLOC(tw.arena, tw.off.layer * p.L);
  } else {
    b.qkv_nz = 1;
    BATCH_ALLOC(b.qkv, sizeof(float) * R * p.qkv_dim);
  }
#undef BATCH_ALLOC
  if ((e = cudaMemset(b.info, 0, sizeof(BatchInfo))) != cudaSuccess) return fail(cuda_status(e));
  if ((e = cudaStreamCreateWithFlags(&bs->cap, cudaStreamNonBlocking)) != cudaSuccess) return fail(cuda_status(e));
  void* gemms[] = {(void*)batch_gemm_kernel<BSRC_NORM_HILO, EPI_QKV>, (void*)batch_gemm_kernel<BSRC_BF16, EPI_RESID>,
                   (void*)batch_gemm_kernel<BSRC_NORM, EPI_SWIGLU>, (void*)batch_gemm_kernel<BSRC_NORM_HILO, EPI_HEADS>};
  for (void* fn : gemms)
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmemHilo) != cudaSuccess)
      return fail(MCD_ERR_CUDA);
  if (bs->use_tc &&
      ((bs->tree ? tc_block_set_smem<true>() : tc_block_set_smem<false>()) != cudaSuccess ||
       cudaFuncSetAttribute(tc_heads_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            tc::Layout<kHeadTileMax, true>::kSmemBytes) != cudaSuccess))
    return fail(MCD_ERR_CUDA);
  *out = bs;
  return MCD_OK;
}

// The tcgen05 GEMMs' copies of layer l's matrices (row-major bf16 sources, device).
mcd_status batch_load_layer(BatchState* bs, const FrameParams& p, cudaStream_t st, const LayerSrc& src, int l) {
  if (!bs || !bs->use_tc) return MCD_OK;
  tc_tile_layer(p, st, src.wq, src.wk, src.wv, src.wo, src.wg, src.wu, src.wd, bs->tw.arena + (size_t)l * bs->tw.off.layer);
  return cudaGetLastError() == cudaSuccess ? MCD_OK : MCD_ERR_CUDA;
}

// The tcgen05 GEMM's copy of LM head P (row-major bf16 [V][H] source, device).
mcd_status batch_load_head(BatchState* bs, const FrameParams& p, cudaStream_t st, const uint8_t* src, int P) {
  if (!bs || !bs->tw.heads) return MCD_OK;
  tc_weight_tile_kernel<<<512, 256, 0, st>>>(reinterpret_cast<const uint16_t*>(src), p.V, p.H, p.V, 0, p.V, 0,
                                             bs->tw.heads + (size_t)(P - 1) * p.V * p.H * 2);
  return cudaGetLastError() == cudaSuccess ? MCD_OK : MCD_ERR_CUDA;
}

static GemmArgs gemm_args(const FrameParams& p, const BatchBufs& b) {
  GemmArgs a;
  memset(&a, 0, sizeof(a));
  a.info = b.info;
  a.head_list = b.head_list;
  a.eps = p.eps;
  a.K = p.K;
  a.V = p.V;
  return a;
}

// k-slices of a residual GEMM: enough CTAs for about two per SM, at least 4 k-chunks each.
static int split_k(dim3 grid, int K, int n_sm) {
  const int ctas = (int)(grid.x * grid.y), chunks = K / kGK;
  int z = 1;
  while (ctas * z < 2 * n_sm && chunks / (2 * z) >= 4) z *= 2;
  return z;
}

// LM heads on the tensor cores, tiles grouped by head (operand: the last residual pass).
static void enqueue_heads(const FrameParams& p, const BatchState* bs, cudaStream_t s) {
  const BatchBufs& b = bs->b;
  const int R = b.R, H = p.H;
  const tc::GemmArgs g{nullptr, b.hq_hi, b.hq_lo, p.V, b.Qcap, H, nullptr, p.err, p.wait_ns, false, 0};
  tc_heads_kernel<<<dim3(tc_head_grid_x(R, p.K, p.P), p.V / tc::kBM, 1), kHeadsThreads,
                    tc::Layout<kHeadTileMax, true>::kSmemBytes, s>>>(g, bs->tw.heads, (size_t)p.V * H * 2, b.logits, p.head_bias,
                                                                     b.info, b.head_list, p.P, p.K, p.V);
}

// The operand a residual pass leaves: the next layer's QKV operand, or after the last layer the LM
// heads' (where they run on the tensor cores; the general heads read the rows' sums of squares).
static NormOut after_layer(const FrameParams& p, const BatchState* bs, int l) {
  const BatchBufs& b = bs->b;
  if (l + 1 < p.L) return NormOut{p.attn_norm + (size_t)(l + 1) * p.H, b.xn_hi, b.xn_lo, nullptr, 0, nullptr};
  if (bs->tw.heads) return NormOut{p.final_norm, b.hq_hi, b.hq_lo, b.head_slot, b.Qcap, nullptr};
  return NormOut{nullptr, nullptr, nullptr, nullptr, 0, b.ss + (size_t)(2 * p.L) * b.R};
}

// Every kernel of one call, in stream order on `s`.
static cudaError_t enqueue_call(const FrameParams& p, const BatchState* bs, const BatchLoop& loop, cudaStream_t s) {
  const BatchBufs& b = bs->b;
  const int R = b.R, L = p.L, H = p.H;
  const dim3 blk(256);
  // The products are dependent launches (their weights stream in while the kernel before them
  // runs); the small kernels between them start the ordinary way.  Frames of 5 calls, 8 / 128
  // streams, when this was introduced: 1235 / 1868 us with ordinary launches, 1169 / 1805 with
  // dependent products, 1208 / 1810 with every kernel dependent, 1275 / 1901 with only the small ones.  Outside the while
  // node the last bodies of a frame are empty: no prefetch there.
  const bool pdl = loop.valid != 0;
  batch_pack_kernel<<<1, 256, 0, s>>>(p, b);
  if (bs->use_tc) batch_embed_tc_kernel<<<R, 256, 0, s>>>(p, b);
  else batch_embed_kernel<<<R, 256, 0, s>>>(p, b);
  for (int l = 0; l < L && bs->use_tc; ++l) {
    const uint8_t* wl = bs->tw.arena + (size_t)l * bs->tw.off.layer;
    const int Rtc = b.Rtc, qd = p.NH * p.D;
    const int* M = &b.info->M;
    // RMSNorm -> QKV (hi + lo operand, written by the embedding or the previous layer's last
    // residual pass)
    tc_launch_qkv(false, wl + bs->tw.off.qkv, b.xn_hi, b.xn_lo, b.qkv, p.qkv_dim, Rtc, H, M, p.err, p.wait_ns, p.n_cta, pdl, s);
    batch_attn_kernel<<<dim3(bs->max_streams, p.NKV), blk, 0, s>>>(p, b, l);      // -> att_t
    // Wo (k-split partials) -> residual, the gate/up operand
    tc_launch_resid<false>(wl + bs->tw.off.o, b.att_t, nullptr, b.part, H, Rtc, qd, M, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid_norm(false, false, R, b.X, b.part, qd, Rtc, H, p.n_cta, M, p.eps,
                         NormOut{p.ffn_norm + (size_t)l * H, b.xn_hi, nullptr, nullptr, 0, nullptr}, s);
    // gate/up -> SwiGLU (into the down product's operand)
    tc_launch_gu<false>(wl + bs->tw.off.gu, b.xn_hi, nullptr, b.act_t, nullptr, Rtc, M, p.F, H, p.err, p.wait_ns, p.n_cta, pdl, s);
    // down (k-split partials) -> residual, the next operand
    tc_launch_resid<false>(wl + bs->tw.off.d, b.act_t, nullptr, b.part, H, Rtc, p.F, M, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid_norm(false, false, R, b.X, b.part, p.F, Rtc, H, p.n_cta, M, p.eps, after_layer(p, bs, l), s);
  }
  for (int l = 0; l < L && !bs->use_tc; ++l) {
    {   // RMSNorm -> QKV
      GemmArgs a = gemm_args(p, b);
      a.W = p.w_qkv + (size_t)l * p.g[MAT_QKV].stride;
      a.g = p.g[MAT_QKV];
      a.X = b.X;
      a.ldx = H;
      a.gain = p.attn_norm + (size_t)l * H;
      a.ss = b.ss + (size_t)(2 * l) * R;
      a.out = b.qkv;
      a.ld = p.qkv_dim;
      batch_gemm_kernel<BSRC_NORM_HILO, EPI_QKV>
          <<<dim3(a.g.M / kGM + (a.g.M % kGM != 0), R / kGN), blk, kGemmSmemHilo, s>>>(a);
    }
    batch_attn_kernel<<<dim3(bs->max_streams, p.NKV), blk, 0, s>>>(p, b, l);
    {   // Wo + residual
      GemmArgs a = gemm_args(p, b);
      a.W = p.w_wo + (size_t)l * p.g[MAT_WO].stride;
      a.g = p.g[MAT_WO];
      a.Xb = b.att;
      a.ldx = p.NH * p.D;
      a.out = b.X;
      a.ld = H;
      const dim3 grid(a.g.M / kGM + (a.g.M % kGM != 0), R / kGN);
      batch_gemm_kernel<BSRC_BF16, EPI_RESID><<<dim3(grid.x, grid.y, split_k(grid, a.g.K, p.n_cta)), blk, kGemmSmem, s>>>(a);
      batch_rowss_kernel<<<R / 8, blk, 0, s>>>(b.X, H, b.ss + (size_t)(2 * l + 1) * R, b.info);
    }
    {   // RMSNorm -> gate/up -> SwiGLU
      GemmArgs a = gemm_args(p, b);
      a.W = p.w_gu + (size_t)l * p.g[MAT_GU].stride;
      a.g = p.g[MAT_GU];
      a.X = b.X;
      a.ldx = H;
      a.gain = p.ffn_norm + (size_t)l * H;
      a.ss = b.ss + (size_t)(2 * l + 1) * R;
      a.act = b.act;
      a.ld = p.F;
      batch_gemm_kernel<BSRC_NORM, EPI_SWIGLU><<<dim3(a.g.M / kGM + (a.g.M % kGM != 0), R / kGN), blk, kGemmSmem, s>>>(a);
    }
    {   // down + residual
      GemmArgs a = gemm_args(p, b);
      a.W = p.w_wd + (size_t)l * p.g[MAT_WD].stride;
      a.g = p.g[MAT_WD];
      a.Xb = b.act;
      a.ldx = p.F;
      a.out = b.X;
      a.ld = H;
      const dim3 grid(a.g.M / kGM + (a.g.M % kGM != 0), R / kGN);
      batch_gemm_kernel<BSRC_BF16, EPI_RESID><<<dim3(grid.x, grid.y, split_k(grid, a.g.K, p.n_cta)), blk, kGemmSmem, s>>>(a);
      batch_rowss_kernel<<<R / 8, blk, 0, s>>>(b.X, H, b.ss + (size_t)(2 * l + 2) * R, b.info);
    }
  }
  if (bs->tw.heads) {
    enqueue_heads(p, bs, s);
  } else {   // final RMSNorm -> LM heads, one grid slice per head
    GemmArgs a = gemm_args(p, b);
    a.W = p.w_head;
    a.g = p.g[MAT_HEAD];
    a.X = b.X;
    a.ldx = H;
    a.gain = p.final_norm;
    a.ss = b.ss + (size_t)(2 * L) * R;
    a.logits = b.logits;
    a.head_bias = p.head_bias;
    batch_gemm_kernel<BSRC_NORM_HILO, EPI_HEADS>
        <<<dim3(a.g.M / kGM + (a.g.M % kGM != 0), R / kGN, p.P), blk, kGemmSmemHilo, s>>>(a);
  }
  batch_topk_kernel<<<R * (p.K + 1) + R, kConsumerThreads, 0, s>>>(p, b);
  batch_accept_kernel<<<bs->max_streams, kConsumerThreads, 0, s>>>(p, b, loop);
  return cudaGetLastError();
}

// Every kernel of one tree call.
static cudaError_t enqueue_tree_call(const FrameParams& p, const BatchState* bs, const BatchLoop& loop, cudaStream_t s) {
  const BatchBufs& b = bs->b;
  const int L = p.L, H = p.H, Rtc = b.Rtc, qd = p.NH * p.D;
  const dim3 blk(256);
  const bool pdl = loop.valid != 0;
  const int* M = &b.info->M;
  batch_tree_pack_kernel<<<1, 128, 0, s>>>(p, b);
  batch_embed_tc_kernel<<<kMaxTreeRows, 256, 0, s>>>(p, b);
  for (int l = 0; l < L; ++l) {
    const uint8_t* wl = bs->tw.arena + (size_t)l * bs->tw.off.layer;
    tc_launch_qkv(true, wl + bs->tw.off.qkv, b.xn_hi, b.xn_lo, b.qkv, p.qkv_dim, Rtc, H, M, p.err, p.wait_ns, p.n_cta, pdl, s);
    batch_tree_rope_kernel<<<(kMaxTreeRows * (p.NH + 2 * p.NKV) + 7) / 8, blk, 0, s>>>(p, b, l);
    batch_tree_attn_kernel<<<(kMaxTreeRows * p.NH + 7) / 8, blk, 0, s>>>(p, b, l);
    tc_launch_resid<true>(wl + bs->tw.off.o, b.att_t, b.att_lo, b.part, H, Rtc, qd, M, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid_norm(true, false, kMaxTreeRows, b.X, b.part, qd, Rtc, H, p.n_cta, M, p.eps,
                         NormOut{p.ffn_norm + (size_t)l * H, b.xn_hi, b.xn_lo, nullptr, 0, nullptr}, s);
    tc_launch_gu<true>(wl + bs->tw.off.gu, b.xn_hi, b.xn_lo, b.act_t, b.act_lo, Rtc, M, p.F, H, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid<true>(wl + bs->tw.off.d, b.act_t, b.act_lo, b.part, H, Rtc, p.F, M, p.err, p.wait_ns, p.n_cta, pdl, s);
    tc_launch_resid_norm(true, false, kMaxTreeRows, b.X, b.part, p.F, Rtc, H, p.n_cta, M, p.eps, after_layer(p, bs, l), s);
  }
  enqueue_heads(p, bs, s);
  batch_topk_kernel<<<kMaxTreeRows * (p.K + 1) + b.R, kConsumerThreads, 0, s>>>(p, b);
  batch_tree_accept_kernel<<<1, kConsumerThreads, 0, s>>>(p, b, loop);
  return cudaGetLastError();
}

// The frame's graph: the while node over the calls.
static cudaError_t build_graph(const FrameParams& p, BatchState* bs) {
  cudaStream_t s = bs->cap;
  cudaError_t e = cudaGraphCreate(&bs->graph, 0);
  if (e != cudaSuccess) return e;
  cudaGraphNode_t loop_node = nullptr;
  BatchLoop loop{0, 1};
  e = cudaGraphConditionalHandleCreate(&loop.handle, bs->graph, 1, cudaGraphCondAssignDefault);
  if (e != cudaSuccess) return e;
  cudaGraphNodeParams np = {};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = loop.handle;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  if ((e = cudaGraphAddNode(&loop_node, bs->graph, nullptr, nullptr, 0, &np)) != cudaSuccess) return e;
  e = cudaStreamBeginCaptureToGraph(s, np.conditional.phGraph_out[0], nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  const cudaError_t q = (bs->tree ? enqueue_tree_call : enqueue_call)(p, bs, loop, s);
  cudaGraph_t body = nullptr;
  e = cudaStreamEndCapture(s, &body);
  if (q != cudaSuccess || e != cudaSuccess) return q != cudaSuccess ? q : e;
  return cudaGraphInstantiate(&bs->exec, bs->graph, 0);
}

mcd_status batch_prepare(BatchState* bs, const FrameParams& p, const cudaStream_t* upload) {
  if (bs->exec) return MCD_OK;
  // the caller may be capturing a stream of its own: nothing here touches it
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  MCD_CHECK(cudaThreadExchangeStreamCaptureMode(&mode));
  const cudaError_t e = build_graph(p, bs);
  (void)cudaThreadExchangeStreamCaptureMode(&mode);
  if (e != cudaSuccess) {
    if (bs->graph) cudaGraphDestroy(bs->graph);
    bs->graph = nullptr;
    return cuda_status(e);
  }
  if (upload) MCD_CHECK(cudaGraphUpload(bs->exec, *upload));
  return MCD_OK;
}

mcd_status batch_decode(BatchState* bs, const FrameParams& p, cudaStream_t stream, int n, const uint32_t* stream_ids,
                        const uint32_t* frame_ids, const float* cond, const int32_t* c0, const float* c0_emb,
                        int32_t* codes_out, mcd_frame_stats* stats, uint8_t* trace) {
  if (n < 1 || n > bs->max_streams) return MCD_ERR_INVALID_ARG;
  // a graph with a conditional node cannot become part of a graph that the caller captures
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  MCD_CHECK(cudaStreamIsCapturing(stream, &capturing));
  const bool unrolled = capturing == cudaStreamCaptureStatusActive;
  if (!unrolled) {
    const mcd_status r = batch_prepare(bs, p);
    if (r != MCD_OK) return r;
  }
  BatchFrame f;
  memset(&f, 0, sizeof(f));
  f.S = n;
  for (int i = 0; i < n; ++i) {
    f.stream_ids[i] = stream_ids[i];
    f.frame_ids[i] = frame_ids[i];
  }
  f.cond = cond;
  f.c0 = c0;
  f.c0emb = c0_emb;
  f.codes_out = codes_out;
  f.stats = stats;
  f.trace = trace;
  f.tree = p.tree;
  batch_begin_kernel<<<1, 256, 0, stream>>>(f, bs->b.frame, bs->b.info, p.st, p.C0V);
  MCD_CHECK(cudaGetLastError());
  if (!unrolled) {
    MCD_CHECK(cudaGraphLaunch(bs->exec, stream));
    return MCD_OK;
  }
  for (int call = 0; call < p.P; ++call) MCD_CHECK((bs->tree ? enqueue_tree_call : enqueue_call)(p, bs, BatchLoop{0, 0}, stream));
  return MCD_OK;
}

}  // namespace mcd
