// The transformer-block products of many rows on the tcgen05 GEMM (mcd_tcgemm.cuh), shared by
// the batched path (many streams per call) and the CodeDecoder prompt prefill: with bf16
// weights and qkv_dim, F, H multiples of 128 the QKV, Wo, gate/up and down products run on
// the tensor cores.  Their operand rows are written as SW128 tiles by the kernel that
// produces them: the normalised rows by the pass that also folds the k-split partial sums of
// the previous residual product into the residual stream (tc_resid_norm_kernel), the
// attention outputs by the attention kernel, the SwiGLU outputs by the gate/up epilogue.
// Every kernel reads its live row count from device memory (*nrows, rows beyond it are
// neither computed nor written).  Internal linkage: each translation unit has its copy.
#pragma once
#include <type_traits>

#include "mcd_internal.cuh"
#include "mcd_tcgemm.cuh"

namespace mcd {
namespace {


// Eight elements 8t.. of a row, times gain and 1/rms, as the hi (and with lo also the remainder)
// halves of a product's operand.
struct NormChunk {
  uint4 hi, lo;
};
__device__ __forceinline__ NormChunk norm_chunk(const float (&x)[8], float inv_rms, const float* __restrict__ gain, int t) {
  const float4 g0 = __ldg(reinterpret_cast<const float4*>(gain + 8 * t));
  const float4 g1 = __ldg(reinterpret_cast<const float4*>(gain + 8 * t + 4));
  const float v[8] = {x[0] * g0.x * inv_rms, x[1] * g0.y * inv_rms, x[2] * g0.z * inv_rms, x[3] * g0.w * inv_rms,
                      x[4] * g1.x * inv_rms, x[5] * g1.y * inv_rms, x[6] * g1.z * inv_rms, x[7] * g1.w * inv_rms};
  uint32_t h[4], l[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    h[q] = pack_bf16x2(v[2 * q], v[2 * q + 1]);
    l[q] = pack_bf16x2(v[2 * q] - bf16_lo_f32(h[q]), v[2 * q + 1] - bf16_hi_f32(h[q]));
  }
  return NormChunk{make_uint4(h[0], h[1], h[2], h[3]), make_uint4(l[0], l[1], l[2], l[3])};
}
// Sum of s over the CTA's 128 threads (one barrier).
__device__ __forceinline__ float block_sum128(float s) {
  __shared__ float red[4];
#pragma unroll
  for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  return red[0] + red[1] + red[2] + red[3];
}

// Row-major bf16 [rows][K] -> an SW128-tiled matrix of R rows (weight load): source row r
// goes to row row0 + (r / grp) * gstride + r % grp (grp = rows: row0 + r).
__global__ void tc_weight_tile_kernel(const uint16_t* __restrict__ src, int rows, int K, int R, int row0, int grp,
                                      int gstride, uint8_t* __restrict__ dst) {
  const long long total = (long long)rows * (K / 8);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / (K / 8)), ch = (int)(i % (K / 8));
    const int dr = row0 + (r / grp) * gstride + r % grp;
    *reinterpret_cast<uint4*>(dst + tc::sw128_offset(R, dr, ch >> 3, ch & 7)) =
        *reinterpret_cast<const uint4*>(src + (size_t)r * K + (size_t)ch * 8);
  }
}

constexpr int kTcBN = 128;        // packed rows per tile: QKV (hi + lo operand), Wo, down
constexpr int kTcSplit = 16;      // k-splits of the residual products (at most)
constexpr int kTcQkvSplit = 4;    // k-splits of the QKV product (at most)
// A product's column tiles and k-splits at Rtc operand rows.
//
// Trees and prompts (free_k): up to 128 rows a product is its weight stream, and a few column
// tiles of 128-row weight tiles would leave most SMs without a share of it: tiles of up to 64
// columns, and as many k-splits as fill the SMs (at most z_max).  A 32-node tree (33 rows): 1422 us
// per frame with QKV, Wo and down on 32 / 48 / 48 CTAs, 1358 on 128 each.
//
// Chain streams: the k-splits do not depend on the row count below 385 rows (QKV unsplit, Wo and
// down six), so a stream's logits are the same bits whatever context it is decoded in.  Its Wo,
// gate/up and down operands are single bf16 values, which turn a sum's last bit into 3e-4 of the
// logits.  Split freely as well, frames of 8 / 16 / 32 streams would take 1021 / 1100 / 1219 us
// instead of 1131 / 1175 / 1278.
struct TcShape {
  int pitch, z;
};
inline TcShape tc_small_shape(int M, int Rtc, int n_sm, int z_max) {
  const int units = Rtc / 16, T = (Rtc + 63) / 64, z = n_sm / ((M / tc::kBM) * T);
  return TcShape{(units + T - 1) / T * 16, z < 1 ? 1 : (z > z_max ? z_max : z)};
}
constexpr int kTcSmallRows = 128;
// Residual products otherwise: six splits, four from 385 rows (512 operand rows: 128-column tiles, 128
// CTAs) on, where more splits' partial sums cost more than they save.
inline TcShape tc_resid_shape(int H, int Rtc, int n_sm, bool free_k) {
  if (free_k && Rtc <= kTcSmallRows) return tc_small_shape(H, Rtc, n_sm, kTcSplit);
  const int n_mt = H / tc::kBM, units = Rtc / 16, z = Rtc > 384 ? 4 : 6;
  int T = n_sm / (n_mt * z);
  if (T < 1) T = 1;
  if (T < (Rtc + 255) / 256) T = (Rtc + 255) / 256;
  if (T > units) T = units;
  return TcShape{(units + T - 1) / T * 16, z};
}
// Non-empty k-splits of a product over K in z splits (gemm_tile's split of the k-slices).
inline int tc_splits(int K, int z) {
  const int nk = K / tc::kBK, per = (nk + z - 1) / z;
  return (nk + per - 1) / per;
}

// Shared memory for the ring of a tile of up to 128 columns: two CTAs of consecutive kernels fit
// an SM together, so the next product's weights stream in while this one finishes.
constexpr int kTcCompact = 100 * 1024;
constexpr int kTcCompactRows = 384;

// Elements lane + 32 i (i < nd) of a row of the QKV product: its nz <= kTcQkvSplit partial sums, zs
// floats apart, added.
__device__ __forceinline__ void qkv_row(float (&x)[4], const float* src, int nd, int lane, int nz, size_t zs) {
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = i < nd ? __ldcg(src + lane + 32 * i) : 0.f;
  if (nz == 1) return;
  float y[kTcQkvSplit - 1][4];
#pragma unroll
  for (int z = 1; z < kTcQkvSplit; ++z)
#pragma unroll
    for (int i = 0; i < 4; ++i) y[z - 1][i] = i < nd && z < nz ? __ldcg(src + z * zs + lane + 32 * i) : 0.f;
#pragma unroll
  for (int z = 0; z < kTcQkvSplit - 1; ++z)
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] += y[z][i];
}

// q, k, v = W (x . g / rms) with the hi + lo operand.
__global__ void __launch_bounds__(tc::kPThreads, 1) tc_qkv_kernel(const tc::GemmArgs g, float* out, int ld) {
  tc::gemm_persistent<kTcBN, true>(g, 1, [&](int m, int n, int, float v) { out[(size_t)n * ld + m] = v; });
}
// The same product, one 128 x pitch tile per CTA; k-split z writes partial sums out[z][Rtc][ld].
constexpr int kQkvThreads = 256;
template <int BN, int kBudget>
__global__ void __launch_bounds__(kQkvThreads, 1) tc_qkv_tile_kernel(const tc::GemmArgs g, float* out, int ld,
                                                                      const int* nrows) {
  tc::TileRun t;
  if (!tc::gemm_tile_run<BN, true, kBudget, true>(g, t)) return;
  const int M = *nrows;
  float* o = out + (size_t)blockIdx.z * g.N * ld;
  tc::gemm_tile_drain<BN>(t, [&](int m, int n, float v) {
    if (n < M) o[(size_t)n * ld + m] = v;
  });
}

// gate/up -> SwiGLU, one 128 x pitch tile per CTA (gemm_tile_run).  A is the interleaved
// gate/up matrix of 2F rows written by tc_tile_layer: rows 0..63 of tile b are the gate rows
// of features 64b..64b+63, rows 64..127 the up rows of the same features.  The accumulator is
// staged in shared memory (the idle operand ring, [column][tile row]) so that a thread holds
// the gate and up values of eight consecutive features of one packed row; it writes
// silu(gate) * up as one 16-byte bf16 chunk of the down product's SW128 operand (k-slice b,
// element (row n, feature m)).  Packed rows at or past *nrows are not written.
// kHilo (trees and prompts): the operand and the result are hi + lo pairs of bf16 (about 16 mantissa bits).
constexpr int kGuThreads = 256;
template <int BN, bool kHilo, int kBudget>
__global__ void __launch_bounds__(kGuThreads, 1) tc_gu_kernel(const tc::GemmArgs g, uint8_t* act_t, uint8_t* act_lo, int Rtc,
                                                               const int* nrows) {
  using L = tc::Layout<BN, kHilo, kBudget>;
  constexpr int kSP = tc::kBM + 4;                  // staged column stride (floats)
  static_assert((size_t)BN * kSP * 4 <= (size_t)L::kStages * L::kStageBytes, "gate/up staging exceeds the ring");
  tc::TileRun t;
  if (!tc::gemm_tile_run<BN, kHilo, kBudget, true>(g, t)) return;
  float* S = reinterpret_cast<float*>(t.smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, part = warp >> 2, n_parts = (int)(blockDim.x >> 7);
  if (t.ok) {
    // warp w drains TMEM lanes 32 (w % 4) .. (tile rows) for the column chunks c = w / 4 mod
    // (warps / 4); a warp's 32 lanes store 32 consecutive floats of one column
    const uint32_t lane_base = t.tmem + ((uint32_t)(quarter * 32) << 16);
    const int r = quarter * 32 + lane, n_ch = t.nw >> 4;
    for (int ch = part; ch < n_ch; ch += n_parts) {
      float v[16];
      tc::tmem_ld16(lane_base + (uint32_t)(16 * ch), v);
#pragma unroll
      for (int j = 0; j < 16; ++j) S[(16 * ch + j) * kSP + r] = v[j];
    }
  }
  __syncthreads();
  if (t.ok) {
    const int M = *nrows, kt = t.m0 / tc::kBM;
    for (int it = threadIdx.x; it < t.nw * 8; it += blockDim.x) {
      const int nl = it >> 3, c = it & 7, n = t.n0 + nl;
      if (n >= M) continue;
      const float4* gs = reinterpret_cast<const float4*>(S + nl * kSP + 8 * c);
      const float4* us = reinterpret_cast<const float4*>(S + nl * kSP + 64 + 8 * c);
      const float4 g0 = gs[0], g1 = gs[1], u0 = us[0], u1 = us[1];
      const float gt[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
      const float up[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = gt[e] / (1.0f + __expf(-gt[e])) * up[e];
      const size_t off = tc::sw128_offset(Rtc, n, kt, c);
      uint32_t h[4], lo[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        h[q] = pack_bf16x2(v[2 * q], v[2 * q + 1]);
        lo[q] = pack_bf16x2(v[2 * q] - bf16_lo_f32(h[q]), v[2 * q + 1] - bf16_hi_f32(h[q]));
      }
      *reinterpret_cast<uint4*>(act_t + off) = make_uint4(h[0], h[1], h[2], h[3]);
      if (kHilo) *reinterpret_cast<uint4*>(act_lo + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
  tc::gemm_tile_free<BN>(t);
}

// Residual products (Wo, down): one 128 x pitch tile per CTA over the k-slices of split
// blockIdx.z; split z writes its partial sums part[z][n][m] (plain stores);
// tc_resid_norm_kernel adds them into the residual stream.
constexpr int kResidThreads = 256;
template <int BN, bool kHilo, int kBudget>
__global__ void __launch_bounds__(kResidThreads, 1) tc_resid_kernel(const tc::GemmArgs g, float* part, int ld, int Rtc,
                                                                     const int* nrows) {
  tc::TileRun t;
  if (!tc::gemm_tile_run<BN, kHilo, kBudget, true>(g, t)) return;
  const int M = *nrows;
  const size_t zoff = (size_t)blockIdx.z * Rtc;
  tc::gemm_tile_drain<BN>(t, [&](int m, int n, float v) {
    if (n < M) part[(zoff + n) * ld + m] = v;
  });
}

// Where a residual pass writes the row's normalised operand: `hi` / `lo` of Rtc rows at the row
// itself; after the last layer, with `slots` (eight per row, -1: none), at those rows of the LM
// heads' operand of slot_rows rows instead.  ss (may be null): the rows' sums of squares.
struct NormOut {
  const float* gain;          // null: no operand
  uint8_t *hi, *lo;
  const int* slots;
  int slot_rows;
  float* ss;
};
// Per packed row (one CTA, thread t owns elements 8t..8t+7): X += the nz partial sums, the
// row's sum of squares (the next RMSNorm), and the next product's normalised operand as SW128
// tiles.
template <int NZ>       // partial sums held in registers (nz <= NZ)
__global__ void __launch_bounds__(128) tc_resid_norm_kernel(float* X, const float* __restrict__ part, int nz, int Rtc,
                                                            int H, const int* nrows, float eps, const NormOut out) {
  tc::pdl_wait();
  tc::pdl_trigger();
  const int r = blockIdx.x;
  if (r >= *nrows) return;
  const int t = threadIdx.x;
  const bool live = t < H / 8;
  float x[8];
  float ss = 0.f;
  if (live) {
    float4* xr = reinterpret_cast<float4*>(X + (size_t)r * H + 8 * t);
    float4 a = xr[0], b = xr[1];
    // every partial's loads issued before the first add, added in split order
    float4 u[NZ], w[NZ];
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
      if (z < nz) {
        const float4* pr = reinterpret_cast<const float4*>(part + ((size_t)z * Rtc + r) * H + 8 * t);
        u[z] = __ldcg(pr);
        w[z] = __ldcg(pr + 1);
      }
    }
#pragma unroll
    for (int z = 0; z < NZ; ++z) {
      if (z < nz) {
        a.x += u[z].x; a.y += u[z].y; a.z += u[z].z; a.w += u[z].w;
        b.x += w[z].x; b.y += w[z].y; b.z += w[z].z; b.w += w[z].w;
      }
    }
    xr[0] = a;
    xr[1] = b;
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
#pragma unroll
    for (int i = 0; i < 8; ++i) ss += x[i] * x[i];
  }
  const float tot = block_sum128(ss);
  if (out.ss && t == 0) out.ss[r] = tot;
  if (!out.gain || !live) return;
  const NormChunk c = norm_chunk(x, rsqrtf(tot / (float)H + eps), out.gain, t);
  if (!out.slots) {
    const size_t off = tc::sw128_offset(Rtc, r, t >> 3, t & 7);
    *reinterpret_cast<uint4*>(out.hi + off) = c.hi;
    if (out.lo) *reinterpret_cast<uint4*>(out.lo + off) = c.lo;
  } else {
    for (int j = 0; j < 8; ++j) {
      const int q = out.slots[8 * r + j];
      if (q < 0) continue;
      const size_t off = tc::sw128_offset(out.slot_rows, q, t >> 3, t & 7);
      *reinterpret_cast<uint4*>(out.hi + off) = c.hi;
      *reinterpret_cast<uint4*>(out.lo + off) = c.lo;
    }
  }
}

// The transformer-block products can use the tensor-core GEMM (shape and dtype limits).
bool tc_block_supported(const FrameParams& p) {
  return p.wdtype == MCD_WEIGHT_BF16 && p.qkv_dim % 128 == 0 && p.F % 128 == 0 && p.H % 128 == 0 &&
         (p.NH * p.D) % 64 == 0 && p.H % 64 == 0 && p.F % 64 == 0 && p.H <= 1024;
}

// SW128 copies of one layer's weights: [qkv | gate/up interleaved (2F rows) | o | d], offsets
// within a layer.
struct TcLayerOffsets {
  size_t qkv = 0, gu = 0, o = 0, d = 0, layer = 0;
};
inline TcLayerOffsets tc_layer_offsets(const FrameParams& p) {
  TcLayerOffsets t;
  const size_t H = p.H, F = p.F, qd = (size_t)p.NH * p.D;
  t.qkv = 0;
  t.gu = t.qkv + (size_t)p.qkv_dim * H * 2;
  t.o = t.gu + 2 * F * H * 2;
  t.d = t.o + H * qd * 2;
  t.layer = t.d + H * F * 2;
  return t;
}
// Tile layer l's row-major bf16 sources (device) into the SW128 copies at base.
inline void tc_tile_layer(const FrameParams& p, cudaStream_t st, const uint8_t* wq, const uint8_t* wk, const uint8_t* wv,
                          const uint8_t* wo, const uint8_t* wg, const uint8_t* wu, const uint8_t* wd, uint8_t* base) {
  const TcLayerOffsets t = tc_layer_offsets(p);
  const int H = p.H, F = p.F, qd = p.NH * p.D, kd = p.NKV * p.D;
  auto tile = [&](const uint8_t* s, int rows, int K, int R, int row0, int grp, int gstride, size_t off) {
    tc_weight_tile_kernel<<<512, 256, 0, st>>>(reinterpret_cast<const uint16_t*>(s), rows, K, R, row0, grp, gstride,
                                               base + off);
  };
  tile(wq, qd, H, p.qkv_dim, 0, qd, 0, t.qkv);
  tile(wk, kd, H, p.qkv_dim, qd, kd, 0, t.qkv);
  tile(wv, kd, H, p.qkv_dim, qd + kd, kd, 0, t.qkv);
  // gate rows 64b.. of tile b at its rows 0..63, the up rows at 64..127 (tc_gu_kernel)
  tile(wg, F, H, 2 * F, 0, 64, 128, t.gu);
  tile(wu, F, H, 2 * F, 64, 64, 128, t.gu);
  tile(wo, H, qd, H, 0, H, 0, t.o);
  tile(wd, H, F, H, 0, F, 0, t.d);
}
// The instantiation of a gate/up or residual product for a tile pitch, as go(std::integral_constant
// BN, budget); a compact ring where two CTAs of consecutive kernels shall share an SM.
template <bool kHilo, class Go>
inline void tc_pick(int pitch, int Rtc, Go go) {
  if (pitch <= 64) go(std::integral_constant<int, 64>{}, std::integral_constant<int, kTcCompact>{});
  else if (!kHilo && pitch <= 128 && Rtc <= kTcCompactRows)
    go(std::integral_constant<int, 128>{}, std::integral_constant<int, kTcCompact>{});
  else if (pitch <= 128) go(std::integral_constant<int, 128>{}, std::integral_constant<int, tc::kStageBudget>{});
  else if (pitch <= 176) go(std::integral_constant<int, 176>{}, std::integral_constant<int, tc::kStageBudget>{});
  else go(std::integral_constant<int, 256>{}, std::integral_constant<int, tc::kStageBudget>{});
}
// Dynamic shared memory of the block kernels (once per translation unit).
template <bool kHilo>
inline cudaError_t tc_block_set_smem() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto fn, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  set(tc_qkv_kernel, tc::PLayout<kTcBN, true>::kSmemBytes);
  set(tc_qkv_tile_kernel<64, kTcCompact>, tc::Layout<64, true, kTcCompact>::kSmemBytes);
  set(tc_qkv_tile_kernel<128, tc::kStageBudget>, tc::Layout<128, true>::kSmemBytes);
  auto both = [&](auto bn, auto budget) {
    constexpr int BN = decltype(bn)::value, B = decltype(budget)::value;
    set(tc_gu_kernel<BN, kHilo, B>, tc::Layout<BN, kHilo, B>::kSmemBytes);
    set(tc_resid_kernel<BN, kHilo, B>, tc::Layout<BN, kHilo, B>::kSmemBytes);
  };
  for (int pitch : {64, 128, 176, 256})
    for (int rows : {16, kTcCompactRows + 16}) tc_pick<kHilo>(pitch, rows, both);
  return e;
}

// Persistent launch shape: one CTA per SM at most, one per tile at least.
inline dim3 tc_grid(int n_tiles, int n_sm) { return dim3(n_tiles < n_sm ? n_tiles : n_sm); }
inline int tc_tiles(int N, int BN, int M, int splits) { return (N / BN) * (M / tc::kBM) * splits; }

// The QKV product's form at n packed rows: the persistent one when its 128-column tiles give at
// least four fifths of the SMs a tile, else one tile per CTA with the columns shared out over
// all SMs (QKV of 4096 x 1024 on 152 SMs: from 385 rows on).  Measured both ways: 512 rows
// (128 streams) 343.9 us per call persistent, 346.2 one tile per CTA; 128 rows (32 streams)
// 267.2 and 265.7; a prompt of 255 rows is 64 tiles of 128 columns against 128 of 64.
inline bool tc_qkv_persistent(int n, int qkv_dim, int n_sm) {
  return tc_tiles((n + kTcBN - 1) / kTcBN * kTcBN, kTcBN, qkv_dim, 1) * 5 >= n_sm * 4;
}
// Operand rows for n packed rows: what the QKV form needs, else the next multiple of 16.
inline int tc_operand_rows(int n, int qkv_dim, int n_sm) {
  const int unit = tc_qkv_persistent(n, qkv_dim, n_sm) ? kTcBN : 16;
  return (n + unit - 1) / unit * unit;
}
// Column tiles and k-splits of the QKV product (tile form); tc_qkv_splits: partial sums it leaves.
inline TcShape tc_qkv_shape(int qkv_dim, int Rtc, int n_sm, bool free_k) {
  if (free_k && Rtc <= kTcSmallRows) return tc_small_shape(qkv_dim, Rtc, n_sm, kTcQkvSplit);
  return TcShape{tc::tile_pitch(qkv_dim, Rtc, n_sm), 1};
}
inline int tc_qkv_splits(int qkv_dim, int Rtc, int H, int n_sm, bool free_k) {
  return tc_qkv_persistent(Rtc, qkv_dim, n_sm) ? 1 : tc_splits(H, tc_qkv_shape(qkv_dim, Rtc, n_sm, free_k).z);
}
// q, k, v of Rtc operand rows, as tc_qkv_splits partial sums out[z][Rtc][qkv_dim].  Below
// tc_qkv_persistent's line the pitch is at most kTcBN: nt
// tiles of 128 columns over n_mt weight tiles with nt n_mt < 0.8 n_sm leave n_sm / n_mt >= nt.
inline void tc_launch_qkv(bool free_k, const uint8_t* w, const uint8_t* xn_hi, const uint8_t* xn_lo, float* out, int qkv_dim, int Rtc,
                          int H, const int* nrows, int* err, unsigned long long wait_ns, int n_sm, bool pdl, cudaStream_t s) {
  tc::GemmArgs g{w, xn_hi, xn_lo, qkv_dim, Rtc, H, nrows, err, wait_ns, pdl, 0};
  if (tc_qkv_persistent(Rtc, qkv_dim, n_sm)) {
    tc::launch(pdl, tc_qkv_kernel, tc_grid(tc_tiles(Rtc, kTcBN, qkv_dim, 1), n_sm), dim3(tc::kPThreads),
                   tc::PLayout<kTcBN, true>::kSmemBytes, s, g, out, qkv_dim);
    return;
  }
  const TcShape sh = tc_qkv_shape(qkv_dim, Rtc, n_sm, free_k);
  g.bn = sh.pitch;
  const dim3 grid((Rtc + g.bn - 1) / g.bn, qkv_dim / tc::kBM, sh.z);
  if (g.bn <= 64)
    tc::launch(pdl, tc_qkv_tile_kernel<64, kTcCompact>, grid, dim3(kQkvThreads), tc::Layout<64, true, kTcCompact>::kSmemBytes,
                   s, g, out, qkv_dim, nrows);
  else
    tc::launch(pdl, tc_qkv_tile_kernel<128, tc::kStageBudget>, grid, dim3(kQkvThreads), tc::Layout<128, true>::kSmemBytes, s,
                   g, out, qkv_dim, nrows);
}

// gate/up -> SwiGLU into the down product's operand.  gu: the interleaved gate/up matrix
// (2F rows); xn: the normalised operand of Rtc rows.  The tile pitch over the packed rows fills
// the SMs with one tile per CTA (three tiles of 176 / 176 / 160 rows at 512 rows, F = 3072).
template <bool kHilo>
inline void tc_launch_gu(const uint8_t* gu, const uint8_t* xn, const uint8_t* xn_lo, uint8_t* act_t, uint8_t* act_lo, int Rtc,
                         const int* nrows, int F, int H, int* err, unsigned long long wait_ns, int n_sm, bool pdl,
                         cudaStream_t s) {
  const int pitch = Rtc <= 64 ? Rtc : tc::tile_pitch(2 * F, Rtc, n_sm);
  const tc::GemmArgs g{gu, xn, xn_lo, 2 * F, Rtc, H, nrows, err, wait_ns, pdl, pitch};
  const dim3 grid((Rtc + pitch - 1) / pitch, 2 * F / tc::kBM);
  tc_pick<kHilo>(pitch, Rtc, [&](auto bn, auto budget) {
    constexpr int BN = decltype(bn)::value, B = decltype(budget)::value;
    tc::launch(pdl, tc_gu_kernel<BN, kHilo, B>, grid, dim3(kGuThreads), tc::Layout<BN, kHilo, B>::kSmemBytes, s, g, act_t,
               act_lo, Rtc, nrows);
  });
}

// Wo or down (A = w: H rows of K, B = act: Rtc rows) -> the partial sums of tc_resid_shape's splits
// (H = 1024: trees and prompts 16 splits of one column tile up to 64 rows, 128 CTAs, and 9 of two up to
// 128, 144 CTAs; otherwise 6 of up to three, 144 CTAs; 4 of four at 512, 128 CTAs).
template <bool kHilo>
inline void tc_launch_resid(const uint8_t* w, const uint8_t* act, const uint8_t* act_lo, float* part, int H, int Rtc, int K,
                            const int* nrows, int* err, unsigned long long wait_ns, int n_sm, bool pdl, cudaStream_t s) {
  const TcShape sh = tc_resid_shape(H, Rtc, n_sm, kHilo);
  const int pitch = sh.pitch;
  const tc::GemmArgs g{w, act, act_lo, H, Rtc, K, nrows, err, wait_ns, pdl, pitch};
  const dim3 grid((Rtc + pitch - 1) / pitch, H / tc::kBM, sh.z);
  tc_pick<kHilo>(pitch, Rtc, [&](auto bn, auto budget) {
    constexpr int BN = decltype(bn)::value, B = decltype(budget)::value;
    tc::launch(pdl, tc_resid_kernel<BN, kHilo, B>, grid, dim3(kResidThreads), tc::Layout<BN, kHilo, B>::kSmemBytes, s, g,
               part, H, Rtc, nrows);
  });
}

// The residual pass of a product over K (tc_resid_norm_kernel) on `rows` CTAs.
inline void tc_launch_resid_norm(bool free_k, bool pdl, int rows, float* X, const float* part, int K, int Rtc, int H, int n_sm,
                                 const int* nrows, float eps, const NormOut& out, cudaStream_t s) {
  const int nz = tc_splits(K, tc_resid_shape(H, Rtc, n_sm, free_k).z);
  if (nz <= 6)
    tc::launch(pdl, tc_resid_norm_kernel<6>, dim3(rows), dim3(128), 0, s, X, part, nz, Rtc, H, nrows, eps, out);
  else
    tc::launch(pdl, tc_resid_norm_kernel<kTcSplit>, dim3(rows), dim3(128), 0, s, X, part, nz, Rtc, H, nrows, eps, out);
}
// Floats of partial sums a residual product leaves at up to Rtc operand rows.
inline size_t tc_part_floats(int Rtc, int H) {
  const size_t small = (size_t)kTcSplit * (Rtc < kTcSmallRows ? Rtc : kTcSmallRows), large = (size_t)6 * Rtc;
  return (small > large ? small : large) * H;
}

}  // namespace
}  // namespace mcd
