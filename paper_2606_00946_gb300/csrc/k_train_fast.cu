// Training step of a bf16 predictor on tensor cores (Sec. 4.3.2 online
// learning; loss and optimiser as in k_train.cu: mean squared error, SGD or
// Adam), built around bf16 operand images.
//
// An "image" of a matrix X [R, C] is X in bf16 laid out exactly as a K-major
// 128-byte-swizzled MMA operand: element (r, c) at byte sw128_offset(r, c, R),
// so the 128 x 64 (or N x 64) tile of rows r0.. and K-block kb is one
// contiguous run of bytes that a single bulk copy lands in shared memory
// ready for tcgen05.mma.  Each product's epilogue writes the images the next
// products read, both row-major (X) and transposed (X^T, for the weight
// gradients, whose reduction runs over the batch):
//
//   gather     A_0 = bf16(zscore(x)) -> img(A_0), img(A_0^T)
//   forward l  Z = A_l W_l^T + b_l (TMEM) -> A_{l+1} = bf16(relu(Z)), mask [Z > 0]
//   last l     ... plus the width-1 output layer: yhat, loss, dz_L = 2 (yhat - y) / B,
//              dW_L, db_L partials, dz_l = bf16(dz_L) bf16(w_L) [Z > 0] -> img(dz_l), img(dz_l^T)
//   backward   dW_l = bf16(dz_l)^T A_l   (split over the batch, fp32 partials)
//              dz_{l-1} = (bf16(dz_l) W_l) [Z_{l-1} > 0] -> images
//   optimiser  gradient = ordered sum of the partials; SGD / Adam on the fp32
//              master; rewrites img(W_l), img(W_l^T) for the next step.
// How these are launched depends on the shape (run_train_fast):
//   hidden layers up to 256   gather; k_tr_chain: every forward layer, the output
//                             layer and the input gradients, a 128-row tile's
//                             activations kept in shared memory; k_tr_dw: the
//                             weight gradients of every layer; optimiser
//   what plan_chain refuses,  gather; k_tr_gemm per product, a weight gradient
//   layers of 384 or 512      beside each input gradient; optimiser
//   train_ctas > 0            one persistent launch, k_tr_step, the same products
//                             as its phases
// Replay admission runs the forward layers alone (k_emb_gather, k_tr_gemm,
// k_emb_rows).
// Bias gradients are column sums of the unrounded dz, formed per 128-row tile
// in the epilogues.  The rounding points are those of the reference path
// (k_train.cu): bf16 operands of every product, fp32 sums, biases and state.
#include <algorithm>
#include <cmath>

#include "blockhash.cuh"
#include "chain_tiles.h"
#include "common.cuh"
#include "sm100.cuh"

namespace ls {
using namespace sm100;

namespace {

constexpr int kT = 512;        // 16 warps: TMEM lane quadrant = warp % 4, column quarter = warp / 4
constexpr int kM = 128;        // rows per tile
constexpr int kMaxChunks = 8;  // K-blocks of 64 per CTA
constexpr int kStageRegion = 4 * (kM * 128 + 256 * 128);  // operand stages (as many as fit, at least four)
constexpr int kTailBar = 256;  // barriers and the TMEM address, before the epilogue scratch

enum { TE_STORE = 0, TE_FWD = 1, TE_FWD_OUT = 2, TE_DX = 3 };

// One product D = A B^T over a K range, tiled as 128-row tiles x n_split
// column parts x splits of K; CTA li -> (column part li % n_split, row tile,
// split), so the column parts of a tile are adjacent (a cluster for TE_FWD_OUT).
struct TrJob {
  int epi;
  int m_tiles, n_split, splits;
  int nchunks;                       // K-blocks of 64 per CTA (the last split may hold fewer)
  int kblocks;                       // K-blocks of the whole product
  int stages;                        // tr_stages(NT)
  int NT;                            // columns per CTA; the product's N = NT * n_split
  const uint8_t* A;                  // image, rA rows
  int rA;
  const uint8_t* B;                  // image, N rows
  int M;                             // valid rows of D
  // TE_STORE: fp32 partial D to C[split][row][col]
  float* C;
  int ldc;
  int64_t split_stride;
  // TE_FWD / TE_FWD_OUT / TE_DX
  const float* bias;                 // layer bias (TE_FWD, TE_FWD_OUT)
  uint8_t* out;                      // row-major image of the result, rows = rows_pad (nullable)
  uint8_t* outT;                     // transposed image, rows = rT
  int rT;
  uint16_t* mask_out;                // TE_FWD: bits of [Z > 0] as [N/16][rows_pad]
  const uint16_t* mask_in;           // TE_DX: bits of the layer input's ReLU
  float* colpart;                    // [m_tiles][N] column sums of dz (TE_FWD_OUT, TE_DX)
  int rows_pad;                      // padded batch (multiple of 128)
  // TE_FWD_OUT: width-1 output layer
  const float* wL;                   // [N] fp32 master weights of the output layer
  const float* bL;                   // [1]
  const float* y;                    // [batch] targets
  int batch;
  float* partWL;                     // [m_tiles][N]
  float* partBL;                     // [m_tiles]
  float* partLoss;                   // [m_tiles]
  // dropout between hidden layers (0 = none): TE_FWD drops units of hidden
  // activation drop_h and scales the kept ones; TE_DX scales the gradient of
  // the dropped activation drop_h (its keep bits are in mask_in)
  int drop_h;
};

// K-blocks of split `split` of job J: splits hold nchunks each, the last what
// is left of the product's kblocks.
__device__ __forceinline__ int tr_chunks(const TrJob& J, int split) {
  return min(J.nchunks, J.kblocks - split * J.nchunks);
}

// Operand stages a product with NT columns per CTA has (a stage: the 128-row
// A tile and the NT-row B tile of one K-block).  With more K-blocks than
// stages, K-block c + stages refills the stage of K-block c.
int tr_stages(int NT) { return std::min(kMaxChunks, kStageRegion / (kM * 128 + NT * 128)); }

struct TrArgs {
  TrJob job[2];
  int n_cta0;                        // CTAs of job 0; the rest run job 1
  int n_cta;                         // CTAs of both jobs
  int* err;
  const DevState* st;                // optimiser step counter (dropout stream)
  uint64_t drop_seed, drop_thr;      // keep <=> (u >> 11) >= drop_thr
  float drop_scale;                  // fp32 1 / (1 - p)
  // replay admission's forward (EMB): records in use of the candidates' tiles
  // and of the kept records' after them; tiles past them are skipped
  const int64_t* counts;
  int tiles_cand;
};

__device__ __forceinline__ uint16_t bf16_bits(float x) {
  __nv_bfloat16 v = __float2bfloat16_rn(x);
  return *reinterpret_cast<uint16_t*>(&v);
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Sum over the warp's 32 lanes of each of 16 per-lane values: afterwards
// lanes u and u + 16 hold the sum for column u.  Fixed order (butterfly).
__device__ __forceinline__ float col_reduce16(float (&v)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 8; s >= 1; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float send = up ? v[i] : v[i + s];
      const float keep = up ? v[i + s] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// Row-major image from packed bf16 pairs: w[h] holds columns c + 2h (low
// half) and c + 2h + 1 (high half) of row j; c % 16 == 0.
__device__ __forceinline__ void store_row16p(uint8_t* img, int rows, int j, int c, const uint32_t (&w)[8]) {
  *reinterpret_cast<uint4*>(img + sw128_offset(j, c, rows)) = make_uint4(w[0], w[1], w[2], w[3]);
  *reinterpret_cast<uint4*>(img + sw128_offset(j, c + 8, rows)) = make_uint4(w[4], w[5], w[6], w[7]);
}

// Where an epilogue's row-major columns go: a CTA's own tile (or nowhere).
struct OwnRow {
  uint8_t* S1;
  __device__ __forceinline__ void operator()(int r, int c, const uint32_t (&w)[8]) const {
    if (S1) store_row16p(S1, kM, r, c, w);
  }
};

// The own tile and, in a cluster of two, the same place in the other CTA,
// counted there on the K-block's barrier (the columns are those of whole
// K-blocks).
struct ClusterRow {
  uint8_t* S1;
  uint32_t peer, peer_bar;  // S1 and the barrier of its first K-block in the other CTA (0: none)
  __device__ __forceinline__ void operator()(int r, int c, const uint32_t (&w)[8]) const {
    if (!S1) return;
    store_row16p(S1, kM, r, c, w);
    if (peer) {
      const uint32_t rb = peer_bar + 8 * (uint32_t)(c >> 6);
      st_async_v4(peer + (uint32_t)sw128_offset(r, c, kM), w[0], w[1], w[2], w[3], rb);
      st_async_v4(peer + (uint32_t)sw128_offset(r, c + 8, kM), w[4], w[5], w[6], w[7], rb);
    }
  }
};

// Transposed image [rowsT x 128] from packed bf16 pairs: element (c + u, r)
// for u < 16, c % 16 == 0, r < 128 the tile row.  The same bytes as
// sw128_offset(c + u, r, rowsT), with the row's swizzle phase (c + u) & 7 =
// u & 7 folded into per-store constants.
__device__ __forceinline__ void store_col16p(uint8_t* imgT, int rowsT, int r, int c, const uint32_t (&w)[8]) {
  uint8_t* base = imgT + (size_t)(r >> 6) * rowsT * 128 + (size_t)c * 128 + (r & 7) * 2;
  const uint32_t cx = (uint32_t)((r & 63) >> 3) << 4;
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    const uint16_t v = (u & 1) ? (uint16_t)(w[u >> 1] >> 16) : (uint16_t)(w[u >> 1] & 0xffffu);
    *reinterpret_cast<uint16_t*>(base + u * 128 + (cx ^ ((uint32_t)(u & 7) << 4))) = v;
  }
}

// Forward epilogue of one warp's columns [cbeg, cbeg + cw) of its 32 tile
// rows (r the thread's row): Z + b, ReLU and, with `drop`, dropout of unit
// n0 + c under the stream h1 (key rowkey + c, rowkey = (row << 20) | n0),
// each activation rounded to bf16 once as packed pairs that both images take
// their bytes from, and the 16-bit masks [Z > 0 and kept].  EMB (a forward with
// no backward): the row-major image alone.
template <bool EMB, class Row>
__device__ __forceinline__ void fwd_cols(uint32_t taddr, const float* s_bias, int cbeg, int cw, const Row& row,
                                         uint8_t* S2, int NT, int r, uint16_t* mask_out, int64_t rows_pad,
                                         bool drop, uint64_t h1, uint64_t rowkey, uint64_t drop_thr,
                                         float drop_scale) {
  for (int c = cbeg; c < cbeg + cw; c += 16) {
    uint32_t v[16];
    tmem_ld16x(taddr + (uint32_t)c, v);
    tmem_wait_ld();
    uint32_t w[8];
    uint32_t bits = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float4 q4 = reinterpret_cast<const float4*>(s_bias + c)[g];
      const float bq[4] = {q4.x, q4.y, q4.z, q4.w};
      float a4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int u = 4 * g + e;
        const float z = __uint_as_float(v[u]) + bq[e];
        float rv = z > 0.0f ? z : 0.0f;
        bool on = z > 0.0f;
        if (drop) {
          const uint64_t hu = bh::mix64(h1 ^ (rowkey + (uint64_t)(c + u)));
          const bool keep = (hu >> 11) >= drop_thr;
          on = on && keep;
          rv = keep ? rv * drop_scale : 0.0f;
        }
        bits |= (on ? 1u : 0u) << u;
        a4[e] = rv;
      }
      w[2 * g] = pack2(a4[0], a4[1]);
      w[2 * g + 1] = pack2(a4[2], a4[3]);
    }
    row(r, c, w);
    if (!EMB) {
      mask_out[(int64_t)(c >> 4) * rows_pad] = (uint16_t)bits;
      store_col16p(S2, NT, r, c, w);
    }
  }
}

// Epilogue scratch of a training-product CTA, after its barriers.
struct EpiSmem {
  static constexpr int kFloats = 256 + 256 + 8 * 256 + 8 * 128 + 128 + 128 + 8;
  float* s_bias;  // [256]
  float* s_w;     // [256] bf16-rounded output weights
  float* red;     // [4][256] column sums by lane quadrant
  float* red2;    // [4][256]
  float* rowq;    // [8][128] row dots by column group
  float* rowdot;  // [128] this CTA's row dots
  float* yrow;    // [128] predictions
  float* wsum;    // [8] warp partials
  __device__ __forceinline__ explicit EpiSmem(uint8_t* at)
      : s_bias(reinterpret_cast<float*>(at)),
        s_w(s_bias + 256),
        red(s_w + 256),
        red2(red + 4 * 256),
        rowq(red2 + 4 * 256),
        rowdot(rowq + 8 * 128),
        yrow(rowdot + 128),
        wsum(yrow + 128) {}
};

// Column c's sum of the four lane quadrants' partials [4][256].
__device__ __forceinline__ float col_total(const float* red, int c) {
  return ((red[c] + red[256 + c]) + red[512 + c]) + red[768 + c];
}

// Input-gradient epilogue of one warp's columns: dz = acc [mask] sc, its
// images (the row-major one through `row`) and the column sums of the 32 rows
// into red.  mask_in: this row's 16-bit words, `stride` apart by 16 columns;
// `bits` the warp's first one, loaded by the caller before it waited for the
// product (each later one is requested a step ahead).
template <class Row>
__device__ __forceinline__ void dx_cols(uint32_t taddr, int cbeg, int cw, const Row& row, uint8_t* S2, int NT, int r,
                                        const uint16_t* mask_in, int64_t stride, uint32_t bits, float sc,
                                        float* red) {
  const int lane = threadIdx.x & 31;
  for (int c = cbeg; c < cbeg + cw; c += 16) {
    uint32_t v[16];
    tmem_ld16x(taddr + (uint32_t)c, v);
    tmem_wait_ld();
    const uint32_t next = c + 16 < cbeg + cw ? mask_in[(int64_t)((c >> 4) + 1) * stride] : 0u;
    float dz[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) dz[u] = ((bits >> u) & 1u) ? __uint_as_float(v[u]) * sc : 0.0f;
    uint32_t w[8];
#pragma unroll
    for (int h = 0; h < 8; ++h) w[h] = pack2(dz[2 * h], dz[2 * h + 1]);
    row(r, c, w);
    store_col16p(S2, NT, r, c, w);
    const float sb = col_reduce16(dz);
    if (lane < 16) red[c + lane] = sb;
    bits = next;
  }
}

// The width-1 output layer behind the last hidden one.
struct OutLayer {
  const float* bL;
  const float* y;
  int batch;
  float* partWL;
  float* partBL;
  float* partLoss;
  float* colpart;
};

// The row dots of a tile's n_split column parts (the ranks of a cluster,
// PAIR_ONLY: at most two), added in rank order, by every thread of every rank's
// epilogue, also after a timed-out wait (ok false): the total of row threadIdx.x.
template <bool PAIR_ONLY>
struct DsmemTotals {
  int n_split;
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  __device__ __forceinline__ float total(bool& ok, const EpiSmem& E) const {
    const int tid = threadIdx.x;
    if (n_split > 1) cluster_sync();
    else __syncthreads();
    float tot = 0.0f;
    if (ok && tid < kM) {
      tot = E.rowdot[tid];
      if (n_split > 1) {
        if (PAIR_ONLY || n_split == 2) {
          const uint32_t me = cluster_ctarank();
          const float other = ld_dsmem_f32(E.rowdot + tid, me ^ 1u);
          tot = me == 0 ? tot + other : other + tot;
        } else {  // four
          float v[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = ld_dsmem_f32(E.rowdot + tid, (uint32_t)k);
          tot = ((v[0] + v[1]) + v[2]) + v[3];
        }
      }
    }
    return tot;
  }
  // the other ranks have read this CTA's row dots, and its yrow is complete
  __device__ __forceinline__ void settle(bool&) const {
    if (n_split > 1) cluster_sync();
    else __syncthreads();
  }
};

// The same for a cluster of two (or one CTA), each rank sending its row dots
// to the other, counted on its barrier (armed before the kernel's first
// cluster barrier), by the 512 threads of the epilogue.
struct SentTotals {
  float* other;  // [128]
  uint64_t* bar;
  int rank, CL;
  __device__ __forceinline__ void sync() const { named_bar_sync(1, kT); }
  __device__ __forceinline__ float total(bool& ok, const EpiSmem& E) const {
    const int tid = threadIdx.x;
    float tot = 0.0f;
    if (ok && tid < kM) {
      tot = E.rowdot[tid];  // (this thread's own store)
      if (CL > 1) {
        const uint32_t to = (uint32_t)rank ^ 1u;
        st_async_f32(map_cluster(other + tid, to), tot, map_cluster(bar, to));
        if (mbar_wait_cl(bar, 0)) tot = rank == 0 ? tot + other[tid] : other[tid] + tot;
        else ok = false;
      }
    }
    return tot;
  }
  __device__ __forceinline__ void settle(bool& ok) const { ok = named_bar_and(1, kT, ok); }
};

// Epilogue of the last hidden layer's columns [n0, n0 + NT) of a 128-row tile
// by the whole CTA: output layer, loss, its gradients and dz.
template <class Totals, class Row>
__device__ __forceinline__ void out_epilogue(bool& ok, const OutLayer& o, uint32_t taddr, int NT, int N, int n0, int mt,
                                             int m0, int ns, const Totals& totals, const Row& row, uint8_t* S2,
                                             const EpiSmem& E) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, cq = warp >> 2;
  const int r = 32 * q + lane, j = m0 + r;
  const int cw = NT / 4, cbeg = cq * cw;
  // pass 1: activations and this warp's part of the output dot product.  With
  // all of 128 or 256 columns in one CTA, each warp keeps its two halves apart
  // and the row dot is added as two CTAs of half the columns add it: the same
  // order, the same bits.
  const bool whole = NT == N && (NT == 128 || NT == 256);
  const bool valid = j < o.batch;
  const float target = valid ? __ldg(o.y + j) : 0.0f, bias_out = __ldg(o.bL);  // (early: they are needed in a chain)
  if (ok) {
    float dot = 0.0f, first = 0.0f;  // (two names: an indexed pair would live in local memory)
    for (int c = cbeg; c < cbeg + cw; c += 16) {
      if (whole && c == cbeg + cw / 2) {
        first = dot;
        dot = 0.0f;
      }
      uint32_t v[16];
      tmem_ld16x(taddr + (uint32_t)c, v);
      tmem_wait_ld();
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const float4 b4 = reinterpret_cast<const float4*>(E.s_bias + c)[g];
        const float4 w4 = reinterpret_cast<const float4*>(E.s_w + c)[g];
        const float b[4] = {b4.x, b4.y, b4.z, b4.w}, wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float z = __uint_as_float(v[4 * g + e]) + b[e];
          dot = fmaf(round_bf16(z > 0.0f ? z : 0.0f), wv[e], dot);
        }
      }
    }
    if (whole) {
      E.rowq[(2 * cq) * 128 + r] = first;
      E.rowq[(2 * cq + 1) * 128 + r] = dot;
    } else {
      E.rowq[cq * 128 + r] = dot;
    }
  }
  totals.sync();
  if (ok && tid < kM) {
    const float lo = ((E.rowq[tid] + E.rowq[128 + tid]) + E.rowq[256 + tid]) + E.rowq[384 + tid];
    E.rowdot[tid] =
        whole ? lo + (((E.rowq[512 + tid] + E.rowq[640 + tid]) + E.rowq[768 + tid]) + E.rowq[896 + tid]) : lo;
  }
  const float tot = totals.total(ok, E);
  if (ok && tid < kM) E.yrow[tid] = tot + bias_out;
  totals.settle(ok);
  if (ok) {
    const float yhat = E.yrow[r];
    const float e = valid ? yhat - target : 0.0f;
    const float dzL = valid ? 2.0f * e / (float)o.batch : 0.0f;
    const float rd = round_bf16(dzL);
    if (ns == 0 && cq == 0) {
      float e2 = e * e, dsum = dzL;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        e2 += __shfl_xor_sync(0xffffffffu, e2, o);
        dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
      }
      if (lane == 0) {
        E.wsum[q] = e2;
        E.wsum[4 + q] = dsum;
      }
    }
    // pass 2 (Z re-read from TMEM, so [Z > 0] is the same test as in pass 1):
    // dW_L partial (sum_j bf16(dz_L[j]) a[j, c]) and dz = bf16(dz_L) bf16(w_L) [Z > 0]
    for (int c = cbeg; c < cbeg + cw; c += 16) {
      uint32_t v[16];
      tmem_ld16x(taddr + (uint32_t)c, v);
      tmem_wait_ld();
      float pw[16], dz[16];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const float4 b4 = reinterpret_cast<const float4*>(E.s_bias + c)[g];
        const float4 w4 = reinterpret_cast<const float4*>(E.s_w + c)[g];
        const float b[4] = {b4.x, b4.y, b4.z, b4.w}, wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float z = __uint_as_float(v[4 * g + e]) + b[e];
          const bool pos = z > 0.0f;
          pw[4 * g + e] = rd * round_bf16(pos ? z : 0.0f);
          dz[4 * g + e] = pos ? rd * wv[e] : 0.0f;
        }
      }
      uint32_t w[8];
#pragma unroll
      for (int h = 0; h < 8; ++h) w[h] = pack2(dz[2 * h], dz[2 * h + 1]);
      row(r, c, w);
      store_col16p(S2, NT, r, c, w);
      const float sw = col_reduce16(pw);
      if (lane < 16) E.red2[q * 256 + c + lane] = sw;
      const float sb = col_reduce16(dz);
      if (lane < 16) E.red[q * 256 + c + lane] = sb;
    }
  }
  totals.sync();
  if (ok) {
    for (int c = tid; c < NT; c += kT) {
      o.partWL[(int64_t)mt * N + n0 + c] = col_total(E.red2, c);
      o.colpart[(int64_t)mt * N + n0 + c] = col_total(E.red, c);
    }
    if (ns == 0 && tid == 0) {
      o.partLoss[mt] = ((E.wsum[0] + E.wsum[1]) + E.wsum[2]) + E.wsum[3];
      o.partBL[mt] = ((E.wsum[4] + E.wsum[5]) + E.wsum[6]) + E.wsum[7];
    }
  }
}

// fp32 tile of a weight-gradient partial: the warp's 32 rows and columns
// [cbeg, cbeg + cw) from TMEM into `tile` (rows of NT floats and 16 bytes more,
// so that the rows of a quarter warp start in different banks).
__device__ __forceinline__ void store_tile(uint32_t taddr, int r, int cbeg, int cw, int NT, uint8_t* tile) {
  uint8_t* row = tile + (size_t)r * (NT * 4 + 16);
  for (int c = cbeg; c < cbeg + cw; c += 16) {
    uint32_t v[16];
    tmem_ld16x(taddr + (uint32_t)c, v);
    tmem_wait_ld();
#pragma unroll
    for (int g = 0; g < 4; ++g)
      *reinterpret_cast<uint4*>(row + (c + 4 * g) * 4) = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
  }
}

// The tile's valid rows to global memory (row pitch ldc floats), a bulk copy
// each, by the first 128 threads once every warp has stored (and fenced).
// Stores from the threads' registers touch 32 lines an instruction and took
// the load-store unit 4K cycles a tile of 128 columns.
__device__ __forceinline__ void copy_tile(float* C, int ldc, int rows, int NT, const uint8_t* tile, bool drain) {
  const int r = threadIdx.x;
  if (r < rows && r < kM) bulk_s2g(C + (int64_t)r * ldc, tile + (size_t)r * (NT * 4 + 16), (uint32_t)NT * 4);
  if (r < kM) {
    if (drain) bulk_commit_wait_all();  // (tr_tile)
    else bulk_commit_wait_read();
  }
}

// Shared memory of a training-product CTA: the operand stages, then the
// barriers (kMaxChunks `full`, `done`, kMaxChunks `used`) and epilogue scratch.
__device__ __forceinline__ uint8_t* tr_tail(uint8_t* smem) { return smem + kStageRegion; }

// The copy of K-block c's operands (`a`: the 128-row tile of A, `b`: the
// columns of B) into stage s.
__device__ __forceinline__ void tr_copy(const TrJob& J, int c, int s, int kb, int m0, int n0, bool a, bool b, uint8_t* smem,
                                        uint64_t* full) {
  const int NT = J.NT, N = NT * J.n_split;
  const uint32_t a_bytes = kM * 128, b_bytes = (uint32_t)NT * 128;
  uint8_t* st = smem + (size_t)s * (a_bytes + b_bytes);
  if (a) bulk_g2s(st, J.A + (size_t)kb * J.rA * 128 + (size_t)m0 * 128, a_bytes, &full[c]);
  if (b) bulk_g2s(st + a_bytes, J.B + (size_t)kb * N * 128 + (size_t)n0 * 128, b_bytes, &full[c]);
}

// The part of tile `bid` that reads nothing the step's earlier products
// write: arm the tile's chunk barriers (for a CTA that runs `many` tiles, the
// barriers it does not use are arrived on with no bytes, so each advances one
// phase per tile),
// copy the weight operand (forward and input-gradient products read the
// weight images, which only the optimiser of the previous step writes) and
// stage the epilogue's bias and output weights (the fp32 master).  A
// per-launch product runs it before waiting for its predecessor.
template <bool RING>
__device__ __forceinline__ void tr_tile_pre(const TrArgs& args, int bid, uint8_t* smem, bool many) {
  const bool second = bid >= args.n_cta0;
  const TrJob& J = args.job[second ? 1 : 0];
  const int li = second ? bid - args.n_cta0 : bid;
  const int ns = li % J.n_split, rest = li / J.n_split;
  const int split = rest / J.m_tiles;
  const int NT = J.NT, n0 = ns * NT, nch = tr_chunks(J, split);
  const uint32_t stage_bytes = kM * 128 + (uint32_t)NT * 128;
  uint8_t* tail = tr_tail(smem);
  uint64_t* full = reinterpret_cast<uint64_t*>(tail);
  float* s_bias = reinterpret_cast<float*>(tail + kTailBar);
  float* s_w = s_bias + 256;
  const int tid = threadIdx.x;
  if (tid == 0) {
    const bool b_static = J.epi != TE_STORE;  // the weight-gradient products read activations
    const int S = RING ? J.stages : kMaxChunks;
    for (int c = 0; c < nch; ++c) {
      mbar_arrive_expect_tx(&full[c], stage_bytes);
      if (b_static && c < S) tr_copy(J, c, c, split * J.nchunks + c, 0, n0, false, true, smem, full);
    }
    if (many)
      for (int c = nch; c < kMaxChunks; ++c) mbar_arrive(&full[c]);
  }
  for (int t = tid; t < NT; t += kT) {
    if (J.bias) s_bias[t] = __ldg(J.bias + n0 + t);
    if (J.epi == TE_FWD_OUT) s_w[t] = round_bf16(__ldg(J.wL + n0 + t));
  }
}

// The operand copies of tile `bid` that tr_tile_pre left (the activation or
// gradient operand; both operands of a weight-gradient product), by one
// thread, onto the barriers tr_tile_pre armed.
template <bool RING>
__device__ __forceinline__ void tr_tile_copies(const TrArgs& args, int bid, uint8_t* smem) {
  const bool second = bid >= args.n_cta0;
  const TrJob& J = args.job[second ? 1 : 0];
  const int li = second ? bid - args.n_cta0 : bid;
  const int ns = li % J.n_split, rest = li / J.n_split;
  const int mt = rest % J.m_tiles, split = rest / J.m_tiles;
  const int m0 = mt * kM;
  const int NT = J.NT, n0 = ns * NT;
  const int nch = RING ? min(tr_chunks(J, split), J.stages) : tr_chunks(J, split);
  uint64_t* full = reinterpret_cast<uint64_t*>(tr_tail(smem));
  for (int c = 0; c < nch; ++c)
    tr_copy(J, c, c, split * J.nchunks + c, m0, n0, true, J.epi == TE_STORE, smem, full);
}

// One output tile (part `bid` of the products in `args`) on this CTA's shared
// memory and TMEM accumulator, after tr_tile_pre of the same tile (and, when
// `copied`, tr_tile_copies).  Every
// mbarrier advances by one phase per tile (parity `par`).  `drain` waits for
// the tile's image stores to reach global memory (other CTAs of the grid read
// them); otherwise only until they have read shared memory.  Returns false
// after a timed-out wait (error latched, copies in flight waited for).
template <bool RING, bool EMB = false>
__device__ __forceinline__ bool tr_tile(const TrArgs& args, int bid, uint8_t* smem, uint32_t tmem, uint32_t par,
                                        bool drain, bool copied) {
  const bool second = bid >= args.n_cta0;
  const TrJob& J = args.job[second ? 1 : 0];
  const int li = second ? bid - args.n_cta0 : bid;
  const int ns = li % J.n_split, rest = li / J.n_split;
  const int mt = rest % J.m_tiles, split = rest / J.m_tiles;
  const int m0 = mt * kM;
  const int NT = J.NT, N = NT * J.n_split, n0 = ns * NT, nch = tr_chunks(J, split);
  const uint32_t a_bytes = kM * 128, b_bytes = (uint32_t)NT * 128;
  const uint32_t stage_bytes = a_bytes + b_bytes;
  uint8_t* tail = tr_tail(smem);
  uint64_t* full = reinterpret_cast<uint64_t*>(tail);           // [kMaxChunks]
  uint64_t* done = full + kMaxChunks;
  uint64_t* used = done + 1;                                    // [kMaxChunks] K-block read by the products
  const EpiSmem E(tail + kTailBar);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = RING ? J.stages : kMaxChunks;
  int copies = min(nch, S);  // K-blocks whose copies were issued (thread 0)
  bool ok = true;
  if (tid == 0) {
    if (!copied) tr_tile_copies<RING>(args, bid, smem);
    const uint32_t idesc = idesc_bf16_f32(kM, NT);
    // RING (hidden layers wider than 256, one tile per launch): there may be
    // more K-blocks than stages, at most twice as many
    for (int c = 0; c < nch; ++c) {
      if (!mbar_wait(&full[c], par)) { ok = false; break; }
      tc_fence_after();
      const uint32_t sa = smem_u32(smem + (size_t)(c < S ? c : c - S) * stage_bytes), sb = sa + a_bytes;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        umma_bf16(tmem, sdesc_sw128(sa + 32u * k), sdesc_sw128(sb + 32u * k), idesc, (c | k) ? 1u : 0u);
      if (RING) {
        // refill the previous K-block's stage once its products have read it
        // (this K-block's products keep the tensor core busy meanwhile)
        if (c + S < nch) umma_commit(&used[c]);
        if (c >= 1 && c - 1 + S < nch) {
          if (!mbar_wait(&used[c - 1], 0)) { ok = false; break; }
          tr_copy(J, c - 1 + S, c - 1, split * J.nchunks + c - 1 + S, m0, n0, true, true, smem, full);
          copies = c + S;
        }
      }
    }
    umma_commit(done);  // arrives once everything issued so far has completed
  }
  __syncwarp();
  if (!mbar_wait(done, par)) ok = false;
  ok = __syncthreads_and(ok) != 0;  // one decision for the whole CTA
  if (!ok) {
    latch_error(args.err, LS_ERR_TIMEOUT);
    // copies that may still be in flight land in this CTA's own shared memory;
    // wait (bounded) for them before the CTA exits
    if (tid == 0)
      for (int c = 0; c < copies; ++c) mbar_wait(&full[c], par);
  }
  tc_fence_after();

  const int q = warp & 3, cq = warp >> 2;
  const int r = 32 * q + lane, j = m0 + r;
  // the epilogues stage their image tiles in the (now free) operand stages,
  // in the images' own byte layout: the row-major tile [128 rows x NT] as
  // NT / 64 runs of 16 KB, the transposed tile [NT rows x 128] as two runs of
  // NT x 128 bytes; bulk copies then write each run with one instruction
  uint8_t* S1 = smem;
  uint8_t* S2 = smem + 65536;
  const int cw = NT / 4, cbeg = cq * cw;  // this warp's columns (CTA-local)
  const uint32_t lane_addr = (uint32_t)(32 * q) << 16;

  if (ok && J.epi == TE_STORE) {
    if (j < J.M) store_tile(tmem + lane_addr, r, cbeg, cw, NT, smem);
    fence_async_smem();
    __syncthreads();
    copy_tile(J.C + (int64_t)split * J.split_stride + (int64_t)m0 * J.ldc + n0, J.ldc, J.M - m0, NT, smem, drain);
  } else if (ok && J.epi == TE_FWD) {
    // dropout stream of this activation at step t = step + 1 (Sec. 4.1: dropout
    // between hidden layers): h1 = mix64(seed ^ ((t << 16) | h)),
    // u = mix64(h1 ^ ((row << 20) | unit)), kept when (u >> 11) >= thr
    uint64_t h1 = 0;
    if (J.drop_h > 0) {
      const uint64_t t = (uint64_t)(*reinterpret_cast<const volatile int64_t*>(&args.st->step) + 1);
      h1 = bh::mix64(args.drop_seed ^ ((t << 16) | (uint64_t)J.drop_h));
    }
    uint16_t* mask_out = J.mask_out + j + (int64_t)(n0 >> 4) * J.rows_pad;
    const bool drop = J.drop_h > 0;
    fwd_cols<EMB>(tmem + lane_addr, E.s_bias, cbeg, cw, OwnRow{S1}, S2, NT, r, mask_out, J.rows_pad, drop, h1,
             ((uint64_t)j << 20) | (uint64_t)n0, args.drop_thr, args.drop_scale);
  } else if (ok && J.epi == TE_DX) {
    const uint16_t* mask = J.mask_in + (int64_t)(n0 >> 4) * J.rows_pad + j;
    dx_cols(tmem + lane_addr, cbeg, cw, OwnRow{J.out ? S1 : nullptr}, S2, NT, r, mask, J.rows_pad,
            mask[(int64_t)(cbeg >> 4) * J.rows_pad], J.drop_h > 0 ? args.drop_scale : 1.0f, E.red + q * 256);
    __syncthreads();
    for (int c = tid; c < NT; c += kT)
      J.colpart[(int64_t)mt * N + n0 + c] = col_total(E.red, c);
  }
  if (!EMB && J.epi == TE_FWD_OUT) {
    const OutLayer o{J.bL, J.y, J.batch, J.partWL, J.partBL, J.partLoss, J.colpart};
    out_epilogue(ok, o, tmem + lane_addr, NT, N, n0, mt, m0, ns, DsmemTotals<!RING>{J.n_split},
                 OwnRow{J.out ? S1 : nullptr}, S2, E);
  }
  if (ok && J.epi != TE_STORE) {
    fence_async_smem();  // staged tiles are read by the bulk copies (async proxy)
    __syncthreads();
    if (tid == 0) {
      if (J.out)
        for (int kb = 0; kb < NT / 64; ++kb)
          bulk_s2g(J.out + ((int64_t)(n0 / 64 + kb) * J.rows_pad + m0) * 128, S1 + (size_t)kb * kM * 128, kM * 128);
      for (int h = 0; !EMB && h < kM / 64; ++h)
        bulk_s2g(J.outT + ((int64_t)(m0 / 64 + h) * J.rT + n0) * 128, S2 + (size_t)h * NT * 128,
                 (uint32_t)NT * 128);
      if (drain) bulk_commit_wait_all();
      else bulk_commit_wait_read();  // before the stages are reused or the CTA exits
    }
  }
  tc_fence_before();
  __syncthreads();
  return ok;
}

// One launch per product (or pair of products): CTA b runs tile b.
template <bool RING, bool EMB>
__global__ void __launch_bounds__(kT, 1) k_tr_gemm(const __grid_constant__ TrArgs args) {
  extern __shared__ uint8_t smem_raw[];
  if (EMB) {  // the tile's rows are in use?  (the counts come from an earlier kernel)
    pdl_trigger();
    pdl_wait();
    const int mt = (int)blockIdx.x / args.job[0].n_split;
    const bool kept = mt >= args.tiles_cand;
    if ((int64_t)(kept ? mt - args.tiles_cand : mt) * kM >= args.counts[kept ? 1 : 0]) return;
  }
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(tr_tail(smem));
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(full + 2 * kMaxChunks + 1);
  const int NT = args.job[(int)blockIdx.x >= args.n_cta0 ? 1 : 0].NT;
  uint32_t tcols = 32;
  while ((int)tcols < NT) tcols <<= 1;
  if (threadIdx.x == 0) {
    // `full` of the tile's K-blocks, `done`, and `used` of those refilled (one
    // thread sets them up one after the other, so only what the tile needs)
    const TrJob& J = args.job[(int)blockIdx.x >= args.n_cta0 ? 1 : 0];
    for (int c = 0; c < J.nchunks; ++c) mbar_init(&full[c], 1);
    mbar_init(&full[kMaxChunks], 1);
    if (RING)
      for (int c = J.stages; c < J.nchunks; ++c) mbar_init(&full[kMaxChunks + 1 + c - J.stages], 1);
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    tmem_alloc(tmem_holder, tcols);
    tmem_relinquish();
  }
  // The next product may start now: its CTAs take SMs this grid leaves idle
  // and run their own prologue while this one works.  Every kernel of the
  // step after the gather starts only after the gather has passed its wait
  // (it lets its successor in behind it), so after the previous step's
  // optimiser has completed: the weight images and the master read before
  // the wait below are final.
  if (!EMB) pdl_trigger();
  tr_tile_pre<RING>(args, (int)blockIdx.x, smem, false);
  // the activation and gradient operands come from the previous kernels of the
  // stream: their copies start as soon as the wait returns
  if (!EMB) pdl_wait();
  if (threadIdx.x == 0) tr_tile_copies<RING>(args, (int)blockIdx.x, smem);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  // image stores may still be in flight when the CTA exits: the grid's
  // completion makes them visible to the next kernel
  tr_tile<RING, EMB>(args, (int)blockIdx.x, smem, tmem, 0, false, true);
  if (threadIdx.x < 32) tmem_dealloc(tmem, tcols);
}

// The forward pass and the input gradients of a step in one launch: one CTA,
// or a cluster of two, per 128-row tile; CTA `rank` has columns [rank * NT,
// ...) of every product.  The tile's activations (then gradients) stay in
// shared memory as the next product's operand: the epilogue stores its columns
// into both CTAs' copies, the other's counted on its barriers.  Two copies in
// turn need no cluster barrier: a rank writes the operand of product p + 1
// once its own product p is done, so after the other has finished product
// p - 1, which read that copy last; the tile that the other may still be
// storing from there keeps out of the way (chain_tiles.h).  Weights stream through a ring of K-blocks
// that is filled ahead across products by a warp of its own; another issues
// the products; sixteen run the epilogues.  Global memory gets only what the
// weight gradients read, the transposed images.  Same tiles, products and
// order of every sum as a launch per product, so the same bits.
//
// Bound by the chain of a tile: per product of 256 columns about 2.6K cycles
// from operand to accumulator and 4-5.5K of epilogue arithmetic and stores
// (11K for the output layer's).  Before, each product was a launch of its own,
// 5.5-8 us with its prologue, loads and tail.  A step (this, the gather, the
// weight gradients and the optimiser; us, a launch per product -> now):
//   128-256-256-256-1  batch 4096  49.8 -> 40.7     64-128-128-128-1  512  34.4 -> 25.4
//   64-128-128-128-1   batch 4096, dropout  41.0 -> 32.3              8192  50.0 -> 32.2
//   128-192-192-1      batch 8192  43.2 -> 33.3     128-256-256-1     8192  51.1 -> 33.8
//   128-256-256-1      batch 4096  35.5 -> 30.6     16-64-1           256  16.2 -> 15.7
// (of which the weight gradients' row copies, see copy_tile: 46.0 -> 41.8 for
// the first, 37.2 -> 34.0 and 37.7 -> 34.5 for the third row; and the mask
// words and targets requested before they are needed, about 1 us of each).
constexpr int kMaxPhases = 2 * (LS_MAX_LAYERS - 1);
constexpr int kMaxRing = 8;
constexpr int kChainT = kT + 64;  // the epilogue's warps, the products' warp, the weights' warp
constexpr int kSmemMax = 227 * 1024;
constexpr int kChainBar = 384;  // barriers and the TMEM address, before the epilogue scratch

struct ChainPhase {
  int epi;             // TE_FWD, TE_FWD_OUT or TE_DX
  int nk;              // K-blocks
  int NT;              // columns per CTA
  int feeds;           // the next product reads the result
  const uint8_t* B;    // weight image, NT * CL rows
  const float* bias;
  uint8_t* outT;       // transposed image of the result, rT rows
  int rT;
  int drop_h;          // as TrJob's
  uint16_t* mask;      // written by TE_FWD, read by TE_DX
  float* colpart;
  int stage[2];        // bytes: where each rank stages the transposed tile, in both operand copies
};

struct ChainArgs {
  ChainPhase ph[kMaxPhases];
  int n, CL;
  int a_bytes;         // one copy of the operand tile
  int stages, stage_bytes;
  uint32_t tmem_cols;
  const uint8_t* A0;   // image of the minibatch, R rows
  int R;
  const float* wL;
  OutLayer out;        // (colpart from the phase)
  int* err;
  const DevState* st;
  uint64_t drop_seed, drop_thr;
  float drop_scale;
};

__global__ void __launch_bounds__(kChainT, 1) k_tr_chain(const __grid_constant__ ChainArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* A = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* ring = A + 2 * (size_t)a.a_bytes;
  uint64_t* afull = reinterpret_cast<uint64_t*>(ring + (size_t)a.stages * a.stage_bytes);  // [2][kMaxChunks]
  uint64_t* done = afull + 2 * kMaxChunks;  // a product's accumulator is complete
  uint64_t* ready = done + 1;               // the epilogue's warps have written the next operand's columns
  uint64_t* xbar = ready + 1;               // the other rank's row dots
  uint64_t* bfull = xbar + 1;               // [kMaxRing]
  uint64_t* bempty = bfull + kMaxRing;      // [kMaxRing]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bempty + kMaxRing);
  volatile int* gave_up = reinterpret_cast<volatile int*>(tmem_holder + 1);
  const EpiSmem E(reinterpret_cast<uint8_t*>(afull) + kChainBar);
  float* other = E.s_bias + EpiSmem::kFloats;  // [128] the other rank's row dots
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int CL = a.CL;
  const int rank = CL > 1 ? (int)cluster_ctarank() : 0;
  const int mt = (int)blockIdx.x / CL, m0 = mt * kM;

  if (tid == 0) {
    for (int c = 0; c < 2 * kMaxChunks; ++c) mbar_init(&afull[c], 1);
    mbar_init(done, 1);
    mbar_init(ready, kT / 32);
    mbar_init(xbar, 1);
    for (int c = 0; c < a.stages; ++c) {
      mbar_init(&bfull[c], 1);
      mbar_init(&bempty[c], 1);
    }
    *gave_up = 0;
    fence_mbar_init();
    if (CL > 1) mbar_arrive_expect_tx(xbar, kM * 4);
  }
  __syncwarp();
  if (warp == 0) {
    tmem_alloc(tmem_holder, a.tmem_cols);
    tmem_relinquish();
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  if (CL > 1) cluster_sync();  // both ranks' barriers are ready for the other's stores
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == kT / 32 + 1) {
    // weights: every product's K-blocks in order through the ring (final
    // before this kernel starts: see k_tr_gemm)
    if (lane == 0) {
      int st = 0, loaded = 0;
      uint32_t par = 0;  // of the reuse a stage waits for
      bool ok = true;
      for (int p = 0; ok && p < a.n; ++p) {
        const uint32_t bytes = (uint32_t)a.ph[p].NT * 128;
        const uint8_t* src = a.ph[p].B + (size_t)rank * bytes;
        for (int c = 0; c < a.ph[p].nk; ++c, src += (size_t)CL * bytes) {
          if (loaded >= a.stages && (!mbar_wait(&bempty[st], par) || *gave_up)) { ok = false; break; }
          mbar_arrive_expect_tx(&bfull[st], bytes);
          bulk_g2s(ring + (size_t)st * a.stage_bytes, src, bytes, &bfull[st]);
          ++loaded;
          if (++st == a.stages) {
            st = 0;
            par = loaded > a.stages ? par ^ 1u : 0u;
          }
        }
      }
      if (!ok) {  // copies under way land in this CTA's shared memory: wait for them (bounded)
        *gave_up = 1;
        for (int u = loaded > a.stages ? loaded - a.stages : 0; u < loaded; ++u)
          if (!mbar_wait(&bfull[u % a.stages], (uint32_t)(u / a.stages) & 1u)) break;
      }
    }
  } else if (warp == kT / 32) {
    // products
    if (lane == 0) {
      pdl_wait();  // the minibatch from the gather
      int cs = 0;
      uint32_t cpar = 0, apar = 0;
      int own0 = 0, own1 = 0;  // K-blocks of the operand that this CTA writes itself
      for (int c = 0; c < a.ph[0].nk; ++c) {
        mbar_arrive_expect_tx(&afull[c], kM * 128);
        bulk_g2s(A + (size_t)c * kM * 128, a.A0 + ((size_t)c * a.R + m0) * 128, kM * 128, &afull[c]);
      }
      bool ok = true;
      for (int p = 0; p < a.n; ++p) {
        const int nk = a.ph[p].nk, NT = a.ph[p].NT;
        const int buf = p & 1;
        const uint32_t sA = smem_u32(A) + (uint32_t)buf * a.a_bytes;
        uint64_t* af = afull + buf * kMaxChunks;
        const uint32_t idesc = idesc_bf16_f32(kM, NT);
        if (p > 0 && !mbar_wait(ready, (uint32_t)(p - 1) & 1u)) ok = false;
        if (*gave_up) ok = false;
        tc_fence_after();
        for (int c = 0; ok && c < nk; ++c) {
          if (c < own0 || c >= own1) {
            const uint32_t bit = (uint32_t)(buf * kMaxChunks + c);
            if (!mbar_wait_cl(&af[c], (apar >> bit) & 1u)) ok = false;
            apar ^= 1u << bit;
            fence_async_smem();  // the other rank's stores, read by the products
          }
          if (ok && !mbar_wait(&bfull[cs], cpar)) ok = false;
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = sA + (uint32_t)c * kM * 128, sb = smem_u32(ring) + (uint32_t)cs * a.stage_bytes;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_bf16(tmem, sdesc_sw128(sa + 32u * k), sdesc_sw128(sb + 32u * k), idesc, (c | k) ? 1u : 0u);
          umma_commit(&bempty[cs]);
          if (++cs == a.stages) {
            cs = 0;
            cpar ^= 1u;
          }
        }
        if (!ok) *gave_up = 1;
        umma_commit(done);
        if (!ok) break;
        // the next operand's blocks of the other rank
        own0 = rank * (NT / 64);
        own1 = own0 + NT / 64;
        if (p + 1 < a.n)
          for (int c = 0; c < a.ph[p + 1].nk; ++c)
            if (c < own0 || c >= own1)
              mbar_arrive_expect_tx(&afull[(buf ^ 1) * kMaxChunks + c], kM * 128);
      }
      if (!ok)  // the minibatch's copies (a rank that gave up sends nothing more)
        for (int c = 0; c < a.ph[0].nk && !(apar >> c & 1u); ++c)
          if (!mbar_wait(&afull[c], 0)) break;
    }
  } else {
    // epilogues
    const int q = warp & 3, cq = warp >> 2;
    const int r = 32 * q + lane, j = m0 + r;
    const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16);
    pdl_wait();  // targets and the step counter
    bool ok = true;
    for (int p = 0; ok && p < a.n; ++p) {
      const ChainPhase& P = a.ph[p];
      const int NT = P.NT, n0 = rank * NT;
      for (int t = tid; t < NT; t += kT) {
        if (P.bias) E.s_bias[t] = __ldg(P.bias + n0 + t);
        if (P.epi == TE_FWD_OUT) E.s_w[t] = round_bf16(__ldg(a.wL + n0 + t));
      }
      const int cw = NT / 4, cbeg = cq * cw, own0 = chain::first_block(rank, NT);
      // the transposed tile for its bulk stores takes K-blocks of the operand
      // just read that the other rank does not write for the next product (it
      // may be at that epilogue already); this one writes there only in its
      // own next epilogue, after the stores have read the tile
      uint8_t* S2 = A + (rank ? P.stage[1] : P.stage[0]);
      uint16_t* mask = P.mask + j + (int64_t)(n0 >> 4) * a.R;
      const uint32_t bits = P.epi == TE_DX ? mask[(int64_t)(cbeg >> 4) * a.R] : 0u;
      if (tid == 0) bulk_commit_wait_read();  // the last product's stores have read S2
      __syncwarp();
      if (!mbar_wait(done, (uint32_t)p & 1u)) ok = false;
      ok = named_bar_and(1, kT, ok && !*gave_up);  // one decision for the whole CTA
      if (!ok) break;
      tc_fence_after();
      uint8_t* S1 = A + (size_t)((p + 1) & 1) * a.a_bytes + (size_t)own0 * kM * 128;
      uint64_t* sb = afull + ((p + 1) & 1) * kMaxChunks + own0;
      const bool send = CL > 1 && P.feeds;
      const ClusterRow row{P.feeds ? S1 : nullptr, send ? map_cluster(S1, (uint32_t)rank ^ 1u) : 0,
                           send ? map_cluster(sb, (uint32_t)rank ^ 1u) : 0};
      if (P.epi == TE_FWD) {
        uint64_t h1 = 0;
        const bool drop = P.drop_h > 0;
        if (drop) {  // (as in tr_tile)
          const uint64_t t = (uint64_t)(*reinterpret_cast<const volatile int64_t*>(&a.st->step) + 1);
          h1 = bh::mix64(a.drop_seed ^ ((t << 16) | (uint64_t)P.drop_h));
        }
        fwd_cols<false>(taddr, E.s_bias, cbeg, cw, row, S2, NT, r, mask, a.R, drop, h1,
                        ((uint64_t)j << 20) | (uint64_t)n0, a.drop_thr, a.drop_scale);
      } else if (P.epi == TE_DX) {
        dx_cols(taddr, cbeg, cw, row, S2, NT, r, mask, a.R, bits, P.drop_h > 0 ? a.drop_scale : 1.0f, E.red + q * 256);
      } else {
        OutLayer o = a.out;
        o.colpart = P.colpart;
        out_epilogue(ok, o, taddr, NT, NT * CL, n0, mt, m0, rank, SentTotals{other, xbar, rank, CL}, row, S2, E);
        if (!ok) break;
      }
      tc_fence_before();
      fence_async_smem();  // the columns are read by products and bulk copies
      __syncwarp();
      if (lane == 0) mbar_arrive(ready);
      named_bar_sync(1, kT);
      if (tid == 0)
        for (int h = 0; h < kM / 64; ++h)
          bulk_s2g(P.outT + ((int64_t)(m0 / 64 + h) * P.rT + n0) * 128, S2 + (size_t)h * NT * 128, (uint32_t)NT * 128);
      if (P.epi == TE_DX)
        for (int c = tid; c < NT; c += kT) P.colpart[(int64_t)mt * NT * CL + n0 + c] = col_total(E.red, c);
    }
    if (tid == 0) {
      bulk_commit_wait_read();
      if (!ok) {
        *gave_up = 1;
        latch_error(a.err, LS_ERR_TIMEOUT);
      }
    }
    tc_fence_before();
  }
  __syncwarp();
  __syncthreads();
  if (CL > 1) cluster_sync();  // no rank leaves while the other may still store to it
  if (CL > 1 && *gave_up) cluster_drain();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, a.tmem_cols);
}

// The weight gradients of every hidden layer in one launch: dW_l = dz_l^T A_l
// as 128-row tiles x column parts x splits of the batch (k_tr_gemm's TE_STORE
// jobs: same tiles, splits and order, so the same bits), two CTAs an SM: bound
// by the operand reads from L2 (25 MB for 128-256-256-256-1 at batch 4096),
// which one launch of all layers keeps going where one launch a layer left
// half the SMs idle.
struct DwJob {
  const uint8_t* A;   // img(dz_l^T), rA rows
  const uint8_t* B;   // img(A_l^T), NT * n_split rows
  float* C;           // [split][M][ldc]
  int rA, M, ldc;
  int NT, n_split, m_tiles;
  int nchunks, kblocks, stages;
};
constexpr int kDwT = 256;
constexpr int kDwStage = kM * (192 * 4 + 16);  // operand stages, then the fp32 tile of at most 192 columns

struct DwArgs {
  DwJob job[LS_MAX_LAYERS - 1];
  int cta0[LS_MAX_LAYERS];  // first CTA of each job
  int n;
  int* err;
};

__global__ void __launch_bounds__(kDwT, 2) k_tr_dw(const __grid_constant__ DwArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kDwStage);  // [kMaxRing]
  uint64_t* empty = full + kMaxRing;                              // [kMaxRing]
  uint64_t* done = empty + kMaxRing;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(done + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int jb = 0;
#pragma unroll
  for (int k = 1; k < LS_MAX_LAYERS - 1; ++k) jb += (k < a.n && (int)blockIdx.x >= a.cta0[k]) ? 1 : 0;
  const DwJob& J = a.job[jb];
  const int li = (int)blockIdx.x - a.cta0[jb];
  const int ns = li % J.n_split, rest = li / J.n_split;
  const int mt = rest % J.m_tiles, split = rest / J.m_tiles;
  const int NT = J.NT, N = NT * J.n_split, n0 = ns * NT, m0 = mt * kM;
  const int nch = min(J.nchunks, J.kblocks - split * J.nchunks), S = J.stages;
  const uint32_t b_bytes = (uint32_t)NT * 128, stage_bytes = kM * 128 + b_bytes;
  uint32_t tcols = 32;
  while ((int)tcols < NT) tcols <<= 1;
  if (tid == 0) {
    for (int c = 0; c < S; ++c) {
      mbar_init(&full[c], 1);
      mbar_init(&empty[c], 1);
    }
    mbar_init(done, 1);
    fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) {
    tmem_alloc(tmem_holder, tcols);
    tmem_relinquish();
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  pdl_wait();  // the transposed images
  bool ok = true;
  if (tid == 0) {
    auto load = [&](int c, int st) {
      const size_t kb = (size_t)(split * J.nchunks + c);
      uint8_t* to = smem + (size_t)st * stage_bytes;
      mbar_arrive_expect_tx(&full[st], stage_bytes);
      bulk_g2s(to, J.A + (kb * J.rA + m0) * 128, kM * 128, &full[st]);
      bulk_g2s(to + kM * 128, J.B + (kb * N + n0) * 128, b_bytes, &full[st]);
    };
    int loaded = 0, st = 0, lst = 0;
    uint32_t par = 0, lpar = 0;
    for (; loaded < nch && loaded < S; ++loaded) load(loaded, loaded);
    const uint32_t idesc = idesc_bf16_f32(kM, NT);
    int c = 0;
    for (; c < nch; ++c) {
      if (!mbar_wait(&full[st], par)) { ok = false; break; }
      tc_fence_after();
      const uint32_t sa = smem_u32(smem + (size_t)st * stage_bytes), sb = sa + kM * 128;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        umma_bf16(tmem, sdesc_sw128(sa + 32u * k), sdesc_sw128(sb + 32u * k), idesc, (c | k) ? 1u : 0u);
      umma_commit(&empty[st]);
      if (++st == S) {
        st = 0;
        par ^= 1u;
      }
      if (c > 0 && loaded < nch) {  // the previous K-block's stage
        if (!mbar_wait(&empty[lst], lpar)) { ok = false; break; }
        load(loaded, lst);
        ++loaded;
        if (++lst == S) {
          lst = 0;
          lpar ^= 1u;
        }
      }
    }
    if (!ok)  // copies under way land in this CTA's shared memory: wait for them (bounded)
      for (; c < loaded; ++c) {
        if (!mbar_wait(&full[st], par)) break;
        if (++st == S) {
          st = 0;
          par ^= 1u;
        }
      }
    umma_commit(done);
  }
  __syncwarp();
  if (!mbar_wait(done, 0)) ok = false;
  ok = __syncthreads_and(ok) != 0;
  if (!ok) latch_error(a.err, LS_ERR_TIMEOUT);
  tc_fence_after();
  const int q = warp & 3, r = 32 * q + lane;
  if (ok && m0 + r < J.M) store_tile(tmem + ((uint32_t)(32 * q) << 16), r, (warp >> 2) * (NT / 2), NT / 2, NT, smem);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  if (ok) copy_tile(J.C + ((int64_t)split * J.M + m0) * J.ldc + n0, J.ldc, J.M - m0, NT, smem, false);
  __syncwarp();
  if (warp == 0) tmem_dealloc(tmem, tcols);
}

// Minibatch gather: row j of the batch (slot idx[j], or (step*B + j) mod
// valid) z-scored and rounded to bf16 into img(A_0) and img(A_0^T); rows past
// the batch and columns past d are zero.  Thread = (row j, 8 columns).
struct GatherArgs {
  int B, rows_pad, d, d_pad;
  const int32_t* idx;
  DevState* st;
  int64_t capacity, replay_base;
  const float* ring_x;
  const float* ring_y;
  const float* mean;
  const float* stdv;
  uint8_t* a0;
  uint8_t* a0t;
  float* y;
  int* err;
};

// Items [first, total) with stride `stride` of the minibatch gather; `lead`:
// this thread also checks the buffer and sets the Adam bias corrections.
__device__ __forceinline__ void tr_gather_items(const GatherArgs& g, int64_t first, int64_t stride, bool lead) {
  const int B = g.B, rows_pad = g.rows_pad, d = g.d, d_pad = g.d_pad;
  const int32_t* __restrict__ idx = g.idx;
  const float* __restrict__ ring_x = g.ring_x;
  const float* __restrict__ ring_y = g.ring_y;
  const float* __restrict__ mean = g.mean;
  const float* __restrict__ stdv = g.stdv;
  uint8_t* __restrict__ a0 = g.a0;
  uint8_t* __restrict__ a0t = g.a0t;
  float* __restrict__ y = g.y;
  int* err = g.err;
  DevState* st = g.st;
  const int64_t step = st->step;
  const int64_t count = st->ring_count;
  const int64_t nF = count < g.capacity ? count : g.capacity;
  const int64_t valid = nF + st->replay_count;  // F u R
  const int64_t replay_base = g.replay_base;
  if (valid < 1 && lead) {
    latch_error(err, LS_ERR_STATE);
    st->train_abort = 1;  // the optimiser of this step leaves every parameter as it is
  }
  if (lead) set_adam_bc(st);
  const int total = rows_pad * (d_pad / 8);  // at most 2^31 / 16 rows of 128 columns
  // rows of a multiple of four columns are read as 16-byte vectors
  const bool vec = (d & 3) == 0;
  for (int64_t e = first; e < total; e += stride) {
    const int ei = (int)e;
    const int j = ei % rows_pad, c0 = (ei / rows_pad) * 8;
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = 0.0f;
    if (j < B && valid > 0) {  // an empty buffer (error latched above) reads nothing: zero rows
      int64_t slot;
      if (idx) {
        slot = idx[j];
        if (slot < 0 || slot >= valid) {
          if (c0 == 0) {
            latch_error(err, LS_ERR_ARG);
            st->train_abort = 1;
          }
          slot = 0;
        }
      } else {
        slot = valid > 0 ? (step * (int64_t)B + j) % valid : 0;
      }
      slot = union_row(slot, nF, replay_base);
      const float* row = ring_x + slot * d;
      if (vec && c0 + 8 <= d) {
        float x[8], mu[8], sd[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 xv = __ldg(reinterpret_cast<const float4*>(row + c0) + h);
          const float4 mv = __ldg(reinterpret_cast<const float4*>(mean + c0) + h);
          const float4 sv = __ldg(reinterpret_cast<const float4*>(stdv + c0) + h);
          x[4 * h] = xv.x, x[4 * h + 1] = xv.y, x[4 * h + 2] = xv.z, x[4 * h + 3] = xv.w;
          mu[4 * h] = mv.x, mu[4 * h + 1] = mv.y, mu[4 * h + 2] = mv.z, mu[4 * h + 3] = mv.w;
          sd[4 * h] = sv.x, sd[4 * h + 1] = sv.y, sd[4 * h + 2] = sv.z, sd[4 * h + 3] = sv.w;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = round_bf16(zscore(x[u], mu[u], sd[u]));
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c0 + u < d) v[u] = round_bf16(zscore(__ldg(row + c0 + u), __ldg(mean + c0 + u), __ldg(stdv + c0 + u)));
      }
      if (c0 == 0) y[j] = ring_y[slot];
    } else if (j < B && c0 == 0) {
      y[j] = 0.0f;
    }
    uint4 qv;
    qv.x = pack2(v[0], v[1]);
    qv.y = pack2(v[2], v[3]);
    qv.z = pack2(v[4], v[5]);
    qv.w = pack2(v[6], v[7]);
    *reinterpret_cast<uint4*>(a0 + sw128_offset(j, c0, rows_pad)) = qv;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      *reinterpret_cast<uint16_t*>(a0t + sw128_offset(c0 + u, j, d_pad)) = bf16_bits(v[u]);
  }
}

__global__ void k_tr_gather(const __grid_constant__ GatherArgs g) {
  pdl_wait();  // the ring and the device counters from the previous kernels of the stream
  pdl_trigger();
  tr_gather_items(g, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x,
                  blockIdx.x == 0 && threadIdx.x == 0);
}

struct OptLayer {
  const float* partW;  // [S][out][ld] split partials of dW (hidden) or [T][in] tile partials (output)
  int S;
  int ld;
  const float* partB;  // [T][out] (hidden) or [T] (output)
  uint8_t* imgW;       // [out rows, in_pad] image of bf16(W) (hidden layers)
  uint8_t* imgWT;      // [in_pad rows, out] image of bf16(W)^T
  int in_pad;
};

struct OptArgs {
  MlpDesc m;
  OptLayer L[LS_MAX_LAYERS];
  int T;               // row tiles of the batch
  int64_t n;           // parameters
  int mode;            // 0: images only, 1: SGD, 2: Adam
  float lr;
  float* p;
  float* mo;
  float* vo;
  DevState* st;
  const float* partLoss;
  int B;
  float* loss_out;
  // one-pass launch: block b holds 256 parameters of layer l, blk0[l] <= b <
  // blk0[l + 1], from the layer's first parameter on (opt_blocks)
  int blk0[LS_MAX_LAYERS + 1];
};

// Gradient (ordered sum of its partials), optimiser update and bf16 image
// writes of parameter e of layer l.  A step whose gather found no record or a
// bad slot (`aborted`) changes nothing: the images already hold the unchanged
// weights.
__device__ __forceinline__ void tr_opt_one(const OptArgs& a, int l, int64_t e, bool aborted, float bc1, float bc2) {
  const MlpDesc& m = a.m;
  const int out = m.w[l + 1], in = m.w[l];
  const OptLayer& P = a.L[l];
  const bool hidden = l + 1 < m.n_layers, is_w = e < m.boff[l];
  int o = 0, i = 0;
  if (is_w) {
    const int u = (int)(e - m.woff[l]);  // index within one layer's weights
    if (hidden) {
      o = u / in;
      i = u - o * in;
    } else {
      i = u;
    }
  } else {
    o = (int)(e - m.boff[l]);
  }
  float p = a.p[e];
  if (a.mode != 0) {
    // the moments do not depend on the gradient: their loads overlap the partials'
    float mo = 0.0f, vo = 0.0f;
    if (a.mode == 2) {
      mo = a.mo[e];
      vo = a.vo[e];
    }
    float g;
    if (hidden)
      g = is_w ? ordered_sum(P.partW + (int64_t)o * P.ld + i, P.S, (int64_t)out * P.ld)
               : ordered_sum(P.partB + o, a.T, out);
    else
      g = is_w ? ordered_sum(P.partW + i, a.T, P.ld) : ordered_sum(P.partB, a.T, 1);
    if (aborted) return;
    if (a.mode == 1) {
      p = p - a.lr * g;
    } else {
      const float me = 0.9f * mo + 0.1f * g;
      const float ve = 0.999f * vo + 0.001f * g * g;
      a.mo[e] = me;
      a.vo[e] = ve;
      const float mh = me / bc1, vh = ve / bc2;
      p = p - a.lr * mh / (sqrtf(vh) + 1e-8f);
    }
    a.p[e] = p;
  }
  if (hidden && is_w) {
    const uint16_t b = bf16_bits(p);
    *reinterpret_cast<uint16_t*>(P.imgW + sw128_offset(o, i, out)) = b;
    *reinterpret_cast<uint16_t*>(P.imgWT + sw128_offset(i, o, P.in_pad)) = b;
  }
}

// The gradient, the update of the fp32 master and the images of every parameter
// in [first, n) with stride `stride` (the persistent step).
__device__ __forceinline__ void tr_opt_items(const OptArgs& a, int64_t first, int64_t stride) {
  const MlpDesc& m = a.m;
  const int nl = m.n_layers;
  const bool aborted = a.mode != 0 && a.st->train_abort != 0;
  const float bc1 = a.st->adam_bc[0], bc2 = a.st->adam_bc[1];  // set by the gather kernel
  for (int64_t e = first; e < a.n; e += stride) {
    // the layer of parameter e: layer starts increase, so count those at or before e
    int l = 0;
#pragma unroll
    for (int k = 1; k < LS_MAX_LAYERS; ++k) l += (k < nl && e >= m.woff[k]) ? 1 : 0;
    tr_opt_one(a, l, e, aborted, bc1, bc2);
  }
}

// The minibatch loss (sum of the tile partials in order), by one warp: the
// lanes load 32 partials at once, every lane adds them in tile order, lane 0
// writes the result.
__device__ __forceinline__ void tr_loss_warp(const OptArgs& a) {
  if (a.mode != 0 && a.loss_out) {
    const int lane = threadIdx.x & 31;
    const bool abort = a.st->train_abort != 0;
    float s = 0.0f;
    for (int t0 = 0; t0 < a.T; t0 += 32) {
      const float v = t0 + lane < a.T ? a.partLoss[t0 + lane] : 0.0f;
      const int n = min(32, a.T - t0);
      for (int k = 0; k < n; ++k) s += __shfl_sync(0xffffffffu, v, k);
    }
    if (lane == 0) *a.loss_out = abort ? __int_as_float(0x7fc00000) : s / (float)a.B;
  }
}

__global__ void __launch_bounds__(256) k_tr_opt(const __grid_constant__ OptArgs a) {
  pdl_wait();  // gradient partials from the previous kernels of the stream
  pdl_trigger();
  const int64_t t = a.st->step + 1;
  const bool aborted = a.mode != 0 && a.st->train_abort != 0;
  const float bc1 = a.st->adam_bc[0], bc2 = a.st->adam_bc[1];  // set by the gather kernel
  {
    // this block's layer and parameters (one pass: a parameter per thread)
    const int nl = a.m.n_layers;
    int l = 0;
#pragma unroll
    for (int k = 1; k < LS_MAX_LAYERS; ++k) l += (k < nl && (int)blockIdx.x >= a.blk0[k]) ? 1 : 0;
    const int64_t e = a.m.woff[l] + (int64_t)((int)blockIdx.x - a.blk0[l]) * 256 + threadIdx.x;
    if (e < a.m.boff[l] + a.m.w[l + 1]) tr_opt_one(a, l, e, aborted, bc1, bc2);
  }
  if (blockIdx.x == 0 && threadIdx.x < 32) tr_loss_warp(a);
  // the last block, once every block has read the counter and the flag
  if (a.mode != 0 && last_block(&a.st->done[DONE_OPT]) && threadIdx.x == 0) {
    if (!aborted) advance_step(a.st, t);
    a.st->train_abort = 0;
  }
}

// ---------------------------------------------------------------------------
// The whole step as one persistent launch of a few CTAs (the rest of the GPU
// stays with routing): the gather, each product of the forward and backward
// passes (a phase: its tiles spread over the CTAs) and the optimiser, with a
// grid barrier between phases.  Same tiles, same epilogues and same order of
// every sum as the launch-per-phase path, so the same bits.
// ---------------------------------------------------------------------------
constexpr uint32_t kGridSpin = 1u << 21;  // barrier polls before giving up (a second or so)

struct StepArgs {
  GatherArgs g;
  TrArgs ph[kMaxPhases];
  int n_ph;
  OptArgs opt;
  uint32_t* bar;  // [0] arrivals, [1] abort flag; zero at launch
};
static_assert(sizeof(StepArgs) <= 32000, "kernel parameters of the persistent step");

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All CTAs meet (arrival `k` of each CTA: target k * gridDim.x).  Generic
// writes before it are visible to every read after it, bulk copies included.
// False for every CTA once one has given up (bounded wait) or failed a tile.
__device__ __forceinline__ bool tr_grid_sync(uint32_t* bar, uint32_t target, int* err) {
  __shared__ int s_go;
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile uint32_t* abort = bar + 1;
    __threadfence();
    atomicAdd(bar, 1u);
    int go = 1;
    for (uint32_t it = 0; ld_acquire_u32(bar) < target; ++it) {
      if (*abort || it >= kGridSpin) {
        if (!*abort) {
          atomicExch(bar + 1, 1u);
          latch_error(err, LS_ERR_TIMEOUT);
        }
        go = 0;
        break;
      }
      __nanosleep(64);
    }
    if (*abort) go = 0;
    s_go = go;
  }
  __syncthreads();
  asm volatile("fence.proxy.async.global;" ::: "memory");
  return s_go != 0;
}

__global__ void __launch_bounds__(kT, 1) k_tr_step(const __grid_constant__ StepArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(tr_tail(smem));
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(full + 2 * kMaxChunks + 1);
  const int tid = threadIdx.x;
  if (tid == 0) {
    for (int c = 0; c <= 2 * kMaxChunks; ++c) mbar_init(&full[c], 1);  // `full`, `done`, `used`
    fence_mbar_init();
  }
  if (tid < 32) {
    tmem_alloc(tmem_holder, 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  int* err = a.g.err;
  const int64_t first = blockIdx.x * (int64_t)kT + tid, stride = (int64_t)gridDim.x * kT;
  uint32_t arrivals = 0;
  tr_gather_items(a.g, first, stride, blockIdx.x == 0 && tid == 0);
  bool go = tr_grid_sync(a.bar, ++arrivals * gridDim.x, err);
  uint32_t par = 0;
  for (int ph = 0; go && ph < a.n_ph; ++ph) {
    const TrArgs& P = a.ph[ph];
    for (int b = blockIdx.x; b < P.n_cta; b += gridDim.x) {
      tr_tile_pre<false>(P, b, smem, true);
      if (!tr_tile<false>(P, b, smem, tmem, par, true, false)) {
        if (tid == 0) atomicExch(a.bar + 1, 1u);
        go = false;
        break;
      }
      par ^= 1u;
    }
    if (go) go = tr_grid_sync(a.bar, ++arrivals * gridDim.x, err);
  }
  if (go) {
    tr_opt_items(a.opt, first, stride);
    if (tr_grid_sync(a.bar, ++arrivals * gridDim.x, err) && blockIdx.x == 0 && tid < 32) {
      tr_loss_warp(a.opt);
      __syncwarp();  // every lane has read the abort flag before lane 0 clears it
      if (tid == 0 && a.opt.mode != 0) {
        if (!a.opt.st->train_abort) advance_step(a.opt.st, a.opt.st->step + 1);
        a.opt.st->train_abort = 0;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid < 32) tmem_dealloc(tmem, 256);
}

int gemm_smem_bytes() {
  return 1024 + kStageRegion + kTailBar + EpiSmem::kFloats * 4;
}

TrArgs tr_args(const Ctx& c, const TrJob& j0, const TrJob* j1, int* err) {
  TrArgs a{};
  a.st = c.st;
  a.drop_seed = c.cfg.dropout_seed;
  a.drop_thr = c.cfg.dropout > 0.0f ? (uint64_t)std::ceil((double)c.cfg.dropout * 9007199254740992.0) : 0;
  a.drop_scale = (float)(1.0 / (1.0 - (double)c.cfg.dropout));
  a.job[0] = j0;
  a.job[0].stages = tr_stages(j0.NT);
  a.n_cta0 = j0.m_tiles * j0.n_split * j0.splits;
  int n = a.n_cta0;
  if (j1) {
    a.job[1] = *j1;
    a.job[1].stages = tr_stages(j1->NT);
    n += j1->m_tiles * j1->n_split * j1->splits;
  }
  a.err = err;
  a.n_cta = n;
  return a;
}

template <bool RING, bool EMB>
cudaError_t launch_tr_as(const TrArgs& a, cudaStream_t s) {
  // the column parts of a TE_FWD_OUT tile exchange row sums through
  // distributed shared memory: one cluster per tile
  const int cl = a.job[0].epi == TE_FWD_OUT ? a.job[0].n_split : 1;
  return launch_smem<k_tr_gemm<RING, EMB>>(dim3(a.n_cta), dim3(kT), (size_t)gemm_smem_bytes(), s, cl, a);
}

cudaError_t launch_tr_args(const Ctx& c, const TrArgs& a, bool emb, cudaStream_t s) {
  if (emb) return c.tf.wide ? launch_tr_as<true, true>(a, s) : launch_tr_as<false, true>(a, s);
  return c.tf.wide ? launch_tr_as<true, false>(a, s) : launch_tr_as<false, false>(a, s);
}

cudaError_t launch_tr_gemm(const Ctx& c, const TrJob& j0, const TrJob* j1, int* err, cudaStream_t s) {
  return launch_tr_args(c, tr_args(c, j0, j1, err), false, s);
}

// Column parts per tile of a product with N columns: two when the columns
// split into halves that are multiples of 64 (each warp then owns a multiple
// of 16 columns); wider layers, 128 columns a part (see plan_train_fast).
int n_split_for(int N) { return N > 256 ? N / 128 : N % 128 == 0 ? 2 : 1; }

// Column parts of a hidden forward product (per-launch path) over T row
// tiles.  256 columns run as four 64-column parts (128 CTAs for a batch of
// 4096: half the epilogue and image stores per SM); wider layers as 128-column
// parts while those fill half the SMs, else 64-column ones.
int n_split_fwd(int N, int T, int sms) {
  if (N > 256) return T * (N / 128) >= sms / 2 ? N / 128 : N / 64;
  return N % 256 == 0 ? 4 : n_split_for(N);
}

// Column parts of the last hidden layer's product, which form a cluster: two
// halves, or four quarters of 512 columns (an accumulator has at most 256).
int n_split_out(int N) { return N == 512 ? 4 : N > 256 ? 2 : n_split_for(N); }

}  // namespace

namespace {

// Shape of the one-launch forward and input-gradient pass (k_tr_chain); CL 0:
// a launch per product.  The CTAs of a tile's cluster are the column parts of
// the output product, so that the row dot products add up in the same order;
// every hidden layer has to split into as many parts of whole K-blocks, and
// two copies of the operand tile and three K-blocks of weights have to fit:
// layers up to 256.  (With one copy and a cluster barrier per product, layers
// of 512 in clusters of four came out even at batch 4096, 55.7 us against
// 56.1, and behind at 256, 45.5 against 40.7: a rank's 32 KB for each of three
// others pass at some 11 bytes a cycle.)  Layers of up to 128 columns stay
// whole once two CTAs a tile would not all be resident; while they are, two are
// the better: 35.2 us against 39.4 at batch 4096 of 64-128-128-128-1 with
// dropout.
struct ChainPlan {
  int CL = 0, a_bytes = 0, stages = 0, stage_bytes = 0, nt_max = 0, smem = 0;
};
ChainPlan plan_chain(const MlpDesc& m, const TrainFast& f, int T, int sms) {
  ChainPlan p;
  const int nh = m.n_layers - 1;
  int w_max = 0;
  for (int l = 1; l <= nh; ++l) w_max = std::max(w_max, m.w[l]);
  const int parts = n_split_out(m.w[nh]);
  const int CL = w_max <= 128 && T * parts > sms ? 1 : parts;
  if (CL > 2) return p;
  for (int l = 1; l <= nh; ++l) {
    if (m.w[l] % (64 * CL) != 0 || m.w[l] / CL > 256) return p;
    p.nt_max = std::max(p.nt_max, m.w[l] / CL);
  }
  p.a_bytes = kM * std::max(f.in_pad[0], w_max) * 2;
  p.stage_bytes = p.nt_max * 128;
  const int fixed = 1024 + 2 * p.a_bytes + kChainBar + (EpiSmem::kFloats + kM) * 4;
  p.stages = std::min(kMaxRing, (kSmemMax - fixed) / p.stage_bytes);
  if (p.stages < 3) return p;
  p.smem = fixed + p.stages * p.stage_bytes;
  p.CL = CL;
  return p;
}

}  // namespace

// The fast path applies to bf16 predictors with at least one hidden layer,
// hidden widths that are multiples of 64 up to 256, or 384 or 512, and an
// input width of at most 256 (padded to 64).  Layers wider than 256 stream
// their K-blocks through the stages and split into parts of 128 columns; 320
// and 448 have no such split into equal parts for the output product's
// cluster of two or four and stay on the general path.  A step of
// 128-512-512-1 at batch 4096 took 214 us on the general path (22 launches,
// fp32 operands converted as they are staged) and takes 66 us here.
bool plan_train_fast(const MlpDesc& m, int max_batch, TrainFast& f) {
  f = TrainFast{};
  if (!m.bf16 || m.n_layers < 2) return false;
  f.in_pad[0] = ((m.w[0] + 63) / 64) * 64;
  if (f.in_pad[0] > 256) return false;
  for (int l = 1; l < m.n_layers; ++l) {
    const bool wide = m.w[l] == 384 || m.w[l] == 512;
    if (m.w[l] % 64 != 0 || (m.w[l] > 256 && !wide)) return false;
    f.wide = f.wide || wide;
    f.in_pad[l] = m.w[l];
  }
  f.rows_max = ((max_batch + kM - 1) / kM) * kM;
  f.on = true;
  f.chain = plan_chain(m, f, 1, 152).CL;
  return true;
}

// dz^T images: one a layer where the weight gradients run after the whole
// backward pass, else two by layer parity.
static int train_dzt_images(const MlpDesc& m, const TrainFast& f) {
  return f.chain ? std::max(2, m.n_layers - 1) : 2;
}

int64_t train_fast_bytes(const MlpDesc& m, const TrainFast& f, int64_t* parts_floats) {
  const int nh = m.n_layers - 1;
  const int64_t R = f.rows_max;
  int64_t bytes = 0;
  for (int l = 0; l < nh; ++l) bytes += 2 * R * f.in_pad[l] * 2;  // A_l, A_l^T
  int hmax = 0;
  for (int l = 1; l <= nh; ++l) hmax = std::max(hmax, m.w[l]);
  const int64_t hpad = ((hmax + 127) / 128) * 128;
  bytes += 2 * R * hmax * 2 + train_dzt_images(m, f) * hpad * R * 2;  // dz images and transposes
  for (int l = 1; l <= nh; ++l) bytes += (int64_t)(m.w[l] / 32) * R * 4;  // masks
  for (int l = 0; l < nh; ++l) bytes += 2 * (int64_t)m.w[l + 1] * f.in_pad[l] * 2;  // weight images
  const int64_t T = R / kM;
  int64_t pf = 0;
  for (int l = 0; l < nh; ++l) pf += (R / 128) * (int64_t)m.w[l + 1] * f.in_pad[l] + T * m.w[l + 1];
  pf += T * m.w[nh] + T + T;  // output layer weight / bias partials, loss partials
  *parts_floats = pf;
  return bytes;
}

// Carve the context's fast-path buffers out of one allocation.
void train_fast_bind(const MlpDesc& m, TrainFast& f, uint8_t* base, float* parts) {
  const int nh = m.n_layers - 1;
  const int64_t R = f.rows_max;
  uint8_t* p = base;
  for (int l = 0; l < nh; ++l) {
    f.imgA[l] = p;
    p += R * f.in_pad[l] * 2;
    f.imgAT[l] = p;
    p += R * f.in_pad[l] * 2;
  }
  int hmax = 0;
  for (int l = 1; l <= nh; ++l) hmax = std::max(hmax, m.w[l]);
  const int64_t hpad = ((hmax + 127) / 128) * 128;
  for (int b = 0; b < 2; ++b) {
    f.imgDZ[b] = p;
    p += R * hmax * 2;
  }
  for (int b = 0; b < train_dzt_images(m, f); ++b) {
    f.imgDZT[b] = p;
    p += hpad * R * 2;
  }
  for (int l = 1; l <= nh; ++l) {
    f.mask[l] = reinterpret_cast<uint16_t*>(p);
    p += (int64_t)(m.w[l] / 32) * R * 4;
  }
  for (int l = 0; l < nh; ++l) {
    f.imgW[l] = p;
    p += (int64_t)m.w[l + 1] * f.in_pad[l] * 2;
    f.imgWT[l] = p;
    p += (int64_t)m.w[l + 1] * f.in_pad[l] * 2;
  }
  const int64_t T = R / kM;
  float* q = parts;
  for (int l = 0; l < nh; ++l) {
    f.partW[l] = q;
    q += (R / 128) * (int64_t)m.w[l + 1] * f.in_pad[l];
    f.partB[l] = q;
    q += T * m.w[l + 1];
  }
  f.partWL = q;
  q += T * m.w[nh];
  f.partBL = q;
  q += T;
  f.partLoss = q;
}

// Blocks of the one-pass optimiser launch: 256 parameters each, within one
// layer.  Returns the grid size.
int opt_blocks(const MlpDesc& m, OptArgs& a) {
  int b = 0;
  for (int l = 0; l < m.n_layers; ++l) {
    a.blk0[l] = b;
    const int64_t n_l = m.boff[l] + m.w[l + 1] - m.woff[l];
    b += (int)((n_l + 255) / 256);
  }
  for (int l = m.n_layers; l <= LS_MAX_LAYERS; ++l) a.blk0[l] = b;
  return b;
}

// bf16 images of the master's hidden-layer weights (after ls_set_params).
cudaError_t train_fast_images(Ctx& c, cudaStream_t s) {
  const MlpDesc& m = c.mlp;
  TrainFast& f = c.tf;
  OptArgs a{};
  a.m = m;
  for (int l = 0; l + 1 < m.n_layers; ++l) {
    a.L[l].imgW = f.imgW[l];
    a.L[l].imgWT = f.imgWT[l];
    a.L[l].in_pad = f.in_pad[l];
  }
  a.n = c.n_params;
  a.mode = 0;
  a.p = c.master;
  a.st = c.st;
  const int grid = opt_blocks(m, a);
  k_tr_opt<<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

namespace {
GatherArgs gather_args(const Ctx& c, int B, const int32_t* idx) {
  GatherArgs g{};
  g.B = B;
  g.rows_pad = ((B + kM - 1) / kM) * kM;
  g.d = c.mlp.w[0];
  g.d_pad = c.tf.in_pad[0];
  g.idx = idx;
  g.st = c.st;
  g.capacity = c.cfg.ring_capacity;
  g.replay_base = c.replay_base;
  g.ring_x = c.ring_x;
  g.ring_y = c.ring_y;
  g.mean = c.mean;
  g.stdv = c.stdv;
  g.a0 = c.tf.imgA[0];
  g.a0t = c.tf.imgAT[0];
  g.y = c.ty;
  g.err = c.d_err;
  return g;
}
}  // namespace

cudaError_t run_train_fast(Ctx& c, int B, const int32_t* idx, int opt, float lr, float* loss_out, cudaStream_t s) {
  const MlpDesc& m = c.mlp;
  TrainFast& f = c.tf;
  const int nh = m.n_layers - 1;  // hidden layers 0..nh-1, output layer nh
  const int R = ((B + kM - 1) / kM) * kM;
  const int T = R / kM;
  // one persistent launch (the products become its phases) or one launch each
  const bool one = c.train_ctas > 0;
  const bool chain = !one && f.chain > 0;
  const ChainPlan cp = chain ? plan_chain(m, f, T, c.sms) : ChainPlan{};
  ChainArgs ca{};
  DwArgs da{};
  int dw_ctas = 0;
  auto chain_phase = [&](const TrJob& J, int K, bool feeds) {
    ChainPhase& P = ca.ph[ca.n++];
    P.epi = J.epi;
    P.nk = K / 64;
    P.NT = J.NT * J.n_split / cp.CL;
    P.feeds = feeds;
    P.B = J.B;
    P.bias = J.bias;
    P.outT = J.outT;
    P.rT = J.rT;
    P.drop_h = J.drop_h;
    P.mask = J.epi == TE_DX ? const_cast<uint16_t*>(J.mask_in) : J.mask_out;
    P.colpart = J.colpart;
  };
  const auto dzt = [&](int l) { return f.imgDZT[chain ? l : l & 1]; };
  static thread_local StepArgs step;
  step = StepArgs{};
  cudaError_t e = cudaSuccess;
  if (!one) {
    e = traced(c, TR_GATHER, 1, s, [&] {
      const int64_t total = (int64_t)R * (f.in_pad[0] / 8);
      const int grid = (int)std::min<int64_t>((total + 255) / 256, (int64_t)c.sms * 8);
      // Long rows that are not whole 16-byte vectors are read word by word and
      // live on L1, which an SM that still runs the step before has set to
      // shared memory: then the gather waits for that step before it starts.
      // (Steps issued one by one, 246-256-1: 8192 rows 42 us chained, 35 so;
      // 32,768 rows 128, 102; 129-256-1 at 16,384 57, 50.  The chained launch is
      // the faster one for short rows, 29-128-1 at 2048 rows 19 us against 21,
      // and small batches.)
      if ((m.w[0] & 3) != 0 && m.w[0] > 64 && R >= 2048) {
        k_tr_gather<<<grid, 256, 0, s>>>(gather_args(c, B, idx));
        return cudaGetLastError();
      }
      return launch_chained(k_tr_gather, dim3(grid), dim3(256), 0, s, 1, gather_args(c, B, idx));
    });
    if (e != cudaSuccess) return e;
  }
  // forward: hidden layers; the last one also runs the output layer and the loss
  for (int l = 0; l < nh; ++l) {
    const bool last = l == nh - 1;
    TrJob J{};
    J.epi = last ? TE_FWD_OUT : TE_FWD;
    J.m_tiles = T;
    // the persistent launch has no clusters: the output layer's row dot
    // products stay within one CTA (all columns of the tile)
    const int N = m.w[l + 1];
    J.n_split = one ? (last ? 1 : n_split_for(N)) : last ? n_split_out(N) : n_split_fwd(N, T, c.sms);
    J.splits = 1;
    J.nchunks = J.kblocks = f.in_pad[l] / 64;
    J.NT = m.w[l + 1] / J.n_split;
    J.A = f.imgA[l];
    J.rA = R;
    J.B = f.imgW[l];
    J.M = R;
    J.bias = c.master + m.boff[l];
    J.rows_pad = R;
    if (!last) {
      J.out = f.imgA[l + 1];
      J.outT = f.imgAT[l + 1];
      J.rT = f.in_pad[l + 1];
      J.mask_out = f.mask[l + 1];
    } else {
      J.out = l > 0 ? f.imgDZ[l & 1] : nullptr;
      J.outT = dzt(l);
      J.rT = ((m.w[l + 1] + 127) / 128) * 128;
      J.colpart = f.partB[l];
      J.wL = c.master + m.woff[nh];
      J.bL = c.master + m.boff[nh];
      J.y = c.ty;
      J.batch = B;
      J.partWL = f.partWL;
      J.partBL = f.partBL;
      J.partLoss = f.partLoss;
    }
    // dropout on hidden activation l + 1 when it feeds another hidden layer
    J.drop_h = (c.cfg.dropout > 0.0f && l + 2 < m.n_layers) ? l + 1 : 0;
    if (one) {
      step.ph[step.n_ph++] = tr_args(c, J, nullptr, c.d_err);
      continue;
    }
    if (chain) {
      chain_phase(J, f.in_pad[l], !last || nh > 1);
      if (last) ca.out = OutLayer{J.bL, J.y, J.batch, J.partWL, J.partBL, J.partLoss, nullptr};
      continue;
    }
    e = traced(c, TR_GEMM_TC_FWD, 1, s, [&] { return launch_tr_gemm(c, J, nullptr, c.d_err, s); });
    if (e != cudaSuccess) return e;
  }
  // backward: dW_l (split over the batch) and, for l > 0, dz_{l-1} in the same launch
  for (int l = nh - 1; l >= 0; --l) {
    const int out = m.w[l + 1];
    TrJob W{};
    W.epi = TE_STORE;
    W.m_tiles = (out + kM - 1) / kM;
    W.n_split = n_split_for(f.in_pad[l]);
    // K-blocks (of 64 batch rows) per CTA: 4 when that still gives 48 CTAs,
    // else 2 (more CTAs, more partials for the optimiser to add); 8 where a
    // wide layer's parts give 96 CTAs all the same (half the partials)
    const int parts = W.m_tiles * W.n_split;
    const int kpc = f.wide && parts * (R / 512) >= 96 ? 8 : parts * (R / 256) >= 48 ? 4 : 2;
    W.kblocks = R / 64;
    W.nchunks = std::min(kpc, W.kblocks);
    W.splits = (W.kblocks + W.nchunks - 1) / W.nchunks;  // the last one may be short
    W.NT = f.in_pad[l] / W.n_split;
    W.A = dzt(l);
    W.rA = ((out + 127) / 128) * 128;
    W.B = f.imgAT[l];
    W.M = out;
    W.C = f.partW[l];
    W.ldc = f.in_pad[l];
    W.split_stride = (int64_t)out * f.in_pad[l];
    f.splits[l] = W.splits;
    TrJob X{};
    if (l > 0) {
      X.epi = TE_DX;
      X.m_tiles = T;
      X.n_split = n_split_for(m.w[l]);
      X.splits = 1;
      X.nchunks = X.kblocks = out / 64;
      X.NT = m.w[l] / X.n_split;
      X.A = f.imgDZ[l & 1];
      X.rA = R;
      X.B = f.imgWT[l];
      X.M = R;
      X.rows_pad = R;
      X.mask_in = f.mask[l];
      X.out = l > 1 ? f.imgDZ[(l - 1) & 1] : nullptr;
      X.outT = dzt(l - 1);
      X.rT = ((m.w[l] + 127) / 128) * 128;
      X.colpart = f.partB[l - 1];
      X.drop_h = (c.cfg.dropout > 0.0f && l < m.n_layers - 1) ? l : 0;  // input a_l was dropped
    }
    if (one) {
      step.ph[step.n_ph++] = tr_args(c, W, l > 0 ? &X : nullptr, c.d_err);
      continue;
    }
    if (chain) {
      if (l > 0) chain_phase(X, out, l > 1);
      da.cta0[da.n] = dw_ctas;
      DwJob& D = da.job[da.n++];
      D = DwJob{W.A, W.B, W.C, W.rA, W.M, W.ldc, W.NT, W.n_split, W.m_tiles, W.nchunks, W.kblocks, 0};
      D.stages = std::min({kMaxRing, W.nchunks, kDwStage / ((kM + W.NT) * 128)});
      dw_ctas += W.m_tiles * W.n_split * W.splits;
      continue;
    }
    e = traced(c, l > 0 ? TR_GEMM_TC_DX : TR_GEMM_TC_DW, 1, s,
               [&] { return launch_tr_gemm(c, W, l > 0 ? &X : nullptr, c.d_err, s); });
    if (e != cudaSuccess) return e;
  }
  if (chain) {
    for (int p = 0; p < ca.n; ++p)
      for (int r = 0; r < 2; ++r)
        ca.ph[p].stage[r] = (p & 1) * cp.a_bytes +
                            chain::stage_block(cp.CL, r, ca.ph[p].NT, ca.ph[p + (p + 1 < ca.n)].NT) * kM * 128;
    ca.CL = cp.CL;
    ca.a_bytes = cp.a_bytes;
    ca.stages = cp.stages;
    ca.stage_bytes = cp.stage_bytes;
    ca.tmem_cols = 32;
    while ((int)ca.tmem_cols < cp.nt_max) ca.tmem_cols <<= 1;
    ca.A0 = f.imgA[0];
    ca.R = R;
    ca.wL = c.master + m.woff[nh];
    const TrArgs t = tr_args(c, TrJob{}, nullptr, c.d_err);  // (the dropout stream)
    ca.err = t.err;
    ca.st = t.st;
    ca.drop_seed = t.drop_seed;
    ca.drop_thr = t.drop_thr;
    ca.drop_scale = t.drop_scale;
    e = traced(c, TR_GEMM_TC_FWD, 1, s, [&] {
      return launch_smem<k_tr_chain>(dim3(T * cp.CL), dim3(kChainT), (size_t)cp.smem, s, cp.CL, ca);
    });
    if (e != cudaSuccess) return e;
    da.err = c.d_err;
    e = traced(c, TR_GEMM_TC_DW, 1, s, [&] {
      const int smem = 1024 + kDwStage + (2 * kMaxRing + 2) * 8;
      return launch_smem<k_tr_dw>(dim3(dw_ctas), dim3(kDwT), (size_t)smem, s, 1, da);
    });
    if (e != cudaSuccess) return e;
  }
  OptArgs a{};
  a.m = m;
  for (int l = 0; l < nh; ++l) {
    a.L[l].partW = f.partW[l];
    a.L[l].S = f.splits[l];
    a.L[l].ld = f.in_pad[l];
    a.L[l].partB = f.partB[l];
    a.L[l].imgW = f.imgW[l];
    a.L[l].imgWT = f.imgWT[l];
    a.L[l].in_pad = f.in_pad[l];
  }
  a.L[nh].partW = f.partWL;
  a.L[nh].ld = m.w[nh];
  a.L[nh].partB = f.partBL;
  a.T = T;
  a.n = c.n_params;
  a.mode = opt == LS_SGD ? 1 : 2;
  a.lr = lr;
  a.p = c.master;
  a.mo = c.adam_m;
  a.vo = c.adam_v;
  a.st = c.st;
  a.partLoss = f.partLoss;
  a.B = B;
  a.loss_out = loss_out ? loss_out : c.loss_tmp;
  if (one) {
    step.g = gather_args(c, B, idx);
    step.opt = a;
    step.bar = c.tr_bar;
    return traced(c, TR_TRAIN_STEP, 1, s, [&] {
      cudaError_t e2 = cudaMemsetAsync(c.tr_bar, 0, 2 * sizeof(uint32_t), s);
      if (e2 != cudaSuccess) return e2;
      const int smem = gemm_smem_bytes();
      e2 = allow_smem<k_tr_step>();
      if (e2 != cudaSuccess) return e2;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(c.train_ctas);
      cfg.blockDim = dim3(kT);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: the grid barrier needs it
      attr[0].val.cooperative = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      return cudaLaunchKernelEx(&cfg, k_tr_step, step);
    });
  }
  return traced(c, TR_OPT, 1, s, [&] {
    const int grid = opt_blocks(m, a);
    return launch_chained(k_tr_opt, dim3(grid), dim3(256), 0, s, 1, a);
  });
}

// ---------------------------------------------------------------------------
// Replay admission's embeddings on the operand images (k_replay.cu)
// ---------------------------------------------------------------------------
namespace {

struct EmbGather {
  int rows, tiles_cand, d, d_pad;  // rows of the image: the candidates' tiles, then the kept records'
  int64_t C, P, base;              // FIFO and pending capacities, first replay row
  const int64_t* counts;           // candidates, kept records
  const DevState* st;
  const float* ring_x;
  const float* ring_y;
  const float* mean;
  const float* stdv;
  uint8_t* a0;
  float* y;
};

// Image rows of the round's records, z-scored and rounded to bf16 (thread =
// (row, 8 columns)); rows past a tile's records are zero, tiles past them are
// left alone.
__global__ void __launch_bounds__(256) k_emb_gather(const __grid_constant__ EmbGather g) {
  pdl_wait();
  pdl_trigger();
  const int64_t m = g.counts[0], nr = g.counts[1];
  const int64_t count = g.st->ring_count, hi = count > g.C ? count - g.C : 0, lo = hi - m;
  const int rc = g.tiles_cand * kM;
  const bool vec = (g.d & 3) == 0;
  const int total = g.rows * (g.d_pad / 8);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int j = e % g.rows, c0 = (e / g.rows) * 8;
    const int64_t i = j < rc ? j : j - rc, used = j < rc ? m : nr;
    if ((i & ~(int64_t)(kM - 1)) >= used) continue;
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = 0.0f;
    float y = 0.0f;
    if (i < used) {
      const int64_t slot = j < rc ? g.C + (lo + i) % g.P : g.base + i;
      const float* row = g.ring_x + slot * g.d;
      if (vec && c0 + 8 <= g.d) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 xv = __ldg(reinterpret_cast<const float4*>(row + c0) + h);
          const float4 mv = __ldg(reinterpret_cast<const float4*>(g.mean + c0) + h);
          const float4 sv = __ldg(reinterpret_cast<const float4*>(g.stdv + c0) + h);
          v[4 * h] = zscore(xv.x, mv.x, sv.x);
          v[4 * h + 1] = zscore(xv.y, mv.y, sv.y);
          v[4 * h + 2] = zscore(xv.z, mv.z, sv.z);
          v[4 * h + 3] = zscore(xv.w, mv.w, sv.w);
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c0 + u < g.d) v[u] = zscore(__ldg(row + c0 + u), __ldg(g.mean + c0 + u), __ldg(g.stdv + c0 + u));
      }
      if (c0 == 0) y = g.ring_y[slot];
    }
    if (c0 == 0) g.y[j] = y;
    *reinterpret_cast<uint4*>(g.a0 + sw128_offset(j, c0, g.rows)) =
        make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
  }
}

// The gradient embeddings of the round, a warp per image row: yhat from the
// last hidden activations (bf16 weights, lanes along them), g = (yhat - y) a
// in bf16 into the embedding image (tiles of 128 rows, a tile's K-blocks
// together) and |bf16(g)|^2 of the rows in use, every sum in the order of the
// general path's k_out_fwd and k_replay_embed.
struct EmbRows {
  int rows, tiles_cand, H;
  int64_t P;
  const int64_t* counts;
  const uint8_t* a;  // image of the last hidden activations
  const float* w;    // output layer
  const float* b;
  const float* y;
  uint8_t* img;
  float* norm;       // [P] candidates, then kept records
};

__global__ void __launch_bounds__(256) k_emb_rows(const __grid_constant__ EmbRows g) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31, rc = g.tiles_cand * kM;
  const int64_t m = g.counts[0], nr = g.counts[1];
  for (int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < g.rows; j += (gridDim.x * blockDim.x) >> 5) {
    const bool kept = j >= rc;
    const int64_t i = kept ? j - rc : j, used = kept ? nr : m;
    if ((i & ~(int64_t)(kM - 1)) >= used) continue;  // a tile without records
    float av[8], z = 0.0f;  // H <= 256
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = lane + 32 * u;
      av[u] = k < g.H ? __uint_as_float((uint32_t)*reinterpret_cast<const uint16_t*>(g.a + sw128_offset(j, k, g.rows)) << 16)
                      : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (lane + 32 * u < g.H) z = fmaf(av[u], round_bf16(__ldg(g.w + lane + 32 * u)), z);
#pragma unroll
    for (int o = 16; o; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const float res = (z + __ldg(g.b)) - g.y[j];
    uint8_t* tile = g.img + (int64_t)(j / kM) * kM * g.H * 2;
    float s = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = lane + 32 * u;
      if (k >= g.H) break;
      const uint16_t b = bf16_bits(res * av[u]);
      const float bv = __uint_as_float((uint32_t)b << 16);
      s = fmaf(bv, bv, s);
      *reinterpret_cast<uint16_t*>(tile + sw128_offset(j % kM, k, kM)) = b;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0 && i < used) g.norm[(kept ? g.P : 0) + i] = s;
  }
}

// Widest image of the embedding forward: layer inputs and the last hidden
// activations.
int emb_width(const MlpDesc& m, const TrainFast& f) {
  int w = m.w[m.n_layers - 1];
  for (int l = 0; l + 1 < m.n_layers; ++l) w = std::max(w, f.in_pad[l]);
  return w;
}

}  // namespace

// Bytes of the two activation images and the targets of an admission round
// over `rows` image rows (0: the embeddings run through the general forward).
int64_t replay_embed_bytes(const MlpDesc& m, const TrainFast& f, int64_t rows) {
  return f.on ? 2 * rows * emb_width(m, f) * 2 + rows * 4 : 0;
}

// Embeddings of the round whose counts and reset norms k_replay_prep left:
// gather, the hidden layers, the embedding rows.  (In chunks of the training
// batch through the general forward, fp32 operands staged by every product:
// 15 launches for pools of 5000; an admission round of 1000 candidates took
// 160 us, 65 us on the images.)
cudaError_t replay_embed_fast(Ctx& c, int64_t P, int64_t Rc, cudaStream_t s) {
  const MlpDesc& m = c.mlp;
  TrainFast& f = c.tf;
  const int nh = m.n_layers - 1;
  const int tc = (int)((P + kM - 1) / kM), T = tc + (int)((Rc + kM - 1) / kM), rows = T * kM;
  const int pad = emb_width(m, f);
  uint8_t* img[2] = {c.remb_img, c.remb_img + (int64_t)rows * pad * 2};
  float* y = reinterpret_cast<float*>(c.remb_img + 2 * (int64_t)rows * pad * 2);
  EmbGather g{};
  g.rows = rows;
  g.tiles_cand = tc;
  g.d = m.w[0];
  g.d_pad = f.in_pad[0];
  g.C = c.cfg.ring_capacity;
  g.P = P;
  g.base = c.replay_base;
  g.counts = c.rcount;
  g.st = c.st;
  g.ring_x = c.ring_x;
  g.ring_y = c.ring_y;
  g.mean = c.mean;
  g.stdv = c.stdv;
  g.a0 = img[0];
  g.y = y;
  cudaError_t e = traced(c, TR_REPLAY, 1, s, [&] {
    const int64_t total = (int64_t)rows * (g.d_pad / 8);
    const int grid = (int)std::min<int64_t>((total + 255) / 256, (int64_t)c.sms * 8);
    return launch_chained(k_emb_gather, dim3(grid), dim3(256), 0, s, 1, g);
  });
  for (int l = 0; e == cudaSuccess && l < nh; ++l) {
    const int N = m.w[l + 1];
    TrJob J{};
    J.epi = TE_FWD;
    J.m_tiles = T;
    J.n_split = n_split_fwd(N, T, c.sms);
    J.splits = 1;
    J.nchunks = J.kblocks = f.in_pad[l] / 64;
    J.NT = N / J.n_split;
    J.A = img[l & 1];
    J.rA = rows;
    J.B = f.imgW[l];
    J.M = rows;
    J.bias = c.master + m.boff[l];
    J.rows_pad = rows;
    J.out = img[(l + 1) & 1];
    TrArgs a = tr_args(c, J, nullptr, c.d_err);
    a.counts = c.rcount;
    a.tiles_cand = tc;
    e = traced(c, TR_REPLAY, 1, s, [&] { return launch_tr_args(c, a, true, s); });
  }
  if (e != cudaSuccess) return e;
  EmbRows r{};
  r.rows = rows;
  r.tiles_cand = tc;
  r.H = m.w[nh];
  r.P = P;
  r.counts = c.rcount;
  r.a = img[nh & 1];
  r.w = c.master + m.woff[nh];
  r.b = c.master + m.boff[nh];
  r.y = y;
  r.img = c.rimg;
  r.norm = c.rnorm;
  return traced(c, TR_REPLAY, 1, s, [&] {
    const int grid = std::min((rows + 7) / 8, c.sms * 8);
    return launch_chained(k_emb_rows, dim3(grid), dim3(256), 0, s, 1, r);
  });
}

}  // namespace ls
