// Sequential-commit routing (Sec. 4.2 cluster snapshot manager and prefix
// KV-cache tracker; Sec. 4.3.1 P1: the gateway routes one request at a time):
// the requests of a batch are routed in order, and each decision is committed
// before the next request is scored -- the chosen instance's queue count grows
// by one and the prompt's full blocks join its cache (the prefix index gains
// the instance's bit for each block key), so a later request with the same
// prefix sees the hit and the longer queue.
//
// The chain of decisions is inherently serial, so what bounds the call is the
// latency of one step.  One cluster of up to eight CTAs walks the requests;
// the instances are split over the CTAs (each holds all weights in shared
// memory and a few instances' rows), and the warps of a CTA work on three
// requests at once:
//   - eight warps score request s (the predictor on CUDA cores, each sum in K
//     order) and send each warp's lowest (score, index) to its slot in every
//     CTA of the cluster;
//   - six warps look up the block keys of request s + 1, z-score its extras
//     and turn the instance masks into hit lengths and pair features, in two
//     versions per instance: as if request s went elsewhere, and as if it went
//     there; two warps insert request s - 1's keys for its chosen instance.
// The slots are written by remote stores that count their bytes on a barrier
// in the receiving CTA, so a step waits for the other CTAs' bids and nothing
// else; nothing on its path is read from global memory (weights, biases and
// the layers' shapes are in shared memory).  The masks looked up for request
// s + 1 hold the commits up to request s - 4 for certain (the lookups start
// with the bids for s - 1, which a CTA sends once its inserting warps have
// finished with s - 4); those of the four requests since are added when the
// masks are read: a block whose key equals the earlier request's key at the
// same position is also held by the instance that request went to (a flag per
// block and earlier request; equal prefixes give equal keys, and a key is only
// ever inserted with its request).
// Measured on 64 requests over 16 instances with 64-128-128-128-1: 3.8 us
// a request (of 18.5 with one CTA doing every stage in turn, a barrier after
// each); the bids' travel, the layers' shared-memory loads and a few hundred
// instructions that each step runs once bound it.
#include "blockhash.cuh"
#include "common.cuh"
#include "seq_steps.h"
#include "sm100.cuh"

namespace ls {
namespace {
using namespace bh;
using namespace sm100;

constexpr int kSeqHalf = 256;          // threads that score
constexpr int kSeqLook = 192;          // threads that look up
constexpr int kSeqIns = 64;            // threads that insert
constexpr int kSeqThreads = kSeqHalf + kSeqLook + kSeqIns;
constexpr int kSeqWarps = kSeqHalf / 32;
constexpr int kSeqCluster = 8;         // CTAs at most
constexpr int kSeqMaxW = 8;            // instance-mask words (512 instances)

struct SeqArgs {
  int n_req, n_inst, d_inst, d_req, q_col;
  const int64_t* tok_off;
  const uint64_t* bkeys;  // block keys of the batch at (tok_off[r] - tok_off[0]) / 16 + b
  int64_t bcap;
  const float* req;
  float* inst;            // [n_inst, d_inst] instance rows (updated in place at the end)
  const float* mean;
  const float* stdv;
  const float* params0;
  const float* params1;
  const DevState* st;
  MlpDesc m;
  int rows;               // instances a CTA has at most
  int xs;                 // elements per activation row (a multiple of 8)
  int bids;               // bids a request gets: warps with a row, over all CTAs
  int wsm;                // 1: the weights are copied into shared memory once per call
  int64_t wbytes;         // size of that weight region
  int woff_s[LS_MAX_LAYERS];      // byte offset of hidden layer l's weights in it
  int hidden_out;         // outputs of all hidden layers
  uint64_t* gkeys;
  uint64_t* gmask;
  uint64_t gslots_mask;
  int32_t* counts;
  int64_t max_keys;
  int32_t* choice;
  float* best;
  float* scores;          // [n_req, n_inst] or NULL
  int32_t* hits;          // [n_req, n_inst] or NULL
  int* err;
};

// Blocks of a prompt whose masks are looked up a request ahead (longer
// prompts' later blocks are looked up when a row still matches there).
constexpr int seq_blocks(int W) { return (W <= 2 ? 3 : 1) * kSeqLook; }

// Index lookups through L2 (ld.global.cg), so that keys the cluster inserted are seen.
template <int W>
__device__ __forceinline__ void seq_lookup(const SeqArgs& a, uint64_t key, uint64_t (&mw)[W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) mw[w] = 0;
  const uint64_t mslots = a.gslots_mask;
  uint64_t s = key & mslots;
  for (uint64_t n = 0; n <= mslots; ++n) {
    if (W == 1) {
      const ulonglong2 e = __ldcg(reinterpret_cast<const ulonglong2*>(a.gkeys) + s);
      if (e.x == key) mw[0] = e.y;
      if (e.x == key || e.x == 0) return;
    } else {
      const uint64_t k = __ldcg(a.gkeys + s);
      if (k == key) {
#pragma unroll
        for (int w = 0; w < W; ++w) mw[w] = __ldcg(a.gmask + s * W + w);
        return;
      }
      if (k == 0) return;
    }
    s = (s + 1) & mslots;
  }
}

// Insertion of `key` for instance `inst` (the protocol of the snapshot's index
// insert: CAS on an empty slot, OR of the instance's bit); true when the bit
// is newly set (one more distinct key of the instance).
template <int W>
__device__ __forceinline__ bool seq_insert(const SeqArgs& a, uint64_t key, int inst) {
  unsigned long long* tab = reinterpret_cast<unsigned long long*>(a.gkeys);
  const int kstride = W == 1 ? 2 : 1;
  uint64_t s = key & a.gslots_mask;
  int64_t slot = -1;
  for (uint64_t n = 0; n <= a.gslots_mask; ++n) {
    const unsigned long long prev = atomicCAS(tab + s * kstride, 0ull, (unsigned long long)key);
    if (prev == 0ull || prev == key) { slot = (int64_t)s; break; }
    s = (s + 1) & a.gslots_mask;
  }
  if (slot < 0) { latch_error(a.err, LS_ERR_TABLE_FULL); return false; }
  const unsigned long long bit = 1ull << (inst & 63);
  unsigned long long* mword = W == 1 ? tab + 2 * slot + 1
                                     : reinterpret_cast<unsigned long long*>(a.gmask + slot * W + (inst >> 6));
  return !(atomicOr(mword, bit) & bit);
}

// (score, instance) as one key whose unsigned order is the selection order:
// NaN after every number, -0 equal to +0, ties to the lower index.
__device__ __forceinline__ uint64_t seq_code(float v, int i) {
  const uint32_t c = v != v ? 0xffffffffu : ord_code(v == 0.0f ? 0.0f : v);
  return ((uint64_t)c << 32) | (uint32_t)i;
}

// v into the 64-bit word at `slot`, its eight bytes counted on the barrier at
// `bar` (addresses in the same CTA of the cluster).
__device__ __forceinline__ void seq_remote_store(uint32_t slot, uint32_t bar, uint64_t v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(slot), "l"(v),
               "r"(bar)
               : "memory");
}

// Waits (bounded) for the bids of a request; once a wait of the CTA has given
// up, none waits any more and the call runs to its end (error latched).  From
// then on the CTA sends no bids, so the others, each after its own wait, stop
// too instead of joining bids of different requests; every CTA comes to the
// cluster barrier at the kernel's end, and none leaves before it.
__device__ __forceinline__ void seq_wait(uint64_t* bar, uint32_t parity, volatile int* gave_up, int* err) {
  if (mbar_try_wait(bar, parity)) return;
  const long long t0 = clock64();
  while (!*gave_up && !mbar_try_wait(bar, parity))
    if (clock64() - t0 > kWaitCycles) {
      *gave_up = 1;
      latch_error(err, LS_ERR_TIMEOUT);
    }
}

// The instance of the lowest of the n (at most 64) codes at `slot`, in every
// lane of the warp.
__device__ __forceinline__ int seq_select(const volatile uint64_t* slot, int n) {
  const int lane = threadIdx.x & 31;
  uint64_t v = lane < n ? slot[lane] : ~0ull;
  const uint64_t u = lane + 32 < n ? slot[lane + 32] : ~0ull;
  v = u < v ? u : v;
  const uint32_t hi = __reduce_min_sync(kFull, (uint32_t)(v >> 32));
  return (int)__reduce_min_sync(kFull, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0xffffffffu);
}

// The barriers below are warp-aligned instructions: the lanes come together first.
__device__ __forceinline__ void seq_half_sync() {
  __syncwarp();
  named_bar_sync(1, kSeqHalf);
}

struct SeqMeta {
  int64_t L, nb, k0;  // prompt length, full blocks, first block key
};

struct SeqLayer {
  int in, out, w, b;  // widths, weights (byte offset), biases (index)
  float inv_out;      // 1 / out
  int rt;             // rows a thread takes (0: weights in global memory)
};

// Byte offsets of the shared-memory arrays (each 16-byte aligned).  Layer
// inputs and activations take `xe` bytes each: 2 in bf16 mode (their values
// are bf16-rounded, so bf16 holds them exactly), 4 in fp32 mode.
// The weight region (`wbytes`, 0 when the weights stay in global memory)
// holds layer l's weights with the outputs adjacent: fp32 W[k][out], or bf16
// pairs (k, k + 1) as [k / 2][out] words (an odd K padded with 0).
struct SeqSmem {
  size_t inst, x0, x1, x2, sc, pre, mask, flag, meta, cand, bar, lay, bias, wl, w, total;
};
__host__ __device__ __forceinline__ size_t seq_al(size_t b) { return (b + 15) & ~(size_t)15; }
__host__ __device__ __forceinline__ SeqSmem seq_smem(int rows, int DI, int xs, int W, int xe, int hidden_out,
                                                     size_t wbytes) {
  SeqSmem o;
  const size_t nb = (size_t)seq_blocks(W);
  o.inst = 0;                                                      // [rows][d_inst]
  o.x0 = seq_al(o.inst + (size_t)rows * (DI > 0 ? DI : 1) * 4);    // [2][rows][xs] feature rows (requests in turn)
  o.x1 = seq_al(o.x0 + 2 * (size_t)rows * xs * xe);                // [rows][xs] activations
  o.x2 = seq_al(o.x1 + (size_t)rows * xs * xe);                    // [rows][xs] activations
  o.sc = seq_al(o.x2 + (size_t)rows * xs * xe);                    // [rows] scores
  o.pre = seq_al(o.sc + (size_t)rows * 4);                         // [2][rows][2][8] pair features and hit length
  o.mask = seq_al(o.pre + 2 * (size_t)rows * 64);                  // [blocks][W] instance masks
  o.flag = seq_al(o.mask + nb * W * 8);                            // [blocks] keys shared with the four before
  o.meta = seq_al(o.flag + nb);                                    // [8]
  o.cand = seq_al(o.meta + 8 * sizeof(SeqMeta));                   // [4][64] bids
  o.bar = seq_al(o.cand + 4 * 64 * 8);                             // [4] barriers of the bids, then a flag
  o.lay = seq_al(o.bar + 4 * 8 + 16);                              // hidden layers
  o.bias = seq_al(o.lay + LS_MAX_LAYERS * sizeof(SeqLayer));       // their biases
  o.wl = seq_al(o.bias + (size_t)hidden_out * 4);                  // [xs] output-layer weights
  o.w = seq_al(o.wl + (size_t)xs * 4);                             // hidden-layer weights (optional)
  o.total = seq_al(o.w + wbytes);
  return o;
}

// Activation element i as fp32 / stored (rounded to bf16 in bf16 mode).
template <bool BF>
__device__ __forceinline__ float seq_xget(const uint8_t* X, int i) {
  return BF ? __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(X)[i] << 16)
            : reinterpret_cast<const float*>(X)[i];
}
template <bool BF>
__device__ __forceinline__ void seq_xset(uint8_t* X, int i, float v) {
  if (BF) reinterpret_cast<__nv_bfloat16*>(X)[i] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(X)[i] = v;
}

// acc + x.lo w.lo + x.hi w.hi, added in that order: two fp32 fused
// multiply-adds of bf16 inputs.
__device__ __forceinline__ void seq_fma_pair(uint32_t x, uint32_t w, float& acc) {
  asm("{\n .reg .b16 xl, xh, wl, wh;\n mov.b32 {xl, xh}, %1;\n mov.b32 {wl, wh}, %2;\n"
      " fma.rn.f32.bf16 %0, xl, wl, %0;\n fma.rn.f32.bf16 %0, xh, wh, %0;\n}"
      : "+f"(acc)
      : "r"(x), "r"(w));
}

// Weights and activations of one thread for KS K steps: eight in bf16 mode
// (pairs in a word), four in fp32 mode.
template <bool BF, int RT, int OT>
struct SeqStep {
  static constexpr int KS = BF ? 8 : 4;
  uint32_t w[4][OT];
  uint4 x[RT];
  __device__ __forceinline__ void load(const uint32_t* wp, int out, const uint8_t* const (&xr)[RT], int byte) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      if (OT == 2) {
        const uint2 v = *reinterpret_cast<const uint2*>(wp + h * out);
        w[h][0] = v.x;
        w[h][OT - 1] = v.y;
      } else {
        w[h][0] = wp[h * out];
      }
    }
#pragma unroll
    for (int q = 0; q < RT; ++q) x[q] = *reinterpret_cast<const uint4*>(xr[q] + byte);
  }
  __device__ __forceinline__ void add(float (&acc)[RT][OT]) const {
#pragma unroll
    for (int h = 0; h < 4; ++h)
#pragma unroll
      for (int q = 0; q < RT; ++q) {
        const uint32_t xv = h == 0 ? x[q].x : h == 1 ? x[q].y : h == 2 ? x[q].z : x[q].w;
#pragma unroll
        for (int c = 0; c < OT; ++c) {
          if (BF) seq_fma_pair(xv, w[h][c], acc[q][c]);
          else acc[q][c] = fmaf(__uint_as_float(xv), __uint_as_float(w[h][c]), acc[q][c]);
        }
      }
  }
};

// A hidden layer with its weights in shared memory: thread per (OT adjacent
// outputs, RT rows), each sum in K order, the bias added after it; ReLU and
// (bf16 mode) rounding.  Shared-memory loads bound it (128 bytes a cycle
// whether or not the lanes share an address): a 16-byte activation load of a
// row, the same for the whole warp, costs as much as four weight words, so a
// thread takes two outputs and up to four rows per load of each.
template <bool BF, int RT, int OT>
__device__ __forceinline__ void seq_layer(const uint8_t* Wt, const uint8_t* xin, uint8_t* xout, const float* bl,
                                          int rows, int in, int out, float inv_out, int xs) {
  constexpr int XE = BF ? 2 : 4, KS = SeqStep<BF, RT, OT>::KS;
  const int oc = out / OT, groups = (rows + RT - 1) / RT;
#pragma unroll 1
  for (int e = threadIdx.x; e < groups * oc; e += kSeqHalf) {
    const int g = (int)(((float)e + 0.5f) * (inv_out * OT));  // e / oc (both far below 2^20)
    const int o = (e - g * oc) * OT, i0 = g * RT;
    const uint8_t* xr[RT];
#pragma unroll
    for (int q = 0; q < RT; ++q) xr[q] = xin + min(i0 + q, rows - 1) * xs * XE;
    float acc[RT][OT];
#pragma unroll
    for (int q = 0; q < RT; ++q)
#pragma unroll
      for (int c = 0; c < OT; ++c) acc[q][c] = 0.0f;
    const uint32_t* wp = reinterpret_cast<const uint32_t*>(Wt) + o;
    const int step = 4 * out, n = in / KS;
    if (n > 0) {  // the loads of one step are in flight while the one before it is added
      SeqStep<BF, RT, OT> s0, s1;
      s0.load(wp, out, xr, 0);
      int t = 0;
#pragma unroll 1
      for (; t + 2 < n; t += 2) {
        s1.load(wp + step, out, xr, 16 * t + 16);
        s0.add(acc);
        wp += 2 * step;
        s0.load(wp, out, xr, 16 * t + 32);
        s1.add(acc);
      }
      if (t + 1 < n) {
        s1.load(wp + step, out, xr, 16 * t + 16);
        s0.add(acc);
        s1.add(acc);
        wp += 2 * step;
      } else {
        s0.add(acc);
        wp += step;
      }
    }
#pragma unroll 1
    for (int k = KS * n; k < in; ++k) {
      const int h = k - KS * n;
#pragma unroll
      for (int c = 0; c < OT; ++c) {
        const uint32_t w = wp[(BF ? h >> 1 : h) * out + c];
        const float wv = __uint_as_float(!BF ? w : (h & 1) ? w & 0xffff0000u : w << 16);
#pragma unroll
        for (int q = 0; q < RT; ++q) acc[q][c] = fmaf(seq_xget<BF>(xr[q], k), wv, acc[q][c]);
      }
    }
#pragma unroll
    for (int c = 0; c < OT; ++c) {
      const float bo = bl[o + c];
#pragma unroll
      for (int q = 0; q < RT; ++q)
        if (i0 + q < rows) seq_xset<BF>(xout, (i0 + q) * xs + o + c, fmaxf(acc[q][c] + bo, 0.0f));
    }
  }
}

// A hidden layer whose weights do not fit in shared memory: a warp takes C
// adjacent output columns, lanes across K, the columns' weights in registers.
// The latency of their loads from L2 bounds it, so those of several columns are
// in flight together (8 requests of 128-512-512-1 over one instance 432 us with
// one column at a time, 286 with two, 236 with four; over 40 instances 1272, 838,
// 661).
template <bool BF>
__device__ __noinline__ void seq_layer_global(const float* __restrict__ Wl, const uint8_t* xin, uint8_t* xout,
                                                 const float* bl, int rows, int in, int out, int xs) {
  constexpr int C = 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int o0 = C * warp; o0 < out; o0 += C * kSeqWarps) {
    float wr[C][16];
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int k = lane + 32 * j;
        wr[c][j] = k < in && o0 + c < out ? __ldg(Wl + (int64_t)(o0 + c) * in + k) : 0.0f;
      }
    for (int i = 0; i < rows; ++i) {
      float part[C];
#pragma unroll
      for (int c = 0; c < C; ++c) part[c] = 0.0f;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int k = lane + 32 * j;
        if (k < in) {
          const float x = seq_xget<BF>(xin, i * xs + k);
#pragma unroll
          for (int c = 0; c < C; ++c) part[c] = fmaf(wr[c][j], x, part[c]);
        }
      }
#pragma unroll
      for (int sft = 16; sft; sft >>= 1)
#pragma unroll
        for (int c = 0; c < C; ++c) part[c] += __shfl_xor_sync(kFull, part[c], sft);
      if (lane == 0)
#pragma unroll
        for (int c = 0; c < C; ++c)
          if (o0 + c < out) seq_xset<BF>(xout, i * xs + o0 + c, fmaxf(part[c] + bl[o0 + c], 0.0f));
    }
  }
}

// Layer weights W [out][in] (published fp32, bf16-valued in bf16 mode) into
// the shared-memory layout, by `n` threads.  Lanes take eight outputs of four
// consecutive 4-value pieces of K: 64-byte runs of each row read, and the
// words written (outputs adjacent) four to a bank.
template <bool BF>
__device__ __noinline__ void seq_stage_weights(const float* __restrict__ Wl, uint8_t* Wt, int in, int out, int t,
                                                  int n) {
  if ((in & 15) == 0 && (out & 7) == 0 && (reinterpret_cast<uintptr_t>(Wl) & 15) == 0) {
    const int warp = t >> 5, lane = t & 31, nw = n >> 5;
    const int kt = in >> 4, tiles = kt * (out >> 3);  // a warp's tile: 8 outputs x 16 K
#pragma unroll 4
    for (int e = warp; e < tiles; e += nw) {
      const int o = (e / kt) * 8 + (lane & 7), k = (e % kt) * 16 + (lane >> 3) * 4;
      const float4 v = __ldg(reinterpret_cast<const float4*>(Wl + (int64_t)o * in + k));
      if (BF) {
        uint32_t* w = reinterpret_cast<uint32_t*>(Wt) + (int64_t)(k >> 1) * out + o;
        w[0] = (__float_as_uint(v.x) >> 16) | (__float_as_uint(v.y) & 0xffff0000u);
        w[out] = (__float_as_uint(v.z) >> 16) | (__float_as_uint(v.w) & 0xffff0000u);
      } else {
        float* w = reinterpret_cast<float*>(Wt) + (int64_t)k * out + o;
        w[0] = v.x;
        w[out] = v.y;
        w[2 * out] = v.z;
        w[3 * out] = v.w;
      }
    }
    return;
  }
  const int kp = BF ? (in + 1) & ~1 : in;
  for (int e = t; e < kp * out; e += n) {
    const int o = e / kp, k = e - o * kp;
    const float v = k < in ? __ldg(Wl + (int64_t)o * in + k) : 0.0f;
    if (BF) reinterpret_cast<uint16_t*>(Wt)[((int64_t)(k >> 1) * out + o) * 2 + (k & 1)] =
        (uint16_t)(__float_as_uint(v) >> 16);
    else reinterpret_cast<float*>(Wt)[(int64_t)k * out + o] = v;
  }
}

// The rest of seq_pre_row's walk, past the blocks looked up ahead (out of
// line: the scoring warps' code of a request should fit the instruction cache
// beside the other warps'): h0 and h1 from h0's value so far.
template <int W>
__device__ __noinline__ int2 seq_pre_tail(const SeqArgs& a, const SeqMeta* meta, int s, int gi, uint32_t patch0,
                                          int h0) {
  const int lane = threadIdx.x & 31, wi = gi >> 6, bi = gi & 63;
  const SeqMeta me = meta[s & 7];
  const int nb = (int)me.nb;
  int h1 = -1;
#pragma unroll 1
  for (int b0 = seq_blocks(W); b0 < nb && h1 < 0; b0 += 32) {
    const int b = b0 + lane;
    bool a0 = true, a1 = true;
    if (b < nb) {
      const uint64_t key = me.k0 + b < a.bcap ? a.bkeys[me.k0 + b] : 0ull;
      a0 = a1 = false;
      if (key) {
        uint64_t mw[W];
        seq_lookup<W>(a, key, mw);
#pragma unroll
        for (int w = 0; w < W; ++w)
          if (w == wi) a0 = (mw[w] >> bi) & 1ull;
        auto same = [&](int q) {  // the request q before this one has the same key here
          const SeqMeta pm = meta[(s - q) & 7];
          return s >= q && b < pm.nb && pm.k0 + b < a.bcap && a.bkeys[pm.k0 + b] == key;
        };
#pragma unroll
        for (int q = 2; q <= 4; ++q)
          if (patch0 & (1u << (q - 1))) a0 = a0 || same(q);
        a1 = a0 || same(1);
      }
    }
    const uint32_t m0 = __ballot_sync(kFull, !a0), m1 = __ballot_sync(kFull, !a1);
    if (h0 < 0 && m0) h0 = b0 + __ffs(m0) - 1;
    if (m1) h1 = b0 + __ffs(m1) - 1;
  }
  return make_int2(h0, h1);
}

// The pair features and hit length of one instance row for request s (masks
// mk, flags fl), by one warp: version 0 with the commits before the
// last one (`patch0`: the flags of the requests two to four back, bits 1 to
// 3, that this instance got), version 1 as if the last request (bit 0) also
// went here.  Version v's feature
// k is left at pre[8 v + k], its hit length at pre[8 v + 6].
template <int W>
__device__ __forceinline__ void seq_pre_row(const SeqArgs& a, const SeqMeta* meta, int s, const uint64_t* mk,
                                            const uint8_t* fl, int gi, uint32_t patch0, float pmu, float psd,
                                            float* pre) {
  constexpr int NB = seq_blocks(W);
  const int lane = threadIdx.x & 31;
  const SeqMeta me = meta[s & 7];
  const int nb = (int)me.nb, nbc = min(nb, NB), wi = gi >> 6, bi = gi & 63;
  const uint32_t patch1 = patch0 | 1u;
  int h0 = -1, h1 = -1;  // first block this instance lacks, without and with the last commit (h0 <= h1)
#pragma unroll 1
  for (int b0 = 0; b0 < nbc && h1 < 0; b0 += 128) {
    uint32_t m0[4], m1[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int b = b0 + 32 * u + lane;
      const bool held = b >= nbc || ((mk[b * W + wi] >> bi) & 1ull);
      const uint32_t f = b < nbc ? fl[b] : 0u;
      m0[u] = __ballot_sync(kFull, !held && !(f & patch0));
      m1[u] = __ballot_sync(kFull, !held && !(f & patch1));
    }
    int t0 = -1, t1 = -1;
#pragma unroll
    for (int u = 3; u >= 0; --u) {
      if (m0[u]) t0 = b0 + 32 * u + __ffs(m0[u]) - 1;
      if (m1[u]) t1 = b0 + 32 * u + __ffs(m1[u]) - 1;
    }
    if (h0 < 0) h0 = t0;
    h1 = t1;
  }
  if (nb > NB && h1 < 0) {  // past the blocks looked up ahead
    const int2 h = seq_pre_tail<W>(a, meta, s, gi, patch0, h0);
    h0 = h.x;
    h1 = h.y;
  }
  h0 = h0 < 0 ? nb : h0;
  h1 = h1 < 0 ? nb : h1;
  // lanes 8 v + k: feature k of version v
  const int k = lane & 7, h = lane & 8 ? h1 : h0;
  const int64_t hit = (int64_t)kBlockTok * h;
  const float fL = (float)me.L, f2 = (float)hit;
  const float f3 = me.L > 0 ? f2 / fL : 0.0f;
  const float raw = k == 0   ? fL
                    : k == 1 ? (float)h
                    : k == 2 ? f2
                    : k == 3 ? f3
                    : k == 4 ? (float)(me.L - hit)
                             : (float)((me.L + kBlockTok - 1) / kBlockTok - h);
  const float z = zscore(raw, pmu, psd);
  if (lane < 16) pre[lane] = k < kPair ? z : __int_as_float(h);
}

template <int W, bool BF>
__global__ void __launch_bounds__(kSeqThreads, 1) k_route_seq(const __grid_constant__ SeqArgs a) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  constexpr int NB = seq_blocks(W), KPT = NB / kSeqLook;  // blocks ahead, and per thread
  constexpr int XE = BF ? 2 : 4;
  const int N = a.n_inst, DI = a.d_inst, DR = a.d_req, R = a.rows, xs = a.xs;
  const MlpDesc& m = a.m;
  const SeqSmem o = seq_smem(R, DI, xs, W, XE, a.hidden_out, a.wsm ? (size_t)a.wbytes : 0);
  float* sinst = reinterpret_cast<float*>(smem_raw + o.inst);
  uint8_t* X0 = smem_raw + o.x0;
  const int x0_bytes = R * xs * XE;  // request s's feature rows: X0 + (s & 1) * x0_bytes
  uint8_t* Wsm = smem_raw + o.w;
  float* sc = reinterpret_cast<float*>(smem_raw + o.sc);
  float* pre = reinterpret_cast<float*>(smem_raw + o.pre);
  SeqLayer* lay = reinterpret_cast<SeqLayer*>(smem_raw + o.lay);
  float* bias = reinterpret_cast<float*>(smem_raw + o.bias);
  float* wl = reinterpret_cast<float*>(smem_raw + o.wl);
  volatile uint64_t* cand = reinterpret_cast<volatile uint64_t*>(smem_raw + o.cand);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + o.bar);
  volatile int* gave_up = reinterpret_cast<volatile int*>(bar + 4);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank(), ranks = gridDim.x;  // one cluster
  // every CTA has a row: the first N % ranks CTAs one more than the others
  const int share = N / (int)ranks, more = N - share * (int)ranks;
  const int i0 = (int)rank * share + min((int)rank, more), rows = share + ((int)rank < more ? 1 : 0);
  const int slots = (int)ranks * min(R, kSeqWarps);  // a slot per warp that may have a row
  const uint32_t bid_bytes = 8u * (uint32_t)a.bids;
  const int64_t base = a.tok_off[0];

  // The bids of request s: slot set s % 4, barrier s % 4 (its phase s / 4).
  // A set is written again four requests later, by CTAs that have this CTA's
  // bids of the three requests between, which it sends only after its own
  // warps are done reading the set (the barriers of seq_steps.h).
  for (int e = tid; e < 256; e += kSeqThreads) cand[e] = ~0ull;  // slots of warps without a row keep this
  if (tid == 0) {
    *gave_up = 0;
    for (int q = 0; q < 4; ++q) {
      mbar_init(&bar[q], 1);
      mbar_arrive_expect_tx(&bar[q], bid_bytes);
    }
    fence_mbar_init();
  }
  __syncthreads();
  cluster_sync();

  if (tid < kSeqHalf) {
    // ---- scoring
    const int sel = *reinterpret_cast<const volatile int32_t*>(&a.st->cur) == 1 ? 1 : 0;
    const float* __restrict__ params = sel ? a.params1 : a.params0;
#pragma unroll 1
    for (int e = tid; e < rows * DI; e += kSeqHalf) {
      const int i = e / DI, k = e - i * DI;
      const float v = a.inst[(int64_t)(i0 + i) * DI + k];
      sinst[e] = v;
      const float z = zscore(v, a.mean[kPair + k], a.stdv[kPair + k]);
      seq_xset<BF>(X0, i * xs + kPair + k, z);
      seq_xset<BF>(X0 + x0_bytes, i * xs + kPair + k, z);
    }
    const int L = m.n_layers, in_last = m.w[L - 1];
    for (int k = tid; k < in_last; k += kSeqHalf) wl[k] = params[m.woff[L - 1] + k];
    {
      int nb = 0;
#pragma unroll 1
      for (int l = 0; l + 1 < L; ++l) {
        const int in = m.w[l], out = m.w[l + 1];
        if (a.wsm) seq_stage_weights<BF>(params + m.woff[l], Wsm + a.woff_s[l], in, out, tid, kSeqHalf);
        for (int k = tid; k < out; k += kSeqHalf) bias[nb + k] = params[m.boff[l] + k];
        const int rt = !a.wsm ? 0 : (out & 1) ? 3 : rows > 2 ? 4 : rows;  // 3: one output and two rows
        if (tid == 0) lay[l] = SeqLayer{in, out, a.woff_s[l], nb, 1.0f / (float)out, rt};
        nb += out;
      }
    }
    const float blast = params[m.boff[L - 1]];
    const float qmu = a.q_col >= 0 ? a.mean[kPair + a.q_col] : 0.0f;
    const float qsd = a.q_col >= 0 ? a.stdv[kPair + a.q_col] : 1.0f;
    // this warp's slot and its set's barrier in the CTA of rank `lane`
    const int seen = (int)rank * min(R, kSeqWarps) + warp;
    uint32_t slot_at = 0, bar_at = 0;
    if (lane < (int)ranks) {
      slot_at = map_cluster(const_cast<const uint64_t*>(cand) + seen, (uint32_t)lane);
      bar_at = map_cluster(bar, (uint32_t)lane);
    }
    int c1 = -1;        // where request s - 1 went
    bool sends = true;  // no wait of this CTA has given up
    seq_half_sync();  // X0 and the weights are complete
#pragma unroll 1
    for (int s = 0; s <= a.n_req; ++s) {
      // Request s is looked up, request s - 3 inserted by this CTA's warps.
      // (Which barriers, and why no arrival meets an earlier use of its
      // barrier: seq_steps.h.)
      __syncwarp();
      if (s < a.n_req) named_bar_sync(seq::bar_looked_up(s), kSeqHalf + kSeqLook);
      if (seq::waits_inserted(s, a.n_req)) named_bar_sync(seq::bar_inserted(s - 2), kSeqHalf + kSeqIns);
      if (s > 0) {
        if (lane == 0 && sends) seq_wait(&bar[(s - 1) & 3], (uint32_t)((s - 1) >> 2) & 1u, gave_up, a.err);
        __syncwarp();
        sends = !*gave_up;
        c1 = seq_select(cand + 64 * ((s - 1) & 3), slots);
        // the other warps may go on with this request's step
        if (seq::tells_look(s, a.n_req)) named_bar_arrive(seq::bar_bids_look(), kSeqHalf + kSeqLook);
        named_bar_arrive(seq::bar_bids_insert(s), kSeqHalf + kSeqIns);
      }
      uint8_t* Xs = X0 + (s & 1) * x0_bytes;
      // 1. the last commit's queue, and this request's pair features given it
      if (tid == kSeqHalf - 1) {
        if (s > 0 && !*gave_up) mbar_arrive_expect_tx(&bar[(s - 1) & 3], bid_bytes);  // for request s + 3
        if (c1 >= i0 && c1 < i0 + rows) {
          const int i = c1 - i0;
          if (a.q_col >= 0) {
            const float v = sinst[i * DI + a.q_col] + 1.0f;
            sinst[i * DI + a.q_col] = v;
            const float z = zscore(v, qmu, qsd);
            seq_xset<BF>(X0, i * xs + kPair + a.q_col, z);
            seq_xset<BF>(X0 + x0_bytes, i * xs + kPair + a.q_col, z);
          }
          a.choice[s - 1] = c1;
          a.best[s - 1] = sc[i];
        }
      }
      if (s == a.n_req) break;
      const float* ps = pre + (s & 1) * R * 16;
#pragma unroll 1
      for (int e = tid; e < rows * 8; e += kSeqHalf) {
        const int i = e >> 3, k = e & 7;
        const float v = ps[16 * i + (i0 + i == c1 ? 8 : 0) + k];
        if (k < kPair) seq_xset<BF>(Xs, i * xs + k, v);
      }
      seq_half_sync();
      // 2. the predictor's hidden layers
      const uint8_t* xin = Xs;
#pragma unroll 1
      for (int l = 0; l + 1 < L; ++l) {
        const SeqLayer y = lay[l];
        uint8_t* xout = smem_raw + ((l & 1) ? o.x2 : o.x1);
        const uint8_t* w = Wsm + y.w;
        if (y.rt == 2) seq_layer<BF, 2, 2>(w, xin, xout, bias + y.b, rows, y.in, y.out, y.inv_out, xs);
        else if (y.rt == 4) seq_layer<BF, 4, 2>(w, xin, xout, bias + y.b, rows, y.in, y.out, y.inv_out, xs);
        else if (y.rt == 1) seq_layer<BF, 1, 2>(w, xin, xout, bias + y.b, rows, y.in, y.out, y.inv_out, xs);
        else if (y.rt == 3) seq_layer<BF, 2, 1>(w, xin, xout, bias + y.b, rows, y.in, y.out, y.inv_out, xs);
        else seq_layer_global<BF>(params + m.woff[l], xin, xout, bias + y.b, rows, y.in, y.out, xs);
        seq_half_sync();
        xin = xout;
      }
      // 3. the output layer, warp per row, and the warp's lowest code to every CTA
      uint64_t bid = ~0ull;
#pragma unroll 1
      for (int i = warp; i < rows; i += kSeqWarps) {
        float part = 0.0f;
#pragma unroll 4
        for (int k = lane; k < in_last; k += 32) part = fmaf(wl[k], seq_xget<BF>(xin, i * xs + k), part);
#pragma unroll
        for (int sft = 16; sft; sft >>= 1) part += __shfl_xor_sync(kFull, part, sft);
        const float z = part + blast;
        const uint64_t code = seq_code(z, i0 + i);
        bid = code < bid ? code : bid;
        if (lane == 0) sc[i] = z;
      }
      if (warp < rows && lane < (int)ranks && sends)
        seq_remote_store(slot_at + 512u * (s & 3), bar_at + 8u * (s & 3), bid);
      __syncwarp();
      if (lane == 0)
#pragma unroll 1
        for (int i = warp; i < rows; i += kSeqWarps) {
          const int64_t at = (int64_t)s * N + i0 + i;
          if (a.scores) a.scores[at] = sc[i];
          if (a.hits) a.hits[at] = __float_as_int(ps[16 * i + (i0 + i == c1 ? 8 : 0) + 6]);
        }
      // the last scores are written; with no hidden layer, the feature rows read
      if (s + 1 == a.n_req || L == 1) seq_half_sync();
    }
    seq_half_sync();
#pragma unroll 1
    for (int e = tid; e < rows * DI; e += kSeqHalf) a.inst[(int64_t)i0 * DI + e] = sinst[e];
  } else if (tid < kSeqHalf + kSeqLook) {
    // ---- lookups: step s prepares request s + 1
    uint64_t* mask = reinterpret_cast<uint64_t*>(smem_raw + o.mask);
    uint8_t* flag = smem_raw + o.flag;
    SeqMeta* meta = reinterpret_cast<SeqMeta*>(smem_raw + o.meta);
    const int pt = tid - kSeqHalf, pw = pt >> 5;
    const int pk = lane & 7;  // this lane's pair feature
    const float pmu = pk < kPair ? a.mean[pk] : 0.0f, psd = pk < kPair ? a.stdv[pk] : 1.0f;
    // keys of requests s - 3 .. s + 2 in k[0] .. k[5] (0: none)
    uint64_t k[6][KPT];
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
      for (int j = 0; j < KPT; ++j) k[q][j] = 0ull;
    // token offsets of requests s + 2 and s + 3 (request r's prompt: [off r, off r + 1))
    auto off = [&](int r) { return a.tok_off[min(r, a.n_req)]; };
    int64_t o2 = off(1), o3 = off(2);
    int64_t LC = o2 - base, nbC = LC / kBlockTok, k0C = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const int64_t b = pt + kSeqLook * j;
      if (b < nbC && b < a.bcap) k[4][j] = a.bkeys[b];
    }
    int c1 = -1, c2 = -1, c3 = -1;  // where requests s - 1, s - 2 and s - 3 went
#pragma unroll 1
    for (int s = -1; s + 1 < a.n_req; ++s) {
      // keys of request s + 2, in flight over the step
      const int64_t LD = s + 2 < a.n_req ? o3 - o2 : 0, nbD = LD / kBlockTok, k0D = (o2 - base) / kBlockTok;
      const int64_t o4 = off(s + 4);
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const int64_t b = pt + kSeqLook * j;
        k[5][j] = b < nbD && k0D + b < a.bcap ? a.bkeys[k0D + b] : 0ull;
      }
      c3 = c2;
      c2 = c1;
      if (s > 0) {  // the bids for request s - 1 are in
        __syncwarp();
        named_bar_sync(seq::bar_bids_look(), kSeqHalf + kSeqLook);
        c1 = seq_select(cand + 64 * ((s - 1) & 3), slots);
      }
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const int b = pt + kSeqLook * j;
        if (b >= nbC) continue;
        uint64_t mw[W];
#pragma unroll
        for (int w = 0; w < W; ++w) mw[w] = 0;
        uint32_t f = 0;
        if (k[4][j]) {
          seq_lookup<W>(a, k[4][j], mw);
#pragma unroll
          for (int q = 0; q < 4; ++q) f |= k[4][j] == k[3 - q][j] ? 1u << q : 0u;
        }
#pragma unroll
        for (int w = 0; w < W; ++w) mask[b * W + w] = mw[w];
        flag[b] = (uint8_t)f;
      }
      if (pt == 0) meta[(s + 1) & 7] = SeqMeta{LC, nbC, k0C};
      __syncwarp();
      named_bar_sync(10, kSeqLook);  // the masks are complete
      float* ps = pre + ((s + 1) & 1) * R * 16;
#pragma unroll 1
      for (int i = pw; i < rows; i += kSeqLook / 32) {
        const int gi = i0 + i;
        seq_pre_row<W>(a, meta, s + 1, mask, flag, gi,
                       (gi == c1 ? 2u : 0u) | (gi == c2 ? 4u : 0u) | (gi == c3 ? 8u : 0u), pmu, psd, ps + 16 * i);
      }
      // the extras, from the last warp on (the first ones have the rows)
      uint8_t* Xn = X0 + ((s + 1) & 1) * x0_bytes;
#pragma unroll 1
      for (int c = kSeqLook - 1 - pt; c < DR; c += kSeqLook) {
        const int col = kPair + DI + c;
        const float z = zscore(a.req[(int64_t)(s + 1) * DR + c], a.mean[col], a.stdv[col]);
#pragma unroll 1
        for (int i = 0; i < rows; ++i) seq_xset<BF>(Xn, i * xs + col, z);
      }
      __syncwarp();
      named_bar_sync(10, kSeqLook);  // the masks are read
      named_bar_arrive(seq::bar_looked_up(s + 1), kSeqHalf + kSeqLook);
#pragma unroll
      for (int q = 0; q < 5; ++q)
#pragma unroll
        for (int j = 0; j < KPT; ++j) k[q][j] = k[q + 1][j];
      nbC = nbD;
      k0C = k0D;
      LC = LD;
      o2 = o3;
      o3 = o4;
    }
  } else {
    // ---- insertion: step s inserts request s - 1 for the instance it went
    // to; the CTAs share its blocks by runs of 32
    const int it = tid - kSeqHalf - kSeqLook;
    int64_t t0 = base;
#pragma unroll 1
    for (int s = 0; s <= a.n_req; ++s) {
      if (s > 0) {
        const int64_t t1 = a.tok_off[s], nb = (t1 - t0) / kBlockTok, k0 = (t0 - base) / kBlockTok;
        t0 = t1;
        int64_t b = (((int64_t)(it >> 5) * ranks + rank) << 5) + lane;
        uint64_t key = b < nb && k0 + b < a.bcap ? a.bkeys[k0 + b] : 0ull;
        __syncwarp();
        named_bar_sync(seq::bar_bids_insert(s), kSeqHalf + kSeqIns);  // the bids for request s - 1 are in
        const int c = seq_select(cand + 64 * ((s - 1) & 3), slots);
        int fresh = 0;
#pragma unroll 1
        while (c >= 0 && b - lane < nb) {  // (warp-uniform)
          const bool add = key && seq_insert<W>(a, key, c);
          fresh += __popc(__ballot_sync(kFull, add));
          b += (int64_t)kSeqIns * ranks;
          key = b < nb && k0 + b < a.bcap ? a.bkeys[k0 + b] : 0ull;
        }
        if (lane == 0 && fresh && (int64_t)atomicAdd(a.counts + c, fresh) + fresh > a.max_keys)
          latch_error(a.err, LS_ERR_TABLE_FULL);
      }
      if (seq::tells_inserted(s, a.n_req)) {
        __threadfence();  // the inserted keys before this CTA's next bids
        __syncwarp();
        named_bar_arrive(seq::bar_inserted(s), kSeqHalf + kSeqIns);
      }
    }
  }
  __syncwarp();
  cluster_sync();  // no CTA leaves while another may still store bids into it
  if (*gave_up) cluster_drain();
}

}  // namespace

// Whether a shape is taken: the bytes one CTA would need for all instances'
// state rows, two fp32 activation rows each and the masks of 512 blocks, 0
// beyond 200 KB (a cluster's CTAs each need less: they share the instances).
size_t route_seq_smem(int n_inst, int d_inst, int wmax, int W) {
  if (W < 1 || W > kSeqMaxW || wmax > 512 || n_inst < 1) return 0;
  size_t b = seq_al((size_t)n_inst * (d_inst > 0 ? d_inst : 1) * 4);
  b = seq_al(b + (size_t)n_inst * wmax * 4);
  b = seq_al(b + (size_t)n_inst * wmax * 4);
  b = seq_al(b + (size_t)n_inst * 4);
  b = seq_al(b + (size_t)n_inst * 4);
  b = seq_al(b + (size_t)512 * W * 8);
  b = seq_al(b + (size_t)16 * W * 8);
  b = seq_al(b + (size_t)W * 8);
  b += 2 * 64;
  return b <= 200 * 1024 ? b : 0;
}

namespace {
template <int W>
cudaError_t seq_kernel(bool bf16, void (*&k)(const SeqArgs)) {
  k = bf16 ? k_route_seq<W, true> : k_route_seq<W, false>;
  return bf16 ? allow_smem<k_route_seq<W, true>>() : allow_smem<k_route_seq<W, false>>();
}
}  // namespace

cudaError_t launch_route_seq(int n_req, int n_inst, int d_inst, int d_req, int q_col, const int64_t* tok_off,
                             const uint64_t* bkeys, int64_t bcap, const float* req, float* inst, const float* mean,
                             const float* stdv, const Published* pub, const DevState* st, const MlpDesc& m,
                             uint64_t* gkeys, uint64_t* gmask, int W, uint64_t gslots_mask, int32_t* counts,
                             int64_t max_keys, int32_t* choice, float* best, float* scores, int32_t* hits, int* err,
                             cudaStream_t s) {
  if (n_req <= 0) return cudaSuccess;
  int wmax = 1;
  for (int l = 0; l <= m.n_layers; ++l) wmax = std::max(wmax, m.w[l]);
  if (!route_seq_smem(n_inst, d_inst, wmax, W)) return cudaErrorInvalidValue;
  int ranks = 1;
  while (ranks < kSeqCluster && 2 * ranks <= n_inst) ranks *= 2;  // a power of two
  SeqArgs a{};
  a.n_req = n_req;
  a.n_inst = n_inst;
  a.d_inst = d_inst;
  a.d_req = d_req;
  a.q_col = q_col;
  a.tok_off = tok_off;
  a.bkeys = bkeys;
  a.bcap = bcap;
  a.req = req;
  a.inst = inst;
  a.mean = mean;
  a.stdv = stdv;
  a.params0 = pub[0].params;
  a.params1 = pub[1].params;
  a.st = st;
  a.m = m;
  for (int l = 0; l + 1 < m.n_layers; ++l) a.hidden_out += m.w[l + 1];
  a.rows = (n_inst + ranks - 1) / ranks;
  a.xs = (wmax + 7) & ~7;
  for (int r = 0; r < ranks; ++r) a.bids += std::min(n_inst / ranks + (r < n_inst % ranks ? 1 : 0), kSeqWarps);
  a.gkeys = gkeys;
  a.gmask = gmask;
  a.gslots_mask = gslots_mask;
  a.counts = counts;
  a.max_keys = max_keys;
  a.choice = choice;
  a.best = best;
  a.scores = scores;
  a.hits = hits;
  a.err = err;
  const int xe = m.bf16 ? 2 : 4;
  size_t wb = 0;
  for (int l = 0; l + 1 < m.n_layers; ++l) {
    a.woff_s[l] = (int)wb;
    const size_t in = m.bf16 ? (m.w[l] + 1) & ~1 : m.w[l];
    wb = seq_al(wb + in * m.w[l + 1] * xe);
  }
  // the weights go to shared memory when they fit beside the rest
  const size_t with_w = seq_smem(a.rows, d_inst, a.xs, W, xe, a.hidden_out, wb).total;
  a.wsm = with_w <= 224 * 1024 ? 1 : 0;
  a.wbytes = a.wsm ? (int64_t)wb : 0;
  const size_t smem = a.wsm ? with_w : seq_smem(a.rows, d_inst, a.xs, W, xe, a.hidden_out, 0).total;
  void (*k)(const SeqArgs) = nullptr;
  cudaError_t e = cudaErrorInvalidValue;
  switch (W) {
    case 1: e = seq_kernel<1>(m.bf16, k); break;
    case 2: e = seq_kernel<2>(m.bf16, k); break;
    case 4: e = seq_kernel<4>(m.bf16, k); break;
    case 8: e = seq_kernel<8>(m.bf16, k); break;
  }
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ranks);
  cfg.blockDim = dim3(kSeqThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ranks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, a);
}

}  // namespace ls
