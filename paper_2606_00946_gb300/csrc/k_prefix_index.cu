// Prefix index over all instances: one open-addressing table maps a block key
// to the bitmask of instances whose cache holds that block (the gateway's
// single logical prefix index of Sec. 4.2, in hash-table form as Sec. 2
// allows).  Hit lengths then need one lookup per (request, block) instead of
// one per (request, block, instance):
//   alive_b = AND_{b' <= b} mask(key_b')   (bits of instances still matching)
//   h_i     = number of leading blocks b with bit i of alive_b set
// which is exactly "leading blocks all cached on instance i, stop at the first
// miss" (Sec. 2: prefix reuse is strictly sequential).
//
// One warp per request: each round hashes the next 32 blocks of the prompt
// (one per lane; the chained prefix state is a warp-wide scan of the linear
// recurrence), looks the 32 keys up at once, and a warp-wide prefix AND of
// their instance masks gives, per lane, the instances still matching every
// block up to it.  An instance that stops matching in the round gets its hit
// length from one ballot, or, when several of a group of 32 stop in it, from a
// bit transpose of their alive masks (a request's first blocks end most of the
// instances: at 256 instances the ballots, a dozen instructions each, were
// most of a walk's first round).  The hit lengths wait in shared memory and the
// row is written once, coalesced, at the end.  The walk stops at the first
// round after which no instance matches, so tokens past the longest hit plus
// one round are never read.  Walks differ in length by orders of magnitude,
// so warps take requests from a shared counter (a warp that finishes a short
// walk takes the next request) rather than a fixed share each, the long ones
// first.  Small batches give each request a CTA (k_prefix_index_coop).
#include "blockhash.cuh"
#include "sm100.cuh"

namespace ls {
namespace {
using namespace bh;

constexpr int kNT = 128;
constexpr int kFewDeaths = 2;  // instances of 32 that end in a round one by one; more, by a transpose

// Slot of `key` in the index (linear probing in aligned 4-slot buckets), -1 if absent.
__device__ __forceinline__ int64_t index_find(const uint64_t* __restrict__ gkeys, uint64_t gmask_slots,
                                              uint64_t key) {
  uint64_t s = key & gmask_slots;
  uint32_t first = (uint32_t)(s & 3u);
  uint64_t b = s & ~(uint64_t)3;
  for (uint64_t n = 0; n <= (gmask_slots >> 2) + 1; ++n) {
    const ulonglong2* q = reinterpret_cast<const ulonglong2*>(gkeys + b);
    const ulonglong2 v01 = __ldg(q), v23 = __ldg(q + 1);
    const uint64_t v[4] = {v01.x, v01.y, v23.x, v23.y};
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      if (j < first) continue;
      if (v[j] == key) return (int64_t)(b + j);
      if (v[j] == 0) return -1;
    }
    first = 0;
    b = (b + 4) & gmask_slots;
  }
  return -1;
}

// With one mask word (at most 64 instances) the index stores each key next to
// its mask, entry e = (ent[2e], ent[2e+1]) = (key, mask), so one 32-byte
// bucket of two entries answers a probe: mask of `key`, 0 if absent.
__device__ __forceinline__ uint64_t index_mask_w1(const uint64_t* __restrict__ ent, uint64_t mslots, uint64_t key) {
  uint64_t s = key & mslots;
  uint32_t first = (uint32_t)(s & 1);
  uint64_t b = s & ~(uint64_t)1;
  for (uint64_t n = 0; n <= (mslots >> 1) + 1; ++n) {
    const ulonglong2* q = reinterpret_cast<const ulonglong2*>(ent + 2 * b);
    const ulonglong2 e0 = __ldg(q), e1 = __ldg(q + 1);
    if (first == 0) {
      if (e0.x == key) return e0.y;
      if (e0.x == 0) return 0;
    }
    if (e1.x == key) return e1.y;
    if (e1.x == 0) return 0;
    first = 0;
    b = (b + 2) & mslots;
  }
  return 0;
}

// Transpose of the warp's 32 x 32 bit matrix: bit b of lane i of the result is
// bit i of lane b's v.
__device__ __forceinline__ uint32_t transpose32(uint32_t v, int lane) {
#pragma unroll
  for (int j = 16; j; j >>= 1) {
    const uint32_t m = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu : j == 2 ? 0x33333333u
                                                                                           : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(kFull, v, j);
    v = (lane & j) ? (v & ~m) | ((y >> j) & m) : (v & m) | ((y & m) << j);
  }
  return v;
}

// Token buffer of a warp's round: the 32 blocks' 2 KB as the 16-byte chunks
// of global memory they lie in, 128 or (prompts start at any token) 129 of
// them, four chunks every 80 bytes: the lanes' 16-byte loads of their own block
// then meet no bank twice.
constexpr uint32_t kRoundBytes = 33 * 80;

// Asynchronous copy of the tokens of blocks [p, p + 32) of a prompt of `len`
// tokens at `base` (one warp; at most the prompt's own tokens are read).  Read
// block by block, a lane each, the same tokens take 16 loads of 32 addresses
// 64 bytes apart, 256 of the 290 shared-memory / L1 cycles of a round.
__device__ __forceinline__ void round_copy(const int32_t* __restrict__ base, int64_t len, int64_t p, uint32_t dst) {
  const int lane = threadIdx.x & 31;
  const uint8_t* src = reinterpret_cast<const uint8_t*>(base + p * kBlockTok);
  const int sh = (int)(reinterpret_cast<uintptr_t>(src) & 15);
  const int64_t left = 4 * (len - p * kBlockTok);     // bytes of the prompt from here on
  const int rem = left < 4096 ? (int)left : 4096;
  const int need = min(rem & ~63, 2048);              // bytes of full blocks in the round
  src -= sh;
  dst += (uint32_t)(lane >> 2) * 80u + (uint32_t)(lane & 3) * 16u;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int c = lane + 32 * i, o = 16 * c - sh;     // chunk, and its first byte's place in the round
    if (o >= need || (i == 4 && lane > 0)) continue;
    if ((o >= 0 || p > 0) && o + 16 <= rem) {
      sm100::cp_async16(dst + 640u * i, src + 16 * c);
    } else {  // the prompt's first or last chunk
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (o + 4 * k >= 0 && o + 4 * k < need) sm100::cp_async4(dst + 640u * i + 4u * k, src + 16 * c + 4 * k);
    }
  }
  sm100::cp_async_commit();
}

// Content hash of the lane's block in a round's buffer.
__device__ __forceinline__ uint64_t round_hash(const int32_t* base, uint32_t buf, int lane) {
  const uint32_t at = buf + (uint32_t)lane * 80u;
  const int s = (int)(reinterpret_cast<uintptr_t>(base) & 15) >> 2;  // words before the block in its first chunk
  const bool s1 = s & 1, s2 = s & 2;  // (the same for the whole warp)
  uint32_t v[8];
  sm100::lds128(at, v);
  uint64_t acc = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q < 3) sm100::lds128(at + 16u * (q + 1), v + 4);
    else if (s) sm100::lds128(at + 80u, v + 4);
    uint32_t u[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) u[j] = s1 ? v[j + 1] : v[j];
    acc ^= word_mix(s2 ? u[2] : u[0], s2 ? u[3] : u[1], 2 * q);
    acc ^= word_mix(s2 ? u[4] : u[2], s2 ? u[5] : u[3], 2 * q + 1);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = v[j + 4];
  }
  return mix64(acc);
}

// The masks of a block key (0 where absent).
template <int W>
__device__ __forceinline__ void index_masks(const uint64_t* __restrict__ gkeys, const uint64_t* __restrict__ gmask,
                                            uint64_t gmask_slots, uint64_t key, uint64_t (&pa)[W]) {
  if (W == 1) {
    pa[0] = index_mask_w1(gkeys, gmask_slots, key);
  } else {
    const int64_t slot = index_find(gkeys, gmask_slots, key);
#pragma unroll
    for (int w = 0; w < W; ++w) pa[w] = slot >= 0 ? __ldg(gmask + slot * W + w) : 0ull;
  }
}

// Instances of mask word w that ended (`died`) among the warp's 32 blocks from
// block p on: hit length p + the number of blocks whose prefix AND x holds
// the instance, kept at ended[64 w + instance bit].
__device__ __forceinline__ void note_ended(uint64_t died, uint64_t x, int64_t p, int w, int lane, int32_t* ended) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t d = (uint32_t)(died >> (32 * h));
    if (__popc(d) > kFewDeaths) {
      const int cnt = __popc(transpose32((uint32_t)(x >> (32 * h)), lane));
      if ((d >> lane) & 1u) ended[64 * w + 32 * h + lane] = (int32_t)(p + cnt);
    } else {
      for (; d; d &= d - 1) {
        const int bit = __ffs(d) - 1;
        const int cnt = __popc(__ballot_sync(kFull, (x >> (32 * h + bit)) & 1ull));
        if (lane == bit) ended[64 * w + 32 * h + lane] = (int32_t)(p + cnt);
      }
    }
  }
}

// G^(lane + 1): the factor by which the state entering 32 blocks reaches lane
// `lane`.
__device__ __forceinline__ uint64_t lane_power(int lane) {
  uint64_t g = 1, b = kG;
  for (unsigned e = (unsigned)lane + 1; e; e >>= 1) {
    if (e & 1) g *= b;
    b *= b;
  }
  return g;
}

template <int W>
__device__ __forceinline__ void all_alive(int n_inst, uint64_t (&alive)[W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int lo = 64 * w;
    alive[w] = n_inst >= lo + 64 ? ~0ull : (n_inst > lo ? ((1ull << (n_inst - lo)) - 1ull) : 0ull);
  }
}

// One request's walk by the NW warps of the CTA: NW * 32 blocks a round.  The
// chained state is affine in the state entering a warp's blocks, so each warp
// scans its own and the warps' totals chain the rest; likewise the prefix AND.
// Two barriers a round; the row of hit lengths is written at the end.
template <int W, int NW>
struct CoopSmem {
  uint64_t tot[NW];
  uint64_t end[NW][W];
  int32_t ended[64 * W];
};
template <int W, int NW>
__device__ __forceinline__ void coop_walk(int64_t t0, int64_t nb, const int32_t* __restrict__ tok,
                                          const uint64_t* __restrict__ gkeys, const uint64_t* __restrict__ gmask,
                                          uint64_t gmask_slots, int n_inst, int32_t* __restrict__ hrow,
                                          const uint64_t* s_glane, CoopSmem<W, NW>& S) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t* base = tok + t0;
  const uintptr_t ab = reinterpret_cast<uintptr_t>(base);
  const int align = (ab & 15) == 0 ? 16 : (ab & 7) == 0 ? 8 : 4;
  uint64_t alive[W];
  all_alive<W>(n_inst, alive);
  uint64_t state = kG;  // s_{-1}
  bool any = n_inst > 0;
  uint32_t tw[16];
  if (threadIdx.x < nb) block_load(base + (int64_t)threadIdx.x * kBlockTok, align, tw);
  for (int64_t p = 0; p < nb && any; p += 32 * NW) {
    const int64_t b = p + threadIdx.x;
    const bool in = b < nb;
    uint64_t B = in ? block_hash(tw) : 0ull;
    if (b + 32 * NW < nb) block_load(base + (b + 32 * NW) * kBlockTok, align, tw);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int off = 1 << k;
      const uint64_t o = __shfl_up_sync(kFull, B, off);
      if (lane >= off) B = gpow(off) * o + B;
    }
    if (lane == 31) S.tot[warp] = B;
    __syncthreads();
    uint64_t mine = state;  // the state entering this warp's blocks
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      if (v == warp) mine = state;
      state = gpow(32) * state + S.tot[v];  // (past the prompt's end only in its last round)
    }
    uint64_t pa[W];
    if (in) {
      index_masks<W>(gkeys, gmask, gmask_slots, key_of(s_glane[lane] * mine + B), pa);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) pa[w] = 0ull;
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const uint64_t y = __shfl_up_sync(kFull, pa[w], 1 << k);
        if (lane >= (1 << k)) pa[w] &= y;
      }
      if (lane == 31) S.end[warp][w] = pa[w];
    }
    __syncthreads();
    any = false;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      uint64_t before = alive[w];  // matching every block before this warp's
#pragma unroll
      for (int v = 0; v < NW; ++v) {
        if (v == warp) before = alive[w];
        alive[w] &= S.end[v][w];
      }
      note_ended(before & ~S.end[warp][w], pa[w] & before, p + 32 * warp, w, lane, S.ended);
      any = any || alive[w] != 0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int i = 64 * w + threadIdx.x;
    // instances matching every full block (or a request without a full block)
    if (threadIdx.x < 64 && i < n_inst) hrow[i] = ((alive[w] >> threadIdx.x) & 1ull) ? (int32_t)nb : S.ended[i];
  }
  __syncthreads();  // the shared memory is free for the next walk
}

// A CTA of NW warps per request: batches of no more requests than CTAs fit on
// the GPU, where a walk's rounds, not the number of walks, take the time (one
// request over 16 instances as a graph replay of the route: 24.6 -> 20.6 us; a
// 256-request route behind a rebuild 71 -> 64 us).  Larger batches fill the GPU
// with a warp per walk; giving only their long prompts whole CTAs gained
// nothing there, the two barriers a round cost what the rounds saved.
template <int W, int NW>
__global__ void __launch_bounds__(32 * NW, W <= 4 ? 32 / NW : 1) k_prefix_index_coop(
    const int32_t* __restrict__ tok, const int64_t* __restrict__ tok_off, const uint64_t* __restrict__ gkeys,
    const uint64_t* __restrict__ gmask, uint64_t gmask_slots, int n_inst, int32_t* __restrict__ hits, DevState* st) {
  __shared__ CoopSmem<W, NW> S;
  __shared__ uint64_t s_glane[32];
  sm100::pdl_wait();  // the previous kernel of the stream is complete
  route_snapshot(st);
  const int64_t t0 = tok_off[blockIdx.x], nb = (tok_off[blockIdx.x + 1] - t0) / kBlockTok;
  if (threadIdx.x < 32) s_glane[threadIdx.x] = lane_power(threadIdx.x);
  __syncthreads();
  coop_walk<W, NW>(t0, nb, tok, gkeys, gmask, gmask_slots, n_inst, hits + (int64_t)blockIdx.x * n_inst, s_glane, S);
  sm100::pdl_trigger();
}

// Up to two mask words the walk stages its tokens (round_copy); beyond, its
// warps read them directly: the buffers would take the L1 that holds index
// lines of the larger tables (256 instances: 1988 us a large route staged,
// 1966 not; 64 instances 334 against 347, 32 instances 56.0 against 57.8).
// `order` (nullable): the requests in the order they are to be taken.
template <int W>
__global__ void __launch_bounds__(kNT, W <= 4 ? 8 : 1) k_prefix_index(int n_req, const int32_t* __restrict__ tok,
                                                      const int64_t* __restrict__ tok_off,
                                                      const uint64_t* __restrict__ gkeys,
                                                      const uint64_t* __restrict__ gmask, uint64_t gmask_slots,
                                                      int n_inst, int32_t* __restrict__ hits, DevState* st,
                                                      const uint32_t* __restrict__ order) {
  constexpr bool kStaged = W <= 2;
  sm100::pdl_wait();  // the previous kernel of the stream is complete
  route_snapshot(st);
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // (lane powers in shared memory: one load per round, no registers held)
  __shared__ uint64_t s_glane[32];
  // hit lengths of the instances that ended in this warp's walk (each written
  // and read by the lane i mod 32)
  __shared__ int32_t s_ended[kNT / 32][64 * W];
  __shared__ __align__(16) uint8_t s_tok[kStaged ? kNT / 32 : 1][2][kStaged ? kRoundBytes : 16];
  if (threadIdx.x < 32) s_glane[lane] = lane_power(lane);
  __syncthreads();
  int32_t* const ended = s_ended[threadIdx.x >> 5];
  const uint32_t tokens = sm100::smem_u32(s_tok[kStaged ? threadIdx.x >> 5 : 0]);
  uint32_t buf = 0;  // the round's token buffer
  for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < n_req;) {
    const int64_t r = order ? (int64_t)order[q] : q;
    const int64_t t0 = tok_off[r], len = tok_off[r + 1] - t0;
    const int64_t nb = len / kBlockTok;
    const int32_t* base = tok + t0;
    uint64_t alive[W];
    all_alive<W>(n_inst, alive);
    uint64_t state = kG;  // s_{-1}
    bool any = n_inst > 0;
    // A round's tokens are requested one round ahead (staged: copied to shared
    // memory; else into registers), so that their load overlaps the index
    // probes of the current round.  A copy that a walk did not come to use goes
    // to the buffer its last round did not read; the next walk starts in the
    // other one and waits for both.
    const uintptr_t ab = reinterpret_cast<uintptr_t>(base);
    const int align = (ab & 15) == 0 ? 16 : (ab & 7) == 0 ? 8 : 4;
    uint32_t tw[16];
    if (kStaged) {
      if (nb > 0) round_copy(base, len, 0, tokens + buf * kRoundBytes);
    } else if (lane < nb) {
      block_load(base + (int64_t)lane * kBlockTok, align, tw);
    }
    for (int64_t p = 0; p < nb && any; p += 32) {
      const int64_t b = p + lane;
      const bool in = b < nb;
      // inclusive scan: B = sum_{j <= lane} G^(lane - j) c_j, then s = G^(lane+1) s_in + B
      uint64_t B = 0ull;
      if (kStaged) {
        sm100::cp_async_wait<0>();
        __syncwarp();
        if (p + 32 < nb) round_copy(base, len, p + 32, tokens + (buf ^ 1u) * kRoundBytes);
        if (in) B = round_hash(base, tokens + buf * kRoundBytes, lane);
        buf ^= 1u;
      } else {
        if (in) B = block_hash(tw);
        if (b + 32 < nb) block_load(base + (b + 32) * kBlockTok, align, tw);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const int off = 1 << k;
        const uint64_t o = __shfl_up_sync(kFull, B, off);
        if (lane >= off) B = gpow(off) * o + B;
      }
      const uint64_t s = s_glane[lane] * state + B;
      const int last = (int)(nb - p < 32 ? nb - p : 32) - 1;
      state = __shfl_sync(kFull, s, last);
      uint64_t pa[W];
      if (in) {
        index_masks<W>(gkeys, gmask, gmask_slots, key_of(s), pa);
      } else {
#pragma unroll
        for (int w = 0; w < W; ++w) pa[w] = 0ull;
      }
      any = false;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        uint64_t x = pa[w];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const uint64_t y = __shfl_up_sync(kFull, x, 1 << k);
          if (lane >= (1 << k)) x &= y;
        }
        x &= alive[w];
        const uint64_t end = __shfl_sync(kFull, x, 31);
        note_ended(alive[w] & ~end, x, p, w, lane, ended);
        alive[w] = end;
        any = any || end != 0;
      }
    }
    if (nb > 0) buf ^= 1u;  // the buffer the last round read
    int32_t* hrow = hits + (int64_t)r * n_inst;
#pragma unroll
    for (int w = 0; w < W; ++w)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int bit = 32 * h + lane, i = 64 * w + bit;
        // instances matching every full block (or requests without a full block)
        if (i < n_inst) hrow[i] = ((alive[w] >> bit) & 1ull) ? (int32_t)nb : ended[i];
      }
    // the next request: from the counter (after each warp's first), else a fixed stride
    if (st) {
      uint32_t nx = 0;
      if (lane == 0) nx = atomicAdd(&st->walk_next, 1u);
      q = warps + (int64_t)__shfl_sync(kFull, nx, 0);
    } else {
      q += warps;
    }
  }
  sm100::cp_async_wait<0>();
  // the counter starts at 0 for the next walk: reset by the last block to finish
  if (st && last_block(&st->done[DONE_WALK]) && threadIdx.x == 0) st->walk_next = 0u;
  sm100::pdl_trigger();  // the next kernel may start once every CTA is here
}

// Instance of key position k: the last i with key_off[i] <= k.
__device__ __forceinline__ int key_instance(const int64_t* __restrict__ key_off, int n_inst, int64_t k) {
  int lo = 0, hi = n_inst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (key_off[mid] <= k) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The requests of a batch by falling prompt length (by its leading three
// binary digits; any order within a class), for the walk to take the long ones
// first: a walk that starts when most are done ends that much later.  One CTA
// (counting sort).
constexpr int kLenClasses = 128;
__device__ __forceinline__ int length_class(int64_t len) {
  const uint32_t n = (uint32_t)(len / kBlockTok < (1 << 28) ? len / kBlockTok : (1 << 28));
  if (n < 4) return kLenClasses - 1 - (int)n;
  const int e = 31 - __clz(n);
  return kLenClasses - 1 - (4 * (e - 1) + (int)((n >> (e - 2)) & 3u));
}

__global__ void __launch_bounds__(1024) k_walk_order(int n_req, const int64_t* __restrict__ tok_off,
                                                     uint32_t* __restrict__ order) {
  __shared__ uint32_t at[kLenClasses];
  sm100::pdl_wait();
  if (threadIdx.x < kLenClasses) at[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll 4
  for (int r = threadIdx.x; r < n_req; r += 1024) atomicAdd(at + length_class(tok_off[r + 1] - tok_off[r]), 1u);
  __syncthreads();
  if (threadIdx.x < 32) {  // class counts to first places, four classes a lane
    uint32_t c[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      c[k] = at[4 * threadIdx.x + k];
      sum += c[k];
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, o);
      if ((int)threadIdx.x >= o) x += y;
    }
    x -= sum;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      at[4 * threadIdx.x + k] = x;
      x += c[k];
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int r = threadIdx.x; r < n_req; r += 1024)
    order[atomicAdd(at + length_class(tok_off[r + 1] - tok_off[r]), 1u)] = (uint32_t)r;
  sm100::pdl_trigger();
}

// Insert (instance, key) pairs.  A new key takes a slot (CAS on 0); the
// instance's bit is OR-ed into the slot's mask; a bit set for the first time
// counts one distinct key of that instance (more than max_keys latches
// LS_ERR_TABLE_FULL, as does a probe sequence that finds no room).  With
// W == 1 keys and masks share the interleaved entry array gkeys (gmask unused).
//
// A warp takes U * 32 consecutive keys, so nearly every warp holds keys of one
// instance: it finds that instance once and adds its distinct keys to the
// instance's counter with one atomic.  (An atomic per key serialised on the few
// counter addresses bounded the kernel: a rebuild of 32 instances of 16,384
// keys with a 256-request route behind it took 384 us, 64 us with one per
// warp.)  A thread's U first probes are in flight together; what remains is two
// dependent L2 atomics per key.
template <int U>
__global__ void __launch_bounds__(256) k_index_insert(const uint64_t* __restrict__ keys,
                                                      const int64_t* __restrict__ key_off, int n_inst,
                                                      int64_t n_keys, uint64_t* gkeys, uint64_t* gmask, int W,
                                                      uint64_t gmask_slots, int32_t* counts, int64_t max_keys,
                                                      int* err) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long* tab = reinterpret_cast<unsigned long long*>(gkeys);
  const int kstride = W == 1 ? 2 : 1;
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c * (32 * U) < n_keys; c += warps) {
    const int64_t base = c * (32 * U);
    const int first = key_instance(key_off, n_inst, base);
    // (the last instance takes whatever follows its first key)
    const bool one = first == n_inst - 1 || base + 32 * U <= key_off[first + 1];
    unsigned long long key[U], prev[U];
    bool in[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t k = base + 32 * u + lane;
      in[u] = k < n_keys;
      key[u] = in[u] ? keys[k] : 0ull;
      if (key[u] == 0) key[u] = 1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      prev[u] = in[u] ? atomicCAS(tab + (key[u] & gmask_slots) * kstride, 0ull, key[u]) : 0ull;
    bool fresh[U];
    int inst[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      fresh[u] = false;
      inst[u] = one ? first : in[u] ? key_instance(key_off, n_inst, base + 32 * u + lane) : 0;
      if (!in[u]) continue;
      uint64_t s = key[u] & gmask_slots;
      bool found = prev[u] == 0ull || prev[u] == key[u];
      for (uint64_t n = 0; !found && n < gmask_slots; ++n) {  // the other slots, linearly
        s = (s + 1) & gmask_slots;
        const unsigned long long p = atomicCAS(tab + s * kstride, 0ull, key[u]);
        found = p == 0ull || p == key[u];
      }
      if (!found) {
        latch_error(err, LS_ERR_TABLE_FULL);
        continue;
      }
      const unsigned long long bit = 1ull << (inst[u] & 63);
      unsigned long long* mword =
          W == 1 ? tab + 2 * s + 1 : reinterpret_cast<unsigned long long*>(gmask + s * W + (inst[u] >> 6));
      fresh[u] = !(atomicOr(mword, bit) & bit);
    }
    if (one) {
      int n = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) n += __popc(__ballot_sync(kFull, fresh[u]));
      if (lane == 0 && n > 0 && (int64_t)atomicAdd(counts + first, n) + n > max_keys)
        latch_error(err, LS_ERR_TABLE_FULL);
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (fresh[u] && (int64_t)atomicAdd(counts + inst[u], 1) >= max_keys) latch_error(err, LS_ERR_TABLE_FULL);
    }
  }
}

}  // namespace

int index_words(int max_instances) { return max_instances <= 64 ? 1 : max_instances <= 128 ? 2 : max_instances <= 256 ? 4 : max_instances <= 512 ? 8 : 0; }

namespace {
using WalkKernel = void (*)(int, const int32_t*, const int64_t*, const uint64_t*, const uint64_t*, uint64_t, int,
                            int32_t*, DevState*, const uint32_t*);
WalkKernel walk_kernel(int W) {
  switch (W) {
    case 1: return k_prefix_index<1>;
    case 2: return k_prefix_index<2>;
    case 4: return k_prefix_index<4>;
    case 8: return k_prefix_index<8>;
  }
  return nullptr;
}

// A CTA of eight or four warps per request while that many CTAs fit.
bool walk_by_cta(int n_req, int W, int sms) { return n_req <= 8 * sms && (W <= 4 || n_req <= sms); }

// CTAs of the walk by warps that are resident at once.
int walk_resident(int W, int sms) {
  static int resident[9] = {};
  if (!resident[W]) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_kernel(W), kNT, 0) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      per_sm = 1;
    }
    resident[W] = per_sm;
  }
  return sms * resident[W];
}

int walk_ctas(int n_req) { return (n_req + kNT / 32 - 1) / (kNT / 32); }  // a warp per request
}  // namespace

// More requests than warps at once: the long ones first (8192 prompts of 8k to
// 32k tokens over 64 instances: a route took 334 us in order, 318 so).
bool prefix_index_sorts(int n_req, int W, int sms) {
  return walk_kernel(W) && !walk_by_cta(n_req, W, sms) && walk_resident(W, sms) < walk_ctas(n_req);
}

cudaError_t launch_walk_order(int n_req, const int64_t* tok_off, uint32_t* order, cudaStream_t s) {
  return launch_chained(k_walk_order, dim3(1), dim3(1024), 0, s, 1, n_req, tok_off, order);
}

cudaError_t launch_prefix_index(int n_req, const int32_t* tok, const int64_t* tok_off, const uint64_t* gkeys,
                                const uint64_t* gmask, int W, uint64_t gmask_slots, int n_inst, int32_t* hits,
                                const uint32_t* order, int sms, DevState* st, cudaStream_t s) {
  if (n_req <= 0) return cudaSuccess;
  const WalkKernel k = walk_kernel(W);
  if (!k) return cudaErrorInvalidValue;
  if (walk_by_cta(n_req, W, sms)) {
    void (*c)(const int32_t*, const int64_t*, const uint64_t*, const uint64_t*, uint64_t, int, int32_t*, DevState*) =
        nullptr;
    const bool wide = n_req <= 4 * sms;
    switch (W) {
      case 1: c = wide ? k_prefix_index_coop<1, 8> : k_prefix_index_coop<1, 4>; break;
      case 2: c = wide ? k_prefix_index_coop<2, 8> : k_prefix_index_coop<2, 4>; break;
      case 4: c = wide ? k_prefix_index_coop<4, 8> : k_prefix_index_coop<4, 4>; break;
      default: c = k_prefix_index_coop<8, 8>; break;  // (at most a request per SM)
    }
    return launch_chained(c, dim3(n_req), dim3(wide ? 256 : 128), 0, s, 1, tok, tok_off, gkeys, gmask, gmask_slots,
                          n_inst, hits, st);
  }
  // as many warps as are resident at once (they then take requests from the
  // counter); with no state to keep the counter in, one warp per request
  const int grid = std::max(1, std::min(walk_ctas(n_req), st ? walk_resident(W, sms) : sms * 16));
  return launch_chained(k, dim3(grid), dim3(kNT), 0, s, 1, n_req, tok, tok_off, gkeys, gmask, gmask_slots, n_inst,
                        hits, st, order);
}

cudaError_t launch_index_insert(const uint64_t* keys, const int64_t* key_off, int n_inst, int64_t n_keys,
                                uint64_t* gkeys, uint64_t* gmask, int W, uint64_t gmask_slots, int32_t* counts,
                                int64_t max_keys, bool cleared, int* err, int sms, cudaStream_t s) {
  if (n_keys <= 0 || n_inst <= 0) return cudaSuccess;
  // Four keys a thread once a cleared table takes more keys than the GPU has
  // threads (whole calls: 1,048,576 keys of 64 instances 39.7 us, 45.4 with one
  // a thread; 2,000,000 of one 105, 136); one while threads are idle (100,000
  // keys of one instance 22.9 us, 38.2 with four) and into a filled table, where
  // the probes find their keys and the second atomic is the longer wait
  // (2,000,000 keys already held 54 us, 85 with four).
  const bool four = cleared && n_keys > (int64_t)sms * 2048;
  const int64_t per = 256 * (four ? 4 : 1);
  const int64_t blocks = std::min<int64_t>((n_keys + per - 1) / per, (int64_t)sms * 32);
  auto* k = four ? k_index_insert<4> : k_index_insert<1>;
  k<<<(int)blocks, 256, 0, s>>>(keys, key_off, n_inst, n_keys, gkeys, gmask, W, gmask_slots, counts, max_keys, err);
  return cudaGetLastError();
}

}  // namespace ls
