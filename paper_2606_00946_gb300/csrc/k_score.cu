// Scoring kernels on CUDA cores: feature assembly (Sec. 4.1 Features,
// Algorithm 4 Normalize), the reward-model forward pass for small or fp32
// predictors (Sec. 4.1 Model architecture), the greedy argmin selector
// (Algorithm 4, argmax reward = argmin predicted TTFT) and the sample ring.
#include "common.cuh"
#include "sm100.cuh"

namespace ls {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float norm_feature(int k, int64_t L, int h, const float* inst,
                                             int d_inst, const float* req, const float* mean,
                                             const float* stdv) {
  return zscore(raw_feature(k, L, h, inst, d_inst, req), mean[k], stdv[k]);
}

__global__ void k_assemble(int n_req, int n_inst, const int64_t* __restrict__ tok_off,
                           const int32_t* __restrict__ hits, const float* __restrict__ inst_state,
                           int d_inst, const float* __restrict__ req_feats, int d_req,
                           const float* __restrict__ mean, const float* __restrict__ stdv,
                           float* __restrict__ x_out) {
  const int d = kPair + d_inst + d_req;
  const int64_t total = (int64_t)n_req * n_inst * d;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / d;
    const int k = (int)(e - row * d);
    const int r = (int)(row / n_inst), i = (int)(row - (int64_t)r * n_inst);
    const int64_t L = tok_off[r + 1] - tok_off[r];
    x_out[e] = norm_feature(k, L, hits[row], inst_state + (int64_t)i * d_inst, d_inst,
                            req_feats + (int64_t)r * d_req, mean, stdv);
  }
}

// The first of the warp's (score, index) candidates in the selection order
// (index -1: none), in every lane.
__device__ __forceinline__ void warp_first(float& bv, int& bi) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float ov = __shfl_xor_sync(kFull, bv, o);
    const int oi = __shfl_xor_sync(kFull, bi, o);
    if (oi >= 0 && (bi < 0 || score_precedes(ov, oi, bv, bi))) { bv = ov; bi = oi; }
  }
}

// Forward pass of tiles of TR pair rows (row = r * n_inst + i) on CUDA cores.
// Activations lie in shared memory as [unit][row], rows adjacent (pitch TR + 4),
// so one 16-byte load gives a thread four rows of a unit; a thread forms RV
// rows x CT outputs (lanes along the outputs, 32 apart), each sum in K order,
// the bias added after it.  What bounds it is the operand loads from shared
// memory: a 16-byte load is 512 bytes for a warp whether or not its lanes share
// the address, so a thread takes as many outputs per activation load as it has
// registers for (four, 128 a warp).  Route calls as graph replays, before (a
// thread per output over 16 rows, so half to three quarters of the threads idle
// below 128 outputs) and now: 64 x 8 rows of 16-64-64-1 18.9 -> 13.2 us, 1024 x
// 32 of 64-128-128-128-1 236 -> 107, 256 x 64 of 64-256-256-1 176 -> 124.
// The weights W^T [in, out] stream from the published copy; when every CTA runs
// one tile and they fit (`SM`), they are staged in shared memory first, all
// loads in flight together.
// Output layer (width 1): one warp per row, lanes split the dot product.
// With whole requests in a tile (`rq` > 0 of them) the selection runs here.
constexpr int kSimtT = 256;
constexpr int kSimtW = kSimtT / 32;

struct SimtArgs {
  MlpDesc mlp;
  const float* pp[2];
  const float* wt[2];
  const int32_t* sel;
  int n_req, n_inst, d_inst, d_req, tr, rq;
  int64_t tiles;
  const int64_t* tok_off;
  const int32_t* hits;
  const float* inst_state;
  const float* req_feats;
  const float* mean;
  const float* stdv;
  float* scores;      // nullable when the selection runs here
  int32_t* choice;
  float* best;
};

struct SimtRow {
  int r, i;  // request and instance
};

// One K step: row values x[RV], weights w[32 c].
template <int RV, int CT>
__device__ __forceinline__ void simt_step(const float* x, const float* w, float (&acc)[CT][RV]) {
  float xv[RV], wv[CT];
#pragma unroll
  for (int q = 0; q < RV / 4; ++q) {
    const float4 t = reinterpret_cast<const float4*>(x)[q];
    xv[4 * q] = t.x;
    xv[4 * q + 1] = t.y;
    xv[4 * q + 2] = t.z;
    xv[4 * q + 3] = t.w;
  }
#pragma unroll
  for (int c = 0; c < CT; ++c) wv[c] = w[32 * c];
#pragma unroll
  for (int c = 0; c < CT; ++c)
#pragma unroll
    for (int q = 0; q < RV; ++q) acc[c][q] = fmaf(xv[q], wv[c], acc[c][q]);
}

// Bias, ReLU and rounding of a thread's outputs o + 32 c for rows r0 ..
template <int RV, int CT>
__device__ __forceinline__ void simt_store(const float (&acc)[CT][RV], const float* __restrict__ bias, float* xout,
                                           int o, int out, int r0, int P, int bf16) {
#pragma unroll
  for (int c = 0; c < CT; ++c) {
    if (o + 32 * c >= out) break;
    const float bo = __ldg(bias + o + 32 * c);
    float* d = xout + (o + 32 * c) * P + r0;
#pragma unroll
    for (int q = 0; q < RV; ++q) {
      float z = acc[c][q] + bo;
      z = z > 0.0f ? z : 0.0f;
      d[q] = bf16 ? round_bf16(z) : z;
    }
  }
}

// A hidden layer with its weights [in][out] in shared memory (readable 32 CT
// floats past their end).
template <int RV, int CT>
__device__ __forceinline__ void simt_layer(const float* W, const float* __restrict__ bias, const float* xin,
                                           float* xout, int in, int out, int tr, int P, int bf16) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = (out + 32 * CT - 1) / (32 * CT), rg = tr / RV;
#pragma unroll 1
  for (int e = warp; e < groups * rg; e += kSimtW) {
    const int g = e / rg, r0 = (e - g * rg) * RV, o = g * 32 * CT + lane;
    float acc[CT][RV];
#pragma unroll
    for (int c = 0; c < CT; ++c)
#pragma unroll
      for (int q = 0; q < RV; ++q) acc[c][q] = 0.0f;
    const float* w = W + o;
    const float* x = xin + r0;
#pragma unroll 4
    for (int k = 0; k < in; ++k, w += out, x += P) simt_step<RV, CT>(x, w, acc);
    simt_store<RV, CT>(acc, bias, xout, o, out, r0, P, bf16);
  }
}

// A hidden layer whose weights stream from the published copy: kSimtK K steps
// of the columns the CTA's warps work on at a time, through kSimtStages
// asynchronous copies that every warp shares.  (Read through L1 by each warp
// for itself, the 164 KB of 64-128-128-128-1 beside two CTAs' activations
// missed it: 105 us for 32,768 rows, a third of the stalls on these loads.)
constexpr int kSimtK = 16;
constexpr int kSimtStages = 3;

template <int RV, int CT>
__device__ __forceinline__ void simt_layer_stream(const float* __restrict__ W, const float* __restrict__ bias,
                                                  const float* xin, float* xout, float* ring, int in, int out, int tr,
                                                  int P, int bf16) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rg = tr / RV;                  // 1, 2, 4 or 8 warps along the rows
  const int cols = kSimtW / rg * 32 * CT;  // columns the warps cover together
  const int g = warp / rg, r0 = (warp - g * rg) * RV;
  const int chunks = (in + kSimtK - 1) / kSimtK;
  const bool vec = (out & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
#pragma unroll 1
  for (int c0 = 0; c0 < out; c0 += cols) {
    const int nc = min(cols, out - c0);
    const auto copy = [&](int chunk) {
      float* st = ring + (chunk % kSimtStages) * kSimtK * cols;
      const int k0 = chunk * kSimtK, nk = min(kSimtK, in - k0);
      const float* src = W + (int64_t)k0 * out + c0;
      if (vec) {
        const int per = cols >> 2, sh = __ffs(per) - 1;  // a power of two
        for (int e = threadIdx.x; e < kSimtK * per; e += kSimtT) {
          const int k = e >> sh, c = 4 * (e & (per - 1));
          if (k < nk && c < nc) sm100::cp_async16(st + k * cols + c, src + (int64_t)k * out + c);
        }
      } else {
        const int sh = __ffs(cols) - 1;
        for (int e = threadIdx.x; e < kSimtK * cols; e += kSimtT) {
          const int k = e >> sh, c = e & (cols - 1);
          if (k < nk && c < nc) sm100::cp_async4(st + k * cols + c, src + (int64_t)k * out + c);
        }
      }
    };
    __syncthreads();  // the ring is free
#pragma unroll
    for (int q = 0; q < kSimtStages - 1; ++q) {
      if (q < chunks) copy(q);
      sm100::cp_async_commit();
    }
    float acc[CT][RV];
#pragma unroll
    for (int c = 0; c < CT; ++c)
#pragma unroll
      for (int q = 0; q < RV; ++q) acc[c][q] = 0.0f;
    const float* x = xin + r0;
#pragma unroll 1
    for (int chunk = 0; chunk < chunks; ++chunk) {
      sm100::cp_async_wait<kSimtStages - 2>();
      __syncthreads();  // the chunk is in, and every warp is done with the one before it
      if (chunk + kSimtStages - 1 < chunks) copy(chunk + kSimtStages - 1);
      sm100::cp_async_commit();
      const float* w = ring + (chunk % kSimtStages) * kSimtK * cols + g * 32 * CT + lane;
      const int nk = min(kSimtK, in - chunk * kSimtK);
      if (nk == kSimtK) {
#pragma unroll 4
        for (int k = 0; k < kSimtK; ++k, x += P) simt_step<RV, CT>(x, w + k * cols, acc);
      } else {
#pragma unroll 1
        for (int k = 0; k < nk; ++k, x += P) simt_step<RV, CT>(x, w + k * cols, acc);
      }
    }
    simt_store<RV, CT>(acc, bias, xout, c0 + g * 32 * CT + lane, out, r0, P, bf16);
  }
}

template <int RV, bool SM>
__global__ void __launch_bounds__(kSimtT, 2) k_score_simt(const __grid_constant__ SimtArgs a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ SimtRow s_row[64];
  sm100::pdl_wait();  // hit lengths and the route's buffer from the prefix kernel
  const MlpDesc& mlp = a.mlp;
  const int b1 = a.sel && *a.sel == 1 ? 1 : 0;  // published buffer of this route
  const float* __restrict__ pp = a.pp[b1];
  const float* __restrict__ wt = a.wt[b1];
  const int tr = a.tr, P = tr + 4, L = mlp.n_layers, d = mlp.w[0];
  float* xa = smem;
  float* xb = smem + mlp.max_width * P;
  float* sc = xb + mlp.max_width * P;  // [tr] scores of the tile
  float* ws = sc + tr;                 // the hidden layers' weights (SM), or the ring they stream through
  const int64_t rows = (int64_t)a.n_req * a.n_inst;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int step = a.rq > 0 ? a.rq * a.n_inst : tr;  // rows of a tile
  if (SM) {
    const int n = (int)mlp.wtoff[L - 1];  // every hidden layer's
#pragma unroll 8
    for (int e = threadIdx.x; e < n; e += kSimtT) ws[e] = __ldg(wt + e);
  }

  // feature k of tile row rr, rounded to bf16 in bf16 mode
  const auto put = [&](float* x, int k, int rr, float v) { x[k * P + rr] = mlp.bf16 ? round_bf16(v) : v; };

  for (int64_t t = blockIdx.x; t < a.tiles; t += gridDim.x) {
    const int64_t row0 = t * step;
    float* x = xa;
    float* y = xb;
    if (threadIdx.x < tr) {
      const int64_t g = row0 + threadIdx.x;
      SimtRow e{0, 0};
      if ((int)threadIdx.x < step && g < rows) {
        e.r = (int)(g / a.n_inst);
        e.i = (int)(g - (int64_t)e.r * a.n_inst);
        const int64_t len = a.tok_off[e.r + 1] - a.tok_off[e.r];
        const int h = a.hits[g];
#pragma unroll
        for (int k = 0; k < kPair; ++k)
          put(x, k, threadIdx.x, zscore(raw_feature(k, len, h, nullptr, 0, nullptr), a.mean[k], a.stdv[k]));
      } else {  // no row here: what the layers form is not used (instance 0's values, 0 elsewhere)
        for (int k = 0; k < d; ++k)
          if (k < kPair || k >= kPair + a.d_inst) x[k * P + threadIdx.x] = 0.0f;
      }
      s_row[threadIdx.x] = e;
    }
    __syncthreads();
    // instance columns: a warp per row, lanes along the columns
#pragma unroll 2
    for (int rr = warp; rr < tr; rr += kSimtW) {
      const int i = s_row[rr].i;
      for (int k = lane; k < a.d_inst; k += 32)
        put(x, kPair + k, rr, zscore(__ldg(a.inst_state + (int64_t)i * a.d_inst + k), a.mean[kPair + k],
                                     a.stdv[kPair + k]));
    }
    // request columns: a warp per request of the tile, its rows share the values
    const int r_first = s_row[0].r, r_last = s_row[min(step, (int)(rows - row0)) - 1].r;
    for (int r = r_first + warp; r <= r_last; r += kSimtW) {
      const int64_t at = (int64_t)r * a.n_inst - row0;
      const int lo = (int)(at < 0 ? 0 : at), hi = (int)min((int64_t)step, at + a.n_inst);
      for (int k = lane; k < a.d_req; k += 32) {
        const int col = kPair + a.d_inst + k;
        const float v = zscore(__ldg(a.req_feats + (int64_t)r * a.d_req + k), a.mean[col], a.stdv[col]);
        for (int rr = lo; rr < hi; ++rr) put(x, col, rr, v);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int l = 0; l + 1 < L; ++l) {
      const int in = mlp.w[l], out = mlp.w[l + 1];
      const float* W = SM ? ws + mlp.wtoff[l] : wt + mlp.wtoff[l];
      const float* bias = pp + mlp.boff[l];
      // four outputs a thread (128 a warp) even where that leaves warps idle:
      // the operand loads, not the warps, are short; two in the low tiles,
      // whose one or two warps would wait for their own latency
      if (SM) {
        if (out > 64 && tr >= 16) simt_layer<RV, 4>(W, bias, x, y, in, out, tr, P, mlp.bf16);
        else simt_layer<RV, 2>(W, bias, x, y, in, out, tr, P, mlp.bf16);
      } else {
        if (out > 64 && tr >= 16) simt_layer_stream<RV, 4>(W, bias, x, y, ws, in, out, tr, P, mlp.bf16);
        else simt_layer_stream<RV, 2>(W, bias, x, y, ws, in, out, tr, P, mlp.bf16);
      }
      __syncthreads();
      float* s = x;
      x = y;
      y = s;
    }
    {  // output layer, width 1
      const int in = mlp.w[L - 1];
      const float* __restrict__ W = wt + mlp.wtoff[L - 1];
      const float bo = __ldg(pp + mlp.boff[L - 1]);
      for (int rr = warp; rr < tr; rr += kSimtW) {
        float s = 0.0f;
        for (int k = lane; k < in; k += 32) s = fmaf(x[k * P + rr], __ldg(W + k), s);
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (lane == 0) {
          sc[rr] = s + bo;
          if (a.scores && rr < step && row0 + rr < rows) a.scores[row0 + rr] = s + bo;
        }
      }
    }
    __syncthreads();
    // the greedy selection of the tile's requests, a warp each
    for (int q = warp; q < a.rq; q += kSimtW) {
      const int64_t r = t * a.rq + q;
      if (r >= a.n_req) break;
      float bv = 0.0f;
      int bi = -1;
      for (int i = lane; i < a.n_inst; i += 32) {
        const float v = sc[q * a.n_inst + i];
        if (bi < 0 || score_precedes(v, i, bv, bi)) { bv = v; bi = i; }
      }
      warp_first(bv, bi);
      if (lane == 0) { a.choice[r] = bi; a.best[r] = bv; }
    }
    __syncthreads();
  }
  sm100::pdl_trigger();
}

// One warp per request: lexicographic (score, index) minimum over instances.
__global__ void k_argmin(int n_req, int n_inst, const float* __restrict__ scores,
                         int32_t* __restrict__ choice, float* __restrict__ best) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (r >= n_req) return;
  const float* s = scores + r * n_inst;
  float bv = 0.0f;
  int bi = -1;
  for (int i = lane; i < n_inst; i += 32) {
    const float v = s[i];
    if (bi < 0 || score_precedes(v, i, bv, bi)) { bv = v; bi = i; }
  }
  warp_first(bv, bi);
  if (lane == 0) { choice[r] = bi; best[r] = bv; }
}

// Record j of the batch -> slot (count + j) mod capacity, count = records
// appended before this batch (device state); the last block advances the
// count by n.  When a batch is longer than the ring only its last `capacity`
// records are kept.  With a pending ring (pending > 0; then n <= capacity)
// the record a slot held, stream position p - capacity, is first copied to
// pending row capacity + (p - capacity) mod pending by the thread that then
// overwrites the same piece; of the records one call evicts only the newest
// `pending` are copied, so no two copies share a row.
__global__ void k_ring_append(int n, int d, const float* __restrict__ x, const float* __restrict__ y,
                              float* ring_x, float* ring_y, DevState* st, int64_t capacity, int64_t pending) {
  const int64_t count = *reinterpret_cast<volatile int64_t*>(&st->ring_count);
  const int64_t first = n > capacity ? n - capacity : 0;
  // piece = 4 consecutive columns of one record (the last piece of a record
  // may be short); pieces of a record share its slot
  const int per = (d + 3) / 4;
  const int64_t total = (int64_t)(n - first) * per;
  const bool vec = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(ring_x) & 15) == 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t jj = e / per;
    const int k = (int)(e - jj * per) * 4;
    const int64_t j = first + jj;
    const int64_t slot = (count + j) % capacity;
    const float* src = x + j * d + k;
    float* dst = ring_x + slot * d + k;
    // only the newest `pending` records this call evicts are kept (older ones
    // would land on the same pending rows)
    if (pending > 0 && count + j >= capacity && count + j - capacity >= count + n - capacity - pending) {
      const int64_t prow = capacity + (count + j - capacity) % pending;
      float* pdst = ring_x + prow * d + k;
      if (vec) {
        *reinterpret_cast<float4*>(pdst) = *reinterpret_cast<const float4*>(dst);
      } else {
        for (int u = 0; u < 4 && k + u < d; ++u) pdst[u] = dst[u];
      }
      if (k == 0) ring_y[prow] = ring_y[slot];
    }
    if (vec) {
      *reinterpret_cast<float4*>(dst) = __ldg(reinterpret_cast<const float4*>(src));
    } else {
      for (int u = 0; u < 4 && k + u < d; ++u) dst[u] = __ldg(src + u);
    }
    if (k == 0) ring_y[slot] = y[j];
  }
  if (last_block(&st->done[DONE_RING]) && threadIdx.x == 0) st->ring_count = count + n;
}

int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

int grid_1d(int64_t n, int threads, int per_sm = 8) {
  int64_t g = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count() * per_sm;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

cudaError_t launch_assemble_features(int n_req, int n_inst, const int64_t* tok_off,
                                     const int32_t* hits, const float* inst_state, int d_inst,
                                     const float* req_feats, int d_req, const float* mean,
                                     const float* stdv, float* x_out, cudaStream_t s) {
  const int64_t total = (int64_t)n_req * n_inst * (kPair + d_inst + d_req);
  if (total <= 0) return cudaSuccess;
  k_assemble<<<grid_1d(total, 256), 256, 0, s>>>(n_req, n_inst, tok_off, hits, inst_state, d_inst,
                                                req_feats, d_req, mean, stdv, x_out);
  return cudaGetLastError();
}

namespace {
// How the CUDA-core scorer splits a batch: rows per tile (the smallest of 4 to
// 64 that leaves a tile per SM or fewer: a small batch spreads over the SMs, a
// large one shares each weight load among many rows), requests per tile when
// the selection runs in the scorer (0: it does not), and whether the weights
// are staged.
struct SimtPlan {
  int tr, rq, staged, smem;
  int64_t tiles;
};

SimtPlan plan_simt(const MlpDesc& m, int n_req, int n_inst, int sms) {
  SimtPlan p{};
  const int64_t rows = (int64_t)n_req * n_inst;
  p.tr = 4;
  while (p.tr < 64 && (rows + p.tr - 1) / p.tr > sms) p.tr *= 2;
  // activations and scores; the weight ring (columns of all warps, see simt_layer_stream)
  const auto bytes = [&](int tr) { return (2 * m.max_width * (tr + 4) + tr) * 4; };
  const auto ring = [&](int tr) {
    const int rg = tr / (tr <= 16 ? 4 : 8), ct = tr >= 16 ? 4 : 2;
    return kSimtStages * kSimtK * (kSimtW / rg) * 32 * ct * 4;
  };
  const int most = 224 * 1024;
  // whole requests per tile, where that leaves a tile per SM or fewer, or at
  // most a quarter of a tile's rows unused; tiles grow to 16 rows for it (a
  // launch saved), not further (fewer SMs at work)
  int tr = p.tr;
  while (tr < 16 && tr < n_inst) tr *= 2;
  if (n_inst <= tr && bytes(tr) + ring(tr) <= most) {
    const int rq = tr / n_inst;
    if ((n_req + rq - 1) / rq <= sms || 4 * rq * n_inst >= 3 * tr) {
      p.tr = tr;
      p.rq = rq;
    }
  }
  while (p.tr > 4 && bytes(p.tr) + ring(p.tr) > most) p.tr /= 2;  // (very wide layers; then without selection)
  p.tiles = p.rq ? (n_req + p.rq - 1) / p.rq : (rows + p.tr - 1) / p.tr;
  p.smem = bytes(p.tr);
  const int64_t w = m.wtoff[m.n_layers - 1] * 4;
  p.staged = p.tiles <= sms && p.smem + w + 512 <= most;
  p.smem += p.staged ? (int)w + 512 : ring(p.tr);
  return p;
}
}  // namespace

bool simt_selects(const MlpDesc& m, int n_req, int n_inst, int sms) { return plan_simt(m, n_req, n_inst, sms).rq > 0; }

cudaError_t launch_score_simt(const MlpDesc& mlp, const Published* pub, const int32_t* sel, int n_req, int n_inst,
                              const int64_t* tok_off, const int32_t* hits, const float* inst_state,
                              int d_inst, const float* req_feats, int d_req, const float* mean,
                              const float* stdv, float* scores, int32_t* choice, float* best, int sms,
                              cudaStream_t s) {
  if (n_req <= 0) return cudaSuccess;
  const SimtPlan p = plan_simt(mlp, n_req, n_inst, sms);
  SimtArgs a{};
  a.mlp = mlp;
  for (int b = 0; b < 2; ++b) {
    a.pp[b] = pub[b].params;
    a.wt[b] = pub[b].wt;
  }
  a.sel = sel;
  a.n_req = n_req;
  a.n_inst = n_inst;
  a.d_inst = d_inst;
  a.d_req = d_req;
  a.tr = p.tr;
  a.rq = choice ? p.rq : 0;
  a.tiles = a.rq ? p.tiles : ((int64_t)n_req * n_inst + p.tr - 1) / p.tr;
  a.tok_off = tok_off;
  a.hits = hits;
  a.inst_state = inst_state;
  a.req_feats = req_feats;
  a.mean = mean;
  a.stdv = stdv;
  a.scores = scores;
  a.choice = choice;
  a.best = best;
  auto* launch = p.tr <= 16 ? (p.staged ? launch_smem<k_score_simt<4, true>, SimtArgs&>
                                        : launch_smem<k_score_simt<4, false>, SimtArgs&>)
                            : (p.staged ? launch_smem<k_score_simt<8, true>, SimtArgs&>
                                        : launch_smem<k_score_simt<8, false>, SimtArgs&>);
  const int grid = (int)std::min<int64_t>(a.tiles, 2 * (int64_t)sms);
  return launch(dim3(grid), dim3(kSimtT), (size_t)p.smem, s, 1, a);
}

cudaError_t launch_argmin(int n_req, int n_inst, const float* scores, int32_t* choice, float* best,
                          cudaStream_t s) {
  if (n_req <= 0) return cudaSuccess;
  const int64_t threads = (int64_t)n_req * 32;
  k_argmin<<<(int)((threads + 255) / 256), 256, 0, s>>>(n_req, n_inst, scores, choice, best);
  return cudaGetLastError();
}

cudaError_t launch_ring_append(int n, int d, const float* x, const float* y, float* ring_x,
                               float* ring_y, DevState* st, int64_t capacity, int64_t pending, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t keep = n > capacity ? capacity : n;
  const int64_t total = keep * ((d + 3) / 4);
  k_ring_append<<<grid_1d(total, 256), 256, 0, s>>>(n, d, x, y, ring_x, ring_y, st, capacity, pending);
  return cudaGetLastError();
}

}  // namespace ls
