// Training step of an fp32 predictor in two launches (Sec. 4.3.2 online
// learning; loss and optimisers as in k_train.cu: mean squared error, SGD or
// Adam, fp32 throughout):
//   k_trs_grad  a CTA takes tiles of 4 to 32 minibatch rows through the whole
//               step on chip: gather and z-score, the forward layers, the
//               output layer and loss, and the backward layers, its gradient
//               partials (every parameter) written to its own row of a buffer;
//   k_trs_opt   each parameter's gradient is the ordered sum of the CTAs'
//               partials, then the update; one warp adds the loss.
// A small predictor's step is bound by launches and by latency, not by its
// arithmetic.  Device time per step as graph replays, 20 launches of the
// general path before and two now: 16-64-64-1 on 256 rows 76 -> 17 us,
// 64-128-128-128-1 on 1024 rows 164 -> 44 us, 64-256-256-1 on 1024 rows
// (weights in chunks) 142 -> 90 us, 16-64-64-1 on 4096 rows 97 -> 42 us.
// Within a CTA shared-memory loads are the bound (a load of 16 bytes a lane
// takes four cycles whether or not the lanes share an address), so a thread
// forms 4 or 8 rows x one or two outputs from each activation load, rows
// adjacent.
//
// Shared memory holds W_l^T [in][out] with an odd pitch (lanes along the
// outputs in the forward layers, along the inputs in the backward ones,
// without bank conflicts either way), the input of every layer [in][rows] and
// two dZ buffers [out][rows].  When the weights do not all fit, a layer's are
// staged in chunks of outputs as they are needed.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "sm100.cuh"

namespace ls {
using namespace sm100;

namespace {

constexpr int kT = 256;
constexpr int kWarps = kT / 32;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kSmemMax = 220 * 1024;
constexpr int64_t kMaxParams = 128 * 1024;  // partials of every CTA: 78 MB at most

struct TrsArgs {
  MlpDesc m;
  int B, tr, tiles;
  int resident;                   // all weights staged once
  int chunk;                      // outputs staged at once (not resident)
  int woff_s[LS_MAX_LAYERS];      // floats: layer l's weights (resident) in the weight region
  int xoff_s[LS_MAX_LAYERS];      // floats: layer l's input
  int x_total, dz_rows;           // floats of all inputs; rows of a dZ buffer
  const int32_t* idx;
  DevState* st;
  int64_t capacity, replay_base;
  const float* ring_x;
  const float* ring_y;
  const float* mean;
  const float* stdv;
  const float* p;                 // master parameters
  float* part;                    // [CTA][n_params + 2]: gradient partials, then the squared errors (high, low)
  int64_t ld;
  int* err;
};

__device__ __forceinline__ int pitch(int out) { return out | 1; }

// Stage outputs [o0, o0 + oc) of layer l: dst[k * pitch(oc) + o - o0] = W[o][k].
__device__ __forceinline__ void trs_stage(const float* __restrict__ W, int in, int o0, int oc, float* dst) {
  const int pt = pitch(oc), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  W += (int64_t)o0 * in;
  if ((in & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0) {
    // 16 bytes a load, eight loads in flight; item e: output e / (in / 4), inputs 4 (e mod (in / 4))
    const int q4 = in >> 2, n = oc * q4;
    const float inv = 1.0f / (float)q4;
#pragma unroll 1
    for (int e0 = threadIdx.x; e0 < n; e0 += 8 * kT) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e0 + u * kT < n) v[u] = __ldg(reinterpret_cast<const float4*>(W) + e0 + u * kT);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * kT;
        if (e >= n) break;
        const int o = (int)(((float)e + 0.5f) * inv);  // e / q4 (e < 2^18: exact)
        float* w = dst + 4 * (e - o * q4) * pt + o;
        w[0] = v[u].x;
        w[pt] = v[u].y;
        w[2 * pt] = v[u].z;
        w[3 * pt] = v[u].w;
      }
    }
    return;
  }
#pragma unroll 1
  for (int k = lane; k < in; k += 32)  // a warp per output, eight rows of loads in flight
#pragma unroll 8
    for (int o = warp; o < oc; o += kWarps) dst[k * pt + o] = __ldg(W + (int64_t)o * in + k);
}

template <int RV>
__device__ __forceinline__ void ld_rows(const float* p, float (&v)[RV]) {
#pragma unroll
  for (int q = 0; q < RV / 4; ++q) {
    const float4 t = reinterpret_cast<const float4*>(p)[q];
    v[4 * q] = t.x;
    v[4 * q + 1] = t.y;
    v[4 * q + 2] = t.z;
    v[4 * q + 3] = t.w;
  }
}

// acc[c][q] += sum over s < n of w[s * ws + c * cs] src[s * tr + q]: one
// thread's CT columns x RV rows of a product whose summed index runs over n
// shared-memory rows of `src` (column c counted only when c < cols).
template <int RV, int CT>
__device__ __forceinline__ void trs_dot(const float* w, int ws, int cs, int cols, const float* src, int tr, int n,
                                        float (&acc)[CT][RV]) {
#pragma unroll 4
  for (int s = 0; s < n; ++s) {
    float x[RV];
    ld_rows<RV>(src + s * tr, x);
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      const float wv = c < cols ? w[s * ws + c * cs] : 0.0f;
#pragma unroll
      for (int q = 0; q < RV; ++q) acc[c][q] = fmaf(wv, x[q], acc[c][q]);
    }
  }
}

// Forward outputs [o0, o0 + oc): out[o][r] = relu(sum_k W[o][k] in[k][r] + b[o]).
template <int RV, int CT>
__device__ __forceinline__ void trs_fwd(const float* w, const float* __restrict__ bias, const float* xin, float* xout,
                                        int in, int o0, int oc, int tr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = (oc + 32 * CT - 1) / (32 * CT), rg = tr / RV;
#pragma unroll 1
  for (int e = warp; e < groups * rg; e += kWarps) {
    const int g = e / rg, r0 = (e - g * rg) * RV, o = g * 32 * CT + lane;
    const int cols = o >= oc ? 0 : (CT == 2 && o + 32 < oc) ? 2 : 1;
    float acc[CT][RV];
#pragma unroll
    for (int c = 0; c < CT; ++c)
#pragma unroll
      for (int q = 0; q < RV; ++q) acc[c][q] = 0.0f;
    trs_dot<RV, CT>(w + o, pitch(oc), 32, cols, xin + r0, tr, in, acc);
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      if (c >= cols) break;
      const float b = __ldg(bias + o0 + o + 32 * c);
      float* d = xout + (o0 + o + 32 * c) * tr + r0;
#pragma unroll
      for (int q = 0; q < RV; ++q) {
        const float z = acc[c][q] + b;
        d[q] = z > 0.0f ? z : 0.0f;
      }
    }
  }
}

// Input gradient from outputs [o0, o0 + oc): dx[k][r] (+)= sum_o W[o][k] dz[o][r],
// and on the last chunk the ReLU mask of the input.
template <int RV, int CT>
__device__ __forceinline__ void trs_dx(const float* w, const float* dz, float* dx, const float* x, int in, int o0,
                                       int oc, bool first, bool last, int tr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = (in + 32 * CT - 1) / (32 * CT), rg = tr / RV, pt = pitch(oc);
#pragma unroll 1
  for (int e = warp; e < groups * rg; e += kWarps) {
    const int g = e / rg, r0 = (e - g * rg) * RV, k = g * 32 * CT + lane;
    const int cols = k >= in ? 0 : (CT == 2 && k + 32 < in) ? 2 : 1;
    float acc[CT][RV];
#pragma unroll
    for (int c = 0; c < CT; ++c)
#pragma unroll
      for (int q = 0; q < RV; ++q) acc[c][q] = 0.0f;
    trs_dot<RV, CT>(w + k * pt, 1, 32 * pt, cols, dz + o0 * tr + r0, tr, oc, acc);
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      if (c >= cols) break;
      const int at = (k + 32 * c) * tr + r0;
#pragma unroll
      for (int q = 0; q < RV; ++q) {
        const float v = first ? acc[c][q] : dx[at + q] + acc[c][q];
        dx[at + q] = !last || x[at + q] > 0.0f ? v : 0.0f;
      }
    }
  }
}

// Weight gradient partial: part[o * in + k] (+)= sum_r dz[o][r] x[k][r], and
// db[o].  A thread takes four outputs x one or two inputs (32 apart).
template <int RV>
__device__ __forceinline__ void trs_dw(const float* dz, const float* x, float* part, float* part_b, int in, int out,
                                       int tr, bool add) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kg = (in + 63) / 64, og = (out + 3) / 4;
#pragma unroll 1
  for (int e = warp; e < kg * og; e += kWarps) {
    const int g = e / kg, o = 4 * g, k = (e - g * kg) * 64 + lane;
    const bool k0 = k < in, k1 = k + 32 < in;
    float acc[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0.0f;
#pragma unroll 1
    for (int r0 = 0; r0 < tr; r0 += RV) {
      float xa[RV], xb[RV];
      ld_rows<RV>(x + (k0 ? k : 0) * tr + r0, xa);
      ld_rows<RV>(x + (k1 ? k + 32 : 0) * tr + r0, xb);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float d[RV];
        ld_rows<RV>(dz + min(o + i, out - 1) * tr + r0, d);
#pragma unroll
        for (int q = 0; q < RV; ++q) {
          acc[i][0] = fmaf(d[q], xa[q], acc[i][0]);
          acc[i][1] = fmaf(d[q], xb[q], acc[i][1]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (o + i >= out) break;
      float* d = part + (int64_t)(o + i) * in + k;
      if (k0) d[0] = add ? d[0] + acc[i][0] : acc[i][0];
      if (k1) d[32] = add ? d[32] + acc[i][1] : acc[i][1];
    }
  }
  for (int o = threadIdx.x; o < out; o += kT) {
    float s = 0.0f;
    for (int r = 0; r < tr; ++r) s += dz[o * tr + r];
    part_b[o] = add ? part_b[o] + s : s;
  }
}

// (one CTA an SM is launched, so a thread may have 255 registers: held to 128
// for a second one, the kernel spilled)
template <int RV>
__global__ void __launch_bounds__(kT, 1) k_trs_grad(const __grid_constant__ TrsArgs a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_y[32], s_dz[32], s_e2[32];
  __shared__ int64_t s_row[32];
  const MlpDesc& m = a.m;
  const int tr = a.tr, L = m.n_layers, nh = L - 1, d = m.w[0];
  float* X = sm;                                // inputs of every layer
  float* dz0 = X + a.x_total;                   // dZ buffers
  float* dz1 = dz0 + a.dz_rows * tr;
  float* Wsm = dz1 + a.dz_rows * tr;            // weights
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* part = a.part + (int64_t)blockIdx.x * a.ld;
  pdl_wait();  // parameters, ring and counters from the previous kernels of the stream
  pdl_trigger();
  const int64_t step = a.st->step, count = a.st->ring_count;
  const int64_t nF = count < a.capacity ? count : a.capacity;
  const int64_t valid = nF + a.st->replay_count;  // F u R
  const int64_t first = valid > 0 ? step * (int64_t)a.B % valid : 0;
  if (blockIdx.x == 0 && tid == 0) {
    if (valid < 1) {
      latch_error(a.err, LS_ERR_STATE);
      a.st->train_abort = 1;  // the optimiser of this step leaves every parameter as it is
    }
    set_adam_bc(a.st);
  }
  if (a.resident)
#pragma unroll 1
    for (int l = 0; l < nh; ++l) trs_stage(a.p + m.woff[l], m.w[l], 0, m.w[l + 1], Wsm + a.woff_s[l]);
  const float b_out = __ldg(a.p + m.boff[nh]);
  double e2 = 0.0;  // thread 0: squared errors of this CTA's tiles
#pragma unroll 1
  for (int t = blockIdx.x; t < a.tiles; t += gridDim.x) {
    const bool add = t != (int)blockIdx.x;
    if (add) __syncthreads();  // the tile before is done with the buffers
    // ---- minibatch rows: slot idx[j] or (step B + j) mod valid, z-scored
    if (tid < tr) {
      const int j = t * tr + tid;
      int64_t row = -1;
      if (j < a.B && valid > 0) {
        int64_t slot;
        if (a.idx) {
          slot = a.idx[j];
          if (slot < 0 || slot >= valid) {
            latch_error(a.err, LS_ERR_ARG);
            a.st->train_abort = 1;
            slot = 0;
          }
        } else {
          slot = first + j;  // (step B + j) mod valid
          if (slot >= valid) slot %= valid;
        }
        row = union_row(slot, nF, a.replay_base);
      }
      s_row[tid] = row;
      s_y[tid] = row >= 0 ? a.ring_y[row] : 0.0f;
    }
    __syncthreads();
#pragma unroll 4
    for (int r = warp; r < tr; r += kWarps) {
      const int64_t row = s_row[r];
      for (int k = lane; k < d; k += 32)
        X[k * tr + r] = row >= 0 ? zscore(__ldg(a.ring_x + row * d + k), a.mean[k], a.stdv[k]) : 0.0f;
    }
    __syncthreads();
    // ---- forward
#pragma unroll 1
    for (int l = 0; l < nh; ++l) {
      const int in = m.w[l], out = m.w[l + 1], step_o = a.resident ? out : a.chunk;
#pragma unroll 1
      for (int o0 = 0; o0 < out; o0 += step_o) {
        const int oc = min(step_o, out - o0);
        float* w = a.resident ? Wsm + a.woff_s[l] : Wsm;
        if (!a.resident) {
          trs_stage(a.p + m.woff[l], in, o0, oc, w);
          __syncthreads();
        }
        const float* bias = a.p + m.boff[l];
        // two outputs a thread once one each would give every warp work
        if (((oc + 31) / 32) * (tr / RV) > kWarps)
          trs_fwd<RV, 2>(w, bias, X + a.xoff_s[l], X + a.xoff_s[l + 1], in, o0, oc, tr);
        else
          trs_fwd<RV, 1>(w, bias, X + a.xoff_s[l], X + a.xoff_s[l + 1], in, o0, oc, tr);
        __syncthreads();
      }
    }
    // ---- output layer (width 1), loss and its gradient: warp per row
    const int in_l = m.w[nh];
    const float* xl = X + a.xoff_s[nh];
    const float* wl = a.p + m.woff[nh];
#pragma unroll 1
    for (int r = warp; r < tr; r += kWarps) {
      float s = 0.0f;
      for (int k = lane; k < in_l; k += 32) s = fmaf(xl[k * tr + r], __ldg(wl + k), s);
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
      if (lane == 0) {
        const float e = t * tr + r < a.B ? (s + b_out) - s_y[r] : 0.0f;
        s_dz[r] = 2.0f * e / (float)a.B;
        s_e2[r] = e * e;
      }
    }
    __syncthreads();
    if (tid == 0) {
      float db = 0.0f;
      for (int r = 0; r < tr; ++r) {
        e2 += (double)s_e2[r];
        db += s_dz[r];
      }
      float* pb = part + m.boff[nh];
      *pb = add ? *pb + db : db;
    }
    for (int k = tid; k < in_l; k += kT) {
      const float w = __ldg(wl + k);
      float g = 0.0f;
      for (int r = 0; r < tr; ++r) {
        const float xv = xl[k * tr + r], dzr = s_dz[r];
        g = fmaf(dzr, xv, g);
        if (nh > 0) dz0[k * tr + r] = xv > 0.0f ? dzr * w : 0.0f;
      }
      float* pw = part + m.woff[nh] + k;
      *pw = add ? *pw + g : g;
    }
    __syncthreads();
    // ---- backward
    float *dz = dz0, *dx = dz1;
#pragma unroll 1
    for (int l = nh - 1; l >= 0; --l) {
      const int in = m.w[l], out = m.w[l + 1], step_o = a.resident ? out : a.chunk;
      const float* x = X + a.xoff_s[l];
      trs_dw<RV>(dz, x, part + m.woff[l], part + m.boff[l], in, out, tr, add);
      if (l > 0) {
#pragma unroll 1
        for (int o0 = 0; o0 < out; o0 += step_o) {
          const int oc = min(step_o, out - o0);
          float* w = a.resident ? Wsm + a.woff_s[l] : Wsm;
          if (!a.resident) {
            __syncthreads();
            trs_stage(a.p + m.woff[l], in, o0, oc, w);
            __syncthreads();
          }
          const bool first = o0 == 0, last = o0 + oc >= out;
          if (((in + 31) / 32) * (tr / RV) > kWarps) trs_dx<RV, 2>(w, dz, dx, x, in, o0, oc, first, last, tr);
          else trs_dx<RV, 1>(w, dz, dx, x, in, o0, oc, first, last, tr);
        }
      }
      __syncthreads();
      float* s = dz;
      dz = dx;
      dx = s;
    }
  }
  if (tid == 0) {
    part[a.ld - 2] = (float)e2;
    part[a.ld - 1] = (float)(e2 - (double)(float)e2);
  }
}

struct TrsOpt {
  int64_t n, ld;
  int parts, B;
  int adam;
  float lr;
  const float* part;
  float* p;
  float* mo;
  float* vo;
  float* loss_out;
  DevState* st;
};

__global__ void __launch_bounds__(128) k_trs_opt(const __grid_constant__ TrsOpt a) {
  pdl_wait();
  pdl_trigger();
  DevState* st = a.st;
  const int64_t t = st->step + 1;
  const bool aborted = st->train_abort != 0;
  const float bc1 = st->adam_bc[0], bc2 = st->adam_bc[1];
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e < a.n) {
    float mo = 0.0f, vo = 0.0f;
    if (a.adam) {
      mo = a.mo[e];
      vo = a.vo[e];
    }
    const float p = a.p[e];
    const float g = ordered_sum(a.part + e, a.parts, a.ld);
    if (!aborted) {
      if (a.adam) {
        const float me = 0.9f * mo + 0.1f * g;
        const float ve = 0.999f * vo + 0.001f * g * g;
        a.mo[e] = me;
        a.vo[e] = ve;
        const float mh = me / bc1, vh = ve / bc2;
        a.p[e] = p - a.lr * mh / (sqrtf(vh) + 1e-8f);
      } else {
        a.p[e] = p - a.lr * g;
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x < 32 && a.loss_out) {  // the loss, by one warp
    double s = 0.0;
    for (int q = threadIdx.x; q < a.parts; q += 32) {
      const float* v = a.part + q * a.ld + a.n;
      s += (double)__ldg(v) + (double)__ldg(v + 1);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    if (threadIdx.x == 0) *a.loss_out = aborted ? __int_as_float(0x7fc00000) : (float)(s / (double)a.B);
  }
  // the last block, once every block has read the counter and the flag
  if (last_block(&st->done[DONE_OPT]) && threadIdx.x == 0) {
    if (!aborted) advance_step(st, t);
    st->train_abort = 0;
  }
}

// Shared-memory floats besides the weights for tiles of `tr` rows.
int64_t trs_floats(const MlpDesc& m, int tr) {
  int64_t x = 0, hmax = 0;
  for (int l = 0; l < m.n_layers; ++l) {
    x += m.w[l];
    if (l > 0) hmax = std::max<int64_t>(hmax, m.w[l]);
  }
  return (x + 2 * hmax) * tr;
}

int64_t trs_resident_floats(const MlpDesc& m) {
  int64_t w = 0;
  for (int l = 0; l + 1 < m.n_layers; ++l) w += (int64_t)m.w[l] * (m.w[l + 1] | 1);
  return w;
}

// The tile height and weight staging for a batch of B rows: the smallest tile
// of 4, 8, 16 or 32 rows that leaves a tile per SM or fewer (small tiles:
// more CTAs, shorter chains in each), with the weights resident when they fit
// and else in chunks of 64 or 32 outputs.  False when not even that fits.
bool trs_plan(const MlpDesc& m, int B, int sms, int& tr, int& chunk, int64_t& floats) {
  int64_t in_max = 0;
  for (int l = 0; l + 1 < m.n_layers; ++l) in_max = std::max<int64_t>(in_max, m.w[l]);
  const int64_t cap = kSmemMax / 4;
  tr = 4;
  while (tr < 32 && ((int64_t)B + tr - 1) / tr > sms) tr *= 2;
  for (; tr >= 4; tr /= 2) {
    const int64_t f = trs_floats(m, tr);
    for (int c : {0, 64, 32}) {
      const int64_t w = c == 0 ? trs_resident_floats(m) : in_max * (c | 1);
      if (f + w <= cap) {
        chunk = c;
        floats = f + w;
        return true;
      }
    }
  }
  return false;
}

}  // namespace

// The fp32 step applies to fp32 predictors of at most kMaxParams parameters
// whose activations fit in shared memory with a weight chunk.
//
// Returns the largest batch it is taken for (0: none); the general path takes
// larger ones.  A CTA shares a weight among the rows of one tile only, so every
// further round of tiles costs as much as the first, in proportion to the
// parameters; the general path pays some seven launches a layer once and its
// products then fill the GPU.  The line: a 32-row tile per SM (fewer rows where
// a tile has fewer), 16 rows where the layers average over 15,000 parameters, and
// none for predictors that are small beside their layer count.  Device time of
// a step as graph replays on 152 SMs, general path / this one, at or below the
// line and above it:
//   no line   64-64, d 16       166 / 103 us at 12,288 rows, 310 / 218 at 32,768
//             80-80-80, d 64    338 / 284 at 16,384
//   32 rows   128, d 64         70 / 46 at 4864       76 / 80 at 6144
//             128-128-128, d 64 215 / 145 at 4864     240 / 307 at 6144
//             192-96, d 128     168 / 137 at 4864     187 / 290 at 6144
//   16 rows   256, d 128        70 / 45 at 2048       82 / 99 at 3072
//             512, d 64         64 / 61 at 2048       80 / 121 at 3072
//             256-256, d 64     166 / 121 at 2048     198 / 250 at 3072
//             1000, d 16 (tiles of 16)  56 / 43 at 1024  96 / 166 at 3072
//   no hidden layer, 32 rows    25 / 25 at 4864       29 / 33 at 6144
int plan_train_f32(const MlpDesc& m, int64_t n_params, int max_batch, int sms, int64_t* part_floats) {
  int tr, chunk;
  int64_t floats;
  if (m.bf16 || n_params > kMaxParams || !trs_plan(m, 1, sms, tr, chunk, floats)) return 0;
  trs_plan(m, INT_MAX, sms, tr, chunk, floats);  // tr: the rows of a tile of a large batch
  const int64_t layers = m.n_layers;
  const bool small = layers > 1 && n_params <= 1200 * layers * layers;
  const int line = small ? INT_MAX : std::min(tr, n_params <= 15000 * layers ? 32 : 16) * sms;
  const int64_t ctas = std::min<int64_t>(sms, (std::min(max_batch, line) + 3) / 4);
  *part_floats = ctas * (n_params + 2);
  return line;
}

cudaError_t run_train_f32(Ctx& c, int B, const int32_t* idx, int opt, float lr, float* loss_out, cudaStream_t s) {
  const MlpDesc& m = c.mlp;
  TrsArgs a{};
  a.m = m;
  a.B = B;
  int64_t floats = 0;
  if (!trs_plan(m, B, c.sms, a.tr, a.chunk, floats)) return cudaErrorInvalidValue;
  a.resident = a.chunk == 0;
  a.tiles = (B + a.tr - 1) / a.tr;
  int64_t w = 0;
  int x = 0, hmax = 0;
  for (int l = 0; l < m.n_layers; ++l) {
    a.woff_s[l] = (int)w;
    if (l + 1 < m.n_layers) w += (int64_t)m.w[l] * (m.w[l + 1] | 1);
    a.xoff_s[l] = x;
    x += m.w[l] * a.tr;
    if (l > 0) hmax = std::max(hmax, m.w[l]);
  }
  a.x_total = x;
  a.dz_rows = hmax;
  a.idx = idx;
  a.st = c.st;
  a.capacity = c.cfg.ring_capacity;
  a.replay_base = c.replay_base;
  a.ring_x = c.ring_x;
  a.ring_y = c.ring_y;
  a.mean = c.mean;
  a.stdv = c.stdv;
  a.p = c.master;
  a.part = c.trs_part;
  a.ld = c.n_params + 2;
  a.err = c.d_err;
  const int ctas = std::min(a.tiles, c.sms);
  cudaError_t e = traced(c, TR_TRAIN_STEP, 1, s, [&] {
    auto* launch = a.tr == 4 ? launch_smem<k_trs_grad<4>, TrsArgs&> : launch_smem<k_trs_grad<8>, TrsArgs&>;
    return launch(dim3(ctas), dim3(kT), (size_t)floats * sizeof(float), s, 1, a);
  });
  if (e != cudaSuccess) return e;
  TrsOpt o{};
  o.n = c.n_params;
  o.ld = a.ld;
  o.parts = ctas;
  o.B = B;
  o.adam = opt == LS_ADAM;
  o.lr = lr;
  o.part = c.trs_part;
  o.p = c.master;
  o.mo = c.adam_m;
  o.vo = c.adam_v;
  o.loss_out = loss_out ? loss_out : c.loss_tmp;
  o.st = c.st;
  return traced(c, TR_OPT, 1, s, [&] {
    return launch_chained(k_trs_opt, dim3((unsigned)((c.n_params + 127) / 128)), dim3(128), 0, s, 1, o);
  });
}

}  // namespace ls
