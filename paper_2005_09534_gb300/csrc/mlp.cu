// Learned predictor of spectral bounds and density of states: a small fully
// connected FP32 network, x -> tanh(W1 x' + b1) -> tanh(W2 . + b2) -> W3 . + b3,
// with x' = (x - x_mean) / x_std and outputs in standardized target units.
// Forward, backward (hand-derived; deterministic reductions, no atomics) and
// the Adam update are plain CUDA kernels.  The network is tiny (about 20k
// parameters), so launches and serial sums are what it costs: with up to
// kFusedMax inputs and hidden units a gradient takes three kernels (everything
// of a batch row; the weight gradients, split over the batch; their sum with
// the Adam update).  Wider networks keep one kernel per layer.
//
// Parameter layout (one contiguous float array):
//   W1 [H x d_in] row-major, b1 [H], W2 [H x H], b2 [H], W3 [d_out x H], b3 [d_out].
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "polfed_internal.h"

struct polfed_mlp {
  int d_in = 0, H = 0, d_out = 0, n_params = 0;
  float* params = nullptr;  // device
  float* m = nullptr;       // Adam first moment
  float* v = nullptr;       // Adam second moment
  float* grad = nullptr;    // device, n_params
  float* scale = nullptr;   // device: x_mean [d_in], 1/x_std [d_in], y_mean [d_out], y_std [d_out]
  float* io = nullptr;      // device: one input row and one output row (polfed_mlp_predict)
  float* work = nullptr;    // activations and deltas
  size_t work_floats = 0;
  std::vector<float> h_scale;  // host copy of scale
  int64_t t = 0;               // Adam step counter
  int device = 0;
};

namespace polfed {
namespace {

// xs[b][i] = (x[b][i] - mean[i]) * inv_std[i]
__global__ void k_mlp_standardize(const float* __restrict__ x, const float* __restrict__ mean,
                                  const float* __restrict__ inv_std, int B, int d, float* __restrict__ xs) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * d) return;
  const int i = e % d;
  xs[e] = (x[e] - mean[i]) * inv_std[i];
}

// out[b][j] = act(sum_i W[j][i] in[b][i] + bias[j]); act = tanh (hidden) or identity
__global__ void k_mlp_layer(const float* __restrict__ W, const float* __restrict__ bias, const float* __restrict__ in,
                            int B, int n_in, int n_out, int tanh_act, float* __restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * n_out) return;
  const int b = e / n_out, j = e % n_out;
  float s = bias[j];
  const float* w = W + (size_t)j * n_in;
  const float* x = in + (size_t)b * n_in;
  for (int i = 0; i < n_in; i++) s = fmaf(w[i], x[i], s);
  out[e] = tanh_act ? tanhf(s) : s;
}

// y[b][o] = ys[b][o] * y_std[o] + y_mean[o]
__global__ void k_mlp_unscale(const float* __restrict__ ys, const float* __restrict__ mean,
                              const float* __restrict__ sd, int B, int d, float* __restrict__ y) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * d) return;
  const int o = e % d;
  y[e] = fmaf(ys[e], sd[o], mean[o]);
}

// r = y - (t - y_mean) / y_std;  dy = r / B;  lp = 0.5 r^2 / B
__global__ void k_mlp_out_delta(const float* __restrict__ y, const float* __restrict__ t,
                                const float* __restrict__ mean, const float* __restrict__ sd, int B, int d_out,
                                float* __restrict__ dy, float* __restrict__ lp) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * d_out) return;
  const int o = e % d_out;
  const float r = y[e] - (t[e] - mean[o]) / sd[o];
  dy[e] = r / (float)B;
  lp[e] = 0.5f * r * r / (float)B;
}

// dW[j][i] = sum_b dz[b][j] in[b][i];  db[j] = sum_b dz[b][j]  (one thread per parameter)
__global__ void k_mlp_wgrad(const float* __restrict__ dz, const float* __restrict__ in, int B, int n_in, int n_out,
                            float* __restrict__ dW, float* __restrict__ db) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int nw = n_out * n_in;
  if (e < nw) {
    const int j = e / n_in, i = e % n_in;
    float s = 0.f;
    for (int b = 0; b < B; b++) s = fmaf(dz[(size_t)b * n_out + j], in[(size_t)b * n_in + i], s);
    dW[e] = s;
  } else if (e < nw + n_out) {
    const int j = e - nw;
    float s = 0.f;
    for (int b = 0; b < B; b++) s += dz[(size_t)b * n_out + j];
    db[j] = s;
  }
}

// dz_prev[b][i] = (sum_j W[j][i] dz[b][j]) * (1 - a_prev[b][i]^2)   (tanh' = 1 - tanh^2)
__global__ void k_mlp_back(const float* __restrict__ W, const float* __restrict__ dz, const float* __restrict__ a_prev,
                           int B, int n_in, int n_out, float* __restrict__ dz_prev) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * n_in) return;
  const int b = e / n_in, i = e % n_in;
  float s = 0.f;
  for (int j = 0; j < n_out; j++) s = fmaf(W[(size_t)j * n_in + i], dz[(size_t)b * n_out + j], s);
  const float a = a_prev[e];
  dz_prev[e] = s * (1.f - a * a);
}

// Adam with bias correction (Kingma & Ba, ICLR 2015, Algorithm 1).
__global__ void k_mlp_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ g, int n, float lr, float b1, float b2, float eps, float c1,
                           float c2) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const float gi = g[e];
  const float mi = b1 * m[e] + (1.f - b1) * gi;
  const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
  m[e] = mi;
  v[e] = vi;
  p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// *out = sum x[0..n), one block, fixed order
__global__ void k_mlp_sum(const float* __restrict__ x, int n, float* __restrict__ out) {
  __shared__ float sh[256];
  float s = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// uniform in [-a, a] from splitmix64, a = sqrt(6 / (fan_in + fan_out)) per weight matrix; biases 0
__global__ void k_mlp_init(float* p, int n, uint64_t seed, int d_in, int H, int d_out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(e + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  const float u = (float)((double)(z >> 40) * (1.0 / 16777216.0)) * 2.f - 1.f;
  const int n1 = H * d_in, n2 = n1 + H, n3 = n2 + H * H, n4 = n3 + H, n5 = n4 + d_out * H;
  float a = 0.f;
  if (e < n1)
    a = sqrtf(6.f / (d_in + H));
  else if (e >= n2 && e < n3)
    a = sqrtf(6.f / (2 * H));
  else if (e >= n4 && e < n5)
    a = sqrtf(6.f / (H + d_out));
  p[e] = a * u;
}

// ------------------------------------------------------- fused batch rows
constexpr int kFusedMax = 512;  // inputs and hidden units of the fused kernels
constexpr int kMaxOut = 64;
constexpr int kRowThreads = 256;

struct RowArgs {
  const float *W1, *b1, *W2, *b2, *W3, *b3, *xm, *xinv, *ym, *ysd;
  const float *x, *t;  // t == nullptr: forward only
  float *xs, *a1, *a2, *dy, *dz2, *dz1, *lossp, *y;
  int B, d_in, H, d_out;
};

// out[j * TB + r] = sum_i W[j * n_in + i] in[i * TB + r]: a warp takes 16 / TB
// rows of W at a time (lanes along i, coalesced) for all TB batch rows and
// reduces its 16 sums by exchanging halves.  fin(j, r, sum) consumes them.
template <int TB, class F>
__device__ __forceinline__ void rows_dot(const float* __restrict__ W, const float* in, int n_in, int n_out, F fin) {
  constexpr int JT = 16 / TB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j0 = warp * JT; j0 < n_out; j0 += JT * (kRowThreads / 32)) {
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; q++) v[q] = 0.f;
#pragma unroll 4
    for (int i = lane; i < n_in; i += 32) {
      float xr[TB];
#pragma unroll
      for (int r = 0; r < TB; r += 4) *reinterpret_cast<float4*>(xr + r) = *reinterpret_cast<const float4*>(in + i * TB + r);
#pragma unroll
      for (int j = 0; j < JT; j++) {
        const float w = j0 + j < n_out ? __ldg(W + (size_t)(j0 + j) * n_in + i) : 0.f;
#pragma unroll
        for (int r = 0; r < TB; r++) v[j * TB + r] = fmaf(w, xr[r], v[j * TB + r]);
      }
    }
#pragma unroll
    for (int m = 16, c = 8; m >= 2; m >>= 1, c >>= 1) {
      const bool up = lane & m;
#pragma unroll
      for (int q = 0; q < 8; q++)
        if (q < c) {
          const float send = up ? v[q] : v[q + c], keep = up ? v[q + c] : v[q];
          v[q] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
    }
    const float s = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
    const int idx = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
    const int j = j0 + idx / TB;
    if (!(lane & 1) && j < n_out) fin(j, idx % TB, s);
  }
}

// Everything of TB batch rows: standardization, the three layers, the output
// delta and loss, and the deltas of both hidden layers.  Bound by latency (a
// CTA's chain of dot products; the weights come from L2, read once per CTA).
// 23 inputs, 2 x 128 hidden units, batch 256: a whole gradient call 194 -> 45 us,
// this kernel 12, the weight gradients 4.5 (101 before, serial over the batch),
// their sum 2 us.
template <int TB>
__global__ void __launch_bounds__(kRowThreads) k_mlp_rows(const RowArgs A) {
  extern __shared__ __align__(16) float sh[];
  const int H = A.H, b0 = blockIdx.x * TB, tid = threadIdx.x;
  float* sx = sh;                    // [d_in][TB]
  float* s1 = sx + A.d_in * TB;      // [H][TB] a1
  float* s2 = s1 + H * TB;           // a2
  float* sd = s2 + H * TB;           // dz2
  float* so = sd + H * TB;           // [d_out][TB] dy
  float* sl = so + A.d_out * TB;     // loss terms
  for (int e = tid; e < A.d_in * TB; e += kRowThreads) {
    const int r = e / A.d_in, i = e - r * A.d_in;
    float v = 0.f;
    if (b0 + r < A.B) {
      const size_t g = (size_t)(b0 + r) * A.d_in + i;
      v = (A.x[g] - A.xm[i]) * A.xinv[i];
      if (A.t) A.xs[g] = v;
    }
    sx[i * TB + r] = v;
  }
  __syncthreads();
  rows_dot<TB>(A.W1, sx, A.d_in, H, [&](int j, int r, float s) {
    s = tanhf(s + A.b1[j]);
    s1[j * TB + r] = s;
    if (A.t && b0 + r < A.B) A.a1[(size_t)(b0 + r) * H + j] = s;
  });
  __syncthreads();
  rows_dot<TB>(A.W2, s1, H, H, [&](int j, int r, float s) {
    s = tanhf(s + A.b2[j]);
    s2[j * TB + r] = s;
    if (A.t && b0 + r < A.B) A.a2[(size_t)(b0 + r) * H + j] = s;
  });
  __syncthreads();
  rows_dot<TB>(A.W3, s2, H, A.d_out, [&](int o, int r, float s) {
    s += A.b3[o];
    const bool in = b0 + r < A.B;
    const size_t g = (size_t)(b0 + r) * A.d_out + o;
    if (!A.t) {
      if (in) A.y[g] = fmaf(s, A.ysd[o], A.ym[o]);
      return;
    }
    const float e = in ? s - (A.t[g] - A.ym[o]) / A.ysd[o] : 0.f;
    const float dy = e / (float)A.B;
    so[o * TB + r] = dy;
    sl[o * TB + r] = 0.5f * e * e / (float)A.B;
    if (in) A.dy[g] = dy;
  });
  if (!A.t) return;
  __syncthreads();
  if (tid == 0) {
    float l = 0.f;
    for (int q = 0; q < A.d_out * TB; q++) l += sl[q];
    A.lossp[blockIdx.x] = l;
  }
  // dz2 = (W3^T dy) (1 - a2^2)
  for (int i = tid; i < H; i += kRowThreads) {
    float z[TB];
#pragma unroll
    for (int r = 0; r < TB; r++) z[r] = 0.f;
    for (int o = 0; o < A.d_out; o++) {
      const float w = __ldg(A.W3 + (size_t)o * H + i);
#pragma unroll
      for (int r = 0; r < TB; r++) z[r] = fmaf(w, so[o * TB + r], z[r]);
    }
#pragma unroll
    for (int r = 0; r < TB; r++) {
      const float a = s2[i * TB + r];
      z[r] *= 1.f - a * a;
      sd[i * TB + r] = z[r];
      if (b0 + r < A.B) A.dz2[(size_t)(b0 + r) * H + i] = z[r];
    }
  }
  __syncthreads();
  // dz1 = (W2^T dz2) (1 - a1^2): one thread per (hidden unit, share of the sum); shares meet in s2
  const int Hr = (H + 31) & ~31, ng = Hr >= kRowThreads ? 1 : kRowThreads / Hr;
  const int g = Hr >= kRowThreads ? 0 : tid / Hr;
  for (int i = Hr >= kRowThreads ? tid : tid - g * Hr; i < H; i += kRowThreads) {
    if (g >= ng) break;
    float z[TB];
#pragma unroll
    for (int r = 0; r < TB; r++) z[r] = 0.f;
    const int jn = (H + ng - 1) / ng, j1 = min(H, (g + 1) * jn);
#pragma unroll 8
    for (int j = g * jn; j < j1; j++) {
      const float w = __ldg(A.W2 + (size_t)j * H + i);
#pragma unroll
      for (int r = 0; r < TB; r += 4) {
        const float4 d = *reinterpret_cast<const float4*>(sd + j * TB + r);
        z[r] = fmaf(w, d.x, z[r]);
        z[r + 1] = fmaf(w, d.y, z[r + 1]);
        z[r + 2] = fmaf(w, d.z, z[r + 2]);
        z[r + 3] = fmaf(w, d.w, z[r + 3]);
      }
    }
#pragma unroll
    for (int r = 0; r < TB; r++) (g == 0 ? s2 : sl + A.d_out * TB + (size_t)(g - 1) * H * TB)[i * TB + r] = z[r];
  }
  __syncthreads();
  for (int e = tid; e < H * TB; e += kRowThreads) {
    const int r = e / H, i = e - r * H;
    float z = s2[i * TB + r];
    for (int q = 1; q < ng; q++) z += sl[A.d_out * TB + (size_t)(q - 1) * H * TB + i * TB + r];
    const float a = s1[i * TB + r];
    if (b0 + r < A.B) A.dz1[(size_t)(b0 + r) * H + i] = z * (1.f - a * a);
  }
}

size_t rows_smem(int TB, int d_in, int H, int d_out) {
  const int Hr = (H + 31) & ~31, ng = Hr >= kRowThreads ? 1 : kRowThreads / Hr;
  return (size_t)TB * (d_in + 3 * H + 2 * d_out + (ng - 1) * H) * sizeof(float);
}

// One of the three weight matrices: dW[j][i] = sum_b dz[b][j] in[b][i], db[j] = sum_b dz[b][j].
struct WMat {
  const float *dz, *in;
  int n_in, n_out, off_w, off_b, tile0;  // offsets in the parameters, first tile
};
struct WArgs {
  WMat m[3];
  int B, rows;  // rows of the batch per split
  int64_t n_params;
  float* part;  // [splits][n_params]
};

// 32 x 32 tiles of the weight gradients over one share of the batch.
__global__ void __launch_bounds__(256) k_mlp_wgrad_tiles(const WArgs A) {
  __shared__ __align__(16) float sz[32][32], si[32][32];
  int q = 2;
  while (q > 0 && (int)blockIdx.x < A.m[q].tile0) q--;
  const WMat m = A.m[q];
  const int tcols = (m.n_in + 31) / 32, tl = blockIdx.x - m.tile0;
  const int j0 = (tl / tcols) * 32, i0 = (tl % tcols) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int b0 = blockIdx.y * A.rows, b1 = min(A.B, b0 + A.rows);
  float acc[4] = {0.f, 0.f, 0.f, 0.f}, ab[4] = {0.f, 0.f, 0.f, 0.f};
  for (int b = b0; b < b1; b += 32) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int r = ty + 8 * u;
      const bool in = b + r < b1;
      sz[r][tx] = in && j0 + tx < m.n_out ? m.dz[(size_t)(b + r) * m.n_out + j0 + tx] : 0.f;
      si[r][tx] = in && i0 + tx < m.n_in ? m.in[(size_t)(b + r) * m.n_in + i0 + tx] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int r = 0; r < 32; r++) {
      const float4 z = *reinterpret_cast<const float4*>(&sz[r][ty * 4]);
      const float x = si[r][tx];
      acc[0] = fmaf(z.x, x, acc[0]);
      acc[1] = fmaf(z.y, x, acc[1]);
      acc[2] = fmaf(z.z, x, acc[2]);
      acc[3] = fmaf(z.w, x, acc[3]);
      ab[0] += z.x;
      ab[1] += z.y;
      ab[2] += z.z;
      ab[3] += z.w;
    }
  }
  float* P = A.part + blockIdx.y * A.n_params;
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const int j = j0 + ty * 4 + u, i = i0 + tx;
    if (j < m.n_out && i < m.n_in) P[m.off_w + (size_t)j * m.n_in + i] = acc[u];
    if (j < m.n_out && i == 0) P[m.off_b + j] = ab[u];
  }
}

// Sum of the shares in order, the Adam update if lr > 0, and (last CTA) the loss.
__global__ void k_mlp_combine(const float* __restrict__ part, int splits, int n, float* __restrict__ grad,
                              float* __restrict__ out, const float* __restrict__ lossp, int n_loss,
                              float* __restrict__ loss, float* __restrict__ p, float* __restrict__ m,
                              float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  __shared__ float sh[256];
  if (blockIdx.x == gridDim.x - 1) {
    float s = 0.f;
    for (int i = threadIdx.x; i < n_loss; i += 256) s += lossp[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
      if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = sh[0];
    return;
  }
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= n) return;
  float s = 0.f;
  for (int q = 0; q < splits; q++) s += part[(size_t)q * n + e];
  grad[e] = s;
  if (out) out[e] = s;
  if (lr > 0.f) {
    const float mi = b1 * m[e] + (1.f - b1) * s;
    const float vi = b2 * v[e] + (1.f - b2) * s * s;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

unsigned nblk(int n) { return (unsigned)((n + 255) / 256); }

struct Views {
  const float *W1, *b1, *W2, *b2, *W3, *b3;
  float *gW1, *gb1, *gW2, *gb2, *gW3, *gb3;
  const float *xm, *xinv, *ym, *ysd;
};

Views views(const polfed_mlp* n) {
  Views v;
  v.W1 = n->params;
  v.b1 = v.W1 + (size_t)n->H * n->d_in;
  v.W2 = v.b1 + n->H;
  v.b2 = v.W2 + (size_t)n->H * n->H;
  v.W3 = v.b2 + n->H;
  v.b3 = v.W3 + (size_t)n->d_out * n->H;
  v.gW1 = n->grad;
  v.gb1 = v.gW1 + (size_t)n->H * n->d_in;
  v.gW2 = v.gb1 + n->H;
  v.gb2 = v.gW2 + (size_t)n->H * n->H;
  v.gW3 = v.gb2 + n->H;
  v.gb3 = v.gW3 + (size_t)n->d_out * n->H;
  v.xm = n->scale;
  v.xinv = v.xm + n->d_in;
  v.ym = v.xinv + n->d_in;
  v.ysd = v.ym + n->d_out;
  return v;
}

// Work buffer: xs [B d_in] | a1 [B H] | a2 [B H] | y [B d_out] | dy [B d_out] | dz2 [B H] | dz1 [B H] | loss [1]
// | loss terms and gradient shares of the fused kernels
struct Work {
  float *xs, *a1, *a2, *y, *dy, *dz2, *dz1, *loss, *lossp, *part;
  int tb, splits;
};

bool fused(const polfed_mlp* n) { return n->d_in <= kFusedMax && n->H <= kFusedMax; }

int ensure_work(polfed_mlp* n, int B, Work* w) {
  // 4 batch rows to a CTA, 8 for large batches (W2 is read once per CTA); shares of at least 64 rows
  w->tb = B <= 1024 ? 4 : 8;
  w->splits = std::max(1, std::min(16, (B + 63) / 64));
  const size_t rows = (size_t)B * (n->d_in + 4 * n->H + 2 * n->d_out) + 64;
  const size_t nl = fused(n) ? ((size_t)(B + w->tb - 1) / w->tb + 63) & ~(size_t)63 : 0;
  const size_t need = rows + (fused(n) ? nl + (size_t)w->splits * n->n_params : 0);
  if (!n->work || n->work_floats < need) {
    if (n->work) cudaFree(n->work);
    n->work = nullptr;
    n->work_floats = 0;
    if (device_malloc((void**)&n->work, need * sizeof(float)) != cudaSuccess) {
      cudaGetLastError();
      return fail(POLFED_ENOMEM, "MLP work allocation failed");
    }
    n->work_floats = need;
  }
  w->xs = n->work;
  w->a1 = w->xs + (size_t)B * n->d_in;
  w->a2 = w->a1 + (size_t)B * n->H;
  w->y = w->a2 + (size_t)B * n->H;
  w->dy = w->y + (size_t)B * n->d_out;
  w->dz2 = w->dy + (size_t)B * n->d_out;
  w->dz1 = w->dz2 + (size_t)B * n->H;
  w->loss = w->dz1 + (size_t)B * n->H;
  w->lossp = n->work + rows;
  w->part = w->lossp + nl;
  return POLFED_OK;
}

// The fused row kernel: forward into y (t == nullptr), or forward and deltas.
int run_rows(polfed_mlp* n, const float* x, const float* t, int B, float* y, const Work& w, cudaStream_t s) {
  const Views v = views(n);
  const RowArgs A{v.W1, v.b1, v.W2, v.b2, v.W3, v.b3, v.xm, v.xinv, v.ym, v.ysd, x, t, w.xs, w.a1, w.a2, w.dy,
                  w.dz2, w.dz1, w.lossp, y, B, n->d_in, n->H, n->d_out};
  const size_t smem = rows_smem(w.tb, n->d_in, n->H, n->d_out);
  const int grid = (B + w.tb - 1) / w.tb;
  if (w.tb == 4)
    k_mlp_rows<4><<<grid, kRowThreads, smem, s>>>(A);
  else
    k_mlp_rows<8><<<grid, kRowThreads, smem, s>>>(A);
  PF_CUDA(cudaGetLastError());
  count_launch();
  return POLFED_OK;
}

// standardized forward pass into the work buffer
int forward(polfed_mlp* n, const float* x, int B, cudaStream_t s, Work* w) {
  PF_CHECK(ensure_work(n, B, w));
  const Views v = views(n);
  k_mlp_standardize<<<nblk(B * n->d_in), 256, 0, s>>>(x, v.xm, v.xinv, B, n->d_in, w->xs);
  k_mlp_layer<<<nblk(B * n->H), 256, 0, s>>>(v.W1, v.b1, w->xs, B, n->d_in, n->H, 1, w->a1);
  k_mlp_layer<<<nblk(B * n->H), 256, 0, s>>>(v.W2, v.b2, w->a1, B, n->H, n->H, 1, w->a2);
  k_mlp_layer<<<nblk(B * n->d_out), 256, 0, s>>>(v.W3, v.b3, w->a2, B, n->H, n->d_out, 0, w->y);
  PF_CUDA(cudaGetLastError());
  count_launch(4);
  return POLFED_OK;
}

// The shared memory that the largest fused network takes, for every network: the limit belongs to the kernel,
// and a call that set its own could lower it under another thread's launch.
int allow_rows_smem() {
  const int big = (int)rows_smem(8, kFusedMax, kFusedMax, kMaxOut);
  PF_CUDA(cudaFuncSetAttribute(k_mlp_rows<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  PF_CUDA(cudaFuncSetAttribute(k_mlp_rows<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  return POLFED_OK;
}

struct AdamStep {
  float lr = 0.f, b1 = 0.9f, b2 = 0.999f, eps = 1e-8f, c1 = 1.f, c2 = 1.f;  // lr == 0: gradient only
};

// gradient of 0.5/B sum |y - t'|^2 into n->grad (and d_grad), with the Adam
// update of the parameters if ad.lr > 0; wide networks: the loss partials go to
// dz1 before it is overwritten (d_out <= H)
int backward(polfed_mlp* n, const float* x, const float* t, int B, cudaStream_t s, float* d_grad, const AdamStep& ad,
             float* loss_host) {
  Work w;
  const Views v = views(n);
  if (fused(n)) {
    PF_CHECK(ensure_work(n, B, &w));
    PF_CHECK(run_rows(n, x, t, B, nullptr, w, s));
    WArgs A{};
    const int H = n->H;
    auto tiles = [](int r, int c) { return ((r + 31) / 32) * ((c + 31) / 32); };
    A.m[0] = WMat{w.dz2, w.a1, H, H, (int)(v.W2 - n->params), (int)(v.b2 - n->params), 0};
    A.m[1] = WMat{w.dz1, w.xs, n->d_in, H, (int)(v.W1 - n->params), (int)(v.b1 - n->params), tiles(H, H)};
    A.m[2] = WMat{w.dy, w.a2, H, n->d_out, (int)(v.W3 - n->params), (int)(v.b3 - n->params),
                  A.m[1].tile0 + tiles(H, n->d_in)};
    A.B = B;
    A.rows = ((B + w.splits - 1) / w.splits + 31) & ~31;
    A.n_params = n->n_params;
    A.part = w.part;
    const int splits = (B + A.rows - 1) / A.rows;
    k_mlp_wgrad_tiles<<<dim3(A.m[2].tile0 + tiles(n->d_out, H), splits), 256, 0, s>>>(A);
    k_mlp_combine<<<nblk(n->n_params) + 1, 256, 0, s>>>(w.part, splits, n->n_params, n->grad, d_grad, w.lossp,
                                                         (B + w.tb - 1) / w.tb, w.loss, n->params, n->m, n->v, ad.lr,
                                                         ad.b1, ad.b2, ad.eps, ad.c1, ad.c2);
    PF_CUDA(cudaGetLastError());
    count_launch(2);
    if (loss_host) PF_CUDA(cudaMemcpyAsync(loss_host, w.loss, sizeof(float), cudaMemcpyDeviceToHost, s));
    return POLFED_OK;
  }
  PF_CHECK(forward(n, x, B, s, &w));
  k_mlp_out_delta<<<nblk(B * n->d_out), 256, 0, s>>>(w.y, t, v.ym, v.ysd, B, n->d_out, w.dy, w.dz1);
  k_mlp_sum<<<1, 256, 0, s>>>(w.dz1, B * n->d_out, w.loss);
  k_mlp_wgrad<<<nblk(n->d_out * n->H + n->d_out), 256, 0, s>>>(w.dy, w.a2, B, n->H, n->d_out, v.gW3, v.gb3);
  k_mlp_back<<<nblk(B * n->H), 256, 0, s>>>(v.W3, w.dy, w.a2, B, n->H, n->d_out, w.dz2);
  k_mlp_wgrad<<<nblk(n->H * n->H + n->H), 256, 0, s>>>(w.dz2, w.a1, B, n->H, n->H, v.gW2, v.gb2);
  k_mlp_back<<<nblk(B * n->H), 256, 0, s>>>(v.W2, w.dz2, w.a1, B, n->H, n->H, w.dz1);
  k_mlp_wgrad<<<nblk(n->H * n->d_in + n->H), 256, 0, s>>>(w.dz1, w.xs, B, n->d_in, n->H, v.gW1, v.gb1);
  PF_CUDA(cudaGetLastError());
  count_launch(7);
  if (ad.lr > 0.f) {
    k_mlp_adam<<<nblk(n->n_params), 256, 0, s>>>(n->params, n->m, n->v, n->grad, n->n_params, ad.lr, ad.b1, ad.b2,
                                                  ad.eps, ad.c1, ad.c2);
    PF_CUDA(cudaGetLastError());
    count_launch();
  }
  if (d_grad)
    PF_CUDA(cudaMemcpyAsync(d_grad, n->grad, (size_t)n->n_params * sizeof(float), cudaMemcpyDeviceToDevice, s));
  if (loss_host) PF_CUDA(cudaMemcpyAsync(loss_host, w.loss, sizeof(float), cudaMemcpyDeviceToHost, s));
  return POLFED_OK;
}

struct DeviceGuard {
  int prev = 0;
  explicit DeviceGuard(int d) {
    cudaGetDevice(&prev);
    cudaSetDevice(d);
  }
  ~DeviceGuard() { cudaSetDevice(prev); }
};

}  // namespace
}  // namespace polfed

using namespace polfed;

extern "C" {

void polfed_mlp_destroy(polfed_mlp* n) {
  if (!n) return;
  DeviceGuard g(n->device);
  cudaFree(n->params);
  cudaFree(n->m);
  cudaFree(n->v);
  cudaFree(n->grad);
  cudaFree(n->scale);
  cudaFree(n->io);
  cudaFree(n->work);
  delete n;
}

int polfed_mlp_create(int32_t d_in, int32_t hidden, int32_t d_out, uint64_t seed, polfed_mlp** out) {
  if (!out) return fail(POLFED_EINVAL, "out is NULL");
  if (d_in < 1 || d_in > 1024 || d_out < 1 || d_out > kMaxOut || hidden < d_out || hidden > 4096)
    return fail(POLFED_EINVAL, "need 1 <= d_in <= 1024, 1 <= d_out <= 64, d_out <= hidden <= 4096");
  polfed_mlp* n = new polfed_mlp();
  n->d_in = d_in;
  n->H = hidden;
  n->d_out = d_out;
  n->n_params = hidden * d_in + hidden + hidden * hidden + hidden + d_out * hidden + d_out;
  cudaGetDevice(&n->device);
  const size_t bytes = (size_t)n->n_params * sizeof(float);
  const size_t sbytes = (size_t)(2 * d_in + 2 * d_out) * sizeof(float);
  if (device_malloc((void**)&n->params, bytes) != cudaSuccess || device_malloc((void**)&n->m, bytes) != cudaSuccess ||
      device_malloc((void**)&n->v, bytes) != cudaSuccess || device_malloc((void**)&n->grad, bytes) != cudaSuccess ||
      device_malloc((void**)&n->scale, sbytes) != cudaSuccess ||
      device_malloc((void**)&n->io, (size_t)(d_in + d_out) * sizeof(float)) != cudaSuccess) {
    cudaGetLastError();
    polfed_mlp_destroy(n);
    return fail(POLFED_ENOMEM, "MLP allocation failed");
  }
  if (const int e = allow_rows_smem()) {
    polfed_mlp_destroy(n);
    return e;
  }
  n->h_scale.assign(2 * d_in + 2 * d_out, 0.f);
  for (int i = 0; i < d_in; i++) n->h_scale[d_in + i] = 1.f;
  for (int o = 0; o < d_out; o++) n->h_scale[2 * d_in + d_out + o] = 1.f;
  int rc = POLFED_OK;
  if (cudaMemset(n->m, 0, bytes) != cudaSuccess || cudaMemset(n->v, 0, bytes) != cudaSuccess ||
      cudaMemset(n->grad, 0, bytes) != cudaSuccess ||
      cudaMemcpy(n->scale, n->h_scale.data(), sbytes, cudaMemcpyHostToDevice) != cudaSuccess)
    rc = POLFED_ECUDA;
  if (rc == POLFED_OK) {
    k_mlp_init<<<nblk(n->n_params), 256>>>(n->params, n->n_params, seed, d_in, hidden, d_out);
    count_launch();
    if (cudaDeviceSynchronize() != cudaSuccess) rc = POLFED_ECUDA;
  }
  if (rc != POLFED_OK) {
    cudaGetLastError();
    polfed_mlp_destroy(n);
    return fail(rc, "MLP initialization failed");
  }
  *out = n;
  return POLFED_OK;
}

int32_t polfed_mlp_num_params(const polfed_mlp* n) { return n ? n->n_params : 0; }

int polfed_mlp_set_params(polfed_mlp* n, const float* host) {
  if (!n || !host) return fail(POLFED_EINVAL, "NULL argument");
  DeviceGuard g(n->device);
  const size_t bytes = (size_t)n->n_params * sizeof(float);
  PF_CUDA(cudaMemcpy(n->params, host, bytes, cudaMemcpyHostToDevice));
  PF_CUDA(cudaMemset(n->m, 0, bytes));
  PF_CUDA(cudaMemset(n->v, 0, bytes));
  n->t = 0;
  return POLFED_OK;
}

int polfed_mlp_get_params(const polfed_mlp* n, float* host) {
  if (!n || !host) return fail(POLFED_EINVAL, "NULL argument");
  DeviceGuard g(n->device);
  PF_CUDA(cudaMemcpy(host, n->params, (size_t)n->n_params * sizeof(float), cudaMemcpyDeviceToHost));
  return POLFED_OK;
}

int polfed_mlp_set_scaling(polfed_mlp* n, const float* x_mean, const float* x_std, const float* y_mean,
                           const float* y_std) {
  if (!n || !x_mean || !x_std || !y_mean || !y_std) return fail(POLFED_EINVAL, "NULL argument");
  for (int i = 0; i < n->d_in; i++)
    if (!(x_std[i] > 0.f) || !std::isfinite(x_std[i]) || !std::isfinite(x_mean[i]))
      return fail(POLFED_EINVAL, "x_std must be finite and > 0");
  for (int o = 0; o < n->d_out; o++)
    if (!(y_std[o] > 0.f) || !std::isfinite(y_std[o]) || !std::isfinite(y_mean[o]))
      return fail(POLFED_EINVAL, "y_std must be finite and > 0");
  for (int i = 0; i < n->d_in; i++) {
    n->h_scale[i] = x_mean[i];
    n->h_scale[n->d_in + i] = 1.f / x_std[i];
  }
  for (int o = 0; o < n->d_out; o++) {
    n->h_scale[2 * n->d_in + o] = y_mean[o];
    n->h_scale[2 * n->d_in + n->d_out + o] = y_std[o];
  }
  DeviceGuard g(n->device);
  PF_CUDA(cudaMemcpy(n->scale, n->h_scale.data(), n->h_scale.size() * sizeof(float), cudaMemcpyHostToDevice));
  return POLFED_OK;
}

int polfed_mlp_forward(polfed_mlp* n, const float* d_x, int32_t B, float* d_y, polfed_stream_t stream) {
  if (!n || !d_x || !d_y || B < 1 || B > (1 << 20)) return fail(POLFED_EINVAL, "bad MLP forward arguments");
  DeviceGuard g(n->device);
  cudaStream_t s = (cudaStream_t)stream;
  Work w;
  if (fused(n)) {
    PF_CHECK(ensure_work(n, B, &w));
    // the CTAs of the row kernel read x and write y in any order: outputs over the inputs go through a copy
    const size_t xb = (size_t)B * n->d_in * sizeof(float), yb = (size_t)B * n->d_out * sizeof(float);
    const bool over = (uintptr_t)d_x < (uintptr_t)d_y + yb && (uintptr_t)d_y < (uintptr_t)d_x + xb;
    PF_CHECK(run_rows(n, d_x, nullptr, B, over ? w.y : d_y, w, s));
    if (over) PF_CUDA(cudaMemcpyAsync(d_y, w.y, yb, cudaMemcpyDeviceToDevice, s));
    PF_CUDA(cudaStreamSynchronize(s));
    return POLFED_OK;
  }
  PF_CHECK(forward(n, d_x, B, s, &w));
  const Views v = views(n);
  k_mlp_unscale<<<nblk(B * n->d_out), 256, 0, s>>>(w.y, v.ym, v.ysd, B, n->d_out, d_y);
  PF_CUDA(cudaGetLastError());
  count_launch();
  PF_CUDA(cudaStreamSynchronize(s));
  return POLFED_OK;
}

int polfed_mlp_grad(polfed_mlp* n, const float* d_x, const float* d_t, int32_t B, float* d_grad, float* loss,
                    polfed_stream_t stream) {
  if (!n || !d_x || !d_t || B < 1 || B > (1 << 20)) return fail(POLFED_EINVAL, "bad MLP gradient arguments");
  DeviceGuard g(n->device);
  cudaStream_t s = (cudaStream_t)stream;
  PF_CHECK(backward(n, d_x, d_t, B, s, d_grad, AdamStep(), loss));
  PF_CUDA(cudaStreamSynchronize(s));
  return POLFED_OK;
}

int polfed_mlp_train_step(polfed_mlp* n, const float* d_x, const float* d_t, int32_t B, float lr, float* loss,
                          polfed_stream_t stream) {
  if (!n || !d_x || !d_t || B < 1 || B > (1 << 20) || !(lr > 0.f))
    return fail(POLFED_EINVAL, "bad MLP training arguments");
  DeviceGuard g(n->device);
  cudaStream_t s = (cudaStream_t)stream;
  n->t++;
  AdamStep ad;
  ad.lr = lr;
  ad.c1 = 1.f - std::pow(ad.b1, (float)n->t);
  ad.c2 = 1.f - std::pow(ad.b2, (float)n->t);
  const int rc = backward(n, d_x, d_t, B, s, nullptr, ad, loss);
  if (rc != POLFED_OK) {
    n->t--;
    return rc;
  }
  PF_CUDA(cudaStreamSynchronize(s));
  return POLFED_OK;
}

int polfed_mlp_features(const polfed_model* model, double W, float* x) {
  if (!model || !model->h || !x) return fail(POLFED_EINVAL, "NULL argument");
  if (model->L < 2 || model->L > 32) return fail(POLFED_EINVAL, "L must be in 2..32");
  for (int i = 0; i < model->L; i++) x[i] = (float)model->h[i];
  x[model->L] = (float)W;
  return POLFED_OK;
}

int polfed_mlp_targets(int32_t L, const double* labels, float* y) {
  if (!labels || !y) return fail(POLFED_EINVAL, "NULL argument");
  if (L < 2 || L > 32) return fail(POLFED_EINVAL, "L must be in 2..32");
  if (!(labels[2] > 0.0) || !std::isfinite(labels[2])) return fail(POLFED_EINVAL, "rho_eps must be > 0");
  y[0] = (float)(labels[0] / L);
  y[1] = (float)(labels[1] / L);
  y[2] = (float)std::log(labels[2]);
  return POLFED_OK;
}

int polfed_mlp_predict(polfed_mlp* n, const polfed_model* model, double W, double* out) {
  if (!n || !model || !out) return fail(POLFED_EINVAL, "NULL argument");
  if (n->d_in != model->L + 1 || n->d_out != 3) return fail(POLFED_EINVAL, "predictor needs d_in = L + 1, d_out = 3");
  std::vector<float> x(n->d_in);
  PF_CHECK(polfed_mlp_features(model, W, x.data()));
  DeviceGuard g(n->device);
  PF_CUDA(cudaMemcpy(n->io, x.data(), n->d_in * sizeof(float), cudaMemcpyHostToDevice));
  PF_CHECK(polfed_mlp_forward(n, n->io, 1, n->io + n->d_in, nullptr));
  float y[3];
  PF_CUDA(cudaMemcpy(y, n->io + n->d_in, sizeof(y), cudaMemcpyDeviceToHost));
  out[0] = (double)y[0] * model->L;
  out[1] = (double)y[1] * model->L;
  out[2] = std::exp((double)y[2]);
  return POLFED_OK;
}

}  // extern "C"
