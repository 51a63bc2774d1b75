// Observables of the eigenpairs (section "Entanglement entropy and level
// statistics"): the mean gap ratio of a sorted spectrum and the half-chain
// entanglement entropy of sector eigenvectors.
//
// Gap ratio: r_i = min(g_i, g_{i+1}) / max(g_i, g_{i+1}), g_i = E_{i+1} - E_i,
// averaged over i.
//
// Entanglement entropy of the bipartition A = sites [x, x + L/2) (mod L), B =
// the rest: S = -sum alpha^2 ln alpha^2 over the Schmidt coefficients alpha.
// In the S^z = 0 sector the amplitude matrix psi[a][b] (a: configuration of A,
// b: configuration of B) is block diagonal in the number k of up spins in A:
// block k is C(L/2, k) x C(L/2, L/2 - k), rows and columns ranked within their
// popcount class by the combinatorial number system.  The alpha^2 of block k
// are the eigenvalues of its Gram matrix G_k = M_k M_k^T, a small symmetric
// projected eigenproblem (the reduced density matrix rho_A restricted to k up
// spins) solved with cuSOLVER's batched symmetric eigensolver.  The blocks of
// one vector hold sum_k C(L/2, k)^2 = C(L, L/2) = N entries, so a vector's
// blocks and Gram matrices each take N doubles.
// A and its complement have the same entropy, so cut x + L/2 repeats cut x:
// L/2 cuts are computed and the average over the L positions x is their mean.
#include <cusolverDn.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "polfed_internal.h"
#include "rows.h"

namespace polfed {

namespace {

// C(n, k) for n, k <= 16 from a per-CTA Pascal triangle
struct SmallBinom {
  uint32_t c[17][17];
};

__device__ void fill_binom(SmallBinom& b) {
  if (threadIdx.x == 0) {
    for (int n = 0; n <= 16; n++)
      for (int k = 0; k <= 16; k++) b.c[n][k] = 0;
    for (int n = 0; n <= 16; n++) {
      b.c[n][0] = 1;
      for (int k = 1; k <= n; k++) b.c[n][k] = b.c[n - 1][k - 1] + (k <= n - 1 ? b.c[n - 1][k] : 0);
    }
  }
  __syncthreads();
}

// colex rank of an h-bit string among those of equal popcount: sum_j C(p_j, j + 1)
__device__ __forceinline__ uint32_t colex_rank(uint32_t a, const SmallBinom& b) {
  uint32_t r = 0;
  int j = 0;
  while (a) {
    const int p = __ffs(a) - 1;
    r += b.c[p][++j];
    a &= a - 1;
  }
  return r;
}

// Scatter the amplitudes of nv vectors into the Schmidt blocks of cut x:
// M[v * N + boff[k] + ra * C_k + rb] = psi_v[r] with s = states[r] rotated so
// that site x is bit 0, a = its low h bits (subsystem A), b = its high h bits.
// blockIdx.y adds to the cut; vector v of cut x goes to M + v * vstride + (x - x0) * dim.
__global__ void k_schmidt_scatter(const uint32_t* __restrict__ states, int64_t dim, int L, int x0,
                                  const double* __restrict__ vecs, int64_t ld, int nv, const int64_t* boff,
                                  double* __restrict__ M, int64_t vstride) {
  __shared__ SmallBinom sb;
  fill_binom(sb);
  const int h = L / 2, x = x0 + blockIdx.y;
  M += (int64_t)blockIdx.y * dim;
  const uint32_t full = (L == 32) ? 0xFFFFFFFFu : ((1u << L) - 1u);
  const uint32_t hmask = (1u << h) - 1u;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < dim; r += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t s = states[r];
    const uint32_t rot = x == 0 ? s : (((s >> x) | (s << (L - x))) & full);
    const uint32_t a = rot & hmask, b = rot >> h;
    const int k = __popc(a);
    const uint32_t Ck = sb.c[h][k];
    const int64_t off = boff[k] + (int64_t)colex_rank(a, sb) * Ck + colex_rank(b, sb);
    for (int v = 0; v < nv; v++) M[v * vstride + off] = vecs[(int64_t)v * ld + r];
  }
}

// G_k = M_k M_k^T for every (vector, block): 32 x 32 output tiles, 256 threads,
// FP64.  Block k of vector v: M at v * N + boff[k], G at goff[k] + v * C_k^2
// (the Gram matrices of one block index are contiguous over the vectors, the
// layout the batched eigensolver takes).
struct GramJob {
  int k, n, tiles;      // block index, C_k, tiles per side
  int64_t boff, goff;   // offsets of M_k in a vector's blocks, of G_k's region
  int64_t tile0;        // first global tile of this block index (over vectors)
};

__global__ void __launch_bounds__(256) k_schmidt_gram(const double* __restrict__ M, int64_t dim, const GramJob* jobs,
                                                      int n_jobs, int nv, double* __restrict__ G) {
  __shared__ double As[32][33], Bs[32][33];
  // find the job of this CTA (jobs in tile0 order)
  const int64_t t = blockIdx.x;
  int j = 0;
  while (j + 1 < n_jobs && jobs[j + 1].tile0 <= t) j++;
  const GramJob J = jobs[j];
  const int64_t local = t - J.tile0;
  const int per_vec = J.tiles * J.tiles;
  const int v = (int)(local / per_vec);
  if (v >= nv) return;
  const int ti = (int)(local % per_vec) / J.tiles, tj = (int)(local % per_vec) % J.tiles;
  const int n = J.n;
  const double* Mk = M + (int64_t)v * dim + J.boff;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;  // 8 rows of 32
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int c0 = 0; c0 < n; c0 += 32) {
    for (int q = 0; q < 4; q++) {
      const int row = ty + 8 * q;
      const int gi = ti * 32 + row, gj = tj * 32 + row, gc = c0 + tx;
      As[row][tx] = (gi < n && gc < n) ? Mk[(int64_t)gi * n + gc] : 0.0;
      Bs[row][tx] = (gj < n && gc < n) ? Mk[(int64_t)gj * n + gc] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < 32; c++) {
      const double bv = Bs[tx][c];
#pragma unroll
      for (int q = 0; q < 4; q++) acc[q] = fma(As[ty + 8 * q][c], bv, acc[q]);
    }
    __syncthreads();
  }
  double* Gk = G + J.goff + (int64_t)v * n * n;
  for (int q = 0; q < 4; q++) {
    const int gi = ti * 32 + ty + 8 * q, gj = tj * 32 + tx;
    if (gi < n && gj < n) Gk[(int64_t)gj * n + gi] = acc[q];  // symmetric: either order
  }
}

// -sum lambda ln lambda over the eigenvalues of every block of vector v
// (lambda <= 0 from rounding contributes nothing); one CTA per vector, fixed
// summation order.  W holds the eigenvalues at the Gram layout's offsets
// divided by C_k (woff[k] + v * C_k).
__global__ void k_schmidt_entropy(const double* __restrict__ W, const int64_t* woff, const int* sizes, int nblk,
                                  int nv, double* out, int64_t out_stride) {
  __shared__ double red[256];
  const int v = blockIdx.x;
  if (v >= nv) return;
  double s = 0.0;
  for (int k = 0; k < nblk; k++) {
    const int n = sizes[k];
    const double* w = W + woff[k] + (int64_t)v * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const double l = w[i];
      if (l > 0.0) s -= l * log(l);
    }
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[(int64_t)v * out_stride] = red[0];
}

// r_i for i = 0..n-3 and their sum, one CTA (fixed order); flag[0] = 1 if the
// values are not ascending, flag[1] = 1 if two consecutive gaps are both zero.
__global__ void k_gap_ratio(const double* __restrict__ e, int n, double* r_out, double* sum_out, int* flag) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int i = threadIdx.x; i + 2 < n; i += blockDim.x) {
    const double g0 = e[i + 1] - e[i], g1 = e[i + 2] - e[i + 1];
    if (g0 < 0.0 || g1 < 0.0) flag[0] = 1;
    const double mx = fmax(g0, g1), mn = fmin(g0, g1);
    double r = 0.0;
    if (mx > 0.0)
      r = mn / mx;
    else
      flag[1] = 1;
    if (r_out) r_out[i] = r;
    s += r;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *sum_out = red[0];
}

// ---------------------------------------------- eigenvalues of small blocks
// Householder tridiagonalization (Golub & Van Loan, section 8.3.1) of
// G = M M^T, one CTA per (vector, cut, block): G in shared memory (lower
// triangle, odd pitch), M staged through it in column chunks.  Writes the
// diagonal and the squared off-diagonals.
//
// GB300 runs 2 FP64 FMAs per SM and clock, so the FP64 pipe bounds all of this:
// the work per block is kept to n^3/2 (Gram) + 2 n^3/3 (reduction) FMAs, the
// square root and the division of a step are taken by one thread only, and
// eigenvalues come from Sturm counts without divisions, most of them in float-float
// (k_schmidt_values).
// Measured: 50 vectors at L = 14 (2800 blocks of 1 to 35 rows) 28.6 -> 0.85 ms
// against the batched library solver, whose 42 solves took 900 launches and a
// synchronization each.  Blocks beyond kTriMax rows do not fit shared memory
// and stay with the library.
constexpr int kTriThreads = 128;
constexpr int kTriMax = 126;  // C(9, 4): blocks of L <= 18
constexpr int kTriChunk = 16;

__host__ __device__ constexpr int tri_pitch(int n) { return n | 1; }
// per (vector, cut): 2^h diagonal and 2^h squared off-diagonal entries by block, h + 1 block scales (padded)
__host__ __device__ constexpr int64_t tri_doubles(int h) { return (2 << h) + 16; }
size_t tri_smem(int n) { return ((size_t)n * tri_pitch(n) + (size_t)n * (kTriChunk + 1) + 2 * n + 4) * sizeof(double); }

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// blockIdx.y chooses among the one or two blocks of this size (boff: in M, toff and k: in T).
__global__ void __launch_bounds__(kTriThreads) k_schmidt_tri(const double* __restrict__ M, int64_t dim, int n,
                                                              int64_t boff0, int64_t boff1, int toff0, int toff1,
                                                              int k0, int k1, int h, double* __restrict__ T) {
  extern __shared__ double sm[];
  const int P = tri_pitch(n), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* A = sm;                               // n x P
  double* C = A + (size_t)n * P;                // n x (chunk + 1)
  double* v = C + (size_t)n * (kTriChunk + 1);  // Householder vector
  double* q = v + n;
  double* sc = q + n;                           // scalars of the step
  const int64_t vc = blockIdx.x;
  const double* Mk = M + vc * dim + (blockIdx.y ? boff1 : boff0);
  double* d = T + vc * tri_doubles(h) + (blockIdx.y ? toff1 : toff0);
  double* e2 = d + (1 << h);
  // Gram, lower triangle: rows r and n-1-r share a line of n+1 entries
  const int half = (n + 1) / 2, ent = half * (n + 1);
  for (int e = tid; e < n * P; e += kTriThreads) A[e] = 0.0;
  for (int c0 = 0; c0 < n; c0 += kTriChunk) {
    __syncthreads();
    for (int e = tid; e < n * kTriChunk; e += kTriThreads) {
      const int i = e / kTriChunk, c = e % kTriChunk;
      C[i * (kTriChunk + 1) + c] = c0 + c < n ? Mk[(int64_t)i * n + c0 + c] : 0.0;
    }
    __syncthreads();
    for (int e = tid; e < ent; e += kTriThreads) {
      const int r = e / (n + 1), c = e - r * (n + 1);
      const bool up = c <= r;
      if (!up && n - 1 - r == r) continue;  // the middle row of odd n
      const int i = up ? r : n - 1 - r, j = up ? c : c - r - 1;
      double s = A[i * P + j];
#pragma unroll
      for (int u = 0; u < kTriChunk; u++) s = fma(C[i * (kTriChunk + 1) + u], C[j * (kTriChunk + 1) + u], s);
      A[i * P + j] = s;
    }
  }
  __syncthreads();
  // Scale by the power of two that brings the trace into [1/2, 1), so that the squares of the reduction
  // neither overflow nor (above the tail it drops) underflow
  if (warp == 0) {
    double t = 0.0;
    for (int i = lane; i < n; i += 32) t += A[i * P + i];
    t = warp_sum(t);
    if (lane == 0) {
      int ex = 0;
      frexp(t, &ex);
      ex = max(ex, -1000);
      const bool fin = t > 0.0 && isfinite(t);
      sc[2] = ldexp(1.0, -ex);
      sc[3] = fin ? 1.0 : 0.0;
      // not fin: t is 0 (an empty block) or not finite
      T[vc * tri_doubles(h) + (2 << h) + (blockIdx.y ? k1 : k0)] = fin ? ldexp(1.0, ex) : t;
    }
  }
  __syncthreads();
  if (sc[3] == 0.0) return;  // k_schmidt_values reads the scale alone
  for (int e = tid; e < n * P; e += kTriThreads) A[e] *= sc[2];
  __syncthreads();
  for (int k = 0; k + 2 < n; k++) {
    // v = x - alpha e_1, x = A[k+1.., k]; beta = 2 / |v|^2
    const int m = n - k - 1;
    const double* x = A + (k + 1) * P + k;
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane; i < m; i += 32)
        if (i > 0) s = fma(x[i * P], x[i * P], s);
      s = warp_sum(s);
      if (lane == 0) {
        const double x0 = x[0];
        double beta = 0.0, v0 = x0;
        double off2 = x0 * x0;
        // a tail below 2^-450 of the trace is taken as zero: its square would leave FP64's range
        if (s > 0x1p-900) {
          off2 = fma(x0, x0, s);
          const double nx = sqrt(off2);
          v0 = x0 + (x0 >= 0.0 ? nx : -nx);
          beta = 2.0 / fma(v0, v0, s);
        }
        sc[0] = beta;
        sc[1] = v0;
        d[k] = A[k * P + k];
        e2[k] = off2;
      }
    }
    __syncthreads();
    const double beta = sc[0], v0 = sc[1];
    if (beta != 0.0) {
      // p = beta A v (four threads per row; the upper triangle by symmetry)
      const double* B = A + (k + 1) * P + (k + 1);
      for (int r0 = 0; r0 < m; r0 += kTriThreads / 4) {
        const int i = r0 + tid / 4, part = tid % 4;
        double s = 0.0;
        if (i < m)
          for (int j = part; j < m; j += 4)
            s = fma(j <= i ? B[i * P + j] : B[j * P + i], j == 0 ? v0 : x[j * P], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (i < m && part == 0) {
          q[i] = beta * s;
          v[i] = i == 0 ? v0 : x[i * P];
        }
      }
      __syncthreads();
      // w = p - (beta p^T v / 2) v, A -= v w^T + w v^T
      if (warp == 0) {
        double s = 0.0;
        for (int i = lane; i < m; i += 32) s = fma(q[i], v[i], s);
        s = warp_sum(s) * (-0.5 * beta);
        for (int i = lane; i < m; i += 32) q[i] = fma(s, v[i], q[i]);
      }
      __syncthreads();
      double* W = A + (k + 1) * P + (k + 1);
      const int hm = (m + 1) / 2, em = hm * (m + 1);
      for (int e = tid; e < em; e += kTriThreads) {
        const int r = e / (m + 1), c = e - r * (m + 1);
        const bool up = c <= r;
        if (!up && m - 1 - r == r) continue;
        const int i = up ? r : m - 1 - r, j = up ? c : c - r - 1;
        W[i * P + j] -= fma(v[i], q[j], q[i] * v[j]);
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    const int k = n - 2;
    if (n >= 2) {
      d[k] = A[k * P + k];
      const double o = A[(k + 1) * P + k];
      e2[k] = o * o;
    }
    d[n - 1] = A[(n - 1) * P + n - 1];
    e2[n - 1] = 0.0;
  }
}

// Number of eigenvalues below x of the tridiagonal (d, e2), by the signs of the
// leading principal minors p_i = (d_i - x) p_{i-1} - e2_{i-1} p_{i-2} (Givens'
// Sturm sequence).  Only signs matter, so both minors are rescaled by a power
// of two after every term (integer arithmetic on the exponents: |p| in [1, 2));
// a minor below 2^-200 of its predecessor counts as -2^-200 of it.
__device__ __forceinline__ int sturm(const double* __restrict__ d, const double* __restrict__ e2, int n, double x) {
  constexpr int kTiny = 1023 - 200;
  int cnt = 0;
  double p = 1.0, pm = 0.0, e = 0.0;
  for (int i = 0; i < n; i++) {
    const double nx = fma(__ldg(d + i) - x, p, -(e * pm));
    e = __ldg(e2 + i);
    const int hi = __double2hiint(nx), ho = __double2hiint(p);
    int ex = (hi >> 20) & 0x7FF;
    const bool tiny = ex < kTiny;
    const int sign = (tiny ? ~ho : hi) & 0x80000000;
    ex = tiny ? kTiny : ex;
    cnt += (uint32_t)(sign ^ ho) >> 31;
    pm = __hiloint2double((ho & 0x800FFFFF) | ((2046 - ex) << 20), __double2loint(p));
    p = __hiloint2double(sign | (tiny ? 0 : hi & 0xFFFFF) | (1023 << 20), tiny ? 0 : __double2loint(nx));
  }
  return cnt;
}

// The same count in float-float arithmetic (2^-46) on the FP32 pipe, for a first
// bracket; d and e2 as (hi, lo).  A minor below 2^-60 of its predecessor counts as
// -2^-60 of it.
__device__ __forceinline__ int sturm_ff(const float2* d, const float2* e2, int n, double x) {
  constexpr int kTiny = 127 - 60;
  const float xh = (float)x;
  const float2 mx = make_float2(-xh, -(float)(x - (double)xh));
  int cnt = 0;
  float2 p = make_float2(1.f, 0.f), pm = make_float2(0.f, 0.f), e = pm;
  for (int i = 0; i < n; i++) {
    const float2 w = df_mul(e, pm), nx = df_add(df_mul(df_add(d[i], mx), p), make_float2(-w.x, -w.y));
    e = e2[i];
    const int hi = __float_as_int(nx.x), ho = __float_as_int(p.x);
    int ex = (hi >> 23) & 0xFF;
    const bool tiny = ex < kTiny;
    const int sign = (tiny ? ~ho : hi) & 0x80000000;
    ex = tiny ? kTiny : ex;
    cnt += (uint32_t)(sign ^ ho) >> 31;
    const float f = __int_as_float((254 - ex) << 23);
    pm = make_float2(p.x * f, p.y * f);
    p = tiny ? make_float2(__int_as_float(sign | 0x3F800000), 0.f) : make_float2(nx.x * f, nx.y * f);
  }
  return cnt;
}

// One thread per eigenvalue, one CTA of 2^h threads per (vector, cut): bisection
// on the Sturm count to 2^-62 of the block's trace (below the rounding of G) or
// to the last bit, then S = -sum lambda ln lambda (lambda <= 0 from rounding
// contributes nothing), summed in fixed order.  `first` holds the offset of each
// block's eigenvalues (h + 2 entries).
// Three FP64 instructions a term, at 2 a clock and SM, bound it: so the first 38
// bisections count in float-float, two FP64 counts confirm the bracket they leave
// (widened by its rounding; the whole interval otherwise) and FP64 goes on from
// there.  50 vectors at L = 14: 737 us with FP64 alone, now 482 us.
struct BlockFirst {
  int v[12];
};
__global__ void __launch_bounds__(512) k_schmidt_values(const double* __restrict__ T, int h, const BlockFirst first,
                                                        double* __restrict__ S) {
  __shared__ double red[512];
  __shared__ float2 fd[512], fe[512];
  const int64_t vc = blockIdx.x;
  const int t = threadIdx.x;
  const double* base = T + vc * tri_doubles(h);
  auto split = [](double v) { return make_float2((float)v, (float)(v - (double)(float)v)); };
  fd[t] = split(base[t]);
  fe[t] = split(base[t + (1 << h)]);
  __syncthreads();
  int k = 0;
  while (t >= first.v[k + 1]) k++;
  const int n = first.v[k + 1] - first.v[k], idx = t - first.v[k];
  const double scale = base[(2 << h) + k];
  double s = 0.0;
  if (scale > 0.0 && isfinite(scale)) {
    const double* d = base + first.v[k];
    const double* e2 = d + (1 << h);
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < 38; it++) {
      const double mid = 0.5 * (lo + hi);
      if (sturm_ff(fd + first.v[k], fe + first.v[k], n, mid) > idx)
        hi = mid;
      else
        lo = mid;
    }
    lo -= 0x1p-39;
    hi += 0x1p-39;
    if (sturm(d, e2, n, lo) > idx || sturm(d, e2, n, hi) <= idx) {
      lo = -0x1p-48;
      hi = 1.0 + 0x1p-48;
    }
    for (int it = 0; it < 64; it++) {
      const double mid = 0.5 * (lo + hi);
      if (mid == lo || mid == hi || hi - lo < 0x1p-62) break;
      if (sturm(d, e2, n, mid) > idx)
        hi = mid;
      else
        lo = mid;
    }
    const double l = 0.5 * (lo + hi) * scale;
    if (l > 0.0) s = -l * log(l);
  } else if (scale != 0.0) {
    s = scale - scale;  // not finite
  }
  red[t] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (t < o) red[t] += red[t + o];
    __syncthreads();
  }
  if (t == 0) S[vc] = red[0];
}

struct StreamMem {
  void* p = nullptr;
  cudaStream_t s = nullptr;
  ~StreamMem() {
    if (p) cudaFreeAsync(p, s);
  }
};

uint64_t binom64(int n, int k) {
  if (k < 0 || k > n) return 0;
  uint64_t r = 1;
  for (int i = 1; i <= k; i++) r = r * (uint64_t)(n - k + i) / (uint64_t)i;
  return r;
}

// All blocks have at most kTriMax rows: every cut of a group of vectors in
// h / 2 + 3 launches.  Sh[v * h + x]: entropy of cut x.
int entropy_small(int L, const uint32_t* d_states, const double* d_vecs, int64_t ld, int n_vec, cudaStream_t s,
                  std::vector<double>& Sh) {
  const int h = L / 2;
  const int64_t dim = (int64_t)binom64(L, h);
  std::vector<int64_t> boff(h + 2, 0);
  BlockFirst first{};
  for (int k = 0; k <= h; k++) {
    const int64_t n = (int64_t)binom64(h, k);
    boff[k + 1] = boff[k] + n * n;
    first.v[k + 1] = first.v[k] + (int)n;
  }
  // blocks of nvb vectors and all cuts within ~1 GiB
  const int nvb = (int)std::max<int64_t>(1, std::min<int64_t>(n_vec, (int64_t)(1 << 30) / (8 * h * (dim + tri_doubles(h)))));
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t bM = up((size_t)nvb * h * dim * 8), bT = up((size_t)nvb * h * tri_doubles(h) * 8), bS = up((size_t)n_vec * h * 8);
  StreamMem mem;
  mem.s = s;
  if (scratch_alloc(&mem.p, bM + bT + bS + 256, s) != POLFED_OK) {
    cudaGetLastError();
    return fail(POLFED_ENOMEM, "device workspace for the Schmidt blocks");
  }
  double* M = (double*)mem.p;
  double* T = (double*)((char*)mem.p + bM);
  double* dS = (double*)((char*)mem.p + bM + bT);
  int64_t* d_boff = (int64_t*)((char*)mem.p + bM + bT + bS);
  PF_CUDA(cudaMemcpyAsync(d_boff, boff.data(), boff.size() * 8, cudaMemcpyHostToDevice, s));
  PF_CUDA(cudaFuncSetAttribute(k_schmidt_tri, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tri_smem(kTriMax)));
  for (int v0 = 0; v0 < n_vec; v0 += nvb) {
    const int nv = std::min(nvb, n_vec - v0);
    const int grid = (int)std::min<int64_t>((dim + 255) / 256, 152 * 8);
    k_schmidt_scatter<<<dim3(grid, h), 256, 0, s>>>(d_states, dim, L, 0, d_vecs + (int64_t)v0 * ld, ld, nv, d_boff, M,
                                                    h * dim);
    for (int k = h / 2; k >= 0; k--) {  // largest blocks first
      const int n = (int)binom64(h, k), k1 = h - k;
      k_schmidt_tri<<<dim3(nv * h, k1 != k ? 2 : 1), kTriThreads, tri_smem(n), s>>>(
          M, dim, n, boff[k], boff[k1], first.v[k], first.v[k1], k, k1, h, T);
    }
    k_schmidt_values<<<nv * h, 1 << h, 0, s>>>(T, h, first, dS + (int64_t)v0 * h);
    PF_CUDA(cudaGetLastError());
    count_launch(h / 2 + 3);
  }
  Sh.resize((size_t)n_vec * h);
  PF_CUDA(cudaMemcpyAsync(Sh.data(), dS, Sh.size() * 8, cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  for (double v : Sh)
    if (!std::isfinite(v)) return fail(POLFED_ECUDA, "eigen-solve of a Schmidt block that is not finite");
  return POLFED_OK;
}

void entropy_out(const std::vector<double>& Sh, int L, int n_vec, int per_cut, double* S) {
  const int h = L / 2;
  for (int v = 0; v < n_vec; v++) {
    if (per_cut) {
      for (int x = 0; x < L; x++) S[(size_t)v * L + x] = Sh[(size_t)v * h + (x % h)];
    } else {
      double a = 0.0;
      for (int x = 0; x < h; x++) a += Sh[(size_t)v * h + x];
      S[v] = a / h;
    }
  }
}

}  // namespace

}  // namespace polfed

using namespace polfed;

extern "C" {

int polfed_gap_ratio(const double* d_evals, int32_t n, double* r_mean, double* d_r, polfed_stream_t stream) {
  clear_error();
  if (!d_evals || !r_mean) return fail(POLFED_EINVAL, "d_evals or r_mean is NULL");
  if (n < 3) return fail(POLFED_EINVAL, "need at least 3 eigenvalues");
  cudaStream_t s = (cudaStream_t)stream;
  StreamMem mem;
  mem.s = s;
  PF_CHECK(scratch_alloc(&mem.p, 64, s));
  double* sum = (double*)mem.p;
  int* flag = (int*)((char*)mem.p + 32);
  PF_CUDA(cudaMemsetAsync(mem.p, 0, 64, s));
  k_gap_ratio<<<1, 1024, 0, s>>>(d_evals, n, d_r, sum, flag);
  PF_CUDA(cudaGetLastError());
  count_launch();
  double hs = 0.0;
  int hf[2] = {0, 0};
  PF_CUDA(cudaMemcpyAsync(&hs, sum, sizeof(double), cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaMemcpyAsync(hf, flag, sizeof(hf), cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  if (hf[0]) return fail(POLFED_EINVAL, "eigenvalues are not in ascending order");
  if (hf[1]) return fail(POLFED_EINVAL, "two consecutive zero gaps: the gap ratio is undefined");
  *r_mean = hs / (double)(n - 2);
  return POLFED_OK;
}

int polfed_entanglement_entropy(polfed_ctx* ctx, int32_t L, const uint32_t* d_states, const double* d_vecs,
                                int64_t ld, int32_t n_vec, int32_t per_cut, double* S) {
  clear_error();
  if (!ctx) return fail(POLFED_EINVAL, "ctx is NULL");
  if (L < 4 || L > 32 || (L & 1)) return fail(POLFED_EINVAL, "L must be even, 4 <= L <= 32");
  if (!d_states || !d_vecs || !S) return fail(POLFED_EINVAL, "NULL pointer");
  const int h = L / 2;
  if (h > 16) return fail(POLFED_EINVAL, "L must be <= 32");
  const int64_t dim = (int64_t)binom64(L, h);
  if (ld < dim) return fail(POLFED_EINVAL, "ld must be >= C(L, L/2)");
  if (n_vec < 1) return fail(POLFED_EINVAL, "n_vec must be >= 1");
  const int dev = ctx_device(ctx);
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(dev);
  struct Restore {
    int d;
    ~Restore() { cudaSetDevice(d); }
  } restore{prev};
  cudaStream_t s = ctx_stream(ctx);
  if ((int64_t)binom64(h, h / 2) <= kTriMax) {
    std::vector<double> Sh;
    PF_CHECK(entropy_small(L, d_states, d_vecs, ld, n_vec, s, Sh));
    entropy_out(Sh, L, n_vec, per_cut, S);
    return POLFED_OK;
  }
  cusolverDnHandle_t solver = (cusolverDnHandle_t)ctx_solver(ctx);
  // blocks k = 0..h (C_k = C(h, k)); Gram regions ordered k = 0, h, 1, h-1, ... so that the two
  // blocks of equal size sit next to each other (one batched eigen-solve per size)
  std::vector<int> sizes(h + 1);
  std::vector<int64_t> boff(h + 2, 0);
  for (int k = 0; k <= h; k++) {
    sizes[k] = (int)binom64(h, k);
    boff[k + 1] = boff[k] + (int64_t)sizes[k] * sizes[k];
  }
  // batch of vectors per pass: blocks + Gram matrices (2 N doubles each) within ~1 GiB
  const int nv_max = (int)std::max<int64_t>(1, std::min<int64_t>(n_vec, (int64_t)(1 << 30) / (16 * dim)));
  std::vector<int> order;  // block order of the Gram regions
  for (int k = 0; k <= h / 2; k++) {
    order.push_back(k);
    if (h - k != k) order.push_back(h - k);
  }
  std::vector<int64_t> goff(h + 1), woff(h + 1);
  {
    int64_t g = 0, w = 0;
    for (int k : order) {
      goff[k] = g;
      woff[k] = w;
      g += (int64_t)nv_max * sizes[k] * sizes[k];
      w += (int64_t)nv_max * sizes[k];
    }
  }
  // Gram jobs (tiles) in block order
  std::vector<GramJob> jobs;
  int64_t tiles_total = 0;
  for (int k = 0; k <= h; k++) {
    GramJob J;
    J.k = k;
    J.n = sizes[k];
    J.tiles = (sizes[k] + 31) / 32;
    J.boff = boff[k];
    J.goff = goff[k];
    J.tile0 = tiles_total;
    tiles_total += (int64_t)nv_max * J.tiles * J.tiles;
    jobs.push_back(J);
  }
  // batched eigensolver workspace per size class
  cusolverDnParams_t params = nullptr;
  if (cusolverDnCreateParams(&params) != CUSOLVER_STATUS_SUCCESS) return fail(POLFED_ECUDA, "cusolverDnCreateParams");
  struct Params {
    cusolverDnParams_t p;
    ~Params() { cusolverDnDestroyParams(p); }
  } pguard{params};
  size_t ws_dev = 0, ws_host = 0;
  for (size_t q = 0; q < order.size();) {
    const int k = order[q];
    const int n = sizes[k];
    const int cnt = (q + 1 < order.size() && sizes[order[q + 1]] == n) ? 2 : 1;
    size_t d = 0, hh = 0;
    if (cusolverDnXsyevBatched_bufferSize(solver, params, CUSOLVER_EIG_MODE_NOVECTOR, CUBLAS_FILL_MODE_LOWER, n,
                                          CUDA_R_64F, nullptr, n, CUDA_R_64F, nullptr, CUDA_R_64F, &d, &hh,
                                          (int64_t)cnt * nv_max) != CUSOLVER_STATUS_SUCCESS)
      return fail(POLFED_ECUDA, "cusolverDnXsyevBatched_bufferSize failed");
    ws_dev = std::max(ws_dev, d);
    ws_host = std::max(ws_host, hh);
    q += cnt;
  }
  const size_t a256 = 255;
  auto up = [&](size_t b) { return (b + a256) & ~a256; };
  const size_t bM = up((size_t)nv_max * dim * 8), bG = up((size_t)nv_max * dim * 8), bW = up((size_t)nv_max * dim * 8);
  const size_t bOff = up((h + 2) * 8 * 3), bJobs = up(jobs.size() * sizeof(GramJob)), bSz = up((h + 1) * 4);
  const size_t bInfo = up((size_t)2 * nv_max * 4), bS = up((size_t)n_vec * h * 8), bWs = up(ws_dev + 16);
  StreamMem mem;
  mem.s = s;
  if (scratch_alloc(&mem.p, bM + bG + bW + bOff + bJobs + bSz + bInfo + bS + bWs, s) != POLFED_OK) {
    cudaGetLastError();
    return fail(POLFED_ENOMEM, "device workspace for the Schmidt blocks");
  }
  char* base = (char*)mem.p;
  double* M = (double*)base;
  double* G = (double*)(base + bM);
  double* Wd = (double*)(base + bM + bG);
  int64_t* d_boff = (int64_t*)(base + bM + bG + bW);
  int64_t* d_woff = d_boff + (h + 2);
  GramJob* d_jobs = (GramJob*)(base + bM + bG + bW + bOff);
  int* d_sizes = (int*)(base + bM + bG + bW + bOff + bJobs);
  int* d_info = (int*)(base + bM + bG + bW + bOff + bJobs + bSz);
  double* d_S = (double*)(base + bM + bG + bW + bOff + bJobs + bSz + bInfo);
  void* d_ws = base + bM + bG + bW + bOff + bJobs + bSz + bInfo + bS;
  std::vector<char> h_ws(ws_host + 16);
  std::vector<int64_t> offs(2 * (h + 2), 0);
  for (int k = 0; k <= h + 1; k++) offs[k] = boff[k];
  for (int k = 0; k <= h; k++) offs[h + 2 + k] = woff[k];
  PF_CUDA(cudaMemcpyAsync(d_boff, offs.data(), offs.size() * 8, cudaMemcpyHostToDevice, s));
  PF_CUDA(cudaMemcpyAsync(d_jobs, jobs.data(), jobs.size() * sizeof(GramJob), cudaMemcpyHostToDevice, s));
  PF_CUDA(cudaMemcpyAsync(d_sizes, sizes.data(), sizes.size() * 4, cudaMemcpyHostToDevice, s));
  std::vector<int> hinfo(2 * nv_max);
  for (int v0 = 0; v0 < n_vec; v0 += nv_max) {
    const int nv = std::min(nv_max, n_vec - v0);
    for (int x = 0; x < h; x++) {
      const int grid = (int)std::min<int64_t>((dim + 255) / 256, 152 * 8);
      k_schmidt_scatter<<<grid, 256, 0, s>>>(d_states, dim, L, x, d_vecs + (int64_t)v0 * ld, ld, nv, d_boff, M, dim);
      PF_CUDA(cudaGetLastError());
      count_launch();
      // tiles of the vectors present (the job table is laid out for nv_max vectors; CTAs of absent
      // vectors return at once)
      k_schmidt_gram<<<(unsigned)tiles_total, 256, 0, s>>>(M, dim, d_jobs, (int)jobs.size(), nv, G);
      PF_CUDA(cudaGetLastError());
      count_launch();
      for (size_t q = 0; q < order.size();) {
        const int k = order[q];
        const int n = sizes[k];
        const int cnt = (q + 1 < order.size() && sizes[order[q + 1]] == n) ? 2 : 1;
        // the regions of the cnt blocks are adjacent; with nv < nv_max the second one starts
        // nv_max matrices after the first, so solve each block's nv matrices separately then
        for (int c = 0; c < cnt; c++) {
          const int kk = order[q + c];
          if (n == 1) {  // a 1 x 1 block is its own eigenvalue
            PF_CUDA(cudaMemcpyAsync(Wd + woff[kk], G + goff[kk], (size_t)nv * 8, cudaMemcpyDeviceToDevice, s));
            continue;
          }
          if (cusolverDnXsyevBatched(solver, params, CUSOLVER_EIG_MODE_NOVECTOR, CUBLAS_FILL_MODE_LOWER, n,
                                     CUDA_R_64F, G + goff[kk], n, CUDA_R_64F, Wd + woff[kk], CUDA_R_64F, d_ws,
                                     ws_dev, h_ws.data(), ws_host, d_info, (int64_t)nv) != CUSOLVER_STATUS_SUCCESS)
            return fail(POLFED_ECUDA, "cusolverDnXsyevBatched failed");
          PF_CUDA(cudaMemcpyAsync(hinfo.data(), d_info, (size_t)nv * 4, cudaMemcpyDeviceToHost, s));
          PF_CUDA(cudaStreamSynchronize(s));
          for (int i = 0; i < nv; i++)
            if (hinfo[i] != 0) return fail(POLFED_ECUDA, "batched eigen-solve info = " + std::to_string(hinfo[i]));
        }
        q += cnt;
      }
      k_schmidt_entropy<<<nv, 256, 0, s>>>(Wd, d_woff, d_sizes, h + 1, nv, d_S + (int64_t)v0 * h + x, h);
      PF_CUDA(cudaGetLastError());
      count_launch();
    }
  }
  std::vector<double> Sh((size_t)n_vec * h);
  PF_CUDA(cudaMemcpyAsync(Sh.data(), d_S, Sh.size() * 8, cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  entropy_out(Sh, L, n_vec, per_cut, S);
  return POLFED_OK;
}

}  // extern "C"
