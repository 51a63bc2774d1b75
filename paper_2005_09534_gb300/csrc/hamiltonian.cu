// Matrix-free H~ application and the Clenshaw evaluation of P^K_sigma(H~) X.
//
// Eq. (1) in the S^z = 0 basis: the diagonal is sum_{bonds} J_l Delta z_i z_j
// + sum_i h_i z_i (z = +-1/2) and every antiparallel pair (i, i+l) connects s
// to s ^ (2^i | 2^(i+l)) with amplitude J_l / 2 (Supplement, "Technical
// details": the off-diagonal elements are constants and are never loaded).
// Rescaling (text before Eq. (3)): H~ = alpha (H - beta), alpha = 2/(e_hi - e_lo),
// beta = (e_hi + e_lo)/2.
//
// Ranking.  Split a state into its low b bits s_lo and high L-b bits s_hi.
// With the combinatorial number system, rank(s) = sum_k C(p_k, k+1) over the
// set bits p_0 < p_1 < ...  The low bits contribute T_lo[s_lo] (the rank of
// s_lo among b-bit strings of its popcount) and the high bits T_hi[s_hi]
// (their indices are shifted by popc(s_lo) = L/2 - popc(s_hi)), so
// rank(s) = T_hi[s_hi] + T_lo[s_lo].  All rows with one s_hi form a contiguous
// "group" of C(b, L/2 - popc(s_hi)) rows starting at T_hi[s_hi].
//
// Kernel layout (rows.h).  A team of four warps owns one group at a time and
// stages the group's rows of the gather source b1 in shared memory.  A row's
// neighbours are then
//   - low bonds (both sites in the low part): rows of the same group -> shared memory;
//   - high bonds (both sites high): row T_hi[s_hi'] + local index, i.e. the
//     same local row of another group -> coalesced loads from L2;
//   - cross bonds (one site in each part): a gather inside a neighbour group.
// Vectors are processed in column slices of 16*LPR bytes (LPR lanes per row,
// 16 bytes per lane), stored slice-major (row stride = slice width).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <mutex>
#include <thread>
#include <type_traits>

#include "polfed_internal.h"
#include "rows.h"

namespace polfed {

// ------------------------------------------------------------- binomials
__constant__ uint32_t c_binom[33][33];
__device__ uint32_t d_binom[33][33];  // for divergent reads
static uint32_t h_binom[33][33];
static std::once_flag h_binom_once;

static void init_binom() {
  std::call_once(h_binom_once, [] {
    memset(h_binom, 0, sizeof(h_binom));
    for (int n = 0; n <= 32; n++) {
      h_binom[n][0] = 1;
      for (int k = 1; k <= n; k++) h_binom[n][k] = h_binom[n - 1][k - 1] + (k <= n - 1 ? h_binom[n - 1][k] : 0);
    }
  });
}

uint32_t binom_host(int n, int k) {
  init_binom();
  if (n < 0 || n > 32 || k < 0 || k > n) return 0;
  return h_binom[n][k];
}

void upload_binomials() {
  init_binom();
  static std::mutex mu;
  static uint64_t done = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  if (dev < 64 && (done >> dev) & 1) return;
  cudaMemcpyToSymbol(c_binom, h_binom, sizeof(h_binom));
  cudaMemcpyToSymbol(d_binom, h_binom, sizeof(h_binom));
  if (dev < 64) done |= (1ull << dev);
}

// -------------------------------------------------------------- geometry
// Low bits of a plan.  Large L: b = 10, a group block of at most C(10,5) * 128 B
// = 32 KB (six teams to an SM).  Smaller L: smaller groups, so that there are
// more of them for the 912 teams (by L alone; a block of several slices has that
// many more work items).  Measured on GB300 (whole calls, b one lower / chosen /
// one higher): L = 14 FP64 K = 200: 1.20, 1.14, 1.37 ms; L = 18 float-float 256
// moments: 3.16, 2.85, 3.33 ms; L = 20 J1-J2 float-float K = 64: 7.93, 7.23, 7.48 ms
// (FP32 per column: 3.74, 3.14, 3.04); L = 22 FP32 K = 200 at b = 8 / 9 / 10: 45.1,
// 40.6, 40.2 ms.
static int clamp_b(int L, int b) {
  if (const char* e = getenv("POLFED_LOWBITS")) b = atoi(e);
  if (b > 10) b = 10;
  if (b < 2) b = 2;
  if (L - b < 2) b = L - 2;
  return b;
}
static int choose_b(int L) { return clamp_b(L, L <= 14 ? L - 9 : (L <= 20 ? L / 2 - 1 : 10)); }
// FP32 moments keep their split too: it decides the order of their sums (policy RF32M).
int moments_b(int kind, int L) { return kind == POLFED_F32 ? clamp_b(L, L - 10) : 0; }

int build_geometry(const polfed_model* m, int b_override, HamGeometry* g) {
  if (!m) return fail(POLFED_EINVAL, "model is NULL");
  if (m->L < 4 || m->L > 32 || (m->L & 1)) return fail(POLFED_EINVAL, "L must be even, 4 <= L <= 32");
  if (!m->h) return fail(POLFED_EINVAL, "model.h is NULL");
  memset(g, 0, sizeof(*g));
  const int L = m->L;
  g->L = L;
  g->n_up = L / 2;
  g->periodic = m->periodic ? 1 : 0;
  g->J1 = m->J1;
  g->J2 = m->J2;
  g->Delta = m->Delta;
  for (int i = 0; i < L; i++) {
    if (!std::isfinite(m->h[i])) return fail(POLFED_EINVAL, "non-finite field h_i");
    g->h[i] = m->h[i];
  }
  if (!std::isfinite(m->J1) || !std::isfinite(m->J2) || !std::isfinite(m->Delta))
    return fail(POLFED_EINVAL, "non-finite coupling");
  g->dim = (int64_t)binom_host(L, L / 2);
  int b = b_override > 0 ? b_override : choose_b(L);
  if (b < 2 || L - b < 2) return fail(POLFED_EINVAL, "bad low/high split");
  g->b = b;
  g->nh = L - b;
  // literal terms of Eq. (1): l = 1, 2 and i = 0..L-1 (j = i + l, wrapped if periodic)
  std::vector<Bond> low, high, cross;
  for (int l = 1; l <= 2; l++) {
    double J = (l == 1) ? m->J1 : m->J2;
    if (J == 0.0) continue;
    for (int i = 0; i < L; i++) {
      int j = i + l;
      if (j >= L) {
        if (!g->periodic) continue;
        j -= L;
      }
      Bond bd{std::min(i, j), std::max(i, j), l};
      if (bd.j < b)
        low.push_back(bd);
      else if (bd.i >= b)
        high.push_back(bd);
      else
        cross.push_back(bd);
    }
  }
  auto by_cls = [](const Bond& x, const Bond& y) { return x.cls < y.cls; };
  std::stable_sort(low.begin(), low.end(), by_cls);
  std::stable_sort(high.begin(), high.end(), by_cls);
  if ((int)low.size() > kMaxBonds || (int)high.size() > kMaxBonds || (int)cross.size() > 8)
    return fail(POLFED_EINVAL, "too many bonds for the table layout");
  for (auto& x : low) {
    g->low_mask[g->n_low1 + g->n_low2] = (1u << x.i) | (1u << x.j);
    (x.cls == 1 ? g->n_low1 : g->n_low2)++;
  }
  for (auto& x : high) {
    g->high_mask[g->n_high1 + g->n_high2] = (1u << (x.i - b)) | (1u << (x.j - b));
    (x.cls == 1 ? g->n_high1 : g->n_high2)++;
  }
  for (auto& x : cross) {
    g->cross_lo[g->n_cross] = x.i;
    g->cross_hi[g->n_cross] = x.j - b;
    g->cross_cls[g->n_cross] = x.cls;
    g->n_cross++;
  }
  int off = 0;
  for (int c = 0; c <= b + 1; c++) {
    g->cls_off[c] = off;
    if (c <= b) off += (int)binom_host(b, c);
  }
  {
    const bool j2 = g->n_low2 + g->n_high2 > 0 || m->J2 != 0.0;
    const int maxcr = j2 ? 6 : 2;
    g->rec_stride = j2 ? 32 : 16;
    if (2 + g->n_low1 + g->n_low2 + maxcr > g->rec_stride) return fail(POLFED_EINVAL, "too many low bonds for the record");
    if (g->n_high1 + g->n_high2 > kMaxHigh) return fail(POLFED_EINVAL, "too many high bonds for the group table");
  }
  g->max_group = 0;
  g->n_groups = 0;
  for (int pc = 0; pc <= g->nh; pc++) {
    int n_lo = g->n_up - pc;
    if (n_lo < 0 || n_lo > b) continue;
    g->max_group = std::max(g->max_group, (int)binom_host(b, n_lo));
    g->n_groups += (int)binom_host(g->nh, pc);
  }
  return POLFED_OK;
}

// ------------------------------------------------------------ table kernels
// First row of the schedule of the groups with popcount pc: classes by
// decreasing group size (sizes depend only on the popcount), groups of a class
// in ascending s_hi.  Neighbours through high bonds share the popcount, so the
// class in work (30 MB of b1 at L = 22) stays in L2.
struct ClassStart {
  int v[34];
};

static ClassStart class_starts(const HamGeometry& g) {
  ClassStart cs{};
  int pcs[34], sizes[34], n = 0;
  for (int pc = 0; pc <= g.nh; pc++) {
    const int n_lo = g.n_up - pc;
    if (n_lo < 0 || n_lo > g.b) continue;
    pcs[n] = pc;
    sizes[n++] = (int)binom_host(g.b, n_lo);
  }
  for (int i = 1; i < n; i++)  // stable insertion sort by decreasing size
    for (int j = i; j > 0 && sizes[j] > sizes[j - 1]; j--) {
      std::swap(sizes[j], sizes[j - 1]);
      std::swap(pcs[j], pcs[j - 1]);
    }
  int pos = 0;
  for (int i = 0; i < n; i++) {
    cs.v[pcs[i]] = pos;
    pos += (int)binom_host(g.nh, pcs[i]);
  }
  return cs;
}

// alpha- and beta-scaled diagonals of one storage type: low part by cls_off +
// local index, then the groups in schedule order (alpha * (F_hi - beta)), then
// the cross patterns.  kind < 0: none.
struct TypedOut {
  int kind;
  double alpha, beta;
  void* out;
  __device__ __forceinline__ void put(int i, double v) const {
    if (kind == POLFED_F32)
      reinterpret_cast<float*>(out)[i] = (float)v;
    else if (kind == POLFED_F64)
      reinterpret_cast<double*>(out)[i] = v;
    else
      reinterpret_cast<float2*>(out)[i] = make_float2((float)v, (float)(v - (double)(float)v));
  }
};

// All tables of a plan in one launch: thread i < n_main does low state i (rank,
// diagonal), high state i (rank, diagonal, its group's place in the schedule and
// the head of its record) and cross pattern i; the threads after them one entry
// of a neighbour record or one neighbour of a group each.  A state's neighbours are ranked again instead of being
// read from another launch's table, with the binomials in shared memory (as
// divergent reads of constant memory they are serialized).  Bound by launches and
// latency: the four kernels this replaces took 21 us and three more launches at
// L = 22, this one 10; an L = 12 call with one column took 52 us, now 40.
constexpr int kTableThreads = 128;
__global__ void __launch_bounds__(kTableThreads) k_tables(const HamGeometry g, const ClassStart cs, HamTables t, int* err,
                                                          TypedOut ty, int n_main) {
  __shared__ uint32_t B[33][33];
  for (int e = threadIdx.x; e < 33 * 33; e += kTableThreads) (&B[0][0])[e] = (&d_binom[0][0])[e];
  __syncthreads();
  const int i = blockIdx.x * kTableThreads + threadIdx.x;
  auto rank_lo = [&](uint32_t a) {
    uint32_t r = 0;
    for (int k = 1; a; a &= a - 1, k++) r += B[__ffs(a) - 1][k];
    return r;
  };
  // first row of a group: its bits sit above n_lo low ones
  auto rank_hi = [&](uint32_t a) {
    uint32_t r = 0;
    for (int k = g.n_up - __popc(a) + 1; a; a &= a - 1, k++) r += B[g.b + __ffs(a) - 1][k];
    return (int)r;
  };
  auto valid = [&](uint32_t a) {
    const int n = g.n_up - __popc(a);
    return n >= 0 && n <= g.b;
  };
  const int RS = g.rec_stride;
  int j = i - n_main;
  if (j >= RS << g.b) {  // one neighbour of a group: kMaxHigh high ones, then 8 cross bonds
    j -= RS << g.b;
    const int e = j % (kMaxHigh + 8);
    const uint32_t grp = (uint32_t)(j / (kMaxHigh + 8));
    if (grp >> g.nh || !valid(grp)) return;
    GroupRec* r = t.grec + cs.v[__popc(grp)] + (int)rank_lo(grp);
    if (e < kMaxHigh) {
      uint32_t m = 0;
      int cnt = 0;
      for (int q = 0; q < g.n_high1 + g.n_high2 && !m; q++)
        if (__popc(grp & g.high_mask[q]) == 1 && cnt++ == e) m = g.high_mask[q];
      r->hn_base[e] = m ? rank_hi(grp ^ m) : 0;
    } else {
      const int k = e - kMaxHigh;
      int base = 0, n = 0;
      if (k < g.n_cross) {
        const uint32_t g2 = grp ^ (1u << g.cross_hi[k]);
        // rows with the bond antiparallel exist only if the neighbouring class is valid
        if (valid(g2)) {
          base = rank_hi(g2);
          n = (int)B[g.b][g.n_up - __popc(g2)];
        }
      }
      r->cr_base[k] = base;
      r->cr_n[k] = n;
    }
    return;
  }
  if (j >= 0) {  // neighbour records (layout in HamTables::rec): one entry, for every row size
    const uint32_t a = (uint32_t)(j / RS);
    const int e = j % RS, l1 = RS == 32 ? 8 : 4;  // l1: first low entry, after the cross neighbours
    auto active = [&](int q0, int n, int want, int* cnt) {  // the want-th active low bond of a class
      uint32_t m = 0;
      *cnt = 0;
      for (int q = q0; q < q0 + n; q++)
        if (__popc(a & g.low_mask[q]) == 1 && (*cnt)++ == want) m = g.low_mask[q];
      return m;
    };
    uint32_t flip = 0, v = 0;
    int n1, n2;
    if (e == 0) {
      for (int q = 0; q < g.n_cross; q++) v |= ((a >> g.cross_lo[q]) & 1u) << q;
    } else if (e == 1) {
      active(0, g.n_low1, -1, &n1);
      active(g.n_low1, g.n_low2, -1, &n2);
      v = (uint32_t)(n1 | (n2 << 8));
    } else if (e < l1) {
      if (e - 2 < g.n_cross) flip = 1u << g.cross_lo[e - 2];
    } else if (e < l1 + 10 || RS == 16) {
      flip = active(0, g.n_low1, e - l1, &n1);
    } else {
      flip = active(g.n_low1, g.n_low2, e - l1 - 10, &n2);
    }
    const uint32_t row = flip ? rank_lo(a ^ flip) + 1 : 0;
    const size_t o = ((size_t)g.cls_off[__popc(a)] + rank_lo(a)) * RS + e;
    for (int q = 0; q < 4; q++) t.rec[q][o] = (uint16_t)(e < 2 ? v : row * (16u << q));
    return;
  }
  if (i < 64) err[i] = 0;
  if (i < (1 << g.b)) {
    const uint32_t a = (uint32_t)i, r = rank_lo(a);
    const int pos = g.cls_off[__popc(a)] + (int)r;
    t.U_lo[pos] = (uint16_t)i;
    double d = 0.0;
    for (int q = 0; q < g.n_low1 + g.n_low2; q++) {
      const double J = q < g.n_low1 ? g.J1 : g.J2;
      d += J * g.Delta * (__popc(a & g.low_mask[q]) == 1 ? -0.25 : 0.25);
    }
    for (int q = 0; q < g.b; q++) d += g.h[q] * (((i >> q) & 1) ? 0.5 : -0.5);
    t.F_lo[i] = d;
    if (ty.kind >= 0) ty.put(pos, ty.alpha * d);
  }
  if (i < (1 << g.nh)) {
    const uint32_t grp = (uint32_t)i;
    const int pc = __popc(grp), n_lo = g.n_up - pc;
    int T = -1;
    double d = 0.0;
    if (valid(grp)) {
      T = rank_hi(grp);
      const int nhb = g.n_high1 + g.n_high2;
      for (int q = 0; q < nhb; q++) {
        const double J = q < g.n_high1 ? g.J1 : g.J2;
        d += J * g.Delta * (__popc(grp & g.high_mask[q]) == 1 ? -0.25 : 0.25);
      }
      for (int q = 0; q < g.nh; q++) d += g.h[g.b + q] * (((i >> q) & 1) ? 0.5 : -0.5);
      const int pos = cs.v[pc] + (int)rank_lo(grp);  // among the nh-bit strings of its popcount
      t.order[pos] = i;
      GroupRec* r = t.grec + pos;
      r->r0 = T;
      r->n_g = (int)B[g.b][n_lo];
      r->cls_base = g.cls_off[n_lo];
      int cnt = 0, cnt1 = 0, need = 0;
      for (int k = 0; k < nhb; k++)
        if (__popc(grp & g.high_mask[k]) == 1) {
          cnt++;
          if (k < g.n_high1) cnt1++;
        }
      r->n_hn = cnt;
      r->n_hn1 = cnt1;
      for (int k = 0; k < g.n_cross; k++)
        if (!((grp >> g.cross_hi[k]) & 1)) need |= 1 << k;  // the low bit must differ from the high bit
      r->need_mask = need;
      r->pad0 = r->pad1 = 0;
      if (ty.kind >= 0) ty.put((1 << g.b) + pos, ty.alpha * (d - ty.beta));
    }
    t.T_hi[i] = T;
    t.F_hi[i] = d;
  }
  if (i < (1 << g.n_cross)) {
    double d = 0.0;
    for (int k = 0; k < g.n_cross; k++) {
      const double J = g.cross_cls[k] == 1 ? g.J1 : g.J2;
      d += J * g.Delta * (((i >> k) & 1) ? -0.25 : 0.25);
    }
    t.C_x[i] = d;
    if (ty.kind >= 0) ty.put((1 << g.b) + g.n_groups + i, ty.alpha * d);
  }
}

// -------------------------------------------------------- bounded waits
// Iteration cap of the grid barrier's waits; a wait that runs out makes the
// kernel stop and the call return POLFED_ETIMEOUT.  polfed_set_wait_limit
// lowers the cap for tests.
constexpr uint32_t kBarrierWaitPolls = 1u << 24;
static std::atomic<uint32_t> g_wait_limit{0};
static uint32_t wait_cap(uint32_t dflt) {
  const uint32_t v = g_wait_limit.load();
  return v == 0 ? dflt : std::min(v, dflt);
}

// ------------------------------------------------------ slice conversions
template <class NT>
struct Conv;
template <>
struct Conv<RF32> {
  static __device__ __forceinline__ float from_d(double v) { return (float)v; }
  static __device__ __forceinline__ float from_f(float v) { return v; }
  static __device__ __forceinline__ double to_d(float v) { return (double)v; }
  static __device__ __forceinline__ float to_f(float v) { return v; }
  static __device__ __forceinline__ float mul(float c, float v) { return c * v; }
  static __device__ __forceinline__ float zero() { return 0.f; }
};
template <>
struct Conv<RF64> {
  static __device__ __forceinline__ double from_d(double v) { return v; }
  static __device__ __forceinline__ double from_f(float v) { return (double)v; }
  static __device__ __forceinline__ double to_d(double v) { return v; }
  static __device__ __forceinline__ float to_f(double v) { return (float)v; }
  static __device__ __forceinline__ double mul(double c, double v) { return c * v; }
  static __device__ __forceinline__ double zero() { return 0.0; }
};
template <>
struct Conv<RDF> {
  static __device__ __forceinline__ float2 from_d(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
  }
  static __device__ __forceinline__ float2 from_f(float v) { return make_float2(v, 0.f); }
  static __device__ __forceinline__ double to_d(float2 v) { return (double)v.x + (double)v.y; }
  static __device__ __forceinline__ float to_f(float2 v) { return v.x + v.y; }
  static __device__ __forceinline__ float2 mul(float2 c, float2 v) { return df_mul(c, v); }
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
};

template <class S>
union V16 {
  int4 i;
  S s[16 / sizeof(S)];
};

// a chunk's elements as they are stored (float-float: both hi, then both lo)
template <class NT>
__device__ __forceinline__ int4 stored(const int4& v) {
  if constexpr (std::is_same<NT, RDF>::value) return make_int4(v.x, v.z, v.y, v.w);
  return v;
}

template <class NT>
__device__ __forceinline__ typename NT::C col_cx_scale(const float* colscale, int c, typename NT::C cscale) {
  if constexpr (std::is_same<NT, RF32>::value) {
    if (colscale) return colscale[c];
  }
  return cscale;
}

// Columns [col0, col0 + ncols) of a row-major ABI block (ld elements per row)
// into consecutive slice buffers of W columns each (`stride` elements apart;
// the last one zero padded), optionally also a scaled copy; records max |x| in
// flag[0] (as float bits).  One thread per 16-byte chunk of a slice row; VIN
// input elements per load where the block's alignment allows it.
template <class NT, class In, int VIN>
__global__ void k_slice_in(const In* __restrict__ in, int64_t dim, int ld, int col0, int ncols, int W, int nsl,
                           int64_t stride, typename NT::S* xs, typename NT::S* a_scaled, typename NT::C cscale,
                           float* flag, const float* colscale, int64_t colstride) {
  using S = typename NT::S;
  constexpr int VEC = 16 / sizeof(S);
  float mx = 0.f;
  const int cps = W / VEC, cpr = cps * nsl;  // chunks per slice row, per block row
  const int64_t n = dim * cpr;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = n < (1ll << 31) ? (int64_t)((uint32_t)e / (uint32_t)cpr) : e / cpr;
    const int q = (int)(e - r * cpr), sl = q / cps, c = (q - sl * cps) * VEC, cc = sl * W + c;
    In raw[VEC];
    const In* src = in + r * ld + col0 + cc;
    if (cc + VEC <= ncols) {
#pragma unroll
      for (int v = 0; v < VEC; v += VIN) {
        struct alignas(VIN * sizeof(In)) Pack {
          In x[VIN];
        };
        const Pack p = *reinterpret_cast<const Pack*>(src + v);
#pragma unroll
        for (int u = 0; u < VIN; u++) raw[v + u] = p.x[u];
      }
    } else {
#pragma unroll
      for (int v = 0; v < VEC; v++) raw[v] = cc + v < ncols ? src[v] : In(0);
    }
    V16<S> o, a;
#pragma unroll
    for (int v = 0; v < VEC; v++) {
      if constexpr (sizeof(In) == 4)
        o.s[v] = Conv<NT>::from_f(raw[v]);
      else
        o.s[v] = Conv<NT>::from_d(raw[v]);
      mx = fmaxf(mx, fabsf((float)raw[v]));
      if (a_scaled)
        a.s[v] = Conv<NT>::mul(col_cx_scale<NT>(colscale ? colscale + sl * colstride : nullptr, c + v, cscale), o.s[v]);
    }
    const int64_t d = sl * stride + r * W + c;
    if (xs) *reinterpret_cast<int4*>(xs + d) = stored<NT>(o.i);
    if (a_scaled) *reinterpret_cast<int4*>(a_scaled + d) = stored<NT>(a.i);
  }
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && flag) atomicMax(reinterpret_cast<int*>(flag), __float_as_int(mx));
}

// Slice buffers -> columns of a row-major ABI block; records max |y| in flag[1]
// and sets flag[2] (int) to 1 on a non-finite value.
template <class NT, class Out, int VOUT>
__global__ void k_slice_out(const typename NT::S* __restrict__ ys, int64_t dim, int W, int nsl, int64_t stride,
                            int ncols, Out* out, int ld, int col0, float* flag) {
  using S = typename NT::S;
  constexpr int VEC = 16 / sizeof(S);
  float mx = 0.f;
  int bad = 0;
  const int cps = W / VEC, cpr = cps * nsl;
  const int64_t n = dim * cpr;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = n < (1ll << 31) ? (int64_t)((uint32_t)e / (uint32_t)cpr) : e / cpr;
    const int q = (int)(e - r * cpr), sl = q / cps, c = (q - sl * cps) * VEC, cc = sl * W + c;
    if (cc >= ncols) continue;
    V16<S> u;
    u.i = stored<NT>(*reinterpret_cast<const int4*>(ys + sl * stride + r * W + c));  // its own inverse
    Out o[VEC];
#pragma unroll
    for (int v = 0; v < VEC; v++) {
      if constexpr (sizeof(Out) == 4)
        o[v] = Conv<NT>::to_f(u.s[v]);
      else
        o[v] = Conv<NT>::to_d(u.s[v]);
      if (cc + v < ncols) {
        if (!isfinite(o[v])) bad = 1;
        mx = fmaxf(mx, fabsf((float)o[v]));
      }
    }
    Out* dst = out + r * ld + col0 + cc;
    if (cc + VEC <= ncols) {
#pragma unroll
      for (int v = 0; v < VEC; v += VOUT) {
        struct alignas(VOUT * sizeof(Out)) Pack {
          Out x[VOUT];
        };
        Pack p;
#pragma unroll
        for (int w = 0; w < VOUT; w++) p.x[w] = o[v + w];
        *reinterpret_cast<Pack*>(dst + v) = p;
      }
    } else {
#pragma unroll
      for (int v = 0; v < VEC; v++)
        if (cc + v < ncols) dst[v] = o[v];
    }
  }
  for (int o = 16; o; o >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if ((threadIdx.x & 31) == 0 && flag) {
    atomicMax(reinterpret_cast<int*>(flag) + 1, __float_as_int(mx));
    if (bad) atomicExch(reinterpret_cast<int*>(flag) + 2, 1);
  }
}

// Typed, alpha/beta-scaled diagonal tables: F_lo by class order | F_hi in
// schedule order | C_x.
__global__ void k_typed(const HamTables t, int nlo, int ngr, int ncx, TypedOut ty) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nlo + ngr + ncx) return;
  double v;
  if (i < nlo)
    v = ty.alpha * t.F_lo[t.U_lo[i]];
  else if (i < nlo + ngr)
    v = ty.alpha * (t.F_hi[t.order[i - nlo]] - ty.beta);
  else
    v = ty.alpha * t.C_x[i - nlo - ngr];
  ty.put(i, v);
}

// --------------------------------------------------------------- host side
size_t elem_bytes(int kind) { return kind == POLFED_F32 ? 4 : 8; }
int slice_width(int kind, int lpr) { return (int)(16 / elem_bytes(kind)) * lpr; }

int choose_lpr(int kind, int n_b) {
  const int vec = (int)(16 / elem_bytes(kind));
  int lpr = 1;
  while (lpr < 8 && vec * lpr < n_b) lpr *= 2;
  return lpr;
}

static int lpr_index(int lpr) { return lpr == 8 ? 3 : (lpr == 4 ? 2 : (lpr == 2 ? 1 : 0)); }

// Offsets of the tables of a geometry in one allocation.
struct PlanLayout {
  size_t Ulo, Thi, Ord, Flo, Fhi, Cx, Grp, Err, Rec, total;
  size_t rec1;  // bytes of one record table
  explicit PlanLayout(const HamGeometry& g) {
    const size_t nlo = (size_t)1 << g.b, nhi = (size_t)1 << g.nh, ncx = (size_t)1 << g.n_cross;
    total = 0;
    auto carve = [&](size_t n) {
      const size_t o = total;
      total += (n + 255) & ~(size_t)255;
      return o;
    };
    Ulo = carve(nlo * 2);
    Thi = carve(nhi * 4);
    Ord = carve(nhi * 4);
    Flo = carve(nlo * 8);
    Fhi = carve(nhi * 8);
    Cx = carve(ncx * 8);
    Grp = carve((size_t)g.n_groups * sizeof(GroupRec));
    Err = carve(256);
    rec1 = (nlo * (size_t)g.rec_stride * 2 + 255) & ~(size_t)255;
    Rec = carve(4 * rec1);
  }
};

static int typed_out(int kind, double e_lo, double e_hi, void* dst, TypedOut* ty) {
  if (kind < 0 || kind > 2) return fail(POLFED_EINVAL, "bad dtype");
  *ty = TypedOut{kind, 1.0, 0.0, dst};
  if (!(e_lo == 0.0 && e_hi == 0.0)) {
    if (!(e_hi > e_lo)) return fail(POLFED_EINVAL, "need e_lo < e_hi");
    ty->alpha = 2.0 / (e_hi - e_lo);
    ty->beta = 0.5 * (e_hi + e_lo);
  }
  return POLFED_OK;
}

// Point the plan's tables into `base` and enqueue the kernels that fill them.
int HamPlan::bind(char* base, cudaStream_t s, int kind, double e_lo, double e_hi, void* typed_dst) {
  const PlanLayout lay(geo);
  tab.U_lo = (uint16_t*)(base + lay.Ulo);
  tab.T_hi = (int32_t*)(base + lay.Thi);
  tab.order = (int32_t*)(base + lay.Ord);
  tab.F_lo = (double*)(base + lay.Flo);
  tab.F_hi = (double*)(base + lay.Fhi);
  tab.C_x = (double*)(base + lay.Cx);
  tab.grec = (GroupRec*)(base + lay.Grp);
  for (int i = 0; i < 4; i++) tab.rec[i] = (uint16_t*)(base + lay.Rec + i * lay.rec1);
  err_flag = (int*)(base + lay.Err);
  bar_base = 0;
  TypedOut ty{-1, 1.0, 0.0, nullptr};
  if (kind >= 0) {
    PF_CHECK(typed_out(kind, e_lo, e_hi, typed_dst, &ty));
    typed[kind] = typed_dst;
    typed_ok[kind] = true;
    typed_lo[kind] = e_lo;
    typed_hi[kind] = e_hi;
  }
  const int n_main = (std::max({64, 1 << geo.b, 1 << geo.nh, 1 << geo.n_cross}) + kTableThreads - 1) / kTableThreads;
  const int n_rec = ((geo.rec_stride << geo.b) + ((kMaxHigh + 8) << geo.nh) + kTableThreads - 1) / kTableThreads;
  k_tables<<<n_main + n_rec, kTableThreads, 0, s>>>(geo, class_starts(geo), tab, err_flag, ty, n_main * kTableThreads);
  PF_CUDA(cudaGetLastError());
  return POLFED_OK;
}

static size_t typed_bytes_of(const HamGeometry& g) {
  return (((size_t)1 << g.b) + ((size_t)1 << g.n_cross) + (size_t)g.n_groups) * 8 + 512;
}

int HamPlan::init(const polfed_model* m, cudaStream_t s, bool stream_ordered, int b_override, int kind, double e_lo,
                  double e_hi) {
  release();
  upload_binomials();
  PF_CHECK(build_geometry(m, b_override, &geo));
  stream = s;
  stream_alloc = stream_ordered;
  const size_t bytes = PlanLayout(geo).total, all = bytes + (kind >= 0 ? typed_bytes_of(geo) : 0);
  if (stream_ordered)
    PF_CHECK(scratch_alloc(&dev, all, s));
  else
    PF_CUDA(device_malloc(&dev, all));
  dev_end = (char*)dev + all;
  return bind((char*)dev, s, kind, e_lo, e_hi, (char*)dev + bytes);
}

int HamPlan::prepare_typed(int kind, double e_lo, double e_hi) {
  if (kind < 0 || kind > 2) return fail(POLFED_EINVAL, "bad dtype");
  if (typed_ok[kind] && typed_lo[kind] == e_lo && typed_hi[kind] == e_hi) return POLFED_OK;
  if (!typed[kind]) {
    if (stream_alloc)
      PF_CHECK(scratch_alloc(&typed[kind], typed_bytes_of(geo), stream));
    else
      PF_CUDA(device_malloc(&typed[kind], typed_bytes_of(geo)));
  }
  typed_ok[kind] = false;
  TypedOut ty;
  PF_CHECK(typed_out(kind, e_lo, e_hi, typed[kind], &ty));
  const int nlo = 1 << geo.b, ncx = 1 << geo.n_cross, n = nlo + geo.n_groups + ncx;
  k_typed<<<(n + 255) / 256, 256, 0, stream>>>(tab, nlo, geo.n_groups, ncx, ty);
  PF_CUDA(cudaGetLastError());
  typed_ok[kind] = true;
  typed_lo[kind] = e_lo;
  typed_hi[kind] = e_hi;
  return POLFED_OK;
}

void HamPlan::release() {
  if (dev) {
    if (stream_alloc)
      cudaFreeAsync(dev, stream);
    else
      cudaFree(dev);
  }
  for (int k = 0; k < 3; k++) {
    if (typed[k] && !(typed[k] >= dev && typed[k] < dev_end)) {  // not part of dev
      if (stream_alloc)
        cudaFreeAsync(typed[k], stream);
      else
        cudaFree(typed[k]);
    }
    typed[k] = nullptr;
    typed_ok[k] = false;
  }
  dev = nullptr;
}

static void split_df(double v, float2& o) {
  o.x = (float)v;
  o.y = (float)(v - (double)o.x);
}

// v in the constant type of `kind`, in its own 8 bytes
static double typed_const(int kind, double v) {
  if (kind == POLFED_F64) return v;
  double out = 0.0;
  if (kind == POLFED_F32) {
    const float f = (float)v;
    memcpy(&out, &f, 4);
  } else {
    float2 f;
    split_df(v, f);
    memcpy(&out, &f, 8);
  }
  return out;
}

// The operator part of a job (buffers, order and coefficients are the caller's).
static StepJob make_job(const HamPlan& p, int kind, int lpr, double invD) {
  const HamGeometry& g = p.geo;
  StepJob j{};
  const size_t es = kind == POLFED_F32 ? 4 : 8, nlo = (size_t)1 << g.b;
  const char* t = (const char*)p.typed[kind];
  j.rec = p.tab.rec[lpr_index(lpr)];
  j.grec = p.tab.grec;
  j.Fc = t;
  j.Fhi = t + nlo * es;
  j.Cx = t + (nlo + (size_t)g.n_groups) * es;
  const double alpha = (p.typed_lo[kind] == 0.0 && p.typed_hi[kind] == 0.0) ? 1.0 : 2.0 / (p.typed_hi[kind] - p.typed_lo[kind]);
  const double o1 = alpha * 0.5 * g.J1, o2 = alpha * 0.5 * g.J2;
  // float-float keeps the couplings apart from cH; FP32 / FP64 take their product
  const double fi = kind == POLFED_DF64 ? 1.0 : 2.0, fl = kind == POLFED_DF64 ? 1.0 : invD;
  j.con[kConS1] = typed_const(kind, fi * o1);
  j.con[kConS2] = typed_const(kind, fi * o2);
  j.con[kConS1Last] = typed_const(kind, fl * o1);
  j.con[kConS2Last] = typed_const(kind, fl * o2);
  j.con[kConInvD] = typed_const(kind, invD);
  j.n_groups = g.n_groups;
  j.n_cross = g.n_cross;
  for (int k = 0; k < g.n_cross; k++)
    if (g.cross_cls[k] == 2) j.c2mask |= 1 << k;
  return j;
}

static int check_operator(const HamPlan& p, int kind) {
  const bool j2 = p.geo.rec_stride == 32;
  if (kind < 0 || kind > 2 || !p.typed_ok[kind])
    return fail(POLFED_EINVAL, "operator tables not prepared for this precision");
  if (p.geo.n_cross > (j2 ? 6 : 2)) return fail(POLFED_EINVAL, "more cross bonds than the kernel handles");
  return POLFED_OK;
}

// Launch the steps of `run`: the grid size (> 0), or a negative status.
static int launch_rows(const StepRun& run, int kind, int lpr, bool j2, StepMode mode, int max_group, int64_t items,
                       bool cooperative, cudaStream_t s, int max_teams = kMaxTeams) {
  switch (kind) {
    case POLFED_F32: return launch_rows_f32(run, lpr, j2, mode, max_group, items, cooperative, max_teams, s);
    case POLFED_F64: return launch_rows_f64(run, lpr, j2, mode, max_group, items, cooperative, max_teams, s);
    case POLFED_DF64: return launch_rows_df(run, lpr, j2, mode, max_group, items, cooperative, max_teams, s);
  }
  return fail(POLFED_EINVAL, "bad dtype");
}

// A cooperative grid fills the GPU and its CTAs wait for one another, so only
// one is in flight per device: a thread holds a turn from a launch to its
// completion.  A call of many launches gives its turn up about every
// kTurnSeconds if another thread waits, and a thread that had the last turn lets
// the other go first, so that a short call does not wait for the end of a long
// one.  What needs no turn (event creation, reading the error flag) stays outside
// it, and turns are not handed over in the order of asking: either leaves the GPU
// idle, 3% of a run of 64 realizations on as many threads.
class Turn {
  struct Queue {
    std::mutex mu;
    std::atomic<int> waiting{0};
    std::atomic<uint64_t> given{0};
  };
  static Queue& queue(int dev) {
    static Queue q[64];
    return q[dev];
  }
  static uint64_t& last(int dev) {
    static thread_local uint64_t l[64];
    return l[dev];
  }
  static int device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev & 63;
  }
  Queue& q_;
  uint64_t& last_;  // this thread's latest turn

  void take() {
    while (q_.waiting.load() > 0 && q_.given.load() == last_) std::this_thread::yield();
    q_.waiting++;
    q_.mu.lock();
    q_.waiting--;
    last_ = ++q_.given;
  }

 public:
  explicit Turn(int dev = device()) : q_(queue(dev)), last_(last(dev)) { take(); }
  ~Turn() { q_.mu.unlock(); }
  Turn(const Turn&) = delete;
  Turn& operator=(const Turn&) = delete;
  void again() {  // between two launches of a long call, none in flight
    if (q_.waiting.load() == 0) return;
    q_.mu.unlock();
    take();
  }
};

constexpr double kTurnSeconds = 0.1;        // of a filter or of moments: the steps of a turn, in one or more launches
constexpr double kBatchTurnSeconds = 0.25;  // of a batched filter: one launch

// An upper estimate of a step's seconds, by the bytes of its slices (measured: 1.7 to 3.6 TB/s in FP32 and
// float-float; half of that and less in FP64, whose pipe bounds it) and by the rows of the busiest team (0.1 to 0.2 us
// each of 128 bytes).  Turns are cut by it.  The end of one costs up to 0.2 ms: an L = 22 run's filters take 56.3 to
// 56.7 s with launches of 448 steps, 56.8 with turns of 196 and 56.9 with turns of 138.
static double step_seconds(int kind, double row_bytes, int64_t items, int max_group) {
  const int64_t teams = 152 * kMaxTeams, rounds = (items + teams - 1) / teams;
  const double rate = kind == POLFED_F64 ? 0.5e12 : 1.5e12;
  return 5e-6 + std::max(4.0 * row_bytes / rate, 0.4e-6 * (double)rounds * max_group);
}

// ------------------------------------------------------------ filter engine
// A block is filtered in column slices of W columns; `ns` slices run in one
// launch: as many as keep their three buffers (x, b_{k+1}, b_{k+2}) in L2
// together, so that small problems fill the GPU and large ones keep the gather
// source resident.
struct FilterShape {
  int lpr, W, nsl, ns;
  size_t slice;  // bytes of one slice buffer
};

static FilterShape slices_of(const HamGeometry& g, int kind, int n_b, size_t limit, int lpr) {
  FilterShape f;
  f.lpr = lpr;
  f.W = slice_width(kind, f.lpr);
  f.nsl = (n_b + f.W - 1) / f.W;
  f.slice = ((size_t)g.dim * f.W * elem_bytes(kind) + 255) & ~(size_t)255;
  f.ns = (int)std::max<size_t>(1, std::min<size_t>((size_t)f.nsl, limit / (3 * f.slice)));
  return f;
}

static FilterShape filter_shape(const HamGeometry& g, int kind, int n_b, size_t limit) {
  return slices_of(g, kind, n_b, limit, choose_lpr(kind, n_b));
}

// The FP32 filter takes 64-byte rows where a slice of 128-byte ones, the gather
// source, is beyond L2 (346 MB at L = 24) and rows gather few neighbours: XXZ,
// 32 columns, K = 40: 18.5 ms with 128 bytes, 17.0 with 64 (21.2 with 32).  Within L2
// (L = 22) they cost 7%; J1-J2 gains nothing (38.1 and 38.3 ms at L = 24).
static FilterShape filter_rows(const HamGeometry& g, int kind, int n_b, size_t limit) {
  const FilterShape f = filter_shape(g, kind, n_b, limit);
  if (kind == POLFED_F32 && f.lpr == 8 && f.slice > ((size_t)160 << 20) && g.rec_stride == 16)
    return slices_of(g, kind, n_b, limit, 4);
  return f;
}

// The launches of a block: sets of ns slices, and the columns that do not fill
// the last slice by themselves in a narrower one.  Small problems, whose slices
// all run together, keep the padded slice: it shares their launch.  L = 20,
// J1-J2, FP32, 37 columns, K = 48: 4.33 ms as two slices of 32, 3.19 as one and
// one of 8 (2.05 and 0.92 in the steps).
struct SlicePart {
  FilterShape f;
  int ns, s0, col0, ncols;  // slices s0.. of columns col0..
};

static std::vector<SlicePart> slice_parts(const HamGeometry& g, int kind, const FilterShape& f, int n_b) {
  std::vector<SlicePart> parts;
  const int rem = n_b % f.W;
  const bool split = f.nsl > f.ns && rem > 0 && choose_lpr(kind, rem) < f.lpr;
  const int nfull = f.nsl - (split ? 1 : 0);
  for (int s0 = 0; s0 < nfull; s0 += f.ns) {
    const int ns = std::min(f.ns, nfull - s0), col0 = s0 * f.W;
    parts.push_back(SlicePart{f, ns, s0, col0, std::min(ns * f.W, n_b - col0)});
  }
  if (split) {
    FilterShape t = filter_shape(g, kind, rem, 0);
    parts.push_back(SlicePart{t, 1, nfull, nfull * f.W, rem});
  }
  return parts;
}

size_t filter_scratch_bytes(const HamPlan& plan, int kind, int n_b) {
  const FilterShape f = filter_shape(plan.geo, kind, n_b, plan.slice_set);
  return 3 * (size_t)f.ns * f.slice + 256;
}

struct SliceBufs {
  char *xs, *ba, *bb;
  SliceBufs(const FilterScratch& scr, const FilterShape& f)
      : xs((char*)scr.xs), ba(xs + f.ns * f.slice), bb(ba + f.ns * f.slice) {}
};

static int carve_scratch(FilterScratch& scr, const FilterShape& f) {
  if (!scr.xs || scr.bytes < 3 * (size_t)f.ns * f.slice + 256) return fail(POLFED_ENOMEM, "filter scratch too small");
  scr.flag = (float*)((char*)scr.xs + 3 * (size_t)f.ns * f.slice);
  return POLFED_OK;
}

static int conv_grid(int64_t chunks) { return (int)std::max<int64_t>(1, std::min<int64_t>((chunks + 255) / 256, 152 * 16)); }

// elements of `es` bytes per vector access at p, p + ld, ... (1, 2 or 4)
static int vec_elems(const void* p, int64_t ld, size_t es) {
  for (int v = (int)(16 / es); v > 1; v /= 2)
    if ((uintptr_t)p % (v * es) == 0 && ld % v == 0) return v;
  return 1;
}

template <class NT, class In>
static int slice_in_t(const void* in, int64_t dim, int ld, int col0, int ncols, const FilterShape& f, int nsl, void* xs,
                      void* as, double scale, float* flag, cudaStream_t s, const float* colscale, int64_t colstride) {
  typename NT::C cs;
  if constexpr (std::is_same<NT, RDF>::value)
    split_df(scale, cs);
  else
    cs = (typename NT::C)scale;
  using S = typename NT::S;
  constexpr int VEC = 16 / sizeof(S);
  const int64_t st = (int64_t)(f.slice / sizeof(S));
  const int grid = conv_grid(dim * (f.W / VEC) * nsl);
  const In* p = (const In*)in;
  const int v = std::min(VEC, vec_elems(p + col0, ld, sizeof(In)));
#define PF_IN(V_) \
  k_slice_in<NT, In, V_><<<grid, 256, 0, s>>>(p, dim, ld, col0, ncols, f.W, nsl, st, (S*)xs, (S*)as, cs, flag, colscale, colstride)
  if (v >= 4) {
    if constexpr (VEC >= 4) PF_IN(4);
  } else if (v == 2) {
    PF_IN(2);
  } else {
    PF_IN(1);
  }
#undef PF_IN
  PF_CUDA(cudaGetLastError());
  count_launch();
  return POLFED_OK;
}

static int slice_in(int kind, int abi_kind, const void* in, int64_t dim, int ld, int col0, int ncols,
                    const FilterShape& f, int nsl, void* xs, void* as, double scale, float* flag, cudaStream_t s,
                    const float* colscale = nullptr, int64_t colstride = 0) {
#define PF_SI(NT_)                                                                                                    \
  return abi_kind == POLFED_F32                                                                                       \
             ? slice_in_t<NT_, float>(in, dim, ld, col0, ncols, f, nsl, xs, as, scale, flag, s, colscale, colstride)  \
             : slice_in_t<NT_, double>(in, dim, ld, col0, ncols, f, nsl, xs, as, scale, flag, s, colscale, colstride)
  switch (kind) {
    case POLFED_F32: PF_SI(RF32);
    case POLFED_F64: PF_SI(RF64);
    default: PF_SI(RDF);
  }
#undef PF_SI
}

template <class NT, class Out>
static int slice_out_t(const void* ys, int64_t dim, const FilterShape& f, int nsl, int ncols, void* out, int ld, int col0,
                       float* flag, cudaStream_t s) {
  using S = typename NT::S;
  constexpr int VEC = 16 / sizeof(S);
  const int64_t st = (int64_t)(f.slice / sizeof(S));
  const int grid = conv_grid(dim * (f.W / VEC) * nsl);
  Out* p = (Out*)out;
  const int v = std::min(VEC, vec_elems(p + col0, ld, sizeof(Out)));
#define PF_OUT(V_) k_slice_out<NT, Out, V_><<<grid, 256, 0, s>>>((const S*)ys, dim, f.W, nsl, st, ncols, p, ld, col0, flag)
  if (v >= 4) {
    if constexpr (VEC >= 4) PF_OUT(4);
  } else if (v == 2) {
    PF_OUT(2);
  } else {
    PF_OUT(1);
  }
#undef PF_OUT
  PF_CUDA(cudaGetLastError());
  count_launch();
  return POLFED_OK;
}

static int slice_out(int kind, int abi_kind, const void* ys, int64_t dim, const FilterShape& f, int nsl, int ncols,
                     void* out, int ld, int col0, float* flag, cudaStream_t s) {
#define PF_SO(NT_)                                                                                  \
  return abi_kind == POLFED_F32 ? slice_out_t<NT_, float>(ys, dim, f, nsl, ncols, out, ld, col0, flag, s) \
                                : slice_out_t<NT_, double>(ys, dim, f, nsl, ncols, out, ld, col0, flag, s)
  switch (kind) {
    case POLFED_F32: PF_SO(RF32);
    case POLFED_F64: PF_SO(RF64);
    default: PF_SO(RDF);
  }
#undef PF_SO
}

// Device time of the step launches of storage kind `kind` between start() and
// stop(), by a pair of CUDA events on the launching stream; credited to the timed
// counters.  Only what has to happen within a turn is done by start() and wait().
struct StepTimer {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaStream_t s;
  int kind;
  int64_t n0 = 0;
  double b0 = 0.0;
  StepTimer(cudaStream_t st, int k) : s(st), kind(k) {
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) drop();
  }
  void start() {
    n0 = counters().all_launches[kind];
    b0 = counters().all_alg_bytes[kind];
    if (e0) cudaEventRecord(e0, s);
  }
  int wait() {  // for the launches
    if (!e0) {
      PF_CUDA(cudaStreamSynchronize(s));
      return POLFED_OK;
    }
    PF_CUDA(cudaEventRecord(e1, s));
    PF_CUDA(cudaEventSynchronize(e1));
    return POLFED_OK;
  }
  int credit() {
    if (!e0) return POLFED_OK;
    float ms = 0.f;
    PF_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    Counters& c = counters();
    const int64_t n = c.all_launches[kind] - n0;
    const double b = c.all_alg_bytes[kind] - b0;
    c.step_gpu_s += 1e-3 * ms;
    c.step_launches += n;
    c.step_alg_bytes += b;
    c.kind_gpu_s[kind] += 1e-3 * ms;
    c.kind_launches[kind] += n;
    c.kind_alg_bytes[kind] += b;
    return POLFED_OK;
  }
  int stop() {
    PF_CHECK(wait());
    return credit();
  }
  void drop() {
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    e0 = e1 = nullptr;
  }
  ~StepTimer() { drop(); }
};

// A step kernel whose bounded wait expired leaves plan.err_flag set.
static int check_timeout(HamPlan& plan, cudaStream_t s) {
  int e = 0;
  PF_CUDA(cudaMemcpyAsync(&e, plan.err_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  if (e) {
    cudaMemsetAsync(plan.err_flag, 0, 256, s);
    plan.bar_base = 0;
    return fail(POLFED_ETIMEOUT, "a bounded device wait in the step kernel expired");
  }
  return POLFED_OK;
}

// The parts of a cooperative run over `ns` slices that its mode does not change.
static int cooperative_run(HamPlan& plan, int kind, const FilterShape& f, int ns, double invD, const SliceBufs& b,
                           cudaStream_t s, StepRun* run) {
  PF_CHECK(check_operator(plan, kind));
  *run = StepRun{};
  run->one = make_job(plan, kind, f.lpr, invD);
  run->one.xs = b.xs;
  run->one.ba = b.ba;
  run->one.bb = b.bb;
  run->n_jobs = ns;
  run->stride = (int64_t)f.slice;
  run->bar = (unsigned*)(plan.err_flag + 16);
  run->err = plan.err_flag;
  run->cap = wait_cap(kBarrierWaitPolls);
  return POLFED_OK;
}

// The Clenshaw steps k = K-1..1 and the final step of Eq. (2) of `ns` slices
// (b_K in ba, X in xs), several steps to a cooperative launch: K = 200 at
// L = 14 costs one launch instead of 200.  coef(n) gives c_n; col (device) the
// per-column rows instead.  The result is in *res.
template <class Coef>
static int run_steps(HamPlan& plan, int kind, const FilterShape& f, int ns, const Coef& coef, int K, double invD,
                     const float* col, int64_t colstride, int colw, const SliceBufs& b, cudaStream_t s, char** res) {
  StepRun run;
  PF_CHECK(cooperative_run(plan, kind, f, ns, invD, b, s, &run));
  const bool j2 = plan.geo.rec_stride == 32;
  run.one.K = K;
  run.one.colcx = col;
  run.colstride = colstride;
  run.one.colw = colw;
  const int64_t items = (int64_t)plan.geo.n_groups * ns;
  const double row = (double)plan.geo.dim * f.W * elem_bytes(kind) * ns;
  const int turn_steps = std::max(1, (int)(kTurnSeconds / step_seconds(kind, row, items, plan.geo.max_group)));
  StepTimer tm(s, kind);
  {
    Turn turn;
    tm.start();  // within the turn: the time of these launches, not of other threads' before them
    for (int st = 0, t0 = 0; st < K; st = run.st1) {
      if (st == t0 + turn_steps) {
        PF_CHECK(tm.stop());
        PF_CHECK(check_timeout(plan, s));
        turn.again();
        tm.start();
        t0 = st;
      }
      run.st0 = st;
      run.st1 = std::min({K, st + kParamSteps, t0 + turn_steps});
      run.bar_base = plan.bar_base;
      double alg = 0.0;
      for (int q = run.st0; q < run.st1; q++) {
        const int k = K - 1 - q;
        double c = col ? 1.0 : coef(k);
        if (!col) {
          if (k == 0) c *= invD;
          run.cx[q - st] = typed_const(kind, c);
        }
        alg += row * (3.0 + (c != 0.0 ? 1.0 : 0.0));
      }
      const int grid = launch_rows(run, kind, f.lpr, j2, col ? kFilterCols : kFilter, plan.geo.max_group, items, true, s);
      if (grid < 0) return grid;
      plan.bar_base += (unsigned)grid * (unsigned)(run.st1 - run.st0 - 1);
      count_step(kind, alg);
    }
    PF_CHECK(tm.wait());
  }
  PF_CHECK(tm.credit());
  PF_CHECK(check_timeout(plan, s));
  *res = (K % 2 == 0) ? b.ba : b.bb;
  return POLFED_OK;
}

template <class Coef>
static int filter_slices(HamPlan& plan, int kind, const FilterShape& f, const Coef& coef, int K, double invD,
                         const float* d_col, const void* in, void* out, int n_b, int abi_kind, FilterScratch& scr,
                         cudaStream_t s) {
  PF_CHECK(carve_scratch(scr, f));
  const int64_t dim = plan.geo.dim;
  const int64_t colstride = d_col ? (int64_t)(K + 1) * f.W : 0;
  PF_CUDA(cudaMemsetAsync(scr.flag, 0, 16, s));
  for (const SlicePart& p : slice_parts(plan.geo, kind, f, n_b)) {
    const SliceBufs b(scr, p.f);
    if (K == 0) {
      PF_CHECK(slice_in(kind, abi_kind, in, dim, n_b, p.col0, p.ncols, p.f, p.ns, nullptr, b.ba, coef(0) * invD, scr.flag, s));
      PF_CHECK(slice_out(kind, abi_kind, b.ba, dim, p.f, p.ns, p.ncols, out, n_b, p.col0, scr.flag, s));
      continue;
    }
    const float* col = d_col ? d_col + p.s0 * colstride : nullptr;
    // b_K = c_K X (in ba); b_{K+1} = 0 is not read by the first step
    PF_CHECK(slice_in(kind, abi_kind, in, dim, n_b, p.col0, p.ncols, p.f, p.ns, b.xs, b.ba, col ? 1.0 : coef(K), scr.flag,
                      s, col ? col + (size_t)K * f.W : nullptr, colstride));
    char* res = nullptr;
    PF_CHECK(run_steps(plan, kind, p.f, p.ns, coef, K, invD, col, colstride, f.W, b, s, &res));
    PF_CHECK(slice_out(kind, abi_kind, res, dim, p.f, p.ns, p.ncols, out, n_b, p.col0, scr.flag, s));
  }
  return POLFED_OK;
}

int filter_block(HamPlan& plan, int kind, const double* c, int K, double invD, const void* in, void* out, int n_b,
                 int abi_kind, FilterScratch& scr, cudaStream_t s) {
  const FilterShape f = filter_rows(plan.geo, kind, n_b, plan.slice_set);
  return filter_slices(plan, kind, f, [c](int n) { return c[n]; }, K, invD, nullptr, in, out, n_b, abi_kind, scr, s);
}

int filter_block_cols(HamPlan& plan, const float* d_coef, int K, const void* in, void* out, int n_b, int abi_kind,
                      FilterScratch& scr, cudaStream_t s) {
  if (K < 1) return fail(POLFED_EINVAL, "per-column filter needs K >= 1");
  const FilterShape f = filter_shape(plan.geo, POLFED_F32, n_b, plan.slice_set);
  return filter_slices(plan, POLFED_F32, f, [](int) { return 1.0; }, K, 1.0, d_coef, in, out, n_b, abi_kind, scr, s);
}

size_t moment_scratch_bytes(const HamPlan& plan, int kind, int n_b) {
  if (kind != POLFED_DF64) return 0;
  const FilterShape f = filter_shape(plan.geo, kind, n_b, plan.slice_set);
  return f.ns * f.slice;
}

// mu[2 st + {0, 1}] += the sums of step st0 + st, in CTA order (one warp a step)
__global__ void k_moment_sums(const double2* __restrict__ part, int n_cta, double* __restrict__ mu) {
  double2 v = make_double2(0.0, 0.0);
  for (int i = threadIdx.x; i < n_cta; i += 32) {
    const double2 u = part[(size_t)blockIdx.x * n_cta + i];
    v.x += u.x;
    v.y += u.y;
  }
  for (int o = 16; o; o >>= 1) {
    v.x += __shfl_xor_sync(~0u, v.x, o);
    v.y += __shfl_xor_sync(~0u, v.y, o);
  }
  if (threadIdx.x == 0) {
    mu[2 * blockIdx.x] += v.x;
    mu[2 * blockIdx.x + 1] += v.y;
  }
}

// The recurrence stays in slice layout from its first step to its last.
// L = 18, 16 columns, float-float with t_n in FP64: a pair of moments took 53 us
// as five launches (slice copies in and out, H~, update, sum), now 22, of which
// about a third is the FP64 pipe (conversions, update and sums of 778k elements).
int moment_steps(HamPlan& plan, int kind, const void* in, int n_b, int half, void* t_odd, void* part, size_t part_bytes,
                 double* mu, FilterScratch& scr, cudaStream_t s) {
  const FilterShape f = filter_shape(plan.geo, kind, n_b, plan.slice_set);
  PF_CHECK(carve_scratch(scr, f));
  const int64_t dim = plan.geo.dim;
  const int abi = kind == POLFED_F32 ? POLFED_F32 : POLFED_F64;
  const bool j2 = plan.geo.rec_stride == 32;
  PF_CUDA(cudaMemsetAsync(mu, 0, (size_t)2 * half * sizeof(double), s));
  for (const SlicePart& p : slice_parts(plan.geo, kind, f, n_b)) {
    const SliceBufs b(scr, p.f);
    PF_CHECK(slice_in(kind, abi, in, dim, n_b, p.col0, p.ncols, p.f, p.ns, b.ba, nullptr, 0.0, nullptr, s));
    if (kind == POLFED_DF64)
      PF_CHECK(slice_in(POLFED_F64, abi, in, dim, n_b, p.col0, p.ncols, p.f, p.ns, b.xs, nullptr, 0.0, nullptr, s));
    StepRun run;
    PF_CHECK(cooperative_run(plan, kind, p.f, p.ns, 1.0, b, s, &run));
    run.one.K = half;
    run.one.low_first = f.lpr == 8 && plan.geo.max_group >= 32;
    run.one.ta = b.xs;
    run.one.tb = (char*)t_odd;
    run.part = (double2*)part;
    const int64_t items = (int64_t)plan.geo.n_groups * p.ns;
    const double row = (double)dim * p.f.W * elem_bytes(kind) * p.ns;
    const int64_t per_step = std::min<int64_t>(items, kMaxMomentCtas) * sizeof(double2);
    const int launch_steps = (int)std::max<int64_t>(1, std::min<int64_t>(kParamSteps, (int64_t)part_bytes / per_step));
    const int turn_steps = std::max(1, (int)(kTurnSeconds / step_seconds(kind, row, items, plan.geo.max_group)));
    {
      Turn turn;
      for (int st = 0, t0 = 0; st < half; st = run.st1) {
        if (st == t0 + turn_steps) {
          PF_CHECK(check_timeout(plan, s));  // synchronizes
          turn.again();
          t0 = st;
        }
        run.st0 = st;
        run.st1 = std::min({half, st + launch_steps, t0 + turn_steps});
        run.bar_base = plan.bar_base;
        const int n = run.st1 - run.st0;
        const int grid = launch_rows(run, kind, p.f.lpr, j2, kMoments, plan.geo.max_group, items, true, s);
        if (grid < 0) return grid;
        plan.bar_base += (unsigned)grid * (unsigned)(n - 1);
        count_step(kind, row * (kind == POLFED_DF64 ? 5.0 : 3.0) * n);
        k_moment_sums<<<n, 32, 0, s>>>((const double2*)part, grid, mu + 2 * st);
        PF_CUDA(cudaGetLastError());
        count_launch();
      }
      PF_CUDA(cudaStreamSynchronize(s));
    }
    PF_CHECK(check_timeout(plan, s));
  }
  return POLFED_OK;
}

// Rows that are whole slices of 16-byte chunks are gathered where they lie: 64
// FP64 columns at L = 22 spent 345 of 1770 us on the copies into slices and out of
// them; in one launch over the block they take 1340 (FP32: 350 and 247).
bool apply_direct(int kind, int abi_kind, int n_b, const void* in, const void* out) {
  const size_t pitch = (size_t)n_b * elem_bytes(kind);
  return kind == abi_kind && kind != POLFED_DF64 && pitch % (16 * choose_lpr(kind, n_b)) == 0 && (uintptr_t)in % 16 == 0 &&
         (uintptr_t)out % 16 == 0;
}

int apply_block(HamPlan& plan, int kind, const void* in, void* out, int n_b, int abi_kind, FilterScratch& scr,
                cudaStream_t s) {
  const FilterShape f = filter_shape(plan.geo, kind, n_b, plan.slice_set);
  if (apply_direct(kind, abi_kind, n_b, in, out)) {
    const size_t pitch = (size_t)n_b * elem_bytes(kind);
    PF_CHECK(check_operator(plan, kind));
    StepRun run{};
    run.one = make_job(plan, kind, f.lpr, 1.0);
    run.one.xs = run.one.ba = (char*)const_cast<void*>(in);
    run.one.bb = (char*)out;
    run.one.K = 1;
    run.one.rowmul = (int)(pitch / (16 * f.lpr));
    run.st1 = 1;
    run.stride = 16 * f.lpr;
    run.err = plan.err_flag;
    run.n_jobs = f.nsl;
    const int grid = launch_rows(run, kind, f.lpr, plan.geo.rec_stride == 32, kDirect, plan.geo.max_group,
                                 (int64_t)plan.geo.n_groups * f.nsl, false, s);
    if (grid < 0) return grid;
    count_step(kind, (double)plan.geo.dim * pitch * 2.0);
    return POLFED_OK;
  }
  PF_CHECK(carve_scratch(scr, f));
  PF_CHECK(check_operator(plan, kind));
  const int64_t dim = plan.geo.dim;
  for (const SlicePart& p : slice_parts(plan.geo, kind, f, n_b)) {
    const SliceBufs b(scr, p.f);
    PF_CHECK(slice_in(kind, abi_kind, in, dim, n_b, p.col0, p.ncols, p.f, p.ns, b.xs, nullptr, 0.0, nullptr, s));
    StepRun run{};
    // one step of order K = 1 with c_0 = 0: out = H~ in, no barrier
    run.one = make_job(plan, kind, p.f.lpr, 1.0);
    run.one.xs = run.one.ba = b.xs;
    run.one.bb = b.bb;
    run.one.K = 1;
    run.st1 = 1;
    run.stride = (int64_t)p.f.slice;
    run.err = plan.err_flag;
    run.n_jobs = p.ns;
    const int grid = launch_rows(run, kind, p.f.lpr, plan.geo.rec_stride == 32, kFilter, plan.geo.max_group,
                                 (int64_t)plan.geo.n_groups * p.ns, false, s);
    if (grid < 0) return grid;
    count_step(kind, (double)dim * p.f.W * elem_bytes(kind) * p.ns * 3.0);
    PF_CHECK(slice_out(kind, abi_kind, b.bb, dim, p.f, p.ns, p.ncols, out, n_b, p.col0, nullptr, s));
  }
  return POLFED_OK;
}

// ------------------------------------------------ batched filter (host side)
namespace {

// jobs | coefficients (8 bytes a step) | flags | barrier and error | slice buffers
struct BatchLayout {
  size_t coef_off, flags_off, bar_off, slices_off, total;
  int n_jobs;
};

FilterShape batch_shape(const HamGeometry& g, int kind, int n_b) {
  FilterShape f;
  f.lpr = kBatchLpr;
  f.W = slice_width(kind, f.lpr);
  f.nsl = f.ns = (n_b + f.W - 1) / f.W;
  f.slice = ((size_t)g.dim * f.W * elem_bytes(kind) + 255) & ~(size_t)255;
  return f;
}

BatchLayout batch_layout(const std::vector<BatchFilterItem>& items, int kind) {
  BatchLayout L{};
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  size_t coefs = 0, slices = 0;
  for (const auto& it : items) {
    const FilterShape f = batch_shape(it.plan->geo, kind, it.n_b);
    L.n_jobs += f.nsl;
    coefs += (size_t)it.K + 1;
    slices += 3 * (size_t)f.nsl * f.slice;
  }
  L.coef_off = al(sizeof(StepJob) * std::max(1, L.n_jobs));
  L.flags_off = L.coef_off + al(sizeof(double) * std::max<size_t>(1, coefs));
  L.bar_off = L.flags_off + al(16 * std::max<size_t>(1, items.size()));
  L.slices_off = L.bar_off + 256;
  L.total = L.slices_off + slices;
  return L;
}

}  // namespace

size_t batch_scratch_bytes(const std::vector<BatchFilterItem>& items, int kind) {
  return batch_layout(items, kind).total;
}

int filter_batched(std::vector<BatchFilterItem>& items, int kind, int abi_kind, void* scratch, size_t bytes,
                   cudaStream_t s, int ctas_per_sm, BatchStats* bst) {
  if (items.empty()) return POLFED_OK;
  if (kind != POLFED_F32 && kind != POLFED_DF64) return fail(POLFED_EINVAL, "batched filter: FP32 or DF64 only");
  const BatchLayout Lo = batch_layout(items, kind);
  if (!scratch || bytes < Lo.total) return fail(POLFED_ENOMEM, "batched filter scratch too small");
  char* base = (char*)scratch;
  const bool j2 = items[0].plan->geo.rec_stride == 32;
  std::vector<StepJob> jobs;
  std::vector<double> coefs;
  jobs.reserve(Lo.n_jobs);
  size_t pos = Lo.slices_off;
  int n_steps = 0, max_group = 1;
  int64_t groups = 0;
  double alg = 0.0;
  PF_CUDA(cudaMemsetAsync(base + Lo.flags_off, 0, Lo.slices_off - Lo.flags_off, s));
  for (size_t q = 0; q < items.size(); q++) {
    BatchFilterItem& it = items[q];
    HamPlan& p = *it.plan;
    const HamGeometry& g = p.geo;
    if ((g.rec_stride == 32) != j2) return fail(POLFED_EINVAL, "batched filter: all jobs must agree on J2 = 0 or not");
    PF_CHECK(check_operator(p, kind));
    const FilterShape f = batch_shape(g, kind, it.n_b);
    float* flag = (float*)(base + Lo.flags_off + 16 * q);
    char* xs = base + pos;
    char* ba = xs + f.nsl * f.slice;
    char* bb = ba + f.nsl * f.slice;
    pos += 3 * (size_t)f.nsl * f.slice;
    if (it.K == 0) {
      PF_CHECK(slice_in(kind, abi_kind, it.in, g.dim, it.n_b, 0, it.n_b, f, f.nsl, nullptr, ba, it.coef[0] * it.invD,
                        flag, s));
      continue;
    }
    PF_CHECK(slice_in(kind, abi_kind, it.in, g.dim, it.n_b, 0, it.n_b, f, f.nsl, xs, ba, it.coef[it.K], flag, s));
    StepJob J = make_job(p, kind, f.lpr, it.invD);
    J.cx = base + Lo.coef_off + coefs.size() * sizeof(double);
    J.K = it.K;
    const size_t first = coefs.size();
    coefs.resize(first + (size_t)it.K + 1);
    char* cp = (char*)(coefs.data() + first);
    const size_t ces = kind == POLFED_F32 ? 4 : 8;
    const double row = (double)g.dim * f.W * elem_bytes(kind);
    double steps = 0.0;
    for (int st = 0; st < it.K; st++) {  // in step order
      const int k = it.K - 1 - st;
      const double c = k >= 1 ? it.coef[k] : it.coef[0] * it.invD;
      const double t = typed_const(kind, c);
      memcpy(cp + (size_t)st * ces, &t, ces);
      // Clenshaw minimum per step: read b_{k+1}, b_{k+2}, write b_k, read X when c_k != 0
      steps += 3.0 + (c != 0.0 ? 1.0 : 0.0);
    }
    for (int sl = 0; sl < f.nsl; sl++) {
      J.xs = xs + sl * f.slice;
      J.ba = ba + sl * f.slice;
      J.bb = bb + sl * f.slice;
      jobs.push_back(J);
      alg += row * steps;
      groups += g.n_groups;
    }
    n_steps = std::max(n_steps, it.K);
    max_group = std::max(max_group, g.max_group);
  }
  if (!jobs.empty()) {
    PF_CUDA(cudaMemcpyAsync(base + Lo.coef_off, coefs.data(), coefs.size() * sizeof(double), cudaMemcpyHostToDevice, s));
    PF_CUDA(cudaMemcpyAsync(base, jobs.data(), jobs.size() * sizeof(StepJob), cudaMemcpyHostToDevice, s));
    StepRun run{};
    run.jobs = (const StepJob*)base;
    run.n_jobs = (int)jobs.size();
    run.st1 = n_steps;
    run.bar = (unsigned*)(base + Lo.bar_off);
    run.err = (int*)(base + Lo.bar_off + 64);
    run.cap = wait_cap(kBarrierWaitPolls);
    int grid = 0;
    const double g0 = counters().step_gpu_s;
    double row = 0.0;  // of a step that every job takes part in
    for (const auto& it : items) {
      const FilterShape f = batch_shape(it.plan->geo, kind, it.n_b);
      row += (double)it.plan->geo.dim * f.W * elem_bytes(kind) * f.nsl;
    }
    const int turn_steps = std::max(1, (int)(kBatchTurnSeconds / step_seconds(kind, row, groups, max_group)));
    StepTimer tm(s, kind);
    {
      Turn turn;
      for (int st = 0; st < n_steps; st += turn_steps) {
        if (st > 0) turn.again();
        run.st0 = st;
        run.st1 = std::min(n_steps, st + turn_steps);
        tm.start();
        grid = launch_rows(run, kind, kBatchLpr, j2, kFilter, max_group, groups, true, s,
                           ctas_per_sm == 1 ? kMaxTeams / 2 : kMaxTeams);
        if (grid < 0) return grid;
        count_step(kind, alg * (run.st1 - run.st0) / n_steps);  // one launch carries every job's steps
        PF_CHECK(tm.stop());
        run.bar_base += (unsigned)grid * (unsigned)(run.st1 - run.st0 - 1);
      }
    }
    int e = 0;
    PF_CUDA(cudaMemcpyAsync(&e, run.err, sizeof(int), cudaMemcpyDeviceToHost, s));
    PF_CUDA(cudaStreamSynchronize(s));
    if (e) return fail(POLFED_ETIMEOUT, "a grid barrier of the batched filter timed out");
    if (bst) {
      bst->n_jobs = (int)jobs.size();
      bst->n_steps = n_steps;
      bst->grid = grid;
      bst->gpu_s = counters().step_gpu_s - g0;
      bst->alg_bytes = alg;
    }
  }
  // outputs: the buffer written by each job's last step
  pos = Lo.slices_off;
  for (size_t q = 0; q < items.size(); q++) {
    BatchFilterItem& it = items[q];
    const FilterShape f = batch_shape(it.plan->geo, kind, it.n_b);
    float* flag = (float*)(base + Lo.flags_off + 16 * q);
    const char* ba = base + pos + f.nsl * f.slice;
    const char* bb = ba + f.nsl * f.slice;
    pos += 3 * (size_t)f.nsl * f.slice;
    PF_CHECK(slice_out(kind, abi_kind, it.K % 2 == 0 ? ba : bb, it.plan->geo.dim, f, f.nsl, it.n_b, it.out, it.n_b, 0,
                       flag, s));
  }
  std::vector<float> fl(4 * items.size());
  PF_CUDA(cudaMemcpyAsync(fl.data(), base + Lo.flags_off, 16 * items.size(), cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  for (size_t q = 0; q < items.size(); q++) {
    int bad = 0;
    memcpy(&bad, &fl[4 * q + 2], 4);
    double csum = 0.0;
    for (int n = 0; n <= items[q].K; n++) csum += std::fabs(items[q].coef[n]);
    const double bound = csum * items[q].invD * std::sqrt((double)items[q].plan->geo.dim) * fl[4 * q] * 1.01 + 1e-300;
    items[q].bounds_error = bad || (double)fl[4 * q + 1] > bound;
  }
  return POLFED_OK;
}

void cheb_coeffs(double sigma, int K, std::vector<double>& c, double& D) {
  // Eq. (2): c_n = sqrt(4 - 3 delta_{0n}) cos(n arccos sigma); D = sum_n c_n T_n(sigma)
  // with T_n(sigma) = cos(n arccos sigma).  At sigma = 0, cos(n pi/2) is 0, +-1 exactly.
  c.assign(K + 1, 0.0);
  D = 0.0;
  const double phi = std::acos(sigma);
  for (int n = 0; n <= K; n++) {
    double cn;
    if (sigma == 0.0) {
      cn = (n & 1) ? 0.0 : ((n / 2) & 1 ? -1.0 : 1.0);
    } else {
      cn = std::cos(n * phi);
    }
    c[n] = (n == 0 ? 1.0 : 2.0) * cn;
    D += c[n] * cn;
  }
}

// ------------------------------------------------------------- basis kernel
// Unrank: the r-th L-bit string with n_up set bits in ascending order, by the
// combinatorial number system (greedy from the top bit).
__global__ void k_basis(int L, int n_up, uint32_t* states, int64_t dim) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < dim; r += (int64_t)gridDim.x * blockDim.x) {
    uint32_t rem = (uint32_t)r, s = 0;
    int k = n_up;
    for (int p = L - 1; p >= 0 && k > 0; p--) {
      const uint32_t c = c_binom[p][k];  // states with the top set bit below p
      if (rem >= c) {
        s |= 1u << p;
        rem -= c;
        k--;
      }
    }
    states[r] = s;
  }
}

int launch_basis(int L, int n_up, uint32_t* d_states, int64_t dim, cudaStream_t s) {
  upload_binomials();
  if (dim == 0) return POLFED_OK;
  int grid = (int)std::min<int64_t>((dim + 255) / 256, 152 * 32);
  k_basis<<<grid, 256, 0, s>>>(L, n_up, d_states, dim);
  PF_CUDA(cudaGetLastError());
  return POLFED_OK;
}

}  // namespace polfed

// ===================================================================== no-alloc
// polfed_cheb_filter_static: the Chebyshev filter with every table and every
// recurrence buffer carved out of one fixed device array instead of allocated
// memory.  It exists for callers that cannot allocate device memory while they
// run, e.g. code executing inside a memory pool or allocator callback, a
// library embedded in a host application that owns all device allocations, or
// a real-time loop that must not call into the allocator.  The array is a
// file-scope __device__ object: every GPU that loads this library holds it
// (kStaticScratchBytes) until the process exits, whether or not it is used.
namespace polfed {

constexpr size_t kStaticScratchBytes = (size_t)32 << 20;  // 32 MiB: dim <= 48620 (L <= 18) at 128-byte slices
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Device address of g_static_scratch per device (host code must not use the
// symbol itself: on the host it names a stand-in, not device memory).
static void* g_static_addr[64] = {nullptr};
static std::mutex g_static_mu;

static int static_scratch_addr(void** out) {
  int dev = 0;
  PF_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(POLFED_EINVAL, "device ordinal out of range for the static scratch table");
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_addr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return fail(POLFED_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_static_addr[dev] = p;
  }
  *out = g_static_addr[dev];
  return POLFED_OK;
}

// c_n of Eq. (2) computed on the fly (same expression as cheb_coeffs) or read
// from the caller's array; no storage.
struct CoefSource {
  const double* user;
  double sigma, phi;
  double operator[](int n) const {
    if (user) return user[n];
    const double cn = (sigma == 0.0) ? ((n & 1) ? 0.0 : ((n / 2) & 1 ? -1.0 : 1.0)) : std::cos(n * phi);
    return (n == 0 ? 1.0 : 2.0) * cn;
  }
  double T(int n) const {  // T_n(sigma)
    return (sigma == 0.0) ? ((n & 1) ? 0.0 : ((n / 2) & 1 ? -1.0 : 1.0)) : std::cos(n * phi);
  }
};

static int static_filter(const polfed_model* model, double e_lo, double e_hi, const CoefSource& c, int K, double invD,
                         const void* d_X, void* d_Y, int n_b, int dtype, cudaStream_t s) {
  upload_binomials();
  HamPlan plan;  // borrowed memory: pointers are cleared before it is destroyed
  struct Unborrow {
    HamPlan& p;
    ~Unborrow() {
      p.dev = nullptr;
      for (int k = 0; k < 3; k++) p.typed[k] = nullptr;
    }
  } unborrow{plan};
  PF_CHECK(build_geometry(model, -1, &plan.geo));
  const HamGeometry& g = plan.geo;
  const size_t tab = PlanLayout(g).total, typ = (typed_bytes_of(g) + 255) & ~(size_t)255;
  // as many slices at a time as the array holds (at least one)
  const size_t room = kStaticScratchBytes > tab + typ + 256 ? kStaticScratchBytes - tab - typ - 256 : 0;
  const FilterShape f = filter_shape(g, dtype, n_b, room);
  const size_t bytes = tab + typ + 3 * (size_t)f.ns * f.slice + 256;
  if (bytes > kStaticScratchBytes)
    return fail(POLFED_ENOMEM, "polfed_cheb_filter_static needs " + std::to_string(bytes) +
                                   " bytes of scratch; the static array holds " + std::to_string(kStaticScratchBytes) +
                                   " (use polfed_cheb_filter for this size)");
  void* base = nullptr;
  PF_CHECK(static_scratch_addr(&base));
  char* d = (char*)base;
  plan.stream = s;
  plan.stream_alloc = false;
  PF_CHECK(plan.bind(d, s, dtype, e_lo, e_hi, d + tab));
  FilterScratch scr;
  scr.xs = d + tab + typ;
  scr.bytes = bytes - tab - typ;
  const int abi = dtype == POLFED_F32 ? POLFED_F32 : POLFED_F64;
  PF_CHECK(filter_slices(plan, dtype, f, [&c](int n) { return c[n]; }, K, invD, nullptr, d_X, d_Y, n_b, abi, scr, s));
  float flag[3] = {0, 0, 0};
  PF_CUDA(cudaMemcpyAsync(flag, scr.flag, sizeof(flag), cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  int bad = 0;
  memcpy(&bad, &flag[2], 4);
  double csum = 0.0;
  for (int n = 0; n <= K; n++) csum += std::fabs(c[n]);
  const double bound = csum * invD * std::sqrt((double)g.dim) * (double)flag[0] * 1.01 + 1e-300;
  if (bad || (double)flag[1] > bound)
    return fail(POLFED_EBOUNDS, "filter output grew beyond the Chebyshev bound: spectrum outside [e_lo, e_hi]");
  return POLFED_OK;
}

}  // namespace polfed

extern "C" int polfed_set_wait_limit(uint32_t polls) {
  polfed::g_wait_limit.store(polls);
  return POLFED_OK;
}

extern "C" int polfed_cheb_filter_static(const polfed_model* model, const uint32_t* d_states, int64_t dim,
                                         double e_lo, double e_hi, double sigma, int32_t K, const double* coeffs,
                                         const void* d_X, void* d_Y, int32_t n_b, int32_t dtype,
                                         polfed_stream_t stream) {
  using namespace polfed;
  clear_error();
  if (!model) return fail(POLFED_EINVAL, "model is NULL");
  if (model->L < 4 || model->L > 32 || (model->L & 1)) return fail(POLFED_EINVAL, "L must be even, 4 <= L <= 32");
  if (dim != (int64_t)binom_host(model->L, model->L / 2)) return fail(POLFED_EINVAL, "dim != C(L, L/2)");
  if (!d_states || !d_X || !d_Y) return fail(POLFED_EINVAL, "NULL device pointer");
  if (n_b < 1 || n_b > 128) return fail(POLFED_EINVAL, "n_b must be in 1..128");
  if (dtype != POLFED_F32 && dtype != POLFED_F64 && dtype != POLFED_DF64) return fail(POLFED_EINVAL, "bad dtype");
  {
    const size_t es = dtype == POLFED_F32 ? 4 : 8;
    const char* x = (const char*)d_X;
    const char* y = (const char*)d_Y;
    const size_t nbytes = (size_t)dim * n_b * es;
    if (x < y + nbytes && y < x + nbytes) return fail(POLFED_EINVAL, "X and Y must not overlap");
  }
  if (!std::isfinite(e_lo) || !std::isfinite(e_hi) || (!(e_lo == 0.0 && e_hi == 0.0) && !(e_lo < e_hi)))
    return fail(POLFED_EINVAL, "need e_lo < e_hi (or both 0)");
  if (K < 0 || K > 10000000) return fail(POLFED_EINVAL, "K must be in 0..1e7");
  if (!coeffs && !(sigma > -1.0 && sigma < 1.0)) return fail(POLFED_EINVAL, "sigma must be in (-1, 1)");
  CoefSource c{coeffs, sigma, coeffs ? 0.0 : std::acos(sigma)};
  double invD = 1.0;
  if (coeffs) {
    for (int n = 0; n <= K; n++)
      if (!std::isfinite(coeffs[n])) return fail(POLFED_EINVAL, "non-finite coefficient");
  } else {
    double D = 0.0;
    for (int n = 0; n <= K; n++) D += c[n] * c.T(n);
    invD = 1.0 / D;
  }
  return static_filter(model, e_lo, e_hi, c, K, invD, d_X, d_Y, n_b, dtype, (cudaStream_t)stream);
}
