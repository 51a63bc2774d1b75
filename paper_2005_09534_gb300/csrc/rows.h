// Device code of the Clenshaw / H~ step: number policies, the group routine and
// the step kernel (one translation unit per storage type instantiates it).
#pragma once

#include <type_traits>

#include "polfed_internal.h"

namespace polfed {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Reads of the work item in shared memory are volatile: they are repeated where
// they are used instead of being held in registers.
__device__ __forceinline__ uint64_t lds64(const void* p) {
  uint64_t v;
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(smem_u32(p)));
  return v;
}
__device__ __forceinline__ int lds32(const void* p) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)));
  return v;
}

// --------------------------------------------------------- number policies
// Float-float arithmetic: a value is hi + lo with |lo| <= ulp(hi)/2.
// two_sum: Knuth (TAOCP vol. 2, 4.2.2); fast_two_sum: Dekker (1971);
// products use the FMA-based exact product error.
__device__ __forceinline__ float2 fast_two_sum(float a, float b) {
  float s = a + b;
  float e = b - (s - a);
  return make_float2(s, e);
}
__device__ __forceinline__ float2 two_sum(float a, float b) {
  float s = a + b;
  float bb = s - a;
  float e = (a - (s - bb)) + (b - bb);
  return make_float2(s, e);
}
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
  float2 s = two_sum(a.x, b.x);
  s.y += a.y + b.y;
  return fast_two_sum(s.x, s.y);
}
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  float p = a.x * b.x;
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  return fast_two_sum(p, e);
}

// The same on two values at once, each in one half of a pair (packed FP32
// instructions; rounding and order are those of the scalar forms).  The
// float-float step issues 2.2 instructions a clock with scalar ones: L = 20,
// J1-J2, 32 columns took 65 us a step and slice, packed 60, and with two rows
// of a thread in flight, which their registers then allow, 56.
struct DF2 {
  float2 h, l;
};
__device__ __forceinline__ float2 pair(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, pair(-1.f), a); }
__device__ __forceinline__ DF2 fast_two_sum(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  return DF2{s, __fadd2_rn(b, sub2(a, s))};
}
__device__ __forceinline__ DF2 two_sum(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b), t = sub2(a, s);  // t = -(s - a)
  return DF2{s, __fadd2_rn(sub2(a, __fadd2_rn(s, t)), __fadd2_rn(b, t))};
}
__device__ __forceinline__ DF2 df_add(const DF2& a, const DF2& b) {
  const DF2 s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, __fadd2_rn(s.l, __fadd2_rn(a.l, b.l)));
}
__device__ __forceinline__ DF2 df_mul(float2 c, const DF2& b) {  // c: one (hi, lo) for both
  const float2 p = __fmul2_rn(pair(c.x), b.h);
  float2 e = __ffma2_rn(pair(c.x), b.h, make_float2(-p.x, -p.y));
  e = __ffma2_rn(pair(c.x), b.l, e);
  e = __ffma2_rn(pair(c.y), b.h, e);
  return fast_two_sum(p, e);
}

// A policy works on 16-byte chunks of a row (int4 as loaded):
//   S, C         storage element and constant type
//   Acc          running sums over a row's neighbours (zero / add1 / add2: coupling class 1 / 2)
//   Coef         the step's constants (make)
//   fin          cX x + cH (d own + o1 sum1 + o2 sum2) + cB b2
// FP32 and FP64 fold cH into the couplings and accumulate s_l v by FMA straight
// into the result; float-float sums first and scales once (a float-float
// product costs as much as two additions).

// Typed constants of a job (StepJob::con), in the order of the enum.
enum { kConS1, kConS2, kConS1Last, kConS2Last, kConInvD, kConN };

struct RF32 {
  static constexpr bool kBondOrder = false;
  using S = float;
  using C = float;
  struct Coef {
    float s1, s2, cH, cX, cB;
  };
  struct Sum {
    float s1, s2;
  };
  static __device__ __forceinline__ Sum load_sum(const Coef* k) {
    return Sum{__int_as_float(lds32(&k->s1)), __int_as_float(lds32(&k->s2))};
  }
  static __device__ __forceinline__ Coef load_fin(const Coef* k) {
    return Coef{0.f, 0.f, __int_as_float(lds32(&k->cH)), __int_as_float(lds32(&k->cX)), __int_as_float(lds32(&k->cB))};
  }
  template <bool J2>
  struct Acc {
    float2 p, q;
  };
  static __device__ __forceinline__ Coef make(const double* con, bool last, bool first, float cx) {
    const float* f = reinterpret_cast<const float*>(con);
    Coef k;
    k.s1 = f[2 * (last ? kConS1Last : kConS1)];
    k.s2 = f[2 * (last ? kConS2Last : kConS2)];
    k.cH = last ? f[2 * kConInvD] : 2.f;
    k.cB = first ? 0.f : (last ? -f[2 * kConInvD] : -1.f);
    k.cX = cx;
    return k;
  }
  static __device__ __forceinline__ bool has_x(const Coef& k) { return k.cX != 0.f; }
  static __device__ __forceinline__ bool has_b(const Coef& k) { return k.cB != 0.f; }
  template <bool J2>
  static __device__ __forceinline__ void zero(Acc<J2>& a) {
    a.p = a.q = make_float2(0.f, 0.f);
  }
  template <bool J2>
  static __device__ __forceinline__ void fma(Acc<J2>& a, float s, const int4& u) {  // packed two-wide FMAs
    const float2 ss = make_float2(s, s);
    a.p = __ffma2_rn(ss, make_float2(__int_as_float(u.x), __int_as_float(u.y)), a.p);
    a.q = __ffma2_rn(ss, make_float2(__int_as_float(u.z), __int_as_float(u.w)), a.q);
  }
  template <bool J2>
  static __device__ __forceinline__ void add1(Acc<J2>& a, const Sum& k, const int4& u) {
    fma<J2>(a, k.s1, u);
  }
  template <bool J2>
  static __device__ __forceinline__ void add2(Acc<J2>& a, const Sum& k, const int4& u) {
    fma<J2>(a, k.s2, u);
  }
  static __device__ __forceinline__ float add3(float a, float b, float c) { return a + b + c; }
  // cxv: per-column cX of the lane's chunk (cols) instead of the step's scalar
  template <bool J2>
  static __device__ __forceinline__ int4 fin(Acc<J2>& a, const Coef& k, float d, const int4& own, const int4& x,
                                             const int4& b, bool hx, bool hb, bool cols, const float4& cxv) {
    fma<J2>(a, k.cH * d, own);
    if (hx) {
      if (cols) {
        a.p = __ffma2_rn(make_float2(cxv.x, cxv.y), make_float2(__int_as_float(x.x), __int_as_float(x.y)), a.p);
        a.q = __ffma2_rn(make_float2(cxv.z, cxv.w), make_float2(__int_as_float(x.z), __int_as_float(x.w)), a.q);
      } else {
        fma<J2>(a, k.cX, x);
      }
    }
    if (hb) fma<J2>(a, k.cB, b);
    return make_int4(__float_as_int(a.p.x), __float_as_int(a.p.y), __float_as_int(a.q.x), __float_as_int(a.q.y));
  }
  // dot += (t . t, t' . t)
  static __device__ __forceinline__ void dots(const int4& t, const int4& n, double2& dot) {
    auto one = [&](int a, int b) {
      const double c = (double)__int_as_float(a);
      dot.x = ::fma(c, c, dot.x);
      dot.y = ::fma((double)__int_as_float(b), c, dot.y);
    };
    one(t.x, n.x);
    one(t.y, n.y);
    one(t.z, n.z);
    one(t.w, n.w);
  }
};

struct RF64 {
  static constexpr bool kBondOrder = false;
  using S = double;
  using C = double;
  struct Coef {
    double s1, s2, cH, cX, cB;
  };
  struct Sum {
    double s1, s2;
  };
  static __device__ __forceinline__ Sum load_sum(const Coef* k) {
    return Sum{__longlong_as_double(lds64(&k->s1)), __longlong_as_double(lds64(&k->s2))};
  }
  static __device__ __forceinline__ Coef load_fin(const Coef* k) {
    return Coef{0.0, 0.0, __longlong_as_double(lds64(&k->cH)), __longlong_as_double(lds64(&k->cX)),
                __longlong_as_double(lds64(&k->cB))};
  }
  template <bool J2>
  struct Acc {
    double p, q;
  };
  static __device__ __forceinline__ Coef make(const double* con, bool last, bool first, double cx) {
    Coef k;
    k.s1 = con[last ? kConS1Last : kConS1];
    k.s2 = con[last ? kConS2Last : kConS2];
    k.cH = last ? con[kConInvD] : 2.0;
    k.cB = first ? 0.0 : (last ? -con[kConInvD] : -1.0);
    k.cX = cx;
    return k;
  }
  static __device__ __forceinline__ bool has_x(const Coef& k) { return k.cX != 0.0; }
  static __device__ __forceinline__ bool has_b(const Coef& k) { return k.cB != 0.0; }
  template <bool J2>
  static __device__ __forceinline__ void zero(Acc<J2>& a) {
    a.p = a.q = 0.0;
  }
  template <bool J2>
  static __device__ __forceinline__ void fma(Acc<J2>& a, double s, const int4& u) {
    a.p = ::fma(s, __hiloint2double(u.y, u.x), a.p);
    a.q = ::fma(s, __hiloint2double(u.w, u.z), a.q);
  }
  template <bool J2>
  static __device__ __forceinline__ void add1(Acc<J2>& a, const Sum& k, const int4& u) {
    fma<J2>(a, k.s1, u);
  }
  template <bool J2>
  static __device__ __forceinline__ void add2(Acc<J2>& a, const Sum& k, const int4& u) {
    fma<J2>(a, k.s2, u);
  }
  static __device__ __forceinline__ double add3(double a, double b, double c) { return a + b + c; }
  template <bool J2>
  static __device__ __forceinline__ int4 fin(Acc<J2>& a, const Coef& k, double d, const int4& own, const int4& x,
                                             const int4& b, bool hx, bool hb, bool, const float4&) {
    fma<J2>(a, d, own);  // d: cH times the diagonal
    if (hx) fma<J2>(a, k.cX, x);
    if (hb) fma<J2>(a, k.cB, b);
    return make_int4(__double2loint(a.p), __double2hiint(a.p), __double2loint(a.q), __double2hiint(a.q));
  }
  static __device__ __forceinline__ void dots(const int4& t, const int4& n, double2& dot) {
    const double c0 = __hiloint2double(t.y, t.x), c1 = __hiloint2double(t.w, t.z);
    dot.x = ::fma(c1, c1, ::fma(c0, c0, dot.x));
    dot.y = ::fma(__hiloint2double(n.w, n.z), c1, ::fma(__hiloint2double(n.y, n.x), c0, dot.y));
  }
};

// FP32 moments.  They are returned in FP64 though each carries FP32 rounding
// noise of 1e-8: other sums of the same neighbours would differ from earlier
// results by that much.  So this policy keeps the sums as they have always been:
// neighbours by plain addition in bond order, then d own + o1 sum1 + o2 sum2.
struct RF32M : RF32 {
  static constexpr bool kBondOrder = true;
  struct Sum {};
  static __device__ __forceinline__ Sum load_sum(const Coef*) { return Sum{}; }
  static __device__ __forceinline__ Coef load_fin(const Coef* k) { return *k; }
  template <bool J2>
  struct Acc {
    float2 p, q, p2, q2;
  };
  template <bool J2>
  static __device__ __forceinline__ void zero(Acc<J2>& a) {
    a.p = a.q = a.p2 = a.q2 = make_float2(0.f, 0.f);
  }
  static __device__ __forceinline__ float2 lo(const int4& u) { return make_float2(__int_as_float(u.x), __int_as_float(u.y)); }
  static __device__ __forceinline__ float2 hi(const int4& u) { return make_float2(__int_as_float(u.z), __int_as_float(u.w)); }
  template <bool J2>
  static __device__ __forceinline__ void add1(Acc<J2>& a, const Sum&, const int4& u) {
    a.p = __fadd2_rn(a.p, lo(u));
    a.q = __fadd2_rn(a.q, hi(u));
  }
  template <bool J2>
  static __device__ __forceinline__ void add2(Acc<J2>& a, const Sum&, const int4& u) {
    a.p2 = __fadd2_rn(a.p2, lo(u));
    a.q2 = __fadd2_rn(a.q2, hi(u));
  }
  template <bool J2>
  static __device__ __forceinline__ int4 fin(Acc<J2>& a, const Coef& k, float d, const int4& own, const int4&,
                                             const int4& b, bool, bool hb, bool, const float4&) {
    auto one = [&](float2 s1, float2 s2, float2 o, float2 bb) {
      const float2 dd = make_float2(d, d), o1 = make_float2(k.s1, k.s1), o2 = make_float2(k.s2, k.s2);
      float2 y = __ffma2_rn(dd, o, __fmul2_rn(o1, s1));
      if constexpr (J2) y = __ffma2_rn(o2, s2, y);
      return hb ? __ffma2_rn(make_float2(2.f, 2.f), y, make_float2(-bb.x, -bb.y)) : y;
    };
    const float2 x = one(a.p, a.p2, lo(own), lo(b)), y = one(a.q, a.q2, hi(own), hi(b));
    return make_int4(__float_as_int(x.x), __float_as_int(x.y), __float_as_int(y.x), __float_as_int(y.y));
  }
};

struct RDF {
  static constexpr bool kBondOrder = false;
  using S = float2;  // (hi, lo); two neighbouring elements are stored as (hi, hi, lo, lo)
  using C = float2;
  struct Coef {
    float2 o1, o2, cH, cX, cB;
    bool exact;  // cX, cH, cB are 0 or +-2^k: multiply hi and lo separately (exact)
  };
  struct Sum {};
  static __device__ __forceinline__ Sum load_sum(const Coef*) { return Sum{}; }
  static __device__ __forceinline__ Coef load_fin(const Coef* k) { return *k; }
  template <bool J2>
  struct Acc {
    DF2 a, c;  // running hi sums, accumulated low parts and rounding errors; c: coupling class 2
  };
  static __device__ __forceinline__ DF2 chunk(const int4& v) {
    return DF2{make_float2(__int_as_float(v.x), __int_as_float(v.y)), make_float2(__int_as_float(v.z), __int_as_float(v.w))};
  }
  static __device__ __forceinline__ bool pow2(float2 v) {
    return v.y == 0.f && (__float_as_uint(v.x) & 0x7FFFFFu) == 0;
  }
  static __device__ __forceinline__ Coef make(const double* con, bool last, bool first, float2 cx) {
    const float2* f = reinterpret_cast<const float2*>(con);
    Coef k;
    k.o1 = f[kConS1];
    k.o2 = f[kConS2];
    const float2 iv = f[kConInvD];
    k.cH = last ? iv : make_float2(2.f, 0.f);
    k.cB = first ? make_float2(0.f, 0.f) : (last ? make_float2(-iv.x, -iv.y) : make_float2(-1.f, 0.f));
    k.cX = cx;
    k.exact = pow2(k.cX) && pow2(k.cH) && pow2(k.cB);
    return k;
  }
  static __device__ __forceinline__ bool has_x(const Coef& k) { return k.cX.x != 0.f; }
  static __device__ __forceinline__ bool has_b(const Coef& k) { return k.cB.x != 0.f; }
  template <bool J2>
  static __device__ __forceinline__ void zero(Acc<J2>& a) {
    a.a = DF2{pair(0.f), pair(0.f)};
    if constexpr (J2) a.c = a.a;
  }
  static __device__ __forceinline__ void acc(DF2& a, const int4& u) {
    const DF2 v = chunk(u), s = two_sum(a.h, v.h);
    a.h = s.h;
    a.l = __fadd2_rn(a.l, __fadd2_rn(s.l, v.l));
  }
  template <bool J2>
  static __device__ __forceinline__ void add1(Acc<J2>& a, const Sum&, const int4& u) {
    acc(a.a, u);
  }
  template <bool J2>
  static __device__ __forceinline__ void add2(Acc<J2>& a, const Sum&, const int4& u) {
    acc(a.c, u);
  }
  static __device__ __forceinline__ float2 add3(float2 a, float2 b, float2 c) { return df_add(df_add(a, b), c); }
  template <bool J2>
  static __device__ __forceinline__ int4 fin(Acc<J2>& a, const Coef& k, float2 d, const int4& own, const int4& x,
                                             const int4& b, bool hx, bool hb, bool, const float4&) {
    DF2 y = df_add(df_mul(d, chunk(own)), df_mul(k.o1, fast_two_sum(a.a.h, a.a.l)));
    if constexpr (J2) y = df_add(y, df_mul(k.o2, fast_two_sum(a.c.h, a.c.l)));
    auto scaled = [](float c, const DF2& v) { return DF2{__fmul2_rn(pair(c), v.h), __fmul2_rn(pair(c), v.l)}; };
    DF2 r;
    if (k.exact) {
      r = scaled(k.cH.x, y);
      if (hx) r = df_add(r, scaled(k.cX.x, chunk(x)));
      if (hb) r = df_add(r, scaled(k.cB.x, chunk(b)));
    } else {
      r = df_mul(k.cH, y);
      if (hx) r = df_add(r, df_mul(k.cX, chunk(x)));
      if (hb) r = df_add(r, df_mul(k.cB, chunk(b)));
    }
    return make_int4(__float_as_int(r.h.x), __float_as_int(r.h.y), __float_as_int(r.l.x), __float_as_int(r.l.y));
  }
  // (double)v of a float by integer operations: with the FP64 pipe's conversions
  // (2 a clock and SM) a pair of moments at L = 18, 16 columns takes 26 us, so 23
  static __device__ __forceinline__ double f2d(int b) {
    const uint32_t a = (uint32_t)b & 0x7FFFFFFFu;
    if (a - 0x00800000u < 0x7F000000u)
      return __hiloint2double((int)(((uint32_t)b & 0x80000000u) | ((a >> 3) + 0x38000000u)), b << 29);
    return a == 0 ? __hiloint2double(b, 0) : (double)__int_as_float(b);
  }
  // y = H~ t_n (two elements): t_{n+1} = 2 y - t_{n-1} in FP64 (y itself for n = 0), its split in r
  static __device__ __forceinline__ double2 moment(const int4& y, const int4& t, const int4& prev, bool hb, double2& dot,
                                                   bool live, int4& r) {
    double v0 = f2d(y.x) + f2d(y.z);
    double v1 = f2d(y.y) + f2d(y.w);
    if (hb) {
      v0 = ::fma(2.0, v0, -__hiloint2double(prev.y, prev.x));
      v1 = ::fma(2.0, v1, -__hiloint2double(prev.w, prev.z));
    }
    if (live) {
      const double c0 = __hiloint2double(t.y, t.x), c1 = __hiloint2double(t.w, t.z);
      dot.x = ::fma(c1, c1, ::fma(c0, c0, dot.x));
      dot.y = ::fma(v1, c1, ::fma(v0, c0, dot.y));
    }
    const float h0 = (float)v0, h1 = (float)v1;
    r = make_int4(__float_as_int(h0), __float_as_int(h1), __float_as_int((float)(v0 - f2d(__float_as_int(h0)))),
                  __float_as_int((float)(v1 - f2d(__float_as_int(h1)))));
    return make_double2(v0, v1);
  }
};

// ------------------------------------------------------------------- jobs
// One column slice of one operator going through its Clenshaw steps.
struct StepJob {
  const uint16_t* rec;  // neighbour records (HamTables::rec)
  const GroupRec* grec;
  const void* Fc;       // typed, alpha-scaled diagonal of the low part, by cls_off + local index
  const void* Fhi;      // of the high part (schedule order, includes -alpha*beta)
  const void* Cx;       // of the cross bonds, by pattern
  const void* cx;       // typed cX in step order (a job of StepRun::jobs)
  const float* colcx;   // FP32: per-column cX, row n = order n (colw floats each), or null
  char *xs, *ba, *bb;   // x, b_{k+1}, b_{k+2} (overwritten by b_k)
  char *ta, *tb;        // moments in float-float: t_n (even n, odd n) in FP64
  double con[kConN];    // typed constants (each in its own 8 bytes)
  int K, n_groups, n_cross, c2mask;
  int colw;
  int rowmul;           // direct: bytes between rows / bytes of a slice's row
  int low_first;        // FP32 moments: low bonds before high ones
};

constexpr int kParamSteps = 448;  // step coefficients that travel in the kernel parameters

// What a step computes: the filter's recurrence, with a scalar or a per-column
// c_n, or t_{n+1} = 2 H~ t_n - t_{n-1} with the sums t_n . t_n and t_{n+1} . t_n,
// or one H~ product on the columns of a row-major block (rows `rowmul` slice rows apart).
enum StepMode { kFilter, kFilterCols, kMoments, kDirect };

struct StepRun {
  StepJob one;            // jobs == nullptr: n_jobs slices of this operator, buffers `stride` bytes apart
  const StepJob* jobs;
  int n_jobs;
  int st0, st1;           // steps of this launch
  int64_t stride, colstride;
  unsigned* bar;          // arrivals of the grid barrier, bar_base before this launch
  unsigned bar_base;
  uint32_t cap;
  int* err;
  double2* part;          // moments: the two sums of each CTA, gridDim.x entries per step from st0 on
  double cx[kParamSteps]; // jobs == nullptr: cX of the steps from st0 on, each in its own 8 bytes
};

// ------------------------------------------------------------ memory helpers
__device__ __forceinline__ void cp_async16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// L2 only: earlier steps of the same launch wrote these rows from other SMs
__device__ __forceinline__ int4 ld_l2(const char* p) {
  int4 v;
  asm volatile("ld.global.cg.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// tables: cached in L1, repeated at the place of use (volatile) to keep registers free
__device__ __forceinline__ uint4 ld_tab(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ld_stream(const char* p) {
  int4 v;
  asm volatile("ld.global.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// ---------------------------------------------------------------- step kernel
constexpr int kTeam = 128;       // threads of a team (4 warps, one group at a time)
constexpr int kMaxTeams = 6;     // 768 threads at 80 registers

__device__ __forceinline__ void team_sync(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(kTeam) : "memory");
}
// What a team needs for its group, in shared memory (double buffered).
template <class NT>
struct alignas(16) WorkItem {
  GroupRec g;
  typename NT::C fhi;
  int64_t pad;
  const char *b1, *x, *rec, *fc, *cxt, *col;  // col: the step's per-column cX
  char* t;                                    // moments in float-float: t_{n-1} in FP64 (x: t_n)
  char* out;                                  // and b2
  typename NT::Coef k;
  int n_cross, c2mask, rowmul, flags;         // flags: 1 = reads x, 2 = reads b2, 4 = low bonds first
};

// One step of one group (the rows sharing s_hi) by a team:
//   out = cX x + cH (H~ b1) + cB b2,  out in place of b2.
template <class NT, int LPR, bool J2, StepMode MODE, int RMAX>
struct GroupStep {
  using C = typename NT::C;
  using Acc = typename NT::template Acc<J2>;
  using Coef = typename NT::Coef;
  using Item = WorkItem<NT>;
  static constexpr int ROWB = 16 * LPR;
  static constexpr int RPW = 32 / LPR;             // rows of a warp's block
  static constexpr int NW = kTeam / 32;
  static constexpr int MAXCR = J2 ? 6 : 2;
  static constexpr int RS = J2 ? 32 : 16;          // uint16 entries of a record
  static constexpr int RSB = 2 * RS;
  static constexpr int STEP = kTeam * 16;          // bytes between a thread's consecutive rows
  // FP64: the diagonal of a row is formed once, not by each of its lanes (see run)
  static constexpr bool ROWD = std::is_same<NT, RF64>::value;
  static constexpr bool T64 = MODE == kMoments && std::is_same<NT, RDF>::value;  // t_n kept in FP64 beside its split

  template <int R>
  static __device__ __forceinline__ void pass(const Item* I, int blk, int n_g, const unsigned char* tile, bool& ready,
                                              int team, double2& dot, const C* dsm) {
    // high neighbours in flight per row (FP32, L = 24, J1-J2: 37.8 ms with two, 37.3 with four; float-float with
    // two rows is faster with two, 7.3 and 7.6 ms; FP64 at L = 14, single rows: 1200 us with four, 1165 with six)
    constexpr int HU = std::is_same<NT, RF32>::value ? 4 : (R == 1 ? (std::is_same<NT, RF64>::value ? 6 : 4) : 2);
    const int l32 = threadIdx.x & 31, lane16 = (l32 % LPR) * 16;
    int row = blk * RPW + l32 / LPR;
    bool live = true;
    if constexpr (R == 1) {
      live = row < n_g;
      row = min(row, n_g - 1);
    }
    const uint32_t ro = (uint32_t)(row * ROWB + lane16);  // in the tile
    const uint32_t mul = MODE == kDirect ? (uint32_t)lds32(&I->rowmul) : 1u;
    const uint32_t pitch = ROWB * mul, gro = MODE == kDirect ? (uint32_t)(row * pitch + lane16) : ro;
    const uint32_t step = STEP * mul;
    const size_t goff = (size_t)(uint32_t)lds32(&I->g.r0) * pitch + gro;
    const int flags = lds32(&I->flags);
    const bool hx = flags & 1, hb = flags & 2;
    const typename NT::Sum k = NT::load_sum(&I->k);
    Acc acc[R];
    int4 xv[R], bv[R];
#pragma unroll
    for (int i = 0; i < R; i++) NT::template zero<J2>(acc[i]);
    // high bonds: the same local rows of other groups
    const char* b1 = (const char*)lds64(&I->b1);
    auto add = [&](Acc& a, bool c1, const int4& u) {
      if (!J2 || c1)
        NT::template add1<J2>(a, k, u);
      else
        NT::template add2<J2>(a, k, u);
    };
    {
      const char* hp = b1 + gro;
      auto high = [&](int k0, int k1, bool c1) {
        int kk = k0;
        for (; kk + HU <= k1; kk += HU) {
          int4 u[HU][R];
#pragma unroll
          for (int j = 0; j < HU; j++) {
            const char* p = hp + (size_t)(uint32_t)lds32(&I->g.hn_base[kk + j]) * pitch;
#pragma unroll
            for (int i = 0; i < R; i++) u[j][i] = ld_l2(p + i * step);
          }
#pragma unroll
          for (int j = 0; j < HU; j++)
#pragma unroll
            for (int i = 0; i < R; i++) add(acc[i], c1, u[j][i]);
        }
        for (; kk < k1; kk++) {
          int4 u[R];
          const char* p = hp + (size_t)(uint32_t)lds32(&I->g.hn_base[kk]) * pitch;
#pragma unroll
          for (int i = 0; i < R; i++) u[i] = ld_l2(p + i * step);
#pragma unroll
          for (int i = 0; i < R; i++) add(acc[i], c1, u[i]);
        }
      };
      const int n_hn1 = lds32(&I->g.n_hn1);
      high(0, n_hn1, true);
      if constexpr (J2) high(n_hn1, lds32(&I->g.n_hn), false);
    }
    // x and b2, when the registers of the high neighbours are free again: loaded
    // first, L = 22, FP32, 64 columns takes 109 us a step and slice, here 101
    if (hx) {
      const char* p = (const char*)lds64(&I->x) + goff;
#pragma unroll
      for (int i = 0; i < R; i++) xv[i] = T64 ? ld_l2(p + i * STEP) : ld_stream(p + i * STEP);
    }
    if (hb) {
      const char* p = (const char*)lds64(T64 ? (const void*)&I->t : (const void*)&I->out) + goff;
#pragma unroll
      for (int i = 0; i < R; i++) bv[i] = ld_l2(p + i * STEP);
    }
    // neighbour records of the rows: header and cross neighbours
    const char* rp0 = (const char*)lds64(&I->rec) + (size_t)(uint32_t)((lds32(&I->g.cls_base) + row) * RSB);
    constexpr int RSTEP = kTeam / LPR * RSB;
    uint4 hd[R];
#pragma unroll
    for (int i = 0; i < R; i++) hd[i] = ld_tab(rp0 + i * RSTEP);
    auto half = [](const uint4& v, int e) {  // entry e = 0..7 of a 16-byte piece
      const uint32_t x = e < 2 ? v.x : (e < 4 ? v.y : (e < 6 ? v.z : v.w));
      return (e & 1) ? (x >> 16) : (x & 0xFFFFu);
    };
    // cross bonds: rows of another group, where the bond is antiparallel
    uint32_t pat[R];
    const int n_cross = lds32(&I->n_cross);
    {
      const uint32_t need = (uint32_t)lds32(&I->g.need_mask);
#pragma unroll
      for (int i = 0; i < R; i++) pat[i] = ~(half(hd[i], 0) ^ need) & ((1u << n_cross) - 1u);
    }
#pragma unroll
    for (int c = 0; c < MAXCR; c++) {
      if (c < n_cross) {
        const char* p = b1 + lane16 + (size_t)(uint32_t)lds32(&I->g.cr_base[c]) * pitch - pitch;
        const bool c1 = !J2 || !((lds32(&I->c2mask) >> c) & 1);
        int4 u[R];
#pragma unroll
        for (int i = 0; i < R; i++)
          if ((pat[i] >> c) & 1) u[i] = ld_l2(p + half(hd[i], 2 + c) * mul);
#pragma unroll
        for (int i = 0; i < R; i++)
          if ((pat[i] >> c) & 1) add(acc[i], c1, u[i]);
      }
    }
    if (!ready) {
      cp_async_wait();
      team_sync(team);
      ready = true;
    }
    // low bonds: rows of the staged group; lists are padded with the zero row at tile offset 0
    const unsigned char* tl = tile + lane16;
    auto low = [&](Acc& a, bool c1, uint32_t e0, uint32_t e1, bool second) {
      const int4 u0 = *reinterpret_cast<const int4*>(tl + e0), u1 = *reinterpret_cast<const int4*>(tl + e1);
      add(a, c1, u0);
      if (!ROWD || second) add(a, c1, u1);  // FP64: not even a padded entry is free
    };
#pragma unroll
    for (int i = 0; i < R; i++) {
      const uint32_t cnt = half(hd[i], 1);
      const int n1 = __reduce_max_sync(~0u, cnt & 0xFF);
      const char* rp = rp0 + i * RSTEP;
      if constexpr (J2) {
        const int n2 = __reduce_max_sync(~0u, cnt >> 8);
        const uint4 q1 = ld_tab(rp + 16), q2 = ld_tab(rp + 32);
        if (n1 > 0) low(acc[i], true, half(q1, 0), half(q1, 1), n1 > 1);
        if (n1 > 2) low(acc[i], true, half(q1, 2), half(q1, 3), n1 > 3);
        if (n1 > 4) low(acc[i], true, half(q1, 4), half(q1, 5), n1 > 5);
        if (n1 > 6) low(acc[i], true, half(q1, 6), half(q1, 7), n1 > 7);
        if (n1 > 8) low(acc[i], true, half(q2, 0), half(q2, 1), n1 > 9);
        const uint4 q3 = ld_tab(rp + 48);
        if (n2 > 0) low(acc[i], false, half(q2, 2), half(q2, 3), n2 > 1);
        if (n2 > 2) low(acc[i], false, half(q2, 4), half(q2, 5), n2 > 3);
        if (n2 > 4) low(acc[i], false, half(q2, 6), half(q2, 7), n2 > 5);
        if (n2 > 6) low(acc[i], false, half(q3, 0), half(q3, 1), n2 > 7);
        if (n2 > 8) low(acc[i], false, half(q3, 2), half(q3, 3), n2 > 9);
      } else {
        if (n1 > 0) low(acc[i], true, half(hd[i], 4), half(hd[i], 5), n1 > 1);
        if (n1 > 2) low(acc[i], true, half(hd[i], 6), half(hd[i], 7), n1 > 3);
        if (n1 > 4) {
          const uint4 q1 = ld_tab(rp + 16);
          low(acc[i], true, half(q1, 0), half(q1, 1), n1 > 5);
          if (n1 > 6) low(acc[i], true, half(q1, 2), half(q1, 3), n1 > 7);
          if (n1 > 8) low(acc[i], true, half(q1, 4), half(q1, 5), n1 > 9);
        }
      }
    }
    {
      const C* fc = (const C*)lds64(&I->fc) + lds32(&I->g.cls_base) + row;
      const C* cxt = (const C*)lds64(&I->cxt);
      char* out = (char*)lds64(&I->out) + goff;
      float4 cxv = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (MODE == kFilterCols) cxv = __ldg(reinterpret_cast<const float4*>((const char*)lds64(&I->col) + lane16));
      const C fhi = I->fhi;
      const Coef kf = NT::load_fin(&I->k);
#pragma unroll
      for (int i = 0; i < R; i++) {
        C d;
        if constexpr (ROWD)
          d = dsm[row + i * (kTeam / LPR)];
        else
          d = NT::add3(__ldg(fc + i * (kTeam / LPR)), fhi, __ldg(cxt + pat[i]));
        const int4 own = *reinterpret_cast<const int4*>(tile + ROWB + ro + i * STEP);
        int4 r;
        if constexpr (T64) {
          const int4 y = NT::template fin<J2>(acc[i], kf, d, own, xv[i], bv[i], false, false, false, cxv);
          const double2 v = NT::moment(y, xv[i], bv[i], hb, dot, R > 1 || live, r);
          if (R > 1 || live) __stcg(reinterpret_cast<double2*>((char*)lds64(&I->t) + goff + i * STEP), v);
        } else {
          r = NT::template fin<J2>(acc[i], kf, d, own, xv[i], bv[i], hx, hb, MODE == kFilterCols, cxv);
          if constexpr (MODE == kMoments)
            if (R > 1 || live) NT::dots(own, r, dot);
        }
        if (R > 1 || live) __stcg(reinterpret_cast<int4*>(out + i * step), r);
      }
    }
  }

  // The same step with the neighbours in bond order (RF32M): high, low, cross
  // bonds, or low, cross, high where the job says so.
  static __device__ __forceinline__ void pass_in_order(const Item* I, int blk, int n_g, const unsigned char* tile,
                                                       bool& ready, int team, double2& dot) {
    const int l32 = threadIdx.x & 31, lane16 = (l32 % LPR) * 16;
    const bool live = blk * RPW + l32 / LPR < n_g;
    const int row = min(blk * RPW + l32 / LPR, n_g - 1);
    const uint32_t ro = (uint32_t)(row * ROWB + lane16);
    const size_t goff = (size_t)(uint32_t)lds32(&I->g.r0) * ROWB + ro;
    const int flags = lds32(&I->flags);
    const char* b1 = (const char*)lds64(&I->b1);
    const typename NT::Sum k = NT::load_sum(&I->k);
    const int4 bv = (flags & 2) ? ld_l2((const char*)lds64(&I->out) + goff) : make_int4(0, 0, 0, 0);
    Acc acc;
    NT::template zero<J2>(acc);
    auto add = [&](bool c1, const int4& u) {
      if (!J2 || c1)
        NT::template add1<J2>(acc, k, u);
      else
        NT::template add2<J2>(acc, k, u);
    };
    const int n_hn = lds32(&I->g.n_hn), n_hn1 = lds32(&I->g.n_hn1), n_cross = lds32(&I->n_cross);
    const uint16_t* rec = (const uint16_t*)lds64(&I->rec) + (size_t)(uint32_t)(lds32(&I->g.cls_base) + row) * RS;
    const uint32_t pat = ~((uint32_t)__ldg(rec) ^ (uint32_t)lds32(&I->g.need_mask)) & ((1u << n_cross) - 1u);
    auto high = [&]() {
      auto src = [&](int j) { return ld_l2(b1 + ro + (size_t)(uint32_t)lds32(&I->g.hn_base[j]) * ROWB); };
      int j = 0;
      for (; j + 4 <= n_hn; j += 4) {
        int4 u[4];
#pragma unroll
        for (int q = 0; q < 4; q++) u[q] = src(j + q);
#pragma unroll
        for (int q = 0; q < 4; q++) add(j + q < n_hn1, u[q]);
      }
      for (; j < n_hn; j++) add(j < n_hn1, src(j));
    };
    if (!(flags & 4)) high();
    if (!ready) {
      cp_async_wait();
      team_sync(team);
      ready = true;
    }
    const uint32_t cnt = __ldg(rec + 1);
    for (int e = 0; e < (int)(cnt & 0xFF); e++)
      add(true, *reinterpret_cast<const int4*>(tile + lane16 + __ldg(rec + low_entry(e, true))));
    if constexpr (J2)
      for (int e = 0; e < (int)(cnt >> 8); e++)
        add(false, *reinterpret_cast<const int4*>(tile + lane16 + __ldg(rec + low_entry(e, false))));
    for (int c = 0; c < n_cross; c++)
      if ((pat >> c) & 1)
        add(!J2 || !((lds32(&I->c2mask) >> c) & 1),
            ld_l2(b1 + lane16 + (size_t)(uint32_t)lds32(&I->g.cr_base[c]) * ROWB - ROWB + __ldg(rec + 2 + c)));
    if (flags & 4) high();
    const C d = NT::add3(__ldg((const C*)lds64(&I->fc) + lds32(&I->g.cls_base) + row), I->fhi,
                         __ldg((const C*)lds64(&I->cxt) + pat));
    const int4 own = *reinterpret_cast<const int4*>(tile + ROWB + ro);
    const int4 r = NT::template fin<J2>(acc, NT::load_fin(&I->k), d, own, bv, bv, false, flags & 2, false,
                                        make_float4(0.f, 0.f, 0.f, 0.f));
    if (live) {
      NT::dots(own, r, dot);
      __stcg(reinterpret_cast<int4*>((char*)lds64(&I->out) + goff), r);
    }
  }
  // entry of the e-th low neighbour in a record
  static __device__ __forceinline__ int low_entry(int e, bool c1) { return J2 ? (c1 ? 8 : 18) + e : 4 + e; }

  static __device__ __forceinline__ void run(const Item* I, unsigned char* tile, int team, int w, double2& dot, C* dsm) {
    const int n_g = lds32(&I->g.n_g);
    {
      const uint32_t mul = MODE == kDirect ? (uint32_t)lds32(&I->rowmul) : 1u;
      const char* src = (const char*)lds64(&I->b1) + (size_t)(uint32_t)lds32(&I->g.r0) * (ROWB * mul);
      const int nb = n_g * ROWB;
      for (int c = (threadIdx.x % kTeam) * 16; c < nb; c += STEP)
        cp_async16(tile + ROWB + c, src + (MODE == kDirect ? c / ROWB * (ROWB * mul) + c % ROWB : c));
      cp_async_commit();
    }
    if constexpr (ROWD) {
      // cH d of the group's rows: 3 FP64 instructions a row instead of 3 for each of its 16-byte chunks, the
      // FP64 pipe being 89% busy (L = 20, 64 columns, K = 40: 16.4 ms, with this and no padded entries 14.6)
      const int cls = lds32(&I->g.cls_base), n_cross = lds32(&I->n_cross);
      const uint32_t need = (uint32_t)lds32(&I->g.need_mask);
      const C cH = NT::load_fin(&I->k).cH;
      for (int r = threadIdx.x % kTeam; r < n_g; r += kTeam) {
        const uint32_t own = __ldg((const uint16_t*)lds64(&I->rec) + (size_t)(cls + r) * RS);
        const uint32_t pat = ~(own ^ need) & ((1u << n_cross) - 1u);
        dsm[r] = cH * NT::add3(__ldg((const C*)lds64(&I->fc) + cls + r), I->fhi, __ldg((const C*)lds64(&I->cxt) + pat));
      }
    }
    bool ready = false;
    const int nblk = (n_g + RPW - 1) / RPW, nfull = n_g / RPW;
    int blk = w;
    if constexpr (NT::kBondOrder) {
      for (; blk < nblk; blk += NW) pass_in_order(I, blk, n_g, tile, ready, team, dot);
    } else {
      if constexpr (RMAX >= 2)
        for (; blk + NW < nfull; blk += 2 * NW) pass<2>(I, blk, n_g, tile, ready, team, dot, dsm);
      for (; blk < nblk; blk += NW) pass<1>(I, blk, n_g, tile, ready, team, dot, dsm);
    }
    if (!ready) {
      cp_async_wait();
      team_sync(team);
    }
  }
};

// Grid barrier of a cooperative launch: arrivals are counted on one monotone
// counter; waits are bounded (cap polls), a wait that runs out sets *err and
// every CTA leaves at its next barrier.  What needs no other CTA's result goes
// between the two halves.
__device__ __forceinline__ void grid_arrive(unsigned* count) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
  }
}
__device__ __forceinline__ bool grid_wait(unsigned* count, unsigned target, int* err, uint32_t cap) {
  int ok = 1;
  if (threadIdx.x == 0) {
    uint32_t it = 0;
    while ((int)(*(volatile unsigned*)count - target) < 0) {
      if (++it > cap) {
        atomicExch(err, 1);
        ok = 0;
        break;
      }
      if ((it & 15) == 0) {
        if (*(volatile int*)err) {
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  return __syncthreads_and(ok) != 0;
}

// Steps st0..st1-1 of every job with st < K.  Work items are (job, group)
// pairs, groups largest first, dealt to the teams of all CTAs in alternating
// direction; CTAs meet at the grid barrier between steps.  The record of a
// team's next group is fetched while the current one is worked on.
//
// What bounds it.  A row reads 9.3 rows of 128 bytes through L2 at L = 22 XXZ
// (itself 1, high bonds 5.8, cross bonds 1, b2 1, x on half of the steps) and
// 5 more from the staged group: 0.84 GB per step against the 0.32 GB a step
// cannot do without, of which 0.34 GB come from DRAM.  The time is the latency
// of those loads (long-scoreboard stalls; issue slots 30%, L2 35%, DRAM 44%
// busy), so the kernel holds as many independent warps as its registers allow
// (six teams of four per SM, each with its own group and barrier), keeps
// uniform values in shared memory and reads everything but the own group
// straight into registers.  A bulk-copy ring that staged every neighbour block
// was slower (129 us per step at L = 22; 360 instead of 190 instructions per
// four rows), deeper per-warp prefetch was too (the scoreboards of a warp make
// its loads wait for one another).
// Many steps per launch save a launch of about 5 us each, which at L <= 18 is
// most of the step: the barrier costs 1.4 us.
// Items are dealt in advance: handed out by an atomic counter instead, neighbouring
// groups drift apart and L = 20 float-float takes 8.5 ms for 7.3, L = 22 42.4 for 40.6.
// Measured, us per step and slice of 128 bytes (one launch per step before):
// L = 14 FP64 37 -> 5.2, L = 18 float-float moments 53 -> 22, L = 20 J1-J2
// float-float 91 -> 56, L = 20 J1-J2 FP32 71 -> 43, L = 22 FP32 128 -> 99,
// L = 24 J1-J2 FP32 1183 -> 760.
template <class NT, int LPR, bool J2, StepMode MODE>
__global__ void __launch_bounds__(kTeam* kMaxTeams, 1) k_step_rows(const __grid_constant__ StepRun R, int tile_bytes) {
  using C = typename NT::C;
  using Item = WorkItem<NT>;
  // rows of a thread in flight (float-float moments hold t_n and t_{n-1} too: 22.6 us a pair with one, 23.8 with two)
  constexpr int RMAX = (std::is_same<NT, RDF>::value && MODE == kMoments) ? 1 : 2;
  extern __shared__ __align__(128) unsigned char smem[];
  const int team = threadIdx.x / kTeam, tt = threadIdx.x % kTeam;
  unsigned char* tile = smem + (size_t)team * tile_bytes;
  Item* items = reinterpret_cast<Item*>(smem + (size_t)(blockDim.x / kTeam) * tile_bytes) + 2 * team;
  // FP64: cH d of the group's rows, behind the items
  C* dsm = reinterpret_cast<C*>(smem + (size_t)(blockDim.x / kTeam) * (tile_bytes + 2 * sizeof(Item))) +
           (size_t)team * (tile_bytes / (16 * LPR));
  const int n_teams = (blockDim.x / kTeam) * gridDim.x;
  const int me = team * gridDim.x + blockIdx.x;  // neighbouring items go to different SMs
  if (tt < LPR) *reinterpret_cast<int4*>(tile + tt * 16) = make_int4(0, 0, 0, 0);  // the zero row
  unsigned target = R.bar_base;
  int st = R.st0, j = 0, base = 0, r = 0;
  // fetch the r-th item of this team into items[r & 1]; false if there is none
  auto fetch = [&]() -> bool {
    const int item = r * n_teams + ((r & 1) ? n_teams - 1 - me : me);
    const StepJob* J = nullptr;
    for (; j < R.n_jobs; j++) {
      J = R.jobs ? R.jobs + j : &R.one;
      const int ng = st < J->K ? J->n_groups : 0;
      if (item < base + ng) break;
      base += ng;
    }
    if (j >= R.n_jobs) return false;
    Item* I = items + (r & 1);
    const int gidx = item - base;
    constexpr int NG = sizeof(GroupRec) / 16;
    if (tt < NG) cp_async16(reinterpret_cast<char*>(&I->g) + tt * 16, reinterpret_cast<const char*>(J->grec + gidx) + tt * 16);
    if (tt == NG)
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(&I->fhi)),
                   "l"(reinterpret_cast<const C*>(J->Fhi) + gidx), "n"(sizeof(C))
                   : "memory");
    cp_async_commit();
    if (tt == 32) {
      const size_t so = R.jobs ? 0 : (size_t)j * R.stride;
      I->b1 = ((st & 1) ? J->bb : J->ba) + so;
      I->out = ((st & 1) ? J->ba : J->bb) + so;
      I->x = J->xs + so;
      I->rec = reinterpret_cast<const char*>(J->rec);
      I->fc = reinterpret_cast<const char*>(J->Fc);
      I->cxt = reinterpret_cast<const char*>(J->Cx);
      I->n_cross = J->n_cross;
      I->c2mask = J->c2mask;
      if constexpr (MODE == kDirect) I->rowmul = J->rowmul;
      const int kk = J->K - 1 - st;
      bool last = kk == 0, first = st == 0;
      C cx = C();
      if constexpr (MODE == kMoments) {  // t_1 = H~ t_0, then 2 H~ t_n - t_{n-1}; FP32 and float-float take H~ t_n and finish it
        last = first = first || !std::is_same<NT, RF64>::value;
        I->x = (st & 1) ? J->tb + so : J->ta + so;
        I->t = (st & 1) ? J->ta + so : J->tb + so;
      } else if constexpr (MODE == kFilterCols) {
        I->col = reinterpret_cast<const char*>(J->colcx + (R.jobs ? 0 : j * R.colstride) + (size_t)kk * J->colw);
      } else {
        cx = R.jobs ? __ldg(reinterpret_cast<const C*>(J->cx) + st) : *reinterpret_cast<const C*>(&R.cx[st - R.st0]);
      }
      const typename NT::Coef k = NT::make(J->con, last, first, cx);
      I->k = k;
      if constexpr (MODE == kMoments)
        I->flags = (std::is_same<NT, RDF>::value ? 1 : 0) | (st > 0 ? 2 : 0) | (J->low_first ? 4 : 0);
      else
        I->flags = (MODE == kFilterCols || NT::has_x(k) ? 1 : 0) | (NT::has_b(k) ? 2 : 0);
    }
    return true;
  };
  bool more = fetch();
  double2 dot = make_double2(0.0, 0.0);
  for (;;) {
    while (more) {
      cp_async_wait();
      team_sync(team);  // the item is complete, the previous group's tile is no longer read
      const Item* I = items + (r & 1);
      r++;
      more = fetch();
      GroupStep<NT, LPR, J2, MODE, RMAX>::run(I, tile, team, tt >> 5, dot, dsm);
    }
    if constexpr (MODE == kMoments) {
      __shared__ double2 wsum[kTeam * kMaxTeams / 32];
      for (int o = 16; o; o >>= 1) {
        dot.x += __shfl_xor_sync(~0u, dot.x, o);
        dot.y += __shfl_xor_sync(~0u, dot.y, o);
      }
      if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = dot;
      __syncthreads();
      if (threadIdx.x == 32) {
        for (int w = 0; w < (int)blockDim.x / 32; w++)
          if (w != 1) dot = make_double2(dot.x + wsum[w].x, dot.y + wsum[w].y);
        R.part[(size_t)(st - R.st0) * gridDim.x + blockIdx.x] = dot;
      }
      dot = make_double2(0.0, 0.0);
    }
    if (++st == R.st1) break;
    grid_arrive(R.bar);
    j = base = r = 0;
    more = fetch();  // the first item of the next step, while the others arrive
    target += gridDim.x;
    if (!grid_wait(R.bar, target, R.err, R.cap)) break;
  }
  cp_async_wait();
}

// Launch the steps of `run` on up to max_teams teams per SM: the grid size (> 0), or a negative status.
int launch_rows_f32(const StepRun& run, int lpr, bool j2, StepMode mode, int max_group, int64_t items, bool cooperative,
                    int max_teams, cudaStream_t s);
int launch_rows_f64(const StepRun& run, int lpr, bool j2, StepMode mode, int max_group, int64_t items, bool cooperative,
                    int max_teams, cudaStream_t s);
int launch_rows_df(const StepRun& run, int lpr, bool j2, StepMode mode, int max_group, int64_t items, bool cooperative,
                   int max_teams, cudaStream_t s);

}  // namespace polfed
