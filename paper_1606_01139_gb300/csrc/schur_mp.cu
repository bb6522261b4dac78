// Projected eigenproblem of a thick restart, for the batched windows: only the
// invariant subspace of the kept Ritz values (smallest |theta|, the 'SM' rule on
// the shifted operator of Eq. 3) is needed to full accuracy, so the order-m
// work runs in FP32 and the accuracy comes from a subspace iteration:
//
//  1. mp_hess_kernel    Householder reduction of H to Hessenberg form, FP32
//  2. mp_chase_kernel   QR iteration to Schur form, FP32, chains of up to 16
//                       single-shift bulges three rows apart until the blocks
//                       that split off have order 32 or less, then a warp per
//                       block; the rotations go to a list, the active block
//                       alone is updated
//  3. mp_apply_kernel   Q = reflectors x rotations, a warp per two rows
//  4. mp_gemm (FP32)    T = Q^H H Q
//  5. mp_order_kernel   the k kept Ritz values to the leading block, all
//                       bubbles moving at once; its rotations applied to Q
//  6. three corrections of V = Q[:, 0:k]:  W = H V, G = V^H W, R = W - V G in
//     double-single; T22 X - X T11 = Q2^H R in FP32 (mp_sylv_kernel);
//     V <- orth(V - Q2 X) (one Newton-Schulz step).  The FP32 solve corrects a
//     factor ~1e-4 per step: 4e-7 |H| -> 1e-10 -> 1e-14, the accuracy of the
//     double-single products (measured on restart matrices of order 150-237).
//  7. the double-single Schur form of G (order k) by the same reduction and
//     chase, its reflectors and rotations applied to V, one more Newton-Schulz
//     step, T = V^H H V; then eigenvectors and residual estimates.
//
// The chain of dependent rotations is what bounds the whole step: the order-m
// double-single kernel (schur_ds.cu, one CTA) takes ~1.9 us per rotation, 17-38
// thousand of them at order 150-208.  An FP32 chase step takes ~0.55 us and
// moves all bulges of a chain (3-7 thousand steps), and the double-single chain
// that remains has order k, a sixth to a half of m.  Measured per restart on one
// GB300: 43 ms -> 5.9 ms at order 150 (15-35 kept), 57 ms -> 9.6 ms at orders
// 163-184 (35-110 kept); |H Z - Z T| / max|H| 0.6-2e-14, |Z^H Z - I| 2e-14 to
// 2e-13 on restart matrices of orders 150-208.
//
// A failure (iteration or list limit, corrections that do not converge, a last
// restart whose kept set hangs on FP32 rounding) is reported as status 1 in
// ordinfo[2]; the caller then runs the double-single kernel of order m on the
// saved matrix.
#include <mutex>
#include <set>
#include <type_traits>
#include <utility>

#include "ds.cuh"
#include "swi_internal.cuh"

namespace swi {

namespace {

constexpr int kNB = 16;             // bulges per chain, rotations per list step
constexpr int kSmall = 32;          // blocks up to this order are finished by a warp each
constexpr int kChaseThreads = 32 * kNB;  // a warp per bulge
constexpr int kMaxM = kMpMaxOrder;
constexpr size_t kSmemMatrix = 220 * 1024;  // largest matrix kept in shared memory

enum { CTL_STATUS = 0, CTL_K0 = 1, CTL_STEPS = 2, CTL_STEPS2 = 3, CTL_HMAX = 4, CTL_STEPSK = 6, CTL_HMAXK = 7,
       CTL_RMAX = 8 /* one per projection: 4 */ };

__device__ __forceinline__ float2 fc(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 f2(double2 v) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ float2 mulf(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// acc += a b, acc += conj(a) b
__device__ __forceinline__ void fma2(float2& c, float2 a, float2 b) {
  c.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
  c.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
}
__device__ __forceinline__ void fma2c(float2& c, float2 a, float2 b) {
  c.x = fmaf(a.x, b.x, fmaf(a.y, b.y, c.x));
  c.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, c.y));
}
__device__ __forceinline__ float norm2(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }
__device__ __forceinline__ float abs1(float2 a) { return fabsf(a.x) + fabsf(a.y); }
__device__ __forceinline__ float2 divf2(float2 a, float2 b) {  // scaled: |b|^2 stays in range
  const float m = fmaxf(fabsf(b.x), fabsf(b.y));
  if (!(m > 0.f)) return fc(0.f, 0.f);
  const float2 q = fc(b.x / m, b.y / m);
  const float d = 1.f / (norm2(q) * m);
  return fc((a.x * q.x + a.y * q.y) * d, (a.y * q.x - a.x * q.y) * d);
}
__device__ __forceinline__ float2 sqrtf2(float2 z) {  // principal square root
  const float m = fmaxf(fabsf(z.x), fabsf(z.y));
  if (!(m > 0.f)) return fc(0.f, 0.f);
  const float x = z.x / m, y = z.y / m;
  const float r = sqrtf(fmaf(x, x, y * y));
  const float t = sqrtf(0.5f * (r + fabsf(x))), s = sqrtf(m);
  return x >= 0.f ? fc(s * t, s * (y / (2.f * t))) : fc(s * (fabsf(y) / (2.f * t)), s * copysignf(t, y));
}
__device__ __forceinline__ float2 shfl_xor2(float2 a, int o) {
  return fc(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
__device__ __forceinline__ float2 warp_sum2(float2 a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float2 b = shfl_xor2(a, o);
    a.x += b.x;
    a.y += b.y;
  }
  return a;
}

// The reduction, the chase and the application of its rotations run in FP32
// (C = float2) on the projected matrix and in double-single (C = ds::dc) on the
// kept block; the overloads below are their arithmetic.
using ds::dc;
using ds::df;
template <class C>
struct RotT;
template <>
struct RotT<float2> {
  float c;
  float2 s;
};
template <>
struct RotT<dc> {
  df c;
  dc s;
};
using Rot = RotT<float2>;

template <class C>
struct Arith;
template <>
struct Arith<float2> {
  using R = float;
  __device__ static float2 from(double2 v) { return f2(v); }
  __device__ static float2 zero() { return fc(0.f, 0.f); }
};
template <>
struct Arith<dc> {
  using R = df;
  __device__ static dc from(double2 v) {
    dc r;
    ds::split_wide(v.x, r.re.h, r.re.l);
    ds::split_wide(v.y, r.im.h, r.im.l);
    return r;
  }
  __device__ static dc zero() { return ds::czero(); }
};
__device__ __forceinline__ float2 head(float2 a) { return a; }
__device__ __forceinline__ float2 head(dc a) { return fc(a.re.h, a.im.h); }
__device__ __forceinline__ float abs1(dc a) { return fabsf(a.re.h) + fabsf(a.im.h); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return fc(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ dc sub(dc a, dc b) { return ds::csub(a, b); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return fc(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ dc add(dc a, dc b) { return ds::cadd(a, b); }
__device__ __forceinline__ float2 scale(float2 a, float t) { return fc(a.x * t, a.y * t); }
__device__ __forceinline__ dc scale(dc a, df t) { return ds::cscale(a, t); }
// running sums: (head, error) pairs in the double-single form, closed by norm()
__device__ __forceinline__ void fma2(dc& c, const dc& a, const dc& b) {
  ds::fma_acc(c.re.h, c.re.l, a.re.h, a.re.l, b.re.h, b.re.l);
  ds::fma_acc(c.im.h, c.im.l, a.re.h, a.re.l, b.im.h, b.im.l);
  ds::fma_acc(c.re.h, c.re.l, -a.im.h, -a.im.l, b.im.h, b.im.l);
  ds::fma_acc(c.im.h, c.im.l, a.im.h, a.im.l, b.re.h, b.re.l);
}
__device__ __forceinline__ void fma2c(dc& c, const dc& a, const dc& b) {
  ds::fma_acc(c.re.h, c.re.l, a.re.h, a.re.l, b.re.h, b.re.l);
  ds::fma_acc(c.im.h, c.im.l, a.re.h, a.re.l, b.im.h, b.im.l);
  ds::fma_acc(c.re.h, c.re.l, a.im.h, a.im.l, b.im.h, b.im.l);
  ds::fma_acc(c.im.h, c.im.l, -a.im.h, -a.im.l, b.re.h, b.re.l);
}
// a + b c and a + b conj(c)
__device__ __forceinline__ float2 fmadd(float2 a, float2 b, float2 c) {
  fma2(a, b, c);
  return a;
}
__device__ __forceinline__ dc fmadd(dc a, dc b, dc c) { return ds::cadd(a, ds::cmul(b, c)); }
__device__ __forceinline__ float2 fmaddc(float2 a, float2 b, float2 c) {
  fma2(a, b, fc(c.x, -c.y));
  return a;
}
__device__ __forceinline__ dc fmaddc(dc a, dc b, dc c) { return ds::cadd(a, ds::cmulc_l(c, b)); }
__device__ __forceinline__ float2 norm(float2 a) { return a; }
__device__ __forceinline__ dc norm(dc a) {
  return dc{ds::two_sum(a.re.h, a.re.l), ds::two_sum(a.im.h, a.im.l)};
}
__device__ __forceinline__ float2 shx(float2 a, int o) { return shfl_xor2(a, o); }
__device__ __forceinline__ df shx(df a, int o) {
  return df{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ dc shx(dc a, int o) { return dc{shx(a.re, o), shx(a.im, o)}; }
template <class C>
__device__ __forceinline__ C lanes_sum(C a, int from) {  // over the lanes that differ in bits < 2 from
  for (int o = from; o > 0; o >>= 1) a = add(a, shx(a, o));
  return a;
}
__device__ __forceinline__ float radd(float a, float b) { return a + b; }
__device__ __forceinline__ df radd(df a, df b) { return ds::add(a, b); }
__device__ __forceinline__ float rshx(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ df rshx(df a, int o) { return shx(a, o); }
__device__ __forceinline__ float cnorm(float2 a) { return norm2(a); }
__device__ __forceinline__ df cnorm(dc a) { return ds::cabs2(a); }
__device__ __forceinline__ float hi(float a) { return a; }
__device__ __forceinline__ float hi(df a) { return a.h; }
__device__ __forceinline__ float rs(float a) { return rsqrtf(a); }
// 1/sqrt(a): the float estimate x and one correction x e (1/2 + 3/8 e), e = 1 - a x^2
// formed in double-single (|e| < 2^-20: the next term is below 2^-60)
__device__ __forceinline__ df rs(df a) {
  const float x = rsqrtf(a.h);
  const float p = x * x;
  const df t = ds::mul(a, df{p, fmaf(x, x, -p)});
  const float e = (1.f - t.h) - t.l;
  return ds::quick_two_sum(x, x * e * fmaf(0.375f, e, 0.5f));
}
__device__ __forceinline__ float rmul(float a, float b) { return a * b; }
__device__ __forceinline__ df rmul(df a, df b) { return ds::mul(a, b); }
__device__ __forceinline__ float two_over(float a) { return 2.f / a; }
__device__ __forceinline__ df two_over(df a) { return ds::div(df{2.f, 0.f}, a); }
__device__ __forceinline__ float rzero(float) { return 0.f; }
__device__ __forceinline__ df rzero(df) { return df{0.f, 0.f}; }
__device__ __forceinline__ void set_re(float2& a, float t) { a.x = t; }
__device__ __forceinline__ void set_re(dc& a, df t) { a.re = t; }
__device__ __forceinline__ void set_one(float2& a) { a.x = 1.f; }
__device__ __forceinline__ void set_one(dc& a) { a.re.h = 1.f; }
__device__ __forceinline__ float2 cneg(float2 a) { return fc(-a.x, -a.y); }
__device__ __forceinline__ dc cneg(dc a) { return dc{ds::neg(a.re), ds::neg(a.im)}; }

// G = [[c, s], [-conj(s), c]] with G [x; y] = [r; 0]; r returned in r.  The
// inputs are brought to order one by a power of two: entries behind a converged
// shift are tiny and their squares would leave the float range.
__device__ __forceinline__ void pow2_scales(float mx, float& sc, float& un) {
  const int be = min(max((__float_as_int(mx) >> 23) & 0xff, 1), 253);
  sc = __int_as_float((254 - be) << 23);
  un = __int_as_float(be << 23);
}
__device__ __forceinline__ Rot make_rot(float2 x, float2 y, float2& r) {
  Rot g;
  {
    const float a2 = norm2(x), n2 = a2 + norm2(y);
    if (a2 > 1e-9f && n2 < 1e9f) {  // the usual case: no scaling needed
      const float t = rsqrtf(a2 * n2);
      g.c = a2 * t;
      g.s = fc(fmaf(x.x, y.x, x.y * y.y) * t, fmaf(x.y, y.x, -x.x * y.y) * t);
      const float q = n2 * t;  // r = x / |x| sqrt(n2) = x n2 t
      r = fc(x.x * q, x.y * q);
      return g;
    }
  }
  float sc, un;
  pow2_scales(fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y))), sc, un);
  const float2 a = fc(x.x * sc, x.y * sc), b = fc(y.x * sc, y.y * sc);
  const float a2 = norm2(a), b2 = norm2(b);
  const float n2 = a2 + b2;
  if (b2 == 0.f) {
    g.c = 1.f;
    g.s = fc(0.f, 0.f);
    r = x;
  } else if (a2 < 1e-18f * n2) {
    const float t = rsqrtf(b2);
    g.c = 0.f;
    g.s = fc(b.x * t, -b.y * t);
    r = fc(b2 * t * un, 0.f);
  } else {
    const float t = rsqrtf(a2 * n2);
    g.c = a2 * t;
    g.s = fc(fmaf(a.x, b.x, a.y * b.y) * t, fmaf(a.y, b.x, -a.x * b.y) * t);
    const float q = n2 * t * un;  // r = x / |x| sqrt(n2) = x n2 t
    r = fc(a.x * q, a.y * q);
  }
  return g;
}
__device__ __forceinline__ float2 scale_f(float2 a, float t) { return fc(a.x * t, a.y * t); }
__device__ __forceinline__ dc scale_f(dc a, float t) {
  return dc{df{a.re.h * t, a.re.l * t}, df{a.im.h * t, a.im.l * t}};
}
__device__ __forceinline__ RotT<dc> make_rot(dc x, dc y, dc& r) {
  RotT<dc> g;
  float sc, un;
  pow2_scales(fmaxf(fmaxf(fabsf(x.re.h), fabsf(x.im.h)), fmaxf(fabsf(y.re.h), fabsf(y.im.h))), sc, un);
  const dc a = scale_f(x, sc), b = scale_f(y, sc);
  const df a2 = ds::cabs2(a), b2 = ds::cabs2(b), n2 = ds::add(a2, b2);
  if (b2.h == 0.f) {
    g.c = df{1.f, 0.f};
    g.s = ds::czero();
    r = x;
  } else if (a2.h < 1e-30f * n2.h) {
    const df t = rs(b2);
    g.c = df{0.f, 0.f};
    g.s = dc{ds::mul(b.re, t), ds::neg(ds::mul(b.im, t))};
    r = scale_f(dc{ds::mul(b2, t), df{0.f, 0.f}}, un);
  } else {
    const df t = rs(ds::mul(a2, n2));
    g.c = ds::mul(a2, t);
    g.s = ds::cscale(ds::cmulc_l(b, a), t);
    r = scale_f(ds::cscale(a, ds::mul(n2, t)), un);
  }
  return g;
}
__device__ __forceinline__ void rot_rows(float2& p, float2& q, const Rot& g) {  // (c p + s q, c q - conj(s) p)
  const float2 a = p, b = q;
  p = fc(fmaf(g.c, a.x, fmaf(g.s.x, b.x, -g.s.y * b.y)), fmaf(g.c, a.y, fmaf(g.s.x, b.y, g.s.y * b.x)));
  q = fc(fmaf(g.c, b.x, -fmaf(g.s.x, a.x, g.s.y * a.y)), fmaf(g.c, b.y, -fmaf(g.s.x, a.y, -g.s.y * a.x)));
}
__device__ __forceinline__ void rot_cols(float2& p, float2& q, const Rot& g) {  // (c p + conj(s) q, c q - s p)
  const float2 a = p, b = q;
  p = fc(fmaf(g.c, a.x, fmaf(g.s.x, b.x, g.s.y * b.y)), fmaf(g.c, a.y, fmaf(g.s.x, b.y, -g.s.y * b.x)));
  q = fc(fmaf(g.c, b.x, -fmaf(g.s.x, a.x, -g.s.y * a.y)), fmaf(g.c, b.y, -fmaf(g.s.x, a.y, g.s.y * a.x)));
}
// x c + y d + z e of double-single values: exact products, heads by TwoSum
__device__ __forceinline__ df dot3(df x, df c, df y, df d, df z, df e) {
  const float p0 = x.h * c.h, p1 = y.h * d.h, p2 = z.h * e.h;
  float t0 = fmaf(x.h, c.h, -p0), t1 = fmaf(y.h, d.h, -p1), t2 = fmaf(z.h, e.h, -p2);
  t0 = fmaf(x.h, c.l, t0);
  t1 = fmaf(y.h, d.l, t1);
  t2 = fmaf(z.h, e.l, t2);
  t0 = fmaf(x.l, c.h, t0);
  t1 = fmaf(y.l, d.h, t1);
  t2 = fmaf(z.l, e.h, t2);
  const df s1 = ds::two_sum(p1, p2);
  const df s0 = ds::two_sum(p0, s1.h);
  return ds::quick_two_sum(s0.h, s0.l + ((s1.l + t0) + (t1 + t2)));
}
__device__ __forceinline__ void rot_rows(dc& p, dc& q, const RotT<dc>& g) {
  const dc a = p, b = q;
  const df sxn = ds::neg(g.s.re), syn = ds::neg(g.s.im);
  p = dc{dot3(a.re, g.c, b.re, g.s.re, b.im, syn), dot3(a.im, g.c, b.im, g.s.re, b.re, g.s.im)};
  q = dc{dot3(b.re, g.c, a.re, sxn, a.im, syn), dot3(b.im, g.c, a.im, sxn, a.re, g.s.im)};
}
__device__ __forceinline__ void rot_cols(dc& p, dc& q, const RotT<dc>& g) {
  const dc a = p, b = q;
  const df sxn = ds::neg(g.s.re), syn = ds::neg(g.s.im);
  p = dc{dot3(a.re, g.c, b.re, g.s.re, b.im, g.s.im), dot3(a.im, g.c, b.im, g.s.re, b.re, syn)};
  q = dc{dot3(b.re, g.c, a.re, sxn, a.im, g.s.im), dot3(b.im, g.c, a.im, sxn, a.re, syn)};
}
__device__ __forceinline__ void put_rot(float4* list, long long at, const Rot& g, int k) {
  list[at] = make_float4(g.c, g.s.x, g.s.y, __int_as_float(k));
}
__device__ __forceinline__ void put_rot(float4* list, long long at, const RotT<dc>& g, int k) {
  list[2 * at] = make_float4(g.c.h, g.c.l, g.s.re.h, g.s.re.l);
  list[2 * at + 1] = make_float4(g.s.im.h, g.s.im.l, 0.f, __int_as_float(k));
}
template <class C>
struct RotEntry {
  RotT<C> g;
  int k;
};
__device__ __forceinline__ void get_rot(const float4* list, long long at, RotEntry<float2>& e) {
  const float4 a = __ldg(list + at);
  e.g = Rot{a.x, fc(a.y, a.z)};
  e.k = __float_as_int(a.w);
}
__device__ __forceinline__ void get_rot(const float4* list, long long at, RotEntry<dc>& e) {
  const float4 a = __ldg(list + 2 * at), b = __ldg(list + 2 * at + 1);
  e.g.c = df{a.x, a.y};
  e.g.s = dc{df{a.z, a.w}, df{b.x, b.y}};
  e.k = __float_as_int(b.w);
}
__device__ __forceinline__ Rot ident(float2) { return Rot{1.f, fc(0.f, 0.f)}; }
__device__ __forceinline__ RotT<dc> ident(dc) { return RotT<dc>{df{1.f, 0.f}, ds::czero()}; }

// packed upper-Hessenberg columns (rows 0 .. j + 2: the subdiagonal and a bulge)
__host__ __device__ __forceinline__ int offh(int j) { return j * (j + 5) / 2; }
// packed upper-triangular rows of an order-m matrix (columns i .. m - 1)
__host__ __device__ __forceinline__ int row_at(int m, int i) { return i * m - i * (i - 1) / 2; }
// packed upper-triangular columns (rows 0 .. j)
__host__ __device__ __forceinline__ int offu(int j) { return j * (j + 1) / 2; }

// The matrix a reduction works on: the projected matrix (FP32) or the kept block
// (double-single, its order on the device alone).
template <class C>
struct Red {
  const double2* A;   // [order][ld]
  int ld, order;      // order < 0: ctl[CTL_K0]
  C *work, *Hp, *Vr;
  typename Arith<C>::R* tau;
  int* len;           // rows of each reflector
  float4* rot;
  int max_steps, hmax_slot, steps_slot;
};
__device__ __forceinline__ int order_of(int order, const int* ctl) { return order < 0 ? ctl[CTL_K0] : order; }

// ---------------------------------------------------------------- 1. Hessenberg form
// One CTA; the matrix row-major in shared memory where it fits, else in global
// memory.  Per column: the reflector, its left product (thread groups over row
// classes, summed in shared memory), then one pass over the rows (a warp per
// row, the row in registers) that applies the left update, forms the right
// product and applies it.  NT x 32 >= the order.  The matrix is scaled to order
// one (pow2_scales of its largest entry; the reflectors and the chase's rotations
// do not see the scale): only squares of entries far below rounding leave the
// float range then, whatever the size of H.
template <class C, int NT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) mp_hess_kernel(const __grid_constant__ Red<C> D, int* ctl, int in_smem) {
  using R = typename Arith<C>::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ C v[NT * 32], w[NT * 32], part[THREADS + 32];
  __shared__ unsigned s_hmax;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (D.order < 0 && ctl[CTL_STATUS] != 0) return;
  const int m = order_of(D.order, ctl);
  C* A = in_smem ? reinterpret_cast<C*>(smem_raw) : D.work;
  if (tid == 0) s_hmax = 0u;
  __syncthreads();
  float hm = 0.f;
  for (int e = tid; e < m * m; e += THREADS) {
    const C h = Arith<C>::from(D.A[(long long)(e / m) * D.ld + e % m]);
    A[e] = h;
    hm = fmaxf(hm, abs1(h));
  }
  atomicMax(&s_hmax, __float_as_uint(hm));
  __syncthreads();
  float sc, un;
  pow2_scales(__uint_as_float(s_hmax), sc, un);
  for (int e = tid; e < m * m; e += THREADS) A[e] = scale_f(A[e], sc);
  __syncthreads();
  for (int c = 0; c + 2 < m; ++c) {
    // every warp forms the same reflector (no barrier for it); nr: rows and
    // columns c + 1 .. c + nr, up to the column's last nonzero.  After a restart
    // (a triangle, two coupling rows, a band) the support grows by two per
    // column, so the first third of the columns is cheap
    R t2 = rzero(R{});
    int nr = 1;
    for (int i = 1 + lane; i < m - 1 - c; i += 32) {
      const C x = A[(c + 1 + i) * m + c];
      if (abs1(x) > 0.f) nr = i + 1;
      t2 = radd(t2, cnorm(x));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      t2 = radd(t2, rshx(t2, o));
      nr = max(nr, __shfl_xor_sync(0xffffffffu, nr, o));
    }
    if (!(hi(t2) > 1e-34f)) {
      if (tid == 0) {
        D.tau[c] = rzero(R{});
        D.len[c] = 0;
      }
      continue;
    }
    const C x0 = A[(c + 1) * m + c];
    const R ax = cnorm(x0), n2 = radd(t2, ax), xn = rmul(n2, rs(n2));
    C alpha;  // -x0 / |x0| ||x||
    if (hi(ax) > 1e-34f) {
      alpha = cneg(scale(scale(x0, rs(ax)), xn));
    } else {
      alpha = Arith<C>::zero();
      set_re(alpha, xn);
      alpha = cneg(alpha);
    }
    const C v0 = sub(x0, alpha);
    const R tau = two_over(radd(cnorm(v0), t2));
    for (int i = tid; i < nr; i += THREADS) {
      const C vi = i == 0 ? v0 : A[(c + 1 + i) * m + c];
      v[i] = vi;
      D.Vr[(long long)c * m + c + 1 + i] = vi;
    }
    if (tid == 0) {
      D.tau[c] = tau;
      D.len[c] = nr;
    }
    __syncthreads();
    const int nc = m - 1 - c;  // columns of the left product
    const int ncp = (nc + 31) & ~31;
    const int G = max(1, THREADS / ncp), g = tid / ncp, jj = tid - g * ncp;
    if (ncp <= THREADS) {
      if (g < G && jj < nc) {
        C a0 = Arith<C>::zero(), a1 = a0;
        int i = g;
        for (; i + G < nr; i += 2 * G) {
          fma2c(a0, v[i], A[(c + 1 + i) * m + c + 1 + jj]);
          fma2c(a1, v[i + G], A[(c + 1 + i + G) * m + c + 1 + jj]);
        }
        if (i < nr) fma2c(a0, v[i], A[(c + 1 + i) * m + c + 1 + jj]);
        part[g * ncp + jj] = add(norm(a0), norm(a1));
      }
      __syncthreads();
      for (int j = tid; j < nc; j += THREADS) {
        C s = part[j];
        for (int q = 1; q < G; ++q) s = add(s, part[q * ncp + j]);
        w[j] = scale(s, tau);
      }
    }
    __syncthreads();
    C vr[NT], wr[NT];
#pragma unroll
    for (int q = 0; q < NT; ++q) {
      const int j = lane + 32 * q;
      vr[q] = j < nr ? v[j] : Arith<C>::zero();
      wr[q] = j < nc ? w[j] : Arith<C>::zero();
    }
    for (int i = warp; i < m; i += THREADS / 32) {
      const bool below = i > c && i - c <= nr;
      C* Ar = A + i * m + c + 1 + lane;
      C row[NT], u = Arith<C>::zero();
#pragma unroll
      for (int q = 0; q < NT; ++q) row[q] = lane + 32 * q < (below ? nc : nr) ? Ar[32 * q] : Arith<C>::zero();
      if (below) {
        const C vi = cneg(v[i - c - 1]);
#pragma unroll
        for (int q = 0; q < NT; ++q)
          if (32 * q < nc) row[q] = fmadd(row[q], vi, wr[q]);
      }
#pragma unroll
      for (int q = 0; q < NT; ++q)
        if (32 * q < nr) fma2(u, row[q], vr[q]);
      u = cneg(scale(lanes_sum(norm(u), 16), tau));
#pragma unroll
      for (int q = 0; q < NT; ++q)
        if (32 * q < nr) {
          if (lane + 32 * q < (below ? nc : nr)) Ar[32 * q] = fmaddc(row[q], u, vr[q]);
        } else if (below && lane + 32 * q < nc) {
          Ar[32 * q] = row[q];
        }
      if (below && lane == 0) A[i * m + c] = i == c + 1 ? alpha : Arith<C>::zero();
    }
    __syncthreads();
  }
  __syncthreads();
  for (int e = tid; e < m * m; e += THREADS) {
    const int j = e / m, i = e % m;
    if (i <= j + 2) D.Hp[offh(j) + i] = i <= j + 1 ? A[i * m + j] : Arith<C>::zero();
  }
  if (tid == 0) {
    if (D.order >= 0) {  // the step's first kernel: the control block starts here
      ctl[CTL_STATUS] = 0;
      ctl[CTL_K0] = 0;
      ctl[CTL_STEPS2] = 0;
      for (int q = 0; q < 4; ++q) ctl[CTL_RMAX + q] = 0;
    }
    ctl[D.steps_slot] = 0;
    ctl[D.hmax_slot] = (int)s_hmax;
  }
}

// ---------------------------------------------------------------- 2. the chase
// eigenvalues of the trailing nb x nb block (approximate: a shift needs no
// more), by one warp: at most one single-shift QR sweep per eigenvalue on an
// FP32 copy in shared memory, lane j owning column j, then row j.  The copy is
// taken relative to the last diagonal entry, so that the shift nearest it keeps
// its full relative accuracy in the double-single form.
__device__ __forceinline__ float2 wilkinson(float2 p, float2 q, float2 r, float2 d) {  // of [[p, q], [r, d]], nearer d
  const float2 t = fc(0.5f * (p.x - d.x), 0.5f * (p.y - d.y)), bc = mulf(q, r);
  float2 s2 = mulf(t, t);
  s2 = sqrtf2(fc(s2.x + bc.x, s2.y + bc.y));
  const float2 r1 = fc(t.x + s2.x, t.y + s2.y), r2 = fc(t.x - s2.x, t.y - s2.y);
  const float2 den = norm2(r1) >= norm2(r2) ? r1 : r2;
  if (!(norm2(den) > 0.f)) return d;
  const float2 z = divf2(bc, den);
  return fc(d.x - z.x, d.y - z.y);
}
template <class C>
__device__ void chain_shifts(const C* H, int ihi, int nb, float2 (*a)[kNB + 1], float2* mu, bool exceptional) {
  const int lane = threadIdx.x & 31, o = ihi - nb + 1;
  const C last = H[offh(ihi) + ihi];
  for (int e = lane; e < nb * nb; e += 32) {
    const int i = e / nb, j = e % nb;
    a[i][j] = i > j + 1 ? fc(0.f, 0.f)
                        : (i == j ? head(sub(H[offh(o + j) + o + i], last)) : head(H[offh(o + j) + o + i]));
  }
  __syncwarp();
  for (int hi = nb - 1; hi > 0; --hi) {
    if (!(abs1(a[hi][hi - 1]) <= 1e-2f * (abs1(a[hi][hi]) + abs1(a[hi - 1][hi - 1])))) {
      const float2 s = wilkinson(a[hi - 1][hi - 1], a[hi - 1][hi], a[hi][hi - 1], a[hi][hi]);
      for (int k = 0; k < hi; ++k) {
        const float2 x = k == 0 ? fc(a[0][0].x - s.x, a[0][0].y - s.y) : a[k][k - 1];
        const float2 y = k == 0 ? a[1][0] : a[k + 1][k - 1];
        float2 r;
        const Rot g = make_rot(x, y, r);
        __syncwarp();
        if (lane < nb && lane >= k - 1) rot_rows(a[k][lane], a[k + 1][lane], g);
        __syncwarp();
        if (lane <= min(k + 2, hi)) rot_cols(a[lane][k], a[lane][k + 1], g);
        __syncwarp();
      }
    }
    __syncwarp();
  }
  if (lane < nb) mu[lane] = a[nb - 1 - lane][nb - 1 - lane];
  __syncwarp();
  if (exceptional && lane < nb) mu[lane].x += 0.75f * abs1(H[offh(ihi - 1) + ihi]);
}

__device__ __forceinline__ float2 plus_f(float2 a, float2 b) { return fc(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ dc plus_f(dc a, float2 b) { return ds::cadd(a, dc{df{b.x, 0.f}, df{b.y, 0.f}}); }
// a subdiagonal entry is negligible below rel x its diagonal neighbours or abs x
// the largest entry: FP32 rounding of the whole reduction is ~1e-6 of |H|, so
// 1e-7 there; the limits of the order-m kernel in double-single
template <class C>
struct Defl;
template <>
struct Defl<float2> {
  static constexpr float rel = 1.2e-7f, abs = 1e-7f;
};
template <>
struct Defl<dc> {
  static constexpr float rel = 4e-15f, abs = 1e-14f;
};

template <class C, bool SMEM>
__global__ void __launch_bounds__(kChaseThreads, 1) mp_chase_kernel(const __grid_constant__ Red<C> D, int* ctl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float2 s_mu[kNB];
  __shared__ float2 s_blk[kNB][kNB + 1];
  __shared__ int s_l, s_nblk, s_next, s_most, s_bad;
  __shared__ short2 s_small[kMaxM / 2 + 1];
  if (ctl[CTL_STATUS] != 0) return;
  const int m = order_of(D.order, ctl), tid = threadIdx.x, lane = tid & 31, b = tid >> 5;
  C* H = SMEM ? reinterpret_cast<C*>(smem_raw) : D.Hp;
  if (SMEM)
    for (int e = tid; e < offh(m); e += kChaseThreads) H[e] = D.Hp[e];
  float sc, un;
  pow2_scales(__int_as_float(ctl[D.hmax_slot]), sc, un);
  const float hmax = __int_as_float(ctl[D.hmax_slot]) * sc;
  int ihi = m - 1, its = 0, sweeps = 0, step = 0, status = 0;
  if (tid == 0) s_nblk = s_next = s_most = s_bad = 0;
  __syncthreads();
  while (ihi > 0) {
    // the largest index with a negligible subdiagonal
    if (tid == 0) s_l = 0;
    __syncthreads();
    for (int i = tid + 1; i <= ihi; i += kChaseThreads) {
      const float t = abs1(H[offh(i - 1) + i - 1]) + abs1(H[offh(i) + i]);
      if (abs1(H[offh(i - 1) + i]) <= fmaxf(Defl<C>::rel * t, Defl<C>::abs * hmax)) atomicMax(&s_l, i);
    }
    __syncthreads();
    const int l = s_l;
    if (l > 0 && tid == 0) H[offh(l - 1) + l] = Arith<C>::zero();
    if (l == ihi) {
      __syncthreads();
      --ihi;
      its = 0;
      continue;
    }
    if (ihi - l < kSmall) {  // left for the second phase
      if (tid == 0) s_small[s_nblk++] = make_short2((short)l, (short)ihi);
      __syncthreads();
      ihi = l - 1;
      its = 0;
      continue;
    }
    ++its;
    const int nb = min(kNB, (ihi - l + 1) / 3);  // at least 11: the blocks here have order 33 and more
    const int T = (ihi - l) + 3 * (nb - 1);
    if (++sweeps > 30 * m + 30 || step + T > D.max_steps) {
      status = 1;
      break;
    }
    const C last = H[offh(ihi) + ihi];
    if (b == 0) chain_shifts(H, ihi, nb, s_blk, s_mu, its % 10 == 0);
    __syncthreads();
    const C mu = plus_f(last, s_mu[min(b, nb - 1)]);
    for (int t = 0; t < T; ++t, ++step) {
      const int k = l + t - 3 * b;
      const bool act = b < nb && k >= l && k < ihi;
      RotT<C> g = ident(C{});
      C r = Arith<C>::zero();
      if (act) {
        C x, y;
        if (k == l) {
          x = sub(H[offh(l) + l], mu);
          y = H[offh(l) + l + 1];
        } else {
          x = H[offh(k - 1) + k];
          y = H[offh(k - 1) + k + 1];
        }
        g = make_rot(x, y, r);
        __syncwarp();  // at the top of a block, x and y lie in the columns rotated next
        // columns k + lane, + 32, ... (two at a time: independent loads in flight);
        // offh(j + 32) - offh(j) = 32 j + 592
        int j = k + lane, at = offh(j) + k, step32 = 32 * j + 592;
        for (; j + 32 <= ihi; j += 64) {
          C *p = H + at, *q = p + step32;
          C h0 = p[0], h1 = p[1], g0 = q[0], g1 = q[1];
          rot_rows(h0, h1, g);
          rot_rows(g0, g1, g);
          p[0] = h0;
          p[1] = h1;
          q[0] = g0;
          q[1] = g1;
          at += 2 * step32 + 1024;
          step32 += 2048;
        }
        if (j <= ihi) {
          C* p = H + at;
          C h0 = p[0], h1 = p[1];
          rot_rows(h0, h1, g);
          p[0] = h0;
          p[1] = h1;
        }
      }
      __syncthreads();
      if (act) {
        const int top = min(k + 2, ihi);
        C *p0 = H + offh(k), *p1 = p0 + k + 3;
        int i = l + lane;
        for (; i + 32 <= top; i += 64) {
          C h0 = p0[i], h1 = p1[i], g0 = p0[i + 32], g1 = p1[i + 32];
          rot_cols(h0, h1, g);
          rot_cols(g0, g1, g);
          p0[i] = h0;
          p1[i] = h1;
          p0[i + 32] = g0;
          p1[i + 32] = g1;
        }
        if (i <= top) {
          C h0 = p0[i], h1 = p1[i];
          rot_cols(h0, h1, g);
          p0[i] = h0;
          p1[i] = h1;
        }
      }
      if (lane == 0) {
        if (act && k > l) {
          H[offh(k - 1) + k] = r;
          H[offh(k - 1) + k + 1] = Arith<C>::zero();
        }
        put_rot(D.rot, (long long)step * kNB + b, g, act ? k : -1);
      }
      __syncthreads();
    }
  }
  __syncthreads();
  // ---- the small blocks, a warp each: single shifts, lane j owning a column of
  // the row rotations, then a row of the column rotations.  A warp's rotations
  // fill its own slot of the list from the last common step on; those of
  // different blocks touch different columns.
  const int nblk = s_nblk;
  int mine = step;
  if (status == 0) {
    for (;;) {
      int q = 0;
      if (lane == 0) q = atomicAdd(&s_next, 1);
      q = __shfl_sync(0xffffffffu, q, 0);
      // one decision for the warp: another warp may set s_bad between two lanes' reads
      if (q >= nblk || __any_sync(0xffffffffu, s_bad)) break;
      const int l0 = s_small[q].x;
      int top = s_small[q].y, it = 0, total = 0;
      while (top > l0) {
        // lane i tests the subdiagonal of row l0 + 1 + i
        const int row = l0 + 1 + lane;
        bool small = false;
        if (row <= top) {
          const float t = abs1(H[offh(row - 1) + row - 1]) + abs1(H[offh(row) + row]);
          small = abs1(H[offh(row - 1) + row]) <= fmaxf(Defl<C>::rel * t, Defl<C>::abs * hmax);
        }
        const unsigned hit = __ballot_sync(0xffffffffu, small);
        const int l = hit ? l0 + 32 - __clz(hit) : l0;
        if (l == top) {
          --top;
          it = 0;
          continue;
        }
        ++it;
        if (++total > 40 * kSmall || mine + top - l > D.max_steps) {
          s_bad = 1;
          break;
        }
        const C last = H[offh(top) + top];
        float2 mf = wilkinson(head(sub(H[offh(top - 1) + top - 1], last)), head(H[offh(top) + top - 1]),
                              head(H[offh(top - 1) + top]), fc(0.f, 0.f));
        if (it % 10 == 0) mf.x += 0.75f * abs1(H[offh(top - 1) + top]);
        const C mu = plus_f(last, mf);
        __syncwarp();
        for (int k = l; k < top; ++k, ++mine) {
          C x, y, r;
          if (k == l) {
            x = sub(H[offh(l) + l], mu);
            y = H[offh(l) + l + 1];
          } else {
            x = H[offh(k - 1) + k];
            y = H[offh(k - 1) + k + 1];
          }
          const RotT<C> g = make_rot(x, y, r);
          __syncwarp();
          const int j = k + lane;
          if (j <= top) {
            C* p = H + offh(j) + k;
            C h0 = p[0], h1 = p[1];
            rot_rows(h0, h1, g);
            p[0] = h0;
            p[1] = h1;
          }
          __syncwarp();
          const int i = l + lane;
          if (i <= min(k + 2, top)) {
            C *p0 = H + offh(k), *p1 = p0 + k + 3;
            C h0 = p0[i], h1 = p1[i];
            rot_cols(h0, h1, g);
            p0[i] = h0;
            p1[i] = h1;
          }
          if (lane == 0) {
            if (k > l) {
              H[offh(k - 1) + k] = r;
              H[offh(k - 1) + k + 1] = Arith<C>::zero();
            }
            put_rot(D.rot, (long long)mine * kNB + b, g, k);
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) atomicMax(&s_most, mine);
  }
  __syncthreads();
  if (s_bad) status = 1;
  if (status == 0) {
    for (int q = mine + lane; q < s_most; q += 32) put_rot(D.rot, (long long)q * kNB + b, ident(C{}), -1);
    step = s_most;
  }
  if (tid == 0) {
    if (status) ctl[CTL_STATUS] = status;
    ctl[D.steps_slot] = status ? 0 : step;
  }
}

// ---------------------------------------------------------------- 3. rows x (reflectors, rotations)
// Rows of Q (or of V) times the reflectors of a reduction (Vr set) and the
// rotations of a list.  Two rows per warp in shared memory; a lane holds one
// row and one of the (at most 16, disjoint) rotations of a step, so the steps of
// a warp need no barrier beyond its own.  src NULL: rows of the identity.
constexpr int kApplyWarps = 4, kRows = 32 / kNB;  // rows per warp
__device__ __forceinline__ double2 to_out(dc a) { return ds::cto(a); }
__device__ __forceinline__ float2 to_out(float2 a) { return a; }
__device__ __forceinline__ float2 load_row(const float2* p, float2) { return *p; }
__device__ __forceinline__ dc load_row(const double2* p, dc) { return Arith<dc>::from(*p); }
template <class C, class E, int AHEAD, int NT>
__global__ void __launch_bounds__(32 * kApplyWarps)
    mp_apply_kernel(const __grid_constant__ Red<C> D, int* ctl, int nrows, const E* src, E* dst, int lds, int reflect) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (ctl[CTL_STATUS] != 0) return;
  const int m = order_of(D.order, ctl);
  const int row = (blockIdx.x * kApplyWarps + warp) * kRows + lane / kNB, b = lane % kNB;
  C* q = reinterpret_cast<C*>(smem_raw) + (size_t)(warp * kRows + lane / kNB) * (m + 1);
  const bool on = row < nrows;
  for (int j = b; j < m; j += kNB) {
    C x = Arith<C>::zero();
    if (on && src) x = load_row(src + (long long)row * lds + j, C{});
    else if (on && j == row) set_one(x);
    q[j] = x;
  }
  __syncwarp();
  if (reflect) {
    // all lanes on one row at a time, the reflector in registers (the next one
    // loaded meanwhile)
    C* q0 = reinterpret_cast<C*>(smem_raw) + (size_t)(warp * kRows) * (m + 1);
    C vn[NT];
    typename Arith<C>::R tn = D.tau[0];
    int ln = D.len[0];
#pragma unroll
    for (int q = 0; q < NT; ++q) vn[q] = lane + 32 * q < ln ? D.Vr[1 + lane + 32 * q] : Arith<C>::zero();
    for (int c = 0; c + 2 < m; ++c) {
      C v[NT];
      const typename Arith<C>::R tau = tn;
      const int len = ln;
#pragma unroll
      for (int q = 0; q < NT; ++q) v[q] = vn[q];
      if (c + 3 < m) {
        tn = D.tau[c + 1];
        ln = D.len[c + 1];
        const C* src_v = D.Vr + (long long)(c + 1) * m + c + 2 + lane;
#pragma unroll
        for (int q = 0; q < NT; ++q) vn[q] = lane + 32 * q < ln ? src_v[32 * q] : Arith<C>::zero();
      }
      if (hi(tau) == 0.f) continue;
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        C* qr = q0 + r * (m + 1) + c + 1 + lane;
        C x[NT], u = Arith<C>::zero();
#pragma unroll
        for (int q = 0; q < NT; ++q) {
          if (32 * q < len) {
            x[q] = lane + 32 * q < len ? qr[32 * q] : Arith<C>::zero();
            fma2(u, x[q], v[q]);
          }
        }
        u = cneg(scale(lanes_sum(norm(u), 16), tau));
#pragma unroll
        for (int q = 0; q < NT; ++q)
          if (lane + 32 * q < len) qr[32 * q] = fmaddc(x[q], u, v[q]);
      }
      __syncwarp();  // columns change lanes with c
    }
  }
  __syncwarp();
  const int n = ctl[D.steps_slot];
  RotEntry<C> pre[AHEAD];
#pragma unroll
  for (int a = 0; a < AHEAD; ++a) {
    pre[a].k = -1;
    if (a < n) get_rot(D.rot, (long long)a * kNB + b, pre[a]);
  }
  for (int s0 = 0; s0 < n; s0 += AHEAD) {
#pragma unroll
    for (int a = 0; a < AHEAD; ++a) {
      const RotEntry<C> e = pre[a];
      pre[a].k = -1;
      if (s0 + a + AHEAD < n) get_rot(D.rot, (long long)(s0 + a + AHEAD) * kNB + b, pre[a]);
      if (e.k >= 0) {
        C h0 = q[e.k], h1 = q[e.k + 1];
        rot_cols(h0, h1, e.g);
        q[e.k] = h0;
        q[e.k + 1] = h1;
      }
      __syncwarp();
    }
  }
  if (on)
    for (int j = b; j < m; j += kNB) dst[(long long)row * lds + j] = to_out(q[j]);
}

// ---------------------------------------------------------------- 4./6. small products
// a correction is left out once the residual is at double-single rounding
__device__ __forceinline__ bool settled(const int* ctl, int it) {
  return __int_as_float(ctl[CTL_RMAX + it]) <= 8e-15f * __int_as_float(ctl[CTL_HMAX]);
}
// 16 x 16 outputs per CTA of 4 x 256 threads, the contraction split over the
// four groups (sums combined in FP64); dimensions from the control block (k is
// known on the device alone).
enum { OP_P = 0, OP_T, OP_W, OP_G, OP_R, OP_Y, OP_F, OP_S, OP_N };
constexpr bool op_ds(int op) { return op == OP_W || op == OP_G || op == OP_R || op == OP_S; }

struct DsC {
  float rh, rl, ih, il;
};
template <bool UNIT>  // UNIT: an entry of orthonormal vectors, of no use below 2^-74
__device__ __forceinline__ DsC ds_split(double2 v) {
  DsC r;
  if constexpr (UNIT) {
    ds::split_flush(v.x, r.rh, r.rl);
    ds::split_flush(v.y, r.ih, r.il);
  } else {
    ds::split_wide(v.x, r.rh, r.rl);
    ds::split_wide(v.y, r.ih, r.il);
  }
  return r;
}

template <int OP>
__global__ void __launch_bounds__(1024) mp_gemm_kernel(const __grid_constant__ MpJob J, const double2* V,
                                                       double2* Vout, int it) {
  constexpr bool DS = op_ds(OP);
  using E = typename std::conditional<DS, DsC, float2>::type;
  __shared__ E sa[4][16][17];
  __shared__ E sb[4][16][16];
  __shared__ double2 red[3][256];
  if (J.ctl[CTL_STATUS] != 0) return;
  if ((OP == OP_Y || OP == OP_F) && settled(J.ctl, it)) return;
  const int m = J.m, k0 = J.ctl[CTL_K0], kc = J.kcap;
  const int rows = (OP == OP_G || OP == OP_S) ? k0 : (OP == OP_Y ? m - k0 : m);
  const int cols = (OP == OP_P || OP == OP_T) ? m : k0;
  const int K = (OP == OP_R || OP == OP_N) ? k0 : (OP == OP_F ? m - k0 : m);
  const int r0 = blockIdx.y * 16, c0 = blockIdx.x * 16;
  if (r0 >= rows || c0 >= cols || (OP == OP_T && r0 > c0 + 15)) return;
  const int tid = threadIdx.x & 255, g = threadIdx.x >> 8;
  const int tx = tid & 15, ty = tid >> 4;
  const double2* Gm = J.G;
  // operands: a(r, k), b(k, c)
  auto lda_d = [&](int r, int k) -> double2 {
    if (OP == OP_W) return J.H[(long long)r * J.ld + k];
    if (OP == OP_G || OP == OP_S) {
      const double2 x = V[(long long)k * kc + r];
      return make_double2(x.x, -x.y);
    }
    return V[(long long)r * kc + k];  // OP_R
  };
  auto ldb_d = [&](int k, int c) -> double2 {
    if (OP == OP_W || OP == OP_S) return V[(long long)k * kc + c];
    if (OP == OP_G) return J.W[(long long)k * kc + c];
    return Gm[(long long)k * J.ld + c];  // OP_R
  };
  auto lda_f = [&](int r, int k) -> float2 {
    if (OP == OP_P) return f2(J.H[(long long)r * J.ld + k]);
    if (OP == OP_T) {
      const float2 x = J.Q[(long long)k * m + r];
      return fc(x.x, -x.y);
    }
    if (OP == OP_Y) {
      const float2 x = J.Q[(long long)k * m + k0 + r];
      return fc(x.x, -x.y);
    }
    if (OP == OP_F) return J.Q[(long long)r * m + k0 + k];
    return f2(V[(long long)r * kc + k]);  // OP_N
  };
  auto ldb_f = [&](int k, int c) -> float2 {
    if (OP == OP_P) return J.Q[(long long)k * m + c];
    if (OP == OP_T) return J.P[(long long)k * m + c];
    if (OP == OP_Y) return J.R32[(long long)k * kc + c];
    if (OP == OP_F) return J.X[(long long)k * kc + c];
    return J.S32[(long long)k * kc + c];  // OP_N
  };
  const int kq = ((K + 3) / 4 + 15) / 16 * 16;  // K of one group, whole stages
  const int kb = g * kq, ke = min(K, kb + kq);
  double vx = 0.0, vy = 0.0;
  if constexpr (DS) {
    float rs = 0.f, re = 0.f, is = 0.f, ie = 0.f;
    for (int kk = 0; kk < kq; kk += 16) {
      const int ka = kb + kk;
      const bool conj_t = OP == OP_G || OP == OP_S;  // a is stored [k][r]: read along r
      const int ar = conj_t ? tx : ty, ak = conj_t ? ty : tx;
      sa[g][ar][ak] = ds_split<OP != OP_W>(r0 + ar < rows && ka + ak < ke ? lda_d(r0 + ar, ka + ak) : make_double2(0.0, 0.0));
      sb[g][ty][tx] = ds_split<OP == OP_W || OP == OP_S>(c0 + tx < cols && ka + ty < ke ? ldb_d(ka + ty, c0 + tx) : make_double2(0.0, 0.0));
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const DsC a = sa[g][ty][q], b = sb[g][q][tx];
        ds::fma_acc(rs, re, a.rh, a.rl, b.rh, b.rl);
        ds::fma_acc(is, ie, a.rh, a.rl, b.ih, b.il);
        ds::fma_acc(rs, re, -a.ih, -a.il, b.ih, b.il);
        ds::fma_acc(is, ie, a.ih, a.il, b.rh, b.rl);
      }
      __syncthreads();
    }
    vx = (double)rs + (double)re;
    vy = (double)is + (double)ie;
  } else {
    float2 acc = fc(0.f, 0.f);
    for (int kk = 0; kk < kq; kk += 16) {
      const int ka = kb + kk;
      const bool conj_t = OP == OP_T || OP == OP_Y;
      const int ar = conj_t ? tx : ty, ak = conj_t ? ty : tx;
      sa[g][ar][ak] = r0 + ar < rows && ka + ak < ke ? lda_f(r0 + ar, ka + ak) : fc(0.f, 0.f);
      sb[g][ty][tx] = c0 + tx < cols && ka + ty < ke ? ldb_f(ka + ty, c0 + tx) : fc(0.f, 0.f);
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 16; ++q) fma2(acc, sa[g][ty][q], sb[g][q][tx]);
      __syncthreads();
    }
    vx = acc.x;
    vy = acc.y;
  }
  if (g > 0) red[g - 1][tid] = make_double2(vx, vy);
  __syncthreads();
  if (g > 0) return;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    vx += red[q][tid].x;
    vy += red[q][tid].y;
  }
  const int r = r0 + ty, c = c0 + tx;
  const bool in = r < rows && c < cols;
  if (OP == OP_R) {  // R = W - V G, rounded to FP32 (it is small), and its largest entry
    float mx = 0.f;
    if (in) {
      const double2 wv = J.W[(long long)r * kc + c];
      const float2 x = f2(make_double2(wv.x - vx, wv.y - vy));
      J.R32[(long long)r * kc + c] = x;
      mx = abs1(x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) atomicMax(reinterpret_cast<unsigned*>(J.ctl + CTL_RMAX + it), __float_as_uint(mx));
    return;
  }
  if (!in) return;
  if (OP == OP_P) J.P[(long long)r * m + c] = fc((float)vx, (float)vy);
  if (OP == OP_T && r <= c) J.T[offu(c) + r] = fc((float)vx, (float)vy);
  if (OP == OP_W) J.W[(long long)r * kc + c] = make_double2(vx, vy);
  if (OP == OP_G) J.G[(long long)r * J.ld + c] = make_double2(vx, vy);
  if (OP == OP_Y) J.X[(long long)r * kc + c] = fc((float)vx, (float)vy);
  if (OP == OP_S) J.S32[(long long)r * kc + c] = fc((float)(vx - (r == c ? 1.0 : 0.0)), (float)vy);
  if (OP == OP_F) {
    const double2 v = V[(long long)r * kc + c];
    Vout[(long long)r * kc + c] = make_double2(v.x - vx, v.y - vy);
  }
  if (OP == OP_N) {
    const double2 v = V[(long long)r * kc + c];
    Vout[(long long)r * kc + c] = make_double2(v.x - 0.5 * vx, v.y - 0.5 * vy);
  }
}

// ---------------------------------------------------------------- 5. ordering
// The kept Ritz values (keep of smallest |theta - i sig_im|, more while the cut
// would split values closer than 2e-6 |H|, at most kmax) move to the leading
// block by adjacent swaps: in every step each kept value below an unkept one
// swaps, all at once (disjoint pairs), so the bubbles travel together.
__global__ void __launch_bounds__(512, 1) mp_order_kernel(const __grid_constant__ MpJob J, int in_smem) {
  extern __shared__ float2 smem[];
  __shared__ float key[kMaxM];
  __shared__ unsigned char sel[kMaxM + 1];
  __shared__ float sorted[kMaxM];
  __shared__ int swq[kMaxM / 2 + 1];
  __shared__ Rot rots[kMaxM / 2 + 1];
  __shared__ int s_cnt, s_k0;
  if (J.ctl[CTL_STATUS] != 0) return;
  const int m = J.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float2* T = in_smem ? smem : J.T;
  if (in_smem)
    for (int e = tid; e < offu(m); e += 512) T[e] = J.T[e];
  __syncthreads();
  const float hmax = __int_as_float(J.ctl[CTL_HMAX]);
  if (tid < m) {
    const float2 t = T[offu(tid) + tid];
    key[tid] = hypotf(t.x, t.y - (float)J.sig_im);
  }
  __syncthreads();
  int rank = 0;
  if (tid < m) {
    const float a = key[tid];
    for (int q = 0; q < m; ++q) rank += key[q] < a || (key[q] == a && q < tid);
    sorted[rank] = a;
  }
  __syncthreads();
  if (tid == 0) {
    int k = min(J.keep, m);
    while (k < m - 1 && k < J.kmax && k < J.kcap && !(sorted[k] - sorted[k - 1] > 2e-6f * hmax)) ++k;
    s_k0 = k;
  }
  __syncthreads();
  const int k0 = s_k0;
  if (tid < m) sel[tid] = rank < k0 ? 1 : 0;
  __syncthreads();
  int step = 0, status = 0;
  for (int it = 0; it < 2 * m; ++it) {
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    if (tid + 1 < m && !sel[tid] && sel[tid + 1]) swq[atomicAdd(&s_cnt, 1)] = tid;
    __syncthreads();
    const int n = s_cnt;
    if (n == 0) break;
    const int ng = (n + kNB - 1) / kNB;
    if (step + ng > J.max_steps2) {
      status = 1;
      break;
    }
    if (tid < ng * kNB) {
      Rot g = ident(float2{});
      if (tid < n) {
        const int q = swq[tid];
        const float2 a = T[offu(q) + q], d = T[offu(q + 1) + q + 1];
        float2 r;
        g = make_rot(T[offu(q + 1) + q], fc(d.x - a.x, d.y - a.y), r);
        rots[tid] = g;
      }
      put_rot(J.rot2, (long long)step * kNB + tid, g, tid < n ? swq[tid] : -1);
    }
    __syncthreads();
    for (int s = warp; s < n; s += 16) {  // rows q, q + 1
      const int q = swq[s];
      const Rot g = rots[s];
      for (int j = q + 2 + lane; j < m; j += 32) {
        float2* p = T + offu(j) + q;
        float2 h0 = p[0], h1 = p[1];
        rot_rows(h0, h1, g);
        p[0] = h0;
        p[1] = h1;
      }
    }
    __syncthreads();
    for (int s = warp; s < n; s += 16) {  // columns q, q + 1
      const int q = swq[s];
      const Rot g = rots[s];
      float2 *p0 = T + offu(q), *p1 = T + offu(q + 1);
      for (int i = lane; i < q; i += 32) {
        float2 h0 = p0[i], h1 = p1[i];
        rot_cols(h0, h1, g);
        p0[i] = h0;
        p1[i] = h1;
      }
      if (lane == 0) {
        const float2 t = p0[q];
        p0[q] = p1[q + 1];
        p1[q + 1] = t;
        sel[q] = 1;
        sel[q + 1] = 0;
      }
    }
    step += ng;
    __syncthreads();
  }
  if (in_smem)
    for (int e = tid; e < offu(m); e += 512) J.T[e] = T[e];
  if (tid < m) J.rad[tid] = sorted[tid];
  for (int i = warp; i < m; i += 16)
    for (int j = i + lane; j < m; j += 32) J.Tr[row_at(m, i) + j - i] = T[offu(j) + i];
  if (tid == 0) {
    J.ctl[CTL_K0] = status ? 0 : k0;
    J.ctl[CTL_STEPS2] = step;
    J.ctl[CTL_STATUS] = status;
  }
}

// V = Q[:, 0:k] in FP64
__global__ void mp_init_kernel(const __grid_constant__ MpJob J, double2* V) {
  if (J.ctl[CTL_STATUS] != 0) return;
  const int k0 = J.ctl[CTL_K0];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < J.m * k0; e += gridDim.x * blockDim.x) {
    const int r = e / k0, c = e % k0;
    const float2 q = J.Q[(long long)r * J.m + c];
    V[(long long)r * J.kcap + c] = make_double2(q.x, q.y);
  }
}

// ---------------------------------------------------------------- 6. T22 X - X T11 = Y
// X (m - k x k, in place of Y) along the anti-diagonals (row from the bottom,
// column from the left): a warp per entry, its row of T22 and column of T11
// against the finished entries.  T22 is read by rows (Tr, packed by rows, in
// shared memory where it fits beside X): a column-packed T22 costs a sector per
// lane and took 1.9 us per anti-diagonal at order 150.
__global__ void __launch_bounds__(1024, 1) mp_sylv_kernel(const __grid_constant__ MpJob J, int where, int it) {
  extern __shared__ float2 smem[];
  if (J.ctl[CTL_STATUS] != 0 || settled(J.ctl, it)) return;
  const int m = J.m, k0 = J.ctl[CTL_K0], p = m - k0, kc = J.kcap;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float floor_ = 1e-7f * __int_as_float(J.ctl[CTL_HMAX]);
  float2* X = where >= 1 ? smem : J.X;
  const int ldx = where >= 1 ? (k0 | 1) : kc;
  if (where >= 1)
    for (int e = tid; e < p * k0; e += 1024) X[(e / k0) * ldx + e % k0] = J.X[(long long)(e / k0) * kc + e % k0];
  // row i of T22: entries [i][i'], i' >= i, at row_at(m, k0 + i) + i' - i
  const float2* R = J.Tr + row_at(m, k0);
  if (where == 2) {
    float2* sR = smem + p * ldx;
    for (int e = tid; e < offu(p); e += 1024) sR[e] = R[e];
    R = sR;
  }
  __syncthreads();
  for (int d = 0; d < p + k0 - 1; ++d) {
    const int j0 = max(0, d - (p - 1)), j1 = min(k0 - 1, d);
    for (int j = j0 + warp; j <= j1; j += 32) {
      const int i = p - 1 - (d - j);
      float2 s = fc(0.f, 0.f);
      // sum_{i' > i} T22[i][i'] x[i'][j] - sum_{j' < j} x[i][j'] T11[j'][j]
      const float2* Ri = R + row_at(p, i);
      for (int q = 1 + lane; q < p - i; q += 32) fma2(s, Ri[q], X[(i + q) * ldx + j]);
      for (int q = lane; q < j; q += 32) {
        const float2 t = J.T[offu(j) + q];
        fma2(s, fc(-t.x, -t.y), X[i * ldx + q]);
      }
      s = warp_sum2(s);
      if (lane == 0) {
        const float2 a = Ri[0], bb = J.T[offu(j) + j];
        float2 den = fc(a.x - bb.x, a.y - bb.y);
        if (abs1(den) < floor_) den = fc(floor_, 0.f);
        const float2 y = X[i * ldx + j];
        X[i * ldx + j] = divf2(fc(y.x - s.x, y.y - s.y), den);
      }
    }
    __syncthreads();
  }
  if (where >= 1)
    for (int e = tid; e < p * k0; e += 1024) J.X[(long long)(e / k0) * kc + e % k0] = X[(e / k0) * ldx + e % k0];
}

// the verdict on the corrections: |H V - V G| beyond double-single rounding
// fails the step
__global__ void mp_verdict_kernel(const __grid_constant__ MpJob J) {
  if (J.ctl[CTL_STATUS] != 0) return;
  const float r = __int_as_float(J.ctl[CTL_RMAX + 3]), h = __int_as_float(J.ctl[CTL_HMAX]);
  if (!(r <= 1e-13f * h)) J.ctl[CTL_STATUS] = 2;
}

// ---------------------------------------------------------------- 7. results
// A warp per kept Ritz value i: Z[:, i] = V[:, i], T[0:i+1, i], theta_i,
// (B V)[:, i], the unit eigenvector s_i of T (FP64 back substitution, the lanes
// sharing each dot product) and ||B V s_i||.  V, W = H V and G = V^H H V are the
// final ones; G is upper triangular to double-single rounding.
__global__ void __launch_bounds__(128) mp_results_kernel(const __grid_constant__ MpJob J, const double2* V) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (J.ctl[CTL_STATUS] != 0) return;
  const int m = J.m, k0 = J.ctl[CTL_K0], kc = J.kcap;
  const int lane = threadIdx.x & 31, i = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (i >= k0) return;
  auto wsum = [](double2 s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    return s;
  };
  for (int r = lane; r < m; r += 32) J.Z[(long long)r * J.ld + i] = V[(long long)r * kc + i];
  for (int r = lane; r < k0; r += 32)
    J.H[(long long)r * J.ld + i] = r <= i ? J.G[(long long)r * J.ld + i] : make_double2(0.0, 0.0);
  const double2 lam = J.G[(long long)i * J.ld + i];
  if (lane == 0) J.theta[i] = lam;
  double2* s = reinterpret_cast<double2*>(smem_raw) + (size_t)(threadIdx.x >> 5) * kc;
  const double smin = fmax(1e-14 * swi::cabs(lam), 1e-290);
  if (lane == 0) s[i] = make_double2(1.0, 0.0);
  __syncwarp();
  double nrm = 1.0;
  for (int j = i - 1; j >= 0; --j) {
    double2 acc = make_double2(0.0, 0.0);
    for (int l = j + 1 + lane; l <= i; l += 32) cfma(acc, J.G[(long long)j * J.ld + l], s[l]);
    acc = wsum(acc);
    double2 den = swi::csub(J.G[(long long)j * J.ld + j], lam);
    if (swi::cabs(den) < smin) den = make_double2(smin, 0.0);
    const double2 x = swi::cdiv(make_double2(-acc.x, -acc.y), den);
    if (lane == 0) s[j] = x;
    nrm += swi::cabs2(x);
    __syncwarp();
  }
  nrm = 1.0 / sqrt(nrm);
  for (int l = lane; l < k0; l += 32)
    J.S[(long long)l * J.ld + i] = l <= i ? swi::cscale(s[l], nrm) : make_double2(0.0, 0.0);
  double r2 = 0.0;
  for (int r = 0; r < J.b; ++r) {
    // row r of B V against s_i: the columns this needs are formed by the warp itself
    double2 acc = make_double2(0.0, 0.0);
    for (int l = lane; l <= i; l += 32) cfma(acc, J.BV[(long long)r * J.ld + l], s[l]);
    acc = wsum(acc);
    r2 += swi::cabs2(acc);
  }
  if (lane == 0) {
    J.resid[i] = sqrt(r2) * nrm;
    for (int r = 0; r < J.b; ++r) J.Bz[(long long)r * J.ld + i] = J.BV[(long long)r * J.ld + i];
  }
}

// B V, a warp per entry
__global__ void mp_couple_kernel(const __grid_constant__ MpJob J, const double2* V) {
  if (J.ctl[CTL_STATUS] != 0) return;
  const int k0 = J.ctl[CTL_K0], lane = threadIdx.x & 31;
  for (int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); e < J.b * k0;
       e += gridDim.x * (blockDim.x >> 5)) {
    const int r = e / k0, c = e % k0;
    double2 s = make_double2(0.0, 0.0);
    for (int q = lane; q < J.m; q += 32) cfma(s, J.B[(long long)r * J.ld + q], V[(long long)q * J.kcap + c]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    if (lane == 0) J.BV[(long long)r * J.ld + c] = s;
  }
}

// The step's outcome: kept count, wanted pairs at the tolerance, status, work.
// The kept set was chosen by FP32 values.  When all wanted pairs are at the
// tolerance (the window would end), the nearest value left out must lie beyond
// the last wanted one by more than those values are off: 16 times the largest
// change of a kept value's distance between the two forms (values of the same
// matrix, of conditions that differ).  If not, the step gives up, and the
// full-order step decides.
__global__ void __launch_bounds__(512) mp_outcome_kernel(const __grid_constant__ MpJob J) {
  __shared__ int s_n;
  __shared__ unsigned s_off;
  __shared__ double s_last;
  const int k0 = J.ctl[CTL_K0], st = J.ctl[CTL_STATUS];
  if (threadIdx.x == 0) {
    s_n = 0;
    s_off = 0u;
    s_last = 0.0;
  }
  __syncthreads();
  if (st == 0)
    for (int i = threadIdx.x; i < k0; i += blockDim.x) {
      const double2 ti = J.theta[i];
      const double ai = swi::cabs(make_double2(ti.x, ti.y - J.sig_im));
      int rank = 0;
      for (int q = 0; q < k0; ++q) {
        const double2 tq = J.theta[q];
        const double aq = swi::cabs(make_double2(tq.x, tq.y - J.sig_im));
        if (aq < ai || (aq == ai && q < i)) ++rank;
      }
      if (rank < J.nwant && J.resid[i] <= J.tol_abs) atomicAdd(&s_n, 1);
      if (rank == J.nwant - 1) s_last = ai;
      atomicMax(&s_off, __float_as_uint((float)fabs(ai - (double)J.rad[rank])));
    }
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool unsure = st == 0 && s_n >= J.nwant && k0 < J.m &&
                        !((double)J.rad[k0] - 16.0 * (double)__uint_as_float(s_off) > s_last);
    J.ordinfo[0] = k0;
    J.ordinfo[1] = s_n;
    J.ordinfo[2] = st != 0 || unsure ? 1 : 0;
    J.ordinfo[3] = (int)(((long long)J.ctl[CTL_STEPSK] * 4 * 2 * k0) >> 10);  // Givens pair updates / 1024
  }
}

template <class K>
void allow_smem(K kernel, size_t bytes) {
  if (bytes > 16 * 1024) smem_opt_in(reinterpret_cast<const void*>(kernel));  // beside the kernels' static share
}

}  // namespace

void smem_opt_in(const void* kernel) {
  static std::mutex mu;
  static std::set<std::pair<int, const void*>> done;
  int dev = 0;
  SWI_CUDA_TRY(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  if (done.count({dev, kernel})) return;
  cudaFuncAttributes fa;
  SWI_CUDA_TRY(cudaFuncGetAttributes(&fa, kernel));
  int most = 0;
  SWI_CUDA_TRY(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  SWI_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    most - (int)fa.sharedSizeBytes));
  done.insert({dev, kernel});
}

size_t mp_schur_bytes(int m, int kcap, int ld, int b) { return mp_schur_layout(nullptr, nullptr, m, kcap, ld, b); }

size_t mp_schur_layout(MpJob* J, void* base, int m, int kcap, int ld, int b) {
  char* p = static_cast<char*>(base);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) & ~size_t(255);
    return p ? static_cast<void*>(p + at) : nullptr;
  };
  const size_t mm = (size_t)m * m, mk = (size_t)m * kcap, kk = (size_t)kcap * kcap;
  MpJob t{};
  t.max_steps = 60 * m + 2000;
  t.max_steps2 = (m + kNB - 1) / kNB * 2 * m;
  t.max_stepsk = 60 * kcap + 2000;
  t.ctl = static_cast<int*>(take(64));
  t.H32 = static_cast<float2*>(take(8 * mm));
  t.Hp = static_cast<float2*>(take(8 * (size_t)offh(m)));
  t.Vr = static_cast<float2*>(take(8 * mm));
  t.tau = static_cast<float*>(take(4 * (size_t)m));
  t.rad = static_cast<float*>(take(4 * (size_t)m));
  t.len = static_cast<int*>(take(4 * (size_t)m));
  t.Q = static_cast<float2*>(take(8 * mm));
  t.P = static_cast<float2*>(take(8 * mm));
  t.T = static_cast<float2*>(take(8 * (size_t)offu(m)));
  t.Tr = static_cast<float2*>(take(8 * (size_t)offu(m)));
  t.rot = static_cast<float4*>(take(16 * (size_t)kNB * t.max_steps));
  t.rot2 = static_cast<float4*>(take(16 * (size_t)kNB * t.max_steps2));
  t.V[0] = static_cast<double2*>(take(16 * mk));
  t.V[1] = static_cast<double2*>(take(16 * mk));
  t.W = static_cast<double2*>(take(16 * mk));
  t.R32 = static_cast<float2*>(take(8 * mk));
  t.X = static_cast<float2*>(take(8 * mk));
  t.S32 = static_cast<float2*>(take(8 * kk));
  t.G = static_cast<double2*>(take(16 * (size_t)kcap * ld));
  t.BV = static_cast<double2*>(take(16 * (size_t)b * ld));
  t.Gd = take(sizeof(dc) * kk);
  t.Gp = take(sizeof(dc) * (size_t)offh(kcap));
  t.Vk = take(sizeof(dc) * kk);
  t.tauk = take(sizeof(df) * (size_t)kcap);
  t.rotk = static_cast<float4*>(take(32 * (size_t)kNB * t.max_stepsk));
  if (J) *J = t;
  return off;
}

// Orders below 48 stay with the full-order kernel.  Measured per call, a quarter
// kept (this form / that one): order 48 1.5 / 4.6 ms, 40 1.4 / 3.4, 32 1.2 / 2.3, 20
// 0.9 / 1.1; the solvers' default bases have 130 vectors and more (150: 6.4 / 41).
// Room for eight values beyond the kept ones is what the cut may need at a tie.
bool mp_schur_takes(int m, int keep, int kmax) {
  return m >= 48 && m <= kMpMaxOrder && keep >= 3 && keep <= kmax && keep + 8 < m;
}

void launch_schur_mp(const SchurJob& S, void* work, int kcap, cudaStream_t s, long long* launches) {
  const int m = S.m;
  if (!mp_schur_takes(m, S.keep, S.kmax) || kcap < S.keep || kcap > S.kmax || S.keep < S.nwant)
    throw Error{SWI_ECUDA, "mixed-precision Schur step: sizes out of range"};
  MpJob J;
  mp_schur_layout(&J, work, m, kcap, S.ld, S.b);
  J.m = m;
  J.ld = S.ld;
  J.b = S.b;
  J.keep = S.keep;
  J.kmax = S.kmax;
  J.kcap = kcap;
  J.nwant = S.nwant;
  J.sig_im = S.sig_im;
  J.tol_abs = S.tol_abs;
  J.H = S.H;
  J.Z = S.Z;
  J.B = S.B;
  J.Bz = S.Bz;
  J.theta = S.theta;
  J.resid = S.resid;
  J.S = S.S;
  J.ordinfo = S.ordinfo;
  long long n = 0;
  auto done = [&]() {
    SWI_CHECK_LAUNCH();
    ++n;
  };
  auto tiles = [](int n_) { return (unsigned)((n_ + 15) / 16); };
  auto row_blocks = [](int n_) { return (unsigned)((n_ + kRows * kApplyWarps - 1) / (kRows * kApplyWarps)); };
  // ---- FP32 Schur form
  const Red<float2> D{S.H, S.ld, m, J.H32, J.Hp, J.Vr, J.tau, J.len, J.rot, J.max_steps, CTL_HMAX, CTL_STEPS};
  const size_t sq = 8 * (size_t)m * m;
  const int hs = sq <= kSmemMatrix - 28 * 1024 ? 1 : 0;  // beside the reflector, its product and partial sums
  auto hess = [&](auto kernel) {
    allow_smem(kernel, hs ? sq : 0);
    kernel<<<1, 1024, hs ? sq : 0, s>>>(D, J.ctl, hs);
  };
  if (m <= 160) hess(mp_hess_kernel<float2, 5, 1024>);
  else if (m <= 256) hess(mp_hess_kernel<float2, 8, 1024>);
  else hess(mp_hess_kernel<float2, 16, 1024>);
  done();
  const size_t ph = 8 * (size_t)offh(m);
  const int cs = ph <= kSmemMatrix ? 1 : 0;
  auto chase = [&](auto kernel, const auto& P, size_t bytes) {
    allow_smem(kernel, bytes);
    kernel<<<1, kChaseThreads, bytes, s>>>(P, J.ctl);
  };
  if (cs) chase(mp_chase_kernel<float2, true>, D, ph);
  else chase(mp_chase_kernel<float2, false>, D, 0);
  done();
  const size_t qs = 8 * (size_t)kApplyWarps * kRows * (m + 1);
  auto applyq = [&](const Red<float2>& P, const float2* src, int reflect) {
    auto go = [&](auto kernel) {
      allow_smem(kernel, qs);
      kernel<<<row_blocks(m), 32 * kApplyWarps, qs, s>>>(P, J.ctl, m, src, J.Q, m, reflect);
    };
    if (m <= 160) go(mp_apply_kernel<float2, float2, 16, 5>);
    else if (m <= 256) go(mp_apply_kernel<float2, float2, 16, 8>);
    else go(mp_apply_kernel<float2, float2, 16, 16>);
  };
  applyq(D, nullptr, 1);
  done();
  const dim3 gmm(tiles(m), tiles(m)), gmk(tiles(kcap), tiles(m)), gkk(tiles(kcap), tiles(kcap));
  mp_gemm_kernel<OP_P><<<gmm, 1024, 0, s>>>(J, nullptr, nullptr, 0);
  done();
  mp_gemm_kernel<OP_T><<<gmm, 1024, 0, s>>>(J, nullptr, nullptr, 0);
  done();
  const size_t pu = 8 * (size_t)offu(m);
  const int os = pu <= kSmemMatrix - 12 * 1024 ? 1 : 0;  // beside the keys and swap lists
  allow_smem(mp_order_kernel, os ? pu : 0);
  mp_order_kernel<<<1, 512, os ? pu : 0, s>>>(J, os);
  done();
  Red<float2> D2 = D;
  D2.rot = J.rot2;
  D2.steps_slot = CTL_STEPS2;
  applyq(D2, J.Q, 0);
  done();
  // ---- the kept subspace to double-single accuracy
  int cur = 0;
  mp_init_kernel<<<(m * kcap + 255) / 256, 256, 0, s>>>(J, J.V[0]);
  done();
  auto orth = [&]() {  // V <- V (3 I - V^H V) / 2
    mp_gemm_kernel<OP_S><<<gkk, 1024, 0, s>>>(J, J.V[cur], nullptr, 0);
    done();
    mp_gemm_kernel<OP_N><<<gmk, 1024, 0, s>>>(J, J.V[cur], J.V[cur ^ 1], 0);
    done();
    cur ^= 1;
  };
  auto project = [&]() {
    mp_gemm_kernel<OP_W><<<gmk, 1024, 0, s>>>(J, J.V[cur], nullptr, 0);
    done();
    mp_gemm_kernel<OP_G><<<gkk, 1024, 0, s>>>(J, J.V[cur], nullptr, 0);
    done();
  };
  auto residual = [&](int it) {
    project();
    mp_gemm_kernel<OP_R><<<gmk, 1024, 0, s>>>(J, J.V[cur], nullptr, it);
    done();
  };
  const size_t xs = 8 * (size_t)(m - S.keep) * (size_t)(kcap | 1), rs22 = 8 * (size_t)offu(m - S.keep);
  const int where = xs + rs22 <= kSmemMatrix ? 2 : (xs <= kSmemMatrix ? 1 : 0);
  const size_t sylv_smem = where == 2 ? xs + rs22 : (where == 1 ? xs : 0);
  allow_smem(mp_sylv_kernel, sylv_smem);
  orth();
  for (int it = 0; it < 3; ++it) {
    residual(it);
    mp_gemm_kernel<OP_Y><<<gmk, 1024, 0, s>>>(J, nullptr, nullptr, it);
    done();
    mp_sylv_kernel<<<1, 1024, sylv_smem, s>>>(J, where, it);
    done();
    mp_gemm_kernel<OP_F><<<gmk, 1024, 0, s>>>(J, J.V[cur], J.V[cur], it);
    done();
    orth();
  }
  residual(3);
  mp_verdict_kernel<<<1, 1, 0, s>>>(J);
  done();
  // ---- the double-single Schur form of the kept block, applied to V
  const Red<dc> K{J.G, S.ld, -1, static_cast<dc*>(J.Gd), static_cast<dc*>(J.Gp), static_cast<dc*>(J.Vk),
                  static_cast<df*>(J.tauk), J.len, J.rotk, J.max_stepsk, CTL_HMAXK, CTL_STEPSK};
  const size_t kq = sizeof(dc) * (size_t)kcap * kcap;
  const int ks = kq <= kSmemMatrix - 44 * 1024 ? 1 : 0;
  auto hessk = [&](auto kernel) {
    allow_smem(kernel, ks ? kq : 0);
    kernel<<<1, 512, ks ? kq : 0, s>>>(K, J.ctl, ks);
  };
  if (kcap <= 96) hessk(mp_hess_kernel<dc, 3, 512>);
  else if (kcap <= 256) hessk(mp_hess_kernel<dc, 8, 512>);
  else hessk(mp_hess_kernel<dc, 16, 512>);
  done();
  const size_t kp = sizeof(dc) * (size_t)offh(kcap);
  const int kc = kp <= kSmemMatrix ? 1 : 0;
  if (kc) chase(mp_chase_kernel<dc, true>, K, kp);
  else chase(mp_chase_kernel<dc, false>, K, 0);
  done();
  const size_t ks_rows = sizeof(dc) * (size_t)kApplyWarps * kRows * (kcap + 1);
  auto applyk = [&](auto kernel) {
    allow_smem(kernel, ks_rows);
    kernel<<<row_blocks(m), 32 * kApplyWarps, ks_rows, s>>>(K, J.ctl, m, J.V[cur], J.V[cur], kcap, 1);
  };
  if (kcap <= 96) applyk(mp_apply_kernel<dc, double2, 8, 3>);
  else if (kcap <= 256) applyk(mp_apply_kernel<dc, double2, 8, 8>);
  else applyk(mp_apply_kernel<dc, double2, 8, 16>);
  done();
  orth();
  project();
  mp_couple_kernel<<<32, 256, 0, s>>>(J, J.V[cur]);
  done();
  const size_t rs_ = sizeof(double2) * 4 * (size_t)kcap;
  mp_results_kernel<<<(unsigned)((kcap + 3) / 4), 128, rs_, s>>>(J, J.V[cur]);
  done();
  mp_outcome_kernel<<<1, 512, 0, s>>>(J);
  done();
  if (launches) *launches += n;
}

}  // namespace swi
