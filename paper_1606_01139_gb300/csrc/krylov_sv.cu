// Gram-Schmidt passes of the single-vector Krylov loop (Section 2.1: one new
// vector per window and step, as in the implicitly restarted Arnoldi method the
// paper runs), batched over the windows of one solve; the same passes serve
// windows that add a block of nb = 2 vectors per step (a template parameter:
// each pass still streams the basis once, for both new vectors).
//
// Every window keeps its basis row-major, Q [N][ld] (a grid point's basis
// coefficients are contiguous), so each pass of classical Gram-Schmidt against
// the new vectors w streams the basis once.  Classical Gram-Schmidt twice is
// three passes: the Gram (FP32 products of the heads), the update fused with
// the second Gram (the accurate pass), and the update by the second pass's
// small coefficients (FP32 products).  Two element types share the kernels
// through an arithmetic policy:
//  - complex64 with FP32 arithmetic (the reduced-precision form);
//  - complex128 in double-single arithmetic: every FP64 operand split into a
//    float head and tail from its bit fields, products exact up to their
//    tails (FMA), sums TwoSum-compensated, ~2^-46 relative per term (GB300's
//    FP64 rate would cap these passes near a third of the HBM bandwidth); the
//    new vectors themselves are kept in split form while they are
//    orthogonalised.
//
//  sv_gram_kernel:   part[chunk][i][b] = sum_{rows of chunk} conj(Q[r, i]) w[r, b]
//                    (a block per 32-column slab and row chunk, one column per lane)
//  sv_update_kernel: w[r, :] -= Q[r, :] c, then the next Gram's partials: one
//                    pass over Q for both (double-single)
//  sv_update_fast_kernel: w[r, :] -= Q[r, :] c for the second pass's small
//                    coefficients (FP32 products of the heads), then the
//                    partials of w^H w
//  sv_wgram_kernel:  part[chunk][a][b] = sum_{rows of chunk} conj(w[r, a]) w[r, b],
//                    of a block as it is or times its Cholesky factor's inverse
//  sv_reduce_kernel: FP64 sums of the chunk partials, added into columns of H;
//                    for w^H w the Cholesky factor of the block (Cholesky-QR)
// Chunks hold at most 1024 rows: the per-lane FP32 (or double-single) partial
// sums stay short, chunks are combined in FP64.
#include <algorithm>

#include "ds.cuh"
#include "swi_internal.cuh"

namespace swi {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// ----------------------------------------------------------------- arithmetic policies
// w^H w entries are accumulated in double-single (heads and error terms of the
// real and imaginary parts) by lane 0 of a warp, on the FP32 pipe
struct Gds {
  float rh, re, ih, ie;
};
__device__ __forceinline__ void gds_acc(Gds& a, float xrh, float xrl, float xih, float xil, float yrh, float yrl,
                                        float yih, float yil) {  // a += conj(x) y
  ds::fma_acc(a.rh, a.re, xrh, xrl, yrh, yrl);
  ds::fma_acc(a.rh, a.re, xih, xil, yih, yil);
  ds::fma_acc(a.ih, a.ie, xrh, xrl, yih, yil);
  ds::fma_acc(a.ih, a.ie, -xih, -xil, yrh, yrl);
}

struct PolC64 {
  using T = float2;   // basis element
  using A = float2;   // accumulator
  using S = float2;   // an element prepared for products (no split in FP32)
  // a += conj(q) * w
  __device__ static void conj_mac(A& a, T q, T w) {
    a.x = fmaf(q.x, w.x, fmaf(q.y, w.y, a.x));
    a.y = fmaf(q.x, w.y, fmaf(-q.y, w.x, a.y));
  }
  __device__ static A shfl_xor(A a, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
  }
  __device__ static T from_c(double2 c) { return make_float2((float)c.x, (float)c.y); }
  // the new vectors w: complex64, like the basis
  using W = float2;
  __device__ static S wload(W v) { return v; }
  __device__ static W wstore(S v) { return v; }
  __device__ static S wsub(S w, A d) { return make_float2(w.x - d.x, w.y - d.y); }
  __device__ static void gacc(Gds& g, S x, S y) { gds_acc(g, x.x, 0.f, x.y, 0.f, y.x, 0.f, y.y, 0.f); }
  __device__ static T out(S v) { return v; }  // a basis entry
  // the FP32 passes: the same arithmetic
  using F = float2;
  __device__ static F fzero() { return make_float2(0.f, 0.f); }
  __device__ static void fconj_mac(F& a, T q, S w) { conj_mac(a, q, w); }
  __device__ static F fadd(F a, F b) { return make_float2(a.x + b.x, a.y + b.y); }
  __device__ static double2 fto_d(F a) { return make_double2(a.x, a.y); }
  __device__ static A fto_A(F a) { return a; }
  __device__ static float2 head2(T c) { return c; }
  // elements staged in shared memory for the accurate pass, and its accumulator
  using ST = float2;
  using AC = float2;
  __host__ __device__ static int ldt(int ncols) { return (ncols + 15) / 16 * 16 + 8; }  // 8-byte rows: offset half a bank cycle
  __device__ static ST stage(T v) { return v; }
  static constexpr bool kStaged = true;  // a copied entry needs no conversion
  __device__ static ST restage(ST v) { return v; }
  __device__ static float2 raw_head(ST v) { return v; }
  __device__ static ST swap(ST v) { return make_float2(v.y, v.x); }
  __device__ static ST of_w(S v) { return v; }
  __device__ static AC azero() { return make_float2(0.f, 0.f); }
  __device__ static void tmac(AC& a, ST q, ST c, ST cs) {  // a += q c
    a = __ffma2_rn(make_float2(q.x, q.x), c, a);
    a = __ffma2_rn(make_float2(-q.y, q.y), cs, a);
  }
  __device__ static void tcmac(AC& a, ST q, ST w, ST wsw) {  // a += conj(q) w
    a = __ffma2_rn(make_float2(q.x, q.x), w, a);
    a = __ffma2_rn(make_float2(q.y, -q.y), wsw, a);
  }
  __device__ static AC tadd(AC a, AC b) { return __fadd2_rn(a, b); }
  __device__ static AC tshx(AC a, int o) { return shfl_xor(a, o); }
  __device__ static double2 tto_d(AC a) { return make_double2(a.x, a.y); }
  __device__ static S wsub_t(S w, AC d) { return wsub(w, d); }
  __device__ static S sshx(S a, int o) { return shfl_xor(a, o); }
  __device__ static S smul2(S a, double2 r, S b, double2 t, bool two) {  // a r + b t, FP64 products
    double re = a.x * r.x - a.y * r.y, im = a.x * r.y + a.y * r.x;
    if (two) {
      re += b.x * t.x - b.y * t.y;
      im += b.x * t.y + b.y * t.x;
    }
    return make_float2((float)re, (float)im);
  }
};

// Operands are split by ds::split_flush (no FP64 instruction on any path): the
// basis entries, new vectors and coefficients of the loop lie far inside its
// range.
__device__ __forceinline__ float hi_fast(double x) {  // the head of ds::split_flush alone
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned int top = (unsigned int)(b >> 32);
  const int e0 = (int)((top >> 20) & 0x7ff);
  const int e = min(max(e0, 949), 1149);
  const unsigned int fb =
      ((unsigned int)(e - 896) << 23 | ((unsigned int)(b >> 29) & 0x7fffffu)) + ((unsigned int)(b >> 28) & 1u);
  return e0 < 949 ? 0.f : __uint_as_float((top & 0x80000000u) | fb);
}

struct PolDs {
  using T = double2;
  struct A {
    float rh, re, ih, ie;
  };
  struct S {  // heads and tails of the real and imaginary parts
    float rh, rl, ih, il;
  };
  __device__ static T from_c(double2 c) { return c; }
  // the new vectors w: kept in split form (heads and tails as floats) while
  // they are orthogonalised, so that forming w - Q c takes no FP64 instruction
  using W = float4;
  __device__ static S wload(W v) { return S{v.x, v.y, v.z, v.w}; }
  __device__ static W wstore(S v) { return make_float4(v.rh, v.rl, v.ih, v.il); }
  __device__ static S wsub(S w, A d) {  // w - d, renormalised to head + tail
    const ds::df r = ds::add(ds::df{w.rh, w.rl}, ds::df{-d.rh, -d.re});
    const ds::df i = ds::add(ds::df{w.ih, w.il}, ds::df{-d.ih, -d.ie});
    return S{r.h, r.l, i.h, i.l};
  }
  __device__ static void gacc(Gds& g, S x, S y) { gds_acc(g, x.rh, x.rl, x.ih, x.il, y.rh, y.rl, y.ih, y.il); }
  __device__ static T out(const S& v) {  // a basis entry (no FP64 instruction)
    return make_double2(ds::join_bits(v.rh, v.rl), ds::join_bits(v.ih, v.il));
  }
  // the FP32 passes: products of the heads in FP32 (the first Gram of
  // classical Gram-Schmidt twice, and the update by the second pass's small
  // coefficients, need no more)
  using F = float2;
  __device__ static F fzero() { return make_float2(0.f, 0.f); }
  __device__ static void fconj_mac(F& a, T q, const S& w) {  // a += conj(q) w
    const float qr = hi_fast(q.x), qi = hi_fast(q.y);
    a.x = fmaf(qr, w.rh, fmaf(qi, w.ih, a.x));
    a.y = fmaf(qr, w.ih, fmaf(-qi, w.rh, a.y));
  }
  __device__ static F fadd(F a, F b) { return make_float2(a.x + b.x, a.y + b.y); }
  __device__ static double2 fto_d(F a) { return make_double2(a.x, a.y); }
  __device__ static A fto_A(F a) { return A{a.x, 0.f, a.y, 0.f}; }
  __device__ static float2 head2(T c) { return make_float2(hi_fast(c.x), hi_fast(c.y)); }
  // elements staged in shared memory for the accurate pass: heads (re, im), tails
  // (re, im), so that real and imaginary parts go through packed FP32x2
  // instructions; the accumulator likewise
  using ST = float4;
  struct AC {
    float2 h, l;
  };
  __host__ __device__ static int ldt(int ncols) { return ncols; }
  __device__ static ST stage(T v) {
    ST o;
    ds::split_flush(v.x, o.x, o.z);
    ds::split_flush(v.y, o.y, o.w);
    return o;
  }
  static constexpr bool kStaged = false;
  // an entry as copied (the bytes of a T)
  __device__ static T raw(ST v) {
    return make_double2(__hiloint2double(__float_as_int(v.y), __float_as_int(v.x)),
                        __hiloint2double(__float_as_int(v.w), __float_as_int(v.z)));
  }
  __device__ static ST restage(ST v) { return stage(raw(v)); }
  __device__ static float2 raw_head(ST v) { return head2(raw(v)); }
  __device__ static ST swap(ST v) { return make_float4(v.y, v.x, v.w, v.z); }
  __device__ static ST of_w(const S& v) { return make_float4(v.rh, v.ih, v.rl, v.il); }
  __device__ static AC azero() { return AC{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
  __device__ static float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
  // a += (uh + ul) (vh + vl) per component: exact product up to its tail, head by
  // TwoSum; nh = -uh, so that the product arrives negated and no operand of a
  // packed instruction needs its sign turned
  __device__ static void mulv(AC& a, float2 uh, float2 nh, float2 ul, float2 vh, float2 vl) {
    const float2 np = __fmul2_rn(nh, vh);
    float2 e = __ffma2_rn(uh, vh, np);
    e = __ffma2_rn(uh, vl, e);
    e = __ffma2_rn(ul, vh, e);
    const float2 t = sub2(a.h, np);
    const float2 bp = sub2(t, a.h);
    const float2 err = sub2(sub2(a.h, sub2(t, bp)), __fadd2_rn(np, bp));
    a.h = t;
    a.l = __fadd2_rn(a.l, __fadd2_rn(err, e));
  }
  __device__ static void tmac(AC& a, ST q, ST c, ST cs) {  // a += q c
    mulv(a, make_float2(q.x, q.x), make_float2(-q.x, -q.x), make_float2(q.z, q.z), make_float2(c.x, c.y),
         make_float2(c.z, c.w));
    mulv(a, make_float2(-q.y, q.y), make_float2(q.y, -q.y), make_float2(-q.w, q.w), make_float2(cs.x, cs.y),
         make_float2(cs.z, cs.w));
  }
  __device__ static void tcmac(AC& a, ST q, ST w, ST wsw) {  // a += conj(q) w
    mulv(a, make_float2(q.x, q.x), make_float2(-q.x, -q.x), make_float2(q.z, q.z), make_float2(w.x, w.y),
         make_float2(w.z, w.w));
    mulv(a, make_float2(q.y, -q.y), make_float2(-q.y, q.y), make_float2(q.w, -q.w), make_float2(wsw.x, wsw.y),
         make_float2(wsw.z, wsw.w));
  }
  __device__ static AC tadd(AC a, AC b) {
    const float2 t = __fadd2_rn(a.h, b.h);
    const float2 bp = sub2(t, a.h);
    const float2 err = __fadd2_rn(sub2(a.h, sub2(t, bp)), sub2(b.h, bp));
    return AC{t, __fadd2_rn(__fadd2_rn(a.l, b.l), err)};
  }
  __device__ static float2 sx(float2 a, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
  }
  __device__ static AC tshx(AC a, int o) { return AC{sx(a.h, o), sx(a.l, o)}; }
  __device__ static double2 tto_d(AC a) {
    return make_double2((double)a.h.x + (double)a.l.x, (double)a.h.y + (double)a.l.y);
  }
  __device__ static S sshx(const S& a, int o) {
    const float2 r = sx(make_float2(a.rh, a.rl), o), i = sx(make_float2(a.ih, a.il), o);
    return S{r.x, r.y, i.x, i.y};
  }
  __device__ static S wsub_t(const S& w, AC d) { return wsub(w, A{d.h.x, d.l.x, d.h.y, d.l.y}); }
  __device__ static S smul2(const S& a, double2 r, const S& b, double2 t, bool two) {  // a r + b t in double-single
    const ST rs = stage(r), ts = stage(t);
    AC s = azero();
    tmac(s, of_w(a), rs, swap(rs));
    if (two) tmac(s, of_w(b), ts, swap(ts));
    const ds::df x = ds::two_sum(s.h.x, s.l.x), y = ds::two_sum(s.h.y, s.l.y);
    return S{x.h, x.l, y.h, y.l};
  }
};

// a basis entry (8 or 16 bytes) from global to shared memory, asynchronously; zero if !on
template <class ST>
__device__ __forceinline__ void copy_entry(ST* dst, const ST* src, bool on) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = on ? (int)sizeof(ST) : 0;
  if constexpr (sizeof(ST) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ----------------------------------------------------------------- Gram pass
template <class Pol, int NB>
__global__ void __launch_bounds__(kThreads) sv_gram_kernel(const __grid_constant__ SvBatch batch, int N, int rpc) {
  using T = typename Pol::T;
  const SvJob& J = batch.job[blockIdx.z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.y * 32 + lane;
  if (blockIdx.y * 32 >= J.ncols) return;  // this job has fewer slabs (uniform over the block)
  using Wt = typename Pol::W;
  const T* __restrict__ Q = static_cast<const T*>(J.Q);
  const Wt* __restrict__ w = static_cast<const Wt*>(J.w);
  const int r0 = blockIdx.x * rpc, r1 = min(N, r0 + rpc);
  const bool on = col < J.ncols;
  __shared__ double2 red[kWarps][NB][32];
  int r = r0 + warp;
  // four rows per iteration, their loads issued together (memory-level
  // parallelism), two interleaved accumulators per column of w
  typename Pol::F a0[NB], a1[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) a0[b] = a1[b] = Pol::fzero();
  for (; r + 3 * kWarps < r1; r += 4 * kWarps) {
    T q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = on ? __ldg(Q + (long long)(r + u * kWarps) * J.ldq + col) : T{};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int b = 0; b < NB; ++b)
        Pol::fconj_mac((u & 1) ? a1[b] : a0[b], q[u], Pol::wload(w[(long long)(r + u * kWarps) * J.ldw + b]));
  }
  for (; r < r1; r += kWarps) {
    const T q0 = on ? __ldg(Q + (long long)r * J.ldq + col) : T{};
#pragma unroll
    for (int b = 0; b < NB; ++b) Pol::fconj_mac(a0[b], q0, Pol::wload(w[(long long)r * J.ldw + b]));
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) red[warp][b][lane] = Pol::fto_d(Pol::fadd(a0[b], a1[b]));
  __syncthreads();
  if (warp == 0 && on) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      double2 s = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < kWarps; ++k) {
        s.x += red[k][b][lane].x;
        s.y += red[k][b][lane].y;
      }
      J.part[(long long)blockIdx.x * J.ldp + col * NB + b] = s;
    }
  }
}

// ----------------------------------------------------------------- update fused with the second Gram
// The accurate pass: w[r, :] -= Q[r, :] c, then the partials of Q^H w, in
// double-single (FP32 in the complex64 form).  A tile of RT rows is staged once
// in shared memory, split into heads and tails as it arrives; the update then
// gives each row to 256 / RT lanes (three to five shuffle levels per row), the
// Gram gives each column to a thread (to 256 / columns row groups when there
// are fewer than 256), which needs no shuffles and no accumulators beyond its
// own column's.  FP32 issue bounds it (192 operations per basis entry at
// nb = 2, half the issue slots when packed), so every entry is split once.
// Measured with its reduction (one window of 48x48x96, ~58 to 116 columns, nb = 2):
// 306 us (354 alone at 116 columns: 59% of the issue slots); a warp per
// row with both products from global memory, splitting twice and reducing over
// 32 lanes, took 459 us (2,000 rows in four windows: 112 us, now 24).
template <class Pol, int RT, int NC2, int NB, int NBUF>
__global__ void __launch_bounds__(kThreads, NC2 == 1 ? 3 : 1)
    sv_update_kernel(const __grid_constant__ SvBatch batch, int N, int rpc) {
  using T = typename Pol::T;
  using ST = typename Pol::ST;
  using AC = typename Pol::AC;
  using Sp = typename Pol::S;
  using Wt = typename Pol::W;
  constexpr int L = kThreads / RT;  // lanes per row of the update
  static_assert(L <= 32, "a row's lanes lie in one warp");
  extern __shared__ __align__(16) unsigned char raw[];
  const SvJob& J = batch.job[blockIdx.y];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ncols = J.ncols, ldt = Pol::ldt(ncols);
  ST* cs = reinterpret_cast<ST*>(raw);  // coefficients [NB][2][ncols]: as they are, parts swapped
  ST* ws = cs + NB * 2 * ncols;         // the tile's new values [RT][NB][2]
  ST* tile = ws + RT * NB * 2;          // [NBUF][RT][ldt]
  for (int e = tid; e < ncols * NB; e += kThreads) {
    const ST v = Pol::stage(Pol::from_c(J.c[e]));
    cs[(e % NB) * 2 * ncols + e / NB] = v;
    cs[((e % NB) * 2 + 1) * ncols + e / NB] = Pol::swap(v);
  }
  const ST* __restrict__ Q = static_cast<const ST*>(J.Q);  // entries as bytes
  Wt* w = static_cast<Wt*>(J.w);
  const int r0 = blockIdx.x * rpc, r1 = min(N, r0 + rpc);
  // Gram role: column(s) gcol, gcol + 256, ..., rows g, g + G, ...
  const int cpad = min(kThreads, (ncols + 31) & ~31), G = kThreads / cpad;
  const int g = tid / cpad, gcol = tid - g * cpad;
  AC acc[NC2][NB];
#pragma unroll
  for (int k = 0; k < NC2; ++k)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[k][b] = Pol::azero();
  const auto fetch = [&](int rb, ST* dst) {
#pragma unroll
    for (int k = 0; k < RT / kWarps; ++k) {
      const int r = warp + k * kWarps, row = rb + r;
      const bool on = row < r1;
      const ST* src = Q + (long long)(on ? row : r0) * J.ldq;
      for (int i = lane; i < ncols; i += 32) copy_entry(dst + r * ldt + i, src + i, on);
    }
    copies_commit();
  };
  ST* const first = tile;
  fetch(r0, tile);
  for (int rb = r0; rb < r1; rb += RT) {
    copies_wait<0>();
    if constexpr (!Pol::kStaged) {  // every thread converts, in place, what it copied
#pragma unroll
      for (int k = 0; k < RT / kWarps; ++k) {
        ST* t = tile + (warp + k * kWarps) * ldt;
#pragma unroll 4
        for (int i = lane; i < ncols; i += 32) t[i] = Pol::restage(t[i]);
      }
    }
    __syncthreads();  // the tile is there, and the last one's products are done
    if (NBUF == 2 && rb + RT < r1) fetch(rb + RT, tile == first ? first + RT * ldt : first);
    {
      const int r = tid / L, sub = tid % L, row = rb + r;
      AC d[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) d[b] = Pol::azero();
      for (int i = sub; i < ncols; i += L) {
        const ST q = tile[r * ldt + i];
#pragma unroll
        for (int b = 0; b < NB; ++b) Pol::tmac(d[b], q, cs[2 * b * ncols + i], cs[(2 * b + 1) * ncols + i]);
      }
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) d[b] = Pol::tadd(d[b], Pol::tshx(d[b], o));
      // lane b of the row forms the row's new value of vector b
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (sub == b) {
          Sp v{};
          if (row < r1) {
            v = Pol::wsub_t(Pol::wload(w[(long long)row * J.ldw + b]), d[b]);
            w[(long long)row * J.ldw + b] = Pol::wstore(v);
          }
          const ST t = Pol::of_w(v);
          ws[(r * NB + b) * 2] = t;
          ws[(r * NB + b) * 2 + 1] = Pol::swap(t);
        }
    }
    __syncthreads();
    if (g < G) {
#pragma unroll 2
      for (int r = g; r < RT; r += G) {
#pragma unroll
        for (int k = 0; k < NC2; ++k) {
          const int i = gcol + k * kThreads;
          if (i < ncols) {
            const ST q = tile[r * ldt + i];
#pragma unroll
            for (int b = 0; b < NB; ++b) Pol::tcmac(acc[k][b], q, ws[(r * NB + b) * 2], ws[(r * NB + b) * 2 + 1]);
          }
        }
      }
    }
    if (NBUF == 2) {
      tile = tile == first ? first + RT * ldt : first;
    } else {
      __syncthreads();
      if (rb + RT < r1) fetch(rb + RT, tile);
    }
  }
  __syncthreads();
  // sums of the row groups (the tile's space holds them; G > 1 only with one column per thread)
  double2* out = J.part + (long long)blockIdx.x * J.ldp;
  double2* red = reinterpret_cast<double2*>(raw);
  if (G > 1) {
    if (g > 0 && g < G && gcol < ncols)
#pragma unroll
      for (int b = 0; b < NB; ++b) red[((g - 1) * NB + b) * cpad + gcol] = Pol::tto_d(acc[0][b]);
    __syncthreads();
  }
  if (g == 0) {
#pragma unroll
    for (int k = 0; k < NC2; ++k) {
      const int i = gcol + k * kThreads;
      if (i < ncols)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          double2 s = Pol::tto_d(acc[k][b]);
          for (int q = 1; q < G; ++q) {
            const double2 v = red[((q - 1) * NB + b) * cpad + i];
            s.x += v.x;
            s.y += v.y;
          }
          out[i * NB + b] = s;
        }
    }
  }
}

// sum over a block of the NB x NB entries held (as FP64) by its threads, into
// out[0 .. NB NB); red: [kWarps][NB * NB]
template <int NB>
__device__ __forceinline__ void block_sum_small(const Gds* g, double2 (*red)[NB * NB], double2* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int e = 0; e < NB * NB; ++e) {
    double2 s = make_double2((double)g[e].rh + (double)g[e].re, (double)g[e].ih + (double)g[e].ie);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    if (lane == 0) red[warp][e] = s;
  }
  __syncthreads();
  if (threadIdx.x < NB * NB) {
    double2 s = red[0][threadIdx.x];
#pragma unroll
    for (int k = 1; k < kWarps; ++k) {
      s.x += red[k][threadIdx.x].x;
      s.y += red[k][threadIdx.x].y;
    }
    out[threadIdx.x] = s;
  }
}

// ----------------------------------------------------------------- the second update (FP32 products) and w^H w
// w[r, :] -= Q[r, :] c for the second pass's small coefficients: products of
// the basis heads in FP32; and the new block's Gram matrix in double-single on
// the way.  HBM-bound: a warp takes R rows at a time and copies the next R into
// its half of shared memory meanwhile (every lane reads only what it copied, so
// nothing waits on another lane); the R x NB products are summed over the lanes
// by halving - every level keeps half the values per lane - so that
// R NB + log2(32 / (R NB)) exchanges serve all of them; then each value's first
// lane forms the row's new entry.
template <class Pol, int NB, int R>
__global__ void __launch_bounds__(kThreads)
    sv_update_fast_kernel(const __grid_constant__ SvBatch batch, int N, int rpc, int stages) {
  using ST = typename Pol::ST;
  using Sp = typename Pol::S;
  using Wt = typename Pol::W;
  constexpr int V = R * NB;  // values per warp pass, index row * NB + b
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ double2 red[kWarps][NB * NB];
  const SvJob& J = batch.job[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ncols = J.ncols;
  ST* ring = reinterpret_cast<ST*>(raw) + (size_t)warp * stages * R * ncols;  // [stages][R][ncols] per warp
  // the coefficients' heads, [NB][ncols] (8 bytes per entry: conflict-free reads)
  float2* cs = reinterpret_cast<float2*>(reinterpret_cast<ST*>(raw) + (size_t)kWarps * stages * R * ncols);
  const ST* __restrict__ Q = static_cast<const ST*>(J.Q);  // entries as bytes
  Wt* w = static_cast<Wt*>(J.w);
  const int r0 = blockIdx.x * rpc, r1 = min(N, r0 + rpc);
  const auto fetch = [&](int r, ST* dst) {
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const bool on = r + u < r1;
      const ST* src = Q + (long long)(on ? r + u : r0) * J.ldq;
      for (int i = lane; i < ncols; i += 32) copy_entry(dst + u * ncols + i, src + i, on);
    }
  };
  int st = 0;
  if (r0 + warp * R < r1) fetch(r0 + warp * R, ring);
  copies_commit();
  for (int e = threadIdx.x; e < ncols * NB; e += kThreads) cs[(e % NB) * ncols + e / NB] = Pol::head2(Pol::from_c(J.c[e]));
  __syncthreads();
  constexpr int kLow = 32 / V;  // lanes left per value
  const int vi = lane / kLow, vrow = vi / NB, vb = vi % NB;
  Gds g[NB * NB];
#pragma unroll
  for (int e = 0; e < NB * NB; ++e) g[e] = Gds{0.f, 0.f, 0.f, 0.f};
  for (int r = r0 + warp * R; r < r1; r += kWarps * R) {
    const int rn = r + kWarps * R;
    if (stages == 2) {
      if (rn < r1) fetch(rn, ring + (st ^ 1) * R * ncols);
      copies_commit();
      copies_wait<1>();
    } else {
      copies_wait<0>();
    }
    const ST* q = ring + st * R * ncols;
    // the value this lane will finish: its old entry, loaded beside the basis
    const bool on = r + vrow < r1;
    Wt* wp = w + (long long)(r + vrow) * J.ldw + vb;
    Sp old{};
    if (on) old = Pol::wload(*wp);
    float2 f[V];
#pragma unroll
    for (int e = 0; e < V; ++e) f[e] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int i = lane; i < ncols; i += 32) {
      float2 c[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) c[b] = cs[b * ncols + i];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const float2 h = Pol::raw_head(q[u * ncols + i]);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          float2& a = f[u * NB + b];
          a.x = fmaf(h.x, c[b].x, fmaf(-h.y, c[b].y, a.x));
          a.y = fmaf(h.x, c[b].y, fmaf(h.y, c[b].x, a.y));
        }
      }
    }
    if (stages == 2) {
      st ^= 1;
    } else {
      if (rn < r1) fetch(rn, ring);
      copies_commit();
    }
#pragma unroll
    for (int n = V / 2, o = 16; n > 0; n >>= 1, o >>= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int e = 0; e < n; ++e) {
        const float2 keep = up ? f[e + n] : f[e], give = up ? f[e] : f[e + n];
        f[e].x = keep.x + __shfl_xor_sync(0xffffffffu, give.x, o);
        f[e].y = keep.y + __shfl_xor_sync(0xffffffffu, give.y, o);
      }
    }
#pragma unroll
    for (int o = kLow / 2; o > 0; o >>= 1) {
      f[0].x += __shfl_xor_sync(0xffffffffu, f[0].x, o);
      f[0].y += __shfl_xor_sync(0xffffffffu, f[0].y, o);
    }
    const Sp v = Pol::wsub(old, Pol::fto_A(f[0]));
    const bool own = on && lane % kLow == 0;
    if (own) *wp = Pol::wstore(v);
    if constexpr (NB == 1) {
      if (own) Pol::gacc(g[0], v, v);
    } else {
      const Sp v1 = Pol::sshx(v, kLow);  // the row's other vector
      if (own && vb == 0) {
        Pol::gacc(g[0], v, v);
        Pol::gacc(g[1], v, v1);
        Pol::gacc(g[2], v1, v);
        Pol::gacc(g[3], v1, v1);
      }
    }
  }
  block_sum_small<NB>(g, red, J.part + (long long)blockIdx.x * J.ldp);
}

// ----------------------------------------------------------------- w^H w of the new block
// A block per row chunk and job, a thread per row (strided): double-single
// products on every lane, FP64 sums across the block.  With r set the row is
// first multiplied by the Cholesky factor's inverse (in place): the first
// normalisation of a 2-vector block with the Gram matrix of the second.
template <class Pol, int NB, bool SCALE>
__global__ void __launch_bounds__(kThreads) sv_wgram_kernel(const __grid_constant__ SvBatch batch, int N, int rpc) {
  using Wt = typename Pol::W;
  const SvJob& J = batch.job[blockIdx.y];
  Wt* w = static_cast<Wt*>(J.w);
  const int r0 = blockIdx.x * rpc, r1 = min(N, r0 + rpc);
  __shared__ double2 red[kWarps][NB * NB];
  double2 ri[NB * NB];
#pragma unroll
  for (int e = 0; e < NB * NB; ++e) ri[e] = SCALE ? J.c[e] : make_double2(0.0, 0.0);
  Gds g[NB * NB];
#pragma unroll
  for (int e = 0; e < NB * NB; ++e) g[e] = Gds{0.f, 0.f, 0.f, 0.f};
  for (int r = r0 + threadIdx.x; r < r1; r += kThreads) {
    typename Pol::S v[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) v[b] = Pol::wload(w[(long long)r * J.ldw + b]);
    if constexpr (SCALE) {
      typename Pol::S o[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) {  // column b of v R^-1 (upper triangular)
        o[b] = Pol::smul2(v[0], ri[b], v[NB - 1], ri[(NB - 1) * NB + b], b > 0);
        w[(long long)r * J.ldw + b] = Pol::wstore(o[b]);
      }
#pragma unroll
      for (int b = 0; b < NB; ++b) v[b] = o[b];
    }
#pragma unroll
    for (int a = 0; a < NB; ++a)
#pragma unroll
      for (int b = 0; b < NB; ++b) Pol::gacc(g[a * NB + b], v[a], v[b]);
  }
  block_sum_small<NB>(g, red, J.part + (long long)blockIdx.x * J.ldp);
}

// ----------------------------------------------------------------- chunk reduction
// A block per 8 entries and job (per 4 entries where the block's Gram matrix is
// summed): the FP64 additions bound it, and a warp instruction takes ~19 cycles of
// an SM's FP64 pipe however few lanes are on, so the entries are spread over
// many SMs and every warp's lanes filled with (entry, chunk) pairs.  With 32
// entries and 1024 threads to a block it took 16 us cold, now 9.
constexpr int kRedThreads = 256;

// upper Cholesky factor R of the Hermitian nb x nb matrix G (G = R^H R), its
// inverse, and whether a pivot fell below 1e-14 of its diagonal entry
__device__ bool chol_small(const double2* G, int nb, double2* R, double2* Ri) {
  bool bad = false;
  for (int e = 0; e < 4; ++e) R[e] = Ri[e] = make_double2(0.0, 0.0);
  const double g00 = G[0].x;
  if (!(g00 > 0.0)) return true;
  const double r00 = sqrt(g00), i00 = 1.0 / r00;
  R[0] = make_double2(r00, 0.0);
  Ri[0] = make_double2(i00, 0.0);
  if (nb == 1) return false;
  const double2 r01 = make_double2(G[1].x * i00, G[1].y * i00);
  const double d = G[3].x - (r01.x * r01.x + r01.y * r01.y);
  if (!(d > 1e-14 * G[3].x)) {
    bad = true;
  }
  const double r11 = d > 0.0 ? sqrt(d) : 0.0;
  R[1] = r01;
  R[3] = make_double2(r11, 0.0);
  if (r11 > 0.0) {
    const double i11 = 1.0 / r11, t = i00 * i11;
    Ri[1] = make_double2(-r01.x * t, -r01.y * t);
    Ri[3] = make_double2(i11, 0.0);
  }
  return bad;
}

__global__ void __launch_bounds__(kRedThreads) sv_reduce_kernel(const __grid_constant__ SvReduceBatch batch) {
  const SvReduceJob& J = batch.job[blockIdx.y];
  const int E = J.mode == 0 ? 8 : 4, lanes = kRedThreads / E;  // entries, chunks at a time
  const int cl = threadIdx.x % E, k = threadIdx.x / E;
  const int i = blockIdx.x * E + cl;
  const int nent = J.mode == 0 ? J.ncols * J.nb : J.nb * J.nb;
  if (blockIdx.x * E >= nent) return;  // uniform over the block
  double2 a0 = make_double2(0.0, 0.0), a1 = a0;
  if (i < nent) {
    int ch = k;
    for (; ch + lanes < J.nchunks; ch += 2 * lanes) {
      const double2 v0 = J.part[(long long)ch * J.ldp + i];
      const double2 v1 = J.part[(long long)(ch + lanes) * J.ldp + i];
      a0.x += v0.x;
      a0.y += v0.y;
      a1.x += v1.x;
      a1.y += v1.y;
    }
    if (ch < J.nchunks) {
      const double2 v0 = J.part[(long long)ch * J.ldp + i];
      a0.x += v0.x;
      a0.y += v0.y;
    }
  }
  __shared__ double2 red[kRedThreads / 32][8];
  __shared__ double2 fin[4];
  a0 = make_double2(a0.x + a1.x, a0.y + a1.y);
  for (int o = E; o < 32; o <<= 1) {
    a0.x += __shfl_xor_sync(0xffffffffu, a0.x, o);
    a0.y += __shfl_xor_sync(0xffffffffu, a0.y, o);
  }
  if ((threadIdx.x & 31) < E) red[threadIdx.x >> 5][cl] = a0;
  __syncthreads();
  if (k == 0 && i < nent) {
    double2 s = red[0][cl];
#pragma unroll
    for (int q = 1; q < kRedThreads / 32; ++q) {
      s.x += red[q][cl].x;
      s.y += red[q][cl].y;
    }
    if (J.mode == 0) {
      if (J.C) J.C[i] = s;
      if (J.H) {
        double2* h = J.H + (long long)(i / J.nb) * J.ldh + i % J.nb;
        *h = make_double2(h->x + s.x, h->y + s.y);
      }
    } else {
      fin[i] = s;
    }
  }
  if (J.mode == 0) return;
  __syncthreads();
  if (threadIdx.x != 0) return;
  double2 R[4], Ri[4];
  const bool bad = chol_small(fin, J.nb, R, Ri);
  const int nb = J.nb;
  if (J.mode == 1) {
    for (int e = 0; e < nb * nb; ++e) {
      J.r[e] = Ri[e];
      J.r[4 + e] = R[e];
    }
    if (nb == 1 && J.H) J.H[0] = R[0];
  } else {
    // R = R2 R1 (both upper triangular, nb = 2)
    const double2* R1 = J.r + 4;
    for (int e = 0; e < 4; ++e) J.r[e] = Ri[e];
    if (J.H) {
      for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b) {
          double2 s = make_double2(0.0, 0.0);
          for (int q = 0; q < 2; ++q) {
            const double2 x = R[a * 2 + q], y = R1[q * 2 + b];
            s.x += x.x * y.x - x.y * y.y;
            s.y += x.x * y.y + x.y * y.x;
          }
          J.H[(long long)a * J.ldh + b] = s;
        }
    }
  }
  if (bad) J.r[8] = make_double2(1.0, 0.0);
}

// ----------------------------------------------------------------- normalisation
// the block times the inverse of its Cholesky factor, into the basis and into
// the newest-vectors block, a thread per row; in the arithmetic of the new
// vectors (six FP64 conversions and eight products per entry cost more than the
// row's traffic on GB300's FP64 pipe)
template <class Pol, int NB>
__global__ void sv_normalize_kernel(const __grid_constant__ SvNormBatch batch, int N) {
  using T = typename Pol::T;
  using Wt = typename Pol::W;
  const SvNormJob& J = batch.job[blockIdx.y];
  double2 r[NB * NB];
#pragma unroll
  for (int e = 0; e < NB * NB; ++e) r[e] = J.r[e];
  const Wt* w = static_cast<const Wt*>(J.w);
  for (long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x; row < N;
       row += (long long)gridDim.x * blockDim.x) {
    typename Pol::S v[NB];
#pragma unroll
    for (int a = 0; a < NB; ++a) v[a] = Pol::wload(w[row * J.ldw + a]);
#pragma unroll
    for (int b = 0; b < NB; ++b) {  // column b of v R^-1 (upper triangular)
      const T o = Pol::out(Pol::smul2(v[0], r[b], v[NB - 1], r[(NB - 1) * NB + b], b > 0));
      static_cast<T*>(J.dst1)[row * J.ld1 + b] = o;
      if (J.dst2) static_cast<T*>(J.dst2)[row * J.ld2 + b] = o;
    }
  }
}

template <class Pol, int RT, int NC2, int NB, int NBUF>
void launch_update_rt(const SvBatch& b, int N, int rpc, int maxcols, cudaStream_t s) {
  using ST = typename Pol::ST;
  const size_t tile = sizeof(ST) * ((size_t)NB * 2 * maxcols + RT * NB * 2 + (size_t)NBUF * RT * Pol::ldt(maxcols));
  // the row groups' sums share the space: (G - 1) NB cpad <= 224 NB entries of 16 bytes
  const size_t smem = std::max(tile, sizeof(double2) * 224 * NB);
  smem_opt_in(reinterpret_cast<const void*>(sv_update_kernel<Pol, RT, NC2, NB, NBUF>));
  sv_update_kernel<Pol, RT, NC2, NB, NBUF><<<dim3((N + rpc - 1) / rpc, b.n), kThreads, smem, s>>>(b, N, rpc);
}

// rows per tile: three blocks of 256 threads share an SM's shared memory with two
// tiles each (a complex128 tile of 32 rows up to 64 columns, 16 rows up to 128)
template <class Pol, int NB>
void launch_update(const SvBatch& b, int N, int rpc, int maxcols, cudaStream_t s) {
  const int wide = sizeof(typename Pol::ST) == 8 ? 2 : 1;
  if (maxcols <= 64 * wide) launch_update_rt<Pol, 32, 1, NB, 2>(b, N, rpc, maxcols, s);
  else if (maxcols <= 128 * wide) launch_update_rt<Pol, 16, 1, NB, 2>(b, N, rpc, maxcols, s);
  else if (maxcols <= 256) launch_update_rt<Pol, 8, 1, NB, 2>(b, N, rpc, maxcols, s);
  else if (maxcols <= 512) launch_update_rt<Pol, 8, 2, NB, 2>(b, N, rpc, maxcols, s);
  else if constexpr (NB == 1) launch_update_rt<Pol, 8, 4, NB, 1>(b, N, rpc, maxcols, s);
  else throw Error{SWI_EINVAL, "Gram-Schmidt pass: at most 512 basis columns with 2-vector blocks"};
}

template <class Pol, int NB, int R>
void launch_update_fast_r(const SvBatch& b, int N, int rpc, int maxcols, int stages, cudaStream_t s) {
  const size_t smem = sizeof(typename Pol::ST) * (size_t)kWarps * stages * R * maxcols + sizeof(float2) * (size_t)maxcols * NB;
  smem_opt_in(reinterpret_cast<const void*>(sv_update_fast_kernel<Pol, NB, R>));
  sv_update_fast_kernel<Pol, NB, R><<<dim3((N + rpc - 1) / rpc, b.n), kThreads, smem, s>>>(b, N, rpc, stages);
}

// rows per warp: three blocks share an SM's shared memory up to 256 columns
// (complex128); past 512 only one stage of one row fits a block
template <class Pol, int NB>
void launch_update_fast(const SvBatch& b, int N, int rpc, int maxcols, cudaStream_t s) {
  const int wide = sizeof(typename Pol::ST) == 8 ? 2 : 1;
  if (maxcols <= 64 * wide) launch_update_fast_r<Pol, NB, 4>(b, N, rpc, maxcols, 2, s);
  else if (maxcols <= 128 * wide) launch_update_fast_r<Pol, NB, 2>(b, N, rpc, maxcols, 2, s);
  else if (maxcols <= 512) launch_update_fast_r<Pol, NB, 1>(b, N, rpc, maxcols, 2, s);
  else if constexpr (NB == 1) launch_update_fast_r<Pol, NB, 1>(b, N, rpc, maxcols, 1, s);
  else throw Error{SWI_EINVAL, "Gram-Schmidt pass: at most 512 basis columns with 2-vector blocks"};
}

template <class Pol, int NB>
void launch_pass_nb(const SvBatch& b, int mode, int N, int rpc, int maxcols, cudaStream_t s) {
  const int nchunks = (N + rpc - 1) / rpc;
  if (mode == SV_GRAM) {
    const dim3 grid(nchunks, (maxcols + 31) / 32, b.n);
    sv_gram_kernel<Pol, NB><<<grid, kThreads, 0, s>>>(b, N, rpc);
  } else if (mode == SV_UPDATE_GRAM) {
    launch_update<Pol, NB>(b, N, rpc, maxcols, s);
  } else if (mode == SV_UPDATE) {
    launch_update_fast<Pol, NB>(b, N, rpc, maxcols, s);
  } else if (mode == SV_SCALE_WGRAM) {
    sv_wgram_kernel<Pol, NB, true><<<dim3(nchunks, b.n), kThreads, 0, s>>>(b, N, rpc);
  } else {
    sv_wgram_kernel<Pol, NB, false><<<dim3(nchunks, b.n), kThreads, 0, s>>>(b, N, rpc);
  }
}

}  // namespace

int sv_rows_per_chunk(int N, int njobs) {
  // one wave of the three blocks an SM holds, over the jobs; at least one tile of
  // 32 rows (2,000 rows in four windows: 252 blocks; chunks of at least 256 rows
  // left 32, each marching 32 rows per warp for ~110 us) and at most 1024 (the
  // bound on the per-lane partial sums: several waves then)
  const long long per = ((long long)N * std::max(njobs, 1) + 3 * 152 - 1) / (3 * 152);
  return (int)std::max<long long>(32, std::min<long long>(1024, (per + 31) / 32 * 32));
}

void launch_sv_pass(const SvBatch& b, int mode, bool ds, int nb, int N, int rpc, cudaStream_t s,
                    long long* launches) {
  if (b.n <= 0) return;
  if (nb != 1 && nb != 2) throw Error{SWI_EINVAL, "Gram-Schmidt pass: blocks of 1 or 2 vectors"};
  int maxcols = 0;
  for (int q = 0; q < b.n; ++q) {
    const int nc = b.job[q].ncols;
    if (nc > 1024 || (mode != SV_WGRAM && mode != SV_SCALE_WGRAM && nc < 1))
      throw Error{SWI_EINVAL, "Gram-Schmidt pass: 1..1024 basis columns"};
    maxcols = std::max(maxcols, nc);
  }
  if (rpc < 8 || rpc > 1024) throw Error{SWI_EINVAL, "Gram-Schmidt pass: rows per chunk out of range"};
  if (ds) {
    if (nb == 1) launch_pass_nb<PolDs, 1>(b, mode, N, rpc, maxcols, s);
    else launch_pass_nb<PolDs, 2>(b, mode, N, rpc, maxcols, s);
  } else {
    if (nb == 1) launch_pass_nb<PolC64, 1>(b, mode, N, rpc, maxcols, s);
    else launch_pass_nb<PolC64, 2>(b, mode, N, rpc, maxcols, s);
  }
  SWI_CHECK_LAUNCH();
  if (launches) ++*launches;
}

void launch_sv_reduce(const SvReduceBatch& b, cudaStream_t s, long long* launches) {
  if (b.n <= 0) return;
  int maxent = 1;
  for (int q = 0; q < b.n; ++q) {
    const SvReduceJob& J = b.job[q];
    if (J.nb != 1 && J.nb != 2) throw Error{SWI_EINVAL, "chunk reduction: blocks of 1 or 2 vectors"};
    if (J.mode != 0 && J.r == nullptr) throw Error{SWI_EINVAL, "chunk reduction: Cholesky output missing"};
    if (J.mode == 2 && J.nb != 2) throw Error{SWI_EINVAL, "chunk reduction: second Cholesky pass needs nb = 2"};
    maxent = std::max(maxent, J.mode == 0 ? J.ncols * J.nb : J.nb * J.nb);
  }
  sv_reduce_kernel<<<dim3((maxent + 7) / 8, b.n), kRedThreads, 0, s>>>(b);
  SWI_CHECK_LAUNCH();
  if (launches) ++*launches;
}

void launch_sv_normalize(const SvNormBatch& b, bool ds, int nb, int N, cudaStream_t s, long long* launches) {
  if (b.n <= 0) return;
  if (nb != 1 && nb != 2) throw Error{SWI_EINVAL, "normalisation: blocks of 1 or 2 vectors"};
  const int blocks = std::min((N + 255) / 256, 1024);
  const dim3 grid(blocks, b.n);
  if (ds) {
    if (nb == 1) sv_normalize_kernel<PolDs, 1><<<grid, 256, 0, s>>>(b, N);
    else sv_normalize_kernel<PolDs, 2><<<grid, 256, 0, s>>>(b, N);
  } else {
    if (nb == 1) sv_normalize_kernel<PolC64, 1><<<grid, 256, 0, s>>>(b, N);
    else sv_normalize_kernel<PolC64, 2><<<grid, 256, 0, s>>>(b, N);
  }
  SWI_CHECK_LAUNCH();
  if (launches) ++*launches;
}

}  // namespace swi
