// The dense contractions of the adjoint of T(E) in double-single arithmetic on
// the FP32 pipes (the FP64-class form):
//
//   M[a][c] = sum_e w_e g_ea g_ec sum_l R[a][l] conj(g_el) L[c][l]
//   dL/dV(r) = 2 Re sum_ac U_ra M_ac U_rc = 2 Re sum_c U_rc sum_{a <= c} S_ac U_ra,
//              S_ac = M_ac + M_ca (a < c), S_aa = M_aa
//
// FP32 issue bounds them: a complex multiply-add is 48 operations (each real
// product exact up to its tail, heads summed by TwoSum), so a thread holds
// several outputs, real and imaginary parts go through packed FP32x2
// instructions (half the issue slots; the rest carry loads and splits), and
// nothing inside the loops touches the FP64 pipe.  Sums run in double-single over
// at most 1,024 terms and in FP64 beyond.  Rows of R and L, and S as a whole, are
// scaled by powers of two before they are split: their sizes follow the absorbers.
//
// Measured on one GB300, 400 pairs of the 48x48x96 grid, 128 energies:
// adjoint 52 ms against 176 (M in native FP64, ~119; U M as an N x n product, then
// a row dot: all of M, and 1.4 GB of scratch).  48 pairs of the 10x10x20 grid, 32
// energies: 0.10 ms against 2.7.
#include <algorithm>

#include "ds.cuh"
#include "swi_internal.cuh"
#include "transport.cuh"

namespace swi {

namespace {

constexpr int kT = 32;     // output tile edge
constexpr int kK = 16;     // contraction depth of one shared-memory stage
constexpr int kThr = 256;  // 16 x 16 threads, 2 x 2 outputs each (rows ty + 16 i, columns tx + 16 j)
constexpr int kFlush = 64;  // stages (1,024 terms) per FP64 flush
constexpr int kNorm = 8;    // terms between two renormalisations of a running sum

struct V4 {  // complex double-single: heads (re, im), tails (re, im)
  float2 h, l;
};
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ V4 ld(float4 v) { return V4{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 split4(double2 v) {
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  if (__double_as_longlong(v.x) << 1) ds::split_bits(v.x, o.x, o.z);
  if (__double_as_longlong(v.y) << 1) ds::split_bits(v.y, o.y, o.w);
  return o;
}
// a += (uh + ul) (vh + vl) per component
__device__ __forceinline__ void mulv(V4& a, float2 uh, float2 ul, float2 vh, float2 vl) {
  const float2 p = __fmul2_rn(uh, vh);
  float2 e = __ffma2_rn(uh, vh, make_float2(-p.x, -p.y));
  e = __ffma2_rn(uh, vl, e);
  e = __ffma2_rn(ul, vh, e);
  const float2 t = add2(a.h, p);
  const float2 bp = sub2(t, a.h);
  const float2 err = add2(sub2(a.h, sub2(t, bp)), sub2(p, bp));
  a.h = t;
  a.l = add2(a.l, add2(err, e));
}
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 pm(float x) { return make_float2(x, -x); }
__device__ __forceinline__ float2 mp(float x) { return make_float2(-x, x); }
__device__ __forceinline__ float2 swp(float2 v) { return make_float2(v.y, v.x); }
// a += conj(x) y, a += x y
__device__ __forceinline__ void cmacc(V4& a, const V4& x, const V4& y) {
  mulv(a, dup(x.h.x), dup(x.l.x), y.h, y.l);
  mulv(a, pm(x.h.y), pm(x.l.y), swp(y.h), swp(y.l));
}
__device__ __forceinline__ void cmac(V4& a, const V4& x, const V4& y) {
  mulv(a, dup(x.h.x), dup(x.l.x), y.h, y.l);
  mulv(a, mp(x.h.y), mp(x.l.y), swp(y.h), swp(y.l));
}
__device__ __forceinline__ V4 zero4() { return V4{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
// head + tail as a pair again (TwoSum).  A running sum's tail collects the heads'
// rounding errors and grows with their number, and its own rounding with it: after
// k terms ~0.08 k 2^-48 of their root sum of squares (a CPU emulation), with this
// every 8 terms 0.3 sqrt(k) 2^-48
__device__ __forceinline__ V4 renorm(const V4& a) {
  const float2 t = add2(a.h, a.l), bb = sub2(t, a.h);
  return V4{t, add2(sub2(a.h, sub2(t, bb)), sub2(a.l, bb))};
}
__device__ __forceinline__ void flush(double2& s, V4& a) {
  s.x += (double)a.h.x + (double)a.l.x;
  s.y += (double)a.h.y + (double)a.l.y;
  a = zero4();
}

// A power of two that brings a largest magnitude (its bits) to [1, 2) (1 where
// there is none, or no finite one), and its inverse: weakly coupled wires have
// projections and an M far below 1, whose products would leave the range of a float.
__device__ __forceinline__ double unit_scale(unsigned long long mx, bool inverse) {
  const unsigned ef = (unsigned)(mx >> 52);
  if (ef == 0 || ef >= 0x7ff) return 1.0;
  const unsigned f = max(2046u - ef, 1u);
  return __longlong_as_double((long long)(inverse ? 2046u - f : f) << 52);
}
__device__ __forceinline__ unsigned long long max_bits(unsigned long long v, double2 m) {
  return max(v, max((unsigned long long)__double_as_longlong(fabs(m.x)), (unsigned long long)__double_as_longlong(fabs(m.y))));
}

// R and L (blockIdx.y) scaled by rows and split, a warp per row; inv[row]: the
// inverse of the row's scale (R first, then L).  Both are linear in the absorbers:
// a row of 1e-20 against one of L of 1e-20 has products that no float holds.
__global__ void __launch_bounds__(kThr) split_rows_kernel(const double2* __restrict__ R, const double2* __restrict__ L,
                                                         int n, float4* __restrict__ Rs, float4* __restrict__ Ls,
                                                         double* __restrict__ inv) {
  const int row = blockIdx.x * (kThr / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= n) return;
  const double2* src = (blockIdx.y ? L : R) + (size_t)row * n;
  float4* dst = (blockIdx.y ? Ls : Rs) + (size_t)row * n;
  unsigned long long v = 0;
  for (int l = lane; l < n; l += 32) v = max_bits(v, src[l]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  const double f = unit_scale(v, false);
  for (int l = lane; l < n; l += 32) dst[l] = split4(cscale(src[l], f));
  if (lane == 0) inv[blockIdx.y * n + row] = unit_scale(v, true);
}

// gt[e][l] = 1/(E_e - eps_l), formed in FP64 and split
__global__ void gtab_ds_kernel(const double2* __restrict__ eps, int n, const double* __restrict__ E, int nE,
                               float4* __restrict__ gt) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nE * n) return;
  const int e = (int)(t / n), l = (int)(t % n);
  gt[t] = split4(cdiv(make_double2(1.0, 0.0), csub(make_double2(E[e], 0.0), eps[l])));
}

// part[s][a][c] = the energies of group s (blockIdx.z) of M, from the rows of R and
// L as they are scaled
__global__ void __launch_bounds__(kThr, 2)
    gradM_ds_kernel(const float4* __restrict__ R, const float4* __restrict__ L, const float4* __restrict__ gt,
                    const double* __restrict__ inv, const double* __restrict__ wts, int n, int nE, int per,
                    double2* __restrict__ part) {
  __shared__ float4 sr[kK][kT + 1], sl[kK][kT + 1];  // R[a][l], conj(g_l) L[c][l]
  const int a0 = blockIdx.y * kT, c0 = blockIdx.x * kT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double2 tot[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) tot[i][j] = make_double2(0.0, 0.0);
  const int e0 = blockIdx.z * per, e1 = min(nE, e0 + per);
  for (int e = e0; e < e1; ++e) {
    const double we = wts[e];
    if (we == 0.0) continue;  // the same for every thread of the block
    const float4* g = gt + (size_t)e * n;
    V4 acc[2][2];
    double2 sum[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        acc[i][j] = zero4();
        sum[i][j] = make_double2(0.0, 0.0);
      }
    int stage = 0;
    for (int l0 = 0; l0 < n; l0 += kK) {
#pragma unroll
      for (int q = 0; q < kK * kT / kThr; ++q) {
        const int f = threadIdx.x + q * kThr, ll = f % kK, row = f / kK;  // 16 consecutive l of one row
        const int l = l0 + ll, a = a0 + row, c = c0 + row;
        sr[ll][row] = a < n && l < n ? __ldg(R + (size_t)a * n + l) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < n && l < n) {
          V4 p = zero4();
          cmacc(p, ld(__ldg(g + l)), ld(__ldg(L + (size_t)c * n + l)));
          p = renorm(p);
          v = make_float4(p.h.x, p.h.y, p.l.x, p.l.y);
        }
        sl[ll][row] = v;
      }
      __syncthreads();
      for (int lb = 0; lb < kK; lb += kNorm) {
#pragma unroll 4
        for (int ll = lb; ll < lb + kNorm; ++ll) {
          V4 xr[2], xl[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            xr[i] = ld(sr[ll][ty + 16 * i]);
            xl[i] = ld(sl[ll][tx + 16 * i]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) cmac(acc[i][j], xr[i], xl[j]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) acc[i][j] = renorm(acc[i][j]);
      }
      __syncthreads();
      if (++stage == kFlush) {
        stage = 0;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) flush(sum[i][j], acc[i][j]);
      }
    }
    // += w_e g_a g_c acc, in FP64 (once per energy)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int a = a0 + ty + 16 * i;
      if (a >= n) continue;
      const float4 ga = g[a];
      const double2 da = make_double2((double)ga.x + (double)ga.z, (double)ga.y + (double)ga.w);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = c0 + tx + 16 * j;
        if (c >= n) continue;
        const float4 gc = g[c];
        const double2 dc = make_double2((double)gc.x + (double)gc.z, (double)gc.y + (double)gc.w);
        flush(sum[i][j], acc[i][j]);
        cfma(tot[i][j], cscale(cmul(da, dc), we), sum[i][j]);
      }
    }
  }
  double2* P = part + (size_t)blockIdx.z * n * n;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int a = a0 + ty + 16 * i;
    if (a >= n) continue;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = c0 + tx + 16 * j;
      if (c < n) P[(size_t)a * n + c] = cscale(cscale(tot[i][j], inv[a]), inv[n + c]);
    }
  }
}

// largest |re| or |im| of M, as its bits (a non-negative double orders like them)
__global__ void absmax_kernel(const double2* __restrict__ M, long long nn, unsigned long long* __restrict__ mx) {
  unsigned long long v = 0;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nn; t += (long long)gridDim.x * blockDim.x) {
    v = max_bits(v, M[t]);
  }
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0 && v) atomicMax(mx, v);
}
// S[a][c] scaled and split, a <= c (zero below the diagonal)
__global__ void symsplit_kernel(const double2* __restrict__ M, int n, const unsigned long long* __restrict__ mx,
                                float4* __restrict__ S) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  const int a = (int)(t / n), c = (int)(t % n);
  double2 v = make_double2(0.0, 0.0);
  if (a <= c) v = M[t];
  if (a < c) v = cadd(v, M[(size_t)c * n + a]);
  S[t] = split4(cscale(v, unit_scale(*mx, false)));
}

// out[r] for the 32 rows r0 .. r0 + 31 of a block: per 32-column tile the sums
// over a <= c, contracted with the same rows of U at once (nothing of size N x n
// is stored).  LONG, past kFlush stages: a tile is contracted after every kFlush
// of them (the loop alone costs the short form 2.5%)
template <bool LONG>
__global__ void __launch_bounds__(kThr, 2)
    rowquad_ds_kernel(const double2* __restrict__ U, const float4* __restrict__ S, int n, long long N,
                      const unsigned long long* __restrict__ mx, double* __restrict__ out) {
  __shared__ float4 su[kK][kT + 1];  // su[a][row] = U[r0 + row][a0 + a]
  __shared__ float4 sm[kK][kT];      // sm[a][col] = S[a0 + a][c0 + col]
  const long long r0 = (long long)blockIdx.x * kT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double row[2] = {0.0, 0.0};
  for (int c0 = 0; c0 < n; c0 += kT)
  for (int as = 0, end = min(n, c0 + kT); as < (LONG ? end : 1); as += kFlush * kK) {
    V4 acc[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j] = zero4();
    const int a1 = LONG ? min(end, as + kFlush * kK) : end;
    for (int a0 = as; a0 < a1; a0 += kK) {
#pragma unroll
      for (int q = 0; q < kK * kT / kThr; ++q) {
        const int f = threadIdx.x + q * kThr;
        {
          const int aa = f % kK, rr = f / kK;  // 16 consecutive columns of one row of U
          const long long r = r0 + rr;
          su[aa][rr] = r < N && a0 + aa < n ? split4(__ldg(U + r * n + a0 + aa)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        {
          const int col = f % kT, ab = f / kT;  // 32 consecutive columns of one row of S
          sm[ab][col] = a0 + ab < n && c0 + col < n ? __ldg(S + (size_t)(a0 + ab) * n + c0 + col)
                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      __syncthreads();
      for (int ab = 0; ab < kK; ab += kNorm) {
#pragma unroll 4
        for (int aa = ab; aa < ab + kNorm; ++aa) {
          V4 xu[2], xm[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            xu[i] = ld(su[aa][ty + 16 * i]);
            xm[i] = ld(sm[aa][tx + 16 * i]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) cmac(acc[i][j], xu[i], xm[j]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) acc[i][j] = renorm(acc[i][j]);
      }
      __syncthreads();
    }
    // Re(acc U[r][c]), one FP64 addition per row, tile and 1,024 terms
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const long long r = r0 + ty + 16 * i;
      if (r >= N) continue;
      float h = 0.f, l = 0.f;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = c0 + tx + 16 * j;
        if (c >= n) continue;
        const float4 u = split4(__ldg(U + r * n + c));
        const V4 x = renorm(acc[i][j]);
        ds::fma_acc(h, l, x.h.x, x.l.x, u.x, u.z);
        ds::fma_acc(h, l, -x.h.y, -x.l.y, u.y, u.w);
      }
      row[i] += (double)h + (double)l;
    }
  }
  // sum over the 16 column lanes (tx) of each half-warp
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) row[i] += __shfl_xor_sync(0xffffffffu, row[i], o);
  if (tx == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const long long r = r0 + ty + 16 * i;
      if (r < N) out[r] = 2.0 * unit_scale(*mx, true) * row[i];
    }
  }
}

__global__ void sum_parts_kernel(const double2* __restrict__ part, int parts, long long nn, double2* __restrict__ M) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nn) return;
  double2 s = part[t];
  for (int q = 1; q < parts; ++q) s = cadd(s, part[(size_t)q * nn + t]);
  M[t] = s;
}

}  // namespace

// Energy groups of the adjoint: about two waves of two blocks per SM over the
// tiles, at most 64 groups (the partial matrices)
int gradM_ds_groups(int n, int nE) {
  const long long nt = (n + kT - 1) / kT;
  const long long k = std::min<long long>({(4 * 152 + nt * nt - 1) / (nt * nt), (long long)nE, 64});
  return (int)std::max<long long>(k, 1);
}

void launch_gradM_ds(const double2* R, const double2* L, const double2* eps, int n, const double* E, const double* w,
                     int nE, int groups, float4* split, double2* part, double2* M, cudaStream_t s,
                     long long* launches) {
  if (n <= 0) return;
  const long long nn = (long long)n * n, ne = (long long)nE * n;
  float4 *Rs = split, *Ls = split + nn, *gt = split + 2 * nn;
  double* inv = reinterpret_cast<double*>(gt + ne);
  split_rows_kernel<<<dim3((unsigned)((n + kThr / 32 - 1) / (kThr / 32)), 2), kThr, 0, s>>>(R, L, n, Rs, Ls, inv);
  SWI_CHECK_LAUNCH();
  gtab_ds_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, s>>>(eps, n, E, nE, gt);
  SWI_CHECK_LAUNCH();
  const unsigned nt = (unsigned)((n + kT - 1) / kT);
  const int per = (nE + groups - 1) / groups, ng = (nE + per - 1) / per;
  double2* dst = ng > 1 ? part : M;
  gradM_ds_kernel<<<dim3(nt, nt, (unsigned)ng), kThr, 0, s>>>(Rs, Ls, gt, inv, w, n, nE, per, dst);
  SWI_CHECK_LAUNCH();
  if (ng > 1) {
    sum_parts_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(part, ng, nn, M);
    SWI_CHECK_LAUNCH();
  }
  if (launches) *launches += ng > 1 ? 4 : 3;
}

void launch_rowquad_ds(const double2* U, const double2* M, int n, long long N, float4* split, double* out,
                       cudaStream_t s, long long* launches) {
  if (n <= 0 || N <= 0) return;
  const long long nn = (long long)n * n;
  unsigned long long* mx = reinterpret_cast<unsigned long long*>(split + nn);
  SWI_CUDA_TRY(cudaMemsetAsync(mx, 0, sizeof(*mx), s));
  absmax_kernel<<<(unsigned)std::min<long long>((nn + 255) / 256, 304), 256, 0, s>>>(M, nn, mx);
  SWI_CHECK_LAUNCH();
  symsplit_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(M, n, mx, split);
  SWI_CHECK_LAUNCH();
  const unsigned grid = (unsigned)((N + kT - 1) / kT);
  if (n > kFlush * kK) rowquad_ds_kernel<true><<<grid, kThr, 0, s>>>(U, split, n, N, mx, out);
  else rowquad_ds_kernel<false><<<grid, kThr, 0, s>>>(U, split, n, N, mx, out);
  SWI_CHECK_LAUNCH();
  if (launches) *launches += 3;
}

}  // namespace swi
