// Shifted stencil Y = (A - sigma_col) X on complex128 vectors, in
// double-single arithmetic: the operator of Eq. 1 applied matrix-free and
// shifted as in Eq. 3, for the Krylov loop of the double-single solver.  Native
// FP64 caps the stencil at GB300's FP64 rate (two DFMA per SM clock, ~0.22
// TB/s of vectors), so it runs on the FP32 pipes, in two kernels:
//
//  pad_ds_kernel      X split once into (hi, lo) floats from its bit fields, into
//                     an array with the 6 ghost layers around the grid filled in
//                     (odd reflection or zero)
//  stencil_ds_kernel  the 37 terms of every output straight from that array: no
//                     boundary cases, no staging, no barrier
//
// FP32 issue bounds the second.  For each distance m the six neighbours are
// summed first (heads by TwoSum, tails plainly) and the sum is multiplied by the
// weight once: 8 operations per neighbour and component and 11 per distance,
// against 12 per neighbour when every term is its own product.  The weights are
// the integers 831600 c_m (the common denominator of the 12th-order formula)
// over 2^21: exact floats without tails; one double-single product by the common
// factor ends the sum.  The copy holds X / 8, so that six neighbours at the top of
// a float's range still have a sum; the factors of the last products are 8 times
// the operator's.  Real and imaginary parts go through packed FP32x2
// instructions, and nothing touches the FP64 pipe (ds::join_bits).  Neighbours
// come from L1, read ahead as far as 128 registers allow (limits of 80 or 64 for
// more warps measured within 5%).  Forms that staged a plane per barrier in shared memory and kept the 13 z values
// of a point in registers (128 registers, 16 warps) or in a shared ring took
// 286-295 us at the first size below and 16 us at the second: the splits' and
// ghosts' code alone was several thousand instructions to fetch per block.
//
// Measured on one GB300, both kernels: 48x48x96, 16 columns 150 us against 500 us
// for one product per term in 16 x 8 x 4 tiles; 10x10x20, 2 columns 10 us
// against 125 us (two blocks marching 16 planes).
// Layout: X, Y are [N][ld] complex128, column index innermost.
#include <algorithm>

#include "ds.cuh"
#include "swi_internal.cuh"

namespace swi {

namespace {

constexpr int kR = 6;
constexpr int kRowsY = 8, kThreadsDs = 32 * kRowsY;
constexpr float kIn = 0.125f, kOut = 8.f;  // scale of the padded copy, and of the factors of its products
// 831600 c_1 .. 831600 c_6, c = 12/7, -15/56, 10/189, -1/112, 2/1925, -1/16632, over 2^21
__host__ __device__ constexpr float weight(int m) {
  return (m == 1 ? 1425600.f : m == 2 ? -222750.f : m == 3 ? 44000.f : m == 4 ? -7425.f : m == 5 ? 864.f : -50.f) /
         2097152.f;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

struct dsc {  // complex double-single: heads (re, im), tails (re, im)
  float2 h, l;
};
__device__ __forceinline__ dsc unpack(float4 v) { return dsc{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }

// s += x: heads by TwoSum, the error and x's tail into the tail
__device__ __forceinline__ void acc_add(dsc& s, const dsc& x) {
  const float2 t = add2(s.h, x.h);
  const float2 bb = sub2(t, s.h);
  const float2 err = add2(sub2(s.h, sub2(t, bb)), sub2(x.h, bb));
  s.h = t;
  s.l = add2(s.l, add2(err, x.l));
}
// a += c s, c an exact real weight
__device__ __forceinline__ void acc_w(dsc& a, float c, const dsc& s) {
  const float2 w = make_float2(c, c);
  const float2 p = __fmul2_rn(w, s.h);
  float2 e = __ffma2_rn(w, s.h, make_float2(-p.x, -p.y));
  e = __ffma2_rn(w, s.l, e);
  acc_add(a, dsc{p, e});
}
// a += c s, c = ch + cl a real factor per component
__device__ __forceinline__ void acc_mul(dsc& a, float2 ch, float2 cl, const dsc& s) {
  const float2 p = __fmul2_rn(ch, s.h);
  float2 e = __ffma2_rn(ch, s.h, make_float2(-p.x, -p.y));
  e = __ffma2_rn(ch, s.l, e);
  e = __ffma2_rn(cl, s.h, e);
  acc_add(a, dsc{p, e});
}

// source index of axis index j on a line of n points; sgn 0: a zero ghost
__device__ __forceinline__ int ghost(int j, int n, bool zero, float& sgn) {
  if (j >= 0 && j < n) return j;
  if (zero || j == -1 || j == n) {
    sgn = 0.f;
    return 0;
  }
  const int s = j < 0 ? -2 - j : 2 * n - j;
  if (s < 0 || s >= n) {  // reflection beyond the far side
    sgn = 0.f;
    return 0;
  }
  sgn = -sgn;
  return s;
}

// P[z + 6][y + 6][(x + 6) nc + c] = X / 8 split, ghosts filled in; a block per rows of
// (y, z), lanes along (x, c).  Only the cells a 37-point cross reads are needed:
// a row with two or more of its coordinates outside is skipped.
__global__ void __launch_bounds__(256) pad_ds_kernel(const double2* __restrict__ X, int ldx, int nc, int nx, int ny,
                                                     int nz, int zero, float4* __restrict__ P) {
  const int px = nx + 2 * kR, py = ny + 2 * kR;
  const long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);  // (z + 6) py + y + 6
  if (row >= (long long)py * (nz + 2 * kR)) return;
  const int z = (int)(row / py) - kR, y = (int)(row % py) - kR;
  const bool zin = z >= 0 && z < nz, yin = y >= 0 && y < ny;
  if (!zin && !yin) return;
  const bool inner = zin && yin;  // else: ghost rows need no x ghosts
  float srow = 1.f;
  const int sz = ghost(z, nz, zero, srow);
  const int sy = ghost(y, ny, zero, srow);
  const double2* src = X + ((long long)sz * ny + sy) * nx * ldx;
  float4* dst = P + row * px * nc;
  const bool near = px * nc < (1 << 22);
  const float inv = 1.f / (float)nc;  // f / nc for f < 2^22 (the half keeps it off the integers)
  for (int f = blockIdx.y * 32 + (threadIdx.x & 31); f < px * nc; f += gridDim.y * 32) {
    const int xx = near ? (int)(((float)f + 0.5f) * inv) : f / nc, c = f - xx * nc, x = xx - kR;
    float s = srow;
    int sx = x;
    if (x < 0 || x >= nx) {
      if (!inner) continue;
      sx = ghost(x, nx, zero, s);
    }
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (s != 0.f) {
      const double2 v = __ldg(src + (long long)sx * ldx + c);
      ds::split_wide(v.x, o.x, o.z);
      ds::split_wide(v.y, o.y, o.w);
      s *= kIn;
      o = make_float4(s * o.x, s * o.y, s * o.z, s * o.w);
    }
    dst[f] = o;
  }
}

__global__ void __launch_bounds__(kThreadsDs, 2)
    stencil_ds_kernel(const float4* __restrict__ P, int nc, int nx, int ny, int nz, const float4* __restrict__ VG,
                      const double* __restrict__ sigma, double cm0, float2 fac,  // 8 c_m = (fac.x + fac.y) weight(m)
                      double2* __restrict__ Y, int ldy, int out_ds, int zchunk) {
  const int xb = (nx * nc + 31) / 32;  // blocks along (x, c)
  const int f = (blockIdx.x % xb) * 32 + (threadIdx.x & 31), y = (blockIdx.x / xb) * kRowsY + (threadIdx.x >> 5);
  if (f >= nx * nc || y >= ny) return;
  const int x = f / nc, c = f - x * nc;
  const int px = nx + 2 * kR, py = ny + 2 * kR;
  const int rowp = px * nc;                     // elements between y neighbours
  const long long planep = (long long)rowp * py;  // and between z neighbours
  const int z0 = blockIdx.y * zchunk, z1 = min(nz, z0 + zchunk);
  ds::df dcen;  // 8 (3 c_0 - sigma)
  ds::split_wide(3.0 * cm0 - sigma[c], dcen.h, dcen.l);
  dcen.h *= kOut;
  dcen.l *= kOut;
  const float4* p = P + (long long)(z0 + kR) * planep + (long long)(y + kR) * rowp + (x + kR) * nc + c;
  for (int z = z0; z < z1; ++z, p += planep) {
    const long long r = ((long long)z * ny + y) * nx + x;
    const float4 vg = __ldg(VG + r);
    dsc k{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int m = 1; m <= kR; ++m) {
      dsc t = unpack(__ldg(p - m * nc));
      acc_add(t, unpack(__ldg(p + m * nc)));
      acc_add(t, unpack(__ldg(p - m * rowp)));
      acc_add(t, unpack(__ldg(p + m * rowp)));
      acc_add(t, unpack(__ldg(p - m * planep)));
      acc_add(t, unpack(__ldg(p + m * planep)));
      acc_w(k, weight(m), t);
    }
    // (d - i g) u: re = d ur + g ui, im = d ui - g ur
    const dsc u = unpack(__ldg(p));
    const ds::df d = ds::add(ds::df{vg.x, vg.y}, dcen);
    dsc a{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    acc_mul(a, make_float2(d.h, d.h), make_float2(d.l, d.l), u);
    acc_mul(a, make_float2(vg.z, -vg.z), make_float2(vg.w, -vg.w),
            dsc{make_float2(u.h.y, u.h.x), make_float2(u.l.y, u.l.x)});
    acc_mul(a, make_float2(fac.x, fac.x), make_float2(fac.y, fac.y), k);
    const ds::df re = ds::two_sum(a.h.x, a.l.x), im = ds::two_sum(a.h.y, a.l.y);
    if (out_ds)
      reinterpret_cast<float4*>(Y)[r * ldy + c] = make_float4(re.h, re.l, im.h, im.l);
    else
      Y[r * ldy + c] = make_double2(ds::join_bits(re.h, re.l), ds::join_bits(im.h, im.l));
  }
}

__global__ void pack_vg_ds_kernel(const double* __restrict__ V, const double* __restrict__ G, long long n,
                                  float4* __restrict__ out) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    float4 o;
    ds::split_bits(V[e], o.x, o.y);
    ds::split_bits(G[e], o.z, o.w);
    out[e] = make_float4(kOut * o.x, kOut * o.y, kOut * o.z, kOut * o.w);
  }
}

long long padded(const StencilParams& P) {
  return (long long)(P.nx + 2 * kR) * (P.ny + 2 * kR) * (P.nz + 2 * kR);
}
// columns per pass: all of a block of at most 32, fewer (at least one) when the
// padded copy would pass 2 GB
int pass_columns(const StencilParams& P, int ncols) {
  const long long most = std::max<long long>(1, (2LL << 30) / (16 * padded(P)));
  return (int)std::min<long long>({(long long)ncols, 32, most});
}

}  // namespace

void launch_pack_vg_ds(const double* V, const double* G, long long n, float4* out, cudaStream_t s) {
  pack_vg_ds_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 4096), 256, 0, s>>>(V, G, n, out);
  SWI_CHECK_LAUNCH();
}

size_t stencil_ds_work_bytes(const StencilParams& P, int ncols) {
  return sizeof(float4) * (size_t)padded(P) * pass_columns(P, std::max(ncols, 1));
}

void launch_stencil_ds(const StencilParams& P, const double2* X, int ldx, double2* Y, int ldy, int ncols, int out_ds,
                       const double* sigma_dev, float4* work, cudaStream_t s, long long* launches) {
  if (ncols <= 0) return;
  if (P.VGds == nullptr || work == nullptr)
    throw Error{SWI_ESTATE, "double-single stencil: the split (V, Gamma) array or the work space is missing"};
  const double fd = P.cm[1] / (double)weight(1);
  const float2 fac = make_float2(kOut * (float)fd, kOut * (float)(fd - (double)(float)fd));
  const int px = P.nx + 2 * kR;
  const long long rows = (long long)(P.ny + 2 * kR) * (P.nz + 2 * kR);
  const int step = pass_columns(P, ncols);
  for (int c0 = 0; c0 < ncols; c0 += step) {
    const int nc = std::min(step, ncols - c0);
    pad_ds_kernel<<<dim3((unsigned)((rows + 7) / 8), std::min((px * nc + 127) / 128, 65535)), 256, 0, s>>>(
        X + c0, ldx, nc, P.nx, P.ny, P.nz, P.bc == SWI_BC_ZERO, work);
    SWI_CHECK_LAUNCH();
    // z chunks: about six rounds of the two blocks an SM holds, so that the
    // last round is short; a block that marches more planes finds its z
    // neighbours in L1
    const long long per = (long long)((P.nx * nc + 31) / 32) * ((P.ny + kRowsY - 1) / kRowsY);
    const int nzc = (int)std::min<long long>(P.nz, std::max<long long>(1, (12LL * 152 + per - 1) / per));
    const int zchunk = std::max((P.nz + nzc - 1) / nzc, (P.nz + 65534) / 65535);
    const dim3 grid((unsigned)per, (P.nz + zchunk - 1) / zchunk);
    stencil_ds_kernel<<<grid, kThreadsDs, 0, s>>>(work, nc, P.nx, P.ny, P.nz, P.VGds, sigma_dev + c0, P.cm[0], fac,
                                                  Y + c0, ldy, out_ds, zchunk);
    SWI_CHECK_LAUNCH();
    if (launches) *launches += 2;
  }
}

}  // namespace swi
