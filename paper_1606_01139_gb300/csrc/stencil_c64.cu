// Shifted stencil Y = (A - sigma_col) X on complex64 vectors with FP32
// arithmetic (Eq. 1 applied matrix-free, shifted as in Eq. 3): the form for
// blocks whose rows are not 16-byte aligned (an odd column count) and for grids
// too small to fill the GPU with the deep tiles of stencil_c64_tma.cu.  A tile of
// (x, y) points fitted to the grid (at most 512 points x columns) x 4 columns, or
// 2 where no more are given, per CTA marches along z: the 13 z values of a point
// in a register queue, the x and y neighbours from the current plane staged into
// shared memory with a 6-point cross-shaped halo (ghosts by odd reflection or
// zero), two buffers so that one barrier per plane suffices.  Latency bounds it,
// so everything a plane needs is loaded two planes ahead and z is cut into whole
// waves of CTAs.  Measured on one GB300: 45x37x91, 7 columns 26 us (fixed tiles of
// 16 x 8 x 4 with a second wave of 28 CTAs took the same); 48x48x96, 2 columns ~20
// us against 47 of the TMA-staged kernel.  Layout: X, Y are [N][ld] complex64
// (float2), column index innermost.
#include <algorithm>

#include "swi_internal.cuh"

namespace swi {

namespace {

constexpr int kR = 6, kThreadsC64 = 512, kSlotsPerThread = 4;
constexpr int kWave = 152;  // CTAs resident at once
constexpr long long kMinTmaBlocks = 72;  // see launch_stencil_c64

// value of column c at axis index j of a line whose in-range extent is n
// (odd reflection about the planes -1 and n, or zero)
template <int BC>
__device__ __forceinline__ bool ghost_src(int j, int n, int& src, float& sgn) {
  if (j >= 0 && j < n) {
    src = j;
    sgn = 1.f;
    return true;
  }
  if (BC == SWI_BC_ZERO) return false;
  if (j <= -2) {
    src = -2 - j;
  } else if (j >= n + 1) {
    src = 2 * n - j;
  } else {
    return false;
  }
  if (src < 0 || src >= n) return false;  // reflection beyond the far side: a zero ghost
  sgn = -1.f;
  return true;
}

template <int BC>
__device__ __forceinline__ float2 load_z(const float2* __restrict__ X, long long pt_col, long long plane_ld, int z,
                                         int nz) {
  int src;
  float sgn;
  if (!ghost_src<BC>(z, nz, src, sgn)) return make_float2(0.f, 0.f);
  const float2 v = __ldg(X + pt_col + (long long)src * plane_ld);
  return make_float2(sgn * v.x, sgn * v.y);
}

template <int BC, int kNC>
__global__ void __launch_bounds__(kThreadsC64, 1)
    stencil_c64_kernel(const __grid_constant__ StencilC64Params P, const float2* __restrict__ X, int ldx,
                       float2* __restrict__ Y, int ldy, int ncols, const float* __restrict__ sigma, int zchunk, int TX,
                       int TY) {
  extern __shared__ float2 s_buf[];  // [2][TY + 12][TX + 12][kNC]
  const int SX = TX + 2 * kR, SY = TY + 2 * kR;
  const int cc = threadIdx.x % kNC, pt = threadIdx.x / kNC;
  const int tx = pt % TX, ty = pt / TX;
  const int tiles_x = (P.nx + TX - 1) / TX;
  const int x0 = (blockIdx.x % tiles_x) * TX, y0 = (blockIdx.x / tiles_x) * TY;
  const int c0 = blockIdx.y * kNC;
  const int x = x0 + tx, y = y0 + ty, c = c0 + cc;
  const bool mine = pt < TX * TY && x < P.nx && y < P.ny && c < ncols;
  const int z0 = blockIdx.z * zchunk, z1 = min(P.nz, z0 + zchunk);
  const long long plane = (long long)P.nx * P.ny;
  const long long plane_ld = plane * ldx;
  const long long prow = (long long)y * P.nx + x;  // point index within a plane
  const long long pt_col = prow * ldx + c;
  float cm[kR + 1];
#pragma unroll
  for (int m = 0; m <= kR; ++m) cm[m] = P.cm[m];
  const float dcen = 3.f * cm[0] - (mine ? sigma[c] : 0.f);

  // staged cells of this thread: shared index, source offset within a plane and
  // sign (0: a zero ghost or an unused cell)
  int soff[kSlotsPerThread], sidx[kSlotsPerThread];
  float ssg[kSlotsPerThread];
  const int slots_a = TY * SX * kNC, slots = slots_a + 2 * kR * TX * kNC;
#pragma unroll
  for (int k = 0; k < kSlotsPerThread; ++k) {
    const int e = threadIdx.x + k * kThreadsC64;
    const int sc = e % kNC;
    int sx, sy;
    if (e < slots_a) {
      sx = (e / kNC) % SX;
      sy = kR + e / (kNC * SX);
    } else {
      const int f = (e - slots_a) / kNC;
      sx = kR + f % TX;
      const int r = f / TX;
      sy = r < kR ? r : r + TY;
    }
    sidx[k] = -1;
    soff[k] = 0;
    ssg[k] = 0.f;
    if (e < slots) {
      sidx[k] = (sy * SX + sx) * kNC + sc;
      int srcx, srcy;
      float sgx, sgy;
      const int gc = c0 + sc;
      if (gc < ncols && ghost_src<BC>(x0 + sx - kR, P.nx, srcx, sgx) && ghost_src<BC>(y0 + sy - kR, P.ny, srcy, sgy)) {
        soff[k] = (srcy * P.nx + srcx) * ldx + gc;
        ssg[k] = sgx * sgy;
      }
    }
  }
  const int buf = SX * SY * kNC;
  const int here = ((kR + ty) * SX + kR + tx) * kNC + cc, row = SX * kNC;

  // z queue: q[k] = X at z - 6 + k, k = 0..12
  float2 q[2 * kR + 1];
#pragma unroll
  for (int k = 0; k < 2 * kR + 1; ++k)
    q[k] = mine ? load_z<BC>(X, pt_col, plane_ld, z0 - kR + k, P.nz) : make_float2(0.f, 0.f);
  // loads two steps ahead, alternating between the A and B register sets:
  // staging values of plane z + 1 / z + 2, queue entries for planes z + 7 / z + 8,
  // V and Gamma of planes z / z + 1
  float2 preA[kSlotsPerThread], preB[kSlotsPerThread];
  const auto load_plane = [&](int z, float2 (&pre)[kSlotsPerThread]) {
    const float2* Xz = X + (long long)z * plane_ld;
#pragma unroll
    for (int k = 0; k < kSlotsPerThread; ++k)
      pre[k] = (z < z1 && ssg[k] != 0.f) ? __ldg(Xz + soff[k]) : make_float2(0.f, 0.f);
  };
  const auto store_plane = [&](int z, const float2 (&pre)[kSlotsPerThread]) {
    float2* nb = s_buf + ((z - z0) & 1) * buf;
#pragma unroll
    for (int k = 0; k < kSlotsPerThread; ++k)
      if (sidx[k] >= 0) nb[sidx[k]] = make_float2(ssg[k] * pre[k].x, ssg[k] * pre[k].y);
  };
  load_plane(z0, preB);
  load_plane(z0 + 1, preA);
  float2 nqA = mine ? load_z<BC>(X, pt_col, plane_ld, z0 + kR + 1, P.nz) : make_float2(0.f, 0.f), nqB = nqA;
  float vA = mine ? __ldg(P.V + (long long)z0 * plane + prow) : 0.f;
  float gA = mine ? __ldg(P.G + (long long)z0 * plane + prow) : 0.f;
  float vB = 0.f, gB = 0.f;
  store_plane(z0, preB);
  __syncthreads();

  const auto step = [&](const int z, float2 (&pcur)[kSlotsPerThread], float2 (&pnxt)[kSlotsPerThread], float2& qcur,
                        float2& qnxt, float& vcur, float& gcur, float& vnxt, float& gnxt) {
    load_plane(z + 2, pnxt);
    qnxt = mine && z + 2 < z1 ? load_z<BC>(X, pt_col, plane_ld, z + kR + 2, P.nz) : make_float2(0.f, 0.f);
    if (mine && z + 1 < z1) {
      vnxt = __ldg(P.V + (long long)(z + 1) * plane + prow);
      gnxt = __ldg(P.G + (long long)(z + 1) * plane + prow);
    }
    if (mine) {
      const float2* s = s_buf + ((z - z0) & 1) * buf + here;
      const float d = dcen + vcur;
      const float2 u = q[kR];
      float2 a = make_float2(fmaf(d, u.x, gcur * u.y), fmaf(d, u.y, -gcur * u.x));
#pragma unroll
      for (int m = 1; m <= kR; ++m) {
        const float2 t = __fadd2_rn(__fadd2_rn(__fadd2_rn(s[-m * kNC], s[m * kNC]), __fadd2_rn(s[-m * row], s[m * row])),
                                    __fadd2_rn(q[kR - m], q[kR + m]));
        a = __ffma2_rn(make_float2(cm[m], cm[m]), t, a);
      }
      Y[((long long)z * plane + prow) * ldy + c] = a;
    }
    if (z + 1 < z1) store_plane(z + 1, pcur);
#pragma unroll
    for (int k = 0; k < 2 * kR; ++k) q[k] = q[k + 1];
    q[2 * kR] = qcur;
    __syncthreads();  // plane z + 1 is staged; plane z's buffer is written after the next barrier at the earliest
  };
  int z = z0;
  for (; z + 1 < z1; z += 2) {
    step(z, preA, preB, nqA, nqB, vA, gA, vB, gB);
    step(z + 1, preB, preA, nqB, nqA, vB, gB, vA, gA);
  }
  if (z < z1) step(z, preA, preB, nqA, nqB, vA, gA, vB, gB);
}

// Tile of at most 512 / kNC points: the extents that cover nx x ny with the
// fewest CTAs and halo cells, each axis cut evenly
void pick_tile(int nx, int ny, int kNC, int& TX, int& TY) {
  double best = 1e300;
  TX = TY = 8;
  for (int t = std::min(8, nx); t <= std::min(nx, 64); ++t) {
    const int u_max = std::min({ny, kThreadsC64 / kNC / t, 32});
    const int bx = (nx + t - 1) / t, by = (ny + u_max - 1) / u_max;
    const int w = (nx + bx - 1) / bx, v = (ny + by - 1) / by;
    const int slots = (v * (w + 2 * kR) + 2 * kR * w) * kNC;
    if (slots > kSlotsPerThread * kThreadsC64) continue;
    // a CTA costs its full width of threads, and its halo
    const double cost = (double)bx * by * (kThreadsC64 + 0.25 * slots);
    if (cost < best) {
      best = cost;
      TX = w;
      TY = v;
    }
  }
}

// Planes per CTA: a chunk of c planes costs about c + 2 plane times (filling the
// queue), so the waves of resident CTAs times that is made small
int pick_zchunk(long long ctas, int nz) {
  int zchunk = nz;
  double best = 1e300;
  for (int n = 1; n <= nz; ++n) {
    const int ch = (nz + n - 1) / n, m = (nz + ch - 1) / ch;
    if (m != n) continue;
    const double t = (double)((ctas * m + kWave - 1) / kWave) * (ch + 2);
    if (t < best) {
      best = t;
      zchunk = ch;
    }
  }
  return zchunk;
}

}  // namespace

void launch_stencil_c64(const StencilC64Params& P, const float2* X, int ldx, float2* Y, int ldy, int ncols,
                        const float* sigma_dev, cudaStream_t s, long long* launches) {
  if (ncols <= 0) return;
  // The TMA-staged kernel (16-byte aligned rows) has blocks of 32 x 8 points x 4
  // columns x at least 24 planes: with few of them, or few of their columns in
  // use, it leaves SMs or lanes idle.  Measured (this kernel / that one, us, each
  // with ~40 of host time): 48x48x96 with 2 columns (48 blocks, half used) 53/83,
  // with 8 (96) 78/80, with 16 (192) 112/88; 45x37x91 with 8 (60) 70/86; 64x64x128
  // with 4 (80) 86/79, with 2 (80, half used) 65/81; 96x96x192 with 2 (288, half
  // used) 112/109
  const long long deep = (long long)((P.nx + 31) / 32) * ((P.ny + 7) / 8) * ((ncols + 3) / 4) * std::max(1, P.nz / 24);
  if (deep * std::min(ncols, 4) >= kMinTmaBlocks * 4 && P.VG != nullptr && stencil_c64_tma_ok(X, ldx)) {
    launch_stencil_c64_tma(P, X, ldx, Y, ldy, ncols, sigma_dev, s, launches);
    return;
  }
  int TX, TY;
  const int kNC = ncols <= 2 ? 2 : 4;
  pick_tile(P.nx, P.ny, kNC, TX, TY);
  const int tiles = ((P.nx + TX - 1) / TX) * ((P.ny + TY - 1) / TY);
  const int cgroups = (ncols + kNC - 1) / kNC;
  const int zchunk = pick_zchunk((long long)tiles * cgroups, P.nz);
  const dim3 grid(tiles, cgroups, (P.nz + zchunk - 1) / zchunk);
  // at most 42 KB: the slots of a tile bound its staged cells
  const size_t smem = sizeof(float2) * 2 * (size_t)(TX + 2 * kR) * (TY + 2 * kR) * kNC;
  auto go = [&](auto kernel) {
    kernel<<<grid, kThreadsC64, smem, s>>>(P, X, ldx, Y, ldy, ncols, sigma_dev, zchunk, TX, TY);
  };
  if (kNC == 2) {
    if (P.bc == SWI_BC_ZERO) go(stencil_c64_kernel<SWI_BC_ZERO, 2>);
    else go(stencil_c64_kernel<SWI_BC_ODD, 2>);
  } else {
    if (P.bc == SWI_BC_ZERO) go(stencil_c64_kernel<SWI_BC_ZERO, 4>);
    else go(stencil_c64_kernel<SWI_BC_ODD, 4>);
  }
  SWI_CHECK_LAUNCH();
  if (launches) ++*launches;
}

}  // namespace swi
