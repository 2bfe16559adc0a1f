// Grid kernels: Yee FDTD curl updates (§2 Maxwell curl equations, FDTD on
// the Yee lattice per ref [9] of the paper), particle load/unload between
// global FP64 coordinates and (cell, offset), and the FP64 diagnostics.
#include <cuda_runtime.h>
#include <math.h>

#include "pic_device.cuh"

namespace pic {

namespace {

int grid_blocks(int64_t n, int per_block) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (n + per_block - 1) / per_block;
  const int64_t cap = (int64_t)nsm * 32;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

template <class R> struct YeeArgs {
  int n[3];
  int absorb;  // x walls absorbing: wall nodes are left to the Mur kernels
  R rdx[3];  // 1/dx_a
  R h;       // time step of this update
  R *E[3];
  R *B[3];
  const R *J[3];
};

// 3D runs: the three updates as launches of their own (2D: k_field_step2).
// B <- B - h curl E, curl E at the B locations.
template <class R>
__global__ void __launch_bounds__(256) k_yee_b(YeeArgs<R> a) {
  after_previous();
  const int n0 = a.n[0], n1 = a.n[1], n2 = a.n[2];
  const int64_t ncell = (int64_t)n0 * n1 * n2;
  const int64_t sy = n0, sz = (int64_t)n0 * n1;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(c % n0);
    const int64_t r = c / n0;
    const int j = (int)(r % n1);
    const int k = (int)(r / n1);
    const int64_t cxp = c + (i + 1 < n0 ? 1 : 1 - n0);
    const int64_t cyp = c + (j + 1 < n1 ? sy : sy - sy * n1);
    const R ex = a.E[0][c], ey = a.E[1][c], ez = a.E[2][c];
    R cx = (a.E[2][cyp] - ez) * a.rdx[1];
    R cy = -(a.E[2][cxp] - ez) * a.rdx[0];
    const R cz = (a.E[1][cxp] - ey) * a.rdx[0] - (a.E[0][cyp] - ex) * a.rdx[1];
    const int64_t czp = c + (k + 1 < n2 ? sz : sz - sz * n2);
    cx -= (a.E[1][czp] - ey) * a.rdx[2];
    cy += (a.E[0][czp] - ex) * a.rdx[2];
    a.B[0][c] -= a.h * cx;
    if (a.absorb && i == n0 - 1) continue;  // By, Bz half a cell beyond the last node
    a.B[1][c] -= a.h * cy;
    a.B[2][c] -= a.h * cz;
  }
}

// E <- E + h (curl B - J), curl B at the E locations.
template <class R>
__global__ void __launch_bounds__(256) k_yee_e(YeeArgs<R> a) {
  after_previous();
  const int n0 = a.n[0], n1 = a.n[1], n2 = a.n[2];
  const int64_t ncell = (int64_t)n0 * n1 * n2;
  const int64_t sy = n0, sz = (int64_t)n0 * n1;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(c % n0);
    const int64_t r = c / n0;
    const int j = (int)(r % n1);
    const int k = (int)(r / n1);
    const int64_t cxm = c - (i > 0 ? 1 : 1 - n0);
    const int64_t cym = c - (j > 0 ? sy : sy - sy * n1);
    const R bx = a.B[0][c], by = a.B[1][c], bz = a.B[2][c];
    R cx = (bz - a.B[2][cym]) * a.rdx[1];
    R cy = -(bz - a.B[2][cxm]) * a.rdx[0];
    const R cz = (by - a.B[1][cxm]) * a.rdx[0] - (bx - a.B[0][cym]) * a.rdx[1];
    const int64_t czm = c - (k > 0 ? sz : sz - sz * n2);
    cx -= (by - a.B[1][czm]) * a.rdx[2];
    cy += (bx - a.B[0][czm]) * a.rdx[2];
    if (a.absorb && i == n0 - 1) continue;  // wall node (Mur) and Ex beyond the last node
    a.E[0][c] += a.h * (cx - a.J[0][c]);
    if (a.absorb && i == 0) continue;       // wall node (Mur)
    a.E[1][c] += a.h * (cy - a.J[1][c]);
    a.E[2][c] += a.h * (cz - a.J[2][c]);
  }
}

// The same two updates with 16-byte vector accesses along x: a thread takes
// W = 16 / sizeof(R) consecutive cells of one row (four FP32 or two FP64
// values per component), on a 3D grid of (x groups, rows, planes), so there
// is no division per cell and every load and store of a warp is 512
// contiguous bytes.  The neighbour across the group's end in x is one extra
// scalar load (cached; the adjacent thread reads it too), with the periodic
// wrap at the ends of the row.  Used when the row length is a multiple of W
// (so every component array is 16-byte aligned); the scalar kernels above
// take the other grids.
template <class R> struct alignas(16) Pack {
  R v[16 / sizeof(R)];
};
template <class R> __device__ __forceinline__ Pack<R> ldp(const R *p) { return *reinterpret_cast<const Pack<R> *>(p); }
template <class R> __device__ __forceinline__ void stp(R *p, const Pack<R> &v) { *reinterpret_cast<Pack<R> *>(p) = v; }

template <class R>
__global__ void __launch_bounds__(256) k_yee_b_vec(YeeArgs<R> a) {
  after_previous();
  constexpr int W = 16 / sizeof(R);
  const int n0 = a.n[0], n1 = a.n[1], n2 = a.n[2];
  const int nq = n0 / W;
  const int iq = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (iq >= nq || j >= n1) return;
  const int64_t sy = n0, sz = (int64_t)n0 * n1;
  const int64_t row = (int64_t)j * sy + (int64_t)k * sz;
  const int64_t c = row + (int64_t)iq * W;
  const int64_t cyp = j + 1 < n1 ? c + sy : c + sy - sy * n1;
  const int64_t cxn = iq + 1 < nq ? c + W : row;  // x + 1 of the group's last cell
  const Pack<R> ex = ldp(a.E[0] + c), ey = ldp(a.E[1] + c), ez = ldp(a.E[2] + c);
  const Pack<R> ex_yp = ldp(a.E[0] + cyp), ez_yp = ldp(a.E[2] + cyp);
  const R ey_xn = a.E[1][cxn], ez_xn = a.E[2][cxn];
  const int64_t czp = k + 1 < n2 ? c + sz : c + sz - sz * n2;
  const Pack<R> ex_zp = ldp(a.E[0] + czp);
  const Pack<R> ey_zp = ldp(a.E[1] + czp);
  Pack<R> bx = ldp(a.B[0] + c), by = ldp(a.B[1] + c), bz = ldp(a.B[2] + c);
  // By, Bz half a cell beyond the last node stay as they are at absorbing walls
  const bool last = a.absorb && iq == nq - 1;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const R eyx = w + 1 < W ? ey.v[w + 1] : ey_xn, ezx = w + 1 < W ? ez.v[w + 1] : ez_xn;
    R cx = (ez_yp.v[w] - ez.v[w]) * a.rdx[1];
    R cy = -(ezx - ez.v[w]) * a.rdx[0];
    const R cz = (eyx - ey.v[w]) * a.rdx[0] - (ex_yp.v[w] - ex.v[w]) * a.rdx[1];
    cx -= (ey_zp.v[w] - ey.v[w]) * a.rdx[2];
    cy += (ex_zp.v[w] - ex.v[w]) * a.rdx[2];
    bx.v[w] -= a.h * cx;
    if (!(last && w == W - 1)) {
      by.v[w] -= a.h * cy;
      bz.v[w] -= a.h * cz;
    }
  }
  stp(a.B[0] + c, bx);
  stp(a.B[1] + c, by);
  stp(a.B[2] + c, bz);
}

template <class R>
__global__ void __launch_bounds__(256) k_yee_e_vec(YeeArgs<R> a) {
  after_previous();
  constexpr int W = 16 / sizeof(R);
  const int n0 = a.n[0], n1 = a.n[1], n2 = a.n[2];
  const int nq = n0 / W;
  const int iq = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (iq >= nq || j >= n1) return;
  const int64_t sy = n0, sz = (int64_t)n0 * n1;
  const int64_t row = (int64_t)j * sy + (int64_t)k * sz;
  const int64_t c = row + (int64_t)iq * W;
  const int64_t cym = j > 0 ? c - sy : c - sy + sy * n1;
  const int64_t cxp = iq > 0 ? c - 1 : row + n0 - 1;  // x - 1 of the group's first cell
  const Pack<R> bx = ldp(a.B[0] + c), by = ldp(a.B[1] + c), bz = ldp(a.B[2] + c);
  const Pack<R> bx_ym = ldp(a.B[0] + cym), bz_ym = ldp(a.B[2] + cym);
  const R by_xp = a.B[1][cxp], bz_xp = a.B[2][cxp];
  const int64_t czm = k > 0 ? c - sz : c - sz + sz * n2;
  const Pack<R> bx_zm = ldp(a.B[0] + czm);
  const Pack<R> by_zm = ldp(a.B[1] + czm);
  const Pack<R> jx = ldp(a.J[0] + c), jy = ldp(a.J[1] + c), jz = ldp(a.J[2] + c);
  Pack<R> ex = ldp(a.E[0] + c), ey = ldp(a.E[1] + c), ez = ldp(a.E[2] + c);
  // at absorbing walls the wall nodes belong to the Mur kernels, and Ex
  // half a cell beyond the last node is not updated
  const bool first = a.absorb && iq == 0, last = a.absorb && iq == nq - 1;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const R byx = w > 0 ? by.v[w - 1] : by_xp, bzx = w > 0 ? bz.v[w - 1] : bz_xp;
    R cx = (bz.v[w] - bz_ym.v[w]) * a.rdx[1];
    R cy = -(bz.v[w] - bzx) * a.rdx[0];
    const R cz = (by.v[w] - byx) * a.rdx[0] - (bx.v[w] - bx_ym.v[w]) * a.rdx[1];
    cx -= (by.v[w] - by_zm.v[w]) * a.rdx[2];
    cy += (bx.v[w] - bx_zm.v[w]) * a.rdx[2];
    const bool wall_hi = last && w == W - 1, wall_lo = first && w == 0;
    if (!wall_hi) ex.v[w] += a.h * (cx - jx.v[w]);
    if (!wall_hi && !wall_lo) {
      ey.v[w] += a.h * (cy - jy.v[w]);
      ez.v[w] += a.h * (cz - jz.v[w]);
    }
  }
  stp(a.E[0] + c, ex);
  stp(a.E[1] + c, ey);
  stp(a.E[2] + c, ez);
}

// Vector path when the row length is a multiple of W and every array is
// 16-byte aligned; block (x groups, rows) with 256 threads.
template <class R> bool yee_vec_ok(const Grid &g, const YeeArgs<R> &a, bool with_j) {
  constexpr int W = 16 / sizeof(R);
  if (g.n[0] % W != 0 || g.n[2] > 65535) return false;
  for (int d = 0; d < 3; ++d) {
    if (reinterpret_cast<uintptr_t>(a.E[d]) % 16 || reinterpret_cast<uintptr_t>(a.B[d]) % 16) return false;
    if (with_j && reinterpret_cast<uintptr_t>(a.J[d]) % 16) return false;
  }
  return true;
}
template <class R> void yee_vec_shape(const Grid &g, dim3 &grid, dim3 &block) {
  constexpr int W = 16 / sizeof(R);
  const int nq = g.n[0] / W;
  const int bx = nq >= 64 ? 64 : 32;
  block = dim3(bx, 256 / bx, 1);
  grid = dim3((nq + bx - 1) / bx, (g.n[1] + block.y - 1) / block.y, g.n[2]);
}

template <class R>
__global__ void k_mur_save(int n0, int n1, int n2, const R *Ey, const R *Ez, double *buf) {
  after_previous();
  const int64_t nyz = (int64_t)n1 * n2;
  const int nodes[4] = {0, 1, n0 - 2, n0 - 1};
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < 8 * nyz; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t jk = q % nyz;
    const int cq = (int)(q / nyz);  // component * 4 + node slot
    const R *E = cq < 4 ? Ey : Ez;
    buf[q] = (double)E[nodes[cq & 3] + (int64_t)n0 * jk];
  }
}

// E(0)^{n+1} = L(0)^{n+1} + S(1)^n + k (S(1)^{n+1} - S(0)^n), S = E - L the
// scattered field, k = (dt - dx)/(dt + dx); the same without L at x = n0-1.
// L = P(row) times the step's four waveform values (LaserStep).
template <class R>
__global__ void k_mur_apply(int n0, int n1, int n2, double dx, double dt, R *Ey, R *Ez, const double *buf,
                            LaserStep ls) {
  after_previous();
  const int64_t nyz = (int64_t)n1 * n2;
  const double kc = (dt - dx) / (dt + dx);
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < 2 * nyz; q += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(q / nyz);  // 0: Ey, 1: Ez
    const int64_t jk = q % nyz;
    R *E = c == 0 ? Ey : Ez;
    const double *o = buf + (int64_t)c * 4 * nyz;
    double l0o = 0.0, l1o = 0.0, l0n = 0.0, l1n = 0.0;
    if (ls.pol == c + 1) {
      if (ls.oblique) {
        // the wall row's own delay and profile (Ey rows at (j + 1/2, k), Ez rows at (j, k + 1/2))
        const int j = (int)(jk % n1), k = (int)(jk / n1);
        const double y = (j + (c == 0 ? 0.5 : 0.0)) * ls.dy, z = (k + (c == 1 ? 0.5 : 0.0)) * ls.dz;
        l0o = laser_wave(ls, 0.0, y, z, ls.t_old);
        l1o = laser_wave(ls, ls.dx, y, z, ls.t_old);
        l0n = laser_wave(ls, 0.0, y, z, ls.t_new);
        l1n = laser_wave(ls, ls.dx, y, z, ls.t_new);
      } else {
        const double p = ls.prof[jk];
        l0o = p * ls.amp[0];
        l1o = p * ls.amp[1];
        l0n = p * ls.amp[2];
        l1n = p * ls.amp[3];
      }
    }
    const int64_t row = (int64_t)n0 * jk;
    const double s0o = o[0 * nyz + jk] - l0o;
    const double s1o = o[1 * nyz + jk] - l1o;
    const double s1n = (double)E[row + 1] - l1n;
    E[row] = (R)(l0n + s1o + kc * (s1n - s0o));
    const double r1o = o[2 * nyz + jk], r0o = o[3 * nyz + jk];
    const double r1n = (double)E[row + n0 - 2];
    E[row + n0 - 1] = (R)(r1o + kc * (r1n - r0o));
  }
}

template <class R>
YeeArgs<R> yee_args(const Grid &g, void *const E[3], void *const B[3], void *const J[3], double h) {
  YeeArgs<R> a;
  a.absorb = g.absorb_lo || g.absorb_hi;
  for (int d = 0; d < 3; ++d) {
    a.n[d] = g.n[d];
    a.rdx[d] = (R)(1.0 / g.dx[d]);
    a.E[d] = static_cast<R *>(E[d]);
    a.B[d] = static_cast<R *>(B[d]);
    a.J[d] = J ? static_cast<const R *>(J[d]) : nullptr;
  }
  a.h = (R)h;
  return a;
}

// ---- the whole field update of a 2D step in one pass ----
// B half, E (with the Mur walls and the incoming wave) and B half from the
// fields E, B into E2, B2, and the next step's J cleared.  A warp takes a
// strip of kStripW columns and `rows` rows, one lane per column with one lane
// of halo below and two above, and marches along y: a row's y neighbours are
// the registers of the passes before and after, its x neighbours come by
// shuffle, so that there is no shared memory and no barrier.  The halo's
// intermediate values are recomputed by every strip that needs them.
//
// Five launches with walls and 132 B per cell before (FP32), 72 B now with
// the 12 that clear J.  Small grids are bound by launches and by the chain of
// dependent passes, large ones by loads in flight: 2048 x 1024 FP32 with walls
// 36 us (4.2 TB/s) where the launches took 55 and their gaps; 64 x 64 FP64 6.2
// us (14.5).
template <class R> struct FieldStep2 {
  int n0, n1, absorb;
  int width, rows;  // output columns and rows of a strip
  unsigned strips;  // strips side by side
  R rdx, rdy, h;    // h: the full step
  const R *E[3], *B[3], *J[3];
  R *E2[3], *B2[3], *Jn[3];
  double kc;  // Mur: (dt - dx) / (dt + dx)
  LaserStep ls;
  unsigned long long *counters;  // escape counters cleared for the next step's pushes
  int ncounters;
};
constexpr int kStripW = 29;

template <class R> __global__ void __launch_bounds__(64) k_field_step2(const __grid_constant__ FieldStep2<R> a) {
  after_previous();
  const int lane = threadIdx.x & 31;
  if (blockIdx.x == 0)
    for (int k = threadIdx.x; k < a.ncounters; k += blockDim.x) a.counters[k] = 0;
  const int x0 = (int)(blockIdx.x % a.strips) * a.width;
  const int y0 = (int)((blockIdx.x / a.strips * (blockDim.x / 32) + (threadIdx.x >> 5)) * a.rows);
  if (y0 >= a.n1) return;
  const int rows = min(a.rows, a.n1 - y0);
  int i = x0 - 1 + lane;  // this lane's column, wrapped
  const bool mine = lane >= 1 && lane <= a.width && i < a.n0;
  i %= a.n0;
  if (i < 0) i += a.n0;
  const bool wall_lo = a.absorb && i == 0, wall_hi = a.absorb && i == a.n0 - 1;
  // the wave at the x = 0 wall: this strip's rows in groups of eight, four
  // values of a row in four lanes (L0, L1 at the old and at the new time)
  const bool wave = a.absorb && a.ls.pol != 0 && x0 == 0;
  double wv = 0.0;
  const bool has_lo = __any_sync(0xffffffffu, wall_lo), has_hi = __any_sync(0xffffffffu, wall_hi);
  const auto row = [&](int j) {  // y0 + j, wrapped (rows -1 .. rows + 1 are asked for)
    int y = y0 + j;
    while (y >= a.n1) y -= a.n1;
    return (y < 0 ? a.n1 - 1 : y) * a.n0 + i;  // (cells stay below 2^30)
  };
  R e[3], en[3], bh[3], bhm[3], ep[3], epm[3], bhp[3];
  R b[3], jv[3], bn[3], jn[3], enn[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int g = row(-1), g1 = row(0);
    e[c] = a.E[c][g];
    en[c] = a.E[c][g1];
    b[c] = a.B[c][g];
    jv[c] = R(0);
    bhm[c] = epm[c] = bhp[c] = R(0);
  }
  const R hh = R(0.5) * a.h;
  for (int j = -1; j <= rows; ++j) {
    // the next pass's loads first
    if (j < rows) {
      const int g1 = row(j + 1), g2 = row(j + 2);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        bn[c] = a.B[c][g1];
        jn[c] = a.J[c][g1];
        enn[c] = a.E[c][g2];
      }
    }
    // B half: B - h/2 curl E (rows j, j + 1)
    {
      const R eyx = __shfl_down_sync(0xffffffffu, e[1], 1), ezx = __shfl_down_sync(0xffffffffu, e[2], 1);
      const R cx = (en[2] - e[2]) * a.rdy;
      const R cy = -(ezx - e[2]) * a.rdx;
      const R cz = (eyx - e[1]) * a.rdx - (en[0] - e[0]) * a.rdy;
      bh[0] = b[0] - hh * cx;
      bh[1] = wall_hi ? b[1] : b[1] - hh * cy;  // By, Bz half a cell beyond the last node
      bh[2] = wall_hi ? b[2] : b[2] - hh * cz;
    }
    // E: E + h (curl B - J) (rows j - 1, j)
    const R byx = __shfl_up_sync(0xffffffffu, bh[1], 1), bzx = __shfl_up_sync(0xffffffffu, bh[2], 1);
    if (j >= 0) {
      const R cx = (bh[2] - bhm[2]) * a.rdy;
      const R cy = -(bh[2] - bzx) * a.rdx;
      const R cz = (bh[1] - byx) * a.rdx - (bh[0] - bhm[0]) * a.rdy;
      ep[0] = wall_hi ? e[0] : e[0] + a.h * (cx - jv[0]);
      ep[1] = wall_hi || wall_lo ? e[1] : e[1] + a.h * (cy - jv[1]);
      ep[2] = wall_hi || wall_lo ? e[2] : e[2] + a.h * (cz - jv[2]);
      if (a.absorb) {
        if (wave && j % 8 == 0) {
          // rows j .. j + 7: value lane % 4 of row lane / 4
          const int y = (y0 + j + lane / 4) % a.n1;
          const int v = lane % 4;
          if (a.ls.oblique)
            wv = laser_wave(a.ls, (v & 1) ? a.ls.dx : 0.0, (y + (a.ls.pol == 1 ? 0.5 : 0.0)) * a.ls.dy,
                            a.ls.pol == 2 ? 0.5 * a.ls.dz : 0.0, v < 2 ? a.ls.t_old : a.ls.t_new);
          else
            wv = a.ls.prof[y] * a.ls.amp[v];
        }
        // (only the warps that hold a wall's column take these branches: left
        // to every warp, the FP64 of the two lines cost three times the rest)
        if (has_lo) {
          double l[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) l[v] = __shfl_sync(0xffffffffu, wv, (j & 7) * 4 + v);
#pragma unroll
          for (int c = 1; c < 3; ++c) {
            // the neighbour inside, at the old and at the new time
            const R oi = __shfl_down_sync(0xffffffffu, e[c], 1), ni = __shfl_down_sync(0xffffffffu, ep[c], 1);
            const bool in = wave && a.ls.pol == c;
            const double s0o = (double)e[c] - (in ? l[0] : 0.0), s1o = (double)oi - (in ? l[1] : 0.0);
            const double s1n = (double)ni - (in ? l[3] : 0.0);
            if (wall_lo) ep[c] = (R)((in ? l[2] : 0.0) + s1o + a.kc * (s1n - s0o));
          }
        }
        if (has_hi)
#pragma unroll
          for (int c = 1; c < 3; ++c) {
            const R ox = __shfl_up_sync(0xffffffffu, e[c], 1), nx = __shfl_up_sync(0xffffffffu, ep[c], 1);
            if (wall_hi) ep[c] = (R)((double)ox + a.kc * ((double)nx - (double)e[c]));
          }
      }
    }
    // B half of the row before: B - h/2 curl E (rows j - 1, j), and the results
    const R eyx = __shfl_down_sync(0xffffffffu, epm[1], 1), ezx = __shfl_down_sync(0xffffffffu, epm[2], 1);
    if (j >= 1 && mine) {
      const R cx = (ep[2] - epm[2]) * a.rdy;
      const R cy = -(ezx - epm[2]) * a.rdx;
      const R cz = (eyx - epm[1]) * a.rdx - (ep[0] - epm[0]) * a.rdy;
      const int g = (y0 + j - 1) * a.n0 + i;
      a.B2[0][g] = bhp[0] - hh * cx;
      a.B2[1][g] = wall_hi ? bhp[1] : bhp[1] - hh * cy;
      a.B2[2][g] = wall_hi ? bhp[2] : bhp[2] - hh * cz;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        a.E2[c][g] = epm[c];
        a.Jn[c][g] = R(0);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      bhm[c] = bhp[c] = bh[c];
      epm[c] = ep[c];
      e[c] = en[c];
      en[c] = enn[c];
      b[c] = bn[c];
      jv[c] = jn[c];
    }
  }
}

// ---- particle load: global (x, y, z) -> (cell, offset) ----
template <class R>
__global__ void k_load(int dims, int n0, int n1, int n2, double rdx0, double rdx1, double rdx2, int absorb, Particles p,
                       int64_t offset, int64_t n, const double *__restrict__ x, const double *__restrict__ y,
                       const double *__restrict__ z, const double *__restrict__ ux, const double *__restrict__ uy,
                       const double *__restrict__ uz, const double *__restrict__ w, const uint32_t *__restrict__ id,
                       uint32_t id_base, unsigned long long *bad) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const double pos[3] = {x[q] * rdx0, y[q] * rdx1, dims == 3 ? z[q] * rdx2 : 0.0};
    const int nn[3] = {n0, n1, n2};
    int ci[3] = {0, 0, 0};
    R off[3] = {R(0), R(0), R(0)};
    // non-finite positions, momenta or weights are not loaded (marked dead)
    bool ok = isfinite(ux[q]) && isfinite(uy[q]) && isfinite(uz[q]) && isfinite(w[q]);
    for (int d = 0; d < dims; ++d) {
      if (!isfinite(pos[d])) {
        ok = false;
        continue;
      }
      const double fl = floor(pos[d]);
      double f = pos[d] - fl;
      long long i = (long long)fl;
      R fr = (R)f;
      if (fr >= R(1)) {  // rounding of the narrowing conversion
        fr = R(0);
        i += 1;
      }
      if (d == 0 && absorb && (pos[0] < kWallLo || pos[0] >= nn[0] - kWallHiMargin)) ok = false;
      i %= nn[d];
      if (i < 0) i += nn[d];
      ci[d] = (int)i;
      off[d] = fr;
    }
    const int64_t s = offset + q;
    if (!ok) {
      atomicAdd(bad, 1ull);
      p.cell[s] = -1;
    } else {
      p.cell[s] = ci[0] + n0 * (ci[1] + n1 * ci[2]);
    }
    for (int d = 0; d < 3; ++d) {
      if (d < dims) static_cast<R *>(p.off[d])[s] = off[d];
    }
    static_cast<R *>(p.u[0])[s] = (R)ux[q];
    static_cast<R *>(p.u[1])[s] = (R)uy[q];
    static_cast<R *>(p.u[2])[s] = (R)uz[q];
    static_cast<R *>(p.w)[s] = (R)w[q];
    p.id[s] = id ? id[q] : id_base + (uint32_t)q;  // no tags given: running index
  }
}

// ---- validation of particle storage copied in from outside (state resume) ----
// A slot below n is valid when it is dead (cell -1) or when its cell lies in
// the grid (and, with absorbing x walls, its position between them), its
// offsets on the grid's axes are in [0, 1) and its momenta and weight are
// finite.  Invalid slots are counted in *bad.
template <class R>
__global__ void k_check_particles(int dims, int n0, int64_t ncell, int absorb, Particles p, int64_t n,
                                  unsigned long long *bad) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int c = p.cell[q];
    if (c == -1) continue;
    bool ok = c >= 0 && (int64_t)c < ncell;
    for (int d = 0; d < dims; ++d) {
      const R f = static_cast<const R *>(p.off[d])[q];
      ok = ok && f >= R(0) && f < R(1);  // false for NaN
    }
    for (int d = 0; d < 3; ++d) ok = ok && isfinite(static_cast<const R *>(p.u[d])[q]);
    ok = ok && isfinite(static_cast<const R *>(p.w)[q]);
    if (ok && absorb) {
      const double X = (double)(c % n0) + (double)static_cast<const R *>(p.off[0])[q];
      ok = X >= kWallLo && X < n0 - kWallHiMargin;
    }
    if (!ok) atomicAdd(bad, 1ull);
  }
}

// ---- particle unload: (cell, offset) -> global FP64 ----
template <class R>
__global__ void k_unload(int dims, int n0, int n1, double dx0, double dx1, double dx2, Particles p,
                         const int64_t *__restrict__ d_count, double *x, double *y, double *z, double *ux, double *uy,
                         double *uz, double *w, uint32_t *id, int32_t *alive) {
  const int64_t n = *d_count;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int c = p.cell[q];
    const int i = c < 0 ? 0 : c % n0;
    const int r = c < 0 ? 0 : c / n0;
    const int j = r % n1;
    const int k = r / n1;
    if (x) x[q] = ((double)i + (double)static_cast<const R *>(p.off[0])[q]) * dx0;
    if (y) y[q] = ((double)j + (double)static_cast<const R *>(p.off[1])[q]) * dx1;
    if (z) z[q] = dims == 3 ? ((double)k + (double)static_cast<const R *>(p.off[2])[q]) * dx2 : 0.0;
    if (ux) ux[q] = (double)static_cast<const R *>(p.u[0])[q];
    if (uy) uy[q] = (double)static_cast<const R *>(p.u[1])[q];
    if (uz) uz[q] = (double)static_cast<const R *>(p.u[2])[q];
    if (w) w[q] = (double)static_cast<const R *>(p.w)[q];
    if (id) id[q] = p.id[q];
    if (alive) alive[q] = c >= 0 ? 1 : 0;
  }
}

template <class Rs, class Rd>
__global__ void k_convert(const Rs *__restrict__ s, Rd *__restrict__ d, int64_t n) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    d[q] = (Rd)s[q];
}

// ---- charge density at the nodes: rho += q w S(X-i) S(Y-j) S(Z-k) ----
template <class R>
__global__ void k_rho(int dims, int order, int n0, int n1, int n2, double q, Particles p,
                      const int64_t *__restrict__ d_count, double *rho) {
  const int64_t n = *d_count;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    const int c = p.cell[s];
    if (c < 0) continue;
    const int ci[3] = {c % n0, (c / n0) % n1, dims == 3 ? c / (n0 * n1) : 0};
    const int nn[3] = {n0, n1, n2};
    int base[3] = {0, 0, 0};
    double wt[3][3] = {{1, 0, 0}, {1, 0, 0}, {1, 0, 0}};
    int ns[3] = {1, 1, 1};
    for (int d = 0; d < dims; ++d) {
      const double f = (double)static_cast<const R *>(p.off[d])[s];
      if (order == 2) {
        const int h = f >= 0.5;
        const double dd = f - h;
        const double a = 0.5 - dd, b = 0.5 + dd;
        wt[d][0] = 0.5 * a * a;
        wt[d][1] = 0.75 - dd * dd;
        wt[d][2] = 0.5 * b * b;
        base[d] = ci[d] + h - 1;
        ns[d] = 3;
      } else {
        wt[d][0] = 1.0 - f;
        wt[d][1] = f;
        base[d] = ci[d];
        ns[d] = 2;
      }
    }
    const double qw = q * (double)static_cast<const R *>(p.w)[s];
    for (int kz = 0; kz < ns[2]; ++kz)
      for (int ky = 0; ky < ns[1]; ++ky)
        for (int kx = 0; kx < ns[0]; ++kx) {
          const int gi = wrapi(base[0] + kx, nn[0]);
          const int gj = wrapi(base[1] + ky, nn[1]);
          const int gk = dims == 3 ? wrapi(base[2] + kz, nn[2]) : 0;
          atomicAdd(rho + gi + (int64_t)n0 * (gj + (int64_t)n1 * gk), qw * wt[0][kx] * wt[1][ky] * wt[2][kz]);
        }
  }
}

template <class R>
__global__ void __launch_bounds__(256)
    k_field_diag(int dims, int n0, int n1, int n2, double rdx0, double rdx1, double rdx2, double rdt, const R *Ex,
                 const R *Ey, const R *Ez, const R *Bx, const R *By, const R *Bz, const R *Jx, const R *Jy,
                 const R *Jz, const double *rho, const double *rho_prev, double *out) {
  __shared__ double sh[32];
  double se = 0, sb = 0, sq = 0, gm = 0, cm = 0, nf = 0;
  // one x row per block and pass (no per-cell index division)
  const int64_t nrows = (int64_t)n1 * n2;
  for (int64_t r = blockIdx.x; r < nrows; r += gridDim.x) {
    const int j = (int)(r % n1), k = (int)(r / n1);
    const int64_t dy = j > 0 ? n0 : (int64_t)n0 - (int64_t)n0 * n1;  // to the y - 1 row, periodic
    const int64_t dz = k > 0 ? (int64_t)n0 * n1 : (int64_t)n0 * n1 - (int64_t)n0 * n1 * n2;
    for (int i = threadIdx.x; i < n0; i += blockDim.x) {
      const int64_t c = r * n0 + i;
      const double ex = Ex[c], ey = Ey[c], ez = Ez[c], bx = Bx[c], by = By[c], bz = Bz[c];
      se += ex * ex + ey * ey + ez * ez;
      sb += bx * bx + by * by + bz * bz;
      if (!isfinite(ex) || !isfinite(ey) || !isfinite(ez) || !isfinite(bx) || !isfinite(by) || !isfinite(bz)) nf += 1;
      const int64_t cxm = c - (i > 0 ? 1 : 1 - n0);
      const int64_t cym = c - dy;
      const int64_t czm = c - dz;
      double div = ((double)Ex[c] - (double)Ex[cxm]) * rdx0 + ((double)Ey[c] - (double)Ey[cym]) * rdx1;
      double dj = ((double)Jx[c] - (double)Jx[cxm]) * rdx0 + ((double)Jy[c] - (double)Jy[cym]) * rdx1;
      if (dims == 3) {
        div += ((double)Ez[c] - (double)Ez[czm]) * rdx2;
        dj += ((double)Jz[c] - (double)Jz[czm]) * rdx2;
      }
      sq += rho[c];
      gm = fmax(gm, fabs(div - rho[c]));
      if (rho_prev) cm = fmax(cm, fabs((rho[c] - rho_prev[c]) * rdt + dj));
    }
  }
  double v;
  v = block_sum(se, sh);
  if (threadIdx.x == 0) atomicAdd(out + 0, v);
  v = block_sum(sb, sh);
  if (threadIdx.x == 0) atomicAdd(out + 1, v);
  v = block_sum(sq, sh);
  if (threadIdx.x == 0) atomicAdd(out + 2, v);
  v = block_max(gm, sh);
  if (threadIdx.x == 0) atomic_max_nonneg(out + 3, v);
  v = block_max(cm, sh);
  if (threadIdx.x == 0) atomic_max_nonneg(out + 4, v);
  v = block_sum(nf, sh);
  if (threadIdx.x == 0) atomicAdd(out + 5, v);
}

// A thread's running sum of per-element terms computed in R.  FP64 runs add
// in FP64.  FP32 runs keep a compensated FP32 sum (Neumaier's variant of
// Kahan summation), which stays off the slow FP64 pipe and is exact to a few
// FP32 ulps of the summed magnitudes; block and grid sums are FP64.
template <class R> struct ThreadSum;
template <> struct ThreadSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct ThreadSum<float> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x;
    c += fabsf(s) >= fabsf(x) ? (s - t) + x : (x - t) + s;  // the rounding error of s + x, exactly
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// sum E^2, sum B^2 (squares in the storage precision)
template <class R>
__global__ void __launch_bounds__(256)
    k_field_energy(int64_t ncell, const R *Ex, const R *Ey, const R *Ez, const R *Bx, const R *By, const R *Bz,
                   double *out) {
  __shared__ double sh[32];
  ThreadSum<R> se, sb;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
    const R ex = Ex[c], ey = Ey[c], ez = Ez[c], bx = Bx[c], by = By[c], bz = Bz[c];
    se.add(ex * ex + ey * ey + ez * ez);
    sb.add(bx * bx + by * by + bz * bz);
  }
  double v = block_sum(se.value(), sh);
  if (threadIdx.x == 0) atomicAdd(out + 0, v);
  v = block_sum(sb.value(), sh);
  if (threadIdx.x == 0) atomicAdd(out + 1, v);
}

template <class R>
__global__ void __launch_bounds__(256)
    k_particle_diag(Particles p, const int64_t *__restrict__ d_count, double m, double *out) {
  __shared__ double sh[32];
  const int64_t n = *d_count;
  const int32_t *__restrict__ cell = p.cell;
  const R *__restrict__ u0 = static_cast<const R *>(p.u[0]);
  const R *__restrict__ u1 = static_cast<const R *>(p.u[1]);
  const R *__restrict__ u2p = static_cast<const R *>(p.u[2]);
  const R *__restrict__ w = static_cast<const R *>(p.w);
  ThreadSum<R> ek;
  int64_t cnt = 0, nf = 0;
  // four slots per thread and pass, every load issued before any is used
  // (a dead slot's momenta are read and dropped rather than skipped, so
  // the loads do not wait for the cell index)
  constexpr int kU = 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t s0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s0 < n; s0 += kU * stride) {
    int c[kU];
    R ux[kU], uy[kU], uz[kU], wq[kU];
#pragma unroll
    for (int k = 0; k < kU; ++k) {
      const int64_t s = s0 + k * stride;
      const bool in = s < n;
      c[k] = in ? cell[s] : -1;
      ux[k] = in ? u0[s] : R(0);
      uy[k] = in ? u1[s] : R(0);
      uz[k] = in ? u2p[s] : R(0);
      wq[k] = in ? w[s] : R(0);
    }
#pragma unroll
    for (int k = 0; k < kU; ++k) {
      if (c[k] < 0) continue;
      // per-particle terms in the storage precision
      const R u2 = ux[k] * ux[k] + uy[k] * uy[k] + uz[k] * uz[k];
      // gamma - 1 = u^2 / (sqrt(1 + u^2) + 1), free of cancellation
      ek.add(wq[k] * (u2 / (sqrt(R(1) + u2) + R(1))));
      ++cnt;
      nf += !isfinite(u2);
    }
  }
  double v = block_sum(ek.value(), sh);
  if (threadIdx.x == 0) atomicAdd(out + 0, m * v);
  v = block_sum((double)cnt, sh);
  if (threadIdx.x == 0) atomicAdd(out + 1, v);
  v = block_sum((double)nf, sh);
  if (threadIdx.x == 0) atomicAdd(out + 2, v);
}

// J and the escape counters cleared for a 3D step's pushes: one launch of the
// step's chain where two memsets took 7 us of a small run's step and broke the
// chain (75 x 50 x 43 smoothed plasma 193 -> 183 us per step).  Bound by the
// stores on large grids, as the memset was.
__global__ void __launch_bounds__(256)
    k_clear(uint4 *__restrict__ p, int64_t n16, uint32_t *__restrict__ rest, int nrest,
            unsigned long long *__restrict__ counters, int ncounters) {
  after_previous();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (int64_t i = t; i < n16; i += (int64_t)gridDim.x * blockDim.x) p[i] = make_uint4(0, 0, 0, 0);
  if (t < nrest) rest[t] = 0;
  if (t < ncounters) counters[t] = 0;
}

// A tape entry's copies: two blocks, each 16-byte aligned and a multiple of 4
// bytes long, in one launch of the step's chain.  Bound by memory.  Two
// asynchronous copies took 45 us an entry beside the reverse sweep, and broke
// the chain; this takes 27 (256 x 256 FP32 run: gradient 34.9 -> 33.1 ms).
struct CopyArgs {
  const uint4 *src[2];
  uint4 *dst[2];
  int64_t n16[2];
  int rest[2];  // 4-byte words past them
};
__global__ void __launch_bounds__(256) k_copy(const __grid_constant__ CopyArgs a) {
  after_previous();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = (int64_t)gridDim.x * blockDim.x;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const uint4 *__restrict__ src = a.src[b];
    uint4 *__restrict__ dst = a.dst[b];
    const int64_t n16 = a.n16[b];
    int64_t i = t;
    for (; i + 3 * n < n16; i += 4 * n) {
      uint4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = src[i + k * n];
#pragma unroll
      for (int k = 0; k < 4; ++k) dst[i + k * n] = v[k];
    }
    for (; i < n16; i += n) dst[i] = src[i];
    if (t < a.rest[b])
      reinterpret_cast<uint32_t *>(dst + n16)[t] = reinterpret_cast<const uint32_t *>(src + n16)[t];
  }
}

// All the smoothing passes along one axis at once: the taps of the passes
// convolved, out = w[0] in + sum_k w[k] (in[-k] + in[+k]), periodic, on `ncomp`
// fields back to back.  The passes of the axes commute, so a launch per axis
// does what a launch per pass, axis and field did (27 launches for J in 3D with
// two passes and compensation, 126 us on 75 x 50 x 43 FP32; three launches and
// 26 us now).  The taps come from the cache: every value is read once per tap.
constexpr int kSmoothRadius = 9;  // eight binomial passes and a compensating one
template <class R> struct SmoothArgs {
  const R *in;
  R *out;
  int n0, n1, n2, ncomp, axis, radius;
  R w[kSmoothRadius + 1];
};
template <class R> __global__ void __launch_bounds__(256) k_smooth_axis(const __grid_constant__ SmoothArgs<R> a) {
  after_previous();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n0) return;
  const int len = a.axis == 0 ? a.n0 : a.axis == 1 ? a.n1 : a.n2;
  const int64_t step = a.axis == 0 ? 1 : a.axis == 1 ? a.n0 : (int64_t)a.n0 * a.n1;
  for (int64_t kc = blockIdx.z; kc < (int64_t)a.n2 * a.ncomp; kc += gridDim.z) {
    for (int j = blockIdx.y * blockDim.y + threadIdx.y; j < a.n1; j += gridDim.y * blockDim.y) {
      const int64_t c = i + a.n0 * (j + a.n1 * kc);
      const int at = a.axis == 0 ? i : a.axis == 1 ? j : (int)(kc % a.n2);
      const R *line = a.in + (c - at * step);
      R v = a.w[0] * a.in[c];
      int lo = at, hi = at;
      for (int k = 1; k <= a.radius; ++k) {
        lo = lo > 0 ? lo - 1 : len - 1;
        hi = hi + 1 < len ? hi + 1 : 0;
        v += a.w[k] * (line[lo * step] + line[hi * step]);
      }
      a.out[c] = v;
    }
  }
}

template <class R>
static cudaError_t smooth_t(const Grid &g, R *f, int ncomp, R *tmp, int passes, int compensate, cudaStream_t st,
                            int *nlaunch, bool *in_tmp) {
  // the taps at 0 .. radius of the passes (1/4, 1/2, 1/4) and (compensate) of
  // (side, alpha, side), alpha = 1 + passes / 2, side = (1 - alpha) / 2
  double w[kSmoothRadius + 2] = {1.0};
  int radius = 0;
  const auto convolve = [&](double alpha) {
    const double side = 0.5 * (1.0 - alpha);
    double o[kSmoothRadius + 2] = {};
    for (int k = 0; k <= radius + 1; ++k)
      o[k] = alpha * w[k] + side * ((k > 0 ? w[k - 1] : w[1]) + (k <= radius ? w[k + 1] : 0.0));
    ++radius;
    for (int k = 0; k <= radius; ++k) w[k] = o[k];
  };
  for (int p = 0; p < passes; ++p) convolve(0.5);
  if (compensate) convolve(1.0 + 0.5 * passes);
  SmoothArgs<R> a;
  a.n0 = g.n[0];
  a.n1 = g.n[1];
  a.n2 = g.n[2];
  a.ncomp = ncomp;
  a.radius = radius;
  for (int k = 0; k <= kSmoothRadius; ++k) a.w[k] = (R)(k <= radius ? w[k] : 0.0);
  const dim3 block(64, 4, 1);
  const int64_t planes = (int64_t)g.n[2] * ncomp;
  const dim3 grid((a.n0 + 63) / 64, (a.n1 + 3) / 4 < 65535 ? (a.n1 + 3) / 4 : 65535, planes < 65535 ? planes : 65535);
  for (a.axis = 0; a.axis < g.dims; ++a.axis) {
    a.in = f;
    a.out = tmp;
    launch_next(k_smooth_axis<R>, grid, block, 0, st, a);
    R *t = f;
    f = tmp;
    tmp = t;
  }
  if (nlaunch) *nlaunch = g.dims;
  *in_tmp = g.dims % 2 == 1;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_smooth(const Grid &g, void *f, int ncomp, bool f64, void *tmp, int passes, int compensate,
                          cudaStream_t st, int *nlaunch, bool *in_tmp) {
  if (f64 || g.prec == 1)
    return smooth_t<double>(g, static_cast<double *>(f), ncomp, static_cast<double *>(tmp), passes, compensate, st,
                            nlaunch, in_tmp);
  return smooth_t<float>(g, static_cast<float *>(f), ncomp, static_cast<float *>(tmp), passes, compensate, st, nlaunch,
                         in_tmp);
}

template <class R> void yee_b_t(const Grid &g, void *const E[3], void *const B[3], double h, cudaStream_t st) {
  auto a = yee_args<R>(g, E, B, nullptr, h);
  if (yee_vec_ok<R>(g, a, false)) {
    dim3 grid, block;
    yee_vec_shape<R>(g, grid, block);
    launch_next(k_yee_b_vec<R>, grid, block, 0, st, a);
  } else {
    const int nb = grid_blocks(g.ncell, 256);
    launch_next(k_yee_b<R>, nb, 256, 0, st, a);
  }
}

template <class R>
void yee_e_t(const Grid &g, void *const E[3], void *const B[3], void *const J[3], double h, cudaStream_t st) {
  auto a = yee_args<R>(g, E, B, J, h);
  if (yee_vec_ok<R>(g, a, true)) {
    dim3 grid, block;
    yee_vec_shape<R>(g, grid, block);
    launch_next(k_yee_e_vec<R>, grid, block, 0, st, a);
  } else {
    const int nb = grid_blocks(g.ncell, 256);
    launch_next(k_yee_e<R>, nb, 256, 0, st, a);
  }
}

cudaError_t launch_copy(void *const dst[2], const void *const src[2], const size_t bytes[2], cudaStream_t st) {
  CopyArgs a;
  for (int b = 0; b < 2; ++b) {
    a.src[b] = static_cast<const uint4 *>(src[b]);
    a.dst[b] = static_cast<uint4 *>(dst[b]);
    a.n16[b] = (int64_t)(bytes[b] / 16);
    a.rest[b] = (int)(bytes[b] % 16 / 4);
    if ((reinterpret_cast<uintptr_t>(dst[b]) | reinterpret_cast<uintptr_t>(src[b])) % 16 || bytes[b] % 4)
      return cudaErrorInvalidValue;
  }
  launch_next(k_copy, grid_blocks((a.n16[0] + a.n16[1] + 3) / 4, 256), 256, 0, st, a);
  return cudaGetLastError();
}

cudaError_t launch_clear(void *mem, size_t bytes, unsigned long long *counters, int ncounters, cudaStream_t st) {
  const int64_t n16 = (int64_t)(bytes / 16);
  int nb = grid_blocks(n16 > ncounters ? n16 : ncounters, 256);
  launch_next(k_clear, nb, 256, 0, st, static_cast<uint4 *>(mem), n16,
              reinterpret_cast<uint32_t *>(static_cast<char *>(mem) + n16 * 16), (int)(bytes % 16 / 4), counters,
              ncounters);
  return cudaGetLastError();
}

cudaError_t launch_yee_b(const Grid &g, void *const E[3], void *const B[3], double h, cudaStream_t st) {
  if (g.prec == 1) yee_b_t<double>(g, E, B, h, st);
  else yee_b_t<float>(g, E, B, h, st);
  return cudaGetLastError();
}

cudaError_t launch_yee_e(const Grid &g, void *const E[3], void *const B[3], void *const J[3], double h,
                         cudaStream_t st) {
  if (g.prec == 1) yee_e_t<double>(g, E, B, J, h, st);
  else yee_e_t<float>(g, E, B, J, h, st);
  return cudaGetLastError();
}

template <class R>
static cudaError_t field_step2_t(const Grid &g, void *const E[3], void *const B[3], void *const J[3],
                                 void *const E2[3], void *const B2[3], void *const Jn[3], const LaserStep &ls,
                                 unsigned long long *counters, int ncounters, cudaStream_t st) {
  FieldStep2<R> a;
  a.n0 = g.n[0];
  a.n1 = g.n[1];
  a.absorb = g.absorb_lo || g.absorb_hi;
  // (the right wall's node needs the column before it: not the first of a strip)
  a.width = kStripW;
  while (a.absorb && a.n0 % a.width == 1) --a.width;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // long strips recompute less (rows + 3 rows are read), short ones give more
  // warps: the longest that make 64 warps per SM (2048 x 1024 FP32: 36 us, 47
  // with 16 warps per SM), down to one row (64 x 64 FP64: 6.2 us, 9.1 with
  // three).  An oblique wave is evaluated for eight rows at a time.
  const int64_t strips = (a.n0 + a.width - 1) / a.width;
  const int least = ls.oblique ? 7 : 1;
  a.rows = 31;
  while (a.rows > least && strips * ((a.n1 + a.rows - 1) / a.rows) < 64 * (int64_t)nsm) a.rows /= 2;
  a.rdx = (R)(1.0 / g.dx[0]);
  a.rdy = (R)(1.0 / g.dx[1]);
  a.h = (R)g.dt;
  for (int d = 0; d < 3; ++d) {
    a.E[d] = static_cast<const R *>(E[d]);
    a.B[d] = static_cast<const R *>(B[d]);
    a.J[d] = static_cast<const R *>(J[d]);
    a.E2[d] = static_cast<R *>(E2[d]);
    a.B2[d] = static_cast<R *>(B2[d]);
    a.Jn[d] = static_cast<R *>(Jn[d]);
  }
  a.kc = (g.dt - g.dx[0]) / (g.dt + g.dx[0]);
  a.ls = ls;
  a.counters = counters;
  a.ncounters = ncounters;
  a.strips = (unsigned)strips;
  launch_next(k_field_step2<R>, (unsigned)(strips * ((a.n1 + 2 * a.rows - 1) / (2 * a.rows))), 64, 0, st, a);
  return cudaGetLastError();
}

cudaError_t launch_field_step2(const Grid &g, void *const E[3], void *const B[3], void *const J[3], void *const E2[3],
                               void *const B2[3], void *const Jn[3], const LaserStep &ls,
                               unsigned long long *counters, int ncounters, cudaStream_t st) {
  if (g.dims != 2) return cudaErrorInvalidValue;
  if (g.prec == 1) return field_step2_t<double>(g, E, B, J, E2, B2, Jn, ls, counters, ncounters, st);
  return field_step2_t<float>(g, E, B, J, E2, B2, Jn, ls, counters, ncounters, st);
}

cudaError_t launch_mur_save(const Grid &g, void *const E[3], double *buf, cudaStream_t st) {
  const int nb = grid_blocks(8LL * g.n[1] * g.n[2], 256);
  if (g.prec == 1)
    launch_next(k_mur_save<double>, nb, 256, 0, st, g.n[0], g.n[1], g.n[2], static_cast<const double *>(E[1]),
                static_cast<const double *>(E[2]), buf);
  else
    launch_next(k_mur_save<float>, nb, 256, 0, st, g.n[0], g.n[1], g.n[2], static_cast<const float *>(E[1]),
                static_cast<const float *>(E[2]), buf);
  return cudaGetLastError();
}

double laser_waveform(const Laser &L, double tau) {
  if (tau <= 0.0 || tau >= L.duration) return 0.0;
  const double env = sin(3.14159265358979323846 * tau / L.duration);
  return env * env * sin(tau);
}

LaserStep laser_step(const Laser &L, const double *prof, double amplitude, const Grid &g, double t_old, double t_new) {
  LaserStep ls{};
  const double dx = g.dx[0];
  ls.pol = L.enabled ? L.pol : 0;
  ls.prof = prof;
  ls.amp[0] = amplitude * laser_waveform(L, t_old);
  ls.amp[1] = amplitude * laser_waveform(L, t_old - dx);
  ls.amp[2] = amplitude * laser_waveform(L, t_new);
  ls.amp[3] = amplitude * laser_waveform(L, t_new - dx);
  ls.oblique = L.enabled && L.angle != 0.0;
  if (ls.oblique) {
    ls.dims = g.dims;
    ls.cos_t = cos(L.angle);
    ls.sin_t = sin(L.angle);
    // E in the x-y plane: its y component is cos(angle) of the amplitude
    ls.a = amplitude * (L.pol == 1 ? ls.cos_t : 1.0);
    ls.y0 = L.angle > 0.0 ? 0.0 : g.n[1] * g.dx[1];  // the wall edge the tilted fronts reach first
    ls.yc = L.yc;
    ls.zc = L.zc;
    ls.inv_w2 = 1.0 / (L.waist * L.waist);
    ls.duration = L.duration;
    ls.t_old = t_old;
    ls.t_new = t_new;
    ls.dx = dx;
    ls.dy = g.dx[1];
    ls.dz = g.dx[2];
  }
  return ls;
}

cudaError_t launch_mur_apply(const Grid &g, void *const E[3], const double *buf, const LaserStep &ls,
                             cudaStream_t st) {
  const int nb = grid_blocks(2LL * g.n[1] * g.n[2], 256);
  if (g.prec == 1)
    launch_next(k_mur_apply<double>, nb, 256, 0, st, g.n[0], g.n[1], g.n[2], g.dx[0], g.dt,
                static_cast<double *>(E[1]), static_cast<double *>(E[2]), buf, ls);
  else
    launch_next(k_mur_apply<float>, nb, 256, 0, st, g.n[0], g.n[1], g.n[2], g.dx[0], g.dt,
                static_cast<float *>(E[1]), static_cast<float *>(E[2]), buf, ls);
  return cudaGetLastError();
}

cudaError_t launch_load(const Grid &g, const Particles &p, int64_t offset, int64_t n, const double *x,
                        const double *y, const double *z, const double *ux, const double *uy, const double *uz,
                        const double *w, const uint32_t *id, uint32_t id_base, unsigned long long *bad,
                        cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int nb = grid_blocks(n, 256);
  const int absorb = g.absorb_lo || g.absorb_hi;
  if (g.prec == 1)
    k_load<double><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.n[1], g.n[2], 1.0 / g.dx[0], 1.0 / g.dx[1], 1.0 / g.dx[2],
                                       absorb, p, offset, n, x, y, z, ux, uy, uz, w, id, id_base, bad);
  else
    k_load<float><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.n[1], g.n[2], 1.0 / g.dx[0], 1.0 / g.dx[1], 1.0 / g.dx[2],
                                      absorb, p, offset, n, x, y, z, ux, uy, uz, w, id, id_base, bad);
  return cudaGetLastError();
}

cudaError_t launch_check_particles(const Grid &g, const Particles &p, int64_t n, unsigned long long *bad,
                                  cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int nb = grid_blocks(n, 256);
  const int absorb = g.absorb_lo || g.absorb_hi;
  if (g.prec == 1)
    k_check_particles<double><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.ncell, absorb, p, n, bad);
  else
    k_check_particles<float><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.ncell, absorb, p, n, bad);
  return cudaGetLastError();
}

cudaError_t launch_unload(const Grid &g, const Particles &p, const int64_t *d_count, int64_t nmax, double *x,
                          double *y, double *z, double *ux, double *uy, double *uz, double *w, uint32_t *id,
                          int32_t *alive, cudaStream_t st) {
  const int nb = grid_blocks(nmax, 256);
  if (g.prec == 1)
    k_unload<double><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.n[1], g.dx[0], g.dx[1], g.dx[2], p, d_count, x, y, z, ux,
                                         uy, uz, w, id, alive);
  else
    k_unload<float><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.n[1], g.dx[0], g.dx[1], g.dx[2], p, d_count, x, y, z, ux,
                                        uy, uz, w, id, alive);
  return cudaGetLastError();
}

cudaError_t launch_field_to_f64(const Grid &g, const void *src, double *dst, cudaStream_t st) {
  const int nb = grid_blocks(g.ncell, 256);
  if (g.prec == 1)
    return cudaMemcpyAsync(dst, src, sizeof(double) * g.ncell, cudaMemcpyDeviceToDevice, st);
  k_convert<float, double><<<nb, 256, 0, st>>>(static_cast<const float *>(src), dst, g.ncell);
  return cudaGetLastError();
}

cudaError_t launch_field_from_f64(const Grid &g, const double *src, void *dst, cudaStream_t st) {
  const int nb = grid_blocks(g.ncell, 256);
  if (g.prec == 1)
    return cudaMemcpyAsync(dst, src, sizeof(double) * g.ncell, cudaMemcpyDeviceToDevice, st);
  k_convert<double, float><<<nb, 256, 0, st>>>(src, static_cast<float *>(dst), g.ncell);
  return cudaGetLastError();
}

cudaError_t launch_to_f64(int prec, const void *src, double *dst, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (prec == 1) return cudaMemcpyAsync(dst, src, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
  k_convert<float, double><<<grid_blocks(n, 256), 256, 0, st>>>(static_cast<const float *>(src), dst, n);
  return cudaGetLastError();
}

cudaError_t launch_from_f64(int prec, const double *src, void *dst, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (prec == 1) return cudaMemcpyAsync(dst, src, sizeof(double) * n, cudaMemcpyDeviceToDevice, st);
  k_convert<double, float><<<grid_blocks(n, 256), 256, 0, st>>>(src, static_cast<float *>(dst), n);
  return cudaGetLastError();
}

cudaError_t launch_rho(const Grid &g, const Particles &p, const int64_t *d_count, int64_t nmax, double q,
                       double *rho, cudaStream_t st) {
  const int nb = grid_blocks(nmax, 256);
  if (g.prec == 1)
    k_rho<double><<<nb, 256, 0, st>>>(g.dims, g.order, g.n[0], g.n[1], g.n[2], q, p, d_count, rho);
  else
    k_rho<float><<<nb, 256, 0, st>>>(g.dims, g.order, g.n[0], g.n[1], g.n[2], q, p, d_count, rho);
  return cudaGetLastError();
}

cudaError_t launch_field_diag(const Grid &g, void *const E[3], void *const B[3], void *const J[3],
                              const double *rho, const double *rho_prev, double *out, cudaStream_t st) {
  const int nb = grid_blocks(g.ncell, 256);
  const double r0 = 1.0 / g.dx[0], r1 = 1.0 / g.dx[1], r2 = 1.0 / g.dx[2], rdt = 1.0 / g.dt;
  if (g.prec == 1) {
    auto c = [](void *v) { return static_cast<const double *>(v); };
    k_field_diag<double><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.n[1], g.n[2], r0, r1, r2, rdt, c(E[0]), c(E[1]),
                                             c(E[2]), c(B[0]), c(B[1]), c(B[2]), c(J[0]), c(J[1]), c(J[2]), rho,
                                             rho_prev, out);
  } else {
    auto c = [](void *v) { return static_cast<const float *>(v); };
    k_field_diag<float><<<nb, 256, 0, st>>>(g.dims, g.n[0], g.n[1], g.n[2], r0, r1, r2, rdt, c(E[0]), c(E[1]),
                                            c(E[2]), c(B[0]), c(B[1]), c(B[2]), c(J[0]), c(J[1]), c(J[2]), rho,
                                            rho_prev, out);
  }
  return cudaGetLastError();
}

cudaError_t launch_field_energy(const Grid &g, void *const E[3], void *const B[3], double *out, cudaStream_t st) {
  const int nb = grid_blocks(g.ncell, 256);
  if (g.prec == 1) {
    auto c = [](void *v) { return static_cast<const double *>(v); };
    k_field_energy<double><<<nb, 256, 0, st>>>(g.ncell, c(E[0]), c(E[1]), c(E[2]), c(B[0]), c(B[1]), c(B[2]), out);
  } else {
    auto c = [](void *v) { return static_cast<const float *>(v); };
    k_field_energy<float><<<nb, 256, 0, st>>>(g.ncell, c(E[0]), c(E[1]), c(E[2]), c(B[0]), c(B[1]), c(B[2]), out);
  }
  return cudaGetLastError();
}

cudaError_t launch_particle_diag(const Grid &g, const Particles &p, const int64_t *d_count, int64_t nmax, double m,
                                 double *out, cudaStream_t st) {
  const int nb = grid_blocks(nmax, 256);
  if (g.prec == 1) k_particle_diag<double><<<nb, 256, 0, st>>>(p, d_count, m, out);
  else k_particle_diag<float><<<nb, 256, 0, st>>>(p, d_count, m, out);
  return cudaGetLastError();
}

}  // namespace pic
