// Fused per-tile particle kernel: field gather -> Boris push -> leap-frog
// move -> Esirkepov current deposit (§2 eqs. 1-4 of the paper, Boris per its
// ref [8], the charge-conserving deposit for the continuity requirement it
// states in §2).
//
// Cell tiles are 8x8x4 in 3D, 16x16 in 2D.  The sort keeps each tile's
// particles in one contiguous, 4-aligned slot range and cuts that range into
// work items of bounded size, which the resident thread blocks take in turn.
// For an item a block stages E and B of the tile plus guard cells in shared
// memory, pushes all its particles, and then deposits them by groups that
// share a nearest node (see k_push) into a J window in shared memory (fixed
// point in FP32 runs), which it adds to the global J.
//
// A particle that has drifted more than D = 1 cell outside its tile since the
// last sort, or whose cell (CIC) or nearest node (TSC) does in this move, is not
// handled here: its slot is appended to an escape list and k_push_escaped
// applies the same arithmetic on global memory afterwards.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "pic_device.cuh"

namespace pic {

namespace {

constexpr int kThreads = 256;

// i mod n for i within a few periods of [0, n) (window coordinates)
__device__ __forceinline__ int wrap_near(int i, int n) {
  while (i < 0) i += n;
  while (i >= n) i -= n;
  return i;
}
constexpr int32_t kEscFlag = 0x40000000;  // set in `cell` while a particle waits for the escape kernel

// Compile-time tile and window geometry.  E, B and J share one window: the
// nodes -O .. (last) around the tile that the gather of a particle up to D
// cells outside it reaches, and that its deposit reaches when its nearest
// node stays within D cells of the tile over the move (a particle that moves
// further takes the escape path).
template <int DIM, int ORDER> struct Geo {
  static constexpr int TX = DIM == 3 ? 8 : 16;
  static constexpr int TY = DIM == 3 ? 8 : 16;
  static constexpr int TZ = DIM == 3 ? 4 : 1;
  static constexpr int D = 1;  // drift allowance (cells)
  static constexpr int LOE = 1, HIE = ORDER == 2 ? 2 : 1;  // gather reach below / above the cell
  static constexpr int O = D + LOE;                        // window index of the tile's first node
  static constexpr int EX = TX + 2 * D + LOE + HIE;
  static constexpr int EY = TY + 2 * D + LOE + HIE;
  static constexpr int EZ = DIM == 3 ? TZ + 2 * D + LOE + HIE : 1;
  static constexpr int EN = EX * EY * EZ;
  static constexpr int JS = EN + 32;    // word-array stride of the fixed-point J window (32 scratch words)
  static constexpr int NS = ORDER + 1;  // gather stencil width, and that of a settled deposit
  static constexpr int NW = ORDER + 2;  // general deposit stencil width
  // Groups: the nearest node (TSC) or the cell (CIC) of a particle's old
  // position, -D .. T - 1 + D (+ 1 for nodes) on every axis.
  static constexpr int KX = TX + 2 * D + (ORDER == 2 ? 1 : 0);
  static constexpr int KY = TY + 2 * D + (ORDER == 2 ? 1 : 0);
  static constexpr int KZ = DIM == 3 ? TZ + 2 * D + (ORDER == 2 ? 1 : 0) : 1;
  static constexpr int KN = KX * KY * KZ;
  static constexpr int KT = KN + 7;  // and the particles whose support changes, by the axes that do (mask 1..7)
};

// Shared memory of k_push, and the most slots a work item may hold (CAP): a
// block keeps the deposit jobs of its whole item, so that the particles of
// one node meet whatever their slots.  FP32 3D items hold a full 8x8x4 tile
// of the 8-per-cell plasma with room to spare at two blocks per SM.
template <class R, int DIM, int ORDER> struct Lay {
  using G = Geo<DIM, ORDER>;
  static constexpr bool F32 = sizeof(R) == 4;
  static constexpr int CAP = F32 ? (DIM == 2 ? 1920 : ORDER == 1 ? 1216 : 2176) : (DIM == 3 ? 2432 : 1664);
  // per SM (FP32: 2D at four, with 64 registers, 10 % slower on the slab; 3D CIC at two 19 %)
  static constexpr int BLOCKS = F32 ? (ORDER == 1 || DIM == 2 ? 3 : 2) : (DIM == 3 ? 1 : 2);
  // a particle (offsets, momenta, weight), then its job (old and new offsets, 2D3V: vz, weight)
  static constexpr int NJ = DIM == 3 ? 7 : 6;
  // particles one thread sums at a time (3D: 6 beat 5, 7, 8, 12 and 16 by up
  // to 5 %, two-stream 15 %; 2D: 8 beat 6 by 2 %)
  static constexpr int TASK = DIM == 3 ? 6 : 8;
  static constexpr int MAXT = CAP / TASK + G::KN;
  static constexpr size_t align16(size_t b) { return (b + 15) / 16 * 16; }
  // E and B, then (once every particle is pushed) the J window
  static constexpr size_t kWin = align16(6 * G::EN * sizeof(R) > 24 * G::JS ? 6 * G::EN * sizeof(R) : 24 * G::JS);
  static constexpr size_t kJob = kWin;                                  // [NJ][CAP] R
  static constexpr size_t kTag = kJob + align16(NJ * CAP * sizeof(R));  // [CAP] u32
  static constexpr size_t kOrder = kTag + 4 * CAP;                      // [CAP] u16
  static constexpr size_t kCount = align16(kOrder + 2 * CAP);           // [KT] u32, then [KT + 1] u16 and the tasks
  static constexpr size_t kTask = kCount + 2 * (G::KT + 1);             // [MAXT] u16
  static constexpr size_t kEnd = kTask + 2 * MAXT > kCount + 4 * G::KT ? kTask + 2 * MAXT : kCount + 4 * G::KT;
  static_assert(G::KT < 1024 && CAP < 4096 && CAP % 32 == 0, "tag packing");
};

template <class R> struct PushArgs {
  int n[3];
  int ntile[2];
  FastDiv dn0, dn1;
  const R *E[3];
  const R *B[3];
  R *J[3];
  int32_t *cell;
  R *off[3];
  R *u[3];
  const R *w;
  float reach;                      // FP32: the largest of the factors dt / dx_a and (2D3V) 1, see WinAcc
  const int32_t *work_tile;         // work item -> tile
  const int64_t *work_pb;           // work item -> first slot
  const int32_t *work_n;            // work item -> slots
  const int32_t *nwork;             // work items
  int64_t slots;                    // slots of the species
  unsigned long long *next_item;    // items taken beyond the first of every block
  int32_t *esc_list;                // slots deferred to k_push_escaped
  unsigned long long *esc_count;
  unsigned long long *q_jobs;       // particles of this launch whose shape support changes
  R qmh;      // q dt / (2 m)
  R dtdx[3];  // dt / dx_a
  R jfac[3];  // -q dx_a / dt  (Esirkepov running-sum scale, times w)
  float pre[3];          // FP32: powers of two that even out the components of the window, see WinAcc
  float jhi[3], jlo[3];  // FP32: the factor of the window's J_a, and what its rounding left out
  R qz;       // q            (2D3V: Jz = q w vz S)
  int absorb;  // absorbing x walls: remove particles leaving [kWallLo, n0 - kWallHiMargin)
  Counters *ctr;
};

// True when a particle at cell index i0 with offset f has left the region
// allowed between absorbing x walls.
template <class R> __device__ __forceinline__ bool outside_walls(int absorb, int i0, R f, int n0) {
  if (!absorb) return false;
  const R X = (R)i0 + f;
  return X < (R)kWallLo || X >= (R)(n0 - kWallHiMargin);
}

// One value copied from global to shared memory asynchronously.
template <class R> __device__ __forceinline__ void copy_async(R *to, const R *from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from),
               "n"((int)sizeof(R))
               : "memory");
}

// Weighted sum of one field component over the gather stencil; the stencil
// offsets are compile-time (row stride SY, plane stride SZ).
template <class R, int NS, int DIM, int SY, int SZ>
__device__ __forceinline__ R gsum(const R *__restrict__ F, const R *wx, const R *wy, const R *wz) {
  R acc = R(0);
#pragma unroll
  for (int c = 0; c < (DIM == 3 ? NS : 1); ++c) {
    R accb = R(0);
#pragma unroll
    for (int b = 0; b < NS; ++b) {
      const R *row = F + c * SZ + b * SY;
      R ra = row[0] * wx[0];
#pragma unroll
      for (int a = 1; a < NS; ++a) ra += row[a] * wx[a];
      accb += ra * wy[b];
    }
    acc += DIM == 3 ? accb * wz[c] : accb;
  }
  return acc;
}

// Shared-memory J window.  FP32 runs accumulate in fixed point: FP32 shared
// atomics are compare-and-swap loops costing several shared-memory
// wavefronts each, integer shared atomics are single native operations, and
// integer sums are exact and independent of order.  The window holds J without
// its factor -q dx_a / dt (2D3V Jz: q), which the flush multiplies in, to more
// than FP32's precision (rounded to FP32 and multiplied into every particle's
// weight it left up to an ulp in J).  A contribution v becomes
// the integer X = rint(v * 2^K), K chosen per work item: each Esirkepov
// contribution of a particle is at most |w| |v_a| dt / dx_a (2D3V Jz:
// |w| |v_z|), so at most its q = |w| min(1, |vx| + |vy| + |vz|), with the
// velocity after the push, times the largest of those factors.  (A component of
// a smaller factor is held times a power of two that makes up for it, so that
// flat cells or a small dt cost no bits.)  2^K keeps what
// is added at a time, up to Lay::TASK particles of one node, below
// 2^kLimitLog2: at most Q = min(TASK max q, sum of q) over the item's jobs.
// (From the sum of q alone the quantum was up to 2^8 coarser and as large an
// error of J as all other roundings: rms 1.3e-7 instead of 7.8e-8 with 8 per
// cell, and 2.3e-6 instead of 9e-8 in the transverse components of beams of 27
// per cell.)  X is kept as two signed 32-bit words, X = hi * 2^16 + lo with
// |lo| <= 2^15, both found with FP32 FMAs and adds only (adding 1.5 * 2^(23 + s)
// rounds a float of magnitude below 2^(22 + s) to a multiple of 2^s held in the
// low mantissa bits), because float-to-64-bit conversions run on the slow FP64
// pipe.  With |X| < 2^37 per addition (the split holds to 2^38: a stored move of
// less than an ulp of its offset may be twice v dt) an item's hi sums stay below
// 2^30, and the lo sums cannot overflow for fewer than 65,536 contributions per
// node (an item holds at most Lay::CAP particles).  FP64 runs use plain double
// shared atomics, keeping FP64 rounding.
template <class R> struct WinAcc;
template <> struct WinAcc<float> {
  int *w;       // [3][2][jn]: per component lo words, then hi words
  int jn;       // word stride: the window's nodes, then 32 scratch words
  int dummy;    // this lane's scratch word (past the nodes)
  float scale;  // 2^K
  float unit;   // 2^-K
  static constexpr int kLimitLog2 = 37;
  static constexpr float kMagic = 12582912.0f;        // 1.5 * 2^23: ulp 1
  static constexpr float kMagicHi = 824633720832.0f;  // 1.5 * 2^39: ulp 2^16
  // Add the contribution p q (already in units of 2^-K): X = p q is split
  // into hi 2^16 + lo without the FP64 pipe.  The first FMA rounds X to a
  // multiple of 2^16 (|X| < 2^37, so the sum stays in [2^39, 2^40), where
  // the float spacing is 2^16) and its bit pattern minus the magic's is hi;
  // the second FMA gives X - hi 2^16 with one rounding, |.| <= 2^15, and a
  // round-to-nearest conversion gives the integer lo (one instruction where
  // adding and removing the 1.5 * 2^23 magic took two).
  __device__ __forceinline__ void add(int comp, int idx, float p, float q) const {
    const float y = fmaf(p, q, kMagicHi);
    const float r = y - kMagicHi;  // hi 2^16, exact
    const float lf = fmaf(p, q, -r);
    const int hi = __float_as_int(y) - __float_as_int(kMagicHi);
    const int lo = __float2int_rn(lf);  // round to nearest even, as the 2^23 magic would
    // Both words are added unconditionally: a branch around the pair (or a
    // predicate on it) cost more than the adds.  A zero contribution goes to
    // the lane's own scratch word instead of the node, so that it does not
    // collide with the other lanes' nodes in their banks (and an outer node
    // past the window's end, whose contributions are all zero, is not
    // touched).
    const int at = (hi | lo) ? idx : dummy;
    const unsigned s = (unsigned)__cvta_generic_to_shared(w + comp * 2 * jn + at);
    asm volatile("red.shared.add.s32 [%0], %1;\n\tred.shared.add.s32 [%2], %3;" ::"r"(s), "r"(lo),
                 "r"(s + 4u * (unsigned)jn), "r"(hi));
  }
  // The largest power of two (within 2^+-100) that keeps Q 2^K below 2^kLimitLog2.
  __device__ __forceinline__ void set_scale(float Q) {
    const int e2 = (int)(__float_as_uint(Q) >> 23) - 126;  // Q < 2^e2
    int K = Q > 0.f ? kLimitLog2 - e2 : 100;
    K = K > 100 ? 100 : (K < -100 ? -100 : K);
    scale = __int_as_float((127 + K) << 23);
    unit = __int_as_float((127 - K) << 23);
  }
  // The node's J: the sum times the component's factor jhi + jlo.
  __device__ __forceinline__ float get(int comp, int idx, float jhi, float jlo) const {
    const int *b = w + comp * 2 * jn + idx;
    const float hi = (float)b[jn];
    return fmaf(hi, 65536.0f * unit * jhi, fmaf(hi, 65536.0f * unit * jlo, (float)b[0] * (unit * jhi)));
  }
};
template <> struct WinAcc<double> {
  double *w;  // [3][jn], plain double sums (the FP64 path keeps FP64 rounding)
  int jn;
  int dummy;  // (unused)
  double scale;  // 1: contributions are passed unscaled
  double unit;
  __device__ __forceinline__ void add(int comp, int idx, double p, double q) const {
    const double x = p * q;
    if (x != 0.0) atomicAdd(w + comp * jn + idx, x);
  }
  __device__ __forceinline__ double get(int comp, int idx, float, float) const { return w[comp * jn + idx]; }
};

// Esirkepov deposit into the shared J window (compile-time strides).
// base: window index of the stencil's first node.  The last running sum of
// each axis is -DS[last] (the running sum over the whole stencil vanishes),
// so it is exactly zero for a particle that keeps its nearest node on that
// axis.  lx, ly, lz: some active lane of the warp uses the last stencil node
// of that axis (warp-uniform); otherwise every contribution on that outer
// shell is zero and is skipped with a uniform branch.
template <class R, int ORDER, int DIM, int SY, int SZ>
__device__ __forceinline__ void deposit_win(const WinAcc<R> &acc, int base, const DepositAxis<R, ORDER> &X,
                                            const DepositAxis<R, ORDER> &Y, const DepositAxis<R, ORDER> &Z, R cx,
                                            R cy, R cz, R qwvz, bool lx, bool ly, bool lz) {
  constexpr int NW = ORDER + 2;
  constexpr int M = NW - 1;
  R Px[M], Py[M], Pz[M];
  {
    R a = R(0), b = R(0), c = R(0);
#pragma unroll
    for (int k = 0; k < M - 1; ++k) {
      a += X.DS[k];
      b += Y.DS[k];
      c += Z.DS[k];
      Px[k] = cx * a;
      Py[k] = cy * b;
      Pz[k] = cz * c;
    }
    Px[M - 1] = -cx * X.DS[NW - 1];
    Py[M - 1] = -cy * Y.DS[NW - 1];
    Pz[M - 1] = -cz * Z.DS[NW - 1];
  }
  if (DIM == 3) {
    // Jx(i+1/2,j,k) += Px[i] (S0y S0z + DSy S0z/2 + S0y DSz/2 + DSy DSz/3), cyclic for y, z
    R hz[NW], tz[NW], hx[NW], tx[NW];
#pragma unroll
    for (int k = 0; k < NW; ++k) {
      hz[k] = Z.S0[k] + R(0.5) * Z.DS[k];
      tz[k] = R(0.5) * Z.S0[k] + Z.DS[k] * R(1.0 / 3.0);
      hx[k] = X.S0[k] + R(0.5) * X.DS[k];
      tx[k] = R(0.5) * X.S0[k] + X.DS[k] * R(1.0 / 3.0);
    }
#pragma unroll
    for (int c = 0; c < NW; ++c) {
      if (c == NW - 1 && !lz) continue;
#pragma unroll
      for (int b = 0; b < NW; ++b) {
        if (b == NW - 1 && !ly) continue;
        const R br = Y.S0[b] * hz[c] + Y.DS[b] * tz[c];
#pragma unroll
        for (int a = 0; a < M; ++a) {
          if (a == M - 1 && !lx) continue;
          acc.add(0, base + c * SZ + b * SY + a, Px[a], br);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < NW; ++c) {
      if (c == NW - 1 && !lz) continue;
#pragma unroll
      for (int a = 0; a < NW; ++a) {
        if (a == NW - 1 && !lx) continue;
        const R br = Z.S0[c] * hx[a] + Z.DS[c] * tx[a];
#pragma unroll
        for (int b = 0; b < M; ++b) {
          if (b == M - 1 && !ly) continue;
          acc.add(1, base + c * SZ + b * SY + a, Py[b], br);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < NW; ++b) {
      if (b == NW - 1 && !ly) continue;
      const R hy = Y.S0[b] + R(0.5) * Y.DS[b];
      const R ty = R(0.5) * Y.S0[b] + Y.DS[b] * R(1.0 / 3.0);
#pragma unroll
      for (int a = 0; a < NW; ++a) {
        if (a == NW - 1 && !lx) continue;
        const R br = X.S0[a] * hy + X.DS[a] * ty;
#pragma unroll
        for (int c = 0; c < M; ++c) {
          if (c == M - 1 && !lz) continue;
          acc.add(2, base + c * SZ + b * SY + a, Pz[c], br);
        }
      }
    }
  } else {
    // 2D3V: Jx = Px (S0y + DSy/2), Jy = Py (S0x + DSx/2),
    //       Jz = q w vz (S0x S0y + DSx S0y/2 + S0x DSy/2 + DSx DSy/3)
#pragma unroll
    for (int b = 0; b < NW; ++b) {
      if (b == NW - 1 && !ly) continue;
      const R hy = Y.S0[b] + R(0.5) * Y.DS[b];
      const R ty = R(0.5) * Y.S0[b] + Y.DS[b] * R(1.0 / 3.0);
#pragma unroll
      for (int a = 0; a < M; ++a) {
        if (a == M - 1 && !lx) continue;
        acc.add(0, base + b * SY + a, Px[a], hy);
      }
#pragma unroll
      for (int a = 0; a < NW; ++a) {
        if (a == NW - 1 && !lx) continue;
        acc.add(2, base + b * SY + a, qwvz, X.S0[a] * hy + X.DS[a] * ty);
      }
    }
#pragma unroll
    for (int a = 0; a < NW; ++a) {
      if (a == NW - 1 && !lx) continue;
      const R hx = X.S0[a] + R(0.5) * X.DS[a];
#pragma unroll
      for (int b = 0; b < M; ++b) {
        if (b == M - 1 && !ly) continue;
        acc.add(1, base + b * SY + a, Py[b], hx);
      }
    }
  }
}

// ---- settled deposit ----------------------------------------------------
// Most particles keep their shape support over a step: for TSC the nearest
// node does not change, for CIC the cell does not.  For them the Esirkepov
// stencil shrinks from ORDER + 2 to ORDER + 1 nodes per axis (3D TSC: 54
// contributions instead of up to 144).  The shape change DS = S1 - S0 is
// taken in the factored form of DepositAxis (TSC, offsets d0, d1 of the two
// positions from their common nearest node, D = d1 - d0, sg = d0 + d1:
//   DS = (D (sg - 1) / 2, -D sg, D (sg + 1) / 2);  CIC: DS = (-D, D)),
// which keeps FP32's relative precision however small the move, where the
// difference of the two shapes would lose it.  The factored values equal
// S1 - S0 in exact arithmetic, so the current still satisfies the discrete
// continuity equation with rho = sum q w S (to FP32 round-off of S).
template <class R, int ORDER> struct SettledAxis {
  static constexpr int NS = ORDER + 1;
  R S0[NS], DS[NS];
  // offsets of the two positions from their nearest node (TSC) or in the cell (CIC)
  __device__ __forceinline__ void set(R d0, R d1) {
    const R dl = d1 - d0;
    if (ORDER == 2) {
      const R sg = d0 + d1;
      tsc3<R>(d0, S0);
      const R hd = R(0.5) * dl;
      DS[0] = hd * (sg - R(1));
      DS[1] = -dl * sg;
      DS[2] = hd * (sg + R(1));
    } else {
      S0[0] = R(1) - d0;
      S0[1] = d0;
      DS[0] = -dl;
      DS[NS - 1] = dl;
    }
  }
};

// A running sum of contributions p q in registers.
// DoubleSum: one FMA (FP64 runs).
// PairSum: FP32 in 3D.  hi starts at WinAcc<float>::kMagicHi, so that every FMA
// rounds its sum to a multiple of 2^16 (|sum| < 2^38, see WinAcc); how far it
// moved is exact, and a second FMA gives what the contribution was short of
// that, at most 2^15, which lo sums.  lo keeps 2^-6 of a unit, and is rounded to
// a whole one when the window takes the sum: finer than the window, which rounds
// every contribution by itself.  Two registers, and four instructions for two
// sums in packed FP32.  (3D TSC takes its 54 sums in two passes over the tasks,
// Jx and Jy and then Jz, to stay within 128 registers.)  One FP32 value (one
// FMA) loses what cancels within a group, and J had 5 to 13 % more error (rms
// against the 64-bit current of the same moves, 48 x 40 x 32 cells with 1 to 32
// particles each).  256^3 plasma of 8 per cell, 20 steps: 200.5 ms with one FP32
// value, 209.1 with the pair, 214.5 with its four instructions unpacked.
// FixedSum: FP32 in 2D.  The two fixed-point words of WinAcc<float>::add, so that
// the sum of a given scale does not depend on the order of the particles at all;
// its stencil has 21 sums where 3D TSC has 54.
struct DoubleSum {
  double v;
  __device__ __forceinline__ void clear() { v = 0.0; }
  __device__ __forceinline__ void add(double p, double q) { v += p * q; }
};
struct PairSum {
  float hi, lo;
  __device__ __forceinline__ void clear() {
    hi = WinAcc<float>::kMagicHi;
    lo = 0.f;
  }
  __device__ __forceinline__ void add(float p, float q) {
    const float y = fmaf(p, q, hi);
    lo += fmaf(p, q, hi - y);
    hi = y;
  }
};
struct FixedSum {
  int hi, lo;
  __device__ __forceinline__ void clear() { hi = lo = 0; }
  __device__ __forceinline__ void add(float p, float q) {
    const float y = fmaf(p, q, WinAcc<float>::kMagicHi);
    const float z = fmaf(p, q, -(y - WinAcc<float>::kMagicHi)) + WinAcc<float>::kMagic;  // rounds to an integer
    hi += __float_as_int(y) - __float_as_int(WinAcc<float>::kMagicHi);
    lo += __float_as_int(z) - __float_as_int(WinAcc<float>::kMagic);
  }
};

// M sums with a common factor q.
template <int M, class S, class R> __device__ __forceinline__ void add_each(S *s, const R *p, R q) {
#pragma unroll
  for (int k = 0; k < M; ++k) s[k].add(p[k], q);
}
// Two PairSums in packed FP32: the same four operations on both at once.
template <> __device__ __forceinline__ void add_each<2, PairSum, float>(PairSum *s, const float *p, float q) {
  asm("{\n\t"
      ".reg .b64 p, q, h, l, y, d;\n\t"
      "mov.b64 p, {%4, %5};\n\t"
      "mov.b64 q, {%6, %6};\n\t"
      "mov.b64 h, {%0, %1};\n\t"
      "mov.b64 l, {%2, %3};\n\t"
      "fma.rn.f32x2 y, p, q, h;\n\t"
      "sub.rn.f32x2 d, h, y;\n\t"
      "fma.rn.f32x2 d, p, q, d;\n\t"
      "add.rn.f32x2 l, l, d;\n\t"
      "mov.b64 {%0, %1}, y;\n\t"
      "mov.b64 {%2, %3}, l;\n\t"
      "}"
      : "+f"(s[0].hi), "+f"(s[1].hi), "+f"(s[0].lo), "+f"(s[1].lo)
      : "f"(p[0]), "f"(p[1]), "f"(q));
}

// The settled contributions of the particles of one node, summed in
// registers: add() one particle, flush() the sums into the J window once per
// group.  Same brackets as deposit_win: Jx gets
// Px (S0y S0z + DSy S0z/2 + S0y DSz/2 + DSy DSz/3), cyclic; in 2D3V
// Jz = q w vz (S0x S0y + DSx S0y/2 + S0x DSy/2 + DSx DSy/3).  The running
// sums of DS along an axis end at -DS[last] (the whole sum vanishes).
// COMPS: the components summed (bit c: J_c); the others' sums take no registers.
template <class R, int DIM, int ORDER, int COMPS> struct GroupSum {
  static constexpr int NS = ORDER + 1, M = ORDER;
  static constexpr int NA = DIM == 3 ? M * NS * NS : M * NS;  // Jx, Jy sums
  static constexpr int NZ = DIM == 3 ? M * NS * NS : NS * NS;  // Jz sums
  static constexpr bool kX = COMPS & 1, kY = COMPS & 2, kZ = COMPS & 4;
  using S = typename std::conditional<sizeof(R) == 8, DoubleSum,
                                      typename std::conditional<DIM == 2, FixedSum, PairSum>::type>::type;
  S jx[NA], jy[NA], jz[NZ];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      if (kX) jx[i].clear();
      if (kY) jy[i].clear();
    }
#pragma unroll
    for (int i = 0; i < NZ; ++i)
      if (kZ) jz[i].clear();
  }
  __device__ __forceinline__ void add(const SettledAxis<R, ORDER> &X, const SettledAxis<R, ORDER> &Y,
                                      const SettledAxis<R, ORDER> &Z, R cx, R cy, R cz, R qwvz) {
    R Px[M], Py[M], Pz[M];
    {
      R ra = R(0), rb = R(0), rc = R(0);
#pragma unroll
      for (int k = 0; k < M - 1; ++k) {
        ra += X.DS[k];
        rb += Y.DS[k];
        Px[k] = cx * ra;
        Py[k] = cy * rb;
        if (DIM == 3) {
          rc += Z.DS[k];
          Pz[k] = cz * rc;
        }
      }
      Px[M - 1] = -cx * X.DS[NS - 1];
      Py[M - 1] = -cy * Y.DS[NS - 1];
      if (DIM == 3) Pz[M - 1] = -cz * Z.DS[NS - 1];
    }
    if constexpr (DIM == 3) {
      R hz[NS], tz[NS], hx[NS], tx[NS];
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        hz[k] = Z.S0[k] + R(0.5) * Z.DS[k];
        tz[k] = R(0.5) * Z.S0[k] + Z.DS[k] * R(1.0 / 3.0);
        hx[k] = X.S0[k] + R(0.5) * X.DS[k];
        tx[k] = R(0.5) * X.S0[k] + X.DS[k] * R(1.0 / 3.0);
      }
#pragma unroll
      for (int c = 0; c < (kX ? NS : 0); ++c)
#pragma unroll
        for (int b = 0; b < NS; ++b) {
          const R br = Y.S0[b] * hz[c] + Y.DS[b] * tz[c];
          add_each<M>(jx + (c * NS + b) * M, Px, br);
        }
#pragma unroll
      for (int c = 0; c < (kY ? NS : 0); ++c)
#pragma unroll
        for (int a = 0; a < NS; ++a) {
          const R br = Z.S0[c] * hx[a] + Z.DS[c] * tx[a];
          add_each<M>(jy + (c * NS + a) * M, Py, br);
        }
#pragma unroll
      for (int b = 0; b < (kZ ? NS : 0); ++b) {
        const R hy = Y.S0[b] + R(0.5) * Y.DS[b];
        const R ty = R(0.5) * Y.S0[b] + Y.DS[b] * R(1.0 / 3.0);
#pragma unroll
        for (int a = 0; a < NS; ++a) {
          const R br = X.S0[a] * hy + X.DS[a] * ty;
          add_each<M>(jz + (b * NS + a) * M, Pz, br);
        }
      }
    } else {
#pragma unroll
      for (int b = 0; b < NS; ++b) {
        const R hy = Y.S0[b] + R(0.5) * Y.DS[b];
        const R ty = R(0.5) * Y.S0[b] + Y.DS[b] * R(1.0 / 3.0);
#pragma unroll
        for (int a = 0; a < M; ++a) jx[b * M + a].add(Px[a], hy);
#pragma unroll
        for (int a = 0; a < NS; ++a) jz[b * NS + a].add(qwvz, X.S0[a] * hy + X.DS[a] * ty);
      }
#pragma unroll
      for (int a = 0; a < NS; ++a) {
        const R hx = X.S0[a] + R(0.5) * X.DS[a];
#pragma unroll
        for (int b = 0; b < M; ++b) jy[a * M + b].add(Py[b], hx);
      }
    }
  }
  // SY, SZ: the window's row and plane strides; the sink adds at a
  // compile-time node offset from the stencil's first node
  template <int SY, int SZ, class Sink> __device__ __forceinline__ void flush(const Sink &out) const {
    if constexpr (DIM == 3) {
#pragma unroll
      for (int c = 0; c < (kX ? NS : 0); ++c)
#pragma unroll
        for (int b = 0; b < NS; ++b)
#pragma unroll
          for (int a = 0; a < M; ++a) out.add(0, c * SZ + b * SY + a, jx[(c * NS + b) * M + a]);
#pragma unroll
      for (int c = 0; c < (kY ? NS : 0); ++c)
#pragma unroll
        for (int a = 0; a < NS; ++a)
#pragma unroll
          for (int b = 0; b < M; ++b) out.add(1, c * SZ + b * SY + a, jy[(c * NS + a) * M + b]);
#pragma unroll
      for (int b = 0; b < (kZ ? NS : 0); ++b)
#pragma unroll
        for (int a = 0; a < NS; ++a)
#pragma unroll
          for (int c = 0; c < M; ++c) out.add(2, c * SZ + b * SY + a, jz[(b * NS + a) * M + c]);
    } else {
#pragma unroll
      for (int b = 0; b < NS; ++b) {
#pragma unroll
        for (int a = 0; a < M; ++a) out.add(0, b * SY + a, jx[b * M + a]);
#pragma unroll
        for (int a = 0; a < NS; ++a) out.add(2, b * SY + a, jz[b * NS + a]);
      }
#pragma unroll
      for (int a = 0; a < NS; ++a)
#pragma unroll
        for (int b = 0; b < M; ++b) out.add(1, b * SY + a, jy[a * M + b]);
    }
  }
};

// Where a group's sums go.  FP32: the fixed-point pair of WinAcc<float>::add
// at one base register plus a compile-time offset; FP64: a double shared
// atomic (zero skipped).
template <class R, int JS> struct GroupSink;
template <int JS> struct GroupSink<float, JS> {
  unsigned sb;  // byte address of the Jx low word of the stencil's first node
  __device__ __forceinline__ void add(int comp, int off, FixedSum s) const { put(comp, off, s.hi, s.lo); }
  __device__ __forceinline__ void add(int comp, int off, PairSum s) const {
    put(comp, off, __float_as_int(s.hi) - __float_as_int(WinAcc<float>::kMagicHi), __float2int_rn(s.lo));
  }
  __device__ __forceinline__ void put(int comp, int off, int hi, int lo) const {
    const unsigned sa = sb + 8u * (unsigned)JS * (unsigned)comp + 4u * (unsigned)off;
    asm volatile("red.shared.add.s32 [%0], %1;\n\tred.shared.add.s32 [%2], %3;" ::"r"(sa), "r"(lo),
                 "r"(sa + 4u * (unsigned)JS), "r"(hi));
  }
};
template <int JS> struct GroupSink<double, JS> {
  double *w;  // Jx value of the stencil's first node (components JS doubles apart)
  __device__ __forceinline__ void add(int comp, int off, DoubleSum s) const {
    if (s.v != 0.0) atomicAdd(w + comp * JS + off, s.v);
  }
};

// A deposit task: up to TASK settled particles of one group, from position
// tk % 4096 of the job order, their sums added to the window.  scale: of Jx, Jy,
// Jz, and (2D3V) of q vz w.
template <class R, int DIM, int ORDER, int COMPS>
__device__ __forceinline__ void deposit_task(const WinAcc<R> &acc, const R *sJob, const uint16_t *sOrder,
                                             const uint32_t *sTag, unsigned tk, const R (&scale)[4]) {
  using G = Geo<DIM, ORDER>;
  using L = Lay<R, DIM, ORDER>;
  constexpr int CAP = L::CAP, SY = G::EX, SZ = G::EX * G::EY;
  int j = tk & 4095u;
  const int je = j + (int)(tk >> 12) + 1;
  int s = sOrder[j];
  const uint32_t group = sTag[s] & 1023u;
  const int kx = group % G::KX, ky = group / G::KX % G::KY, kz = DIM == 3 ? group / (G::KX * G::KY) : 0;
  // the stencil's first node: one below the nearest node (TSC), the cell's (CIC)
  constexpr int o = ORDER == 2 ? 0 : 1;
  const int jb = (kx + o) + (ky + o) * SY + (DIM == 3 ? (kz + o) * SZ : 0);
  GroupSum<R, DIM, ORDER, COMPS> g;
  g.clear();
  while (true) {
    SettledAxis<R, ORDER> X, Y, Z;
    X.set(sJob[s], sJob[DIM * CAP + s]);
    Y.set(sJob[CAP + s], sJob[(DIM + 1) * CAP + s]);
    const R w = sJob[(L::NJ - 1) * CAP + s];
    R qwvz = R(0);
    if (DIM == 3) Z.set(sJob[2 * CAP + s], sJob[5 * CAP + s]);
    else qwvz = scale[3] * w * sJob[4 * CAP + s];
    if (++j < je) s = sOrder[j];
    g.add(X, Y, Z, scale[0] * w, scale[1] * w, scale[2] * w, qwvz);
    if (j >= je) break;
  }
  GroupSink<R, sizeof(R) == 4 ? G::JS : G::EN> out;
  if constexpr (sizeof(R) == 4) out.sb = (unsigned)__cvta_generic_to_shared(acc.w) + 4u * (unsigned)jb;
  else out.w = acc.w + jb;
  g.template flush<SY, SZ>(out);
}

// A particle's tag, left by the push for the deposit: its group (10 bits),
// for a particle whose support changes the move of its nearest node (CIC: of
// its cell) as 1 + {-1, 0, 1} in 2 bits per axis, its rank within its sort
// key (12 bits), and kTagChange; or kTagIdle, or kTagEscape (kTagIdle among
// its bits).
constexpr uint32_t kTagChange = 1u << 30, kTagIdle = 1u << 31, kTagEscape = kTagIdle | kTagChange;

// How many deposit tasks a group of c particles makes: pieces of T, and one
// for the rest, counted by length class in 10-bit fields, the longest first
// (T = 6: one class per length; T = 8: 8, 6 or 7, 5, 4, 2 or 3, 1).  The
// threads of a warp take tasks of one class, so that their loops have the same
// length.
constexpr int kClasses = 6;
template <int T> __device__ __forceinline__ int task_class(unsigned len) {
  if (T == 6) return 6 - (int)len;
  return len >= 8 ? 0 : len >= 6 ? 1 : len >= 5 ? 2 : len >= 4 ? 3 : len >= 2 ? 4 : 5;
}
template <int T> __device__ __forceinline__ unsigned long long task_counts(unsigned c) {
  static_assert(T == 6 || T == 8, "classes");
  const unsigned full = c / T, rest = c % T;
  return (unsigned long long)full + (rest ? 1ull << (10 * task_class<T>(rest)) : 0ull);
}

// A moved offset x (at most one cell away under the Courant limit) brought
// back into [0, 1): the cell shift sh, and the offset.  A carry that rounds to
// 1 is clamped and counted.
template <class R> __device__ __forceinline__ R carry(R x, int &sh, unsigned &clamp);
template <> __device__ __forceinline__ float carry<float>(float x, int &sh, unsigned &clamp) {
  const float fl = floorf(x);
  sh = (int)fl;
  x -= fl;
  if (x >= 1.f) {
    x = below_one<float>();
    ++clamp;
  }
  return x;
}
template <> __device__ __forceinline__ double carry<double>(double x, int &sh, unsigned &clamp) {
  sh = (x >= 1.0) ? 1 : ((x < 0.0) ? -1 : 0);
  x -= (double)sh;
  if (x >= 1.0) {
    x = below_one<double>();
    ++clamp;
  }
  return x;
}

// The per-particle physics shared by the tile kernel and the escape kernel:
// given gathered E, B, advance u and move.
template <class R, int ORDER, int DIM>
__device__ __forceinline__ void push_move(const PushArgs<R> &a, R u[3], const R E[3], const R B[3], const R f[3],
                                          R fn[3], int s[3], R &ig, unsigned &clamp) {
  boris<R, DIM == 2>(a.qmh, E, B, u);
  ig = inv_gamma<R>(u);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    fn[d] = R(0);
    s[d] = 0;
  }
#pragma unroll
  for (int d = 0; d < DIM; ++d) fn[d] = carry<R>(f[d] + a.dtdx[d] * u[d] * ig, s[d], clamp);
}

// As many blocks as fit the GPU, each taking work items in turn.  For an item:
// its particles and the E, B window are staged by asynchronous copies; every
// particle is gathered, pushed, moved and written back, leaving its deposit
// job and tag in its place; the jobs are counting-sorted by nearest node
// (indices only); those whose support changes are deposited one by one on the
// general stencil, the settled ones a group at a time, summed in registers;
// the J window is added to global J while the next item's particles arrive.
//
// What bounds it: shared-memory wavefronts (72 % of the time at 128^3) and
// instruction issue (66 %), not HBM.  Depositing each particle by itself cost
// 54 contributions of seven instructions, two of them shared reductions of 3.2
// wavefronts; a group sum costs two packed instructions per contribution and the
// reductions once per group.  The gather's 162 shared loads per particle are
// the largest part left.  3D TSC FP32 thermal plasma at 8 per cell, 16.8M
// particles (ncu): 1.655 ms depositing particle by particle, 1.110 by groups,
// 1.030 with asynchronous staging, blocks that stay, and tasks of six, 1.010
// with the sort's item sizes, 1.069 with the sums kept exact (the group sums
// before were one FP32 value); 1884, 1626, 1520, 1520 and 1666 instructions per
// 32 particles.  Two particles per thread in
// packed FP32 (FFMA2) needed 16 % fewer instructions and the same time.
template <class R, int DIM, int ORDER, bool EC>
__global__ void __launch_bounds__(kThreads, Lay<R, DIM, ORDER>::BLOCKS) k_push(const PushArgs<R> a) {
  // (k_push_escaped, set up early, would crowd the SMs whose blocks end first:
  // foil 128 -> 142 ms, hot 2D plasma 3.5 -> 4.1)
  after_previous<false>();
  using G = Geo<DIM, ORDER>;
  using L = Lay<R, DIM, ORDER>;
  constexpr int NS = G::NS, CAP = L::CAP;
  constexpr int SY = G::EX, SZ = G::EX * G::EY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R *sF = reinterpret_cast<R *>(smem_raw);  // 6 * EN: Ex Ey Ez Bx By Bz, then the J window
  R *sJob = reinterpret_cast<R *>(smem_raw + L::kJob);
  uint32_t *sTag = reinterpret_cast<uint32_t *>(smem_raw + L::kTag);
  uint16_t *sOrder = reinterpret_cast<uint16_t *>(smem_raw + L::kOrder);
  uint32_t *sCount = reinterpret_cast<uint32_t *>(smem_raw + L::kCount);
  uint16_t *sStart = reinterpret_cast<uint16_t *>(smem_raw + L::kCount);  // over the counts, once read
  uint16_t *sTask = reinterpret_cast<uint16_t *>(smem_raw + L::kTask);
  __shared__ unsigned int s_clamp, s_absorbed, s_next;
  __shared__ float s_q;          // sum and (as bits) maximum of q, see WinAcc
  __shared__ unsigned int s_qmax;
  __shared__ unsigned int s_wsum[kThreads / 32];
  __shared__ unsigned long long s_wcls[kThreads / 32];
  __shared__ int64_t s_pb;  // the block's next item: first slot, slots, tile
  __shared__ int s_n, s_tile;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // The item's particles, copied into their slots' places in shared memory
  // (cell, offsets, momenta, weight: the arrays that their jobs will take),
  // 16 bytes per asynchronous copy: runs and items start and end on multiples
  // of four slots.
  const auto stage_particles = [&](int64_t pb, int n) {
    const auto copy = [&](void *to, const void *from, int bytes) {
      const unsigned d = (unsigned)__cvta_generic_to_shared(to);
      for (int i = tid * 16; i < bytes; i += kThreads * 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + i), "l"(static_cast<const char *>(from) + i)
                     : "memory");
    };
    if (!PIC_CHECK(n >= 0 && n <= CAP && n % 4 == 0 && pb % 4 == 0 && pb >= 0 && pb + n <= a.slots, a.ctr)) return;
    copy(sTag, a.cell + pb, n * (int)sizeof(int32_t));
#pragma unroll
    for (int d = 0; d < DIM; ++d) copy(sJob + d * CAP, a.off[d] + pb, n * (int)sizeof(R));
#pragma unroll
    for (int d = 0; d < 3; ++d) copy(sJob + (DIM + d) * CAP, a.u[d] + pb, n * (int)sizeof(R));
    copy(sJob + (L::NJ - 1) * CAP, a.w + pb, n * (int)sizeof(R));
  };

  const unsigned nwork = (unsigned)*a.nwork;
  if (blockIdx.x >= nwork) return;
  int t = a.work_tile[blockIdx.x];
  int64_t pb = a.work_pb[blockIdx.x];
  int n = a.work_n[blockIdx.x];
  stage_particles(pb, n);
  while (t >= 0) {
#ifdef PIC_CHECKED
    if (!PIC_CHECK(n >= 0 && n <= CAP && n % 4 == 0 && pb % 4 == 0 && pb >= 0 && pb + n <= a.slots, a.ctr)) n = 0;
#endif
    int t0[3];
    bool edge = false;  // the window crosses the grid's seam
    {
      const int tx = t % a.ntile[0];
      const int r = t / a.ntile[0];
      t0[0] = tx * G::TX;
      t0[1] = (r % a.ntile[1]) * G::TY;
      t0[2] = (r / a.ntile[1]) * G::TZ;
      constexpr int EE[3] = {G::EX, G::EY, G::EZ};
#pragma unroll
      for (int d = 0; d < DIM; ++d) edge = edge || t0[d] < G::O || t0[d] - G::O + EE[d] > a.n[d];
    }
    // ---- stage E, B of the tile + guard (periodic wrap of global indices), RL
    // threads per row ----
    {
      constexpr int RL = G::EX <= 16 ? 16 : 32;
      const int x = tid % RL;
      if (x < G::EX) {
        int gi = t0[0] - G::O + x;
        if (edge) gi = wrap_near(gi, a.n[0]);
        for (int r = tid / RL; r < G::EY * G::EZ; r += kThreads / RL) {
          const int z = DIM == 3 ? r / G::EY : 0, y = r - z * G::EY;
          int gj = t0[1] - G::O + y, gk = DIM == 3 ? t0[2] - G::O + z : 0;
          if (edge) {
            gj = wrap_near(gj, a.n[1]);
            if (DIM == 3) gk = wrap_near(gk, a.n[2]);
          }
          const int g = gi + a.n[0] * (gj + a.n[1] * gk);  // (cells stay below 2^30)
          const int q = x + r * G::EX;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            copy_async(sF + c * G::EN + q, a.E[c] + g);
            copy_async(sF + (3 + c) * G::EN + q, a.B[c] + g);
          }
        }
      }
    }
    for (int q = tid; q < G::KT; q += kThreads) sCount[q] = 0;
    if (tid == 0) {
      s_clamp = s_absorbed = s_next = 0;
      s_q = 0.f;
      s_qmax = 0;
    }
    unsigned long long taken = 0;
    if (tid == 0) taken = atomicAdd(a.next_item, 1ull);  // (its result is first needed after the push)
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // ---- gather, Boris, move, write back; leave a deposit job and its tag.
    // The slots are cell-sorted, so a warp's lanes sit in a few neighbouring
    // cells and mostly read the same field nodes (shared-memory broadcasts).
    unsigned my_clamp = 0, my_absorbed = 0;
    float my_q = 0.f, my_qmax = 0.f;
    for (int s = tid; s < n; s += kThreads) {
      const int c = (int)sTag[s];
      uint32_t tag = kTagIdle;
      // (a single pass, left early by particles that do not deposit)
      if (c >= 0 && PIC_CHECK(c / a.n[0] / a.n[1] < a.n[2], a.ctr)) do {
        const int64_t p = pb + s;
        // decode the cell and its position relative to the tile
        const uint32_t r0 = a.dn0.div((uint32_t)c);
        int ci[3];
        ci[0] = c - (int)r0 * a.n[0];
        if (DIM == 3) {
          const uint32_t r1 = a.dn1.div(r0);
          ci[1] = (int)r0 - (int)r1 * a.n[1];
          ci[2] = (int)r1;
        } else {
          ci[1] = (int)r0;
          ci[2] = 0;
        }
        int l[3] = {0, 0, 0};
        bool inw = true;
        constexpr int TT[3] = {G::TX, G::TY, G::TZ};
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
          int dl = ci[d] - t0[d];
          if (edge) {
            if (dl > TT[d] - 1 + G::D) dl -= a.n[d];
            if (dl < -G::D) dl += a.n[d];
          }
          l[d] = dl;
          inw = inw && (unsigned)(dl + G::D) < (unsigned)(TT[d] + 2 * G::D);
        }
        tag = kTagEscape;
        if (!inw) break;
        R f[3], u[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          f[d] = d < DIM ? sJob[d * CAP + s] : R(0);
          u[d] = sJob[(DIM + d) * CAP + s];
        }
        const R w = sJob[(L::NJ - 1) * CAP + s];
        // ---- gather (§2: g-weighted average of the grid fields) ----
        R fn[3], ig;
        int sh[3];
        unsigned clamp = 0;
        {
          GatherAxis<R, ORDER> gx, gy, gz;
          gx.set(f[0], EC);
          gy.set(f[1], EC);
          gz.set(f[2], EC);
#ifdef PIC_CHECKED
          {
            // every gather stencil inside the E/B window (checked builds)
            const GatherAxis<R, ORDER> *ga[3] = {&gx, &gy, &gz};
            constexpr int EW[3] = {G::EX, G::EY, G::EZ};
            bool ok = true;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
              const int lo = l[d] + (ga[d]->relp < ga[d]->reld ? ga[d]->relp : ga[d]->reld) + G::O;
              const int hi = l[d] + (ga[d]->relp > ga[d]->reld ? ga[d]->relp : ga[d]->reld) + G::O + NS - 1;
              ok = ok && lo >= 0 && hi < EW[d];
            }
            if (!PIC_CHECK(ok, a.ctr)) {
              tag = kTagIdle;
              break;  // leaves the particle as it was
            }
          }
#endif
          const int xp = l[0] + gx.relp + G::O, xd = l[0] + gx.reld + G::O;
          const int yp = (l[1] + gy.relp + G::O) * SY, yd = (l[1] + gy.reld + G::O) * SY;
          const int zp = DIM == 3 ? (l[2] + gz.relp + G::O) * SZ : 0;
          const int zd = DIM == 3 ? (l[2] + gz.reld + G::O) * SZ : 0;
          R E[3], B[3];
          E[0] = gsum<R, NS, DIM, SY, SZ>(sF + 0 * G::EN + xd + yp + zp, gx.wd, gy.wp, gz.wp);
          E[1] = gsum<R, NS, DIM, SY, SZ>(sF + 1 * G::EN + xp + yd + zp, gx.wp, gy.wd, gz.wp);
          E[2] = gsum<R, NS, DIM, SY, SZ>(sF + 2 * G::EN + xp + yp + zd, gx.wp, gy.wp, gz.wd);
          B[0] = gsum<R, NS, DIM, SY, SZ>(sF + 3 * G::EN + xp + yd + zd, gx.wp, gy.wd, gz.wd);
          B[1] = gsum<R, NS, DIM, SY, SZ>(sF + 4 * G::EN + xd + yp + zd, gx.wd, gy.wp, gz.wd);
          B[2] = gsum<R, NS, DIM, SY, SZ>(sF + 5 * G::EN + xd + yd + zp, gx.wd, gy.wd, gz.wp);
          // ---- Boris push (§2 eq. 3) and leap-frog move ----
          push_move<R, ORDER, DIM>(a, u, E, B, f, fn, sh, ig, clamp);
        }
        // offsets from the nearest node (TSC) or in the cell (CIC), before and
        // after, and how far that node or cell moved
        R d0[3], d1[3];
        int k[3] = {0, 0, 0}, key[3] = {0, 0, 0};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (d >= DIM) {
            d0[d] = d1[d] = R(0);
            continue;
          }
          const int h0 = ORDER == 2 && f[d] >= R(0.5), h1 = ORDER == 2 && fn[d] >= R(0.5);
          d0[d] = f[d] - R(h0);
          d1[d] = fn[d] - R(h1);
          k[d] = sh[d] + h1 - h0;
          key[d] = l[d] + h0 + G::D;
          constexpr int KK[3] = {G::KX, G::KY, G::KZ};
          inw = inw && (unsigned)(key[d] + k[d]) < (unsigned)KK[d];
        }
        if (!inw) break;
        tag = kTagIdle;
        my_clamp += clamp;  // (the escape kernel counts its own)

        // ---- the new state ----
        int nc = c + sh[0] + a.n[0] * (DIM == 3 ? sh[1] + a.n[1] * sh[2] : sh[1]);
        if (edge) {
          int i[3];
#pragma unroll
          for (int d = 0; d < DIM; ++d) {
            i[d] = ci[d] + sh[d];
            if (i[d] < 0) i[d] = a.n[d] - 1;
            if (i[d] >= a.n[d]) i[d] = 0;
          }
          nc = DIM == 3 ? i[0] + a.n[0] * (i[1] + a.n[1] * i[2]) : i[0] + a.n[0] * i[1];
        }
        if (outside_walls<R>(a.absorb, ci[0] + sh[0], fn[0], a.n[0])) {
          nc = -1;  // removed at an absorbing wall after depositing its move
          ++my_absorbed;
        }
        a.cell[p] = nc;
#pragma unroll
        for (int d = 0; d < DIM; ++d) a.off[d][p] = fn[d];
#pragma unroll
        for (int d = 0; d < 3; ++d) a.u[d][p] = u[d];

        // ---- the deposit job ----
        // A particle that keeps its place (and, in 2D3V, has vz = 0) or has no
        // weight deposits nothing (a cold target before the pulse reaches it).
        const R vz = u[2] * ig;
        const bool change = (k[0] | k[1] | k[2]) != 0;
        if (w == R(0) ||
            !(change || d0[0] != d1[0] || d0[1] != d1[1] || (DIM == 3 ? d0[2] != d1[2] : vz != R(0))))
          break;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
          sJob[d * CAP + s] = d0[d];
          sJob[(DIM + d) * CAP + s] = d1[d];
        }
        if (DIM == 2) sJob[4 * CAP + s] = vz;  // (the weight stays in its place)
        const uint32_t group = (uint32_t)(key[0] + G::KX * (key[1] + G::KY * key[2]));
        uint32_t sort_key = group;
        tag = group;
        if (change) {
          sort_key = G::KN - 1 + (k[0] != 0) + 2 * (k[1] != 0) + 4 * (k[2] != 0);
          tag |= (uint32_t)((k[0] + 1) << 10 | (k[1] + 1) << 12 | (k[2] + 1) << 14) | kTagChange;
        }
        tag |= atomicAdd(&sCount[sort_key], 1u) << 16;
        // |v| <= min(1, |vx| + |vy| + |vz|)
        if (sizeof(R) == 4) {
          const float q = fabsf((float)w) *
                          fminf(1.f, (fabsf((float)u[0]) + fabsf((float)u[1]) + fabsf((float)u[2])) * (float)ig);
          my_q += q;
          my_qmax = fmaxf(my_qmax, q);
        }
      } while (0);
      sTag[s] = tag;
    }
    if (sizeof(R) == 4) {
      for (int o = 16; o > 0; o >>= 1) my_q += __shfl_xor_sync(0xffffffffu, my_q, o);
      const unsigned qmax = __reduce_max_sync(0xffffffffu, __float_as_uint(my_qmax));
      if (lane == 0 && my_q > 0.f) {
        atomicAdd(&s_q, my_q);
        atomicMax(&s_qmax, qmax);
      }
    }
    if (my_clamp) atomicAdd(&s_clamp, my_clamp);
    if (my_absorbed) atomicAdd(&s_absorbed, my_absorbed);
    __syncthreads();
    // the next item, read meanwhile
    int t_next = -1, n_next = 0;
    int64_t pb_next = 0;
    if (tid == 0) {
      if (s_clamp) atomicAdd(&a.ctr->clamped, (unsigned long long)s_clamp);
      if (s_absorbed) atomicAdd(&a.ctr->absorbed, (unsigned long long)s_absorbed);
      const unsigned long long next = taken + gridDim.x;
      if (next < nwork) {
        t_next = a.work_tile[next];
        pb_next = a.work_pb[next];
        n_next = a.work_n[next];
      }
    }

    // ---- counting sort of the jobs: key starts, and the deposit tasks.  Each
    // thread takes KPT consecutive keys; one block scan carries the job count
    // and the task counts of every length class.
    constexpr int KPT = (G::KT + kThreads - 1) / kThreads;
    uint32_t cnt[KPT], sum = 0;
    unsigned long long cls = 0;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
      const int q = tid * KPT + i;
      cnt[i] = q < G::KT ? sCount[q] : 0u;
      sum += cnt[i];
      if (q < G::KN) cls += task_counts<L::TASK>(cnt[i]);
    }
    const uint32_t sum0 = sum;
    const unsigned long long cls0 = cls;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, sum, o);
      const unsigned long long x = __shfl_up_sync(0xffffffffu, cls, o);
      if (lane >= o) {
        sum += v;
        cls += x;
      }
    }
    if (lane == 31) {
      s_wsum[warp] = sum;
      s_wcls[warp] = cls;
    }
    // the J window replaces E and B
    for (int q = tid; q < (int)(L::kWin / 16); q += kThreads) reinterpret_cast<int4 *>(smem_raw)[q] = int4{0, 0, 0, 0};
    __syncthreads();
    // the warps' sums, scanned by the first lanes of every warp
    uint32_t wv = s_wsum[lane % (kThreads / 32)];
    unsigned long long wx = s_wcls[lane % (kThreads / 32)];
#pragma unroll
    for (int o = 1; o < kThreads / 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, wv, o);
      const unsigned long long x = __shfl_up_sync(0xffffffffu, wx, o);
      if (lane >= o) {
        wv += v;
        wx += x;
      }
    }
    const uint32_t njob = __shfl_sync(0xffffffffu, wv, kThreads / 32 - 1);
    const unsigned long long all = __shfl_sync(0xffffffffu, wx, kThreads / 32 - 1);
    const int below = warp > 0 ? warp - 1 : 0;
    const uint32_t vb = __shfl_sync(0xffffffffu, wv, below);
    const unsigned long long xb = __shfl_sync(0xffffffffu, wx, below);
    uint32_t at = sum - sum0 + (warp > 0 ? vb : 0u);
    const unsigned long long pos = cls - cls0 + (warp > 0 ? xb : 0ull);
    int ntask = 0;
    {
      int first[kClasses];  // this thread's next task of each class; a class follows the longer ones
#pragma unroll
      for (int q = 0; q < kClasses; ++q) {
        first[q] = ntask + (int)((pos >> (10 * q)) & 1023u);
        ntask += (int)((all >> (10 * q)) & 1023u);
      }
#pragma unroll
      for (int i = 0; i < KPT; ++i) {
        const int q = tid * KPT + i;
        if (q <= G::KT) sStart[q] = (uint16_t)at;
        if (q < G::KN) {
          unsigned from = at, left = cnt[i];
          for (; left >= L::TASK; left -= L::TASK, from += L::TASK)
            sTask[first[0]++] = (uint16_t)(from | (L::TASK - 1) << 12);
          if (left) {
            const int cl = task_class<L::TASK>(left);
            int where = 0;
#pragma unroll
            for (int z = 0; z < kClasses; ++z)
              if (z == cl) where = first[z]++;
            sTask[where] = (uint16_t)(from | (left - 1) << 12);
          }
        }
        at += cnt[i];
      }
    }
    if (tid == 0) {
      s_tile = t_next;
      s_pb = pb_next;
      s_n = n_next;
    }
    __syncthreads();
    // every thread takes part in every pass: a warp appends the particles that
    // are left to k_push_escaped (state untouched) with one atomic
    for (int s0 = 0; s0 < n; s0 += kThreads) {
      const int s = s0 + tid;
      const uint32_t tag = s < n ? sTag[s] : kTagIdle;
      const unsigned esc = __ballot_sync(0xffffffffu, tag == kTagEscape);
      if (esc) {
        unsigned long long slot = 0;
        if (lane == 0) slot = atomicAdd(a.esc_count, (unsigned long long)__popc(esc));
        slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(esc & ((1u << lane) - 1u));
        if (tag == kTagEscape && PIC_CHECK(slot < (unsigned long long)a.slots, a.ctr)) {
          a.cell[pb + s] |= kEscFlag;
          a.esc_list[slot] = (int32_t)(pb + s);
        }
      }
      if (tag & kTagIdle) continue;
      uint32_t sort_key = tag & 1023u;
      if (tag & kTagChange)
        sort_key = G::KN - 1 + (((tag >> 10) & 3u) != 1u) + 2 * (((tag >> 12) & 3u) != 1u) +
                   4 * (((tag >> 14) & 3u) != 1u);
      const uint32_t q = sStart[sort_key] + ((tag >> 16) & 4095u);
      if (!PIC_CHECK(q < (uint32_t)CAP, a.ctr)) continue;
      sOrder[q] = (uint16_t)s;
    }
    WinAcc<R> acc;
    acc.w = reinterpret_cast<decltype(acc.w)>(smem_raw);
    acc.jn = sizeof(R) == 4 ? G::JS : G::EN;
    acc.dummy = G::EN + lane;
    acc.scale = acc.unit = R(1);
    if constexpr (sizeof(R) == 4)  // 1.01: room for the FP32 rounding of the sum
      acc.set_scale(1.01f * a.reach * fminf(L::TASK * __uint_as_float(s_qmax), s_q));
    __syncthreads();

    // ---- deposit: warps take the next 32 particles whose support changes (the
    // longest work, in order of the axes that do), then the next 32 tasks,
    // longest first (kParts = 2: all of them for Jx and Jy, then again for Jz)
    constexpr int kParts = DIM == 3 && ORDER == 2 && L::F32 ? 2 : 1;
    const int nset = sStart[G::KN], nchg = (int)njob - nset, nchg32 = (nchg + 31) & ~31;
    const int ntask32 = (ntask + 31) & ~31;
    const int nunit = nchg32 + (kParts == 2 ? ntask32 : 0) + ntask;
    if (tid == 0 && nchg > 0) atomicAdd(a.q_jobs, (unsigned long long)nchg);
    // (FP32: the factors come in with the flush, and the scales are powers of two)
    const R jf0 = L::F32 ? acc.scale * a.pre[0] : a.jfac[0], jf1 = L::F32 ? acc.scale * a.pre[1] : a.jfac[1];
    const R jf2 = L::F32 ? acc.scale * a.pre[2] : a.jfac[2], jz = L::F32 ? jf2 : a.qz;  // jz: 2D3V
    for (;;) {
      unsigned base = 0;
      if (lane == 0) base = atomicAdd(&s_next, 32u);
      base = __shfl_sync(0xffffffffu, base, 0);
      if ((int)base >= nunit) break;
      const int unit = (int)base + lane;
      if ((int)base >= nchg32) {
        const bool second = kParts == 2 && (int)base >= nchg32 + ntask32;
        const int i = unit - nchg32 - (second ? ntask32 : 0);
        if (i >= ntask) continue;
        const R c[4] = {jf0, jf1, jf2, jz};
        if (kParts == 1) deposit_task<R, DIM, ORDER, 7>(acc, sJob, sOrder, sTag, sTask[i], c);
        else if (second) deposit_task<R, DIM, ORDER, 4>(acc, sJob, sOrder, sTag, sTask[i], c);
        else deposit_task<R, DIM, ORDER, 3>(acc, sJob, sOrder, sTag, sTask[i], c);
      } else {
        // (lanes past the last one add nothing, so that the whole warp votes below)
        bool have = unit < nchg;
        const int s = sOrder[nset + (have ? unit : (int)base)];
        const uint32_t tag = sTag[s];
        const int group = tag & 1023u;
        const int kx = group % G::KX, ky = group / G::KX % G::KY, kz = DIM == 3 ? group / (G::KX * G::KY) : 0;
        DepositAxis<R, ORDER> X, Y, Z;
        X.set_nodes(sJob[s], (int)((tag >> 10) & 3u) - 1, sJob[DIM * CAP + s]);
        Y.set_nodes(sJob[CAP + s], (int)((tag >> 12) & 3u) - 1, sJob[(DIM + 1) * CAP + s]);
        R w = sJob[(L::NJ - 1) * CAP + s];
        R qwvz = R(0);
        if (DIM == 3) {
          Z.set_nodes(sJob[2 * CAP + s], (int)((tag >> 14) & 3u) - 1, sJob[5 * CAP + s]);
        } else {
          Z.zero();
          qwvz = jz * w * sJob[4 * CAP + s];
        }
        const int bx = kx + 1 + X.rel, by = ky + 1 + Y.rel, bz = DIM == 3 ? kz + 1 + Z.rel : 0;
#ifdef PIC_CHECKED
        {
          // the nodes that receive a current inside the window (checked builds)
          const DepositAxis<R, ORDER> *da[3] = {&X, &Y, &Z};
          const int b0[3] = {bx, by, bz};
          constexpr int JW[3] = {G::EX, G::EY, G::EZ};
          bool ok = true;
#pragma unroll
          for (int d = 0; d < DIM; ++d) {
            const bool last = da[d]->S0[G::NW - 1] != R(0) || da[d]->DS[G::NW - 1] != R(0);
            ok = ok && b0[d] >= 0 && b0[d] + G::NW - 2 + (last ? 1 : 0) < JW[d];
          }
          if (!PIC_CHECK(ok, a.ctr)) have = false;
        }
#endif
        if (!have) w = qwvz = R(0);
        // does some lane of this warp use the last stencil node of an axis?
        const bool lx = __any_sync(0xffffffffu, X.S0[G::NW - 1] != R(0) || X.DS[G::NW - 1] != R(0));
        const bool ly = __any_sync(0xffffffffu, Y.S0[G::NW - 1] != R(0) || Y.DS[G::NW - 1] != R(0));
        const bool lz = DIM == 3 && __any_sync(0xffffffffu, Z.S0[G::NW - 1] != R(0) || Z.DS[G::NW - 1] != R(0));
        deposit_win<R, ORDER, DIM, SY, SZ>(acc, bx + by * SY + bz * SZ, X, Y, Z, jf0 * w, jf1 * w, jf2 * w, qwvz, lx, ly,
                                           lz);
      }
    }
    __syncthreads();

    // ---- the next item's particles start on their way (their places are free)
    t = s_tile;
    pb = s_pb;
    n = s_n;
    if (t >= 0) stage_particles(pb, n);

    // ---- flush the J window into global J (nothing moved: no current) ----
    if (njob > 0) {
    if (sizeof(R) == 4 && (a.n[0] & 3) == 0) {
      // FP32 with rows of a multiple of four cells: runs of four nodes along x
      // aligned in global memory, one vector reduction each (every element
      // added atomically); a run reaching past the window's x ends adds zeros
      // there.  A run never straddles the periodic seam.
      const int xs = t0[0] - G::O;               // the window's first node, global x (unwrapped)
      const int a0 = xs - (((xs % 4) + 4) & 3);  // the multiple of 4 at or below it
      constexpr int NG = (G::EX + 6) / 4;        // runs per window row (the last may start past it)
      for (int q = tid; q < NG * G::EY * G::EZ; q += kThreads) {
        const int m = q % NG, row = q / NG;
        const int y = row % G::EY, z = row / G::EY;
        const int wx0 = a0 + 4 * m - xs;  // window x of the run's first node
        if (wx0 >= G::EX) continue;
        const int gi = wrap_near(a0 + 4 * m, a.n[0]);
        const int gj = wrap_near(t0[1] - G::O + y, a.n[1]);
        const int gk = DIM == 3 ? wrap_near(t0[2] - G::O + z, a.n[2]) : 0;
        const int g = gi + a.n[0] * (gj + a.n[1] * gk);  // (cells stay below 2^30)
        const int wrow = z * SZ + y * SY;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int wx = wx0 + e;
            v[e] = (wx >= 0 && wx < G::EX) ? (float)acc.get(c, wrow + wx, a.jhi[c], a.jlo[c]) : 0.f;
          }
          if (v[0] != 0.f || v[1] != 0.f || v[2] != 0.f || v[3] != 0.f)
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a.J[c] + g), "f"(v[0]), "f"(v[1]),
                         "f"(v[2]), "f"(v[3])
                         : "memory");
        }
      }
    } else {
      for (int q = tid; q < G::EN; q += kThreads) {
        const int x = q % G::EX;
        const int y = (q / G::EX) % G::EY;
        const int z = q / SZ;
        const int gi = wrap_near(t0[0] - G::O + x, a.n[0]);
        const int gj = wrap_near(t0[1] - G::O + y, a.n[1]);
        const int gk = DIM == 3 ? wrap_near(t0[2] - G::O + z, a.n[2]) : 0;
        const int g = gi + a.n[0] * (gj + a.n[1] * gk);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const R v = acc.get(c, q, a.jhi[c], a.jlo[c]);
          if (v != R(0)) atomicAdd(a.J[c] + g, v);
        }
      }
    }
    }
    __syncthreads();  // the window is free again
  }
}

// Particles deferred by the tile kernel: the same gather / Boris / move /
// Esirkepov arithmetic, reading E, B from and adding J to global memory with
// periodic index wrapping.
template <class R, int DIM, int ORDER, bool EC>
__global__ void __launch_bounds__(kThreads) k_push_escaped(const PushArgs<R> a) {
  after_previous();
  constexpr int NS = ORDER + 1;
  constexpr int NW = ORDER + 2;
  const unsigned long long nesc = *a.esc_count;
  unsigned my_clamp = 0;
  for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < nesc;
       q += (unsigned long long)gridDim.x * blockDim.x) {
    const int64_t p = a.esc_list[q];
    if (!PIC_CHECK(p >= 0 && p < a.slots, a.ctr)) continue;
    const int c = a.cell[p] & ~kEscFlag;
    if (!PIC_CHECK(c >= 0 && c / a.n[0] / a.n[1] < a.n[2], a.ctr)) continue;
    int ci[3];
    ci[0] = c % a.n[0];
    ci[1] = (c / a.n[0]) % a.n[1];
    ci[2] = DIM == 3 ? c / (a.n[0] * a.n[1]) : 0;
    R f[3], u[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      f[d] = d < DIM ? a.off[d][p] : R(0);
      u[d] = a.u[d][p];
    }
    GatherAxis<R, ORDER> ga[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) ga[d].set(f[d], EC);
    const int64_t sy = a.n[0], sz = (int64_t)a.n[0] * a.n[1];
    auto fetch = [&](const R *F, const bool dual[3]) {
      R acc = R(0);
      for (int cz = 0; cz < (DIM == 3 ? NS : 1); ++cz) {
        const int kz = DIM == 3 ? wrapi(ci[2] + (dual[2] ? ga[2].reld : ga[2].relp) + cz, a.n[2]) : 0;
        const R wz = DIM == 3 ? (dual[2] ? ga[2].wd[cz] : ga[2].wp[cz]) : R(1);
        for (int by = 0; by < NS; ++by) {
          const int ky = wrapi(ci[1] + (dual[1] ? ga[1].reld : ga[1].relp) + by, a.n[1]);
          const R wy = dual[1] ? ga[1].wd[by] : ga[1].wp[by];
          for (int ax = 0; ax < NS; ++ax) {
            const int kx = wrapi(ci[0] + (dual[0] ? ga[0].reld : ga[0].relp) + ax, a.n[0]);
            const R wx = dual[0] ? ga[0].wd[ax] : ga[0].wp[ax];
            acc += F[kx + sy * ky + sz * kz] * (wx * wy * wz);
          }
        }
      }
      return acc;
    };
    const bool sE[3][3] = {{true, false, false}, {false, true, false}, {false, false, true}};
    const bool sB[3][3] = {{false, true, true}, {true, false, true}, {true, true, false}};
    R E[3], B[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      E[k] = fetch(a.E[k], sE[k]);
      B[k] = fetch(a.B[k], sB[k]);
    }
    R fn[3], ig;
    int s[3];
    push_move<R, ORDER, DIM>(a, u, E, B, f, fn, s, ig, my_clamp);
    DepositAxis<R, ORDER> da[3];
    da[0].set(f[0], s[0], fn[0]);
    da[1].set(f[1], s[1], fn[1]);
    if (DIM == 3) da[2].set(f[2], s[2], fn[2]);
    else da[2].zero();
    const R wq = a.w[p];
    // global Esirkepov with wrapped node indices
    R P[3][NW - 1];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      R run = R(0);
      for (int k = 0; k < NW - 2; ++k) {
        run += da[d].DS[k];
        P[d][k] = a.jfac[d] * wq * run;
      }
      P[d][NW - 2] = -a.jfac[d] * wq * da[d].DS[NW - 1];  // the full running sum vanishes
    }
    int gx[NW], gy[NW], gz[NW];
    for (int k = 0; k < NW; ++k) {
      gx[k] = wrapi(ci[0] + da[0].rel + k, a.n[0]);
      gy[k] = wrapi(ci[1] + da[1].rel + k, a.n[1]);
      gz[k] = DIM == 3 ? wrapi(ci[2] + da[2].rel + k, a.n[2]) : 0;
    }
    const DepositAxis<R, ORDER> &X = da[0], &Y = da[1], &Z = da[2];
    if (DIM == 3) {
      for (int cz = 0; cz < NW; ++cz)
        for (int by = 0; by < NW; ++by)
          for (int ax = 0; ax < NW; ++ax) {
            const int64_t g = gx[ax] + sy * gy[by] + sz * gz[cz];
            const R bx = Y.S0[by] * (Z.S0[cz] + R(0.5) * Z.DS[cz]) + Y.DS[by] * (R(0.5) * Z.S0[cz] + Z.DS[cz] * R(1.0 / 3.0));
            const R byy = Z.S0[cz] * (X.S0[ax] + R(0.5) * X.DS[ax]) + Z.DS[cz] * (R(0.5) * X.S0[ax] + X.DS[ax] * R(1.0 / 3.0));
            const R bz = X.S0[ax] * (Y.S0[by] + R(0.5) * Y.DS[by]) + X.DS[ax] * (R(0.5) * Y.S0[by] + Y.DS[by] * R(1.0 / 3.0));
            if (ax < NW - 1) atomicAdd(a.J[0] + g, P[0][ax] * bx);
            if (by < NW - 1) atomicAdd(a.J[1] + g, P[1][by] * byy);
            if (cz < NW - 1) atomicAdd(a.J[2] + g, P[2][cz] * bz);
          }
    } else {
      const R qwvz = a.qz * wq * u[2] * ig;
      for (int by = 0; by < NW; ++by)
        for (int ax = 0; ax < NW; ++ax) {
          const int64_t g = gx[ax] + sy * gy[by];
          const R hy = Y.S0[by] + R(0.5) * Y.DS[by];
          const R ty = R(0.5) * Y.S0[by] + Y.DS[by] * R(1.0 / 3.0);
          const R hx = X.S0[ax] + R(0.5) * X.DS[ax];
          if (ax < NW - 1) atomicAdd(a.J[0] + g, P[0][ax] * hy);
          if (by < NW - 1) atomicAdd(a.J[1] + g, P[1][by] * hx);
          atomicAdd(a.J[2] + g, qwvz * (X.S0[ax] * hy + X.DS[ax] * ty));
        }
    }
    if (outside_walls<R>(a.absorb, ci[0] + s[0], fn[0], a.n[0])) {
      a.cell[p] = -1;  // removed at an absorbing wall after depositing its move
      atomicAdd(&a.ctr->absorbed, 1ull);
      continue;
    }
    int nc[3] = {ci[0], ci[1], ci[2]};
#pragma unroll
    for (int d = 0; d < DIM; ++d) nc[d] = wrapi(ci[d] + s[d], a.n[d]);
    a.cell[p] = nc[0] + a.n[0] * (nc[1] + a.n[1] * nc[2]);
#pragma unroll
    for (int d = 0; d < DIM; ++d) a.off[d][p] = fn[d];
#pragma unroll
    for (int d = 0; d < 3; ++d) a.u[d][p] = u[d];
  }
  if (my_clamp) atomicAdd(&a.ctr->clamped, (unsigned long long)my_clamp);
  // escaped particle-steps are counted by the host-visible counter
  if (blockIdx.x == 0 && threadIdx.x == 0 && nesc) atomicAdd(&a.ctr->escaped, nesc);
}

template <class R, int DIM, int ORDER, bool EC>
cudaError_t launch_t(const Grid &g, void *const E[3], void *const B[3], void *const J[3], const Particles &p,
                     const WorkSplit &ws, int32_t *esc_list, unsigned long long *esc_count, double q, double m,
                     Counters *ctr, cudaStream_t st, int *nlaunch) {
  if (ws.plan.cand[0] > Lay<R, DIM, ORDER>::CAP || ws.nwork > 0x7fffffff) return cudaErrorInvalidValue;
  PushArgs<R> a;
  a.work_tile = ws.work_tile;
  a.work_pb = ws.work_pb;
  a.work_n = ws.work_n;
  a.nwork = ws.count;
  a.slots = ws.slots;
  a.next_item = esc_count + 2;
  a.reach = DIM == 2 ? 1.f : 0.f;
  for (int d = 0; d < 3; ++d) {
    a.n[d] = g.n[d];
    a.E[d] = static_cast<const R *>(E[d]);
    a.B[d] = static_cast<const R *>(B[d]);
    a.J[d] = static_cast<R *>(J[d]);
    a.off[d] = static_cast<R *>(p.off[d]);
    a.u[d] = static_cast<R *>(p.u[d]);
    a.dtdx[d] = (R)(g.dt / g.dx[d]);
    a.jfac[d] = (R)(-q * g.dx[d] / g.dt);
    if (d < DIM) a.reach = std::fmax(a.reach, (float)(g.dt / g.dx[d]) * 1.000001f);
  }
  for (int d = 0; d < 3; ++d) {
    const bool z2 = DIM == 2 && d == 2;
    // the power of two next below what J_d's factor dt / dx_d lacks to the largest (at least 1)
    const double lacks = a.reach / (z2 ? 1.0 : g.dt / g.dx[d]);
    a.pre[d] = (float)std::exp2(std::floor(std::log2(std::fmin(lacks, 16777216.0))));
    const double jwin = (z2 ? q : -q * g.dx[d] / g.dt) / a.pre[d];
    a.jhi[d] = (float)jwin;
    a.jlo[d] = (float)(jwin - (double)a.jhi[d]);
  }
  a.ntile[0] = g.ntile[0];
  a.ntile[1] = g.ntile[1];
  a.dn0 = make_fastdiv((uint32_t)g.n[0]);
  a.dn1 = make_fastdiv((uint32_t)g.n[1]);
  a.cell = p.cell;
  a.w = static_cast<const R *>(p.w);
  a.esc_list = esc_list;
  a.esc_count = esc_count;
  a.q_jobs = esc_count + 1;
  a.qmh = (R)(q * g.dt / (2.0 * m));
  a.qz = (R)q;
  a.absorb = g.absorb_lo || g.absorb_hi;
  a.ctr = ctr;
  constexpr size_t smem = Lay<R, DIM, ORDER>::kEnd;
  auto fn = k_push<R, DIM, ORDER, EC>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t nb = (int64_t)nsm * Lay<R, DIM, ORDER>::BLOCKS;  // as many blocks as fit: they take items in turn
  e = launch_next(fn, (unsigned)(ws.nwork < nb ? ws.nwork : nb), kThreads, smem, st, a);
  if (e != cudaSuccess) return e;
  e = launch_next(k_push_escaped<R, DIM, ORDER, EC>, nsm, kThreads, 0, st, a);
  if (e != cudaSuccess) return e;
  if (nlaunch) *nlaunch = 2;
  return cudaGetLastError();
}

// Charge density at the nodes for the diagnostics, rho += q w S(X-i)S(Y-j)S(Z-k),
// one block per tile like k_push, particles taken in the same lane-spread
// order (a warp's lanes about one cell apart, so that their atomics hit
// different nodes).  The block's window sums are exact fixed point, scaled
// from a bound on the tile's charge (|rho_node| <= sum |q w|), so the window
// does not depend on the order of the additions; each node then receives
// one FP64 add per tile that reaches it.  Particles more than one cell
// outside their tile add to the global array directly.
//  FP32 runs: weights and products in FP32 (their positions carry FP32
//   rounding anyway), the tile's bound scaled to 2^37 and each product split
//   into int32 words hi 2^16 + lo by FP32 FMAs, as in the push's current
//   window; each particle's contributions sum exactly to its charge (the
//   last node takes the remainder), so the total charge is conserved; a
//   tile of more than kMaxWindowSlots particles is flushed in pieces so that
//   the lo sums cannot overflow.
//  FP64 runs: weights in FP64, the bound scaled to 2^61, one 64-bit word per
//   node.
template <class R, int DIM, int ORDER>
__global__ void __launch_bounds__(kThreads)
    k_rho_tile(int n0, int n1, int n2, int ntile0, int ntile1, FastDiv dn0, FastDiv dn1, const int32_t *__restrict__ cell,
               const R *__restrict__ off0, const R *__restrict__ off1, const R *__restrict__ off2,
               const R *__restrict__ w, const int64_t *__restrict__ tile_start, double q, double *rho,
               Counters *ctr) {
  using G = Geo<DIM, ORDER>;
  constexpr int NS = ORDER + 1;
  constexpr int RX = G::EX, RY = G::EY, RZ = G::EZ;  // window: cell-1 .. cell+2 around the tile (+ drift)
  constexpr int RN = RX * RY * RZ;
  constexpr bool kF32 = sizeof(R) == 4;
  __shared__ unsigned long long win[RN];  // FP32: int32 lo words [0, RN), hi words [RN, 2 RN)
  int *wlo = reinterpret_cast<int *>(win);
  __shared__ double s_sum;
  const int t = blockIdx.x;
  const int64_t pb = tile_start[t], pe = tile_start[t + 1];
  if (pb >= pe) return;
  const int tid = threadIdx.x;
  int t0[3];
  t0[0] = (t % ntile0) * G::TX;
  t0[1] = ((t / ntile0) % ntile1) * G::TY;
  t0[2] = (t / ntile0 / ntile1) * G::TZ;
  if (tid == 0) s_sum = 0.0;
  __syncthreads();
  {
    R part = R(0);
    for (int64_t p = pb + tid; p < pe; p += kThreads)
      if (cell[p] >= 0) part += fabs(w[p]);
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0 && part > R(0)) atomicAdd(&s_sum, (double)part);
  }
  __syncthreads();
  // 1.01: room for the rounding of the sum above
  const double Q = fabs(q) * s_sum * 1.01;
  int e2 = 0;
  if (Q > 0.0) frexp(Q, &e2);  // Q < 2^e2
  int K = Q > 0.0 ? (kF32 ? WinAcc<float>::kLimitLog2 : 61) - e2 : 0;
  K = K > 100 ? 100 : (K < -100 ? -100 : K);
  const double scale = ldexp(1.0, K);
  const R *offs[3] = {off0, off1, off2};
  const int nn[3] = {n0, n1, n2};
  constexpr int TT[3] = {G::TX, G::TY, G::TZ};
  const int lane = tid & 31, warp = tid >> 5;
  const int e = 8 * lane + ((warp + (lane >> 2)) & 7);  // lane-spread slot of a 256-slot chunk
  for (int64_t s0 = pb; s0 < pe; s0 += kMaxWindowSlots) {
    const int64_t se = pe - s0 < kMaxWindowSlots ? pe : s0 + kMaxWindowSlots;
    for (int i = tid; i < (kF32 ? 2 * RN : RN); i += kThreads) {
      if (kF32) wlo[i] = 0;
      else win[i] = 0ull;
    }
    __syncthreads();
    for (int64_t c0 = s0; c0 < se; c0 += kThreads) {
      const int64_t p = c0 + e;
      if (p >= se) continue;
      const int c = cell[p];
      if (c < 0) continue;
      const uint32_t r0 = dn0.div((uint32_t)c);
      const int ci[3] = {c - (int)r0 * n0, DIM == 3 ? (int)(r0 - dn1.div(r0) * n1) : (int)r0,
                         DIM == 3 ? (int)dn1.div(r0) : 0};
      int l[3] = {0, 0, 0};
      bool inw = true;
      int base[3] = {0, 0, 0};
      R wt[3][NS];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (d >= DIM) {
          wt[d][0] = R(1);
          for (int k = 1; k < NS; ++k) wt[d][k] = R(0);
          continue;
        }
        int dl = ci[d] - t0[d];
        if (dl > TT[d] - 1 + G::D) dl -= nn[d];
        if (dl < -G::D) dl += nn[d];
        l[d] = dl;
        inw = inw && dl >= -G::D && dl <= TT[d] - 1 + G::D;
        const R f = offs[d][p];
        if (ORDER == 2) {
          const int h = f >= R(0.5);
          const R dd = f - R(h), a = R(0.5) - dd, b = R(0.5) + dd;
          wt[d][0] = R(0.5) * a * a;
          wt[d][1] = R(0.75) - dd * dd;
          wt[d][NS - 1] = R(0.5) * b * b;
          base[d] = h - 1;
        } else {
          wt[d][0] = R(1) - f;
          wt[d][NS - 1] = f;
          base[d] = 0;
        }
      }
      // q w S_x, in window units (2^K) for particles in the window
      const R qw = inw ? (R)(q * scale) * w[p] : (R)q * w[p];
      R qwx[NS];
#pragma unroll
      for (int kx = 0; kx < NS; ++kx) qwx[kx] = qw * wt[0][kx];
      // FP32 runs: the particle's last node takes its whole charge minus what
      // the other nodes received, so that its integer contributions sum to
      // the integer q w 2^K exactly (and a particle outside the window adds
      // q w minus the other FP64 products): the FP32 weights need not sum to
      // one exactly for the total charge to be conserved.
      int hi_t = 0, lo_t = 0;
      double v_t = 0.0;
      if (kF32) {
        if (inw) {
          const float y = qw + WinAcc<float>::kMagicHi;  // |q w 2^K| < 2^37: hi 2^16 + lo as below
          hi_t = __float_as_int(y) - __float_as_int(WinAcc<float>::kMagicHi);
          lo_t = __float_as_int((qw - (y - WinAcc<float>::kMagicHi)) + WinAcc<float>::kMagic) -
                 __float_as_int(WinAcc<float>::kMagic);
        } else {
          v_t = (double)qw;
        }
      }
#pragma unroll
      for (int kz = 0; kz < (DIM == 3 ? NS : 1); ++kz)
#pragma unroll
        for (int ky = 0; ky < NS; ++ky) {
          const R wyz = wt[1][ky] * wt[2][kz];
#pragma unroll
          for (int kx = 0; kx < NS; ++kx) {
            const bool last = kF32 && kx == NS - 1 && ky == NS - 1 && kz == (DIM == 3 ? NS - 1 : 0);
            if (inw) {
              const int ix = l[0] + base[0] + kx + G::D + G::LOE;
              const int iy = l[1] + base[1] + ky + G::D + G::LOE;
              const int iz = DIM == 3 ? l[2] + base[2] + kz + G::D + G::LOE : 0;
              if (!PIC_CHECK(ix >= 0 && ix < RX && iy >= 0 && iy < RY && iz >= 0 && iz < RZ, ctr)) continue;
              const int at = ix + RX * (iy + RY * iz);
              if constexpr (kF32) {
                // X = qwx wyz 2^K < 2^37 as hi 2^16 + lo, the push's split
                int hi, lo;
                if (last) {
                  hi = hi_t;
                  lo = lo_t;
                  const int carry = (lo + 32768) >> 16;  // back to |lo| <= 2^15
                  hi += carry;
                  lo -= carry * 65536;
                } else {
                  const float y = fmaf(qwx[kx], wyz, WinAcc<float>::kMagicHi);
                  const float r = y - WinAcc<float>::kMagicHi;
                  const float lf = fmaf(qwx[kx], wyz, -r);
                  hi = __float_as_int(y) - __float_as_int(WinAcc<float>::kMagicHi);
                  lo = __float_as_int(lf + WinAcc<float>::kMagic) - __float_as_int(WinAcc<float>::kMagic);
                  hi_t -= hi;
                  lo_t -= lo;
                }
                atomicAdd(wlo + at, lo);
                atomicAdd(wlo + RN + at, hi);
              } else {
                atomicAdd(&win[at], (unsigned long long)__double2ll_rn(qwx[kx] * wyz));
              }
            } else {
              double v = (double)qwx[kx] * (double)wyz;
              if (last) v = v_t;
              else v_t -= v;
              const int gi = wrapi(ci[0] + base[0] + kx, n0), gj = wrapi(ci[1] + base[1] + ky, n1);
              const int gk = DIM == 3 ? wrapi(ci[2] + base[2] + kz, n2) : 0;
              atomicAdd(rho + gi + (int64_t)n0 * (gj + (int64_t)n1 * gk), v);
            }
          }
        }
    }
    __syncthreads();
    for (int i = tid; i < RN; i += kThreads) {
      const long long X = kF32 ? (long long)wlo[RN + i] * 65536 + wlo[i] : (long long)win[i];
      if (X == 0) continue;
      const int x = i % RX, y = (i / RX) % RY, z = i / (RX * RY);
      const int gi = wrap_near(t0[0] - G::D - G::LOE + x, n0);
      const int gj = wrap_near(t0[1] - G::D - G::LOE + y, n1);
      const int gk = DIM == 3 ? wrap_near(t0[2] - G::D - G::LOE + z, n2) : 0;
      atomicAdd(rho + gi + (int64_t)n0 * (gj + (int64_t)n1 * gk), (double)X / scale);
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_rho_tiled(const Grid &g, const Particles &p, const int64_t *tile_start, double q, double *rho,
                             Counters *ctr, cudaStream_t st) {
  if (g.ntiles > 0x7fffffff) return cudaErrorInvalidValue;
  const FastDiv d0 = make_fastdiv((uint32_t)g.n[0]), d1 = make_fastdiv((uint32_t)g.n[1]);
  const unsigned nb = (unsigned)g.ntiles;
#define PIC_RHO_CASE(K, R, D, O)                                                                                 \
  case K:                                                                                                        \
    k_rho_tile<R, D, O><<<nb, kThreads, 0, st>>>(g.n[0], g.n[1], g.n[2], g.ntile[0], g.ntile[1], d0, d1, p.cell, \
                                                  static_cast<const R *>(p.off[0]), static_cast<const R *>(p.off[1]), \
                                                  static_cast<const R *>(p.off[2]), static_cast<const R *>(p.w),  \
                                                  tile_start, q, rho, ctr);                                      \
    break;
  switch ((g.prec == 1 ? 100 : 0) + g.dims * 10 + g.order) {
    PIC_RHO_CASE(21, float, 2, 1)
    PIC_RHO_CASE(22, float, 2, 2)
    PIC_RHO_CASE(31, float, 3, 1)
    PIC_RHO_CASE(32, float, 3, 2)
    PIC_RHO_CASE(121, double, 2, 1)
    PIC_RHO_CASE(122, double, 2, 2)
    PIC_RHO_CASE(131, double, 3, 1)
    PIC_RHO_CASE(132, double, 3, 2)
    default: return cudaErrorInvalidValue;
  }
#undef PIC_RHO_CASE
  return cudaGetLastError();
}

// Tile shape compiled into the push kernel for a given dimensionality.
void push_tile_shape(int dims, int tile[3]) {
  tile[0] = dims == 3 ? Geo<3, 2>::TX : Geo<2, 2>::TX;
  tile[1] = dims == 3 ? Geo<3, 2>::TY : Geo<2, 2>::TY;
  tile[2] = dims == 3 ? Geo<3, 2>::TZ : 1;
}

// The layout of the kernel that serves a grid.
template <class F> static auto with_layout(const Grid &g, F f) {
  switch ((g.prec == 1 ? 100 : 0) + g.dims * 10 + g.order) {
    case 21: return f(Lay<float, 2, 1>{});
    case 22: return f(Lay<float, 2, 2>{});
    case 31: return f(Lay<float, 3, 1>{});
    case 121: return f(Lay<double, 2, 1>{});
    case 122: return f(Lay<double, 2, 2>{});
    case 131: return f(Lay<double, 3, 1>{});
    case 132: return f(Lay<double, 3, 2>{});
    default: return f(Lay<float, 3, 2>{});
  }
}
size_t push_smem_bytes(const Grid &g) {
  return with_layout(g, [](auto l) { return (size_t)decltype(l)::kEnd; });
}
ItemPlan push_item_plan(const Grid &g) {
  ItemPlan pl;
  const int cap = with_layout(g, [](auto l) { return (int)decltype(l)::CAP; });
  pl.blocks = with_layout(g, [](auto l) { return (int)decltype(l)::BLOCKS; });
  // an item's own cost in slots, from the instructions of the same particles
  // cut differently (2D: 434; 3D TSC: 345; FP64 particles cost far more each)
  pl.fixed = g.prec == 1 ? 120 : 400;
  for (int j = 0; j < kItemCands; ++j) {
    // eight sizes per halving, down to a twelfth: close enough that the items of
    // few tiles can fill the SMs' last round (eight sizes, none below 256,
    // against these: 64^2 FP64 CIC push 39.5 -> 37.3 us, 75 x 50 x 43 FP32 CIC
    // 105 -> 93 us, 2D foil of 0.33M particles 27.8 -> 20.9 us)
    pl.cand[j] = (int)(cap * std::exp2(-j / 8.0)) / kTilePad * kTilePad;
    // 2D FP32: a tile of up to 512 slots stays whole.  An item's window does not
    // depend on the order of its particles, but the windows of its and its
    // neighbours' items are added to J in any order: with one item per tile most
    // nodes receive two values at most, whose sum has no order, so that small
    // differentiable runs mostly repeat themselves to the last bit.  Nodes near a
    // tile's corner receive up to four, escaped particles add theirs by
    // themselves, and larger tiles may be cut: there nothing promises it.
    if (g.dims == 2 && g.prec == 0 && pl.cand[j] < 512) pl.cand[j] = 512;
  }
  int dev = 0;
  pl.nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&pl.nsm, cudaDevAttrMultiProcessorCount, dev);
  return pl;
}

cudaError_t launch_push(const Grid &g, void *const E[3], void *const B[3], void *const J[3], const Particles &p,
                        const WorkSplit &ws, int32_t *esc_list, unsigned long long *esc_count, double q, double m,
                        Counters *ctr, cudaStream_t st, int *nlaunch) {
  const int key = (g.prec == 1 ? 100 : 0) + g.dims * 10 + g.order;
#define PIC_PUSH_CASE(K, R, D, O)                                                                        \
  case K:                                                                                                \
    return g.gather_ec ? launch_t<R, D, O, true>(g, E, B, J, p, ws, esc_list, esc_count, q, m, ctr, st, nlaunch) \
                       : launch_t<R, D, O, false>(g, E, B, J, p, ws, esc_list, esc_count, q, m, ctr, st, nlaunch);
  switch (key) {
    PIC_PUSH_CASE(21, float, 2, 1)
    PIC_PUSH_CASE(22, float, 2, 2)
    PIC_PUSH_CASE(31, float, 3, 1)
    PIC_PUSH_CASE(32, float, 3, 2)
    PIC_PUSH_CASE(121, double, 2, 1)
    PIC_PUSH_CASE(122, double, 2, 2)
    PIC_PUSH_CASE(131, double, 3, 1)
    PIC_PUSH_CASE(132, double, 3, 2)
    default: return cudaErrorInvalidValue;
  }
#undef PIC_PUSH_CASE
}

}  // namespace pic
