// One particle tile of the push: gather + Boris + move + Esirkepov deposition + rebin, shared by the
// linear push (k_particles.cu) and the cubic and momentum-conserving push (k_push_ho.cu). See
// k_particles.cu for the particle storage.
#pragma once
#include "common.cuh"
#include "fastmath.cuh"

namespace picgb {

// Threads per push block: 8 warps; the 3D FP32 kernel 4, so that three blocks fit an SM at 168 registers: the
// 16 cell groups of a tile are four rounds of them, and one block's prologue and epilogue run beside the
// others' particles (128x128x512 pass 21.15 -> 20.2 ms against two blocks of 6 warps). Cubic shapes
// (ORDER 3): the 51 register sums of the 2D window leave 168 registers a thread, two blocks of 6 warps
// in FP32; 3D FP64 6 warps (their stages have to fit in shared memory).
template <typename T, int NDIM, int ORDER = 1>
struct PushThreads {
  static constexpr int value = ORDER == 3 ? (NDIM == 3 ? (sizeof(T) == 4 ? 384 : 192) : (sizeof(T) == 4 ? 192 : 256))
                                          : (NDIM == 3 && sizeof(T) == 4) ? 128 : 256;
};

// The tile's compile-time extents by shape order.
template <typename T, int NDIM, int ORDER>
struct PushTileOf {
  using type = PTile<T, NDIM>;
};
template <typename T, int NDIM>
struct PushTileOf<T, NDIM, 3> {
  using type = HoTile<T, NDIM>;
};

// Per-warp double-buffered stage of an item (32 packs of 4 slots, cell by cell): [32][4][4] values q,
// [32][4][RW] values r, [32][4] weights per stage (SpeciesBuf's arrays), then [stage][32][4] ids. The
// four slots of pack p of a cell follow those of pack p - 1, so slot k of the cell's 4 LPC is element k
// from the cell's first lane.
template <typename T, int NDIM>
struct PushStage {
  static constexpr int RW = NDIM == 3 ? 2 : 1;
  static constexpr int ELEMS = 32 * (16 + 4 * RW + 4);  // per stage
  static constexpr __host__ __device__ size_t per_warp_elems() {
    return 2 * ELEMS + (2 * 32 * 4 * sizeof(unsigned) + sizeof(T) - 1) / sizeof(T);
  }
  static __device__ __forceinline__ T* q(T* base, int stage, int lane) { return base + stage * ELEMS + lane * 16; }
  static __device__ __forceinline__ T* r(T* base, int stage, int lane) {
    return base + stage * ELEMS + 32 * 16 + lane * 4 * RW;
  }
  static __device__ __forceinline__ T* w(T* base, int stage, int lane) {
    return base + stage * ELEMS + 32 * (16 + 4 * RW) + lane * 4;
  }
  static __device__ __forceinline__ unsigned* id(T* base, int stage, int lane) {
    return reinterpret_cast<unsigned*>(base + 2 * ELEMS) + (stage * 32 + lane) * 4;
  }
};

// FP32 2D: each lane takes two particles of its cell at a time, with the arithmetic of the pair
// in packed FP32x2 instructions (one instruction advances both particles) and the two rebins
// interleaved, so one dependent chain carries two particles.
template <typename T, int NDIM>
struct PushPaired {
  static constexpr bool value = sizeof(T) == 4 && NDIM == 2;
};

// WIN: the gather reads every particle's nodes from one window of its cell (gather_window), as the
// cubic and the momentum-conserving gathers do; a paired push then keeps every node twice, so that one
// 8-byte load yields the packed operand for both particles.
template <typename T, int NDIM, int ORDER = 1, bool WIN = false>
struct PushSmem {
  using TL = typename PushTileOf<T, NDIM, ORDER>::type;
  static constexpr int TX = TL::TX, TY = TL::TY, TZ = TL::TZ;
  static constexpr int NCL = TX * TY * TZ;
  static constexpr int H = (ORDER + 1) / 2;
  // gather tile: nodes [X0-H, X0+TX+H) per direction (y only in 3D)
  static constexpr int GX = TX + 2 * H, GY = (NDIM == 3 ? TY + 2 * H : 1), GZ = TZ + 2 * H, GN = GX * GY * GZ;
  static constexpr int GCOPY = WIN && PushPaired<T, NDIM>::value ? 2 : 1;  // stored values per node
  // current tile: nodes [X0-H, X0+TX+H]
  static constexpr int JX = TX + 2 * H + 1, JY = (NDIM == 3 ? TY + 2 * H + 1 : 1), JZ = TZ + 2 * H + 1;
  static constexpr int JN = JX * JY * JZ;
  // particles leaving the tile, buffered per block: [7][LVB] values (ox oy oz dux duy duz w), LVB
  // keys, LVB ids and the buffer's counter; written to the global leaver list once per tile
  // (3D: within the shared memory of one block per SM in FP64, of three in FP32)
  static constexpr int LVB = NDIM == 3 ? (sizeof(T) == 8 ? 128 : 256) : 512;
  static constexpr size_t lv_bytes() { return (size_t)LVB * (7 * sizeof(T) + 2 * sizeof(int)) + 16; }
  static constexpr size_t bytes() {
    return sizeof(T) * (6 * GN * GCOPY + 3 * JN) + sizeof(int) * (4 * NCL) + 16 +
           sizeof(T) * PushStage<T, NDIM>::per_warp_elems() * (PushThreads<T, NDIM, ORDER>::value / 32) + 16 + lv_bytes();
  }
};

// Per-direction interpolation weights of a particle at cell-relative offset o:
// integer-node S1 (base 0: nodes 0, 1), half-node S1 (Uniform: base -1 or 0), half-node S0
// (Galerkin: node 0). Bases are relative to the particle's cell.
template <typename T>
struct DirW {
  T i0, i1;     // integer nodes 0 and 1
  int hb;       // half-node base (-1 or 0)
  T h0, h1;     // half nodes hb, hb+1
};

template <typename T>
__device__ __forceinline__ DirW<T> dir_weights(T o) {
  DirW<T> d;
  d.i0 = T(1) - o;
  d.i1 = o;
  if (o < T(0.5)) {
    d.hb = -1;
    T g = o + T(0.5);
    d.h0 = T(1) - g;
    d.h1 = g;
  } else {
    d.hb = 0;
    T g = o - T(0.5);
    d.h0 = T(1) - g;
    d.h1 = g;
  }
  return d;
}

// One direction of the gather: returns (base, w0, w1, two) for stagger st and scheme.
template <typename T, int SCHEME>
__device__ __forceinline__ void pick(const DirW<T>& d, int st, int& base, T& w0, T& w1, bool& two) {
  if (!st) {
    base = 0; w0 = d.i0; w1 = d.i1; two = true;
  } else if (SCHEME == 0) {  // Galerkin: S0 along a half-staggered direction
    base = 0; w0 = T(1); w1 = T(0); two = false;
  } else {                   // Uniform: S1 at the half-integer nodes
    base = d.hb; w0 = d.h0; w1 = d.h1; two = true;
  }
}

// Stagger of Ex Ey Ez Bx By Bz along x, y, z.
__device__ __constant__ int c_stag[6][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {0, 1, 1}, {1, 0, 1}, {1, 1, 0}};

template <typename T, int NDIM, int SCHEME>
__device__ __forceinline__ T gather_comp(const T* __restrict__ sgc, int c, int lx, int ly, int lz, const DirW<T>& dx,
                                         const DirW<T>& dy, const DirW<T>& dz) {
  using S = PushSmem<T, NDIM>;
  int bx, by = 0, bz;
  T x0, x1, y0 = T(1), y1 = T(0), z0, z1;
  bool tx, ty = false, tz;
  pick<T, SCHEME>(dx, c_stag[c][0], bx, x0, x1, tx);
  if (NDIM == 3) pick<T, SCHEME>(dy, c_stag[c][1], by, y0, y1, ty);
  pick<T, SCHEME>(dz, c_stag[c][2], bz, z0, z1, tz);
  // smem index of node (lx+bx, ly+by, lz+bz), +1 halo offset per direction
  const int ix = lx + bx + 1, iy = (NDIM == 3 ? ly + by + 1 : 0), iz = lz + bz + 1;
  const T* p = sgc + (iz * S::GY + iy) * S::GX + ix;
  T acc;
  {
    T r0 = x0 * p[0] + (tx ? x1 * p[1] : T(0));
    T r1 = T(0);
    if (ty) {
      const T* q = p + S::GX;
      r1 = x0 * q[0] + (tx ? x1 * q[1] : T(0));
    }
    acc = z0 * (y0 * r0 + y1 * r1);
  }
  if (tz) {
    const T* p2 = p + S::GX * S::GY;
    T r0 = x0 * p2[0] + (tx ? x1 * p2[1] : T(0));
    T r1 = T(0);
    if (ty) {
      const T* q = p2 + S::GX;
      r1 = x0 * q[0] + (tx ? x1 * q[1] : T(0));
    }
    acc += z1 * (y0 * r0 + y1 * r1);
  }
  return acc;
}

// One direction of an Esirkepov move of displacement d (|d| < 1 cell) from offset o in [0,1):
// the 3-node window (origin a = -1 or 0 relative to the cell), the start shapes S0 and the shape
// changes dS on it, and the new cell shift and offset. dS is formed from d itself (slope times
// the move on the linear piece of the spline), not as S(o + d) - S(o), so that moves far below one
// ulp of the offset (the transverse drift of a cold relativistic beam) keep full relative
// precision; the three dS always sum to zero (charge conservation).
template <typename T>
struct EsirDir {
  int a, shift;
  T off;
  T S0[3], dS[3];
};

// Comparisons of the push's values. FP64: integer tests on the IEEE bit patterns, exact for every
// value that is not a NaN (the offsets and displacements compared here are finite), which keeps
// them off the narrow FP64 pipe that bounds the FP64 push. FP32: plain comparisons.
template <typename T>
__device__ __forceinline__ bool is_neg(T x) {  // x < 0 (-0 is not)
  if constexpr (sizeof(T) == 8) return (unsigned long long)__double_as_longlong(x) > 0x8000000000000000ull;
  else return x < T(0);
}
template <typename T>
__device__ __forceinline__ bool is_pos(T x) {  // x > 0
  if constexpr (sizeof(T) == 8) return __double_as_longlong(x) > 0;
  else return x > T(0);
}
template <typename T>
__device__ __forceinline__ bool ge_one(T x) {  // x >= 1
  if constexpr (sizeof(T) == 8) return __double_as_longlong(x) >= 0x3FF0000000000000ll;
  else return x >= T(1);
}
template <typename T>
__device__ __forceinline__ bool abs_lt_one(T x) {  // -1 < x < 1; false for a NaN or an infinity
  if constexpr (sizeof(T) == 8) return (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll) < 0x3FF0000000000000ll;
  else return x > T(-1) && x < T(1);
}

template <typename T>
__device__ __forceinline__ EsirDir<T> esir_dir(T o, T d) {
  EsirDir<T> e;
  const T x1 = o + d;
  if (is_neg(x1)) {  // into the cell below: window nodes -1, 0, 1
    e.a = -1;
    e.S0[0] = T(0); e.S0[1] = T(1) - o; e.S0[2] = o;
    e.dS[0] = -x1; e.dS[2] = -o; e.dS[1] = -(e.dS[0] + e.dS[2]);
    e.off = T(1) + x1;
    e.shift = -1;
    if (ge_one(e.off)) { e.off = T(0); e.shift = 0; }
  } else {
    e.a = 0;
    e.S0[0] = T(1) - o; e.S0[1] = o; e.S0[2] = T(0);
    const T am = T(1) - o;  // distance to the upper face
    const T c = d - am;     // x1 - 1, without the rounding of x1
    if (ge_one(x1) && is_pos(c)) {  // into the cell above: nodes 0, 1, 2
      e.dS[0] = -am; e.dS[2] = c; e.dS[1] = -(e.dS[0] + e.dS[2]);
      e.off = c;
      e.shift = 1;
    } else {  // same cell (or onto the upper face within rounding)
      e.dS[0] = -d; e.dS[1] = d; e.dS[2] = T(0);
      if (ge_one(x1)) { e.off = T(0); e.shift = 1; }
      else { e.off = x1; e.shift = 0; }
    }
  }
  return e;
}

// Layout of one particle's current contributions: index i -> (component, node offset in the
// 3-node window). 2D: 6 Jx (b*2+a), 6 Jz (6+a*2+b), 9 Jy (12+b*3+a). 3D: 18 Jx ((c*3+b)*2+a),
// 18 Jy (18+(c*3+a)*2+b), 18 Jz (36+(b*3+a)*2+c); a, b, c are the x, y, z node offsets.
template <int NDIM>
struct DepLayout;
template <>
struct DepLayout<2> {
  static constexpr int NV = 21;
  static __device__ __forceinline__ void at(int i, int& comp, int& a, int& b, int& c) {
    b = 0;
    if (i < 6) { comp = 0; c = i >> 1; a = i & 1; }
    else if (i < 12) { comp = 2; a = (i - 6) >> 1; c = (i - 6) & 1; }
    else { comp = 1; c = (i - 12) / 3; a = (i - 12) % 3; }
  }
};
template <>
struct DepLayout<3> {
  static constexpr int NV = 54;
  static __device__ __forceinline__ void at(int i, int& comp, int& a, int& b, int& c) {
    if (i < 18) { comp = 0; a = i & 1; b = (i >> 1) % 3; c = (i >> 1) / 3; }
    else if (i < 36) { const int m = i - 18; comp = 1; b = m & 1; a = (m >> 1) % 3; c = (m >> 1) / 3; }
    else { const int m = i - 36; comp = 2; c = m & 1; a = (m >> 1) % 3; b = (m >> 1) / 3; }
  }
};

// Periodic index of g in [-n, 2n) without a modulo (callers guarantee the range: near_ok, or a
// neighbour cell index in [-1, n]).
__device__ __forceinline__ int wrap_near_p(int g, int n) { return g < 0 ? g + n : (g >= n ? g - n : g); }

// Reciprocals and square roots: FP32 the hardware's estimates (relative error ~1e-7, inside the 1e-5
// per-step bar), FP64 one third-order step from them (fastmath.cuh).

// Galerkin gather (order 0 along each half-staggered direction, order 1 elsewhere): the nodes are
// the same for every particle of a cell, so they are read once per lane and each component is an
// affine or bilinear function of the cell offsets. Node (a, b, c) of a component is its value at
// offsets (a, b, c) from the cell's own node in the shared-memory tile.
template <typename T, int NDIM>
struct GalCache;

template <typename T>
struct GalCache<T, 2> {
  // Ex: x half -> S0; z -> S1. Ey: S1 x, S1 z. Ez: S1 x; z half -> S0. Bx: S1 x; S0 z.
  // By: S0 x, S0 z. Bz: S0 x; S1 z.
  T ex0, ex1, ey00, ey10, ey01, ey11, ez0, ez1, bx0, bx1, by0, bz0, bz1;
  __device__ __forceinline__ void load(const T* sg, int lx, int ly, int lz) {
    using S = PushSmem<T, 2>;
    const int p = (lz + 1) * S::GX + lx + 1;
    const T* e = sg;
    ex0 = e[p]; ex1 = e[p + S::GX] - ex0;
    e = sg + S::GN;
    ey00 = e[p]; ey10 = e[p + 1] - ey00; ey01 = e[p + S::GX] - ey00; ey11 = e[p + S::GX + 1] - e[p + S::GX] - ey10;
    e = sg + 2 * S::GN;
    ez0 = e[p]; ez1 = e[p + 1] - ez0;
    e = sg + 3 * S::GN;
    bx0 = e[p]; bx1 = e[p + 1] - bx0;
    by0 = sg[4 * S::GN + p];
    e = sg + 5 * S::GN;
    bz0 = e[p]; bz1 = e[p + S::GX] - bz0;
  }
  __device__ __forceinline__ void interp(T ox, T, T oz, T (&F)[6]) const {
    F[0] = ex0 + oz * ex1;
    F[1] = ey00 + ox * ey10 + oz * (ey01 + ox * ey11);
    F[2] = ez0 + ox * ez1;
    F[3] = bx0 + ox * bx1;
    F[4] = by0;
    F[5] = bz0 + oz * bz1;
  }
};

template <typename T>
struct GalCache<T, 3> {
  // Ex: S0 x, bilinear (y, z). Ey: S0 y, bilinear (x, z). Ez: S0 z, bilinear (x, y).
  // Bx: S0 y, z, linear x. By: S0 x, z, linear y. Bz: S0 x, y, linear z.
  T e[3][4], b[3][2];
  __device__ __forceinline__ void bil(const T* f, int p, int s1, int s2, T (&o)[4]) {
    o[0] = f[p];
    o[1] = f[p + s1] - o[0];
    o[2] = f[p + s2] - o[0];
    o[3] = f[p + s1 + s2] - f[p + s2] - o[1];
  }
  __device__ __forceinline__ void load(const T* sg, int lx, int ly, int lz) {
    using S = PushSmem<T, 3>;
    const int p = ((lz + 1) * S::GY + ly + 1) * S::GX + lx + 1;
    const int sx = 1, sy = S::GX, sz = S::GX * S::GY;
    bil(sg, p, sy, sz, e[0]);
    bil(sg + S::GN, p, sx, sz, e[1]);
    bil(sg + 2 * S::GN, p, sx, sy, e[2]);
    b[0][0] = sg[3 * S::GN + p]; b[0][1] = sg[3 * S::GN + p + sx] - b[0][0];
    b[1][0] = sg[4 * S::GN + p]; b[1][1] = sg[4 * S::GN + p + sy] - b[1][0];
    b[2][0] = sg[5 * S::GN + p]; b[2][1] = sg[5 * S::GN + p + sz] - b[2][0];
  }
  __device__ __forceinline__ void interp(T ox, T oy, T oz, T (&F)[6]) const {
    F[0] = e[0][0] + oy * e[0][1] + oz * (e[0][2] + oy * e[0][3]);
    F[1] = e[1][0] + ox * e[1][1] + oz * (e[1][2] + ox * e[1][3]);
    F[2] = e[2][0] + ox * e[2][1] + oy * (e[2][2] + ox * e[2][3]);
    F[3] = b[0][0] + ox * b[0][1];
    F[4] = b[1][0] + oy * b[1][1];
    F[5] = b[2][0] + oz * b[2][1];
  }
};

// Esirkepov contributions of one particle, written as sums into the 3-node window of its own
// cell (layout of DepLayout). With f = S0 + dS/2 per direction, the 2D out-of-plane weight
// S0x S0z + dSx S0z/2 + S0x dSz/2 + dSx dSz/3 equals fx fz + dSx dSz / 12, and the running sums
// of the in-plane weights at the two half-nodes are dS[0] and -dS[2] times the transverse factor.
template <typename T, int NVP>
__device__ __forceinline__ void deposit2(T (&acc)[NVP], const EsirDir<T>& X, const EsirDir<T>& Z, T cx, T cy, T cz) {
  T fx[3], fz[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    fx[a] = X.S0[a] + T(0.5) * X.dS[a];
    fz[a] = Z.S0[a] + T(0.5) * Z.dS[a];
  }
  const T gx0 = cx * X.dS[0], gx1 = -cx * X.dS[2];
  const T gz0 = cz * Z.dS[0], gz1 = -cz * Z.dS[2];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    acc[b * 2 + 0] += gx0 * fz[b];
    acc[b * 2 + 1] += gx1 * fz[b];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    acc[6 + a * 2 + 0] += gz0 * fx[a];
    acc[6 + a * 2 + 1] += gz1 * fx[a];
  }
  T hx[3], kx[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    hx[a] = cy * fx[a];
    kx[a] = cy * X.dS[a] * T(1.0 / 12.0);
  }
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[12 + b * 3 + a] += hx[a] * fz[b] + kx[a] * Z.dS[b];
}

// Same contributions added to shared memory at the window origin (wx, wz) (tile indices).
template <typename T, int NDIM>
__device__ __forceinline__ void deposit2_smem(T* sj, int wx, int wz, EsirDir<T> X, EsirDir<T> Z, T cx, T cy, T cz) {
  using S = PushSmem<T, NDIM>;
  T v[DepLayout<2>::NV];
#pragma unroll
  for (int i = 0; i < DepLayout<2>::NV; ++i) v[i] = T(0);
  deposit2<T, DepLayout<2>::NV>(v, X, Z, cx, cy, cz);
  const int key = wz * S::JX + wx;
#pragma unroll
  for (int i = 0; i < DepLayout<2>::NV; ++i) {
    int comp, a, b, c;
    DepLayout<2>::at(i, comp, a, b, c);
    atomicAdd(sj + comp * S::JN + key + c * S::JX + a, v[i]);
  }
}

// 3D: W_a = dS_a T(b1, b2) with T = f f + dS dS / 12 over the two transverse directions.
template <typename T, int NVP>
__device__ __forceinline__ void deposit3(T (&acc)[NVP], const EsirDir<T>& X, const EsirDir<T>& Y, const EsirDir<T>& Z,
                                         T cx, T cy, T cz) {
  T fx[3], fy[3], fz[3], kx[3], ky[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    fx[a] = X.S0[a] + T(0.5) * X.dS[a];
    fy[a] = Y.S0[a] + T(0.5) * Y.dS[a];
    fz[a] = Z.S0[a] + T(0.5) * Z.dS[a];
    kx[a] = X.dS[a] * T(1.0 / 12.0);
    ky[a] = Y.dS[a] * T(1.0 / 12.0);
  }
  const T gx0 = cx * X.dS[0], gx1 = -cx * X.dS[2];
  const T gy0 = cy * Y.dS[0], gy1 = -cy * Y.dS[2];
  const T gz0 = cz * Z.dS[0], gz1 = -cz * Z.dS[2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int b = 0; b < 3; ++b) {  // Jx(a+1/2, b, c)
      const T t = fy[b] * fz[c] + ky[b] * Z.dS[c];
      acc[(c * 3 + b) * 2 + 0] += gx0 * t;
      acc[(c * 3 + b) * 2 + 1] += gx1 * t;
    }
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // Jy(a, b+1/2, c)
      const T t = fx[a] * fz[c] + kx[a] * Z.dS[c];
      acc[18 + (c * 3 + a) * 2 + 0] += gy0 * t;
      acc[18 + (c * 3 + a) * 2 + 1] += gy1 * t;
    }
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // Jz(a, b, c+1/2)
      const T t = fx[a] * fy[b] + kx[a] * Y.dS[b];
      acc[36 + (b * 3 + a) * 2 + 0] += gz0 * t;
      acc[36 + (b * 3 + a) * 2 + 1] += gz1 * t;
    }
}

template <typename T, int NDIM>
__device__ __forceinline__ void deposit3_smem(T* sj, int wx, int wy, int wz, EsirDir<T> X, EsirDir<T> Y, EsirDir<T> Z,
                                           T cx, T cy, T cz) {
  using S = PushSmem<T, NDIM>;
  T v[DepLayout<3>::NV];
#pragma unroll
  for (int i = 0; i < DepLayout<3>::NV; ++i) v[i] = T(0);
  deposit3<T, DepLayout<3>::NV>(v, X, Y, Z, cx, cy, cz);
  const int key = (wz * S::JY + wy) * S::JX + wx;
#pragma unroll
  for (int i = 0; i < DepLayout<3>::NV; ++i) {
    int comp, a, b, c;
    DepLayout<3>::at(i, comp, a, b, c);
    atomicAdd(sj + comp * S::JN + key + (c * S::JY + b) * S::JX + a, v[i]);
  }
}

// The sums each lane keeps in registers: the Esirkepov window of a particle that starts in its own
// cell, does not step back across a face, and does not cross its cell's upper face in x (nor, in
// 3D, in y). Such a particle's shape changes vanish at the window's third transverse node (S0 and
// dS are zero there), so its contributions there are exactly zero: of the 3-node window only
// x nodes 0-1 (2D: 13 of the 21 sums; 3D: y nodes 0-1 too, 20 of the 54) carry it. Every other
// particle (a transverse face crossed, or a step back) adds its full window to shared memory.
// 2D layout: 3 Jx (node a = 0, z node c = i), 4 Jz (3 + a*2 + c), 6 Jy (7 + c*2 + a).
// 3D layout: 6 Jx (a = 0; c*2 + b), 6 Jy (b = 0; 6 + c*2 + a), 8 Jz (12 + (b*2 + a)*2 + c).
// Cubic, 2D (ORDER 3; nodes from one below the cell: x 0-3, z 0-4): 15 Jx (c*3 + a), 16 Jz
// (15 + a*4 + c), 20 Jy (31 + c*4 + a). Cubic in 3D deposits after the push (deposit3_cubic).
template <int NDIM, int ORDER = 1>
struct RegLayout;
template <>
struct RegLayout<2, 3> {
  static constexpr int NV = 51;
  static __device__ __forceinline__ void at(int i, int& comp, int& a, int& b, int& c) {
    b = 0;
    if (i < 15) { comp = 0; c = i / 3; a = i - 3 * c; }
    else if (i < 31) { comp = 2; a = (i - 15) >> 2; c = (i - 15) & 3; }
    else { comp = 1; c = (i - 31) >> 2; a = (i - 31) & 3; }
  }
};
template <>
struct RegLayout<3, 3> {
  static constexpr int NV = 1;  // no sums are kept across rounds
  static __device__ __forceinline__ void at(int, int&, int&, int&, int&) {}
};
template <>
struct RegLayout<2, 1> {
  static constexpr int NV = 13;
  static __device__ __forceinline__ void at(int i, int& comp, int& a, int& b, int& c) {
    b = 0;
    if (i < 3) { comp = 0; a = 0; c = i; }
    else if (i < 7) { comp = 2; a = (i - 3) >> 1; c = (i - 3) & 1; }
    else { comp = 1; c = (i - 7) >> 1; a = (i - 7) & 1; }
  }
};
template <>
struct RegLayout<3, 1> {
  static constexpr int NV = 20;
  static __device__ __forceinline__ void at(int i, int& comp, int& a, int& b, int& c) {
    if (i < 6) { comp = 0; a = 0; b = i & 1; c = i >> 1; }
    else if (i < 12) { const int k = i - 6; comp = 1; b = 0; a = k & 1; c = k >> 1; }
    else { const int k = i - 12; comp = 2; c = k & 1; a = (k >> 1) & 1; b = k >> 2; }
  }
};

// Rounds of a full item: 4 particles a lane, one or (paired) two per round.
template <typename T, int NDIM>
struct PushRounds {
  static constexpr int value = PushPaired<T, NDIM>::value ? 2 : 4;
};

// Work assignment of the push kernel: a warp takes CPW = 32/LPC cells of its tile at a time,
// LPC lanes per cell. The cell's particles are split into packs of 4 consecutive slots of one
// species (electron packs first); an item is LPC packs of every cell of the group, copied by one lane
// each (16-byte copies: 8-byte ones cost the 3D push 40 %). Within an item the cell's lanes take its
// 4 LPC slots in turn, one window of LPC slots (a paired push: two windows) per round, and the warp
// runs only the rounds that its fullest cell needs. A cell of 17 + 16 particles costs its warp 9 rounds
// of single particles (12 when every lane walked its own pack), and with 4 + 4 particles all four
// lanes work (two of them before). Measured on 512x1024 FP32 cells, push per step: 16 per species at
// c dt/dz = 0.5 (even cells) 330 -> 311 us and 0.3 523 -> 507 us, 8 per species 319 -> 231 us, 4 per
// species 241 -> 174 us; 256x512 FP64 at 0.3 1.99 -> 1.76 ms; 3D 64x64x256 0.87 -> 0.84 ms. Each lane sums
// the Esirkepov contributions of its particles in registers (the window of RegLayout: every
// particle that neither steps back across a face nor crosses a transverse face); at the end one
// segmented butterfly transpose-reduction over the cell's LPC lanes leaves PER = NVP/LPC of the
// cell's NVP (padded) sums in each lane, added to shared memory with distinct addresses. The other
// particles add their full 3-node window to shared memory directly.
template <int NDIM, int LPC, int ORDER = 1>
struct PushPlan {
  static constexpr int NV = RegLayout<NDIM, ORDER>::NV;
  static constexpr int PER = (NV + LPC - 1) / LPC;
  static constexpr int NVP = PER * LPC;
  static constexpr int CPW = 32 / LPC;
  // An item's 4 LPC slots of a cell form four windows of LPC slots, one per lane each. Which window the
  // cell (c-th of the group) starts a full item with: neighbouring cells start with different ones,
  // because the same window of neighbouring cells lies in the same shared-memory banks.
  static __device__ __forceinline__ int first_window(int c) { return LPC == 4 ? (c >> 1) + (c & 1) : c; }
};

// Crowded cells. A cell with many more packs than its group's others would keep its warp on its LPC lanes, so
// the group leaves it out and the warp then takes it by itself, its packs spread over all lanes (an item is
// 32 of them). A step with 1500 more particles per species in eight cells: momentum-conserving 128x256 FP32
// 495 -> 98 us, FP64 3.5 -> 0.59 ms, cubic FP64 7.6 -> 1.26 ms, 3D 24^3 FP32 1359 -> 138 us; 20,000 in one
// cell, cubic FP32 8.3 -> 0.97 ms (6.3 when a cell had a warp). Even cells pay 0.4 % of the 3D pass, 1.4 %
// of the cubic FP32 one (6.18 -> 6.27 ms on 512x1024).
template <typename T, int NDIM, int ORDER, bool WIN>
struct PushCrowd {
  static constexpr bool value = WIN ? NDIM == 2 : NDIM == 3 && sizeof(T) == 4;
};

// Resident blocks per SM the push kernel is compiled for (register budget).
template <typename T, int NDIM, int ORDER = 1>
struct PushMinBlocks {
  static constexpr int value = sizeof(T) == 8 || (NDIM == 3 && ORDER == 3) ? 1 : (NDIM == 3 ? 3 : 2);
};

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// ---------------------------------------------------------------------------------------------
// Cubic shapes and the momentum-conserving gather.
// ---------------------------------------------------------------------------------------------
// Centred B-splines.
template <typename T>
__device__ __forceinline__ T bspl(int n, T t) {
  const T a = t < T(0) ? -t : t;
  if (n == 0) return (t >= T(-0.5) && t < T(0.5)) ? T(1) : T(0);
  if (n == 1) return a < T(1) ? T(1) - a : T(0);
  if (n == 2) {
    if (a <= T(0.5)) return T(0.75) - a * a;
    if (a < T(1.5)) return T(0.5) * (T(1.5) - a) * (T(1.5) - a);
    return T(0);
  }
  if (a <= T(1)) return T(2.0 / 3.0) - a * a + T(0.5) * a * a * a;
  if (a < T(2)) return (T(2) - a) * (T(2) - a) * (T(2) - a) * T(1.0 / 6.0);
  return T(0);
}

// S_n(a0 - d) - S_n(a0) for the particle shape (n = 1 or 3): on one polynomial piece from the
// displacement (linear: slope times -d; cubic: the terminating Taylor series), else the difference.
template <typename T>
__device__ __forceinline__ T shape_change(int n, T a0, T d) {
  const T a1 = a0 - d;
  if (n == 1) {
    const int p0 = (a0 > T(-1)) + (a0 > T(0)) + (a0 >= T(1)), p1 = (a1 > T(-1)) + (a1 > T(0)) + (a1 >= T(1));
    if (p0 == p1) return p0 == 1 ? -d : (p0 == 2 ? d : T(0));
    return bspl(1, a1) - bspl(1, a0);
  }
  const int p0 = (a0 > T(-2)) + (a0 > T(-1)) + (a0 > T(0)) + (a0 > T(1)) + (a0 >= T(2));
  const int p1 = (a1 > T(-2)) + (a1 > T(-1)) + (a1 > T(0)) + (a1 > T(1)) + (a1 >= T(2));
  if (p0 != p1) return bspl(3, a1) - bspl(3, a0);
  T d1, d2, d3;  // P', P'', P''' of the piece at a0
  switch (p0) {
    case 1: d1 = T(0.5) * (T(2) + a0) * (T(2) + a0); d2 = T(2) + a0; d3 = T(1); break;
    case 2: d1 = -T(2) * a0 - T(1.5) * a0 * a0; d2 = -T(2) - T(3) * a0; d3 = T(-3); break;
    case 3: d1 = -T(2) * a0 + T(1.5) * a0 * a0; d2 = -T(2) + T(3) * a0; d3 = T(3); break;
    case 4: d1 = -T(0.5) * (T(2) - a0) * (T(2) - a0); d2 = T(2) - a0; d3 = T(-1); break;
    default: return T(0);
  }
  return -d * (d1 - d * (T(0.5) * d2 - d * d3 * T(1.0 / 6.0)));
}

// Stagger of Ex Ey Ez Bx By Bz along x, y, z (compile-time, so that the gather's orders and loop
// bounds fold for each unrolled component).
__host__ __device__ constexpr int stag_ho(int c, int axis) {
  return axis == 0 ? (c == 0 || c == 4 || c == 5) : (axis == 1 ? (c == 1 || c == 3 || c == 5) : (c == 2 || c == 3 || c == 4));
}

// One value, or the values of a particle pair in one packed FP32x2 operand.
template <typename T>
struct Lanes1 {
  using V = T;
  static __device__ __forceinline__ V set(T a) { return a; }
  static __device__ __forceinline__ V node(const T* p) { return *p; }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return ::fma(a, b, c); }
  static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
  static __device__ __forceinline__ V add(V a, V b) { return a + b; }
  static __device__ __forceinline__ V neg(V a) { return -a; }
  static __device__ __forceinline__ V pick_low(V a, V lo, V hi) { return a < T(0.5) ? lo : hi; }
  using B = bool;
  static __device__ __forceinline__ V sel(B m, V a, V b) { return m ? a : b; }
};
struct Bool2 {
  bool x, y;
};
struct Lanes2 {
  using V = float2;
  static __device__ __forceinline__ V set(float a) { return make_float2(a, a); }
  static __device__ __forceinline__ V node(const float* p) { return *reinterpret_cast<const float2*>(p); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ V pick_low(V a, V lo, V hi) {
    return make_float2(a.x < 0.5f ? lo.x : hi.x, a.y < 0.5f ? lo.y : hi.y);
  }
  using B = Bool2;
  static __device__ __forceinline__ V sel(B m, V a, V b) { return make_float2(m.x ? a.x : b.x, m.y ? a.y : b.y); }
};

// Weights of the cubic spline on the nodes -1, 0, 1, 2 of the cell for an offset o in [0, 1].
template <class L, typename T, typename V>
__device__ __forceinline__ void cubic_weights(V o, V (&w)[4]) {
  const V p = L::add(L::set(T(1)), L::neg(o));
  const V o2 = L::mul(o, o), p2 = L::mul(p, p);
  const V six = L::set(T(1.0 / 6.0)), half = L::set(T(0.5)), two3 = L::set(T(2.0 / 3.0));
  w[0] = L::mul(L::mul(p2, p), six);
  w[3] = L::mul(L::mul(o2, o), six);
  w[1] = L::fma(o2, L::fma(half, o, L::set(T(-1))), two3);  // 2/3 - o^2 + o^3 / 2
  w[2] = L::fma(p2, L::fma(half, p, L::set(T(-1))), two3);
}

// Nodes of one direction of the gather: NI integer nodes from FI on, NS half-staggered ones from FS
// on, relative to the cell. Every particle of a cell reads the same nodes: the Uniform cubic gather on
// half-staggered nodes takes five, with a zero weight at one end (the range of its four depends on the
// half of the cell the particle is in).
template <int ORDER, int SCHEME>
struct WinNodes {
  static constexpr int NI = ORDER + 1, FI = -(ORDER - 1) / 2;
  static constexpr int NS = SCHEME == 0 ? ORDER : ORDER + 2, FS = ORDER == 3 ? (SCHEME == 0 ? -1 : -2) : 0;
};
template <class L, typename T, typename V, int ORDER, int SCHEME>
__device__ __forceinline__ void win_weights(V o, V (&wi)[4], V (&ws)[5]) {
  if constexpr (ORDER == 1) {
    wi[0] = L::add(L::set(T(1)), L::neg(o));
    wi[1] = o;
  } else {
    cubic_weights<L, T, V>(o, wi);
    if constexpr (SCHEME == 0) {  // quadratic spline about the half node: t = o - 1/2
      const V t = L::add(o, L::set(T(-0.5))), half = L::set(T(0.5));
      const V q = L::add(half, L::neg(t)), r = L::add(half, t);
      ws[0] = L::mul(half, L::mul(q, q));
      ws[1] = L::fma(L::neg(t), t, L::set(T(0.75)));
      ws[2] = L::mul(half, L::mul(r, r));
    } else if constexpr (SCHEME == 1) {
      const V f = L::pick_low(o, L::add(o, L::set(T(0.5))), L::add(o, L::set(T(-0.5))));
      V c[4];
      cubic_weights<L, T, V>(f, c);
      const V z = L::set(T(0));
      ws[0] = L::pick_low(o, c[0], z);
      ws[1] = L::pick_low(o, c[1], c[0]);
      ws[2] = L::pick_low(o, c[2], c[1]);
      ws[3] = L::pick_low(o, c[3], c[2]);
      ws[4] = L::pick_low(o, z, c[3]);
    }
  }
}

// Component C of the gather from the window of cell (lx, ly, lz). The momentum-conserving scheme
// (2) reads integer nodes only: its tile holds the node averages.
template <class L, typename T, typename V, int NDIM, int ORDER, int SCHEME, int C>
__device__ __forceinline__ V window_comp(const T* sg, int lx, int ly, int lz, const V (&xi)[4], const V (&xs)[5],
                                         const V (&yi)[4], const V (&ys)[5], const V (&zi)[4], const V (&zs)[5]) {
  using S = PushSmem<T, NDIM, ORDER, true>;
  using W = WinNodes<ORDER, SCHEME>;
  constexpr bool SX = SCHEME != 2 && stag_ho(C, 0), SY = SCHEME != 2 && stag_ho(C, 1), SZ = SCHEME != 2 && stag_ho(C, 2);
  constexpr int NX = SX ? W::NS : W::NI, NY = NDIM == 3 ? (SY ? W::NS : W::NI) : 1, NZ = SZ ? W::NS : W::NI;
  const int ix = lx + S::H + (SX ? W::FS : W::FI), iz = lz + S::H + (SZ ? W::FS : W::FI);
  const int iy = NDIM == 3 ? ly + S::H + (SY ? W::FS : W::FI) : 0;
  const T* p = sg + (C * S::GN + (iz * S::GY + iy) * S::GX + ix) * S::GCOPY;
  V acc = L::set(T(0));
#pragma unroll
  for (int c = 0; c < NZ; ++c) {
    V plane = L::set(T(0));
#pragma unroll
    for (int b = 0; b < NY; ++b) {
      const T* q = p + (c * S::GY + b) * S::GX * S::GCOPY;
      V row = L::mul(SX ? xs[0] : xi[0], L::node(q));
#pragma unroll
      for (int a = 1; a < NX; ++a) row = L::fma(SX ? xs[a] : xi[a < 4 ? a : 3], L::node(q + a * S::GCOPY), row);
      if (NDIM == 3) plane = L::fma(SY ? ys[b] : yi[b < 4 ? b : 3], row, plane);
      else plane = row;
    }
    acc = L::fma(SZ ? zs[c] : zi[c < 4 ? c : 3], plane, acc);
  }
  return acc;
}

template <class L, typename T, typename V, int NDIM, int ORDER, int SCHEME>
__device__ __forceinline__ void gather_window(const T* sg, int lx, int ly, int lz, V ox, V oy, V oz, V (&F)[6]) {
  V xi[4], xs[5], yi[4], ys[5], zi[4], zs[5];
  win_weights<L, T, V, ORDER, SCHEME>(ox, xi, xs);
  if (NDIM == 3) win_weights<L, T, V, ORDER, SCHEME>(oy, yi, ys);
  win_weights<L, T, V, ORDER, SCHEME>(oz, zi, zs);
  F[0] = window_comp<L, T, V, NDIM, ORDER, SCHEME, 0>(sg, lx, ly, lz, xi, xs, yi, ys, zi, zs);
  F[1] = window_comp<L, T, V, NDIM, ORDER, SCHEME, 1>(sg, lx, ly, lz, xi, xs, yi, ys, zi, zs);
  F[2] = window_comp<L, T, V, NDIM, ORDER, SCHEME, 2>(sg, lx, ly, lz, xi, xs, yi, ys, zi, zs);
  F[3] = window_comp<L, T, V, NDIM, ORDER, SCHEME, 3>(sg, lx, ly, lz, xi, xs, yi, ys, zi, zs);
  F[4] = window_comp<L, T, V, NDIM, ORDER, SCHEME, 4>(sg, lx, ly, lz, xi, xs, yi, ys, zi, zs);
  F[5] = window_comp<L, T, V, NDIM, ORDER, SCHEME, 5>(sg, lx, ly, lz, xi, xs, yi, ys, zi, zs);
}

// The staged copies made ready for gather_window: averaged from the Yee locations to the nodes for
// the momentum-conserving scheme (node i gets (v[i-1] + v[i]) / 2 along each half-staggered direction, x
// then y then z), and every node stored twice for a paired push. Each thread holds its results in
// registers across a barrier, so the tile is rewritten in place. The lowest node along a staggered
// direction has no neighbour in the tile and keeps its value; no particle of the tile reads it.
template <typename T, int NDIM, int ORDER, int SCHEME>
__device__ __forceinline__ void window_nodes(T* sg) {
  using S = PushSmem<T, NDIM, ORDER, true>;
  constexpr int NT = PushThreads<T, NDIM, ORDER>::value, NE = (6 * S::GN + NT - 1) / NT;
  const int tid = threadIdx.x;
  T v[NE];
#pragma unroll
  for (int m = 0; m < NE; ++m) {
    const int e = tid + m * NT;
    v[m] = T(0);
    if (e >= 6 * S::GN) continue;
    if (SCHEME != 2) {
      v[m] = sg[e];
      continue;
    }
    const int c = e / S::GN, rem = e - c * S::GN;
    const int lz = rem / (S::GX * S::GY), ly = (rem / S::GX) % S::GY, lx = rem % S::GX;
    const int sx = stag_ho(c, 0) && lx > 0 ? 1 : 0;
    const int sy = NDIM == 3 && stag_ho(c, 1) && ly > 0 ? S::GX : 0;
    const int sz = stag_ho(c, 2) && lz > 0 ? S::GX * S::GY : 0;
    const T* p = sg + e;
    auto ax = [&](const T* q) { return sx ? T(0.5) * (q[0] + q[-sx]) : q[0]; };
    auto ay = [&](const T* q) { return sy ? T(0.5) * (ax(q) + ax(q - sy)) : ax(q); };
    v[m] = sz ? T(0.5) * (ay(p) + ay(p - sz)) : ay(p);
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < NE; ++m) {
    const int e = tid + m * NT;
    if (e >= 6 * S::GN) continue;
    sg[e * S::GCOPY] = v[m];
    if (S::GCOPY == 2) sg[e * 2 + 1] = v[m];
  }
  __syncthreads();
}

// One direction of a move d from offset o: the distance am to the upper face and the offset c past it
// (d - am, without the rounding of o + d), whether the particle steps back (`down`) or into the next cell
// (`up`), and its new cell shift and offset; the cases and rounding of esir_dir, without branches (a
// divergent branch costs the FP64 pipe both sides).
template <typename T>
__device__ __forceinline__ void move_one(T x1, T c, bool& down, bool& up, int& sh, T& off) {
  down = is_neg(x1);
  const bool top = !down && ge_one(x1);
  up = top && is_pos(c);
  const T below = T(1) + x1;
  const bool back = down && ge_one(below);  // rounding put it back on this cell's lower face
  off = down ? (back ? T(0) : below) : (top ? (up ? c : T(0)) : x1);
  sh = down ? (back ? 0 : -1) : (top ? 1 : 0);
}
template <typename T>
struct Move1 {
  T am, c, off;
  bool down, up;
  int sh;
  __device__ __forceinline__ Move1(T o, T d) {
    am = T(1) - o;
    c = d - am;
    move_one(o + d, c, down, up, sh, off);
  }
};
// The same for a pair.
struct PairMove {
  float2 am, c;
  Bool2 down, up;
  int sha, shb;
  float offa, offb;
};
__device__ __forceinline__ PairMove pair_move(float2 o, float2 d) {
  PairMove m;
  const float2 x1 = __fadd2_rn(o, d);
  m.am = __fadd2_rn(make_float2(1.f, 1.f), make_float2(-o.x, -o.y));
  m.c = __fadd2_rn(d, make_float2(-m.am.x, -m.am.y));
  move_one(x1.x, m.c.x, m.down.x, m.up.x, m.sha, m.offa);
  move_one(x1.y, m.c.y, m.down.y, m.up.y, m.shb, m.offb);
  return m;
}

// The shapes of a linear move that fits the register window: f = S0 + dS / 2 on the cell's nodes. A
// transverse direction stays in its cell (dS = -d, d); along z, with e0 = am or d (into the next cell or
// not) and e2 = c or 0, the shape changes are -e0, e0 - e2, e2.
template <class L, typename T>
struct LinearZ {
  using V = typename L::V;
  V e0, e1, e2, f0, f1, f2;
  __device__ __forceinline__ LinearZ(V o, V d, V am, V c, typename L::B up) {
    e0 = L::sel(up, am, d);
    e2 = L::sel(up, c, L::set(T(0)));
    e1 = L::add(e0, L::neg(e2));
    f0 = L::fma(L::set(T(-0.5)), e0, am);
    f1 = L::fma(L::set(T(0.5)), e1, o);
    f2 = L::mul(L::set(T(0.5)), e2);
  }
};

// 2D linear deposit into the register layout, one particle or a pair (one accumulator half each). The
// weights are the Esirkepov ones in the form of deposit2; the coefficients of a particle that does not
// fit the register window are zero.
template <class L, typename T, int NVP>
__device__ __forceinline__ void deposit2_lin(typename L::V (&acc)[NVP], typename L::V ox, typename L::V dx,
                                             typename L::V amx, const LinearZ<L, T>& Z, typename L::V cx,
                                             typename L::V cy, typename L::V cz) {
  using V = typename L::V;
  const V fx0 = L::fma(L::set(T(-0.5)), dx, amx), fx1 = L::fma(L::set(T(0.5)), dx, ox);
  const V gx0 = L::neg(L::mul(cx, dx));
  acc[0] = L::fma(gx0, Z.f0, acc[0]);
  acc[1] = L::fma(gx0, Z.f1, acc[1]);
  acc[2] = L::fma(gx0, Z.f2, acc[2]);
  const V gz0 = L::neg(L::mul(cz, Z.e0)), gz1 = L::neg(L::mul(cz, Z.e2));
  acc[3] = L::fma(gz0, fx0, acc[3]);
  acc[4] = L::fma(gz1, fx0, acc[4]);
  acc[5] = L::fma(gz0, fx1, acc[5]);
  acc[6] = L::fma(gz1, fx1, acc[6]);
  const V h0 = L::mul(cy, fx0), h1 = L::mul(cy, fx1);
  const V k1 = L::mul(L::mul(cy, dx), L::set(T(1.0 / 12.0))), k0 = L::neg(k1);
  acc[7] = L::fma(h0, Z.f0, L::fma(k1, Z.e0, acc[7]));  // k0 dS0 = -k1 (-e0)
  acc[8] = L::fma(h1, Z.f0, L::fma(k0, Z.e0, acc[8]));
  acc[9] = L::fma(h0, Z.f1, L::fma(k0, Z.e1, acc[9]));
  acc[10] = L::fma(h1, Z.f1, L::fma(k1, Z.e1, acc[10]));
  acc[11] = L::fma(h0, Z.f2, L::fma(k0, Z.e2, acc[11]));
  acc[12] = L::fma(h1, Z.f2, L::fma(k1, Z.e2, acc[12]));
}

// 3D linear deposit into the register layout (the weights of deposit3): x and y stay in their cell.
template <typename T, int NVP>
__device__ __forceinline__ void deposit3_lin(T (&acc)[NVP], T ox, T dx, T oy, T dy, const LinearZ<Lanes1<T>, T>& Z,
                                             T cx, T cy, T cz) {
  const T fx0 = fma(T(-0.5), dx, T(1) - ox), fx1 = fma(T(0.5), dx, ox);
  const T fy0 = fma(T(-0.5), dy, T(1) - oy), fy1 = fma(T(0.5), dy, oy);
  const T kx = dx * T(1.0 / 12.0), ky = dy * T(1.0 / 12.0);
  const T fz[3] = {Z.f0, Z.f1, Z.f2}, ez[3] = {-Z.e0, Z.e1, Z.e2};
  const T gx = -(cx * dx), gy = -(cy * dy), g0 = -(cz * Z.e0), g1 = -(cz * Z.e2);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const T wy = ky * ez[c], wx = kx * ez[c];
    acc[c * 2 + 0] = fma(gx, fma(fy0, fz[c], -wy), acc[c * 2 + 0]);  // Jx(1/2, b, c)
    acc[c * 2 + 1] = fma(gx, fma(fy1, fz[c], wy), acc[c * 2 + 1]);
    acc[6 + c * 2 + 0] = fma(gy, fma(fx0, fz[c], -wx), acc[6 + c * 2 + 0]);  // Jy(a, 1/2, c)
    acc[6 + c * 2 + 1] = fma(gy, fma(fx1, fz[c], wx), acc[6 + c * 2 + 1]);
  }
  const T w = kx * dy;
  const T t[4] = {fma(fx0, fy0, w), fma(fx1, fy0, -w), fma(fx0, fy1, -w), fma(fx1, fy1, w)};
#pragma unroll
  for (int i = 0; i < 4; ++i) {  // Jz(a, b, c + 1/2), i = b * 2 + a
    acc[12 + 2 * i] = fma(g0, t[i], acc[12 + 2 * i]);
    acc[13 + 2 * i] = fma(g1, t[i], acc[13 + 2 * i]);
  }
}
// A particle outside the register window: its full window, into shared memory.
template <typename T>
__device__ __noinline__ void deposit2_far(T* sj, int lx, int lz, T ox, T oz, T dx, T dz, T cx, T cy, T cz) {
  const EsirDir<T> X = esir_dir(ox, dx), Z = esir_dir(oz, dz);
  deposit2_smem<T, 2>(sj, lx + X.a + 1, lz + Z.a + 1, X, Z, cx, cy, cz);
}
template <typename T>
__device__ __noinline__ void deposit3_far(T* sj, int lx, int ly, int lz, T ox, T oy, T oz, T dx, T dy, T dz, T cx, T cy,
                                          T cz) {
  const EsirDir<T> X = esir_dir(ox, dx), Y = esir_dir(oy, dy), Z = esir_dir(oz, dz);
  deposit3_smem<T, 3>(sj, lx + X.a + 1, ly + Y.a + 1, lz + Z.a + 1, X, Y, Z, cx, cy, cz);
}

// One direction of a cubic Esirkepov move: S0 + dS / 2 and the shape change dS on the nodes -1 .. 3 of
// the start cell for a move d that stays in the cell or enters the next one up (`up`, at offset c
// there), formed from the displacement itself on one polynomial piece (full relative precision for small
// moves) and as the difference across the face. One particle or (Lanes2) a pair.
template <typename V>
struct CubicDir {
  V m[5], dS[5];
};
template <class L, typename T, bool UP>
__device__ __forceinline__ CubicDir<typename L::V> cubic_dir(typename L::V o, typename L::V d, typename L::B up,
                                                             typename L::V c) {
  using V = typename L::V;
  CubicDir<V> r;
  V s[4], e[5];
  cubic_weights<L, T, V>(o, s);
  const V p = L::add(L::set(T(1)), L::neg(o)), d2 = L::mul(d, d), d6 = L::mul(d, L::set(T(1.0 / 6.0)));
  const V three = L::set(T(3));
  const V pd = L::mul(p, L::add(p, L::neg(d))), od = L::mul(o, L::add(o, d));
  e[0] = L::neg(L::mul(d6, L::fma(three, pd, d2)));
  e[3] = L::mul(d6, L::fma(three, od, d2));
  e[1] = L::mul(d, L::fma(L::set(T(1.5)), od, L::fma(L::set(T(-2)), o, L::fma(L::set(T(0.5)), d2, L::neg(d)))));
  e[2] = L::neg(L::add(L::add(e[0], e[1]), e[3]));
  e[4] = L::set(T(0));
  if constexpr (UP) {
    V n[4];
    cubic_weights<L, T, V>(c, n);
    e[0] = L::sel(up, L::neg(s[0]), e[0]);
#pragma unroll
    for (int a = 1; a < 4; ++a) e[a] = L::sel(up, L::add(n[a - 1], L::neg(s[a])), e[a]);
    e[4] = L::sel(up, n[3], e[4]);
  }
#pragma unroll
  for (int a = 0; a < 5; ++a) r.dS[a] = e[a];
#pragma unroll
  for (int a = 0; a < 4; ++a) r.m[a] = L::fma(L::set(T(0.5)), e[a], s[a]);
  r.m[4] = L::mul(L::set(T(0.5)), e[4]);
  return r;
}
// running sums of dS, the weights of the current on the four edges (all five dS sum to zero)
template <class L, typename V>
__device__ __forceinline__ void cubic_run(const CubicDir<V>& r, V (&P)[4]) {
  P[0] = r.dS[0];
  P[1] = L::add(r.dS[0], r.dS[1]);
  P[2] = L::neg(L::add(r.dS[3], r.dS[4]));
  P[3] = L::neg(r.dS[4]);
}

// acc += a b for one particle, or for both of a pair
template <typename T>
__device__ __forceinline__ void add_prod(T& acc, T a, T b) {
  acc += a * b;
}
__device__ __forceinline__ void add_prod(float& acc, float2 a, float2 b) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
}

// 2D cubic deposit into the register layout: x stays in its cell, z stays or steps up (a particle that
// does otherwise comes with zero coefficients).
template <class L, typename T, int NVP, typename V>
__device__ __forceinline__ void deposit2_cubic(T (&acc)[NVP], const CubicDir<V>& X, const CubicDir<V>& Z, V cx, V cy,
                                               V cz) {
  V PX[4], PZ[4];
  cubic_run<L>(X, PX);
  cubic_run<L>(Z, PZ);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const V g = L::mul(cx, PX[a]);
#pragma unroll
    for (int c = 0; c < 5; ++c) add_prod(acc[c * 3 + a], g, Z.m[c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const V g = L::mul(cz, PZ[c]);
#pragma unroll
    for (int a = 0; a < 4; ++a) add_prod(acc[15 + a * 4 + c], g, X.m[a]);
  }
  const V k = L::mul(cy, L::set(T(1.0 / 12.0)));
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const V h = L::mul(cy, X.m[a]), q = L::mul(k, X.dS[a]);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      add_prod(acc[31 + c * 4 + a], h, Z.m[c]);
      add_prod(acc[31 + c * 4 + a], q, Z.dS[c]);
    }
  }
}

// Any cubic move of less than a cell, straight into the tile's current: the window nodes -2 .. 3 of
// the start cell. The rare particles that step back or cross a transverse face take this path.
template <typename T, int NDIM>
__device__ __noinline__ void deposit_general(T* sj, int lx, int ly, int lz, T ox, T oy, T oz, T dx, T dy, T dz, T cx,
                                             T cy, T cz) {
  using S = PushSmem<T, NDIM, 3, true>;
  constexpr int NW = 6;
  T Tx[NW], Ty[NW], Tz[NW], ex[NW], ey[NW], ez[NW];
#pragma unroll 1
  for (int a = 0; a < NW; ++a) {
    const T node = T(a - 2);
    ex[a] = shape_change(3, node - ox, dx);
    Tx[a] = bspl(3, node - ox) + T(0.5) * ex[a];
    ez[a] = shape_change(3, node - oz, dz);
    Tz[a] = bspl(3, node - oz) + T(0.5) * ez[a];
    ey[a] = NDIM == 3 ? shape_change(3, node - oy, dy) : T(0);
    Ty[a] = NDIM == 3 ? bspl(3, node - oy) + T(0.5) * ey[a] : T(0);
  }
  // window node 0 (two below the cell) is current-tile index (lx, ly, lz)
  T* w0 = sj + (lz * S::JY + (NDIM == 3 ? ly : 0)) * S::JX + lx;
  if constexpr (NDIM == 2) {
#pragma unroll 1
    for (int b = 0; b < NW; ++b) {
      T px = T(0), pz = T(0);
#pragma unroll 1
      for (int a = 0; a < NW; ++a) {
        px += ex[a];  // the last running sum closes to zero
        pz += ez[a];
        if (a < NW - 1) {
          const T vx = cx * px * Tz[b], vz = cz * pz * Tx[b];
          if (vx != T(0)) atomicAdd(w0 + b * S::JX + a, vx);
          if (vz != T(0)) atomicAdd(w0 + 2 * S::JN + a * S::JX + b, vz);
        }
        const T vy = cy * (Tx[a] * Tz[b] + ex[a] * ez[b] * T(1.0 / 12.0));
        if (vy != T(0)) atomicAdd(w0 + S::JN + b * S::JX + a, vy);
      }
    }
  } else {
#pragma unroll 1
    for (int t2 = 0; t2 < NW; ++t2)
#pragma unroll 1
      for (int t1 = 0; t1 < NW; ++t1) {
        const T gx = Ty[t1] * Tz[t2] + ey[t1] * ez[t2] * T(1.0 / 12.0);  // Jx: (y, z) = (t1, t2)
        const T gy = Tx[t1] * Tz[t2] + ex[t1] * ez[t2] * T(1.0 / 12.0);  // Jy: (x, z) = (t1, t2)
        const T gz = Tx[t1] * Ty[t2] + ex[t1] * ey[t2] * T(1.0 / 12.0);  // Jz: (x, y) = (t1, t2)
        T px = T(0), py = T(0), pz = T(0);
#pragma unroll 1
        for (int a = 0; a < NW - 1; ++a) {
          px += ex[a];
          py += ey[a];
          pz += ez[a];
          const T vx = cx * px * gx, vy = cy * py * gy, vz = cz * pz * gz;
          if (vx != T(0)) atomicAdd(w0 + (t2 * S::JY + t1) * S::JX + a, vx);
          if (vy != T(0)) atomicAdd(w0 + S::JN + (t2 * S::JY + a) * S::JX + t1, vy);
          if (vz != T(0)) atomicAdd(w0 + 2 * S::JN + (a * S::JY + t2) * S::JX + t1, vz);
        }
      }
  }
}

// The same in 2D for the n particles that an item of the paired push has queued (`far`: their slots in the
// stage, which holds offsets, displacements, v_y and charge), eight lanes per particle: lane a forms the
// shapes of window node a of both directions, and the lanes add a row of nodes at a time, to addresses of
// their own. Few particles of a beam come here, but every eighth of a hot load: 2.1M of u_th = 1 at gamma
// = 3 on 256x512 cells, a step 998 us with deposit_general called by the lane or two of a round that have one
// (646 us when a warp took a cell), 419 us so.
inline __device__ __noinline__ void deposit_queue(float* sj, const float* sq, const float* sr, const float* sw,
                                                  const unsigned char* far, int n, int cell0, int per_cell, float jfx,
                                                  float jfy, float jfz) {
  using S = PushSmem<float, 2, 3, true>;
  const int lane = threadIdx.x & 31, a = lane & 7;
#pragma unroll 1
  for (int f0 = 0; f0 < n; f0 += 4) {
    const bool on = f0 + (lane >> 3) < n && a < 6;
    const int e = far[min(f0 + (lane >> 3), n - 1)], cl = cell0 + e / per_cell;
    float q[4];
    ld4(sq + 4 * e, q);
    const float w = on ? sw[e] : 0.f, node = (float)(a - 2);
    const float ex = on ? shape_change(3, node - q[0], q[2]) : 0.f, ez = on ? shape_change(3, node - q[1], q[3]) : 0.f;
    const float Tx = on ? bspl(3, node - q[0]) + 0.5f * ex : 0.f, Tz = on ? bspl(3, node - q[1]) + 0.5f * ez : 0.f;
    float px = ex, pz = ez;  // running sums; the last closes to zero
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const float tx = __shfl_up_sync(0xffffffffu, px, o, 8), tz = __shfl_up_sync(0xffffffffu, pz, o, 8);
      if (a >= o) {
        px += tx;
        pz += tz;
      }
    }
    if (a >= 5) px = pz = 0.f;
    const float vx = w * jfx * px, vz = w * jfz * Tx, cy = w * sr[e] * jfy, vy = cy * Tx, ky = cy * ex * (1.f / 12.f);
    // window node 0 (two below the cell) is current-tile index of the cell itself
    float* j = sj + (cl / S::TX) * S::JX + cl % S::TX + a;
#pragma unroll
    for (int b = 0; b < 6; ++b) {
      const float Tb = __shfl_sync(0xffffffffu, Tz, b, 8), eb = __shfl_sync(0xffffffffu, ez, b, 8);
      const float pb = __shfl_sync(0xffffffffu, pz, b, 8);
      const float v0 = vx * Tb, v1 = fmaf(vy, Tb, ky * eb), v2 = vz * pb;
      if (v0 != 0.f) atomicAdd(j + b * S::JX, v0);
      if (v1 != 0.f) atomicAdd(j + S::JN + b * S::JX, v1);
      if (v2 != 0.f) atomicAdd(j + 2 * S::JN + b * S::JX, v2);
    }
  }
}

// 3D cubic deposit of one item and one component (0 Jx, 1 Jy, 2 Jz). The window of all components has 184
// sums, more than a thread can hold beside the push, so the push leaves each particle's offsets,
// displacements and charge (zero: nothing to add) in its stage slot and the three components are summed
// one after another, 60 to 64 sums at a time, over the lane's particles of the item, then over the
// cell's lanes. Positions: x and y stay in their cell, z stays or steps up. Layouts: Jx (c*4 + b)*3 + a,
// Jy (c*4 + a)*3 + b, Jz (b*4 + a)*4 + c, on nodes from one below the cell (origin `j`).
template <typename T, int LPC, int COMP>
__device__ __forceinline__ void deposit3_cubic(const T* stq, const T* str, const T* stw, int sl, int nrnd, int rnd0,
                                               T coef, T* j) {
  using S = PushSmem<T, 3, 3, true>;
  constexpr int NV = COMP == 2 ? 64 : 60, PER = (NV + LPC - 1) / LPC, NVP = PER * LPC;
  const int lane = threadIdx.x & 31;
  T acc[NVP];
#pragma unroll
  for (int i = 0; i < NVP; ++i) acc[i] = T(0);
#pragma unroll 1
  for (int rnd = 0; rnd < nrnd; ++rnd) {
    const int k = sl + LPC * ((rnd + rnd0) & 3);
    T q[4], e[2];
    ld4(stq + 4 * k, q);
    ld2(str + 2 * k, e);
    const T ox = q[0], oy = q[1], oz = q[2], dx = q[3], dy = e[0], dz = e[1], qw = coef * stw[k];
    const T c = dz - (T(1) - oz);
    using L1 = Lanes1<T>;
    const CubicDir<T> X = cubic_dir<L1, T, false>(ox, dx, false, T(0)), Y = cubic_dir<L1, T, false>(oy, dy, false, T(0));
    const CubicDir<T> Z = cubic_dir<L1, T, true>(oz, dz, ge_one(oz + dz) && is_pos(c), c);
    const CubicDir<T>& A = COMP == 0 ? X : (COMP == 1 ? Y : Z);  // along the component
    const CubicDir<T>& B = COMP == 0 ? Y : X;                    // the fast transverse direction
    const CubicDir<T>& C = COMP == 2 ? Y : Z;                    // the slow one (Z: five nodes)
    constexpr int NA = COMP == 2 ? 4 : 3, NC = COMP == 2 ? 4 : 5;
    T P[4];
    cubic_run<L1>(A, P);
#pragma unroll
    for (int a = 0; a < NA; ++a) P[a] *= qw;
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const T t = B.m[b] * C.m[k] + B.dS[b] * T(1.0 / 12.0) * C.dS[k];
#pragma unroll
        for (int a = 0; a < NA; ++a) acc[(k * 4 + b) * NA + a] += P[a] * t;
      }
  }
#pragma unroll
  for (int sh = LPC / 2; sh >= 1; sh >>= 1) {
    const bool up = (lane & sh) != 0;
#pragma unroll
    for (int i = 0; i < PER * sh; ++i) {
      const T send = up ? acc[i] : acc[i + PER * sh];
      const T keep = up ? acc[i + PER * sh] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
    }
  }
#pragma unroll
  for (int m = 0; m < PER; ++m) {
    const int i = sl * PER + m;
    if (i >= NV || acc[m] == T(0)) continue;
    int a, b, c;
    if (COMP == 2) { c = i & 3; a = (i >> 2) & 3; b = i >> 4; }
    else if (COMP == 1) { const int k = i / 3; b = i - 3 * k; a = k & 3; c = k >> 2; }
    else { const int k = i / 3; a = i - 3 * k; b = k & 3; c = k >> 2; }
    atomicAdd(j + COMP * S::JN + (c * S::JY + b) * S::JX + a, acc[m]);
  }
}

template <typename T, int NDIM, int SCHEME, int LPC, int ORDER = 1>
__device__ __forceinline__ void push_tile(const RunDev<T>& r, const int tile) {
  constexpr bool WIN = ORDER == 3 || SCHEME == 2;    // the gather reads the cell's window of nodes
  constexpr bool LATE = NDIM == 3 && ORDER == 3;     // the deposit follows the push of each item
  constexpr bool QUEUE = PushPaired<T, NDIM>::value && ORDER == 3;  // so do the far deposits
  constexpr bool CROWD = PushCrowd<T, NDIM, ORDER, WIN>::value;     // crowded cells apart from their group
  using S = PushSmem<T, NDIM, ORDER, WIN>;
  using PL = PushPlan<NDIM, LPC, ORDER>;
  constexpr int TX = S::TX, TY = S::TY, NCL = S::NCL;
  constexpr int NV = PL::NV, PER = PL::PER, NVP = PL::NVP, CPW = PL::CPW;
  constexpr int PUSH_THREADS = PushThreads<T, NDIM, ORDER>::value, NWARP = PUSH_THREADS / 32;
  static_assert(NCL % CPW == 0, "cells per tile must be a multiple of the cells per warp");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sg = reinterpret_cast<T*>(smem_raw);
  T* sj = sg + 6 * S::GN * S::GCOPY;
  int* sn = reinterpret_cast<int*>(sj + 3 * S::JN);  // [species][cell] particle counts (input)
  int* scnt = sn + 2 * NCL;                          // [species][cell] output counts of this tile

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // per-warp stages start on a 16-byte boundary after the counts (cp.async destinations)
  const size_t stage_off = ((size_t)(reinterpret_cast<unsigned char*>(scnt + 2 * NCL) - smem_raw) + 15) & ~(size_t)15;
  using SG = PushStage<T, NDIM>;
  T* stg = reinterpret_cast<T*>(smem_raw + stage_off) + (size_t)warp * SG::per_warp_elems();
  // the tile's leaver buffer follows every warp's stage
  const size_t lv_off = (stage_off + sizeof(T) * SG::per_warp_elems() * NWARP + 15) & ~(size_t)15;
  T* lvv = reinterpret_cast<T*>(smem_raw + lv_off);
  int* lvk = reinterpret_cast<int*>(lvv + 7 * S::LVB);
  unsigned* lvi = reinterpret_cast<unsigned*>(lvk + S::LVB);
  int* lvn = reinterpret_cast<int*>(lvi + S::LVB);
  const int tix = tile % r.ntx;
  const int tiy = (tile / r.ntx) % r.nty;
  const int tiz = tile / (r.ntx * r.nty);
  // the run's tile extents (r.tex <= TX ...): cells past them stay empty, as at the grid's edge
  const int X0 = tix * r.tex, Y0 = tiy * r.tey, Z0 = tiz * r.tez;
  const int wx = min(r.tex, r.nx - X0), wy = min(r.tey, r.ny - Y0), wz = min(r.tez, r.nz - Z0);
  const long long nxy = (long long)r.nx * r.ny;

  const bool has_w = r.in[0].w != nullptr;
  const bool has_id = r.in[0].id != nullptr;
  const int sl = lane % LPC;  // lane within its cell group

  // 1. field copies of the tile and its halo into shared memory (periodic wrap); zero the current
  const bool near_ok = r.nx >= S::GX && r.nz >= S::GZ && (NDIM == 2 || r.ny >= S::GY);
  // global index of node (lx, ly, lz) of a tile region that starts H nodes below the tile (cells < 2^30);
  // it lies within one period of the grid when the grid is at least as wide as the region
  auto node_at = [&](int lx, int ly, int lz) -> int {
    const int gx = X0 - S::H + lx, gy = Y0 - S::H + ly, gz = Z0 - S::H + lz;
    const int kx = near_ok ? wrap_near_p(gx, r.nx) : wrapi(gx, r.nx);
    const int ky = NDIM == 3 ? (near_ok ? wrap_near_p(gy, r.ny) : wrapi(gy, r.ny)) : 0;
    const int kz = near_ok ? wrap_near_p(gz, r.nz) : wrapi(gz, r.nz);
    return (kz * r.ny + ky) * r.nx + kx;
  };
  // the planes this tile uses (wz of TZ), one index computation per node for all components: a step of
  // an empty 512x1024 FP32 grid, which is these prologues and epilogues alone, took 47 us with one per
  // component and node
  const int gn = S::GX * S::GY * (wz + 2 * S::H), jn = S::JX * S::JY * (wz + 2 * S::H + 1);
  const int ncl = TX * TY * wz;
  const int ngrp = (ncl + CPW - 1) / CPW;  // cell groups of the tile
  for (int e = tid; e < gn; e += PUSH_THREADS) {
    const int o = node_at(e % S::GX, (e / S::GX) % S::GY, e / (S::GX * S::GY));
#pragma unroll
    for (int c = 0; c < 6; ++c) copy1_async(sg + c * S::GN + e, r.g[c] + o);
  }
  for (int e = tid; e < jn; e += PUSH_THREADS) {
#pragma unroll
    for (int c = 0; c < 3; ++c) sj[c * S::JN + e] = T(0);
  }
  // 2. particle counts of the tile's cells, copied in the same asynchronous batch as the fields (one
  // global round trip for both); then clamped, and the input counts zeroed (they are the next
  // step's output counts). Each thread reads back only the counts it copied itself.
  for (int cl = tid; cl < ngrp * CPW; cl += PUSH_THREADS) {
    const int lx = cl % TX, ly = (cl / TX) % TY, lz = cl / (TX * TY);
    if (lx < wx && ly < wy && lz < wz) {
      const long long cell = (long long)(Z0 + lz) * nxy + (long long)(Y0 + ly) * r.nx + X0 + lx;
      copy1_async(sn + cl, r.in[0].cnt + cell);
      copy1_async(sn + NCL + cl, r.in[1].cnt + cell);
    } else {
      sn[cl] = 0;
      sn[NCL + cl] = 0;
    }
    scnt[cl] = 0;
    scnt[NCL + cl] = 0;
  }
  // One item into a stage: slots [4 it LPC, 4 (it + 1) LPC) of the packs of the lane's cell, whose bin
  // starts at slot bin0 and holds nq0 packs of species 0 of nq in all. The q values go slot by slot over
  // the cell's lanes (neighbouring lanes copy neighbouring slots), the rest one pack per lane. fix: only
  // the packs of species 1.
  auto copy_item = [&](long long bin0, int it, int nq0, int nq, int stage, bool fix) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = j * LPC + sl, pk = it * LPC + (k >> 2);
      if (pk >= nq || (fix && pk < nq0)) continue;
      const bool s1 = pk >= nq0;
      const long long slot = bin0 + 4 * (s1 ? pk - nq0 : pk) + (k & 3);
      copy_async<4 * sizeof(T)>(SG::q(stg, stage, lane - sl) + 4 * k, (s1 ? r.in[1].q : r.in[0].q) + 4 * slot);
    }
    const int pk = it * LPC + sl;
    if (pk >= nq || (fix && pk < nq0)) return;
    const bool s1 = pk >= nq0;
    const long long slot = bin0 + 4 * (s1 ? pk - nq0 : pk);
    copy_async<4 * SG::RW * sizeof(T)>(SG::r(stg, stage, lane), (s1 ? r.in[1].r : r.in[0].r) + SG::RW * slot);
    if (has_w) copy_async<4 * sizeof(T)>(SG::w(stg, stage, lane), (s1 ? r.in[1].w : r.in[0].w) + slot);
    if (has_id) copy_async<16>(SG::id(stg, stage, lane), (s1 ? r.in[1].id : r.in[0].id) + slot);
  };
  // The first item of the warp's first cell group, in the same batch although the counts are not in
  // yet: packs of species 0 only, as the item holds whenever its cell has that many (slots below cap, a
  // multiple of 4: inside the cell's own bin). Its packs of species 1 are copied once the counts are known.
  {
    const int c = warp * CPW + lane / LPC;  // every warp has a first group (NCL / CPW >= NWARP)
    const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
    if (lx < wx && ly < wy && lz < wz)
      copy_item(((long long)(Z0 + lz) * nxy + (long long)(Y0 + ly) * r.nx + X0 + lx) * r.cap, 0, r.cap >> 2, r.cap >> 2, 0,
                false);
  }
  static_assert(NCL / CPW >= NWARP, "every warp needs a first cell group");
  cp_async_commit();
  cp_async_wait_all();
  int npush = 0;  // particles of the cells whose counts this thread reads (cubic 3D: that it pushes)
  for (int cl = tid; cl < ncl; cl += PUSH_THREADS) {
    const int lx = cl % TX, ly = (cl / TX) % TY, lz = cl / (TX * TY);
    if (lx < wx && ly < wy && lz < wz) {
      const long long cell = (long long)(Z0 + lz) * nxy + (long long)(Y0 + ly) * r.nx + X0 + lx;
      const int m0 = min(sn[cl], r.cap), m1 = min(sn[NCL + cl], r.cap);  // the excess of a full bin waits in the spill list
      sn[cl] = m0;
      sn[NCL + cl] = m1;
      if (!LATE) npush += m0 + m1;
      r.in[0].cnt[cell] = 0;
      r.in[1].cnt[cell] = 0;
    }
  }
  // cell groups after each warp's first one are handed out in the order warps ask for them, so
  // warps whose groups hold more packs do fewer groups
  __shared__ int s_next_group;
  // per warp: the slots of the present item whose deposit leaves the register window
  __shared__ unsigned char s_far[QUEUE ? NWARP : 1][QUEUE ? 128 : 1];
  if (tid == 0) {
    *lvn = 0;
    s_next_group = PUSH_THREADS / 32;
  }
  __syncthreads();
  if constexpr (SCHEME == 2 || S::GCOPY == 2) window_nodes<T, NDIM, ORDER, SCHEME>(sg);

  T kin = T(0);
  // current per particle of the uniform weight and unit W (2D Jy: and unit v_y)
  const T cwx = r.wconst * r.jfx, cwy = r.wconst * (NDIM == 3 ? r.jfy : r.jfy2d), cwz = r.wconst * r.jfz;

  // Items of this warp: (cell group, pack round). The packs of the next item are copied into the
  // warp's shared-memory stage with cp.async while the current item is computed.
  // A job is the cells of a group, or (CROWD) one crowded cell of it, whose place in the group is `one` (else
  // -1); crowd: the lanes of the group's crowded cells.
  auto group_iters = [&](int g, unsigned& crowd) -> int {
    const int c = g * CPW + lane / LPC;
    const int nq = ((sn[c] + 3) >> 2) + ((sn[NCL + c] + 3) >> 2);
    crowd = 0;
    if constexpr (CROWD) {
      const int most = __reduce_max_sync(0xffffffffu, nq);
      if (most > 8 * LPC) {  // twice the group's mean and eight items more
        const int mean = __reduce_add_sync(0xffffffffu, nq) >> 5;
        crowd = __ballot_sync(0xffffffffu, nq > 2 * mean + 8 * LPC);
        return __reduce_max_sync(0xffffffffu, crowd >> lane & 1u ? 0 : (nq + LPC - 1) / LPC);
      }
      return (most + LPC - 1) / LPC;
    }
    return __reduce_max_sync(0xffffffffu, (nq + LPC - 1) / LPC);
  };
  // The lane's cell and the counts that the job takes of it; returns which LPC packs of it are the lane's.
  auto lane_cell = [&](int g, int it, int one, unsigned crowd, int& c, int& n0, int& n1) -> int {
    c = g * CPW + (one >= 0 ? one : lane / LPC);
    n0 = sn[c];
    n1 = sn[NCL + c];
    if (CROWD && one < 0 && crowd >> lane & 1u) n0 = n1 = 0;
    return one >= 0 ? it * CPW + lane / LPC : it;
  };
  auto issue = [&](int g, int it, int one, unsigned crowd, int stage, bool fix) {
    int c, n0, n1;
    const int itl = lane_cell(g, it, one, crowd, c, n0, n1);
    const int nq0 = (n0 + 3) >> 2, nq = nq0 + ((n1 + 3) >> 2);
    const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
    copy_item(((long long)(Z0 + lz) * nxy + (long long)(Y0 + ly) * r.nx + X0 + lx) * r.cap, itl, nq0, nq, stage, fix);
  };

  auto take_group = [&]() -> int {
    int v = 0;
    if (lane == 0) v = atomicAdd(&s_next_group, 1);
    return __shfl_sync(0xffffffffu, v, 0);
  };
  int g = warp, it = 0, one = -1, giters = 0;
  unsigned crowd = 0, left = 0;  // the group's crowded cells: their lanes, and those still to be taken (a lane each)
  const unsigned heads = CROWD ? __ballot_sync(0xffffffffu, sl == 0) : 0u;
  // The next job after group g's: its next crowded cell, or another group's cells.
  auto next_job = [&](int& g, int& one, int& giters, unsigned& crowd, unsigned& left, bool first) {
    for (;;) {
      if (CROWD && left != 0) {
        one = (__ffs(left) - 1) / LPC;
        left &= left - 1;
        const int c = g * CPW + one;
        giters = (((sn[c] + 3) >> 2) + ((sn[NCL + c] + 3) >> 2) + 31) >> 5;
        return;
      }
      if (!first) g = take_group();
      first = false;
      one = -1;
      giters = g < ngrp ? group_iters(g, crowd) : 0;
      if (CROWD) left = g < ngrp ? crowd & heads : 0u;
      if (g >= ngrp || giters > 0) return;
    }
  };
  next_job(g, one, giters, crowd, left, true);
  int stage = 0;
  // the first group's first item was copied speculatively
  if (g < ngrp) issue(g, 0, one, crowd, 0, g == warp && one < 0);
  cp_async_commit();
  // the register sums; a linear paired push keeps one half per particle of the pair until the group's end
  constexpr bool ACC2 = PushPaired<T, NDIM>::value && ORDER == 1;
  T acc[NVP];
  float2 acc2[ACC2 ? NVP : 1];
  GalCache<T, NDIM> gc;  // Galerkin nodes of the lane's cell, loaded once per cell group
  while (g < ngrp) {
    // prefetch the next item
    int ng = g, nit = it + 1, niters = giters, none = one;
    unsigned ncrowd = crowd;
    if (nit >= giters) {
      nit = 0;
      next_job(ng, none, niters, ncrowd, left, false);
    }
    if (ng < ngrp) issue(ng, nit, none, ncrowd, stage ^ 1, false);
    cp_async_commit();
    cp_async_wait_1();
    __syncwarp();

    int cl, n0, n1;
    const int itl = lane_cell(g, it, one, crowd, cl, n0, n1);
    const int nq0 = (n0 + 3) >> 2, nq = nq0 + ((n1 + 3) >> 2);
    // the lanes of an empty cell stand in a cell that holds particles: a pair's empty slots go through the
    // arithmetic, and an empty cell's fields may be anything (not finite, or past the tile's last plane not staged)
    if constexpr (PushPaired<T, NDIM>::value) {
      const unsigned live = __ballot_sync(0xffffffffu, nq > 0);
      if (nq == 0) cl = g * CPW + (__ffs(live) - 1) / LPC;
    }
    const int lx = cl % TX, ly = (cl / TX) % TY, lz = min(cl / (TX * TY), wz - 1);
    const int gi = X0 + lx, gj = Y0 + ly, gk = Z0 + lz;
    const int okey = ((lz + 1) * S::JY + (NDIM == 3 ? ly + 1 : 0)) * S::JX + lx + 1;  // cell-origin window
    if (it == 0) {
      if (SCHEME == 0 && !WIN) gc.load(sg, lx, ly, lz);
#pragma unroll
      for (int i = 0; i < NVP; ++i) acc[i] = T(0);
#pragma unroll
      for (int i = 0; i < (ACC2 ? NVP : 1); ++i) acc2[i] = make_float2(0.f, 0.f);
    }
    // rounds of this item: up to the last slot in use of the fullest cell
    constexpr int NR = PushRounds<T, NDIM>::value, U = 4 / NR;
    int nk = 4 * (nq - itl * LPC);  // slots of the cell's packs from this item on, then the last pack's empty ones
    if (nk > 0 && nk <= 4 * LPC) nk -= 4 * (nq > nq0 ? nq - nq0 : nq0) - (nq > nq0 ? n1 : n0);
    const int nrnd = min(NR, (__reduce_max_sync(0xffffffffu, nk) + U * LPC - 1) / (U * LPC));
    const int win0 = U == 2 || nrnd == NR ? PL::first_window(lane / LPC) : 0;
    const T* stq = SG::q(stg, stage, lane - sl);  // slot k of the cell: stq[4 k], str[RW k], stw[k], sti[k]
    const T* str = SG::r(stg, stage, lane - sl);
    const T* stw = SG::w(stg, stage, lane - sl);
    const unsigned* sti = SG::id(stg, stage, lane - sl);
    // whether slot k of the cell's 4 LPC holds a particle, and its species
    const int k1 = 4 * (nq0 - itl * LPC), end0 = n0 - 4 * itl * LPC, end1 = n1 + k1;
    auto slot_of = [&](int k, int& s) -> bool {
      if constexpr (LATE) {  // the cubic 3D push is 2 % slower with the shorter form
        const int q = itl * LPC + (k >> 2);
        s = q >= nq0 ? 1 : 0;
        return q < nq && (s ? n1 + 4 * nq0 : n0) > 4 * q + (k & 3);
      }
      s = k >= k1 ? 1 : 0;
      return k < (s ? end1 : end0);
    };
    int nfar = 0;
#pragma unroll 1
    for (int rnd = 0; rnd < nrnd; ++rnd) {
      if constexpr (PushPaired<T, NDIM>::value) {
        const float2 u02 = make_float2(r.u0, r.u0), one2 = make_float2(1.f, 1.f);
        const float2 dtdx2 = make_float2(r.dtdx, r.dtdx), dtdz2 = make_float2(r.dtdz, r.dtdz);
        const unsigned lt = (1u << lane) - 1u;
        {
          // the pair: the lane's slots in two windows
          const int ka = sl + LPC * ((win0 + 2 * rnd) & (2 * nrnd - 1));
          const int kb = sl + LPC * ((win0 + 2 * rnd + 1) & (2 * nrnd - 1));
          int s_a, s_b;
          const bool va = slot_of(ka, s_a), vb = slot_of(kb, s_b);
          const float2 hh = make_float2(s_a ? r.hq : -r.hq, s_b ? r.hq : -r.hq);
          float qa[4], qb[4];
          ld4(stq + 4 * ka, qa);
          ld4(stq + 4 * kb, qb);
          // an empty slot stands in as a particle at rest with no weight (finite, deposits nothing)
          const float oxa = va ? qa[0] : 0.5f, oza = va ? qa[1] : 0.5f;
          const float uxa = va ? qa[2] : 0.f, uya = va ? qa[3] : 0.f, uza = va ? str[ka] : 0.f;
          const float oxb = vb ? qb[0] : 0.5f, ozb = vb ? qb[1] : 0.5f;
          const float uxb = vb ? qb[2] : 0.f, uyb = vb ? qb[3] : 0.f, uzb = vb ? str[kb] : 0.f;
          const float wa = va ? (has_w ? stw[ka] : r.wconst) : 0.f, wb = vb ? (has_w ? stw[kb] : r.wconst) : 0.f;
          // gather
          float2 F2[6];
          float Fa[6], Fb[6];
          if constexpr (WIN) {
            gather_window<Lanes2, float, float2, 2, ORDER, SCHEME>(sg, lx, 0, lz, make_float2(oxa, oxb), make_float2(0.f, 0.f),
                                                                   make_float2(oza, ozb), F2);
          } else if (SCHEME == 0) {
            gc.interp(oxa, 0.f, oza, Fa);
            gc.interp(oxb, 0.f, ozb, Fb);
          } else {
            const DirW<float> xa = dir_weights(oxa), za = dir_weights(oza), xb = dir_weights(oxb),
                              zb = dir_weights(ozb), y0 = dir_weights(0.f);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              Fa[c] = gather_comp<float, 2, SCHEME>(sg + c * S::GN, c, lx, 0, lz, xa, y0, za);
              Fb[c] = gather_comp<float, 2, SCHEME>(sg + c * S::GN, c, lx, 0, lz, xb, y0, zb);
            }
          }
          if constexpr (!WIN) {
#pragma unroll
            for (int c = 0; c < 6; ++c) F2[c] = make_float2(Fa[c], Fb[c]);
          }
          const float2 Ex = F2[0], Ey = F2[1], Ez = F2[2], Bx = F2[3], By = F2[4], Bz = F2[5];
          // relativistic Boris of the pair, momenta relative to the drift u0 z_hat
          const float2 mx = fma2(hh, Ex, make_float2(uxa, uxb));
          const float2 my = fma2(hh, Ey, make_float2(uya, uyb));
          const float2 mz = fma2(hh, Ez, make_float2(uza, uzb));
          const float2 Mz = add2(u02, mz);
          float2 m2 = fma2(mx, mx, one2);
          m2 = fma2(my, my, m2);
          m2 = fma2(Mz, Mz, m2);
          const float2 hig = mul2(hh, WIN ? fine_rsqrt(m2) : make_float2(fast_rsqrt(m2.x), fast_rsqrt(m2.y)));
          const float2 tx = mul2(hig, Bx), ty = mul2(hig, By), tz = mul2(hig, Bz);
          float2 t2 = fma2(tx, tx, one2);
          t2 = fma2(ty, ty, t2);
          t2 = fma2(tz, tz, t2);
          const float2 sf = WIN ? fine_two_over(t2) : make_float2(two_over(t2.x), two_over(t2.y));
          const float2 sx = mul2(sf, tx), sy = mul2(sf, ty), sz = mul2(sf, tz);
          const float2 qx = fma2(my, tz, fma2(neg2(Mz), ty, mx));
          const float2 qy = fma2(Mz, tx, fma2(neg2(mx), tz, my));
          const float2 qz = fma2(mx, ty, fma2(neg2(my), tx, Mz));
          const float2 ux2 = fma2(qy, sz, fma2(neg2(qz), sy, fma2(hh, Ex, mx)));
          const float2 uy2 = fma2(qz, sx, fma2(neg2(qx), sz, fma2(hh, Ey, my)));
          const float2 uz2 = fma2(qx, sy, fma2(neg2(qy), sx, fma2(hh, Ez, mz)));
          const float2 Uz = add2(u02, uz2);
          float2 u2 = mul2(ux2, ux2);
          u2 = fma2(uy2, uy2, u2);
          u2 = fma2(Uz, Uz, u2);
          const float2 gp = add2(one2, u2);
          const float2 ign = WIN ? fine_rsqrt(gp) : make_float2(fast_rsqrt(gp.x), fast_rsqrt(gp.y));
          if (r.kin) {  // gamma - 1 = u^2 / (gamma + 1)
            const float2 g1 = fma2(gp, ign, one2);
            const float2 k = WIN ? fine_kinetic(u2, gp, ign) : make_float2(fast_div(u2.x, g1.x), fast_div(u2.y, g1.y));
            kin = fmaf(wa, k.x, kin);
            kin = fmaf(wb, k.y, kin);
          }
          const float2 vy2 = mul2(uy2, ign);
          const float2 ddx2 = mul2(dtdx2, mul2(ux2, ign)), ddz2 = mul2(dtdz2, mul2(Uz, ign));
          float dxa = ddx2.x, dza = ddz2.x, dxb = ddx2.y, dzb = ddz2.y;
          float nuxa = ux2.x, nuya = uy2.x, nuza = uz2.x, vya = vy2.x;
          float nuxb = ux2.y, nuyb = uy2.y, nuzb = uz2.y, vyb = vy2.y;
          if (!(dxa > -1.f && dxa < 1.f && dza > -1.f && dza < 1.f)) {
            flag_error(r.err, ERR_NONFINITE);
            dxa = dza = nuxa = nuya = nuza = vya = 0.f;
          }
          if (!(dxb > -1.f && dxb < 1.f && dzb > -1.f && dzb < 1.f)) {
            flag_error(r.err, ERR_NONFINITE);
            dxb = dzb = nuxb = nuyb = nuzb = vyb = 0.f;
          }
          // Esirkepov deposits: in registers where the window fits (RegLayout), the coefficients zero
          // otherwise, and the rest (a step back or across an x face) to shared memory
          const float2 o_x = make_float2(oxa, oxb), o_z = make_float2(oza, ozb);
          const float2 d_x = make_float2(dxa, dxb), d_z = make_float2(dza, dzb);
          const PairMove X = pair_move(o_x, d_x), Z = pair_move(o_z, d_z);
          const bool rega = !(X.down.x || X.up.x || Z.down.x), regb = !(X.down.y || X.up.y || Z.down.y);
          const float2 qw = make_float2(s_a ? wa : -wa, s_b ? wb : -wb);
          const float2 qr = make_float2(rega ? qw.x : 0.f, regb ? qw.y : 0.f);
          const float2 jx2 = make_float2(r.jfx, r.jfx), jy2 = make_float2(r.jfy2d, r.jfy2d), jz2 = make_float2(r.jfz, r.jfz);
          const float2 vyp = make_float2(vya, vyb);
          if constexpr (ORDER == 3)
            deposit2_cubic<Lanes2, float, NVP, float2>(acc, cubic_dir<Lanes2, float, false>(o_x, d_x, Bool2{}, o_x),
                                                       cubic_dir<Lanes2, float, true>(o_z, d_z, Z.up, Z.c), mul2(qr, jx2),
                                                       mul2(mul2(qr, vyp), jy2), mul2(qr, jz2));
          else
            deposit2_lin<Lanes2, float, NVP>(acc2, o_x, d_x, X.am, LinearZ<Lanes2, float>(o_z, d_z, Z.am, Z.c, Z.up),
                                             mul2(qr, jx2), mul2(mul2(qr, vyp), jy2), mul2(qr, jz2));
          if constexpr (QUEUE) {
            if (__any_sync(0xffffffffu, (!rega && va) || (!regb && vb))) {
              // into the stage: displacements, v_y and charge of the slot
              auto queue = [&](bool far, int k, float dx, float dz, float vy, float w) {
                const unsigned m = __ballot_sync(0xffffffffu, far);
                if (far) {
                  const_cast<float*>(stq)[4 * k + 2] = dx;
                  const_cast<float*>(stq)[4 * k + 3] = dz;
                  const_cast<float*>(str)[k] = vy;
                  const_cast<float*>(stw)[k] = w;
                  s_far[warp][nfar + __popc(m & lt)] = (unsigned char)((lane - sl) * 4 + k);
                }
                nfar += __popc(m);
              };
              queue(!rega && va, ka, dxa, dza, vya, qw.x);
              queue(!regb && vb, kb, dxb, dzb, vyb, qw.y);
            }
          } else {
            if (!rega && va) deposit2_far(sj, lx, lz, oxa, oza, dxa, dza, qw.x * r.jfx, qw.x * vya * r.jfy2d, qw.x * r.jfz);
            if (!regb && vb) deposit2_far(sj, lx, lz, oxb, ozb, dxb, dzb, qw.y * r.jfx, qw.y * vyb * r.jfy2d, qw.y * r.jfz);
          }
          // destinations: a cell of this tile (key (cell * 2 + species) in the tile) or, leaving
          // the tile, the global cell (key global cell * 2 + species)
          int dka = -1 - lane, dkb = -1 - lane;
          bool lva = false, lvb = false;
          if (va) {
            const int nlx = lx + X.sha, nlz = lz + Z.sha;
            if (nlx >= 0 && nlx < wx && nlz >= 0 && nlz < wz) {
              dka = (nlz * TX + nlx) * 2 + s_a;
            } else {
              lva = true;
              dka = (wrap_near_p(gk + Z.sha, r.nz) * r.nx + wrap_near_p(gi + X.sha, r.nx)) * 2 + s_a;
            }
          }
          if (vb) {
            const int nlx = lx + X.shb, nlz = lz + Z.shb;
            if (nlx >= 0 && nlx < wx && nlz >= 0 && nlz < wz) {
              dkb = (nlz * TX + nlx) * 2 + s_b;
            } else {
              lvb = true;
              dkb = (wrap_near_p(gk + Z.shb, r.nz) * r.nx + wrap_near_p(gi + X.shb, r.nx)) * 2 + s_b;
            }
          }
          // rebin of the pair: consecutive slots per (destination, species) for each particle of the
          // pair, the two reservations interleaved
          const bool sta = va && !lva, stb = vb && !lvb;
          const unsigned pa = __match_any_sync(0xffffffffu, sta ? dka : -1 - lane);
          const unsigned pb = __match_any_sync(0xffffffffu, stb ? dkb : -1 - lane);
          const int lda = __ffs(pa) - 1, ldb = __ffs(pb) - 1;
          int ba = 0, bb = 0;
          if (sta && lane == lda) ba = atomicAdd(scnt + (dka & 1) * NCL + (dka >> 1), __popc(pa));
          if (stb && lane == ldb) bb = atomicAdd(scnt + (dkb & 1) * NCL + (dkb >> 1), __popc(pb));
          ba = __shfl_sync(0xffffffffu, ba, lda) + __popc(pa & lt);
          bb = __shfl_sync(0xffffffffu, bb, ldb) + __popc(pb & lt);
          const bool fa = sta && ba >= r.cap, fb = stb && bb >= r.cap;  // full bins: on to k_migrate
          // leavers: the tile's shared buffer (one reservation for the pair), then the global list
          // for full bins and once the shared buffer is full. Most rounds have neither: after one vote they
          // only store their particles (with the slots' shorter test and the particle count from the
          // prologue: 512x1024 FP32 pass 8.53 -> 7.99 ms, Uniform at c dt/dz = 0.3 12.14 -> 11.54 ms)
          int lsa = 0, lsb = 0;
          long long goa = 0, gob = 0;
          bool ga = false, gb = false;
          const bool plain = !__any_sync(0xffffffffu, lva || lvb || fa || fb);
          if (!plain) {
            const unsigned lma = __ballot_sync(0xffffffffu, lva), lmb = __ballot_sync(0xffffffffu, lvb);
            int b0 = 0;
            if (lane == 0) b0 = atomicAdd(lvn, __popc(lma) + __popc(lmb));
            b0 = __shfl_sync(0xffffffffu, b0, 0);
            lsa = b0 + __popc(lma & lt);
            lsb = b0 + __popc(lma) + __popc(lmb & lt);
            ga = fa || (lva && lsa >= S::LVB);
            gb = fb || (lvb && lsb >= S::LVB);
            const unsigned gma = __ballot_sync(0xffffffffu, ga), gmb = __ballot_sync(0xffffffffu, gb);
            if (gma | gmb) {
              if (lane == 0) b0 = atomicAdd(r.lv_count, __popc(gma) + __popc(gmb));
              b0 = __shfl_sync(0xffffffffu, b0, 0);
              goa = (long long)b0 + __popc(gma & lt);
              gob = (long long)b0 + __popc(gma) + __popc(gmb & lt);
            }
          }
          const int gcell = gk * r.nx + gi;  // cells < 2^30
          auto put = [&](int dk, int dcell, int jo, float nox, float noz, float ux, float uy, float uz, float w,
                         unsigned id) {
            const long long o = (long long)dcell * r.cap + jo;
            const bool s1 = (dk & 1) != 0;
            st4((s1 ? r.out[1].q : r.out[0].q) + 4 * o, nox, noz, ux, uy);
            (s1 ? r.out[1].r : r.out[0].r)[o] = uz;
            if (has_w) (s1 ? r.out[1].w : r.out[0].w)[o] = w;
            if (has_id) (s1 ? r.out[1].id : r.out[0].id)[o] = id;
          };
          auto place = [&](bool st, bool full, bool lv, bool g, int dk, int jo, int ls, long long go, float nox,
                           float noz, float ux, float uy, float uz, float w, unsigned id, int shx, int shz) {
            const int dcell = gcell + shz * r.nx + shx;  // a cell of this tile when st
            if (st && !full) {
              put(dk, dcell, jo, nox, noz, ux, uy, uz, w, id);
            } else if (g) {
              if (go < r.lv_cap) list_put(r.lv, go, full ? dcell * 2 + (dk & 1) : dk, nox, 0.f, noz, ux, uy, uz, w, id);
              else flag_error(r.err, ERR_OVERFLOW);
            } else if (lv) {
              lvk[ls] = dk;
              lvv[ls] = nox;
              lvv[2 * S::LVB + ls] = noz;
              lvv[3 * S::LVB + ls] = ux;
              lvv[4 * S::LVB + ls] = uy;
              lvv[5 * S::LVB + ls] = uz;
              if (has_w) lvv[6 * S::LVB + ls] = w;
              if (has_id) lvi[ls] = id;
            }
          };
          if (plain) {
            if (va) put(dka, gcell + Z.sha * r.nx + X.sha, ba, X.offa, Z.offa, nuxa, nuya, nuza, wa, has_id ? sti[ka] : 0u);
            if (vb) put(dkb, gcell + Z.shb * r.nx + X.shb, bb, X.offb, Z.offb, nuxb, nuyb, nuzb, wb, has_id ? sti[kb] : 0u);
          } else {
            if (va)
              place(sta, fa, lva, ga, dka, ba, lsa, goa, X.offa, Z.offa, nuxa, nuya, nuza, wa, has_id ? sti[ka] : 0u,
                    X.sha, Z.sha);
            if (vb)
              place(stb, fb, lvb, gb, dkb, bb, lsb, gob, X.offb, Z.offb, nuxb, nuyb, nuzb, wb, has_id ? sti[kb] : 0u,
                    X.shb, Z.shb);
          }
        }
      } else {
      {
        const int k = sl + LPC * ((rnd + win0) & 3);
        int s;
        const bool valid = slot_of(k, s);
        const SpeciesBuf<T> pout = s ? r.out[1] : r.out[0];
        int dkey = -1 - lane;  // unique per lane when there is no particle
        bool leave = false;
        T nox = T(0), noy = T(0), noz = T(0), ux = T(0), uy = T(0), uz = T(0);
        const T w = (has_w && valid) ? stw[k] : r.wconst;
        if (valid) {
          T p4[4];
          ld4(stq + 4 * k, p4);
          const T o_x = p4[0], o_y = NDIM == 3 ? p4[1] : T(0), o_z = NDIM == 3 ? p4[2] : p4[1];
          if constexpr (NDIM == 3) {
            T p2[2];
            ld2(str + 2 * k, p2);
            ux = p4[3];
            uy = p2[0];
            uz = p2[1];
          } else {
            ux = p4[2];
            uy = p4[3];
            uz = str[k];
          }
          // gather
          T F[6];
          if constexpr (WIN) {
            gather_window<Lanes1<T>, T, T, NDIM, ORDER, SCHEME>(sg, lx, ly, lz, o_x, o_y, o_z, F);
          } else if (SCHEME == 0) {
            gc.interp(o_x, o_y, o_z, F);
          } else {
            const DirW<T> dwx = dir_weights(o_x), dwy = dir_weights(o_y), dwz = dir_weights(o_z);
#pragma unroll
            for (int c = 0; c < 6; ++c)
              F[c] = gather_comp<T, NDIM, SCHEME>(sg + c * S::GN, c, lx, ly, lz, dwx, dwy, dwz);
          }
          // relativistic Boris, momenta relative to the drift u0 z_hat (FP64: every operation here counts, its
          // pipe bounds this kernel)
          const T h = s ? r.hq : -r.hq;
          const T mx = fma(h, F[0], ux), my = fma(h, F[1], uy), mz = fma(h, F[2], uz);
          const T Mz = r.u0 + mz;
          const T mm = fma(Mz, Mz, fma(my, my, fma(mx, mx, T(1))));
          const T hig = h * (WIN ? fine_rsqrt(mm) : fast_rsqrt(mm));
          const T tx = hig * F[3], ty = hig * F[4], tz = hig * F[5];
          const T tt = fma(tz, tz, fma(ty, ty, fma(tx, tx, T(1))));
          const T sf = WIN ? fine_two_over(tt) : two_over(tt);
          const T sx = sf * tx, sy = sf * ty, sz = sf * tz;
          const T qx = fma(my, tz, fma(-Mz, ty, mx));
          const T qy = fma(Mz, tx, fma(-mx, tz, my));
          const T qz = fma(mx, ty, fma(-my, tx, Mz));
          ux = fma(qy, sz, fma(-qz, sy, fma(h, F[0], mx)));
          uy = fma(qz, sx, fma(-qx, sz, fma(h, F[1], my)));
          uz = fma(qx, sy, fma(-qy, sx, fma(h, F[2], mz)));
          const T Uz = r.u0 + uz;
          const T u2 = fma(Uz, Uz, fma(uy, uy, ux * ux)), gp = T(1) + u2;
          const T ign = WIN ? fine_rsqrt(gp) : fast_rsqrt(gp);
          T vy = uy * ign;
          if (r.kin)  // gamma - 1 = u^2 / (gamma + 1)
            kin = fma(w, WIN ? fine_kinetic(u2, gp, ign) : fast_div(u2, fma(gp, ign, T(1))), kin);
          if (LATE) ++npush;
          // move (cell-relative displacement in grid units)
          T ddx = r.dtdx * (ux * ign), ddy = NDIM == 3 ? r.dtdy * vy : T(0), ddz = r.dtdz * (Uz * ign);
          if (!(abs_lt_one(ddx) && abs_lt_one(ddy) && abs_lt_one(ddz))) {
            flag_error(r.err, ERR_NONFINITE);
            ddx = ddy = ddz = T(0);
            ux = uy = uz = T(0);
            vy = T(0);
          }
          const Move1<T> X(o_x, ddx), Y(o_y, ddy), Z(o_z, ddz);
          // Esirkepov deposit: summed in registers when the window fits RegLayout (no step back across
          // a face and no transverse crossing; zero coefficients otherwise), else straight to shared memory
          const bool own = !(X.down || X.up || Z.down || (NDIM == 3 && (Y.down || Y.up)));
          T cx = has_w ? w * r.jfx : cwx, cz = has_w ? w * r.jfz : cwz;
          T cy = NDIM == 3 ? (has_w ? w * r.jfy : cwy) : (has_w ? w * r.jfy2d : cwy) * vy;
          cx = s ? cx : -cx;
          cy = s ? cy : -cy;
          cz = s ? cz : -cz;
          const T rx = own ? cx : T(0), ry = own ? cy : T(0), rz = own ? cz : T(0);
          if constexpr (LATE) {  // summed after the item's push, from the particle's stage slot
            const_cast<T*>(stq)[4 * k + 3] = ddx;
            st2(const_cast<T*>(str) + 2 * k, ddy, ddz);
            const_cast<T*>(stw)[k] = own ? (s ? w : -w) : T(0);
            if (!own) deposit_general<T, 3>(sj, lx, ly, lz, o_x, o_y, o_z, ddx, ddy, ddz, cx, cy, cz);
          } else if constexpr (ORDER == 3) {
            deposit2_cubic<Lanes1<T>, T, NVP, T>(acc, cubic_dir<Lanes1<T>, T, false>(o_x, ddx, false, T(0)),
                                                 cubic_dir<Lanes1<T>, T, true>(o_z, ddz, Z.up, Z.c), rx, ry, rz);
            if (!own) deposit_general<T, 2>(sj, lx, 0, lz, o_x, T(0), o_z, ddx, T(0), ddz, cx, cy, cz);
          } else {
            const LinearZ<Lanes1<T>, T> LZ(o_z, ddz, Z.am, Z.c, Z.up);
            if constexpr (NDIM == 2) {
              deposit2_lin<Lanes1<T>, T, NVP>(acc, o_x, ddx, X.am, LZ, rx, ry, rz);
              if (!own) deposit2_far(sj, lx, lz, o_x, o_z, ddx, ddz, cx, cy, cz);
            } else {
              deposit3_lin<T, NVP>(acc, o_x, ddx, o_y, ddy, LZ, rx, ry, rz);
              if (!own) deposit3_far(sj, lx, ly, lz, o_x, o_y, o_z, ddx, ddy, ddz, cx, cy, cz);
            }
          }
          // new cell and offsets
          nox = X.off;
          noy = NDIM == 3 ? Y.off : T(0);
          noz = Z.off;
          const int nlx = lx + X.sh, nly = NDIM == 3 ? ly + Y.sh : 0, nlz = lz + Z.sh;
          if (nlx >= 0 && nlx < wx && nly >= 0 && nly < wy && nlz >= 0 && nlz < wz) {
            dkey = ((nlz * TY + nly) * TX + nlx) * 2 + s;  // stays in this tile
          } else {
            leave = true;  // global destination, as cell * 2 + species
            // one cell across a face: the index stays within [-1, n] (cells < 2^30: int keys)
            const int ni = wrap_near_p(gi + X.sh, r.nx);
            const int nj = NDIM == 3 ? wrap_near_p(gj + Y.sh, r.ny) : 0;
            const int nk = wrap_near_p(gk + Z.sh, r.nz);
            dkey = ((nk * r.ny + nj) * r.nx + ni) * 2 + s;
          }
        }
        if (LATE && !valid) {  // an empty slot: finite values and no charge for the deposit
          st4(const_cast<T*>(stq) + 4 * k, T(0), T(0), T(0), T(0));
          st2(const_cast<T*>(str) + 2 * k, T(0), T(0));
          const_cast<T*>(stw)[k] = T(0);
        }
        // rebin. Destination in this tile: lanes with the same (cell, species) reserve consecutive
        // slots with one shared-memory atomic on the tile's output counts. Destination in another
        // tile: the particle is appended to the leaver list (one global atomic per warp), which
        // k_migrate inserts after this kernel.
        const bool stay = valid && !leave;
        const unsigned peers = __match_any_sync(0xffffffffu, stay ? dkey : -1 - lane);
        const int leader = __ffs(peers) - 1;
        const int rank = __popc(peers & ((1u << lane) - 1u));
        int base = 0;
        if (stay && lane == leader) base = atomicAdd(scnt + (dkey & 1) * NCL + (dkey >> 1), __popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        // a full destination bin: the particle goes through the global leaver list instead, and
        // k_migrate spills it when the bin is still full there (nothing is dropped)
        const bool full = stay && base + rank >= r.cap;
        long long fglob = 0, lglob = 0;
        int lslot = 0;
        if (__any_sync(0xffffffffu, full || (valid && leave))) {  // most rounds: neither
          const unsigned fmask = __ballot_sync(0xffffffffu, full);
          if (fmask) {
            const int fl = __ffs(fmask) - 1;
            int fb = 0;
            if (lane == fl) fb = atomicAdd(r.lv_count, __popc(fmask));
            fb = __shfl_sync(0xffffffffu, fb, fl);
            fglob = (long long)fb + __popc(fmask & ((1u << lane) - 1u));
          }
          // leavers: a slot in the tile's shared-memory buffer (one shared atomic per warp), or, once
          // the buffer is full, straight in the global list
          const unsigned lmask = __ballot_sync(0xffffffffu, valid && leave);
          if (lmask) {
            const int lleader = __ffs(lmask) - 1;
            int b = 0;
            if (lane == lleader) b = atomicAdd(lvn, __popc(lmask));
            b = __shfl_sync(0xffffffffu, b, lleader);
            lslot = b + __popc(lmask & ((1u << lane) - 1u));
            const unsigned gmask = __ballot_sync(0xffffffffu, valid && leave && lslot >= S::LVB);
            if (gmask) {
              const int gl = __ffs(gmask) - 1;
              int gb = 0;
              if (lane == gl) gb = atomicAdd(r.lv_count, __popc(gmask));
              gb = __shfl_sync(0xffffffffu, gb, gl);
              lglob = (long long)gb + __popc(gmask & ((1u << lane) - 1u));
            }
          }
        }
        if (stay) {
          const int j = base + rank;
          const int dl = dkey >> 1;
          const int dx = dl % TX, dy = (dl / TX) % TY, dz = dl / (TX * TY);
          const int dcell = ((Z0 + dz) * r.ny + Y0 + dy) * r.nx + X0 + dx;  // cells < 2^30
          if (!full) {
            const long long o = (long long)dcell * r.cap + j;
            part_put(pout, NDIM, o, nox, noy, noz, ux, uy, uz);
            if (has_w) pout.w[o] = w;
            if (has_id) pout.id[o] = sti[k];
          } else if (fglob < r.lv_cap) {
            list_put(r.lv, fglob, dcell * 2 + (dkey & 1), nox, noy, noz, ux, uy, uz, w, has_id ? sti[k] : 0u);
          } else {
            flag_error(r.err, ERR_OVERFLOW);
          }
        } else if (valid && lslot < S::LVB) {
          lvk[lslot] = dkey;
          lvv[lslot] = nox;
          if (NDIM == 3) lvv[S::LVB + lslot] = noy;
          lvv[2 * S::LVB + lslot] = noz;
          lvv[3 * S::LVB + lslot] = ux;
          lvv[4 * S::LVB + lslot] = uy;
          lvv[5 * S::LVB + lslot] = uz;
          if (has_w) lvv[6 * S::LVB + lslot] = w;
          if (has_id) lvi[lslot] = sti[k];
        } else if (valid) {
          const long long o = lglob;
          if (o < r.lv_cap) {
            r.lv.key[o] = dkey;
            r.lv.ox[o] = nox;
            if (NDIM == 3) r.lv.oy[o] = noy;
            r.lv.oz[o] = noz;
            r.lv.dux[o] = ux;
            r.lv.duy[o] = uy;
            r.lv.duz[o] = uz;
            if (has_w) r.lv.w[o] = w;
            if (has_id) r.lv.id[o] = sti[k];
          } else {
            flag_error(r.err, ERR_OVERFLOW);
          }
        }
      }
      }
    }
    if constexpr (QUEUE) {
      if (nfar > 0) {
        __syncwarp();
        deposit_queue(sj, SG::q(stg, stage, 0), SG::r(stg, stage, 0), SG::w(stg, stage, 0), s_far[warp], nfar,
                      g * CPW + max(one, 0), one < 0 ? 4 * LPC : 128, r.jfx, r.jfy2d, r.jfz);
      }
    }
    if constexpr (LATE) {
      __syncwarp();
      T* j = sj + okey;
      deposit3_cubic<T, LPC, 0>(stq, str, stw, sl, nrnd, win0, r.jfx, j);
      deposit3_cubic<T, LPC, 1>(stq, str, stw, sl, nrnd, win0, r.jfy, j);
      deposit3_cubic<T, LPC, 2>(stq, str, stw, sl, nrnd, win0, r.jfz, j);
    }
    if (!LATE && it == giters - 1) {
      // 3. segmented transpose-reduction of the cell's register sums over its LPC lanes
      if constexpr (ACC2) {
#pragma unroll
        for (int i = 0; i < NVP; ++i) acc[i] = acc2[i].x + acc2[i].y;
      }
#pragma unroll
      for (int sh = LPC / 2; sh >= 1; sh >>= 1) {
        const bool up = (lane & sh) != 0;
#pragma unroll
        for (int j = 0; j < PER * sh; ++j) {
          const T send = up ? acc[j] : acc[j + PER * sh];
          const T keep = up ? acc[j + PER * sh] : acc[j];
          acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
        }
      }
#pragma unroll
      for (int m = 0; m < PER; ++m) {
        const int i = sl * PER + m;
        if (i < NV && acc[m] != T(0)) {
          int comp, a, b, c;
          RegLayout<NDIM, ORDER>::at(i, comp, a, b, c);
          atomicAdd(sj + comp * S::JN + okey + (c * S::JY + b) * S::JX + a, acc[m]);
        }
      }
    }
    __syncwarp();  // the stage just read is refilled by the next iteration's prefetch
    g = ng;
    it = nit;
    one = none;
    crowd = ncrowd;
    giters = niters;
    stage ^= 1;
  }
  cp_async_wait_all();
  __syncthreads();

  // 4. the tile's buffered leavers: one reservation in the global list, then a coalesced copy
  __shared__ int lv_base;
  const int nlv = min(*lvn, S::LVB);
  if (tid == 0) lv_base = nlv > 0 ? atomicAdd(r.lv_count, nlv) : 0;
  __syncthreads();
  for (int e = tid; e < nlv; e += PUSH_THREADS) {
    const long long o = (long long)lv_base + e;
    if (o < r.lv_cap) {
      r.lv.key[o] = lvk[e];
      r.lv.ox[o] = lvv[e];
      if (NDIM == 3) r.lv.oy[o] = lvv[S::LVB + e];
      r.lv.oz[o] = lvv[2 * S::LVB + e];
      r.lv.dux[o] = lvv[3 * S::LVB + e];
      r.lv.duy[o] = lvv[4 * S::LVB + e];
      r.lv.duz[o] = lvv[5 * S::LVB + e];
      if (has_w) r.lv.w[o] = lvv[6 * S::LVB + e];
      if (has_id) r.lv.id[o] = lvi[e];
    } else {
      flag_error(r.err, ERR_OVERFLOW);
    }
  }

  // 5. output counts of the tile's cells (leavers from other tiles are added by k_migrate); a count
  // past the capacity (particles sent on through the leaver list) is stored as the capacity
  for (int cl = tid; cl < ncl; cl += PUSH_THREADS) {
    const int lx = cl % TX, ly = (cl / TX) % TY, lz = cl / (TX * TY);
    if (lx < wx && ly < wy && lz < wz) {
      const long long cell = (long long)(Z0 + lz) * nxy + (long long)(Y0 + ly) * r.nx + X0 + lx;
      r.out[0].cnt[cell] = min(scnt[cl], r.cap);
      r.out[1].cnt[cell] = min(scnt[NCL + cl], r.cap);
    }
  }

  // 6. flush the tile's current to global memory
  for (int e = tid; e < jn; e += PUSH_THREADS) {
    const T v0 = sj[e], v1 = sj[S::JN + e], v2 = sj[2 * S::JN + e];
    if (v0 == T(0) && v1 == T(0) && v2 == T(0)) continue;
    const int o = node_at(e % S::JX, (e / S::JX) % S::JY, e / (S::JX * S::JY));
    if (v0 != T(0)) atomicAdd(r.j[0] + o, v0);
    if (v1 != T(0)) atomicAdd(r.j[1] + o, v1);
    if (v2 != T(0)) atomicAdd(r.j[2] + o, v2);
  }

  // 7. kinetic energy and particle count of this step: per-thread partial sums in the working
  // precision, FP64 across the warp, the block and the grid
  if (r.kin) {
    __shared__ double skin[NWARP];
    __shared__ int swcnt[NWARP];
    double kd = (double)kin;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kd += __shfl_xor_sync(0xffffffffu, kd, o);
    const int nd = __reduce_add_sync(0xffffffffu, npush);
    if (lane == 0) {
      skin[warp] = kd;
      swcnt[warp] = nd;
    }
    __syncthreads();
    if (tid == 0) {
      double t = 0;
      long long c = 0;
      for (int w2 = 0; w2 < NWARP; ++w2) {
        t += skin[w2];
        c += swcnt[w2];
      }
      atomicAdd(r.kin, t);
      atomicAdd(r.kin + 1, (double)c);
    }
  }
}

}  // namespace picgb
