// Field advance of the GRPIC cycle: magnetic half-step (Sec. 3.1, Eq. 10) and electric full
// step (Sec. 3.2, Eq. 12) on the staggered Yee lattice (Sec. 3, Fig. 2).
//
// Prognostic pair: covariant b = (F_yz, F_zx, F_xy) on faces, contravariant d = (F^x4, F^y4,
// F^z4) on edges.  Each update needs the other form of the tensor at its own lattice points:
//   B step:  e_i = F_i4 at the d^i edges,  b_out = b_base - coef curl e(b_src, d)   (forward diff.)
//   E step:  h = F^jk at the b faces,       d_out = d + dx4 (4 pi/c J - div h)       (backward diff.)
// The missing components at a lattice point are the mean of the 2 or 4 nearest points of
// their own lattice; the conversion uses the metric evaluated at that point.  With g_mn = eta + f k k
// (Eqs. 4-6), |k| = 1 and G = f / (1 + f), lowering the tensor of Eq. 8 and eliminating gives
//   e = -d + G [k x b + d - k (k.d)],      h = b - G [b + d x k - k (k.b)]
// (from h = [b - f d x k + f k (k.b)] / (1 + f) and e = f k x h + (f - 1) d - f k (k.d): the k (k.b) and
// k (k.(d x k)) terms vanish in k x h).  e_L needs neither b_L nor its eight-point mean.
//
// A B half-step is one launch, and so is the literal E step; the time-centred E step is two, the midpoint predictor
// d* = d + (dx4/2) rhs(b, d) into memory that is free by then (the idle b buffer) and the update from h(b, d*).
// A block owns a 32 x BY patch of (x, y) columns and marches up z through a chunk of planes: it evaluates the
// conversion for the whole patch of the next plane into shared memory and updates the cells whose stencil lies inside
// the patch.  Neighbouring patches overlap by the stencil's reach, one cell, so each cell is written exactly once by
// one block, from inputs that no block of the launch modifies.  The output is another buffer than the inputs
// (every cell written; a copy where the location is not advanced), except the time-centred second B half-step, which
// overwrites the b^{n-1/2} buffer it reads only at the cell it writes.  Per cell a launch moves the words that it reads
// and writes once: the conversions live in registers and shared memory,
// and in FP32 the metric is evaluated where it is needed instead of being read from memory (48 B per cell and step, as
// much as the fields themselves).  In FP64 it is read from a table (launch_metric_table): its 40 operations at each
// of three locations are two thirds of the kernel's, and the FP64 pipe takes longer for them than HBM for 96 B
// (B step at 96^3: 420 us evaluated, 138 us read).
//
// What bounds them: FP32 the issue of instructions, FP64 the FP64 pipe.  Hence sums over pairs of planes are
// carried from one plane of the march to the next instead of being formed again, a patch synchronises once a plane,
// and FP64 reciprocals and roots are FastOps64's.
// Measured (GB300, microseconds a launch, no layers; before: the E step as one march with a halo of 3, IEEE FP64
// divides and roots, the metric evaluated in FP64, patches over all cells and chunks of at least 4 planes):
//            FP32 64^3   128^3      192^3       64x64x128   FP64 32^3    64^3         96^3
//   B half   24 -> 14   80 -> 45    222 -> 132   39 -> 18    129 -> 15   425 -> 47   1053 -> 138
//   E step   35 -> 30  140 -> 107   411 -> 330   56 -> 40    215 -> 32  1114 -> 104  2193 -> 318  (both launches)
// At 192^3 FP32 moves 38 B (B half) and 62 + 74 B (E) per cell: 2.0 and 2.9 TB/s, 30 and 43 % of the measured copy
// rate; it issues about 500 instructions a cell and plane of the march.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "metric.cuh"

namespace grpic {

namespace {

// Half-cell offsets of the six field locations: 0..2 = d^x, d^y, d^z (edges),
// 3..5 = b_x, b_y, b_z (faces).
__host__ __device__ constexpr int half(int loc, int ax) {
  return (loc < 3) ? (loc == ax ? 1 : 0) : ((loc - 3) == ax ? 0 : 1);
}
// Neighbour range, along one axis, of source lattice s around a point of target lattice t.
__host__ __device__ constexpr int nb_lo(int t, int s, int ax) {
  return half(s, ax) == half(t, ax) ? 0 : (half(t, ax) == 1 ? 0 : -1);
}
__host__ __device__ constexpr int nb_hi(int t, int s, int ax) {
  return half(s, ax) == half(t, ax) ? 0 : (half(t, ax) == 1 ? 1 : 0);
}

// Square root with its reciprocal, reciprocal and quotient: the hardware approximations in FP32 (relative error
// ~1e-7, below the FP32 rounding of the stencil sums), FastOps64 in FP64.
__device__ __forceinline__ float root_t(float v, float& inv) {
  inv = rsqrtf(v);
  return v * inv;
}
__device__ __forceinline__ double root_t(double v, double& inv) { return FastOps64::root_and_rsqrt(v, &inv); }
__device__ __forceinline__ float rcp_t(float v) { return __fdividef(1.f, v); }
__device__ __forceinline__ double rcp_t(double v) { return FastOps64::rcp(v); }
__device__ __forceinline__ float div_t(float a, float b) { return a * __fdividef(1.f, b); }
__device__ __forceinline__ double div_t(double a, double b) { return FastOps64::div(a, b); }
// A product that stays one (in FP64, where the metric table has to hold what the kernels would evaluate, no product is
// left for the compiler to fuse with a sum, which it does differently from place to place).
__device__ __forceinline__ float mul_t(float a, float b) { return a * b; }
__device__ __forceinline__ double mul_t(double a, double b) { return __dmul_rn(a, b); }

// Conversions between FP64 and the field type with integer operations (the hardware's run on the FP64 pipe).
template <typename T>
__device__ __forceinline__ T narrow_t(double v) {
  if constexpr (sizeof(T) == sizeof(float))
    return narrow(v);
  else
    return v;
}
__device__ __forceinline__ double widen_t(float v) { return widen(v); }
__device__ __forceinline__ double widen_t(double v) { return v; }

constexpr int kTX = 32;  // threads (cells) of a patch along x: one warp per row

// Metric at a point.  FP32: f and k of Eqs. 4-5; FP64: G = f / (1 + f) and k.
template <typename T>
struct Pt {
  T f, k0, k1, k2;
};

// Location l of the cell whose lower corner is (xr, yr, zr) relative to the
// centre.  The quartic's root r^2 by the cancellation-free branch form with
// D = sqrt(p^2 + 4 a^2 z^2), p = R^2 - a^2; since the root satisfies r^4 + a^2 z^2 = r^2 (2 r^2 - p)
// = r^2 D, f = 2 m r^3 / (r^4 + a^2 z^2) = 2 m r / D and G = 2 m r / (D + 2 m r).  Excised locations
// (and r = 0) take the flat metric, as the conversions there do.
template <typename T>
__device__ __forceinline__ Pt<T> metric_pt(const FieldConsts<T>& K, int l, T xr, T yr, T zr, bool excised) {
  Pt<T> P;
  P.f = T(0);
  P.k0 = T(0);
  P.k1 = T(0);
  P.k2 = T(1);
  if (excised || !K.massive) return P;
  const T X = half(l, 0) ? xr + T(0.5) : xr;
  const T Y = half(l, 1) ? yr + T(0.5) : yr;
  const T Z = half(l, 2) ? zr + T(0.5) : zr;
  const T q = K.a2 * Z * Z;
  const T p = fma(X, X, fma(Y, Y, fma(Z, Z, -K.a2)));
  const T disc = fma(p, p, T(4) * q);
  T rD, ir;  // 1 / D, 1 / r
  const T D = root_t(disc, rD);
  const T r2 = p >= T(0) ? T(0.5) * (p + D) : div_t(T(2) * q, D - p);
  if (!(r2 > T(0))) return P;
  const T r = root_t(r2, ir);
  const T irho2 = rcp_t(r2 + K.a2);
  if constexpr (sizeof(T) == sizeof(float)) {
    P.f = K.two_m * r * rD;
  } else {
    const T F = mul_t(K.two_m, r);
    P.f = div_t(F, D + F);
  }
  P.k0 = (r * X - mul_t(K.a, Y)) * irho2;
  P.k1 = (r * Y + mul_t(K.a, X)) * irho2;
  P.k2 = Z * ir;
  return P;
}

// Metric at location l of cell c: from the FP64 table when there is one, else evaluated.
template <typename T>
__device__ __forceinline__ Pt<T> metric_at(const FieldConsts<T>& K, const double2* __restrict__ met, long long ncell,
                                           long long c, int l, T xr, T yr, T zr, bool excised) {
  if constexpr (sizeof(T) == sizeof(double)) {
    if (met) {
      const double2 a = __ldg(met + 2 * l * ncell + c), b = __ldg(met + (2 * l + 1) * ncell + c);
      return Pt<T>{a.x, a.y, b.x, b.y};
    }
  }
  return metric_pt<T>(K, l, xr, yr, zr, excised);
}

// e_L = -d_L + G [(k x b)_L + d_L - k_L (k.d)] at an edge: dL is d_L there, sdM, sdN the sums of the four
// nearest points of the other two d components (M = L + 1, N = L + 2 mod 3), sbM, sbN the sums of the two nearest
// points of b_M and b_N.
template <int L, typename T>
__device__ __forceinline__ T edge_e(const Pt<T>& P, T dL, T sdM, T sdN, T sbM, T sbN) {
  const T kL = L == 0 ? P.k0 : (L == 1 ? P.k1 : P.k2);
  const T kM = L == 0 ? P.k1 : (L == 1 ? P.k2 : P.k0);
  const T kN = L == 0 ? P.k2 : (L == 1 ? P.k0 : P.k1);
  T G = P.f;
  if constexpr (sizeof(T) == sizeof(float)) G = P.f * rcp_t(T(1) + P.f);
  const T kd = fma(kL, dL, T(0.25) * fma(kM, sdM, kN * sdN));
  const T t = fma(T(0.5), fma(kM, sbN, -(kN * sbM)), fma(-kL, kd, dL));
  return fma(G, t, -dL);
}

// h_Q at a face: bQ is b_Q there, sbM, sbN the sums of the four nearest points of the other two b components (M = Q +
// 1, N = Q + 2 mod 3), sdM, sdN the sums of the two nearest points of d_M and d_N; (d x k)_Q = d_M k_N - d_N k_M.
// FP64: b_Q - G [b_Q - k_Q (k.b) + (d x k)_Q].
// FP32: [b_Q - f (d x k)_Q + f k_Q (k.b)] / (1 + f) as it stands.  Where b is large beside d (a strong
// uniform field), d is what the differences of these h leave of their rounding to FP32, so another form of equal
// accuracy gives another d (measured 3e-5 apart on the 64 x 64 x 128 disk set-up, each 4e-5 from FP64).
template <int Q, typename T>
__device__ __forceinline__ T face_h(const Pt<T>& P, T bQ, T sbM, T sbN, T sdM, T sdN) {
  const T kQ = Q == 0 ? P.k0 : (Q == 1 ? P.k1 : P.k2);
  const T kM = Q == 0 ? P.k1 : (Q == 1 ? P.k2 : P.k0);
  const T kN = Q == 0 ? P.k2 : (Q == 1 ? P.k0 : P.k1);
  if constexpr (sizeof(T) == sizeof(float)) {
    T b[3];
    b[Q] = bQ;
    b[(Q + 1) % 3] = sbM * 0.25f;
    b[(Q + 2) % 3] = sbN * 0.25f;
    const T dM = sdM * 0.5f, dN = sdN * 0.5f;
    const T dxk = dM * kN - dN * kM;
    const T kb = P.k0 * b[0] + P.k1 * b[1] + P.k2 * b[2];
    return (bQ - P.f * dxk + P.f * kQ * kb) * rcp_t(1.f + P.f);
  } else {
    const T kb = fma(kQ, bQ, T(0.25) * fma(kM, sbM, kN * sbN));
    const T t = fma(T(0.5), fma(kN, sdM, -(kM * sdN)), fma(-kQ, kb, bQ));
    return fma(-P.f, t, bQ);
  }
}

constexpr int kSX = kTX + 2;   // staged columns: the patch and a one-cell halo

// Three components of one z plane of a patch with a one-cell halo, staged in shared memory.
template <typename T, int BY>
struct Plane3 {
  T v[3][BY + 2][kSX];
};

// 4 pi / c J^al in the field type: FP64 J rounded to FP32 with integer operations (this GPU runs
// conversions on its reduced-rate FP64 pipe), then scaled in FP32.
template <typename T>
__device__ __forceinline__ T source(const FieldConsts<T>& K, double J) {
  if constexpr (sizeof(T) == sizeof(float))
    return narrow(J) * K.four_pi_c;
  else
    return K.four_pi_c * J;
}

__device__ __forceinline__ bool adv(uint16_t w, int l) { return (w >> l) & 1u; }
__device__ __forceinline__ bool exc(uint16_t w, int l) { return (w >> (8 + l)) & 1u; }
__device__ __forceinline__ bool in_layer(uint16_t w) { return (w & kLayerBit) != 0u; }

// ---- absorbing layers -------------------------------------------------------------------------
// Relaxation per step at location l of cell (i, j, k): the larger of the outer layer's
// k_out ((W + 1 - s) / W)^2 where s <= W, s being 1 + the cell's distance in cells to the outer two
// index layers (s = 1 at the first advanced cell), and the inner layer's
// k_in (r_abs - r) / (r_abs - r_exc) where r_exc <= r < r_abs (r at the location, in FP64).  The
// outer profile is evaluated in the field type from integers and constants converted on the host;
// the inner one is tabulated once, in FP64, over the box of cells around the hole that holds every
// location with r < r_abs, and looked up in cells flagged for it (kInnerBit).  The field kernels
// then run no FP64 operation for the layers (this GPU's FP64 pipe, which also does its
// conversions, is narrow).

// A small non-negative int as a float without a conversion instruction: the float with the bits
// of 2^23 + v, minus 2^23; exact for 0 <= v < 2^23.
__device__ __forceinline__ float small_int_to_float(int v) { return __int_as_float(0x4B000000 | v) - 8388608.f; }

template <typename T>
__device__ __forceinline__ T outer_kappa(const Grid& g, int i, int j, int k) {
  const int s = 1 + min(min(min(i - 2, g.nx - 3 - i), min(j - 2, g.ny - 3 - j)), min(k - 2, g.nz - 3 - k));
  if (s < 1 || s > g.w_out) return T(0);  // (k_out = 0 gives 0 below)
  T k_out, inv_w, n;
  if constexpr (sizeof(T) == sizeof(float)) {
    k_out = g.k_out_f;
    inv_w = g.inv_w_f;
    n = small_int_to_float(g.w_out + 1 - s);
  } else {
    k_out = g.k_out;
    inv_w = g.inv_w;
    n = (double)(g.w_out + 1 - s);
  }
  const T u = n * inv_w;
  return k_out * u * u;
}

// The inner layer's relaxation at location l of cell (i, j, k), in FP64.
__device__ inline double inner_kappa(const Grid& g, int l, int i, int j, int k) {
  if (!(g.k_in > 0.0) || !(g.r_abs > g.r_exc)) return 0.0;
  const Kerr<double> K = kerr_eval<double>(i + 0.5 * half(l, 0) - g.xc, j + 0.5 * half(l, 1) - g.yc,
                                           k + 0.5 * half(l, 2) - g.zc, g.m, g.a);
  if (K.flat || K.r < g.r_exc || K.r >= g.r_abs) return 0.0;
  return g.k_in * (g.r_abs - K.r) / (g.r_abs - g.r_exc);
}

// Index of location l of cell (i, j, k) in the inner layer's table (the cell must lie in the box).
__host__ __device__ __forceinline__ long long kin_index(const Grid& g, int l, int i, int j, int k) {
  return (((long long)l * g.kboxn[2] + (k - g.kbox0[2])) * g.kboxn[1] + (j - g.kbox0[1])) * g.kboxn[0] +
         (i - g.kbox0[0]);
}

// v relaxed toward the target t at location l of cell (i, j, k) with flags w and outer relaxation k_outer:
// t + (1 - kappa)(v - t).
template <typename T>
__device__ __forceinline__ T relax(const Grid& g, const T* kin, uint16_t w, T k_outer, T t, T v, int l, int i, int j,
                                   int k) {
  T kap = k_outer;
  if (w & kInnerBit) kap = fmax(kap, __ldg(kin + kin_index(g, l, i, j, k)));
  return t + (T(1) - kap) * (v - t);
}

// Asynchronous 4- or 8-byte copy global -> shared, and the commit / wait of the thread's copy groups.
template <typename T>
__device__ __forceinline__ void cp_async(T* dst, const T* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N of this thread's most recent copy groups are still in flight
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The staged halo patch of a block: (BY + 2) x kSX elements, at most two per thread (threads
// 32 x BY); element e of the patch is column e % kSX, row e / kSX, at grid (x0 - 1 + column,
// y0 - 1 + row) where (x0, y0) is the grid position of thread (0, 0).  Columns and rows beyond the grid are left out,
// and planes beyond it take the nearest one: only cells of the outer index layer reach them, and those are not
// converted.  (Copies that clamp the columns too, many lanes reading one address, made a patch at a grid's edge twice
// as slow.)
template <int BY>
struct Stager {
  int s0, s1;       // element in a staged component; negative: none
  unsigned o0, o1;  // x + y nx of the element
  __device__ Stager(const Grid& g, int x0, int y0) {
    const int t = threadIdx.y * kTX + threadIdx.x;
    auto off = [&](int e, int& s) {
      const int x = x0 - 1 + e % kSX, y = y0 - 1 + e / kSX;  // (x0, y0 >= 1)
      s = e < (BY + 2) * kSX && x < g.nx && y < g.ny ? e : -1;
      return (unsigned)(x + y * g.nx);
    };
    o0 = off(t, s0);
    o1 = off(t + kTX * BY, s1);
  }
  // start copying plane p of the three arrays src into dst
  template <typename T>
  __device__ __forceinline__ void stage(const Grid& g, const T* const* src, int p, Plane3<T, BY>& dst) const {
    const long long pz = (long long)min(max(p, 0), g.nz - 1) * g.nx * g.ny;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const T* const plane = src[q] + pz;
      T* const to = &dst.v[q][0][0];
      if (s0 >= 0) cp_async(to + s0, plane + o0);
      if (s1 >= 0) cp_async(to + s1, plane + o1);
    }
  }
};

// The outer two index layers are never advanced: a step into another buffer copies them, each block its share (blocks
// of their own beside the patches filled both slots of an SM with patches while other SMs had none: FP64 at 64^3 80 us
// instead of 46).  Cells by index: the z layers, then the y layers of the planes between them, then the x layers of the
// rows between those.
__device__ __forceinline__ int outer_layer(int q, int n) { return q < 2 ? q : n - 4 + q; }  // q = 0..3
template <typename T>
__device__ __forceinline__ void copy_shell(const Grid& g, const T* const* src, T* const* dst, long long block,
                                           long long blocks) {
  const unsigned plane = g.nx * g.ny, xrow = 4u * g.nx, xcol = 4u * (g.ny - 4);
  const long long nz4 = 4ll * plane, ny4 = (long long)xrow * (g.nz - 4);
  const long long cells = g.ncell - (long long)(g.nx - 4) * (g.ny - 4) * (g.nz - 4);
  const int threads = blockDim.x * blockDim.y;
  for (long long s = block * threads + threadIdx.y * kTX + threadIdx.x; s < cells; s += blocks * threads) {
    int x, y, z;
    if (s < nz4) {
      const unsigned q = (unsigned)(s / plane), e = (unsigned)(s - (long long)q * plane);
      y = e / g.nx;
      x = e - y * g.nx;
      z = outer_layer((int)q, g.nz);
    } else if (s < nz4 + ny4) {
      const unsigned r = (unsigned)((s - nz4) / xrow), e = (unsigned)(s - nz4 - (long long)r * xrow);
      y = e / g.nx;
      x = e - y * g.nx;
      y = outer_layer(y, g.ny);
      z = 2 + (int)r;
    } else {
      const unsigned r = (unsigned)((s - nz4 - ny4) / xcol), e = (unsigned)(s - nz4 - ny4 - (long long)r * xcol);
      x = outer_layer((int)(e & 3u), g.nx);
      y = 2 + (int)(e >> 2);
      z = 2 + (int)r;
    }
    const long long c = ((long long)z * g.ny + y) * g.nx + x;
    T v[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = src[q][c];
#pragma unroll
    for (int q = 0; q < 3; ++q) dst[q][c] = v[q];
  }
}

__device__ __forceinline__ void decode_tile(const TileGrid& t, long long q, int& tx, int& ty, int& zs) {
  tx = (int)(q % t.ntx);
  const long long r = q / t.ntx;
  ty = (int)(r % t.nty);
  zs = 2 + (int)(r / t.nty) * t.zchunk;
}

// ---- B half-step ------------------------------------------------------------------------------
// Patch: threads (tx, ty) at x = x0 + tx, y = y0 + ty; e at the patch of each plane P of the chunk and of
// the plane above it; cells with tx < 31 and ty < BY - 1 are updated (the curl reaches +1).  Iteration P reads the
// staged planes P and P + 1 (P + 2 in flight), the sums over plane P - 1 are carried in registers, and e of plane
// P - 1 is in the other half of E: one barrier a plane.
template <typename T, int BY>
struct BStepSmem {
  Plane3<T, BY> Sb[4], Sd[4];
  T E[2][3][BY][kTX];
};

template <typename T, int BY>
__device__ __forceinline__ void b_step_tile(const Grid& g, const BStepArgs<T>& A, const TileGrid& t, int block,
                                            BStepSmem<T, BY>& sm) {
  int tile_x, tile_y, zs;
  decode_tile(t, block, tile_x, tile_y, zs);
  const int ze = min(zs + t.zchunk, g.nz - 2);
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int cx = tx + 1, cy = ty + 1;  // the cell in the staged planes
  const int x0 = 2 + tile_x * (kTX - 1), y0 = 2 + tile_y * (BY - 1);
  const int x = x0 + tx, y = y0 + ty;
  const bool in_xy = x < g.nx && y < g.ny;
  const bool conv_xy = x >= 1 && x <= g.nx - 2 && y >= 1 && y <= g.ny - 2;
  const bool out_xy = x <= g.nx - 3 && y <= g.ny - 3 && tx < kTX - 1 && ty < BY - 1;
  const T xr = (T)x - A.K.xc, yr = (T)y - A.K.yc;
  const Stager<BY> st(g, x0, y0);
  for (int q = zs - 1; q <= zs + 1; ++q) {
    st.stage(g, A.src, q, sm.Sb[q & 3]);
    st.stage(g, A.d, q, sm.Sd[q & 3]);
  }
  cp_async_commit();
  if (!A.inplace) copy_shell<T>(g, A.base, A.out, block, t.count());
  cp_async_wait<0>();
  __syncthreads();
  // carried from plane P - 1: d_z summed over the x and the y pair, b; from plane P: d_x, d_y and their sums with
  // the neighbour below in x and in y
  T d2x_m, d2y_m, b_m[3], d0, d0x, d1, d1y;
  {
    const Plane3<T, BY>&B = sm.Sb[(zs - 1) & 3], &D = sm.Sd[(zs - 1) & 3], &C = sm.Sd[zs & 3];
    d2x_m = D.v[2][cy][cx] + D.v[2][cy][cx + 1];
    d2y_m = D.v[2][cy][cx] + D.v[2][cy + 1][cx];
#pragma unroll
    for (int q = 0; q < 3; ++q) b_m[q] = B.v[q][cy][cx];
    d0 = C.v[0][cy][cx];
    d0x = d0 + C.v[0][cy][cx - 1];
    d1 = C.v[1][cy][cx];
    d1y = d1 + C.v[1][cy - 1][cx];
  }
  T em[3] = {T(0), T(0), T(0)};  // e of plane P - 1 at the cell
  const int splane = g.nx * g.ny;
  long long cP = ((long long)zs * g.ny + y) * g.nx + x;  // the cell in plane P
  T zr = (T)zs - A.K.zc;
  // loaded one iteration ahead: the flags of plane P + 1 and, for the in-place update, b^{n-1/2} of plane P
  uint16_t w_prev = 0, w = in_xy ? __ldg(A.loc + cP) : (uint16_t)0;
  T old_next[3] = {T(0), T(0), T(0)};
  for (int P = zs; P <= ze; ++P) {
    if (P < ze) {
      st.stage(g, A.src, P + 2, sm.Sb[(P + 2) & 3]);
      st.stage(g, A.d, P + 2, sm.Sd[(P + 2) & 3]);
    }
    cp_async_commit();
    const uint16_t w_next = in_xy && P < ze ? __ldg(A.loc + cP + splane) : (uint16_t)0;
    const int p = P - 1;
    const bool upd = p >= zs && out_xy;
    T old[3] = {b_m[0], b_m[1], b_m[2]};
    if (A.inplace) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        old[q] = old_next[q];
        if (out_xy && P < ze) old_next[q] = A.base[q][cP];
      }
    }
    cp_async_wait<1>();  // planes up to P + 1 have landed
    __syncthreads();
    // e at plane P
    const Plane3<T, BY>&B = sm.Sb[P & 3], &D = sm.Sd[P & 3], &N = sm.Sd[(P + 1) & 3];
    const T b0 = B.v[0][cy][cx], b1 = B.v[1][cy][cx], b2 = B.v[2][cy][cx];
    const T d2 = D.v[2][cy][cx];
    const T d2x = d2 + D.v[2][cy][cx + 1], d2y = d2 + D.v[2][cy + 1][cx];
    const T n0 = N.v[0][cy][cx], n1 = N.v[1][cy][cx];
    const T n0x = n0 + N.v[0][cy][cx - 1], n1y = n1 + N.v[1][cy - 1][cx];
    T e[3] = {T(0), T(0), T(0)};
    if (conv_xy) {  // (the planes of the march, 2 .. n - 2, are all converted)
      auto metric = [&](int l) { return metric_at<T>(A.K, A.met, g.ncell, cP, l, xr, yr, zr, exc(w, l)); };
      e[0] = edge_e<0>(metric(0), d0,
                       d1y + (D.v[1][cy][cx + 1] + D.v[1][cy - 1][cx + 1]), d2x_m + d2x, b_m[1] + b1,
                       B.v[2][cy - 1][cx] + b2);
      e[1] = edge_e<1>(metric(1), d1, d2y_m + d2y,
                       d0x + (D.v[0][cy + 1][cx] + D.v[0][cy + 1][cx - 1]), B.v[2][cy][cx - 1] + b2, b_m[0] + b0);
      e[2] = edge_e<2>(metric(2), d2, d0x + n0x, d1y + n1y,
                       B.v[0][cy - 1][cx] + b0, B.v[1][cy][cx - 1] + b1);
    }
    T(&E)[3][BY][kTX] = sm.E[P & 1];
#pragma unroll
    for (int q = 0; q < 3; ++q) E[q][ty][tx] = e[q];
    // b update at plane P - 1 from e of planes P - 1 (the neighbours' in shared memory) and P (own)
    if (upd) {
      const long long c = cP - splane;
      const T(&Em)[3][BY][kTX] = sm.E[p & 1];
      // curl e at the three faces: b_x = F_yz: d_y e_z - d_z e_y; b_y = F_zx: d_z e_x - d_x e_z;
      // b_z = F_xy: d_x e_y - d_y e_x
      const T cu[3] = {(Em[2][ty + 1][tx] - em[2]) - (e[1] - em[1]), (e[0] - em[0]) - (Em[2][ty][tx + 1] - em[2]),
                       (Em[1][ty][tx + 1] - em[1]) - (Em[0][ty + 1][tx] - em[0])};
      T v[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) v[q] = adv(w_prev, 3 + q) ? fma(-A.coef, cu[q], old[q]) : old[q];
      if (A.tgt[0] && in_layer(w_prev)) {
        const T ko = outer_kappa<T>(g, x, y, p);
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (adv(w_prev, 3 + q)) v[q] = relax<T>(g, A.kin, w_prev, ko, A.tgt[q][c], v[q], 3 + q, x, y, p);
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) A.out[q][c] = v[q];
    }
    d2x_m = d2x;
    d2y_m = d2y;
    b_m[0] = b0;
    b_m[1] = b1;
    b_m[2] = b2;
    d0 = n0;
    d0x = n0x;
    d1 = n1;
    d1y = n1y;
#pragma unroll
    for (int q = 0; q < 3; ++q) em[q] = e[q];
    w_prev = w;
    w = w_next;
    cP += splane;
    zr += T(1);
  }
  cp_async_wait<0>();
}

// ---- E step -----------------------------------------------------------------------------------
// d_out = d + coef (4 pi/c J - div h(b, x)) at advanced edge locations.  The time-centred step is two launches: the
// predictor d* (x = d, coef = dx4 / 2) and the update (x = d*, coef = dx4); the literal step is one (x = d).
// (One launch for both, with h of d and of d* in one march, overlaps patches by 3 cells instead of 1 and needs
// two barriers a plane and 80 registers: slower at every size, see the figures above.)
// Patch: threads (tx, ty) at x = x0 + tx, y = y0 + ty, h at the patch of each plane of the chunk and of the plane
// below it; cells with tx >= 1 and ty >= 1 are updated (the divergence reaches -1).  Iteration q reads the staged
// planes q and q + 1 (q + 2 in flight) for h of plane q and updates plane q - 1 from the h that the last iteration
// left in the other half of H: one barrier a plane.
template <typename T, int BY>
struct EStepSmem {
  Plane3<T, BY> Sb[4], Sx[4];
  T H[2][3][BY][kTX];
};

template <typename T, int BY>
__device__ __forceinline__ void e_step_tile(const Grid& g, const EStepArgs<T>& A, const TileGrid& t, int block,
                                            EStepSmem<T, BY>& sm) {
  int tile_x, tile_y, zs;
  decode_tile(t, block, tile_x, tile_y, zs);
  const int ze = min(zs + t.zchunk, g.nz - 2);
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int cx = tx + 1, cy = ty + 1;
  const int x0 = 1 + tile_x * (kTX - 1), y0 = 1 + tile_y * (BY - 1);
  const int x = x0 + tx, y = y0 + ty;
  const bool conv_xy = x <= g.nx - 2 && y <= g.ny - 2;  // (x, y >= 1)
  const bool out_xy = x <= g.nx - 3 && y <= g.ny - 3 && tx >= 1 && ty >= 1;
  const bool own = A.x[0] == A.d[0];
  const T xr = (T)x - A.K.xc, yr = (T)y - A.K.yc;
  const Stager<BY> st(g, x0, y0);
  for (int q = zs - 2; q <= zs; ++q) {
    st.stage(g, A.b, q, sm.Sb[q & 3]);
    st.stage(g, A.x, q, sm.Sx[q & 3]);
  }
  cp_async_commit();
  copy_shell<T>(g, A.d, A.out, block, t.count());
  cp_async_wait<0>();
  __syncthreads();
  // carried from plane q - 1: b_x summed over the x pair, b_y over the y pair; h, d and J there, and h of plane q - 2
  T b0x_m, b1y_m;
  {
    const Plane3<T, BY>& B = sm.Sb[(zs - 2) & 3];
    b0x_m = B.v[0][cy][cx] + B.v[0][cy][cx + 1];
    b1y_m = B.v[1][cy][cx] + B.v[1][cy + 1][cx];
  }
  T hm[3] = {T(0), T(0), T(0)}, hmm[2] = {T(0), T(0)}, dm[3] = {T(0), T(0), T(0)};
  double jm[3] = {0.0, 0.0, 0.0};
  const int splane = g.nx * g.ny;
  long long cq = ((long long)(zs - 1) * g.ny + y) * g.nx + x;  // the cell in plane q
  T zr = (T)(zs - 1) - A.K.zc;
  uint16_t w_prev = 0, w = conv_xy ? __ldg(A.loc + cq) : (uint16_t)0;  // flags of planes q - 1, q
  for (int q = zs - 1; q <= ze; ++q) {
    if (q + 2 <= ze) {
      st.stage(g, A.b, q + 2, sm.Sb[(q + 2) & 3]);
      st.stage(g, A.x, q + 2, sm.Sx[(q + 2) & 3]);
    }
    cp_async_commit();
    // loaded one iteration ahead: the flags of plane q + 1, J and (where it is not staged) d of plane q
    const uint16_t w_next = conv_xy && q < ze ? __ldg(A.loc + cq + splane) : (uint16_t)0;
    double jq[3] = {0.0, 0.0, 0.0};
    T dq[3] = {T(0), T(0), T(0)};
    if (out_xy && q < ze) {
#pragma unroll
      for (int al = 0; al < 3; ++al) jq[al] = __ldg(A.J[al] + cq);
      if (!own) {
#pragma unroll
        for (int al = 0; al < 3; ++al) dq[al] = __ldg(A.d[al] + cq);
      }
    }
    cp_async_wait<1>();  // planes up to q + 1 have landed
    __syncthreads();
    T h[3] = {T(0), T(0), T(0)};
    if (q < ze && conv_xy) {
      const Plane3<T, BY>&B = sm.Sb[q & 3], &Bn = sm.Sb[(q + 1) & 3], &X = sm.Sx[q & 3], &Xn = sm.Sx[(q + 1) & 3];
      auto metric = [&](int l) { return metric_at<T>(A.K, A.met, g.ncell, cq, l, xr, yr, zr, exc(w, l)); };
      // (sums over points in the order z, y, x)
      const T b0 = B.v[0][cy][cx], b0r = B.v[0][cy][cx + 1], b1 = B.v[1][cy][cx], b1u = B.v[1][cy + 1][cx];
      const T b2 = B.v[2][cy][cx], b2n = Bn.v[2][cy][cx];
      const T x0v = X.v[0][cy][cx], x1v = X.v[1][cy][cx], x2v = X.v[2][cy][cx];
      h[0] = face_h<0>(metric(3), b0, B.v[1][cy][cx - 1] + b1 + B.v[1][cy + 1][cx - 1] + b1u,
                       B.v[2][cy][cx - 1] + b2 + Bn.v[2][cy][cx - 1] + b2n, x1v + Xn.v[1][cy][cx],
                       x2v + X.v[2][cy + 1][cx]);
      h[1] = face_h<1>(metric(4), b1, B.v[2][cy - 1][cx] + b2 + Bn.v[2][cy - 1][cx] + b2n,
                       B.v[0][cy - 1][cx] + B.v[0][cy - 1][cx + 1] + b0 + b0r, x2v + X.v[2][cy][cx + 1],
                       x0v + Xn.v[0][cy][cx]);
      h[2] = face_h<2>(metric(5), b2, b0x_m + b0 + b0r, b1y_m + b1 + b1u, x0v + X.v[0][cy + 1][cx],
                       x1v + X.v[1][cy][cx + 1]);
      b0x_m = b0 + b0r;
      b1y_m = b1 + b1u;
      if (own) {
        dq[0] = x0v;
        dq[1] = x1v;
        dq[2] = x2v;
      }
    }
#pragma unroll
    for (int al = 0; al < 3; ++al) sm.H[q & 1][al][ty][tx] = h[al];
    // d_out at plane q - 1: div_al h, F^{al nu} = +-h_q with q = 3 - al - nu, backward differences (Eq. 12)
    const int p = q - 1;
    if (p >= zs && out_xy) {
      const long long c = cq - splane;
      const T(&M)[3][BY][kTX] = sm.H[p & 1];
      const T dv[3] = {(hm[2] - M[2][ty - 1][tx]) - (hm[1] - hmm[1]), (hm[0] - hmm[0]) - (hm[2] - M[2][ty][tx - 1]),
                       (hm[1] - M[1][ty][tx - 1]) - (hm[0] - M[0][ty - 1][tx])};
      T v[3];
#pragma unroll
      for (int al = 0; al < 3; ++al)
        v[al] = adv(w_prev, al) ? dm[al] + (source<T>(A.K, jm[al]) - dv[al]) * A.coef : dm[al];
      if (A.tgt[0] && in_layer(w_prev)) {
        const T ko = outer_kappa<T>(g, x, y, p);
#pragma unroll
        for (int al = 0; al < 3; ++al)
          if (adv(w_prev, al)) v[al] = relax<T>(g, A.kin, w_prev, ko, A.tgt[al][c], v[al], al, x, y, p);
      }
#pragma unroll
      for (int al = 0; al < 3; ++al) A.out[al][c] = v[al];
    }
    hmm[0] = hm[0];
    hmm[1] = hm[1];
#pragma unroll
    for (int al = 0; al < 3; ++al) {
      hm[al] = h[al];
      dm[al] = dq[al];
      jm[al] = jq[al];
    }
    w_prev = w;
    w = w_next;
    cq += splane;
    zr += T(1);
  }
  cp_async_wait<0>();
}

// Resident blocks per SM: 64 registers a thread for the FP32 patches, 128 for the FP64 ones.
constexpr int patch_blocks(size_t word, int rows) { return (word == 4 ? 32 : 16) / rows; }

// Chunks of at most z planes, as many as nzi planes take, made as equal as they can be.
inline int even_chunk(int nzi, int z) {
  const int nc = (nzi + z - 1) / z;
  return (nzi + nc - 1) / nc;
}

// Patches over the advanced cells [2, n-3] per axis (31 x (rows - 1) cells each), and the split of z that minimises the
// estimated time: a chunk marches `halo` planes beyond its own and the busiest of the `slots` runs
// ceil(patches / slots) of them.
TileGrid tile_grid(const Grid& g, int rows, int slots, double* cost_out = nullptr) {
  TileGrid t;
  const int ox = kTX - 1, oy = rows - 1;
  const int halo = 2;
  const int nzi = g.nz - 4;
  t.ntx = (g.nx - 4 + ox - 1) / ox;
  t.nty = (g.ny - 4 + oy - 1) / oy;
  double best = 1e300;
  for (int z = std::min(nzi, 64); z >= 1; --z) {  // (by the length: by the number of chunks, a long grid has too many)
    const int zc = even_chunk(nzi, z);
    const long long nt = (long long)t.ntx * t.nty * ((nzi + zc - 1) / zc);
    const double per_slot = std::ceil((double)nt / slots);
    const double cost = per_slot * (zc + halo);  // time ~ blocks of the busiest slot x planes marched
    if (cost < best * 0.999) {
      best = cost;
      t.zchunk = zc;
    }
  }
  t.ntz = (nzi + t.zchunk - 1) / t.zchunk;
  if (cost_out) *cost_out = best;
  return t;
}

template <typename T, int BY>
__global__ void __launch_bounds__(kTX * BY, patch_blocks(sizeof(T), BY))
    k_b_step(const Grid g, const BStepArgs<T> A, const TileGrid t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<BStepSmem<T, BY>*>(smem_raw);
  b_step_tile<T, BY>(g, A, t, blockIdx.x, sm);
}

template <typename T, int BY>
__global__ void __launch_bounds__(kTX * BY, patch_blocks(sizeof(T), BY))
    k_e_step(const Grid g, const EStepArgs<T> A, const TileGrid t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<EStepSmem<T, BY>*>(smem_raw);
  e_step_tile<T, BY>(g, A, t, blockIdx.x, sm);
}

// ---- batched: one block per entry of a table of (instance, patch) work items ---------------------
// which (B): 0 first half (b[0] -> b[1]), 1 second half; (E): 0 predictor (into b[1], free by then), 1 update.
// The instance's d buffer parity is read from the device (flipped by launch_batch_flip_d at the end of a step).
template <typename T>
__device__ __forceinline__ const FieldConsts<T>& inst_consts(const InstDesc<T>& D) {
  if constexpr (sizeof(T) == sizeof(float))
    return D.K32;
  else
    return D.K64;
}

template <typename T>
__device__ __forceinline__ BStepArgs<T> batch_b_args(const InstDesc<T>& D, int which, bool literal) {
  BStepArgs<T> A;
  const int dc = *D.dcur;
  A.K = inst_consts(D);
  const T dx4 = A.K.dx4;
  for (int q = 0; q < 3; ++q) {
    A.d[q] = D.FS.d[dc][q];
    if (which == 0) {
      A.src[q] = D.FS.b[0][q];
      A.base[q] = D.FS.b[0][q];
      A.out[q] = D.FS.b[1][q];
    } else {
      A.src[q] = D.FS.b[1][q];
      A.base[q] = literal ? D.FS.b[1][q] : D.FS.b[0][q];
      A.out[q] = D.FS.b[0][q];
    }
  }
  for (int q = 0; q < 3; ++q) A.tgt[q] = which == 1 ? D.FS.tgt[3 + q] : nullptr;
  A.kin = D.FS.kin;
  A.loc = D.FS.loc;
  A.met = D.FS.met;
  A.coef = (which == 1 && !literal) ? dx4 : dx4 * T(0.5);
  A.inplace = which == 1 && !literal;
  return A;
}

template <typename T>
__device__ __forceinline__ EStepArgs<T> batch_e_args(const InstDesc<T>& D, int which, bool literal) {
  EStepArgs<T> A;
  const int dc = *D.dcur;
  A.K = inst_consts(D);
  const bool pred = which == 0;
  for (int q = 0; q < 3; ++q) {
    A.b[q] = D.FS.b[0][q];
    A.d[q] = D.FS.d[dc][q];
    A.x[q] = pred || literal ? D.FS.d[dc][q] : D.FS.b[1][q];
    A.out[q] = pred ? D.FS.b[1][q] : D.FS.d[dc ^ 1][q];
    A.J[q] = D.FS.J[q];
    A.tgt[q] = pred ? nullptr : D.FS.tgt[q];
  }
  A.coef = pred ? A.K.dx4 * T(0.5) : A.K.dx4;
  A.kin = D.FS.kin;
  A.loc = D.FS.loc;
  A.met = D.FS.met;
  return A;
}

template <typename T, int BY>
__global__ void __launch_bounds__(kTX * BY, patch_blocks(sizeof(T), BY))
    k_batch_b_step(const InstDesc<T>* __restrict__ desc, const BlockEntry* __restrict__ blk, int which, bool literal) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BStepArgs<T> A;  // (in registers, as a kernel parameter is not, it would spill)
  __shared__ Grid g;
  auto& sm = *reinterpret_cast<BStepSmem<T, BY>*>(smem_raw);
  const BlockEntry e = blk[blockIdx.x];
  const InstDesc<T>& D = desc[e.inst];
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    A = batch_b_args(D, which, literal);
    g = D.g;
  }
  const TileGrid t = D.tiles;
  __syncthreads();
  b_step_tile<T, BY>(g, A, t, e.block, sm);
}

template <typename T, int BY>
__global__ void __launch_bounds__(kTX * BY, patch_blocks(sizeof(T), BY))
    k_batch_e_step(const InstDesc<T>* __restrict__ desc, const BlockEntry* __restrict__ blk, int which, bool literal) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ EStepArgs<T> A;
  __shared__ Grid g;
  auto& sm = *reinterpret_cast<EStepSmem<T, BY>*>(smem_raw);
  const BlockEntry e = blk[blockIdx.x];
  const InstDesc<T>& D = desc[e.inst];
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    A = batch_e_args(D, which, literal);
    g = D.g;
  }
  const TileGrid t = D.tiles;
  __syncthreads();
  e_step_tile<T, BY>(g, A, t, e.block, sm);
}

template <typename T>
__global__ void k_batch_zero_j(const InstDesc<T>* __restrict__ desc, const BlockEntry* __restrict__ blk, int nblk) {
  for (int bi = blockIdx.x; bi < nblk; bi += gridDim.x) {
    const BlockEntry e = blk[bi];
    const InstDesc<T>& D = desc[e.inst];
    const long long c = (long long)e.block * blockDim.x + threadIdx.x;
    if (c < D.g.ncell) {
      D.FS.J[0][c] = 0.0;
      D.FS.J[1][c] = 0.0;
      D.FS.J[2][c] = 0.0;
    }
  }
}

template <typename T>
__global__ void k_batch_flip_d(const InstDesc<T>* __restrict__ desc, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) *desc[i].dcur ^= 1;
}

// ---- location flags --------------------------------------------------------------------------
// bit l: location l of the cell is advanced (cell in [2, n-3]^3 and r >= r_excise); bit 6: an
// advanced location of the cell has a relaxation kappa > 0; bit 7: one from the inner layer;
// bit 8 + l: location l is excised
// (r < r_excise, or r = 0), where conversions take the flat metric.  Decided once, in FP64.
__global__ void k_location_flags(const Grid g, uint16_t* __restrict__ loc) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const int i = (int)(c % g.nx);
  const int j = (int)((c / g.nx) % g.ny);
  const int k = (int)(c / ((long long)g.nx * g.ny));
  const bool inner = i >= 2 && i <= g.nx - 3 && j >= 2 && j <= g.ny - 3 && k >= 2 && k <= g.nz - 3;
  unsigned w = 0;
#pragma unroll
  for (int l = 0; l < 6; ++l) {
    const double X = i + 0.5 * half(l, 0) - g.xc;
    const double Y = j + 0.5 * half(l, 1) - g.yc;
    const double Z = k + 0.5 * half(l, 2) - g.zc;
    const Kerr<double> K = kerr_eval<double>(X, Y, Z, g.m, g.a);
    const bool excised = K.flat || K.r < g.r_exc;
    if (excised) w |= 1u << (8 + l);
    if (inner && !excised) {
      w |= 1u << l;
      if (outer_kappa<double>(g, i, j, k) > 0.0) w |= kLayerBit;
      // (the box holds every such cell by construction; checked so that no lookup can leave it)
      const bool in_box = i >= g.kbox0[0] && i < g.kbox0[0] + g.kboxn[0] && j >= g.kbox0[1] &&
                          j < g.kbox0[1] + g.kboxn[1] && k >= g.kbox0[2] && k < g.kbox0[2] + g.kboxn[2];
      if (in_box && inner_kappa(g, l, i, j, k) > 0.0) w |= kLayerBit | kInnerBit;
    }
  }
  loc[c] = (uint16_t)w;
}

// ---- initial conditions / conversions ----------------------------------------------------
// b_Q = h_Q + f (v x k)_Q at its face with v = k x h + d, the contravariant (h, d) uniform (g = eta + f k k
// lowers the tensor of Eq. 8).  FP64-pipe bound: FastOps64, and the excised locations from the flags.
// At 128^3: 847 -> 577 us.
template <int Q, typename T>
__device__ __forceinline__ T uniform_b(const Grid& g, int i, int j, int k, bool excised, const double h[3],
                                       const double d[3]) {
  if (excised || !(g.m > 0.0)) return (T)h[Q];
  constexpr int L = 3 + Q, M = (Q + 1) % 3, N = (Q + 2) % 3;
  const Kerr<double> K = kerr_eval_fast(i + 0.5 * half(L, 0) - g.xc, j + 0.5 * half(L, 1) - g.yc,
                                        k + 0.5 * half(L, 2) - g.zc, g.m, g.a);
  const double kv[3] = {K.k0, K.k1, K.k2};
  const double vM = fma(kv[N], h[Q], fma(-kv[Q], h[N], d[M])), vN = fma(kv[Q], h[M], fma(-kv[M], h[Q], d[N]));
  return narrow_t<T>(fma(K.f, fma(vM, kv[N], -(kv[M] * vN)), h[Q]));
}

template <typename T>
__global__ void k_uniform_field(const Grid g, const Fields<T> F, const uint16_t* __restrict__ loc, double E0, double E1,
                                double E2, double B0, double B1, double B2) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const int i = (int)(c % g.nx);
  const int j = (int)((c / g.nx) % g.ny);
  const int k = (int)(c / ((long long)g.nx * g.ny));
  const uint16_t w = loc[c];
  const double h[3] = {B0, B1, B2};
  const double d[3] = {-E0, -E1, -E2};
  F.d[0][c] = (T)d[0];
  F.d[1][c] = (T)d[1];
  F.d[2][c] = (T)d[2];
  F.b[0][c] = uniform_b<0, T>(g, i, j, k, exc(w, 3), h, d);
  F.b[1][c] = uniform_b<1, T>(g, i, j, k, exc(w, 4), h, d);
  F.b[2][c] = uniform_b<2, T>(g, i, j, k, exc(w, 5), h, d);
}

// ---- read-out of the contravariant face components --------------------------------------------
// Sum of the points of source lattice SL nearest to the point of target lattice TL in cell
// (i, j, k), from global memory.
template <int TL, int SL, typename T>
__device__ __forceinline__ T sum_g(const T* __restrict__ F, const Grid& g, int i, int j, int k) {
  constexpr int lx = nb_lo(TL, SL, 0), hx = nb_hi(TL, SL, 0);
  constexpr int ly = nb_lo(TL, SL, 1), hy = nb_hi(TL, SL, 1);
  constexpr int lz = nb_lo(TL, SL, 2), hz = nb_hi(TL, SL, 2);
  T s = T(0);
#pragma unroll
  for (int dz = lz; dz <= hz; ++dz)
#pragma unroll
    for (int dy = ly; dy <= hy; ++dy)
#pragma unroll
      for (int dx = lx; dx <= hx; ++dx) s += F[((long long)(k + dz) * g.ny + (j + dy)) * g.nx + (i + dx)];
  return s;
}

template <int Q, typename T>
__device__ __forceinline__ double face_h_g(const Grid& g, const FieldConsts<T>& K, const Fields<T>& F, int i, int j,
                                           int k, bool excised) {
  constexpr int L = 3 + Q, M = (Q + 1) % 3, N = (Q + 2) % 3;
  const Pt<T> P = metric_pt<T>(K, L, (T)i - K.xc, (T)j - K.yc, (T)k - K.zc, excised);
  return (double)face_h<Q>(P, F.b[Q][((long long)k * g.ny + j) * g.nx + i], sum_g<L, 3 + M>(F.b[M], g, i, j, k),
                           sum_g<L, 3 + N>(F.b[N], g, i, j, k), sum_g<L, M>(F.d[M], g, i, j, k),
                           sum_g<L, N>(F.d[N], g, i, j, k));
}

// h (F^yz, F^zx, F^xy) at every b face of the cells 1 .. n-2 per axis, as the E step converts the
// field; zero on the outer index layer.
template <typename T>
__global__ void k_contra_h(const Grid g, const FieldConsts<T> K, const Fields<T> F, const uint16_t* __restrict__ loc,
                           double* __restrict__ h0, double* __restrict__ h1, double* __restrict__ h2) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const int i = (int)(c % g.nx);
  const int j = (int)((c / g.nx) % g.ny);
  const int k = (int)(c / ((long long)g.nx * g.ny));
  if (i < 1 || j < 1 || k < 1 || i > g.nx - 2 || j > g.ny - 2 || k > g.nz - 2) {
    h0[c] = h1[c] = h2[c] = 0.0;
    return;
  }
  const uint16_t w = loc[c];
  h0[c] = face_h_g<0, T>(g, K, F, i, j, k, exc(w, 3));
  h1[c] = face_h_g<1, T>(g, K, F, i, j, k, exc(w, 4));
  h2[c] = face_h_g<2, T>(g, K, F, i, j, k, exc(w, 5));
}

template <typename T>
__global__ void k_convert_in(T* __restrict__ dst, const double* __restrict__ src, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) dst[i] = narrow_t<T>(src[i]);
}
template <typename T>
__global__ void k_convert_out(double* __restrict__ dst, const T* __restrict__ src, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) dst[i] = widen_t(src[i]);
}

inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

template <typename T>
void launch_contra_h(const Grid& g, const Fields<T>& F, const uint16_t* loc, double* h3, cudaStream_t st) {
  k_contra_h<T><<<blocks_for(g.ncell, 256), 256, 0, st>>>(g, field_consts<T>(g), F, loc, h3, h3 + g.ncell,
                                                   h3 + 2 * g.ncell);
}
template void launch_contra_h<float>(const Grid&, const Fields<float>&, const uint16_t*, double*, cudaStream_t);
template void launch_contra_h<double>(const Grid&, const Fields<double>&, const uint16_t*, double*, cudaStream_t);

void launch_location_flags(const Grid& g, uint16_t* loc, cudaStream_t st) {
  k_location_flags<<<blocks_for(g.ncell, 256), 256, 0, st>>>(g, loc);
}

template <typename T>
__global__ void k_inner_kappa_table(const Grid g, T* __restrict__ kin, long long n) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int i = g.kbox0[0] + (int)(e % g.kboxn[0]);
  long long r = e / g.kboxn[0];
  const int j = g.kbox0[1] + (int)(r % g.kboxn[1]);
  r /= g.kboxn[1];
  const int k = g.kbox0[2] + (int)(r % g.kboxn[2]);
  const int l = (int)(r / g.kboxn[2]);
  kin[e] = (T)inner_kappa(g, l, i, j, k);
}

template <typename T>
void launch_inner_kappa_table(const Grid& g, T* kin, cudaStream_t st) {
  const long long n = 6ll * g.kboxn[0] * g.kboxn[1] * g.kboxn[2];
  if (n > 0) k_inner_kappa_table<T><<<blocks_for(n, 256), 256, 0, st>>>(g, kin, n);
}
template void launch_inner_kappa_table<float>(const Grid&, float*, cudaStream_t);
template void launch_inner_kappa_table<double>(const Grid&, double*, cudaStream_t);

__global__ void k_metric_table(const Grid g, const FieldConsts<double> K, const uint16_t* __restrict__ loc,
                               double2* __restrict__ met) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.ncell) return;
  const int i = (int)(c % g.nx);
  const int j = (int)((c / g.nx) % g.ny);
  const int k = (int)(c / ((long long)g.nx * g.ny));
  const uint16_t w = loc[c];
#pragma unroll 1
  for (int l = 0; l < 6; ++l) {
    const Pt<double> P = metric_pt<double>(K, l, i - K.xc, j - K.yc, k - K.zc, exc(w, l));
    met[2 * l * g.ncell + c] = make_double2(P.f, P.k0);
    met[(2 * l + 1) * g.ncell + c] = make_double2(P.k1, P.k2);
  }
}

void launch_metric_table(const Grid& g, const uint16_t* loc, double2* met, cudaStream_t st) {
  k_metric_table<<<blocks_for(g.ncell, 256), 256, 0, st>>>(g, field_consts<double>(g), loc, met);
}

// Dynamic shared memory of the field kernels (above the 48 KB default): set once per kernel.
template <typename K>
void allow_smem(K kernel, size_t bytes) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T, int BY>
void launch_b_rows(const Grid& g, const BStepArgs<T>& A, const TileGrid& t, cudaStream_t st) {
  constexpr size_t smem = sizeof(BStepSmem<T, BY>);
  static bool once = (allow_smem(k_b_step<T, BY>, smem), true);
  (void)once;
  k_b_step<T, BY><<<(unsigned)t.count(), dim3(kTX, BY), smem, st>>>(g, A, t);
}

template <typename T, int BY>
void launch_e_rows(const Grid& g, const EStepArgs<T>& A, const TileGrid& t, cudaStream_t st) {
  constexpr size_t smem = sizeof(EStepSmem<T, BY>);
  static bool once = (allow_smem(k_e_step<T, BY>, smem), true);
  (void)once;
  k_e_step<T, BY><<<(unsigned)t.count(), dim3(kTX, BY), smem, st>>>(g, A, t);
}

// FP32 patches (and the batched FP64 ones) have 16 rows.  Other FP64 patches, bound by the FP64 pipe whatever their
// shape, take the rows (8 or 16) with the lower estimated time: 16 waste less on the overlap, 8 divide a small grid
// more evenly.
// B step at 32^3 FP64: 8 rows 78 us, 16 rows 144 us (metric evaluated); E step at 64^3: 16 rows 393 us, 8 rows 607 us.
template <typename T>
TileGrid choose_rows(const Grid& g, int sms, int* rows) {
  double c16 = 0.0, c8 = 0.0;
  const TileGrid t16 = tile_grid(g, 16, sms * patch_blocks(sizeof(T), 16), &c16);
  *rows = 16;
  if (sizeof(T) == sizeof(float)) return t16;
  const TileGrid t8 = tile_grid(g, 8, sms, &c8);  // (two blocks share an SM's FP64 pipe)
  if (0.5 * c8 >= c16) return t16;
  *rows = 8;
  return t8;
}

template <typename T>
void launch_b_step(const Grid& g, const BStepArgs<T>& A, int sms, cudaStream_t st) {
  int rows;
  const TileGrid t = choose_rows<T>(g, sms, &rows);
  if constexpr (sizeof(T) == sizeof(double)) {
    if (rows == 8) return launch_b_rows<T, 8>(g, A, t, st);
  }
  launch_b_rows<T, 16>(g, A, t, st);
}

template <typename T>
void launch_e_step(const Grid& g, const EStepArgs<T>& A, int sms, cudaStream_t st) {
  int rows;
  const TileGrid t = choose_rows<T>(g, sms, &rows);
  if constexpr (sizeof(T) == sizeof(double)) {
    if (rows == 8) return launch_e_rows<T, 8>(g, A, t, st);
  }
  launch_e_rows<T, 16>(g, A, t, st);
}

// Patches of the instances of a batch (16 rows), the z chunks the ones (of one length for all) that minimise the
// estimated time as in tile_grid.
constexpr int kBatchRows = 16;
void batch_field_tiles(const Grid* const* grids, int n, size_t word, int sms, TileGrid* tiles) {
  const int slots = sms * patch_blocks(word, kBatchRows);
  for (int i = 0; i < n; ++i) tiles[i] = tile_grid(*grids[i], kBatchRows, 1);
  double best = 1e300;
  int zbest = 64;
  for (int zc = 64; zc >= 1; zc -= zc > 16 ? 4 : 1) {
    long long nt = 0;
    for (int i = 0; i < n; ++i)
      nt += (long long)tiles[i].ntx * tiles[i].nty * ((grids[i]->nz - 4 + zc - 1) / zc);
    const double cost = std::ceil((double)nt / slots) * (zc + 2);
    if (cost < best * 0.999) {
      best = cost;
      zbest = zc;
    }
  }
  for (int i = 0; i < n; ++i) {
    tiles[i].zchunk = zbest;
    tiles[i].ntz = (grids[i]->nz - 4 + zbest - 1) / zbest;
  }
}

template <typename T>
void launch_batch_b_half(const BatchTables<T>& bt, int which, bool literal, cudaStream_t st) {
  constexpr int BY = kBatchRows;
  constexpr size_t smem = sizeof(BStepSmem<T, BY>);
  static bool once = (allow_smem(k_batch_b_step<T, BY>, smem), true);
  (void)once;
  if (bt.ntile == 0) return;
  k_batch_b_step<T, BY><<<bt.ntile, dim3(kTX, BY), smem, st>>>(bt.desc, bt.tile, which, literal);
}

template <typename T>
void launch_batch_e_step(const BatchTables<T>& bt, int which, bool literal, cudaStream_t st) {
  constexpr int BY = kBatchRows;
  constexpr size_t smem = sizeof(EStepSmem<T, BY>);
  static bool once = (allow_smem(k_batch_e_step<T, BY>, smem), true);
  (void)once;
  if (bt.ntile == 0) return;
  k_batch_e_step<T, BY><<<bt.ntile, dim3(kTX, BY), smem, st>>>(bt.desc, bt.tile, which, literal);
}

template <typename T>
void launch_batch_zero_j(const BatchTables<T>& bt, cudaStream_t st) {
  k_batch_zero_j<T><<<std::min(bt.nall, bt.persist_blocks), 256, 0, st>>>(bt.desc, bt.all, bt.nall);
}

template <typename T>
void launch_batch_flip_d(const BatchTables<T>& bt, int ninst, cudaStream_t st) {
  k_batch_flip_d<T><<<(ninst + 127) / 128, 128, 0, st>>>(bt.desc, ninst);
}

template <typename T>
void launch_uniform_field(const Grid& g, const Fields<T>& F, const uint16_t* loc, const double E[3], const double B[3],
                          cudaStream_t st) {
  k_uniform_field<T><<<blocks_for(g.ncell, 256), 256, 0, st>>>(g, F, loc, E[0], E[1], E[2], B[0], B[1], B[2]);
}

__global__ void k_add_f64(double* __restrict__ dst, const double* __restrict__ src, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) dst[i] += src[i];
}

void launch_add_f64(double* dst, const double* src, long long n, cudaStream_t st) {
  if (n > 0) k_add_f64<<<blocks_for(n, 256), 256, 0, st>>>(dst, src, n);
}

template <typename T>
void launch_convert_in(T* dst, const double* src, long long n, cudaStream_t st) {
  k_convert_in<T><<<blocks_for(n, 256), 256, 0, st>>>(dst, src, n);
}
template <typename T>
void launch_convert_out(double* dst, const T* src, long long n, cudaStream_t st) {
  k_convert_out<T><<<blocks_for(n, 256), 256, 0, st>>>(dst, src, n);
}

#define GRPIC_INST_FIELDS(T)                                                                             \
  template void launch_b_step<T>(const Grid&, const BStepArgs<T>&, int, cudaStream_t);                  \
  template void launch_e_step<T>(const Grid&, const EStepArgs<T>&, int, cudaStream_t);                  \
  template void launch_uniform_field<T>(const Grid&, const Fields<T>&, const uint16_t*, const double*,   \
                                        const double*, cudaStream_t);                                    \
  template void launch_convert_in<T>(T*, const double*, long long, cudaStream_t);                       \
  template void launch_convert_out<T>(double*, const T*, long long, cudaStream_t);                      \
  template void launch_batch_b_half<T>(const BatchTables<T>&, int, bool, cudaStream_t);                 \
  template void launch_batch_e_step<T>(const BatchTables<T>&, int, bool, cudaStream_t);                      \
  template void launch_batch_zero_j<T>(const BatchTables<T>&, cudaStream_t);                            \
  template void launch_batch_flip_d<T>(const BatchTables<T>&, int, cudaStream_t);

GRPIC_INST_FIELDS(float)
GRPIC_INST_FIELDS(double)

}  // namespace grpic
