// Diagnostics of the current: charge density at the nodes and the Gauss-law residual.
//
// rho (or J^4 / c with gamma): cloud-in-cell charge of each particle at the 8 nodes around it,
// weights trilinear in the position (the sqrt(-det g) sub-volumes of Sec. 3.3 reduce to that, det g
// being -1), times gamma = u^4 / c for the time component of J = rho gamma v (Sec. 4).
// Gauss residual at node (i, j, k): div E - 4 pi rho with E^a = -d^a = -F^{a4} and backward
// differences of the edge-centred d (the node's own edge minus the one below it on each axis),
// the discrete divergence that the E step (Eq. 12) and the zig-zag deposit keep consistent: with
// the gamma-free deposit in flat space it changes per step by exactly -4 pi times the deposit's
// 3-D continuity defect.
//
// Invariants of each particle's motion: the normalisation g_mn u^m u^n = -c^2 (Eq. 7), kept by the
// exact dynamics in any field (F is antisymmetric), and the Killing energy E = -u_4 and axial
// momentum L = u_phi = x u_y - y u_x (covariant components, position from the centre), kept along
// field-free orbits (the metric is stationary and axisymmetric; Eq. 3).  Evaluated in FP64 from the
// stored state.
#include <cmath>

#include "common.cuh"
#include "metric.cuh"

namespace grpic {

namespace {

__device__ __forceinline__ double to_f64(float v) { return widen(v); }
__device__ __forceinline__ double to_f64(double v) { return v; }

// The cloud of one particle in FP64: eight atomics.  The weights are formed without the charge, so that their rounding is
// the same for particles of opposite charge at one place (a pair plasma's start) and cancels with it.
template <typename T>
__device__ __forceinline__ void cloud64(const Particles<T>& P, long long i, double q, int nx, int ny, int nz,
                                        double inv_c, bool with_gamma, double* __restrict__ rho) {
  const double x[3] = {to_f64(P.x[0][i]), to_f64(P.x[1][i]), to_f64(P.x[2][i])};
  const int nn[3] = {nx, ny, nz};
  int c[3];
  double w[3];
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    double fl;
    floor_split(x[ax], c[ax], fl);
    const int k = min(max(c[ax], 0), nn[ax] - 2);
    w[ax] = x[ax] - (k == c[ax] ? fl : (double)k);
    c[ax] = k;
  }
  const double qq = with_gamma ? q * to_f64(P.u[3][i]) * inv_c : q;
  const double wx[2] = {1.0 - w[0], w[0]}, wy[2] = {1.0 - w[1], w[1]}, wz[2] = {1.0 - w[2], w[2]};
  double* r = rho + ((long long)c[2] * ny + c[1]) * nx + c[0];
#pragma unroll
  for (int dj = 0; dj < 2; ++dj)
#pragma unroll
    for (int di = 0; di < 2; ++di) {
      const double wxy = wx[di] * wy[dj];
#pragma unroll
      for (int dk = 0; dk < 2; ++dk) atomicAdd(r + (long long)dk * nx * ny + dj * nx + di, qq * (wxy * wz[dk]));
    }
}

__global__ void k_charge_density(const Particles<double> P, double q, int nx, int ny, int nz, double inv_c,
                                 bool with_gamma, double* __restrict__ rho) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= P.n || i >= (long long)(*P.n_dev) || P.key[i] == kDead) return;
  cloud64(P, i, q, nx, ny, nz, inv_c, with_gamma, rho);
}

// v = (hi 2^64 + lo) 2^-s in FP64, v > 0 and below 2^(32 W), rounded once (halves upwards): the integers become the
// bits of the result, since conversions would run on the FP64 pipe.
template <int W>
__device__ __forceinline__ double scaled_double(unsigned long long hi, unsigned long long lo, int s) {
  unsigned w[4] = {(unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32)};
  int top = 32 * W - 1;  // the position of bit 31 of the leading word
#pragma unroll
  for (int k = 1; k < W; ++k)
    if (w[W - 1] == 0) {
#pragma unroll
      for (int q = W - 1; q > 0; --q) w[q] = w[q - 1];
      w[0] = 0;
      top -= 32;
    }
  const int lz = __clz(w[W - 1]);
  const unsigned m1 = __funnelshift_l(w[W - 2], w[W - 1], lz);
  const unsigned m0 = __funnelshift_l(W > 2 ? w[W - 3] : 0u, w[W - 2], lz);
  // the leading one of m1 >> 11 adds 1 to the exponent field
  const unsigned long long m = ((unsigned long long)m1 << 21 | m0 >> 11) + ((m0 >> 10) & 1u);
  return __longlong_as_double((long long)m + ((long long)((1022 + top - lz - s) << 20) << 32));
}

// FP32 positions.  One FP64 warp instruction takes 16 cycles of an SM, and the eight weights of a particle, its
// floors and conversions took about 36 of them besides eight atomics.  But a weight of an FP32 coordinate x >= 1 is
// an integer multiple of 2^-23, so the sum of a node's weights over the particles of a cell is an exact integer (69
// bits, with gamma 32 more), rounded once when it is complete.  A warp finds the runs of equal cells among its
// particles (after a sort nearly all particles of a cell) and cuts them to kRun; a few lanes take a run from shared
// memory: one FP64 multiplication and one atomic a node for up to kRun particles.  Without gamma four lanes a run,
// each an x pair of its nodes (the lower node's sum is that of w_y w_z less the upper's); with gamma eight, for the
// wider products make the pair slower (136 us for 123 below).  kRun = 8: the sums stay in 64-bit parts, and with 8
// particles a cell the 4 or 5 runs of a warp fill its lanes.
// gamma: u^4 as a 32-bit integer times a power of two common to the warp, exact while the exponents of its particles
// lie within 8.  A warp with a wider range, or a coordinate below 1 or beyond the last cell, takes cloud64.
// Bound by instruction issue (73 % of the slots).  Measured (6.4 M particles a species, 8 a cell, 96^3): 487 -> 82 us a
// species, with gamma 123.
constexpr int kRun = 8;
template <bool GAMMA>
__global__ void __launch_bounds__(256)
    k_charge_density_runs(const Particles<float> P, double q, int nx, int ny, int nz, double inv_c,
                          double* __restrict__ rho) {
  __shared__ uint4 s_w[8][32];   // 2^23 (w_x, w_y, w_z) and u^4 of the lanes' particles
  __shared__ int2 s_run[8][32];  // the runs: cell, first lane | length << 8
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool live = false;
  float x[3] = {1.f, 1.f, 1.f}, u = 1.f;
  if (i < P.n) {  // all loads in flight together
    const int n = *P.n_dev;
    const uint32_t key = P.key[i];
    x[0] = P.x[0][i];
    x[1] = P.x[1][i];
    x[2] = P.x[2][i];
    if (GAMMA) u = P.u[3][i];
    live = i < n && key != kDead;
  }
  // (NaN fails)
  bool exact = x[0] >= 1.f && x[0] < (float)(nx - 1) && x[1] >= 1.f && x[1] < (float)(ny - 1) && x[2] >= 1.f &&
               x[2] < (float)(nz - 1);
  const int ub = __float_as_int(u), e = ub >> 23;  // (the sign makes e negative)
  int emax = 0;
  if (GAMMA) {
    emax = __reduce_max_sync(0xffffffffu, live ? e : 0);
    exact = exact && (!live || (e >= 1 && e < 255 && emax - e <= 8));
  }
  if (!__all_sync(0xffffffffu, exact || !live)) {
    if (live) cloud64(P, i, q, nx, ny, nz, inv_c, GAMMA, rho);
    return;
  }
  const int c0 = (int)x[0], c1 = (int)x[1], c2 = (int)x[2];
  const int cell = live ? (c2 * ny + c1) * nx + c0 : -1;
  const float one = 8388608.f;
  uint4 v;
  v.x = (unsigned)((x[0] - (float)c0) * one);
  v.y = (unsigned)((x[1] - (float)c1) * one);
  v.z = (unsigned)((x[2] - (float)c2) * one);
  v.w = GAMMA && live ? (unsigned)((ub & 0x7fffff) | 0x800000) << (8 - (emax - e)) : 0u;
  s_w[warp][lane] = v;
  const int before = __shfl_up_sync(0xffffffffu, cell, 1);
  const unsigned starts = __ballot_sync(0xffffffffu, lane == 0 || cell != before);
  const unsigned upto = 0xffffffffu >> (31 - lane);  // this lane and those before it
  const int start = 31 - __clz(starts & upto);
  const bool head = live && ((lane - start) % kRun) == 0;
  const unsigned heads = __ballot_sync(0xffffffffu, head);
  if (head) {
    const unsigned later = starts & ~upto;
    const int end = later ? __ffs(later) - 1 : 32;
    s_run[warp][__popc(heads & upto) - 1] = make_int2(cell, lane | (min(end - lane, kRun) << 8));
  }
  __syncwarp();
  const double scale = GAMMA ? q * inv_c : q;
  // integer sums are in units of 2^-69, with gamma u^4 = U 2^(emax - 158)
  const int bits = GAMMA ? 69 + 158 - emax : 69;
  constexpr int kLanes = GAMMA ? 8 : 4;
  const int tasks = kLanes * __popc(heads);
  for (int t = lane; t < tasks; t += 32) {
    const int2 run = s_run[warp][t / kLanes];
    const int first = run.y & 255, len = run.y >> 8;
    const int sgy = t & 1 ? 1 : -1, sgz = t & 2 ? 1 : -1, sgx = t & 4 ? 1 : -1;
    const int ofy = t & 1 ? 0 : 0x800000, ofz = t & 2 ? 0 : 0x800000, ofx = t & 4 ? 0 : 0x800000;
    double* r = rho + ((long long)run.x + (t & 1 ? nx : 0) + (t & 2 ? nx * ny : 0));
    unsigned long long hi = 0, lo = 0, sum = 0, sum_hi = 0;
    for (int p = first; p < first + len; ++p) {
      const uint4 w = s_w[warp][p];
      const unsigned wy = (unsigned)((int)w.y * sgy + ofy), wz = (unsigned)((int)w.z * sgz + ofz);
      const unsigned long long a = (unsigned long long)wy * wz;
      if (GAMMA) {
        const unsigned long long b = (unsigned long long)(unsigned)((int)w.x * sgx + ofx) * w.w, l = a * b;
        lo += l;
        hi += __umul64hi(a, b) + (lo < l);
      } else {
        sum += a;
        lo += (unsigned long long)(unsigned)a * w.x;
        sum_hi += (unsigned long long)(unsigned)(a >> 32) * w.x;
      }
    }
    if (GAMMA) {
      if (hi | lo) atomicAdd(r + (t & 4 ? 1 : 0), scale * scaled_double<4>(hi, lo, bits));
    } else {
      const unsigned long long l = lo;
      lo += sum_hi << 32;
      hi = (sum_hi >> 32) + (lo < l);
      const unsigned long long rest = (sum << 23) - lo, rest_hi = (sum >> 41) - hi - ((sum << 23) < lo);
      if (rest | rest_hi) atomicAdd(r, scale * scaled_double<3>(rest_hi, rest, bits));
      if (hi | lo) atomicAdd(r + 1, scale * scaled_double<3>(hi, lo, bits));
    }
  }
}

// res = div E - 4 pi rho; the max of |res| over nodes [lo, n - 1 - lo]^3 goes to *maxabs
// (atomicMax on the bit pattern of the non-negative double).
template <typename T>
__global__ void k_gauss(const T* __restrict__ dx, const T* __restrict__ dy, const T* __restrict__ dz,
                        const double* __restrict__ rho, int nx, int ny, int nz, int lo, double* __restrict__ res,
                        unsigned long long* maxabs) {
  const unsigned node = blockIdx.x * blockDim.x + threadIdx.x;  // (ncell < 2^31)
  double worst = 0.0;
  if (node < (unsigned)(nx * ny * nz)) {
    const int idx = (int)node, i = idx % nx, r = idx / nx, j = r % ny, k = r / ny;
    double div = 0.0;
    if (i > 0) div -= to_f64(dx[idx]) - to_f64(dx[idx - 1]);
    if (j > 0) div -= to_f64(dy[idx]) - to_f64(dy[idx - nx]);
    if (k > 0) div -= to_f64(dz[idx]) - to_f64(dz[idx - nx * ny]);
    const double v = div - 4.0 * M_PI * rho[idx];
    if (res) res[idx] = v;
    if (i >= lo && j >= lo && k >= lo && i <= nx - 1 - lo && j <= ny - 1 - lo && k <= nz - 1 - lo) worst = fabs(v);
  }
  // warp maximum of the bit patterns (a NaN is above any number, fmax passes over it: taken as 0), one atomic per warp
  unsigned long long w = (unsigned long long)__double_as_longlong(worst);
  if (w > 0x7ff0000000000000ull) w = 0;
  const unsigned whi = __reduce_max_sync(0xffffffffu, (unsigned)(w >> 32));
  const unsigned wlo = __reduce_max_sync(0xffffffffu, (unsigned)(w >> 32) == whi ? (unsigned)w : 0u);
  if ((threadIdx.x & 31) == 0 && (whi | wlo)) atomicMax(maxabs, ((unsigned long long)whi << 32) | wlo);
}

// Sums and maxima of the invariant statistics (maxima of non-negative doubles as bit patterns).
struct InvAcc {
  unsigned long long n, tracked;
  double norm_sum, e_sum, l_sum;
  unsigned long long norm_max, e_max, l_max;
  unsigned long long max_id;
};

__device__ __forceinline__ void warp_sum_max(double v, double* sum, unsigned long long* mx) {
  double s = v, m = v;
  for (int off = 16; off > 0; off >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, off);
    m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
  }
  if ((threadIdx.x & 31) == 0) {
    if (s != 0.0) atomicAdd(sum, s);
    if (m > 0.0) atomicMax(mx, (unsigned long long)__double_as_longlong(m));
  }
}

template <typename T>
__global__ void k_max_id(const Particles<T> P, unsigned long long* max_id) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const bool live = i < P.n && i < (long long)(*P.n_dev) && P.key[i] != kDead;
  // ids are 32-bit: one warp maximum, then one atomic per warp (a live id may be 0, so the warp
  // publishes only when it has a live particle)
  const unsigned v = live ? P.id[i] : 0u;
  const unsigned m = __reduce_max_sync(0xffffffffu, v);
  const unsigned any = __ballot_sync(0xffffffffu, live);
  if (any && (threadIdx.x & 31) == 0) atomicMax(max_id, (unsigned long long)m);
}

// mode 0: record E and L of the tracked particles (id % stride == 0) at slot id / stride; mode 1:
// compare with the recorded values.  The norm statistics cover every live particle.
template <typename T>
__global__ void k_invariants(const Grid g, const Particles<T> P, int mode, int stride, double* __restrict__ e0,
                             double* __restrict__ l0, long long nslots, InvAcc* acc) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const bool live = i < P.n && i < (long long)(*P.n_dev) && P.key[i] != kDead;
  double norm = 0.0, de = 0.0, dl = 0.0;
  bool cmp = false;
  if (live) {
    const double X = (double)P.x[0][i] - g.xc, Y = (double)P.x[1][i] - g.yc, Z = (double)P.x[2][i] - g.zc;
    const double u[4] = {(double)P.u[0][i], (double)P.u[1][i], (double)P.u[2][i], (double)P.u[3][i]};
    const Kerr<double> K = kerr_eval<double>(X, Y, Z, g.m, g.a);
    const double f = K.flat ? 0.0 : K.f;
    // u_m = g_mn u^n = eta_mn u^n + f k_m (k.u), k_4 = 1
    const double s = K.k0 * u[0] + K.k1 * u[1] + K.k2 * u[2] + u[3];
    const double uc[4] = {u[0] + f * s * K.k0, u[1] + f * s * K.k1, u[2] + f * s * K.k2, -u[3] + f * s};
    const double c2 = g.c * g.c;
    norm = fabs(u[0] * uc[0] + u[1] * uc[1] + u[2] * uc[2] + u[3] * uc[3] + c2) / c2;
    const double E = -uc[3], L = X * uc[1] - Y * uc[0];
    const unsigned id = P.id[i];
    if (id % (unsigned)stride == 0u) {
      const long long slot = id / (unsigned)stride;
      if (slot < nslots) {
        if (mode == 0) {
          e0[slot] = E;
          l0[slot] = L;
        } else if (!isnan(e0[slot])) {
          cmp = true;
          de = fabs(E - e0[slot]) / g.c;
          dl = fabs(L - l0[slot]) / g.c;
        }
      }
    }
  }
  const unsigned nl = __popc(__ballot_sync(0xffffffffu, live)), nc = __popc(__ballot_sync(0xffffffffu, cmp));
  if ((threadIdx.x & 31) == 0) {
    if (nl) atomicAdd(&acc->n, (unsigned long long)nl);
    if (nc) atomicAdd(&acc->tracked, (unsigned long long)nc);
  }
  warp_sum_max(norm, &acc->norm_sum, &acc->norm_max);
  warp_sum_max(de, &acc->e_sum, &acc->e_max);
  warp_sum_max(dl, &acc->l_sum, &acc->l_max);
}

}  // namespace

template <typename T>
void launch_invariants(const Grid& g, const Particles<T>& P, int mode, int stride, double* e0, double* l0,
                       long long nslots, void* acc, cudaStream_t stream) {
  if (P.n <= 0) return;
  k_invariants<T><<<(unsigned)((P.n + 255) / 256), 256, 0, stream>>>(g, P, mode, stride, e0, l0, nslots,
                                                                     static_cast<InvAcc*>(acc));
}

template <typename T>
void launch_max_id(const Particles<T>& P, unsigned long long* max_id, cudaStream_t stream) {
  if (P.n <= 0) return;
  k_max_id<T><<<(unsigned)((P.n + 255) / 256), 256, 0, stream>>>(P, max_id);
}

size_t invariant_acc_bytes() { return sizeof(InvAcc); }

template void launch_invariants<float>(const Grid&, const Particles<float>&, int, int, double*, double*, long long,
                                       void*, cudaStream_t);
template void launch_invariants<double>(const Grid&, const Particles<double>&, int, int, double*, double*,
                                        long long, void*, cudaStream_t);
template void launch_max_id<float>(const Particles<float>&, unsigned long long*, cudaStream_t);
template void launch_max_id<double>(const Particles<double>&, unsigned long long*, cudaStream_t);

template <typename T>
void launch_charge_density(const Particles<T>& P, double q, const Grid& g, bool with_gamma, double* rho,
                           cudaStream_t stream) {
  if (P.n <= 0) return;
  const unsigned nb = (unsigned)((P.n + 255) / 256);
  if constexpr (sizeof(T) == sizeof(float)) {
    if (with_gamma)
      k_charge_density_runs<true><<<nb, 256, 0, stream>>>(P, q, g.nx, g.ny, g.nz, 1.0 / g.c, rho);
    else
      k_charge_density_runs<false><<<nb, 256, 0, stream>>>(P, q, g.nx, g.ny, g.nz, 1.0 / g.c, rho);
  } else {
    k_charge_density<<<nb, 256, 0, stream>>>(P, q, g.nx, g.ny, g.nz, 1.0 / g.c, with_gamma, rho);
  }
}

template <typename T>
void launch_gauss(const Fields<T>& F, const double* rho, const Grid& g, int lo, double* res,
                  unsigned long long* maxabs, cudaStream_t stream) {
  k_gauss<T><<<(unsigned)((g.ncell + 255) / 256), 256, 0, stream>>>(F.d[0], F.d[1], F.d[2], rho, g.nx, g.ny, g.nz,
                                                                     lo, res, maxabs);
}

template void launch_charge_density<float>(const Particles<float>&, double, const Grid&, bool, double*,
                                           cudaStream_t);
template void launch_charge_density<double>(const Particles<double>&, double, const Grid&, bool, double*,
                                            cudaStream_t);
template void launch_gauss<float>(const Fields<float>&, const double*, const Grid&, int, double*,
                                  unsigned long long*, cudaStream_t);
template void launch_gauss<double>(const Fields<double>&, const double*, const Grid&, int, double*,
                                   unsigned long long*, cudaStream_t);

}  // namespace grpic
