// Kernels of the fused gather + GR-RK4 push + curved-metric deposit (the per-particle work is
// in push_core.cuh): the single-kernel push (FP64, and FP32-mixed without the near/far split),
// the near-hole pass of the split FP32-mixed push, the batched push, and particle load/unload.
#include <algorithm>
#include <cmath>

#include "push_core.cuh"

namespace grpic {

namespace {

template <typename T, int Q, bool MIXED, int THREADS>
__global__ void __launch_bounds__(THREADS, 4 * (128 / THREADS))
    k_push_deposit(const Grid g, const Fields<T> F, const Particles<T> P, const Consts<T> C, DevStatus* st) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  unsigned flags = 0, n64 = 0;
  bool active = i < P.n && i < (long long)(*P.n_dev);
  if (active) active = P.key[i] != kDead;
  if (active) push_particle<T, Q, MIXED>(g, F, P, C, i, st, flags, n64, P.key + i);
  warp_status(st, flags, n64, active);
}

// Block-cooperative copy of a trivially copyable struct (a multiple of 4 bytes) into shared memory.
__device__ __forceinline__ void copy_words(void* dst, const void* src, size_t bytes) {
  unsigned* d = static_cast<unsigned*>(dst);
  const unsigned* s = static_cast<const unsigned*>(src);
  for (unsigned w = threadIdx.x; w < bytes / 4; w += blockDim.x) d[w] = s[w];
}

// Near-hole pass of the split FP32-mixed push: the particles listed by the classification
// (whose stages and quadrature nodes may fall inside r < r_fp64).  Persistent blocks take
// 128-entry chunks of the list from a cursor (count[1]) until it is exhausted: the FP64 work
// per particle varies a lot, so a dynamic queue keeps the SMs evenly loaded.  Consecutive list
// entries come from consecutive cell-sorted particles, so a warp stays local.  The far kernel
// runs at the same time and tells near from far particles by the kNear mark in P.key, so the
// new sort keys go to keys[j] (by list slot) and are copied back after both end.
template <int Q>
__global__ void __launch_bounds__(128, 4) k_push_near(const Grid g, const Fields<float> F, const Particles<float> P,
                                                        const Consts<float> C, DevStatus* st,
                                                        const uint32_t* __restrict__ list, uint32_t* __restrict__ keys,
                                                        int* count) {
  __shared__ int s_base;
  const int n = count[0];
  for (;;) {
    if (threadIdx.x == 0) s_base = atomicAdd(count + 1, (int)blockDim.x);
    __syncthreads();
    const int base = s_base;
    __syncthreads();
    if (base >= n) break;
    const int j = base + threadIdx.x;
    const bool active = j < n;
    unsigned flags = 0, n64 = 0;
    if (active) push_particle<float, Q, true>(g, F, P, C, (long long)list[j], st, flags, n64, keys + j);
    warp_status(st, flags, n64, active);
  }
}

// After the join: the near particles' new sort keys back into P.key.
__global__ void k_near_keys(uint32_t* __restrict__ key, const uint32_t* __restrict__ list,
                            const uint32_t* __restrict__ keys, const int* count) {
  const int n = *count;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) key[list[j]] = keys[j];
}

// Batched FP64 push: one CTA per (instance * 4 + species, block) work item; each block belongs to one
// instance and species, so the warp-level status stays per instance.  The block stages its
// instance descriptor (with the host-built launch constants) in shared memory.  The block -> item map is the same
// coprime permutation as k_push_select's (perm; 1 = in order).
template <int Q>
__global__ void __launch_bounds__(128, 4) k_push_deposit_batch(const InstDesc<double>* __restrict__ desc,
                                                                 const BlockEntry* __restrict__ blk, int nblk,
                                                                 unsigned perm) {
  __shared__ Grid sg;
  __shared__ Fields<double> sF;
  __shared__ SpeciesDesc<double> sS;
  __shared__ DevStatus* sst;
  __shared__ int s_cur;
  const int bi = (int)spread_chunk(blockIdx.x, (unsigned)nblk, perm, kBatchSpreadLog2);
  const BlockEntry e = blk[bi];
  // stage the descriptor parts this block needs with one coalesced copy by all threads (the
  // launch constants were built on the host)
  const InstDesc<double>& D = desc[e.inst >> 2];
  copy_words(&sg, &D.g, sizeof(Grid));
  copy_words(&sS, &D.sp[e.inst & 3], sizeof(SpeciesDesc<double>));
  if (threadIdx.x == 0) {
    sst = D.st;
    s_cur = *D.sp[e.inst & 3].cur;
    // the push of a batched step runs after the first B half-step: b^n is in b buffer 1
    const int dc = *D.dcur;
    for (int q = 0; q < 3; ++q) {
      sF.d[q] = D.FS.d[dc][q];
      sF.b[q] = D.FS.b[1][q];
      sF.J[q] = D.FS.J[q];
    }
  }
  __syncthreads();
  const Particles<double>& sP = sS.buf[s_cur];
  const long long i = (long long)e.block * blockDim.x + threadIdx.x;
  unsigned flags = 0, n64 = 0;
  bool active = i < sP.n && i < (long long)(*sP.n_dev);
  if (active) active = sP.key[i] != kDead;
  if (active) push_particle<double, Q, false>(sg, sF, sP, sS.C, i, sst, flags, n64, sP.key + i);
  warp_status(sst, flags, n64, active);
}

// ---- load / unload ---------------------------------------------------------------------
__device__ __forceinline__ float from_f64(double v, float) { return narrow(v); }
__device__ __forceinline__ double from_f64(double v, double) { return v; }

// v > 0, infinity included (from the bits; NaN fails)
__device__ __forceinline__ bool positive(double v) {
  return (unsigned long long)__double_as_longlong(v) - 1 < 0x7ff0000000000000ull;
}

// Is the point inside r <= r_+?  Screened in FP32 (far from the hole nothing else is evaluated), decided by the IEEE
// evaluation.
__device__ __forceinline__ bool inside_horizon(const Grid& g, double X, double Y, double Z) {
  const float xf = narrow(X), yf = narrow(Y), zf = narrow(Z), rp = (float)g.r_plus + fabsf((float)g.a);
  if (xf * xf + yf * yf + zf * zf > 1.01f * rp * rp + 1e-3f) return false;  // r >= R - |a| > r_+
  const Kerr<double> K = kerr_eval<double>(X, Y, Z, g.m, g.a);
  return K.flat || K.r <= g.r_plus;
}

// Completion of u^a from its spatial part.  Covariant u_i (umode 1): g^mn u_m u_n = -c^2 with g^mn = eta^mn - f k^m
// k^n, k^m = (k_i, -1), is (1 + f) u_4^2 - 2 f (k.u) u_4 - C = 0, C = |u|^2 - f (k.u)^2 + c^2; for its roots
// u_4 = [f (k.u) -+ S] / (1 + f), S^2 = f^2 (k.u)^2 + (1 + f) C, u^4 = -u_4 + f (k.u - u_4) is +-S, so the
// future-directed one has u^4 = S.  Contravariant u^i (umode 2): (1 - f) u4^2 - 2 f (k.u) u4 - C = 0 with
// C = |u|^2 + f (k.u)^2 + c^2, u^4 = [f (k.u) + S] / (1 - f), S^2 = f^2 (k.u)^2 + (1 - f) C.
// The load is bound by the FP64 pipe: one FP64 evaluation of the metric by FastOps64 and 20 operations a particle
// (two IEEE evaluations and the two roots of each quadratic before: 5.1 ms for 15.6 M particles of an FP32-mixed
// context; 2.2 ms with the constants formed and the signs compared in FP64 as well; now 2.0 ms).
// FP64 products of the grid's constants, formed once on the host.
struct LoadConsts {
  double two_m, a2, a2_4, c2;
};
template <typename T>
__global__ void k_load(const Grid g, const Particles<T> P, long long n, const double* __restrict__ x4,
                       const double* __restrict__ u4, const uint32_t* __restrict__ ids, int umode, double ct_now,
                       const LoadConsts C, DevStatus* st) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x[3] = {x4[i], x4[n + i], x4[2 * n + i]};
  unsigned bad = 0;
  const int nn[3] = {g.nx, g.ny, g.nz};
  int cell[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    double fl;
    floor_split(x[q], cell[q], fl);
    // x in [1, n - 2] (NaN fails both)
    const bool whole = __double_as_longlong(x[q]) == __double_as_longlong(fl);
    if (!(cell[q] >= 1 && (cell[q] < nn[q] - 2 || (cell[q] == nn[q] - 2 && whole)))) bad |= ST_LOAD_INVALID;
    cell[q] = min(max(cell[q], 0), nn[q] - 2);
  }
  double u[4] = {u4[i], u4[n + i], u4[2 * n + i], umode == 0 ? u4[3 * n + i] : 0.0};
  // the removal rule (r <= r_+) applies from the start: such particles are dropped at load
  const double X = x[0] - g.xc, Y = x[1] - g.yc, Z = x[2] - g.zc;
  bool inside = false;
  if (!bad && g.m > 0.0) {
    inside = inside_horizon(g, X, Y, Z);
    if (inside) atomicAdd(&st->removed_horizon, 1ull);
  }
  if (!bad && !inside && umode != 0) {
    const Kerr<double> K = kerr_eval_fast(X, Y, Z, C.two_m, g.a, C.a2, C.a2_4);
    const double f = K.f, kk[3] = {K.k0, K.k1, K.k2};
    const double ku = fma(kk[0], u[0], fma(kk[1], u[1], kk[2] * u[2]));
    const double fk = f * ku;
    const double uu = fma(u[0], u[0], fma(u[1], u[1], fma(u[2], u[2], C.c2)));
    if (umode == 1) {
      const double A = 1.0 + f;
      const double S2 = fma(fk, fk, A * fma(-fk, ku, uu));
      // (S^2 beyond FP64: loaded with an infinite u^4, which the first step reports, where the metric is not flat)
      if (!positive(S2) || (!finite_t(S2) && !positive(f))) {
        bad |= ST_LOAD_INVALID;
      } else {
        // raise: u^i = u_i - f k_i (k.u - u_4), k.u - u_4 = (k.u + S) / (1 + f)
        const double S = CheckedOps64::root(S2);
        const double fkul = f * ((ku + S) * FastOps64::rcp(A));
#pragma unroll
        for (int q = 0; q < 3; ++q) u[q] = fma(-kk[q], fkul, u[q]);
        u[3] = S;
      }
    } else {
      const double A = 1.0 - f;
      const double S2 = fma(fk, fk, A * fma(fk, ku, uu));
      if (!(A > 0.0)) {
        bad |= ST_LOAD_ERGO;
      } else if (!(S2 >= 0.0)) {
        bad |= ST_LOAD_INVALID;
      } else {
        u[3] = CheckedOps64::div(fk + CheckedOps64::root(S2), A);
        if (!(u[3] > 0.0)) bad |= ST_LOAD_INVALID;
      }
    }
  }
  if (bad) atomicOr(&st->flags, bad);
#pragma unroll
  for (int q = 0; q < 3; ++q) P.x[q][i] = from_f64(x[q], T());
  P.x[3][i] = from_f64(x4[3 * n + i] - ct_now, T());
#pragma unroll
  for (int q = 0; q < 4; ++q) P.u[q][i] = from_f64(u[q], T());
  P.id[i] = ids[i];
  P.key[i] = inside ? kDead : (uint32_t)(((long long)cell[2] * g.ny + cell[1]) * g.nx + cell[0]);
}

template <typename T>
__global__ void k_unload(const Particles<T> P, long long n, double* __restrict__ x4, double* __restrict__ u4,
                         uint32_t* __restrict__ ids, double ct_now) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  // (widened with integer operations: the conversions would run on the FP64 pipe)
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (x4) x4[q * n + i] = to_f64(P.x[q][i]);
  }
  if (x4) x4[3 * n + i] = to_f64(P.x[3][i]) + ct_now;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (u4) u4[q * n + i] = to_f64(P.u[q][i]);
  if (ids) ids[i] = P.id[i];
}

inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

template <typename T, bool MIXED, int THREADS>
void launch_push_q(const Grid& g, const Fields<T>& F, const Particles<T>& P, const Species& sp, DevStatus* st,
                   cudaStream_t stream) {
  const unsigned nb = blocks_for(P.n, THREADS);
  const Consts<T> C = make_consts<T>(g, sp);
  if (g.quad_order == 1)
    k_push_deposit<T, 1, MIXED, THREADS><<<nb, THREADS, 0, stream>>>(g, F, P, C, st);
  else if (g.quad_order == 3)
    k_push_deposit<T, 3, MIXED, THREADS><<<nb, THREADS, 0, stream>>>(g, F, P, C, st);
  else
    k_push_deposit<T, 2, MIXED, THREADS><<<nb, THREADS, 0, stream>>>(g, F, P, C, st);
}

// FP64 runs pure double; FP32 runs the mixed policy.
template <>
void launch_push_deposit<double>(const Grid& g, const Fields<double>& F, const Particles<double>& P,
                                 const Species& sp, DevStatus* st, bool, double, cudaStream_t stream) {
  if (P.n <= 0) return;
  if (small_push(P.n))
    launch_push_q<double, false, 32>(g, F, P, sp, st, stream);
  else
    launch_push_q<double, false, 128>(g, F, P, sp, st, stream);
}
template <>
void launch_push_deposit<float>(const Grid& g, const Fields<float>& F, const Particles<float>& P,
                                const Species& sp, DevStatus* st, bool, double, cudaStream_t stream) {
  if (P.n > 0) launch_push_q<float, true, 128>(g, F, P, sp, st, stream);
}

void launch_push_near(const Grid& g, const Fields<float>& F, const Particles<float>& P, const Species& sp,
                      DevStatus* st, const uint32_t* list, uint32_t* keys, int* count, int nblocks,
                      cudaStream_t stream) {
  if (P.n <= 0 || nblocks <= 0) return;
  const Consts<float> C = make_consts<float>(g, sp);
  if (g.quad_order == 1)
    k_push_near<1><<<nblocks, 128, 0, stream>>>(g, F, P, C, st, list, keys, count);
  else if (g.quad_order == 3)
    k_push_near<3><<<nblocks, 128, 0, stream>>>(g, F, P, C, st, list, keys, count);
  else
    k_push_near<2><<<nblocks, 128, 0, stream>>>(g, F, P, C, st, list, keys, count);
}

void launch_near_keys(const Particles<float>& P, const uint32_t* list, const uint32_t* keys, const int* count,
                      int nblocks, cudaStream_t stream) {
  if (P.n <= 0 || nblocks <= 0) return;
  k_near_keys<<<nblocks, 256, 0, stream>>>(P.key, list, keys, count);
}

void launch_batch_push(const BatchTables<double>& bt, int quad_order, cudaStream_t stream) {
  // one block per work item: each block stages its instance descriptor once, and the hardware
  // scheduler balances instances of very different cost
  const unsigned nb = (unsigned)bt.npart;
  if (bt.npart == 0) return;
  const unsigned perm = spread_multiplier(nb, kBatchSpreadLog2);
  if (quad_order == 1)
    k_push_deposit_batch<1><<<nb, 128, 0, stream>>>(bt.desc, bt.part, bt.npart, perm);
  else if (quad_order == 3)
    k_push_deposit_batch<3><<<nb, 128, 0, stream>>>(bt.desc, bt.part, bt.npart, perm);
  else
    k_push_deposit_batch<2><<<nb, 128, 0, stream>>>(bt.desc, bt.part, bt.npart, perm);
}

template <typename T>
void launch_load_particles(const Grid& g, const Particles<T>& P, long long n, const double* x4, const double* u4,
                           const uint32_t* ids, int umode, double ct_now, DevStatus* st, cudaStream_t stream) {
  if (n <= 0) return;
  k_load<T><<<blocks_for(n, 256), 256, 0, stream>>>(g, P, n, x4, u4, ids, umode, ct_now,
                                              LoadConsts{2.0 * g.m, g.a * g.a, 4.0 * (g.a * g.a), g.c * g.c}, st);
}

template <typename T>
void launch_unload_particles(const Particles<T>& P, long long n, double* x4, double* u4, uint32_t* ids,
                             double ct_now, cudaStream_t stream) {
  if (n <= 0) return;
  k_unload<T><<<blocks_for(n, 256), 256, 0, stream>>>(P, n, x4, u4, ids, ct_now);
}

template void launch_load_particles<float>(const Grid&, const Particles<float>&, long long, const double*,
                                           const double*, const uint32_t*, int, double, DevStatus*, cudaStream_t);
template void launch_load_particles<double>(const Grid&, const Particles<double>&, long long, const double*,
                                            const double*, const uint32_t*, int, double, DevStatus*,
                                            cudaStream_t);
template void launch_unload_particles<float>(const Particles<float>&, long long, double*, double*, uint32_t*,
                                             double, cudaStream_t);
template void launch_unload_particles<double>(const Particles<double>&, long long, double*, double*, uint32_t*,
                                              double, cudaStream_t);

}  // namespace grpic
