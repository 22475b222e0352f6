// Directional second derivatives for force matching (the double backward of
// a loss on forces): along a direction v of the positions,
//   dtheta_tan = d/dt dE/dtheta (x + t v)   (mixed second derivative . v)
//   force_tan  = d/dt F (x + t v) = -H v     (Hessian-vector product)
// The energy/force code is run once with dual numbers (value, tangent): the
// pair vectors carry the tangent v_j - v_i, and every generated function
// (moments, contraction and its reverse pass, pair adjoint) propagates it.
// The tangent of dE/dxi_alpha is sum_i dB_alpha(i)/dt; the tangent of
// dE/dc[mu][k][zi][zj] is sum over pairs of d(Q_k S_mu)/dt; species energies
// have zero tangent.
#pragma once
#include <type_traits>

#include "efv_split.cuh"

namespace mtp {

template <class S>
__device__ __forceinline__ Dual<S> rsqrt_r(Dual<S> a) {
  const S r = rsqrt_r(a.v);
  return {r, S(-0.5) * r * r * r * a.t};
}

struct TangentArgs {
  EfvArgs base;
  const double* v;          // [N][3] direction
  double* dtheta_tan;       // [n_params]
  double* force_tan;        // [N][3] or null
};

// Dual pair vector: value from the precision's own geometry, tangent v_j - v_i.
template <class S>
struct TangentGeom {
  PairGeom<S> g;
  S vx, vy, vz;
  __device__ __forceinline__ void load_centre(const TangentArgs& t, int64_t i, const S* cell) {
    g.load_centre(t.base, i, cell);
    vx = S(t.v[3 * i]); vy = S(t.v[3 * i + 1]); vz = S(t.v[3 * i + 2]);
  }
  __device__ __forceinline__ void vec(const TangentArgs& t, int32_t j, const typename PairGeom<S>::Load& l,
                                      int32_t img, Dual<S>& dx, Dual<S>& dy, Dual<S>& dz) const {
    S x, y, z;
    g.vec(t.base, l, img, x, y, z);
    dx = Dual<S>(x, S(__ldg(t.v + 3 * (int64_t)j)) - vx);
    dy = Dual<S>(y, S(__ldg(t.v + 3 * (int64_t)j + 1)) - vy);
    dz = Dual<S>(z, S(__ldg(t.v + 3 * (int64_t)j + 2)) - vz);
  }
};

// Blocks per SM stated to ptxas (0: none).  The FP64 form of level 16, left to
// itself, it compiles for 32 registers (53 KB of stack, 245 KB of spills a thread);
// with two blocks stated it takes 255 (18 KB, 61 KB): 10,404 atoms 6.1 -> 3.1 ms.
// The other forms need no such hint, and level 8 in FP32 would lose resident blocks.
template <class LV, class S> constexpr int tangent_min_blocks() {
  return LV::LEVEL >= 16 && sizeof(S) == 8 ? 2 : 0;
}

template <class LV, class S>
__global__ void __launch_bounds__(kEfvThreads, (tangent_min_blocks<LV, S>())) tangent_kernel(const TangentArgs t) {
  using R = Dual<S>;
  constexpr int NMU = LV::NMU;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const EfvArgs& a = t.base;
  EfvShared<S, NMU, true> sm;     // coefficients and (tangent) accumulators in S
  sm.template setup<false>(a, smem_raw);
  sm.zero_gradients();
  __syncthreads();
  const int64_t i0 = a.atom_begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool active = i0 < a.atom_end;
  const int64_t i = active ? i0 : a.atom_begin;   // a lane without an atom runs no pairs
  S Bt[LV::NBASIS];
#pragma unroll
  for (int k = 0; k < LV::NBASIS; ++k) Bt[k] = S(0);
  {
    TangentGeom<S> geom;
    geom.load_centre(t, i, cell_of<S>(a));
    const int zi = species_at(a.z, i, a.n_species);
    const int64_t beg = __ldg(a.offsets + i), end = active ? __ldg(a.offsets + i + 1) : beg;
    R M[LV::NCOMP];
#pragma unroll
    for (int c = 0; c < LV::NCOMP; ++c) M[c] = R(0);
    const R rcut = R(sm.rcut), mid = R(sm.mid), scale = R(sm.scale);
    for (int64_t k = beg; k < end; ++k) {
      const int32_t j = __ldg(a.nbr_j + k);
      const int32_t img = __ldg(a.nbr_img + k);
      const auto l = geom.g.fetch(a, j);
      R dx, dy, dz;
      geom.vec(t, j, l, img, dx, dy, dz);
      const R r2 = fmadd(dz, dz, fmadd(dy, dy, dx * dx));
      const R rinv = rsqrt_r(r2);
      const R r = r2 * rinv;
      R f[NMU];
      radial<R, NMU, false, false>(sm.c + (zi * sm.S + l.species) * sm.cstride, sm.nq, r, mid, scale, rcut, f,
                                   (R*)nullptr, (R*)nullptr);
      LV::template moments<R>(M, f, dx * rinv, dy * rinv, dz * rinv);
    }
    R D[LV::NCOMP], B[LV::NBASIS];
    (void)LV::template contract<R, true>(M, sm.xi, D, B);
#pragma unroll
    for (int k = 0; k < LV::NBASIS; ++k) Bt[k] = B[k].t;
    S fx = S(0), fy = S(0), fz = S(0);
    const bool own_acc = sm.S <= kAccSpecies;
    S acc[kAccSpecies * NMU * kMaxQ];
    if (own_acc) {
      for (int u = 0; u < sm.S * NMU * sm.nq; ++u) acc[u] = S(0);
    }
    for (int64_t k = beg; k < end; ++k) {
      const int32_t j = __ldg(a.nbr_j + k);
      const int32_t img = __ldg(a.nbr_img + k);
      const auto l = geom.g.fetch(a, j);
      R dx, dy, dz;
      geom.vec(t, j, l, img, dx, dy, dz);
      const R r2 = fmadd(dz, dz, fmadd(dy, dy, dx * dx));
      const R rinv = rsqrt_r(r2);
      const R r = r2 * rinv;
      R f[NMU], df[NMU], q[kMaxQ];
      radial<R, NMU, true, true>(sm.c + (zi * sm.S + l.species) * sm.cstride, sm.nq, r, mid, scale, rcut, f, df, q);
      R gx, gy, gz, Smu[NMU];
      LV::template pair_adjoint<R>(D, f, df, dx * rinv, dy * rinv, dz * rinv, rinv, gx, gy, gz, Smu);
      fx += gx.t; fy += gy.t; fz += gz.t;
      if (t.force_tan) {
        atomicAdd(t.force_tan + 3 * (int64_t)j, -(double)gx.t);
        atomicAdd(t.force_tan + 3 * (int64_t)j + 1, -(double)gy.t);
        atomicAdd(t.force_tan + 3 * (int64_t)j + 2, -(double)gz.t);
      }
      if (own_acc) {
        S* dst = acc + l.species * NMU * sm.nq;
#pragma unroll
        for (int mu = 0; mu < NMU; ++mu) {
#pragma unroll
          for (int kk = 0; kk < kMaxQ; ++kk)
            if (kk < sm.nq) dst[mu * sm.nq + kk] += (q[kk] * Smu[mu]).t;
        }
      } else {
        S* dst = sm.dc + (zi * sm.S + l.species) * NMU * sm.nq;
#pragma unroll
        for (int mu = 0; mu < NMU; ++mu) {
#pragma unroll
          for (int kk = 0; kk < kMaxQ; ++kk)
            if (kk < sm.nq) atomicAdd(dst + mu * sm.nq + kk, (q[kk] * Smu[mu]).t);
        }
      }
    }
    if (own_acc) add_warp_gradients(sm, 0, NMU * sm.nq, zi, active, [&](int u) { return acc[u]; });
    if (t.force_tan && active) {
      atomicAdd(t.force_tan + 3 * i, (double)fx);
      atomicAdd(t.force_tan + 3 * i + 1, (double)fy);
      atomicAdd(t.force_tan + 3 * i + 2, (double)fz);
    }
  }
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < LV::NBASIS; ++k) {
    const double v = warp_sum((double)Bt[k]);
    if (lane == 0) atomicAdd(sm.dxi + k, S(v));
  }
  __syncthreads();
  const int S_ = sm.S, SS = sm.SS, nq = sm.nq;
  for (int k = threadIdx.x; k < SS * NMU * nq; k += blockDim.x) {
    const int p = k / (NMU * nq);
    const int mk = k % (NMU * nq);
    atomicAdd(t.dtheta_tan + S_ + (int64_t)mk * SS + p, (double)sm.dc[k]);
  }
  for (int k = threadIdx.x; k < sm.m; k += blockDim.x)
    atomicAdd(t.dtheta_tan + S_ + (int64_t)NMU * nq * SS + k, (double)sm.dxi[k]);
}

// Levels with component groups run the tangent as three kernels, as the
// energy does: dual moments per component group and share of the neighbours,
// the tile program on dual numbers, dual adjoint sweeps.
template <class LV, class S, int G>
__device__ __forceinline__ void tangent_moments(const TangentArgs& t, const EfvShared<S, LV::NMU, true>& sm,
                                                const SplitShare& s, int64_t n) {
  using R = Dual<S>;
  constexpr int NMU = LV::NMU;
  const EfvArgs& a = t.base;
  TangentGeom<S> geom;
  geom.load_centre(t, s.i, cell_of<S>(a));
  const int zi = species_at(a.z, s.i, a.n_species);
  const R rcut = R(sm.rcut), mid = R(sm.mid), scale = R(sm.scale);
  R Mg[LV::NCOMP];
#pragma unroll
  for (int c = 0; c < LV::NCOMP; ++c) Mg[c] = R(0);
  for (int64_t k = s.beg; k < s.end; ++k) {
    const int32_t j = __ldg(a.nbr_j + k);
    const int32_t img = __ldg(a.nbr_img + k);
    const auto l = geom.g.fetch(a, j);
    R dx, dy, dz;
    geom.vec(t, j, l, img, dx, dy, dz);
    const R r2 = fmadd(dz, dz, fmadd(dy, dy, dx * dx));
    const R rinv = rsqrt_r(r2);
    const R r = r2 * rinv;
    R f[NMU];
    radial<R, NMU, false, false>(sm.c + (zi * sm.S + l.species) * sm.cstride, sm.nq, r, mid, scale, rcut, f,
                                 (R*)nullptr, (R*)nullptr);
    LV::template moments_group<G, R>(Mg, f, dx * rinv, dy * rinv, dz * rinv);
  }
  if (s.t < tile_padded(n)) {
    R* buf = static_cast<R*>(a.mbuf) + (int64_t)(blockIdx.y >> 1) * (tile_padded(n) * LV::NCOMP);
    LV::template store_group<G, R>(Mg, buf + tile_offset<R>(s.t, LV::NCOMP), tile_atoms<R>());
  }
}

template <class LV, class S>
__global__ void __launch_bounds__(kEfvThreads) tangent_moments_kernel(const TangentArgs t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EfvShared<S, LV::NMU, true> sm;
  sm.template setup<false>(t.base, smem_raw);
  __syncthreads();
  const int64_t n = t.base.atom_end - t.base.atom_begin;
  SplitShare s;
  if (!s.setup(t.base, n)) return;
  if ((blockIdx.y & 1) == 0) tangent_moments<LV, S, 0>(t, sm, s, n);
  else tangent_moments<LV, S, 1>(t, sm, s, n);
}

template <class LV, class S, int G>
__device__ __forceinline__ void tangent_adjoint(const TangentArgs& t, const EfvShared<S, LV::NMU, true>& sm,
                                                const SplitShare& s, int64_t n) {
  using R = Dual<S>;
  constexpr int NMU = LV::NMU;
  constexpr int mu_lo = LV::GROUP_MU_LO[G], mu_hi = LV::GROUP_MU_HI[G];
  const EfvArgs& a = t.base;
  TangentGeom<S> geom;
  geom.load_centre(t, s.i, cell_of<S>(a));
  const int zi = species_at(a.z, s.i, a.n_species);
  const R rcut = R(sm.rcut), mid = R(sm.mid), scale = R(sm.scale);
  S fx = S(0), fy = S(0), fz = S(0);
  const bool own_acc = sm.S <= kAccSpecies;
  S acc[kAccSpecies * NMU * kMaxQ];
  if (own_acc) {
    for (int v = 0; v < sm.S * NMU * sm.nq; ++v) acc[v] = S(0);
  }
  R Dg[LV::NCOMP];
  const R* buf = static_cast<const R*>(a.mbuf) + (int64_t)a.n_parts * (tile_padded(n) * LV::NCOMP);
  LV::template load_group<G, R>(buf + tile_offset<R>(s.active ? s.t : 0, LV::NCOMP), tile_atoms<R>(), Dg);
  for (int64_t k = s.beg; k < s.end; ++k) {
    const int32_t j = __ldg(a.nbr_j + k);
    const int32_t img = __ldg(a.nbr_img + k);
    const auto l = geom.g.fetch(a, j);
    R dx, dy, dz;
    geom.vec(t, j, l, img, dx, dy, dz);
    const R r2 = fmadd(dz, dz, fmadd(dy, dy, dx * dx));
    const R rinv = rsqrt_r(r2);
    const R r = r2 * rinv;
    R f[NMU], df[NMU], q[kMaxQ];
    radial<R, NMU, true, true>(sm.c + (zi * sm.S + l.species) * sm.cstride, sm.nq, r, mid, scale, rcut, f, df, q);
    R gx, gy, gz, Smu[NMU];
    LV::template pair_adjoint_group<G, R>(Dg, f, df, dx * rinv, dy * rinv, dz * rinv, rinv, gx, gy, gz, Smu);
    fx += gx.t; fy += gy.t; fz += gz.t;
    if (t.force_tan) {
      atomicAdd(t.force_tan + 3 * (int64_t)j, -(double)gx.t);
      atomicAdd(t.force_tan + 3 * (int64_t)j + 1, -(double)gy.t);
      atomicAdd(t.force_tan + 3 * (int64_t)j + 2, -(double)gz.t);
    }
    if (own_acc) {
      S* dst = acc + l.species * NMU * sm.nq;
#pragma unroll
      for (int mu = mu_lo; mu < mu_hi; ++mu) {
#pragma unroll
        for (int kk = 0; kk < kMaxQ; ++kk)
          if (kk < sm.nq) dst[mu * sm.nq + kk] += (q[kk] * Smu[mu]).t;
      }
    } else {
      S* dst = sm.dc + (zi * sm.S + l.species) * NMU * sm.nq;
#pragma unroll
      for (int mu = mu_lo; mu < mu_hi; ++mu) {
#pragma unroll
        for (int kk = 0; kk < kMaxQ; ++kk)
          if (kk < sm.nq) atomicAdd(dst + mu * sm.nq + kk, (q[kk] * Smu[mu]).t);
      }
    }
  }
  if (own_acc)
    add_warp_gradients(sm, mu_lo * sm.nq, mu_hi * sm.nq, zi, s.active, [&](int u) { return acc[u]; });
  if (t.force_tan && s.active) {
    atomicAdd(t.force_tan + 3 * s.i, (double)fx);
    atomicAdd(t.force_tan + 3 * s.i + 1, (double)fy);
    atomicAdd(t.force_tan + 3 * s.i + 2, (double)fz);
  }
}

template <class LV, class S>
__global__ void __launch_bounds__(kEfvThreads) tangent_adjoint_kernel(const TangentArgs t) {
  constexpr int NMU = LV::NMU;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const EfvArgs& a = t.base;
  EfvShared<S, NMU, true> sm;
  sm.template setup<false>(a, smem_raw);
  sm.zero_gradients();
  __syncthreads();
  const int64_t n = a.atom_end - a.atom_begin;
  SplitShare s;
  if (s.setup(a, n)) {
    if ((blockIdx.y & 1) == 0) tangent_adjoint<LV, S, 0>(t, sm, s, n);
    else tangent_adjoint<LV, S, 1>(t, sm, s, n);
  }
  __syncthreads();
  const int S_ = sm.S, SS = sm.SS, nq = sm.nq;
  for (int k = threadIdx.x; k < SS * NMU * nq; k += blockDim.x) {
    const int p = k / (NMU * nq);
    const int mk = k % (NMU * nq);
    atomicAdd(t.dtheta_tan + S_ + (int64_t)mk * SS + p, (double)sm.dc[k]);
  }
}

// The tangent's accumulators are thread-private in either precision: staging only.
template <class S, int NMU>
size_t tangent_smem(const EfvArgs& a, int threads) {
  const size_t base = (efv_smem_bytes<S, NMU, true>(a.n_species * a.n_species, a.n_q, a.m) + 15) & ~size_t(15);
  const size_t stage = efv_stage_bytes<S, true>(a.n_species, threads);
  return base + stage <= kMaxBlockSmem ? base + stage : base;
}

template <class LV, class S>
int tangent_split_launch(const TangentArgs& t, cudaStream_t stream) {
  const EfvArgs& a = t.base;
  const int64_t n = a.atom_end - a.atom_begin;
  const int threads = sizeof(S) == 8 ? fp64_threads(n, 2 * a.n_parts) : kEfvThreads;
  const dim3 grid((unsigned)((n + threads - 1) / threads), 2 * a.n_parts);
  const size_t bytes = tangent_smem<S, LV::NMU>(a, threads);
  int rc;
  if ((rc = set_smem(tangent_moments_kernel<LV, S>, bytes)) != MTP_OK) return rc;
  if ((rc = set_smem(tangent_adjoint_kernel<LV, S>, bytes)) != MTP_OK) return rc;
  tangent_moments_kernel<LV, S><<<grid, threads, bytes, stream>>>(t);
  if ((rc = tile_contract_launch<LV, Dual<S>, true>(a, t.dtheta_tan, stream)) != MTP_OK) return rc;
  tangent_adjoint_kernel<LV, S><<<grid, threads, bytes, stream>>>(t);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("tangent split kernels (level %d): %s", LV::LEVEL, cudaGetErrorString(e));
    return MTP_ERR_CUDA;
  }
  return MTP_OK;
}

// One kernel (levels with one component group).  Two rules, with whole calls in us:
//   staging area: everywhere (level 8, 10,404 atoms mixed 141 -> 93) but at level 16
//   in FP32 with more than one block per SM, where the spills want the cache that
//   the area takes (two species: 21,296 atoms 600 -> 487, 182,250 atoms 4,051 ->
//   3,166; three: 704 -> 632, 4,237 -> 4,160).  With one species all lanes' sums meet
//   on the same addresses, and the line is at four blocks (21,296 atoms 433 against
//   483, 182,250 atoms 3,245 -> 2,587); with four the area stays (69,696 atoms 1,566
//   against 1,674);
//   the blocks that a last, partial wave leaves, from half a block of 128 to one for
//   every SM, go in a launch of their own: in one launch the SMs that finish first
//   take several of them each (54,000 atoms FP64: level 8 2,385 -> 1,946, level 12
//   4,795 -> 4,052, level 16 10,310 -> 8,675).  With 4 blocks left over, or 103 of 64
//   threads, the launch would cost 3 to 5%.
template <class LV, class S>
int tangent_fused_launch(const TangentArgs& t, cudaStream_t stream) {
  const EfvArgs& a = t.base;
  const int64_t n = a.atom_end - a.atom_begin, sms = device_sms();
  const int threads = sizeof(S) == 8 ? fp64_threads(n, 1) : kEfvThreads;
  const int64_t blocks = (n + threads - 1) / threads;
  auto kern = tangent_kernel<LV, S>;
  const bool staged = LV::LEVEL < 16 || sizeof(S) == 8 || a.n_species >= kAccSpecies ||
                      blocks <= (a.n_species == 1 ? 4 : 1) * sms;
  const size_t bytes =
      staged ? tangent_smem<S, LV::NMU>(a, threads) : efv_smem_bytes<S, LV::NMU, true>(a.n_species * a.n_species, a.n_q, a.m);
  const int rc = set_smem(kern, bytes);
  if (rc != MTP_OK) return rc;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, bytes) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  int64_t rest = blocks % (per_sm * sms);
  if (rest == blocks || rest > sms || 2 * rest * threads < sms * kEfvThreads) rest = 0;
  TangentArgs part = t;
  if (rest) part.base.atom_end = a.atom_begin + (blocks - rest) * threads;
  kern<<<(unsigned)(blocks - rest), threads, bytes, stream>>>(part);
  if (rest) {
    part.base.atom_begin = part.base.atom_end;
    part.base.atom_end = a.atom_end;
    kern<<<(unsigned)rest, threads, bytes, stream>>>(part);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("tangent kernel launch (level %d): %s", LV::LEVEL, cudaGetErrorString(e));
    return MTP_ERR_CUDA;
  }
  return MTP_OK;
}

template <class LV>
int tangent_launch(const TangentArgs& t, int precision, cudaStream_t stream) {
  const EfvArgs& a = t.base;
  const int64_t n = a.atom_end - a.atom_begin;
  if (n <= 0) return MTP_OK;
  if constexpr (LV::NGROUPS > 1) {   // the caller always provides the scratch
    return precision == MTP_MIXED ? tangent_split_launch<LV, float>(t, stream)
                                  : tangent_split_launch<LV, double>(t, stream);
  } else {
    return precision == MTP_MIXED ? tangent_fused_launch<LV, float>(t, stream)
                                  : tangent_fused_launch<LV, double>(t, stream);
  }
}

}  // namespace mtp
