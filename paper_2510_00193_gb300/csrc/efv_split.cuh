// Levels with component groups (18 and 20: 201 and 295 moment components, too
// many for registers) and a scratch buffer a.mbuf run as three kernels: the
// neighbour sweeps need many registers per thread, the contraction the whole
// shared memory of an SM.
//
// Sweeps: one thread per atom, component group (mu = 0, mu >= 1: a group's
// moments or adjoints fit in registers) and share of the atom's neighbours
// (a.n_parts of them); blockIdx.y = 2 share + group.  Every share writes its
// own partial moments, which the contraction adds when it loads them, so the
// shares never wait for one another.  Scratch layout: tile_offset.
#pragma once
#include "efv_kernel.cuh"
#include "tile_contract.cuh"

namespace mtp {

// This thread's atom of the range and its share of the neighbours.
struct SplitShare {
  int64_t t, i, beg, end;
  bool active;
  __device__ __forceinline__ bool setup(const EfvArgs& a, int64_t n) {
    t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    active = t < n;
    i = a.atom_begin + (active ? t : 0);
    const int part = blockIdx.y >> 1;
    int64_t b, e;
    list_row(a, i, b, e);
    const int64_t len = e - b;
    beg = b + len * part / a.n_parts;
    end = active ? b + len * (part + 1) / a.n_parts : beg;
    return __any_sync(0xffffffffu, t < tile_padded(n));
  }
};

template <class LV, class R, int G>
__device__ __forceinline__ void split_moments(const EfvArgs& a, const EfvShared<R, LV::NMU, false>& sm,
                                              const SplitShare& s, int64_t n) {
  PairGeom<R> geom;
  geom.load_centre(a, s.i, cell_of<R>(a));
  const int zi = species_at(a.z, s.i, a.n_species);
  R Mg[LV::NCOMP];
#pragma unroll
  for (int c = 0; c < LV::NCOMP; ++c) Mg[c] = R(0);
  moment_sweep<LV, R, false, G, true>(a, sm, geom, a.cell, zi, s.beg, s.end, Mg);
  // the atoms that pad the last tile get zero moments
  if (s.t < tile_padded(n)) {
    R* buf = static_cast<R*>(a.mbuf) + (int64_t)(blockIdx.y >> 1) * (tile_padded(n) * LV::NCOMP);
    LV::template store_group<G, R>(Mg, buf + tile_offset<R>(s.t, LV::NCOMP), tile_atoms<R>());
  }
}

template <class LV, class R>
__global__ void __launch_bounds__(kEfvThreads) split_moments_kernel(const EfvArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EfvShared<R, LV::NMU, false> sm;
  sm.setup(a, smem_raw);
  __syncthreads();
  const int64_t n = a.atom_end - a.atom_begin;
  SplitShare s;
  if (!s.setup(a, n)) return;
  if ((blockIdx.y & 1) == 0) split_moments<LV, R, 0>(a, sm, s, n);
  else split_moments<LV, R, 1>(a, sm, s, n);
}

// The mixed path's dE/dc accumulators: [entry of one group][thread], one more
// column than threads.  One group's entries without a staging area, instead of
// all groups' with one, let two blocks share an SM at level 20 with n_q = 10
// (132 KB a block before: 108,000 atoms 1.64 ms for this kernel, 1.07 now).
template <class LV> constexpr int largest_group_mus() {
  int mus = 0;
  for (int g = 0; g < LV::NGROUPS; ++g) {
    const int n = LV::GROUP_MU_HI[g] - LV::GROUP_MU_LO[g];
    mus = n > mus ? n : mus;
  }
  return mus;
}
template <class LV>
__host__ __device__ inline size_t split_columns_bytes(int S, int nq, int threads) {
  constexpr int mus = largest_group_mus<LV>();
  return sizeof(float) * (size_t)S * mus * nq * (threads + 1);
}

template <class LV, class R, bool DTHETA, int G>
__device__ __forceinline__ void split_adjoint(const EfvArgs& a, const EfvShared<R, LV::NMU, DTHETA>& sm,
                                              const SplitShare& s, int64_t n, R* w) {
  constexpr int NMU = LV::NMU;
  PairGeom<R> geom;
  geom.load_centre(a, s.i, cell_of<R>(a));
  const int zi = species_at(a.z, s.i, a.n_species);
  R fx = R(0), fy = R(0), fz = R(0);
  constexpr int mu_lo = LV::GROUP_MU_LO[G], mu_hi = LV::GROUP_MU_HI[G];
  constexpr bool kColumns = sizeof(R) == 4;   // FP32: in shared memory, FP64: thread-private
  R acc_local[(DTHETA && !kColumns) ? kAccSpecies * NMU * kMaxQ : 1];
  GroupAccView<R> acc({acc_local, 1}, NMU * sm.nq, 0);
  if (kColumns)
    acc = GroupAccView<R>({sm.acc ? sm.acc + threadIdx.x : nullptr, (int)blockDim.x + 1}, (mu_hi - mu_lo) * sm.nq,
                          mu_lo * sm.nq);
  const bool own_acc = DTHETA && sm.S <= kAccSpecies && acc.p != nullptr;
  if (own_acc) {
    for (int u = 0; u < sm.S * acc.per; ++u) acc[u] = R(0);
  }
  R Dg[LV::NCOMP];
  const R* buf = static_cast<const R*>(a.mbuf) + (int64_t)a.n_parts * (tile_padded(n) * LV::NCOMP);
  LV::template load_group<G, R>(buf + tile_offset<R>(s.active ? s.t : 0, LV::NCOMP), tile_atoms<R>(), Dg);
  adjoint_sweep<LV, R, DTHETA, G, true>(a, sm, geom, a.cell, zi, s.beg, s.end, Dg, fx, fy, fz, w, acc, own_acc);
  if (own_acc) {
    if constexpr (kColumns) add_warp_columns(sm, sm.acc, mu_lo * sm.nq, mu_hi * sm.nq, zi, s.active);
    else add_warp_gradients(sm, mu_lo * sm.nq, mu_hi * sm.nq, zi, s.active, [&](int t) { return acc[t]; });
  }
  if (!s.active) return;
  scatter_force(a, s.i, fx, fy, fz);
  if (!isfinite((double)fx) || !isfinite((double)fy) || !isfinite((double)fz))
    flag_status(a.status, MTP_ERR_NONFINITE);
}

template <class LV, class R, bool DTHETA>
__global__ void __launch_bounds__(kEfvThreads) split_adjoint_kernel(const EfvArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EfvShared<R, LV::NMU, DTHETA> sm;
  sm.template setup<false>(a, smem_raw);
  if (DTHETA && sizeof(R) == 4 && sm.S <= kAccSpecies) {
    const size_t off = (efv_smem_bytes<R, LV::NMU, DTHETA>(sm.SS, sm.nq, sm.m) + 15) & ~size_t(15);
    if (dynamic_smem_size() >= off + split_columns_bytes<LV>(sm.S, sm.nq, blockDim.x))
      sm.acc = reinterpret_cast<R*>(smem_raw + off);
  }
  sm.zero_gradients();
  __syncthreads();
  const int64_t n = a.atom_end - a.atom_begin;
  R w[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
  SplitShare s;
  if (s.setup(a, n)) {
    if ((blockIdx.y & 1) == 0) split_adjoint<LV, R, DTHETA, 0>(a, sm, s, n, w);
    else split_adjoint<LV, R, DTHETA, 1>(a, sm, s, n, w);
  }
  efv_block_flush<LV, R, DTHETA>(sm, 0.0, w, a.e_total, a.virial, a.dtheta, kFlushEW | kFlushDc);
}

// Contraction kernel: one block per resident slot of the device, each taking
// tile after tile.
template <class LV, class R, bool WANT_B>
int tile_contract_launch(const EfvArgs& a, double* theta, cudaStream_t stream) {
  auto kern = tile_contract_kernel<LV, R, WANT_B>;
  constexpr size_t bytes = tile_smem_bytes<LV, R>();
  int rc = set_smem(kern, bytes);
  if (rc != MTP_OK) return rc;
  const int64_t n = a.atom_end - a.atom_begin;
  const int64_t tiles = (n + tile_atoms<R>() - 1) / tile_atoms<R>();
  constexpr int resident = (int)(227 * 1024 / (bytes + 1024)) < 2 ? (int)(227 * 1024 / (bytes + 1024)) : 2;
  static_assert(resident >= 1, "a tile's slots fit in the shared memory of an SM");
  const int64_t grid = std::min<int64_t>(tiles, (int64_t)device_sms() * resident);
  kern<<<(unsigned)grid, kTileThreads, bytes, stream>>>(a, theta);
  return MTP_OK;
}

template <class LV, class R, bool DTHETA>
int efv_split_launch(const EfvArgs& a, cudaStream_t stream) {
  const int SS = a.n_species * a.n_species;
  const int64_t n = a.atom_end - a.atom_begin;
  if (n <= 0) return MTP_OK;
  // every thread of the last block that pads a tile must exist: a block's threads are whole tiles
  const int threads = sizeof(R) == 8 ? fp64_threads(n, 2 * a.n_parts) : kEfvThreads;
  const dim3 grid((unsigned)((n + threads - 1) / threads), 2 * a.n_parts);
  const size_t b0 = efv_smem_bytes<R, LV::NMU, false>(SS, a.n_q, a.m);
  const size_t base = (efv_smem_bytes<R, LV::NMU, DTHETA>(SS, a.n_q, a.m) + 15) & ~size_t(15);
  size_t b1 = base;
  if (DTHETA && a.n_species <= kAccSpecies) {
    const size_t more = sizeof(R) == 4 ? split_columns_bytes<LV>(a.n_species, a.n_q, threads)
                                       : efv_stage_bytes<R, DTHETA>(a.n_species, threads);
    if (base + more <= kMaxBlockSmem) b1 += more;
  }
  int rc;
  if ((rc = set_smem(split_moments_kernel<LV, R>, b0)) != MTP_OK) return rc;
  if ((rc = set_smem(split_adjoint_kernel<LV, R, DTHETA>, b1)) != MTP_OK) return rc;
  split_moments_kernel<LV, R><<<grid, threads, b0, stream>>>(a);
  if constexpr (std::is_same<R, float>::value) {
    // the scratch of a chunked call is sized for its first, largest range
    if (a.graphs && n >= kGraphAtoms) rc = graphs_launch<LV::LEVEL>(a, DTHETA, stream);
    else rc = tile_contract_launch<LV, R, DTHETA>(a, a.dtheta, stream);
  } else {
    rc = tile_contract_launch<LV, R, DTHETA>(a, a.dtheta, stream);
  }
  if (rc != MTP_OK) return rc;
  split_adjoint_kernel<LV, R, DTHETA><<<grid, threads, b1, stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("efv split kernels (level %d): %s", LV::LEVEL, cudaGetErrorString(e));
    return MTP_ERR_CUDA;
  }
  return MTP_OK;
}

template <class LV, class R, bool DTHETA>
int efv_launch_typed(const EfvArgs& a, cudaStream_t stream) {
  if constexpr (LV::NGROUPS > 1) {
    if (a.mbuf) return efv_split_launch<LV, R, DTHETA>(a, stream);
  }
  const int SS = a.n_species * a.n_species;
  const int64_t n = a.atom_end - a.atom_begin;
  if (n <= 0) return MTP_OK;
  const int threads = sizeof(R) == 8 ? fp64_threads(n, 1) : kEfvFusedThreads;
  const size_t base = (efv_smem_bytes<R, LV::NMU, DTHETA>(SS, a.n_q, a.m) + 15) & ~size_t(15);
  const size_t bytes = base + efv_acc_bytes<R, LV::NMU, DTHETA>(base, a.n_species, a.n_q, threads);
  auto kern = efv_kernel<LV, R, DTHETA>;
  // the single-group levels with the common radial basis size n_q = 8 run with
  // n_q fixed at compile time (FP64, 48,546 atoms with dE/dtheta: 3.5 -> 2.9 ms;
  // loops up to kMaxQ predicate FP64 operations away that still take their turn
  // in the pipe)
  if constexpr (LV::NGROUPS == 1) {
    if (a.n_q == kFixedQ) kern = efv_kernel<LV, R, DTHETA, kFixedQ>;
  }
  const int rc = set_smem(kern, bytes);
  if (rc != MTP_OK) return rc;
  kern<<<(unsigned)((n + threads - 1) / threads), threads, bytes, stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("efv kernel launch (level %d): %s", LV::LEVEL, cudaGetErrorString(e));
    return MTP_ERR_CUDA;
  }
  return MTP_OK;
}

template <class LV>
int efv_launch(const EfvArgs& a, int precision, bool want_dtheta, cudaStream_t stream) {
  if (precision == MTP_MIXED) {
    return want_dtheta ? efv_launch_typed<LV, float, true>(a, stream) : efv_launch_typed<LV, float, false>(a, stream);
  }
  return want_dtheta ? efv_launch_typed<LV, double, true>(a, stream) : efv_launch_typed<LV, double, false>(a, stream);
}

}  // namespace mtp
