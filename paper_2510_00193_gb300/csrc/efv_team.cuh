// Energy/force kernel in which the W warps of a block share 32 atoms (lane =
// atom; fewer in small systems, with several lanes per atom): the block-parallel variant (the paper keeps a separate GPU pair style
// that spreads one atom's work over a team of threads for small systems, Sec.
// 2.1, Table 1, and Sec. 4).  With one thread per atom a system of a few
// thousand atoms leaves most of the GPU idle, and every thread walks ~26-54
// pairs twice and a contraction of ~10k instructions in sequence.  Here
//   sweep 1: warp w takes the w-th share of every lane's pairs; the partial
//            moments meet in shared memory ([w][component][lane], no bank
//            conflicts) and are added component by component;
//   contract: warp p runs part p of the generated contraction on all 32
//            atoms (part_values<p>, then part_adjoint<p> once the graph values
//            of all parts are there), so the warps execute different code on
//            the same atoms and no work is repeated but the recomputed nodes;
//            the parts' shares of D = dE_i/dM are added as the moments were;
//   sweep 2: warp w takes its share of the pairs again; F_i is added across
//            the warps in shared memory, F_j -= g is scattered.
// Taken for systems whose blocks fit in one wave (the rule stands at the call);
// above that the instruction streams of four different contraction parts on an
// SM cost more than the idle lanes of one thread per atom.  Level 16, mixed
// energies and forces, this kernel / one thread per atom (whole call, us):
// 2,000 atoms 39 / 60, 8,192 45 / 57, 16,000 74 / 57; with dE/dtheta 2,000 atoms
// 49 / 108, 16,000 171 / 111; FP64 128 atoms 115 / 224 (the form before), 1,152
// 137 / 464, 3,432 272 / 959, 8,704 558 / 941, 16,000 1,081 / 953.  With 32 atoms
// per block always, FP64 at 128 atoms took 269 us: four SMs' FP64 pipes.
// The form before (one warp per atom, every lane running the whole contraction)
// took 59 us at 2,000 atoms.  Bound: instruction fetch (ncu: 4.4 of 8.3 warps per
// issue wait for instructions at 2,000 atoms).
// Levels with component groups (18 and 20) run the split kernels at every size.
#pragma once
#include "efv_kernel.cuh"

namespace mtp {

// Many species with a large radial basis: the coefficients leave no room for
// the shares (the caller takes one thread per atom then).
constexpr int kTeamNoRoom = 1000;
constexpr int kTeamMinAtoms = 2;
constexpr int kTeamWarps = 4;   // 8 measured slower above 2,000 atoms (the extra warps wait through the contraction)

// A lane's column of a [k][32] array in shared memory.
template <class R> struct LaneColumn {
  R* p;
  __device__ __forceinline__ R& operator[](int k) const { return p[k * 32]; }
};
template <class R> struct GraphColumn {
  R* p;
  __device__ __forceinline__ R operator()(int g) const { return p[g * 32]; }
  __device__ __forceinline__ void put(int g, R v) const { p[g * 32] = v; }
};

template <class LV, class R>
__host__ __device__ __forceinline__ size_t team_buf_bytes(int W) {
  // partial moments / D shares, their sum, graph values, energies of the parts, forces of the warps
  const size_t shares = W > LV::NPARTS ? W : LV::NPARTS;
  return sizeof(R) * 32 * (shares * LV::NSWEPT + LV::NSWEPT + LV::NGRAPH + LV::NPARTS + 3 * (size_t)W);
}

template <class LV, class R>
__device__ __forceinline__ void team_values(int p, LaneColumn<R> M, GraphColumn<R> G) {
  if (p == 0) LV::template part_values_0<R>(M, G);
  else if (p == 1) LV::template part_values_1<R>(M, G);
  else if (p == 2) LV::template part_values_2<R>(M, G);
  else LV::template part_values_3<R>(M, G);
}

template <class LV, class R, bool WANT_B, class BV>
__device__ __forceinline__ R team_adjoint(int p, LaneColumn<R> M, GraphColumn<R> G,
                                          const typename ScalarOf<R>::T* xi, LaneColumn<R> share, BV B) {
  auto put = [&](const R (&D)[LV::NSWEPT]) {
#pragma unroll
    for (int k = 0; k < LV::NSWEPT; ++k) share[k] = D[k];
  };
  R D[LV::NSWEPT];
  R e;
  if (p == 0) { e = LV::template part_adjoint_0<R, WANT_B>(M, G, xi, D, B); put(D); }
  else if (p == 1) { e = LV::template part_adjoint_1<R, WANT_B>(M, G, xi, D, B); put(D); }
  else if (p == 2) { e = LV::template part_adjoint_2<R, WANT_B>(M, G, xi, D, B); put(D); }
  else { e = LV::template part_adjoint_3<R, WANT_B>(M, G, xi, D, B); put(D); }
  return e;
}

template <class LV, class R, bool DTHETA, int W, int NQ>
__global__ void __launch_bounds__(32 * W, 2) efv_team_kernel(const EfvArgs a, const int atoms) {
  static_assert(LV::NGROUPS == 1, "levels with one component group");
  static_assert(LV::NPARTS == 4, "four parts");
  constexpr int NMU = LV::NMU, NSW = LV::NSWEPT, NP = LV::NPARTS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EfvShared<R, NMU, DTHETA> sm;
  sm.setup(a, smem_raw);
  sm.zero_gradients();
  const int SS = a.n_species * a.n_species;
  constexpr int SHARES = W > NP ? W : NP;
  R* shares = reinterpret_cast<R*>(smem_raw + ((efv_smem_bytes<R, NMU, DTHETA>(SS, a.n_q, a.m) + 15) & ~size_t(15)) +
                                   efv_own_bytes<R, NMU, DTHETA>(a.n_species, a.n_q, 32 * W) +
                                   efv_stage_bytes<R, DTHETA>(a.n_species, 32 * W));
  R* total = shares + SHARES * NSW * 32;
  R* graphs = total + NSW * 32;
  R* energy = graphs + LV::NGRAPH * 32;
  R* force = energy + NP * 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // lane = atom + atoms * sub: the lanes of an atom take shares of its pairs too,
  // and run the contraction on the same values
  const int subs = 32 / atoms, sub = lane / atoms;
  const int64_t i0 = a.atom_begin + (int64_t)blockIdx.x * atoms + (lane & (atoms - 1));
  const bool active = i0 < a.atom_end, owner = active && sub == 0;
  const int64_t i = active ? i0 : a.atom_begin;
  __syncthreads();
  PairGeom<R> geom;
  geom.load_centre(a, i, cell_of<R>(a));
  const int zi = species_at(a.z, i, a.n_species);
  int64_t row, row_end;
  list_row(a, i, row, row_end);
  const int len = active ? (int)(row_end - row) : 0;
  const int share = warp * subs + sub, all = W * subs;
  const int64_t beg = row + (int64_t)len * share / all, end = row + (int64_t)len * (share + 1) / all;
  const LaneColumn<R> mine{shares + (size_t)warp * NSW * 32 + lane}, sum{total + lane};
  // sum over the lanes of one atom (every one of them receives it)
  auto add_subs = [&](R v) {
    for (int o = atoms; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  // adds the shares of `count` warps, component by component
  auto add_shares = [&](int count, bool across) {
    for (int k = warp; k < NSW; k += W) {
      R s = shares[k * 32 + lane];
      for (int v = 1; v < count; ++v) s += shares[(v * NSW + k) * 32 + lane];
      sum[k] = across ? add_subs(s) : s;
    }
  };
  {
    R M[LV::NCOMP];
#pragma unroll
    for (int c = 0; c < LV::NCOMP; ++c) M[c] = R(0);
    moment_sweep<LV, R, DTHETA, -1, false, NQ>(a, sm, geom, a.cell, zi, beg, end, M);
    LV::template store_swept<R>(M, mine);
  }
  __syncthreads();
  add_shares(W, true);
  __syncthreads();
  const GraphColumn<R> G{graphs + lane};
  for (int p = warp; p < NP; p += W) team_values<LV, R>(p, sum, G);
  __syncthreads();
  for (int p = warp; p < NP; p += W) {
    const LaneColumn<R> share{shares + (size_t)p * NSW * 32 + lane};
    R e;
    if constexpr (DTHETA)
      e = team_adjoint<LV, R, true>(p, sum, G, sm.xi, share, WarpBasisSink<R>{sm.dxi, lane, owner});
    else
      e = team_adjoint<LV, R, false>(p, sum, G, sm.xi, share, (R*)nullptr);
    energy[p * 32 + lane] = e;
  }
  __syncthreads();
  add_shares(NP, false);
  double e_i = 0.0;
  if (warp == 0 && owner) {
    for (int p = 0; p < NP; ++p) e_i += (double)energy[p * 32 + lane];
    e_i += a.species_energy[zi];
    a.e_atom[i] = e_i;
    if (DTHETA) atomicAdd(sm.cnt + zi, 1);
  }
  __syncthreads();
  R w[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
  R fx = R(0), fy = R(0), fz = R(0);
  // dE/dc of this thread's pairs, per neighbour species (as in efv_atom)
  R acc_local[(DTHETA && sizeof(R) == 8) ? kAccSpecies * NMU * kMaxQ : 1];
  const AccView<R> acc = own_accumulators<R, NQ>(sm.acc, acc_local);
  const bool own_acc = DTHETA && sm.S <= kAccSpecies && acc.p != nullptr;
  if (own_acc) {
    for (int t = 0; t < sm.S * NMU * sm.nq; ++t) acc[t] = R(0);
  }
  {
    R D[LV::NCOMP];
    LV::template load_swept<R>(D, sum);
    adjoint_sweep<LV, R, DTHETA, -1, false, NQ>(a, sm, geom, a.cell, zi, beg, end, D, fx, fy, fz, w, acc, own_acc);
  }
  force[(warp * 3 + 0) * 32 + lane] = fx;
  force[(warp * 3 + 1) * 32 + lane] = fy;
  force[(warp * 3 + 2) * 32 + lane] = fz;
  __syncthreads();
  if (own_acc) add_warp_gradients(sm, 0, NMU * sm.nq, zi, active, [&](int t) { return acc[t]; });
  if (warp == 0) {
    for (int v = 1; v < W; ++v) {
      fx += force[(v * 3 + 0) * 32 + lane];
      fy += force[(v * 3 + 1) * 32 + lane];
      fz += force[(v * 3 + 2) * 32 + lane];
    }
    fx = add_subs(fx);
    fy = add_subs(fy);
    fz = add_subs(fz);
  }
  if (warp == 0 && owner) {
    scatter_force(a, i, fx, fy, fz);
    if (!isfinite(e_i) || !isfinite((double)fx) || !isfinite((double)fy) || !isfinite((double)fz))
      flag_status(a.status, MTP_ERR_NONFINITE);
  }
  efv_block_flush<LV, R, DTHETA>(sm, e_i, w, a.e_total, a.virial, a.dtheta);
}

template <class LV, class R, bool DTHETA>
int efv_team_launch_typed(const EfvArgs& a, cudaStream_t stream) {
  const int SS = a.n_species * a.n_species;
  const size_t bytes = ((efv_smem_bytes<R, LV::NMU, DTHETA>(SS, a.n_q, a.m) + 15) & ~size_t(15)) +
                       efv_own_bytes<R, LV::NMU, DTHETA>(a.n_species, a.n_q, 32 * kTeamWarps) +
                       efv_stage_bytes<R, DTHETA>(a.n_species, 32 * kTeamWarps) +
                       team_buf_bytes<LV, R>(kTeamWarps);
  if (bytes > kMaxBlockSmem) return kTeamNoRoom;
  auto kern = efv_team_kernel<LV, R, DTHETA, kTeamWarps, 0>;
  if (a.n_q == kFixedQ) kern = efv_team_kernel<LV, R, DTHETA, kTeamWarps, kFixedQ>;
  int rc = set_smem(kern, bytes);
  if (rc != MTP_OK) return rc;
  const int64_t n = a.atom_end - a.atom_begin;
  if (n <= 0) return MTP_OK;
  // fewer atoms per block while the blocks still fit one to an SM: the lanes of
  // an atom share its pairs, and the pipes of more SMs take part
  int atoms = 32;
  const int64_t sms = device_sms();
  while (atoms > kTeamMinAtoms && (n + atoms / 2 - 1) / (atoms / 2) <= sms) atoms /= 2;
  kern<<<(unsigned)((n + atoms - 1) / atoms), 32 * kTeamWarps, bytes, stream>>>(a, atoms);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("team kernel launch (level %d): %s", LV::LEVEL, cudaGetErrorString(e));
    return MTP_ERR_CUDA;
  }
  return MTP_OK;
}

template <class LV>
int efv_team_launch(const EfvArgs& a, int precision, bool want_dtheta, cudaStream_t stream) {
  if (precision == MTP_MIXED)
    return want_dtheta ? efv_team_launch_typed<LV, float, true>(a, stream)
                       : efv_team_launch_typed<LV, float, false>(a, stream);
  return want_dtheta ? efv_team_launch_typed<LV, double, true>(a, stream)
                     : efv_team_launch_typed<LV, double, false>(a, stream);
}

}  // namespace mtp
