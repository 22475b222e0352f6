// Contraction of the levels with component groups (18 and 20) in FP32 for
// large systems: one thread per atom, straight-line code.  The whole
// contraction is far larger than the instruction cache (level 20: some 50,000
// instructions), so it is cut into groups of graphs, each a kernel of its own
// whose code fits: the values of the graphs, then the basis products with E
// and the graph adjoints, then per group its graphs' nodes again and their
// reverse pass.  Operands stay in registers, where the tile program
// (tile_contract.cuh) reads each of its ~31,000 terms' operands from shared
// memory; moments and the D accumulators pass between the kernels through
// memory (about 12 KB per atom at level 20), and so do the graph values
// (G[graph][atom]).
//
// Measured, level 20, 108,000 atoms, mixed: contraction 3.60 ms (tile program)
// -> 0.59 ms (values 104, products 48, adjoints 435 us); the whole evaluation
// 4.22 -> 1.41 ms.  Below 4,096 atoms the tile program stays: these kernels would
// run on less than half a wave each.  Tile program / these, whole call (us):
//   level 18:  2,048 atoms 87/109, 2,916 111/119, 4,000 129/119, 5,808 170/143, 8,788 217/141
//   level 20:  2,048 117 to 127/213, 4,000 202/222, 4,840 208/227, 5,808 271/255, 8,788 374/266
// with dE/dtheta at level 20: 4,000 239/271, 4,840 241/271, 5,808 328/327.  One
// line for both levels: each loses up to a tenth close to it, level 18 below,
// level 20 above.
// Bound: instruction issue at 8 warps per SM (255 registers); the groups that
// touch many components (281 of 295 in one) also wait for their D columns.
#pragma once
#include <utility>

#include "efv_kernel.cuh"
#include "tile_contract.cuh"

namespace mtp {

// Partial moments of the neighbour sweep's shares added into the first.
static __global__ void __launch_bounds__(256) sum_shares_kernel(float* __restrict__ mom, int64_t part, int n_parts) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= part) return;
  float s = mom[k];
  for (int p = 1; p < n_parts; ++p) s += mom[p * part + k];
  mom[k] = s;
}

template <class GR, int NCOMP, int K>
__global__ void __launch_bounds__(kEfvThreads) graph_values_kernel(const float* __restrict__ mom, int64_t n,
                                                                   float* __restrict__ G, int64_t gld) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  GR::template values<K>(mom + tile_offset<float>(t, NCOMP), tile_atoms<float>(), G + t, gld);
}

// Sums basis values over the warp: 32 of them pass through shared memory, and
// lane e adds value e of all lanes (in four chains) into the block's dE/dxi.
// The products kernel does little else, so five shuffles and an atomic per
// value were most of its time (108,000 atoms with dE/dtheta: 266 -> 63 us, 48
// without).  The values come in the order of their indices.
template <int M> struct StagedBasisSink {
  float* stage;   // the warp's [32][33]
  float* dxi;
  int lane;
  bool active;
  __device__ __forceinline__ void operator()(int a, float v) const {
    stage[(a & 31) * 33 + lane] = active ? v : 0.f;
    if ((a & 31) == 31 || a == M - 1) {
      __syncwarp();
      if (lane <= (a & 31)) {
        const float* row = stage + lane * 33;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int l = 0; l < 32; ++l) s[l & 3] += row[l];
        atomicAdd(dxi + (a & ~31) + lane, (s[0] + s[1]) + (s[2] + s[3]));
      }
      __syncwarp();
    }
  }
};

// Shared memory of the products kernel: no pair coefficients, so it does not
// grow with the species or n_q, and the staging area always fits beside the sums.
template <class LV, bool DTHETA> constexpr size_t graph_products_bytes() {
  return efv_sums_bytes<float, LV::NBASIS>() + (DTHETA ? sizeof(float) * 33 * kEfvThreads : 0);
}

template <class GR, class LV, bool DTHETA>
__global__ void __launch_bounds__(kEfvThreads) graph_products_kernel(const EfvArgs a, const float* __restrict__ G,
                                                                     float* __restrict__ GB, int64_t gld) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EfvShared<float, LV::NMU, DTHETA> sm;
  sm.template setup_sums<LV::NBASIS>(a, smem_raw);
  __syncthreads();
  const int64_t n = a.atom_end - a.atom_begin;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool active = t < n;
  double e_i = 0.0;
  const float w[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // lanes without an atom run along on the first one (the basis values are summed across the warp)
  const int64_t u = active ? t : 0;
  if (__any_sync(0xffffffffu, active)) {
    // the scratch has room for the padding atoms of the last block's warps: see split_scratch_bytes
    float* stage = reinterpret_cast<float*>(smem_raw + efv_sums_bytes<float, LV::NBASIS>());
    const StagedBasisSink<LV::NBASIS> sink{stage + (threadIdx.x >> 5) * 32 * 33, sm.dxi, (int)(threadIdx.x & 31),
                                           active};
    const float e = GR::template products<DTHETA>(G + u, gld, sm.xi, GB + t, sink);
    if (active) {
      const int64_t i = a.atom_begin + t;
      const int zi = species_at(a.z, i, a.n_species);
      e_i = a.species_energy[zi] + (double)e;
      a.e_atom[i] = e_i;
      if (!isfinite(e_i)) flag_status(a.status, MTP_ERR_NONFINITE);
      if (DTHETA) atomicAdd(sm.cnt + zi, 1);
    }
  }
  efv_block_flush<LV, float, DTHETA>(sm, e_i, w, a.e_total, a.virial, a.dtheta, kFlushEW | kFlushDxi);
}

template <class GR, int NCOMP, int K>
__global__ void __launch_bounds__(kEfvThreads) graph_adjoint_kernel(const float* __restrict__ mom, int64_t n,
                                                                    const float* __restrict__ GB, int64_t gld,
                                                                    float* __restrict__ D) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int64_t at = tile_offset<float>(t, NCOMP);
  GR::template adjoint<K>(mom + at, tile_atoms<float>(), GB + t, gld, D + at);
}

template <class GR, class LV, bool DTHETA, int... V, int... A>
int graphs_launch_seq(const EfvArgs& a, cudaStream_t stream, std::integer_sequence<int, V...>,
                      std::integer_sequence<int, A...>) {
  const int64_t n = a.atom_end - a.atom_begin;
  if (n <= 0) return MTP_OK;
  const int64_t part = tile_padded(n) * LV::NCOMP, gld = graph_padded(n);
  float* mom = static_cast<float*>(a.mbuf);
  float* D = mom + part * a.n_parts;
  float* G = D + part;
  float* GB = G + gld * LV::NGRAPH;
  const unsigned grid = (unsigned)((n + kEfvThreads - 1) / kEfvThreads);
  constexpr size_t bytes = graph_products_bytes<LV, DTHETA>();
  static_assert(bytes <= 48 * 1024, "within the default limit of a launch");
  if (a.n_parts > 1)
    sum_shares_kernel<<<(unsigned)((part + 255) / 256), 256, 0, stream>>>(mom, part, a.n_parts);
  (graph_values_kernel<GR, LV::NCOMP, V><<<grid, kEfvThreads, 0, stream>>>(mom, n, G, gld), ...);
  graph_products_kernel<GR, LV, DTHETA><<<grid, kEfvThreads, bytes, stream>>>(a, G, GB, gld);
  (graph_adjoint_kernel<GR, LV::NCOMP, A><<<grid, kEfvThreads, 0, stream>>>(mom, n, GB, gld, D), ...);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("graph kernels (level %d): %s", LV::LEVEL, cudaGetErrorString(e));
    return MTP_ERR_CUDA;
  }
  return MTP_OK;
}

template <class GR, class LV>
int graphs_launch_typed(const EfvArgs& a, bool want_dtheta, cudaStream_t stream) {
  using Vs = std::make_integer_sequence<int, GR::VALUE_GROUPS>;
  using As = std::make_integer_sequence<int, GR::ADJOINT_GROUPS>;
  return want_dtheta ? graphs_launch_seq<GR, LV, true>(a, stream, Vs(), As())
                     : graphs_launch_seq<GR, LV, false>(a, stream, Vs(), As());
}

}  // namespace mtp
