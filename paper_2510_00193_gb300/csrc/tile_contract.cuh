// Contraction and reverse pass of the levels with component groups (18 and
// 20) for tiles of atoms: one block holds every value and adjoint of its
// tile's atoms in shared memory and runs the level's tile program (phases of
// independent dot products S[dst] (+)= sum w S[x] S[y] over the slots of one
// array; the reverse pass gathers, so no two threads add to one slot).
//
// A slot is a row of 32 bytes, one entry per atom of the tile: 8 atoms in
// FP32, 4 in FP64 and FP32 dual numbers, 2 in FP64 dual numbers.  Two threads
// share a record, each on 16 bytes of the row (one vector load per operand),
// so a term's indices are decoded once for several atoms.  Level 20 has 6,082
// slots (195 KB: one block of 16 warps per SM), level 18 2,302 (74 KB).
//
// Measured (whole evaluation, FCC level 20, against one thread per atom
// interpreting the program on local-memory arrays, or one warp per atom with
// shared-memory atomics for small systems): 2,016 atoms mixed 2.38 -> 0.134 ms,
// 108,000 atoms mixed 10.4 -> 4.2 ms (there the graph kernels of efv_graphs.cuh
// now take 1.41), one FP64 force-matching step of 4,000 atoms 41.3 -> 5.8 ms.
//
// Bound: on the FP32 path latency, 23 phases of which 8 hold a single slab
// (about 800 cycles each of a tile's 70,000; 14 of 23 warps per issue wait at
// barriers), and the shared-memory reads
// between them (two 16-byte reads per term and thread; the order of the terms
// puts the four rows that a quarter warp reads in different bank groups where
// it can: 24.8 instead of 31.0 thousand wavefronts per tile); on the FP64 path
// its pipe, 57% busy over the whole dual kernel.
#pragma once
#include <type_traits>

#include "efv_kernel.cuh"

namespace mtp {

constexpr int kTileThreads = 1024;
constexpr int kTileRowBytes = 32;
constexpr int kTileLanes = 16;   // records per warp (two threads each), as the programs are encoded

template <class R> constexpr int tile_atoms() { return kTileRowBytes / (int)sizeof(R); }

// atoms of a range rounded up to whole tiles of every type
__host__ __device__ __forceinline__ int64_t tile_padded(int64_t n) { return (n + 7) & ~int64_t(7); }

// Where atom t of the range keeps component c in the split kernels' scratch:
// tile after tile, [tile][c][atom of the tile], so that a tile's rows are
// contiguous.  Returns the address of component 0; components are
// tile_atoms<R>() entries apart.
template <class R>
__device__ __forceinline__ int64_t tile_offset(int64_t t, int ncomp) {
  constexpr int AB = tile_atoms<R>();
  return (t / AB) * ((int64_t)ncomp * AB) + (t % AB);
}

// 16 bytes of a row: the entries of 16 / sizeof(R) atoms.
template <class R> struct RowVec {
  static constexpr int N = 16 / (int)sizeof(R);
  R e[N];
};

template <class R> __device__ __forceinline__ RowVec<R> row_load(const unsigned char* p) {
  union { float4 f; double2 d; } u;
  RowVec<R> v;
  u.f = *reinterpret_cast<const float4*>(p);
  if constexpr (std::is_same<R, float>::value) {
    v.e[0] = u.f.x; v.e[1] = u.f.y; v.e[2] = u.f.z; v.e[3] = u.f.w;
  } else if constexpr (std::is_same<R, double>::value) {
    v.e[0] = u.d.x; v.e[1] = u.d.y;
  } else if constexpr (std::is_same<R, Dual<float>>::value) {
    v.e[0] = Dual<float>(u.f.x, u.f.y); v.e[1] = Dual<float>(u.f.z, u.f.w);
  } else {
    v.e[0] = Dual<double>(u.d.x, u.d.y);
  }
  return v;
}

template <class R> __device__ __forceinline__ void row_store(unsigned char* p, const RowVec<R>& v) {
  if constexpr (std::is_same<R, float>::value) {
    *reinterpret_cast<float4*>(p) = make_float4(v.e[0], v.e[1], v.e[2], v.e[3]);
  } else if constexpr (std::is_same<R, double>::value) {
    *reinterpret_cast<double2*>(p) = make_double2(v.e[0], v.e[1]);
  } else if constexpr (std::is_same<R, Dual<float>>::value) {
    *reinterpret_cast<float4*>(p) = make_float4(v.e[0].v, v.e[0].t, v.e[1].v, v.e[1].t);
  } else {
    *reinterpret_cast<double2*>(p) = make_double2(v.e[0].v, v.e[0].t);
  }
}

__device__ __forceinline__ float scaled(float a, float w) { return a * w; }
__device__ __forceinline__ double scaled(double a, double w) { return a * w; }
template <class S> __device__ __forceinline__ Dual<S> scaled(Dual<S> a, S w) { return {a.v * w, a.t * w}; }

// One term of a record: acc += w S[x] S[y].
template <class R, bool UNIT>
__device__ __forceinline__ void tile_term(const unsigned char* rows, const typename ScalarOf<R>::T* wt, uint32_t t,
                                          RowVec<R>& acc) {
  const RowVec<R> x = row_load<R>(rows + ((t & 0x1FFFu) << 5));
  const RowVec<R> y = row_load<R>(rows + ((t >> 8) & 0x3FFE0u));
  if constexpr (UNIT) {
#pragma unroll
    for (int k = 0; k < RowVec<R>::N; ++k) acc.e[k] = fmadd(x.e[k], y.e[k], acc.e[k]);
  } else {
    const typename ScalarOf<R>::T w = wt[t >> 26];
#pragma unroll
    for (int k = 0; k < RowVec<R>::N; ++k) acc.e[k] = fmadd(scaled(x.e[k], w), y.e[k], acc.e[k]);
  }
}

// `count` (1 to 4, the same for all lanes) terms of one chunk.
template <class R, bool UNIT>
__device__ __forceinline__ void tile_chunk(const unsigned char* rows, const typename ScalarOf<R>::T* wt, uint32_t t0,
                                           uint32_t t1, uint32_t t2, uint32_t t3, int count, RowVec<R>& acc) {
  if (count == 4) {
    tile_term<R, UNIT>(rows, wt, t0, acc);
    tile_term<R, UNIT>(rows, wt, t1, acc);
    tile_term<R, UNIT>(rows, wt, t2, acc);
    tile_term<R, UNIT>(rows, wt, t3, acc);
  } else if (count == 3) {
    tile_term<R, UNIT>(rows, wt, t0, acc);
    tile_term<R, UNIT>(rows, wt, t1, acc);
    tile_term<R, UNIT>(rows, wt, t2, acc);
  } else if (count == 2) {
    tile_term<R, UNIT>(rows, wt, t0, acc);
    tile_term<R, UNIT>(rows, wt, t1, acc);
  } else {
    tile_term<R, UNIT>(rows, wt, t0, acc);
  }
}

// One slab: each pair of threads runs one record, whose first chunk is in w0;
// two more chunks are on their way while one runs (a chunk's work is shorter
// than a read from L2).  `terms` is the number of terms of the longest record
// (shorter ones are filled up with 0 * 0), and the first `unit` chunks hold
// weights 1 only.  FP64 runs exactly these terms, the weights only where they
// are (its pipe is the bound); FP32 runs whole chunks, of one kind per slab:
// there each warp's latency counts, and the branches cost more than the filler
// (2,016 atoms: 157 against 137 us per evaluation).
template <class R, bool UNIT>
__device__ __forceinline__ void tile_slab(unsigned char* rows, const typename ScalarOf<R>::T* wt,
                                          const uint4* __restrict__ prog, uint4 w0, int terms, int unit) {
  constexpr bool EXACT = sizeof(typename ScalarOf<R>::T) == 8;
  const uint32_t dst = w0.x & 0x1FFFu;
  uint4 w1 = w0, w2 = w0;
  if (terms > 3) w1 = __ldg(prog + kTileLanes);
  if (terms > 7) w2 = __ldg(prog + 2 * kTileLanes);
  RowVec<R> acc;
  if (w0.x & 0x2000u) {
    acc = row_load<R>(rows + (dst << 5));
  } else {
#pragma unroll
    for (int k = 0; k < RowVec<R>::N; ++k) acc.e[k] = R(0);
  }
  if constexpr (EXACT) {
    uint32_t t0 = w0.y, t1 = w0.z, t2 = w0.w, t3 = w0.w;
    int count = min(terms, 3);
    while (true) {
      terms -= count;
      if (unit > 0) tile_chunk<R, true>(rows, wt, t0, t1, t2, t3, count, acc);
      else tile_chunk<R, false>(rows, wt, t0, t1, t2, t3, count, acc);
      if (terms <= 0) break;
      --unit;
      t0 = w1.x; t1 = w1.y; t2 = w1.z; t3 = w1.w;
      w1 = w2;
      prog += kTileLanes;
      if (terms > 8) w2 = __ldg(prog + 2 * kTileLanes);
      count = min(terms, 4);
    }
  } else {
    tile_term<R, UNIT>(rows, wt, w0.y, acc);
    tile_term<R, UNIT>(rows, wt, w0.z, acc);
    tile_term<R, UNIT>(rows, wt, w0.w, acc);
    for (terms -= 3; terms > 0; terms -= 4) {
      const uint4 w = w1;
      w1 = w2;
      prog += kTileLanes;
      if (terms > 8) w2 = __ldg(prog + 2 * kTileLanes);
      tile_term<R, UNIT>(rows, wt, w.x, acc);
      tile_term<R, UNIT>(rows, wt, w.y, acc);
      tile_term<R, UNIT>(rows, wt, w.z, acc);
      tile_term<R, UNIT>(rows, wt, w.w, acc);
    }
  }
  if (dst != 0x1FFFu) row_store<R>(rows + (dst << 5), acc);
}

// slab, phase: the program's slab descriptors and phase bounds, in shared
// memory.  The first chunk of a warp's next slab is read while it runs the one
// before, across the barrier between two phases too (a phase's slabs follow
// the last one's, so its first slab of this warp is known by then).
template <class LV, class R>
__device__ __forceinline__ void tile_phases(unsigned char* rows, const typename ScalarOf<R>::T* wt,
                                            const uint2* slab, const int* phase, int from, int to) {
  constexpr int W = kTileThreads / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint4* __restrict__ base = LV::tile_prog() + (lane >> 1);
  rows += (lane & 1) * 16;
  int start = phase[from], end = phase[from + 1];
  int s = 0, ns = 0;
  uint4 w;                                       // first chunk of slab s
  bool ready = false;
  for (int p = from; p < to; ++p) {
    const int next_end = phase[min(p + 2, (int)LV::TILE_PHASES)];
    if (!ready) {                                // the first phase, or the warp had no slab in the last one
      s = start + warp;
      ns = s + W < end ? s + W : end + warp;
      w = __ldg(base + slab[min(s, LV::TILE_SLABS - 1)].x);
    }
    ready = s < end;
    while (s < end) {
      const uint2 sl = slab[s];
      const uint4 nw = __ldg(base + slab[min(ns, LV::TILE_SLABS - 1)].x);
      const int stop = ns < end ? end : next_end;
      const int n2 = ns + W < stop ? ns + W : stop + warp;
      const int terms = (int)(sl.y >> 8), unit = (int)(sl.y & 0xFFu);
      if constexpr (sizeof(typename ScalarOf<R>::T) == 8) tile_slab<R, false>(rows, wt, base + sl.x, w, terms, unit);
      else if (unit == (terms + 4) >> 2) tile_slab<R, true>(rows, wt, base + sl.x, w, terms, unit);
      else tile_slab<R, false>(rows, wt, base + sl.x, w, terms, unit);
      s = ns; w = nw;
      ns = n2;
    }
    start = end;
    end = next_end;
    __syncthreads();
  }
}

// Shared memory: the slots, the weight table, one row of partial energies per
// warp, the slab descriptors and phase bounds, the species counts.
template <class LV, class R>
__host__ __device__ constexpr size_t tile_smem_bytes() {
  return (size_t)LV::TILE_SLOTS * kTileRowBytes + 64 * sizeof(double) + (kTileThreads / 32) * kTileRowBytes +
         (size_t)LV::TILE_SLABS * sizeof(uint2) + sizeof(int) * (LV::TILE_PHASES + 1 + kMaxSpecies);
}

// a.mbuf: a.n_parts buffers of partial moments (the neighbour sweep's shares,
// added here) and then the adjoints D = dE/dM, each [tile][NCOMP][atoms].
// R = S: site energies, their sum and (WANT_B) dE/dxi and the species counts
// into theta; R = Dual<S>: theta receives the tangent of dE/dxi.
template <class LV, class R, bool WANT_B>
__global__ void __launch_bounds__(kTileThreads) tile_contract_kernel(const EfvArgs a, double* __restrict__ theta) {
  using S = typename ScalarOf<R>::T;
  constexpr bool DUAL = !std::is_same<R, S>::value;
  constexpr int AB = tile_atoms<R>(), H = 2, N = RowVec<R>::N;
  constexpr int C = LV::NCOMP;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* rows = smem;
  S* wt = reinterpret_cast<S*>(smem + (size_t)LV::TILE_SLOTS * kTileRowBytes);
  R* esum = reinterpret_cast<R*>(smem + (size_t)LV::TILE_SLOTS * kTileRowBytes + 64 * sizeof(double));
  uint2* slab = reinterpret_cast<uint2*>(esum + (kTileThreads / 32) * AB);
  int* phase = reinterpret_cast<int*>(slab + LV::TILE_SLABS);
  int* cnt = phase + LV::TILE_PHASES + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const S* __restrict__ xi;
  if constexpr (sizeof(S) == 4) xi = a.xi_f;
  else xi = a.xi_d;
  if (tid < LV::TILE_WEIGHTS) wt[tid] = (S)LV::tile_weight()[tid];
  for (int k = tid; k < LV::TILE_SLABS; k += kTileThreads) slab[k] = LV::tile_slab()[k];
  if (tid <= LV::TILE_PHASES) phase[tid] = LV::tile_phase()[tid];
  if (tid < kMaxSpecies) cnt[tid] = 0;
  if (tid < AB) {
    reinterpret_cast<R*>(rows + (size_t)LV::TILE_ONE * kTileRowBytes)[tid] = R(1);
    reinterpret_cast<R*>(rows + (size_t)LV::TILE_ZERO * kTileRowBytes)[tid] = R(0);
  }
  const int64_t n = a.atom_end - a.atom_begin;
  const int64_t part = tile_padded(n) * C;       // entries of one buffer
  const int64_t tiles = (n + AB - 1) / AB;
  const R* __restrict__ mom = static_cast<const R*>(a.mbuf);
  R* __restrict__ dout = static_cast<R*>(a.mbuf) + part * a.n_parts;
  double e_sum = 0.0;                            // lane 0 of warps < AB: site energies of column `warp`
  constexpr int BPT = (LV::NBASIS + kTileThreads - 1) / kTileThreads;
  double b_sum[BPT];                             // dE/dxi of basis values tid, tid + kTileThreads, ...
#pragma unroll
  for (int k = 0; k < BPT; ++k) b_sum[k] = 0.0;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t mine = tile * AB + warp;         // the atom whose site energy lane 0 of warps < AB forms
    int zi = 0;
    double e0 = 0.0;
    if constexpr (!DUAL) {
      if (warp < AB && lane == 0 && mine < n) {
        zi = species_at(a.z, a.atom_begin + mine, a.n_species);
        e0 = a.species_energy[zi];
      }
    }
    // moments into the component rows, the shares of the sweep's parts added
    for (int u = tid; u < C * H; u += kTileThreads) {
      const unsigned char* src = reinterpret_cast<const unsigned char*>(mom + tile * (C * AB)) + u * 16;
      RowVec<R> v = row_load<R>(src);
      for (int p = 1; p < a.n_parts; ++p) {
        const RowVec<R> q = row_load<R>(src + (size_t)p * part * sizeof(R));
#pragma unroll
        for (int k = 0; k < N; ++k) v.e[k] += q.e[k];
      }
      row_store<R>(rows + u * 16, v);
    }
    __syncthreads();
    tile_phases<LV, R>(rows, wt, slab, phase, 0, LV::TILE_FORWARD);
    // basis values: site energies, dE/dxi, and the seeds of the reverse pass
    RowVec<R> e;
#pragma unroll
    for (int k = 0; k < N; ++k) e.e[k] = R(0);
    const int half = tid & 1;
    for (int b = tid >> 1; b < LV::NBASIS; b += kTileThreads / 2) {
      const int slot = __ldg(LV::tile_basis() + b);
      const S w = __ldg(xi + b);
      RowVec<R> seed;
      if constexpr (!DUAL) {
        const RowVec<R> v = row_load<R>(rows + (size_t)slot * kTileRowBytes + half * 16);
#pragma unroll
        for (int k = 0; k < N; ++k) e.e[k] = fmadd(R(w), v.e[k], e.e[k]);
      }
#pragma unroll
      for (int k = 0; k < N; ++k) seed.e[k] = R(w);
      row_store<R>(rows + (size_t)(LV::TILE_AOFF + slot) * kTileRowBytes + half * 16, seed);
    }
    if constexpr (WANT_B) {
#pragma unroll
      for (int k = 0; k < BPT; ++k) {
        const int b = tid + k * kTileThreads;
        if (b < LV::NBASIS) {
          const unsigned char* p = rows + (size_t)__ldg(LV::tile_basis() + b) * kTileRowBytes;
          const RowVec<R> v0 = row_load<R>(p), v1 = row_load<R>(p + 16);
          S s = S(0);
#pragma unroll
          for (int q = 0; q < N; ++q) {
            if constexpr (DUAL) s += v0.e[q].t + v1.e[q].t;
            else s += v0.e[q] + v1.e[q];
          }
          b_sum[k] += (double)s;
        }
      }
    }
    if constexpr (!DUAL) {
#pragma unroll
      for (int o = 2; o < 32; o <<= 1) {
#pragma unroll
        for (int k = 0; k < N; ++k) e.e[k] += __shfl_xor_sync(0xffffffffu, e.e[k], o);
      }
      if (lane < 2) row_store<R>(reinterpret_cast<unsigned char*>(esum + warp * AB) + lane * 16, e);
    }
    __syncthreads();
    if constexpr (!DUAL) {
      if (warp < AB) {                             // one warp per column (a serial sum: 5,000 cycles of a tile's 74,000)
        const double ei = warp_sum((double)esum[lane * AB + warp]) + e0;
        if (lane == 0 && mine < n) {
          a.e_atom[a.atom_begin + mine] = ei;
          e_sum += ei;
          if (!isfinite(ei)) flag_status(a.status, MTP_ERR_NONFINITE);
          if (WANT_B) atomicAdd(cnt + zi, 1);
        }
      }
    }
    tile_phases<LV, R>(rows, wt, slab, phase, LV::TILE_FORWARD, LV::TILE_PHASES);
    {
      unsigned char* dst = reinterpret_cast<unsigned char*>(dout + tile * (C * AB));
      const unsigned char* src = rows + (size_t)LV::TILE_AOFF * kTileRowBytes;
      for (int u = tid; u < C * H; u += kTileThreads) row_store<R>(dst + u * 16, row_load<R>(src + u * 16));
    }
    __syncthreads();
  }
  if constexpr (!DUAL) {
    if (warp < AB && lane == 0) atomicAdd(a.e_total, e_sum);
  }
  if constexpr (WANT_B) {
    const int64_t xoff = a.n_species + (int64_t)LV::NMU * a.n_q * a.n_species * a.n_species;
#pragma unroll
    for (int k = 0; k < BPT; ++k) {
      const int b = tid + k * kTileThreads;
      if (b < LV::NBASIS) atomicAdd(theta + xoff + b, b_sum[k]);
    }
    if constexpr (!DUAL) {
      if (tid < a.n_species) atomicAdd(theta + tid, (double)cnt[tid]);
    }
  }
}

}  // namespace mtp
