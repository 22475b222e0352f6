// Cell-list construction of the full periodic neighbour list.
//
// Atoms are binned in fractional coordinates.  Along axis k the cell has
// plane spacing h_k = 1 / |column k of H^-1|; a pair closer than R_cut
// differs by at most R_cut / h_k in fractional coordinate k, so with nb_k bins
// it lies at most R_k = floor(R_cut nb_k / h_k) + 1 bins away.  Periodic axes
// are searched over unwrapped bin offsets t in [b - R_k, b + R_k]; bin
// t mod nb_k together with the wrap q = floor(t / nb_k) gives each image of
// each candidate exactly once (several images for cells thinner than R_cut).
// The in/out decision is the exact FP64 expression of the list definition:
// d = (x_j + s) - x_i, s = (n1 a + n2 b) + n3 c, r^2 = (dx dx + dy dy) + dz dz,
// each operation separately rounded (explicit _rn intrinsics, no contraction),
// wherever an FP32 estimate with a proven error bound cannot decide it.
//
// Measured (build of 500,000 BCC atoms at R_cut 5 A: 1.31 -> 0.54 ms; list and
// level-16 evaluation of 14,858 atoms 0.434 -> 0.214 ms) against two searches
// by one thread per atom that handled each found neighbour inside the candidate
// loop, and a sorting network over 64-bit keys.  What it rests on:
//   - one search: count_kernel leaves what it finds, order_kernel makes rows;
//   - the candidate loop only tests and sets bits, so a warp stays together
//     (one warp per atom with lanes on rows was 2x slower: 25 scattered loads a
//     step);
//   - bins of R_cut x R_cut x R_cut/4 (9 runs of ~20 slots);
//   - a tighter bound on the FP32 error: each exact decision costs a warp some
//     40 FP64 instructions, and there were 0.3 per atom (now 0.01).
// Bound now: instruction issue (count 172 us, order 211 us at 500,000 atoms).
#include <cub/device/device_scan.cuh>
#include <cuda/std/functional>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "mtp_internal.cuh"
#include "scratch_plan.h"

namespace mtp {

struct NbrGeom {
  double cell[9];
  float cellf[9];
  float rc2_hi;       // prefilter bound: rc^2 plus the worst FP32 rounding of r^2
  float rc2_lo;       // below it (and above rz2) a candidate is inside whatever the rounding
  float rz2;          // FP32 r^2 above which the exact r^2 is certainly positive
  double hinv[9];
  double origin[3];   // fractional origin of the bin grid (0 on periodic axes)
  double width[3];    // fractional width of one bin
  double inv_width[3];
  int nb[3];
  int reach[3];
  int pbc[3];
  bool unique;        // no atom can be the neighbour of another through two images
  double rc2;
};

// Order-preserving map of doubles onto unsigned integers (for atomic min/max).
__device__ __forceinline__ unsigned long long ordered_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
static double unordered_bits(unsigned long long b) {
  const unsigned long long r = (b >> 63) ? (b & 0x7fffffffffffffffull) : ~b;
  double v;
  memcpy(&v, &r, sizeof(v));
  return v;
}

// Bin of a fractional coordinate along axis k.
__device__ __forceinline__ int bin_coord(double s, const NbrGeom& g, int k) {
  const int b = (int)floor((s - g.origin[k]) * g.inv_width[k]);
  return min(max(b, 0), g.nb[k] - 1);
}
// Bin coordinates of an atom in one word (at most 1024 bins per axis).
__device__ __forceinline__ int pack_bin(int b0, int b1, int b2) { return b0 | (b1 << 10) | (b2 << 20); }
__device__ __forceinline__ int bin_index(int p, const NbrGeom& g) {
  return ((p & 1023) * g.nb[1] + ((p >> 10) & 1023)) * g.nb[2] + (p >> 20);
}

// Wrapped position and wrap counts of every atom.  PERIODIC (every axis is):
// the bins are known beforehand, so the atom is also binned here (its rank in
// the bin is its place in the bin's slots).  Otherwise the fractional
// coordinates and their extent along the open axes come first, and
// bin_count_kernel bins the atoms once the host has laid the bins.
// meta: wrap counts and the packed bin.
template <bool PERIODIC>
__global__ void wrap_kernel(const double* __restrict__ x, int64_t n, NbrGeom g, double* __restrict__ sw,
                            int4* __restrict__ meta, unsigned long long* __restrict__ extent, float4* __restrict__ xw,
                            int* __restrict__ rank, int* __restrict__ bin_count, int* __restrict__ status) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
  if (i < n) {
    const double px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2];
    if (!isfinite(px) || !isfinite(py) || !isfinite(pz)) atomicCAS(status, 0, MTP_ERR_NONFINITE);
    double sv[3];
    int wv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      double s = px * g.hinv[0 + k] + py * g.hinv[3 + k] + pz * g.hinv[6 + k];
      int w = 0;
      if (PERIODIC || g.pbc[k]) {
        const double f = floor(s);
        w = (int)f;
        s -= f;
        if (s >= 1.0) { s -= 1.0; w += 1; }
        if (s < 0.0) s = 0.0;
      }
      sv[k] = s;
      wv[k] = w;
      if (!PERIODIC) {
        sw[3 * i + k] = s;
        lo[k] = hi[k] = ordered_bits(s);
      }
    }
    // wrapped Cartesian position in FP32, for the distance prefilter
    xw[i] = make_float4((float)(sv[0] * g.cell[0] + sv[1] * g.cell[3] + sv[2] * g.cell[6]),
                        (float)(sv[0] * g.cell[1] + sv[1] * g.cell[4] + sv[2] * g.cell[7]),
                        (float)(sv[0] * g.cell[2] + sv[1] * g.cell[5] + sv[2] * g.cell[8]), 0.f);
    int bin = 0;
    if (PERIODIC) {
      bin = pack_bin(bin_coord(sv[0], g, 0), bin_coord(sv[1], g, 1), bin_coord(sv[2], g, 2));
      rank[i] = atomicAdd(bin_count + bin_index(bin, g), 1);
    }
    meta[i] = make_int4(wv[0], wv[1], wv[2], bin);
  }
  if (PERIODIC) return;
  // min/max of the fractional coordinates (used to lay bins over open axes)
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (g.pbc[k]) continue;
    for (int o = 16; o > 0; o >>= 1) {
      lo[k] = min(lo[k], __shfl_down_sync(0xffffffffu, lo[k], o));
      hi[k] = max(hi[k], __shfl_down_sync(0xffffffffu, hi[k], o));
    }
    if ((threadIdx.x & 31) == 0) {
      atomicMin(extent + 2 * k, lo[k]);
      atomicMax(extent + 2 * k + 1, hi[k]);
    }
  }
}

__global__ void bin_count_kernel(const double* __restrict__ sw, int64_t n, NbrGeom g, int4* __restrict__ meta,
                                 int* __restrict__ rank, int* __restrict__ bin_count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int bin = pack_bin(bin_coord(sw[3 * i], g, 0), bin_coord(sw[3 * i + 1], g, 1), bin_coord(sw[3 * i + 2], g, 2));
  rank[i] = atomicAdd(bin_count + bin_index(bin, g), 1);
  meta[i].w = bin;
}

// Atoms in bin order: their FP32 wrapped positions, and their wrap counts and
// indices, by slot (the candidate loops read them without a dependent gather).
__global__ void bin_fill_kernel(const int4* __restrict__ meta, int64_t n, NbrGeom g, const int* __restrict__ bin_start,
                                const int* __restrict__ rank, const float4* __restrict__ xw,
                                float4* __restrict__ bin_xw, int4* __restrict__ bin_meta) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int4 m = meta[i];
  const int slot = bin_start[bin_index(m.w, g)] + rank[i];
  bin_xw[slot] = xw[i];
  bin_meta[slot] = make_int4(m.x, m.y, m.z, (int)i);
}

__device__ __forceinline__ int floor_div(int t, int m) { return t >= 0 ? t / m : -((-t + m - 1) / m); }
// floor(t / m); most searches leave the cell by less than one period
__device__ __forceinline__ int wrap_count(int t, int m) {
  if (t >= 0 && t < m) return 0;
  if (t < 0 && t >= -m) return -1;
  if (t >= m && t < 2 * m) return 1;
  return floor_div(t, m);
}

// Canonical order of a list entry, (j, n1, n2, n3) lexicographic: j, then the
// image with n1 in the highest bits (pack_image has it in the lowest).
__device__ __forceinline__ uint32_t image_key(int32_t img) {
  const uint32_t u = (uint32_t)img;
  return ((u & 1023u) << 20) | (u & 0xFFC00u) | (u >> 20);
}
__device__ __forceinline__ unsigned long long row_key(int32_t j, int32_t img) {
  return ((unsigned long long)(uint32_t)j << 30) | image_key(img);
}

constexpr int kSearchThreads = 128;
// Columns of found neighbours above this size (some 10 million atoms at 60
// neighbours) are given back after the build.  Below it the list keeps them and
// a build in place allocates nothing: giving them back costs a build of 9.8
// million atoms 1.3 of 8.0 ms (4.2 GB).
constexpr size_t kColumnsKept = size_t(4) << 30;
constexpr int kRowBuffer = 1536;   // entries per warp kept in shared memory while their rows are put in order

// Places the buffered entries lane, lane + 32, ... (R of them from entry
// `first` on) of one row (cnt entries, padded to a multiple of 4 with
// j = 0xFFFFFFFF) in canonical order: entry e goes to the position
// equal to the number of entries before it.  UNIQUE: no atom appears twice in
// a row, so j alone decides.
template <int R, bool UNIQUE>
__device__ __forceinline__ void place_row(const uint32_t* bj, const uint32_t* bi, int cnt, int first, int lane,
                                          int32_t* __restrict__ out_j, int32_t* __restrict__ out_img) {
  uint32_t mj[R], mi[R], mk[R];
  int rank[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = first + 32 * r + lane;
    mj[r] = e < cnt ? bj[e] : 0xFFFFFFFFu;
    mi[r] = e < cnt ? bi[e] : 0u;
    mk[r] = UNIQUE ? 0u : image_key((int32_t)mi[r]);
    rank[r] = 0;
  }
  for (int t = 0; t < cnt; t += 4) {
    const uint4 o = *reinterpret_cast<const uint4*>(bj + t);
    if (UNIQUE) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        rank[r] += (int)(o.x < mj[r]) + (int)(o.y < mj[r]) + (int)(o.z < mj[r]) + (int)(o.w < mj[r]);
    } else {
      const uint4 p = *reinterpret_cast<const uint4*>(bi + t);
      const uint32_t oj[4] = {o.x, o.y, o.z, o.w};
      const uint32_t ok[4] = {image_key((int32_t)p.x), image_key((int32_t)p.y), image_key((int32_t)p.z),
                              image_key((int32_t)p.w)};
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int q = 0; q < 4; ++q) rank[r] += (int)(oj[q] < mj[r] || (oj[q] == mj[r] && ok[q] < mk[r]));
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (first + 32 * r + lane < cnt) {
      out_j[rank[r]] = (int32_t)mj[r];
      out_img[rank[r]] = (int32_t)mi[r];
    }
  }
}

template <bool UNIQUE>
__device__ __forceinline__ void place_row_any(const uint32_t* bj, const uint32_t* bi, int cnt, int lane,
                                              int32_t* __restrict__ out_j, int32_t* __restrict__ out_img) {
  if (cnt <= 32) place_row<1, UNIQUE>(bj, bi, cnt, 0, lane, out_j, out_img);
  else
    for (int first = 0; first < cnt; first += 64) place_row<2, UNIQUE>(bj, bi, cnt, first, lane, out_j, out_img);
}

// What the candidate search reads.
struct SearchArgs {
  const double* x;
  const int4* meta;        // per atom: wrap counts, packed bin
  const int* bin_start;    // [bins + 1]
  const float4* bin_xw;    // per slot: FP32 wrapped position
  const int4* bin_meta;    // per slot: wrap counts, atom index
  int64_t n;
  int* status;
};

// Exact decision for the candidate at slot u with bin wraps q.
__device__ __noinline__ bool exact_inside(const SearchArgs& s, const NbrGeom& g, int4 mi, int u, int q0, int q1,
                                          int q2) {
  const int4 mj = __ldg(s.bin_meta + u);
  const int i = mi.w, j = mj.w;
  const int n1 = q0 + mi.x - mj.x, n2 = q1 + mi.y - mj.y, n3 = q2 + mi.z - mj.z;
  const double sx = __dadd_rn(__dadd_rn(__dmul_rn((double)n1, g.cell[0]), __dmul_rn((double)n2, g.cell[3])),
                              __dmul_rn((double)n3, g.cell[6]));
  const double sy = __dadd_rn(__dadd_rn(__dmul_rn((double)n1, g.cell[1]), __dmul_rn((double)n2, g.cell[4])),
                              __dmul_rn((double)n3, g.cell[7]));
  const double sz = __dadd_rn(__dadd_rn(__dmul_rn((double)n1, g.cell[2]), __dmul_rn((double)n2, g.cell[5])),
                              __dmul_rn((double)n3, g.cell[8]));
  const double dx = __dsub_rn(__dadd_rn(s.x[3 * (int64_t)j], sx), s.x[3 * (int64_t)i]);
  const double dy = __dsub_rn(__dadd_rn(s.x[3 * (int64_t)j + 1], sy), s.x[3 * (int64_t)i + 1]);
  const double dz = __dsub_rn(__dadd_rn(s.x[3 * (int64_t)j + 2], sz), s.x[3 * (int64_t)i + 2]);
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  return r2 < g.rc2 && r2 > 0.0;
}

// Visits the neighbours of the atom at a slot: hits(u0, mask, q0, q1, q2) for
// runs of up to 32 slots from u0 on, mask marking those inside the cutoff.
// The searched bins form rows along the last axis, and the bins of a row are
// consecutive slots between periodic wraps.  The loop over a run only tests
// distances in FP32 (wrapped positions plus the bin wrap) and sets bits, so
// the lanes of a warp, whose atoms are neighbours in bin order and read nearby
// slots, stay together; what FP32 cannot decide (a distance between rc2_lo and
// rc2_hi or near 0, bounds that exceed what its rounding can move it by) is
// decided by the exact FP64 expression afterwards.
// Of every run only the share sub of `shares` equal ones is visited.
template <class Hits>
__device__ __forceinline__ void search_atom(const SearchArgs& s, const NbrGeom& g, int4 mi, float4 pw, int sub,
                                            int shares, Hits&& hits) {
  const int bin = __ldg(s.meta + mi.w).w;
  const int b0 = bin & 1023, b1 = (bin >> 10) & 1023, b2 = bin >> 20;
  for (int t0 = b0 - g.reach[0]; t0 <= b0 + g.reach[0]; ++t0) {
    int q0 = 0, c0 = t0;
    if (g.pbc[0]) { q0 = wrap_count(t0, g.nb[0]); c0 = t0 - q0 * g.nb[0]; }
    else if (t0 < 0 || t0 >= g.nb[0]) continue;
    for (int t1 = b1 - g.reach[1]; t1 <= b1 + g.reach[1]; ++t1) {
      int q1 = 0, c1 = t1;
      if (g.pbc[1]) { q1 = wrap_count(t1, g.nb[1]); c1 = t1 - q1 * g.nb[1]; }
      else if (t1 < 0 || t1 >= g.nb[1]) continue;
      int t2 = b2 - g.reach[2], t2_hi = b2 + g.reach[2];
      if (!g.pbc[2]) {
        t2 = max(t2, 0);
        t2_hi = min(t2_hi, g.nb[2] - 1);
      }
      const int* row = s.bin_start + (c0 * g.nb[1] + c1) * g.nb[2];
      while (t2 <= t2_hi) {
        const int q2 = g.pbc[2] ? wrap_count(t2, g.nb[2]) : 0;
        const int c2 = t2 - q2 * g.nb[2];
        const int c2_end = min(g.nb[2] - 1, c2 + (t2_hi - t2));   // bins c2 .. c2_end share the wrap q2
        int u_beg = __ldg(row + c2), u_end = __ldg(row + c2_end + 1);
        if (shares > 1) {
          const int len = u_end - u_beg;
          u_end = u_beg + len * (sub + 1) / shares;
          u_beg += len * sub / shares;
        }
        t2 += c2_end - c2 + 1;
        const float fq0 = (float)q0, fq1 = (float)q1, fq2 = (float)q2;
        const float shx = fq0 * g.cellf[0] + fq1 * g.cellf[3] + fq2 * g.cellf[6] - pw.x;
        const float shy = fq0 * g.cellf[1] + fq1 * g.cellf[4] + fq2 * g.cellf[7] - pw.y;
        const float shz = fq0 * g.cellf[2] + fq1 * g.cellf[5] + fq2 * g.cellf[8] - pw.z;
        for (int u0 = u_beg; u0 < u_end; u0 += 32) {
          const int len = min(32, u_end - u0);
          unsigned in = 0u, maybe = 0u;
          // four candidates at a time: their loads are in flight together (past the end the last one again)
          for (int k = 0; k < len; k += 4) {
            float r2f[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 qw = __ldg(s.bin_xw + u0 + min(k + q, len - 1));
              const float fx = qw.x + shx, fy = qw.y + shy, fz = qw.z + shz;
              r2f[q] = fx * fx + fy * fy + fz * fz;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const unsigned bit = k + q < len ? 1u << (k + q) : 0u;
              if (!(r2f[q] >= g.rc2_hi)) maybe |= bit;
              if (r2f[q] < g.rc2_lo && r2f[q] > g.rz2) in |= bit;
            }
          }
          maybe &= ~in;
          while (maybe) {
            const int k = __ffs(maybe) - 1;
            maybe &= maybe - 1;
            if (exact_inside(s, g, mi, u0 + k, q0, q1, q2)) in |= 1u << k;
          }
          if (in) hits(u0, in, q0, q1, q2);
        }
      }
    }
  }
}

__device__ __forceinline__ bool image_overflows(int n1, int n2, int n3) {
  return n1 < -511 || n1 > 511 || n2 < -511 || n2 > 511 || n3 < -511 || n3 > 511;
}

// A found neighbour in one word: its slot and the bin wraps (each -1, 0 or 1).
constexpr int kSlotBits = 27;
__device__ __forceinline__ uint32_t pack_wraps(int q0, int q1, int q2) {
  return (uint32_t)((q0 + 1) + 3 * (q1 + 1) + 9 * (q2 + 1)) << kSlotBits;
}

// Neighbour counts; `lanes` threads (a power of two up to 4) per atom, in bin
// order, each visiting its share of every row's run of slots.  With `found` (the common
// case) every thread also leaves what it found in its column of
// found[entry][column], entries < depth, which order_kernel turns into list
// rows; a column that runs over sets status[1], and fill_kernel searches again
// instead.  A pair whose image leaves +-511 makes the call fail; it has a wrap
// count above 200 on one of its atoms or a bin wrap above 111, and every pair
// is visited from both sides, so only such atoms look at the images here.
__global__ void __launch_bounds__(kSearchThreads) count_kernel(const SearchArgs s, const NbrGeom g, int lanes,
                                                               uint32_t* __restrict__ found, int depth,
                                                               int* __restrict__ column_count,
                                                               int* __restrict__ counts) {
  const int64_t col = (int64_t)blockIdx.x * kSearchThreads + threadIdx.x;
  const int64_t cols = s.n * lanes;
  const bool active = col < cols;
  const int64_t slot = active ? col / lanes : 0;
  const int sub = (int)(threadIdx.x & (lanes - 1));
  const float4 pw = __ldg(s.bin_xw + slot);
  const int4 mi = __ldg(s.bin_meta + slot);
  const bool far = mi.x < -200 || mi.x > 200 || mi.y < -200 || mi.y > 200 || mi.z < -200 || mi.z > 200;
  int mine = 0;
  uint32_t* out = found + col;
  if (active) {
    search_atom(s, g, mi, pw, sub, lanes, [&](int u0, unsigned in, int q0, int q1, int q2) {
      if (far || abs(q0) > 111 || abs(q1) > 111 || abs(q2) > 111) {
        for (unsigned m = in; m; m &= m - 1) {
          const int4 mj = __ldg(s.bin_meta + u0 + __ffs(m) - 1);
          if (image_overflows(q0 + mi.x - mj.x, q1 + mi.y - mj.y, q2 + mi.z - mj.z))
            atomicCAS(s.status, 0, MTP_ERR_NEIGHBOR_OVERFLOW);
        }
      }
      if (found) {
        const uint32_t wraps = pack_wraps(q0, q1, q2);
        for (; in; in &= in - 1) {
          if (mine < depth) *out = (uint32_t)(__ffs(in) - 1 + u0) | wraps;
          out += cols;
          ++mine;
        }
      } else {
        mine += __popc(in);
      }
    });
    if (found) {
      column_count[col] = mine;
      if (mine > depth) s.status[1] = 1;
    }
  }
  for (int o = 1; o < lanes; o <<= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if (active && sub == 0) counts[mi.w] = mine;
}

// List rows from what count_kernel found: a block gathers the columns of its
// atoms and forms (j, image) of every entry, then one warp per atom orders the
// row and writes it; the blocks also write the offsets.  May run before the
// host knows the pair count or whether the build failed: does nothing if the
// pairs do not fit in `capacity`, a column ran over or an error is recorded, so
// that a list built in place keeps its offsets and rows until they are replaced
// together.
constexpr int kOrderWarps = 8;
constexpr int kOrderBuffer = 512;   // entries of one row
template <int LANES>
__global__ void __launch_bounds__(32 * kOrderWarps) order_kernel(const SearchArgs s, const NbrGeom g,
                                                                 const uint32_t* __restrict__ found,
                                                                 const int* __restrict__ column_count,
                                                                 const int64_t* __restrict__ offsets, int64_t capacity,
                                                                 int64_t* __restrict__ out_offsets,
                                                                 int32_t* __restrict__ out_j,
                                                                 int32_t* __restrict__ out_img) {
  __shared__ __align__(16) uint32_t buf[kOrderWarps][2][kOrderBuffer];
  __shared__ int start[kOrderWarps * LANES];   // by column of the block: its place in the row
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t total = __ldg(offsets + s.n);
  if (total > capacity || __ldg(s.status) != 0 || __ldg(s.status + 1) != 0) return;
  const int64_t slot0 = (int64_t)blockIdx.x * kOrderWarps, cols = s.n * LANES;
  const int atoms = (int)min((int64_t)kOrderWarps, s.n - slot0);
  // the block's share of the offsets, by atom index (one sector; by the atoms of its slots: eight)
  if ((int)threadIdx.x < atoms) out_offsets[slot0 + threadIdx.x] = __ldg(offsets + slot0 + threadIdx.x);
  if (blockIdx.x == 0 && threadIdx.x == 0) out_offsets[s.n] = total;
  constexpr int width = kOrderWarps * LANES;
  // the block's columns side by side: a sector of `found` holds the same entry of 8 columns
  const int c = threadIdx.x % width;
  const int a = c / LANES;
  const int64_t col = slot0 * LANES + c;
  const int cnt_c = a < atoms ? __ldg(column_count + col) : 0;
  if (threadIdx.x < width) {
    int pos = cnt_c;   // inclusive sum over the columns of the same atom
    for (int o = 1; o < LANES; o <<= 1) {
      const int v = __shfl_up_sync(__activemask(), pos, o, LANES);
      if ((c & (LANES - 1)) >= o) pos += v;
    }
    start[c] = pos;
  }
  __syncthreads();
  if (a < atoms) {
    const int4 mi = __ldg(s.bin_meta + slot0 + a);
    const int at = start[c] - cnt_c;
    for (int k = threadIdx.x / width; k < cnt_c; k += 32 * kOrderWarps / width) {
      const uint32_t f = __ldg(found + (int64_t)k * cols + col);
      const int4 mj = __ldg(s.bin_meta + (f & ((1u << kSlotBits) - 1u)));
      const int q = (int)(f >> kSlotBits);
      const int q2 = q / 9, q1 = (q - 9 * q2) / 3, q0 = q - 9 * q2 - 3 * q1;
      buf[a][0][at + k] = (uint32_t)mj.w;
      buf[a][1][at + k] = (uint32_t)pack_image(q0 - 1 + mi.x - mj.x, q1 - 1 + mi.y - mj.y, q2 - 1 + mi.z - mj.z);
    }
  }
  const int cnt = warp < atoms ? start[(warp + 1) * LANES - 1] : 0;   // this warp's row
  if (lane < ((4 - (cnt & 3)) & 3)) buf[warp][0][cnt + lane] = 0xFFFFFFFFu;
  __syncthreads();
  if (warp >= atoms) return;
  const int64_t base = __ldg(offsets + __ldg(s.bin_meta + slot0 + warp).w);
  if (g.unique) place_row_any<true>(buf[warp][0], buf[warp][1], cnt, lane, out_j + base, out_img + base);
  else place_row_any<false>(buf[warp][0], buf[warp][1], cnt, lane, out_j + base, out_img + base);
}

// List rows where the count left no usable columns: the search again, thread by thread into the
// warp's shared buffer (as many of the warp's atoms at a time as fit), then
// the warp orders one row after the other and writes it.
__global__ void __launch_bounds__(kSearchThreads) fill_kernel(const SearchArgs s, const NbrGeom g,
                                                              const int64_t* __restrict__ offsets, int64_t capacity,
                                                              int64_t* __restrict__ out_offsets,
                                                              int32_t* __restrict__ out_j,
                                                              int32_t* __restrict__ out_img) {
  __shared__ __align__(16) uint32_t buf[kSearchThreads / 32][2][kRowBuffer];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t slot = (int64_t)blockIdx.x * kSearchThreads + threadIdx.x;
  const int64_t total = __ldg(offsets + s.n);
  if (total > capacity) return;
  if (slot < s.n) out_offsets[slot] = __ldg(offsets + slot);
  if (slot == 0) out_offsets[s.n] = total;
  uint32_t* bj = buf[warp][0];
  uint32_t* bi = buf[warp][1];
  bool todo = slot < s.n;
  float4 pw = make_float4(0.f, 0.f, 0.f, 0.f);
  int4 mi = make_int4(0, 0, 0, 0);
  int cnt = 0;
  int64_t base = 0;
  if (todo) {
    pw = __ldg(s.bin_xw + slot);
    mi = __ldg(s.bin_meta + slot);
    base = __ldg(offsets + mi.w);
    const int64_t c64 = __ldg(offsets + mi.w + 1) - base;
    cnt = (int)c64;
    if (cnt > kRowBuffer) {
      // a row that does not fit: straight to the list, ordered by insertion (never at the densities here)
      int64_t at = base;
      search_atom(s, g, mi, pw, 0, 1, [&](int u0, unsigned in, int q0, int q1, int q2) {
        for (; in; in &= in - 1) {
          const int u = u0 + __ffs(in) - 1;
          const int4 mj = __ldg(s.bin_meta + u);
          const int32_t jj = mj.w;
          const int32_t im = pack_image(q0 + mi.x - mj.x, q1 + mi.y - mj.y, q2 + mi.z - mj.z);
          const unsigned long long kp = row_key(jj, im);
          int64_t q = at++;
          while (q > base && row_key(out_j[q - 1], out_img[q - 1]) > kp) {
            out_j[q] = out_j[q - 1];
            out_img[q] = out_img[q - 1];
            --q;
          }
          out_j[q] = jj;
          out_img[q] = im;
        }
      });
      todo = false;
    }
    if (cnt == 0) todo = false;
  }
  while (__any_sync(0xffffffffu, todo)) {
    // the first of the remaining atoms whose rows (rounded up to 4 entries) fit together
    const int mine = todo ? (cnt + 3) & ~3 : 0;
    int pos = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, pos, o);
      if (lane >= o) pos += v;
    }
    const bool now = todo && pos <= kRowBuffer;
    pos -= mine;
    if (now) {
      int at = pos;
      search_atom(s, g, mi, pw, 0, 1, [&](int u0, unsigned in, int q0, int q1, int q2) {
        for (; in; in &= in - 1) {
          const int u = u0 + __ffs(in) - 1;
          const int4 mj = __ldg(s.bin_meta + u);
          if (at < pos + cnt) {
            bj[at] = (uint32_t)mj.w;
            bi[at] = (uint32_t)pack_image(q0 + mi.x - mj.x, q1 + mi.y - mj.y, q2 + mi.z - mj.z);
          }
          ++at;
        }
      });
      for (int e = pos + cnt; e < pos + mine; ++e) bj[e] = 0xFFFFFFFFu;
      todo = false;
    }
    __syncwarp();
    for (unsigned rows = __ballot_sync(0xffffffffu, now); rows; rows &= rows - 1) {
      const int a = __ffs(rows) - 1;
      const int p = __shfl_sync(0xffffffffu, pos, a), c = __shfl_sync(0xffffffffu, cnt, a);
      const int64_t b = __shfl_sync(0xffffffffu, base, a);
      if (g.unique) place_row_any<true>(bj + p, bi + p, c, lane, out_j + b, out_img + b);
      else place_row_any<false>(bj + p, bi + p, c, lane, out_j + b, out_img + b);
    }
    __syncwarp();
  }
}

static void invert3(const double* m, double* inv) {
  const double a = m[0], b = m[1], c = m[2], d = m[3], e = m[4], f = m[5], gg = m[6], h = m[7], k = m[8];
  const double det = a * (e * k - f * h) - b * (d * k - f * gg) + c * (d * h - e * gg);
  inv[0] = (e * k - f * h) / det;
  inv[1] = (c * h - b * k) / det;
  inv[2] = (b * f - c * e) / det;
  inv[3] = (f * gg - d * k) / det;
  inv[4] = (a * k - c * gg) / det;
  inv[5] = (c * d - a * f) / det;
  inv[6] = (d * h - e * gg) / det;
  inv[7] = (b * gg - a * h) / det;
  inv[8] = (a * e - b * d) / det;
}

int build_neighbors(mtp_nlist* nl, const double* x, int64_t n, const double* cell, const int32_t* pbc, double r_cut,
                    cudaStream_t stream) {
  NbrGeom g;
  for (int k = 0; k < 9; ++k) g.cell[k] = cell[k];
  const double det = cell[0] * (cell[4] * cell[8] - cell[5] * cell[7]) - cell[1] * (cell[3] * cell[8] - cell[5] * cell[6]) +
                     cell[2] * (cell[3] * cell[7] - cell[4] * cell[6]);
  if (!(std::fabs(det) > 0.0) || !std::isfinite(det)) {
    set_error("mtp_build_neighbors: cell is singular or not finite (det = %g)", det);
    return MTP_ERR_ARG;
  }
  invert3(cell, g.hinv);
  double h[3];
  for (int k = 0; k < 3; ++k) {
    // s = x H^-1 (x a row vector): column k of H^-1 maps x to s_k
    const double c0 = g.hinv[0 + k], c1 = g.hinv[3 + k], c2 = g.hinv[6 + k];
    h[k] = 1.0 / std::sqrt(c0 * c0 + c1 * c1 + c2 * c2);
    g.pbc[k] = pbc[k] ? 1 : 0;
  }
  g.rc2 = r_cut * r_cut;
  for (int k = 0; k < 9; ++k) g.cellf[k] = (float)cell[k];

  const int T = 256;
  const unsigned blocks = (unsigned)((n + T - 1) / T);
  int rc;
  const int64_t n1 = std::max<int64_t>(n, 1);
  const bool periodic = g.pbc[0] && g.pbc[1] && g.pbc[2];
  // Memory the build needs; where it does not fit beside the columns of found
  // neighbours (this build's or an earlier one's), those go, and the rows are searched twice.
  uint32_t* found = nullptr;
  auto need = [&](DevBuf& buf, size_t bytes) {
    int e = MTP_OK;
    allocate_dropping([&]() { return (e = buf.ensure(bytes)) == MTP_OK; },
                      [&]() {
                        if (!nl->columns.ptr) return false;
                        nl->columns.release();
                        found = nullptr;
                        return true;
                      });
    return e;
  };
  if ((rc = need(nl->wrapped, (sizeof(float4) + sizeof(int4) + sizeof(double) * 3) * n1 + 64)) != MTP_OK) return rc;
  float4* xw = nl->wrapped.as<float4>();
  int4* meta = reinterpret_cast<int4*>(xw + n1);
  double* sw = reinterpret_cast<double*>(meta + n1);
  unsigned long long* extent = reinterpret_cast<unsigned long long*>(sw + 3 * n1);
  if ((rc = need(nl->bin_atoms, (sizeof(float4) + sizeof(int4) + sizeof(int)) * n1)) != MTP_OK) return rc;
  float4* bin_xw = nl->bin_atoms.as<float4>();
  int4* bin_meta = reinterpret_cast<int4*>(bin_xw + n1);
  int* rank = reinterpret_cast<int*>(bin_meta + n1);
  if ((rc = need(nl->status, sizeof(int) * 4)) != MTP_OK) return rc;
  int* status = nl->status.as<int>();
  MTP_TRY_CUDA(cudaMemsetAsync(status, 0, 2 * sizeof(int), stream));
  unsigned long long ext_bits[6];
  if (!periodic) {
    // the extent of the atoms along the open axes decides their bins
    const unsigned long long ext_init[6] = {~0ull, 0ull, ~0ull, 0ull, ~0ull, 0ull};
    MTP_TRY_CUDA(cudaMemcpyAsync(extent, ext_init, sizeof(ext_init), cudaMemcpyHostToDevice, stream));
    if (n > 0) wrap_kernel<false><<<blocks, T, 0, stream>>>(x, n, g, sw, meta, extent, xw, nullptr, nullptr, status);
    MTP_TRY_CUDA(cudaGetLastError());
    int wrap_status = 0;
    MTP_TRY_CUDA(cudaMemcpyAsync(ext_bits, extent, sizeof(ext_bits), cudaMemcpyDeviceToHost, stream));
    MTP_TRY_CUDA(cudaMemcpyAsync(&wrap_status, status, sizeof(int), cudaMemcpyDeviceToHost, stream));
    MTP_TRY_CUDA(cudaStreamSynchronize(stream));
    if (wrap_status == MTP_ERR_NONFINITE) {
      set_error("mtp_build_neighbors: non-finite position");
      return MTP_ERR_NONFINITE;
    }
  }
  int64_t nbins = 1;
  for (int k = 0; k < 3; ++k) {
    if (g.pbc[k]) {
      // bins of one cutoff along the first two axes (a search of 9 rows) and of
      // a quarter along the last, where a row's bins are one run of slots: 9 x
      // 2.25 R_cut^3 searched, in runs of about 20 atoms.  Bins of half a cutoff
      // along every axis search less (15.6 R_cut^3) but in 25 runs of about 5
      // atoms, whose set-up and uneven lengths cost more than the candidates.
      g.nb[k] = std::max(1, (int)std::floor((k == 2 ? 4.0 : 1.0) * h[k] / r_cut));
      g.nb[k] = (int)std::min<int64_t>(g.nb[k], 1024);
      g.origin[k] = 0.0;
      g.width[k] = 1.0 / g.nb[k];
    } else {
      double lo = 0.0, hi = 0.0;
      if (n > 0) {
        lo = unordered_bits(ext_bits[2 * k]);
        hi = unordered_bits(ext_bits[2 * k + 1]);
      }
      const double w = r_cut / h[k];   // fractional width of one cutoff
      g.origin[k] = lo;
      g.width[k] = w;
      int64_t nbk = (int64_t)std::floor((hi - lo) / w) + 1;
      g.nb[k] = (int)std::max<int64_t>(1, std::min<int64_t>(nbk, 1024));
      if (nbk > 1024) g.width[k] = (hi - lo) / 1023.999;
    }
    g.reach[k] = (int)std::floor(r_cut * g.nb[k] / h[k] * (1.0 + 1e-9) * (g.pbc[k] ? 1.0 : 0.0)) + 1;
    if (!g.pbc[k]) g.reach[k] = std::max(1, (int)std::ceil(r_cut / (g.width[k] * h[k])));
    g.inv_width[k] = 1.0 / g.width[k];
    nbins *= g.nb[k];
  }
  // two images of one atom are at least the smallest plane spacing of a
  // periodic axis apart, and both lie within R_cut of the centre
  g.unique = true;
  for (int k = 0; k < 3; ++k)
    if (g.pbc[k] && h[k] <= 2.0 * r_cut * (1.0 + 1e-9)) g.unique = false;
  {
    // FP32 prefilter margin.  With u = 2^-24, a component of the pair vector is
    // (xw_j + (shift - xw_i)): xw carries u P (P bounds the wrapped positions'
    // component, the sum over k of |H_k| times the wrapped fractional range),
    // the shift at most 5 u S (three products of rounded cell entries with the
    // bin wraps, two sums; S is the sum over k of |H_k| max |q_k|), the
    // difference u (S + P) more and the sum u (2 R_cut) for a pair that can
    // matter: u (3 P + 6 S + 2 R_cut) together.  err is that vector's norm, half
    // more, and the rounding of r^2 itself is covered by the factors 1 +- 1e-6.
    double err2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      double P = 0.0, S = 0.0;
      for (int k = 0; k < 3; ++k) {
        double span = 1.0;
        if (!g.pbc[k] && n > 0)
          span = std::max(std::fabs(unordered_bits(ext_bits[2 * k])), std::fabs(unordered_bits(ext_bits[2 * k + 1])));
        const double qmax = g.pbc[k] ? (double)((g.reach[k] + g.nb[k] - 1) / g.nb[k]) : 0.0;
        P += std::fabs(cell[3 * k + c]) * span;
        S += std::fabs(cell[3 * k + c]) * qmax;
      }
      const double e = 3.0 * P + 6.0 * S + 2.0 * r_cut;
      err2 += e * e;
    }
    const double err = 1.5 * std::ldexp(1.0, -24) * std::sqrt(err2);
    g.rc2_hi = (float)((r_cut + err) * (r_cut + err) * (1.0 + 1e-6));
    // the same bound the other way: an FP32 distance below R_cut - err (and
    // above 2 err) puts the exact one inside (0, R_cut), so the FP64 test is
    // needed only in the two shells around 0 and R_cut
    const double lo = r_cut - err;
    g.rc2_lo = lo > 0.0 ? (float)(lo * lo * (1.0 - 1e-6)) : 0.0f;
    g.rz2 = (float)(4.0 * err * err * (1.0 + 1e-6)) + 1e-30f;
  }
  if ((rc = need(nl->bins, sizeof(int) * (nbins + 1))) != MTP_OK) return rc;
  int* bin_count = nl->bins.as<int>();
  if ((rc = need(nl->bin_start, sizeof(int) * (nbins + 1))) != MTP_OK) return rc;
  int* bin_start = nl->bin_start.as<int>();
  MTP_TRY_CUDA(cudaMemsetAsync(bin_count, 0, sizeof(int) * (nbins + 1), stream));
  if (n > 0) {
    if (periodic)
      wrap_kernel<true><<<blocks, T, 0, stream>>>(x, n, g, nullptr, meta, nullptr, xw, rank, bin_count, status);
    else
      bin_count_kernel<<<blocks, T, 0, stream>>>(sw, n, g, meta, rank, bin_count);
  }
  MTP_TRY_CUDA(cudaGetLastError());
  // the scans run over one entry more: bin_start[nbins] and offsets[n] are the totals
  size_t tmp_bytes = 0;
  MTP_TRY_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tmp_bytes, bin_count, bin_start, (int)(nbins + 1), stream));
  size_t tmp2 = 0;
  MTP_TRY_CUDA(cub::DeviceScan::ExclusiveScan(nullptr, tmp2, (int*)nullptr, (int64_t*)nullptr, ::cuda::std::plus<>{},
                                              (int64_t)0, (int)(n + 1), stream));
  tmp_bytes = std::max(tmp_bytes, tmp2);
  // counts, the new offsets, the scans' temporary storage
  const size_t counts_bytes = sizeof(int) * (size_t)((n + 4) & ~int64_t(3)), offsets_bytes = sizeof(int64_t) * (n + 1);
  if ((rc = need(nl->counts, counts_bytes + ((offsets_bytes + 15) & ~size_t(15)) + tmp_bytes + 64)) != MTP_OK)
    return rc;
  int* counts = nl->counts.as<int>();
  int64_t* offsets = reinterpret_cast<int64_t*>(reinterpret_cast<char*>(counts) + counts_bytes);
  void* tmp = reinterpret_cast<char*>(offsets) + ((offsets_bytes + 15) & ~size_t(15));
  MTP_TRY_CUDA(cub::DeviceScan::ExclusiveSum(tmp, tmp_bytes, bin_count, bin_start, (int)(nbins + 1), stream));
  MTP_TRY_CUDA(cudaMemsetAsync(counts + n, 0, sizeof(int), stream));
  const unsigned search_blocks = (unsigned)((n + kSearchThreads - 1) / kSearchThreads);
  // Columns of found neighbours.  Threads per atom: more for small systems,
  // whose search is a chain of dependent loads on too few threads.  Entries per
  // column: half more than the mean density gives, and some.
  // BCC at R_cut 5 A, build in place with 1 / 2 / 4 threads (us): 2,000 atoms
  // 129 / 115 / 111, 16,000 145 / 133 / 121, 31,250 153 / 141 / 139, 50,460
  // 171 / 158 / 162, 98,568 200 / 200 / 215, 203,136 282 / 292 / 337; hence 4 up to
  // 50,000 atoms and 2 up to 100,000 (some 1,300 threads per SM).
  int lanes = 1;
  while (lanes < 4 && 2 * n * lanes <= 200000) lanes *= 2;
  const double mean = (double)n / std::fabs(det) * 4.1887902047863905 * r_cut * r_cut * r_cut;
  int depth = (int)std::min(1.5 * mean / lanes + 16.0, (double)kOrderBuffer);
  bool columns = n < (int64_t(1) << kSlotBits) && depth * lanes <= kOrderBuffer;
  for (int k = 0; k < 3; ++k)
    if (g.pbc[k] && g.reach[k] > g.nb[k]) columns = false;   // a bin wrap beyond +-1
  int* column_count = nullptr;
  // without room for them the rows are searched twice
  if (n > 0 && columns && nl->columns.try_ensure(sizeof(int) * (size_t)n * lanes * (depth + 1))) {
    column_count = nl->columns.as<int>();
    found = reinterpret_cast<uint32_t*>(column_count + n * lanes);
  }
  const SearchArgs sa{x, meta, bin_start, bin_xw, bin_meta, n, status};
  if (n > 0) {
    bin_fill_kernel<<<blocks, T, 0, stream>>>(meta, n, g, bin_start, rank, xw, bin_xw, bin_meta);
    count_kernel<<<(unsigned)((n * lanes + kSearchThreads - 1) / kSearchThreads), kSearchThreads, 0, stream>>>(
        sa, g, lanes, found, depth, column_count, counts);
  }
  MTP_TRY_CUDA(cudaGetLastError());
  MTP_TRY_CUDA(cub::DeviceScan::ExclusiveScan(tmp, tmp_bytes, counts, offsets, ::cuda::std::plus<>{}, (int64_t)0,
                                              (int)(n + 1), stream));
  // a list that is rebuilt usually has room for the new rows: its fill is
  // queued before the host has the pair count, and does nothing if it has not
  auto list_room = [&]() { return (int64_t)(std::min(nl->nbr_j.bytes, nl->nbr_img.bytes) / sizeof(int32_t)); };
  auto order = [&]() {
    auto kern = lanes == 1 ? order_kernel<1> : lanes == 2 ? order_kernel<2> : order_kernel<4>;
    kern<<<(unsigned)((n + kOrderWarps - 1) / kOrderWarps), 32 * kOrderWarps, 0, stream>>>(
        sa, g, found, column_count, offsets, list_room(), nl->offsets.as<int64_t>(), nl->nbr_j.as<int32_t>(),
        nl->nbr_img.as<int32_t>());
  };
  int64_t total = 0;
  int st[2] = {0, 0};
  MTP_TRY_CUDA(cudaMemcpyAsync(&total, offsets + n, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  MTP_TRY_CUDA(cudaMemcpyAsync(st, status, sizeof(st), cudaMemcpyDeviceToHost, stream));
  const int64_t room = found && nl->offsets.bytes >= offsets_bytes ? list_room() : 0;
  if (room > 0) order();
  MTP_TRY_CUDA(cudaGetLastError());
  MTP_TRY_CUDA(cudaStreamSynchronize(stream));
  if (st[0] == MTP_ERR_NONFINITE) {
    set_error("mtp_build_neighbors: non-finite position");
    return MTP_ERR_NONFINITE;
  }
  if (st[0] != 0) {
    set_error("mtp_build_neighbors: a neighbour image exceeds +-511 cells (cell too thin for the cutoff)");
    return MTP_ERR_NEIGHBOR_OVERFLOW;
  }
  // the build succeeded: from here on the list is the new one.  An allocation
  // that fails leaves an empty list (its arrays are gone)
  nl->n_atoms = 0;
  nl->n_pairs = 0;
  const size_t row_bytes = sizeof(int32_t) * std::max<int64_t>(total, 1);
  if ((rc = need(nl->offsets, offsets_bytes)) != MTP_OK || (rc = need(nl->nbr_j, row_bytes)) != MTP_OK ||
      (rc = need(nl->nbr_img, row_bytes)) != MTP_OK)
    return rc;
  if (total == 0) {
    MTP_TRY_CUDA(cudaMemcpyAsync(nl->offsets.ptr, offsets, offsets_bytes, cudaMemcpyDeviceToDevice, stream));
  } else if (!found || st[1]) {
    fill_kernel<<<search_blocks, kSearchThreads, 0, stream>>>(sa, g, offsets, list_room(), nl->offsets.as<int64_t>(),
                                                              nl->nbr_j.as<int32_t>(), nl->nbr_img.as<int32_t>());
  } else if (total > room) {
    order();
  }
  MTP_TRY_CUDA(cudaGetLastError());
  if (nl->columns.bytes > kColumnsKept) nl->columns.release();   // waits for order_kernel
  for (int k = 0; k < 9; ++k) nl->cell[k] = cell[k];
  for (int k = 0; k < 3; ++k) nl->pbc[k] = g.pbc[k];
  nl->r_cut = r_cut;
  nl->n_atoms = n;
  nl->n_pairs = total;
  return MTP_OK;
}

}  // namespace mtp
