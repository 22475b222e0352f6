// Internal definitions of the GB300 MTP library (not part of the C-ABI).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "mtp.h"

namespace mtp {

void set_error(const char* fmt, ...);

#define MTP_TRY_CUDA(call)                                                                      \
  do {                                                                                          \
    cudaError_t e_ = (call);                                                                    \
    if (e_ != cudaSuccess) {                                                                    \
      mtp::set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return e_ == cudaErrorMemoryAllocation ? MTP_ERR_OOM : MTP_ERR_CUDA;                      \
    }                                                                                           \
  } while (0)

// Device buffer that only grows.  Memory that a stream capture has recorded is
// not freed when the buffer grows (the graph may be replayed at any later
// time), only by release().
struct DevBuf {
  void* ptr = nullptr;
  size_t bytes = 0;
  bool in_graph = false;       // a capture has recorded ptr
  std::vector<void*> kept;     // outgrown memory that captures have recorded
  int ensure(size_t want);
  bool try_ensure(size_t want);   // for scratch that a call can do without
  void release();
  template <class T> T* as() const { return static_cast<T*>(ptr); }
};

constexpr int kMaxSpecies = 16;
constexpr int kMaxQ = 16;
constexpr int kImageBias = 512;  // image components are stored as n + 512 in 10 bits each

__host__ __device__ inline int32_t pack_image(int n1, int n2, int n3) {
  return (int32_t)(((uint32_t)(n1 + kImageBias)) | ((uint32_t)(n2 + kImageBias) << 10) |
                   ((uint32_t)(n3 + kImageBias) << 20));
}
__host__ __device__ inline void unpack_image(int32_t p, int& n1, int& n2, int& n3) {
  uint32_t u = (uint32_t)p;
  n1 = (int)(u & 1023u) - kImageBias;
  n2 = (int)((u >> 10) & 1023u) - kImageBias;
  n3 = (int)((u >> 20) & 1023u) - kImageBias;
}

// Species index of atom i as the kernels use it: a value outside 0..S-1
// (reported through the status word by the entry point's checks) is read as
// species 0, so that no table lookup leaves its array.
__device__ __forceinline__ int species_at(const int32_t* z, int64_t i, int S) {
  const int v = __ldg(z + i);
  return (unsigned)v < (unsigned)S ? v : 0;
}

// Everything an energy/force launch needs, passed by value.
struct EfvArgs {
  int64_t atom_begin, atom_end, n_atoms;
  const int64_t* offsets;
  const int64_t* row_counts;   // nullptr: row i is offsets[i] .. offsets[i + 1]; else offsets[i] .. + row_counts[i]
  const int32_t* nbr_j;
  const int32_t* nbr_img;
  const double* x;          // FP64 path
  const long long* xq;      // mixed path: 32.32 fixed-point fractional coordinates [N][3]
  const int32_t* z;
  double cell[9];
  float cellf[9];
  int n_species, n_q, n_mu, m;
  double r_min, r_cut;
  const double* species_energy;
  const double* radial_d;   // [n_mu][n_q][S][S]
  const double* xi_d;
  const float* radial_f;
  const float* xi_f;
  double* e_atom;
  double* forces;
  float* forces_f;          // mixed path: FP32 force accumulator [N][3], converted at the end
  double* virial;
  double* e_total;
  double* dtheta;           // nullable
  int* status;
  void* mbuf;               // levels with component groups: scratch of the split kernels in the working precision,
                            // n_parts buffers of partial moments, then the adjoints (nullptr: one fused kernel)
  int n_parts;              // shares into which the split kernels cut each atom's neighbours
  int graphs;               // mbuf has room for the graph values (straight-line contraction)
  const int32_t* order;     // kernels with one thread per atom: thread t of the range takes atom order[t] (nullptr: t)
};

// Atom of thread t of the range.
__device__ __forceinline__ int64_t thread_atom(const EfvArgs& a, int64_t t) {
  return a.atom_begin + (a.order ? (int64_t)__ldg(a.order + t) : t);
}
// List row of atom i.
__device__ __forceinline__ void list_row(const EfvArgs& a, int64_t i, int64_t& beg, int64_t& end) {
  beg = __ldg(a.offsets + i);
  end = a.row_counts ? beg + __ldg(a.row_counts + i) : __ldg(a.offsets + i + 1);
}

// Everything an evaluation needs before its own kernels, in one launch (a
// call on a few hundred atoms is bound by launches: separate clears of the
// energy, virial, gradient and force arrays cost more than its kernels):
// the outputs that the kernels add to are cleared and every species index is
// checked; MIXED: x (FP64) -> 32.32 fixed-point fractional coordinates
// s = x H^-1 (not wrapped: the pair difference plus the image is then exact),
// species in slot 3.
struct PrepArgs {
  const double* x;
  const int32_t* z;
  int64_t n, n_params;
  double h[9];          // H^-1, MIXED: times 2^32 (exact)
  int n_species;
  long long* xq;        // MIXED
  float* forces_f;      // MIXED, nullable
  double* forces;       // FP64 path, nullable
  double* virial;       // [6], nullable
  double* e_total;      // nullable
  double* dtheta;       // [n_params], nullable
  int* status;
};
int launch_prep(const PrepArgs& a, bool mixed, cudaStream_t s);
// order[t], t < atom_end - atom_begin: the range's atoms (relative to
// atom_begin), every 1,024 consecutive ones sorted by the length of their rows.
int launch_row_order(const EfvArgs& a, int32_t* order, cudaStream_t s);
// Whether work queued on s goes into a graph (or cannot be queued at all).
bool is_capturing(cudaStream_t s);
// H^-1 of the cell rows, times `scale`.
void inverse_rows(const double* cell, double scale, double* hi);

// Shares of each atom's neighbours in the split sweeps (levels with component
// groups) of n atoms.  One thread per atom, component group and share: at 255
// registers two 128-thread blocks are resident per SM, and a small system
// leaves most of them empty, so its neighbours are cut into shares until one
// wave is full (level 20, 4,000 atoms, FP64: one share left 32 blocks for 152
// SMs).  The contraction adds the shares' moments when it loads them.
constexpr int kSplitMaxParts = 16;
// SMs of the current device.
inline int device_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
    return 1;
  return n;
}
inline int split_parts(int64_t n, int sms) {
  const int64_t blocks = 2 * ((n + 127) / 128);
  int parts = 1;
  while (parts < kSplitMaxParts && 2 * parts * blocks <= 2 * (int64_t)sms) parts *= 2;
  return parts;
}
// Row length of the graph values G[graph][atom]: whole blocks of 128 threads.
__host__ __device__ inline int64_t graph_padded(int64_t n) { return (n + 127) / 128 * 128; }
// From this many atoms of a range on, the mixed path of the levels with
// component groups contracts with the straight-line graph kernels (times on both
// sides stand there).
constexpr int64_t kGraphAtoms = 4096;
// The straight-line contraction of level LEVEL (generated).
template <int LEVEL> int graphs_launch(const EfvArgs& a, bool want_dtheta, cudaStream_t s);

using EfvLaunch = int (*)(const EfvArgs&, int precision, bool want_dtheta, cudaStream_t);
// FP64 basis rows of listed atoms (list == nullptr: atoms atom_begin..), optional FP64 column sums.
using RowsLaunch = int (*)(const EfvArgs&, const int32_t* list, int64_t n_rows, double* rows, int64_t ld,
                           double* bsum, cudaStream_t);

struct BatchArgs;
using BatchLaunch = int (*)(const BatchArgs&, int precision, bool want_dtheta, int threads, cudaStream_t);
struct TangentArgs;
using TangentLaunch = int (*)(const TangentArgs&, int precision, cudaStream_t);

struct LevelEntry {
  int level;
  EfvLaunch efv;
  RowsLaunch rows;
  BatchLaunch batch;
  TangentLaunch tangent;
  int split_comps;   // components per atom of the EfvArgs::mbuf scratch (0: the level needs none)
  int split_graphs;  // graphs per atom of that scratch (0: the level needs none)
  EfvLaunch team;    // kernel whose warps share atoms (levels with component groups: the split kernels)
};

const LevelEntry* find_level(int level);

// Tensor-core grade (grade_tc.cu).
constexpr int kTcSlices = 7;      // BF16 slices per operand
constexpr int kTcMaxBasis = 128;  // padded basis size of the tensor-core product
size_t tc_x_bytes(int64_t n_rows);
size_t tc_y_bytes();
int tc_prepare(const double* rows, int64_t n, int m, const double* a_inv, const double* amax,
               unsigned long long* colmax, uint16_t* ys, int* fexp, int* dexp, int* fmax, uint16_t* xs, int* erow,
               int* status, cudaStream_t s);
int tc_gemm(const uint16_t* xs, const uint16_t* ys, const int* fexp, const int* erow, int64_t n,
            unsigned long long* gbits, int* status, float* dbg, cudaStream_t s);
int tc_finalize(const unsigned long long* gbits, int64_t n, const int* erow, const int* fmax, double tau_sel,
                double tau_brk, double* gamma, uint8_t* flags, unsigned long long* gmax_bits, int32_t* list,
                unsigned* list_n, cudaStream_t s);

}  // namespace mtp

struct mtp_handle {
  int device = 0;
  int level = 0, n_species = 0, n_q = 0, n_mu = 0, m = 0, n_comp = 0;
  double r_min = 0, r_cut = 0;
  int64_t n_params = 0;
  const mtp::LevelEntry* ops = nullptr;
  std::vector<double> h_species, h_radial, h_xi;
  mtp::DevBuf species, radial_d, xi_d, radial_f, xi_f, status;
  mtp::DevBuf xq;        // fixed-point positions scratch
  mtp::DevBuf forces_f;  // FP32 force accumulator (mixed path)
  mtp::DevBuf grade;     // grade scratch: counters, row maxima, column sums, FP64 basis rows
  mtp::DevBuf mbuf;      // moment/adjoint scratch of the split kernels (levels with component groups)
  mtp::DevBuf order;     // atoms by row length (launch_row_order)
  int efv_variant = 0;   // 0: tuned or by size, 1: thread per atom, 2: warps share atoms
  int8_t tuned[2][64] = {};   // [precision][floor(log2 N)]: 0 untuned, else the faster variant
};

struct mtp_nlist {
  int device = 0;
  int64_t n_atoms = 0, n_pairs = 0;
  double r_cut = 0;
  double cell[9] = {0};
  int pbc[3] = {0, 0, 0};
  mtp::DevBuf offsets, nbr_j, nbr_img;
  const int64_t* row_counts = nullptr;   // entries of row i from offsets[i] on (nullptr: up to offsets[i + 1])
  mtp::DevBuf counts, bins, bin_start, bin_atoms, wrapped, columns, status;
};

namespace mtp {
// mtp_compute_efv with the device word that takes its error status.
int compute_efv(mtp_handle* h, const mtp_nlist* nl, const double* x, const int32_t* z, int64_t n, const double* cell,
                int32_t precision, int64_t chunk_atoms, double* e_atom, double* forces, double* virial,
                double* e_total, double* dtheta, int* status, cudaStream_t s);
}  // namespace mtp
