// pg_host.h -- host-side objects behind the C ABI and the kernel launchers.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <map>
#include <string>
#include <vector>

#include "../../include/parcels_gb.h"
#include "pg_device.cuh"

namespace pg {

void set_error(const char *fmt, ...);
void clear_error();

// Every device allocation of the library goes through these two, so the
// accounting (and failure injection in tests) has one place.
cudaError_t dev_alloc(void **p, size_t bytes);
void dev_free(void *p);

// Count of kernel launches made by the library (all threads, all devices).
void note_launches(int n);

struct Slot {
  void *buf = nullptr;        // interleaved slab in storage format
  float *scales = nullptr;    // [nf] FP32 scales of this slot
  int s = -1;                 // snapshot held (-1: none)
  cudaEvent_t ready = nullptr;   // upload finished (recorded on the side stream)
  cudaEvent_t free = nullptr;    // last use finished (recorded on the compute stream)
};

// Device arrays of one particle set (positions in one of the two forms), in
// one allocation: a set is made and freed with two calls of the allocator
// instead of fifteen (with one kernel for the start state, a batch of 24 sets
// 15.7 -> 10.8 ms).
struct PsetArrays {
  void *base = nullptr;       // the allocation
  void *x = nullptr, *y = nullptr, *z = nullptr;
  int32_t *ci = nullptr, *cj = nullptr, *ck = nullptr;
  float *fx = nullptr, *fy = nullptr, *fz = nullptr;
  double *time = nullptr;
  uint64_t *id = nullptr;
  uint32_t *step = nullptr;
  uint8_t *status = nullptr;
  double *age = nullptr;      // [cap]
  double *var = nullptr;      // [nvar][cap] sampled variables
  double *hstep = nullptr;    // [cap] RKF45 step lengths
  void free_all() {
    dev_free(base);
    *this = PsetArrays();
  }
};

// Allocate the arrays of `cap` particles with `nvar` sampled variables.  Ages and
// step lengths start as zeros from entry `first` on -- the entries that the
// caller does not write at once -- because a re-sort leaves arrays that no kernel
// has used where they are, and swaps the two sets: every entry of either has to
// hold the zero of a new particle by then.
pg_status alloc_arrays(PsetArrays &A, int pos, int64_t cap, int nvar, int64_t first = 0);

// Arrays of one output slot (device or pinned host), cap rows each.
struct OutputView {
  uint64_t *id = nullptr;
  double *lon = nullptr, *lat = nullptr, *depth = nullptr, *age = nullptr;
  double *vars = nullptr;       // [nvar][cap]
  uint8_t *status = nullptr;
  uint32_t *count = nullptr;    // rows written
};

struct OutputSlot {
  void *d = nullptr;            // device slot
  void *h = nullptr;            // pinned host copy
  cudaEvent_t packed = nullptr, copied = nullptr;
  double time = 0.0;
  bool pending = false;
};

// Two-slot pinned output ring of a particle set (output.cu).
struct OutputRing {
  int64_t cap = 0;
  int nvar = 0;
  OutputSlot slot[2];
  uint32_t *d_tiles = nullptr;  // tile counts and offsets of the compaction
  cudaStream_t cs = nullptr;    // the copy stream
  int next = 0;                 // slot of the next output
  ~OutputRing();
  void release();
  cudaError_t prepare(int64_t need_cap, int need_nvar);
  // pack the output at time t into slot `next` on `st` and copy it to the
  // host on the copy stream; indexed: rows of alive particles and of those
  // deleted at or after t_prev (direction sgn)
  cudaError_t enqueue(const pg_pset *ps, double t, double t_prev, double sgn, int indexed,
                      cudaStream_t st);
  // wait for slot k's copy; host views of its arrays and its time
  cudaError_t wait(int k, OutputView &hv, double &t);
  static OutputView view(const void *base, int64_t rows_cap, int nv);
};

}  // namespace pg

struct pg_fieldset {
  int device = 0;
  // constants carried by the field set (Sect. 3), read by the behaviours
  std::map<std::string, double> constants;
  int interp = 0;               // velocities: 0 linear, 1 nearest
  // scalar fields (tracers) sampled into particle variables, resident only
  int ntr = 0;
  std::string tr_name[2];
  int tr_interp[2] = {0, 0};
  std::vector<void *> tr_slabs; // [2 * nt] planar slabs (null until loaded)
  const void **d_ttab = nullptr;// device copy of tr_slabs
  int sm_count = 0;
  int nx = 0, ny = 0, nz = 0, mesh = 0, periodic = 0, nfields = 0, storage = 0;
  std::vector<double> lon, lat, depth;
  double *d_axes64 = nullptr;   // lon | lat | depth
  float *d_axes32 = nullptr;
  int uni[3] = {0, 0, 0};
  double x0[3] = {0, 0, 0}, inv_d[3] = {0, 0, 0};
  // time axis
  int nt = 0;
  std::vector<double> times;
  double period = 0.0;
  double *d_times = nullptr;
  // storage
  size_t nodes = 0;             // nx * ny * nz
  size_t slab_bytes = 0;        // interleaved slab in storage format
  std::vector<void *> slabs;    // resident snapshots (null until loaded)
  std::vector<float> h_scales;  // [nt * nf]
  const void **d_tab = nullptr; // device table [nt]
  float *d_scales = nullptr;    // device [nt * nf]
  unsigned *d_amax = nullptr;   // scratch of the quantiser
  void *d_stage = nullptr;      // planar staging buffer (host-sourced uploads)
  size_t stage_bytes = 0;
  // streaming
  bool streaming = false;
  std::vector<const void *> src_ptrs;
  pg_snapshot_cb cb = nullptr;
  void *cb_user = nullptr;
  int src_dtype = PG_F32;
  std::vector<pg::Slot> slot = std::vector<pg::Slot>(4);   // the ring (>= 4 slots)
  void *h_pinned = nullptr;     // pinned staging for callback sources
  cudaStream_t side = nullptr;
  cudaEvent_t stage_free = nullptr;
  int64_t uploads = 0;          // streamed snapshot uploads
  int64_t upload_h2d_bytes = 0; // of which host-to-device bytes
};

struct pg_kernel {
  int scheme = PG_RK4;
  unsigned beh = 0;
  double kh = 0.0, w_sink = 0.0;   // NaN: the field set's constant of that name
};

struct pg_pset {
  pg_fieldset *fs = nullptr;
  int pos = PG_POS_F32;
  uint64_t seed = 0;
  int64_t n = 0, cap = 0;
  void *base = nullptr;                                 // the arrays' allocation
  void *x = nullptr, *y = nullptr, *z = nullptr;       // positions (plain forms)
  int32_t *ci = nullptr, *cj = nullptr, *ck = nullptr;  // cell form
  float *fx = nullptr, *fy = nullptr, *fz = nullptr;
  double *time = nullptr;
  uint64_t *id = nullptr;
  uint32_t *step = nullptr;
  uint8_t *status = nullptr;
  double *age = nullptr;               // [cap] age in seconds (age behaviour)
  double *var = nullptr;               // [nvar][cap] sampled variables
  double *hstep = nullptr;             // [cap] RKF45 step lengths (0: start from dt)
  int nvar = 0;                        // the field set's scalar fields at creation
  // whether ages and RKF45 step lengths can be other than the zeros that all
  // entries of both sets of arrays start with (alloc_arrays, new particles);
  // until then a re-sort leaves them
  bool age_used = false, hstep_used = false;
  double t_min = 0.0, t_max = 0.0;     // range of particle times
  pg_tune tune{256, 0, 0};             // chunk_steps 0: chosen per execute
  unsigned long long *d_counter = nullptr;
  int *d_err = nullptr;
  // re-sort: second set of arrays (same capacity) and scratch, on first use
  pg::PsetArrays alt;
  int64_t alt_cap = 0;
  void *sort_scratch = nullptr;
  size_t sort_scratch_bytes = 0;
  double *diag_scratch = nullptr;
  // trajectory output ring, on first use
  pg::OutputRing *out = nullptr;
  // optional CUDA-event timing of the advection launches
  bool timing = false;
  std::vector<cudaEvent_t> ev;        // pairs (start, stop) per launch
  size_t ev_used = 0;
  double timed_ms = 0.0;
  int64_t timed_launches = 0;
};

namespace pg {

cudaError_t launch_repack(const void *src, int src_dtype, int nf, size_t nodes, void *dst,
                          int storage, float *scales_out, unsigned *amax_scratch, int sm_count,
                          cudaStream_t st);

// Advection chunk for lon/lat/depth positions.  real: PG_POS_F64 / PG_POS_F32.
cudaError_t launch_advect_plain(const StepArgs &a, int real, int storage, int block,
                                cudaStream_t st);

// Advection chunk for cell-index + offset positions.
cudaError_t launch_advect_cell(const StepArgs &a, int storage, int block, cudaStream_t st);
cudaError_t launch_to_cell(const GridArgs &g, const double *lon, const double *lat,
                           const double *dep, int32_t *ci, int32_t *cj, int32_t *ck, float *fx,
                           float *fy, float *fz, int64_t n, int sm, cudaStream_t st);
cudaError_t launch_from_cell(const GridArgs &g, const int32_t *ci, const int32_t *cj,
                             const int32_t *ck, const float *fx, const float *fy, const float *fz,
                             double *lon, double *lat, double *dep, int64_t n, int sm,
                             cudaStream_t st);

// Grid argument block of a field set (defined in capi.cu).
GridArgs grid_args_of(const pg_fieldset *fs);

// One network step of the learned flow map: the particles' features packed
// as the tcgen05 inference kernel's input tiles, the network, the displacement
// applied to the particles in its last epilogue (surrogate_features.cuh).
struct SurrogateStepIO {
  GridArgs g;
  FieldArgs f;
  float *lon, *lat, *dep;
  double *time;
  uint32_t *step;
  uint8_t *status;
  int64_t n;
  double horizon;
  int *ferr;                  // device word: feature error (time range, missing slab)
};
// A layer's weight and bias gradient (gemm_tn_splitk_tc, mlp_tc.cu).
struct WeightGrad {
  const __nv_bfloat16 *A, *B;   // [batch x Mrows], [batch x N]
  int64_t lda, ldb;
  int Mrows, N;
  float *out;                   // [Mrows x N]
  const float *bpart;           // [nparts x Mrows]
  int nparts;
  float *bout;                  // [Mrows]
};
// Whether the network's engine and shape allow the fused step.
bool mlp_fused_step_ok(const pg_mlp *net);
// Bytes of the packed features of a step on n particles.
size_t mlp_fused_step_scratch(int64_t n);
// The fused step (weights packed first if needed) with the features in xpk;
// reads back the network's and the features' error words.
pg_status mlp_fused_step(pg_mlp *net, const SurrogateStepIO &io, uint8_t *xpk, cudaStream_t st);

// Kernel argument block of a kernel on a field set: NaN parameters and those
// of the settle and age behaviours from the field set's constants (capi.cu).
pg_status resolve_kernel(const pg_kernel *k, const pg_fieldset *fs, uint64_t seed, KernArgs &a);

// The device arrays of a particle set, and replacing them (capi.cu).
PsetArrays pset_arrays(const pg_pset *ps);
void pset_set_arrays(pg_pset *ps, const PsetArrays &A);

// Advection chunk with the worked example's behaviours or nearest-neighbour
// interpolation on FP32 positions and FP32 storage (advect_f32_ext.cu).
cudaError_t launch_advect_plain_ext(const StepArgs &a, int block, cudaStream_t st);

// Element size of one position coordinate for a position form.
inline size_t pos_elem(int pos) { return pos == PG_POS_F64 ? 8 : 4; }
inline size_t storage_elem(int storage) {
  return storage == PG_F64 ? 8 : (storage == PG_F32 ? 4 : 2);
}

}  // namespace pg

namespace pg {

// Geometry kind of a grid; the FP32 kernels are compiled once per kind.
inline int geo_of(const GridArgs &g) {
  return g.mesh != 1 ? GEO_FLAT : (g.periodic ? GEO_SPH_PER : GEO_SPH);
}

// Shape of a launch over n particles of a set that does not fill the chip.
// Block: the given one, halved (to a warp at least) while the blocks would
// not give every multiprocessor two -- 10,000 FP64 particles in 40 blocks of
// 256 used 40 of 152.  Lanes: 32 particles per warp, fewer, in powers of two,
// while the warps are at most `sparse` per multiprocessor: such a launch
// lasts as long as its slowest warp's chain of stages, and a warp takes the
// slow path of a stage (a cell change: searches and dependent loads, four
// times the rest of the stage) whenever one of its lanes does.
// FP64 (one pipe per multiprocessor, 16 clocks a warp instruction whatever
// its lanes): one warp per multiprocessor (10,000 particles: 8.4 ms with 32
// lanes, 10.5 ms with 16).
constexpr int kSparseWarps = 8, kSparseWarps64 = 1;
inline void launch_shape(int64_t n, int block, int sms, int sparse, int &b, int &lanes) {
  b = block;
  lanes = 32;
  if (sms <= 0) return;
  while (lanes > 1 && (n + lanes / 2 - 1) / (lanes / 2) <= (int64_t)sms * sparse) lanes /= 2;
  const int64_t threads = (n + lanes - 1) / lanes * 32;
  while (b >= 64 && b % 64 == 0 && threads <= (int64_t)b * (2 * sms - 1)) b /= 2;
}

// Launch a chunk kernel over a.p.n particles, one thread each.  The block
// size is clamped to what the kernel's register use allows (queried once per
// kernel).
template <void (*Kernel)(StepArgs)>
inline cudaError_t launch_clamped(const StepArgs &a, int block, cudaStream_t st,
                                  int sparse = kSparseWarps) {
  static int max_threads = 0;
  static int sms = 0;
  if (max_threads == 0) {
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, Kernel);
    int dev = 0, q = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&q, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms = q;
    max_threads = at.maxThreadsPerBlock;
  }
  StepArgs s = a;
  int b;
  launch_shape(a.p.n, block > max_threads ? (max_threads / 32) * 32 : block, sms, sparse, b, s.lanes);
  const int64_t threads = (a.p.n + s.lanes - 1) / s.lanes * 32;
  const int64_t grid = (threads + b - 1) / b;
  Kernel<<<(unsigned)grid, b, 0, st>>>(s);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace pg
