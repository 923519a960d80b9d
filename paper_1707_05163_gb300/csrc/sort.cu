// sort.cu -- Morton re-sort with compaction, and FP64 moments.
//
// Re-sort: particles are bucketed by the Morton code of their (coarsened)
// cell indices, so that neighbouring threads advect particles in
// neighbouring cells and their field gathers share cache lines; deleted
// particles go to one last bucket behind all alive ones, so later launches
// cover only the alive prefix.  It is a counting sort: histogram, exclusive
// scan, scatter, then one gather of every particle array into the second set
// of arrays.  Order inside a bucket is not fixed; no particle's arithmetic
// depends on it.
//
// Moments: FP64 sums over alive particles, per block in a fixed order and
// then over blocks in a fixed order, so the result does not depend on timing.
#include "pg_host.h"

namespace pg {

namespace {

constexpr int kMaxKeyBits = 22;
constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanBlock * kScanItems;

struct MortonSpec {
  int dims;
  int bits[3];
  int shift[3];
  int total;
};

// Bits of the Morton key: all cell bits of each axis, then the finest bits
// dropped (largest axis first) until the key has at most about twice as many
// buckets as particles (between 2^8 and 2^22 buckets).
MortonSpec morton_spec(const pg_fieldset *fs, int64_t n) {
  int max_bits = 1;
  while (max_bits < kMaxKeyBits && ((int64_t)1 << max_bits) < 2 * n) ++max_bits;
  if (max_bits < 8) max_bits = 8;
  MortonSpec m{};
  const int nodes[3] = {fs->nx, fs->ny, fs->nz};
  m.dims = fs->nz > 1 ? 3 : 2;
  m.total = 0;
  for (int d = 0; d < m.dims; ++d) {
    int b = 0;
    while ((1 << b) < nodes[d]) ++b;
    m.bits[d] = b;
    m.shift[d] = 0;
    m.total += b;
  }
  while (m.total > max_bits) {
    int w = 0;
    for (int d = 1; d < m.dims; ++d)
      if (m.bits[d] > m.bits[w]) w = d;
    --m.bits[w];
    ++m.shift[w];
    --m.total;
  }
  return m;
}

template <typename Real>
__device__ __forceinline__ int cell_index(const Real *x, int n, int uni, Real x0, Real inv, Real p) {
  int i;
  if (uni) {
    const Real f = floor((p - x0) * inv);
    i = f >= (Real)0 ? (f > (Real)(n - 1) ? n - 1 : (int)f) : 0;     // 0 for NaN too
  } else {
    int lo = 0, hi = n - 1;
    if (!(p >= x[0])) return 0;
    if (!(p < x[n - 1])) return n - 1;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (x[mid] <= p) lo = mid; else hi = mid;
    }
    i = lo;
  }
  return i;
}

__device__ __forceinline__ uint32_t morton(const int (&c)[3], const MortonSpec &m) {
  uint32_t key = 0;
  int pos = 0;
  int maxb = 0;
  for (int d = 0; d < m.dims; ++d) maxb = m.bits[d] > maxb ? m.bits[d] : maxb;
  for (int b = 0; b < maxb; ++b)
    for (int d = 0; d < m.dims; ++d)
      if (b < m.bits[d]) key |= (uint32_t)(((c[d] >> m.shift[d]) >> b) & 1) << pos++;
  return key;
}

// Bucket of every particle and the buckets' counts.  Cells are found in the
// positions' own precision (GridArgs' axes in it): the order only decides
// which particles are neighbours, and FP64 searches took 0.57 ms for 10M FP32
// positions.
__device__ __forceinline__ const double *sort_axis(const GridArgs &g, int a, double) {
  return a == 0 ? g.lon : (a == 1 ? g.lat : g.depth);
}
__device__ __forceinline__ const float *sort_axis(const GridArgs &g, int a, float) {
  return a == 0 ? g.lonf : (a == 1 ? g.latf : g.depthf);
}
__device__ __forceinline__ double sort_x0(const GridArgs &g, int a, double) { return g.x0[a]; }
__device__ __forceinline__ float sort_x0(const GridArgs &g, int a, float) { return g.x0f[a]; }
__device__ __forceinline__ double sort_inv(const GridArgs &g, int a, double) { return g.inv_d[a]; }
__device__ __forceinline__ float sort_inv(const GridArgs &g, int a, float) { return g.inv_df[a]; }

template <typename Real>
__global__ void bucket_kernel(GridArgs g, MortonSpec m, const Real *x, const Real *y,
                              const Real *z, const int32_t *ci, const int32_t *cj,
                              const int32_t *ck, const uint8_t *status, int64_t n,
                              uint32_t dead, uint32_t *key, uint32_t *count) {
  const Real o = (Real)0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    uint32_t k = dead;
    if (status[p] == 0) {
      int c[3] = {0, 0, 0};
      if (ci) {
        c[0] = ci[p]; c[1] = cj[p]; c[2] = ck ? ck[p] : 0;
      } else {
        Real lon = x[p];
        if (g.periodic) {
          Real r = lon - sort_x0(g, 0, o);
          if (!(r >= (Real)0 && r < (Real)360)) {
            r = fmod(r, (Real)360);
            if (r < (Real)0) r += (Real)360;
            lon = sort_x0(g, 0, o) + r;
          }
        }
        c[0] = cell_index(sort_axis(g, 0, o), g.nx, g.uni[0], sort_x0(g, 0, o), sort_inv(g, 0, o), lon);
        c[1] = cell_index(sort_axis(g, 1, o), g.ny, g.uni[1], sort_x0(g, 1, o), sort_inv(g, 1, o), y[p]);
        if (g.nz > 1)
          c[2] = cell_index(sort_axis(g, 2, o), g.nz, g.uni[2], sort_x0(g, 2, o), sort_inv(g, 2, o), z[p]);
      }
      k = morton(c, m);
    }
    key[p] = k;
    atomicAdd(&count[k], 1u);
  }
}

// Exclusive scan of m counts, tile by tile (1024 threads x 4 items).
__global__ void scan_tiles_kernel(const uint32_t *in, uint32_t *out, uint32_t *tile_sums,
                                  int64_t m) {
  __shared__ uint32_t s[kScanBlock];
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t local = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < m ? in[base + i] : 0u;
    local += v[i];
  }
  s[threadIdx.x] = local;
  __syncthreads();
  for (int o = 1; o < kScanBlock; o <<= 1) {
    const uint32_t add = threadIdx.x >= (unsigned)o ? s[threadIdx.x - o] : 0u;
    __syncthreads();
    s[threadIdx.x] += add;
    __syncthreads();
  }
  uint32_t run = s[threadIdx.x] - local;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < m) out[base + i] = run;
    run += v[i];
  }
  if (threadIdx.x == kScanBlock - 1) tile_sums[blockIdx.x] = s[threadIdx.x];
}

__global__ void scan_add_kernel(uint32_t *out, const uint32_t *tile_off, int64_t m) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  const uint32_t add = tile_off[blockIdx.x];
  for (int i = threadIdx.x; i < kScanTile; i += blockDim.x)
    if (base + i < m) out[base + i] += add;
}

__global__ void scatter_kernel(const uint32_t *key, uint32_t *offset, uint32_t *perm, int64_t n) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t at = atomicAdd(&offset[key[p]], 1u);
    perm[at] = (uint32_t)p;
  }
}

// Arrays of a set's state moved in one pass: entry p of dst from entry perm[p]
// of src (perm null: entry p).  A permuted pass is bound by its scattered
// reads, so arrays share a pass only while they stay in L2 together (129 MB on
// the chip this library is compiled for, source and destination): the passes of
// a set of up to a million particles take them all (one launch in place of
// twelve); of 10M particles, all at once were 1.03 ms, and passes of at most
// kPassBytes 0.39 ms.
constexpr int kPassArrays = 8;
constexpr size_t kPassBytes = (size_t)48 << 20;
struct StatePass {
  const void *src[kPassArrays];
  void *dst[kPassArrays];
  int el[kPassArrays];      // 8, 4 or 1 bytes
  int n = 0;
};
__global__ void __launch_bounds__(256) state_pass_kernel(const __grid_constant__ StatePass a,
                                                         const uint32_t *perm, int64_t n) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = perm ? (int64_t)perm[p] : p;
    unsigned long long v[kPassArrays];
#pragma unroll
    for (int j = 0; j < kPassArrays; ++j)
      if (j < a.n)
        v[j] = a.el[j] == 8   ? reinterpret_cast<const unsigned long long *>(a.src[j])[q]
               : a.el[j] == 4 ? reinterpret_cast<const uint32_t *>(a.src[j])[q]
                              : reinterpret_cast<const uint8_t *>(a.src[j])[q];
#pragma unroll
    for (int j = 0; j < kPassArrays; ++j)
      if (j < a.n) {
        if (a.el[j] == 8) reinterpret_cast<unsigned long long *>(a.dst[j])[p] = v[j];
        else if (a.el[j] == 4) reinterpret_cast<uint32_t *>(a.dst[j])[p] = (uint32_t)v[j];
        else reinterpret_cast<uint8_t *>(a.dst[j])[p] = (uint8_t)v[j];
      }
  }
}

void launch_state_pass(const pg_pset *ps, const PsetArrays &src, const PsetArrays &dst,
                       const uint32_t *perm, int grid, cudaStream_t st) {
  StatePass a;
  size_t bytes = 0;
  auto flush = [&]() {
    if (a.n == 0) return;
    state_pass_kernel<<<grid, 256, 0, st>>>(a, perm, ps->n);
    note_launches(1);
    a.n = 0;
    bytes = 0;
  };
  auto move = [&](const void *s, void *d, int el) {
    const size_t b = (size_t)ps->n * el;
    if (a.n == kPassArrays || (perm && a.n > 0 && bytes + b > kPassBytes)) flush();
    a.src[a.n] = s; a.dst[a.n] = d; a.el[a.n] = el;
    ++a.n;
    bytes += b;
  };
  if (ps->pos == PG_POS_CELL) {
    move(src.ci, dst.ci, 4); move(src.cj, dst.cj, 4); move(src.ck, dst.ck, 4);
    move(src.fx, dst.fx, 4); move(src.fy, dst.fy, 4); move(src.fz, dst.fz, 4);
  } else {
    const int el = (int)pos_elem(ps->pos);
    move(src.x, dst.x, el); move(src.y, dst.y, el); move(src.z, dst.z, el);
  }
  move(src.step, dst.step, 4);
  move(src.status, dst.status, 1);
  move(src.time, dst.time, 8);
  move(src.id, dst.id, 8);
  if (ps->age_used) move(src.age, dst.age, 8);
  if (ps->hstep_used) move(src.hstep, dst.hstep, 8);
  for (int j = 0; j < ps->nvar; ++j)
    move(src.var + (size_t)j * ps->cap, dst.var + (size_t)j * ps->cap, 8);
  flush();
}

int grid_of(int64_t n, int sm) {
  int64_t g = (n + 255) / 256;
  if (g > (int64_t)sm * 32) g = (int64_t)sm * 32;
  return (int)(g < 1 ? 1 : g);
}

// Exclusive scan of m entries in place of `out` (in may equal out).
cudaError_t exclusive_scan(const uint32_t *in, uint32_t *out, int64_t m, uint32_t *tmp,
                           cudaStream_t st) {
  const int64_t tiles = (m + kScanTile - 1) / kScanTile;
  uint32_t *sums = tmp;                 // [tiles]
  uint32_t *sums_out = tmp + tiles;     // [tiles]
  uint32_t *dummy = tmp + 2 * tiles;    // [1]
  scan_tiles_kernel<<<(unsigned)tiles, kScanBlock, 0, st>>>(in, out, sums, m);
  if (tiles > 1) {
    // tiles <= kScanTile, so one tile scans all tile sums
    scan_tiles_kernel<<<1, kScanBlock, 0, st>>>(sums, sums_out, dummy, tiles);
    scan_add_kernel<<<(unsigned)tiles, 256, 0, st>>>(out, sums_out, m);
    note_launches(2);
  }
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

// Exclusive scan of m 32-bit entries (m at most scan_max_entries()) with a
// scratch of scan_scratch_words(m) words; in may equal out.
int64_t scan_max_entries() { return (int64_t)kScanTile * kScanTile; }
size_t scan_scratch_words(int64_t m) { return (size_t)(2 * ((m + kScanTile - 1) / kScanTile) + 1); }
cudaError_t exclusive_scan_u32(const uint32_t *in, uint32_t *out, int64_t m, uint32_t *tmp,
                               cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  if (m > scan_max_entries()) return cudaErrorInvalidValue;
  return exclusive_scan(in, out, m, tmp, st);
}

// n_alive == nullptr: keep the particle arrays where they are (the sorted
// copy is copied back) and read nothing back to the host, so the whole
// re-sort is a fixed sequence of device operations (capturable in a graph).
// Scratch and the second array set must then already exist
// (prepare_resort).
cudaError_t prepare_resort(pg_pset *ps) {
  const int64_t n = ps->n;
  if (n == 0) return cudaSuccess;
  const MortonSpec m = morton_spec(ps->fs, n);
  const int64_t nb = ((int64_t)1 << m.total) + 1;
  const int64_t tiles = (nb + kScanTile - 1) / kScanTile;
  const size_t need = sizeof(uint32_t) * ((size_t)n * 2 + (size_t)nb * 2 + (size_t)tiles * 2 + 1);
  cudaError_t e;
  if (ps->sort_scratch_bytes < need) {
    dev_free(ps->sort_scratch);
    ps->sort_scratch = nullptr;
    ps->sort_scratch_bytes = 0;
    if ((e = dev_alloc(&ps->sort_scratch, need)) != cudaSuccess) return e;
    ps->sort_scratch_bytes = need;
  }
  // the second set has exactly the first one's capacity: the sampled
  // variables are laid out with the capacity as their stride
  if (ps->alt_cap != ps->cap) {
    ps->alt.free_all();
    ps->alt_cap = 0;
    const pg_status r = alloc_arrays(ps->alt, ps->pos, ps->cap, ps->nvar);
    if (r) return r == PG_ERR_NOMEM ? cudaErrorMemoryAllocation : cudaErrorUnknown;
    ps->alt_cap = ps->cap;
  }
  return cudaSuccess;
}

cudaError_t launch_resort(pg_pset *ps, cudaStream_t st, int64_t *n_alive) {
  const int64_t n = ps->n;
  if (n_alive) *n_alive = n;
  if (n == 0) return cudaSuccess;
  if (n >= (int64_t)0xFFFFFFFFll) return cudaErrorInvalidValue;
  const pg_fieldset *fs = ps->fs;
  const MortonSpec m = morton_spec(fs, n);
  const uint32_t dead = 1u << m.total;
  const int64_t nb = (int64_t)dead + 1;
  cudaError_t e;
  if ((e = prepare_resort(ps)) != cudaSuccess) return e;
  uint32_t *key = (uint32_t *)ps->sort_scratch;
  uint32_t *perm = key + n;
  uint32_t *count = perm + n;
  uint32_t *offset = count + nb;
  uint32_t *tmp = offset + nb;
  const int sm = fs->sm_count;
  const GridArgs g = grid_args_of(fs);
  if ((e = cudaMemsetAsync(count, 0, sizeof(uint32_t) * nb, st)) != cudaSuccess) return e;
  const int gr = grid_of(n, sm);
  if (ps->pos == PG_POS_F64)
    bucket_kernel<double><<<gr, 256, 0, st>>>(g, m, (const double *)ps->x, (const double *)ps->y,
                                              (const double *)ps->z, nullptr, nullptr, nullptr,
                                              ps->status, n, dead, key, count);
  else if (ps->pos == PG_POS_F32)
    bucket_kernel<float><<<gr, 256, 0, st>>>(g, m, (const float *)ps->x, (const float *)ps->y,
                                             (const float *)ps->z, nullptr, nullptr, nullptr,
                                             ps->status, n, dead, key, count);
  else
    bucket_kernel<float><<<gr, 256, 0, st>>>(g, m, nullptr, nullptr, nullptr, ps->ci, ps->cj,
                                             fs->nz > 1 ? ps->ck : nullptr, ps->status, n, dead,
                                             key, count);
  note_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = exclusive_scan(count, offset, nb, tmp, st)) != cudaSuccess) return e;
  uint32_t dead_count = 0;
  if (n_alive &&
      (e = cudaMemcpyAsync(&dead_count, count + dead, 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return e;
  scatter_kernel<<<gr, 256, 0, st>>>(key, offset, perm, n);
  note_launches(1);
  PsetArrays &B = ps->alt;
  launch_state_pass(ps, pset_arrays(ps), B, perm, gr, st);
  // fixed-pointer mode: the sorted arrays back in place
  if (!n_alive) launch_state_pass(ps, B, pset_arrays(ps), nullptr, gr, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (!n_alive) return cudaSuccess;
  // swap the two array sets
  const PsetArrays A = pset_arrays(ps);
  pset_set_arrays(ps, B);
  B = A;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  *n_alive = n - (int64_t)dead_count;
  return cudaSuccess;
}

// ----------------------------------------------------------------- moments

namespace {

constexpr int kMomBlocks = 256;
constexpr int kMomThreads = 256;

template <typename Real>
__device__ __forceinline__ void pos_of(const Real *x, const Real *y, const Real *z,
                                       const int32_t *ci, const int32_t *cj, const int32_t *ck,
                                       const float *fx, const float *fy, const float *fz,
                                       const GridArgs &g, int64_t p, double &a, double &b,
                                       double &c) {
  if (ci) {   // uniform axes: x0 + (index + offset) * spacing
    a = g.x0[0] + ((double)ci[p] + (double)fx[p]) * g.d[0];
    b = g.x0[1] + ((double)cj[p] + (double)fy[p]) * g.d[1];
    c = ck ? g.x0[2] + ((double)ck[p] + (double)fz[p]) * g.d[2] : 0.0;
  } else {
    a = (double)x[p]; b = (double)y[p]; c = (double)z[p];
  }
}

// Block b sums the contiguous range [b*chunk, (b+1)*chunk) in index order,
// thread-strided, then combines threads in a fixed tree.
template <typename Real>
__global__ void moments_kernel(GridArgs g, const Real *x, const Real *y, const Real *z,
                               const int32_t *ci, const int32_t *cj, const int32_t *ck,
                               const float *fx, const float *fy, const float *fz,
                               const uint8_t *status, int64_t n, double *partial) {
  __shared__ double sh[7][kMomThreads];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t beg = (int64_t)blockIdx.x * chunk;
  const int64_t end = beg + chunk < n ? beg + chunk : n;
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int64_t p = beg + threadIdx.x; p < end; p += blockDim.x) {
    if (status[p] != 0) continue;
    double a, b, c;
    pos_of<Real>(x, y, z, ci, cj, ck, fx, fy, fz, g, p, a, b, c);
    acc[0] += 1.0; acc[1] += a; acc[2] += b; acc[3] += c;
    acc[4] += a * a; acc[5] += b * b; acc[6] += c * c;
  }
  for (int q = 0; q < 7; ++q) sh[q][threadIdx.x] = acc[q];
  __syncthreads();
  for (int o = kMomThreads / 2; o > 0; o >>= 1) {
    if (threadIdx.x < (unsigned)o)
      for (int q = 0; q < 7; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 7; ++q) partial[blockIdx.x * 7 + q] = sh[q][0];
}

__global__ void moments_final_kernel(const double *partial, int nblocks, double *out) {
  const int q = threadIdx.x;
  if (q < 7) {
    double s = 0.0;
    for (int b = 0; b < nblocks; ++b) s += partial[b * 7 + q];
    out[q] = s;
  }
}

}  // namespace

cudaError_t launch_moments(const pg_pset *ps_c, double *out7, cudaStream_t st) {
  pg_pset *ps = const_cast<pg_pset *>(ps_c);
  cudaError_t e;
  if (!ps->diag_scratch) {
    if ((e = dev_alloc((void **)&ps->diag_scratch, sizeof(double) * (kMomBlocks * 7 + 8))) !=
        cudaSuccess)
      return e;
  }
  const pg_fieldset *fs = ps->fs;
  const GridArgs g = grid_args_of(fs);
  double *partial = ps->diag_scratch;
  double *res = partial + kMomBlocks * 7;
  const int64_t n = ps->n;
  if (ps->pos == PG_POS_F64)
    moments_kernel<double><<<kMomBlocks, kMomThreads, 0, st>>>(
        g, (const double *)ps->x, (const double *)ps->y, (const double *)ps->z, nullptr, nullptr,
        nullptr, nullptr, nullptr, nullptr, ps->status, n, partial);
  else if (ps->pos == PG_POS_F32)
    moments_kernel<float><<<kMomBlocks, kMomThreads, 0, st>>>(
        g, (const float *)ps->x, (const float *)ps->y, (const float *)ps->z, nullptr, nullptr,
        nullptr, nullptr, nullptr, nullptr, ps->status, n, partial);
  else
    moments_kernel<float><<<kMomBlocks, kMomThreads, 0, st>>>(
        g, nullptr, nullptr, nullptr, ps->ci, ps->cj, fs->nz > 1 ? ps->ck : nullptr, ps->fx,
        ps->fy, fs->nz > 1 ? ps->fz : nullptr, ps->status, n, partial);
  moments_final_kernel<<<1, 32, 0, st>>>(partial, kMomBlocks, res);
  note_launches(2);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(out7, res, sizeof(double) * 7, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return e;
  return cudaStreamSynchronize(st);
}

}  // namespace pg
