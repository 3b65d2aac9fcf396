// C ABI of libtetm (include/tetm.h): solve lifetime, geometry, bunch,
// stepping, wake, diagnostics and checkpoints. Host logic only; the update
// and reduction kernels live in kernels_step.cu and kernels_diag.cu.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <unistd.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <vector>

#include "tetm_internal.h"
#include <nvtx3/nvToolsExt.h>

using namespace tetm;

namespace tetm {

Layout make_layout(int nx, int ny, int nz, int elem_bytes) {
  Layout L;
  L.nx = nx;
  L.ny = ny;
  L.nz = nz;
  // i = 0 after the guard columns: at column 8 in float32 (the 56-column tiles
  // of the slab kernel then write whole 32-byte sectors, and its tensor copies
  // start on 16-byte boundaries), at 2 in float64
  L.ox = elem_bytes == 4 ? 8 : 2;
  // rows on 32-byte sectors; float32 rows a multiple of 16 entries, so the
  // byte-wide activity rows are 16-byte strides for tensor copies
  const int align = elem_bytes == 4 ? 16 : 32 / elem_bytes;
  long long px = L.ox + nx + 3;                    // >= 2 zero columns past nx, plus one
                                                   // so a column pair starting at nx + 1 stays in the row
  px = (px + align - 1) / align * align;
  L.px = px;
  L.sz = (long long)(ny + 4) * px;
  L.count = (long long)(nz + 3) * L.sz;            // planes -1 .. nz+1
  return L;
}

}  // namespace tetm

namespace {

// ---------------------------------------------------------------------------
// Geometry on the device (staircase reading of the material matrices)
// ---------------------------------------------------------------------------
struct GeomIn {
  const uint8_t* pec;    // per cell of the whole grid or nullptr
  const double* eps;     // per cell of the whole grid or nullptr
  const double* mu;      // per cell of the whole grid or nullptr
  int nx, ny, nz;        // nz: planes of this solve
  int k_off, nz_all;     // z-slab: global plane of local plane 0, planes of the whole grid
  double dx, dy, dz;
};

// cell (ci, cj, ck) of this solve (ck local): PEC outside the whole grid
__device__ __forceinline__ bool gpec(const GeomIn& g, long ci, long cj, long ck) {
  ck += g.k_off;
  if (ci < 0 || cj < 0 || ck < 0 || ci >= g.nx || cj >= g.ny || ck >= g.nz_all) return true;
  return g.pec ? g.pec[ci + (long)g.nx * (cj + (long)g.ny * ck)] != 0 : false;
}
__device__ __forceinline__ double gval(const double* a, const GeomIn& g, long ci, long cj, long ck) {
  return a ? a[ci + (long)g.nx * (cj + (long)g.ny * (ck + g.k_off))] : 1.0;
}

// Edge along `axis` at node (i,j,k): the four cells around it.
__device__ double edge_minv(const GeomIn& g, int axis, long i, long j, long k) {
  long c[4][3];
  double len, area;
  if (axis == 0) {
    long t[4][3] = {{i, j - 1, k - 1}, {i, j, k - 1}, {i, j - 1, k}, {i, j, k}};
    memcpy(c, t, sizeof(c)); len = g.dx; area = g.dy * g.dz;
  } else if (axis == 1) {
    long t[4][3] = {{i - 1, j, k - 1}, {i, j, k - 1}, {i - 1, j, k}, {i, j, k}};
    memcpy(c, t, sizeof(c)); len = g.dy; area = g.dx * g.dz;
  } else {
    long t[4][3] = {{i - 1, j - 1, k}, {i, j - 1, k}, {i - 1, j, k}, {i, j, k}};
    memcpy(c, t, sizeof(c)); len = g.dz; area = g.dx * g.dy;
  }
  double e = 0.0;
  for (int q = 0; q < 4; ++q) {
    if (gpec(g, c[q][0], c[q][1], c[q][2])) return 0.0;
    e += gval(g.eps, g, c[q][0], c[q][1], c[q][2]);
  }
  return len / (kEps0 * 0.25 * e * area);
}

// Face normal to `axis` at node (i,j,k): the two cells sharing it.
__device__ double face_minv(const GeomIn& g, int axis, long i, long j, long k) {
  long c[2][3];
  double len, area;
  if (axis == 0) {
    long t[2][3] = {{i - 1, j, k}, {i, j, k}};
    memcpy(c, t, sizeof(c)); len = g.dx; area = g.dy * g.dz;
  } else if (axis == 1) {
    long t[2][3] = {{i, j - 1, k}, {i, j, k}};
    memcpy(c, t, sizeof(c)); len = g.dy; area = g.dx * g.dz;
  } else {
    long t[2][3] = {{i, j, k - 1}, {i, j, k}};
    memcpy(c, t, sizeof(c)); len = g.dz; area = g.dx * g.dy;
  }
  double r = 0.0;
  for (int q = 0; q < 2; ++q) {
    if (gpec(g, c[q][0], c[q][1], c[q][2])) return 0.0;
    r += 1.0 / gval(g.mu, g, c[q][0], c[q][1], c[q][2]);
  }
  return len * 0.5 * r / (kMu0 * area);
}

// Per-entry arrays of a component (material runs; nullptr where not kept): the
// steps' coefficient s M^-1 and, for the balances, which would otherwise divide
// at every use, M^-1 in float64 (float64 fields; M by recip_coef) or M and a2
// M^-1 as (hi, lo) float32 pairs whose sum is the float64 value to 2^-48
// (float32).
struct EntryOut {
  void* u;
  double s;
  double* minv;
  float2 *mp, *ap;
  double a2;
};
struct EntryOuts {
  EntryOut c[6];
};
template <typename T>
__device__ __forceinline__ void put_entry(const EntryOut& o, long long id, double v) {
  auto pair = [](double x) {
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
  };
  if (v == 0.0) return;
  static_cast<T*>(o.u)[id] = (T)(o.s * v);
  if constexpr (sizeof(T) == 8) {
    o.minv[id] = v;
  } else {
    o.mp[id] = pair(1.0 / v);
    if (o.ap) o.ap[id] = pair(o.a2 * v);
  }
}

// Activity bits (and the per-entry arrays, zero on entry) of the node entries of planes
// k_first .. nz: k_first = 0 for a whole grid, -1 for a z-slab whose plane
// below its first one is a ghost plane with the geometry of the whole grid; the
// nodes 0 .. n-1 of planes 0 .. nz-1 that carry a field are added to *active.
// Every entry of a node touches the node's own cell, so a node of a PEC cell
// has none, and with one material (no arrays) an entry carries a field where
// the cells around it are open and its constant is not zero (a bit of live).
// The six float64 quotients per node, which the mask alone does not need, were
// the time: 4.9 ms for 256 x 256 x 1024 nodes, so 0.3 (and the activity count, a
// pass of its own, 0.7). With arrays the entries' M^-1 become their
// coefficients here and only float64 fields keep them: in arrays of their own
// they were a quarter of the device memory of a float32 solve (1.5 GB for 192 x
// 192 x 768 nodes), written, read back and released for 1.6 ms.
template <typename T, bool ARRAYS>
__global__ void __launch_bounds__(256) build_geometry(GeomIn g, Layout L, int k_first, unsigned per_plane, unsigned live,
                                                      uint8_t* mask, EntryOuts out, unsigned long long* active) {
  const int k = k_first + (int)(blockIdx.x / per_plane);
  const unsigned q = (blockIdx.x % per_plane) * blockDim.x + threadIdx.x;
  const int i = (int)(q % (unsigned)(g.nx + 1)), j = (int)(q / (unsigned)(g.nx + 1));
  unsigned m = 0;
  if (j <= g.ny && !gpec(g, i, j, k)) {
    const long long id = L.idx(i, j, k);
    if constexpr (ARRAYS) {
      const double v[6] = {edge_minv(g, 0, i, j, k), edge_minv(g, 1, i, j, k), edge_minv(g, 2, i, j, k),
                           face_minv(g, 0, i, j, k), face_minv(g, 1, i, j, k), face_minv(g, 2, i, j, k)};
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        if (v[c] != 0.0) m |= 1u << c;
        put_entry<T>(out.c[c], id, v[c]);
      }
    } else {
      const bool x = !gpec(g, i - 1, j, k), y = !gpec(g, i, j - 1, k), z = !gpec(g, i, j, k - 1);
      if (y && z && !gpec(g, i, j - 1, k - 1)) m |= 1u << kEX;
      if (x && z && !gpec(g, i - 1, j, k - 1)) m |= 1u << kEY;
      if (x && y && !gpec(g, i - 1, j - 1, k)) m |= 1u << kEZ;
      if (x) m |= 1u << kHX;
      if (y) m |= 1u << kHY;
      if (z) m |= 1u << kHZ;
      m &= live;
    }
    mask[id] = (uint8_t)m;
  }
  const int n = __syncthreads_count(m != 0 && k >= 0 && k < g.nz);  // (the cell (i, j, k) is open: i < nx, j < ny)
  if (threadIdx.x == 0 && n) atomicAdd(active, (unsigned long long)n);
}

// M = 1/M^-1 per entry (0 where M^-1 is 0: an entry without a field), float64
// fields: a pass of its own, so that the cell arrays are released before the M
// arrays are made and a solve needs no more memory to be created than to be kept
__global__ void recip_coef(const double* minv, long long n, double* out) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) out[q] = minv[q] != 0.0 ? 1.0 / minv[q] : 0.0;
}

// flags |= 1: a value is not a finite number >= 1, |= 2: not all are equal
__global__ void scan_cells(const double* a, long long n, int* flags) {
  const double first = a[0];
  int f = 0;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    const double v = a[q];
    if (!(v >= 1.0) || !isfinite(v)) f |= 1;
    if (v != first) f |= 2;
  }
  f = __reduce_or_sync(0xffffffffu, f);
  if ((threadIdx.x & 31) == 0 && f) atomicOr(flags, f);
}

// Canonical FIT layout <-> device layout, for planes [k0, k0 + nk).
template <typename T>
__global__ void to_canonical(const T* src, Layout L, int k0, int nk, double* dst) {
  const long long total = (long long)(L.nx + 1) * (L.ny + 1) * nk;
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= total) return;
  const int i = (int)(q % (L.nx + 1));
  const int j = (int)((q / (L.nx + 1)) % (L.ny + 1));
  const int k = k0 + (int)(q / ((long long)(L.nx + 1) * (L.ny + 1)));
  dst[q] = (double)src[L.idx(i, j, k)];
}
template <typename T>
__global__ void from_canonical(const double* src, Layout L, int k0, int nk, const uint8_t* mask,
                               int comp, T* dst) {
  const long long total = (long long)(L.nx + 1) * (L.ny + 1) * nk;
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= total) return;
  const int i = (int)(q % (L.nx + 1));
  const int j = (int)((q / (L.nx + 1)) % (L.ny + 1));
  const int k = k0 + (int)(q / ((long long)(L.nx + 1) * (L.ny + 1)));
  const long long id = L.idx(i, j, k);
  dst[id] = ((mask[id] >> comp) & 1) ? (T)src[q] : T(0);
}

// Per tile and plane (tile-major): 1 where one of the tile's own cells carries
// a field in that plane; a warp per (tile, plane).
__global__ void tile_activity(const uint8_t* mask, Layout L, int tx, int ty, int tiles_x, long long n,
                              uint8_t* act) {
  const int lane = threadIdx.x & 31;
  const long long step = (long long)gridDim.x * blockDim.x / 32;
  for (long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / 32; q < n; q += step) {
    const int tile = (int)(q / L.nz), k = (int)(q % L.nz);
    const int i0 = (tile % tiles_x) * tx, j0 = (tile / tiles_x) * ty;
    bool any = false;
    for (int c = lane; c - lane < tx * ty && !any; c += 32) {
      const int i = i0 + c % tx, j = j0 + c / tx;
      any = __any_sync(0xffffffffu, c < tx * ty && i < L.nx && j < L.ny && mask[L.idx(i, j, k)] != 0);
    }
    if (lane == 0) act[q] = any ? 1 : 0;
  }
}

// Entries of one component that hold a non-zero value where the activity bit
// is clear: the guard ring around the cells and the entries of PEC objects,
// which every update leaves at zero (the canary of an out-of-place write).
template <typename T>
__global__ void guard_scan(const T* f, const uint8_t* mask, long long count, int comp,
                           unsigned long long* out) {
  unsigned long long c = 0;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < count;
       q += (long long)gridDim.x * blockDim.x)
    if (f[q] != T(0) && !((mask[q] >> comp) & 1)) ++c;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

double phi(double x) { return 0.5 * erfc(-x / sqrt(2.0)); }

}  // namespace


namespace {

int cuda_fail(cudaError_t e) {
  cudaGetLastError();  // answered here: the next launch's check must not see it again
  if (e == cudaErrorMemoryAllocation) return TETM_E_NOMEM;
  return TETM_E_CUDA;
}
#define CK(call)                                  \
  do {                                            \
    cudaError_t e_ = (call);                      \
    if (e_ != cudaSuccess) return cuda_fail(e_);  \
  } while (0)

int dalloc(tetm_solver* s, void** p, size_t bytes) {
  cudaError_t e = dev_alloc(p, bytes, s->stream);
  if (e != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    return cuda_fail(e);
  }
  s->device_bytes += (long long)bytes;
  return TETM_OK;
}

bool grid_ok(const tetm_grid* g) {
  return g && g->nx >= 2 && g->ny >= 2 && g->nz >= 2 && g->dx > 0 && g->dy > 0 && g->dz > 0 &&
         g->cdt >= 0 && (g->precision == TETM_FP64 || g->precision == TETM_FP32) &&
         isfinite(g->dx) && isfinite(g->dy) && isfinite(g->dz) && isfinite(g->cdt) &&
         (long long)g->nx * g->ny < (1LL << 31) && (long long)(g->nx + 1) * (g->ny + 1) * (g->nz + 1) < (1LL << 40);
}

double cdt_of(const tetm_grid* g) { return g->cdt > 0 ? g->cdt : g->dz; }

}  // namespace

namespace {
std::mutex g_pool_mu;
cudaMemPool_t g_pool[64];
uint64_t g_pool_keep = 0;

cudaMemPool_t lib_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(g_pool_mu);
  if (!g_pool[dev]) {
    cudaMemPoolProps props;
    memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    uint64_t keep = g_pool_keep;
    cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    g_pool[dev] = p;
  }
  return g_pool[dev];
}
}  // namespace

cudaError_t tetm::dev_alloc(void** p, size_t bytes, cudaStream_t st) {
  *p = nullptr;
  cudaMemPool_t pool = lib_pool();
  if (!pool) return cudaErrorMemoryAllocation;
  return cudaMallocFromPoolAsync(p, bytes ? bytes : 16, pool, st);
}

// One value of every page is read here first. The GPU reads pageable memory
// through the host's page tables, and a page that the CPU has not used for a
// while costs it a fault of some 10 us: 226 MB last used 0.2 s ago took 35 to 65
// ms to copy on a host that had been busy for a minute, 1.3 ms with the reads
// before it, which take 0.1 ms (pages of 64 KB).
cudaError_t tetm::upload(void* dst, const void* src, size_t bytes, cudaStream_t st) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, src) != cudaSuccess)
    cudaGetLastError();
  else if (at.type == cudaMemoryTypeUnregistered) {  // (pinned memory needs none)
    static const long sys = sysconf(_SC_PAGESIZE);
    const size_t page = sys > 0 ? (size_t)sys : 4096;
    const volatile unsigned char* p = static_cast<const volatile unsigned char*>(src);
    for (size_t q = 0; q < bytes; q += page) (void)p[q];
    if (bytes) (void)p[bytes - 1];
  }
  return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
}

void tetm::dev_free(void* p, cudaStream_t st) {
  if (p) cudaFreeAsync(p, st);
}

namespace {

// per tile of tx x ty nodes and plane (tile-major): 1 where one of its own
// cells carries a field
int tile_planes(tetm_solver* s, int tx, int ty, std::vector<uint8_t>* act) {
  const Layout& L = s->L;
  const int tiles_x = (L.nx + tx - 1) / tx, tiles_y = (L.ny + ty - 1) / ty;
  const size_t n = (size_t)tiles_x * tiles_y * L.nz;
  try {
    act->resize(n);
  } catch (const std::bad_alloc&) {
    return TETM_E_NOMEM;
  }
  uint8_t* d = nullptr;
  CK(dev_alloc((void**)&d, n, s->stream));
  tile_activity<<<(unsigned)std::min<size_t>((n + 7) / 8, 1u << 16), 256, 0, s->stream>>>(
      s->mask, L, tx, ty, tiles_x, (long long)n, d);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(act->data(), d, n, cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  dev_free(d, s->stream);
  return e == cudaSuccess ? TETM_OK : cuda_fail(e);
}

// The items (tile, chunk of cz planes) with an active plane, in grid order:
// items that run at the same time are neighbours and share their halo rows
// through L2 (ordering the list by work instead was measured 1.3x slower).
void items_of(const std::vector<uint8_t>& act, int nz, int cz, std::vector<int>* list) {
  const int tiles = (int)(act.size() / (size_t)nz);
  list->clear();
  for (int k0 = 0, c = 0; k0 < nz; k0 += cz, ++c)
    for (int t = 0; t < tiles; ++t)
      if (memchr(act.data() + (size_t)t * nz + k0, 1, (size_t)std::min(cz, nz - k0))) list->push_back(c * tiles + t);
}

// items[cz]: how many those are, cz = lo .. hi
std::vector<long long> count_items(const std::vector<uint8_t>& act, int nz, int lo, int hi) {
  std::vector<long long> items((size_t)hi + 1, 0);
  std::vector<int> before((size_t)nz + 1);  // active planes of the tile below a plane
  for (size_t t = 0; t < act.size() / (size_t)nz; ++t) {
    before[0] = 0;
    for (int k = 0; k < nz; ++k) before[(size_t)k + 1] = before[(size_t)k] + act[t * nz + k];
    if (!before[(size_t)nz]) continue;
    for (int cz = lo; cz <= hi; ++cz)
      for (int k0 = 0; k0 < nz; k0 += cz)
        items[(size_t)cz] += before[(size_t)std::min(k0 + cz, nz)] > before[(size_t)k0];
  }
  return items;
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return sms;
}

}  // namespace

void tetm::work_list(const tetm_solver* s, int cz, std::vector<int>* list) { items_of(s->act, s->L.nz, cz, list); }

// Planes per work item of the slab kernel, where the caller set none. Every
// item takes about cz + 2 planes' time (the plane below the chunk, and filling
// the pipeline) and the GPU holds two per SM at once, so a step takes
// ceil(items / slots) rounds of cz + 2 planes. Measured on eight one-material
// geometries (48 x 48 x 192 to 256 x 256 x 1024, every cz of 4..24 and every
// third to 62), the cz of the fewest such planes was the fastest in six, 1 and
// 10% off in the others; in three material ones 0 to 6%. Against 32 planes
// always: 32.8 -> 10.3 us per step on 48 x 48 x 192, 96.8 -> 63.5 on 128 x 128
// x 600 (342 items at 32 planes are two rounds, 288 at 38 one).
// Of `share` solves that step together each has its part of many rounds, so
// the last one counts by half: items * share / slots + 1/2 on average, at least
// one, and no more than kChunk planes, since the others may leave early (a batch
// of 16: 406 ms at 20 to 32 planes, 441 at 8, 423 at 64).
int tetm::choose_chunk(const std::vector<uint8_t>& act, int nz, int share, double* out) {
  const int sms = sm_count();
  const int top = std::min(share == 1 ? kMaxChunk : kChunk, std::max(nz, kMinChunk));
  if (sms < 1) return kChunk;
  const double slots = 2.0 * sms;
  const std::vector<long long> items = count_items(act, nz, kMinChunk, top);
  int best = kMinChunk;
  double least = 0.0;
  for (int cz = kMinChunk; cz <= top; ++cz) {
    const double r = (double)items[(size_t)cz] * share / slots;
    const double cost = (share == 1 ? ceil(r) : std::max(r + 0.5, 1.0)) * (cz + 2);
    if (cz == kMinChunk || cost <= least) {  // of equals the longest: fewest planes read twice
      best = cz;
      least = cost;
    }
  }
  if (out) *out = least;
  return best;
}

namespace {

// Planes per work item for a chunk the caller set on the shape 56 x 28, whose
// items own 12 rows: the set number, or, where that leaves the last round of
// the GPU's slots so empty that the step takes a tenth longer by the cost of
// choose_chunk, the best one of no less than half of it. The same chunk makes
// more than twice the items it made at 28 rows, and one round of those can
// become two with the second nearly empty.
int fit_chunk(const std::vector<uint8_t>& act, int nz, int cz) {
  const int sms = sm_count(), hi = std::min(cz, nz), lo = std::max(kMinChunk, (hi + 1) / 2);
  if (sms < 1 || lo >= hi) return cz;
  const double slots = 2.0 * sms;
  const std::vector<long long> items = count_items(act, nz, lo, hi);
  auto cost = [&](int c) { return ceil((double)items[(size_t)c] / slots) * (c + 2); };
  int best = hi;
  for (int c = hi - 1; c >= lo; --c)
    if (cost(c) < cost(best)) best = c;
  return cost(best) < 0.9 * cost(hi) ? best : cz;
}

}  // namespace

// All of it is made before anything of the solve changes: a rebuild that fails
// leaves the shape, the item list and the partials as they were, fit for each
// other (a list read under another tile shape would walk past the grid).
int tetm::rebuild_work(tetm_solver* s) try {
  const Layout& L = s->L;
  const int rows = slab_rows(s->tile_x, s->tile_y);
  const int tiles_x = (L.nx + s->tile_x - 1) / s->tile_x, tiles_y = (L.ny + rows - 1) / rows;
  const long long tiles = (long long)tiles_x * tiles_y;
  const int cz_min = s->auto_chunk() ? kMinChunk : s->chunk_z;
  if (tiles * ((L.nz + cz_min - 1) / cz_min) >= (1LL << 31)) return TETM_E_ARG;
  std::vector<uint8_t> act;
  const int rc = tile_planes(s, s->tile_x, rows, &act);
  if (rc != TETM_OK) return rc;
  const int cz = s->own_chunk ? s->chunk_z : s->auto_chunk() ? choose_chunk(act, L.nz, 1) : kChunk;
  const int item_z = s->own_chunk && rows != s->tile_y ? fit_chunk(act, L.nz, cz) : cz;
  std::vector<int> list;
  items_of(act, L.nz, item_z, &list);
  int* work = nullptr;
  double* part = nullptr;
  const int cap = std::max(2048, 3 * (int)list.size());  // balance reductions keep three partials per work item
  cudaError_t e = cudaSuccess;
  if (cap > s->diag.cap) e = dev_alloc((void**)&part, sizeof(double) * (size_t)cap, s->stream);
  if (e == cudaSuccess && !list.empty()) {
    e = dev_alloc((void**)&work, sizeof(int) * list.size(), s->stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(work, list.data(), sizeof(int) * list.size(), cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  }
  if (e != cudaSuccess) {
    dev_free(work, s->stream);
    dev_free(part, s->stream);
    return cuda_fail(e);
  }
  if (part) {
    dev_free(s->diag.part, s->stream);
    s->diag.part = part;
    s->diag.cap = cap;
  }
  dev_free(s->work, s->stream);
  s->work = work;
  s->tiles_x = tiles_x;
  s->tiles_y = tiles_y;
  s->chunk_z = cz;
  s->item_z = item_z;
  s->n_chunks = (L.nz + item_z - 1) / item_z;
  s->n_work = (int)list.size();
  s->work_host = std::move(list);
  s->act = std::move(act);
  s->work_dirty = false;
  return TETM_OK;
} catch (const std::bad_alloc&) {
  return TETM_E_NOMEM;
}

int tetm::reshape(tetm_solver* s, int tile_x, int tile_y, int chunk_z, bool own_shape, bool own_chunk) {
  const int x = s->tile_x, y = s->tile_y, z = s->chunk_z;
  const bool os = s->own_shape, oc = s->own_chunk;
  s->tile_x = tile_x;
  s->tile_y = tile_y;
  s->chunk_z = chunk_z;
  s->own_shape = own_shape;
  s->own_chunk = own_chunk;
  const int rc = rebuild_work(s);
  if (rc != TETM_OK) {
    s->tile_x = x;
    s->tile_y = y;
    s->chunk_z = z;
    s->own_shape = os;
    s->own_chunk = oc;
  }
  return rc;
}

namespace {

// Work items of the float64 band kernels: the column hulls of the active
// entries per (plane, band) from the device, the list from them.
int build_band(tetm_solver* s) try {
  const int rows = band_rows(s->active_cells);
  const size_t n = (size_t)((s->L.ny + rows - 1) / rows) * (size_t)s->L.nz;
  std::vector<int2> h(n);
  int2* d = nullptr;
  CK(dev_alloc((void**)&d, sizeof(int2) * n, s->stream));
  cudaError_t e = launch_band_hulls(s->mask, s->L, rows, d, s->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), d, sizeof(int2) * n, cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  dev_free(d, s->stream);
  if (e != cudaSuccess) return cuda_fail(e);
  std::vector<int4> items;
  band_list(s->L, rows, h, &items, &s->band_smem);
  s->n_band = (int)items.size();
  s->band_cells = 0;
  for (const int4& v : items) s->band_cells += (long long)(v.w & 0xFFFF) * (v.w >> 16);
  if (items.empty()) return TETM_OK;
  const int rc = dalloc(s, (void**)&s->band, sizeof(int4) * items.size());
  if (rc != TETM_OK) return rc;
  CK(cudaMemcpyAsync(s->band, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  return TETM_OK;
} catch (const std::bad_alloc&) {
  return TETM_E_NOMEM;
}

// Work items of the half-step kernels, where they are the faster float32 step
// (none otherwise). An item of `run` planes takes about run + 2 planes' time
// (its two launches each fill once), kHalfBlocks of them per SM at once, in the
// units of choose_chunk as long as latency bounds both. Up to kHalfCells active
// cells it does: us per step on the sweep | the halves at the run chosen here,
// 10.2 | 4.1 at 7e3 active cells, 10.2 | 5.2 at 1.1e5, 12.3 | 7.9 at 2.9e5,
// 14.4 | 10.8 at 3.7e5, 20.5 | 14.7 at 6.3e5; beyond, the halves' fuller SMs and
// 64 bytes per node cost more: 20.5 | 21.2 at 8.7e5, 28.7 | 31.8 at 1.4e6.
constexpr long long kHalfCells = 3LL << 18;
int build_half(tetm_solver* s) try {
  const int nz = s->L.nz, sms = sm_count();
  if (sms < 1 || s->n_work == 0 || s->active_cells > kHalfCells) return TETM_OK;
  double sweep = 0.0;
  choose_chunk(s->act, nz, 1, &sweep);
  const double slots = (double)kHalfBlocks * sms;
  std::vector<uint8_t> act;
  int rc = tile_planes(s, kHalfX, kHalfY, &act);
  if (rc != TETM_OK) return rc;
  const std::vector<long long> items = count_items(act, nz, 1, kMaxRun);
  for (int run = 1; run <= kMaxRun; ++run) {
    const double cost = ceil((double)items[(size_t)run] / slots) * (run + 2);
    if (cost >= sweep) continue;
    s->half_run = run;
    sweep = cost;
  }
  if (!s->half_run) return TETM_OK;
  std::vector<int> list;
  items_of(act, nz, s->half_run, &list);
  s->n_half = (int)list.size();
  rc = dalloc(s, (void**)&s->half, sizeof(int) * list.size());
  if (rc != TETM_OK) return rc;
  CK(cudaMemcpyAsync(s->half, list.data(), sizeof(int) * list.size(), cudaMemcpyHostToDevice, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  return TETM_OK;
} catch (const std::bad_alloc&) {
  return TETM_E_NOMEM;
}

}  // namespace

template <typename T>
StepArgs<T> tetm::step_args(tetm_solver* s, bool fused) {
  StepArgs<T> a;
  for (int c = 0; c < 6; ++c) {
    a.in[c] = (const T*)s->set[s->cur][c];
    a.out[c] = fused ? (T*)s->set[1 - s->cur][c] : (T*)s->set[s->cur][c];
    a.co.u[c] = (T)(((c == kEZ || c == kHZ) ? 2.0 * s->alpha : s->alpha) * s->minv_c[c]);
    a.co.ua[c] = (const T*)s->ua[c];
  }
  a.cstep = (unsigned)(field_step(s->L, s->esz) / 16);
  a.co.mask = s->mask;
  a.L = s->L;
  a.n = s->step;
  a.b.on = s->bunch ? 1 : 0;
  a.b.i0 = s->i0;
  a.b.j0 = s->j0;
  a.b.c0 = s->c0;
  a.b.kshift = s->kshift - s->k_lo;  // plane indices of the kernels are local to a z-slab
  a.b.m_min = s->m_min;
  a.b.m_max = s->m_max;
  a.b.inv_q = s->bunch ? 1.0 / s->q : 0.0;
  a.b.J = (const T*)s->J;
  a.b.W = s->W;
  {
    const int nw = s->bunch ? s->m_max - s->m_min + 1 : 0;
    const double eta0 = kMu0 * kC;
    a.b.obs_on = (s->bunch && s->obs_on) ? 1 : 0;
    a.b.obs_i = s->obs_i;
    a.b.obs_j = s->obs_j;
    a.b.WX = s->bunch ? s->W + nw : nullptr;
    a.b.WY = s->bunch ? s->W + 2 * nw : nullptr;
    const double iq = s->bunch ? 1.0 / s->q : 0.0;
    // E_x - c mu0 H_y and E_y + c mu0 H_x times dz/Q, with e = E * (edge
    // length) and h = H * (dual edge length): dy for h_y, dx for h_x
    a.b.tw_ex = s->g.dz * iq / s->g.dx;
    a.b.tw_hy = -eta0 * s->g.dz * iq / s->g.dy;
    a.b.tw_ey = s->g.dz * iq / s->g.dy;
    a.b.tw_hx = eta0 * s->g.dz * iq / s->g.dx;
  }
  a.tiles_x = s->tiles_x;
  a.tiles_y = s->tiles_y;
  a.chunk_z = s->item_z;
  a.n_chunks = s->n_chunks;
  a.work = s->work;
  a.n_work = s->n_work;
  return a;
}
template StepArgs<float> tetm::step_args<float>(tetm_solver*, bool);
template StepArgs<double> tetm::step_args<double>(tetm_solver*, bool);

namespace {

// Queue the FP64 balances of the step just taken into device slots:
// rec[0] = n, rec[1] = W^{n,e}, rec[2] = max|qe - qbunch|, rec[3] = max|qh|,
// rec[4] = max|qbunch|. No host synchronisation.
WorkView work_view(const tetm_solver* s) {
  WorkView v;
  v.items = s->work;
  v.n_items = s->n_work;
  v.tile_x = s->tile_x;
  v.tile_y = slab_rows(s->tile_x, s->tile_y);
  v.chunk_z = s->item_z;
  v.tiles_x = s->tiles_x;
  v.tiles_y = s->tiles_y;
  return v;
}

template <typename T>
int queue_balances(tetm_solver* s, double* rec) {
  const double zc = ((double)(s->step + s->kshift - s->k_lo - 1) + 0.5 - s->c0) * s->g.dz;
  CK(launch_bunch_charge(s->bunch ? s->q : 0.0, s->bunch ? s->sigma : 1.0, s->g.dz, zc, s->g.nz,
                         s->qline, rec + 4, (double)s->step, rec, s->stream));
  const T *cur[6], *prv[6];
  const double *ma[6], *mr[6];
  for (int c = 0; c < 6; ++c) {
    cur[c] = (const T*)s->set[s->cur][c];
    prv[c] = (const T*)s->set[1 - s->cur][c];
    ma[c] = s->minv_a[c];
    mr[c] = s->m_a[c];
  }
  const WorkView wv = work_view(s);
  if constexpr (sizeof(T) == 4) {
    if (!s->uniform) {  // float32 fields, material arrays: one float32-pair pass
      CK(launch_balances_mat_f32((const float* const*)cur, (const float* const*)prv, s->mask, s->mp, s->ap, s->L,
                                 s->alpha, s->bunch ? s->qline : nullptr, s->i0, s->j0, wv, s->diag, rec + 1,
                                 rec + 2, rec + 3, s->stream));
      return TETM_OK;
    }
  }
  if (s->uniform) {  // one pass for both
    CK(launch_balances<T>(cur, prv, s->mask, s->minv_c, s->L, s->alpha, s->bunch ? s->qline : nullptr, s->i0,
                          s->j0, wv, s->diag, rec + 1, rec + 2, rec + 3, s->stream));
    return TETM_OK;
  }
  if constexpr (sizeof(T) == 8) {  // float64 fields, material arrays: two float64 passes
    CK(launch_energy<T>(cur, s->mask, s->minv_c, ma, mr, s->L, s->alpha, wv, s->diag, rec + 1, s->stream));
    CK(launch_charge<T>(cur, prv, s->mask, s->minv_c, ma, mr, s->L, s->alpha,
                        s->bunch ? s->qline : nullptr, s->i0, s->j0, wv, s->diag, rec + 2, rec + 3,
                        s->stream));
  }
  return TETM_OK;
}

// Yee's scheme (Eq. (7)): the fused launch (ping-pong) for one material,
// else the two in-place reference launches
template <typename T>
int do_yee_steps(tetm_solver* s, int n) {
  const bool fused = s->kernel == TETM_KERNEL_FUSED && s->uniform;
  for (int q = 0; q < n; ++q) {
    StepArgs<T> a = step_args<T>(s, fused);
    for (int c = 0; c < 6; ++c) a.co.u[c] = (T)(2.0 * s->alpha * s->minv_c[c]);  // dt M^-1
    a.b.on = 0;
    a.b.obs_on = 0;
    if (fused) {
      if (s->n_work > 0) CK(launch_yee_fused_step<T>(a, s->stream));
      s->cur = 1 - s->cur;
    } else {
      CK(launch_yee_reference_step<T>(a, s->stream));
    }
    s->step += 1;
  }
  return TETM_OK;
}

template <typename T>
int do_steps(tetm_solver* s, int n) {
  if (s->scheme == TETM_SCHEME_YEE) return do_yee_steps<T>(s, n);
  bool last_pair = false;
  for (int q = 0; q < n; ++q) {
    const bool bal = s->bal_every > 0 && (s->step + 1) % s->bal_every == 0;
    if (s->kernel == TETM_KERNEL_TWOSTEP) {
      // a pair of steps per launch, unless a balance or a transverse gather
      // falls after its first step or a balance after its second (it needs
      // the state before)
      const bool bal2 = s->bal_every > 0 && (s->step + 2) % s->bal_every == 0;
      StepArgs<T> a = step_args<T>(s, true);
      last_pair = q + 1 < n && !bal && !bal2 && !(s->bunch && s->obs_on);
      if (last_pair) {
        if (s->n_work > 0) CK(launch_fused_two_steps<T>(a, s->tile_x, s->tile_y, s->stream));
        s->cur = 1 - s->cur;
        s->step += 2;
        ++q;
        continue;
      }
      if (s->n_work > 0) CK(launch_fused_step<T>(a, s->tile_x, s->tile_y, s->stream));
      if (s->bunch && s->obs_on) CK(launch_transverse_after_step<T>(a, s->stream));
      s->cur = 1 - s->cur;
    } else if (s->kernel == TETM_KERNEL_FUSED) {
      StepArgs<T> a = step_args<T>(s, true);
      if (s->n_work > 0) {
        const bool band = sizeof(T) == 8 && s->bands(), half = sizeof(T) == 4 && s->halves();
        if (band) {
          if constexpr (sizeof(T) == 8) CK(launch_band_step(a, s->band, s->n_band, s->band_smem, s->stream));
          a.b.obs_on = 0;  // the transverse wake is in
        } else if (half) {
          if constexpr (sizeof(T) == 4) CK(launch_half_step(a, s->half, s->n_half, s->half_run, s->stream));
          a.b.obs_on = 0;
        } else if (warp_shape_ok(s->tile_x, s->tile_y)) {
          CK(launch_fused_warp_step<T>(a, s->tile_x, s->tile_y, s->stream));
        } else if (slab_shape_ok(s->tile_x, s->tile_y, !s->uniform)) {
          if constexpr (sizeof(T) == 4) {
            CK(launch_fused_slab_step(a, s->sched, s->stream));
          } else {
            return TETM_E_UNSUPPORTED;
          }
        } else {
          CK(launch_fused_step<T>(a, s->tile_x, s->tile_y, s->stream));
        }
      }
      if (a.b.obs_on) CK(launch_transverse_after_step<T>(a, s->stream));
      s->cur = 1 - s->cur;
    } else {
      if (q == n - 1 || bal) {  // keep y^n beside y^{n+1} for the charge balance
        for (int c = 0; c < 6; ++c)
          CK(cudaMemcpyAsync(s->set[1 - s->cur][c], s->set[s->cur][c], (size_t)s->L.count * s->esz,
                             cudaMemcpyDeviceToDevice, s->stream));
      }
      StepArgs<T> a = step_args<T>(s, false);
      CK(launch_reference_step<T>(a, s->stream));
    }
    s->step += 1;
    if (bal) {
      double* rec = s->hist + 5 * (s->hist_count % s->hist_cap);
      int rc = queue_balances<T>(s, rec);
      if (rc) return rc;
      s->hist_count += 1;
    }
  }
  // after a pair the other field set holds the state two steps back
  if (n > 0) s->prev_valid = !last_pair;
  return TETM_OK;
}

int ensure_staging(tetm_solver* s) {
  if (s->staging) return TETM_OK;
  const long long plane = (long long)(s->L.nx + 1) * (s->L.ny + 1);
  long long nk = std::max(1LL, std::min((long long)s->L.nz + 1, (16LL << 20) / plane));
  s->staging_elems = nk * plane;
  return dalloc(s, (void**)&s->staging, sizeof(double) * (size_t)s->staging_elems);
}

template <typename T>
int get_fields_t(tetm_solver* s, int comp, double* host) {
  const long long plane = (long long)(s->L.nx + 1) * (s->L.ny + 1);
  const int nk_max = (int)(s->staging_elems / plane);
  for (int k0 = 0; k0 <= s->L.nz; k0 += nk_max) {
    const int nk = std::min(nk_max, s->L.nz + 1 - k0);
    const long long n = plane * nk;
    to_canonical<T><<<(unsigned)((n + 255) / 256), 256, 0, s->stream>>>(
        (const T*)s->set[s->cur][comp], s->L, k0, nk, s->staging);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(host + plane * k0, s->staging, sizeof(double) * (size_t)n,
                       cudaMemcpyDeviceToHost, s->stream));
    CK(cudaStreamSynchronize(s->stream));
  }
  return TETM_OK;
}

template <typename T>
int set_fields_t(tetm_solver* s, int comp, const double* host) {
  const long long plane = (long long)(s->L.nx + 1) * (s->L.ny + 1);
  const int nk_max = (int)(s->staging_elems / plane);
  for (int k0 = 0; k0 <= s->L.nz; k0 += nk_max) {
    const int nk = std::min(nk_max, s->L.nz + 1 - k0);
    const long long n = plane * nk;
    CK(cudaMemcpyAsync(s->staging, host + plane * k0, sizeof(double) * (size_t)n,
                       cudaMemcpyHostToDevice, s->stream));
    from_canonical<T><<<(unsigned)((n + 255) / 256), 256, 0, s->stream>>>(
        s->staging, s->L, k0, nk, s->mask, comp, (T*)s->set[s->cur][comp]);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(s->stream));
  }
  return TETM_OK;
}

// releases every device array of the solve, in the order of its stream
void free_all(tetm_solver* s) {
  cudaStream_t st = s->stream;
  for (int b = 0; b < 2; ++b) dev_free(s->set[b][0], st);
  for (int c = 0; c < 6; ++c) {
    dev_free(s->minv_a[c], st);
    dev_free(s->m_a[c], st);
    dev_free(s->mp[c], st);
    dev_free(s->ap[c], st);
    dev_free(s->ua[c], st);
  }
  dev_free(s->mask, st);
  dev_free(s->work, st);
  dev_free(s->band, st);
  dev_free(s->half, st);
  dev_free(s->J, st);
  dev_free(s->W, st);
  dev_free(s->qline, st);
  dev_free(s->diag.part, st);
  dev_free(s->diag.out, st);
  dev_free(s->hist, st);
  dev_free(s->staging, st);
  dev_free(s->sched, st);
}

}  // namespace

extern "C" {

const char* tetm_strerror(int code) {
  switch (code) {
    case TETM_OK: return "ok";
    case TETM_E_ARG: return "bad argument";
    case TETM_E_UNSTABLE: return "time step violates the stability bound of Eq. (25)";
    case TETM_E_NOT_MAGIC: return "bunch and wake need c*dt == dz";
    case TETM_E_NOMEM: return "out of memory";
    case TETM_E_CUDA: return "CUDA runtime error";
    case TETM_E_STATE: return "call not valid in the current solver state";
    case TETM_E_TIMEOUT: return "bounded device wait timed out";
    case TETM_E_DIVERGED: return "energy is not finite: the run diverged";
    case TETM_E_UNSUPPORTED: return "unsupported option combination";
    case TETM_E_TOO_LARGE: return "grid larger than the fixed scratch of tetm_energy_noalloc";
    default: return "unknown error";
  }
}

int64_t tetm_bytes_needed(const tetm_grid* g) {
  if (!grid_ok(g)) return 0;
  const size_t esz = g->precision == TETM_FP64 ? 8 : 4;
  const Layout L = make_layout(g->nx, g->ny, g->nz, (int)esz);
  return (int64_t)(12 * esz + 1) * L.count + (int64_t)(1 << 20);
}

}  // extern "C"

namespace {

// The flags of scan_cells for an array of n host values, which stays on the
// device in *out; -1 with nothing there where the device cannot.
int scan_on_device(const double* a, long long n, cudaStream_t st, double** out) {
  double* d = nullptr;
  int *f = nullptr, h = -1;
  if (dev_alloc((void**)&d, sizeof(double) * (size_t)n, st) == cudaSuccess &&
      dev_alloc((void**)&f, sizeof(int), st) == cudaSuccess && cudaMemsetAsync(f, 0, sizeof(int), st) == cudaSuccess &&
      upload(d, a, sizeof(double) * (size_t)n, st) == cudaSuccess) {
    scan_cells<<<1024, 256, 0, st>>>(d, n, f);
    if (cudaGetLastError() != cudaSuccess || cudaMemcpyAsync(&h, f, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      h = -1;
  }
  dev_free(f, st);
  if (h < 0) {
    dev_free(d, st);
    d = nullptr;
    cudaGetLastError();
  }
  *out = d;
  return h;
}

// Checks the material arrays (every value a finite number >= 1) and whether
// each holds one value only. On the host a pass over an array takes 0.74 ns per
// cell (20.9 ms for the 2.8e7 cells of a 192 x 192 x 768 grid), on the device
// its upload, which the geometry of a grid with several materials needs anyway,
// and 0.05 ms; so above kScanCells the arrays go up first and stay in dcell when
// they are not uniform. Where the device refuses (none there, no memory left)
// the host looks, so that a wrong value is a wrong argument there too.
constexpr long long kScanCells = 1 << 16;  // 48 us on the host, as much as a launch and its two copies
int cell_materials(const double* eps_r, const double* mu_r, long long ncell, cudaStream_t st, bool* uniform,
                   double* dcell[2]) {
  int flags = 0;
  for (int w = 0; w < 2; ++w) {
    const double* a = w == 0 ? eps_r : mu_r;
    if (!a) continue;
    int f = -1;
    if (ncell > kScanCells) f = scan_on_device(a, ncell, st, &dcell[w]);
    if (f < 0) {
      f = 0;
      for (long long q = 0; q < ncell && !(f & 1); ++q) f |= (!(a[q] >= 1.0) || !isfinite(a[q]) ? 1 : 0) | (a[q] != a[0] ? 2 : 0);
    }
    flags |= f;
    if (f & 1) break;
  }
  *uniform = !(flags & 2);
  if (*uniform || (flags & 1))
    for (int w = 0; w < 2; ++w) {
      dev_free(dcell[w], st);
      dcell[w] = nullptr;
    }
  return flags & 1 ? TETM_E_ARG : TETM_OK;
}

// A solve of planes [k_lo, k_lo + g->nz) of a grid of nz_all planes (the
// whole grid: k_lo = 0, nz_all = g->nz); the cell arrays cover the whole grid.
int create_impl(const tetm_grid* g, int k_lo, int nz_all, const double* eps_r, const double* mu_r,
                const uint8_t* pec, cudaStream_t st, tetm_solver** out) {
  if (!out) return TETM_E_ARG;
  *out = nullptr;
  if (!grid_ok(g)) return TETM_E_ARG;
  const double cdt = cdt_of(g);
  const double lim_t = 1.0 / sqrt(1.0 / (g->dx * g->dx) + 1.0 / (g->dy * g->dy));
  if (cdt > g->dz * (1.0 + 1e-12) || cdt > lim_t * (1.0 + 1e-12)) return TETM_E_UNSTABLE;
  const long long ncell = (long long)g->nx * g->ny * nz_all;
  // materials: physical (>= 1) and finite; uniform if every cell has the same value
  bool uniform = true;
  double eps_u = 1.0, mu_u = 1.0;
  double* dcell[2] = {nullptr, nullptr};  // eps_r, mu_r on the device (not uniform)
  const int checked = cell_materials(eps_r, mu_r, ncell, st, &uniform, dcell);
  if (checked != TETM_OK) return checked;
  if (eps_r) eps_u = eps_r[0];
  if (mu_r) mu_u = mu_r[0];
  int dev_count = 0;
  if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count < 1) {
    cudaGetLastError();
    return TETM_E_CUDA;
  }
  tetm_solver* s = new (std::nothrow) tetm_solver();
  if (!s) {
    for (double* d : dcell) dev_free(d, st);
    return TETM_E_NOMEM;
  }
  s->g = *g;
  s->g.cdt = cdt;
  s->k_lo = k_lo;
  s->nz_all = nz_all;
  s->esz = g->precision == TETM_FP64 ? 8 : 4;
  s->L = make_layout(g->nx, g->ny, g->nz, (int)s->esz);
  s->alpha = 0.5 * cdt / kC;
  s->stream = st;
  s->scheme = TETM_SCHEME_TETM;
  s->kernel = TETM_KERNEL_FUSED;
  s->uniform = uniform;
  s->vacuum = uniform && eps_u == 1.0 && mu_u == 1.0;
  // float32: the slab kernel (kernels_slab.cu; named 56 x 12 with
  // coefficient arrays); float64: the band kernels (kernels_band.cu), the
  // warp-tiled kernel (kernels_warp.cu) once a shape is set
  s->tile_x = s->esz == 4 ? 56 : 28;
  s->tile_y = s->esz == 4 ? (uniform ? 28 : 12) : 20;
  s->chunk_z = kChunk;
  int rc = TETM_OK;
  const size_t fstep = field_step(s->L, s->esz), fbytes = 5 * fstep + (size_t)s->L.count * s->esz;
  for (int b = 0; b < 2 && rc == TETM_OK; ++b) {
    rc = dalloc(s, &s->set[b][0], fbytes);
    if (rc != TETM_OK) break;
    for (int c = 1; c < 6; ++c) s->set[b][c] = (char*)s->set[b][0] + c * fstep;
    rc = cudaMemsetAsync(s->set[b][0], 0, fbytes, s->stream) == cudaSuccess ? TETM_OK : TETM_E_CUDA;
  }
  if (rc == TETM_OK) rc = dalloc(s, (void**)&s->mask, (size_t)s->L.count);
  if (rc == TETM_OK) rc = cudaMemsetAsync(s->mask, 0, (size_t)s->L.count, s->stream) == cudaSuccess ? TETM_OK : TETM_E_CUDA;
  if (rc == TETM_OK) rc = dalloc(s, (void**)&s->diag.part, sizeof(double) * 2048);
  if (rc == TETM_OK) rc = dalloc(s, (void**)&s->diag.out, sizeof(double) * 8);
  if (rc == TETM_OK) rc = dalloc(s, (void**)&s->sched, 2 * sizeof(int));
  if (rc == TETM_OK) rc = cudaMemsetAsync(s->sched, 0, 2 * sizeof(int), s->stream) == cudaSuccess ? TETM_OK : TETM_E_CUDA;
  s->diag.cap = 2048;
  s->hist_cap = 4096;
  if (rc == TETM_OK) rc = dalloc(s, (void**)&s->hist, sizeof(double) * 5 * (size_t)s->hist_cap);
  if (rc == TETM_OK) rc = dalloc(s, (void**)&s->qline, sizeof(double) * (size_t)(g->nz + 1));
  EntryOuts eo;
  memset(&eo, 0, sizeof(eo));
  if (rc == TETM_OK && !uniform) {
    const size_t n = (size_t)s->L.count;
    auto zeroed = [&](void** p, size_t bytes) {
      if (rc == TETM_OK) rc = dalloc(s, p, bytes);
      if (rc == TETM_OK && cudaMemsetAsync(*p, 0, bytes, s->stream) != cudaSuccess) rc = TETM_E_CUDA;
    };
    for (int c = 0; c < 6; ++c) {
      const bool a2 = c == kHX || c == kHY || c == kEX || c == kEY;
      zeroed(&s->ua[c], n * s->esz);
      if (s->esz == 8) {
        zeroed((void**)&s->minv_a[c], n * sizeof(double));
      } else {
        zeroed((void**)&s->mp[c], n * sizeof(float2));
        if (a2) zeroed((void**)&s->ap[c], n * sizeof(float2));
      }
      eo.c[c] = EntryOut{s->ua[c],    (c == kEZ || c == kHZ) ? 2.0 * s->alpha : s->alpha,
                         s->minv_a[c], s->mp[c], s->ap[c], s->alpha * s->alpha};
    }
  }
  // upload the cell arrays, build the mask (and the per-entry arrays) on the device
  GeomIn gi;
  gi.pec = nullptr;
  gi.eps = nullptr;
  gi.mu = nullptr;
  gi.nx = g->nx; gi.ny = g->ny; gi.nz = g->nz;
  gi.k_off = k_lo;
  gi.nz_all = nz_all;
  gi.dx = g->dx; gi.dy = g->dy; gi.dz = g->dz;
  uint8_t* dpec = nullptr;
  if (rc == TETM_OK && pec) {
    if (dev_alloc((void**)&dpec, (size_t)ncell, s->stream) != cudaSuccess ||
        upload(dpec, pec, (size_t)ncell, s->stream) != cudaSuccess)
      rc = TETM_E_CUDA;
    gi.pec = dpec;
  }
  if (rc == TETM_OK && !uniform) {
    for (int w = 0; w < 2 && rc == TETM_OK; ++w) {
      const double* a = w == 0 ? eps_r : mu_r;
      if (a && !dcell[w] &&
          (dev_alloc((void**)&dcell[w], sizeof(double) * (size_t)ncell, s->stream) != cudaSuccess ||
           upload(dcell[w], a, sizeof(double) * (size_t)ncell, s->stream) != cudaSuccess))
        rc = TETM_E_CUDA;
    }
    gi.eps = dcell[0];
    gi.mu = dcell[1];
  }
  unsigned long long* cnt = nullptr;
  if (rc == TETM_OK && dev_alloc((void**)&cnt, sizeof(*cnt), s->stream) != cudaSuccess) rc = TETM_E_CUDA;
  if (rc == TETM_OK) {
    const int k_first = k_lo > 0 ? -1 : 0;  // a z-slab's ghost plane below takes the whole grid's geometry
    const unsigned per_plane = (unsigned)(((long long)(g->nx + 1) * (g->ny + 1) + 255) / 256);
    const long long blocks = (long long)per_plane * (g->nz + 1 - k_first);
    // the components whose M^-1 is not zero with one material
    const double e = kEps0 * 0.25 * 4.0, h = 0.5 * 2.0;
    const double v[6] = {g->dx / (e * (g->dy * g->dz)), g->dy / (e * (g->dx * g->dz)), g->dz / (e * (g->dx * g->dy)),
                         g->dx * h / (kMu0 * (g->dy * g->dz)), g->dy * h / (kMu0 * (g->dx * g->dz)),
                         g->dz * h / (kMu0 * (g->dx * g->dy))};
    unsigned live = 0;
    for (int c = 0; c < 6; ++c)
      if (v[c] != 0.0) live |= 1u << c;
    unsigned long long n = 0;
    cudaMemsetAsync(cnt, 0, sizeof(*cnt), s->stream);
    if (uniform)
      build_geometry<float, false><<<(unsigned)blocks, 256, 0, s->stream>>>(gi, s->L, k_first, per_plane, live, s->mask, eo, cnt);
    else if (s->esz == 8)
      build_geometry<double, true><<<(unsigned)blocks, 256, 0, s->stream>>>(gi, s->L, k_first, per_plane, live, s->mask, eo, cnt);
    else
      build_geometry<float, true><<<(unsigned)blocks, 256, 0, s->stream>>>(gi, s->L, k_first, per_plane, live, s->mask, eo, cnt);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(&n, cnt, sizeof(n), cudaMemcpyDeviceToHost, s->stream) != cudaSuccess ||
        cudaStreamSynchronize(s->stream) != cudaSuccess)
      rc = TETM_E_CUDA;
    s->active_cells = (long long)n;
  }
  dev_free(cnt, s->stream);
  dev_free(dpec, s->stream);
  for (double* d : dcell) dev_free(d, s->stream);
  if (!uniform && s->esz == 8)
    for (int c = 0; c < 6 && rc == TETM_OK; ++c) {
      rc = dalloc(s, (void**)&s->m_a[c], sizeof(double) * (size_t)s->L.count);
      if (rc != TETM_OK) break;
      recip_coef<<<(unsigned)((s->L.count + 255) / 256), 256, 0, s->stream>>>(s->minv_a[c], s->L.count, s->m_a[c]);
      if (cudaGetLastError() != cudaSuccess) rc = TETM_E_CUDA;
    }
  // per-component constants for the uniform case (vacuum or one material)
  const double dx = g->dx, dy = g->dy, dz = g->dz;
  s->minv_c[kEX] = dx / (kEps0 * eps_u * dy * dz);
  s->minv_c[kEY] = dy / (kEps0 * eps_u * dx * dz);
  s->minv_c[kEZ] = dz / (kEps0 * eps_u * dx * dy);
  s->minv_c[kHX] = dx / (kMu0 * mu_u * dy * dz);
  s->minv_c[kHY] = dy / (kMu0 * mu_u * dx * dz);
  s->minv_c[kHZ] = dz / (kMu0 * mu_u * dx * dy);
  if (rc == TETM_OK) rc = rebuild_work(s);
  // (a z-slab keeps the fused sweep, which recomputes its ghost plane's TM half)
  if (rc == TETM_OK && s->esz == 8 && !s->is_slab()) rc = build_band(s);
  if (rc == TETM_OK && s->esz == 4 && s->uniform && !s->is_slab()) rc = build_half(s);
  if (rc != TETM_OK) {
    free_all(s);
    delete s;
    cudaGetLastError();
    return rc;
  }
  *out = s;
  return TETM_OK;
}

}  // namespace

extern "C" {

int tetm_create(const tetm_grid* g, const double* eps_r, const double* mu_r, const uint8_t* pec,
                tetm_solver** out) {
  return create_impl(g, 0, g ? g->nz : 0, eps_r, mu_r, pec, nullptr, out);
}

int tetm_create_on_stream(const tetm_grid* g, const double* eps_r, const double* mu_r, const uint8_t* pec,
                          void* stream, tetm_solver** out) {
  return create_impl(g, 0, g ? g->nz : 0, eps_r, mu_r, pec, (cudaStream_t)stream, out);
}

int tetm_pool_reserve(uint64_t bytes) {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  g_pool_keep = bytes;
  for (cudaMemPool_t p : g_pool)
    if (p && cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &bytes) != cudaSuccess) {
      cudaGetLastError();
      return TETM_E_CUDA;
    }
  return TETM_OK;
}

int tetm_create_slab(const tetm_grid* g, int32_t k_lo, int32_t k_hi, const double* eps_r, const double* mu_r,
                     const uint8_t* pec, tetm_solver** out) {
  if (!out) return TETM_E_ARG;
  *out = nullptr;
  if (!g || k_lo < 0 || k_hi > g->nz || k_hi - k_lo < 2) return TETM_E_ARG;
  tetm_grid local = *g;
  local.nz = k_hi - k_lo;
  return create_impl(&local, k_lo, g->nz, eps_r, mu_r, pec, nullptr, out);
}

void tetm_destroy(tetm_solver* s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream); else cudaDeviceSynchronize();
  free_all(s);
  delete s;
}

int tetm_set_stream(tetm_solver* s, void* st) {
  if (!s) return TETM_E_ARG;
  s->stream = (cudaStream_t)st;
  return TETM_OK;
}

int tetm_set_kernel(tetm_solver* s, int32_t kernel) {
  if (!s || (kernel != TETM_KERNEL_FUSED && kernel != TETM_KERNEL_REFERENCE && kernel != TETM_KERNEL_TWOSTEP))
    return TETM_E_ARG;
  if (s->in_batch) return TETM_E_STATE;
  if (kernel == TETM_KERNEL_TWOSTEP &&
      (!s->uniform || s->is_slab() || s->scheme != TETM_SCHEME_TETM || !fused2_shape_ok(s->tile_x, s->tile_y)))
    return TETM_E_UNSUPPORTED;
  if (kernel == TETM_KERNEL_REFERENCE && s->is_slab()) return TETM_E_UNSUPPORTED;  // it updates ghost planes in place
  // (Yee's scheme runs material arrays on the reference updates whatever the kernel)
  if (kernel == TETM_KERNEL_FUSED && !s->uniform && s->tile_x != 28 && !slab_shape_ok(s->tile_x, s->tile_y, true) &&
      s->scheme == TETM_SCHEME_TETM)
    return TETM_E_UNSUPPORTED;
  s->kernel = kernel;
  return TETM_OK;
}

int tetm_set_tiling(tetm_solver* s, int32_t tile_x, int32_t tile_y, int32_t chunk_z) {
  if (!s) return TETM_E_ARG;
  if (s->in_batch) return TETM_E_STATE;
  const int tx = tile_x ? tile_x : s->tile_x;
  const int ty = tile_y ? tile_y : s->tile_y;
  const int cz = chunk_z ? chunk_z : s->chunk_z;
  if (s->scheme == TETM_SCHEME_YEE) {  // Yee's fused kernel has one tile shape
    if (tx != s->tile_x || ty != s->tile_y) return TETM_E_UNSUPPORTED;
    if (cz < 4) return TETM_E_ARG;
    return reshape(s, tx, ty, cz, s->own_shape, s->own_chunk || chunk_z);
  }
  const bool slab_u = slab_shape_ok(tx, ty, false), slab_m = slab_shape_ok(tx, ty, true);
  if ((!fused_shape_ok(tx, ty) && !warp_shape_ok(tx, ty) && !slab_u && !slab_m) || cz < 4)
    return TETM_E_ARG;
  // per-entry coefficients (general materials) run on the warp-tiled kernel
  // and on the slab kernel as 56 x 12; one material there as 56 x 28
  if (!s->uniform && tx != 28 && !slab_m && s->kernel == TETM_KERNEL_FUSED)
    return TETM_E_UNSUPPORTED;
  if (s->uniform && slab_m && !slab_u) return TETM_E_UNSUPPORTED;
  // the slab kernel is float32 only
  if ((slab_u || slab_m) && s->esz != 4) return TETM_E_UNSUPPORTED;
  if (s->kernel == TETM_KERNEL_TWOSTEP && !fused2_shape_ok(tx, ty)) return TETM_E_UNSUPPORTED;
  const bool own_shape = s->own_shape || tile_x || tile_y || chunk_z, own_chunk = s->own_chunk || chunk_z;
  if (tx == s->tile_x && ty == s->tile_y && cz == s->chunk_z && s->work) {
    s->own_shape = own_shape;
    s->own_chunk = own_chunk;
    return TETM_OK;
  }
  return reshape(s, tx, ty, cz, own_shape, own_chunk);
}

int tetm_set_scheme(tetm_solver* s, int32_t scheme) {
  if (!s || (scheme != TETM_SCHEME_TETM && scheme != TETM_SCHEME_YEE)) return TETM_E_ARG;
  if (scheme == s->scheme) return TETM_OK;
  if (s->is_slab() || s->kernel == TETM_KERNEL_TWOSTEP) return TETM_E_UNSUPPORTED;
  if (s->step != 0 || s->bunch || s->in_batch || s->bal_every > 0) return TETM_E_STATE;
  int tx, ty;
  if (scheme == TETM_SCHEME_YEE) {
    const double dx = s->g.dx, dy = s->g.dy, dz = s->g.dz;
    const double lim = 1.0 / sqrt(1.0 / (dx * dx) + 1.0 / (dy * dy) + 1.0 / (dz * dz));  // Eq. (8)
    if (s->g.cdt > lim * (1.0 + 1e-12)) return TETM_E_UNSTABLE;
    yee_shape((int)s->esz, &tx, &ty);
  } else {  // the TE/TM scheme's default work shape
    tx = s->esz == 4 ? 56 : 28;
    ty = s->esz == 4 ? (s->uniform ? 28 : 12) : 20;
  }
  const int rc = reshape(s, tx, ty, s->chunk_z, s->own_shape, s->own_chunk);
  if (rc == TETM_OK) s->scheme = scheme;
  return rc;
}

int tetm_set_bunch(tetm_solver* s, double sigma_z, double charge, int32_t i0, int32_t j0) {
  if (!s || !(sigma_z > 0) || !isfinite(sigma_z) || charge == 0 || !isfinite(charge)) return TETM_E_ARG;
  if (i0 < 1 || i0 > s->g.nx - 1 || j0 < 1 || j0 > s->g.ny - 1) return TETM_E_ARG;
  if (s->scheme == TETM_SCHEME_YEE) return TETM_E_UNSUPPORTED;
  if (fabs(s->g.cdt - s->g.dz) > 1e-12 * s->g.dz) return TETM_E_NOT_MAGIC;
  if (s->step != 0 || s->bunch) return TETM_E_STATE;
  const double dz = s->g.dz;
  const int c0 = (int)ceil(5.0 * sigma_z / dz - 1e-12);
  const int m_max = (int)ceil(15.0 * sigma_z / dz - 1e-12);
  if (c0 < 1 || c0 > (1 << 20)) return TETM_E_ARG;
  std::vector<double> qc((size_t)(2 * c0));
  for (int d = -c0; d < c0; ++d) {
    const double lo = std::max((double)d * dz, -5.0 * sigma_z);
    const double hi = std::min((double)(d + 1) * dz, 5.0 * sigma_z);
    qc[(size_t)(d + c0)] = hi > lo ? charge * (phi(hi / sigma_z) - phi(lo / sigma_z)) : 0.0;
  }
  const int nw = m_max + c0 + 2;
  void* J = nullptr;
  double* W = nullptr;
  if (dev_alloc(&J, s->esz * qc.size(), s->stream) != cudaSuccess ||
      dev_alloc((void**)&W, 3 * sizeof(double) * nw, s->stream) != cudaSuccess) {
    dev_free(J, s->stream);
    dev_free(W, s->stream);
    cudaGetLastError();
    return TETM_E_NOMEM;
  }
  // J from a host vector that lives until the stream has read it (the
  // synchronisation below), all on the solve's stream
  int rc = TETM_OK;
  std::vector<double> j64;
  std::vector<float> j32;
  cudaError_t e = cudaSuccess;
  if (s->esz == 8) {
    j64.resize(qc.size());
    for (size_t q = 0; q < qc.size(); ++q) j64[q] = kC * qc[q] / dz;
    e = cudaMemcpyAsync(J, j64.data(), sizeof(double) * j64.size(), cudaMemcpyHostToDevice, s->stream);
  } else {
    j32.resize(qc.size());
    for (size_t q = 0; q < qc.size(); ++q) j32[q] = (float)(kC * qc[q] / dz);
    e = cudaMemcpyAsync(J, j32.data(), sizeof(float) * j32.size(), cudaMemcpyHostToDevice, s->stream);
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(W, 0, 3 * sizeof(double) * nw, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e != cudaSuccess) rc = TETM_E_CUDA;
  if (rc != TETM_OK) {
    dev_free(J, s->stream);
    dev_free(W, s->stream);
    cudaGetLastError();
    return rc;
  }
  s->J = J;
  s->W = W;
  s->device_bytes += (long long)(s->esz * qc.size() + 3 * sizeof(double) * nw);
  s->qcell = qc;
  s->bunch = true;
  s->i0 = i0;
  s->j0 = j0;
  s->obs_on = false;
  s->obs_i = i0;
  s->obs_j = j0;
  s->c0 = c0;
  s->m_min = -c0 - 1;
  s->m_max = m_max;
  s->sigma = sigma_z;
  s->q = charge;
  return TETM_OK;
}

int tetm_step(tetm_solver* s, int32_t n) {
  if (!s || n < 0) return TETM_E_ARG;
  if (s->in_batch) return TETM_E_STATE;
  if (s->kernel == TETM_KERNEL_FUSED && s->work_dirty) {
    int rc = rebuild_work(s);
    if (rc) return rc;
  }
  nvtxRangePushA("tetm_step");  // a range in a profiler's timeline (no cost without one)
  const int rc = s->esz == 8 ? do_steps<double>(s, n) : do_steps<float>(s, n);
  nvtxRangePop();
  return rc;
}

int tetm_sync(tetm_solver* s) {
  if (!s) return TETM_E_ARG;
  CK(cudaStreamSynchronize(s->stream));
  return TETM_OK;
}

int tetm_wake(tetm_solver* s, double* out, int32_t cap, int32_t* n_out, double* s0, double* ds) {
  if (!s) return TETM_E_ARG;
  if (!s->bunch) return TETM_E_STATE;
  const int nw = s->m_max - s->m_min + 1;
  if (n_out) *n_out = nw;
  if (s0) *s0 = s->m_min * s->g.dz;
  if (ds) *ds = s->g.dz;
  if (out) {
    if (cap < nw) return TETM_E_ARG;
    CK(cudaMemcpyAsync(out, s->W, sizeof(double) * nw, cudaMemcpyDeviceToHost, s->stream));
  }
  CK(cudaStreamSynchronize(s->stream));
  return TETM_OK;
}

int tetm_set_observer(tetm_solver* s, int32_t i, int32_t j) {
  if (!s) return TETM_E_ARG;
  if (s->in_batch || !s->bunch || s->step != 0) return TETM_E_STATE;
  if (i < 0 || i > s->g.nx - 1 || j < 0 || j > s->g.ny - 1) return TETM_E_ARG;
  s->obs_on = true;
  s->obs_i = i;
  s->obs_j = j;
  return TETM_OK;
}

int tetm_transverse_wake(tetm_solver* s, double* wx, double* wy, int32_t cap, int32_t* n_out, double* s0,
                         double* ds) {
  if (!s) return TETM_E_ARG;
  if (!s->bunch || !s->obs_on) return TETM_E_STATE;
  const int nw = s->m_max - s->m_min + 1;
  if (n_out) *n_out = nw;
  if (s0) *s0 = s->m_min * s->g.dz;
  if (ds) *ds = s->g.dz;
  if ((wx || wy) && cap < nw) return TETM_E_ARG;
  if (wx) CK(cudaMemcpyAsync(wx, s->W + nw, sizeof(double) * nw, cudaMemcpyDeviceToHost, s->stream));
  if (wy) CK(cudaMemcpyAsync(wy, s->W + 2 * nw, sizeof(double) * nw, cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  return TETM_OK;
}

int tetm_energy(tetm_solver* s, double* w) {
  if (!s || !w) return TETM_E_ARG;
  if (s->scheme != TETM_SCHEME_TETM) return TETM_E_UNSUPPORTED;
  const double *ma[6], *mr[6];
  for (int c = 0; c < 6; ++c) {
    ma[c] = s->minv_a[c];
    mr[c] = s->m_a[c];
  }
  cudaError_t e;
  if (s->esz == 8) {
    const double* f[6];
    for (int c = 0; c < 6; ++c) f[c] = (const double*)s->set[s->cur][c];
    e = s->uniform ? launch_balances<double>(f, nullptr, s->mask, s->minv_c, s->L, s->alpha, nullptr, 0, 0,
                                             work_view(s), s->diag, s->diag.out, nullptr, nullptr, s->stream)
                   : launch_energy<double>(f, s->mask, s->minv_c, ma, mr, s->L, s->alpha, work_view(s), s->diag,
                                           s->diag.out, s->stream);
  } else {
    const float* f[6];
    for (int c = 0; c < 6; ++c) f[c] = (const float*)s->set[s->cur][c];
    e = s->uniform ? launch_balances<float>(f, nullptr, s->mask, s->minv_c, s->L, s->alpha, nullptr, 0, 0,
                                            work_view(s), s->diag, s->diag.out, nullptr, nullptr, s->stream)
                   : launch_balances_mat_f32(f, nullptr, s->mask, s->mp, s->ap, s->L, s->alpha, nullptr, 0, 0,
                                             work_view(s), s->diag, s->diag.out, nullptr, nullptr, s->stream);
  }
  CK(e);
  CK(cudaMemcpyAsync(w, s->diag.out, sizeof(double), cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  return isfinite(*w) ? TETM_OK : TETM_E_DIVERGED;
}

int tetm_charge_residual(tetm_solver* s, double* max_e, double* max_h, double* q_scale) {
  if (!s) return TETM_E_ARG;
  if (s->scheme != TETM_SCHEME_TETM) return TETM_E_UNSUPPORTED;
  if (!s->prev_valid || s->step < 1) return TETM_E_STATE;
  int rc = s->esz == 8 ? queue_balances<double>(s, s->diag.out) : queue_balances<float>(s, s->diag.out);
  if (rc) return rc;
  double h[5];
  CK(cudaMemcpyAsync(h, s->diag.out, sizeof(h), cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  if (max_e) *max_e = h[2];
  if (max_h) *max_h = h[3];
  if (q_scale) *q_scale = h[4];
  return TETM_OK;
}

int tetm_set_balance_every(tetm_solver* s, int32_t every) {
  if (!s || every < 0) return TETM_E_ARG;
  // a z-slab's ghost planes of the new state arrive only with the next exchange
  if (every > 0 && s->is_slab()) return TETM_E_UNSUPPORTED;
  if (every > 0 && s->scheme != TETM_SCHEME_TETM) return TETM_E_UNSUPPORTED;
  s->bal_every = every;
  return TETM_OK;
}

int tetm_balance_history(tetm_solver* s, double* out, int32_t cap, int32_t* n_out) {
  if (!s) return TETM_E_ARG;
  const long long n = std::min<long long>(s->hist_count, s->hist_cap);
  if (n_out) *n_out = (int32_t)n;
  if (out && n > 0) {
    if (cap < n) return TETM_E_ARG;
    std::vector<double> h((size_t)(5 * s->hist_cap));
    CK(cudaMemcpyAsync(h.data(), s->hist, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s->stream));
    CK(cudaStreamSynchronize(s->stream));
    const long long first = s->hist_count - n;
    for (long long r = 0; r < n; ++r) {
      const long long slot = (first + r) % s->hist_cap;
      memcpy(out + 5 * r, h.data() + 5 * slot, 5 * sizeof(double));
    }
  } else {
    CK(cudaStreamSynchronize(s->stream));
  }
  return TETM_OK;
}

int tetm_get_fields(tetm_solver* s, int32_t comp, double* host) {
  if (!s || !host || comp < 0 || comp > 5) return TETM_E_ARG;
  int rc = ensure_staging(s);
  if (rc) return rc;
  return s->esz == 8 ? get_fields_t<double>(s, comp, host) : get_fields_t<float>(s, comp, host);
}

int tetm_set_fields(tetm_solver* s, int32_t comp, const double* host) {
  if (!s || !host || comp < 0 || comp > 5) return TETM_E_ARG;
  if (s->in_batch) return TETM_E_STATE;
  int rc = ensure_staging(s);
  if (rc) return rc;
  rc = s->esz == 8 ? set_fields_t<double>(s, comp, host) : set_fields_t<float>(s, comp, host);
  s->prev_valid = false;
  return rc;
}

int tetm_check_guards(tetm_solver* s, int64_t* violations) {
  if (!s || !violations) return TETM_E_ARG;
  unsigned long long* cnt = nullptr;
  unsigned long long h = 0;
  CK(dev_alloc((void**)&cnt, sizeof(*cnt), s->stream));
  cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(*cnt), s->stream);
  for (int b = 0; b < 2 && e == cudaSuccess; ++b)
    for (int c = 0; c < 6 && e == cudaSuccess; ++c) {
      if (s->esz == 8)
        guard_scan<double><<<1024, 256, 0, s->stream>>>((const double*)s->set[b][c], s->mask, s->L.count, c, cnt);
      else
        guard_scan<float><<<1024, 256, 0, s->stream>>>((const float*)s->set[b][c], s->mask, s->L.count, c, cnt);
      e = cudaGetLastError();
    }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  dev_free(cnt, s->stream);
  CK(e);
  *violations = (int64_t)h;
  return TETM_OK;
}

int64_t tetm_plane_bytes(tetm_solver* s, int32_t dir) {
  if (!s || (dir != TETM_PLANES_UP && dir != TETM_PLANES_DOWN)) return 0;
  return (int64_t)(dir == TETM_PLANES_UP ? 6 : 2) * s->L.sz * (int64_t)s->esz;
}

int tetm_export_plane(tetm_solver* s, int32_t dir, void* buf) {
  if (!s || !buf || (dir != TETM_PLANES_UP && dir != TETM_PLANES_DOWN)) return TETM_E_ARG;
  if (s->scheme != TETM_SCHEME_TETM || s->in_batch) return TETM_E_STATE;
  const size_t pb = (size_t)s->L.sz * s->esz;
  // up: every component of the last plane the solve owns; down: e_x, e_y of its first
  const int k = dir == TETM_PLANES_UP ? s->L.nz - 1 : 0;
  const int comps[6] = {kEX, kEY, kEZ, kHX, kHY, kHZ};
  const int nc = dir == TETM_PLANES_UP ? 6 : 2;
  char* p = static_cast<char*>(buf);
  for (int q = 0; q < nc; ++q) {
    const char* src = static_cast<const char*>(s->set[s->cur][comps[q]]) + (size_t)(k + 1) * pb;
    CK(cudaMemcpyAsync(p + q * pb, src, pb, cudaMemcpyDefault, s->stream));
  }
  return TETM_OK;
}

int tetm_import_plane(tetm_solver* s, int32_t dir, const void* buf) {
  if (!s || !buf || (dir != TETM_PLANES_UP && dir != TETM_PLANES_DOWN)) return TETM_E_ARG;
  if (s->scheme != TETM_SCHEME_TETM || s->in_batch) return TETM_E_STATE;
  // a message moving up fills the ghost plane below the first owned plane
  // (needs a neighbour below: k_lo > 0); one moving down fills e_x, e_y of
  // the plane above the last owned one (needs a neighbour above)
  if (dir == TETM_PLANES_UP ? s->k_lo == 0 : s->k_lo + s->L.nz >= s->nz_all) return TETM_E_STATE;
  const size_t pb = (size_t)s->L.sz * s->esz;
  const int k = dir == TETM_PLANES_UP ? -1 : s->L.nz;
  const int comps[6] = {kEX, kEY, kEZ, kHX, kHY, kHZ};
  const int nc = dir == TETM_PLANES_UP ? 6 : 2;
  const char* p = static_cast<const char*>(buf);
  for (int q = 0; q < nc; ++q) {
    char* dst = static_cast<char*>(s->set[s->cur][comps[q]]) + (size_t)(k + 1) * pb;
    CK(cudaMemcpyAsync(dst, p + q * pb, pb, cudaMemcpyDefault, s->stream));
  }
  return TETM_OK;
}

int tetm_get_info(tetm_solver* s, tetm_info* info) {
  if (!s || !info) return TETM_E_ARG;
  memset(info, 0, sizeof(*info));
  info->step = s->step;
  info->device_bytes = s->device_bytes;
  info->active_cells = s->active_cells;
  const bool fused = s->scheme == TETM_SCHEME_TETM && s->kernel == TETM_KERNEL_FUSED && !s->in_batch;
  info->processed_cells = fused && s->bands()    ? s->band_cells
                          : fused && s->halves() ? (long long)s->n_half * kHalfX * kHalfY * s->half_run
                                                 : (long long)s->n_work * s->tile_x * slab_rows(s->tile_x, s->tile_y) * s->item_z;
  info->kernel = s->kernel;
  info->precision = s->g.precision;
  info->tile_x = s->tile_x;
  info->tile_y = s->tile_y;
  info->chunk_z = s->chunk_z;
  info->work_items = s->n_work;
  info->wake_len = s->bunch ? s->m_max - s->m_min + 1 : 0;
  info->uniform_material = s->uniform ? 1 : 0;
  return TETM_OK;
}

// Checkpoint format: a fixed header, the six arrays of the current state in
// the device layout, then the wake accumulators.
struct CkptHeader {
  char magic[8];
  int32_t nx, ny, nz, precision;
  double dx, dy, dz, cdt;
  int64_t step;
  int64_t count;
  int32_t bunch, nw;
  int64_t kshift;
  int32_t obs_i, obs_j;
};

int tetm_save(tetm_solver* s, void* buf, size_t cap, size_t* used) {
  if (!s) return TETM_E_ARG;
  if (s->scheme != TETM_SCHEME_TETM) return TETM_E_UNSUPPORTED;
  const int nw = s->bunch ? s->m_max - s->m_min + 1 : 0;
  const size_t fb = (size_t)s->L.count * s->esz;
  const size_t need = sizeof(CkptHeader) + 6 * fb + 3 * sizeof(double) * (size_t)nw;
  if (used) *used = need;
  if (!buf) return TETM_OK;
  if (cap < need) return TETM_E_ARG;
  CkptHeader h;
  memset(&h, 0, sizeof(h));
  memcpy(h.magic, "TETMCKP3", 8);
  h.nx = s->g.nx; h.ny = s->g.ny; h.nz = s->g.nz; h.precision = s->g.precision;
  h.dx = s->g.dx; h.dy = s->g.dy; h.dz = s->g.dz; h.cdt = s->g.cdt;
  h.step = s->step;
  h.count = s->L.count;
  h.bunch = s->bunch;
  h.nw = nw;
  h.kshift = s->kshift;
  h.obs_i = (s->bunch && s->obs_on) ? s->obs_i : -1;  // -1: no transverse wake
  h.obs_j = (s->bunch && s->obs_on) ? s->obs_j : -1;
  char* p = (char*)buf;
  memcpy(p, &h, sizeof(h));
  p += sizeof(h);
  for (int c = 0; c < 6; ++c, p += fb)
    CK(cudaMemcpyAsync(p, s->set[s->cur][c], fb, cudaMemcpyDeviceToHost, s->stream));
  if (nw) CK(cudaMemcpyAsync(p, s->W, 3 * sizeof(double) * nw, cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  return TETM_OK;
}

int tetm_load(tetm_solver* s, const void* buf, size_t size) {
  if (!s || !buf || size < sizeof(CkptHeader)) return TETM_E_ARG;
  if (s->scheme != TETM_SCHEME_TETM) return TETM_E_UNSUPPORTED;
  if (s->in_batch) return TETM_E_STATE;
  CkptHeader h;
  memcpy(&h, buf, sizeof(h));
  const int nw = s->bunch ? s->m_max - s->m_min + 1 : 0;
  const size_t fb = (size_t)s->L.count * s->esz;
  if (memcmp(h.magic, "TETMCKP3", 8) != 0 || h.nx != s->g.nx || h.ny != s->g.ny || h.nz != s->g.nz ||
      h.precision != s->g.precision || h.count != s->L.count || h.bunch != (int)s->bunch || h.nw != nw ||
      h.dx != s->g.dx || h.dy != s->g.dy || h.dz != s->g.dz || h.cdt != s->g.cdt ||
      h.kshift != s->kshift)
    return TETM_E_ARG;
  const int oi = (s->bunch && s->obs_on) ? s->obs_i : -1, oj = (s->bunch && s->obs_on) ? s->obs_j : -1;
  if (h.obs_i != oi || h.obs_j != oj) return TETM_E_ARG;
  if (size < sizeof(CkptHeader) + 6 * fb + 3 * sizeof(double) * (size_t)nw) return TETM_E_ARG;
  const char* p = (const char*)buf + sizeof(h);
  for (int c = 0; c < 6; ++c, p += fb)
    CK(cudaMemcpyAsync(s->set[s->cur][c], p, fb, cudaMemcpyHostToDevice, s->stream));
  if (nw) CK(cudaMemcpyAsync(s->W, p, 3 * sizeof(double) * nw, cudaMemcpyHostToDevice, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  s->step = h.step;
  s->prev_valid = false;
  return TETM_OK;
}

}  // extern "C"
