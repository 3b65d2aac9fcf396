// Float64 step in two launches, one per half (Sec. 4.2, Eq. (23)): the TM half
// (U1..U5) of every plane, then the TE half (U6..U10).
//
// What bounds it: the float64 pipe. A warp's float64 instruction takes the
// SM's pipe for about 20 cycles however many of its lanes are active (9.66 ns
// measured), 36 of them per 32 cells and step (61 us for 0.86 M cells), while
// the 128 bytes a cell moves in two launches are a third of that time at the
// HBM rate. So the split is made for few float64 instructions and full warps:
//  * no march along z: a half reads the other half's results from memory, so
//    no plane is computed twice (the fused sweeps recompute the TM half of the
//    plane below each z-chunk) and every (plane, band) pair is independent.
//    A 24 x 24 x 96 pipe is 288 work items instead of 6 serial marches of 792
//    rows each, and a 96 x 96 x 384 collimator 2000 instead of 108;
//  * a work item is a band of rows of one plane, cut to the columns between
//    the first and last that carry a field there (the pipe wall around a round
//    pipe costs nothing), at most 64 wide;
//  * inside an item the nodes of each stage are numbered consecutively and
//    dealt to the threads, whatever the width, with exactly the halo the
//    stage needs: the halo is one node, not two, and costs 0.8 rows and 0.8
//    columns of a half's work (the warp-tiled sweep: 4 of 24 rows, 4 of 32
//    columns, 1 of 33 planes);
//  * intermediates (hx~, hy~, ez' / ex~, ey~, hz') stay in shared memory.
// Per node the operations and their order are those of the other step
// kernels, so the results are the same bits.
// Measured per step, warp-tiled sweep (28 x 20 x 32) -> bands: 24 x 24 x 96
// pipe 1101 -> 14.05 us; collimators 96 x 96 x 384 1189 -> 98 us, 192 x 192 x
// 384 1200 -> 317 us, 256 x 256 x 1024 2042 -> 1387 us (85% of the float64
// pipe's rate at 36 instructions per active cell); with coefficient arrays,
// 96 x 96 x 384, 1151 -> 101 us. 256 threads against 128: the small pipe 14.2
// against 16.5 us, the others the same. The loads of a node do not wait for
// its activity byte, and the launches overlap their starts (launch_pdl): the
// small pipe took 19.7 us without.
#include <algorithm>

#include "tetm_internal.h"

namespace tetm {
namespace {

constexpr int kBThreads = 256;
constexpr int kBandCols = 64;  // columns of an item at most

// this thread's nodes of a stage: node t of rows x width nodes, t = thread,
// thread + kBThreads, ...
struct Walk {
  int r, c;
  const int w, rows;
  __device__ __forceinline__ Walk(int rows_, int w_) : r((int)threadIdx.x / w_), c((int)threadIdx.x % w_), w(w_), rows(rows_) {}
  __device__ __forceinline__ bool ok() const { return r < rows; }
  __device__ __forceinline__ void next() {
    c += kBThreads;
    while (c >= w) {
      c -= w;
      ++r;
    }
  }
};

struct BandItem {
  int k, j0, i0, w, rows;  // owned nodes: rows j0 .. j0 + rows - 1, columns i0 .. i0 + w - 1 of plane k
  long long base;          // layout index of (i0, j0, k)
};
__device__ __forceinline__ BandItem band_item(const int4* items, const Layout& L) {
  const int4 v = items[blockIdx.x];
  BandItem it;
  it.k = v.x;
  it.j0 = v.y;
  it.i0 = v.z;
  it.w = v.w & 0xFFFF;
  it.rows = v.w >> 16;
  it.base = L.idx(it.i0, it.j0, it.k);
  return it;
}

// doubles of shared memory of an item: two arrays of (rows + 2)(w + 1), two of
// (rows + 1)(w + 2), one of (rows + 1)(w + 1)
__host__ __device__ constexpr int band_doubles(int rows, int w) {
  return 2 * (rows + 2) * (w + 1) + 2 * (rows + 1) * (w + 2) + (rows + 1) * (w + 1);
}

// the coefficient of component c at an entry that carries it
template <bool MAT>
__device__ __forceinline__ double coef(const StepArgs<double>& a, int c, long long id) {
  if constexpr (MAT)
    return a.co.ua[c][id];
  else
    return a.co.u[c];
}

// TM half of a band: hx~ on the owned rows, one below (for ez' of the first)
// and one above, columns to one right of the owned; hy~ to one row above, one
// column left and right; ez' to one row above and one column right; then the
// owned hx', hy'. An entry without a field holds zero and stays zero.
template <bool MAT>
__global__ void __launch_bounds__(kBThreads, 4) band_tm(const StepArgs<double> a, const int4* __restrict__ items) {
  extern __shared__ double band_sm[];
  const Layout L = a.L;
  const BandItem it = band_item(items, L);
  const long long PX = L.px, SZ = L.sz;
  const int R = it.rows, W = it.w, wx = W + 1, wy = W + 2;
  double* const hxa = band_sm;              // rows -1 .. R, columns 0 .. W
  double* const dey = hxa + (R + 2) * wx;   // e_y of plane k+1 minus plane k, there
  double* const hya = dey + (R + 2) * wx;   // rows 0 .. R, columns -1 .. W
  double* const dex = hya + (R + 1) * wy;
  double* const ezn = dex + (R + 1) * wy;   // rows 0 .. R, columns 0 .. W
  const uint8_t* __restrict__ mk = a.co.mask + it.base;
  // (no __restrict__: it would let the compiler load a field before pdl_wait)
  const double* ex = a.in[kEX] + it.base;
  const double* ey = a.in[kEY] + it.base;
  const double* ez = a.in[kEZ] + it.base;
  const double* hx = a.in[kHX] + it.base;
  const double* hy = a.in[kHY] + it.base;
  pdl_trigger();
  pdl_wait();
  for (Walk t(R + 2, wx); t.ok(); t.next()) {
    const long long id = (t.r - 1) * PX + t.c;
    const unsigned m = mk[id];
    const double y0 = ey[id], y1 = ey[id + SZ], z0 = ez[id], z1 = ez[id + PX], h0 = hx[id];
    double h = 0.0, d = 0.0;
    if (m & 8) {
      d = y1 - y0;
      h = h0 + coef<MAT>(a, kHX, it.base + id) * (d - (z1 - z0));                  // U1
    }
    hxa[t.r * wx + t.c] = h;
    dey[t.r * wx + t.c] = d;
  }
  for (Walk t(R + 1, wy); t.ok(); t.next()) {
    const long long id = t.r * PX + t.c - 1;
    const unsigned m = mk[id];
    const double x0 = ex[id], x1 = ex[id + SZ], z0 = ez[id], z1 = ez[id + 1], h0 = hy[id];
    double h = 0.0, d = 0.0;
    if (m & 16) {
      d = x1 - x0;
      h = h0 + coef<MAT>(a, kHY, it.base + id) * (-d + (z1 - z0));                 // U2
    }
    hya[t.r * wy + t.c] = h;
    dex[t.r * wy + t.c] = d;
  }
  __syncthreads();
  for (Walk t(R + 1, wx); t.ok(); t.next()) {
    const long long id = t.r * PX + t.c;
    double e = 0.0;
    if (mk[id] & 4) {
      const double* x = hxa + (t.r + 1) * wx + t.c;
      const double* y = hya + t.r * wy + t.c + 1;
      double cur = (x[-wx] - x[0]) - (y[-1] - y[0]);
      const bool line = a.b.on && it.i0 + t.c == a.b.i0 && it.j0 + t.r == a.b.j0;
      if (line) {  // the bunch current on its line
        const long long dd = (long long)it.k - (a.n + a.b.kshift) + a.b.c0;
        if (dd >= -a.b.c0 && dd < a.b.c0) cur -= a.b.J[dd + a.b.c0];
      }
      e = ez[id] + coef<MAT>(a, kEZ, it.base + id) * cur;                           // U3
      if (t.r < R && t.c < W) {
        a.out[kEZ][it.base + id] = e;
        // one item owns the line's node of a plane: a sample gets one addition a step
        if (line) add_wake(a.b, (a.n + a.b.kshift) - it.k - a.b.c0, e);
      }
    }
    ezn[t.r * wx + t.c] = e;
  }
  __syncthreads();
  for (Walk t(R, W); t.ok(); t.next()) {
    const long long id = t.r * PX + t.c;
    const unsigned m = mk[id];
    const double* e = ezn + t.r * wx + t.c;
    if (m & 8)
      a.out[kHX][it.base + id] = hxa[(t.r + 1) * wx + t.c] + coef<MAT>(a, kHX, it.base + id) *
                                 (dey[(t.r + 1) * wx + t.c] - (e[wx] - e[0]));      // U4
    if (m & 16)
      a.out[kHY][it.base + id] = hya[t.r * wy + t.c + 1] + coef<MAT>(a, kHY, it.base + id) *
                                 (-dex[t.r * wy + t.c + 1] + (e[1] - e[0]));        // U5
  }
}

// TE half, the mirror image: ex~ to one row below and above and one column
// left, ey~ to one row below and one column left and right, hz' to one row
// below and one column left, then the owned ex', ey'. It reads the new h_x,
// h_y of its plane and of the plane below, which band_tm has written.
template <bool MAT>
__global__ void __launch_bounds__(kBThreads, 4) band_te(const StepArgs<double> a, const int4* __restrict__ items) {
  extern __shared__ double band_sm[];
  const Layout L = a.L;
  const BandItem it = band_item(items, L);
  const long long PX = L.px, SZ = L.sz;
  const int R = it.rows, W = it.w, wx = W + 1, wy = W + 2;
  double* const exa = band_sm;              // rows -1 .. R, columns -1 .. W-1
  double* const dhy = exa + (R + 2) * wx;   // new h_y of plane k-1 minus plane k, there
  double* const eya = dhy + (R + 2) * wx;   // rows -1 .. R-1, columns -1 .. W
  double* const dhx = eya + (R + 1) * wy;
  double* const hzn = dhx + (R + 1) * wy;   // rows -1 .. R-1, columns -1 .. W-1
  const uint8_t* __restrict__ mk = a.co.mask + it.base;
  const double* ex = a.in[kEX] + it.base;
  const double* ey = a.in[kEY] + it.base;
  const double* hz = a.in[kHZ] + it.base;
  const double* hx = a.out[kHX] + it.base;
  const double* hy = a.out[kHY] + it.base;
  pdl_trigger();
  pdl_wait();
  // the transverse wake of the observer line's node, from the old e_x, e_y and
  // the new h_x, h_y, beside the rest (as a launch of its own behind the step it
  // made the small pipe 14.2 us instead of 14.05, 17.4 when its start overlapped)
  const int oi = a.b.obs_i - it.i0, oj = a.b.obs_j - it.j0;
  if (a.b.obs_on && threadIdx.x == 0 && oi >= 0 && oi < W && oj >= 0 && oj < R) {
    const long long id = oj * PX + oi;
    gather_wx(a.b, a.n, it.k, ex[id], hy[id]);
    gather_wy(a.b, a.n, it.k, ey[id], hx[id]);
  }
  for (Walk t(R + 2, wx); t.ok(); t.next()) {
    const long long id = (t.r - 1) * PX + t.c - 1;
    const unsigned m = mk[id];
    double e = 0.0, d = 0.0;
    const double y0 = hy[id], y1 = hy[id - SZ], z0 = hz[id], e0 = ex[id];
    if (m & 1) {
      d = y1 - y0;
      e = e0 + coef<MAT>(a, kEX, it.base + id) * (d - (hz[id - PX] - z0));         // U6
    }
    exa[t.r * wx + t.c] = e;
    dhy[t.r * wx + t.c] = d;
  }
  for (Walk t(R + 1, wy); t.ok(); t.next()) {
    const long long id = (t.r - 1) * PX + t.c - 1;
    const unsigned m = mk[id];
    double e = 0.0, d = 0.0;
    const double x0 = hx[id], x1 = hx[id - SZ], z0 = hz[id], e0 = ey[id];
    if (m & 2) {
      d = x1 - x0;
      e = e0 + coef<MAT>(a, kEY, it.base + id) * (-d + (hz[id - 1] - z0));         // U7
    }
    eya[t.r * wy + t.c] = e;
    dhx[t.r * wy + t.c] = d;
  }
  __syncthreads();
  for (Walk t(R + 1, wx); t.ok(); t.next()) {
    const long long id = (t.r - 1) * PX + t.c - 1;
    double h = 0.0;
    if (mk[id] & 32) {
      const double* x = exa + t.r * wx + t.c;
      const double* y = eya + t.r * wy + t.c;
      h = hz[id] + coef<MAT>(a, kHZ, it.base + id) * ((x[wx] - x[0]) - (y[1] - y[0]));  // U8
      if (t.r > 0 && t.c > 0) a.out[kHZ][it.base + id] = h;
    }
    hzn[t.r * wx + t.c] = h;
  }
  __syncthreads();
  for (Walk t(R, W); t.ok(); t.next()) {
    const long long id = t.r * PX + t.c;
    const unsigned m = mk[id];
    const double* h = hzn + (t.r + 1) * wx + t.c + 1;
    if (m & 1)
      a.out[kEX][it.base + id] = exa[(t.r + 1) * wx + t.c + 1] + coef<MAT>(a, kEX, it.base + id) *
                                 (dhy[(t.r + 1) * wx + t.c + 1] - (h[-wx] - h[0]));   // U9
    if (m & 2)
      a.out[kEY][it.base + id] = eya[(t.r + 1) * wy + t.c + 1] + coef<MAT>(a, kEY, it.base + id) *
                                 (-dhx[(t.r + 1) * wy + t.c + 1] + (h[-1] - h[0]));   // U10
  }
}

// First and last + 1 column with an active entry among rows [band * rows, +
// rows) of plane k (first = last: none); one warp per (plane, band).
__global__ void band_hulls(const uint8_t* mask, Layout L, int rows, int bands, int2* out) {
  const int lane = threadIdx.x & 31;
  const long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (q >= (long long)bands * L.nz) return;
  const int band = (int)(q % bands), k = (int)(q / bands);
  int lo = L.nx, hi = 0;
  for (int j = band * rows; j < min((band + 1) * rows, L.ny); ++j)
    for (int i = lane; i < L.nx; i += 32)
      if (mask[L.idx(i, j, k)]) {
        lo = min(lo, i);
        hi = max(hi, i + 1);
      }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) out[q] = make_int2(lo, max(lo, hi));
}

}  // namespace

// Rows of a band: 16 rows halve the halo rows of 8 (0.8 of a row's work per
// band), 8 rows make twice as many items. us per step with 8 | 16 rows: 22.8 |
// 33.9 at 0.11 M active cells, 98 | 106 at 0.86 M, 199.5 | 199.5 at 2.06 M,
// 318 | 317 at 3.5 M, 1441 | 1387 at 16.5 M.
int band_rows(long long active_cells) { return active_cells >= (2LL << 20) ? 16 : 8; }

cudaError_t launch_band_hulls(const uint8_t* mask, const Layout& L, int rows, int2* out, cudaStream_t st) {
  const int bands = (L.ny + rows - 1) / rows;
  const long long warps = (long long)bands * L.nz;
  band_hulls<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(mask, L, rows, bands, out);
  return cudaGetLastError();
}

void band_list(const Layout& L, int rows, const std::vector<int2>& hulls, std::vector<int4>* items, int* smem) {
  const int bands = (L.ny + rows - 1) / rows;
  items->clear();
  int top = 0;
  for (int k = 0; k < L.nz; ++k)
    for (int b = 0; b < bands; ++b) {
      const int2 h = hulls[(size_t)k * bands + b];
      const int width = h.y - h.x, r = std::min(rows, L.ny - b * rows);
      if (width <= 0) continue;
      const int segs = (width + kBandCols - 1) / kBandCols, w = (width + segs - 1) / segs;
      for (int i = h.x; i < h.y; i += w) {
        const int wi = std::min(w, h.y - i);
        items->push_back(make_int4(k, b * rows, i, wi | (r << 16)));
        top = std::max(top, band_doubles(r, wi));
      }
    }
  *smem = top * (int)sizeof(double);
}

cudaError_t launch_band_step(const StepArgs<double>& a, const int4* items, int n, int smem, cudaStream_t st) {
  cudaError_t e;
  if (a.co.ua[0]) {
    e = launch_pdl(band_tm<true>, n, kBThreads, smem, st, a, items);
    if (e == cudaSuccess) e = launch_pdl(band_te<true>, n, kBThreads, smem, st, a, items);
  } else {
    e = launch_pdl(band_tm<false>, n, kBThreads, smem, st, a, items);
    if (e == cudaSuccess) e = launch_pdl(band_te<false>, n, kBThreads, smem, st, a, items);
  }
  return e;
}

}  // namespace tetm
