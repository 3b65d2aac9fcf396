// Float32 step of a small grid in two launches, one per half (Sec. 4.2, Eq.
// (23)): the TM half (U1..U5) of every plane, then the TE half (U6..U10).
//
// What bounds it: latency. The block-tiled sweep (kernels_slab.cu) computes the
// TM half of the plane below each chunk again and runs 4 planes at least one
// after the other, 10.3 us a step however small the grid. A half reads the
// other's results from memory instead, so planes are independent: an item is
// 56 x 14 nodes of a run of planes, as short as one, in the shortest case two
// memory round trips per launch. Two launches move 64 bytes of fields per node
// instead of 48, which a grid that fits the L2 does not notice; on large ones
// the sweep is faster (the rule is at build_half in capi.cu).
// A thread holds two rows of four columns (64 x 16 loaded, 128 threads, four
// blocks per SM): of the neighbour rows a pair reads, one is its own, so a half
// exchanges two rows per pair through shared memory, with two block barriers
// per plane. e_x, e_y (new h_x, h_y) of the plane above (below) are carried
// along the run. Per node the operations and their order are those of the other
// step kernels, so the results are the same bits.
// Measured per step, sweep -> halves: 24 x 24 x 96 pipe 10.3 -> 4.7 us, 48 x
// 48 x 192 cavity 10.3 -> 5.2, 56 x 56 x 224 pipe 12.3 -> 7.9 (runs of two), 72
// x 72 x 300 pipe 20.5 -> 14.7 (four), 96 x 96 x 384 pipe 28.8 -> 31.8, 256 x
// 256 x 1024 collimator 200 -> 273. Five blocks of 96 registers spill in the TE
// half: 5.9 on 48 x 48 x 192; 8 loaded rows: the same times, more halo. Inputs
// loaded a plane ahead spill or halve the blocks: 6.9.
#include <algorithm>

#include "quads.cuh"
#include "tetm_internal.h"

namespace tetm {
namespace {

constexpr int kRows = kHalfY + 2;            // loaded rows; columns: 64
constexpr int kThreads = 16 * kRows / 2;     // 128
constexpr int kPad = (kRows / 2 + 2) * 16;   // quads of an exchange buffer, one row of them spare at each end

// A thread's part of a work item: its pair of rows, columns gi .. gi + 3.
struct HalfItem {
  int k0, k1;          // planes
  int gi, gj;          // node of the quad's first column, first row
  bool in[2], own[2];  // the row's quad lies inside the arrays; its tile owns it
  long long off;       // layout index of (gi, gj, k0)
};

__device__ __forceinline__ HalfItem half_item(const StepArgs<float>& a, int item, int run, int q, int rp) {
  HalfItem t;
  const int tx = (a.L.nx + kHalfX - 1) / kHalfX, ty = (a.L.ny + kHalfY - 1) / kHalfY, nt = tx * ty;
  const int tile = item % nt;
  t.k0 = item / nt * run;
  t.k1 = min(t.k0 + run, a.L.nz);
  t.gi = tile % tx * kHalfX - 4 + 4 * q;
  t.gj = tile / tx * kHalfY - 1 + 2 * rp;
  const bool inx = t.gi + a.L.ox + 4 <= a.L.px;
  const bool qx = q >= 1 && q <= 14;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int b = 2 * rp + r;
    t.in[r] = inx && t.gj + r < a.L.ny + 2;
    t.own[r] = qx && b >= 1 && b <= kHalfY && t.gj + r < a.L.ny;
  }
  t.off = (long long)(t.k0 + 1) * a.L.sz + (long long)(t.gj + 2) * a.L.px + t.gi + a.L.ox;
  return t;
}

// component c's coefficient of the quad's entries that carry it, else zero
__device__ __forceinline__ P4 coq(unsigned w, int c, float u) {
  auto at = [&](int e) { return (w & (1u << (8 * e + c))) ? u : 0.f; };
  return P4{pk(at(0), at(1)), pk(at(2), at(3))};
}

// entry (row r, column e) of a pair of quads, without an indexed register array
__device__ __forceinline__ float pick(const P4 (&v)[2], int r, int e) {
  const P4 q = r ? v[1] : v[0];
  const f2 h = e < 2 ? q.a : q.b;
  return e & 1 ? hi(h) : lo(h);
}

// TM half (U1..U5): owned rows 1 .. kHalfY of the box. What a neighbour row or
// column outside the box would give is whatever lies there; it reaches one node
// in, never an owned one (e_z of the row above the box is loaded).
__global__ void __launch_bounds__(kThreads, kHalfBlocks) half_tm(const StepArgs<float> a, const int* __restrict__ items, int run) {
  __shared__ float4 xs[2 * kPad];
  const int q = threadIdx.x & 15, rp = threadIdx.x >> 4;
  float* const x1 = reinterpret_cast<float*>(xs) + ((rp + 1) * 16 + q) * 4;
  float* const x2 = x1 + 4 * kPad;
  const HalfItem t = half_item(a, items[blockIdx.x], run, q, rp);
  const long long SZ = a.L.sz, PX = a.L.px;
  const float uHX = a.co.u[kHX], uHY = a.co.u[kHY], uEZ = a.co.u[kEZ];
  const uint8_t* mk = a.co.mask + t.off;
  unsigned w[2], wn[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    w[r] = ld_word_if(mk + r * PX, t.in[r]);
    wn[r] = ld_word_if(mk + r * PX + SZ, t.in[r]);
  }
  // the row above the pair, for e_z there
  const bool inu = t.in[1] && t.gj + 2 < a.L.ny + 2;
  unsigned wu = ld_word_if(mk + 2 * PX, inu);
  long long g = t.off;
  pdl_trigger();
  pdl_wait();
  P4 ex[2], ey[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    ex[r] = ldg_if(a.in[kEX] + g + r * PX, hw(w[r], kEX));
    ey[r] = ldg_if(a.in[kEY] + g + r * PX, hw(w[r], kEY));
  }
  // the pair holds the bunch line node (one thread of the owning tile, and halo ones)
  const bool line = a.b.on && t.gj <= a.b.j0 && t.gj + 1 >= a.b.j0 && a.b.i0 >= t.gi && a.b.i0 < t.gi + 4;
  for (int k = t.k0; k < t.k1; ++k) {
    P4 ez[2], hx[2], hy[2], dex[2], dey[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const P4 x1n = ldg_if(a.in[kEX] + g + SZ + r * PX, hw(wn[r], kEX));
      const P4 y1n = ldg_if(a.in[kEY] + g + SZ + r * PX, hw(wn[r], kEY));
      ez[r] = ldg_if(a.in[kEZ] + g + r * PX, hw(w[r], kEZ));
      hx[r] = ldg_if(a.in[kHX] + g + r * PX, hw(w[r], kHX));
      hy[r] = ldg_if(a.in[kHY] + g + r * PX, hw(w[r], kHY));
      dex[r] = x1n;
      dey[r] = y1n;
    }
    const P4 ezu = ldg_if(a.in[kEZ] + g + 2 * PX, hw(wu, kEZ));
    unsigned w2[2] = {0u, 0u}, wu2 = 0u;
    if (k + 1 < t.k1) {
#pragma unroll
      for (int r = 0; r < 2; ++r) w2[r] = ld_word_if(mk + r * PX + 2 * SZ, t.in[r]);
      wu2 = ld_word_if(mk + 2 * PX + SZ, inu);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const P4 x1n = dex[r], y1n = dey[r];
      dex[r] = sub4(x1n, ex[r]);
      dey[r] = sub4(y1n, ey[r]);
      ex[r] = x1n;
      ey[r] = y1n;
      hx[r] = fma4(coq(w[r], kHX, uHX), sub4(dey[r], sub4(r ? ezu : ez[1], ez[r])), hx[r]);  // U1
      hy[r] = fma4(coq(w[r], kHY, uHY), sub4(diff_right(ez[r]), dex[r]), hy[r]);             // U2
    }
    stp(x1, hx[1]);
    __syncthreads();
    const P4 hxd = ldp(x1 - 64);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      P4 cur = sub4(sub4(r ? hx[0] : hxd, hx[r]), diff_left(hy[r]));
      if (line && t.gj + r == a.b.j0) {
        const long long dd = (long long)k - (a.n + a.b.kshift) + a.b.c0;
        if (dd >= -a.b.c0 && dd < a.b.c0) {
          const float jj = a.b.J[dd + a.b.c0];
          const int e = a.b.i0 - t.gi;
          cur = sub4(cur, P4{pk(e == 0 ? jj : 0.f, e == 1 ? jj : 0.f), pk(e == 2 ? jj : 0.f, e == 3 ? jj : 0.f)});
        }
      }
      ez[r] = fma4(coq(w[r], kEZ, uEZ), cur, ez[r]);                                          // U3
    }
    stp(x2, ez[0]);
    __syncthreads();
    const P4 eznu = ldp(x2 + 64);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      hx[r] = fma4(coq(w[r], kHX, uHX), sub4(dey[r], sub4(r ? eznu : ez[1], ez[r])), hx[r]);  // U4
      hy[r] = fma4(coq(w[r], kHY, uHY), sub4(diff_right(ez[r]), dex[r]), hy[r]);              // U5
      const unsigned ms = t.own[r] ? w[r] : 0u;
      stg_if(a.out[kEZ] + g + r * PX, ez[r], hw(ms, kEZ));
      stg_if(a.out[kHX] + g + r * PX, hx[r], hw(ms, kHX));
      stg_if(a.out[kHY] + g + r * PX, hy[r], hw(ms, kHY));
      if (line && t.own[r] && t.gj + r == a.b.j0 && a.b.i0 < a.L.nx) {
        const int e = a.b.i0 - t.gi;
        add_wake(a.b, (a.n + a.b.kshift) - k - a.b.c0,
                 e == 0 ? lo(ez[r].a) : e == 1 ? hi(ez[r].a) : e == 2 ? lo(ez[r].b) : hi(ez[r].b));
      }
      w[r] = wn[r];
      wn[r] = w2[r];
    }
    wu = wu2;
    g += SZ;
    mk += SZ;
  }
}

// TE half (U6..U10), the mirror image; it reads the new h_x, h_y of its planes
// and of the plane below, which half_tm has written, and gathers the observer
// line's transverse wake, whose old e_x, e_y and new h_x, h_y it holds.
__global__ void __launch_bounds__(kThreads, kHalfBlocks) half_te(const StepArgs<float> a, const int* __restrict__ items, int run) {
  __shared__ float4 xs[2 * kPad];
  const int q = threadIdx.x & 15, rp = threadIdx.x >> 4;
  float* const x1 = reinterpret_cast<float*>(xs) + ((rp + 1) * 16 + q) * 4;
  float* const x2 = x1 + 4 * kPad;
  const HalfItem t = half_item(a, items[blockIdx.x], run, q, rp);
  const long long SZ = a.L.sz, PX = a.L.px;
  const float uEX = a.co.u[kEX], uEY = a.co.u[kEY], uHZ = a.co.u[kHZ];
  const uint8_t* mk = a.co.mask + t.off;
  unsigned w[2], wp[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    wp[r] = ld_word_if(mk + r * PX - SZ, t.in[r]);
    w[r] = ld_word_if(mk + r * PX, t.in[r]);
  }
  // the row below the pair, for h_z there
  unsigned wd = ld_word_if(mk - PX, t.in[0]);
  long long g = t.off;
  pdl_trigger();
  pdl_wait();
  P4 hxp[2], hyp[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    hxp[r] = ldg_if(a.out[kHX] + g - SZ + r * PX, hw(wp[r], kHX));
    hyp[r] = ldg_if(a.out[kHY] + g - SZ + r * PX, hw(wp[r], kHY));
  }
  const int orow = a.b.obs_j - t.gj, ocol = a.b.obs_i - t.gi;
  const bool obs = a.b.obs_on && ocol >= 0 && ocol < 4 && ((orow == 0 && t.own[0]) || (orow == 1 && t.own[1]));
  for (int k = t.k0; k < t.k1; ++k) {
    P4 hz[2], ex[2], ey[2], dhx[2], dhy[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      dhx[r] = ldg_if(a.out[kHX] + g + r * PX, hw(w[r], kHX));
      dhy[r] = ldg_if(a.out[kHY] + g + r * PX, hw(w[r], kHY));
      hz[r] = ldg_if(a.in[kHZ] + g + r * PX, hw(w[r], kHZ));
      ex[r] = ldg_if(a.in[kEX] + g + r * PX, hw(w[r], kEX));
      ey[r] = ldg_if(a.in[kEY] + g + r * PX, hw(w[r], kEY));
    }
    const P4 hzd = ldg_if(a.in[kHZ] + g - PX, hw(wd, kHZ));
    unsigned w2[2] = {0u, 0u}, wd2 = 0u;
    if (k + 1 < t.k1) {
#pragma unroll
      for (int r = 0; r < 2; ++r) w2[r] = ld_word_if(mk + r * PX + SZ, t.in[r]);
      wd2 = ld_word_if(mk - PX + SZ, t.in[0]);
    }
    if (obs) {
      gather_wx(a.b, a.n, k, pick(ex, orow, ocol), pick(dhy, orow, ocol));
      gather_wy(a.b, a.n, k, pick(ey, orow, ocol), pick(dhx, orow, ocol));
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const P4 hxn = dhx[r], hyn = dhy[r];
      dhx[r] = sub4(hxp[r], hxn);
      dhy[r] = sub4(hyp[r], hyn);
      hxp[r] = hxn;
      hyp[r] = hyn;
      ex[r] = fma4(coq(w[r], kEX, uEX), sub4(dhy[r], sub4(r ? hz[0] : hzd, hz[r])), ex[r]);  // U6
      ey[r] = fma4(coq(w[r], kEY, uEY), sub4(diff_left(hz[r]), dhx[r]), ey[r]);              // U7
    }
    stp(x1, ex[0]);
    __syncthreads();
    const P4 exu = ldp(x1 + 64);
#pragma unroll
    for (int r = 0; r < 2; ++r)
      hz[r] = fma4(coq(w[r], kHZ, uHZ), sub4(sub4(r ? exu : ex[1], ex[r]), diff_right(ey[r])), hz[r]);  // U8
    stp(x2, hz[1]);
    __syncthreads();
    const P4 hznd = ldp(x2 - 64);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      ex[r] = fma4(coq(w[r], kEX, uEX), sub4(dhy[r], sub4(r ? hz[0] : hznd, hz[r])), ex[r]);  // U9
      ey[r] = fma4(coq(w[r], kEY, uEY), sub4(diff_left(hz[r]), dhx[r]), ey[r]);               // U10
      const unsigned ms = t.own[r] ? w[r] : 0u;
      stg_if(a.out[kHZ] + g + r * PX, hz[r], hw(ms, kHZ));
      stg_if(a.out[kEX] + g + r * PX, ex[r], hw(ms, kEX));
      stg_if(a.out[kEY] + g + r * PX, ey[r], hw(ms, kEY));
      w[r] = w2[r];
    }
    wd = wd2;
    g += SZ;
    mk += SZ;
  }
}

}  // namespace

cudaError_t launch_half_step(const StepArgs<float>& a, const int* items, int n, int run, cudaStream_t st) {
  cudaError_t e = launch_pdl(half_tm, n, kThreads, 0, st, a, items, run);
  if (e == cudaSuccess) e = launch_pdl(half_te, n, kThreads, 0, st, a, items, run);
  return e;
}

}  // namespace tetm
