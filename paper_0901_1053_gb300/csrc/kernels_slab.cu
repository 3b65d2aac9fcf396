// Block-tiled fused step, float32 (Sec. 4.2, Eq. (23)).
//
// Two CTAs of 256 threads per SM take (tile, z chunk) work items in turn. A
// tile owns 56 x 12 nodes and loads 64 x 16 (4 halo columns and 2 halo rows on
// each side: the ten updates reach two nodes sideways), so one CTA's barriers
// and copy waits overlap the other's work. Thread t holds the four consecutive
// columns 4 (t mod 16) .. +3 of row t / 16 (a quad), so its loads and stores
// are 16-byte vectors, and marches through the chunk plane by plane with the
// z-state of its quad in registers (old e_x, e_y, new h_x, h_y of the planes
// below): no per-row state in shared memory.
//
// What bounds it: latency behind the block barriers at 16 warps per SM. No pipe
// is full: on 256 x 256 x 512 L1/TEX is at 58% (its shared-memory and
// load/store data pipe 51), DRAM 55, SM 46, and of a warp's 7.4 cycles per
// issued instruction 1.9 are a barrier, 1.0 global loads, 0.9 shared memory, 0.5
// the arithmetic pipes. With one material on 256 x 256 x 2048 a step takes 395
// us, of which the arithmetic and barriers alone take 209 us, and all inputs
// from L2 instead of DRAM 373 us. Tried on the way (us
// per step on 256 x 256 x 1024 / 2048 and on a 16-solve batch's longest
// solve): one CTA of 512 threads on 64 x 32 boxes in scalar arithmetic 225 /
// 402 / 534; the same with packed pairs of float32 (half the issue slots for
// the same roundings) 210 / 394 / 582; 64 x 16 boxes in two CTAs, packed, 204 /
// 395 / 476 and 32.8 instead of 54.7 on 48 x 48 x 192, where a grid of few
// tiles makes 2.3 times the items. The rows loaded in vain (4 of 16 instead of
// 4 of 32) cost less than the waits of a lone CTA. A ring for all six inputs
// instead of register loads, and tensor-map copies into it, were slower (more
// shared-memory reads between the same barriers), and so were later loads of
// e_x, e_y (238 us), a sweep unrolled by three planes (264 us: code size) and
// one that gathers the transverse wake itself (1.3 us more, the launch 1.5 less
// only on small grids). With coefficient arrays packed pairs save nothing (192 x
// 192 x 768, a quarter open: 151.4 against 148.8 us).
//
// Only entries that carry a field move through the per-thread loads and
// stores. Each thread reads the activity bytes of its quad (one 32-bit word
// per plane, a few planes ahead) and
//  * loads h_x, h_y, e_x, e_y of the quad (16-byte loads one plane ahead) only
//    when one of its four nodes carries that component, else takes zero (an
//    entry without a field holds zero for ever);
//  * stores each new component of the quad only when one of its nodes
//    carries it (the other field set's entry already holds that zero).
// e_z and h_z are the inputs a node reads at its neighbours; they (and with
// material arrays the six per-entry coefficient arrays, read at the node)
// arrive through rings of two planes in shared memory: each thread copies its
// own quad of every array into the slot with a 16-byte asynchronous copy, or
// writes zeros without a read where none of the quad's nodes carries that
// component (an entry without a field, and its coefficient, hold zero), so the
// rings read no pipe wall. Completion by the thread's copy group, publication
// by a block barrier.
//
// The intermediates a stage reads one row up or down (hx~, ez', ex~, hz') go
// through shared-memory buffers, those one column left or right through warp
// shuffles. Six stages per plane:
//   S1 hx~, hy~ (U1, U2)  | S2 ez' (U3, + current) | S3 hx', hy' (U4, U5)
//   S4 ex~, ey~ (U6, U7)  | S5 hz' (U8)            | S6 ex', ey' (U9, U10)
// With one material they run plane by plane, a block barrier after S1, S2,
// S4 and S5 (two buffers). With coefficient arrays the sweep is skewed by half
// a step: iteration i runs S1..S3 of plane i+1 (the TM half reads only old
// fields) beside S4..S6 of plane i (the TE half reads the new h_x, h_y of
// planes i and i-1), as pairs A = S1|S4, B = S2|S5, C = S3|S6 with a barrier
// after A and after B (four buffers: C reads what B wrote, and the next A
// writes only buffers that other threads last read in B); the copies then
// have two planes of work to land. (The skew costs the one-material sweep more
// instructions than its barriers do: its coefficients come from the activity
// words, and a third plane of e_x, e_y rides in registers.) Per node the
// arithmetic and its order are the same in both, so the results are the same
// bits.
// The column of i = 0 sits at 8 in the float32 layout, so the 224-byte rows a
// tile writes start and end on 32-byte sectors and no two tiles write into
// the same sector.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "quads.cuh"
#include "tetm_internal.h"

namespace tetm {

namespace {

constexpr int kSX = 64, kSY = 16;    // loaded columns, rows
constexpr int kOX = 56, kOY = 12;    // owned columns, rows
constexpr int kQ = kSX / 4;          // column quads per row
constexpr int kSThreads = kQ * kSY;  // 256
constexpr int kNamedY = 28;          // tetm_set_tiling names the one-material shape 56 x 28, the other 56 x 12

// One material: a two-plane ring of e_z and h_z (one coefficient per
// component, switched by the activity bytes) and two exchange buffers, laid
// out in one array with a spare row at the end, so that a read one row or
// one column past a buffer's edge stays inside it (see slab_item).
struct SlabSmemU {
  static constexpr int SD = 2;             // planes in the ring (the next plane lands while this one is worked on)
  static constexpr int kP = kSY * kSX;     // one box plane
  float f[(2 * SD + 2) * kP + kSX];        // e_z slots, h_z slots, x1, x2, spare row
  int next[2];                             // the CTA's next work item (dynamic schedule)
  __device__ __forceinline__ float* ez(int s) { return f + s * kP; }
  __device__ __forceinline__ float* hz(int s) { return f + (SD + s) * kP; }
  __device__ __forceinline__ float* x1() { return f + 2 * SD * kP; }
  __device__ __forceinline__ float* x2() { return f + (2 * SD + 1) * kP; }
};
// Material arrays: two-plane rings of e_z and h_z with the six per-entry
// coefficient arrays (alpha M^-1, 2 alpha M^-1 for e_z and h_z), and the four
// exchange buffers of the skewed sweep (hx~, ez', ex~, hz'), 82 KB, in one
// array with a spare row at the end (reads past a buffer's edge stay inside).
struct SlabSmemM {
  static constexpr int kP = kSY * kSX;
  float f[20 * kP + kSX];  // e_z slots (2), h_z slots (2), 2 x 6 coefficient planes, x1..x4, spare row
  int next[2];
  __device__ __forceinline__ float* ez(int s) { return f + s * kP; }
  __device__ __forceinline__ float* hz(int s) { return f + (2 + s) * kP; }
  __device__ __forceinline__ float* co(int s, int c) { return f + (4 + 6 * s + c) * kP; }
  __device__ __forceinline__ float* x(int b) { return f + (15 + b) * kP; }  // b = 1..4: planes 16..19
};
template <bool MAT>
using SlabSmem = typename std::conditional<MAT, SlabSmemM, SlabSmemU>::type;


// 16 bytes into shared memory by an asynchronous copy, or (c false) 16 zero
// bytes without a global read
__device__ __forceinline__ void cp16_or_zero(void* sdst, const void* gsrc, bool c) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(su32(sdst)), "l"(gsrc), "r"(c ? 16u : 0u)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
struct Q4 {
  float v[4];
};
__device__ __forceinline__ Q4 q4(float4 a) { return Q4{{a.x, a.y, a.z, a.w}}; }
__device__ __forceinline__ Q4 ld4_if(const float* p, unsigned c) {
  Q4 r;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n mov.f32 %0, 0f00000000;\n mov.f32 %1, 0f00000000;\n"
      " mov.f32 %2, 0f00000000;\n mov.f32 %3, 0f00000000;\n"
      " @q ld.global.v4.f32 {%0,%1,%2,%3}, [%4];\n}"
      : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3])
      : "l"(p), "r"(c));
  return r;
}
__device__ __forceinline__ void st4_if(float* p, const Q4& v, unsigned c) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q st.global.v4.f32 [%0], {%1,%2,%3,%4};\n}" ::"l"(p),
               "f"(v.v[0]), "f"(v.v[1]), "f"(v.v[2]), "f"(v.v[3]), "r"(c)
               : "memory");
}
__device__ __forceinline__ Q4 lds4(const float* p) { return q4(*reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void sts4(float* p, const Q4& a) {
  *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}

// One (tile, z-chunk) work item of solve a with one material (the ten
// updates of every plane of the chunk, plane by plane: four block barriers
// per plane). SHARED: a lies in shared memory (batches) instead of the
// parameter space. There each array's address is its set's pointer, kept in
// registers, plus a multiple of cstep: the twelve pointers were a shared-memory
// read each in every plane, ahead of the access that needs it (batch of 16
// solves: 558 us per step of the longest, so 476). From the
// parameter space the twelve pointers are free, and one running pointer per
// set was measured 1.7 times slower.
//
// The reads of a neighbour one row or column outside the 64 x 16 box take
// whatever the neighbouring shared-memory words or lanes hold, without an
// edge test. Each of the six stages reaches one node sideways, and a value
// computed from an outside neighbour is wrong only on the box's outermost
// row or column; through the stages that error reaches at most two rows and
// two columns in, all of them halo (the tile owns rows 2..13 and columns
// 4..59 of the box), and halo nodes are never stored.
template <bool SHARED>
__device__ __forceinline__ void slab_item(const StepArgs<float>& a, int item, SlabSmemU& S) {
  constexpr int kSD = SlabSmemU::SD;
  const int tid = threadIdx.x, q = tid % kQ, row = tid / kQ;
  const Layout L = a.L;
  const long long SZ = L.sz, PX = L.px;
  const float uEX = a.co.u[kEX], uEY = a.co.u[kEY], uEZ = a.co.u[kEZ];
  const float uHX = a.co.u[kHX], uHY = a.co.u[kHY], uHZ = a.co.u[kHZ];
  const int ntile = a.tiles_x * a.tiles_y;
  const P4 zero{0ull, 0ull};
  const float* const in0 = a.in[0];
  float* const out0 = a.out[0];
  const uint8_t* const mask = a.co.mask;
  const unsigned cs = a.cstep;
  auto in_of = [&](int c) -> const float* {
    if constexpr (SHARED)
      return reinterpret_cast<const float*>(reinterpret_cast<const char*>(in0) + (unsigned long long)cs * (16u * c));
    else
      return a.in[c];
  };
  auto out_of = [&](int c) -> float* {
    if constexpr (SHARED)
      return reinterpret_cast<float*>(reinterpret_cast<char*>(out0) + (unsigned long long)cs * (16u * c));
    else
      return a.out[c];
  };
  const int tile = item % ntile, chunk = item / ntile;
  const int gx0 = (tile % a.tiles_x) * kOX - 4;  // global i of loaded column 0
  const int gy0 = (tile / a.tiles_x) * kOY - 2;  // global j of loaded row 0
  const int k0 = chunk * a.chunk_z, k1 = min(k0 + a.chunk_z, L.nz);
  const int kstart = k0 - 1;
  const int nplanes = k1 - kstart;
  const int cx = gx0 + L.ox;                   // layout column of loaded column 0

  // this thread's quad; a quad with an active node lies inside its layout
  // row (columns i <= nx + 2 < px - ox), so every predicated access is a
  // whole 16-byte vector (a quad across i = nx stores the zeros its entries
  // past the cells compute: zero input, zero coefficient)
  const int gi = gx0 + 4 * q, gj = gy0 + row;
  const bool inq = gj + 2 < L.ny + 4 && cx + 4 * q + 4 <= PX;  // the quad lies inside the arrays
  const long long qoff = (long long)(gj + 2) * PX + cx + 4 * q;
  const bool own_q = q >= 1 && q <= kQ - 2 && row >= 2 && row < kSY - 2 && gj < L.ny;
  auto gidx = [&](int k) { return (long long)(k + 1) * SZ + qoff; };
  auto word = [&](int k) -> unsigned { return ld_word_if(mask + gidx(k), inq); };
  auto load_if = [&](const float* base, int k, unsigned p) -> P4 { return ldg_if(base + gidx(k), p); };
  // plane k into its slot: each thread copies the quad of its own node row
  // and columns of e_z, h_z, only where one of the quad's nodes carries that
  // component (zeros otherwise: the entry holds zero), so the ring reads no
  // pipe wall; completion by the thread's copy group and the block barrier
  // after it
  auto issue_q = [&](int k, unsigned mw) {
    const int s = (k - kstart) % kSD;
    const long long g = inq ? gidx(k) : 0;
    cp16_or_zero(S.ez(s) + row * kSX + 4 * q, in_of(kEZ) + g, has(mw, kEZ));
    cp16_or_zero(S.hz(s) + row * kSX + 4 * q, in_of(kHZ) + g, has(mw, kHZ));
  };
  // activity words of planes k .. k + kSD (m[0] of the plane being worked
  // on; m[kSD] of the plane whose copy is issued next); z-state and the
  // register prefetch (plane k: hx, hy of k; ex, ey of k+1)
  unsigned m[kSD + 1];
#pragma unroll
  for (int i = 0; i <= kSD; ++i) m[i] = kstart + i <= k1 ? word(kstart + i) : 0u;
#pragma unroll
  for (int i = 0; i < kSD; ++i) {
    if (i < nplanes) issue_q(kstart + i, m[i]);
    cp_commit();
  }
  cp_wait<kSD - 1>();
  __syncthreads();  // plane kstart's slot is in
  P4 ex0 = load_if(in_of(kEX), kstart, hw(m[0], kEX)), ey0 = load_if(in_of(kEY), kstart, hw(m[0], kEY));
  P4 hxc = load_if(in_of(kHX), kstart, hw(m[0], kHX)), hyc = load_if(in_of(kHY), kstart, hw(m[0], kHY));
  P4 ex1 = load_if(in_of(kEX), kstart + 1, hw(m[1], kEX)), ey1 = load_if(in_of(kEY), kstart + 1, hw(m[1], kEY));
  P4 hxp = zero, hyp = zero;
  const bool line_row = a.b.on && gj == a.b.j0;
  const bool line_q = line_row && a.b.i0 >= gi && a.b.i0 < gi + 4;  // the quad holds the bunch line node

  for (int k = kstart; k < k1; ++k) {
    const int s = (k - kstart) % kSD;
    // next plane's register inputs and the activity word kSD + 1 planes on, early
    P4 hxn_in, hyn_in, exn_in, eyn_in;
    unsigned mn = 0u;
    const bool more = k + 1 < k1;
    if (more) {
      hxn_in = load_if(in_of(kHX), k + 1, hw(m[1], kHX));
      hyn_in = load_if(in_of(kHY), k + 1, hw(m[1], kHY));
      exn_in = load_if(in_of(kEX), k + 2, hw(m[2], kEX));
      eyn_in = load_if(in_of(kEY), k + 2, hw(m[2], kEY));
      if (k + kSD + 1 <= k1) mn = word(k + kSD + 1);
    }
    // slot inputs: e_z, h_z of this quad and its neighbours
    const float* sez = S.ez(s) + row * kSX + 4 * q;
    const float* shz = S.hz(s) + row * kSX + 4 * q;
    const P4 ez = ldp(sez);
    const P4 ezU = ldp(sez + kSX);
    const P4 hz = ldp(shz);
    const P4 hzD = ldp(shz - kSX);
    float* const x1 = S.x1() + row * kSX + 4 * q;  // this thread's quad in the exchange buffers
    float* const x2 = S.x2() + row * kSX + 4 * q;
    // one coefficient per component, switched by the activity bytes
    const unsigned w = m[0];
    auto co = [&](int c, float u) {
      auto at = [&](int e) { return (w & (1u << (8 * e + c))) ? u : 0.f; };
      return P4{pk(at(0), at(1)), pk(at(2), at(3))};
    };
    const P4 cHX = co(kHX, uHX), cHY = co(kHY, uHY), cEZ = co(kEZ, uEZ);
    const P4 cEX = co(kEX, uEX), cEY = co(kEY, uEY), cHZ = co(kHZ, uHZ);
    const P4 dey = sub4(ey1, ey0), dex = sub4(ex1, ex0);
    const P4 hxa = fma4(cHX, sub4(dey, sub4(ezU, ez)), hxc);        // U1
    const P4 hya = fma4(cHY, sub4(diff_right(ez), dex), hyc);       // U2
    stp(x1, hxa);
    __syncthreads();  // (1) the slot is read and hx~ is out
    if (k + kSD < k1) issue_q(k + kSD, m[kSD]);  // into the freed slot
    cp_commit();
    // S2: ez' = ez + 2a M^-1 (P_y^T hx~ - P_x^T hy~ - jj_z)
    P4 cur = sub4(sub4(ldp(x1 - kSX), hxa), diff_left(hya));
    if (line_q) {  // the bunch current on its line (one quad of a tile row)
      const long long dd = (long long)k - (a.n + a.b.kshift) + a.b.c0;
      if (dd >= -a.b.c0 && dd < a.b.c0) {
        const float jj = a.b.J[dd + a.b.c0];
        const int e = a.b.i0 - gi;
        cur = sub4(cur, P4{pk(e == 0 ? jj : 0.f, e == 1 ? jj : 0.f), pk(e == 2 ? jj : 0.f, e == 3 ? jj : 0.f)});
      }
    }
    const P4 ezn = fma4(cEZ, cur, ez);                              // U3
    stp(x2, ezn);
    __syncthreads();  // (2)
    // S3: hx', hy'
    const P4 hxn = fma4(cHX, sub4(dey, sub4(ldp(x2 + kSX), ezn)), hxa);  // U4
    const P4 hyn = fma4(cHY, sub4(diff_right(ezn), dex), hya);           // U5
    const bool st = k >= k0 && own_q;
    const unsigned ms = st ? m[0] : 0u;  // the plane's word where this thread stores
    stg_if(out_of(kEZ) + gidx(k), ezn, hw(ms, kEZ));
    stg_if(out_of(kHX) + gidx(k), hxn, hw(ms, kHX));
    stg_if(out_of(kHY) + gidx(k), hyn, hw(ms, kHY));
    if (st && line_q && a.b.i0 < L.nx) {
      const int e = a.b.i0 - gi;  // the quad's entry on the bunch line (no indexed register array)
      add_wake(a.b, (a.n + a.b.kshift) - k - a.b.c0,
               e == 0 ? lo(ezn.a) : e == 1 ? hi(ezn.a) : e == 2 ? lo(ezn.b) : hi(ezn.b));
    }
    // S4: ex~, ey~ with the new hx, hy of this plane and of the plane below
    const P4 dhy = sub4(hyp, hyn), dhx = sub4(hxp, hxn);
    const P4 exa = fma4(cEX, sub4(dhy, sub4(hzD, hz)), ex0);        // U6
    const P4 eya = fma4(cEY, sub4(diff_left(hz), dhx), ey0);        // U7
    stp(x1, exa);
    __syncthreads();  // (3)
    // S5: hz'
    const P4 hzn = fma4(cHZ, sub4(sub4(ldp(x1 + kSX), exa), diff_right(eya)), hz);  // U8
    stp(x2, hzn);
    cp_wait<kSD - 1>();  // this thread's copies of the next plane are in
    __syncthreads();  // (4) (and the next plane's slot is in)
    // S6: ex', ey'
    const P4 exn = fma4(cEX, sub4(dhy, sub4(ldp(x2 - kSX), hzn)), exa);  // U9
    const P4 eyn = fma4(cEY, sub4(diff_left(hzn), dhx), eya);            // U10
    stg_if(out_of(kEX) + gidx(k), exn, hw(ms, kEX));
    stg_if(out_of(kEY) + gidx(k), eyn, hw(ms, kEY));
    stg_if(out_of(kHZ) + gidx(k), hzn, hw(ms, kHZ));
    // carry the z-state, take the prefetched inputs
    hxp = hxn;
    hyp = hyn;
    ex0 = ex1;
    ey0 = ey1;
#pragma unroll
    for (int i = 0; i < kSD; ++i) m[i] = m[i + 1];
    m[kSD] = mn;
    if (more) {
      hxc = hxn_in;
      hyc = hyn_in;
      ex1 = exn_in;
      ey1 = eyn_in;
    }
  }
  cp_wait<0>();
  __syncthreads();  // every thread is done with the ring before the next item refills it
}

// One (tile, z-chunk) work item of solve a with per-entry coefficient
// arrays, skewed by half a step: iteration i runs the TM half of plane i+1
// (U1..U5, which reads only old fields) beside the TE half of plane i
// (U6..U10, which reads the new h_x, h_y of planes i and i-1), two block
// barriers per iteration. Neighbour reads past the box edge go without edge
// tests, as in slab_item (the two-node halo absorbs what they return).
__device__ __forceinline__ void slab_item_mat(const StepArgs<float>& a, int item, SlabSmemM& S) {
  const int tid = threadIdx.x, q = tid % kQ, row = tid / kQ;
  const Layout L = a.L;
  const long long SZ = L.sz, PX = L.px;
  const int ntile = a.tiles_x * a.tiles_y;
  const Q4 zero{{0.f, 0.f, 0.f, 0.f}};
  const int tile = item % ntile, chunk = item / ntile;
  const int gx0 = (tile % a.tiles_x) * kOX - 4;  // global i of loaded column 0
  const int gy0 = (tile / a.tiles_x) * kOY - 2;  // global j of loaded row 0
  const int k0 = chunk * a.chunk_z, k1 = min(k0 + a.chunk_z, L.nz);
  const int kstart = k0 - 1;                   // the plane below the chunk: its new h_x, h_y feed U6, U7 of k0
  const int cx = gx0 + L.ox;                   // layout column of loaded column 0

  // this thread's quad; a quad with an active node lies inside its layout
  // row (columns i <= nx + 2 < px - ox), so every predicated access is a
  // whole 16-byte vector (a quad across i = nx stores the zeros its entries
  // past the cells compute: zero input, zero coefficient)
  const int gi = gx0 + 4 * q, gj = gy0 + row;
  const bool inq = gj + 2 < L.ny + 4 && cx + 4 * q + 4 <= PX;  // the quad lies inside the arrays
  const long long qoff = (long long)(gj + 2) * PX + cx + 4 * q;
  const bool own_q = q >= 1 && q <= kQ - 2 && row >= 2 && row < kSY - 2 && gj < L.ny;
  const int qo = row * kSX + 4 * q;  // this thread's quad in a box plane
  float* const x1 = S.x(1) + qo;     // and in the exchange buffers
  float* const x2 = S.x(2) + qo;
  float* const x3 = S.x(3) + qo;
  float* const x4 = S.x(4) + qo;
  auto gidx = [&](int k) { return (long long)(k + 1) * SZ + qoff; };
  auto word = [&](int k) -> unsigned { return ld_word_if(a.co.mask + gidx(k), inq); };
  auto load_if = [&](const float* base, int k, unsigned p) -> Q4 { return ld4_if(base + gidx(k), p); };
  // e_z of plane k with the coefficient arrays of h_x, h_y, e_z (the TM
  // half), h_z of plane k with those of e_x, e_y, h_z (the TE half), into
  // their slots: each thread copies the quads of its own
  // node row and columns, only where one of the quad's nodes carries that
  // component (zeros otherwise: the entry and its coefficient hold zero), so
  // the ring reads no pipe wall; completion by the thread's copy group and
  // the block barrier after it
  auto issue_ez = [&](int k, unsigned mw) {
    const int s = (k - kstart) & 1;
    const long long g = inq ? gidx(k) : 0;
    const int o = row * kSX + 4 * q;
    cp16_or_zero(S.ez(s) + o, a.in[kEZ] + g, has(mw, kEZ));
    cp16_or_zero(S.co(s, kHX) + o, a.co.ua[kHX] + g, has(mw, kHX));
    cp16_or_zero(S.co(s, kHY) + o, a.co.ua[kHY] + g, has(mw, kHY));
    cp16_or_zero(S.co(s, kEZ) + o, a.co.ua[kEZ] + g, has(mw, kEZ));
  };
  auto issue_hz = [&](int k, unsigned mw) {
    const int s = (k - kstart) & 1;
    const long long g = inq ? gidx(k) : 0;
    const int o = row * kSX + 4 * q;
    cp16_or_zero(S.hz(s) + o, a.in[kHZ] + g, has(mw, kHZ));
    cp16_or_zero(S.co(s, kEX) + o, a.co.ua[kEX] + g, has(mw, kEX));
    cp16_or_zero(S.co(s, kEY) + o, a.co.ua[kEY] + g, has(mw, kEY));
    cp16_or_zero(S.co(s, kHZ) + o, a.co.ua[kHZ] + g, has(mw, kHZ));
  };
  // Iteration i works on the TM half of plane i+1 and the TE half of plane
  // i; m[j] is the activity word of plane i + j. The ring holds e_z of
  // planes i+1, i+2 and h_z of planes i, i+1; after the first barrier the
  // slots read in A take e_z of i+3 and h_z of i+2 (two planes of work to
  // land). Registers: old e_x, e_y of planes i, i+1, i+2 (exA, exB, exC),
  // old h_x, h_y of plane i+1, new h_x, h_y of planes i (hxn) and i-1 (hxp),
  // and the loads of the next iteration, one iteration ahead.
  unsigned m[4];
  m[0] = 0u;  // plane kstart - 1: no TE half there
#pragma unroll
  for (int j = 1; j < 4; ++j) m[j] = kstart + j - 1 <= k1 ? word(kstart + j - 1) : 0u;
  issue_ez(kstart, m[1]);
  if (kstart + 1 < k1) issue_ez(kstart + 1, m[2]);
  cp_commit();
  Q4 exA = zero, eyA = zero;
  Q4 exB = load_if(a.in[kEX], kstart, hw(m[1], kEX)), eyB = load_if(a.in[kEY], kstart, hw(m[1], kEY));
  Q4 exC = load_if(a.in[kEX], kstart + 1, hw(m[2], kEX)), eyC = load_if(a.in[kEY], kstart + 1, hw(m[2], kEY));
  Q4 hxc = load_if(a.in[kHX], kstart, hw(m[1], kHX)), hyc = load_if(a.in[kHY], kstart, hw(m[1], kHY));
  Q4 hxp = zero, hyp = zero, hxn = zero, hyn = zero;
  const bool line_row = a.b.on && gj == a.b.j0;
  const bool line_q = line_row && a.b.i0 >= gi && a.b.i0 < gi + 4;  // the quad holds the bunch line node
  cp_wait<0>();
  __syncthreads();  // e_z of planes kstart, kstart + 1 is in

  for (int i = kstart - 1; i < k1; ++i) {
    const bool tm = i + 1 < k1;  // the TM half of plane p = i + 1 (block-uniform)
    const bool te = i >= k0;     // the TE half of plane i (block-uniform)
    const int p = i + 1;
    const int se = (p - kstart) & 1, sh = (i - kstart) & 1;
    // the next iteration's register inputs and the activity word four planes on, early
    Q4 hxn_in = zero, hyn_in = zero, exn_in = zero, eyn_in = zero;
    unsigned mn = 0u;
    if (i + 3 <= k1) {
      hxn_in = load_if(a.in[kHX], i + 2, hw(m[2], kHX));
      hyn_in = load_if(a.in[kHY], i + 2, hw(m[2], kHY));
      exn_in = load_if(a.in[kEX], i + 3, hw(m[3], kEX));
      eyn_in = load_if(a.in[kEY], i + 3, hw(m[3], kEY));
      if (i + 4 <= k1) mn = word(i + 4);
    }
    // A warp none of whose quads carries a component in a plane (PEC rows of
    // a tile at the pipe wall) computes nothing there: every value it would
    // compute is zero (an entry without a field and its coefficients hold
    // zero), so it writes zeros where its neighbours read them and keeps to
    // the barriers and the ring.
    const bool wtm = __any_sync(0xffffffffu, m[1] != 0u || line_q);
    const bool wte = __any_sync(0xffffffffu, m[0] != 0u);
    float cHX[4], cHY[4], cEZ[4], cEX[4], cEY[4], cHZ[4];
    // ---- A: S1 of plane p (hx~, hy~: U1, U2) | S4 of plane i (ex~, ey~: U6, U7)
    Q4 ez = zero, hxa = zero, hya = zero;
    if (tm) {
      if (wtm) {
        const float* sez = S.ez(se) + qo;
        ez = lds4(sez);
        const Q4 ezU = lds4(sez + kSX);
        const float ezR = sez[4];
        const Q4 c0 = lds4(S.co(se, kHX) + qo), c1 = lds4(S.co(se, kHY) + qo);
        const Q4 c2 = lds4(S.co(se, kEZ) + qo);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          cHX[e] = c0.v[e];
          cHY[e] = c1.v[e];
          cEZ[e] = c2.v[e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float dey = eyC.v[e] - eyB.v[e], dex = exC.v[e] - exB.v[e];
          const float ezx = e < 3 ? ez.v[e + 1] : ezR;
          hxa.v[e] = hxc.v[e] + cHX[e] * (dey - (ezU.v[e] - ez.v[e]));   // U1
          hya.v[e] = hyc.v[e] + cHY[e] * (-dex + (ezx - ez.v[e]));      // U2
        }
      }
      sts4(x1, hxa);
    }
    Q4 hz = zero, exa = zero, eya = zero;
    if (te) {
      if (wte) {
        const float* shz = S.hz(sh) + qo;
        hz = lds4(shz);
        const Q4 hzD = lds4(shz - kSX);
        const float hzL = shz[-1];
        const Q4 c0 = lds4(S.co(sh, kEX) + qo), c1 = lds4(S.co(sh, kEY) + qo);
        const Q4 c2 = lds4(S.co(sh, kHZ) + qo);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          cEX[e] = c0.v[e];
          cEY[e] = c1.v[e];
          cHZ[e] = c2.v[e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float hzl = e > 0 ? hz.v[e - 1] : hzL;
          exa.v[e] = exA.v[e] + cEX[e] * ((hyp.v[e] - hyn.v[e]) - (hzD.v[e] - hz.v[e]));   // U6
          eya.v[e] = eyA.v[e] + cEY[e] * (-(hxp.v[e] - hxn.v[e]) + (hzl - hz.v[e]));       // U7
        }
      }
      sts4(x3, exa);
    }
    __syncthreads();  // (1) the slots are read; hx~ and ex~ are out
    if (i + 3 < k1) issue_ez(i + 3, m[3]);  // into the freed slots
    if (i + 2 < k1) issue_hz(i + 2, m[2]);
    cp_commit();
    // ---- B: S2 of plane p (ez': U3 with the bunch current) | S5 of plane i (hz': U8)
    Q4 ezn = zero;
    if (tm) {
      if (wtm) {
        const Q4 hxaD = lds4(x1 - kSX);
        const float hyaL = left_any(hya.v[3]);
        float cur[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float hyl = e > 0 ? hya.v[e - 1] : hyaL;
          cur[e] = (hxaD.v[e] - hxa.v[e]) - (hyl - hya.v[e]);
        }
        if (line_q) {  // the bunch current on its line (one quad of a tile row)
          const long long dd = (long long)p - (a.n + a.b.kshift) + a.b.c0;
          if (dd >= -a.b.c0 && dd < a.b.c0) {
            const float jj = a.b.J[dd + a.b.c0];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (gi + e == a.b.i0) cur[e] -= jj;
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) ezn.v[e] = ez.v[e] + cEZ[e] * cur[e];   // U3
      }
      sts4(x2, ezn);
    }
    Q4 hzn = zero;
    if (te) {
      if (wte) {
        const Q4 exaU = lds4(x3 + kSX);
        const float eyaR = right_any(eya.v[0]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float eyx = e < 3 ? eya.v[e + 1] : eyaR;
          hzn.v[e] = hz.v[e] + cHZ[e] * ((exaU.v[e] - exa.v[e]) - (eyx - eya.v[e]));      // U8
        }
      }
      sts4(x4, hzn);
    }
    cp_wait<1>();     // this thread's copies issued one iteration ago are in
    __syncthreads();  // (2) ez' and hz' are out (and the slots the next A reads are in)
    // ---- C: S3 of plane p (hx', hy': U4, U5) | S6 of plane i (ex', ey': U9, U10)
    // (hx~, ez', ex~, hz' of the thread's own quad come back from the
    // exchange buffers rather than stay in registers across the barrier)
    Q4 hxN = zero, hyN = zero;
    if (tm && wtm) {
      const Q4 hxa2 = lds4(x1);
      const Q4 ezn2 = lds4(x2);
      const Q4 eznU = lds4(x2 + kSX);
      const float eznR = right_any(ezn2.v[0]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float dey = eyC.v[e] - eyB.v[e], dex = exC.v[e] - exB.v[e];
        const float ezx = e < 3 ? ezn2.v[e + 1] : eznR;
        hxN.v[e] = hxa2.v[e] + cHX[e] * (dey - (eznU.v[e] - ezn2.v[e]));  // U4
        hyN.v[e] = hya.v[e] + cHY[e] * (-dex + (ezx - ezn2.v[e]));      // U5
      }
      const bool st = p >= k0 && own_q;
      const unsigned ms = st ? m[1] : 0u;
      st4_if(a.out[kEZ] + gidx(p), ezn2, hw(ms, kEZ));
      st4_if(a.out[kHX] + gidx(p), hxN, hw(ms, kHX));
      st4_if(a.out[kHY] + gidx(p), hyN, hw(ms, kHY));
      if (st && line_q && a.b.i0 < L.nx) {
        const int e = a.b.i0 - gi;  // the quad's entry on the bunch line (no indexed register array)
        const float v = e == 0 ? ezn2.v[0] : e == 1 ? ezn2.v[1] : e == 2 ? ezn2.v[2] : ezn2.v[3];
        add_wake(a.b, (a.n + a.b.kshift) - p - a.b.c0, v);
      }
    }
    if (te && wte) {
      const Q4 exa2 = lds4(x3);
      const Q4 hzn2 = lds4(x4);
      const Q4 hznD = lds4(x4 - kSX);
      const float hznL = left_any(hzn2.v[3]);
      Q4 exn, eyn;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float hzl = e > 0 ? hzn2.v[e - 1] : hznL;
        exn.v[e] = exa2.v[e] + cEX[e] * ((hyp.v[e] - hyn.v[e]) - (hznD.v[e] - hzn2.v[e]));   // U9
        eyn.v[e] = eya.v[e] + cEY[e] * (-(hxp.v[e] - hxn.v[e]) + (hzl - hzn2.v[e]));       // U10
      }
      const unsigned ms = own_q ? m[0] : 0u;
      st4_if(a.out[kEX] + gidx(i), exn, hw(ms, kEX));
      st4_if(a.out[kEY] + gidx(i), eyn, hw(ms, kEY));
      st4_if(a.out[kHZ] + gidx(i), hzn2, hw(ms, kHZ));
    }
    // carry the z-state, take the loads made for the next iteration
    hxp = hxn;
    hyp = hyn;
    hxn = hxN;
    hyn = hyN;
    exA = exB;
    eyA = eyB;
    exB = exC;
    eyB = eyC;
    exC = exn_in;
    eyC = eyn_in;
    hxc = hxn_in;
    hyc = hyn_in;
    m[0] = m[1];
    m[1] = m[2];
    m[2] = m[3];
    m[3] = mn;
  }
  cp_wait<0>();
  __syncthreads();  // every thread is done with the ring before the next item refills it
}

template <bool MAT>
__global__ void __launch_bounds__(kSThreads, 2)
    fused_step_slab(const StepArgs<float> a, int* sched) {
  using Smem = SlabSmem<MAT>;
  extern __shared__ __align__(128) unsigned char slab_raw[];
  Smem& S = *reinterpret_cast<Smem*>(slab_raw);
  const int tid = threadIdx.x;
  const int nitems = a.work ? a.n_work : a.tiles_x * a.tiles_y * a.n_chunks;
  // every block is resident at once, so the next launch's start (2 us of 205 per
  // step on 256 x 256 x 1024) hides behind this one's end
  pdl_trigger();
  pdl_wait();

  // Items in list order: the first per CTA by its index, then (with a
  // schedule counter) whichever item is next when the CTA gets free, fetched
  // one item ahead. Items that run at the same time stay neighbours (shared
  // halo rows in L2) and CTAs that drew cheap items (much PEC) take more.
  const int G = gridDim.x;
  int wi = blockIdx.x, par = 0;
  while (wi < nitems) {
    if (tid == 0 && sched) S.next[par] = G + atomicAdd(sched, 1);
    const int item = a.work ? a.work[wi] : wi;
    if constexpr (MAT)
      slab_item_mat(a, item, S);
    else
      slab_item<false>(a, item, S);
    wi = sched ? S.next[par] : wi + G;
    par ^= 1;
  }
  // the last CTA to finish resets the schedule counter for the next launch
  if (tid == 0 && sched) {
    __threadfence();
    if (atomicAdd(sched + 1, 1) == G - 1) {
      atomicExch(sched, 0);
      atomicExch(sched + 1, 0);
    }
  }
}

// Batches: one launch steps every active member (one material, float32);
// work = (member, item) pairs, the member's arguments from device memory,
// copied into shared memory for each item.
__global__ void __launch_bounds__(kSThreads, 2)
fused_step_slab_batch(const BatchMember<float>* __restrict__ members, const int2* __restrict__ work,
                      const int* __restrict__ n_work_p, int* sched) {
  using Smem = SlabSmem<false>;
  extern __shared__ __align__(128) unsigned char slab_raw[];
  Smem& S = *reinterpret_cast<Smem*>(slab_raw);
  __shared__ StepArgs<float> sargs;
  static_assert(sizeof(StepArgs<float>) % 4 == 0, "StepArgs copied as 32-bit words");
  const int tid = threadIdx.x;
  const int G = gridDim.x;
  const int n_work = *n_work_p;  // written before the launch (stream order)
  int wi = blockIdx.x, par = 0;
  while (wi < n_work) {
    if (tid == 0 && sched) S.next[par] = G + atomicAdd(sched, 1);
    const int2 w = work[wi];
    const BatchMember<float>& mb = members[w.x];
    if (mb.active) {
      // the member's arguments into shared memory once per item: what the
      // sweep reads again from global memory (where the single-solve kernel
      // has its parameter space) is a load on the critical path
      {
        const unsigned* s4 = reinterpret_cast<const unsigned*>(&mb.a);
        unsigned* d4 = reinterpret_cast<unsigned*>(&sargs);
        for (int i = tid; i < (int)(sizeof(StepArgs<float>) / 4); i += kSThreads) d4[i] = s4[i];
      }
      __syncthreads();
      slab_item<true>(sargs, w.y, S);
    } else {
      // an item of a member past its limit: no work, but the ticket thread 0
      // wrote above must be visible before every thread reads it (slab_item
      // ends with a block barrier; this branch needs its own)
      __syncthreads();
    }
    wi = sched ? S.next[par] : wi + G;
    par ^= 1;
  }
  if (tid == 0 && sched) {
    __threadfence();
    if (atomicAdd(sched + 1, 1) == G - 1) {
      atomicExch(sched, 0);
      atomicExch(sched + 1, 0);
    }
  }
}

// After a batch step: every active member swaps its field sets, counts the step
// and retires at its limit; when one does, the items of retired members leave the
// work list (in place, in order). A block that drew such an item paid the round
// trips of its ticket, its list entry and its member's flag, 1.4 us each, and
// late in a batch most of the list was of that kind (16 solves of 228 to 856
// steps: 407 ms of stepping, so 399). One block of 1024 threads.
__global__ void __launch_bounds__(1024) batch_advance_slab(BatchMember<float>* members, int n, int2* work, int* n_work_p) {
  __shared__ int warp_sum[32];
  int retired = 0;
  for (int i = threadIdx.x; i < n; i += 1024) {
    BatchMember<float>& m = members[i];
    if (!m.active) continue;
    for (int c = 0; c < 6; ++c) {
      float* t = m.a.out[c];
      m.a.out[c] = const_cast<float*>(m.a.in[c]);
      m.a.in[c] = t;
    }
    m.a.n += 1;
    m.cur ^= 1;
    if (m.a.n >= m.limit) {
      m.active = 0;
      retired = 1;
    }
  }
  if (!__syncthreads_or(retired)) return;
  const int total = *n_work_p, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int kept = 0;
  for (int base = 0; base < total; base += 1024) {
    const int i = base + threadIdx.x;
    int2 w = make_int2(0, 0);
    bool keep = false;
    if (i < total) {
      w = work[i];
      keep = members[w.x].active != 0;
    }
    const unsigned b = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) warp_sum[warp] = __popc(b);
    __syncthreads();  // (and every entry of this run is read before any is written)
    int before = 0, run = 0;
    for (int k = 0; k < 32; ++k) {
      if (k < warp) before += warp_sum[k];
      run += warp_sum[k];
    }
    if (keep) work[kept + before + __popc(b & ((1u << lane) - 1))] = w;
    kept += run;
    __syncthreads();  // the sums are read
  }
  if (threadIdx.x == 0) *n_work_p = kept;
}

}  // namespace

bool slab_shape_ok(int tx, int ty, bool mat) { return tx == kOX && ty == (mat ? kOY : kNamedY); }
int slab_rows(int tx, int ty) { return tx == kOX && ty == kNamedY ? kOY : ty; }

namespace {
template <bool MAT>
cudaError_t launch_slab(const StepArgs<float>& a, int* sched, cudaStream_t st) {
  static int sms = 0;
  const size_t smem = sizeof(SlabSmem<MAT>);
  if (!sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fused_step_slab<MAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) {
      sms = 0;
      return e;
    }
  }
  const int items = a.work ? a.n_work : a.tiles_x * a.tiles_y * a.n_chunks;
  if (items <= 0) return cudaSuccess;
  return launch_pdl(fused_step_slab<MAT>, std::min(items, 2 * sms), kSThreads, smem, st, a, sched);
}
}  // namespace

cudaError_t launch_fused_slab_batch(BatchMember<float>* members, int n_members, int2* work, int* n_work, int n_bound,
                                    int* sched, int nz_max, cudaStream_t st) {
  static int sms = 0;
  const size_t smem = sizeof(SlabSmem<false>);
  if (!sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fused_step_slab_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) {
      sms = 0;
      return e;
    }
  }
  if (n_bound > 0) {
    fused_step_slab_batch<<<std::min(n_bound, 2 * sms), kSThreads, smem, st>>>(members, work, n_work, sched);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = launch_transverse_after_batch_step<float>(members, n_members, nz_max, st);
  if (e != cudaSuccess) return e;
  batch_advance_slab<<<1, 1024, 0, st>>>(members, n_members, work, n_work);
  return cudaGetLastError();
}

cudaError_t launch_fused_slab_step(const StepArgs<float>& a, int* sched, cudaStream_t st) {
  // per-entry coefficient arrays (material runs) stream through the ring too
  if (a.co.ua[0]) return launch_slab<true>(a, sched, st);
  return launch_slab<false>(a, sched, st);
}

}  // namespace tetm
