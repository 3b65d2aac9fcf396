// Quads of four consecutive float32 nodes as the slab and half-step kernels
// hold them: predicated 16-byte accesses, packed arithmetic, neighbours by
// shuffle (16 lanes hold a row of 64 columns, two rows per warp).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace tetm {

__device__ __forceinline__ unsigned su32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// loads and stores under a predicate, without a branch (zero where not loaded).
// Only what a solve never changes (the activity bytes) goes through the
// non-coherent path: a launch that overlaps the one ahead is on the GPU while
// that one still writes the fields.
__device__ __forceinline__ unsigned ld_word_if(const uint8_t* p, bool c) {
  unsigned v;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n mov.u32 %0, 0;\n @q ld.global.nc.u32 %0, [%1];\n}"
      : "=r"(v)
      : "l"(p), "r"((unsigned)c));
  return v;
}
// the quad's word holds one activity byte per node: component c of any node
__device__ __forceinline__ bool has(unsigned m, int c) { return (m & (0x01010101u << c)) != 0u; }
// the same as a word, nonzero where true (a predicate operand for the
// accesses below, without a conversion from bool)
__device__ __forceinline__ unsigned hw(unsigned m, int c) { return m & (0x01010101u << c); }

// Pairs of float32 in 64-bit registers: one packed instruction rounds each
// half as the scalar one does. A quad is two pairs.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lo(f2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a;
}
__device__ __forceinline__ float hi(f2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return b;
}
struct P4 {
  f2 a, b;  // columns 0, 1 and 2, 3
};
__device__ __forceinline__ P4 fma4(const P4& c, const P4& x, const P4& y) {
  P4 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.a) : "l"(c.a), "l"(x.a), "l"(y.a));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.b) : "l"(c.b), "l"(x.b), "l"(y.b));
  return r;
}
__device__ __forceinline__ P4 sub4(const P4& x, const P4& y) {
  P4 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.a) : "l"(x.a), "l"(y.a));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(x.b), "l"(y.b));
  return r;
}
// 16-byte accesses straight from and to register pairs
__device__ __forceinline__ P4 ldp(const float* p) {
  P4 r;
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(r.a), "=l"(r.b) : "r"(su32(p)) : "memory");
  return r;
}
__device__ __forceinline__ void stp(float* p, const P4& v) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(su32(p)), "l"(v.a), "l"(v.b) : "memory");
}
__device__ __forceinline__ P4 ldg_if(const float* p, unsigned c) {
  P4 r;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n mov.b64 %0, 0;\n mov.b64 %1, 0;\n"
      " @q ld.global.v2.b64 {%0, %1}, [%2];\n}"
      : "=l"(r.a), "=l"(r.b)
      : "l"(p), "r"(c));
  return r;
}
__device__ __forceinline__ void stg_if(float* p, const P4& v, unsigned c) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n @q st.global.v2.b64 [%0], {%1, %2};\n}" ::"l"(p),
               "l"(v.a), "l"(v.b), "r"(c)
               : "memory");
}

// the neighbouring quad's value one column left (x-1) or right (x+1) of this
// quad (lanes: one row per half warp); at the tile edge a lane takes a value
// of the other half warp's row, which only halo nodes read
__device__ __forceinline__ float left_any(float v3) { return __shfl_up_sync(0xffffffffu, v3, 1); }
__device__ __forceinline__ float right_any(float v0) { return __shfl_down_sync(0xffffffffu, v0, 1); }

// the quad one column on minus the quad, and the quad one column back minus it
// (an exchanged column more: see slab_item)
__device__ __forceinline__ P4 diff_right(const P4& v) {
  const float r = right_any(lo(v.a));
  return P4{pk(hi(v.a) - lo(v.a), lo(v.b) - hi(v.a)), pk(hi(v.b) - lo(v.b), r - hi(v.b))};
}
__device__ __forceinline__ P4 diff_left(const P4& v) {
  const float l = left_any(hi(v.b));
  return P4{pk(l - lo(v.a), lo(v.a) - hi(v.a)), pk(hi(v.a) - lo(v.b), lo(v.b) - hi(v.b))};
}

}  // namespace tetm
