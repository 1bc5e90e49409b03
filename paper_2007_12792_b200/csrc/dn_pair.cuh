// Packed pairs of floats (f32x2): the lower half belongs to the left side of the grid, the upper one to the side mirrored
// at x = 1/2.  Shared by the mirrored-pair kernels.
#pragma once

namespace dn {
namespace {

typedef unsigned long long u64;

struct f2 { u64 v; };
__device__ __forceinline__ f2 mk2(float lo, float hi) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ f2 dup2(float x) { return mk2(x, x); }
__device__ __forceinline__ void un2(const f2 a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v)); }
__device__ __forceinline__ float lo2(const f2 a) { float l, h; un2(a, l, h); return l; }
__device__ __forceinline__ float hi2(const f2 a) { float l, h; un2(a, l, h); return h; }
__device__ __forceinline__ f2 operator+(const f2 a, const f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 operator-(const f2 a, const f2 b) { f2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 operator*(const f2 a, const f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 fma2(const f2 a, const f2 b, const f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r; }
__device__ __forceinline__ f2 neg2(const f2 a) { f2 r; r.v = a.v ^ 0x8000000080000000ull; return r; }

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The polynomial with coefficients g[0..M] at c and at -c (cc = c^2): E(cc) + c O(cc) and E(cc) - c O(cc).  The halves of a
// pair are whatever g holds (two Gauss rows, two Gauss planes); c and cc hold the same value twice.
template <int M, int N>
__device__ __forceinline__ void exponents(const f2 (&g)[N], const f2 c, const f2 cc, f2& left, f2& right) {
    constexpr int ME = M / 2 * 2, MO = (M - 1) / 2 * 2 + 1;       // highest even and odd power
    f2 E = g[ME], O = g[MO];
#pragma unroll
    for (int i = ME - 2; i >= 0; i -= 2) E = fma2(E, cc, g[i]);
#pragma unroll
    for (int i = MO - 2; i >= 1; i -= 2) O = fma2(O, cc, g[i]);
    left = fma2(O, c, E);
    right = fma2(neg2(O), c, E);
}

__device__ __forceinline__ void cp4(unsigned d, const float* gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp4_if(unsigned d, const float* gsrc, int pred) {      // predicated, no branch
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void cp16_if(unsigned d, const float* gsrc, int pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

}  // namespace
}  // namespace dn
