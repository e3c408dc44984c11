// packed.cuh -- the per-site arithmetic on packed pairs: a complex value is one
// 64-bit register pair (re, im), and the f32x2 operations of sm_100 and later
// work on both halves in one instruction, each rounded as the scalar operation
// is.  Shared by the two-step and the resident sweeps, which are issue-bound.
#pragma once
#include "lbmbt_internal.cuh"
#include "sweep_common.cuh"

namespace lbmbt {
namespace {

using u64 = unsigned long long;   // one complex value (re, im) as a packed pair

__device__ __forceinline__ u64 pk(float x, float y)
{
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpk(u64 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c)
{
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b)
{
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ u64 sub2(u64 a, u64 b)
{
    u64 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Transform of a value pulled across a face (see pull()).
__device__ __forceinline__ u64 face2(u64 p, int bc, float2 f)
{
    if (bc == BC_MIR) return p;
    float2 v = unpk(p);
    if (bc == BC_MIR_CONJ) v.y = -v.y;
    v = cmul(v, f);
    return pk(v.x, v.y);
}

// Membrane link: v <- o + s (v - o) (mix() of sweep_common.cuh) where bit `B` of
// mk is set, by predication: in tissue nearly every warp has some such lane in
// every direction, and a divergent branch per direction and column costs more.
template <unsigned B>
__device__ __forceinline__ void mix_if(unsigned mk, u64& v, u64 o, u64 s2)
{
    asm("{\n\t.reg .pred p;\n\t.reg .b32 b;\n\t.reg .b64 d;\n\t"
        "and.b32 b, %1, %4;\n\tsetp.ne.u32 p, b, 0;\n\t"
        "sub.rn.f32x2 d, %0, %2;\n\t"
        "@p fma.rn.f32x2 %0, %3, d, %2;\n\t}"
        : "+l"(v)
        : "r"(mk), "l"(o), "l"(s2), "n"(B));
}

// react() and collide_w() of sweep_common.cuh for the first N populations (the
// others are 0 and stay 0): g <- g + g q, M = sum g, g <- g + omega (w M - g), the
// last as g - omega (g - w M), which rounds the same.  Returns M.
template <int N>
__device__ __forceinline__ u64 react_collide(u64 (&g)[N], float2 q, float om, float w0 = W0, float wi = WI)
{
    // the inner product takes the halves crosswise: two scalar operations, where a
    // packed one would need them swapped first
    const u64 qx = pk(q.x, q.x);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const float2 v = unpk(g[i]);
        g[i] = fma2(g[i], qx, pk(__fmaf_rn(-v.y, q.y, v.x), __fmaf_rn(v.x, q.y, v.y)));
    }
    u64 m = g[0];
#pragma unroll
    for (int i = 1; i < N; ++i) m = add2(m, g[i]);
    const u64 no = pk(-om, -om), n0 = pk(-w0, -w0), ni = pk(-wi, -wi);
#pragma unroll
    for (int i = 0; i < N; ++i) g[i] = fma2(no, fma2(i == 0 ? n0 : ni, m, g[i]), g[i]);
    return m;
}

}  // namespace
}  // namespace lbmbt
