// Packed fp32 pairs (fma/add/mul/sub.f32x2, sm_100 and later) and the
// reverse tree of a LUT node written on them.
//
// A packed instruction does two fp32 operations for one issue slot; the FP32
// pipe itself is no faster (measured on GB300, lanes per SM and clock: 124.7
// scalar FFMA, 55-60 packed).  The node kernels are limited by issue slots
// as much as by the pipe, so halving the slots of their tree is what gains.
#pragma once

#include "common.cuh"

namespace bitlogic {

using f32x2 = unsigned long long;   // .lo = first value, .hi = second

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Reverse tree over the two halves of a table at once: element 0 of every
// pair belongs to the half whose top input is 0, element 1 to the other.
// The half of 2^(k-1) entries is evaluated as 4-entry Moebius quads over
// (x_0, x_1) under a lerp tree over x_2 .. x_{k-2}; quad m has coefficients
// cq[4m .. 4m+3] = (c0, c1, c2, c3), value (c0 + c1 x0) + x1 (c2 + c3 x0), and
// entry a of the quad has corner weight W[a].  x, omx (1 - x) and W hold the
// same value in both elements.  Returns the subtree's values, adds
// adjoint * d value / d x_i into dx[i] (the first subtree initialises it) and
// the leaf adjoints into acc.
template <int LV, int M, int H, int k>
__device__ __forceinline__ f32x2 bwd_tree_quad2(const f32x2 (&cq)[H], const f32x2 (&x)[k - 1],
                                                const f32x2 (&omx)[k - 1], const f32x2 (&W)[4], f32x2 adj,
                                                f32x2 (&dx)[k - 1], f32x2 (&acc)[H]) {
    if constexpr (LV == 1) {
        const f32x2 in0 = fma2(cq[4 * M + 1], x[0], cq[4 * M]);
        const f32x2 in1 = fma2(cq[4 * M + 3], x[0], cq[4 * M + 2]);
        const f32x2 dv0 = fma2(cq[4 * M + 3], x[1], cq[4 * M + 1]);
        if constexpr (M == 0) {
            dx[0] = mul2(adj, dv0);
            dx[1] = mul2(adj, in1);
        } else {
            dx[0] = fma2(adj, dv0, dx[0]);
            dx[1] = fma2(adj, in1, dx[1]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[4 * M + a] = fma2(adj, W[a], acc[4 * M + a]);
        return fma2(x[1], in1, in0);
    } else {
        const f32x2 lo = bwd_tree_quad2<LV - 1, 2 * M, H, k>(cq, x, omx, W, mul2(adj, omx[LV]), dx, acc);
        const f32x2 hi = bwd_tree_quad2<LV - 1, 2 * M + 1, H, k>(cq, x, omx, W, mul2(adj, x[LV]), dx, acc);
        const f32x2 diff = sub2(hi, lo);
        if constexpr (M == 0) dx[LV] = mul2(adj, diff);
        else dx[LV] = fma2(adj, diff, dx[LV]);
        return fma2(x[LV], diff, lo);
    }
}

// A table over kt inputs in shared memory, its two halves interleaved (value a
// of half h at word 2 a + h), -> the packed Moebius quads.  Loading whole
// pairs keeps them in register pairs: pairs assembled from two loads were
// moved together again at every use.
template <int kt>
__device__ __forceinline__ void packed_quads(const float* t, f32x2 (&cq)[1 << (kt - 1)]) {
    constexpr int H = 1 << (kt - 1);
#pragma unroll
    for (int m = 0; m < H / 4; ++m) {
        const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(t + 8 * m);
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(t + 8 * m + 4);
        cq[4 * m] = p.x;
        cq[4 * m + 1] = sub2(p.y, p.x);
        cq[4 * m + 2] = sub2(q.x, p.x);
        cq[4 * m + 3] = sub2(sub2(q.y, q.x), cq[4 * m + 1]);
    }
}

// One sample of a table over kt >= 3 inputs x[0 .. kt-1] with output adjoint
// g: adds g * w_a into acc (element h of acc[a] is entry a + h 2^(kt-1)),
// stores g * dv/dx_i in dx[i] (i < kt) and returns the value v.
template <int kt, int N>
__device__ __forceinline__ float node_sample2(const f32x2 (&cq)[1 << (kt - 1)], const float (&x)[N], float g,
                                              float (&dx)[N], f32x2 (&acc)[1 << (kt - 1)]) {
    static_assert(kt >= 3 && N >= kt, "quads under at least one packed input");
    constexpr int H = 1 << (kt - 1);
    const f32x2 one = pack2(1.f, 1.f);
    f32x2 x2[kt - 1], omx2[kt - 1], dx2[kt - 1];
#pragma unroll
    for (int i = 0; i < kt - 1; ++i) {
        x2[i] = pack2(x[i], x[i]);
        omx2[i] = sub2(one, x2[i]);
    }
    const f32x2 W[4] = {mul2(omx2[0], omx2[1]), mul2(x2[0], omx2[1]), mul2(omx2[0], x2[1]), mul2(x2[0], x2[1])};
    const f32x2 adj = mul2(pack2(g, g), pack2(1.f - x[kt - 1], x[kt - 1]));
    const f32x2 v = bwd_tree_quad2<kt - 2, 0, H, kt>(cq, x2, omx2, W, adj, dx2, acc);
    float v0, v1;
    unpack2(v, v0, v1);
    const float diff = v1 - v0;
    dx[kt - 1] = g * diff;
#pragma unroll
    for (int i = 0; i < kt - 1; ++i) {
        float a, b;
        unpack2(dx2[i], a, b);
        dx[i] = a + b;
    }
    return fmaf(x[kt - 1], diff, v0);
}

// Value of the subtree at level LV, index M of both table halves: 8-entry
// Moebius subtables by Horner steps (levels 0 to 2) under lerps.  A subtable's
// steps are written level by level, which the compiler schedules better than
// the nested form (4.05 -> 4.02 ms for the step at 128000 nodes x 2048
// samples; two or four samples at a time, to read each coefficient pair once
// for all, gave no more: 4.02 and 4.14 ms).
template <int LV, int M, int N, int n>
__device__ __forceinline__ f32x2 fwd_tree2(const f32x2 (&cf)[N], const f32x2 (&x)[n]) {
    if constexpr (LV == 2) {
        f32x2 t[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = fma2(cf[8 * M + 2 * j + 1], x[0], cf[8 * M + 2 * j]);
        t[0] = fma2(x[1], t[1], t[0]);
        t[2] = fma2(x[1], t[3], t[2]);
        return fma2(x[2], t[2], t[0]);
    } else {
        const f32x2 lo = fwd_tree2<LV - 1, 2 * M>(cf, x);
        const f32x2 hi = fwd_tree2<LV - 1, 2 * M + 1>(cf, x);
        return fma2(x[LV], sub2(hi, lo), lo);
    }
}

}  // namespace bitlogic
