// Stores of post-collision populations shared by the step kernels: the
// ghost-row values next to a wall, and the words a pair of neighbouring
// 16-bit nodes is stored as.
#pragma once

#include "lbm_device.cuh"
#include "lbm_f2.cuh"

namespace lbm {

// Wall ghost-row stores of a node next to a wall: the populations leaving
// through the wall come back reversed at the next pull (half-way bounce-back
// of f; of g adiabatic, or anti-bounce-back on a fixed-temperature segment).
// fo0.., go0..: the post-collision populations (for shifted formats, their
// deviations from the rest populations) of the three directions that leave
// through the wall: (4, 7, 8) at the bottom, (2, 5, 6) at the top. They come in
// the arithmetic's precision and are rounded once, to nearest. Opposite
// directions have equal rest populations.
template <class S, class C, bool OPEN>
__device__ __noinline__ void wall_store(S* __restrict__ out, const Geometry& G, const KC<C>& k, int x, int y,
                                        C fo0, C fo1, C fo2, C go0, C go1, C go2, C rho) {
    constexpr int SW = sizeof(S) == 2 ? 64 : 32;  // a line's elements
    const bool bottom = (y == 0);
    const int yg = bottom ? -1 : G.ny;
    const C Tw = bottom ? k.T_bottom : k.T_top;
    // n^eq of the wall at rest is linear in its temperature
    C ga1, gd1;
    g_rest_wall(k, rho, C(1), ga1, gd1);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int opp = bottom ? (j == 0 ? 2 : (j == 1 ? 5 : 6)) : (j == 0 ? 4 : (j == 1 ? 7 : 8));
        // x step of the leaving direction: 0 for 4/2; 7 and 6 go left, 8 and 5 right
        const int ex = j == 0 ? 0 : (bottom ? (j == 1 ? -1 : 1) : (j == 1 ? 1 : -1));
        const S fv = Store<S, C>::cvt(j == 0 ? fo0 : (j == 1 ? fo1 : fo2));
        C go = j == 0 ? go0 : (j == 1 ? go1 : go2);
        int xg = x + ex;
        xg = xg < 0 ? xg + G.nx : (xg >= G.nx ? xg - G.nx : xg);
        C T_link = Tw;
        if (bottom && G.hot_len > 0) {
            const int dxh = xg - G.hot_x0;  // (hot_x0 lies in the lattice)
            if ((dxh < 0 ? dxh + G.nx : dxh) < G.hot_len) T_link = k.T_hot;
        }
        if (T_link > C(0)) {
            const C rest = Store<S, C>::SHIFTED ? k.rest[9 + opp] : C(0);
            go = (C(2) * T_link * (j == 0 ? ga1 : gd1) - (go + rest)) - rest;
        }
        const S gv = Store<S, C>::cvt(go);
        S* const q = out + G.at(opp, xg, yg);
        q[0] = fv;
        q[9 * SW] = gv;
        if (!(OPEN && (G.open & 12)) && (xg < GHOST_COLS || xg >= G.nx - GHOST_COLS)) {  // the periodic copy
            S* const c = out + G.at(opp, xg < GHOST_COLS ? xg + G.nx : xg - G.nx, yg);
            c[0] = fv;
            c[9 * SW] = gv;
        }
    }
}

// One population of a node pair (x even, x + 1) as stored: a 32-bit word of two
// 16-bit values with node x in the low half; nearest rounding (rn) or stochastic (sr, 32 random bits: the
// upper 16 drive node x + 1, the lower 16 node x).
template <class S>
struct PairWord;
template <>
struct PairWord<__half> {
    using W = uint32_t;
    static __device__ __forceinline__ W rn(F2 v) {
        uint32_t d;
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x));
        return d;
    }
    static __device__ __forceinline__ W sr(F2 v, uint32_t r) {
        uint32_t d;
        asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x), "r"(r));
        return d;
    }
};
template <>
struct PairWord<__nv_bfloat16> {
    using W = uint32_t;
    static __device__ __forceinline__ W rn(F2 v) {
        uint32_t d;
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x));
        return d;
    }
    static __device__ __forceinline__ W sr(F2 v, uint32_t r) {
        uint32_t d;
        asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.v.y), "f"(v.v.x), "r"(r));
        return d;
    }
};

}  // namespace lbm
