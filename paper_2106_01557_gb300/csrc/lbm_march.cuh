// The row-marching engine of the fused f+g step (Eq. 12a-c, 13, 14), shared by
// the single-lattice step (lbm_march.cu) and the batched step (lbm_batch.cu).
//
// A warp owns a strip of 32 nodes in x (one per lane: FP64, FP32) or 64 (two
// neighbouring nodes per lane in packed FP32x2 arithmetic: 16-bit storage)
// and a run of rows, and walks the rows upwards on its own: nothing in the
// body of a step waits for another warp.
//
// A warp reads and writes lines of its strip straight from and to registers,
// every address an immediate offset from three pointers (the lane's own
// column, the one left and the one right of it). Per row y it
//  1. turns the f populations pulled by row y + 1, loaded during the previous
//     row, into moments: moment 0 is the density the pair force of row y needs
//     above it, and the moments themselves are what row y + 1 collides, so
//     every population is loaded and summed once;
//  2. starts the loads of f pulled by row y + 2 and g pulled by row y + 1, in
//     flight while the row is computed;
//  3. collides row y with the densities of rows y - 1, y and y + 1 (rolled in
//     registers; left and right neighbours by shuffles) and stores it; lanes
//     next to an edge add the periodic ghost columns and rows, the wall's
//     reflections or the open sides' ghosts.
// The densities beside a strip come from one more load per row: lanes 0-8 pull
// the nine populations of the node left of it, lanes 16-24 those of the node
// right of it, and a butterfly over the half-warps sums them in the order of
// moments9.
//
// Measured on 4096 x 1024 with walls (us per step; before, the step staged
// 64-wide tiles of all 18 planes in shared memory by tensor copies, with a
// density pass and a block barrier per tile): FP32 115.0 -> 105.3 (a copy without
// the collision took 104.6 then: what is left is mostly the memory mix), FP16 107.5
// -> 85.9 (bound by the packed arithmetic of 12 warps per SM); with launches that
// overlap (lbm_launch.cuh) and the later changes 103.4 (5.84 TB/s) and 80.4.
// Tried for the rows: a ring of tensor-copied boxes per warp (124, whatever the
// depth: about 10 cycles of the copy engine per line of 128 bytes), 16-byte
// asynchronous copies into a shared-memory ring (124: bound by the shared-
// memory pipe), prefetching 2 to 8 rows ahead into L2 (118 to 142), streaming
// hints on loads (114) and stores (107), the rows of all strips next to each
// other instead of the strips (112 at equal occupancy).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_f2.cuh"
#include "lbm_launch.cuh"
#include "lbm_ptx.cuh"
#include "lbm_store.cuh"

namespace lbm {

__host__ __device__ constexpr int EXm(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }

__host__ __device__ constexpr int EYm(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }

constexpr int MW = 4;  // warps per block

template <class S>
struct MarchCfg {
    static constexpr int NPL = sizeof(S) == 2 ? 2 : 1;                         // nodes per lane
    static constexpr int BPS = sizeof(S) == 8 ? 2 : (sizeof(S) == 4 ? 4 : 3);  // blocks per SM (registers)
    static constexpr int SW = 32 * NPL;                                        // strip width
    static constexpr int ROW = ROW_LINES * SW;                                 // elements per row of a strip
};

// A step is launched while the step before it still runs (lbm_launch.cuh), so
// its loads of the state are ordinary ones: the read-only path (__ldg, or a
// restricted pointer) is for memory that nobody writes while the kernel lives.

// The nine populations of one DF pulled at this lane's node(s), as stored.
// c, l, r: the DF's line 0 in the pulling row, at the lane's (first) column,
// the column left of it and the column right of its last.
template <class S, int NPL>
struct Pulled {
    S v[9];
    __device__ __forceinline__ void load(const S* c, const S* l, const S* r) {
        using Cf = MarchCfg<S>;
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = (EXm(i) == 0 ? c : (EXm(i) > 0 ? l : r))[i * Cf::SW - EYm(i) * Cf::ROW];
    }
    template <class C>
    __device__ __forceinline__ void get(C o[9]) const {
#pragma unroll
        for (int i = 0; i < 9; ++i) o[i] = Store<S, C>::raw(v[i]);
    }
};
// two nodes (x even, x + 1) of 16-bit storage: one word where the pull does
// not move in x, else two 16-bit loads
template <class S>
struct Pulled<S, 2> {
    uint32_t w[9];           // e_x = 0: both nodes, else node x
    unsigned short b[9];     // e_x != 0: node x + 1
    __device__ __forceinline__ void load(const S* c, const S* l, const S* r) {
        using Cf = MarchCfg<S>;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int o = i * Cf::SW - EYm(i) * Cf::ROW;
            if (EXm(i) == 0) {
                w[i] = *reinterpret_cast<const uint32_t*>(c + o);
            } else {
                w[i] = *reinterpret_cast<const unsigned short*>(EXm(i) > 0 ? l + o : c + o + 1);
                b[i] = *reinterpret_cast<const unsigned short*>(EXm(i) > 0 ? c + o : r + o);
            }
        }
    }
    static __device__ __forceinline__ float f(unsigned short h) {
        S s;
        memcpy(&s, &h, 2);
        return Store<S, float>::raw(s);
    }
    __device__ __forceinline__ void get(F2 o[9]) const {
#pragma unroll
        for (int i = 0; i < 9; ++i)
            o[i] = F2(f((unsigned short)(w[i] & 0xffffu)), EXm(i) == 0 ? f((unsigned short)(w[i] >> 16)) : f(b[i]));
    }
};

// per-thread sums of the conservation record
template <class C>
struct Rec {
    C mass, mx, my, ek, et, u2max, bad;
};

// a value of a node, or of a node pair: the sum, and the larger of a and it (a
// where it is NaN: the record's largest speed is that of the nodes that have one)
__device__ __forceinline__ float vsum(float a) { return a; }
__device__ __forceinline__ double vsum(double a) { return a; }
__device__ __forceinline__ float vsum(F2 a) { return a.v.x + a.v.y; }
__device__ __forceinline__ float vmax(float a, float b) { return b > a ? b : a; }
__device__ __forceinline__ double vmax(double a, double b) { return b > a ? b : a; }
__device__ __forceinline__ float vmax(float a, F2 b) { return vmax(vmax(a, b.v.x), b.v.y); }
// Conservation record of the entering state at a node, or a node pair whose
// second node lies in the lattice if v1. The total energy rho e_k - a rho^2 -
// kappa / 2 rho lap(rho), lap = 2 (axes / 3 + diagonals / 12 - 5 rho / 3).
template <class V, class K, class C>
__device__ __forceinline__ void record(const K& k, const V rn[9], const NodeMacro<V>& s, bool v1, Rec<C>& acc) {
    V rho = s.rho;
    const V ax = (rn[1] + rn[2]) + (rn[3] + rn[4]), dg = (rn[5] + rn[6]) + (rn[7] + rn[8]);
    V ek = s.rek;
    V et = ek - rho * (k.rec_rho * rho + k.rec_ax * ax + k.rec_dg * dg);
    V jx = rho * s.uhx, jy = rho * s.uhy;
    V u2 = s.uhx * s.uhx + s.uhy * s.uhy;
    if constexpr (std::is_same<V, F2>::value) {
        if (bad_node(rho.v.x, s.T.v.x, u2.v.x)) acc.bad += 1.f;
        if (v1 && bad_node(rho.v.y, s.T.v.y, u2.v.y)) acc.bad += 1.f;
        if (!v1) rho.v.y = jx.v.y = jy.v.y = ek.v.y = et.v.y = u2.v.y = 0.f;
    } else {
        if (bad_node(rho, s.T, u2)) acc.bad += C(1);
    }
    acc.mass += vsum(rho);
    acc.mx += vsum(jx);
    acc.my += vsum(jy);
    acc.ek += vsum(ek);
    acc.et += vsum(et);
    acc.u2max = vmax(acc.u2max, u2);
}

// The lanes' sums of a record, reduced over the warp: lanes 4 q .. 4 q + 3 hold
// quantity q (7: nothing). Each of the first three exchanges halves the
// quantities a lane still carries, so 9 additions take the place of 35: a
// twelfth of a one-row warp's FP64 operations.
template <class C>
__device__ __forceinline__ C reduce_record(const Rec<C>& acc, int lane) {
    C v[8];
    const C* a = &acc.mass;
#pragma unroll
    for (int q = 0; q < 7; ++q) v[q] = a[q];
    v[7] = C(0);
    auto join = [](C x, C y, bool largest) { return largest ? (y > x ? y : x) : x + y; };  // (quantity 5 is a maximum)
    bool five = true;  // is place `at` quantity 5 if the lane keeps it?
#pragma unroll
    for (int s = 16, n = 4; s >= 4; s >>= 1, n >>= 1) {
        const bool up = lane & s;
        five = five && up == ((5 & n) != 0);
#pragma unroll
        for (int j = 0; j < n; ++j) {
            const C w = __shfl_xor_sync(0xffffffffu, up ? v[j] : v[n + j], s);
            const C x = up ? v[n + j] : v[j];
            v[j] = j == (5 & (n - 1)) ? join(x, w, five) : x + w;
        }
    }
#pragma unroll
    for (int s = 2; s >= 1; s >>= 1) v[0] = join(v[0], __shfl_xor_sync(0xffffffffu, v[0], s), five);
    return v[0];
}

// the constants a step computes with
template <class V, class L>
__device__ __forceinline__ const KC<V>& march_constants(const L& l) {
    if constexpr (std::is_same<V, F2>::value) {
        static_assert(sizeof(KC<F2>) == sizeof(KC<float2>), "F2 is a float2");
        return reinterpret_cast<const KC<F2>&>(l.kp);
    } else if constexpr (std::is_same<V, double>::value) {
        return l.kd;
    } else {
        return l.kf;
    }
}

// What a warp marches over
template <class S, class C>
struct Strip {
    const S* in;               // the state read and the state written
    S* out;
    const double* phi;         // CUBIC
    int xs, y0, y1;            // first column, rows
    unsigned long long wait_ns;  // bound on the wait for the first rows
    bool sr;                   // stochastic rounding of 16-bit storage, keyed by
    const double* steps;       // the step count
};

// Rows y0 .. y1 - 1 of a strip. False if the wait for the first rows ran out
// (nothing is stored then).
// kv: the constants in the arithmetic's type (k, or both lanes of k).
// NODE_DITHER: stochastic rounding from every node's own seed, not the pair's.
// flush(acc): called after every 16 rows and after the last, where runs can be
// long, to carry the lanes' sums on in more bits. (Between two loops over rows: as
// a branch of the loop it costs twice the time.)
struct NoFlush {};
template <class S, class C, bool OPEN, bool CUBIC, bool NODE_DITHER, class K, class Flush = NoFlush>
__device__ __forceinline__ bool march_rows(const KC<C>& k, const K& kv, const Geometry& G, const Strip<S, C>& w,
                                           Rec<C>& acc, Flush flush = Flush()) {
    using Cf = MarchCfg<S>;
    constexpr int NPL = Cf::NPL, SW = Cf::SW, ROW = Cf::ROW;
    using V = typename std::conditional<NPL == 2, F2, C>::type;
    constexpr bool SH = Store<S, C>::SHIFTED;
    const int lane = threadIdx.x % 32;
    const int x = w.xs + NPL * lane;
    const bool v0 = x < G.nx, v1 = x + 1 < G.nx;
    const bool xper = !(OPEN && (G.open & 12));

    // the population of a node beside the strip that this lane pulls: place j
    // of a half-warp holds the direction that stands j-th in moments9's tree
    const int hj = lane & 15;
    const int hd = hj == 0 ? 1 : hj == 1 ? 3 : hj == 2 ? 2 : hj == 3 ? 4 : hj == 4 ? 5 : hj == 5 ? 7 : hj == 6 ? 6 : hj == 7 ? 8 : 0;
    const int hx = lane < 16 ? w.xs - 1 : w.xs + SW;
    const int hey = (hd == 2 || hd == 5 || hd == 6) ? 1 : ((hd == 4 || hd == 7 || hd == 8) ? -1 : 0);
    const S* hp = w.in + G.at(hd, hx - EXm(hd), w.y0 - 1 - hey);
    // line 0 of row y0 - 1 at the lane's own, left and right columns
    const S* pc = w.in + G.at(0, x, w.y0 - 1);
    const S* pl = w.in + G.at(0, x - 1, w.y0 - 1);
    const S* pr = w.in + G.at(0, x + NPL, w.y0 - 1);
    after_previous_grid();  // (a warp's second run of rows finds it done)
    if (w.wait_ns == 0) return false;
    // stochastic rounding is keyed by the step count
    const uint32_t step_key = SH && w.sr ? fmix32((uint32_t)(long long)__ldcg(w.steps) * 0x9e3779b9u + 0x7f4a7c15u) : 0u;
    auto halo_load = [&]() { return hj < 9 ? *hp : S(0.f); };
    auto next_row = [&]() {
        pc += ROW;
        pl += ROW;
        pr += ROW;
        hp += ROW;
    };
    const C r0 = SH ? k.mrest[0] : C(0);
    auto halo_sum = [&](S h) {
        C t = Store<S, C>::raw(h);
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        t += r0;
        if (OPEN && (G.open & 12) && (hx < 0 || hx >= G.nx)) t = k.rho_open;
        return t;
    };
    // a row's densities left of and right of this lane's node(s); at: of a pair,
    // the halves in between
    struct Dens {
        V l, r;
        C c;  // scalar form: at the node
        __device__ __forceinline__ V at() const {
            if constexpr (NPL == 2) return F2(l.v.y, r.v.x);
            else return c;
        }
    };
    auto dens = [&](V r, C h) {
        Dens d;
        if constexpr (NPL == 2) {
            float a = __shfl_up_sync(0xffffffffu, r.v.y, 1), b = __shfl_down_sync(0xffffffffu, r.v.x, 1);
            a = lane == 0 ? h : a;
            b = lane == 31 ? h : b;
            if (OPEN && (G.open & 12)) {  // beyond the right side
                if (x >= G.nx) r.v.x = k.rho_open;
                if (x + 1 >= G.nx) r.v.y = k.rho_open;
                if (x + 2 >= G.nx) b = k.rho_open;
            }
            d.l = F2(a, r.v.x);
            d.r = F2(r.v.y, b);
            d.c = 0.f;
        } else {
            if (OPEN && (G.open & 12) && x >= G.nx) r = k.rho_open;
            const C a = __shfl_up_sync(0xffffffffu, r, 1), b = __shfl_down_sync(0xffffffffu, r, 1);
            d.l = lane == 0 ? h : a;
            d.c = r;
            d.r = lane == 31 ? h : b;
        }
        return d;
    };
    const V ro = V(OPEN ? k.rho_open : C(0));
    const Dens dopen = {ro, ro, OPEN ? k.rho_open : C(0)};

    NodeMacro<V> s;
    V mn[9];  // f moments of the row after the one being collided
    Dens dm, dc;
    Pulled<S, NPL> rf, rg;
    S hn;
    {
        const uint64_t t0 = globaltimer_ns();
        Pulled<S, NPL> rm, rc;
        rm.load(pc, pl, pr);
        const S hm = halo_load();
        next_row();
        rc.load(pc, pl, pr);
        const S hc = halo_load();
        rg.load(pc + 9 * SW, pl + 9 * SW, pr + 9 * SW);
        next_row();
        rf.load(pc, pl, pr);
        hn = halo_load();
        V l[9];
        rm.get(l);
        dm = dens(density_of<SH>(l, kv.mrest), halo_sum(hm));
        rc.get(l);
        moments_of<SH>(l, kv.mrest, mn);
        dc = dens(mn[0], halo_sum(hc));
        if (w.y0 == 0 && G.walls) {
            if (OPEN && (G.open & 1)) dm = dopen;
            else dm = dc;  // beyond a wall: the adjacent node's density
        }
        // (later rows are not timed: with a timer read per row the step of a 4096 x
        // 1024 lattice in FP16 went from 79.5 to 82.7 us then, of a 128 x 128 one in FP32
        // from 3.93 to 4.03, and a load cannot be given up)
        C last;
        if constexpr (NPL == 2) last = dc.r.v.x;
        else last = dc.c;
        if (__any_sync(0xffffffffu, globaltimer_ns_after(last, t0) - t0 > w.wait_ns)) return false;
    }
    // (pc, pl and pr stand at row y0 + 1, row y + 1 in the loop)
    S* po = w.out + G.at(0, x, w.y0);
    // nodes with copies in the ghost columns
    const bool xg = v0 && xper && (x < GHOST_COLS || x + NPL > G.nx - GHOST_COLS);

    int y = w.y0;
#pragma unroll 1
    do {
        const int ye = std::is_same<Flush, NoFlush>::value || w.y1 - y <= 16 ? w.y1 : y + 16;
#pragma unroll 1
        for (; y < ye; ++y) {
            V rn[9];
            {
                V l[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) s.m[i] = mn[i];
                rf.get(l);
                // beyond the run only the density is wanted: worth a branch in FP64
                if (sizeof(C) < 8 || y + 1 < w.y1) moments_of<SH>(l, kv.mrest, mn);
                else mn[0] = density_of<SH>(l, kv.mrest);
                rg.get(l);
                moments_of<SH>(l, kv.nrest, s.n);
            }
            const S hcur = hn;
            if (y + 1 < w.y1) {
                rg.load(pc + 9 * SW, pl + 9 * SW, pr + 9 * SW);
                next_row();
                rf.load(pc, pl, pr);
                hn = halo_load();
            }
            Dens dp = dens(mn[0], halo_sum(hcur));
            if (y == G.ny - 1 && G.walls) {
                if (OPEN && (G.open & 2)) dp = dopen;
                else dp = dc;
            }
            rn[0] = dc.at();
            rn[1] = dc.r;
            rn[2] = dp.at();
            rn[3] = dc.l;
            rn[4] = dm.at();
            rn[5] = dp.r;
            rn[6] = dp.l;
            rn[7] = dm.l;
            rn[8] = dm.r;
            dm = dc;
            dc = dp;
            macro_of(kv, rn, s);
            if (v0) record(kv, rn, s, v1, acc);
            V R7 = V(0);
            if constexpr (CUBIC) {
                // -c (d_x(rho u_x^3) - d_y(rho u_y^3)), periodic central differences
                const long long n = (long long)G.nx * G.ny;
                const int ym = y == 0 ? G.ny - 1 : y - 1, yp = y == G.ny - 1 ? 0 : y + 1;
                auto r7 = [&](int xq) {
                    xq = xq < G.nx ? xq : G.nx - 1;
                    const int xm = xq == 0 ? G.nx - 1 : xq - 1, xp = xq == G.nx - 1 ? 0 : xq + 1;
                    const double dpx = 0.5 * (__ldcg(w.phi + (long long)y * G.nx + xp) - __ldcg(w.phi + (long long)y * G.nx + xm));
                    const double dpy = 0.5 * (__ldcg(w.phi + n + (long long)yp * G.nx + xq) - __ldcg(w.phi + n + (long long)ym * G.nx + xq));
                    return -k.c * ((C)dpx - (C)dpy);
                };
                if constexpr (NPL == 2) R7 = F2(r7(x), r7(x + 1));
                else R7 = r7(x);
            }
            V f[9], g[9];
            collide<SH, CUBIC>(kv, f, g, s, R7);

            // ---- next to a wall: the reflections this node owns -----------------
            // From the values of the collision. In 16-bit storage before the row is
            // rounded, after which they are no longer needed; otherwise, and with open
            // sides, whose ghosts need them to the end, after the row is stored (before
            // it: 512 x 512 in FP32 9.32 -> 9.44 us per step, open 11.2 -> 11.5).
            constexpr bool EARLY = SH && !OPEN;
            auto reflect = [&]() {
                if (!(G.walls && (y == 0 || y == G.ny - 1) && v0)) return;
#pragma unroll
                for (int q = 0; q < NPL; ++q) {
                    if (q == 1 && !v1) break;
                    auto of = [&](V v) -> C {
                        if constexpr (NPL == 2) return q ? v.v.y : v.v.x;
                        else return v;
                    };
                    // (a side that is open has its own ghosts instead)
                    if (y == 0 && !(OPEN && (G.open & 1)))
                        wall_store<S, C, OPEN>(w.out, G, k, x + q, y, of(f[4]), of(f[7]), of(f[8]), of(g[4]), of(g[7]), of(g[8]), of(s.rho));
                    if (y == G.ny - 1 && !(OPEN && (G.open & 2)))
                        wall_store<S, C, OPEN>(w.out, G, k, x + q, y, of(f[2]), of(f[5]), of(f[6]), of(g[2]), of(g[5]), of(g[6]), of(s.rho));
                }
            };
            if constexpr (EARLY) reflect();
            // ---- the row as stored ----------------------------------------------
            using W = typename std::conditional<NPL == 2, uint32_t, S>::type;  // a lane's share of a line
            W wv[18];
            if constexpr (NPL == 2) {
                using PW = PairWord<S>;
                if (NODE_DITHER && w.sr) {
                    // from each node's own seed: a word for the pair (f_i, g_i)
                    const uint32_t h0 = fmix32((uint32_t)(y * G.nx + x) ^ step_key), h1 = fmix32((uint32_t)(y * G.nx + x + 1) ^ step_key);
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const uint32_t r0 = h0 * NODE_DITHER_K[i], r1 = h1 * NODE_DITHER_K[i];
                        wv[i] = PW::sr(f[i], __byte_perm(r0, r1, 0x7632));
                        wv[9 + i] = PW::sr(g[i], __byte_perm(r0, r1, 0x5410));
                    }
                } else if (w.sr) {
                    // from the pair's seed: a word for each population
                    const uint32_t h = fmix32((uint32_t)(y * G.nx + x) ^ step_key);
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        wv[i] = PW::sr(f[i], h * (0x9e3779b9u * (2u * i + 1u)));
                        wv[9 + i] = PW::sr(g[i], h * (0x9e3779b9u * (2u * i + 19u)));
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        wv[i] = PW::rn(f[i]);
                        wv[9 + i] = PW::rn(g[i]);
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    wv[i] = Store<S, C>::cvt(f[i]);
                    wv[9 + i] = Store<S, C>::cvt(g[i]);
                }
            }
            S* const o = po;
            po += ROW;
            if (NPL == 1 ? v0 : v1) {
#pragma unroll
                for (int i = 0; i < 18; ++i) *reinterpret_cast<W*>(o + i * SW) = wv[i];
            }
            // rows next to the periodic seam also have a copy beyond it
            int dup = 0;
            if (!G.walls) dup = y < 2 ? G.ny : (y >= G.ny - 2 ? -G.ny : 0);
            if (v0 && (xg || dup || (NPL == 2 && !v1))) {
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    if (r == 1 && !dup) break;
                    const int yr = y + (r ? dup : 0);
                    S* q = w.out + G.at(0, x, yr);
                    S* ql = w.out + G.at(0, x < GHOST_COLS ? x + G.nx : x - G.nx, yr);                   // copy of node x
                    S* qr = w.out + G.at(0, x + 1 < GHOST_COLS ? x + 1 + G.nx : x + 1 - G.nx, yr);       // of node x + 1
                    const bool cl = xper && (x < GHOST_COLS || x >= G.nx - GHOST_COLS);
                    const bool cr = NPL == 2 && xper && v1 && (x + 1 < GHOST_COLS || x + 1 >= G.nx - GHOST_COLS);
#pragma unroll
                    for (int i = 0; i < 18; ++i) {
                        if constexpr (NPL == 2) {
                            const unsigned short lo = (unsigned short)(wv[i] & 0xffffu), hi = (unsigned short)(wv[i] >> 16);
                            unsigned short* h = reinterpret_cast<unsigned short*>(q + i * SW);
                            h[0] = lo;
                            if (v1) h[1] = hi;
                            if (cl) *reinterpret_cast<unsigned short*>(ql + i * SW) = lo;
                            if (cr) *reinterpret_cast<unsigned short*>(qr + i * SW) = hi;
                        } else {
                            if (r) q[i * SW] = wv[i];
                            if (cl) ql[i * SW] = wv[i];
                        }
                    }
                }
            }
            if constexpr (!EARLY) reflect();
            // ---- next to an open side: the ghosts this node owns ----------------
            if constexpr (OPEN) {
                if (v0 && (((G.open & 1) && y == 0) || ((G.open & 2) && y == G.ny - 1) || ((G.open & 4) && x == 0) ||
                           ((G.open & 8) && x + NPL >= G.nx))) {
#pragma unroll
                    for (int q = 0; q < NPL; ++q) {
                        const int xq = x + q;
                        if (!(((G.open & 1) && y == 0) || ((G.open & 2) && y == G.ny - 1) || ((G.open & 4) && xq == 0) ||
                              ((G.open & 8) && xq == G.nx - 1)) || xq >= G.nx)
                            continue;
                        Pops9<C> pf, pg;
                        if constexpr (NPL == 2) {
#pragma unroll
                            for (int i = 0; i < 9; ++i) {
                                pf.v[i] = q ? f[i].v.y : f[i].v.x;
                                pg.v[i] = q ? g[i].v.y : g[i].v.x;
                            }
                            if (q == 0) open_store<S, C>(w.out, G, k, xq, y, pf, pg, s.rho.v.x, s.uhx.v.x, s.uhy.v.x, s.T.v.x);
                            else open_store<S, C>(w.out, G, k, xq, y, pf, pg, s.rho.v.y, s.uhx.v.y, s.uhy.v.y, s.T.v.y);
                        } else {
#pragma unroll
                            for (int i = 0; i < 9; ++i) {
                                pf.v[i] = f[i];
                                pg.v[i] = g[i];
                            }
                            open_store<S, C>(w.out, G, k, xq, y, pf, pg, s.rho, s.uhx, s.uhy, s.T);
                        }
                    }
                }
            }
        }
        if constexpr (!std::is_same<Flush, NoFlush>::value) flush(acc);
    } while (!std::is_same<Flush, NoFlush>::value && y < w.y1);
    return true;
}

}  // namespace lbm
