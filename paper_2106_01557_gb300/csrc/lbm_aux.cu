// Kernels around the time step: initial populations from macroscopic fields,
// population import/export, and the macroscopic fields / conservation record
// of the current state. They compute in FP64 and convert to the storage type
// at the end; k_init, k_rho and k_moments also come in an FP32 form for
// 32- and 16-bit storage (per-node arithmetic in FP32, sums in FP64), which
// the surrogate rollout uses. None is on the per-step path.
//
// Addressing: the stored state holds post-collision populations; the
// post-streaming population l_i(x) sits at x - e_i (pull streaming,
// Eq. 12a). Ghost columns and rows always hold valid copies (or, next to a
// wall, the reflected value), so a read at x - e_i needs no wrap.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

namespace {

constexpr int AUX_NT = 256;    // threads of a block that adds up a record
constexpr int FIELD_NT = 64;    // of the passes that have one node per thread

template <class S>
__device__ __forceinline__ double load_d(const S* buf, const Geometry& G, int p, int x, int y, double rest) {
    const S v = buf[G.at(p, x, y)];
    if constexpr (sizeof(S) == 2) return rest + (double)Store<S, float>::ld(v, 0.0f);
    else return (double)v;
}

template <class S>
__device__ __forceinline__ S to_store(double v, double rest) {
    if constexpr (sizeof(S) == 2) return Store<S, float>::st((float)(v - rest), 0.0f);
    else return (S)v;
}

// load_d in the compute type C (identical to it for C = double)
template <class S, class C>
__device__ __forceinline__ C load_c(const S* buf, const Geometry& G, int p, int x, int y, C rest) {
    const S v = buf[G.at(p, x, y)];
    if constexpr (sizeof(S) == 2) return rest + (C)Store<S, float>::ld(v, 0.0f);
    else return (C)v;
}
__device__ __forceinline__ int ex_of(int i) {
    return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__device__ __forceinline__ int ey_of(int i) {
    return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}

// Write post-streaming population l_i(x, y) so that the next pull finds it:
// at x - e_i (wrapped in x unless the left and right sides are open; wrapped
// in y when periodic; a ghost row or column at a wall or an open side).
template <class S>
__device__ __forceinline__ void scatter(S* buf, const Geometry& G, int p, int i, int x, int y, S v) {
    int xs = x - ex_of(i), ys = y - ey_of(i);
    if (!(G.open & 12)) xs = xs < 0 ? xs + G.nx : (xs >= G.nx ? xs - G.nx : xs);
    if (!G.walls) ys = ys < 0 ? ys + G.ny : (ys >= G.ny ? ys - G.ny : ys);
    put<S>(buf, G, p, xs, ys, v);
}

// What the kernels of whole fields below have in common. A node's neighbours
// in the state lie at constant offsets from its row in three columns, so one
// 64-bit address is formed per column and not one per population.
template <class S>
struct NodeAt {
    static constexpr int SW = sizeof(S) == 2 ? 64 : 32;  // strip width
    static constexpr int ROW = ROW_LINES * SW;
    int x, y;
    long long idx;     // y nx + x
    long long col[3];  // line 0 of row y in columns x - 1, x, x + 1
    bool inner;        // three or more nodes from every edge: no neighbour wraps, no copies
    __device__ __forceinline__ NodeAt(const Geometry& G, long long i) : idx(i) {
        y = (int)((uint32_t)i / (uint32_t)G.nx);  // (a lattice has at most 2^31 nodes)
        x = (int)((uint32_t)i - (uint32_t)y * (uint32_t)G.nx);
#pragma unroll
        for (int d = -1; d <= 1; ++d) col[d + 1] = G.at(0, x + d, y);
        inner = x >= 3 && x < G.nx - 3 && y >= 3 && y < G.ny - 3;
    }
    // element that population i of the DF whose lines begin at p is pulled from
    __device__ __forceinline__ long long from(int p, int i) const { return col[1 - EX(i)] + ((p + i) * SW - EY(i) * ROW); }
    static __device__ constexpr int EX(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
    static __device__ constexpr int EY(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }
    // the density of the node and its neighbours as the pair force sees them
    template <class C>
    __device__ __forceinline__ void densities(const double* __restrict__ rho, const Geometry& G, double rho_open, C rn[9]) const;
    // the pulled values of a DF, without the rest populations
    template <class C>
    __device__ __forceinline__ void pull(const S* __restrict__ buf, int p, C l[9]) const {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const S v = __ldg(buf + from(p, i));
            if constexpr (sizeof(S) == 8) l[i] = v;
            else l[i] = (C)Store<S, float>::raw(v);
        }
    }
};

// density at (x, y) as the pair force sees it: the open sides' fixed
// density beyond them, the adjacent fluid node's beyond a wall, periodic
// images elsewhere
__device__ __forceinline__ double rho_nb(const double* rho, const Geometry& G, double rho_open, int x, int y) {
    if (G.open && beyond_open(G, x, y)) return rho_open;
    x = x < 0 ? x + G.nx : (x >= G.nx ? x - G.nx : x);
    if (G.walls) y = y < 0 ? 0 : (y >= G.ny ? G.ny - 1 : y);
    else y = y < 0 ? y + G.ny : (y >= G.ny ? y - G.ny : y);
    return rho[(long long)y * G.nx + x];
}

template <class S>
template <class C>
__device__ __forceinline__ void NodeAt<S>::densities(const double* __restrict__ rho, const Geometry& G, double rho_open,
                                                     C rn[9]) const {
    if (inner) {
#pragma unroll
        for (int i = 0; i < 9; ++i) rn[i] = (C)__ldg(rho + idx + EX(i) + EY(i) * G.nx);
    } else {
#pragma unroll 1
        for (int dy = -1; dy <= 1; ++dy) {
            const double a = rho_nb(rho, G, rho_open, x - 1, y + dy), b = rho_nb(rho, G, rho_open, x, y + dy),
                         c = rho_nb(rho, G, rho_open, x + 1, y + dy);
            if (dy < 0) { rn[7] = (C)a; rn[4] = (C)b; rn[8] = (C)c; }
            else if (dy == 0) { rn[3] = (C)a; rn[0] = (C)b; rn[1] = (C)c; }
            else { rn[6] = (C)a; rn[2] = (C)b; rn[5] = (C)c; }
        }
    }
}

// Populations of the state (rho, u, T). In FP64 bound by the FP64 arithmetic
// (1/64 of the FP32 rate): no division but the equation of state's, the
// rest populations of shifted storage come off as three moments, and the
// moments m_4 = -m_3, m_6 = -m_5, n_7 = n_8 = 0 are used as such. 256 x 256,
// FP32 storage, FP64 arithmetic: 37.7 us before (180 FP64 operations and 8
// divisions per node, blocks of 256), 28.7 (147, 64). At 4096 x 1024 in FP32
// the fields in and out take 436 us instead of 606, in FP16 408 instead of 757
// (64-bit index divisions and one 64-bit address per population before).
template <class S, class C>
__global__ void __launch_bounds__(FIELD_NT) k_init(const __grid_constant__ Launch L, const double* __restrict__ rho, const double* __restrict__ ux,
                       const double* __restrict__ uy, const double* __restrict__ T, S* __restrict__ buf) {
    const Geometry& G = L.geo;
    const KC<C>& k = kc<C>(L);
    const long long at = blockIdx.x * (long long)FIELD_NT + threadIdx.x;
    if (at >= (long long)G.nx * G.ny) return;
    const NodeAt<S> d(G, at);
    NodeMacro<C> s;
    C rn[9];
    d.densities(rho, G, L.kd.rho_open, rn);
    const C r = rn[0], vx = (C)__ldg(ux + at) * k.c_inv, vy = (C)__ldg(uy + at) * k.c_inv;
    const C third = C(1.0 / 3.0), twelfth = C(1.0 / 12.0);
    s.rho = r;
    s.gx = third * (rn[1] - rn[3]) + twelfth * ((rn[5] - rn[7]) + (rn[8] - rn[6]));
    s.gy = third * (rn[2] - rn[4]) + twelfth * ((rn[5] - rn[7]) + (rn[6] - rn[8]));
    s.Fhx = k.G2c * r * s.gx + r * k.axc;
    s.Fhy = k.G2c * r * s.gy + r * k.ayc;
    s.uhx = vx;
    s.uhy = vy;
    s.q = k.c2 * (s.Fhx * vx + s.Fhy * vy);
    s.T = (C)__ldg(T + at);
    s.rek = r * (k.cv * s.T + C(0.5) * k.c2 * (vx * vx + vy * vy));
    C f[9], g[9];
    if (L.cubic) {
        C meq[9], Fm[9], neq[9], qm[9];
        equilibria(k, s, meq, Fm, neq, qm, true);
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            meq[j] -= k.half_dt * Fm[j];
            neq[j] -= k.half_dt * qm[j];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            meq[j] -= k.mrest[j];
            neq[j] -= k.nrest[j];
        }
        populations9(meq, f);
        populations9(neq, g);
    } else {
        // m^eq - dt/2 F_m and n^eq - dt/2 q_m (SM Eq. S3, S4), written out
        const C pbe = p_BE(k, r, s.T), eta = pbe * k.cs2_inv - r;
        const C rux = r * vx, ruy = r * vy;
        const C A3 = C(3) * ((rux * vx + ruy * vy) - k.dt * (s.Fhx * vx + s.Fhy * vy));
        const C jx = rux - k.half_dt * s.Fhx, jy = ruy - k.half_dt * s.Fhy;
        const C m7 = (rux - k.dt * s.Fhx) * vx - (ruy - k.dt * s.Fhy) * vy;
        const C m8 = jx * vy - k.half_dt * s.Fhy * vx;
        populations_jj(r - k.mrest[0], (C(2) * (eta - r) + A3) - k.mrest[1], (r + k.beta * eta - A3) - k.mrest[2], jx, jy, m7, m8, f);
        const C hq = k.half_dt * s.q, h = (s.rek + pbe) - hq;
        populations_jj((s.rek - hq) - k.nrest[0], (C(-4) * s.rek + k.c4g1_Cref * s.T - k.g1 * hq) - k.nrest[1],
                       (C(4) * s.rek - k.c4g2_Cref * s.T - k.g2 * hq) - k.nrest[2], h * vx, h * vy, C(0), C(0), g);
    }
    auto as_stored = [](C v) {
        if constexpr (sizeof(S) == 2) return Store<S, float>::st((float)v, 0.0f);
        else return (S)v;
    };
    if (d.inner) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            buf[d.from(0, i)] = as_stored(f[i]);
            buf[d.from(9, i)] = as_stored(g[i]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            scatter<S>(buf, G, i, i, d.x, d.y, as_stored(f[i]));
            scatter<S>(buf, G, 9 + i, i, d.x, d.y, as_stored(g[i]));
        }
    }
}

template <class S>
__global__ void k_set_pops(const Launch L, const double* __restrict__ f, const double* __restrict__ g,
                           S* __restrict__ buf) {
    const Geometry& G = L.geo;
    const long long n = (long long)G.nx * G.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(idx % G.nx), y = (int)(idx / G.nx);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            scatter<S>(buf, G, i, i, x, y, to_store<S>(f[i * n + idx], (double)L.kf.rest[i]));
            scatter<S>(buf, G, 9 + i, i, x, y, to_store<S>(g[i * n + idx], (double)L.kf.rest[9 + i]));
        }
    }
}

template <class S>
__global__ void k_get_pops(const Launch L, const S* __restrict__ buf, double* __restrict__ f,
                           double* __restrict__ g) {
    const Geometry& G = L.geo;
    const long long n = (long long)G.nx * G.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(idx % G.nx), y = (int)(idx / G.nx);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            f[i * n + idx] = load_d<S>(buf, G, i, x - ex_of(i), y - ey_of(i), (double)L.kf.rest[i]);
            g[i * n + idx] = load_d<S>(buf, G, 9 + i, x - ex_of(i), y - ey_of(i), (double)L.kf.rest[9 + i]);
        }
    }
}

template <class S, class C>
__global__ void __launch_bounds__(FIELD_NT) k_rho(const __grid_constant__ Launch L, const S* __restrict__ buf, double* __restrict__ rho) {
    const Geometry& G = L.geo;
    const long long at = blockIdx.x * (long long)FIELD_NT + threadIdx.x;
    if (at >= (long long)G.nx * G.ny) return;
    const NodeAt<S> d(G, at);
    C l[9], m[9];
    d.pull(buf, 0, l);
    moments_of<sizeof(S) == 2>(l, kc<C>(L).mrest, m);
    rho[at] = (double)m[0];
}

// rho u_x^3 and rho u_y^3 (u over c) of every node, phi [2][ny][nx], for
// the cubic-term elimination; rho_f: the density field (k_rho). Periodic
// boxes only.
template <class S, class C>
__global__ void k_phi(const Launch L, const S* __restrict__ buf, const double* __restrict__ rho_f,
                      double* __restrict__ phi) {
    const Geometry& G = L.geo;
    const KC<C>& k = kc<C>(L);
    const long long n = (long long)G.nx * G.ny;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(idx % G.nx), y = (int)(idx / G.nx);
        C f[9], g[9], rn[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            f[i] = load_c<S, C>(buf, G, i, x - ex_of(i), y - ey_of(i), (C)L.kf.rest[i]);
            g[i] = C(0);
            rn[i] = (C)rho_nb(rho_f, G, (double)L.kd.rho_open, x + ex_of(i), y + ey_of(i));
        }
        NodeMacro<C> s;
        node_macro(k, f, g, rn, s);
        phi[idx] = (double)(s.rho * s.uhx * s.uhx * s.uhx);
        phi[n + idx] = (double)(s.rho * s.uhy * s.uhy * s.uhy);
    }
}

// Macroscopic fields (Eq. 13, 14; 14.5 us at 256 x 256 in FP64) and, with RECORD, the FP64 conservation
// record reduced deterministically into stats[0..6].
template <class S, class C, bool RECORD>
__global__ void __launch_bounds__(RECORD ? AUX_NT : FIELD_NT)
    k_moments(const __grid_constant__ Launch L, const S* __restrict__ buf, const double* __restrict__ rho_f, double* __restrict__ o_rho,
              double* __restrict__ o_ux, double* __restrict__ o_uy, double* __restrict__ o_T,
              double* __restrict__ partials, double* __restrict__ stats, unsigned* __restrict__ counter) {
    const Geometry& G = L.geo;
    const KC<C>& k = kc<C>(L);
    const long long n = (long long)G.nx * G.ny;
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const NodeAt<S> d(G, idx);
        C f[9], g[9], rn[9];
        d.pull(buf, 0, f);
        d.pull(buf, 9, g);
        d.densities(rho_f, G, L.kd.rho_open, rn);
        NodeMacro<C> s;
        node_macro<sizeof(S) == 2>(k, f, g, rn, s);
        if (o_rho) o_rho[idx] = (double)s.rho;
        if (o_ux) o_ux[idx] = (double)(s.uhx * k.c);
        if (o_uy) o_uy[idx] = (double)(s.uhy * k.c);
        if (o_T) o_T[idx] = (double)s.T;
        if constexpr (RECORD) {
            const C ax = (rn[1] + rn[2]) + (rn[3] + rn[4]), dg = (rn[5] + rn[6]) + (rn[7] + rn[8]);
            const C u2 = s.uhx * s.uhx + s.uhy * s.uhy;
            acc[0] += (double)s.rho;
            acc[1] += (double)(s.rho * s.uhx);
            acc[2] += (double)(s.rho * s.uhy);
            acc[3] += (double)s.rek;
            acc[4] += (double)(s.rek - s.rho * (k.rec_rho * s.rho + k.rec_ax * ax + k.rec_dg * dg));
            acc[5] = fmax(acc[5], (double)u2);
            if (bad_node(s.rho, s.T, u2)) acc[6] += 1.0;  // as the step kernel counts them
        }
    }
    if constexpr (!RECORD) return;
    acc[1] *= L.kd.c;
    acc[2] *= L.kd.c;
    acc[5] *= L.kd.c2;
    __shared__ double red[AUX_NT / 32][7];
    __shared__ bool last;
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
#pragma unroll
    for (int q = 0; q < 7; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double w = __shfl_down_sync(0xffffffffu, acc[q], o);
            acc[q] = (q == 5) ? fmax(acc[q], w) : acc[q] + w;
        }
    if (lane == 0)
        for (int q = 0; q < 7; ++q) red[warp][q] = acc[q];
    __syncthreads();
    if (tid == 0) {
        double t[7] = {0, 0, 0, 0, 0, 0, 0};
        for (int w = 0; w < AUX_NT / 32; ++w)
            for (int q = 0; q < 7; ++q) t[q] = (q == 5) ? fmax(t[q], red[w][q]) : t[q] + red[w][q];
        for (int q = 0; q < 7; ++q) partials[(size_t)blockIdx.x * NQ + q] = t[q];
        __threadfence();
        last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // every thread combines the blocks tid, tid + AUX_NT, ... (independent L2
    // loads), then a fixed-order tree over the threads: the same record on
    // every run
    double t[7] = {0, 0, 0, 0, 0, 0, 0};
    for (unsigned b = tid; b < gridDim.x; b += AUX_NT)
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            const double pv = __ldcg(partials + (size_t)b * NQ + q);
            t[q] = (q == 5) ? fmax(t[q], pv) : t[q] + pv;
        }
#pragma unroll
    for (int q = 0; q < 7; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double w = __shfl_xor_sync(0xffffffffu, t[q], o);
            t[q] = (q == 5) ? fmax(t[q], w) : t[q] + w;
        }
    __syncthreads();  // red[] of the block pass is no longer needed
    if (lane == 0)
        for (int q = 0; q < 7; ++q) red[warp][q] = t[q];
    __syncthreads();
    if (tid == 0) {
        double u[7] = {0, 0, 0, 0, 0, 0, 0};
        for (int w = 0; w < AUX_NT / 32; ++w)
            for (int q = 0; q < 7; ++q) u[q] = (q == 5) ? fmax(u[q], red[w][q]) : u[q] + red[w][q];
        for (int q = 0; q < 7; ++q) stats[q] = (q == 5) ? sqrt(u[q]) : u[q];
        *counter = 0u;
    }
}

// Elements of a checkpoint file's planes from and into the strips, a thread per
// element of the file. Bound by the copy to or from the host (4096 x 1024 in FP32:
// save 118 -> 65 ms, load 140 -> 36 ms against rows copied by the host).
template <class E, bool SAVE>
__global__ void __launch_bounds__(AUX_NT) k_file(const Geometry G, const FilePlanes F, E* __restrict__ state, long long e, long long n,
                                                 E* __restrict__ file) {
    for (long long i = blockIdx.x * (long long)AUX_NT + threadIdx.x; i < n; i += (long long)gridDim.x * AUX_NT) {
        const long long row = (e + i) / F.pitch;
        const int x = (int)((e + i) - row * F.pitch) - F.px, p = (int)(row / F.nyp), y = (int)(row - (long long)p * F.nyp) - 2;
        const bool read = x >= -GHOST_COLS && x < G.nx + GHOST_COLS && y < G.ny + 2;
        if constexpr (SAVE) file[i] = read ? state[G.at(p, x, y)] : E(0);
        else if (read) state[G.at(p, x, y)] = file[i];
    }
}

template <bool SAVE>
cudaError_t launch_file(int esize, const Geometry& g, const FilePlanes& F, void* state, long long e, long long n, void* file,
                        cudaStream_t s) {
    const long long b = (n + AUX_NT - 1) / AUX_NT;
    const unsigned grid = (unsigned)(b < 65536 ? b : 65536);
    switch (esize) {
        case 2: k_file<uint16_t, SAVE><<<grid, AUX_NT, 0, s>>>(g, F, static_cast<uint16_t*>(state), e, n, static_cast<uint16_t*>(file)); break;
        case 4: k_file<uint32_t, SAVE><<<grid, AUX_NT, 0, s>>>(g, F, static_cast<uint32_t*>(state), e, n, static_cast<uint32_t*>(file)); break;
        case 8: k_file<uint64_t, SAVE><<<grid, AUX_NT, 0, s>>>(g, F, static_cast<uint64_t*>(state), e, n, static_cast<uint64_t*>(file)); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

int aux_blocks(const Geometry& g) {
    const long long n = (long long)g.nx * g.ny;
    long long b = (n + AUX_NT - 1) / AUX_NT;
    return (int)(b < 4096 ? b : 4096);
}

int field_blocks(const Geometry& g) { return (int)(((long long)g.nx * g.ny + FIELD_NT - 1) / FIELD_NT); }

template <class S>
struct AuxT {
    // fast: FP32 per-node arithmetic (32- and 16-bit storage only)
    static cudaError_t init(const Launch& L, const double* rho, const double* ux, const double* uy, const double* T,
                            void* buf, cudaStream_t s, bool fast) {
        if constexpr (sizeof(S) < 8) {
            if (fast) {
                k_init<S, float><<<field_blocks(L.geo), FIELD_NT, 0, s>>>(L, rho, ux, uy, T, static_cast<S*>(buf));
                return cudaGetLastError();
            }
        }
        k_init<S, double><<<field_blocks(L.geo), FIELD_NT, 0, s>>>(L, rho, ux, uy, T, static_cast<S*>(buf));
        return cudaGetLastError();
    }
    // in the step's compute type: FP64 for FP64 storage, FP32 otherwise
    static cudaError_t phi(const Launch& L, const void* buf, double* rho_scratch, double* out, cudaStream_t s) {
        using C = typename std::conditional<sizeof(S) == 8, double, float>::type;
        k_rho<S, C><<<field_blocks(L.geo), FIELD_NT, 0, s>>>(L, static_cast<const S*>(buf), rho_scratch);
        k_phi<S, C><<<aux_blocks(L.geo), AUX_NT, 0, s>>>(L, static_cast<const S*>(buf), rho_scratch, out);
        return cudaGetLastError();
    }
    static cudaError_t set(const Launch& L, const double* f, const double* g, void* buf, cudaStream_t s) {
        k_set_pops<S><<<aux_blocks(L.geo), AUX_NT, 0, s>>>(L, f, g, static_cast<S*>(buf));
        return cudaGetLastError();
    }
    static cudaError_t get(const Launch& L, const void* buf, double* f, double* g, cudaStream_t s) {
        k_get_pops<S><<<aux_blocks(L.geo), AUX_NT, 0, s>>>(L, static_cast<const S*>(buf), f, g);
        return cudaGetLastError();
    }
    template <class C>
    static cudaError_t moments_in(const Launch& L, const S* buf, double* rho_scratch, double* rho, double* ux,
                                  double* uy, double* T, double* partials, double* stats, unsigned* counter,
                                  cudaStream_t s) {
        k_rho<S, C><<<field_blocks(L.geo), FIELD_NT, 0, s>>>(L, buf, rho_scratch);
        if (partials)
            k_moments<S, C, true><<<aux_blocks(L.geo), AUX_NT, 0, s>>>(L, buf, rho_scratch, rho, ux, uy, T, partials, stats, counter);
        else
            k_moments<S, C, false><<<field_blocks(L.geo), FIELD_NT, 0, s>>>(L, buf, rho_scratch, rho, ux, uy, T, nullptr, nullptr, nullptr);
        return cudaGetLastError();
    }
    static cudaError_t moments(const Launch& L, const void* buf, double* rho_scratch, double* rho, double* ux,
                               double* uy, double* T, double* partials, double* stats, unsigned* counter,
                               cudaStream_t s, bool fast) {
        const S* b = static_cast<const S*>(buf);
        if constexpr (sizeof(S) < 8)
            if (fast) return moments_in<float>(L, b, rho_scratch, rho, ux, uy, T, partials, stats, counter, s);
        return moments_in<double>(L, b, rho_scratch, rho, ux, uy, T, partials, stats, counter, s);
    }
};

}  // namespace

int moments_blocks(const Geometry& g) { return aux_blocks(g); }

cudaError_t launch_state_to_file(int esize, const Geometry& g, const FilePlanes& F, const void* buf, long long e, long long n,
                                 void* out, cudaStream_t s) {
    return launch_file<true>(esize, g, F, const_cast<void*>(buf), e, n, out, s);
}
cudaError_t launch_file_to_state(int esize, const Geometry& g, const FilePlanes& F, const void* in, long long e, long long n,
                                 void* buf, cudaStream_t s) {
    return launch_file<false>(esize, g, F, buf, e, n, const_cast<void*>(in), s);
}

#define LBM_DISPATCH(storage, call)                                  \
    switch (storage) {                                               \
        case S_F64: return AuxT<double>::call;                       \
        case S_F32: return AuxT<float>::call;                        \
        case S_F16: return AuxT<__half>::call;                       \
        case S_BF16: return AuxT<__nv_bfloat16>::call;               \
    }                                                                \
    return cudaErrorInvalidValue;

cudaError_t launch_init(int storage, const Launch& L, const double* rho, const double* ux, const double* uy,
                        const double* T, void* buf, cudaStream_t s, bool fast) {
    LBM_DISPATCH(storage, init(L, rho, ux, uy, T, buf, s, fast))
}
cudaError_t launch_cubic_phi(int storage, const Launch& L, const void* buf, double* rho_scratch, double* phi,
                             cudaStream_t s) {
    LBM_DISPATCH(storage, phi(L, buf, rho_scratch, phi, s))
}
cudaError_t launch_set_pops(int storage, const Launch& L, const double* f, const double* g, void* buf,
                            cudaStream_t s) {
    LBM_DISPATCH(storage, set(L, f, g, buf, s))
}
cudaError_t launch_get_pops(int storage, const Launch& L, const void* buf, double* f, double* g, cudaStream_t s) {
    LBM_DISPATCH(storage, get(L, buf, f, g, s))
}
cudaError_t launch_moments(int storage, const Launch& L, const void* buf, double* rho_scratch, double* rho,
                           double* ux, double* uy, double* T, double* partials, double* stats, unsigned* counter,
                           cudaStream_t s, bool fast) {
    LBM_DISPATCH(storage, moments(L, buf, rho_scratch, rho, ux, uy, T, partials, stats, counter, s, fast))
}

}  // namespace lbm
