// Internal declarations shared by the host runtime and the kernels of liblbm.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbm {

// Device status word bits (set by kernels, read and cleared by the host).
enum : int { ST_TIMEOUT = 1, ST_NONFINITE = 2 };

// Number of FP64 quantities in one conservation record.
constexpr int NQ = 8;

// Physical and model scalars in the kernel's compute type. Everything the
// collision needs is precomputed here so that a node update does no
// parameter arithmetic.
template <class C>
struct KC {
    C c, c2, dt, half_dt;
    C c_inv;         // 1 / c
    C G2c;           // G^2 / c   (F^ = F / c)
    C axc, ayc;      // a / c
    C a, half_kappa; // Eq. 16 a and kappa / 2 (total-energy diagnostic)
    C cs2_inv;       // 1 / c_s^2
    C RK, aK_eff, b4;   // p_BE = RK rho T Z(b4 rho) + aK_eff rho^2
    C inv_cv, cv, Cref;
    C g1, g2, beta, kS, hS, bS;
    C se, seps, sq, sp, sige, sigeps, sigp;
    C tauj_v, dtauj, rho_v, inv_drho;
    C qc;            // G^2 dt^2 / 12 of SM Eq. S6a (dx = 1)
    // products of the constants above, formed once on the host
    C we_kS_seps;    // (s_e/2 - 1) k s_eps
    C we_hS;         // (s_e/2 - 1) h
    C wp_bS;         // (s_p/2 - 1) b
    C six_qc;        // 6 qc
    C dt_g1, dt_g2, hdt_g1, hdt_g2;  // dt gamma_1, dt gamma_2, dt/2 gamma_1, dt/2 gamma_2
    C c4g1_Cref, c4g2_Cref;          // (4 + gamma_1) C_ref, (4 - gamma_2) C_ref
    C c2_third;      // c^2 / 3
    C rec_rho, rec_ax, rec_dg;  // total energy: a - 5 kappa / 3, kappa / 3, kappa / 12
    C T_bottom, T_top, T_hot;
    C rho_open, T_open;  // state of the open sides
    C rest[18];      // shifted-storage rest populations (f 0..8, g 9..17)
    C mrest[3], nrest[3];  // moments 0-2 of the f and g rest populations (the others vanish)
};

// Ghost columns that hold periodic copies: a pull reads one column beyond
// the lattice and the density beside it pulls from a second.
constexpr int GHOST_COLS = 2;

// The stored state is cut into strips of 32 nodes in x (64 for 16-bit
// storage), the width of a warp: [strip][row][18 lines][strip width]. A line
// holds one population of a row of a strip (128 bytes; 256 in FP64), so within
// a strip every address is a compile-time offset from one pointer. Lines:
// f_0 .. f_8, g_0 .. g_8. Column x of the lattice is column x + width of the
// state (the first strip holds the ghost columns left of the lattice), node
// row y its row y + 2.
constexpr int ROW_LINES = 18;

struct Geometry {
    int nx, ny, walls;
    int lsw;         // log2 of the strip width
    int nyp;         // rows of a strip (ny + 4)
    int strips;      // one more on each side than the lattice takes
    // element of population p (f_i: i, g_i: 9 + i) of the node at (x, y)
    __host__ __device__ __forceinline__ long long at(int p, int x, int y) const {
        const int xx = x + (1 << lsw);
        return (((((long long)(xx >> lsw) * nyp + (y + 2)) * ROW_LINES) + p) << lsw) + (xx & ((1 << lsw) - 1));
    }
    __host__ __device__ __forceinline__ long long elems() const { return ((long long)strips * nyp * ROW_LINES) << lsw; }
    int hot_x0, hot_len;
    int sms;         // multiprocessors of the device: a step's grid is one wave of resident blocks
    int open;        // open sides: 1 bottom, 2 top, 4 left, 8 right (left and right only together with all)
};

// Is lattice point (x, y) beyond an open side? (x is periodic unless the
// left and right sides are open.)
__host__ __device__ __forceinline__ bool beyond_open(const Geometry& G, int x, int y) {
    return ((G.open & 1) && y < 0) || ((G.open & 2) && y >= G.ny) || ((G.open & 4) && x < 0) ||
           ((G.open & 8) && x >= G.nx);
}

struct Launch {
    Geometry geo;
    KC<float> kf;
    KC<double> kd;
    KC<float2> kp;  // kf in both lanes, for the packed arithmetic of 16-bit storage
    int rounding;  // 16-bit storage: 0 nearest, 1 stochastic
    // bound in ns on a warp's wait for its first rows; 0: no waiting
    unsigned long long tile_wait_ns;
    int cubic;  // eliminate the cubic velocity terms (periodic single cases)
};

// default bound: 2 s
constexpr unsigned long long TILE_WAIT_NS_DEFAULT = 2000000000ull;

// Storage kinds
enum { S_F64 = 0, S_F32 = 1, S_F16 = 2, S_BF16 = 3 };

// Host-side launchers. All return cudaError_t of the launch.
// rho u_x^3 and rho u_y^3 of every node of a state (for the cubic-term
// elimination): the density field into rho_scratch, then phi [2][ny][nx]
cudaError_t launch_cubic_phi(int storage, const Launch& L, const void* buf, double* rho_scratch, double* phi,
                             cudaStream_t s);
// The row-marching step (lbm_march.cu): `groups` blocks of `warps` adjacent
// strips each across x, `chunks` chunks of rows.
struct MarchGrid {
    int groups, warps, chunks;
    int combine_prev;  // that many extra blocks combine the record of the step before (prev)
    int combine_here;  // the last block to finish combines this step's record
};
int march_strip(int storage);  // width of a warp's strip
MarchGrid march_grid(int storage, const Geometry& g);  // with combine_prev as a step after another takes it
// The grid of one step of a call. first: the record of the step before is
// combined already; last: no step follows in the call, so this one combines its
// own record. A launch has one writer of the record: the blocks that combine the
// record before run unordered beside the block that combines this one, and what
// they would write is replaced by it.
inline MarchGrid step_grid(MarchGrid m, bool first, bool last) {
    if (first || last) m.combine_prev = 0;
    m.combine_here = last ? 1 : 0;
    return m;
}
// partials: [groups * chunks][NQ]; cnt_in, cnt_out: the step count before and
// after the step (two places, so that every block can read it); phi: with
// L.cubic, [2][ny][nx] rho u_x^3 and rho u_y^3 (u over c) of the state
// entering the step (launch_cubic_phi), otherwise unused
cudaError_t launch_march(int storage, const Launch& L, const void* in, void* out,
                         const MarchGrid& mg, double* partials, const double* prev, double* stats, const double* cnt_in,
                         double* cnt_out, unsigned* counter, int* status, cudaStream_t s, const double* phi = nullptr);
// the record of a finished step whose partials no later step combined
cudaError_t launch_record_finish(const double* partials, int nblk, double* stats, cudaStream_t s);

// fast: FP32 per-node arithmetic for 32- and 16-bit storage (sums in FP64);
// FP64 storage always computes in FP64
cudaError_t launch_init(int storage, const Launch& L, const double* rho, const double* ux,
                        const double* uy, const double* T, void* buf, cudaStream_t s, bool fast = false);
cudaError_t launch_set_pops(int storage, const Launch& L, const double* f, const double* g, void* buf,
                            cudaStream_t s);
cudaError_t launch_get_pops(int storage, const Launch& L, const void* buf, double* f, double* g,
                            cudaStream_t s);
cudaError_t launch_moments(int storage, const Launch& L, const void* buf, double* rho_scratch,
                           double* rho, double* ux, double* uy, double* T, double* partials,
                           double* stats, unsigned* counter, cudaStream_t s, bool fast = false);
int moments_blocks(const Geometry& g);

// A checkpoint file holds the state as 18 planes (f_0 .. f_8, g_0 .. g_8) of node
// rows -2 .. ny + 1 (and on to `nyp` rows), each row from 128 bytes before its
// column 0 (px elements) to a whole number of 128 bytes that takes the 16 bytes of
// ghost columns beyond the last.
struct FilePlanes {
    int px, nyp;
    long long pitch;
    __host__ __device__ __forceinline__ long long elems() const { return 18 * pitch * nyp; }
};
// elements e .. e + n - 1 of the file from the stored state (zero where a step
// reads nothing), and into it; esize: bytes of a stored value
cudaError_t launch_state_to_file(int esize, const Geometry& g, const FilePlanes& F, const void* buf, long long e, long long n,
                                 void* out, cudaStream_t s);
cudaError_t launch_file_to_state(int esize, const Geometry& g, const FilePlanes& F, const void* in, long long e, long long n,
                                 void* buf, cudaStream_t s);

// Conservation record of caller-owned [9][ny][nx] FP64 populations with all
// scratch in a fixed device array (lbm_noalloc.cu); allocates nothing.
long long noalloc_max_nodes();
cudaError_t launch_record_noalloc(const Launch& L, const double* f, const double* g, double* out,
                                  cudaStream_t s);

}  // namespace lbm

// Access the surrogate's host code needs to a single-case handle (lbm_host.cpp).
struct lbm_handle;
int lbm_internal_fail(int code, const char* msg);
size_t lbm_internal_state_bytes(const lbm_handle* h);
int lbm_internal_snapshot(lbm_handle* h, void* dst);       // device copy of the current state
int lbm_internal_restore(lbm_handle* h, const void* src);  // and back
// lbm_set_fields from device fields [4][n] with FP32 per-node arithmetic
// (32- and 16-bit storage), synchronous
int lbm_internal_set_fields_fast(lbm_handle* h, const double* fields);
// the fields [4][n] (device, may be null) and the conservation record of the
// current state in one FP32 pass (sums in FP64), synchronous
int lbm_internal_read_fast(lbm_handle* h, double* fields, double out[6]);
cudaStream_t lbm_internal_stream(const lbm_handle* h);
// the handle's step count, host and device copies (the device copy keys the
// stochastic rounding of 16-bit storage); synchronous
int lbm_internal_set_steps(lbm_handle* h, int64_t steps);
void lbm_internal_rho_bounds(const lbm_handle* h, double* rho_v, double* rho_l, int* nx, int* ny);
