// Internal definitions of the GB300 r-cell engine (not part of the C ABI).
//
// Data layout in HBM (one context = a batch of r-cells):
//   * Atoms of all cells live in one padded array; cell c owns the slots
//     [atom_off[c], atom_off[c] + ntile[c]*TILE), of which the first n[c] are
//     real atoms.  A tile of TILE = 128 consecutive slots never spans two
//     cells, so every CTA works for exactly one r-cell.
//   * Positions: float4 {x, y, z, 0}, Cartesian in the cell's triangular MD box
//     (ping-pong pair so one kernel can read x(t) of all neighbours while it
//     writes x(t+dt) of its own atoms).  Velocities: float4 {vx, vy, vz, 0}.
//   * Inside a cell, atoms are kept sorted by neighbour bin (counting sort at
//     every list rebuild); `tag` maps a slot back to the caller's atom index.
//     Bins are at least r_list / 2 wide (in perpendicular width), so the
//     candidates of an atom lie in the 5 x 5 x 5 bins around its own.
//   * Verlet list: per tile, [max_nb/4][TILE] groups of four int32 entries
//     j_global | (image << 27) (one 16-byte load per lane per group, coalesced
//     across the tile); the image slot 0..26 selects one of the 27 periodic
//     shift vectors of the cell.  The last group is filled up with null entries
//     (slot 27), whose displacement is far beyond any cutoff.
//   * Per-cell FP64 state: box H, stretch R(t-1), Q, R, F of the last
//     deformation, Philox force-evaluation counter, status word.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/rcell.h"

#define RC_TILE 128
#define RC_IDX_BITS 27
#define RC_IDX_MASK ((1u << RC_IDX_BITS) - 1u)
#define RC_MAX_BONDS 4
#define RC_MAX_BINS_PER_CELL 8192
#define RC_SAMPLE_W 14  // per-step sample record: K[6], W[6], pe, ke

// per-step force-kernel modes
// (MODE_FORCE: forces and the FIRE minimiser's power sums only)
enum { MODE_EVAL = 0, MODE_SETUP = 1, MODE_STEP = 2, MODE_LAST = 3, MODE_FORCE = 4 };

// Everything a kernel needs, passed by value.
struct KParams {
    int pot;
    int units;
    float eps, sigma, rc2, rlist2, skin_half2, skin2;
    float sc_n, sc_m, sc_c;
    float k_fene, R02, wca2;
    float dt, fm;         // fm = (force -> acceleration) / mass
    float inv_tau;        // 0 when the thermostat is off
    float noise;          // sqrt(2 kT fm_units / (m tau dt))
    float mvv2e;          // m v^2 -> energy units, times mass (per atom)
    uint64_t seed;
    int max_nb;
    float max_step;       // > 0: displacement limit per step
    int n_tiles;          // tiles of RC_TILE atoms in the batch
    int max_cell;         // atoms of its largest cell
    int n_sm;             // SMs of the device (tile order of the pair kernels)
    int wait_polls;       // polls of a bounded device-side wait before it gives up
    int masked;           // cells are switched off: the pair kernels take their tiles from act_tiles
};

struct KArrays {
    // per cell
    const int *cell_n, *cell_off, *tile_cell, *cell_tile0;
    const float *Hf;     // 8 floats per cell: h00 h01 h02 h11 h12 h22 . .
    const float *Hif;    // inverse, same layout
    const float4 *shift; // periodic shift tables, RC_SHIFT_W entries per cell
    const int *nbins;    // 4 ints per cell
    const int *bin_off;  // first bin slot per cell
    int *bin_start;      // bin_off[c] .. + nbins+1
    int *status;
    int *need_rebuild, *built;
    unsigned long long *rebuilds;  // per cell: neighbour-list builds so far
    int *act_tiles, *n_act;  // tiles of the active cells, in order, and their number (when masked)
    const int *active;   // per cell: 0 = skipped by every MD kernel (state frozen)
    const unsigned long long *evals;
    double *series;      // [cell][slot][RC_SAMPLE_W]
    int series_cap;
    double *fire_acc;    // [cell][4] and [cell]: f.v, |v|^2, |f|^2 and max |f|^2 bits (MODE_FORCE)
    unsigned *fire_fmax2;
    double *eval_acc;    // [cell][8]: pe, W xx yy zz xy xz yz, pad
    // per atom
    float4 *x0, *x1;     // ping-pong
    float4 *v, *xref, *xr, *f;
    int *tag;
    int4 *partner;       // cell-local indices, -1 = none
    int *nbr, *nnb;
    int *bin_of;         // packed bin: b0 << 20 | b1 << 10 | b2 (each below 1024: at least 4 bins per axis)
    // sort scratch
    float4 *x_tmp, *v_tmp;
    int *tag_tmp, *newpos, *oldidx, *binid;
    int4 *partner_tmp;
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11), from the published round
// definition: words (c0..c3), key (k0,k1); per round
//   (hi0,lo0) = M0*c0, (hi1,lo1) = M1*c2,
//   c <- (hi1^c1^k0, lo1, hi0^c3^k1, lo0), then key += (W0, W1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 rc_philox(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; r++) {
        unsigned int hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        unsigned int hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// Three standard normals for (tag, cell, force evaluation, seed): uniforms
// u = (k + 1/2) 2^-32 and two Box-Muller pairs, of which three values are used.
__device__ __forceinline__ float3 rc_normals3(unsigned int tag, unsigned int cell, unsigned long long ev,
                                              unsigned long long seed) {
    uint4 o = rc_philox(make_uint4(tag, cell, (unsigned int)ev, (unsigned int)(ev >> 32)),
                        make_uint2((unsigned int)seed, (unsigned int)(seed >> 32)));
    const float s = 2.3283064365386963e-10f, h = 1.1641532182693481e-10f;
    float u0 = fmaf((float)o.x, s, h), u1 = fmaf((float)o.y, s, h);
    float u2 = fmaf((float)o.z, s, h), u3 = fmaf((float)o.w, s, h);
    float r0 = sqrtf(-2.0f * logf(u0)), r1 = sqrtf(-2.0f * logf(u2));
    float s0, c0, s1, c1;
    sincospif(2.0f * u1, &s0, &c0);
    sincospif(2.0f * u3, &s1, &c1);
    return make_float3(r0 * c0, r0 * s0, r1 * c1);
}

__device__ __forceinline__ void rc_set_status(int *status, int cell, int code) { atomicCAS(&status[cell], 0, code); }

// Periodic image shift tables.  The MD box H is stored FP32-exact (the FP64
// box of the deformation is rounded once), so the Cartesian shift
// sh = H (sx, sy, sz) of image (sx, sy, sz), s in {-1, 0, 1}, is exact in FP64
// and split into an FP32 value plus an FP32 remainder `lo` (nonzero only for
// combinations of tilted box vectors).  The displacement x_j + sh - x_i is then
// formed as ((x_j + sn) - (x_i - sp)) + lo with sn = min(sh, 0), sp = max(sh, 0):
// x_j + sn and x_i - sp subtract numbers of similar size (exact), so only the
// final subtraction rounds -- the result is the correctly rounded displacement
// instead of one carrying an error of half an ulp of the box length.
// Per image slot: a = {min(sh,0) (3), lo.x}, b = {max(sh,0) (3), lo.y}; the z
// shift n2 * H_zz is exact in FP32, so lo.z = 0.  Two 16-byte shared loads per pair.
//
// Images are numbered by slot k = (code + 14) mod 27 of the image code
// code = (sx+1) + 3(sy+1) + 9(sz+1): the central image (code 13) is slot 0, so
// a list entry j | k << RC_IDX_BITS of the central image is the bare index j.
// Slot 27 is the null entry that fills up a list's last group: its shift puts
// the neighbour 1e18 length units away.
//
// The tables belong to the box: k_deform writes them (FP64, which this GPU runs
// at 1/64 of the FP32 rate) and the pair kernels copy theirs to shared memory.
// Built by every CTA of every launch instead, they kept each CTA's first
// barrier waiting for 27 threads of FP64 work (force kernel on 10.24 M beads
// 1984 -> 1956 us, on one 256-atom cell 20.3 -> 19.5 us).
constexpr int RC_SLOT_CENTRAL = 0;
constexpr unsigned RC_SLOT_NULL = 27;
constexpr int RC_SLOTS = 28, RC_SHIFT_W = 2 * RC_SLOTS;
struct ShiftTab {
    float4 ab[RC_SHIFT_W];  // a of every slot, then b
    __device__ __forceinline__ const float4 &a(unsigned slot) const { return ab[slot]; }
    __device__ __forceinline__ const float4 &b(unsigned slot) const { return ab[RC_SLOTS + slot]; }
};

__host__ __device__ __forceinline__ int rc_image_slot(int sx, int sy, int sz) {
    return ((sx + 1) + 3 * (sy + 1) + 9 * (sz + 1) + 14) % 27;
}

// entry `slot` of the table of the box H (upper triangular, h00 h01 h02 h11 h12 h22)
__device__ __forceinline__ void rc_build_shift(float4 *tab, const float *H, int slot) {
    if (slot == (int)RC_SLOT_NULL) {
        tab[slot] = make_float4(1e18f, 1e18f, 1e18f, 0.f);
        tab[RC_SLOTS + slot] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const int code = (slot + 13) % 27;
    const double sx = (double)(code % 3 - 1), sy = (double)((code / 3) % 3 - 1), sz = (double)(code / 9 - 1);
    const double hx = (double)H[0] * sx + (double)H[1] * sy + (double)H[2] * sz;
    const double hy = (double)H[3] * sy + (double)H[4] * sz;
    const double hz = (double)H[5] * sz;
    const float fx = (float)hx, fy = (float)hy, fz = (float)hz;
    tab[slot] = make_float4(fminf(fx, 0.f), fminf(fy, 0.f), fminf(fz, 0.f), (float)(hx - fx));
    tab[RC_SLOTS + slot] = make_float4(fmaxf(fx, 0.f), fmaxf(fy, 0.f), fmaxf(fz, 0.f), (float)(hy - fy));
}

// cell c's table to shared memory (call with all threads; syncs)
__device__ __forceinline__ void rc_load_shifts(ShiftTab &T, const float4 *shift, int c) {
    if (threadIdx.x < RC_SHIFT_W) T.ab[threadIdx.x] = shift[(size_t)c * RC_SHIFT_W + threadIdx.x];
    __syncthreads();
}

// The central image has all-zero table entries, so its displacement is
// x_j - x_i bit for bit (rc_disp_central).  Lists hold their central entries
// first, so the lanes of a warp walk long runs of central entries together.
__device__ __forceinline__ float3 rc_disp(const float4 &xi, const float4 &xj, const ShiftTab &T, int slot) {
    const float4 sa = T.a(slot), sb = T.b(slot);
    return make_float3(((xj.x + sa.x) - (xi.x - sb.x)) + sa.w, ((xj.y + sa.y) - (xi.y - sb.y)) + sb.w,
                       (xj.z + sa.z) - (xi.z - sb.z));
}

// rc_disp with the slot's entries sa = T.a(slot) and xs = {x_i - T.b(slot) (3),
// T.b(slot).w} formed once for several neighbours of the same image slot
__device__ __forceinline__ float3 rc_disp_pre(const float4 &xj, const float4 &sa, const float4 &xs) {
    return make_float3(((xj.x + sa.x) - xs.x) + sa.w, ((xj.y + sa.y) - xs.y) + xs.w, (xj.z + sa.z) - xs.z);
}

__device__ __forceinline__ float3 rc_disp_central(const float4 &xi, const float4 &xj) {
    return make_float3(xj.x - xi.x, xj.y - xi.y, xj.z - xi.z);
}

// Programmatic dependent launch of the MD-step kernels (sort, list, density,
// force): each is launched with programmatic stream serialisation, so that its
// CTAs can be scheduled while the previous kernel of the stream drains, and
// begins with rc_pdl_wait(), which returns once that kernel has completed and
// its memory operations are visible -- before any access to shared state.  It
// then allows its own dependent to be scheduled (rc_pdl_trigger).  Launched
// without the attribute, the wait returns at once.
__device__ __forceinline__ void rc_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void rc_pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// cluster > 1: the grid (a multiple of it) runs in thread-block clusters of that many CTAs.
template <class... KArgs, class... Args>
void rc_launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, int cluster,
                   Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Surrogate input of one increment: u = (F - F_prev (row-major, 9), E = (F^T F - I)/2 in
// Voigt order xx yy zz xy xz yz (6))
__device__ __forceinline__ void rc_features(const double *fp, const double *f, float *o) {
    for (int k = 0; k < 9; k++) o[k] = (float)(f[k] - fp[k]);
    double C[9];
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) C[3 * a + b] = f[a] * f[b] + f[3 + a] * f[3 + b] + f[6 + a] * f[6 + b];
    o[9] = (float)(0.5 * (C[0] - 1.0));
    o[10] = (float)(0.5 * (C[4] - 1.0));
    o[11] = (float)(0.5 * (C[8] - 1.0));
    o[12] = (float)(0.5 * C[1]);
    o[13] = (float)(0.5 * C[2]);
    o[14] = (float)(0.5 * C[5]);
}

// Ensemble statistics of point i of n (Sm: n_members x n x 6): the members' mean
// stress into mu, returns their relative spread
__device__ __forceinline__ float rc_ensemble(const float *__restrict__ Sm, int n_members, int n, int i, float s_floor,
                                             float (&mu)[6]) {
    float var = 0.0f, nrm = 0.0f;
    for (int c = 0; c < 6; c++) {
        float s = 0.0f;
        for (int k = 0; k < n_members; k++) s += Sm[((size_t)k * n + i) * 6 + c];
        mu[c] = s / n_members;
        float q = 0.0f;
        for (int k = 0; k < n_members; k++) {
            const float d = Sm[((size_t)k * n + i) * 6 + c] - mu[c];
            q += d * d;
        }
        var += n_members > 1 ? q / (n_members - 1) : 0.0f;
        nrm += mu[c] * mu[c];
    }
    return sqrtf(var) / fmaxf(sqrtf(nrm), s_floor);
}

// per-cell state of the FIRE minimiser (k_fire.cu)
struct FireState {
    double *acc;      // [cell][4]: f.v, |v|^2, |f|^2, pad
    unsigned *fmax2;  // max |f_i|^2 as float bits
    float *dt, *alpha, *mixa, *mixb;
    int *npos, *done, *iters, *it, *zero;
    int *moving;  // per cell: 1 while the cell minimises (stands in for the activity mask meanwhile)
};

// host-side launchers (defined in the kernel translation units)
void rc_launch_sort(const KParams &p, const KArrays &a, int cur, int n_cells, cudaStream_t s);
void rc_launch_nlist(const KParams &p, const KArrays &a, int cur, int n_cells, cudaStream_t s);
// stage_atoms > 0: every CTA first copies its whole r-cell (stage_atoms = the
// largest cell of the batch) into shared memory and gathers neighbours there
// coop_tiles > 0: the cooperative walk on that many tiles (of the active ones, when masked)
void rc_launch_density(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int stage_atoms,
                       int coop_tiles, cudaStream_t s);
void rc_launch_force(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int mode, int slot,
                     int step_index, int stage_atoms, int coop_tiles, cudaStream_t s);
int rc_coop_max_tiles(int n_sm);
// act_tiles and n_act from the activity mask
void rc_launch_active_tiles(const KArrays &a, int n_cells, cudaStream_t s);
int rc_stage_max_atoms();
void rc_prepare_staged(int max_cell_atoms);
void rc_launch_deform_impl(const double *F, double *H, double *Rprev, double *Q, double *R, double *Fst, double *dR,
                           const double *H0, float *Hf, float *Hif, float4 *shift, int *status, int *need_rebuild,
                           int *nbins, const int *bin_cap, const int *active, double rlist, int n_cells, int n_sm,
                           cudaStream_t s);
// the shift table of cell c from its box
void rc_launch_shift(const float *Hf, float4 *shift, int c, cudaStream_t s);
void rc_launch_remap(const KArrays &a, const double *dR, int cur, int n_tiles, cudaStream_t s);
void rc_launch_stress(const double *series, int n_avg, int series_cap, const double *H, const double *Q,
                      const double *F, double pconv, double *rot_scratch, double *sig_fem, double *sig_se,
                      double *sig_md, double *P, int n_cells, cudaStream_t s);
void rc_launch_static_pk1(const KParams &p, const KArrays &a, int cur, int n_tiles, const float *mcell, double *acc,
                          cudaStream_t s);
void rc_launch_fire_init(const FireState &s, const int *status, const int *active, int n_cells, float dt0,
                         cudaStream_t st);
void rc_launch_fire_zero_v(const KArrays &a, const FireState &s, int n_tiles, int all_cells, cudaStream_t st);
void rc_launch_fire_iteration(const KParams &p, const KArrays &a, int cur, const FireState &s, int n_tiles, int n_cells,
                              float f_tol, float dt_max, float dmax, int *n_left, cudaStream_t st);
void rc_launch_static_prep(const double *H, const double *H0, float *mcell, double *acc, int n_cells,
                           cudaStream_t st);
void rc_launch_static_finish(const double *acc, const double *H0, const double *Q, const double *F, double pconv,
                             double *P, double *sig, const int *status, int n_cells, cudaStream_t st);
void rc_launch_advance(unsigned long long *evals, const int *active, int n_cells, int n, cudaStream_t s);
void rc_launch_keep_frozen(const KArrays &a, int cur_new, int n_tiles, cudaStream_t s);

// finite elements (k_fe.cu)
void fe_launch_geometry(int npe, const double *X, const int *conn, int ne, double rho0, double *gradN, double *V0,
                        double *mass, int *err, cudaStream_t s);
void fe_launch_apply_bc(const int *mask, const double *val, const double *g, double lambda, double dlambda, double *d,
                        int n3, cudaStream_t s);
void fe_launch_F(int npe, const int *conn, const double *gradN, const double *d, double *F, int ne, cudaStream_t s);
void fe_launch_fint(int npe, const double *X, const int *conn, const double *gradN, const double *V0, const double *P,
                    const double *d, double hg, double *fint, int ne, cudaStream_t s);
void fe_launch_update(const int *mask, const double *mass, const double *fint, double dt, double damping,
                      double *d, double *v, int n3, cudaStream_t s);
// one FE step with the surrogate, in three kernels around the members' forward
// pass (see k_fe.cu)
struct FeStepArgs {
    int ne, n3;  // elements; 3 x nodes
    const int *conn, *mask;
    const double *X, *gradN, *V0, *val, *g;
    double lambda, dlambda, hg;
    double *d, *fint, *F, *F_prev, *P;
    const double *P_md;
    float *u;
    const float *Sm;  // members' stresses, n_members x ne x 6
    int n_members;
    float s_floor, on, off;
    int force_md, *md_flag, *n_frozen, kmax;
    float *s_mean, *spread, *spread_out;
    int *host_flag, *host_frozen;  // pinned host memory
    double *F_hist;
};
void fe_launch_step_begin(int npe, const FeStepArgs &a, cudaStream_t s);
void fe_launch_step_decide(const FeStepArgs &a, cudaStream_t s);
void fe_launch_step_end(int npe, const FeStepArgs &a, cudaStream_t s);
void fe_launch_replay_mask(const int *md_flag, const int *n_frozen, int j, int *mask, int ne, cudaStream_t s);

// the forward pass of sur_step (k_mlp.cu): every member's stresses at n points,
// device, n_members x n x 6 in *Sm; h is advanced
struct sur_ctx;
int sur_step_members(sur_ctx *s, const float *u, int n, float *h, const float **Sm, int *n_members);
