// Force evaluation fused with the velocity-Verlet / Langevin update and the
// per-cell virial reduction -- one launch per MD step (two for Sutton-Chen,
// whose embedding term needs every rho_i before any force).
//
// Thread mapping: a CTA owns one tile of RC_TILE atoms of one r-cell; TPA
// consecutive lanes share one atom and split its Verlet list (TPA in 1,2,4,8),
// combining their partial sums with xor-shuffles.  Neighbour positions are
// gathered as float4 (16-byte, read-only path); atoms of a cell are stored
// bin-sorted, so the gathers of a warp hit a few L1/L2 lines.
//
// Arithmetic: pair math in FP32 (fused multiply-adds); per-atom virial and
// energy partials in FP32; per-warp sums promoted to FP64 before the per-cell
// atomic accumulation.
//
// Per step (mode STEP): f(t) from x(t); v(t) = v(t-dt/2) + dt/2 a(t) with
// a = f/m - v/tau + noise (Langevin friction on the velocity held at force
// time); sample K = sum m v(t) (x) v(t), W(t), PE(t); then v(t+dt/2) = v(t) +
// dt/2 a(t), x(t+dt) = x(t) + dt v(t+dt/2) written to the other position
// buffer, and the skin test that schedules the next neighbour rebuild.
#include "rc_internal.cuh"

namespace {

// lanes that share one atom: TPA, or 1 for the lean walk (TPA == 0)
__host__ __device__ constexpr int lanes_of(int tpa) { return tpa > 0 ? tpa : 1; }

template <int TPA>
__device__ __forceinline__ float sub_sum(float v) {
#pragma unroll
    for (int d = 1; d < TPA; d <<= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Where neighbour records come from: the global array through the read-only
// path, or the whole r-cell staged in shared memory (index minus cell offset).
struct GlobalSrc {
    const float4 *__restrict__ p;
    __device__ __forceinline__ float4 operator()(unsigned j) const { return __ldg(p + j); }
};
struct SharedSrc {
    const float4 *p;
    int off;
    __device__ __forceinline__ float4 operator()(unsigned j) const { return p[(int)j - off]; }
};

// Largest cell (in atoms) whose records are staged in shared memory.
constexpr int RC_STAGE_MAX_ATOMS = 12800;  // 200 KB of float4
constexpr unsigned RC_STAGE_CHUNK = 32768;  // bytes per bulk copy
constexpr int RC_SPIN_LIMIT = 1 << 22;

// Copy n float4 records (16-byte aligned) from global memory into shared memory
// with TMA bulk copies that complete on one mbarrier; every thread waits with a
// bounded spin of `polls` polls.  On a timeout the cell is flagged RC_ETIMEOUT
// and false returned, after a second wait (RC_SPIN_LIMIT polls, independent of
// `polls`) for the copies already issued, so that none is in flight when the
// CTA leaves.
__device__ __forceinline__ bool stage_records(float4 *dst, const float4 *src, int n, int *status, int c, int polls) {
    __shared__ __align__(8) unsigned long long s_bar;
    const unsigned bar = (unsigned)__cvta_generic_to_shared(&s_bar);
    const unsigned bytes = (unsigned)n * 16u;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        const unsigned d0 = (unsigned)__cvta_generic_to_shared(dst);
        for (unsigned o = 0; o < bytes; o += RC_STAGE_CHUNK) {
            const unsigned sz = min(RC_STAGE_CHUNK, bytes - o);
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(d0 + o),
                "l"(reinterpret_cast<const char *>(src) + o), "r"(sz), "r"(bar)
                : "memory");
        }
    }
    unsigned done = 0;
    for (int it = 0; it < polls && !done; it++)
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar)
            : "memory");
    // the whole block agrees, so that either every thread goes on or every thread leaves
    if (__syncthreads_and(done)) return true;
    if (threadIdx.x == 0) rc_set_status(status, c, RC_ETIMEOUT);
    for (int it = 0; it < RC_SPIN_LIMIT && !done; it++)  // let a late copy land before leaving
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar)
            : "memory");
    __syncthreads();
    return false;
}

// List groups are read once per pass: loaded without allocating in L1, which
// then keeps the neighbour records that the atoms of a tile share.
__device__ __forceinline__ int4 ld_list(const int4 *p) {
    int4 v;
    asm("ld.global.nc.L1::no_allocate.v4.s32 {%0, %1, %2, %3}, [%4];"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p));
    return v;
}

// Tile order of the pair kernels.  The grid is padded to a multiple R of the
// SM count S, and block b takes tile (b mod S) R + b / S: blocks b, b + S,
// b + 2S, ... -- those that the first wave deals to one SM -- get consecutive
// tiles, the spatial neighbours of one r-cell, whose shared neighbour records
// then stay in that SM's L1.  Blocks past the last tile return at once (-1).
// When cells are switched off, the same over the tiles of the others: by tile
// number, three active cells of 32 x 4000 atoms ran on 14 SMs and took as long
// as all 32.
__device__ __forceinline__ int tile_of_block(const KParams &p, const KArrays &a) {
    const int at = (int)(blockIdx.x % p.n_sm), row = (int)(blockIdx.x / p.n_sm);
    if (!p.masked) {
        const int t = at * ((int)gridDim.x / p.n_sm) + row;
        return t < p.n_tiles ? t : -1;
    }
    const int n = *a.n_act, rows = (n + p.n_sm - 1) / p.n_sm, k = at * rows + row;
    return row < rows && k < n ? a.act_tiles[k] : -1;
}
inline unsigned pair_grid(const KParams &p) {
    return (unsigned)(((p.n_tiles + p.n_sm - 1) / p.n_sm) * p.n_sm);
}

// Displacements and pair evaluations of one list group (entries e, records
// c0..c3).  Warp-uniform fast paths: all four entries of the image slot 0 (the
// central image: x_j - x_i, the bits rc_disp gives for it) in every converged
// lane, or one image slot per lane's group (the runs of a stencil bin): one
// shift-table read and one x_i - sp per group instead of one per entry, the same
// arithmetic as rc_disp.  Null entries, which fill up a list's last group, have a
// slot of their own whose displacement no cutoff reaches.
//
// fn is straight-line code: no branch on the cutoff,
// which about two thirds of the lanes pass, so that the four evaluations
// interleave.  The pair kernels are bound by the instructions they issue and the
// L1 wavefronts of their gathers (0.7 of the issue slots, 0.6 of the L1 data
// pipe on 320 000 beads); against a branch per entry and a check for the list's
// end: force step without / with a sample 1956 / 2304 -> 1771 / 2117 us on
// 10.24 M beads (lean walk), 56 / 61 -> 45 / 53 us on 160 000, density and force
// of 128 000 copper atoms 71 + 80 -> 66 + 74 us.  (Packed FP32 arithmetic,
// add / mul / fma.f32x2 on two neighbours, took another 2 to 6 % off the lean
// walk but sums in another order; in the pipelined walk it spills.)
template <class Fn>
__device__ __forceinline__ void eval_group(const int4 &e, const float4 &c0, const float4 &c1, const float4 &c2,
                                           const float4 &c3, const float4 &xi, const ShiftTab &T, Fn &&fn) {
    const unsigned s0 = (unsigned)e.x >> RC_IDX_BITS;
    const unsigned am = __activemask();
    float3 d0, d1, d2, d3;
    if (__all_sync(am, ((unsigned)(e.x | e.y | e.z | e.w) >> RC_IDX_BITS) == RC_SLOT_CENTRAL)) {
        d0 = rc_disp_central(xi, c0);
        d1 = rc_disp_central(xi, c1);
        d2 = rc_disp_central(xi, c2);
        d3 = rc_disp_central(xi, c3);
    } else if (__all_sync(am, (((unsigned)(e.x ^ e.y) | (unsigned)(e.x ^ e.z) | (unsigned)(e.x ^ e.w)) >> RC_IDX_BITS) == 0)) {
        const float4 sa = T.a(s0), sb = T.b(s0);
        const float4 xs = make_float4(xi.x - sb.x, xi.y - sb.y, xi.z - sb.z, sb.w);
        d0 = rc_disp_pre(c0, sa, xs);
        d1 = rc_disp_pre(c1, sa, xs);
        d2 = rc_disp_pre(c2, sa, xs);
        d3 = rc_disp_pre(c3, sa, xs);
    } else {
        d0 = rc_disp(xi, c0, T, s0);
        d1 = rc_disp(xi, c1, T, (unsigned)e.y >> RC_IDX_BITS);
        d2 = rc_disp(xi, c2, T, (unsigned)e.z >> RC_IDX_BITS);
        d3 = rc_disp(xi, c3, T, (unsigned)e.w >> RC_IDX_BITS);
    }
    fn(c0, d0);
    fn(c1, d1);
    fn(c2, d2);
    fn(c3, d3);
}

// Walk one atom's Verlet list (this lane's share: groups sub, sub+TPA, ... of
// four entries).  Each group is one 16-byte load.  The loop is software
// pipelined: while the pairs of group g are evaluated, the four neighbour
// records of the next group are already being gathered and the list entries of
// the group after that are being loaded, so the gather latency overlaps the
// pair arithmetic.  fn(xj, d) receives the neighbour's record and the exact
// periodic displacement d = x_j(image) - x_i.
// TPA == 0 is the lean walk: one lane per atom, only the next group's entries
// loaded ahead -- fewer registers, so that more warps per SM hide the latency
// instead (the force kernel is compiled for 10 resident CTAs then, the density
// kernel for 12), which pays when the batch has enough tiles to fill them.
template <int TPA, class Src, class Fn>
__device__ __forceinline__ void for_each_neighbor(const int4 *__restrict__ nb4, int nn, int sub, const Src &src,
                                                  const float4 &xi, const ShiftTab &T, Fn &&fn) {
    const int ng = (nn + 3) >> 2;
    if constexpr (TPA == 0) {
        if (ng == 0) return;
        int4 e = ld_list(nb4);
        for (int g = 0; g < ng; g++) {
            // the list streams from DRAM: ask L2 for the group after next now, so
            // that its load finds it there (no register holds it meanwhile)
            if (g + 3 < ng) asm volatile("prefetch.global.L2 [%0];" ::"l"(nb4 + (size_t)(g + 3) * RC_TILE));
            const float4 c0 = src((unsigned)e.x & RC_IDX_MASK), c1 = src((unsigned)e.y & RC_IDX_MASK);
            const float4 c2 = src((unsigned)e.z & RC_IDX_MASK), c3 = src((unsigned)e.w & RC_IDX_MASK);
            int4 en = e;
            if (g + 1 < ng) en = ld_list(nb4 + (size_t)(g + 1) * RC_TILE);
            eval_group(e, c0, c1, c2, c3, xi, T, fn);
            e = en;
        }
        return;
    }
    int g = sub;
    if (g >= ng) return;
    int4 e = ld_list(nb4 + (size_t)g * RC_TILE);
    float4 c0 = src((unsigned)e.x & RC_IDX_MASK), c1 = src((unsigned)e.y & RC_IDX_MASK);
    float4 c2 = src((unsigned)e.z & RC_IDX_MASK), c3 = src((unsigned)e.w & RC_IDX_MASK);
    int gn = g + TPA;
    int4 en = e;
    if (gn < ng) en = ld_list(nb4 + (size_t)gn * RC_TILE);
    while (true) {
        const int gnn = gn + TPA;
        float4 n0 = c0, n1 = c1, n2 = c2, n3 = c3;
        int4 enn = en;
        if (gn < ng) {  // next stage: gather group gn, load the entries of group gnn
            n0 = src((unsigned)en.x & RC_IDX_MASK);
            n1 = src((unsigned)en.y & RC_IDX_MASK);
            n2 = src((unsigned)en.z & RC_IDX_MASK);
            n3 = src((unsigned)en.w & RC_IDX_MASK);
            if (gnn < ng) enn = ld_list(nb4 + (size_t)gnn * RC_TILE);
        }
        eval_group(e, c0, c1, c2, c3, xi, T, fn);
        if (gn >= ng) break;
        g = gn;
        gn = gnn;
        e = en;
        en = enn;
        c0 = n0;
        c1 = n1;
        c2 = n2;
        c3 = n3;
    }
}

// One neighbour's part in rho, zero beyond the cutoff: (a/r)^2 for m = 6, else
// (a/r)^m, and the sum with it
template <bool M6>
__device__ __forceinline__ float density_term(const KParams &p, const float3 &d) {
    const float r2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    const float ar2 = r2 < p.rc2 ? p.sigma * p.sigma * __fdividef(1.0f, r2) : 0.0f;
    return M6 || !(r2 < p.rc2) ? ar2 : powf(ar2, 0.5f * p.sc_m);
}
template <bool M6>
__device__ __forceinline__ float density_sum(float rho, float q) {
    return M6 ? fmaf(q * q, q, rho) : __fadd_rn(rho, q);
}

// dE/dr / r of one pair, and in e its energy in units of eps / 2 (SC) or 2 eps
// (LJ); both zero beyond the cutoff, where 1 / r^2 counts as zero
template <int POT, bool M6>
__device__ __forceinline__ float pair_term(const KParams &p, const float4 &xi, const float4 &xj, const float3 &d, float &e) {
    const float r2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    const float ir2 = r2 < p.rc2 ? __fdividef(1.0f, r2) : 0.0f;
    const float sr2 = p.sigma * p.sigma * ir2;
    if (POT == RC_POT_SC) {
        float arm, arn;
        if (M6) {
            arm = sr2 * sr2 * sr2;                     // (a/r)^6
            arn = arm * sr2 * (p.sigma * rsqrtf(r2));  // (a/r)^9
        } else {
            // (zero beyond the cutoff by themselves: a negative exponent gives infinity there)
            arm = r2 < p.rc2 ? powf(sr2, 0.5f * p.sc_m) : 0.0f;
            arn = r2 < p.rc2 ? powf(sr2, 0.5f * p.sc_n) : 0.0f;
        }
        e = arn;
        // eps / r^2 [ -n (a/r)^n + c m/2 (rho_i^-1/2 + rho_j^-1/2) (a/r)^m ]
        return p.eps * ir2 * fmaf(0.5f * p.sc_c * p.sc_m * (xi.w + xj.w), arm, -p.sc_n * arn);
    }
    const float sr6 = sr2 * sr2 * sr2;
    e = sr6 * (sr6 - 1.0f);
    // -24 eps (2 (s/r)^12 - (s/r)^6) / r^2
    return -(24.0f * p.eps) * ir2 * sr6 * (2.0f * sr6 - 1.0f);
}

// Sutton-Chen density pass: rho_i = sum_j (a/r_ij)^m over r < rc; writes
// xr_i = {x_i, rho_i^{-1/2}} for the force pass.
// resident CTAs per SM the density pass is compiled for (a register cap of
// 65536 / (128 x this) at one lane per atom): 12 for the lean walk, else 7 --
// a 128 000-atom batch (1000 tiles) in one wave on 152 SMs
constexpr int density_min_ctas(int tpa) { return tpa == 0 ? 12 : (7 / tpa > 0 ? 7 / tpa : 1); }

template <int TPA, bool M6, bool STG>
__global__ void __launch_bounds__(RC_TILE *lanes_of(TPA), density_min_ctas(TPA)) k_density(KParams p, KArrays a, int cur) {
    extern __shared__ __align__(16) float4 s_cell[];
    rc_pdl_wait();
    rc_pdl_trigger();
    const int t = tile_of_block(p, a);
    if (t < 0) return;
    const int c = a.tile_cell[t];
    if (a.status[c] != 0 || !a.active[c]) return;
    __shared__ ShiftTab s_tab;
    rc_load_shifts(s_tab, a.shift, c);

    const int at = threadIdx.x / lanes_of(TPA), sub = threadIdx.x % lanes_of(TPA);
    const int n = a.cell_n[c], off = a.cell_off[c];
    const int li = (t - a.cell_tile0[c]) * RC_TILE + at;
    const float4 *__restrict__ X = cur ? a.x1 : a.x0;
    if (STG && !stage_records(s_cell, X + off, n, a.status, c, p.wait_polls)) return;
    const bool live = li < n;
    const int g = off + li;
    float rho = 0.0f;
    float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) {
        xi = X[g];
        const int nn = a.nnb[g];
        const int4 *__restrict__ nb = reinterpret_cast<const int4 *>(a.nbr) + (size_t)t * (p.max_nb / 4) * RC_TILE + at;
        auto body = [&](const float4 &, const float3 &d) { rho = density_sum<M6>(rho, density_term<M6>(p, d)); };
        if (STG) for_each_neighbor<TPA>(nb, nn, sub, SharedSrc{s_cell, off}, xi, s_tab, body);
        else for_each_neighbor<TPA>(nb, nn, sub, GlobalSrc{X}, xi, s_tab, body);
    }
    rho = sub_sum<TPA>(rho);
    if (live && sub == 0) a.xr[g] = make_float4(xi.x, xi.y, xi.z, rho > 0.0f ? rsqrtf(rho) : 0.0f);
}

// Block reduction of NV <= 16 per-atom float values into FP64, then one
// atomicAdd per value into dst[0..NV).  Within a warp the values are halved
// together (lanes 16 .. 31 take over values 8 .. 15, and so on): 16 shuffles
// instead of 5 NV, the same pairwise sums.
template <int NV, int NT>
__device__ __forceinline__ void block_reduce_add(float (&v)[NV], double *dst) {
    static_assert(NV <= 16, "one value per lane pair");
    __shared__ double s_part[NT / 32][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float w[16];
#pragma unroll
    for (int k = 0; k < 16; k++) w[k] = k < NV ? v[k < NV ? k : 0] : 0.0f;
#pragma unroll
    for (int d = 16, h = 8; h >= 1; d >>= 1, h >>= 1) {
        const bool up = lane & d;
#pragma unroll
        for (int k = 0; k < h; k++) {
            const float mine = up ? w[k + h] : w[k], other = up ? w[k] : w[k + h];
            w[k] = mine + __shfl_xor_sync(0xffffffffu, other, d);
        }
    }
    w[0] += __shfl_xor_sync(0xffffffffu, w[0], 1);
    if ((lane & 1) == 0) s_part[warp][lane >> 1] = (double)w[0];  // lane bits 16 8 4 2: the value's bits 8 4 2 1
    if (NT == 32) __syncwarp();
    else __syncthreads();
    if (threadIdx.x < NV) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < NT / 32; w++) s += s_part[w][threadIdx.x];
        atomicAdd(dst + threadIdx.x, s);
    }
}

// What follows the sums over an atom's neighbours (force f, virial w, energy pe):
// the embedding energy, the chain bonds, and the integration step or, in
// MODE_EVAL and MODE_FORCE, the result.  One thread per atom (own), NT threads per block;
// bonded[k] is the record of atom k of the cell.
template <int POT, int NT>
__device__ __forceinline__ void finish_atom(const KParams &p, const KArrays &a, int cur, int mode, int slot, int step_index,
                                            int c, int g, bool own, const float4 &xi, const ShiftTab &s_tab,
                                            const float4 *bonded, float fx, float fy, float fz, float w0, float w1,
                                            float w2, float w3, float w4, float w5, float pe) {
    if (own && POT == RC_POT_SC && xi.w > 0.0f) pe -= p.eps * p.sc_c / xi.w;  // embedding -eps c sqrt(rho_i)

    if (own && POT == RC_POT_KG) {
        // FENE + WCA on the (at most four) bond partners; each bond is seen from
        // both ends, so each end takes half of the virial and energy.
        const int4 pr = a.partner[g];
        const int q[4] = {pr.x, pr.y, pr.z, pr.w};
        const float *Hi = a.Hif + 8 * c;
#pragma unroll
        for (int b = 0; b < RC_MAX_BONDS; b++) {
            if (q[b] < 0) continue;
            const float4 xj = bonded[q[b]];
            // minimum image: pick the integer shift from fractional coordinates, then
            // form the displacement through the exact shift table
            const float ex = xj.x - xi.x, ey = xj.y - xi.y, ez = xj.z - xi.z;
            const float f2 = Hi[5] * ez, f1 = Hi[3] * ey + Hi[4] * ez, f0 = Hi[0] * ex + Hi[1] * ey + Hi[2] * ez;
            const int n0 = -(int)rintf(f0), n1 = -(int)rintf(f1), n2 = -(int)rintf(f2);
            if (n0 < -1 || n0 > 1 || n1 < -1 || n1 > 1 || n2 < -1 || n2 > 1) {
                rc_set_status(a.status, c, RC_EBOND);
                continue;
            }
            const float3 dd = rc_disp(xi, xj, s_tab, rc_image_slot(n0, n1, n2));
            const float dx = dd.x, dy = dd.y, dz = dd.z;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (!(r2 < p.R02)) {
                rc_set_status(a.status, c, RC_EBOND);
                continue;
            }
            const float ratio = r2 / p.R02;
            float gr = p.k_fene / (1.0f - ratio);
            float U = -0.5f * p.k_fene * p.R02 * log1pf(-ratio);
            if (r2 < p.wca2) {
                const float sr2 = p.sigma * p.sigma / r2, sr6 = sr2 * sr2 * sr2;
                gr -= 24.0f * p.eps * sr6 * (2.0f * sr6 - 1.0f) / r2;
                U += 4.0f * p.eps * sr6 * (sr6 - 1.0f) + p.eps;
            }
            fx = fmaf(gr, dx, fx);
            fy = fmaf(gr, dy, fy);
            fz = fmaf(gr, dz, fz);
            const float hx = -0.5f * gr * dx, hy = -0.5f * gr * dy;
            w0 = fmaf(hx, dx, w0);
            w1 = fmaf(hy, dy, w1);
            w2 = fmaf(-0.5f * gr * dz, dz, w2);
            w3 = fmaf(hx, dy, w3);
            w4 = fmaf(hx, dz, w4);
            w5 = fmaf(hy, dz, w5);
            pe += 0.5f * U;
        }
    }

    if (mode == MODE_EVAL) {
        if (own) a.f[g] = make_float4(fx, fy, fz, pe);
        float v[7] = {own ? pe : 0.f, own ? w0 : 0.f, own ? w1 : 0.f, own ? w2 : 0.f,
                      own ? w3 : 0.f, own ? w4 : 0.f, own ? w5 : 0.f};
        block_reduce_add<7, NT>(v, a.eval_acc + 8 * c);
        return;
    }

    if (mode == MODE_FORCE) {  // the sums over the cell that decide its next FIRE move
        float v[3] = {0.f, 0.f, 0.f};
        if (own) {
            const float4 vv = a.v[g];
            a.f[g] = make_float4(fx, fy, fz, 0.0f);
            // (explicit rounding: the minimiser's branches turn on these sums' last bits)
            v[0] = fmaf(fz, vv.z, fmaf(fx, vv.x, __fmul_rn(fy, vv.y)));
            v[1] = fmaf(vv.z, vv.z, fmaf(vv.x, vv.x, __fmul_rn(vv.y, vv.y)));
            v[2] = fmaf(fz, fz, fmaf(fx, fx, __fmul_rn(fy, fy)));
        }
        float f2max = v[2];
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) f2max = fmaxf(f2max, __shfl_xor_sync(0xffffffffu, f2max, d));
        if ((threadIdx.x & 31) == 0) atomicMax(&a.fire_fmax2[c], __float_as_uint(f2max));  // non-negative: ordered as their bits
        block_reduce_add<3, NT>(v, a.fire_acc + 4 * c);
        return;
    }

    // ---- velocity Verlet + Langevin ----
    float kxx = 0.f, kyy = 0.f, kzz = 0.f, kxy = 0.f, kxz = 0.f, kyz = 0.f;
    if (own) {
        float4 vv = a.v[g];
        float ax = fx * p.fm, ay = fy * p.fm, az = fz * p.fm;
        if (p.inv_tau > 0.0f) {
            const float3 z = rc_normals3((unsigned)a.tag[g], (unsigned)c, a.evals[c] + (unsigned long long)step_index,
                                         p.seed);
            ax += fmaf(-vv.x, p.inv_tau, p.noise * z.x);
            ay += fmaf(-vv.y, p.inv_tau, p.noise * z.y);
            az += fmaf(-vv.z, p.inv_tau, p.noise * z.z);
        }
        const float hdt = 0.5f * p.dt;
        if (mode != MODE_SETUP) {  // complete v(t)
            vv.x = fmaf(hdt, ax, vv.x);
            vv.y = fmaf(hdt, ay, vv.y);
            vv.z = fmaf(hdt, az, vv.z);
            kxx = p.mvv2e * vv.x * vv.x;
            kyy = p.mvv2e * vv.y * vv.y;
            kzz = p.mvv2e * vv.z * vv.z;
            kxy = p.mvv2e * vv.x * vv.y;
            kxz = p.mvv2e * vv.x * vv.z;
            kyz = p.mvv2e * vv.y * vv.z;
        }
        if (mode == MODE_LAST) {
            a.v[g] = vv;
        } else {
            vv.x = fmaf(hdt, ax, vv.x);
            vv.y = fmaf(hdt, ay, vv.y);
            vv.z = fmaf(hdt, az, vv.z);
            if (p.max_step > 0.0f) {
                const float s2 = p.dt * p.dt * (vv.x * vv.x + vv.y * vv.y + vv.z * vv.z);
                if (s2 > p.max_step * p.max_step) {
                    const float f = p.max_step * rsqrtf(s2);
                    vv.x *= f;
                    vv.y *= f;
                    vv.z *= f;
                }
            }
            float4 xn = make_float4(fmaf(p.dt, vv.x, xi.x), fmaf(p.dt, vv.y, xi.y), fmaf(p.dt, vv.z, xi.z), 0.0f);
            a.v[g] = vv;
            (cur ? a.x0 : a.x1)[g] = xn;
            const float4 xr0 = a.xref[g];
            const float ddx = xn.x - xr0.x, ddy = xn.y - xr0.y, ddz = xn.z - xr0.z;
            const float d2 = ddx * ddx + ddy * ddy + ddz * ddz;
            if (d2 > p.skin_half2) a.need_rebuild[c] = 1;
            const float step2 = p.dt * p.dt * (vv.x * vv.x + vv.y * vv.y + vv.z * vv.z);
            if (!(step2 <= p.skin_half2)) rc_set_status(a.status, c, isfinite(step2) ? RC_ELOST : RC_ENAN);
        }
    }
    if (slot >= 0) {
        float v[13] = {kxx, kyy, kzz, kxy, kxz, kyz,
                       own ? w0 : 0.f, own ? w1 : 0.f, own ? w2 : 0.f, own ? w3 : 0.f, own ? w4 : 0.f, own ? w5 : 0.f,
                       own ? pe : 0.f};
        block_reduce_add<13, NT>(v, a.series + ((size_t)c * a.series_cap + slot) * RC_SAMPLE_W);
    }
}

// Resident CTAs per SM the force kernel is compiled for at one lane per atom
// (caps its registers at 65536 / (128 * RC_FORCE_MIN_CTAS)).  7 keeps a
// 128 000-atom batch (1000 tiles) in one wave on 152 SMs; 1 leaves the
// register count to the compiler.  The lean walk takes 10 (48 registers), with a
// sample 8 (64 registers): on the 80 000 tiles of a 10.24 M-bead batch 12 (40
// registers) ran 1.3 times as long, the force step at 9 and 8 1 and 4 % longer,
// the sampling step at 7 and 6 7 % longer.
#ifndef RC_FORCE_MIN_CTAS
#define RC_FORCE_MIN_CTAS 7
#endif
constexpr int force_min_ctas(int tpa, bool sample) {
    return tpa == 0 ? (sample ? 8 : 10) : (RC_FORCE_MIN_CTAS / tpa > 0 ? RC_FORCE_MIN_CTAS / tpa : 1);
}

// WHAT the walk sums: the force alone in an MD step; force, virial and energy
// where a stress sample is recorded (slot >= 0) or in MODE_EVAL; the force alone,
// rounded as it is beside the virial, for the FIRE minimiser, whose branches turn
// on the last bit of f . v (160 000 beads: 80 us per iteration with the virial and
// a kernel of its own for the power sums, 68 us so).
enum { SUM_STEP = 0, SUM_ALL = 1, SUM_FORCE = 2 };
inline int what_of(int mode, int slot) {
    return slot >= 0 || mode == MODE_EVAL ? SUM_ALL : mode == MODE_FORCE ? SUM_FORCE : SUM_STEP;
}

template <int POT, int TPA, bool M6, bool STG, int WHAT>
__global__ void __launch_bounds__(RC_TILE *lanes_of(TPA), force_min_ctas(TPA, WHAT == SUM_ALL)) k_force(KParams p, KArrays a, int cur, int mode, int slot,
                                                       int step_index) {
    extern __shared__ __align__(16) float4 s_cell[];
    rc_pdl_wait();
    rc_pdl_trigger();
    const int t = tile_of_block(p, a);
    if (t < 0) return;
    const int c = a.tile_cell[t];
    if (a.status[c] != 0 || !a.active[c]) return;
    __shared__ ShiftTab s_tab;
    rc_load_shifts(s_tab, a.shift, c);

    const int at = threadIdx.x / lanes_of(TPA), sub = threadIdx.x % lanes_of(TPA);
    const int n = a.cell_n[c], off = a.cell_off[c];
    const int li = (t - a.cell_tile0[c]) * RC_TILE + at;
    const bool live = li < n;
    const int g = off + li;
    const float4 *__restrict__ X = cur ? a.x1 : a.x0;
    const float4 *__restrict__ XG = (POT == RC_POT_SC) ? a.xr : X;  // gathered array
    if (STG && !stage_records(s_cell, XG + off, n, a.status, c, p.wait_polls)) return;

    float fx = 0.f, fy = 0.f, fz = 0.f;
    float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;  // xx yy zz xy xz yz
    float pe = 0.f;
    float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) {
        xi = XG[g];
        const int nn = a.nnb[g];
        const int4 *__restrict__ nb = reinterpret_cast<const int4 *>(a.nbr) + (size_t)t * (p.max_nb / 4) * RC_TILE + at;
        auto body = [&](const float4 &xj, const float3 &d) {
            float e;
            const float gr = pair_term<POT, M6>(p, xi, xj, d, e);
            if (WHAT == SUM_STEP) {
                fx = fmaf(gr, d.x, fx);
                fy = fmaf(gr, d.y, fy);
                fz = fmaf(gr, d.z, fz);
                return;
            }
            const float gx = gr * d.x, gy = gr * d.y, gz = gr * d.z;
            fx = __fadd_rn(fx, gx);
            fy = __fadd_rn(fy, gy);
            fz = __fadd_rn(fz, gz);
            if (WHAT == SUM_ALL) {  // w, pe: scaled once per atom after the walk
                w0 = fmaf(gx, d.x, w0);
                w1 = fmaf(gy, d.y, w1);
                w2 = fmaf(gz, d.z, w2);
                w3 = fmaf(gx, d.y, w3);
                w4 = fmaf(gx, d.z, w4);
                w5 = fmaf(gy, d.z, w5);
                pe = __fadd_rn(pe, e);
            }
        };
        if (STG) for_each_neighbor<TPA>(nb, nn, sub, SharedSrc{s_cell, off}, xi, s_tab, body);
        else for_each_neighbor<TPA>(nb, nn, sub, GlobalSrc{XG}, xi, s_tab, body);
        if (WHAT == SUM_ALL) {
            pe *= POT == RC_POT_SC ? 0.5f * p.eps : 2.0f * p.eps;
            w0 *= -0.5f;
            w1 *= -0.5f;
            w2 *= -0.5f;
            w3 *= -0.5f;
            w4 *= -0.5f;
            w5 *= -0.5f;
        }
    }
    fx = sub_sum<TPA>(fx);
    fy = sub_sum<TPA>(fy);
    fz = sub_sum<TPA>(fz);
    if (WHAT == SUM_ALL) {
        w0 = sub_sum<TPA>(w0);
        w1 = sub_sum<TPA>(w1);
        w2 = sub_sum<TPA>(w2);
        w3 = sub_sum<TPA>(w3);
        w4 = sub_sum<TPA>(w4);
        w5 = sub_sum<TPA>(w5);
        pe = sub_sum<TPA>(pe);
    }
    const float4 *bonded = STG ? s_cell : X + off;
    finish_atom<POT, RC_TILE * lanes_of(TPA)>(p, a, cur, mode, slot, step_index, c, g, live && sub == 0, xi, s_tab, bonded,
                                              fx, fy, fz, w0, w1, w2, w3, w4, w5, pe);
}

// ---------------------------------------------------------------------------
// The cooperative walk, for batches too small to fill the chip: sixteen lanes
// share an atom, in CTAs of 32 atoms (a quarter of a tile).  Each lane evaluates
// one list entry of a round of sixteen and leaves the displacement and dE/dr / r
// in shared memory; then lane r < 10 adds component r of force, virial (xx yy zz
// xy xz yz) and energy over the sixteen entries in list order, four at a time per
// shared load, so that every sum has the bits of the one-lane walk and a batch
// can change between the two at any step.  The last round's missing entries are
// null entries.  The first warp then finishes the 32 atoms as k_force does.
// One lane per atom is a chain of one gather latency per group of four entries
// (236 entries in copper at skin 1.5 A) however few tiles there are: the 256-atom
// LJ cell's step takes 10.7 us instead of 16.3, that of three active 4000-atom
// copper cells of 32 takes 41 us instead of 93.
// ---------------------------------------------------------------------------
constexpr int COOP_LANES = 16, COOP_ATOMS = 32, COOP_THREADS = COOP_LANES * COOP_ATOMS;
constexpr int COOP_PER_TILE = RC_TILE / COOP_ATOMS, COOP_ROW = COOP_LANES + 4, COOP_COMP = COOP_ATOMS * COOP_ROW + 4;

// this CTA's tile, or -1
__device__ __forceinline__ int coop_tile(const KParams &p, const KArrays &a) {
    const int k = (int)(blockIdx.x / COOP_PER_TILE);
    if (!p.masked) return k < p.n_tiles ? k : -1;
    return k < *a.n_act ? a.act_tiles[k] : -1;
}

// The rounds of one atom's list (entry k at nb[(k / 4) 4 TILE + k % 4]; both
// atoms of a warp take the same number): eval(xj, d) on this lane's entry, then
// sum() with all sixteen results in place.  The next round's gathers are in
// flight meanwhile.
template <class Eval, class Sum>
__device__ __forceinline__ void coop_walk(const int *__restrict__ nb, int nn, unsigned self, const float4 *__restrict__ X,
                                          const float4 &xi, const ShiftTab &T, Eval &&eval, Sum &&sum) {
    const int l = threadIdx.x % COOP_LANES;
    int rounds = (nn + COOP_LANES - 1) / COOP_LANES;
    rounds = max(rounds, __shfl_xor_sync(0xffffffffu, rounds, COOP_LANES));
    const auto entry = [&](int r) {
        const int k = r * COOP_LANES + l;
        return k < nn ? (unsigned)__ldg(nb + (size_t)(k >> 2) * (4 * RC_TILE) + (k & 3)) : self | RC_SLOT_NULL << RC_IDX_BITS;
    };
    unsigned e = entry(0), en = entry(1);
    float4 xj = __ldg(X + (e & RC_IDX_MASK));
    for (int r = 0; r < rounds; r++) {
        const float4 xn = __ldg(X + (en & RC_IDX_MASK));
        const unsigned enn = entry(r + 2);
        const unsigned slot = e >> RC_IDX_BITS;
        eval(xj, __all_sync(0xffffffffu, slot == RC_SLOT_CENTRAL) ? rc_disp_central(xi, xj) : rc_disp(xi, xj, T, slot));
        __syncwarp();
        sum();
        __syncwarp();
        e = en;
        en = enn;
        xj = xn;
    }
}

template <bool M6, int CTAS>
__global__ void __launch_bounds__(COOP_THREADS, CTAS) k_density_coop(KParams p, KArrays a, int cur) {
    __shared__ ShiftTab s_tab;
    __shared__ __align__(16) float s_q[COOP_ATOMS][COOP_ROW];
    rc_pdl_wait();
    rc_pdl_trigger();
    const int t = coop_tile(p, a);
    if (t < 0) return;
    const int c = a.tile_cell[t];
    if (a.status[c] != 0 || !a.active[c]) return;
    rc_load_shifts(s_tab, a.shift, c);
    const int at = threadIdx.x / COOP_LANES, l = threadIdx.x % COOP_LANES;
    const int in_tile = (int)(blockIdx.x % COOP_PER_TILE) * COOP_ATOMS + at;
    const int li = (t - a.cell_tile0[c]) * RC_TILE + in_tile, n = a.cell_n[c], off = a.cell_off[c];
    const int g = off + min(li, n - 1);
    const float4 *__restrict__ X = cur ? a.x1 : a.x0;
    const float4 xi = X[g];
    float rho = 0.0f;
    coop_walk(a.nbr + (size_t)t * p.max_nb * RC_TILE + 4 * in_tile, li < n ? a.nnb[g] : 0, (unsigned)g, X, xi, s_tab,
              [&](const float4 &, const float3 &d) { s_q[at][l] = density_term<M6>(p, d); },
              [&] {
#pragma unroll
                  for (int k = 0; k < COOP_LANES; k += 4) {  // (every lane; lane 0's is used)
                      const float4 q = *reinterpret_cast<const float4 *>(&s_q[at][k]);
                      rho = density_sum<M6>(rho, q.x);
                      rho = density_sum<M6>(rho, q.y);
                      rho = density_sum<M6>(rho, q.z);
                      rho = density_sum<M6>(rho, q.w);
                  }
              });
    if (li < n && l == 0) a.xr[g] = make_float4(xi.x, xi.y, xi.z, rho > 0.0f ? rsqrtf(rho) : 0.0f);
}

template <int POT, bool M6, int WHAT, int CTAS>
__global__ void __launch_bounds__(COOP_THREADS, CTAS) k_force_coop(KParams p, KArrays a, int cur, int mode, int slot, int step_index) {
    __shared__ ShiftTab s_tab;
    __shared__ __align__(16) float s_pair[WHAT == SUM_ALL ? 5 : 4][COOP_COMP];  // d (3), dE/dr / r, energy: [atom][entry]
    __shared__ float s_sum[COOP_ATOMS][11];
    rc_pdl_wait();
    rc_pdl_trigger();
    const int t = coop_tile(p, a);
    if (t < 0) return;
    const int c = a.tile_cell[t];
    if (a.status[c] != 0 || !a.active[c]) return;
    rc_load_shifts(s_tab, a.shift, c);
    const int at = threadIdx.x / COOP_LANES, l = threadIdx.x % COOP_LANES;
    const int n = a.cell_n[c], off = a.cell_off[c];
    const int in0 = (int)(blockIdx.x % COOP_PER_TILE) * COOP_ATOMS, li0 = (t - a.cell_tile0[c]) * RC_TILE + in0;
    const float4 *__restrict__ X = cur ? a.x1 : a.x0;
    const float4 *__restrict__ XG = (POT == RC_POT_SC) ? a.xr : X;
    {
        const int li = li0 + at, g = off + min(li, n - 1);
        const float4 xi = XG[g];
        // lane r adds force component r, virial component r - 3 = (ia, ib), or the energy
        const int ia = l < 3 ? l : (l < 6 ? l - 3 : (l < 8 ? 0 : 1)), ib = l < 6 ? l - 3 : (l == 6 ? 1 : 2);
        const bool f = l < 3, w = l >= 3 && l < 9;
        const int row = at * COOP_ROW;
        const float *pa = &s_pair[l == 9 && WHAT == SUM_ALL ? 4 : ia][row], *pb = &s_pair[w ? ib : 0][row], *pg = &s_pair[3][row];
        float acc = 0.0f;
        const auto one = [&](float gr, float da, float db) {
            const float v = gr * da;
            if (WHAT == SUM_STEP) acc = fmaf(gr, da, acc);
            else if (WHAT == SUM_FORCE) acc = __fadd_rn(acc, v);
            else acc = w ? fmaf(v, db, acc) : __fadd_rn(acc, f ? v : da);
        };
        coop_walk(a.nbr + (size_t)t * p.max_nb * RC_TILE + 4 * (in0 + at), li < n ? a.nnb[g] : 0, (unsigned)g, XG, xi, s_tab,
                  [&](const float4 &xj, const float3 &d) {
                      float e;
                      const float gr = pair_term<POT, M6>(p, xi, xj, d, e);
                      s_pair[0][row + l] = d.x;
                      s_pair[1][row + l] = d.y;
                      s_pair[2][row + l] = d.z;
                      s_pair[3][row + l] = gr;
                      if (WHAT == SUM_ALL) s_pair[WHAT == SUM_ALL ? 4 : 0][row + l] = e;
                  },
                  [&] {
                      if (l < (WHAT == SUM_ALL ? 10 : 3)) {
#pragma unroll
                          for (int k = 0; k < COOP_LANES; k += 4) {
                              const float4 gr = *reinterpret_cast<const float4 *>(pg + k),
                                           da = *reinterpret_cast<const float4 *>(pa + k);
                              float4 db = da;
                              if (WHAT == SUM_ALL) db = *reinterpret_cast<const float4 *>(pb + k);
                              one(gr.x, da.x, db.x);
                              one(gr.y, da.y, db.y);
                              one(gr.z, da.z, db.z);
                              one(gr.w, da.w, db.w);
                          }
                      }
                  });
        if (l < (WHAT == SUM_ALL ? 10 : 3)) s_sum[at][l] = acc;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x, li = li0 + lane, g = off + min(li, n - 1);
    const float *r = s_sum[lane];
    float w[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (WHAT == SUM_ALL) {
#pragma unroll
        for (int k = 0; k < 6; k++) w[k] = -0.5f * r[3 + k];
        w[6] = (POT == RC_POT_SC ? 0.5f * p.eps : 2.0f * p.eps) * r[9];
    }
    finish_atom<POT, 32>(p, a, cur, mode, slot, step_index, c, g, li < n, XG[g], s_tab, X + off, r[0], r[1], r[2], w[0], w[1],
                         w[2], w[3], w[4], w[5], w[6]);
}

// Eq. PK1 (Sec. 2.2): per cell, the sum over ordered pairs inside rc of
// dE/dr_ij r_ij (x) R_ij / r_ij with R_ij = M r_ij, M = H(0) H^{-1} (upper
// triangular, m[6] per cell: m00 m01 m02 m11 m12 m22), plus the Kremer-Grest
// bonds, each seen from both ends.  FP32 per atom, FP64 per cell into
// acc[9 c + 3 a + b]; the caller scales by 1 / (2 Omega_0).
template <int POT, bool M6>
__global__ void __launch_bounds__(RC_TILE) k_static_pk1(KParams p, KArrays a, int cur, const float *__restrict__ mcell,
                                                        double *acc) {
    const int t = blockIdx.x;
    const int c = a.tile_cell[t];
    if (a.status[c] != 0 || !a.active[c]) return;
    __shared__ ShiftTab s_tab;
    rc_load_shifts(s_tab, a.shift, c);
    const float *m = mcell + 6 * c;
    const float m00 = m[0], m01 = m[1], m02 = m[2], m11 = m[3], m12 = m[4], m22 = m[5];
    const int n = a.cell_n[c], off = a.cell_off[c];
    const int li = (t - a.cell_tile0[c]) * RC_TILE + threadIdx.x;
    const int g = off + li;
    const float4 *__restrict__ X = cur ? a.x1 : a.x0;
    const float4 *__restrict__ XG = (POT == RC_POT_SC) ? a.xr : X;
    float T[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    auto add = [&](float gr, const float3 &d) {  // gr = dE/dr / r
        const float R0 = fmaf(m00, d.x, fmaf(m01, d.y, m02 * d.z)), R1 = fmaf(m11, d.y, m12 * d.z), R2 = m22 * d.z;
        const float gx = gr * d.x, gy = gr * d.y, gz = gr * d.z;
        T[0] = fmaf(gx, R0, T[0]); T[1] = fmaf(gx, R1, T[1]); T[2] = fmaf(gx, R2, T[2]);
        T[3] = fmaf(gy, R0, T[3]); T[4] = fmaf(gy, R1, T[4]); T[5] = fmaf(gy, R2, T[5]);
        T[6] = fmaf(gz, R0, T[6]); T[7] = fmaf(gz, R1, T[7]); T[8] = fmaf(gz, R2, T[8]);
    };
    if (li < n) {
        const float4 xi = XG[g];
        const int nn = a.nnb[g];
        const int4 *__restrict__ nb =
            reinterpret_cast<const int4 *>(a.nbr) + (size_t)t * (p.max_nb / 4) * RC_TILE + threadIdx.x;
        for_each_neighbor<1>(nb, nn, 0, GlobalSrc{XG}, xi, s_tab, [&](const float4 &xj, const float3 &d) {
            float e;
            add(pair_term<POT, M6>(p, xi, xj, d, e), d);
        });
        if (POT == RC_POT_KG) {
            const int4 pr = a.partner[g];
            const int q[4] = {pr.x, pr.y, pr.z, pr.w};
            const float *Hi = a.Hif + 8 * c;
#pragma unroll
            for (int b = 0; b < RC_MAX_BONDS; b++) {
                if (q[b] < 0) continue;
                const float4 xj = X[off + q[b]];
                const float ex = xj.x - xi.x, ey = xj.y - xi.y, ez = xj.z - xi.z;
                const float f2 = Hi[5] * ez, f1 = Hi[3] * ey + Hi[4] * ez, f0 = Hi[0] * ex + Hi[1] * ey + Hi[2] * ez;
                const int n0 = -(int)rintf(f0), n1 = -(int)rintf(f1), n2 = -(int)rintf(f2);
                if (n0 < -1 || n0 > 1 || n1 < -1 || n1 > 1 || n2 < -1 || n2 > 1) continue;
                const float3 dd = rc_disp(xi, xj, s_tab, rc_image_slot(n0, n1, n2));
                const float r2 = fmaf(dd.x, dd.x, fmaf(dd.y, dd.y, dd.z * dd.z));
                if (!(r2 < p.R02)) continue;
                float gr = p.k_fene / (1.0f - r2 / p.R02);
                if (r2 < p.wca2) {
                    const float sr2 = p.sigma * p.sigma / r2, sr6 = sr2 * sr2 * sr2;
                    gr -= 24.0f * p.eps * sr6 * (2.0f * sr6 - 1.0f) / r2;
                }
                add(gr, dd);
            }
        }
    }
    block_reduce_add<9, RC_TILE>(T, acc + 9 * c);
}

template <class K>
void set_smem(K kernel, int bytes) {
    if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <int POT, bool M6, bool STG, int WHAT>
void launch_force_tpa(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int mode, int slot,
                      int step_index, int smem, cudaStream_t s) {
    switch (tpa) {
    case 0: rc_launch_pdl(k_force<POT, 0, M6, STG, WHAT>, pair_grid(p), RC_TILE * 1, smem, s, 1, p, a, cur, mode, slot, step_index); break;
    case 1: rc_launch_pdl(k_force<POT, 1, M6, STG, WHAT>, pair_grid(p), RC_TILE * 1, smem, s, 1, p, a, cur, mode, slot, step_index); break;
    case 2: rc_launch_pdl(k_force<POT, 2, M6, STG, WHAT>, pair_grid(p), RC_TILE * 2, smem, s, 1, p, a, cur, mode, slot, step_index); break;
    case 4: rc_launch_pdl(k_force<POT, 4, M6, STG, WHAT>, pair_grid(p), RC_TILE * 4, smem, s, 1, p, a, cur, mode, slot, step_index); break;
    default: rc_launch_pdl(k_force<POT, 8, M6, STG, WHAT>, pair_grid(p), RC_TILE * 8, smem, s, 1, p, a, cur, mode, slot, step_index); break;
    }
}

template <int POT, bool M6, bool STG>
void launch_force_pot(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int mode, int slot,
                      int step_index, int smem, cudaStream_t s) {
    const int what = what_of(mode, slot);
    if constexpr (!STG) {
        if (what == SUM_FORCE) {
            launch_force_tpa<POT, M6, STG, SUM_FORCE>(p, a, cur, n_tiles, tpa, mode, slot, step_index, smem, s);
            return;
        }
    }
    if (what == SUM_STEP)
        launch_force_tpa<POT, M6, STG, SUM_STEP>(p, a, cur, n_tiles, tpa, mode, slot, step_index, smem, s);
    else  // (with staging, the minimiser too)
        launch_force_tpa<POT, M6, STG, SUM_ALL>(p, a, cur, n_tiles, tpa, mode, slot, step_index, smem, s);
}

template <bool M6, bool STG>
void launch_density_m(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int smem, cudaStream_t s) {
    switch (tpa) {
    case 0: rc_launch_pdl(k_density<0, M6, STG>, pair_grid(p), RC_TILE * 1, smem, s, 1, p, a, cur); break;
    case 1: rc_launch_pdl(k_density<1, M6, STG>, pair_grid(p), RC_TILE * 1, smem, s, 1, p, a, cur); break;
    case 2: rc_launch_pdl(k_density<2, M6, STG>, pair_grid(p), RC_TILE * 2, smem, s, 1, p, a, cur); break;
    case 4: rc_launch_pdl(k_density<4, M6, STG>, pair_grid(p), RC_TILE * 4, smem, s, 1, p, a, cur); break;
    default: rc_launch_pdl(k_density<8, M6, STG>, pair_grid(p), RC_TILE * 8, smem, s, 1, p, a, cur); break;
    }
}

template <int POT, bool M6, int WHAT>
void prepare_pot_s(int bytes) {
    set_smem(k_force<POT, 0, M6, true, WHAT>, bytes);
    set_smem(k_force<POT, 1, M6, true, WHAT>, bytes);
    set_smem(k_force<POT, 2, M6, true, WHAT>, bytes);
    set_smem(k_force<POT, 4, M6, true, WHAT>, bytes);
    set_smem(k_force<POT, 8, M6, true, WHAT>, bytes);
}

template <int POT, bool M6>
void prepare_pot(int bytes) {
    prepare_pot_s<POT, M6, SUM_ALL>(bytes);
    prepare_pot_s<POT, M6, SUM_STEP>(bytes);
}

template <bool M6>
void prepare_density(int bytes) {
    set_smem(k_density<0, M6, true>, bytes);
    set_smem(k_density<1, M6, true>, bytes);
    set_smem(k_density<2, M6, true>, bytes);
    set_smem(k_density<4, M6, true>, bytes);
    set_smem(k_density<8, M6, true>, bytes);
}

}  // namespace

int rc_stage_max_atoms() { return RC_STAGE_MAX_ATOMS; }

void rc_prepare_staged(int max_cell_atoms) {
    const int bytes = max_cell_atoms * 16;
    prepare_pot<RC_POT_SC, true>(bytes);
    prepare_pot<RC_POT_SC, false>(bytes);
    prepare_pot<RC_POT_LJ, false>(bytes);
    prepare_pot<RC_POT_KG, false>(bytes);
    prepare_density<true>(bytes);
    prepare_density<false>(bytes);
}

// Largest number of tiles for which the cooperative walk is taken: it executes
// more instructions than one lane per atom and wins while those leave the chip
// idle.  us per MD step, one lane / cooperative: LJ copper 18 / 14 (28 tiles),
// 37 / 21 (70), 43 / 33 (140), 49 / 47 (280), 52 / 58 (420); Sutton-Chen 67 / 32
// (64), 99 / 68 (224), 110 / 95 (320), 140 / 177 (640); Kremer-Grest 32 / 18 (80),
// 46 / 40 (240), 47 / 46 (320), 52 / 64 (480).  One line for the three potentials,
// where LJ and Kremer-Grest cross; Sutton-Chen crosses between 320 and 640 tiles, so
// just above the line it runs a tenth longer than it could.
int rc_coop_max_tiles(int n_sm) { return 2 * n_sm; }

namespace {
// CTAs per SM it is compiled for: two (64 registers) while they hold the whole
// batch, else three (40 registers; Kremer-Grest, 240 tiles: 44 -> 40 us)
bool coop_two(const KParams &p, int coop_tiles) { return coop_tiles * COOP_PER_TILE <= 2 * p.n_sm; }
}  // namespace

void rc_launch_density(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int stage_atoms, int coop_tiles,
                       cudaStream_t s) {
    const bool m6 = p.sc_m == 6.0f;
    const int smem = stage_atoms * 16;
    if (coop_tiles > 0) {
        const auto k = coop_two(p, coop_tiles) ? (m6 ? k_density_coop<true, 2> : k_density_coop<false, 2>)
                                               : (m6 ? k_density_coop<true, 3> : k_density_coop<false, 3>);
        rc_launch_pdl(k, coop_tiles * COOP_PER_TILE, COOP_THREADS, 0, s, 1, p, a, cur);
    } else if (stage_atoms > 0) {
        if (m6) launch_density_m<true, true>(p, a, cur, n_tiles, tpa, smem, s);
        else launch_density_m<false, true>(p, a, cur, n_tiles, tpa, smem, s);
    } else {
        if (m6) launch_density_m<true, false>(p, a, cur, n_tiles, tpa, 0, s);
        else launch_density_m<false, false>(p, a, cur, n_tiles, tpa, 0, s);
    }
}

namespace {

template <int POT, bool M6>
void launch_force(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int mode, int slot, int step_index,
                  int stage_atoms, int coop_tiles, cudaStream_t s) {
    const int what = what_of(mode, slot);
    if (coop_tiles > 0) {
        const auto k = coop_two(p, coop_tiles)
                           ? (what == SUM_ALL     ? k_force_coop<POT, M6, SUM_ALL, 2>
                              : what == SUM_FORCE ? k_force_coop<POT, M6, SUM_FORCE, 2>
                                                  : k_force_coop<POT, M6, SUM_STEP, 2>)
                           : (what == SUM_ALL     ? k_force_coop<POT, M6, SUM_ALL, 3>
                              : what == SUM_FORCE ? k_force_coop<POT, M6, SUM_FORCE, 3>
                                                  : k_force_coop<POT, M6, SUM_STEP, 3>);
        rc_launch_pdl(k, coop_tiles * COOP_PER_TILE, COOP_THREADS, 0, s, 1, p, a, cur, mode, slot, step_index);
    } else if (stage_atoms > 0)
        launch_force_pot<POT, M6, true>(p, a, cur, n_tiles, tpa, mode, slot, step_index, stage_atoms * 16, s);
    else
        launch_force_pot<POT, M6, false>(p, a, cur, n_tiles, tpa, mode, slot, step_index, 0, s);
}

}  // namespace

void rc_launch_force(const KParams &p, const KArrays &a, int cur, int n_tiles, int tpa, int mode, int slot,
                     int step_index, int stage_atoms, int coop_tiles, cudaStream_t s) {
    const auto go = p.pot == RC_POT_KG   ? launch_force<RC_POT_KG, false>
                    : p.pot == RC_POT_LJ ? launch_force<RC_POT_LJ, false>
                    : p.sc_m == 6.0f && p.sc_n == 9.0f ? launch_force<RC_POT_SC, true>
                                                       : launch_force<RC_POT_SC, false>;
    go(p, a, cur, n_tiles, tpa, mode, slot, step_index, stage_atoms, coop_tiles, s);
}

void rc_launch_static_pk1(const KParams &p, const KArrays &a, int cur, int n_tiles, const float *mcell, double *acc,
                          cudaStream_t s) {
    if (p.pot == RC_POT_SC) {
        if (p.sc_m == 6.0f && p.sc_n == 9.0f) k_static_pk1<RC_POT_SC, true><<<n_tiles, RC_TILE, 0, s>>>(p, a, cur, mcell, acc);
        else k_static_pk1<RC_POT_SC, false><<<n_tiles, RC_TILE, 0, s>>>(p, a, cur, mcell, acc);
    } else if (p.pot == RC_POT_KG) {
        k_static_pk1<RC_POT_KG, false><<<n_tiles, RC_TILE, 0, s>>>(p, a, cur, mcell, acc);
    } else {
        k_static_pk1<RC_POT_LJ, false><<<n_tiles, RC_TILE, 0, s>>>(p, a, cur, mcell, acc);
    }
}
