// Neighbour-list build for triclinic r-cells (one list per cell, all cells of a
// batch in one launch of each kernel).
//
//  k_sort  : one thread-block cluster per rebuilt r-cell, or one CTA where many
//            small ones rebuild.  Wraps positions into
//            the current box through fractional coordinates, bins atoms on an
//            n0 x n1 x n2 grid over the fractional cube (n_d = floor(2 w_d /
//            r_list), w_d the perpendicular width: bins at least r_list / 2
//            wide), counting-sorts them by bin (stable, so the order is
//            deterministic) and permutes every per-atom array.
//  k_nlist : one warp per four atoms.  The candidates are the 5 x 5 x 5 bins
//            around an atom's own with explicit periodic image shifts (about 0.58 of
//            the candidates of 27 bins r_list wide), less the bins that lie
//            wholly beyond r_list; with n_d >= 2 (w_d >= 2 r_list gives
//            n_d >= 4) the offsets -2..2 map to distinct (bin, image) pairs
//            with images in -1..1, so each (j, image) within r_list is stored
//            exactly once.
//
// Both are bound by latency, not by a rate: in most MD steps a few cells
// rebuild, at steps of their own, and the step waits for the slowest of them.
// So one cell is spread over many SMs, and neither kernel's grid grows with the
// batch (no block per tile that only finds that its cell has nothing to do).
#include <cooperative_groups.h>

#include <type_traits>

#include "rc_internal.cuh"

namespace {

namespace cg = cooperative_groups;

// The cells of a batch for which flag(c) holds, in order, at most LIST_CAP from
// cell `from` on, into s_list by the whole block; returns their number and sets
// `next` to the first cell not looked at.
constexpr int LIST_CAP = 1024;
template <class Flag>
__device__ __forceinline__ int compact_cells(int *s_list, int *s_warp, int n_cells, int from, Flag &&flag) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int to = min(n_cells, from + LIST_CAP);
    int total = 0;
    for (int c0 = from; c0 < to; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const bool on = c < to && flag(c);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) s_warp[warp] = __popc(m);
        __syncthreads();
        int before = total;
        for (int w = 0; w < nw; w++) {
            const int k = s_warp[w];
            if (w < warp) before += k;
            total += k;
        }
        if (on) s_list[before + __popc(m & ((1u << lane) - 1u))] = c;
        __syncthreads();
    }
    return total;
}

// ---------------------------------------------------------------------------
// k_sort.  A cluster of SORT_CL CTAs sorts one cell: the bin counters are
// spread over the CTAs' shared memory (bin b in CTA b / per), counted with
// atomics on distributed shared memory.  Where more cells rebuild than there are
// clusters and they are small (spread_pays), each CTA sorts a cell of its own
// instead, with all counters in its shared memory.  Either way the value an atomic
// returns is an atom's arrival number in its bin, which depends on timing.  So the
// atoms of a bin are first listed in arrival order, and each then takes its place by
// the number of atoms of the bin that precede it in the current order: a stable,
// deterministic order without a serial pass (bins hold a few atoms).
// Measured per MD step: 32 cells of 5000 beads, two or three of which rebuild in
// a step, 29.8 -> 14.7 us against one CTA per cell with a serial one-warp ranking
// (64 cells of 5000 to 20000 beads: 96 -> 24 us).  A full sort of 320 000 beads
// takes 46 us, of one 256-atom cell about 15 us (six cluster barriers and their
// dependent loads).
// ---------------------------------------------------------------------------
constexpr int SORT_CL = 8, SORT_THREADS = 512;
constexpr int SORT_SCAN = 2 * SORT_THREADS;  // bins the block scans at a time
static_assert(RC_MAX_BINS_PER_CELL / SORT_CL % SORT_SCAN == 0, "the scan takes whole rounds");

// exclusive scan of s[0 .. n) in place (n a multiple of SORT_SCAN), returns the total
__device__ __forceinline__ int block_exclusive_scan(int *s, int n, int *s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int total = 0;
    for (int b0 = 2 * threadIdx.x; b0 < n; b0 += SORT_SCAN) {
        const int a = s[b0], b = s[b0 + 1];
        int v = a + b;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += y;
        }
        if (lane == 31) s_warp[warp] = v;
        __syncthreads();
        int base = total;
        for (int w = 0; w < SORT_THREADS / 32; w++) {
            const int k = s_warp[w];
            if (w < warp) base += k;
            total += k;
        }
        s[b0] = base + v - a - b;
        s[b0 + 1] = base + v - b;
        __syncthreads();
    }
    return total;
}

// Cell c, by the cluster (SPREAD; this is its CTA `rank`) or by this CTA alone;
// BATCH atoms per thread whose loads are issued together.
template <bool SPREAD, int BATCH>
__device__ void sort_cell(const KParams &p, const KArrays &a, int cur, int c, int rank, int *s_cnt, int *s_warp,
                          int *s_total, cg::cluster_group &cluster) {
    constexpr int SPAN = SPREAD ? SORT_CL * SORT_THREADS : SORT_THREADS;
    const auto sync = [&] {
        if constexpr (SPREAD) cluster.sync();
        else __syncthreads();
    };
    const int n = a.cell_n[c], off = a.cell_off[c];
    const int nb0 = a.nbins[4 * c], nb1 = a.nbins[4 * c + 1], nb2 = a.nbins[4 * c + 2];
    const int nbt = nb0 * nb1 * nb2, per = SPREAD ? (nbt + SORT_CL - 1) / SORT_CL : nbt;  // bins of a CTA
    const int scan = (per + SORT_SCAN - 1) / SORT_SCAN * SORT_SCAN;
    const float *H = a.Hf + 8 * c, *Hi = a.Hif + 8 * c;
    const float h00 = H[0], h01 = H[1], h02 = H[2], h11 = H[3], h12 = H[4], h22 = H[5];
    const float i00 = Hi[0], i01 = Hi[1], i02 = Hi[2], i11 = Hi[3], i12 = Hi[4], i22 = Hi[5];
    float4 *X = cur ? a.x1 : a.x0;
    const bool kg = p.pot == RC_POT_KG;
    const int me = (SPREAD ? rank * SORT_THREADS : 0) + threadIdx.x;
    int *bs = a.bin_start + a.bin_off[c];
    const auto counter = [&](int bin) {
        if constexpr (SPREAD) return cluster.map_shared_rank(s_cnt, bin / per) + bin % per;
        else return s_cnt + bin;
    };

    for (int b = threadIdx.x; b < scan; b += SORT_THREADS) s_cnt[b] = 0;
    sync();
    // wrap, bin and count; a copy of every per-atom array into the staging arrays,
    // BATCH atoms per thread at a time, all their loads issued before any store
    for (int i0 = me; i0 < n; i0 += SPAN * BATCH) {
        float4 xb[BATCH], vb[BATCH];
        int tb[BATCH];
        int4 pb[BATCH];
#pragma unroll
        for (int k = 0; k < BATCH; k++) {
            const int i = i0 + k * SPAN;
            if (i < n) {
                xb[k] = X[off + i];
                vb[k] = a.v[off + i];
                tb[k] = a.tag[off + i];
                if (kg) pb[k] = a.partner[off + i];
            }
        }
#pragma unroll
        for (int k = 0; k < BATCH; k++) {
            const int i = i0 + k * SPAN;
            if (i >= n) break;
            const int g = off + i;
            const float4 x = xb[k];
            float s2 = i22 * x.z, s1 = i11 * x.y + i12 * x.z, s0 = i00 * x.x + i01 * x.y + i02 * x.z;
            float f0 = floorf(s0), f1 = floorf(s1), f2 = floorf(s2);
            float w0 = s0 - f0, w1 = s1 - f1, w2 = s2 - f2;
            float xw = x.x - (h00 * f0 + h01 * f1 + h02 * f2);
            float yw = x.y - (h11 * f1 + h12 * f2);
            float zw = x.z - h22 * f2;
            int b0 = min(max((int)(w0 * nb0), 0), nb0 - 1);
            int b1 = min(max((int)(w1 * nb1), 0), nb1 - 1);
            int b2 = min(max((int)(w2 * nb2), 0), nb2 - 1);
            int bin = (b0 * nb1 + b1) * nb2 + b2;
            a.x_tmp[g] = make_float4(xw, yw, zw, 0.0f);
            a.binid[g] = bin;
            a.v_tmp[g] = vb[k];
            a.tag_tmp[g] = tb[k];
            if (kg) a.partner_tmp[g] = pb[k];
            a.newpos[g] = atomicAdd(counter(bin), 1);  // arrival number, replaced by the place below
        }
    }
    sync();
    // first atom of every bin: scan of the CTA's bins, plus the totals of the CTAs before
    const int own = block_exclusive_scan(s_cnt, scan, s_warp), bin0 = SPREAD ? rank * per : 0;
    int base = 0;
    if constexpr (SPREAD) {
        if (threadIdx.x == 0) *s_total = own;
        sync();
        for (int r = 0; r < rank; r++) base += *cluster.map_shared_rank(s_total, r);
    }
    for (int b = threadIdx.x; b < per && bin0 + b < nbt; b += SORT_THREADS) {
        const int v = s_cnt[b] + base;
        s_cnt[b] = v;
        bs[bin0 + b] = v;
    }
    if (bin0 == 0 && threadIdx.x == 0) bs[nbt] = n;
    sync();
    // the atoms of every bin in arrival order
    for (int i = me; i < n; i += SPAN) a.oldidx[off + *counter(a.binid[off + i]) + a.newpos[off + i]] = i;
    sync();
    // every atom to its place: the first of its bin plus the number of its
    // bin's atoms before it.  Another CTA's writes are read past the L1 cache.
    for (int i0 = me; i0 < n; i0 += SPAN * BATCH) {
        int bb[BATCH], tb[BATCH];
        float4 xb[BATCH], vb[BATCH];
#pragma unroll
        for (int k = 0; k < BATCH; k++) {
            const int i = i0 + k * SPAN;
            if (i < n) {
                const int g = off + i;
                bb[k] = a.binid[g];
                xb[k] = a.x_tmp[g];
                vb[k] = a.v_tmp[g];
                tb[k] = a.tag_tmp[g];
            }
        }
#pragma unroll
        for (int k = 0; k < BATCH; k++) {
            const int i = i0 + k * SPAN;
            if (i >= n) break;
            const int lo = __ldcg(bs + bb[k]), hi = __ldcg(bs + bb[k] + 1);
            int q = lo;
            for (int s = lo; s < hi; s++) q += __ldcg(a.oldidx + off + s) < i ? 1 : 0;
            a.newpos[off + i] = q;
            q += off;
            X[q] = xb[k];
            a.xref[q] = xb[k];
            a.v[q] = vb[k];
            a.tag[q] = tb[k];
            const int b2 = bb[k] % nb2, b01 = bb[k] / nb2;
            a.bin_of[q] = (b01 / nb1) << 20 | (b01 % nb1) << 10 | b2;
        }
    }
    if (kg) {  // bonded partners renumbered
        sync();
        for (int i0 = me; i0 < n; i0 += SPAN * BATCH) {
            int4 pb[BATCH];
            int qb[BATCH];
#pragma unroll
            for (int k = 0; k < BATCH; k++) {
                const int i = i0 + k * SPAN;
                if (i < n) {
                    pb[k] = a.partner_tmp[off + i];
                    qb[k] = a.newpos[off + i];
                }
            }
#pragma unroll
            for (int k = 0; k < BATCH; k++) {
                const int i = i0 + k * SPAN;
                if (i < n) {
                    const int4 pr = pb[k];
                    const int *np = a.newpos + off;
                    a.partner[off + qb[k]] =
                        make_int4(pr.x >= 0 ? __ldcg(np + pr.x) : -1, pr.y >= 0 ? __ldcg(np + pr.y) : -1,
                                  pr.z >= 0 ? __ldcg(np + pr.z) : -1, pr.w >= 0 ? __ldcg(np + pr.w) : -1);
                }
            }
        }
    }
    sync();  // no CTA's counters change while another one reads them
}

// Whether n_go cells are sorted sooner by the n_cl clusters, in turn, than by one
// CTA each (the CTAs in turn, and no sooner than the largest cell): the same answer
// in every CTA.  Times of one cell in us: by a cluster 9 + 0.8 per thousand atoms,
// by a CTA 6 + 5.  A sort of all cells, all by clusters / as chosen here: 64 cells of
// 256 atoms 28 / 12 us, 1024 of 256 457 / 37, 48 of 2048 29 / 19, 48 of 4000 31 / 28
// (clusters), 256 of 4000 149 / 40, 1024 of 500 beads 598 / 48; a step of 1024 cells of
// 256 atoms, 44 of which rebuild in it, 111 / 97.
__device__ __forceinline__ bool spread_pays(const KArrays &a, const int *s_list, int n_go, int n_cl, int *s_warp, int *s_max) {
    int sum = 0, top = 0;
    for (int k = threadIdx.x; k < n_go; k += SORT_THREADS) {
        const int n = a.cell_n[s_list[k]];
        sum += n;
        top = max(top, n);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, d);
        top = max(top, __shfl_xor_sync(0xffffffffu, top, d));
    }
    if ((threadIdx.x & 31) == 0) {
        s_warp[threadIdx.x >> 5] = sum;
        s_max[threadIdx.x >> 5] = top;
    }
    __syncthreads();
    sum = top = 0;
    for (int w = 0; w < SORT_THREADS / 32; w++) {
        sum += s_warp[w];
        top = max(top, s_max[w]);
    }
    __syncthreads();
    const int n_ctas = n_cl * SORT_CL;
    const float mean = (float)sum / n_go;
    const float spread = ((n_go + n_cl - 1) / n_cl) * (9.0f + 0.8e-3f * mean);
    const float alone = fmaxf(((n_go + n_ctas - 1) / n_ctas) * (6.0f + 5e-3f * mean), 6.0f + 5e-3f * top);
    return spread <= alone;
}

// MANY: a batch of more cells than there are clusters, none of more atoms than a
// cluster has threads.  It has both ways to sort a cell, at one atom per thread
// and without a spill (at two it spills more than the other one, 64 cells of 5000 to
// 20 000 beads run 1 % longer); the other one has clusters only.
template <bool MANY>
__global__ void __launch_bounds__(SORT_THREADS, 2) k_sort(KParams p, KArrays a, int cur, int n_cells) {
    __shared__ int s_cnt[MANY ? RC_MAX_BINS_PER_CELL : RC_MAX_BINS_PER_CELL / SORT_CL];
    __shared__ int s_list[LIST_CAP], s_warp[SORT_THREADS / 32], s_max[SORT_THREADS / 32], s_total;
    rc_pdl_wait();
    rc_pdl_trigger();
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = blockIdx.x % SORT_CL, id = blockIdx.x / SORT_CL, n_cl = gridDim.x / SORT_CL;
    int next = blockIdx.x;  // this CTA's next cell to sort alone
    // the cells to rebuild: the same list in every CTA (k_nlist, after this
    // kernel, clears their flags), dealt to the clusters or CTAs in turn
    for (int from = 0; from < n_cells; from += LIST_CAP) {
        const int n_go = compact_cells(s_list, s_warp, n_cells, from, [&](int c) {
            const bool go = a.need_rebuild[c] && a.status[c] == 0 && a.active[c];
            if (blockIdx.x == 0) a.built[c] = go;
            return go;
        });
        if (!MANY || n_go <= n_cl || spread_pays(a, s_list, n_go, n_cl, s_warp, s_max)) {
            for (int k = id; k < n_go; k += n_cl)
                sort_cell<true, MANY ? 1 : 2>(p, a, cur, s_list[k], rank, s_cnt, s_warp, &s_total, cluster);
        } else {
            for (; next < n_go; next += gridDim.x)
                sort_cell<false, 1>(p, a, cur, s_list[next], 0, s_cnt, s_warp, &s_total, cluster);
            next -= n_go;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// k_nlist.  A warp builds the lists of NL_ATOMS consecutive atoms (sorted by
// bin, so they are neighbours along the third axis; atoms of another bin row are
// taken in a round of their own).  Lane r < 25 takes row (o0, o1) = (r / 5 - 2,
// r % 5 - 2) of the stencil: bins are numbered with the third index fastest, so
// the bins of a row that the atoms need, two on either side of them, are one
// contiguous range of sorted atoms, in up to three segments by their image along
// the third axis (the unwrapped bins, those wrapped below 0 and above n2 - 1).
// The lane drops the bins at its row's ends that are farther than r_list from
// the atoms' bounding box, a scan over the lanes gives every row's place, and
// the rows' candidates -- index and image slot, the very list entry -- go to a
// window in shared memory, NL_WIN at a time.  Then the 32 lanes load one
// candidate each, test it against every atom and append it to the lists of those
// within r_list in order (ballot), so a list is the one a single thread would
// have made: central-image entries first (the pair kernels' fast path), then the
// images, row by row.  The end of each list is a ring of 64 entries in shared
// memory, written out as whole groups of four, 32 entries at a time; the last
// group is filled up with null entries (RC_SLOT_NULL).
// Bound by the instructions of the candidate tests (about 380 candidates in 12
// rounds per four beads at r_list = 2.9 sigma) at the 16 warps per SM that 128
// registers allow; 24 warps at 80 registers spill and run 17 % slower, one atom
// per warp 40 %.  Measured per MD step against one thread per atom, whose segments diverged
// from its neighbours' and whose entries went out as scattered 4-byte stores:
// 32 cells of 5000 beads 79.8 -> 21.5 us, 64 cells of 5000 to 20000 beads 144
// -> 48 us, 512 cells of 20000 beads 989 -> 751 us (0.95 ns per bead rebuilt).
// ---------------------------------------------------------------------------
constexpr int NL_CTAS = 2, NL_THREADS = 256, NL_WARPS = NL_THREADS / 32, NL_WIN = 640, NL_ATOMS = 4, NL_PIECE = 8, NL_RING = 64;
constexpr int NL_GROUP = NL_WARPS * NL_ATOMS;  // atoms a CTA takes at a time
constexpr int NL_CELLS = LIST_CAP / NL_THREADS, NL_WALK = 8;
constexpr unsigned NL_FULL = 0xffffffffu;

// smallest |v| of an interval [lo, hi]
__device__ __forceinline__ float gap(float lo, float hi) { return fmaxf(fmaxf(lo, -hi), 0.0f); }

template <bool KG>
__global__ void __launch_bounds__(NL_THREADS, NL_CTAS) k_nlist(KParams p, KArrays a, int cur, int n_cells) {
    __shared__ int s_list[LIST_CAP], s_first[LIST_CAP + 1], s_warp[NL_WARPS], s_pieces[NL_WARPS];
    __shared__ unsigned s_win[NL_WARPS][NL_WIN];
    __shared__ __align__(16) unsigned s_ring[NL_WARPS][NL_ATOMS][NL_RING + 4];
    rc_pdl_wait();
    rc_pdl_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int o0 = lane / 5 - 2, o1 = lane % 5 - 2;  // this lane's stencil row (lanes 25 .. 31: none)
    const float4 *__restrict__ X = cur ? a.x1 : a.x0;
    unsigned *win = s_win[warp];
    unsigned(*ring)[NL_RING + 4] = s_ring[warp];
    int next = blockIdx.x;  // this CTA's next piece
    for (int from = 0; from < n_cells; from += LIST_CAP) {
        const int n_go = compact_cells(s_list, s_warp, n_cells, from, [&](int c) {
            const bool go = a.built[c] != 0;
            if (go && blockIdx.x == 0) {
                a.need_rebuild[c] = 0;
                a.rebuilds[c]++;
            }
            return go;
        });
        if (n_go == 0) continue;
        // Pieces of consecutive atoms, cell after cell, dealt to the CTAs in turn:
        // up to NL_PIECE groups of atoms, fewer where that would leave CTAs without work
        int n_of[NL_CELLS], all = 0;
#pragma unroll
        for (int j = 0; j < NL_CELLS; j++) {
            const int k = NL_CELLS * threadIdx.x + j;
            n_of[j] = k < n_go ? a.cell_n[s_list[k]] : 0;
            all += n_of[j];
        }
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) all += __shfl_xor_sync(NL_FULL, all, d);
        if (lane == 0) s_warp[warp] = all;
        __syncthreads();
        all = 0;
        for (int w = 0; w < NL_WARPS; w++) all += s_warp[w];
        const int piece = NL_GROUP * min(NL_PIECE, max(1, all / (4 * NL_GROUP * (int)gridDim.x)));
        // A CTA walks a short list cell by cell (0.5 us sooner in steps where a few cells
        // rebuild); in a long one it looks up the cell of its next piece in the numbers of
        // pieces before every cell.  (Walked, 1024 cells of 256 atoms took 547 us, looked
        // up 394; 4096 of them 2155 / 1482; 512 of 2048 980 / 913.)
        const bool walk = n_go <= NL_WALK;
        if (!walk) {
            int before = 0;
#pragma unroll
            for (int j = 0; j < NL_CELLS; j++) before += (n_of[j] + piece - 1) / piece;
            const int own = before;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(NL_FULL, before, d);
                if (lane >= d) before += y;
            }
            if (lane == 31) s_pieces[warp] = before;
            before -= own;
            __syncthreads();
            for (int w = 0; w < warp; w++) before += s_pieces[w];
#pragma unroll
            for (int j = 0; j < NL_CELLS; j++) {
                s_first[NL_CELLS * threadIdx.x + j] = before;
                before += (n_of[j] + piece - 1) / piece;
            }
            if (threadIdx.x == NL_THREADS - 1) s_first[LIST_CAP] = before;  // all pieces
            __syncthreads();
        }
        for (int k = 0; walk ? k < n_go : next < s_first[LIST_CAP];) {
            if (!walk) {
                k = 0;
                for (int d = LIST_CAP / 2; d >= 1; d >>= 1)
                    if (s_first[k + d] <= next) k += d;
                next -= s_first[k];
            }
            const int c = s_list[k], n = a.cell_n[c], pieces = (n + piece - 1) / piece;
            if (next >= pieces) {
                next -= pieces;
                k++;
                continue;
            }
            const int off = a.cell_off[c], t0 = a.cell_tile0[c];
            const int nb0 = a.nbins[4 * c], nb1 = a.nbins[4 * c + 1], nb2 = a.nbins[4 * c + 2];
            const float *H = a.Hf + 8 * c;
            const float4 *tab = a.shift + (size_t)c * RC_SHIFT_W;
            const int *bs = a.bin_start + a.bin_off[c];
            // r_list, and 4e-6 of the box for what positions, bins and their edges may be
            // off: a few roundings (6e-8 each), both to lower and to higher bins
            const float reach = sqrtf(p.rlist2) + 4e-6f * (fabsf(H[0]) + fabsf(H[1]) + fabsf(H[2]) + fabsf(H[3]) +
                                                           fabsf(H[4]) + fabsf(H[5]));
            const float r0 = 1.0f / nb0, r1 = 1.0f / nb1, r2 = 1.0f / nb2;
            const float reach2 = reach * reach, to_bins = nb2 / H[5];
            // entry k of atom li of the cell lives at word 4 * ((t * max_nb/4 + k/4) * TILE + at) + k%4
            const auto out = [&](int li) {
                return reinterpret_cast<int4 *>(a.nbr) + (size_t)(t0 + li / RC_TILE) * (p.max_nb / 4) * RC_TILE + li % RC_TILE;
            };
            for (; next < pieces; next += gridDim.x)
            for (int i0 = next * piece + warp * NL_ATOMS; i0 < min(n, (next + 1) * piece); i0 += NL_GROUP) {
                const int g0 = off + i0;
                int px[NL_ATOMS], py[NL_ATOMS], cnt[NL_ATOMS];  // bond partners, entries found
                bool more = false;                              // an atom with a third bond
#pragma unroll
                for (int m = 0; m < NL_ATOMS; m++) {
                    cnt[m] = 0;
                    if (KG) {
                        const int4 pr = a.partner[off + min(i0 + m, n - 1)];
                        px[m] = pr.x < 0 ? -1 : off + pr.x;
                        py[m] = pr.y < 0 ? -1 : off + pr.y;
                        more = more || pr.z >= 0 || pr.w >= 0;
                    }
                }
                unsigned todo = (1u << min(NL_ATOMS, n - i0)) - 1u;
                while (todo) {  // the atoms of one bin row (the others of the four are put far away)
                    const int b01 = a.bin_of[g0 + __ffs(todo) - 1] >> 10;
                    int z_min = 1024, z_max = -1;
                    float x_lo = 3e38f, x_hi = -3e38f, y_lo = 3e38f, y_hi = -3e38f, z_lo = 3e38f, z_hi = -3e38f;
                    unsigned act = 0;
                    float3 xa[NL_ATOMS];
#pragma unroll
                    for (int m = 0; m < NL_ATOMS; m++) {
                        const int g = off + min(i0 + m, n - 1), bin = a.bin_of[g];
                        const float4 xi = X[g];
                        const bool on = (todo >> m & 1u) && bin >> 10 == b01;
                        xa[m] = on ? make_float3(xi.x, xi.y, xi.z) : make_float3(-1e18f, -1e18f, -1e18f);
                        if (on) {
                            act |= 1u << m;
                            z_min = min(z_min, bin & 1023);
                            z_max = max(z_max, bin & 1023);
                            x_lo = fminf(x_lo, xi.x);
                            x_hi = fmaxf(x_hi, xi.x);
                            y_lo = fminf(y_lo, xi.y);
                            y_hi = fmaxf(y_hi, xi.y);
                            z_lo = fminf(z_lo, xi.z);
                            z_hi = fmaxf(z_hi, xi.z);
                        }
                    }
                    todo &= ~act;
                    // ---- this lane's row ----
                    int start0 = 0, len0 = 0, start1 = 0, len1 = 0, start2 = 0, len2 = 0, s0 = 0, s1 = 0;
                    if (lane < 25) {
                        const int u0 = (b01 >> 10) + o0, u1 = (b01 & 1023) + o1;
                        // extent of the row's bins (all of z that can matter) along x and y
                        const float f0 = u0 * r0, f1 = u1 * r1, f2 = (z_min - 2) * r2, e2 = (z_max + 3) * r2;
                        const float e0 = f0 + r0, e1 = f1 + r1;
                        const float gx = gap(H[0] * f0 + fminf(H[1] * f1, H[1] * e1) + fminf(H[2] * f2, H[2] * e2) - x_hi,
                                             H[0] * e0 + fmaxf(H[1] * f1, H[1] * e1) + fmaxf(H[2] * f2, H[2] * e2) - x_lo);
                        const float gy = gap(H[3] * f1 + fminf(H[4] * f2, H[4] * e2) - y_hi,
                                             H[3] * e1 + fmaxf(H[4] * f2, H[4] * e2) - y_lo);
                        const float rem = reach2 - gx * gx - gy * gy;
                        if (rem >= 0.0f) {  // the stretch of z that is left within r_list
                            const float rz = sqrtf(rem);
                            const int lo = max(z_min - 2, (int)floorf((z_lo - rz) * to_bins)),
                                      hi = min(z_max + 2, (int)floorf((z_hi + rz) * to_bins));
                            s0 = u0 < 0 ? -1 : (u0 >= nb0 ? 1 : 0);
                            s1 = u1 < 0 ? -1 : (u1 >= nb1 ? 1 : 0);
                            const int *rb = bs + ((u0 - s0 * nb0) * nb1 + u1 - s1 * nb1) * nb2;
                            const int l0 = max(lo, 0), h0 = min(hi, nb2 - 1);
                            if (l0 <= h0) {
                                start0 = rb[l0];
                                len0 = rb[h0 + 1] - start0;
                            }
                            if (lo < 0) {
                                start1 = rb[nb2 + lo];
                                len1 = rb[nb2 + min(hi, -1) + 1] - start1;
                            }
                            if (hi >= nb2) {
                                start2 = rb[max(lo - nb2, 0)];
                                len2 = rb[hi - nb2 + 1] - start2;
                            }
                        }
                    }
                    // ---- places: central segments of all rows first, then each row's images ----
                    const bool central = (s0 | s1) == 0;
                    const int nc = central ? len0 : 0, ni = len0 - nc + len1 + len2;
                    int vc = nc, vi = ni;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const int yc = __shfl_up_sync(NL_FULL, vc, d), yi = __shfl_up_sync(NL_FULL, vi, d);
                        if (lane >= d) {
                            vc += yc;
                            vi += yi;
                        }
                    }
                    const int tc = __shfl_sync(NL_FULL, vc, 31), total = tc + __shfl_sync(NL_FULL, vi, 31);
                    const int at_i = tc + vi - ni;  // first place of this row's images
                    const int at0 = central ? vc - nc : at_i, at1 = central ? at_i : at_i + len0;
                    const unsigned w0 = (unsigned)(off + start0) | ((unsigned)rc_image_slot(s0, s1, 0) << RC_IDX_BITS);
                    const unsigned w1 = (unsigned)(off + start1) | ((unsigned)rc_image_slot(s0, s1, -1) << RC_IDX_BITS);
                    const unsigned w2 = (unsigned)(off + start2) | ((unsigned)rc_image_slot(s0, s1, 1) << RC_IDX_BITS);
                    for (int base = 0; base < total; base += NL_WIN) {
                        {
                            unsigned w = w0;
                            int at = at0 - base;
                            const int n01 = len0 + len1, n_all = n01 + len2;
                            for (int j = 0; j < n_all; j++) {
                                at = j == len0 ? at1 - base : at;
                                w = j == len0 ? w1 : w;
                                w = j == n01 ? w2 : w;  // follows the second segment
                                if ((unsigned)at < (unsigned)NL_WIN) win[at] = w;
                                w++;
                                at++;
                            }
                        }
                        __syncwarp();
                        const int end = min(total - base, NL_WIN);
                        // the last round's lanes without a candidate test a null entry
                        for (int b = end + lane; b < ((end + 31) & ~31); b += 32) win[b] = (unsigned)(off + i0) | RC_SLOT_NULL << RC_IDX_BITS;
                        __syncwarp();
                        // one candidate per lane against all atoms: straight-line code (a
                        // candidate that is not kept goes to the ring's spare word)
                        const auto batch = [&](int b, auto img, auto branched) {
                            const unsigned w = win[b + lane];
                            const int j = (int)(w & RC_IDX_MASK);
                            const float4 xj = X[j];
                            float4 sa, sb;
                            if (decltype(img)::value) {
                                const float4 *ts = tab + (w >> RC_IDX_BITS);
                                sa = __ldg(ts);
                                sb = __ldg(ts + RC_SLOTS);
                            }
                            bool keep[NL_ATOMS];
                            unsigned mask[NL_ATOMS];
                            int crossed = 0;
#pragma unroll
                            for (int m = 0; m < NL_ATOMS; m++) {
                                float3 d;
                                if (decltype(img)::value)
                                    d = rc_disp_pre(xj, sa, make_float4(xa[m].x - sb.x, xa[m].y - sb.y, xa[m].z - sb.z, sb.w));
                                else d = make_float3(xj.x - xa[m].x, xj.y - xa[m].y, xj.z - xa[m].z);
                                const float r2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
                                // the atom itself and its bond partners (any image) are left out
                                keep[m] = (r2 < p.rlist2) & (w != (unsigned)(g0 + m));
                                if (KG) keep[m] = keep[m] & (j != px[m]) & (j != py[m]);
                                if (decltype(branched)::value) {
                                    const int4 pr = a.partner[g0 + m];
                                    keep[m] = keep[m] && (pr.z < 0 || j != off + pr.z) && (pr.w < 0 || j != off + pr.w);
                                }
                                mask[m] = __ballot_sync(NL_FULL, keep[m]);
                            }
#pragma unroll
                            for (int m = 0; m < NL_ATOMS; m++) {
                                const int at = (cnt[m] + __popc(mask[m] & lt)) & 63;
                                ring[m][keep[m] ? at : NL_RING] = w;
                                const int now = cnt[m] + __popc(mask[m]);
                                crossed |= cnt[m] ^ now;
                                cnt[m] = now;
                            }
                            if (crossed & ~31) {  // 32 more entries of a list complete (beyond the capacity: dropped)
                                __syncwarp();
#pragma unroll
                                for (int m = 0; m < NL_ATOMS; m++)
                                {
                                    const int before = (cnt[m] - __popc(mask[m])) >> 5, e = 8 * before + lane;
                                    if (cnt[m] >> 5 != before && lane < 8 && 4 * e < p.max_nb)
                                        out(i0 + m)[(size_t)e * RC_TILE] = reinterpret_cast<const int4 *>(ring[m])[e & 15];
                                }
                                __syncwarp();
                            }
                        };
                        int b = 0;
                        if (KG && more) {
                            for (; b < end; b += 32) batch(b, std::true_type{}, std::true_type{});
                        } else {
                            for (; b < end && base + b + 32 <= tc; b += 32) batch(b, std::false_type{}, std::false_type{});
                            for (; b < end; b += 32) batch(b, std::true_type{}, std::false_type{});
                        }
                        __syncwarp();
                    }
                }
                // what is left of each list, with null entries up to a whole group
                const int m = lane >> 3, sub = lane & 7;
                static_assert(NL_ATOMS * 8 == 32, "eight lanes per atom");
                int left = cnt[0];
#pragma unroll
                for (int k2 = 1; k2 < NL_ATOMS; k2++) left = m == k2 ? cnt[k2] : left;
                const int li = i0 + m;
                if (li < n && sub < (-left & 3)) ring[m][(left + sub) & 63] = (unsigned)(off + li) | (RC_SLOT_NULL << RC_IDX_BITS);
                __syncwarp();
                const int e = 8 * (left >> 5) + sub;
                if (li < n) {
                    if (4 * e < min(left, p.max_nb)) out(li)[(size_t)e * RC_TILE] = reinterpret_cast<const int4 *>(ring[m])[e & 15];
                    if (sub == 0) {
                        if (left > p.max_nb) rc_set_status(a.status, c, RC_EOVERFLOW);
                        a.nnb[off + li] = min(left, p.max_nb);
                    }
                }
                __syncwarp();
            }
            next += walk ? -pieces : s_first[k];
            k++;
        }
        if (!walk) next -= s_first[LIST_CAP];
        __syncthreads();
    }
}

}  // namespace

void rc_launch_sort(const KParams &p, const KArrays &a, int cur, int n_cells, cudaStream_t s) {
    // as many clusters as two CTAs per SM allow, at most one per cell
    const int n_cl = min(n_cells, max(1, 2 * p.n_sm / SORT_CL));
    const bool many = n_cells > n_cl && p.max_cell <= SORT_CL * SORT_THREADS;
    rc_launch_pdl(many ? k_sort<true> : k_sort<false>, n_cl * SORT_CL, SORT_THREADS, 0, s, SORT_CL, p, a, cur, n_cells);
}

void rc_launch_nlist(const KParams &p, const KArrays &a, int cur, int n_cells, cudaStream_t s) {
    // NL_CTAS CTAs per SM, at most one per NL_GROUP atoms of the batch
    const int ctas = min(NL_CTAS * p.n_sm, p.n_tiles * (RC_TILE / NL_GROUP));
    rc_launch_pdl(p.pot == RC_POT_KG ? k_nlist<true> : k_nlist<false>, ctas, NL_THREADS, 0, s, 1, p, a, cur, n_cells);
}
