// Tiled single-pass kernel family: the whole time step (moments, pseudopotential,
// 25-point forces of Eq. (FFF), shifted BGK collision of Eq. (be), streaming)
// in one pass over the populations.
//
// Work item = one column strip of TX sites x one segment of TY rows of one cell.
// A CTA has TX column threads (one species and two adjacent columns each: lanes
// 0-15 of a warp species A, 16-31 species B of the same 32 columns) and one
// service warp (TMA issue, halo columns of psi/rho, row sums of sampled steps).
// It walks its segment row by row:
//   * TMA (cp.async.bulk.tensor, 4-D map [cell][q][y][x]) brings whole rows of all
//     18 populations into a ring of D shared-memory slots, several rows ahead,
//     each slot completing on its own mbarrier; a row is TX main columns plus
//     16-byte halo boxes on both sides (periodic wrap in x by coordinates);
//   * when row y+2 lands, its rho_s and psi_s (for the TX columns and 2 halo
//     columns per side) go into a 6-row ring, so rows y-2..y+2 of psi/rho are
//     on chip when row y is collided: the 25-point stencil reads shared memory;
//   * row y is collided from its populations still in the slot ring and pushed
//     to the other ping-pong buffer with plain coalesced stores (x-shifted by
//     -1/0/+1 element), bounce-back rows handled in place; with FP16 storage the
//     stores round to nearest or stochastically (Store<T>, Dither).
// HBM traffic per site update is one read and one write of the 18 populations;
// halo rows/columns are re-read by neighbouring work items (mostly from L2).
// The grid is persistent (CTAs loop over work items).  Every mbarrier wait is
// bounded: on timeout the CTA records ERR_TIMEOUT, drains its copies in flight
// (also bounded) and leaves.
#pragma once

#include <limits>
#include <type_traits>

#include "lb_internal.h"
#include "lb_pair.cuh"
#include "lbhb.h"
#include "tma.cuh"

namespace lbhb {

constexpr int RING = 6;  // psi/rho rows on chip: 5 read by a collision + 1 being written

__host__ __device__ constexpr int al128(int b) { return (b + 127) / 128 * 128; }

// Row-slot ring depth: about three rows in flight beyond the three in use.
// FP64 rows are consumed at the FP64 pipe's pace (a seventh of the FP32 rate),
// so one row in flight covers the memory latency, and the smaller ring lets two
// CTAs share an SM.
__host__ __device__ constexpr int ring_depth(int tx, int elem)
{
    return elem == 8 ? 4 : (6 * al128(18 * tx * elem) + 12 * al128(18 * (16 / elem) * elem) <= 96 * 1024) ? 6 : 5;
}
// Words between the species-A and species-B psi/rho rings, chosen so that a
// half-warp reading A and the other half reading B hit disjoint banks.
__host__ __device__ constexpr int ring_species_stride(int tx)
{
    return RING * (tx + 4) + ((16 - (RING * (tx + 4)) % 32) + 32) % 32;
}

// Threads per CTA: a thread per (species, column pair), TX threads, plus one
// service warp that issues the TMA copies and computes the four halo columns
// of psi/rho, so the column warps all do the same work between two barriers.
__host__ __device__ constexpr int tiled_threads(int tx) { return tx + 32; }

// Dynamic shared memory of a CTA: row slots, psi/rho rings, mbarriers, and two
// rows of per-site profile values (sampled steps).
__host__ __device__ constexpr int tiled_smem_bytes(int tx, int elem)
{
    return ring_depth(tx, elem) * (al128(18 * tx * elem) + 2 * al128(18 * (16 / elem) * elem)) +
           4 * ring_species_stride(tx) * (elem == 8 ? 8 : 4) + ring_depth(tx, elem) * 8 + 2 * tx * (elem == 8 ? 8 : 4);
}
// CTAs of a plain step per SM that shared memory admits (228 KB per SM, 1 KB of
// it reserved per CTA), at most 4: the register budget the compiler is held to,
// so that registers do not admit fewer.  Sampled steps (a tenth of the launches,
// with more live values) are held to at most 3.
__host__ __device__ constexpr int tiled_min_ctas(int tx, int elem)
{
    return 233472 / (tiled_smem_bytes(tx, elem) + 1024) < 1   ? 1
         : 233472 / (tiled_smem_bytes(tx, elem) + 1024) > 4 ? 4
                                                             : 233472 / (tiled_smem_bytes(tx, elem) + 1024);
}

// Service warp, sampled steps: the sums of u_x over each 32-column group of one
// row of a strip (ub: TX values), one FP64 partial per group as the column warps
// would have written it.  Lane l takes NW = TX/32 consecutive columns of group
// l / (32/NW), then a segmented warp sum; FP32 values are carried as an
// unevaluated (hi, lo) pair (error-free two-sum), ~2^-48 relative.  Not inlined,
// so its registers do not add to the column warps' in the hot loop.
template <class C, int TX>
__device__ __noinline__ void profile_row_sums(const C* ub, int lane, double* __restrict__ prof_part, int cell,
                                              int nx, int nrows, int x0, int row)
{
    constexpr int NW = TX / 32, SEG = 32 / NW;
    const int grp = lane / SEG, t = lane % SEG;
    const double part = group_sum<NW>(lane, [&](int q) { return ub[grp * 32 + t * NW + q]; });
    const int nbx = (nx + 31) / 32;  // 32-column groups of the lattice; a narrow last strip has fewer
    if (t == 0 && (x0 >> 5) + grp < nbx) prof_part[((long long)cell * nbx + (x0 >> 5) + grp) * nrows + row] = part;
}

// Kernel families (FAM):
//   FAM_FULL  every strip is TX columns wide (nx a multiple of TX) and every cell
//             has one relaxation time (BGK);
//   FAM_FULL_BIG  the same, for lattices far larger than the L2 (full_big): ring rows
//             are computed per row instead of kept, stores without the streaming hint,
//             1/rho and psi/rho by the fast division;
//   FAM_GEN   the last strip may be narrower (its extra columns masked) and the
//             species may relax with times of their own (BGK);
//   FAM_MRT   as FAM_GEN, with the multiple-relaxation-time collision;
//   FAM_ANY, FAM_ANY_MRT  as these for any width, odd ones too, in FP32 storage.  The
//             halo columns of such a row have no aligned place for a TMA box: the
//             service warp copies them word by word (cp.async, on the row's mbarrier),
//             and the last pair of an odd width updates its first site only.  1021 x 509
//             FP32 18.8 us per step where the generic pair takes 39.5 (its two
//             passes move 232 bytes per site and its loads wait one by one).
constexpr int FAM_FULL = 0, FAM_FULL_BIG = 1, FAM_GEN = 2, FAM_MRT = 3, FAM_ANY = 4, FAM_ANY_MRT = 5, N_FAM = 6;
template <class T, int TX, bool SAMPLE, int FAM>
__global__ void __launch_bounds__(tiled_threads(TX),
                                  SAMPLE ? (tiled_min_ctas(TX, (int)sizeof(T)) < 3 ? tiled_min_ctas(TX, (int)sizeof(T)) : 3)
                                         : tiled_min_ctas(TX, (int)sizeof(T)))
    tiled_step_kernel(const __grid_constant__ CUtensorMap tm_main,
                                                            const __grid_constant__ CUtensorMap tm_halo,
                                                            const T* __restrict__ fin, T* __restrict__ fout, Geom g,
                                                            int bc, RowMap rm,
                                                            int ty,
                                                            int n_strips, int n_seg,
                                                            const CellDev* __restrict__ cells,
                                                            double* __restrict__ prof_part,
                                                            double* __restrict__ wall_part,
                                                            unsigned* __restrict__ err, uint32_t skip_row_arg)
{
    using C = typename Store<T>::C;
    using V = P2<C>;  // a lane pair: one species at the thread's two sites
    constexpr bool FULL = FAM == FAM_FULL || FAM == FAM_FULL_BIG, MRT = FAM == FAM_MRT || FAM == FAM_ANY_MRT, ANY = FAM >= FAM_ANY;
    // Ring rows kept in registers and streaming stores of the whole pairs: FP32, 8 x
    // 1024^2 MRT 216.4 -> 209.6 us, 48 x 64^2 10.5 -> 10.3, 1021 x 509 18.4 -> 18.0;
    // FP16, at its register limit, loses 1.5 %, and so does the memory-bound FAM_FULL_BIG
    constexpr bool KEEP = std::is_same<T, float>::value && FAM != FAM_FULL_BIG;
    constexpr bool DIV = FAM == FAM_FULL_BIG;  // rho_rcp, psi_over_rho
    // stored populations are scale * g (scale 1 except for the dithered FP16 storage)
    constexpr C scale = C(Store<T>::scale), inv_scale = C(1) / scale;
    constexpr int E = (int)sizeof(T);
    constexpr int H = 16 / E;            // halo columns per side brought by TMA
    constexpr int W = TX + 4;            // ring row: columns -2 .. TX+1
    constexpr int D = ring_depth(TX, E);
    constexpr int SS = ring_species_stride(TX);
    constexpr int MAIN_AL = al128(18 * TX * E);
    constexpr int HALO_AL = al128(18 * H * E);
    constexpr int SLOT = MAIN_AL + 2 * HALO_AL;
    constexpr uint32_t TX_BYTES = 18 * TX * E + (ANY ? 0 : 2 * 18 * H * E);
    static_assert(!ANY || std::is_same<T, float>::value, "a halo column of the any-width form is one 4-byte word");

    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* fring = smem;
    // rings [RING][W], SS apart: psi of A, rho of B, psi of B, rho of A, so that a
    // lane's psi and its partner's rho lie at one distance from each other
    unsigned char* const rings = smem + D * SLOT;
    uint64_t* bars = reinterpret_cast<uint64_t*>(rings + 4 * SS * (int)sizeof(C));
    // sampled steps: u_x of each site of the last two rows, summed by the service warp
    C* ubuf = reinterpret_cast<C*>(bars + D);

    constexpr int NW = TX / 32;               // column warps (32 columns x 2 species each)
    const int t = threadIdx.x;
    const int lane = t & 31, warp = t >> 5;
    const bool svc = warp == NW;              // the service warp
    const bool producer = svc && lane == 0;   // issues the TMA copies
    const bool issuer = ANY ? svc : producer;  // keeps the issue cursor
    // column warps: lanes 0-15 species A, 16-31 species B, columns c0 and c0+1;
    // service warp: lanes 0-3 species A, 4-7 species B of the halo columns
    const int sp = svc ? (lane >> 2) & 1 : lane >> 4;
    const int c0 = svc ? 0 : warp * 32 + 2 * (lane & 15);
    // a pipeline that timed out in an earlier launch of the same batch does not
    // run again (each later launch would otherwise wait out its own bound); the
    // decision is taken once per CTA, at the barrier that publishes the mbarriers
    bool stale = false;
    if (t == 0) {
        stale = (*reinterpret_cast<volatile unsigned*>(err) & ERR_TIMEOUT) != 0u;
        for (int d = 0; d < D; ++d) mbar_init(&bars[d], ANY ? 33 : 1);
        fence_mbar_init();
        prefetch_tensormap(&tm_main);
        prefetch_tensormap(&tm_halo);
    }
    if (__syncthreads_or(stale)) return;

    // failure-injection hook (tests only): CTA 0 leaves the copy of its row
    // skip_row_arg unissued, so the waits for it run out; ~0u: none
    const uint32_t skip_row = blockIdx.x == 0 ? skip_row_arg : ~0u;
    const long long per_cell = (long long)n_strips * n_seg;
    const long long items = per_cell * g.n_cells;
    uint32_t nrow = 0;  // global index of row 0 of the current item (rows consumed before it)
    bool aborted = false;
    bool bad = false;  // watchdog: a non-finite or non-positive density seen in this item

    // Issue cursor (producer): the next row to load may belong to a later item
    // of this CTA, so the row pipeline does not drain between items.  Global
    // row n always lives in slot n % D with mbarrier phase (n / D) & 1.  The
    // geometry of the item being issued is cached (one division per item).
    long long iw = blockIdx.x;
    int ik = 0, icell = 0, ix0 = 0, iy0 = 0, iR = 0, ixl = 0, ixr = 0;
    int ihc = 0;  // ANY: this lane's halo column (lane & 3: columns -2, -1, TX, TX + 1 of the strip, periodic)
    uint32_t n_issued = 0;
    auto halo_column = [&](int x0) {
        const int h = lane & 3, x = h < 2 ? x0 - 2 + h : min(x0 + TX, g.nx) + h - 2;
        return x < 0 ? x + g.nx : x >= g.nx ? x - g.nx : x;
    };
    auto load_item = [&]() {
        if (iw >= items) return;
        icell = (int)(iw / per_cell);
        const int irem = (int)(iw - (long long)icell * per_cell);
        const int iseg = irem / n_strips;
        ix0 = (irem - iseg * n_strips) * TX;
        iy0 = rm.ylo + iseg * ty;
        iR = min(ty, rm.ylo + rm.nown - iy0) + 4;
        ixl = ix0 >= H ? ix0 - H : g.nx - H;
        ixr = ix0 + TX < g.nx ? ix0 + TX : 0;
        if constexpr (ANY) ihc = halo_column(ix0);
    };
    if (issuer) load_item();
    auto issue_upto = [&](uint32_t limit) {
        while (n_issued < limit && iw < items) {
            const int slot = (int)(n_issued % D);
            unsigned char* dst = fring + slot * SLOT;
            const int yp = stencil_load_row(iy0 - 2 + ik, g.ny, rm, bc);
            if (n_issued != skip_row) {
                if (producer) {
                    mbar_arrive_expect_tx(&bars[slot], TX_BYTES);
                    tma_load_4d(dst, &tm_main, ix0, yp, 0, icell, &bars[slot]);
                }
                if constexpr (ANY) {
                    // word (population q, halo column h) at 4 q + h, h = lane & 3
                    const T* const row = fin + (long long)icell * g.cellstride + (long long)yp * g.pitch + ihc;
                    for (int e = lane; e < 72; e += 32)
                        cp_async4(dst + MAIN_AL + 4 * e, row + (long long)(e >> 2) * g.plane);
                    cp_async_arrive(&bars[slot]);
                } else {
                    tma_load_4d(dst + MAIN_AL, &tm_halo, ixl, yp, 0, icell, &bars[slot]);
                    tma_load_4d(dst + MAIN_AL + HALO_AL, &tm_halo, ixr, yp, 0, icell, &bars[slot]);
                }
            }
            ++n_issued;
            if (++ik == iR) {
                ik = 0;
                iw += gridDim.x;
                load_item();
            }
        }
    };

    for (long long w = blockIdx.x; w < items && !aborted; w += gridDim.x) {
        const int cell = (int)(w / per_cell);
        const int rem = (int)(w % per_cell);
        const int seg = rem / n_strips, strip = rem % n_strips;
        const int x0 = strip * TX, y0 = rm.ylo + seg * ty;  // buffer row of the item's first row
        const int rows = min(ty, rm.ylo + rm.nown - y0);
        const int R = rows + 4;  // logical rows y0-2 .. y0+rows+1
        // per-cell parameters as scalars (no runtime-indexed arrays: they would
        // live in local memory)
        const ParamSet<C>& pg = params<C>(cells[cell]);
        ParamSet<C> p;
        p.rho0 = pg.rho0;
        p.inv_rho0 = pg.inv_rho0;
        p.u_wall = pg.u_wall;
        p.f0 = pg.f0;
        p.two_over_ny = pg.two_over_ny;
        // this lane's species relaxes with tau_s; mix weighs the partner species'
        // moments in the common velocity (1, and one_time, for one relaxation time)
        const C tau_s = FULL || !sp ? pg.tau : pg.tau_b, omega_s = FULL || !sp ? pg.omega : pg.omega_b;
        const C mix = FULL ? C(1) : (sp ? pg.mix[1] : pg.mix[0]);
        const bool one_time = FULL || pg.mix[0] == C(1);
        // tau = 1 for both species: f* = f^eq.  Uniform over the item, so both
        // half-warps take the same path (a cell with tau_A = 1 != tau_B runs the
        // general update in both)
        const bool unit_omega = FULL ? pg.omega == C(1) : (pg.omega == C(1) && pg.omega_b == C(1));
        // multiple-relaxation-time coefficients of this lane's species (mrt_delta)
        V mh[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) mh[q] = V(MRT ? (sp ? pg.mrt_h[1][q] : pg.mrt_h[0][q]) : C(0));
        // the same values as lane pairs
        const Couplings<V> cp(pg, sp);
        const V tau2 = V(tau_s), ntau2 = V(-tau_s), omega2 = V(omega_s), mix2 = V(mix);
        const V rho0_2 = V(p.rho0), inv_rho0_2 = V(p.inv_rho0);
        const C rho_bar = sp ? pg.rho_bar[1] : pg.rho_bar[0];
        const V rho_bar2 = V(rho_bar);
        // columns of this strip inside the lattice (the last strip of a width that
        // is not a multiple of TX is narrower; the TMA box reads zeros beyond it)
        const int wv = FULL ? TX : min(TX, g.nx - x0);
        const bool act = FULL || c0 < wv;                 // the pair's first column
        const bool act_b = FULL || c0 + (ANY ? 1 : 0) < wv;  // its second (the same unless the width is odd)
        // destination columns of the two sites x, x+1 shifted by -1/0/+1 (periodic)
        const int x = x0 + c0;
        const int col_m = x == 0 ? g.nx - 1 : x - 1, col_p2 = x + 2 == g.nx ? 0 : x + 2;
        const int col_p1 = ANY && x + 1 == g.nx ? 0 : x + 1;
        T* const dst_s = fout + (long long)cell * g.cellstride + (long long)sp * 9 * g.plane;
        T* const dst_x = dst_s + x;  // column x, plane 0 of the species, row 0
        // warps holding column 0 or column nx - 1 wrap their x-shifted stores
        // periodically; the others store each direction's two sites at fixed
        // offsets from one address
        const bool xedge = (x0 == 0 && warp == 0) || (x0 + 32 * warp + 32 >= g.nx);

        // rings of the previous item are no longer read; the watchdog flags of its
        // rows are reported
        if (__syncthreads_or(bad) && t == 0) atomicOr(err, ERR_NONFINITE);
        bad = false;

        if (issuer) issue_upto(nrow + D);  // rows of earlier items are all done
        // Byte offsets of this thread, advanced by one row per iteration instead of
        // computed from row numbers: its place in a ring row (two columns left of the
        // lane's first; the service warp: of its halo column) and in a row slot
        constexpr int RW = W * (int)sizeof(C);                           // a ring row
        constexpr int PARTNER = SS * (int)sizeof(C);                     // from psi to the partner's rho
        const int own = (sp ? -SS : 3 * SS) * (int)sizeof(C);            // from psi to the lane's own rho
        const int hpos = (lane & 3) < 2 ? lane & 3 : wv + (lane & 3);    // service warp
        const int ring0 = (sp * 2 * SS + (svc ? hpos - 2 : c0)) * (int)sizeof(C), ring_end = ring0 + RING * RW;
        const int slot0 = svc ? 0 : (sp * 9 * TX + c0) * E;
        // rho_s, psi_s of the row in the slot at `slot` into the ring row at `ring` (own
        // species, own two columns; the service warp takes the halo columns)
        auto psi_stage = [&](int slot, int ring) {
            C* const to = reinterpret_cast<C*>(rings + ring) + 2;
            C* const to_rho = reinterpret_cast<C*>(rings + ring + own) + 2;
            if (!svc) {
                if (!act) return;  // its ring positions belong to the halo or to nobody
                const T* src = reinterpret_cast<const T*>(fring + slot);
                V r = Pair<T>::ld(src);
#pragma unroll
                for (int i = 1; i < 9; ++i) r = r + Pair<T>::ld(src + i * TX);
                if constexpr (Store<T>::shifted) {  // sum of the shifts w_i rho_bar is rho_bar
                    if constexpr (Store<T>::scale != 1)
                        r = vfma(r, V(inv_scale), rho_bar2);
                    else
                        r = r + rho_bar2;
                }
                const V ps = lane_psi(r, rho0_2, inv_rho0_2);
                if (ANY && !act_b) {  // the next position is a halo column
                    *to = ps.a();
                    *to_rho = r.a();
                } else {
                    Pair<C>::st(to, ps);
                    Pair<C>::st(to_rho, r);
                }
            } else if (lane < 8) {
                // halo column h: 0,1 -> columns -2,-1 (left box); 2,3 -> TX, TX+1 (right box)
                const int h = lane & 3;
                const unsigned char* const base = fring + slot;
                const T* src = reinterpret_cast<const T*>(base + (h < 2 ? MAIN_AL : MAIN_AL + HALO_AL)) + sp * 9 * H +
                               (h < 2 ? H - 2 + h : h - 2);
                C acc = C(0);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    if constexpr (ANY)
                        acc += to_c(reinterpret_cast<const T*>(base + MAIN_AL)[(sp * 9 + i) * 4 + h]);
                    else
                        acc += to_c(src[i * H]);
                }
                if (Store<T>::shifted) acc = acc * inv_scale + rho_bar;
                *to = psi_of(acc, p.rho0, p.inv_rho0);
                *to_rho = acc;
            }
        };

        bool ok = true;
        // slot, and the phase of its barrier, of the row that is staged next (global row nrow + k)
        int sb = (int)(nrow % (uint32_t)D);
        uint32_t ph = (nrow / (uint32_t)D) & 1u;
        auto next_slot = [&]() {
            if (++sb == D) {
                sb = 0;
                ph ^= 1u;
            }
        };
        // Ring rows of logical rows j .. j + 4, read by the collision of row j + 2: all
        // five kept and rotated where registers are free (KEEP), else four of them from the first
        int rr[5] = {ring0, ring0 + RW, ring0 + 2 * RW, ring0 + 3 * RW, ring0 + 4 * RW};
        for (int k = 0; k < 4; ++k) {
            ok = mbar_wait_bounded(&bars[sb], ph) && ok;
            psi_stage(slot0 + sb * SLOT, ring0 + k * RW);
            next_slot();
        }
        if constexpr (D < 5) {
            // a four-slot ring holds rows 0..3 only: rows 4 and 5 go into the slots of
            // rows 0 and 1 once every thread has staged those (the loop below waits
            // for row j + 4 before its own barrier)
            __syncthreads();
            if (issuer) issue_upto(nrow + 2u + (uint32_t)D);
        }
        for (int j = 0; j < rows; ++j) {
            int ring_row[5];
#pragma unroll
            for (int d = 0; d < 5; ++d)
                ring_row[d] = KEEP ? rr[d] : rr[0] + d * RW >= ring_end ? rr[0] + (d - RING) * RW : rr[0] + d * RW;
            const int s2 = slot0 + (sb >= 2 ? sb - 2 : sb + D - 2) * SLOT;  // slot of row j + 2
            ok = mbar_wait_bounded(&bars[sb], ph) && ok;
            psi_stage(slot0 + sb * SLOT, ring_row[4]);
            next_slot();
#pragma unroll
            for (int d = 0; d < 4; ++d) rr[d] = ring_row[d + 1];
            rr[4] = ring_row[4] + RW == ring_end ? ring0 : ring_row[4] + RW;
            // barrier: psi/rho of row j+4 visible, collision of row j+1 finished
            // everywhere; it also tells every thread whether any wait ran out
            if (__syncthreads_or(ok ? 0 : 1)) {
                aborted = true;
                break;
            }
            // rows 0 .. j+1 of this item are done with their slots
            if (issuer) issue_upto(nrow + (uint32_t)(j + 2 + D));
            if (svc) {
                if (SAMPLE && j > 0)  // its row finished before this barrier
                    profile_row_sums<C, TX>(ubuf + ((j - 1) & 1) * TX, lane, prof_part, cell, g.nx, rm.nown, x0,
                                            y0 + j - 1 - rm.ylo);
                continue;
            }
            // ---- collide logical row k = j + 2 (lattice row y), sites x and x+1
            const int y = y0 + j, gy = y - rm.ylo + rm.y0g;  // buffer row, row of the global cell
            const T* fm = reinterpret_cast<const T*>(fring + s2);
            // populations as stored: f for FP32/FP64, the shifted g for FP16; a
            // lane pair per direction (sites x, x+1)
            V f[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = Pair<T>::ld(fm + i * TX);
            // psi window rows k-2..k+2 and rho_s' window rows k-1..k+1, columns
            // c0-2..c0+3 as three pairs; window column 2 + o is site o
            V v[5][3], e[3][3];
#pragma unroll
            for (int d = 0; d < 5; ++d) {
                const C* const ps = reinterpret_cast<const C*>(rings + ring_row[d]);
#pragma unroll
                for (int m = 0; m < 3; ++m) v[d][m] = Pair<C>::ld(ps + 2 * m);
                if (d == 0 || d == 4) continue;
#pragma unroll
                for (int m = 0; m < 3; ++m) e[d - 1][m] = Pair<C>::ld(ps + PARTNER / (int)sizeof(C) + 2 * m);
            }
            const V rho_s = Pair<C>::ld(reinterpret_cast<const C*>(rings + ring_row[2] + own) + 2);
            const V rho_p = e[1][1];  // the partner species' densities at the same two sites
            // pair differences d_q = psi(r + c_q) - psi(r - c_q) of both sites
            V dps[12], dro[4];
            window_diffs(v, e, dps, dro);
            const Pull<V> pu = cp.pull(dps, dro);
            const V jx_s = mom_x<V>(f), jy_s = mom_y<V>(f);
            const V jx_p(__shfl_xor_sync(0xffffffffu, jx_s.a(), 16), __shfl_xor_sync(0xffffffffu, jx_s.b(), 16));
            const V jy_p(__shfl_xor_sync(0xffffffffu, jy_s.a(), 16), __shfl_xor_sync(0xffffffffu, jy_s.b(), 16));
            // common velocity: (j_own + mix j_partner) / (rho_own + mix rho_partner)
            V jwx, jwy, rho_w;
            if constexpr (FULL) {  // one relaxation time: the barycentric velocity
                jwx = jx_s + jx_p;
                jwy = jy_s + jy_p;
                rho_w = rho_s + rho_p;
            } else {
                jwx = vfma(mix2, jx_p, jx_s);
                jwy = vfma(mix2, jy_p, jy_s);
                rho_w = vfma(mix2, rho_p, rho_s);
            }
            if constexpr (Store<T>::scale != 1) {
                jwx = jwx * V(inv_scale);
                jwy = jwy * V(inv_scale);
            }
            const V inv_rho = rho_rcp<DIV>(rho_w);
            const V ux = jwx * inv_rho, uy = jwy * inv_rho;
            const C fx_body = body_force_x<C>(p, gy);
            const bool body_raw = !one_time && !is_zero(fx_body);  // the force needs the raw 1/rho
            const V rho_t = FULL ? rho_w : rho_s + rho_p;        // total density of each site
            V ax = V(fx_body) * inv_rho;
            if (body_raw) ax = V(fx_body) * lane_rcp(rho_t);
            // watchdog: a non-finite or non-positive total density anywhere in the
            // item is reported through the error word when the item ends
            if (act) bad |= !(density_ok(rho_t.a()) && (density_ok(rho_t.b()) || (ANY && !act_b)));
            V fs[9], Fx;
            if constexpr (MRT && Store<T>::shifted) {
                collide_species_shifted<V, false, true>(f, rho_s, rho_bar2, v[2][1], ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx, V(scale), mh);
            } else if constexpr (MRT) {
                collide_species<V, false, true>(f, rho_s, v[2][1], ux, uy, ax, pu, tau2, ntau2, omega2,
                                                fs, &Fx, mh);
            } else if constexpr (Store<T>::shifted) {
                if (unit_omega)
                    collide_species_shifted<V, true>(f, rho_s, rho_bar2, v[2][1], ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx, V(scale));
                else
                    collide_species_shifted<V, false>(f, rho_s, rho_bar2, v[2][1], ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx, V(scale));
            } else {
                if (unit_omega)
                    collide_species<V, true, false, DIV>(f, rho_s, v[2][1], ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx);
                else
                    collide_species<V, false, false, DIV>(f, rho_s, v[2][1], ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx);
            }

            // stochastic rounding: one stream per thread and row, seeded from the
            // sites and their densities
            Dither dz;
            if constexpr (Store<T>::dithered)
                dz.seed(((uint32_t)cell * 0x9E3779B1u) ^ ((uint32_t)gy << 15) ^ ((uint32_t)x << 1) ^ (uint32_t)sp,
                        __float_as_uint(rho_s.a()) ^ (__float_as_uint(rho_s.b()) * 0x85EBCA6Bu));
            // push streaming; rows next to a Couette wall bounce back in place
            const bool wall_lo = bc == 1 && gy == 0, wall_hi = bc == 1 && gy == rm.nyg - 1;
            const int pl = (int)g.plane;  // < 2^31 / 18, checked on the host
            // destination rows y-1, y, y+1: periodic in a whole cell; a slab streams
            // into its ghost rows (the populations that leave it)
            const int row3[3] = {(!rm.slab && y == 0 ? g.ny - 1 : y - 1) * g.pitch, y * g.pitch,
                                 (!rm.slab && y == g.ny - 1 ? 0 : y + 1) * g.pitch};
            const int colA[3] = {col_m, x, col_p1};  // site x,   shifts -1, 0, +1
            const int colB[3] = {x, x + 1, col_p2};  // site x+1, shifts -1, 0, +1
            C dpx_site = C(0);
            if (act) {  // columns beyond the lattice store nothing
                if (!(wall_lo || wall_hi) && !xedge) {
                    // interior row (uniform over the CTA), away from the x edge (uniform
                    // over the warp): one address per direction, no wall tests
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const int cy = q_cy(i), cx = q_cx(i);
                        T* const q = dst_x + (i * pl + row3[cy + 1]);
                        if (cx == 0) {
                            if constexpr (KEEP)  // whole sectors: first out of the L2
                                __stcs(reinterpret_cast<float2*>(q), make_float2(fs[i].a(), fs[i].b()));
                            else
                                st_pair<T, C>(q, fs[i].a(), fs[i].b(), dz);
                        } else {
                            st_one<T, C>(q + cx, fs[i].a(), dz);
                            st_one<T, C>(q + cx + 1, fs[i].b(), dz);
                        }
                    }
                } else if (!(wall_lo || wall_hi)) {
                    // interior row on a warp at the x edge: periodic columns
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const int cy = q_cy(i), cx = q_cx(i);
                        if (cx == 0 && (!ANY || act_b)) {
                            st_pair<T, C>(dst_s + i * pl + row3[cy + 1] + x, fs[i].a(), fs[i].b(), dz);
                        } else {
                            st_one<T, C>(dst_s + i * pl + row3[cy + 1] + colA[cx + 1], fs[i].a(), dz);
                            if (!ANY || act_b)
                                st_one<T, C>(dst_s + i * pl + row3[cy + 1] + colB[cx + 1], fs[i].b(), dz);
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const int cy = q_cy(i), cx = q_cx(i);
                        const bool into_wall = (cy < 0 && wall_lo) || (cy > 0 && wall_hi);
                        if (into_wall) {
                            C dpa, dpb;
                            const C uw = cy < 0 ? -p.u_wall : p.u_wall;
                            // bounce in the f representation (for shifted storage the shift
                            // is put back first; opposite directions carry equal weights,
                            // so the same shift is removed again)
                            const C sh = Store<T>::shifted ? C(q_w(i)) * rho_bar : C(0);
                            const C ba = bounce<C>(i, fs[i].a() * inv_scale + sh, rho_s.a(), uw, &dpa);
                            const C bb = bounce<C>(i, fs[i].b() * inv_scale + sh, rho_s.b(), uw, &dpb);
                            if (!ANY || act_b) {
                                st_pair<T, C>(dst_s + q_opp(i) * pl + row3[1] + x, (ba - sh) * scale, (bb - sh) * scale,
                                              dz);
                                dpx_site += dpa + dpb;
                            } else {
                                st_one<T, C>(dst_s + q_opp(i) * pl + row3[1] + x, (ba - sh) * scale, dz);
                                dpx_site += dpa;
                            }
                        } else if (cx == 0 && (!ANY || act_b)) {
                            st_pair<T, C>(dst_s + i * pl + row3[cy + 1] + x, fs[i].a(), fs[i].b(), dz);
                        } else {
                            st_one<T, C>(dst_s + i * pl + row3[cy + 1] + colA[cx + 1], fs[i].a(), dz);
                            if (!ANY || act_b)
                                st_one<T, C>(dst_s + i * pl + row3[cy + 1] + colB[cx + 1], fs[i].b(), dz);
                        }
                    }
                }
            }
            if (SAMPLE) {
                // force-corrected velocity (j + F/2)/rho of the observables, from the
                // raw barycentric momentum and density
                V jxo = jwx, inv_r = inv_rho;
                if (!one_time) {
                    jxo = jx_s + jx_p;
                    if constexpr (Store<T>::scale != 1) jxo = jxo * V(inv_scale);
                    inv_r = lane_rcp(rho_t);
                }
                // one site per lane: species-A lanes take column x, species-B
                // lanes column x+1; each lane sends its partner the force the
                // partner's site needs, so one shuffle gives F_x of both species
                const C fx_partner = __shfl_xor_sync(0xffffffffu, sp ? Fx.a() : Fx.b(), 16);
                const C Fx_t = (sp ? Fx.b() : Fx.a()) + fx_partner;
                const C up = ((sp ? jxo.b() : jxo.a()) + C(0.5) * Fx_t) * (sp ? inv_r.b() : inv_r.a());
                // the row sums of u_x are the service warp's (svc_profile, after the
                // next barrier): sums carried as an unevaluated pair (error-free
                // two-sum), then added in FP64, ~2^-48 relative
                ubuf[(j & 1) * TX + c0 + sp] = (ANY && sp ? act_b : act) ? up : C(0);
                if (wall_lo || wall_hi) {
                    const double wsum = warp_sum_compensated2(dpx_site, C(0));
                    const int nbx = (g.nx + 31) / 32, wg = (x0 >> 5) + warp;
                    if (lane == 0 && wg < nbx) wall_part[((long long)cell * nbx + wg) * 2 + (wall_lo ? 1 : 0)] = wsum;
                }
            }
        }
        if (SAMPLE && !aborted) {
            __syncthreads();  // the last row's u_x values are in place
            if (svc)
                profile_row_sums<C, TX>(ubuf + ((rows - 1) & 1) * TX, lane, prof_part, cell, g.nx, rm.nown, x0,
                                        y0 + rows - 1 - rm.ylo);
        }
        if (aborted) {
            if (producer) {
                atomicOr(err, ERR_TIMEOUT);
                // drain the copies still in flight before shared memory is released
                for (uint32_t n = nrow; n < n_issued; ++n)
                    if (n != skip_row) mbar_wait_bounded(&bars[n % D], (n / D) & 1u, 500000000ull);
            }
            __syncthreads();
            break;
        }
        nrow += (uint32_t)R;
    }
    if (__syncthreads_or(bad) && t == 0) atomicOr(err, ERR_NONFINITE);
}

template <class T, int TX, int FAM>
static const void* kernel_ptr(bool sample)
{
    return sample ? reinterpret_cast<const void*>(&tiled_step_kernel<T, TX, true, FAM>)
                  : reinterpret_cast<const void*>(&tiled_step_kernel<T, TX, false, FAM>);
}

template <class T, int TX>
static const void* kernel_ptr(bool sample, int fam)
{
    if constexpr (std::is_same<T, float>::value && (TX == 64 || TX == 128)) {  // tiled_any_supported
        if (fam == FAM_ANY) return kernel_ptr<T, TX, FAM_ANY>(sample);
        if (fam == FAM_ANY_MRT) return kernel_ptr<T, TX, FAM_ANY_MRT>(sample);
    }
    if constexpr (std::is_same<T, float>::value && TX == 128)  // full_big
        if (fam == FAM_FULL_BIG) return kernel_ptr<T, TX, FAM_FULL_BIG>(sample);
    return fam == FAM_FULL ? kernel_ptr<T, TX, FAM_FULL>(sample)
         : fam == FAM_GEN  ? kernel_ptr<T, TX, FAM_GEN>(sample)
                           : kernel_ptr<T, TX, FAM_MRT>(sample);
}

// The kernel of storage type T (instantiated in a file of its own per type, so that
// they compile side by side: lb_tiled_f32.cu, ...).
template <class T>
const void* tiled_kernel(int tx, bool sample, int fam)
{
    switch (tx) {
    case 32: return kernel_ptr<T, 32>(sample, fam);
    case 64: return kernel_ptr<T, 64>(sample, fam);
    case 128: return kernel_ptr<T, 128>(sample, fam);
    default: return kernel_ptr<T, 256>(sample, fam);
    }
}

}  // namespace lbhb
