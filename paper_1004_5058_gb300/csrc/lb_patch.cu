// Patch kernel: many time steps of a small lattice in one launch.
//
// The tiled kernel (lb_tiled.cuh) walks rows: a segment costs its rows plus six
// one after another, however few there are, and every step is a launch.  A
// lattice of 64^2 sites then keeps 8 SMs busy for 12 rows.  Here a thread block
// takes a patch of BX x BY sites and updates all of it at once, so the whole
// chip works on a lattice of any size, and a block goes on to the next step as
// soon as the blocks around it have finished this one.
//
// A block per patch (blocks loop over patches where there are more patches than
// resident blocks): every thread holds one species at two adjacent columns of
// one row (lanes 0-15 of a warp species A, 16-31 species B of the same sites,
// as in the tiled kernel, so both give the same bits).
//   * the 9 populations of the pair come straight from L2 into registers; the
//     pairs of the two-site halo around the patch are loaded and summed by the
//     same threads, so rho_s and psi_s of patch and halo are in shared memory
//     after one barrier;
//   * the pair is collided and pushed to the other ping-pong buffer.
// The halo's densities are computed again by every block that needs them: a
// second round of loads for 0.7 of a patch's sites, where an exchange of densities
// would cost a second wait per step.
//
// Bound: latency.  A step is the chain flag -> populations -> densities -> collision
// -> stores -> flag, two trips through L2 and a release that waits for the stores:
// 3.2 us at 64^2 FP32 (a launch of the tiled kernel per step: 9.3 us with 8-row
// segments, 6.0 with 2-row ones).  In FP64 that chain is long by its FP64 instructions,
// 64 cycles each on a sub-partition: 11 us at 64^2 (102 before; the pipes 28 % busy,
// two warps on an SM's four), 45 at 256^2, where the pipes fill; two sites per thread
// took 19.3 us at 64^2 where one took 12.3.
//
// Steps are ordered by one flag per patch (the number of steps it has behind it):
// a patch starts step s when all patches within three sites of it have finished
// step s - 1.  Those hold every site it reads (two sites away, populations pushed
// there from one further out), and every reader of the sites it overwrites.  The
// launch is cooperative, so all blocks are resident and every wait ends; it is
// bounded all the same (ERR_TIMEOUT).
#include <algorithm>
#include <limits>

#include "lb_internal.h"
#include "lb_pair.cuh"
#include "lbhb.h"
#include "tma.cuh"

namespace lbhb {

struct PatchArgs {
    void* in[2];   // step s reads in[s & 1] and writes out[s & 1]
    void* out[2];
    Geom g;
    int bc, npx, npy;  // patches per row and column of a cell
    int steps;
    int first, every;  // sampled steps of this launch: first, first + every, ... (first < 0: none)
    const CellDev* cells;
    // sampled steps k = 0, 1, ... of this launch, in the compute type: u_x of every
    // site [k][cell][ny][nx], and what the walls deliver [k][cell][top, bottom]
    // [species][PatchLane::DW][columns / sites per lane]
    void *u, *dp;
    unsigned* err;
    unsigned* flags;  // [cell][npy][npx] steps done
    unsigned long long wait_ns;  // bound of each wait for a flag
    unsigned withhold;           // failure injection (tests): patch 0 never sets its flag
};

// Pair p, p + 1 of stored elements through L2 (the data other blocks of this
// launch wrote are never in this SM's L1).
__device__ __forceinline__ P2<float> ld_pair(const float* p) { return P2<float>(__ldcg(reinterpret_cast<const float2*>(p))); }
__device__ __forceinline__ P2<float> half_pair(unsigned u)
{
    __half2 h;
    memcpy(&h, &u, 4);
    return P2<float>(__half22float2(h));
}
__device__ __forceinline__ P2<float> ld_pair(const __half* p) { return half_pair(__ldcg(reinterpret_cast<const unsigned*>(p))); }
__device__ __forceinline__ P2<float> ld_pair(const half_sr* p) { return half_pair(__ldcg(reinterpret_cast<const unsigned*>(p))); }
__device__ __forceinline__ float ld_one(const float* p) { return __ldcg(p); }
__device__ __forceinline__ float half_one(unsigned short u)
{
    __half h;
    memcpy(&h, &u, 2);
    return __half2float(h);
}
__device__ __forceinline__ float ld_one(const __half* p) { return half_one(__ldcg(reinterpret_cast<const unsigned short*>(p))); }
__device__ __forceinline__ float ld_one(const half_sr* p) { return half_one(__ldcg(reinterpret_cast<const unsigned short*>(p))); }

// What a thread holds of one species: two adjacent sites of a row, or one in
// FP64, whose pipe takes 64 cycles per warp instruction on each of the SM's four
// sub-partitions: half as many instructions per warp on twice as many warps.
template <class T> struct PatchLane {
    using V = P2<float>;
    static constexpr int NS = 2;
    static constexpr int DW = 1;  // wall momentum of the pair, three links summed
};
template <> struct PatchLane<double> {
    using V = P1;
    static constexpr int NS = 1;
    static constexpr int DW = 3;  // of each link, so that pairs of sites can be summed link by link
};
__device__ __forceinline__ double first(P1 v) { return v.x; }
__device__ __forceinline__ float first(P2<float> v) { return v.a(); }
__device__ __forceinline__ double second(P1 v) { return v.x; }
__device__ __forceinline__ float second(P2<float> v) { return v.b(); }
__device__ __forceinline__ P1 from_partner(P1 v) { return P1(__shfl_xor_sync(0xffffffffu, v.x, 16)); }
__device__ __forceinline__ P2<float> from_partner(P2<float> v)
{
    return P2<float>(__shfl_xor_sync(0xffffffffu, v.a(), 16), __shfl_xor_sync(0xffffffffu, v.b(), 16));
}

// The half-stencil differences of psi and of the partner's density around one
// lane, read from shared memory: ps and ro point at the window's first element
// (two columns left, two rows above; ro one row above), W words per row.
template <int W> __device__ __forceinline__ void lane_window(const float* ps, const float* ro, P2<float> d[12],
                                                            P2<float> de[4], P2<float>* psi, P2<float>* rho_p)
{
    P2<float> v[5][3], e[3][3];
#pragma unroll
    for (int r = 0; r < 5; ++r)
#pragma unroll
        for (int m = 0; m < 3; ++m) v[r][m] = Pair<float>::ld(ps + r * W + 2 * m);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int m = 0; m < 3; ++m) e[r][m] = Pair<float>::ld(ro + r * W + 2 * m);
    *psi = v[2][1];
    *rho_p = e[1][1];
    window_diffs(v, e, d, de);
}
template <int W> __device__ __forceinline__ void lane_window(const double* ps, const double* ro, P1 d[12], P1 de[4],
                                                            P1* psi, P1* rho_p)
{
    *psi = P1(ps[2 * W + 2]);
    *rho_p = P1(ro[W + 2]);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int o = hs_dy(k) * W + hs_dx(k);
        d[k] = P1(ps[2 * W + 2 + o]) - P1(ps[2 * W + 2 - o]);
        if (k < 4) de[k] = P1(ro[W + 2 + o]) - P1(ro[W + 2 - o]);
    }
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Waits until *p has reached v, for at most `ns` of wall time; false when the time ran out.
__device__ __noinline__ bool wait_flag_bounded(const unsigned* p, unsigned v, unsigned long long ns)
{
    if ((int)(ld_acquire(p) - v) >= 0) return true;
    const uint64_t t0 = global_ns();
    for (uint32_t it = 1;; ++it) {
        if ((int)(ld_acquire(p) - v) >= 0) return true;
        if ((it & 63u) == 0 && global_ns() - t0 > ns) return false;
    }
}

// Column of the lattice at periodic distance (x may lie up to a patch and its
// halo outside, which is several times round on the narrowest lattices).
__device__ __forceinline__ int column(int x, int nx)
{
    if (x < 0) x += nx;
    if (x >= nx) x -= nx;
    return x < 0 || x >= nx ? ((x % nx) + nx) % nx : x;
}

constexpr int PATCH_THREADS = 512;  // at most 128 registers
// Words of a shared row: the patch's columns and two on each side.
__host__ __device__ constexpr int patch_row_words(int pw, int ns) { return ns * pw + 4; }

// PW lanes per row of a patch and species (BX = PW x sites per lane columns); a
// warp covers 16 / PW rows, the block's warps lie below one another.
template <class T, int PW, bool MRT>
__global__ void __launch_bounds__(PATCH_THREADS) patch_steps_kernel(const __grid_constant__ PatchArgs a)
{
    using C = typename Store<T>::C;
    using V = typename PatchLane<T>::V;
    constexpr int NS = PatchLane<T>::NS;
    constexpr C scale = C(Store<T>::scale), inv_scale = C(1) / scale;
    constexpr int BX = NS * PW, RPW = 16 / PW, W = patch_row_words(PW, NS);
    constexpr int SIDE = 2 / NS, R = PW + 2 * SIDE;  // lanes of the halo on each side, lanes of a row with halo
    extern __shared__ __align__(16) unsigned char patch_smem[];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int sp = lane >> 4, pl = lane & (PW - 1), row = warp * RPW + ((lane & 15) / PW);
    const int BY = (int)(blockDim.x >> 5) * RPW, SS = (BY + 4) * W;
    C* const psi_s = reinterpret_cast<C*>(patch_smem);  // [species][BY + 4][W]
    C* const rho_s_ = psi_s + 2 * SS;
    const Geom& g = a.g;
    const int nx = g.nx, ny = g.ny, pitch = g.pitch, pl_el = (int)g.plane;
    bool bad = false;  // watchdog: a non-finite or non-positive density at an updated site

    // a launch behind one that timed out does not wait out its own bound
    if (__syncthreads_or(t == 0 && (*reinterpret_cast<volatile unsigned*>(a.err) & ERR_TIMEOUT) != 0u)) return;

    // patches p = blockIdx.x, + gridDim.x, ...: the strides of (px, py, cell)
    const int per_cell = a.npx * a.npy, n_patches = per_cell * g.n_cells;
    const int d_cell = (int)gridDim.x / per_cell, d_rem = (int)gridDim.x - d_cell * per_cell;
    const int d_py = d_rem / a.npx, d_px = d_rem - d_py * a.npx;
    const int cell_0 = (int)blockIdx.x / per_cell, rem_0 = (int)blockIdx.x - cell_0 * per_cell;
    const int py_0 = rem_0 / a.npx, px_0 = rem_0 - py_0 * a.npx;

    int slot = 0;  // sampled steps so far
    for (int s = 0; s < a.steps; ++s) {
        const T* const fin = reinterpret_cast<const T*>(a.in[s & 1]);
        T* const fout = reinterpret_cast<T*>(a.out[s & 1]);
        const bool sample = a.first >= 0 && s >= a.first && (s - a.first) % a.every == 0;
        int cell = cell_0, py = py_0, px = px_0;
        for (int p = blockIdx.x; p < n_patches; p += gridDim.x) {
            const int x0 = px * BX, y0 = py * BY;
            if (s > 0) {
                bool late = false;
                if (warp == 0 && lane < 25) {
                    // patches that hold a site within three of this one: those at the
                    // corners of distance 1 and 3 (a narrow last patch lies between)
                    const int i = lane % 5, j = lane / 5;
                    const int ex = min(x0 + BX, nx) - 1, ey = min(y0 + BY, ny) - 1;
                    const int qx = column(i < 2 ? x0 - 3 + 2 * i : (i == 2 ? x0 : ex + 2 * i - 5), nx);
                    int qy = j < 2 ? y0 - 3 + 2 * j : (j == 2 ? y0 : ey + 2 * j - 5);
                    qy = a.bc == 0 ? column(qy, ny) : min(max(qy, 0), ny - 1);
                    late = !wait_flag_bounded(a.flags + (cell * a.npy + qy / BY) * a.npx + qx / BX, (unsigned)s, a.wait_ns);
                }
                if (__syncthreads_or(late)) {
                    if (t == 0) atomicOr(a.err, ERR_TIMEOUT);
                    return;
                }
            }
            const ParamSet<C>& pg = params<C>(a.cells[cell]);
            const V rho0_2 = V(pg.rho0), inv_rho0_2 = V(pg.inv_rho0);
            const T* const fc = fin + (long long)cell * g.cellstride;

            // densities of a pair at logical columns X, X + 1 and row Y of species q
            auto load_pair = [&](int X, int Y, int q, V f[9]) {
                const int yy = stencil_row(min(Y, ny + 1), ny, a.bc);
                const int xa = column(X, nx), xb = column(X + 1, nx);
                const T* const src = fc + (q * 9 * pl_el + yy * pitch);
                if constexpr (NS == 1) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) f[i] = V(__ldcg(src + (i * pl_el + xa)));
                } else if (xb == xa + 1 && (xa & 1) == 0) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) f[i] = ld_pair(src + (i * pl_el + xa));
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i) f[i] = V(ld_one(src + (i * pl_el + xa)), ld_one(src + (i * pl_el + xb)));
                }
            };
            auto put_pair = [&](const V f[9], int q, int srow, int pi) {
                V r = f[0];
#pragma unroll
                for (int i = 1; i < 9; ++i) r = r + f[i];
                if constexpr (Store<T>::shifted) {
                    const V rb = V(q ? pg.rho_bar[1] : pg.rho_bar[0]);
                    if constexpr (Store<T>::scale != 1)
                        r = vfma(r, V(inv_scale), rb);
                    else
                        r = r + rb;
                }
                const int k = q * SS + srow * W + NS * pi;
                *reinterpret_cast<V*>(psi_s + k) = lane_psi(r, rho0_2, inv_rho0_2);
                *reinterpret_cast<V*>(rho_s_ + k) = r;
            };
            const int x = x0 + NS * pl, y = y0 + row;
            V f[9];
            load_pair(x, y, sp, f);
            // the halo ring: two rows above and below, two columns on each side
            const int ring = 4 * R + 2 * SIDE * BY;
            for (int u = t; u < 2 * ring; u += (int)blockDim.x) {
                const int q = u >= ring ? 1 : 0, v = u - q * ring;
                int srow, pi;
                if (v < 4 * R) {
                    const int rr = v / R;
                    pi = v - rr * R;
                    srow = rr < 2 ? rr : BY + rr;
                } else {
                    const int k = (v - 4 * R) & (2 * SIDE - 1);
                    srow = 2 + (v - 4 * R) / (2 * SIDE);
                    pi = k < SIDE ? k : PW + k;
                }
                V h[9];
                load_pair(x0 - 2 + NS * pi, y0 - 2 + srow, q, h);
                put_pair(h, q, srow, pi);
            }
            put_pair(f, sp, row + 2, pl + SIDE);
            __syncthreads();

            // ---- collide the pair (the tiled kernel's arithmetic)
            const bool act_a = x < nx && y < ny, act_b = NS == 2 && x + 1 < nx && y < ny;
            const C tau_s = sp ? pg.tau_b : pg.tau, omega_s = sp ? pg.omega_b : pg.omega;
            const Couplings<V> cp(pg, sp);
            const V tau2 = V(tau_s), ntau2 = V(-tau_s), omega2 = V(omega_s), mix2 = V(sp ? pg.mix[1] : pg.mix[0]);
            const C rho_bar = sp ? pg.rho_bar[1] : pg.rho_bar[0];
            const bool one_time = pg.mix[0] == C(1);
            const bool unit_omega = pg.omega == C(1) && pg.omega_b == C(1);
            V dps[12], dro[4], psi, rho_p;
            lane_window<W>(psi_s + sp * SS + row * W + NS * pl, rho_s_ + (1 - sp) * SS + (row + 1) * W + NS * pl, dps, dro,
                           &psi, &rho_p);
            const V rho_s = *reinterpret_cast<const V*>(rho_s_ + sp * SS + (row + 2) * W + NS * pl + 2);
            const Pull<V> pu = cp.pull(dps, dro);
            const V jx_s = mom_x<V>(f), jy_s = mom_y<V>(f);
            const V jx_p = from_partner(jx_s), jy_p = from_partner(jy_s);
            V jwx = vfma(mix2, jx_p, jx_s), jwy = vfma(mix2, jy_p, jy_s);
            const V rho_w = vfma(mix2, rho_p, rho_s);
            if constexpr (Store<T>::scale != 1) {
                jwx = jwx * V(inv_scale);
                jwy = jwy * V(inv_scale);
            }
            const V inv_rho = lane_rcp(rho_w);
            const V ux = jwx * inv_rho, uy = jwy * inv_rho;
            const C fx_body = body_force_x<C>(pg, y);
            const V rho_t = rho_s + rho_p;
            V ax = V(fx_body) * inv_rho;
            if (!one_time && !is_zero(fx_body)) ax = V(fx_body) * lane_rcp(rho_t);
            bad |= (act_a && !density_ok(first(rho_t))) ||
                   (act_b && !density_ok(second(rho_t)));
            V fs[9], Fx;
            if constexpr (MRT) {
                V mh[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) mh[q] = V(sp ? pg.mrt_h[1][q] : pg.mrt_h[0][q]);
                if constexpr (Store<T>::shifted)
                    collide_species_shifted<V, false, true>(f, rho_s, V(rho_bar), psi, ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx, V(scale), mh);
                else
                    collide_species<V, false, true>(f, rho_s, psi, ux, uy, ax, pu, tau2, ntau2,
                                                    omega2, fs, &Fx, mh);
            } else if constexpr (Store<T>::shifted) {
                if (unit_omega)
                    collide_species_shifted<V, true>(f, rho_s, V(rho_bar), psi, ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx, V(scale));
                else
                    collide_species_shifted<V, false>(f, rho_s, V(rho_bar), psi, ux, uy, ax, pu, tau2, ntau2, omega2, fs, &Fx, V(scale));
            } else {
                if (unit_omega)
                    collide_species<V, true>(f, rho_s, psi, ux, uy, ax, pu, tau2, ntau2, omega2, fs,
                                             &Fx);
                else
                    collide_species<V, false>(f, rho_s, psi, ux, uy, ax, pu, tau2, ntau2, omega2, fs,
                                              &Fx);
            }
            Dither dz;
            if constexpr (Store<T>::dithered)
                dz.seed(((uint32_t)cell * 0x9E3779B1u) ^ ((uint32_t)y << 15) ^ ((uint32_t)x << 1) ^ (uint32_t)sp,
                        __float_as_uint(first(rho_s)) ^ (__float_as_uint(second(rho_s)) * 0x85EBCA6Bu));

            // ---- push streaming, walls in place
            T* const dst = fout + (long long)cell * g.cellstride;
            const int off = sp * 9 * pl_el + x;  // element offsets stay below 2^31 (patch_supported)
            const int row3[3] = {(y == 0 ? ny - 1 : y - 1) * pitch, y * pitch, (y == ny - 1 ? 0 : y + 1) * pitch};
            const bool wall_lo = a.bc == 1 && y == 0, wall_hi = a.bc == 1 && y == ny - 1;
            C dpx_site = C(0);
            // this thread's place in the wall momenta of a sampled step
            constexpr int DW = PatchLane<T>::DW;
            const int n_units = (nx + NS - 1) / NS;
            C* const dp = reinterpret_cast<C*>(a.dp) +
                          (((long long)(slot * g.n_cells + cell) * 2 + (wall_lo ? 1 : 0)) * 2 + sp) * DW * n_units + x / NS;
            int link = 0;
            if (x0 > 0 && x0 + BX < nx && y0 + BY <= ny && !(wall_lo || wall_hi)) {
                // away from the edges in x (uniform over the block): fixed offsets
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const int cy = q_cy(i), cx = q_cx(i);
                    T* const q = dst + (i * pl_el + off + row3[cy + 1]);
                    if constexpr (NS == 1) {
                        q[cx] = first(fs[i]);
                    } else if (cx == 0) {
                        st_pair<T, C>(q, first(fs[i]), second(fs[i]), dz);
                    } else {
                        st_one<T, C>(q + cx, first(fs[i]), dz);
                        st_one<T, C>(q + cx + 1, second(fs[i]), dz);
                    }
                }
            } else if (act_a) {
                // periodic columns, the last column of an odd width, walls
                const int to_m = x == 0 ? nx - 1 : -1;                      // x - 1
                const int to_1 = x + 1 == nx ? -x : 1;                      // x + 1
                const int to_2 = x + 2 >= nx ? x + 2 - nx - x : 2;          // x + 2
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const int cy = q_cy(i), cx = q_cx(i);
                    const bool into_wall = (cy < 0 && wall_lo) || (cy > 0 && wall_hi);
                    if (into_wall) {
                        C dpa, dpb;
                        const C uw = cy < 0 ? -pg.u_wall : pg.u_wall;
                        const C sh = Store<T>::shifted ? C(q_w(i)) * rho_bar : C(0);
                        const C ba = bounce<C>(i, first(fs[i]) * inv_scale + sh, first(rho_s), uw, &dpa);
                        const C bb = bounce<C>(i, second(fs[i]) * inv_scale + sh, second(rho_s), uw, &dpb);
                        T* const q = dst + (q_opp(i) * pl_el + off + row3[1]);
                        if (act_b) {
                            st_pair<T, C>(q, (ba - sh) * scale, (bb - sh) * scale, dz);
                            dpx_site += dpa + dpb;
                        } else {
                            st_one<T, C>(q, (ba - sh) * scale, dz);
                            dpx_site += dpa;
                        }
                        if (NS == 1 && sample) dp[link++ * n_units] = dpa;
                    } else {
                        T* const q = dst + (i * pl_el + off + row3[cy + 1]);
                        if (cx == 0 && act_b) {
                            st_pair<T, C>(q, first(fs[i]), second(fs[i]), dz);
                        } else {
                            st_one<T, C>(q + (cx < 0 ? to_m : cx > 0 ? to_1 : 0), first(fs[i]), dz);
                            if (act_b) st_one<T, C>(q + (cx < 0 ? 0 : to_2), second(fs[i]), dz);
                        }
                    }
                }
            }
            if (sample) {
                // u_x = (j + F/2)/rho: species-A lanes take column x, species-B lanes x + 1
                V jxo = jwx, inv_r = inv_rho;
                if (!one_time) {
                    jxo = jx_s + jx_p;
                    if constexpr (Store<T>::scale != 1) jxo = jxo * V(inv_scale);
                    inv_r = lane_rcp(rho_t);
                }
                const C fx_partner = __shfl_xor_sync(0xffffffffu, sp ? first(Fx) : second(Fx), 16);
                const C Fx_t = (sp ? second(Fx) : first(Fx)) + fx_partner;
                const C up = ((sp ? second(jxo) : first(jxo)) + C(0.5) * Fx_t) * (sp ? second(inv_r) : first(inv_r));
                if (sp ? act_b : act_a)  // one site per thread: species-A lanes
                    reinterpret_cast<C*>(a.u)[((long long)(slot * g.n_cells + cell) * ny + y) * nx + x + sp] = up;
                if (NS == 2 && act_a && (wall_lo || wall_hi)) *dp = dpx_site;
            }
            // every thread is done with shared memory and has stored its pair
            __syncthreads();
            if (t == 0 && a.steps > 1 && p >= (int)a.withhold) st_release(a.flags + p, (unsigned)(s + 1));
            cell += d_cell;
            py += d_py;
            px += d_px;
            if (px >= a.npx) {
                px -= a.npx;
                ++py;
            }
            if (py >= a.npy) {
                py -= a.npy;
                ++cell;
            }
        }
        slot += sample ? 1 : 0;
    }
    if (__syncthreads_or(bad) && t == 0) atomicOr(a.err, ERR_NONFINITE);
}

// Adds the sampled steps of a launch to the time sums, in the order of the tiled
// kernel with TX = 32 NW columns and its accumulation (so the sums are the same
// bit for bit): per step the 32-column groups one after another, then the step.
// One warp per row of a cell.
template <class C, int NS, int DW, int NW>
__global__ void __launch_bounds__(128) patch_finish_kernel(const C* __restrict__ u, const C* __restrict__ dp, int samples,
                                                           int nx, int ny, int n_cells, int bc,
                                                           double* __restrict__ acc_prof, double* __restrict__ acc_wall)
{
    const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= n_cells * ny) return;
    const int cell = w / ny, y = w - cell * ny, groups = (nx + 31) / 32, n_units = (nx + NS - 1) / NS;
    constexpr int SEG = 32 / NW;
    double acc = acc_prof[w];
    for (int k = 0; k < samples; ++k) {
        const C* row = u + ((long long)(k * n_cells + cell) * ny + y) * nx;
        double sum = 0.0;
        for (int b0 = 0; b0 < groups; b0 += NW) {
            const double part = group_sum<NW>(lane, [&](int q) {
                const int x = b0 * 32 + lane * NW + q;
                return x < nx ? row[x] : C(0);
            });
#pragma unroll
            for (int m = 0; m < NW; ++m)
                if (b0 + m < groups) sum += __shfl_sync(0xffffffffu, part, m * SEG);
        }
        acc += sum;
    }
    if (lane == 0) acc_prof[w] = acc;
    if (bc != 1 || (y != 0 && y != ny - 1)) return;
    const int wall = y == 0 ? 1 : 0, sp = lane >> 4;
    acc = acc_wall[cell * 2 + wall];
    for (int k = 0; k < samples; ++k) {
        const C* d = dp + (((long long)(k * n_cells + cell) * 2 + wall) * 2 + sp) * DW * n_units;
        double sum = 0.0;
        for (int b = 0; b < groups; ++b) {
            const int x = b * 32 + 2 * (lane & 15);
            C v = C(0);
            if constexpr (NS == 2) {
                if (x < nx) v = d[x / 2];
            } else {
#pragma unroll
                for (int i = 0; i < DW; ++i)
                    v += (x < nx ? d[i * n_units + x] : C(0)) + (x + 1 < nx ? d[i * n_units + x + 1] : C(0));
            }
            sum += __shfl_sync(0xffffffffu, warp_sum_compensated2(v, C(0)), 0);
        }
        acc += sum;
    }
    if (lane == 0) acc_wall[cell * 2 + wall] = acc;
}

// ------------------------------------------------------------- host side --
struct PatchPlan {
    Geom g;
    int prec, bc, pw, by;
    int npx, npy;
    int grid[2];  // resident blocks: BGK, MRT
    size_t smem;
    int mrt = 0;
    int slots;  // sampled steps a launch may hold
    bool withhold = false;  // failure injection for the next launch (tests)
    void* mem = nullptr;  // one allocation: the sampled steps' values and the flags
    void *u, *dp;
    unsigned* flags;
};

template <class T, int PW> static const void* patch_kernel(bool mrt)
{
    return mrt ? reinterpret_cast<const void*>(&patch_steps_kernel<T, PW, true>)
               : reinterpret_cast<const void*>(&patch_steps_kernel<T, PW, false>);
}
static const void* patch_kernel(int prec, int pw, bool mrt)
{
    switch (prec) {
    case LB_FP32: return patch_kernel<float, 16>(mrt);
    case LB_FP64: return pw == 8 ? patch_kernel<double, 8>(mrt) : patch_kernel<double, 16>(mrt);
    case LB_FP16_SHIFTED_SR: return patch_kernel<half_sr, 16>(mrt);
    default: return patch_kernel<__half, 16>(mrt);
    }
}

void patch_destroy(PatchPlan* p)
{
    if (!p) return;
    cudaFree(p->mem);
    delete p;
}

// Patches of 32 x 8 sites (FP64: 16 x 8): 8 warps, so that a block hides some of
// its own latency, and 0.7 (FP64: 0.9) halo sites per site.  Measured against 4,
// 9, 12 and 16 rows and 8- and 16-column patches on 64^2 .. 512^2 cells: at 256^2
// FP32 5.98 us per step against 9.4 (32 x 4) and 10.1 (16 x 8).  Up to 10240 sites
// FP64 takes 8 x 4 patches: 64^2 then has 128 of them, one for nearly every SM, whose
// FP64 pipes are the bound; above, 16 columns by the 5 to 8 rows that spread best
// (256^2: 7 rows 44.8 us, 8 rows 49.6).  us per step, 8 x 4 / 16 columns: 32^2 9.6 /
// 11.7, 64^2 11.2 / 12.1, 101 x 83 11.8 / 13.2, 96 x 106 12.7 / 13.2, 104^2 13.7 / 13.4,
// 112^2 13.3 / 14.0, 120^2 14.9 / 13.8, 128^2 17.1 / 14.0; two cells of 64^2 13.2 / 12.3,
// four 17.4 / 15.4.
PatchPlan* patch_create(const Geom& g, int prec, int bc)
{
    if (18 * g.plane >= (1LL << 31)) return nullptr;  // 32-bit element offsets inside a cell
    int dev = 0, sms = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop) return nullptr;
    const bool few = prec == LB_FP64 && (long long)g.nx * g.ny * g.n_cells <= 10240;
    const int pw = few ? 8 : 16;
    int by = few ? 4 : 8;
    if (prec == LB_FP64 && !few) {
        // bound by the SMs' FP64 pipes: the height that gives the fullest SM least to do
        auto load = [&](int h) {
            const long long n = (long long)((g.nx + 15) / 16) * ((g.ny + h - 1) / h) * g.n_cells;
            return ((n + sms - 1) / sms) * (h + 3);  // rows of a patch, and its halo's densities
        };
        for (int h = 7; h >= 5; --h)
            if (load(h) < load(by)) by = h;
    }
    PatchPlan* p = new PatchPlan();
    p->g = g;
    p->prec = prec;
    p->bc = bc;
    p->pw = pw;
    p->by = by;
    const int ns = prec == LB_FP64 ? 1 : 2;  // PatchLane
    p->npx = (g.nx + ns * pw - 1) / (ns * pw);
    p->npy = (g.ny + by - 1) / by;
    p->smem = (size_t)4 * (by + 4) * patch_row_words(pw, ns) * (prec == LB_FP64 ? 8 : 4);
    const long long n = (long long)p->npx * p->npy * g.n_cells;
    const int threads = 32 * by / (16 / pw);
    for (int m = 0; m < 2; ++m) {
        int occ = 0;
        if (n >= (1LL << 30) ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, patch_kernel(prec, pw, m != 0), threads, p->smem) !=
                cudaSuccess ||
            occ < 1) {
            cudaGetLastError();
            patch_destroy(p);
            return nullptr;
        }
        p->grid[m] = (int)std::min<long long>(n, (long long)occ * sms);
    }
    // up to 32 sampled steps per launch in 4 MB (at least one)
    const size_t cb = prec == LB_FP64 ? 8 : 4, u_bytes = cb * g.n_cells * g.ny * g.nx;
    const size_t dp_bytes = cb * g.n_cells * 4 * (prec == LB_FP64 ? 3 * (size_t)g.nx : (size_t)(g.nx + 1) / 2);
    p->slots = (int)std::max<size_t>(1, std::min<size_t>(32, (4u << 20) / u_bytes));
    const size_t u_all = (u_bytes * p->slots + 15) / 16 * 16, dp_all = (dp_bytes * p->slots + 15) / 16 * 16;
    if (cudaMalloc(&p->mem, u_all + dp_all + sizeof(unsigned) * n) != cudaSuccess) {
        cudaGetLastError();
        patch_destroy(p);
        return nullptr;
    }
    p->u = p->mem;
    p->dp = (char*)p->mem + u_all;
    p->flags = (unsigned*)((char*)p->mem + u_all + dp_all);
    return p;
}

int patch_max_samples(const PatchPlan* p) { return p->slots; }

// Steps of about 2 ms, so that other streams' kernels get their turn, and at most 512.
// us per step measured / by this line: FP32 64^2 3.2 / 3.2, 256^2 6.6 / 6.9; FP64 64^2
// 11 / 11, 128^2 14 / 20, 256^2 45 / 54, 320^2 75 / 80; MRT rows take up to 1.5 times as
// long.  A launch costs about 6 us.
int patch_max_steps(const PatchPlan* p)
{
    const double sites = (double)p->g.n_cells * p->g.nx * p->g.ny;
    const double us = (p->prec == LB_FP64 ? 8.0 + 7e-4 * sites : 3.0 + 6e-5 * sites) * (p->mrt ? 1.5 : 1.0);
    return (int)std::min(512.0, std::max(1.0, 2000.0 / us));
}

void patch_inject_withhold(PatchPlan* p) { p->withhold = true; }

void patch_set_collision(PatchPlan* p, int collision) { p->mrt = collision == TILED_MRT; }

// (the launches' own codes: cudaGetLastError would also return an error that an
// earlier call of the same thread left behind)
template <class C, int NS, int DW>
static cudaError_t launch_patch_finish(const PatchPlan* p, int samples, int tile_x, double* acc_prof, double* acc_wall,
                                       cudaStream_t st)
{
    const Geom& g = p->g;
    const void* k;
    switch (tile_x) {
    case 64: k = reinterpret_cast<const void*>(&patch_finish_kernel<C, NS, DW, 2>); break;
    case 128: k = reinterpret_cast<const void*>(&patch_finish_kernel<C, NS, DW, 4>); break;
    case 256: k = reinterpret_cast<const void*>(&patch_finish_kernel<C, NS, DW, 8>); break;
    default: k = reinterpret_cast<const void*>(&patch_finish_kernel<C, NS, DW, 1>); break;
    }
    const C *u = (const C*)p->u, *dp = (const C*)p->dp;
    int nx = g.nx, ny = g.ny, n_cells = g.n_cells, bc = p->bc;
    void* args[] = {(void*)&u, (void*)&dp, (void*)&samples, (void*)&nx, (void*)&ny, (void*)&n_cells, (void*)&bc,
                    (void*)&acc_prof, (void*)&acc_wall};
    return cudaLaunchKernel(k, dim3((n_cells * ny + 3) / 4), dim3(128), args, 0, st);
}

cudaError_t launch_patch_steps(PatchPlan* p, void* src, void* dst, int steps, int first, int every, bool swap, int tile_x,
                               const CellDev* cells, double* acc_prof, double* acc_wall, unsigned* err,
                               cudaStream_t st, int* n_launches)
{
    const int samples = first < 0 ? 0 : (steps - 1 - first) / every + 1;
    cudaError_t e = cudaSuccess;
    if (samples > p->slots) return cudaErrorInvalidValue;
    PatchArgs a{};
    a.in[0] = src;
    a.out[0] = dst;
    a.in[1] = swap ? dst : src;
    a.out[1] = swap ? src : dst;
    a.g = p->g;
    a.bc = p->bc;
    a.npx = p->npx;
    a.npy = p->npy;
    a.steps = steps;
    a.first = first;
    a.every = every > 0 ? every : 1;
    a.cells = cells;
    a.u = p->u;
    a.dp = p->dp;
    a.err = err;
    a.flags = p->flags;
    a.wait_ns = p->withhold ? 200000000ull : 1500000000ull;  // a step takes microseconds
    a.withhold = p->withhold ? 1u : 0u;
    p->withhold = false;  // one launch only
    if (steps > 1) e = cudaMemsetAsync(p->flags, 0, sizeof(unsigned) * p->g.n_cells * p->npx * p->npy, st);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&a};
    e = cudaLaunchCooperativeKernel(patch_kernel(p->prec, p->pw, p->mrt != 0), dim3(p->grid[p->mrt]),
                                    dim3(32 * p->by / (16 / p->pw)), args, p->smem, st);
    if (e != cudaSuccess) return e;
    *n_launches += 1;
    if (samples > 0) {
        e = p->prec == LB_FP64 ? launch_patch_finish<double, 1, 3>(p, samples, tile_x, acc_prof, acc_wall, st)
                               : launch_patch_finish<float, 2, 1>(p, samples, tile_x, acc_prof, acc_wall, st);
        *n_launches += 1;
    }
    return e;
}

}  // namespace lbhb
