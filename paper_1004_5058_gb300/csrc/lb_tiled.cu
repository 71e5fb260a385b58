// Host side of the tiled kernel family (lb_tiled.cuh): tensor maps, tile and grid
// choice, launches.
#include <cudaTypedefs.h>

#include <algorithm>

#include "lb_tiled.cuh"

namespace lbhb {

extern template const void* tiled_kernel<float>(int, bool, int);
extern template const void* tiled_kernel<double>(int, bool, int);
extern template const void* tiled_kernel<__half>(int, bool, int);
extern template const void* tiled_kernel<half_sr>(int, bool, int);

struct SlotGeom {
    int main_b, halo_b, main_al, halo_al, slot_b, tx_bytes, halo;
};

__host__ __device__ inline SlotGeom slot_geom(int tx, int elem)
{
    SlotGeom s;
    s.halo = 16 / elem;
    s.main_b = 18 * tx * elem;
    s.halo_b = 18 * s.halo * elem;
    s.main_al = al128(s.main_b);
    s.halo_al = al128(s.halo_b);
    s.slot_b = s.main_al + 2 * s.halo_al;
    s.tx_bytes = s.main_b + 2 * s.halo_b;
    return s;
}

struct TiledPlan {
    Geom g;     // the whole population buffer (for a slab: its own rows and two ghost rows each side)
    RowMap rm;  // the rows a step updates
    int elem, bc, tx, ty, depth;
    int n_strips, n_seg;
    bool any;        // any width: the FAM_ANY kernels
    bool big;        // full_big
    int grid[N_FAM][2];  // persistent CTAs: [kernel family FAM_*][plain 0 / sampled 1]
    size_t smem;
    CUtensorMap tm_main[2], tm_halo[2];
    void* f[2];
    uint32_t skip_row = ~0u;  // failure injection for the next launch (tests)
    int collision = TILED_BGK_ONE_TIME;  // the cells' collision (tiled_set_collision)
};

// ------------------------------------------------------------- host side --
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

static int depth_for(int tx, int elem) { return ring_depth(tx, elem); }

static size_t smem_bytes(int tx, int elem, int depth)
{
    const SlotGeom sg = slot_geom(tx, elem);
    const int cb = elem == 8 ? 8 : 4;
    // slots, psi/rho rings, mbarriers, and two rows of per-site profile values
    const size_t b = (size_t)depth * sg.slot_b + (size_t)4 * ring_species_stride(tx) * cb + (size_t)depth * 8 +
                     (size_t)2 * tx * cb;
    return b;
}
static_assert(tiled_smem_bytes(128, 4) == 74032, "shared memory of the FP32 128-column tile");

// FP64: row times of an SM with `per_sm` work items of ty rows (the four halo rows only
// pass through psi: 2 rows' worth).  As many items at a time as the SM holds CTAs; a row
// of theirs takes the FP64 pipes of its four sub-partitions in turn, or one warp's time
// on one of them where fewer than four column warps run, and one CTA alone leaves the
// pipe idle for an eighth of the time.  Counting every row as if it filled the pipe gave
// 12 x (160 x 300) in 32 columns 60-row segments, two warps on an SM, and 565 us per
// step; 30-row ones take 345.  2 x (480 x 1000) 929 -> 564, 24 x (96 x 96) 231 -> 146.
static double fp64_row_times(long long per_sm, int ty, int tile_x)
{
    const int occ = tiled_min_ctas(tile_x, 8);
    double t = 0.0;
    for (long long left = per_sm; left > 0; left -= occ)
        t += (ty + 2) * std::max(1.0, (double)std::min<long long>(left, occ) * (tile_x / 32) / 4.0);
    return per_sm == 1 ? 1.13 * t : t;
}

// Segment height from a model of the time of a launch: work items = strips x
// segments x cells; an item walks its rows, four halo rows and about 1.5 row-times
// of start-up one after another, and a row takes longer the more column warps share
// the SM.  us per row measured on 384^2 .. 1024^2 FP32 cells: 0.75 with one
// 128-column CTA per SM, 0.93 with two, 1.2 with three (a service warp counts half).  More items than resident
// CTAs run in rounds.  FP64 rows share the SM's FP64 pipe: see fp64_row_times.
// Heights below 8 (the least before) pay on lattices that do not fill the chip: us
// per step at 8 rows / at the model's choice: 512^2 FP32 12.3 / 10.8 (5 rows), 48
// cells of 64^2 12.3 / 10.6 (6), 512^2 FP16 13.5 / 11.9 (5), FP64 177 / 161 (14).
// A narrower last strip counts as a strip: leaving it out gave 1000 x 1000 FP32
// 16-row segments in two rounds, 38.4 us, where 18 rows take one, 30.0 us.
static int pick_segment_rows(const Geom& g, int nrows, int tile_x, int elem, int sms, int occ)
{
    const long long strips = (g.nx + tile_x - 1) / tile_x;
    int best = 32;
    double best_cost = 1e300;
    for (int ty = 2; ty <= 256 && ty <= nrows; ++ty) {
        const long long items = strips * g.n_cells * ((nrows + ty - 1) / ty);
        const long long per_sm = (items + sms - 1) / sms;  // items of the fullest SM
        double cost;
        if (elem == 8) {
            cost = fp64_row_times(per_sm, ty, tile_x);
        } else {
            const long long rounds = (items + (long long)sms * occ - 1) / ((long long)sms * occ);
            const double warps = (double)std::min<long long>(per_sm, occ) * (tile_x / 32 + 0.5);
            cost = (double)rounds * (ty + 5.5) * (0.6 + 0.04 * warps);
        }
        if (cost < best_cost - 1e-9) {
            best_cost = cost;
            best = ty;
        }
    }
    return best;
}

bool tiled_supported(const Geom& g, int elem, int tile_x, int tile_y)
{
    if (tile_x != 32 && tile_x != 64 && tile_x != 128 && tile_x != 256) return false;
    // tile_y 0: chosen by the fill model.  nx need not be a multiple of the tile
    // (the last strip is narrower) but must be even (column pairs) and its rows
    // 16-byte multiples (TMA strides and halo coordinates).
    if (tile_y < 0 || g.nx % 2 != 0 || g.ny < 5) return false;
    if (g.nx < tile_x || (g.nx * elem) % 16 != 0) return false;
    if (18 * g.plane >= (1LL << 31)) return false;  // 32-bit element offsets inside a cell
    if (smem_bytes(tile_x, elem, depth_for(tile_x, elem)) > 227 * 1024) return false;
    return encode_fn() != nullptr;
}

bool tiled_any_supported(const Geom& g, int elem, int tile_x)
{
    return elem == 4 && (tile_x == 64 || tile_x == 128) && g.nx >= tile_x && g.ny >= 5 && 18 * g.plane < (1LL << 31) &&
           encode_fn() != nullptr;
}

int tiled_partials_nbx(const Geom& g, int) { return (g.nx + 31) / 32; }

static const void* pick_any(int prec, int tx, bool sample, int fam)
{
    switch (prec) {
    case LB_FP32: return tiled_kernel<float>(tx, sample, fam);
    case LB_FP64: return tiled_kernel<double>(tx, sample, fam);
    case LB_FP16_SHIFTED_SR: return tiled_kernel<half_sr>(tx, sample, fam);
    default: return tiled_kernel<__half>(tx, sample, fam);
    }
}

// Whether FAM_FULL launches run as FAM_FULL_BIG: FP32 in 128-column tiles whose two
// buffers are more than twice the L2 (129 MB), so that a step streams from memory and
// rows that finish sooner only spread the CTAs' accesses.  us per step, FAM_FULL /
// FAM_FULL_BIG: 1024^2 (151 MB) 28.4 / 28.8, 16 x 512^2 (604 MB) 101.4 / 100.9,
// 8 x 1024^2 (1.2 GB) 202.0 / 199.9; 1024 x 64^2 (604 MB, 64 columns) 118.8 / 122.3.
// Their row copies also fetch 256 bytes into the L2 at a time, where 128 serve the
// others: 128 / 256 bytes, 8 x 1024^2 202.0 / 200.9, 16 x 512^2 101.7 / 101.4, two
// relaxation times 200.9 / 199.8, 4096^2 419 / 421; 512^2, which the L2 holds, 10.67 / 10.78.
static bool full_big(const Geom& g, int prec, int tile_x)
{
    return prec == LB_FP32 && tile_x == 128 && 2 * 18 * g.plane * g.n_cells * 4 > (256LL << 20);
}

// The family a launch runs: the full-width one when the strips are whole and
// every cell has one relaxation time and BGK, else the general or MRT one.
static int launch_family(const TiledPlan* p)
{
    if (p->any) return p->collision == TILED_MRT ? FAM_ANY_MRT : FAM_ANY;
    if (p->collision == TILED_MRT) return FAM_MRT;
    if (p->g.nx % p->tx != 0 || p->collision != TILED_BGK_ONE_TIME) return FAM_GEN;
    return p->big ? FAM_FULL_BIG : FAM_FULL;
}

static bool encode(CUtensorMap* m, void* base, const Geom& g, int elem, int box_x, bool big)
{
    auto fn = encode_fn();
    if (!fn) return false;
    const CUtensorMapDataType dt = elem == 4   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : elem == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64
                                               : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, 18, (cuuint64_t)g.n_cells};
    cuuint64_t strides[3] = {(cuuint64_t)g.pitch * elem, (cuuint64_t)g.plane * elem,
                             (cuuint64_t)g.cellstride * elem};
    cuuint32_t box[4] = {(cuuint32_t)box_x, 1, 18, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = fn(m, dt, 4, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, big ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

TiledPlan* tiled_create(const Geom& g, const RowMap& rm, int prec, int elem, int bc, void* f0, void* f1, int tile_x,
                        int tile_y, bool any, int collision, const char** err_msg)
{
    if (any ? !tiled_any_supported(g, elem, tile_x) : !tiled_supported(g, elem, tile_x, tile_y)) {
        if (err_msg) *err_msg = "shape/tile not supported by the tiled kernel";
        return nullptr;
    }
    TiledPlan* p = new TiledPlan();
    p->g = g;
    p->rm = rm;
    p->elem = elem;
    p->bc = bc;
    p->any = any;
    p->collision = collision;
    p->tx = tile_x;
    p->ty = tile_y;
    p->big = full_big(g, prec, tile_x);
    p->depth = depth_for(tile_x, elem);
    p->n_strips = (g.nx + tile_x - 1) / tile_x;
    p->smem = smem_bytes(tile_x, elem, p->depth);
    p->f[0] = f0;
    p->f[1] = f1;
    const int halo = 16 / elem;
    for (int b = 0; b < 2; ++b)
        if (!encode(&p->tm_main[b], b ? f1 : f0, g, elem, tile_x, p->big) ||
            !encode(&p->tm_halo[b], b ? f1 : f0, g, elem, halo, p->big)) {
            if (err_msg) *err_msg = "cuTensorMapEncodeTiled failed";
            delete p;
            return nullptr;
        }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // occupancy of each kernel: the full-width family (nx a multiple of the tile,
    // one relaxation time), the general one and the MRT one, each plain and
    // sampled; which family runs depends on the cells' collision, which lb_load
    // may change, so all are prepared.  Plain and sampled launches of a family
    // share the work items (the segment height) but each runs as many persistent
    // CTAs as fit (the sampled variant holds more registers)
    const bool full_ok = g.nx % tile_x == 0;
    const int full = p->big ? FAM_FULL_BIG : FAM_FULL, no_full = p->big ? FAM_FULL : FAM_FULL_BIG;
    int occ[N_FAM][2] = {};
    for (int s = 0; s < 2 * N_FAM; ++s) {
        const int fam = s >> 1, smp = s & 1;
        if (any != (fam >= FAM_ANY) || (fam == full && !full_ok) || fam == no_full) continue;
        const void* k = pick_any(prec, tile_x, smp != 0, fam);
        // the whole unified L1/shared array as shared memory: the CTAs' rings
        // are what sets how many fit on an SM
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p->smem) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess) {
            cudaGetLastError();
            if (err_msg) *err_msg = "cudaFuncSetAttribute(max dynamic smem) failed";
            delete p;
            return nullptr;
        }
        int o = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k, tiled_threads(tile_x), p->smem) != cudaSuccess ||
            o < 1) {
            cudaGetLastError();
            if (err_msg) *err_msg = "tiled kernel does not fit on an SM";
            delete p;
            return nullptr;
        }
        occ[fam][smp] = o;
    }
    // segment height for the plain kernel of the family that these cells run: by the BGK
    // kernel's CTAs per SM, which the MRT kernel's registers do not allow in 64 columns,
    // MRT cells got segments in a little over one round.  us per step with those / these:
    // 16 x (96 x 512) 48.3 / 32.7, 8 x (192 x 400) 30.7 / 21.5, 8 x 320^2 38.0 / 27.9
    if (p->ty <= 0) p->ty = pick_segment_rows(g, rm.nown, tile_x, elem, sms, occ[launch_family(p)][0]);
    p->n_seg = (rm.nown + p->ty - 1) / p->ty;
    const long long items = (long long)p->n_strips * p->n_seg * g.n_cells;
    for (int fam = 0; fam < N_FAM; ++fam)
        for (int smp = 0; smp < 2; ++smp)
            p->grid[fam][smp] = occ[fam][smp] > 0 ? (int)std::min(items, (long long)sms * occ[fam][smp]) : 0;
    return p;
}

void tiled_destroy(TiledPlan* p) { delete p; }

void tiled_inject_skip(TiledPlan* p, uint32_t row) { p->skip_row = row; }

void tiled_set_collision(TiledPlan* p, int collision) { p->collision = collision; }

void tiled_tiles(const TiledPlan* p, int* tx, int* ty)
{
    *tx = p->tx;
    *ty = p->ty;
}

void tiled_launch_shape(const TiledPlan* p, int* grid_plain, int* grid_sampled, int* threads, int* smem)
{
    const int fam = launch_family(p);
    if (grid_plain) *grid_plain = p->grid[fam][0];
    if (grid_sampled) *grid_sampled = p->grid[fam][1];
    if (threads) *threads = tiled_threads(p->tx);
    if (smem) *smem = (int)p->smem;
}

template <class T>
cudaError_t launch_tiled_step(TiledPlan* p, int src, const CellDev* cells, bool sample, double* prof_part,
                              double* wall_part, unsigned* err, cudaStream_t st, int* n_launches)
{
    const T* from = reinterpret_cast<const T*>(p->f[src]);
    T* dst = reinterpret_cast<T*>(p->f[1 - src]);
    const int fam = launch_family(p);
    const void* k = tiled_kernel<T>(p->tx, sample, fam);
    Geom g = p->g;
    RowMap rm = p->rm;
    int bc = p->bc, ty = p->ty, ns = p->n_strips, nseg = p->n_seg;
    uint32_t skip = p->skip_row;
    p->skip_row = ~0u;  // one launch only
    void* args[] = {(void*)&p->tm_main[src], (void*)&p->tm_halo[src], (void*)&from, (void*)&dst, (void*)&g, (void*)&bc,
                    (void*)&rm, (void*)&ty, (void*)&ns, (void*)&nseg, (void*)&cells, (void*)&prof_part,
                    (void*)&wall_part, (void*)&err, (void*)&skip};
    cudaError_t e = cudaLaunchKernel(k, dim3(p->grid[fam][sample ? 1 : 0]), dim3(tiled_threads(p->tx)), args,
                                     p->smem, st);
    *n_launches += 1;
    return e;
}

template cudaError_t launch_tiled_step<float>(TiledPlan*, int, const CellDev*, bool, double*, double*, unsigned*,
                                              cudaStream_t, int*);
template cudaError_t launch_tiled_step<double>(TiledPlan*, int, const CellDev*, bool, double*, double*, unsigned*,
                                               cudaStream_t, int*);
template cudaError_t launch_tiled_step<__half>(TiledPlan*, int, const CellDev*, bool, double*, double*, unsigned*,
                                               cudaStream_t, int*);
template cudaError_t launch_tiled_step<half_sr>(TiledPlan*, int, const CellDev*, bool, double*, double*, unsigned*,
                                                cudaStream_t, int*);

}  // namespace lbhb
