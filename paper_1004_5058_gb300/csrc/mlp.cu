// Flow-curve surrogate kernels (include/lbhb_mlp.h): BF16 tensor-core products
// (mma.sync m16n8k16) with FP32 accumulation for inference, and a training step
// (forward, loss, backward) fused into one kernel per slab of the batch, followed by
// an ordered reduction with Adam on FP32 master weights.
//
// Both kernels keep every layer's weights in shared memory and walk over slabs of
// the batch; a layer's 128 columns are split over four warps per 16 rows, because
// what bounds these sizes is the chain of dependent layers within a slab, and most
// of a layer's instructions are its columns' tanh.  Batch rows beyond the live batch
// are zeros, so padded rows and columns never contribute.  Gradients are sums of
// per-CTA partials reduced in a fixed order, so results are reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "lbhb_mlp.h"
#include "lb_internal.h"
#include "tma.cuh"

namespace {

typedef __nv_bfloat16 bf16;

constexpr int NIN = 5, KIN = 16, HID = 128, NOUT = 2, NOUTP = 16;
constexpr long long OFF_W1 = 0, OFF_B1 = OFF_W1 + HID * NIN, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID,
                    OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID * HID, OFF_W4 = OFF_B3 + HID,
                    OFF_B4 = OFF_W4 + NOUT * HID, NPARAM = OFF_B4 + NOUT;

struct LayerDef {
    int in, in_p, out, out_p;
    long long offW, offB;
};
__host__ __device__ constexpr LayerDef layer_def(int l)
{
    return l == 0   ? LayerDef{NIN, KIN, HID, HID, OFF_W1, OFF_B1}
           : l == 1 ? LayerDef{HID, HID, HID, HID, OFF_W2, OFF_B2}
           : l == 2 ? LayerDef{HID, HID, HID, HID, OFF_W3, OFF_B3}
                    : LayerDef{HID, HID, NOUT, NOUTP, OFF_W4, OFF_B4};
}

__device__ __forceinline__ void mma_bf16(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// tanh on the special-function unit (tanh.approx.f32: relative error about
// 2^-11, a quarter of the BF16 rounding the activation then takes), for the
// training kernel's forward pass.  Inference keeps tanhf.
__device__ __forceinline__ float act_tanh(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float bce_logits(float z, float y)
{
    return fmaxf(z, 0.f) - z * y + log1pf(expf(-fabsf(z)));
}

// FP32 masters -> padded BF16 weights [out_p][in_p], padded FP32 biases.
__global__ void refresh_kernel(const float* __restrict__ p, bf16* w1, bf16* w2, bf16* w3, bf16* w4, float* b1, float* b2,
                               float* b3, float* b4)
{
    bf16* W[4] = {w1, w2, w3, w4};
    float* Bp[4] = {b1, b2, b3, b4};
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    int base = 0;
    for (int l = 0; l < 4; ++l) {
        const LayerDef L = layer_def(l);
        const int nw = L.out_p * L.in_p;
        if (k >= base && k < base + nw) {
            const int o = (k - base) / L.in_p, i = (k - base) % L.in_p;
            const float v = (o < L.out && i < L.in) ? p[L.offW + (long long)o * L.in + i] : 0.f;
            W[l][o * L.in_p + i] = __float2bfloat16_rn(v);
        }
        base += nw;
        if (k >= base && k < base + L.out_p) {
            const int o = k - base;
            Bp[l][o] = o < L.out ? p[L.offB + o] : 0.f;
        }
        base += L.out_p;
    }
}

constexpr int MAX_BINS = 256;  // bins of the serving error-budget table

}  // namespace

// --------------------------------------------------- pieces of both kernels --
constexpr int LD = HID + 8;   // padded 128-wide rows: no bank conflicts on fragment loads
constexpr int LDZ = KIN + 8;  // padded 16-wide rows
// all weights in shared memory: W1 [128][LDZ], W2, W3 [128][LD], W4 [16][LD]
constexpr int W_ELEMS = HID * LDZ + 2 * HID * LD + NOUTP * LD;
__host__ __device__ constexpr int w_at(int l) { return l == 0 ? 0 : l == 1 ? HID * LDZ : l == 2 ? HID * LDZ + HID * LD : HID * LDZ + 2 * HID * LD; }

// 16-byte asynchronous global -> shared copies, in commit groups
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldsm_x4(uint32_t r[4], const bf16* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t r[4], const bf16* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

// Copies of all weights into Ws and of the biases into bs, three groups in the order
// of use: biases, W1 | W2 | W3, W4.
constexpr int BIASES = 3 * HID + NOUTP;
template <int THREADS>
__device__ __forceinline__ void stage_all_weights(bf16* Ws, float* bs, const bf16* const W[4], const float* const bias[4],
                                                  int tid)
{
    if (tid < BIASES / 4) {
        const int l = tid / (HID / 4);
        cp_async16(bs + 4 * tid, bias[l] + 4 * tid - l * HID);
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        const LayerDef L = layer_def(l);
        const int ld = l == 0 ? LDZ : LD;
        bf16* const to = Ws + w_at(l);
        for (int e = tid; e < L.out_p * (L.in_p / 8); e += THREADS) {
            const int r = e / (L.in_p / 8), c8 = (e % (L.in_p / 8)) * 8;
            cp_async16(to + r * ld + c8, W[l] + (long long)r * L.in_p + c8);
        }
        if (l != 2) cp_async_commit();
    }
}

// acc = a warp's 16 x 8 NT product of rows r0 .. r0 + 15 of `in` (K wide) with the
// weights Ws[n0 + n][k]: K-steps of 16 in increasing order (NT even).  The operand
// fragments come from ldmatrix: the A tile as four 8 x 8 matrices (rows 0-7 | 8-15)
// x (k 0-7 | 8-15), two n-tiles of B per load.
template <int NT, int K>
__device__ __forceinline__ void rows_times_weights(float (&acc)[NT][4], const bf16* in, int ld_in, const bf16* Ws,
                                                   int ld_w, int r0, int n0, int lane)
{
#pragma unroll
    for (int ni = 0; ni < NT; ++ni)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[ni][r] = 0.f;
    const int j = lane >> 3, rr = lane & 7;
#pragma unroll
    for (int ks = 0; ks < K; ks += 16) {
        uint32_t a[4];
        ldsm_x4(a, in + (r0 + rr + (j & 1) * 8) * ld_in + ks + (j >> 1) * 8);
#pragma unroll
        for (int np = 0; np < NT / 2; ++np) {
            uint32_t b[4];  // (n 0-7, k 0-7 | 8-15), (n 8-15, k 0-7 | 8-15) of the n-tile pair
            ldsm_x4(b, Ws + (n0 + np * 16 + rr + (j >> 1) * 8) * ld_w + ks + (j & 1) * 8);
            mma_bf16(acc[2 * np], a[0], a[1], a[2], a[3], b[0], b[1]);
            mma_bf16(acc[2 * np + 1], a[0], a[1], a[2], a[3], b[2], b[3]);
        }
    }
}

// z = (x - center) / half_range of ROWS batch rows from b0 on, padded to KIN columns
// (zero rows past B)
template <int ROWS, int THREADS>
__device__ __forceinline__ void normalise_rows(bf16* Z, int ld, const float* x, int b0, int B, const float* center,
                                               const float* half, int tid)
{
    for (int e = tid; e < ROWS * KIN; e += THREADS) {
        const int r = e / KIN, c = e % KIN, b = b0 + r;
        float v = 0.f;
        if (b < B && c < NIN) v = (x[b * NIN + c] - center[c]) / half[c];
        Z[r * ld + c] = __float2bfloat16_rn(v);
    }
}

// ----------------------------------------------------------- inference --
// The whole call in one kernel: a CTA takes slabs of 32 queries through the
// normalisation, the three tanh layers and the output layer with every activation in
// shared memory, then makes the fallback decision (mlp_serve) or writes the pair of
// outputs (mlp_forward).  Per 16-wide slice of K one m16n8k16 BF16 product in
// increasing K, bias and tanh in FP32, activations rounded to BF16.
// Warps: 16 rows x 32 columns each, two row groups, four column groups.
// 64 queries on four warps of 16 rows x 128 columns (192 tanh per lane one after
// another) took 14.4 us for up to 4096 queries and 57 us for 65536 (CUDA events over
// back-to-back calls); these take 8.2 and 41, and the pass with a launch per layer
// that mlp_forward ran took 47 and 132.  Bound: the chain of four layers.
constexpr int SRV_ROWS = 32, SRV_THREADS = 256;
constexpr size_t SRV_SMEM = sizeof(bf16) * (2 * SRV_ROWS * LD + W_ELEMS);  // 97 KB: two CTAs per SM

struct ServeArgs {
    const float* x;
    int B;
    const bf16* W[4];
    const float* bias[4];
    const float *center, *half;
    float scale, margin;
    const int* over_budget;
    int n_bins;
    float ls_lo, ls_hi;
    float *stress, *logit;
    int* fallback;
    float* out;  // mlp_forward: [B][2], and no fallback decision
};

__global__ void __launch_bounds__(SRV_THREADS, 2) serve_fused_kernel(ServeArgs a)
{
    extern __shared__ __align__(16) unsigned char srv_smem[];
    bf16* const act0 = reinterpret_cast<bf16*>(srv_smem);
    bf16* const act1 = act0 + SRV_ROWS * LD;
    bf16* const Ws = act1 + SRV_ROWS * LD;
    __shared__ __align__(16) float bias_s[BIASES];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3, r0 = (warp & 1) * 16, n0 = (warp >> 1) * 32;
    stage_all_weights<SRV_THREADS>(Ws, bias_s, a.W, a.bias, tid);
    const int n_slabs = (a.B + SRV_ROWS - 1) / SRV_ROWS;
    for (int slab = blockIdx.x; slab < n_slabs; slab += gridDim.x) {
        const int b0 = slab * SRV_ROWS;
        __syncthreads();  // the previous slab is done with the activations
        normalise_rows<SRV_ROWS, SRV_THREADS>(act0, LD, a.x, b0, a.B, a.center, a.half, tid);
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            // layer l's weights and inputs (the copies have long landed after the first slab)
            if (l == 0) cp_async_wait<2>();
            if (l == 1) cp_async_wait<1>();
            if (l == 2) cp_async_wait<0>();
            __syncthreads();
            const bf16* const in = (l & 1) ? act1 : act0;
            bf16* const out = (l & 1) ? act0 : act1;
            float acc[4][4];
            if (l == 0)
                rows_times_weights<4, KIN>(acc, in, LD, Ws, LDZ, r0, n0, lane);
            else
                rows_times_weights<4, HID>(acc, in, LD, Ws + w_at(l), LD, r0, n0, lane);
#pragma unroll
            for (int ni = 0; ni < 4; ++ni)
#pragma unroll
                for (int r = 0; r < 4; r += 2) {
                    const int row = r0 + g + (r >= 2 ? 8 : 0), col = n0 + ni * 8 + 2 * t4;
                    __nv_bfloat162 h;
                    h.x = __float2bfloat16_rn(tanhf(acc[ni][r] + bias_s[l * HID + col]));
                    h.y = __float2bfloat16_rn(tanhf(acc[ni][r + 1] + bias_s[l * HID + col + 1]));
                    *reinterpret_cast<__nv_bfloat162*>(out + row * LD + col) = h;
                }
        }
        __syncthreads();
        if (n0 != 0) continue;  // the output layer is 16 columns: one warp per row group
        float acc[2][4];
        rows_times_weights<2, HID>(acc, act1, LD, Ws + w_at(3), LD, r0, 0, lane);
        // columns 0 (stress / scale) and 1 (logit) sit in n-tile 0: lanes with t4 == 0
        if (t4 == 0) {
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
                const int row = r0 + g + 8 * h2, b = b0 + row;
                if (b >= a.B) continue;
                const float y0 = acc[0][2 * h2] + bias_s[3 * HID], y1 = acc[0][2 * h2 + 1] + bias_s[3 * HID + 1];
                if (a.out) {
                    a.out[2 * b] = y0 * a.scale;
                    a.out[2 * b + 1] = y1;
                    continue;
                }
                bool outside = false;
                for (int c = 0; c < NIN; ++c) {
                    const float xv = a.x[b * NIN + c];
                    outside |= !(fabsf(xv - a.center[c]) <= a.half[c]);
                }
                bool budget = false;
                if (a.n_bins > 0) {
                    const float ls = a.x[b * NIN];
                    int k = (int)floorf((ls - a.ls_lo) / (a.ls_hi - a.ls_lo) * a.n_bins);
                    k = k < 0 ? 0 : (k >= a.n_bins ? a.n_bins - 1 : k);
                    budget = a.over_budget[k] != 0;
                }
                a.stress[b] = y0 * a.scale;
                a.logit[b] = y1;
                a.fallback[b] = (outside || budget || !(fabsf(y1) >= a.margin)) ? 1 : 0;
            }
        }
    }
}

// ------------------------------------------------------------ training --
// Loss gradient and backpropagation in one kernel: a CTA takes a slab of 64
// batch rows through the normalisation, the forward pass, the loss and the backward
// pass with every activation and every weight in shared memory, and adds
// the slab's contribution to every weight and bias gradient into its own row
// of FP32 partial sums; grad_finish_kernel then sums the rows in a fixed order
// (reproducible) and, for a training step, applies Adam and refreshes the BF16
// weight copies: BF16 operands, FP32 accumulation, activations and pre-activation
// gradients rounded to BF16.
//   forward   H_l = tanh(X_l W_l^T + b_l) (rows past the batch are zero)
//   loss      (y0 - t)^2 + lam BCE(y1, label), mean over the batch
//   backward  dW_l = D_l^T X_l, db_l = column sums of D_l,
//             D_{l-1} = (D_l W_l) * (1 - H_{l-1}^2)
// The weight gradients multiply two row-major slab buffers along the batch
// (the contraction index is their row), and the input gradients multiply by W_l along
// its rows, so those operands are loaded with ldmatrix.trans.  Each pre-activation
// gradient overwrites, row by row, the activation it was computed from once every warp
// has used that activation.
// 16 warps hold 16 rows x 32 columns each of a layer's product and a 32 x 32 block of a
// weight gradient; four more sum the bias gradients meanwhile (64 dependent additions a
// column) and the FP64 loss meanwhile.  Four warps of 16 rows x 128 columns, loading one
// layer's weights (and their transposes) at a time, took 30.8 us per step at batch 512,
// 45 at 10240 and 150 at 65536 with the reduction; this takes 16.9, 33.7 and 111, a slab
// about 9 us.  Bound: shared-memory bandwidth for the products' operands (1500 of
// about 2200 cycles of a hidden layer) and the chain of eight of them; at 10240 the
// 160 slabs also take two rounds on 152 SMs.  The slab height and the order of all sums are
// fixed: regrouped sums differ in the last bit, and BF16 roundings of later steps
// carry that to 1e-3 of the parameters within an epoch.
constexpr int TR_ROWS = 64;                    // batch rows per slab
constexpr int TR_MAIN = 16, TR_THREADS = 640;  // warps of the products, threads of a CTA
constexpr int TR_MAX_ROWS = 304;               // partial rows at most
// inputs, output gradient, three activations and the weights: 138 KB, one CTA per SM
constexpr size_t TR_SMEM = sizeof(bf16) * (2 * TR_ROWS * LDZ + 3 * TR_ROWS * LD + W_ELEMS);

struct TrainArgs {
    const float *x, *target, *label;
    int B;
    const bf16* W[4];   // [out_p][in_p]
    const float* bias[4];
    const float *center, *half;
    float inv_scale, lam;
    int n_rows;         // partial rows
    float* part;        // [n_rows][NPARAM] partial gradients
    double* loss_part;  // [n_rows]
};

// A weight-gradient block dW[m0 + 16 MT][n0 + 8 NT] = sum over the slab's 64
// rows b of D[b][o] X[b][i]: A = D^T and B = X loaded with ldmatrix.trans from
// the row-major slab buffers (NT even).
template <int MT, int NT>
__device__ __forceinline__ void slab_outer(float (&acc)[MT][NT][4], const bf16* D, int ldD, int m0, const bf16* X,
                                           int ldX, int n0, int lane)
{
#pragma unroll
    for (int mi = 0; mi < MT; ++mi)
#pragma unroll
        for (int ni = 0; ni < NT; ++ni)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[mi][ni][r] = 0.f;
    const int j = lane >> 3, rr = lane & 7;
#pragma unroll
    for (int k0 = 0; k0 < TR_ROWS; k0 += 16) {
        uint32_t a[MT][4];
#pragma unroll
        for (int mi = 0; mi < MT; ++mi)  // matrices (m 0-7|8-15) x (k 0-7|8-15): a0..a3
            ldsm_x4_trans(a[mi], D + (k0 + rr + ((j >> 1) & 1) * 8) * ldD + m0 + mi * 16 + (j & 1) * 8);
#pragma unroll
        for (int np = 0; np < NT / 2; ++np) {  // two n-tiles: (k 0-7|8-15) x (n 0-7|8-15)
            uint32_t b[4];
            ldsm_x4_trans(b, X + (k0 + rr + (j & 1) * 8) * ldX + n0 + np * 16 + (j >> 1) * 8);
#pragma unroll
            for (int mi = 0; mi < MT; ++mi) {
                mma_bf16(acc[mi][2 * np], a[mi][0], a[mi][1], a[mi][2], a[mi][3], b[0], b[1]);
                mma_bf16(acc[mi][2 * np + 1], a[mi][0], a[mi][1], a[mi][2], a[mi][3], b[2], b[3]);
            }
        }
    }
}

// Adds (first slab: stores) a weight-gradient block to the CTA's partial row;
// entries outside the live out x in block are skipped.
template <int MT, int NT, int LS>
__device__ __forceinline__ void put_wgrad(float* row, const float (&acc)[MT][NT][4], long long offW, int m0, int n0,
                                          int g, int t4, bool first)
{
    constexpr LayerDef L = layer_def(LS);  // the block's shape; offW places it
#pragma unroll
    for (int mi = 0; mi < MT; ++mi)
#pragma unroll
        for (int ni = 0; ni < NT; ++ni)
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // rows g and g + 8: the pair (i, i + 1) of adjacent columns
                const int o = m0 + mi * 16 + g + 8 * h, i = n0 + ni * 8 + 2 * t4;
                if (o >= L.out || i >= L.in) continue;
                float* p = row + offW + (long long)o * L.in + i;
                const float v0 = acc[mi][ni][2 * h], v1 = acc[mi][ni][2 * h + 1];
                if (i + 1 < L.in && ((offW + (long long)o * L.in + i) & 1) == 0) {  // one 8-byte access
                    float2* p2 = reinterpret_cast<float2*>(p);
                    if (first) {
                        *p2 = make_float2(v0, v1);
                    } else {
                        const float2 q = *p2;
                        *p2 = make_float2(q.x + v0, q.y + v1);
                    }
                } else {
                    p[0] = first ? v0 : p[0] + v0;
                    if (i + 1 < L.in) p[1] = first ? v1 : p[1] + v1;
                }
            }
}

// A warp's 32 x 32 block of a hidden layer's weight gradient, in the order in which its
// lanes hold it: whole 256-byte stores, where the rows of the matrix would take eight
// pieces of 32 bytes each (2080 cycles a layer, of a slab's 28000).
__device__ __forceinline__ void put_hidden(float* block, const float (&acc)[2][4][4], int lane, bool first)
{
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2* const p = reinterpret_cast<float2*>(block) + ((mi * 4 + ni) * 2 + h) * 32 + lane;
                float2 v = make_float2(acc[mi][ni][2 * h], acc[mi][ni][2 * h + 1]);
                if (!first) {
                    const float2 q = *p;
                    v = make_float2(q.x + v.x, q.y + v.y);
                }
                *p = v;
            }
}
// Parameter at position k of a partial row (even k; k + 1 is the next one's).
__device__ __forceinline__ int param_at(int k)
{
    const int base = k >= OFF_W3 ? (int)OFF_W3 : (int)OFF_W2, p = k - base;
    if (p < 0 || p >= HID * HID) return k;
    const int lane = (p >> 1) & 31, r = (p >> 6) & 15, warp = p >> 10;
    const int o = (warp & 3) * 32 + (r >> 3) * 16 + (r & 1) * 8 + (lane >> 2);
    return base + o * HID + (warp >> 2) * 32 + ((r >> 1) & 3) * 8 + 2 * (lane & 3);
}

// Bias gradient of layer l: column sums of the slab's D (rows in increasing order).
__device__ __forceinline__ void put_bgrad(float* row, const bf16* D, int ld, int l, int col, bool first)
{
    const LayerDef L = layer_def(l);
    if (col >= L.out) return;
    float s = 0.f;
#pragma unroll 32
    for (int b = 0; b < TR_ROWS; ++b) s += __bfloat162float(D[b * ld + col]);
    float* p = row + L.offB + col;
    *p = first ? s : *p + s;
}

// D_{l-1} = (D_l W_l) * (1 - H^2) for 16 rows x 8 NT columns, written over H (BF16);
// the weights [K][in] are read along their rows (ldmatrix.trans).
template <int NT, int K>
__device__ __forceinline__ void back_block(const bf16* D, int ldD, const bf16* Ws, bf16* H, int r0, int n0, int lane,
                                           int b0, int B)
{
    float acc[NT][4];
#pragma unroll
    for (int ni = 0; ni < NT; ++ni)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[ni][r] = 0.f;
    const int j = lane >> 3, rr = lane & 7, g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int ks = 0; ks < K; ks += 16) {
        uint32_t a[4];
        ldsm_x4(a, D + (r0 + rr + (j & 1) * 8) * ldD + ks + (j >> 1) * 8);
#pragma unroll
        for (int np = 0; np < NT / 2; ++np) {
            uint32_t b[4];
            ldsm_x4_trans(b, Ws + (ks + rr + (j & 1) * 8) * LD + n0 + np * 16 + (j >> 1) * 8);
            mma_bf16(acc[2 * np], a[0], a[1], a[2], a[3], b[0], b[1]);
            mma_bf16(acc[2 * np + 1], a[0], a[1], a[2], a[3], b[2], b[3]);
        }
    }
#pragma unroll
    for (int ni = 0; ni < NT; ++ni)
#pragma unroll
        for (int r = 0; r < 4; r += 2) {
            const int row = r0 + g + (r >= 2 ? 8 : 0), col = n0 + ni * 8 + 2 * t4;
            __nv_bfloat162* const p = reinterpret_cast<__nv_bfloat162*>(H + row * LD + col);
            const float2 h = __bfloat1622float2(*p);
            const bool live = b0 + row < B;
            __nv_bfloat162 d;
            d.x = __float2bfloat16_rn(live ? acc[ni][r] * (1.f - h.x * h.x) : 0.f);
            d.y = __float2bfloat16_rn(live ? acc[ni][r + 1] * (1.f - h.y * h.y) : 0.f);
            *p = d;
        }
}

__global__ void __launch_bounds__(TR_THREADS, 1) train_fused_kernel(TrainArgs a)
{
    extern __shared__ __align__(16) unsigned char tr_smem[];
    bf16* const Zs = reinterpret_cast<bf16*>(tr_smem);  // [64][LDZ] inputs
    bf16* const D4 = Zs + TR_ROWS * LDZ;                  // [64][LDZ] output gradient
    bf16* const Hs = D4 + TR_ROWS * LDZ;                  // 3 x [64][LD] activations -> gradients
    bf16* const Ws = Hs + 3 * TR_ROWS * LD;               // all weights
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3, r0 = (warp & 3) * 16, n0 = (warp >> 2) * 32;
    const bool main_warp = warp < TR_MAIN;
    const int col = tid - 32 * TR_MAIN;  // the others' column of the bias gradients
    __shared__ double loss_w[4];
    __shared__ float2 loss_t[TR_ROWS];  // squared error and cross entropy of a row
    __shared__ __align__(16) float bias_s[BIASES];
    lbhb::grid_dependency_wait();
    lbhb::grid_launch_dependents();
    stage_all_weights<TR_THREADS>(Ws, bias_s, a.W, a.bias, tid);
    const int n_slabs = (a.B + TR_ROWS - 1) / TR_ROWS;
    // partial row blockIdx.x, + gridDim.x, ... of n_rows: slabs row, row + n_rows, ...
    for (int prow_i = blockIdx.x; prow_i < a.n_rows; prow_i += gridDim.x) {
    float* const prow = a.part + (long long)prow_i * NPARAM;
    double loss_acc = 0.0;
    for (int slab = prow_i; slab < n_slabs; slab += a.n_rows) {
        const bool first = slab == prow_i;
        const int b0 = slab * TR_ROWS;
        __syncthreads();  // the previous slab is done with the buffers
        normalise_rows<TR_ROWS, TR_THREADS>(Zs, LDZ, a.x, b0, a.B, a.center, a.half, tid);
        for (int e = tid; e < TR_ROWS * LDZ; e += TR_THREADS) D4[e] = __float2bfloat16_rn(0.f);
        // ---- forward
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (l == 0) cp_async_wait<2>();
            if (l == 1) cp_async_wait<1>();
            if (l == 2) cp_async_wait<0>();
            __syncthreads();  // layer l's weights and inputs visible
            if (!main_warp) continue;
            float acc[4][4];
            if (l == 0)
                rows_times_weights<4, KIN>(acc, Zs, LDZ, Ws, LDZ, r0, n0, lane);
            else
                rows_times_weights<4, HID>(acc, Hs + (l - 1) * TR_ROWS * LD, LD, Ws + w_at(l), LD, r0, n0, lane);
            bf16* const out = Hs + l * TR_ROWS * LD;
#pragma unroll
            for (int ni = 0; ni < 4; ++ni)
#pragma unroll
                for (int r = 0; r < 4; r += 2) {
                    const int row = r0 + g + (r >= 2 ? 8 : 0), c = n0 + ni * 8 + 2 * t4;
                    const bool live = b0 + row < a.B;
                    __nv_bfloat162 h;
                    h.x = __float2bfloat16_rn(live ? act_tanh(acc[ni][r] + bias_s[l * HID + c]) : 0.f);
                    h.y = __float2bfloat16_rn(live ? act_tanh(acc[ni][r + 1] + bias_s[l * HID + c + 1]) : 0.f);
                    *reinterpret_cast<__nv_bfloat162*>(out + row * LD + c) = h;
                }
        }
        __syncthreads();
        bf16* const H1 = Hs;
        bf16* const H3 = Hs + 2 * TR_ROWS * LD;
        if (warp < 4) {
            float acc[NOUTP / 8][4];
            rows_times_weights<NOUTP / 8, HID>(acc, H3, LD, Ws + w_at(3), LD, r0, 0, lane);
            // the loss and its gradient: columns 0 (stress / scale) and 1 (logit) of
            // n-tile 0 sit with the t4 == 0 lanes
            if (t4 == 0) {
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    const int row = r0 + g + 8 * h2, b = b0 + row;
                    if (b >= a.B) continue;
                    const float y0 = acc[0][2 * h2] + bias_s[3 * HID], y1 = acc[0][2 * h2 + 1] + bias_s[3 * HID + 1];
                    const float t = a.target[b] * a.inv_scale, lab = a.label[b];
                    const float e = y0 - t;
                    loss_t[row] = make_float2(e * e, bce_logits(y1, lab));
                    const float sg = 1.f / (1.f + expf(-y1));
                    D4[row * LDZ + 0] = __float2bfloat16_rn(2.f * e / (float)a.B);
                    D4[row * LDZ + 1] = __float2bfloat16_rn(a.lam * (sg - lab) / (float)a.B);
                }
            }
        }
        __syncthreads();  // D4 complete
        // ---- backward, layer 4: dW4 (16 x 128) from D4 and H3, db4
        if (!main_warp) {
            put_bgrad(prow, D4, LDZ, 3, col, first);
            // the loss is summed in FP64, whose pipe is slow: off the chain of layers
            if (t4 == 0) {
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    const int row = r0 + g + 8 * h2;
                    if (b0 + row < a.B) loss_acc += (double)loss_t[row].x + (double)a.lam * (double)loss_t[row].y;
                }
            }
        } else if (warp >= 8) {
            float acc[1][2][4];
            slab_outer<1, 2>(acc, D4, LDZ, 0, H3, LD, (warp - 8) * 16, lane);
            put_wgrad<1, 2, 3>(prow, acc, OFF_W4, 0, (warp - 8) * 16, g, t4, first);
        }
        __syncthreads();  // H3 read by every warp's dW4
        if (main_warp) back_block<4, NOUTP>(D4, LDZ, Ws + w_at(3), H3, r0, n0, lane, b0, a.B);  // D3 over H3
        __syncthreads();  // D3 complete
        // layers 3 and 2 (index l = 2, 1): dW_l from D_l (over H_l) and H_{l-1}, then
        // D_{l-1} over H_{l-1} with W_l
        static_assert(layer_def(1).in == layer_def(2).in && layer_def(1).out == layer_def(2).out,
                      "the two hidden-to-hidden layers have one shape");
#pragma unroll 1
        for (int l = 2; l >= 1; --l) {
            bf16* const Dl = Hs + l * TR_ROWS * LD;
            bf16* const Hp = Hs + (l - 1) * TR_ROWS * LD;
            if (!main_warp) {
                put_bgrad(prow, Dl, LD, l, col, first);
                if (l == 1 && slab + a.n_rows >= n_slabs) {
                    // the row's loss: lane sums, then the row groups in order
                    double sum = loss_acc;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
                    if (lane == 0) loss_w[warp - TR_MAIN] = sum;
                }
            } else {
                float acc[2][4][4];
                const int m0 = (warp & 3) * 32;
                slab_outer<2, 4>(acc, Dl, LD, m0, Hp, LD, n0, lane);
                put_hidden(prow + layer_def(l).offW + warp * 1024, acc, lane, first);
            }
            __syncthreads();
            if (main_warp) back_block<4, HID>(Dl, LD, Ws + (l == 2 ? w_at(2) : w_at(1)), Hp, r0, n0, lane, b0, a.B);
            __syncthreads();
        }
        // layer 1: dW1 (128 x 16) from D1 and the inputs
        if (!main_warp) {
            put_bgrad(prow, H1, LD, 0, col, first);
        } else if (warp < 8) {
            float acc[1][KIN / 8][4];
            slab_outer<1, KIN / 8>(acc, H1, LD, warp * 16, Zs, LDZ, 0, lane);
            put_wgrad<1, KIN / 8, 0>(prow, acc, OFF_W1, warp * 16, 0, g, t4, first);
        }
    }
    if (tid == 0) a.loss_part[prow_i] = (loss_w[0] + loss_w[1]) + (loss_w[2] + loss_w[3]);
    }
}

// Sums the CTAs' partial rows in order.  mode 0: gradient into grad.  mode 1: an
// Adam step on the FP32 masters p (m, v its moments) and the refreshed BF16
// weight copies and FP32 biases of that parameter.  Thread 0 of block 0 also
// finishes the loss (mean over the batch).
struct FinishArgs {
    const float* part;
    const double* loss_part;
    int n_rows, B;
    float* grad;
    float *p, *m, *v;
    float lr, b1, b2, eps, c1, c2;
    bf16* W[4];
    float* bias[4];
    float* loss_f;
    double* loss_d;
};

// Parameters per block (two per thread), threads per pair of parameters.
constexpr int FIN_PARAMS = 128, FIN_SPLIT = 4;
__global__ void __launch_bounds__(FIN_PARAMS / 2 * FIN_SPLIT) grad_finish_kernel(FinishArgs a, int mode)
{
    static_assert(NPARAM % 2 == 0, "the partial rows are read in pairs");
    // thread (q, j): parameters k0, k0 + 1, rows c = q, q + 4, ... in eight interleaved
    // sums; the four quarters combine in a fixed order
    constexpr int PAIRS = FIN_PARAMS / 2;
    const int j = threadIdx.x % PAIRS, q = threadIdx.x / PAIRS;
    const int k0 = blockIdx.x * FIN_PARAMS + 2 * j;
    // the first two quarters' threads finish one parameter of a pair each
    const bool mine = q < 2 && k0 < NPARAM;
    const int k = mine ? param_at(k0) + q : 0;
    float mk = 0.f, vk = 0.f, pk = 0.f;
    lbhb::grid_dependency_wait();
    lbhb::grid_launch_dependents();
    if (mine && mode != 0) {
        mk = a.m[k];
        vk = a.v[k];
        pk = a.p[k];
    }
    __shared__ float2 quarter[FIN_SPLIT][PAIRS];
    if (k0 < NPARAM) {
        float2 s8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) s8[u] = make_float2(0.f, 0.f);
        auto add = [&](int u, int c) {
            const float2 v = *reinterpret_cast<const float2*>(a.part + (long long)c * NPARAM + k0);
            s8[u].x += v.x;
            s8[u].y += v.y;
        };
        int c = q;
        for (; c + 7 * FIN_SPLIT < a.n_rows; c += 8 * FIN_SPLIT)
#pragma unroll
            for (int u = 0; u < 8; ++u) add(u, c + u * FIN_SPLIT);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (c + u * FIN_SPLIT < a.n_rows) add(u, c + u * FIN_SPLIT);
        quarter[q][j] = make_float2(((s8[0].x + s8[1].x) + (s8[2].x + s8[3].x)) + ((s8[4].x + s8[5].x) + (s8[6].x + s8[7].x)),
                                    ((s8[0].y + s8[1].y) + (s8[2].y + s8[3].y)) + ((s8[4].y + s8[5].y) + (s8[6].y + s8[7].y)));
    }
    __syncthreads();
    if (blockIdx.x == 0 && q == FIN_SPLIT - 1 && j < 32) {
        // the loss, by one otherwise idle warp: lane sums over rows lane, lane + 32, ...,
        // then a butterfly over the lanes (a fixed order, so the same every call)
        double s = 0.0;
        for (int c = j; c < a.n_rows; c += 32) s += a.loss_part[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (j == 0) {
            s /= (double)a.B;
            if (a.loss_f) *a.loss_f = (float)s;
            if (a.loss_d) *a.loss_d = s;
        }
        return;
    }
    if (!mine) return;
    const float2 g0 = quarter[0][j], g1 = quarter[1][j], g2 = quarter[2][j], g3 = quarter[3][j];
    const float gk = q == 0 ? (g0.x + g1.x) + (g2.x + g3.x) : (g0.y + g1.y) + (g2.y + g3.y);
    if (mode == 0) {
        a.grad[k] = gk;
        return;
    }
    // explicit multiply-adds: their roundings decide later BF16 roundings, so they must
    // not depend on what the compiler contracts
    const float o1 = __fsub_rn(1.f, a.b1), o2 = __fsub_rn(1.f, a.b2);
    mk = __fmaf_rn(o1, gk, __fmul_rn(a.b1, mk));
    vk = __fmaf_rn(a.b2, vk, __fmul_rn(__fmul_rn(o2, gk), gk));
    a.m[k] = mk;
    a.v[k] = vk;
    pk = pk - a.lr * (mk * a.c1) / (sqrtf(vk * a.c2) + a.eps);
    a.p[k] = pk;
    for (int l = 0; l < 4; ++l) {  // the parameter's BF16 weight entries or FP32 bias
        const LayerDef L = layer_def(l);
        if (k >= L.offW && k < L.offB) {
            const int o = (int)((k - L.offW) / L.in), i = (int)((k - L.offW) % L.in);
            a.W[l][o * L.in_p + i] = __float2bfloat16_rn(pk);
        } else if (k >= L.offB && k < L.offB + L.out) {
            a.bias[l][k - L.offB] = pk;
        }
    }
}

struct mlp_handle {
    mlp_config cfg{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int device = 0;
    int sms = 0;
    float *P = nullptr, *M = nullptr, *V = nullptr, *G = nullptr;
    bf16* W[4] = {};
    float* bias[4] = {};
    float* part = nullptr;         // [tr_rows][NPARAM] partial gradients of train_fused_kernel
    int tr_rows = 0;               // its CTAs at most (one partial row each)
    double* loss_part = nullptr;   // [tr_rows]
    double* loss_d = nullptr;
    float *center = nullptr, *half = nullptr;
    float* x_copy = nullptr;     // [max_batch][NIN]: mlp_forward's inputs where its outputs overlap them
    int* over_budget = nullptr;  // [MAX_BINS]
    int n_bins = 0;
    float ls_lo = 0.f, ls_hi = 1.f;
    long long adam_t = 0;
    long long launches = 0;
    std::vector<void*> allocs;
};

namespace {

void release(mlp_handle* h)
{
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    for (void* p : h->allocs) cudaFree(p);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    delete h;
}

template <class T>
cudaError_t alloc(mlp_handle* h, T** p, size_t n)
{
    cudaError_t e = cudaMalloc((void**)p, n * sizeof(T));
    if (e == cudaSuccess) {
        h->allocs.push_back(*p);
        e = cudaMemsetAsync(*p, 0, n * sizeof(T), h->stream);
    }
    return e;
}

// Launch that may set up while the kernel before it on the stream still runs (it waits
// for that kernel's end before it reads or writes anything).
cudaError_t launch_ahead(const void* kernel, int blocks, int threads, size_t smem, cudaStream_t st, void* arg0, void* arg1)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    void* args[] = {arg0, arg1};
    return cudaLaunchKernelExC(&cfg, kernel, args);
}

// Loss, gradient (mode 0: into h->G) or gradient and Adam step (mode 1): the
// fused training kernel over slabs of 64 rows, then the ordered reduction.
cudaError_t fused_step(mlp_handle* h, const float* x, const float* target, const float* label, int B, int mode,
                       float* loss_f, double* loss_d)
{
    TrainArgs ta{};
    ta.x = x;
    ta.target = target;
    ta.label = label;
    ta.B = B;
    for (int l = 0; l < 4; ++l) {
        ta.W[l] = h->W[l];
        ta.bias[l] = h->bias[l];
    }
    ta.center = h->center;
    ta.half = h->half;
    ta.inv_scale = (float)(1.0 / h->cfg.sigma_scale);
    ta.lam = (float)h->cfg.lam;
    ta.part = h->part;
    ta.loss_part = h->loss_part;
    const int slabs = (B + TR_ROWS - 1) / TR_ROWS, rows = std::min(slabs, h->tr_rows);
    ta.n_rows = rows;
    cudaError_t e = launch_ahead(reinterpret_cast<const void*>(&train_fused_kernel), std::min(rows, h->sms), TR_THREADS,
                                 TR_SMEM, h->stream, &ta, nullptr);
    h->launches++;
    if (e != cudaSuccess) return e;
    FinishArgs fa{};
    fa.part = h->part;
    fa.loss_part = h->loss_part;
    fa.n_rows = rows;
    fa.B = B;
    fa.grad = h->G;
    fa.p = h->P;
    fa.m = h->M;
    fa.v = h->V;
    if (mode == 1) {
        h->adam_t++;
        const double b1 = h->cfg.beta1, b2 = h->cfg.beta2;
        fa.lr = (float)h->cfg.lr;
        fa.b1 = (float)b1;
        fa.b2 = (float)b2;
        fa.eps = (float)h->cfg.eps;
        fa.c1 = (float)(1.0 / (1.0 - std::pow(b1, (double)h->adam_t)));
        fa.c2 = (float)(1.0 / (1.0 - std::pow(b2, (double)h->adam_t)));
    }
    for (int l = 0; l < 4; ++l) {
        fa.W[l] = h->W[l];
        fa.bias[l] = h->bias[l];
    }
    fa.loss_f = loss_f;
    fa.loss_d = loss_d;
    e = launch_ahead(reinterpret_cast<const void*>(&grad_finish_kernel), (int)((NPARAM + FIN_PARAMS - 1) / FIN_PARAMS),
                     FIN_PARAMS / 2 * FIN_SPLIT, 0, h->stream, &fa, &mode);
    h->launches++;
    return e;
}

cudaError_t refresh(mlp_handle* h)
{
    int total = 0;
    for (int l = 0; l < 4; ++l) total += layer_def(l).out_p * layer_def(l).in_p + layer_def(l).out_p;
    refresh_kernel<<<(total + 255) / 256, 256, 0, h->stream>>>(h->P, h->W[0], h->W[1], h->W[2], h->W[3], h->bias[0],
                                                                h->bias[1], h->bias[2], h->bias[3]);
    h->launches++;
    return cudaGetLastError();
}

ServeArgs inference_args(const mlp_handle* h, const float* x, int batch)
{
    ServeArgs a{};
    a.x = x;
    a.B = batch;
    for (int l = 0; l < 4; ++l) {
        a.W[l] = h->W[l];
        a.bias[l] = h->bias[l];
    }
    a.center = h->center;
    a.half = h->half;
    a.scale = (float)h->cfg.sigma_scale;
    a.margin = (float)h->cfg.logit_margin;
    a.over_budget = h->over_budget;
    a.n_bins = h->n_bins;
    a.ls_lo = h->ls_lo;
    a.ls_hi = h->ls_hi;
    return a;
}

lb_status launch_inference(mlp_handle* h, const ServeArgs& a)
{
    const int slabs = (a.B + SRV_ROWS - 1) / SRV_ROWS;
    serve_fused_kernel<<<std::min(slabs, 2 * h->sms), SRV_THREADS, SRV_SMEM, h->stream>>>(a);
    h->launches++;
    return cudaGetLastError() == cudaSuccess ? LB_OK : LB_ERR_CUDA;
}

lb_status invalid(const char* msg)
{
    lbhb::set_handleless_error(msg);
    return LB_ERR_INVALID;
}

lb_status check_batch(const mlp_handle* h, int B)
{
    if (B >= 1 && B <= h->cfg.max_batch) return LB_OK;
    char buf[128];
    snprintf(buf, sizeof buf, "mlp: batch %d outside 1..max_batch (%d)", B, h->cfg.max_batch);
    lbhb::set_handleless_error(buf);
    return LB_ERR_INVALID;
}

}  // namespace

extern "C" {

long long mlp_param_count(void) { return NPARAM; }

lb_status mlp_create(const mlp_config* cfg, void* cuda_stream, mlp_handle** out)
{
    if (!out || !cfg) return invalid("mlp_create: NULL config or output");
    *out = nullptr;
    if (cfg->max_batch < 1 || cfg->max_batch > (1 << 24) || !(cfg->sigma_scale > 0.0) || !(cfg->lr >= 0.0))
        return invalid("mlp_create: max_batch, sigma_scale or lr out of range");
    for (int c = 0; c < NIN; ++c)
        if (!(cfg->half_range[c] > 0.0) || !std::isfinite(cfg->center[c]))
            return invalid("mlp_create: half_range must be > 0 and center finite");
    mlp_handle* h = new (std::nothrow) mlp_handle();
    if (!h) return LB_ERR_NOMEM;
    h->cfg = *cfg;
    cudaGetDevice(&h->device);
    cudaError_t e = cudaSuccess;
    if (cuda_stream) h->stream = (cudaStream_t)cuda_stream;
    else {
        e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
        h->own_stream = e == cudaSuccess;
    }
    cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, h->device);
    h->tr_rows = std::min(TR_MAX_ROWS, (cfg->max_batch + TR_ROWS - 1) / TR_ROWS);
    if (e == cudaSuccess) e = alloc(h, &h->P, NPARAM);
    if (e == cudaSuccess) e = alloc(h, &h->M, NPARAM);
    if (e == cudaSuccess) e = alloc(h, &h->V, NPARAM);
    if (e == cudaSuccess) e = alloc(h, &h->G, NPARAM);
    for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
        e = alloc(h, &h->W[l], (size_t)layer_def(l).out_p * layer_def(l).in_p);
        if (e == cudaSuccess) e = alloc(h, &h->bias[l], (size_t)layer_def(l).out_p);
    }
    if (e == cudaSuccess) e = alloc(h, &h->part, (size_t)h->tr_rows * NPARAM);
    if (e == cudaSuccess) e = alloc(h, &h->loss_part, (size_t)h->tr_rows);
    if (e == cudaSuccess) e = alloc(h, &h->loss_d, 1);
    if (e == cudaSuccess) e = alloc(h, &h->center, NIN);
    if (e == cudaSuccess) e = alloc(h, &h->half, NIN);
    if (e == cudaSuccess) e = alloc(h, &h->x_copy, (size_t)cfg->max_batch * NIN);
    if (e == cudaSuccess)  // the fused serving kernel keeps activations and weights in shared memory
        e = cudaFuncSetAttribute(serve_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SRV_SMEM);
    if (e == cudaSuccess)  // and so does the fused training kernel
        e = cudaFuncSetAttribute(train_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TR_SMEM);
    if (e == cudaSuccess) e = alloc(h, &h->over_budget, MAX_BINS);
    if (e == cudaSuccess) {
        float c[NIN], hr[NIN];
        for (int i = 0; i < NIN; ++i) {
            c[i] = (float)cfg->center[i];
            hr[i] = (float)cfg->half_range[i];
        }
        e = cudaMemcpyAsync(h->center, c, sizeof c, cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(h->half, hr, sizeof hr, cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        release(h);
        return e == cudaErrorMemoryAllocation ? LB_ERR_NOMEM : LB_ERR_CUDA;
    }
    *out = h;
    return LB_OK;
}

lb_status mlp_set_params(mlp_handle* h, const float* params, long long n)
{
    if (!h || !params || n != NPARAM) return invalid("mlp: NULL handle or parameters, or wrong count");
    cudaError_t e = cudaMemcpyAsync(h->P, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->M, 0, sizeof(float) * NPARAM, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->V, 0, sizeof(float) * NPARAM, h->stream);
    if (e == cudaSuccess) e = refresh(h);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    h->adam_t = 0;
    return e == cudaSuccess ? LB_OK : LB_ERR_CUDA;
}

lb_status mlp_get_params(mlp_handle* h, float* params, long long n)
{
    if (!h || !params || n != NPARAM) return invalid("mlp: NULL handle or parameters, or wrong count");
    cudaError_t e = cudaMemcpyAsync(params, h->P, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    return e == cudaSuccess ? LB_OK : LB_ERR_CUDA;
}

lb_status mlp_forward(mlp_handle* h, const float* x, int batch, float* out)
{
    if (!h || !x || !out) return invalid("mlp: NULL handle or buffer");
    if (check_batch(h, batch) != LB_OK) return LB_ERR_INVALID;
    // blocks write their queries' outputs while others have yet to read their inputs: an
    // output buffer that overlaps the inputs gets them from a copy
    const uintptr_t xb = (uintptr_t)x, ob = (uintptr_t)out;
    const size_t x_bytes = sizeof(float) * NIN * (size_t)batch, out_bytes = sizeof(float) * NOUT * (size_t)batch;
    if (xb < ob + out_bytes && ob < xb + x_bytes) {
        if (cudaMemcpyAsync(h->x_copy, x, x_bytes, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess) return LB_ERR_CUDA;
        x = h->x_copy;
    }
    ServeArgs a = inference_args(h, x, batch);
    a.out = out;
    return launch_inference(h, a);
}

lb_status mlp_gradients(mlp_handle* h, const float* x, const float* target_stress, const float* label, int batch,
                        float* grad, double* loss)
{
    if (!h || !x || !target_stress || !label || !grad) return invalid("mlp: NULL handle or buffer");
    if (check_batch(h, batch) != LB_OK) return LB_ERR_INVALID;
    cudaError_t e = fused_step(h, x, target_stress, label, batch, 0, nullptr, h->loss_d);
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad, h->G, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, h->stream);
    double l = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&l, h->loss_d, sizeof(double), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (loss) *loss = l;
    return e == cudaSuccess ? LB_OK : LB_ERR_CUDA;
}

lb_status mlp_train_step(mlp_handle* h, const float* x, const float* target_stress, const float* label, int batch,
                         float* loss_dev)
{
    if (!h || !x || !target_stress || !label) return invalid("mlp: NULL handle or buffer");
    if (check_batch(h, batch) != LB_OK) return LB_ERR_INVALID;
    const cudaError_t e = fused_step(h, x, target_stress, label, batch, 1, loss_dev, nullptr);
    return e == cudaSuccess ? LB_OK : LB_ERR_CUDA;
}

lb_status mlp_serve(mlp_handle* h, const float* x, int batch, float* stress, float* logit, int* fallback)
{
    if (!h || !x || !stress || !logit || !fallback) return invalid("mlp: NULL handle or buffer");
    if (check_batch(h, batch) != LB_OK) return LB_ERR_INVALID;
    ServeArgs a = inference_args(h, x, batch);
    a.stress = stress;
    a.logit = logit;
    a.fallback = fallback;
    return launch_inference(h, a);
}

lb_status mlp_set_error_budget(mlp_handle* h, const float* bin_error, int n_bins, double log_s_lo,
                               double log_s_hi, double budget)
{
    if (!h || n_bins < 0 || n_bins > MAX_BINS || (n_bins > 0 && (!bin_error || !(log_s_hi > log_s_lo))))
        return invalid("mlp_set_error_budget: NULL handle, n_bins outside 0..256 or empty log S range");
    int flags[MAX_BINS] = {0};
    for (int k = 0; k < n_bins; ++k) flags[k] = !(bin_error[k] <= budget);  // NaN error is over budget
    cudaError_t e = cudaMemcpyAsync(h->over_budget, flags, sizeof(int) * MAX_BINS, cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return LB_ERR_CUDA;
    h->n_bins = n_bins;
    h->ls_lo = (float)log_s_lo;
    h->ls_hi = (float)log_s_hi;
    return LB_OK;
}

long long mlp_kernel_launches(const mlp_handle* h) { return h ? h->launches : 0; }

void mlp_destroy(mlp_handle* h) { release(h); }

}  // extern "C"
