// gnn.cu -- learned edge preconditioner of the Newmark solve: inference,
// training (forward, backward, Adam) and the flexible PCG that uses it.
//
// The paper has no learned component; the CG step of its Newmark update
// (Sec. III) is where this library plugs one in.  The network, on the graph of
// the interior-edge system A (nodes = DOFs, edges = nonzeros of A):
//
//   d = diag(A), Ahat = D^-1/2 A D^-1/2, a_i = log d_i - mean(log d)
//   rho = sqrt(mean_i r_i^2 / d_i), x_i = r_i / (sqrt(d_i) rho)
//   h0_i = relu(U x_i + V a_i + c)                                   (32 wide)
//   g_l = Ahat h_{l-1},  h_l,i = relu(W_l h_{l-1,i} + Q_l g_l,i + b_l), l = 1..3
//   y_i = o . h_3,i + d0
//   z_i = r_i / d_i + rho y_i / sqrt(d_i)        (Jacobi when y = 0)
//
// Weights are kept as FP32 master values and used as their bfloat16
// roundings; activations and accumulations are FP32, the Jacobi part and
// everything the solver sums are FP64.  Training minimises, over residuals
// taken from Jacobi-PCG solves of the same system,
//   L = (z^T A z - 2 z^T r) / (r^T D^-1 r),
// the A-norm error of z against A^-1 r up to a constant (no solve needed).
//
// Layout: activations row-major (32 floats = 128 B per row), rows in an order
// of their own (by row length, then canonical edge).  Both passes work on tiles
// of rows in shared memory and gather four whole feature rows an instruction.
// Training keeps FP32 multiply-adds and one summation order; a preconditioner
// application runs its layers on the tensor cores (k_layer_tc: TF32 products of split
// activations).  Every reduction (weight gradients, rho, the loss, the PCG dot
// products) uses per-block partials combined in a fixed order: results do not
// depend on scheduling.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "sim.h"

namespace fp {
namespace {

constexpr int kH = 32;
constexpr int kT = 256;                 // threads per block
constexpr int kW = kT / 32;             // warps per block
constexpr int kGB = 456;                // blocks of the row kernels whose FP32 sums go by block (3 per SM)
constexpr int kRowBlocks = 152 * 6;     // most blocks of the others: all rows at once on small meshes
constexpr int kLayer = 2 * kH * kH + kH;
constexpr int kOffU = 0, kOffV = kH, kOffC = 2 * kH, kOffL = 3 * kH;
constexpr int kOffO = kOffL + 3 * kLayer, kOffD0 = kOffO + kH;
constexpr int kNA = 2 * kH + 3;         // per-lane accumulators of a layer's backward
static_assert(kOffD0 + 1 == kGnnParams, "parameter layout");

__device__ __forceinline__ float bf(const unsigned short *t, int i) {
    return __bfloat162float(__ushort_as_bfloat16(t[i]));
}

// ---- deterministic sums: per-block partials, then one block in fixed order ----
template <int N>
__device__ __forceinline__ void block_partial(double v[N], double *part) {
    __shared__ double sh[N][kW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < N; c++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xFFFFFFFFu, v[c], o);
        if (lane == 0) sh[c][warp] = v[c];
    }
    __syncthreads();
    if (threadIdx.x < N) {
        double s = 0.0;
        for (int w = 0; w < kW; w++) s += sh[threadIdx.x][w];
        part[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = s;
    }
}

__global__ void k_final_sums(int nb, int nv, const double *__restrict__ part, double *__restrict__ out) {
    // one warp per value: lanes add blocks lane, lane+32, ... then a shuffle tree
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    if (c >= nv) return;
    double s = 0.0;
    for (int b = lane; b < nb; b += 32) s += part[(size_t)c * nb + b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
    if (lane == 0) out[c] = s;
}

// the sum of nb partials, by one warp in the order of k_final_sums, handed to
// the whole block
__device__ __forceinline__ double block_total(int nb, const double *__restrict__ part) {
    __shared__ double total;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int b = threadIdx.x; b < nb; b += 32) s += part[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
        if (threadIdx.x == 0) total = s;
    }
    __syncthreads();
    return total;
}

// sum_i (x1_i y1_i), sum_i (x2_i y2_i) (x2 may be NULL), scaled by w_i when w != NULL
__global__ void __launch_bounds__(kT) k_dot2(int n, const double *__restrict__ x1, const double *__restrict__ y1,
                                            const double *__restrict__ x2, const double *__restrict__ y2,
                                            const double *__restrict__ w, double *part) {
    double v[2] = {0.0, 0.0};
    for (int i = blockIdx.x * kT + threadIdx.x; i < n; i += gridDim.x * kT) {
        const double s = w ? w[i] : 1.0;
        v[0] = fma(x1[i] * s, y1[i], v[0]);
        if (x2) v[1] = fma(x2[i] * s, y2[i], v[1]);
    }
    block_partial<2>(v, part);
}

// ---- static inputs: Ahat (SELL layout, FP32), 1/sqrt(d), log d ----
__global__ void k_prep_rows(int n, const int *__restrict__ edge, const double *__restrict__ Dinv,
                            double *__restrict__ isd, double *__restrict__ logd) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        isd[i] = sqrt(Dinv[edge[i]]);
        logd[i] = -log(Dinv[edge[i]]);
    }
}

// the columns of the network's rows: the rows of the edges that share a tet,
// in increasing order (insertion in place), then the row itself
__global__ void k_rows_cols(int n, int nsl, const int *__restrict__ sp, const int *__restrict__ sw,
                            const int *__restrict__ canon, const int *__restrict__ tptr, const int *__restrict__ tref,
                            const int *__restrict__ tet_edge, const int *__restrict__ row, int *__restrict__ col) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 32 * nsl) return;
    int *c = col + sp[i >> 5] + (i & 31);
    const int w = sw[i >> 5];
    int m = 0;
    if (i < n)
        for (int a = tptr[canon[i]]; a < tptr[canon[i] + 1]; a++)
            for (int k = 0; k < 6; k++) {
                const int e = tet_edge[6 * (size_t)(tref[a] / 6) + k];
                if (e >= n) continue;
                const int x = row[e];
                int j = m;
                while (j > 0 && c[32 * (j - 1)] > x) j--;
                if ((j > 0 && c[32 * (j - 1)] == x) || m >= w) continue;
                for (int q = m++; q > j; q--) c[32 * q] = c[32 * (q - 1)];
                c[32 * j] = x;
            }
    for (; m < w; m++) c[32 * m] = min(i, n - 1);
}

// (element values are looked up in A's rows, whose padding has the value 0)
__global__ void k_prep_ahat(int n, int nsl, const int *__restrict__ sp, const int *__restrict__ sw,
                            const int *__restrict__ col, const int *__restrict__ edge, const int *__restrict__ asp,
                            const int *__restrict__ asw, const int *__restrict__ acol, const double *__restrict__ val,
                            const double *__restrict__ isd, const double *__restrict__ logd,
                            const double *__restrict__ mean_logd, float *__restrict__ ahat,
                            float *__restrict__ feat_a) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int sl = t >> 5, lane = t & 31;
    if (sl >= nsl) return;
    const int i = sl * 32 + lane, kb = sp[sl] + lane, kw = sw[sl];
    const double si = i < n ? isd[i] : 0.0;
    const int e = i < n ? edge[i] : 0, ab = asp[e >> 5] + (e & 31), aw = asw[e >> 5];
    int last = -1;   // columns increase along a row; padding repeats the row itself
    for (int j = 0; j < kw; j++) {
        const int k = kb + 32 * j, c = col[k];
        double v = 0.0;
        if (i < n && c > last) {
            const int ce = edge[c];
            for (int q = 0; q < aw; q++)
                if (acol[ab + 32 * q] == ce) v += val[ab + 32 * q];
            last = c;
        }
        ahat[k] = i < n ? (float)(v * si * isd[c]) : 0.0f;
    }
    if (i < n) feat_a[i] = (float)(logd[i] - mean_logd[0] / n);
}

__global__ void k_sum(int n, const double *__restrict__ a, double *part) {
    double v[1] = {0.0};
    for (int i = blockIdx.x * kT + threadIdx.x; i < n; i += gridDim.x * kT) v[0] += a[i];
    block_partial<1>(v, part);
}

// rho^2 n = sum r_i^2 / d_i
__global__ void __launch_bounds__(kT) k_rnorm(int n, const int *__restrict__ edge, const double *__restrict__ r,
                                             const double *__restrict__ Dinv, double *part) {
    double v[1] = {0.0};
    for (int i = blockIdx.x * kT + threadIdx.x; i < n; i += gridDim.x * kT) {
        const double re = r[edge[i]];
        v[0] = fma(re * Dinv[edge[i]], re, v[0]);
    }
    block_partial<1>(v, part);
}

__device__ __forceinline__ double rho_of(const double *nrm, int n) { return sqrt(nrm[0] / n); }
// (by one thread of the block: division and root in every warp of it hold the
// FP64 pipes for longer than a small kernel's own work)
__device__ __forceinline__ double block_rho(const double *nrm, int n) {
    __shared__ double rho;
    if (threadIdx.x == 0) rho = rho_of(nrm, n);
    __syncthreads();
    return rho;
}

// ---- forward ----
// The warp's 32 rows are scaled a lane each and the features formed row by row:
// a lane per feature that scales its row itself repeats the row's FP64
// division 32 times (136 -> 15 us at 220,256 rows).  nrm_part: the partials
// of n rho^2; block 0 leaves their sum in nrm.
template <bool KEEP>
__global__ void __launch_bounds__(kT) k_embed(int n, const int *__restrict__ edge, const double *__restrict__ r,
                                             const double *__restrict__ isd,
                                             int n_part, const double *__restrict__ nrm_part, double *__restrict__ nrm,
                                             const float *__restrict__ feat_a,
                                             const unsigned short *__restrict__ th, float *__restrict__ xin,
                                             float *__restrict__ pre0, float *__restrict__ h0) {
    __shared__ double s_rho;
    const int lane = threadIdx.x & 31;
    const double total = block_total(n_part, nrm_part);
    if (threadIdx.x == 0) {
        s_rho = sqrt(total / n);
        if (blockIdx.x == 0) nrm[0] = total;
    }
    __syncthreads();
    const double rho = s_rho;
    const float U = bf(th, kOffU + lane), V = bf(th, kOffV + lane), c = bf(th, kOffC + lane);
    for (int base = (blockIdx.x * kW + (threadIdx.x >> 5)) * 32; base < n; base += gridDim.x * kT) {
        const int i = base + lane, m = min(32, n - base);
        float x = 0.0f, fa = 0.0f;
        if (lane < m) {
            x = rho > 0.0 ? (float)(r[edge[i]] * isd[i] / rho) : 0.0f;
            fa = feat_a[i];
            if (KEEP) xin[i] = x;
        }
#pragma unroll 4
        for (int k = 0; k < m; k++) {
            const float p = fmaf(U, __shfl_sync(0xFFFFFFFFu, x, k), fmaf(V, __shfl_sync(0xFFFFFFFFu, fa, k), c));
            if (KEEP) pre0[(size_t)(base + k) * kH + lane] = p;
            h0[(size_t)(base + k) * kH + lane] = fmaxf(p, 0.0f);
        }
    }
}

constexpr int kTileRows = 16;
constexpr int kSRow = 2 * kH + 4;       // padded row of S: conflict-free fragment loads

__device__ __forceinline__ void load4(const float *p, float v[4]) {
    const float4 x = *reinterpret_cast<const float4 *>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
}

__device__ __forceinline__ void fma4(float4 &acc, float a, float4 v) {
    acc.x = fmaf(a, v.x, acc.x);
    acc.y = fmaf(a, v.y, acc.y);
    acc.z = fmaf(a, v.z, acc.z);
    acc.w = fmaf(a, v.w, acc.w);
}

// acc[p] += sum_j Ahat_ij v_j for the rows i = 16 tile + rs + 4p (rs = lane >> 3)
// and their features 4 (lane & 7) .. + 3, entries in increasing order: each
// 16-byte gather of the warp reads four whole 128-byte feature rows, and a
// row's column and weight are read by the eight lanes that use them.  SELL padding
// has weight 0 and names an existing row.
__device__ __forceinline__ void aggregate_tile(int tile, const int *__restrict__ sp, const int *__restrict__ sw,
                                               const int *__restrict__ col, const float *__restrict__ ahat,
                                               const float *__restrict__ v, float4 acc[4]) {
    const int lane = threadIdx.x & 31, rs = lane >> 3, q8 = lane & 7;
    const int sl = tile >> 1, kb0 = sp[sl] + (tile & 1) * kTileRows, kw = sw[sl];
#pragma unroll 2
    for (int j = 0; j < kw; j++) {
        int c[4];
        float a[4];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int e = kb0 + rs + 4 * p + 32 * j;
            c[p] = col[e];
            a[p] = ahat[e];
        }
#pragma unroll
        for (int p = 0; p < 4; p++)
            fma4(acc[p], a[p], __ldg(reinterpret_cast<const float4 *>(v + (size_t)c[p] * kH + 4 * q8)));
    }
}

// one message-passing layer of the training forward pass; the last one also
// forms z.  It stores the aggregates and pre-activations the backward pass
// reads (a preconditioner application uses k_layer_tc below instead).  FP32
// throughout, each sum in one fixed order.  A warp takes 16 consecutive
// rows: the tile's h and g go to shared memory and each lane forms 4 features
// of 4 rows, so that 16 words read from shared memory serve 32 multiply-adds
// (the words that come back from shared memory or by shuffles bound it: 152 a
// row with a warp per row, 244 us at 220,256 rows; 68 with a feature a lane,
// 86 us; 32 now, 77 us).
template <bool LAST>
__global__ void __launch_bounds__(kT) k_layer(int n, const int *__restrict__ sp, const int *__restrict__ sw,
                                             const int *__restrict__ col, const float *__restrict__ ahat,
                                             const float *__restrict__ hp, const unsigned short *__restrict__ th,
                                             int off, float *__restrict__ g, float *__restrict__ pre,
                                             float *__restrict__ h, const int *__restrict__ edge,
                                             const double *__restrict__ r, const double *__restrict__ Dinv,
                                             const double *__restrict__ isd, const double *__restrict__ nrm,
                                             double *__restrict__ z) {
    extern __shared__ __align__(16) float layer_sh[];
    float *Wt = layer_sh, *Qt = Wt + kH * kH;
    float *S = Qt + kH * kH + (threadIdx.x >> 5) * kTileRows * kSRow;
    for (int t = threadIdx.x; t < kH * kH; t += kT) {
        const int f = t >> 5, k = t & 31;   // W[f][k] -> Wt[k][f]
        Wt[k * kH + f] = bf(th, off + t);
        Qt[k * kH + f] = bf(th, off + kH * kH + t);
    }
    const double rho = LAST ? block_rho(nrm, n) : 0.0;
    __syncthreads();
    const int lane = threadIdx.x & 31, rs = lane >> 3, q8 = lane & 7;
    float b[4], o[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
        b[u] = bf(th, off + 2 * kH * kH + 4 * q8 + u);
        o[u] = LAST ? bf(th, kOffO + 4 * q8 + u) : 0.0f;
    }
    const float d0 = LAST ? bf(th, kOffD0) : 0.0f;
    const int ntiles = (n + kTileRows - 1) / kTileRows;
    for (int tile = blockIdx.x * kW + (threadIdx.x >> 5); tile < ntiles; tile += gridDim.x * kW) {
        const int row0 = tile * kTileRows;
        float4 acc[4];
#pragma unroll
        for (int p = 0; p < 4; p++) acc[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        aggregate_tile(tile, sp, sw, col, ahat, hp, acc);
        __syncwarp();   // the previous tile has been read
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int i = row0 + rs + 4 * p;
            float *srow = S + (rs + 4 * p) * kSRow + 4 * q8;
            float4 hv = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (i < n) {
                hv = __ldg(reinterpret_cast<const float4 *>(hp + (size_t)i * kH + 4 * q8));
                *reinterpret_cast<float4 *>(g + (size_t)i * kH + 4 * q8) = acc[p];
            }
            *reinterpret_cast<float4 *>(srow) = hv;
            *reinterpret_cast<float4 *>(srow + kH) = acc[p];
        }
        __syncwarp();
        // rows rs + 4p, features 4 q8 + u
        float v[4][4];
#pragma unroll
        for (int p = 0; p < 4; p++)
#pragma unroll
            for (int u = 0; u < 4; u++) v[p][u] = b[u];
#pragma unroll 2
        for (int k = 0; k < kH; k += 4) {
            float hk[4][4], gk[4][4];
#pragma unroll
            for (int p = 0; p < 4; p++) {
                load4(S + (rs + 4 * p) * kSRow + k, hk[p]);
                load4(S + (rs + 4 * p) * kSRow + kH + k, gk[p]);
            }
#pragma unroll
            for (int t = 0; t < 4; t++) {
                float w[4], q[4];
                load4(Wt + (k + t) * kH + 4 * q8, w);
                load4(Qt + (k + t) * kH + 4 * q8, q);
#pragma unroll
                for (int p = 0; p < 4; p++)
#pragma unroll
                    for (int u = 0; u < 4; u++) v[p][u] = fmaf(q[u], gk[p][t], fmaf(w[u], hk[p][t], v[p][u]));
            }
        }
        float yrow = 0.0f;
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int i = row0 + rs + 4 * p;
            const float4 hn = make_float4(fmaxf(v[p][0], 0.0f), fmaxf(v[p][1], 0.0f), fmaxf(v[p][2], 0.0f), fmaxf(v[p][3], 0.0f));
            if (i < n) {
                *reinterpret_cast<float4 *>(pre + (size_t)i * kH + 4 * q8) = make_float4(v[p][0], v[p][1], v[p][2], v[p][3]);
                *reinterpret_cast<float4 *>(h + (size_t)i * kH + 4 * q8) = hn;
            }
            if (LAST) {
                // the 32 features added as a tree: f + 16, + 8, + 4, + 2, + 1
                float y[4] = {o[0] * hn.x, o[1] * hn.y, o[2] * hn.z, o[3] * hn.w};
#pragma unroll
                for (int t = 4; t > 0; t >>= 1)
#pragma unroll
                    for (int u = 0; u < 4; u++) y[u] += __shfl_down_sync(0xFFFFFFFFu, y[u], t, 8);
                const float yi = (y[0] + y[2]) + (y[1] + y[3]);
                const float yr = __shfl_sync(0xFFFFFFFFu, yi, 0, 8);
                if (q8 == p) yrow = yr;
            }
        }
        if (LAST && q8 < 4 && row0 + rs + 4 * q8 < n) {
            const int i = row0 + rs + 4 * q8, e = edge[i];
            z[e] = fma(r[e], Dinv[e], rho * (double)(yrow + d0) * isd[i]);
        }
    }
}
constexpr int kLayerShared = (2 * kH * kH + kW * kTileRows * kSRow) * (int)sizeof(float);

// ---- inference layer on the tensor cores ----
// The preconditioner application inside the flexible PCG (no backward pass,
// so nothing but h is stored).  A warp takes a tile of 16 consecutive rows,
// half of one SELL slice, so every row of the tile has the slice's width.
//  1. Aggregation: lane (rs = lane >> 3, q = lane & 7) sums features
//     4q .. 4q + 3 of rows rs, rs + 4, rs + 8, rs + 12 over the rows'
//     entries, so each 16-byte gather of a warp reads four whole 128-byte
//     feature rows (eight lanes per row).  Half-row gathers (16 rows of 64
//     bytes per instruction) kept the L1 at its throughput limit for a
//     quarter of the useful bytes; this layout measured 76 -> 46 ms per
//     Newmark solve.  The rows' own h and aggregates g go to the warp's tile
//     S[16][64] in shared memory.
//  2. The 16 x 64 by 64 x 32 product [h g] [W Q]^T on mma.sync m16n8k8 TF32
//     with FP32 accumulation.  The weights are bfloat16 values, exact in TF32;
//     each activation is split as hi + lo with hi = TF32(a), lo = TF32(a - hi)
//     (two products per tile), so the products carry ~22 significant bits,
//     as close to the FP32 layer as the FP32 sums themselves.
// Fragment layouts (PTX ISA, m16n8k8 .tf32; g = lane >> 2, t = lane & 3):
//   A: a0 (g, t), a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4)
//   B: b0 (k = t, n = g), b1 (k = t + 4, n = g)
//   C: c0 (g, 2t), c1 (g, 2t + 1), c2 (g + 8, 2t), c3 (g + 8, 2t + 1)
constexpr int kTcBlocksPerSm = 4;

__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void mma_tf32(float c[4], const uint32_t a[4], float2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(__float_as_uint(b.x)), "r"(__float_as_uint(b.y)));
}

template <bool LAST>
__global__ void __launch_bounds__(kT, kTcBlocksPerSm) k_layer_tc(int n, const int *__restrict__ sp,
                                                                 const int *__restrict__ sw,
                                                                 const int *__restrict__ col,
                                                                 const float *__restrict__ ahat,
                                                                 const float *__restrict__ hp,
                                                                 const unsigned short *__restrict__ th, int off,
                                                                 float *__restrict__ h, const int *__restrict__ edge, const double *__restrict__ r,
                                                                 const double *__restrict__ Dinv,
                                                                 const double *__restrict__ isd,
                                                                 const double *__restrict__ nrm,
                                                                 double *__restrict__ z,
                                                                 const double *__restrict__ zo,
                                                                 double *__restrict__ part) {
    // B fragments of [W Q]^T for k-step ks and column tile nt at Bf[(ks * 4 + nt) * 32 + lane]
    __shared__ __align__(16) float2 Bf[8 * 4 * 32];
    __shared__ __align__(16) float S[kW][kTileRows * kSRow];
    __shared__ float bsh[kH], osh[kH];
    for (int q = threadIdx.x; q < 8 * 4 * 32; q += kT) {
        const int ks = q >> 7, nt = (q >> 5) & 3, ln = q & 31;
        const int f = nt * 8 + (ln >> 2), k0 = ks * 8 + (ln & 3), k1 = k0 + 4;
        // column k of [W Q]^T row f: W[f][k] for k < 32, Q[f][k - 32] after
        const float w0 = k0 < kH ? bf(th, off + f * kH + k0) : bf(th, off + kH * kH + f * kH + (k0 - kH));
        const float w1 = k1 < kH ? bf(th, off + f * kH + k1) : bf(th, off + kH * kH + f * kH + (k1 - kH));
        Bf[q] = make_float2(w0, w1);
    }
    if (threadIdx.x < kH) {
        bsh[threadIdx.x] = bf(th, off + 2 * kH * kH + threadIdx.x);
        osh[threadIdx.x] = LAST ? bf(th, kOffO + threadIdx.x) : 0.0f;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rs = lane >> 3, q8 = lane & 7;   // aggregation: rows rs + 4p, features 4 q8 .. 4 q8 + 3
    const int g = lane >> 2, t4 = lane & 3;
    float *Sw = S[warp];
    const float d0 = LAST ? bf(th, kOffD0) : 0.0f;
    const double rho = LAST ? block_rho(nrm, n) : 0.0;
    double dots[2] = {0.0, 0.0};   // (r, z), (r, z_old)
    const int ntiles = (n + kTileRows - 1) / kTileRows;
    for (int tile = blockIdx.x * kW + warp; tile < ntiles; tile += gridDim.x * kW) {
        const int row0 = tile * kTileRows;
        float4 acc[4], hv[4];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            acc[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            hv[p] = acc[p];
        }
        aggregate_tile(tile, sp, sw, col, ahat, hp, acc);
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int i = row0 + rs + 4 * p;
            if (i < n) hv[p] = __ldg(reinterpret_cast<const float4 *>(hp + (size_t)i * kH + 4 * q8));
        }
        __syncwarp();   // the previous tile's fragment loads are done
#pragma unroll
        for (int p = 0; p < 4; p++) {
            float *srow = Sw + (rs + 4 * p) * kSRow + 4 * q8;
            *reinterpret_cast<float4 *>(srow) = hv[p];         // columns 0..31: h
            *reinterpret_cast<float4 *>(srow + kH) = acc[p];   // columns 32..63: g
        }
        __syncwarp();
        float c[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; nt++) {
            const float b0 = bsh[nt * 8 + 2 * t4], b1 = bsh[nt * 8 + 2 * t4 + 1];
            c[nt][0] = b0;
            c[nt][1] = b1;
            c[nt][2] = b0;
            c[nt][3] = b1;
        }
#pragma unroll
        for (int ks = 0; ks < 8; ks++) {
            const float *s0 = Sw + g * kSRow + ks * 8 + t4;
            const float av[4] = {s0[0], s0[8 * kSRow], s0[4], s0[8 * kSRow + 4]};
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                hi[q] = to_tf32(av[q]);
                lo[q] = to_tf32(av[q] - __uint_as_float(hi[q]));
            }
#pragma unroll
            for (int nt = 0; nt < 4; nt++) {
                const float2 b = Bf[(ks * 4 + nt) * 32 + lane];
                mma_tf32(c[nt], lo, b);
                mma_tf32(c[nt], hi, b);
            }
        }
        const int i0 = tile * kTileRows + g, i1 = i0 + 8;
        if (!LAST) {
#pragma unroll
            for (int nt = 0; nt < 4; nt++) {
                const int f = nt * 8 + 2 * t4;
                if (i0 < n)
                    *reinterpret_cast<float2 *>(h + (size_t)i0 * kH + f) =
                        make_float2(fmaxf(c[nt][0], 0.0f), fmaxf(c[nt][1], 0.0f));
                if (i1 < n)
                    *reinterpret_cast<float2 *>(h + (size_t)i1 * kH + f) =
                        make_float2(fmaxf(c[nt][2], 0.0f), fmaxf(c[nt][3], 0.0f));
            }
        } else {
            float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
            for (int nt = 0; nt < 4; nt++) {
                const int f = nt * 8 + 2 * t4;
                y0 = fmaf(osh[f], fmaxf(c[nt][0], 0.0f), y0);
                y0 = fmaf(osh[f + 1], fmaxf(c[nt][1], 0.0f), y0);
                y1 = fmaf(osh[f], fmaxf(c[nt][2], 0.0f), y1);
                y1 = fmaf(osh[f + 1], fmaxf(c[nt][3], 0.0f), y1);
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                y0 += __shfl_xor_sync(0xFFFFFFFFu, y0, o);
                y1 += __shfl_xor_sync(0xFFFFFFFFu, y1, o);
            }
            if (t4 == 0) {
                const int ii[2] = {i0, i1};
                const float yy[2] = {y0, y1};
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const int i = ii[q];
                    if (i >= n) continue;
                    const int e = edge[i];
                    const double ri = r[e], zi = fma(ri, Dinv[e], rho * (double)(yy[q] + d0) * isd[i]);
                    z[e] = zi;
                    if (zo) {
                        dots[0] = fma(ri, zi, dots[0]);
                        dots[1] = fma(ri, zo[e], dots[1]);
                    }
                }
            }
        }
    }
    if (LAST && zo) block_partial<2>(dots, part);
}

// ---- backward ----
// gy_i = dL/dy_i = 2 (A z - r)_i rho / (sqrt(d_i) N), N = n rho^2; loss partials z.(Az) - 2 z.r
__global__ void __launch_bounds__(kT) k_gy(int n, int nsl, const int *__restrict__ sp, const int *__restrict__ sw,
                                          const int *__restrict__ col, const double *__restrict__ val,
                                          const double *__restrict__ z, const double *__restrict__ r,
                                          const int *__restrict__ row, const double *__restrict__ isd,
                                          const double *__restrict__ nrm, double *__restrict__ gy, double *part) {
    const int lane = threadIdx.x & 31;
    const double N = nrm[0], rho = block_rho(nrm, n);
    double v[1] = {0.0};
    for (int sl = blockIdx.x * kW + (threadIdx.x >> 5); sl < nsl; sl += gridDim.x * kW) {
        const int kb = sp[sl] + lane, kw = sw[sl];
        double s = 0.0;
        for (int j = 0; j < kw; j++) s = fma(val[kb + 32 * j], z[col[kb + 32 * j]], s);
        const int i = sl * 32 + lane;
        if (i < n) {
            const int g = row[i];
            gy[g] = N > 0.0 ? 2.0 * (s - r[i]) * rho * isd[g] / N : 0.0;
            v[0] += z[i] * s - 2.0 * z[i] * r[i];
        }
    }
    block_partial<1>(v, part);
}

// Adds a warp's per-lane accumulators acc[0..NA) into the block's shared sum in
// warp order, then writes the block's partials part[block][q * 32 + lane].
template <int NA>
__device__ __forceinline__ void block_accumulate(const float acc[NA], float *sh, float *part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int w = 0; w < kW; w++) {
        if (warp == w) {
#pragma unroll
            for (int q = 0; q < NA; q++) sh[q * 32 + lane] = (w == 0 ? 0.0f : sh[q * 32 + lane]) + acc[q];
        }
        __syncthreads();
    }
    for (int t = threadIdx.x; t < NA * 32; t += kT) part[(size_t)blockIdx.x * NA * 32 + t] = sh[t];
}

// Layer l backward.  dpre = dh * [pre > 0]; dW[f][k] += dpre_f h_k, dQ[f][k] +=
// dpre_f g_k, db[f] += dpre_f (and, for the last layer, do[f], dd0); writes
// own = W^T dpre into dh_out and t = Q^T dpre into tq (aggregated next).
// A warp takes kBwdRows of its rows at a time through shared memory, the next ones
// in flight meanwhile (128 registers leave 16 warps an SM).  A lane holds 8 x 4
// entries of dW and dQ and forms 4 entries of own or t for 4 rows, 48 words
// read from shared memory a row.  220,256 rows: 210 us with a warp per row and
// 160 words read or shuffled, 131 without the fetch ahead, 73 us now.  A
// warp's rows stay a grid apart and are added in increasing order, one sum per entry, so
// the sums do not depend on this split.
constexpr int kBwdRows = 8;
constexpr int kBRow = 4 * kH + 4, kARow = kH + 4;   // padded rows: no bank conflicts

// 16 or 8 bytes of global memory to shared memory, asynchronously; zeros where !ok
template <int BYTES>
__device__ __forceinline__ void copy_async(float *dst, const void *src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(ok ? BYTES : 0)
                 : "memory");
}

template <bool LAST>
__global__ void __launch_bounds__(kT, 2) k_layer_bwd(int n, const float *__restrict__ hp,
                                                    const float *__restrict__ g, const float *__restrict__ pre,
                                                    const float *__restrict__ hcur, const float *__restrict__ dh_in,
                                                    const double *__restrict__ gy,
                                                    const unsigned short *__restrict__ th, int off,
                                                    float *__restrict__ dh_out, float *__restrict__ tq,
                                                    float *__restrict__ part) {
    extern __shared__ __align__(16) float bwd_sh[];
    float *WQ = bwd_sh;                                             // W, then Q
    float *acc_sh = WQ + 2 * kH * kH;                               // dW, then dQ: [f][k]
    float *vec_sh = acc_sh + 2 * kH * kARow;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // two batches of rows a warp: h, g, pre (then dpre), dh (last layer: h of the layer), gy
    float *rows_sh = vec_sh + 3 * 32 + warp * 2 * kBwdRows * kBRow;
    for (int t = threadIdx.x; t < 2 * kH * kH; t += kT) WQ[t] = bf(th, off + t);
    __syncthreads();
    const float o = LAST ? bf(th, kOffO + lane) : 0.0f;
    const int f0 = 8 * (lane >> 3), k0 = 4 * (lane & 7);            // entries of dW, dQ
    const int m0 = 4 * (lane >> 4), q = (lane >> 3) & 1;            // rows, own (0) or t (1), ...
    const float *M = WQ + q * kH * kH + k0;                         // ... entries k0 .. k0 + 3
    float *out = q ? tq : dh_out;
    float aw[8][4], aq[8][4], vec[3] = {0.0f, 0.0f, 0.0f};          // vec: db, do, dd0
#pragma unroll
    for (int f = 0; f < 8; f++)
#pragma unroll
        for (int u = 0; u < 4; u++) aw[f][u] = aq[f][u] = 0.0f;
    const int stride = gridDim.x * kW;
    // four rows an instruction, eight lanes a row (a row past the end: zeros)
    auto fetch = [&](int i0, float *S) {
#pragma unroll
        for (int half = 0; half < 2; half++) {
            const int m = 4 * half + (lane >> 3), i = i0 + m * stride;
            const bool ok = i < n;
            const size_t at = (size_t)(ok ? i : 0) * kH + k0;
            float *row = S + m * kBRow + k0;
            copy_async<16>(row, hp + at, ok);
            copy_async<16>(row + kH, g + at, ok);
            copy_async<16>(row + 2 * kH, pre + at, ok);
            copy_async<16>(row + 3 * kH, (LAST ? hcur : dh_in) + at, ok);
        }
        if (LAST && lane < kBwdRows) {
            const int i = i0 + lane * stride;
            copy_async<8>(S + lane * kBRow + 4 * kH, gy + (i < n ? i : 0), i < n);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int i0 = blockIdx.x * kW + warp;
    fetch(i0, rows_sh);
    for (int buf = 0; i0 < n; i0 += kBwdRows * stride, buf ^= 1) {
        float *S = rows_sh + buf * kBwdRows * kBRow;
        fetch(i0 + kBwdRows * stride, rows_sh + (buf ^ 1) * kBwdRows * kBRow);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kBwdRows; m++) {
            float *row = S + m * kBRow;
            float dh = row[3 * kH + lane];
            if (LAST) {
                const float gyi = (float)*reinterpret_cast<const double *>(row + 4 * kH);
                vec[1] = fmaf(gyi, dh, vec[1]);
                vec[2] += gyi;
                dh = gyi * o;
            }
            const float dp = row[2 * kH + lane] > 0.0f ? dh : 0.0f;
            vec[0] += dp;
            row[2 * kH + lane] = dp;
        }
        __syncwarp();
#pragma unroll 2
        for (int m = 0; m < kBwdRows; m++) {
            float d[8], h4[4], g4[4];
            load4(S + m * kBRow + 2 * kH + f0, d);
            load4(S + m * kBRow + 2 * kH + f0 + 4, d + 4);
            load4(S + m * kBRow + k0, h4);
            load4(S + m * kBRow + kH + k0, g4);
#pragma unroll
            for (int f = 0; f < 8; f++)
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    aw[f][u] = fmaf(d[f], h4[u], aw[f][u]);
                    aq[f][u] = fmaf(d[f], g4[u], aq[f][u]);
                }
        }
        float y[4][4];
#pragma unroll
        for (int m = 0; m < 4; m++)
#pragma unroll
            for (int u = 0; u < 4; u++) y[m][u] = 0.0f;
#pragma unroll 2
        for (int f = 0; f < kH; f += 4) {
            float d[4][4];
#pragma unroll
            for (int m = 0; m < 4; m++) load4(S + (m0 + m) * kBRow + 2 * kH + f, d[m]);
#pragma unroll
            for (int t = 0; t < 4; t++) {
                float w[4];
                load4(M + (f + t) * kH, w);
#pragma unroll
                for (int m = 0; m < 4; m++)
#pragma unroll
                    for (int u = 0; u < 4; u++) y[m][u] = fmaf(w[u], d[m][t], y[m][u]);
            }
        }
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const int i = i0 + (m0 + m) * stride;
            if (i < n) *reinterpret_cast<float4 *>(out + (size_t)i * kH + k0) = make_float4(y[m][0], y[m][1], y[m][2], y[m][3]);
        }
        __syncwarp();   // the batch has been read: the next fetch may overwrite it
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // the warps' sums in warp order, then the block's partials [q * 32 + f]
    for (int w = 0; w < kW; w++) {
        if (warp == w) {
#pragma unroll
            for (int f = 0; f < 8; f++) {
                float *pw = acc_sh + (f0 + f) * kARow + k0, *pq = pw + kH * kARow;
                float sw4[4] = {0.0f, 0.0f, 0.0f, 0.0f}, sq4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (w > 0) {
                    load4(pw, sw4);
                    load4(pq, sq4);
                }
                *reinterpret_cast<float4 *>(pw) = make_float4(sw4[0] + aw[f][0], sw4[1] + aw[f][1], sw4[2] + aw[f][2], sw4[3] + aw[f][3]);
                *reinterpret_cast<float4 *>(pq) = make_float4(sq4[0] + aq[f][0], sq4[1] + aq[f][1], sq4[2] + aq[f][2], sq4[3] + aq[f][3]);
            }
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float x = c == 2 && lane > 0 ? 0.0f : vec[c];
                vec_sh[c * 32 + lane] = (w == 0 ? 0.0f : vec_sh[c * 32 + lane]) + x;
            }
        }
        __syncthreads();
    }
    float *dst = part + (size_t)blockIdx.x * kNA * 32;
    for (int t = threadIdx.x; t < kNA * 32; t += kT) {
        const int c = t >> 5, f = t & 31;
        dst[t] = c < kH ? acc_sh[f * kARow + c] : c < 2 * kH ? acc_sh[(kH + f) * kARow + c - kH] : vec_sh[t - 2 * kH * 32];
    }
}

constexpr int kBwdShared = (2 * kH * kH + 2 * kH * kARow + 3 * 32 + kW * 2 * kBwdRows * kBRow) * (int)sizeof(float);

// dh_out_i += sum_j Ahat_ij tq_j (a tile of 16 rows per warp: 92 -> 60 us at 220,256
// rows, bound by the gathers from L2)
__global__ void __launch_bounds__(kT) k_agg_bwd(int n, const int *__restrict__ sp, const int *__restrict__ sw,
                                               const int *__restrict__ col, const float *__restrict__ ahat,
                                               const float *__restrict__ tq, float *__restrict__ dh) {
    const int lane = threadIdx.x & 31, rs = lane >> 3, q8 = lane & 7;
    const int ntiles = (n + kTileRows - 1) / kTileRows;
    for (int tile = blockIdx.x * kW + (threadIdx.x >> 5); tile < ntiles; tile += gridDim.x * kW) {
        float4 acc[4];
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int i = tile * kTileRows + rs + 4 * p;
            acc[p] = i < n ? *reinterpret_cast<const float4 *>(dh + (size_t)i * kH + 4 * q8)
                           : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        aggregate_tile(tile, sp, sw, col, ahat, tq, acc);
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const int i = tile * kTileRows + rs + 4 * p;
            if (i < n) *reinterpret_cast<float4 *>(dh + (size_t)i * kH + 4 * q8) = acc[p];
        }
    }
}

__global__ void __launch_bounds__(kT) k_embed_bwd(int n, const float *__restrict__ xin, const float *__restrict__ feat_a,
                                                 const float *__restrict__ pre0, const float *__restrict__ dh0,
                                                 float *__restrict__ part) {
    __shared__ float acc_sh[3 * 32];
    const int lane = threadIdx.x & 31, stride = gridDim.x * kW;
    float acc[3] = {0.0f, 0.0f, 0.0f};
    // eight rows' loads in flight, added in order (a row past the end adds zeros)
    for (int i0 = blockIdx.x * kW + (threadIdx.x >> 5); i0 < n; i0 += 8 * stride) {
        float pr[8], dh[8], xi[8], fa[8];
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int i = i0 + m * stride;
            pr[m] = dh[m] = xi[m] = fa[m] = 0.0f;
            if (i < n) {
                pr[m] = pre0[(size_t)i * kH + lane];
                dh[m] = dh0[(size_t)i * kH + lane];
                xi[m] = xin[i];
                fa[m] = feat_a[i];
            }
        }
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const float dp = pr[m] > 0.0f ? dh[m] : 0.0f;
            acc[0] = fmaf(dp, xi[m], acc[0]);
            acc[1] = fmaf(dp, fa[m], acc[1]);
            acc[2] += dp;
        }
    }
    block_accumulate<3>(acc, acc_sh, part);
}

// grad[dst[q*32 + lane]] = sum over blocks of part[block][q*32 + lane] (FP64, fixed
// order), for the four tables of one backward pass: three layers of kNA x 32
// partials, then the embedding's 3 x 32.  A block takes 32 of them, its warps
// every eighth partial (a thread per parameter added the 456 in one chain: 4
// launches of 66 us -> one of 20).
constexpr int kFinalBlocks = 3 * kNA + 3;
__global__ void __launch_bounds__(kT) k_grad_final(const float *__restrict__ part, const int *__restrict__ dst,
                                                  double *__restrict__ grad) {
    __shared__ double sh[kW][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tab = min((int)blockIdx.x / kNA, 3), q = blockIdx.x - tab * kNA, na = tab < 3 ? kNA : 3;
    const float *p = part + (size_t)tab * kGB * kNA * 32 + q * 32 + lane;
    double s = 0.0;
#pragma unroll 8
    for (int b = warp; b < kGB; b += kW) s += (double)p[(size_t)b * na * 32];
    sh[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        for (int w = 1; w < kW; w++) s += sh[w][lane];
        const int d = dst[tab * kNA * 32 + q * 32 + lane];
        if (d >= 0) grad[d] = s;
    }
}

__global__ void k_adam(int np, float *__restrict__ theta, float *__restrict__ m, float *__restrict__ v,
                       const double *__restrict__ grad, float lr, float b1, float b2, float eps, float c1, float c2,
                       unsigned short *__restrict__ th_bf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    const float gi = (float)grad[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float t = theta[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    theta[i] = t;
    th_bf[i] = __bfloat16_as_ushort(__float2bfloat16_rn(t));
}

__global__ void k_to_bf16(int np, const float *__restrict__ theta, unsigned short *__restrict__ th_bf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < np) th_bf[i] = __bfloat16_as_ushort(__float2bfloat16_rn(theta[i]));
}

// ---- flexible PCG vector steps ----
// q = A p, and (p, q)
__global__ void __launch_bounds__(kT) k_spmv_dot(int n, int nsl, const int *__restrict__ sp, const int *__restrict__ sw,
                                                const int *__restrict__ col, const double *__restrict__ val,
                                                const double *__restrict__ p, double *__restrict__ q, double *part) {
    const int lane = threadIdx.x & 31;
    double v[1] = {0.0};
    for (int sl = blockIdx.x * kW + (threadIdx.x >> 5); sl < nsl; sl += gridDim.x * kW) {
        const int kb = sp[sl] + lane, kw = sw[sl];
        double s = 0.0;
#pragma unroll 8
        for (int j = 0; j < kw; j++) s = fma(val[kb + 32 * j], p[col[kb + 32 * j]], s);
        const int i = sl * 32 + lane;
        if (i < n) {
            q[i] = s;
            v[0] = fma(p[i], s, v[0]);
        }
    }
    block_partial<1>(v, part);
}

// x += alpha p, r -= alpha q with alpha = rz / (p, q), the latter from its
// partials; then (r, r) and (r, D^-1 r)
__global__ void __launch_bounds__(kT) k_fpcg_xr(int n, double rz, int n_part, const double *__restrict__ pq_part,
                                               const double *__restrict__ p, const double *__restrict__ q,
                                               const double *__restrict__ Dinv, double *__restrict__ x,
                                               double *__restrict__ r, double *part) {
    __shared__ double s_alpha;
    const double pq = block_total(n_part, pq_part);
    if (threadIdx.x == 0) s_alpha = rz / pq;
    __syncthreads();
    const double alpha = s_alpha;
    double v[2] = {0.0, 0.0};
    for (int i = blockIdx.x * kT + threadIdx.x; i < n; i += gridDim.x * kT) {
        x[i] = fma(alpha, p[i], x[i]);
        const double ri = fma(-alpha, q[i], r[i]);
        r[i] = ri;
        v[0] = fma(ri, ri, v[0]);
        v[1] = fma(ri * Dinv[i], ri, v[1]);
    }
    block_partial<2>(v, part);
}

// out[0] = (r, r) from na partials, out[1], out[2] = (r, z), (r, z_old) from nb
// partials each: a warp a value
__global__ void k_fpcg_sums(int na, const double *__restrict__ a, int nb, const double *__restrict__ b,
                            double *__restrict__ out) {
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const double *v = c == 0 ? a : b + (size_t)(c - 1) * nb;
    const int m = c == 0 ? na : nb;
    double s = 0.0;
    for (int k = lane; k < m; k += 32) s += v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
    if (lane == 0) out[c] = s;
}

// p = z + beta p, beta = beta_num / rz_old
__global__ void k_fpcg_p(int n, double beta, const double *__restrict__ z, double *__restrict__ p) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = fma(beta, p[i], z[i]);
}

__global__ void k_jacobi(int n, const double *__restrict__ Dinv, const double *__restrict__ r, double *__restrict__ z) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) z[i] = Dinv[i] * r[i];
}

__global__ void k_resid(int n, int nsl, const int *__restrict__ sp, const int *__restrict__ sw,
                        const int *__restrict__ col, const double *__restrict__ val, const double *__restrict__ b,
                        const double *__restrict__ x, double *__restrict__ r) {
    const int lane = threadIdx.x & 31;
    for (int sl = blockIdx.x * kW + (threadIdx.x >> 5); sl < nsl; sl += gridDim.x * kW) {
        const int kb = sp[sl] + lane, kw = sw[sl];
        double s = 0.0;
        for (int j = 0; j < kw; j++) s = fma(val[kb + 32 * j], x[col[kb + 32 * j]], s);
        const int i = sl * 32 + lane;
        if (i < n) r[i] = b[i] - s;
    }
}

// deterministic [0, 1) hash of (seed, i): SplitMix64 finaliser
double hash01(unsigned long long seed, unsigned long long i) {
    unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

// a thread per row (220,256 rows: A p and (p, q) 24 -> 16 us, the embedding 17 ->
// 14 us against 456 blocks, whose warps took two slices in turn)
int row_blocks(int n) { return std::max(1, std::min((n + kT - 1) / kT, kRowBlocks)); }

// a warp per 16-row tile
int tiles_grid(int n) { return std::max(1, std::min((n + kW * kTileRows - 1) / (kW * kTileRows), 152 * 16)); }

// the tensor-core layer: one 16-row tile per warp at a time, kTcBlocksPerSm blocks per SM
int tc_grid(int n) {
    static int sms = 0;
    if (sms <= 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            sms <= 0)
            sms = 1;
    }
    const int tiles = (n + kTileRows - 1) / kTileRows;
    return std::max(1, std::min((tiles + kW - 1) / kW, sms * kTcBlocksPerSm));
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int gnn_reduce_launch(Sim *s, int nv, double *out, int nb = kGB) {
    GnnState &G = s->gnn;
    { k_final_sums<<<1, 32 * nv, 0, s->stream>>>(nb, nv, G.part.p, out); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

// The network's row order and its SELL-32 pattern, packed: padding names the
// row itself
static int gnn_rows(Sim *s) {
    GnnState &G = s->gnn;
    const Mesh *m = s->mesh;
    const int n = m->n_int_edges, nsl = (n + 31) / 32;
    // rows by (length, canonical edge): counted, then placed in canonical order
    int most = 0;
    for (int e = 0; e < n; e++) most = std::max(most, m->h_row_len[e]);
    std::vector<int> at(most + 2, 0), edge_of(n), row_of(n), canon(n);
    for (int e = 0; e < n; e++) at[m->h_row_len[e] + 1]++;
    for (int l = 0; l <= most; l++) at[l + 1] += at[l];
    for (int c = 0; c < m->n_edges; c++) {
        const int e = m->h_edge_internal[c];
        if (e >= n) continue;
        const int i = at[m->h_row_len[e]]++;
        edge_of[i] = e;
        row_of[e] = i;
        canon[i] = c;
    }
    std::vector<int> ptr(nsl + 1, 0), width(nsl, 0);
    for (int sl = 0; sl < nsl; sl++) {
        width[sl] = m->h_row_len[edge_of[std::min(n, 32 * sl + 32) - 1]];
        ptr[sl + 1] = ptr[sl] + 32 * width[sl];
    }
    G.rows.n_rows = n;
    G.rows.n_slices = nsl;
    G.rows.n_elems = ptr[nsl];
    DevBuf<int> canon_dev;
    int rc;
    if ((rc = G.rows.ptr.upload(ptr)) || (rc = G.rows.width.upload(width)) || (rc = G.rows.col.alloc(ptr[nsl])) ||
        (rc = G.edge_of.upload(edge_of)) || (rc = G.row_of.upload(row_of)) || (rc = canon_dev.upload(canon)))
        return rc;
    if (n > 0) {
        { k_rows_cols<<<(32 * nsl + 255) / 256, 256, 0, s->stream>>>(n, nsl, G.rows.ptr.p, G.rows.width.p, canon_dev.p, m->e2t.rowptr.p, m->e2t.col.p, m->tet_edge.p, G.row_of.p, G.rows.col.p); note_launch(); }
        FP_CUDA(cudaGetLastError());
        FP_CUDA(cudaStreamSynchronize(s->stream));
    }
    return PIC_OK;
}

int gnn_prepare(Sim *s) {
    GnnState &G = s->gnn;
    if (G.ready) return PIC_OK;
    const Mesh *m = s->mesh;
    const int n = m->n_int_edges;
    const size_t nn = (size_t)std::max(n, 1), nh = nn * kH;
    FP_CUDA(cudaFuncSetAttribute(k_layer_bwd<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdShared));
    FP_CUDA(cudaFuncSetAttribute(k_layer_bwd<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdShared));
    int rc;
    if ((rc = gnn_rows(s))) return rc;
    const long long nel = std::max(G.rows.n_elems, 1LL);
    if ((rc = G.theta.alloc(kGnnParams)) || (rc = G.theta_bf.alloc(kGnnParams)) || (rc = G.adam_m.alloc(kGnnParams)) ||
        (rc = G.adam_v.alloc(kGnnParams)) || (rc = G.grad.alloc(kGnnParams)) || (rc = G.ahat.alloc(nel)) ||
        (rc = G.isd.alloc(nn)) || (rc = G.logd.alloc(nn)) || (rc = G.feat_a.alloc(nn)) || (rc = G.xin.alloc(nn)) ||
        (rc = G.gy.alloc(nn)) || (rc = G.dh.alloc(nh)) || (rc = G.dh2.alloc(nh)) || (rc = G.tq.alloc(nh)) ||
        (rc = G.part.alloc(std::max<size_t>(8 * (size_t)kGB, 3 * (size_t)kRowBlocks + 2 * (size_t)tc_grid(n)))) || (rc = G.sc.alloc(16)) ||
        (rc = G.wpart.alloc(4 * (size_t)kGB * kNA * 32)) || (rc = G.dst.alloc(4 * kNA * 32)))
        return rc;
    for (int l = 0; l < 4; l++)
        if ((rc = G.h[l].alloc(nh)) || (rc = G.pre[l].alloc(nh)) || (rc = G.g[l].alloc(l ? nh : 1))) return rc;
    if ((rc = G.r.alloc(nn)) || (rc = G.z.alloc(nn)) || (rc = G.zold.alloc(nn)) || (rc = G.p.alloc(nn)) ||
        (rc = G.q.alloc(nn)))
        return rc;
    // gradient destinations of the per-lane accumulators: layer l (1..3) at
    // table l-1, the embedding at table 3
    std::vector<int> dst(4 * kNA * 32, -1);
    for (int l = 1; l <= 3; l++) {
        int *d = dst.data() + (l - 1) * kNA * 32;
        const int off = kOffL + (l - 1) * kLayer;
        for (int k = 0; k < kH; k++)
            for (int f = 0; f < kH; f++) {
                d[k * 32 + f] = off + f * kH + k;                // dW[f][k]
                d[(kH + k) * 32 + f] = off + kH * kH + f * kH + k;   // dQ[f][k]
            }
        for (int f = 0; f < kH; f++) d[2 * kH * 32 + f] = off + 2 * kH * kH + f;
        if (l == 3) {
            for (int f = 0; f < kH; f++) d[(2 * kH + 1) * 32 + f] = kOffO + f;
            d[(2 * kH + 2) * 32 + 0] = kOffD0;
        }
    }
    {
        int *d = dst.data() + 3 * kNA * 32;
        for (int f = 0; f < kH; f++) {
            d[f] = kOffU + f;
            d[32 + f] = kOffV + f;
            d[64 + f] = kOffC + f;
        }
    }
    FP_CUDA(cudaMemcpyAsync(G.dst.p, dst.data(), sizeof(int) * dst.size(), cudaMemcpyHostToDevice, s->stream));
    if (n > 0) {
        { k_prep_rows<<<(n + 255) / 256, 256, 0, s->stream>>>(n, G.edge_of.p, s->Dinv.p, G.isd.p, G.logd.p); note_launch(); }
        { k_sum<<<kGB, kT, 0, s->stream>>>(n, G.logd.p, G.part.p); note_launch(); }
        if ((rc = gnn_reduce_launch(s, 1, G.sc.p + 8))) return rc;
        const int nsl = G.rows.n_slices;
        { k_prep_ahat<<<(nsl * 32 + 255) / 256, 256, 0, s->stream>>>(n, nsl, G.rows.ptr.p, G.rows.width.p, G.rows.col.p, G.edge_of.p, m->As.ptr.p, m->As.width.p, m->As.col.p, s->A_val.p, G.isd.p, G.logd.p, G.sc.p + 8, G.ahat.p, G.feat_a.p); note_launch(); }
    }
    FP_CUDA(cudaGetLastError());
    G.ready = 1;
    // default weights: small uniform values from a fixed hash, output layer 0
    // (the network starts as the Jacobi preconditioner)
    std::vector<float> th(kGnnParams, 0.0f);
    for (int i = 0; i < kOffO; i++) {
        const int fan = i < kOffL ? 2 : 2 * kH;
        th[i] = (float)((2.0 * hash01(0x6E6E, i) - 1.0) * std::sqrt(3.0 / fan));
    }
    return gnn_set_weights(s, th.data(), kGnnParams);
}

int gnn_set_weights(Sim *s, const float *w, long long np) {
    GnnState &G = s->gnn;
    if (np != kGnnParams) {
        set_error("GNN weights: expected " + std::to_string(kGnnParams) + " values");
        return PIC_ERR_INVALID_ARG;
    }
    FP_CUDA(cudaMemcpyAsync(G.theta.p, w, sizeof(float) * kGnnParams, cudaMemcpyHostToDevice, s->stream));
    FP_CUDA(cudaMemsetAsync(G.adam_m.p, 0, sizeof(float) * kGnnParams, s->stream));
    FP_CUDA(cudaMemsetAsync(G.adam_v.p, 0, sizeof(float) * kGnnParams, s->stream));
    { k_to_bf16<<<(kGnnParams + 255) / 256, 256, 0, s->stream>>>(kGnnParams, G.theta.p, G.theta_bf.p); note_launch(); }
    FP_CUDA(cudaGetLastError());
    FP_CUDA(cudaStreamSynchronize(s->stream));
    G.adam_t = 0;
    return PIC_OK;
}

int gnn_get_weights(Sim *s, float *w, long long np) {
    if (np != kGnnParams) {
        set_error("GNN weights: expected " + std::to_string(kGnnParams) + " values");
        return PIC_ERR_INVALID_ARG;
    }
    FP_CUDA(cudaMemcpyAsync(w, s->gnn.theta.p, sizeof(float) * kGnnParams, cudaMemcpyDeviceToHost, s->stream));
    FP_CUDA(cudaStreamSynchronize(s->stream));
    return PIC_OK;
}

// z = P(r) on interior edges (internal order, device arrays); with `keep`
// the activations a backward pass needs are stored.  G.sc[0] receives n rho^2,
// from the n_part partials at nrm_part (NULL: formed here).  With zo, the partials
// of (r, z) and (r, zo) go to dot_part, tc_grid(n) each.
static int gnn_forward_dots(Sim *s, const double *r, double *z, bool keep, int n_part, const double *nrm_part, const double *zo,
                            double *dot_part) {
    GnnState &G = s->gnn;
    const int n = s->mesh->n_int_edges;
    if (n == 0) return PIC_OK;
    const DevSell &A = G.rows;
    cudaStream_t st = s->stream;
    if (!nrm_part) {
        { k_rnorm<<<kGB, kT, 0, st>>>(n, G.edge_of.p, r, s->Dinv.p, G.part.p); note_launch(); }
        nrm_part = G.part.p;
        n_part = kGB;
    }
    const int rb = row_blocks(n);
    if (keep) { k_embed<true><<<rb, kT, 0, st>>>(n, G.edge_of.p, r, G.isd.p, n_part, nrm_part, G.sc.p, G.feat_a.p, G.theta_bf.p, G.xin.p, G.pre[0].p, G.h[0].p); note_launch(); }
    else { k_embed<false><<<rb, kT, 0, st>>>(n, G.edge_of.p, r, G.isd.p, n_part, nrm_part, G.sc.p, G.feat_a.p, G.theta_bf.p, G.xin.p, G.pre[0].p, G.h[0].p); note_launch(); }
    const int gr = tiles_grid(n), gt = tc_grid(n);
    for (int l = 1; l <= 3; l++) {
        const int off = kOffL + (l - 1) * kLayer;
        // without keep, layers 1 and 2 ping-pong between h[0] and h[1]
        const float *hin = keep ? G.h[l - 1].p : G.h[(l - 1) & 1].p;
        float *hout = keep ? G.h[l].p : G.h[l & 1].p;
        if (l < 3 && keep) { k_layer<false><<<gr, kT, kLayerShared, st>>>(n, A.ptr.p, A.width.p, A.col.p, G.ahat.p, hin, G.theta_bf.p, off, G.g[l].p, G.pre[l].p, hout, G.edge_of.p, r, s->Dinv.p, G.isd.p, G.sc.p, z); note_launch(); }
        else if (l < 3) { k_layer_tc<false><<<gt, kT, 0, st>>>(n, A.ptr.p, A.width.p, A.col.p, G.ahat.p, hin, G.theta_bf.p, off, hout, G.edge_of.p, r, s->Dinv.p, G.isd.p, G.sc.p, z, nullptr, nullptr); note_launch(); }
        else if (keep) { k_layer<true><<<gr, kT, kLayerShared, st>>>(n, A.ptr.p, A.width.p, A.col.p, G.ahat.p, hin, G.theta_bf.p, off, G.g[l].p, G.pre[l].p, hout, G.edge_of.p, r, s->Dinv.p, G.isd.p, G.sc.p, z); note_launch(); }
        else { k_layer_tc<true><<<gt, kT, 0, st>>>(n, A.ptr.p, A.width.p, A.col.p, G.ahat.p, hin, G.theta_bf.p, off, hout, G.edge_of.p, r, s->Dinv.p, G.isd.p, G.sc.p, z, zo, dot_part); note_launch(); }
    }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

int gnn_forward(Sim *s, const double *r, double *z, bool keep) {
    return gnn_forward_dots(s, r, z, keep, 0, nullptr, nullptr, nullptr);
}

// loss and dL/dtheta (into G.grad, device) for residual r; loss -> G.sc[1]
int gnn_backward(Sim *s, const double *r, const double *z) {
    GnnState &G = s->gnn;
    const Mesh *m = s->mesh;
    const int n = m->n_int_edges;
    const DevSell &A = m->As;
    cudaStream_t st = s->stream;
    int rc;
    if (n == 0) {
        FP_CUDA(cudaMemsetAsync(G.grad.p, 0, sizeof(double) * kGnnParams, st));
        FP_CUDA(cudaMemsetAsync(G.sc.p + 1, 0, sizeof(double), st));
        return PIC_OK;
    }
    { k_gy<<<row_blocks(n), kT, 0, st>>>(n, A.n_slices, A.ptr.p, A.width.p, A.col.p, s->A_val.p, z, r, G.row_of.p, G.isd.p, G.sc.p, G.gy.p, G.part.p); note_launch(); }
    if ((rc = gnn_reduce_launch(s, 1, G.sc.p + 1, row_blocks(n)))) return rc;
    // dh of layer l lives in cur; the layer writes W^T dpre into nxt and Q^T dpre into tq
    float *cur = G.dh.p, *nxt = G.dh2.p;
    for (int l = 3; l >= 1; l--) {
        const int off = kOffL + (l - 1) * kLayer;
        float *wpart = G.wpart.p + (size_t)(l - 1) * kGB * kNA * 32;
        if (l == 3) { k_layer_bwd<true><<<kGB, kT, kBwdShared, st>>>(n, G.h[2].p, G.g[3].p, G.pre[3].p, G.h[3].p, nullptr, G.gy.p, G.theta_bf.p, off, nxt, G.tq.p, wpart); note_launch(); }
        else { k_layer_bwd<false><<<kGB, kT, kBwdShared, st>>>(n, G.h[l - 1].p, G.g[l].p, G.pre[l].p, G.h[l].p, cur, G.gy.p, G.theta_bf.p, off, nxt, G.tq.p, wpart); note_launch(); }
        { k_agg_bwd<<<tiles_grid(n), kT, 0, st>>>(n, G.rows.ptr.p, G.rows.width.p, G.rows.col.p, G.ahat.p, G.tq.p, nxt); note_launch(); }
        std::swap(cur, nxt);
    }
    { k_embed_bwd<<<kGB, kT, 0, st>>>(n, G.xin.p, G.feat_a.p, G.pre[0].p, cur, G.wpart.p + 3 * (size_t)kGB * kNA * 32); note_launch(); }
    { k_grad_final<<<kFinalBlocks, kT, 0, st>>>(G.wpart.p, G.dst.p, G.grad.p); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

int gnn_loss_grad(Sim *s, const double *r, double *loss, double *grad_host) {
    int rc;
    if ((rc = gnn_forward(s, r, s->gnn.z.p, true)) || (rc = gnn_backward(s, r, s->gnn.z.p))) return rc;
    double sc[2];
    FP_CUDA(cudaMemcpyAsync(sc, s->gnn.sc.p, sizeof(double) * 2, cudaMemcpyDeviceToHost, s->stream));
    if (grad_host)
        FP_CUDA(cudaMemcpyAsync(grad_host, s->gnn.grad.p, sizeof(double) * kGnnParams, cudaMemcpyDeviceToHost, s->stream));
    FP_CUDA(cudaStreamSynchronize(s->stream));
    if (loss) *loss = sc[0] > 0.0 ? sc[1] / sc[0] : 0.0;
    return PIC_OK;
}

int gnn_train(Sim *s, const pic_gnn_train_cfg *cfg, double *loss_out) {
    GnnState &G = s->gnn;
    const Mesh *m = s->mesh;
    const int n = m->n_int_edges;
    int rc;
    if ((rc = gnn_prepare(s))) return rc;
    if (n == 0) {
        if (loss_out) *loss_out = 0.0;
        return PIC_OK;
    }
    // residual samples: Jacobi-PCG on the last Newmark system from x = 0,
    // stopped after m iterations, m = 0, 1, 2, 4, ... (the residuals CG meets)
    const int ns = std::max(1, std::min(cfg->samples, 16));
    if ((rc = G.samples.alloc((size_t)ns * n))) return rc;
    for (int k = 0; k < ns; k++) {
        const int iters = k == 0 ? 0 : (1 << (k - 1));
        if ((rc = newmark_truncated_residual(s, iters, G.samples.p + (size_t)k * n))) return rc;
    }
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    double last = 0.0;
    for (int t = 0; t < cfg->steps; t++) {
        const double *r = G.samples.p + (size_t)(t % ns) * n;
        if ((rc = gnn_forward(s, r, G.z.p, true)) || (rc = gnn_backward(s, r, G.z.p))) return rc;
        G.adam_t++;
        const float c1 = 1.0f - std::pow(b1, (float)G.adam_t), c2 = 1.0f - std::pow(b2, (float)G.adam_t);
        { k_adam<<<(kGnnParams + 255) / 256, 256, 0, s->stream>>>(kGnnParams, G.theta.p, G.adam_m.p, G.adam_v.p, G.grad.p, (float)cfg->lr, b1, b2, eps, c1, c2, G.theta_bf.p); note_launch(); }
        FP_CUDA(cudaGetLastError());
    }
    // mean loss over the samples with the trained weights
    for (int k = 0; k < ns; k++) {
        double L = 0.0;
        if ((rc = gnn_loss_grad(s, G.samples.p + (size_t)k * n, &L, nullptr))) return rc;
        last += L / ns;
    }
    G.trained = 1;
    if (loss_out) *loss_out = last;
    return PIC_OK;
}

// Flexible PCG (Polak-Ribiere beta) on the Newmark system with the network
// as preconditioner; Jacobi takes over for the rest of the solve when the
// network's direction is not a descent direction (r.z <= 0 or not finite) or
// the residual stops falling for 20 iterations.
int fpcg_newmark(Sim *s, int *iters_out) {
    GnnState &G = s->gnn;
    const Mesh *m = s->mesh;
    const int n = m->n_int_edges;
    const DevSell &A = m->As;
    cudaStream_t st = s->stream;
    const int ge = (n + 255) / 256;
    int rc;
    double *b = s->rhs.p, *x = s->x.p, *r = G.r.p, *z = G.z.p, *zo = G.zold.p, *p = G.p.p, *q = G.q.p;
    auto dots = [&](const double *x1, const double *y1, const double *x2, const double *y2, double out[2]) -> int {
        { k_dot2<<<kGB, kT, 0, st>>>(n, x1, y1, x2, y2, nullptr, G.part.p); note_launch(); }
        int rc2 = gnn_reduce_launch(s, 2, G.sc.p + 4);
        if (rc2) return rc2;
        FP_CUDA(cudaMemcpyAsync(out, G.sc.p + 4, sizeof(double) * 2, cudaMemcpyDeviceToHost, st));
        FP_CUDA(cudaStreamSynchronize(st));
        return PIC_OK;
    };
    auto precond = [&](const double *rr, double *zz, bool jac) -> int {
        if (jac) {
            { k_jacobi<<<ge, 256, 0, st>>>(n, s->Dinv.p, rr, zz); note_launch(); }
            FP_CUDA(cudaGetLastError());
            return PIC_OK;
        }
        return gnn_forward(s, rr, zz, false);
    };
    { k_resid<<<row_blocks(n), kT, 0, st>>>(n, A.n_slices, A.ptr.p, A.width.p, A.col.p, s->A_val.p, b, x, r); note_launch(); }
    double bb_rr[2];
    if ((rc = dots(b, b, r, r, bb_rr))) return rc;
    const double bb = bb_rr[0], tol2 = s->cfg.cg_tol * s->cfg.cg_tol;
    double rr = bb_rr[1];
    int it = 0;
    bool jac = false;
    if (bb == 0.0) {
        FP_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n, st));
        *iters_out = 0;
        return PIC_OK;
    }
    if ((rc = precond(r, z, jac))) return rc;
    double rz[2];
    if ((rc = dots(r, z, nullptr, nullptr, rz))) return rc;
    if (!(rz[0] > 0.0) || !std::isfinite(rz[0])) {
        jac = true;
        if ((rc = precond(r, z, jac)) || (rc = dots(r, z, nullptr, nullptr, rz))) return rc;
    }
    double rzo = rz[0], best = rr;
    int since_best = 0;
    FP_CUDA(cudaMemcpyAsync(p, z, sizeof(double) * n, cudaMemcpyDeviceToDevice, st));
    while (!(rr <= tol2 * bb)) {
        if (it >= s->cfg.cg_max_iters) {
            s->host_status |= ST_CG_NO_CONV;
            set_error("flexible PCG did not reach the tolerance");
            return PIC_ERR_CG_NO_CONVERGENCE;
        }
        // x += alpha p, r -= alpha A p, alpha = r.z / p.A p: partial sums go
        // from kernel to kernel, and the host waits once an iteration
        const int rb = row_blocks(n);
        double *pq_part = G.part.p, *rr_part = pq_part + rb, *dot_part = rr_part + 2 * rb;
        { k_spmv_dot<<<rb, kT, 0, st>>>(n, A.n_slices, A.ptr.p, A.width.p, A.col.p, s->A_val.p, p, q, pq_part); note_launch(); }
        { k_fpcg_xr<<<rb, kT, 0, st>>>(n, rzo, rb, pq_part, p, q, s->Dinv.p, x, r, rr_part); note_launch(); }
        std::swap(z, zo);
        double d1[2], d2[2];
        if (jac) {
            if ((rc = precond(r, z, jac)) || (rc = dots(r, z, r, zo, d1)) || (rc = dots(r, r, nullptr, nullptr, d2))) return rc;
        } else {
            if ((rc = gnn_forward_dots(s, r, z, false, rb, rr_part + rb, zo, dot_part))) return rc;
            { k_fpcg_sums<<<1, 96, 0, st>>>(rb, rr_part, tc_grid(n), dot_part, G.sc.p + 4); note_launch(); }
            FP_CUDA(cudaGetLastError());
            double v[3];
            FP_CUDA(cudaMemcpyAsync(v, G.sc.p + 4, sizeof(v), cudaMemcpyDeviceToHost, st));
            FP_CUDA(cudaStreamSynchronize(st));
            d2[0] = v[0];
            d1[0] = v[1];
            d1[1] = v[2];
        }
        it++;
        rr = d2[0];
        bool restart = false;
        if (rr < best) {
            best = rr;
            since_best = 0;
        } else if (++since_best >= 20 && !jac) {
            jac = restart = true;
        }
        if (!jac && (!(d1[0] > 0.0) || !std::isfinite(d1[0]))) jac = restart = true;
        double beta;
        if (restart) {
            // Jacobi-PCG from here on, restarted along z = D^-1 r
            if ((rc = precond(r, z, true)) || (rc = dots(r, z, nullptr, nullptr, d1))) return rc;
            beta = 0.0;
            G.fell_back = 1;
        } else {
            beta = (d1[0] - d1[1]) / rzo;   // Polak-Ribiere
        }
        rzo = d1[0];
        { k_fpcg_p<<<ge, 256, 0, st>>>(n, beta, z, p); note_launch(); }
        FP_CUDA(cudaGetLastError());
    }
    *iters_out = it;
    return PIC_OK;
}

}  // namespace fp
