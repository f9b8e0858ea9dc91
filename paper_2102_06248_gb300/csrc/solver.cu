// solver.cu -- the field half of the step (Sec. II.B with Sec. III.A):
// Newmark right-hand side driven by Gbar, Jacobi-preconditioned CG on
// A = [*eps] + dt^2/4 [*S] (FP64, bandwidth-bound CSR), completion of the
// solve on the gradient subspace, Faraday update of b, and the conservation
// diagnostics.  All reductions run in a fixed order (deterministic).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "sim.h"
#include "stream.cuh"

namespace fp {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 152 * 16;             // 16 blocks of 256 threads per SM

// ---- deterministic block / grid reductions ----
template <int N>
__device__ __forceinline__ void block_sum(double v[N], double *sh /* [N][kThreads/32] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < N; c++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xFFFFFFFFu, v[c], o);
        if (lane == 0) sh[c * (kThreads / 32) + warp] = v[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < N; c++) {
            double s = 0.0;
            for (int w = 0; w < kThreads / 32; w++) s += sh[c * (kThreads / 32) + w];
            v[c] = s;
        }
    }
    __syncthreads();
}

template <int N>
__device__ __forceinline__ void block_max(double v[N], double *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < N; c++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[c] = fmax(v[c], __shfl_down_sync(0xFFFFFFFFu, v[c], o));
        if (lane == 0) sh[c * (kThreads / 32) + warp] = v[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < N; c++) {
            double s = 0.0;
            for (int w = 0; w < kThreads / 32; w++) s = fmax(s, sh[c * (kThreads / 32) + w]);
            v[c] = s;
        }
    }
    __syncthreads();
}

// Writes this block's N partials; returns true in the block that arrives
// last, after which all partials are visible to it.
template <int N>
__device__ __forceinline__ bool arrive(const double v[N], double *part, unsigned *counter) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < N; c++) part[(size_t)c * gridDim.x + blockIdx.x] = v[c];
        __threadfence();
        const unsigned t = atomicAdd(counter, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// in the last block: sum (or max) over all blocks' partials in block order
template <int N, bool MAX>
__device__ __forceinline__ void grid_combine(double out[N], const double *part, double *sh) {
#pragma unroll
    for (int c = 0; c < N; c++) {
        double s = 0.0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads) {
            const double v = ((volatile const double *)part)[(size_t)c * gridDim.x + b];
            s = MAX ? fmax(s, v) : s + v;
        }
        out[c] = s;
    }
    if (MAX) block_max<N>(out, sh);
    else block_sum<N>(out, sh);
}

// ---------------------------------------------------------------------------
// SELL-32 kernels on the Newmark pattern (thread per row, warp per slice):
// the 32 rows of a slice read their j-th entries as one coalesced 128-byte
// (columns) and 256-byte (values) access.
// ---------------------------------------------------------------------------
constexpr int kSlicesPerBlock = kThreads / 32;

#define SELL_LOOP(n_slices, n) SELL_LOOP_AT(n_slices, n, sp, sw)
#define SELL_LOOP_AT(n_slices, n, sp, sw)                                                              \
    const int lane = threadIdx.x & 31;                                                                 \
    for (int sl = blockIdx.x * kSlicesPerBlock + (threadIdx.x >> 5); sl < (n_slices);                 \
         sl += gridDim.x * kSlicesPerBlock) {                                                          \
        const int r = sl * 32 + lane;                                                                  \
        const bool rv = r < (n);                                                                       \
        const int kb = (sp)[sl] + lane, kw = (sw)[sl];

// face vector hb = H (b + b') (Newmark Maxwell form) or H b (backward
// difference, ONE_LEVEL)
template <bool ONE_LEVEL>
__global__ void __launch_bounds__(kThreads) k_face_hb(int n, int n_slices, const int *__restrict__ sp,
                                                      const int *__restrict__ sw, const int *__restrict__ col,
                                                      const double *__restrict__ Hv, const double *__restrict__ b,
                                                      const double *__restrict__ bp, double *__restrict__ hb) {
    SELL_LOOP(n_slices, n)
        double acc = 0.0;
#pragma unroll 4
        for (int j = 0; j < kw; j++) {
            const int k = kb + 32 * j, c = col[k];
            acc = fma(Hv[k], ONE_LEVEL ? b[c] : b[c] + bp[c], acc);
        }
        if (rv) hb[r] = acc;
    }
}

// Per-row combinations the SELL kernels below gather, formed once per row
// instead of once per stored entry (FP64 instructions are the scarce ones):
// x = 2e - e' (the predictor) and y = 2e + e'.
__global__ void k_rhs_pre(int n, const double *__restrict__ e, const double *__restrict__ ep, double *__restrict__ x,
                          double *__restrict__ y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const double ei = e[i], epi = ep[i];
        x[i] = fma(2.0, ei, -epi);
        y[i] = fma(2.0, ei, epi);
    }
}

// wave form: rhs = M (2e - e') - dt^2/4 K (2e + e') - (g^{n+1} - 2g^n + g^{n-1})
__global__ void __launch_bounds__(kThreads) k_rhs_we_sell(int n, int n_slices, const int *__restrict__ sp,
                                                          const int *__restrict__ sw, const int *__restrict__ col,
                                                          const double *__restrict__ Mv, const double *__restrict__ Kv,
                                                          double c4, const double *__restrict__ x,
                                                          const double *__restrict__ y, const double *__restrict__ gn,
                                                          const double *__restrict__ g, const double *__restrict__ gp,
                                                          double *__restrict__ rhs) {
    SELL_LOOP(n_slices, n)
        double sm = 0.0, sk = 0.0;
#pragma unroll 4
        for (int j = 0; j < kw; j++) {
            const int k = kb + 32 * j;
            const int c = col[k];
            sm = fma(Mv[k], x[c], sm);
            sk = fma(Kv[k], y[c], sk);
        }
        if (rv) rhs[r] = sm - c4 * sk - (gn[r] - 2.0 * g[r] + gp[r]);
    }
}

// Maxwell form: rhs = M e' - dt^2/4 K (2e + e') + dt C^T H (b + b') - (G^{n+1} - G^{n-1})
__global__ void __launch_bounds__(kThreads) k_rhs_mfem_sell(int n, int n_slices, const int *__restrict__ sp,
                                                            const int *__restrict__ sw, const int *__restrict__ col,
                                                            const double *__restrict__ Mv, const double *__restrict__ Kv,
                                                            double c4, double dt, const double *__restrict__ ep,
                                                            const double *__restrict__ y, const double *__restrict__ gn,
                                                            const double *__restrict__ gp, const int *__restrict__ efp,
                                                            const int *__restrict__ efc,
                                                            const signed char *__restrict__ efs,
                                                            const double *__restrict__ hb, double *__restrict__ rhs) {
    SELL_LOOP(n_slices, n)
        double sm = 0.0, sk = 0.0, sc = 0.0;
#pragma unroll 4
        for (int j = 0; j < kw; j++) {
            const int k = kb + 32 * j;
            const int c = col[k];
            sm = fma(Mv[k], ep[c], sm);
            sk = fma(Kv[k], y[c], sk);
        }
        if (rv) {
            for (int k = efp[r]; k < efp[r + 1]; k++) sc += (double)efs[k] * hb[efc[k]];
            rhs[r] = sm - c4 * sk + dt * sc - (gn[r] - gp[r]);
        }
    }
}

// backward difference: rhs = M e + dt C^T H b - (G^{n+1} - G^n)
__global__ void __launch_bounds__(kThreads) k_rhs_bd_sell(int n, int n_slices, const int *__restrict__ sp,
                                                          const int *__restrict__ sw, const int *__restrict__ col,
                                                          const double *__restrict__ Mv, double dt,
                                                          const double *__restrict__ e, const double *__restrict__ gn,
                                                          const double *__restrict__ g, const int *__restrict__ efp,
                                                          const int *__restrict__ efc,
                                                          const signed char *__restrict__ efs,
                                                          const double *__restrict__ hb, double *__restrict__ rhs) {
    SELL_LOOP(n_slices, n)
        double sm = 0.0, sc = 0.0;
#pragma unroll 4
        for (int j = 0; j < kw; j++) {
            const int k = kb + 32 * j;
            sm = fma(Mv[k], e[col[k]], sm);
        }
        if (rv) {
            for (int k = efp[r]; k < efp[r + 1]; k++) sc += (double)efs[k] * hb[efc[k]];
            rhs[r] = sm + dt * sc - (gn[r] - g[r]);
        }
    }
}

// absorbing walls: rhs += I (a u + c v) on the few rows with surface entries
// (wave form: a = dt/(2c), u = e', c = 0; Newmark Maxwell form: a = -dt/c,
// u = e, c = -dt/(2c), v = e')
__global__ void k_rhs_impedance(int nr, const int *__restrict__ row, const int *__restrict__ ptr,
                                const int *__restrict__ col, const double *__restrict__ val, double a,
                                const double *__restrict__ u, double c, const double *__restrict__ v,
                                double *__restrict__ rhs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nr) return;
    double su = 0.0, sv = 0.0;
    for (int k = ptr[i]; k < ptr[i + 1]; k++) {
        su = fma(val[k], u[col[k]], su);
        if (v) sv = fma(val[k], v[col[k]], sv);
    }
    rhs[row[i]] += a * su + c * sv;
}

// t = 2e - e' - x (wave form), e' - x (Newmark Maxwell form) or e - x
// (backward difference), formed once per row
__global__ void k_gc_t(int n, int form, const double *__restrict__ e, const double *__restrict__ ep,
                       const double *__restrict__ x, double *__restrict__ t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        t[i] = form == PIC_FORM_WE ? fma(2.0, e[i], -ep[i]) - x[i] : form == PIC_FORM_MFEM ? ep[i] - x[i] : e[i] - x[i];
}

// w = M t - (second difference of Gbar), t from k_gc_t
__global__ void __launch_bounds__(kThreads) k_gc_w_sell(int n, int n_slices, const int *__restrict__ sp,
                                                        const int *__restrict__ sw, const int *__restrict__ col,
                                                        const double *__restrict__ Mv, int form,
                                                        const double *__restrict__ t, const double *__restrict__ gn,
                                                        const double *__restrict__ g, const double *__restrict__ gp,
                                                        double *__restrict__ w) {
    SELL_LOOP(n_slices, n)
        double s = 0.0;
#pragma unroll 4
        for (int j = 0; j < kw; j++) {
            const int k = kb + 32 * j;
            s = fma(Mv[k], t[col[k]], s);
        }
        if (rv)
            w[r] = s - (form == PIC_FORM_WE ? gn[r] - 2.0 * g[r] + gp[r] : form == PIC_FORM_MFEM ? gn[r] - gp[r] : gn[r] - g[r]);
    }
}

// What a step's diagnostics read from the fields, in one launch: over the
// edges the true residual of the Newmark system and M e (kept for the node
// diagnostics), e^T M e; over the tets max |D b|; over the faces b^T H b; the
// push blocks' kinetic energies.  Every block takes its share of each, so the
// warps that stream the matrices (bound by FP64 and bytes) run beside those
// that gather, and one arrival of the blocks replaces four.
// (6^3 cube, a step of launches: 539 -> 514 us with the shorter sort.)
struct DiagArgs {
    // Newmark pattern
    int n, n_slices;
    const int *sp, *sw, *col;
    const double *Mv, *Kv, *Iv;
    double c4, ci;
    const double *x, *rhs;
    double *me;
    // tets
    int nt;
    const int4 *tf;
    const signed char *sign;
    // faces
    int nf, f_slices;
    const int *fp, *fw, *fcol;
    const double *Hv, *b;
    // push blocks
    int n_ke;
    const double *ke;
    double *part;
    DiagDev *dg;
};

template <bool IMPEDANCE>
__global__ void __launch_bounds__(kThreads) k_diag_fields(const DiagArgs a) {
    __shared__ double sh[5 * kThreads / 32];
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const int first = blockIdx.x * kThreads + threadIdx.x, stride = gridDim.x * kThreads;
    {
        SELL_LOOP_AT(a.n_slices, a.n, a.sp, a.sw)
            double sm = 0.0, sk = 0.0, si = 0.0;
#pragma unroll 4
            for (int j = 0; j < kw; j++) {
                const int k = kb + 32 * j;
                const double xj = a.x[a.col[k]];
                sm += a.Mv[k] * xj;
                sk += a.Kv[k] * xj;
                if (IMPEDANCE) si += a.Iv[k] * xj;
            }
            if (rv) {
                a.me[r] = sm;
                const double res = a.rhs[r] - (sm + a.c4 * sk + a.ci * si);
                acc[0] += res * res;
                acc[1] += a.rhs[r] * a.rhs[r];
                acc[2] += a.x[r] * sm;
            }
        }
    }
    {
        SELL_LOOP_AT(a.f_slices, a.nf, a.fp, a.fw)
            double s = 0.0;
#pragma unroll 4
            for (int j = 0; j < kw; j++) {
                const int k = kb + 32 * j;
                s = fma(a.Hv[k], a.b[a.fcol[k]], s);
            }
            if (rv) acc[3] = fma(a.b[r], s, acc[3]);
        }
    }
    for (int t = first; t < a.nt; t += stride) {
        const int4 f = a.tf[t];
        const double s = a.sign[t];
        acc[5] = fmax(acc[5], fabs(s * (a.b[f.x] - a.b[f.y] + a.b[f.z] - a.b[f.w])));
    }
    for (int p = first; p < a.n_ke; p += stride) acc[4] += a.ke[p];
    block_sum<5>(acc, sh);
    block_max<1>(acc + 5, sh);
    if (arrive<6>(acc, a.part, &a.dg->count)) {
        double tot[6];
        grid_combine<5, false>(tot, a.part, sh);
        grid_combine<1, true>(tot + 5, a.part + 5 * (size_t)gridDim.x, sh);
        if (threadIdx.x == 0) {
            if (a.n > 0) {
                a.dg->relres = tot[1] > 0.0 ? sqrt(tot[0] / tot[1]) : 0.0;
                a.dg->energy_e = 0.5 * tot[2];
            }
            a.dg->energy_b = 0.5 * tot[3];
            a.dg->energy_k = tot[4];
            a.dg->divb_abs = tot[5];
            a.dg->count = 0;
        }
    }
}

__global__ void k_recip_diag_mk(int n, const double *__restrict__ md, const double *__restrict__ kd, double c4,
                                const double *__restrict__ id, double ci, double *__restrict__ dinv) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dinv[i] = 1.0 / (md[i] + c4 * kd[i] + (id ? ci * id[i] : 0.0));
}

int grid_for_slices(int n_slices) {
    return std::max(1, std::min(kMaxBlocks, (n_slices + kSlicesPerBlock - 1) / kSlicesPerBlock));
}

// d_k = (G_int^T w)_k for interior node k
__global__ void k_gc_d(int nin, const int *__restrict__ int_node, const int *__restrict__ ptr,
                       const int *__restrict__ idx, const signed char *__restrict__ sgn, int n_int_edges,
                       const double *__restrict__ w, double *__restrict__ d) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nin) return;
    const int node = int_node[k];
    double s = 0.0;
    for (int a = ptr[node]; a < ptr[node + 1]; a++) {
        const int e = idx[a];
        if (e < n_int_edges) s += (double)sgn[a] * w[e];
    }
    d[k] = s;
}

// x_e += psi(head) - psi(tail) (psi = 0 on wall nodes)
__global__ void k_gc_apply(int n, const int2 *__restrict__ en, const int *__restrict__ node_int,
                           const double *__restrict__ psi, double *__restrict__ x) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int2 ab = en[e];
    const int ia = node_int[ab.x], ib = node_int[ab.y];
    x[e] += (ib >= 0 ? psi[ib] : 0.0) - (ia >= 0 ? psi[ia] : 0.0);
}

// e = -G phi on interior edges (initial electrostatic field)
__global__ void k_minus_grad(int n, const int2 *__restrict__ en, const int *__restrict__ node_int,
                             const double *__restrict__ phi_int, double *__restrict__ e, double *__restrict__ e2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int2 ab = en[i];
    const int ia = node_int[ab.x], ib = node_int[ab.y];
    const double v = -((ib >= 0 ? phi_int[ib] : 0.0) - (ia >= 0 ? phi_int[ia] : 0.0));
    e[i] = v;
    e2[i] = v;
}

// gather / scatter between node vectors and the interior-node compact vectors
__global__ void k_node_to_int(int nin, const int *__restrict__ int_node, const double *__restrict__ a,
                              const double *__restrict__ b, double *__restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nin) return;
    const int n = int_node[k];
    out[k] = a[n] + (b ? b[n] : 0.0);
}
__global__ void k_int_to_node(int nin, const int *__restrict__ int_node, const double *__restrict__ v,
                              double *__restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nin) return;
    out[int_node[k]] = v[k];
}


// Faraday: wave equation b^{n+1} = b^n - dt/2 C (e^{n+1} + e^n);
// Maxwell-solver row b^{n+1} = b^{n-1} - 2 dt C (e^{n+1}/4 + e^n/2 + e^{n-1}/4);
// backward difference b^{n+1} = b^n - dt C e^{n+1}
__global__ void k_faraday(int nf, const int4 *__restrict__ f2e, int form, double dt, const double *__restrict__ x,
                          const double *__restrict__ e, const double *__restrict__ ep, const double *__restrict__ b,
                          const double *__restrict__ bp, double *__restrict__ bn) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nf) return;
    const int4 t = f2e[f];
    const double cx = x[t.x] + x[t.y] - x[t.z];
    if (form == PIC_FORM_BD) {
        bn[f] = b[f] - dt * cx;
        return;
    }
    const double ce = e[t.x] + e[t.y] - e[t.z];
    if (form == PIC_FORM_WE) {
        bn[f] = b[f] - 0.5 * dt * (cx + ce);
    } else {
        const double cp = ep[t.x] + ep[t.y] - ep[t.z];
        bn[f] = bp[f] - 2.0 * dt * (0.25 * cx + 0.5 * ce + 0.25 * cp);
    }
}

// node diagnostics: continuity (all nodes), Gauss (interior nodes), charge scale
__global__ void __launch_bounds__(kThreads) k_diag_nodes(int nn, const int *__restrict__ ptr, const int *__restrict__ idx,
                                                         const signed char *__restrict__ sgn, int n_int_edges,
                                                         const double *__restrict__ dgv, const double *__restrict__ me,
                                                         const double *__restrict__ rho, const double *__restrict__ rho_p,
                                                         const double *__restrict__ wall, const double *__restrict__ wall_p,
                                                         const double *__restrict__ rho_bg,
                                                         const unsigned char *__restrict__ bnd, double *part, DiagDev *dg) {
    __shared__ double sh[3 * kThreads / 32];
    double acc[3] = {0.0, 0.0, 0.0};
    for (int n = blockIdx.x * kThreads + threadIdx.x; n < nn; n += gridDim.x * kThreads) {
        double gtd = 0.0, gme = 0.0;
        for (int a = ptr[n]; a < ptr[n + 1]; a++) {
            const int e = idx[a];
            const double s = (double)sgn[a];
            gtd += s * dgv[e];
            if (e < n_int_edges) gme += s * me[e];
        }
        const double q = rho[n] + wall[n];
        const double cont = q - (rho_p[n] + wall_p[n]) - gtd;
        acc[0] = fmax(acc[0], fabs(cont));
        if (!bnd[n]) acc[1] = fmax(acc[1], fabs(gme + q + rho_bg[n]));
        acc[2] = fmax(acc[2], fabs(q));
    }
    block_max<3>(acc, sh);
    if (arrive<3>(acc, part, &dg->count)) {
        double tot[3];
        grid_combine<3, true>(tot, part, sh);
        if (threadIdx.x == 0) {
            dg->cont_abs = tot[0];
            dg->gauss_abs = tot[1];
            dg->rho_max = tot[2];
            dg->count = 0;
        }
    }
}

// max_n |a_n + b_n| (deterministic; max is order-free)
__global__ void __launch_bounds__(kThreads) k_max_abs_sum(int n, const double *__restrict__ a, const double *__restrict__ b,
                                                          double *part, unsigned *counter, double *out) {
    __shared__ double sh[kThreads / 32];
    double acc[1] = {0.0};
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads)
        acc[0] = fmax(acc[0], fabs(a[i] + b[i]));
    block_max<1>(acc, sh);
    if (arrive<1>(acc, part, counter)) {
        double tot[1];
        grid_combine<1, true>(tot, part, sh);
        if (threadIdx.x == 0) {
            *out = tot[0];
            *counter = 0;
        }
    }
}

// ---------------------------------------------------------------------------
// Persistent Jacobi-PCG on a SELL-32 matrix (the Newmark operator A = M +
// dt^2/4 K on interior edges, and the node Laplacian G^T M G of the gradient
// completion and of the start-up solve).  One cooperative launch runs the whole
// solve.
//
// Sec. III leaves the linear solver open; this one is shaped by the FP64 rate
// of the part it runs on, which is far below its memory and FP32 rates, so the
// iteration is arranged to issue as few FP64 instructions as possible:
//  * the Chronopoulos-Gear recurrence of PCG: the SpMV acts on the
//    preconditioned residual u = D^-1 r alone (w = A u, one multiply-add per
//    stored entry), and the search direction's image s = A p follows from
//    s = w + beta s, so one global reduction per iteration yields
//    gamma = (r,u), delta = (w,u) and (r,r), from which
//    beta = gamma'/gamma and alpha = gamma'/(delta - beta gamma'/alpha);
//  * a reduction forms few FP64 sums, and the scalars of an iteration are
//    formed by one warp of each block (grid_reduce); max|r| travels as the bit
//    pattern of a nonnegative double, whose integer order is its numeric
//    order, so it costs no FP64 instruction.
// The matrix is streamed through shared memory by bulk copies (stream.cuh),
// each warp a contiguous run of slices.  Every thread owns the rows of its
// warp in the vector phase and in the SpMV; only the gathered vector (u, or the
// correction iterate) is read across blocks, by plain loads that L1 may keep:
// the grid barrier between the phases is a release/acquire pair, so they see
// the other blocks' writes.  The grid barriers are one release-add on a
// counter that only grows plus acquire-loads; every wait is bounded, past its
// bound the kernel records a timeout and every block leaves.
// Measured on the 64^3 plasma ball (1.8M rows, MIXED, 60 iterations): 4.44 ->
// 2.72 ms a solve, 45 us an iteration: the stream of 150 MB of records takes
// 22 us of them at the copy rate (it was 232 MB), the vector phase 4 us, the
// two barriers and the reduction 9 us.
// ---------------------------------------------------------------------------
constexpr int kMaxPcgBlocks = 4 * kThreads;    // most blocks of one solve
// Block (one per SM) and bytes of a warp's ring of a single solve: the FP64
// PCG and anything on wide records, and the refinement on narrow ones
template <bool REFINE, bool WIDE>
struct PcgShape {
    // (refinement, bound by the gathers that its warps have in flight: 512,
    // 768, 1024 threads 3.50, 2.79, 2.88 ms per Newmark solve of the 64^3
    // plasma ball, 128, 80, 64 registers; FP64, bound by the FP64 pipes: 512
    // and 768 threads 1.75 and 1.87 ms on 40^3)
    static constexpr int threads = REFINE && !WIDE ? 768 : 512;
    static constexpr int ring = REFINE && !WIDE ? 2 * Record<double, false>::bytes : 8192;
};
// block of the multigrid completion (one per SM; 512 threads: 1.81 ms against
// 1.44 ms on the 64^3 plasma ball, its phases wait on dependent loads)
constexpr int kMgThreads = 1024;
constexpr int kBatchRing = 2 * Record<double, false>::bytes;      // ... in the batched kernels
constexpr int kBatchRingWide = 2 * Record<double, true>::bytes;
// A matrix up to this size is left to stay in L2 between iterations, a larger
// one is loaded evict-first so that the vectors stay (FP32 records of 67, 74
// and 150 MB on the 48^3, 32x32x128 and 64^3 meshes: kept 4.40, 2.00, 3.92 ms
// a solve, evict-first 4.46, 1.95, 3.15 ms)
constexpr size_t kKeepInL2 = 70u << 20;
constexpr int kSlicesPerPcgBlock = 4;          // a small system takes a block per four slices
constexpr int kSmemSlices = 1024;              // slice widths a block keeps in shared memory
constexpr long kSpinLimit = 1L << 22;          // about a second of polling
constexpr int kMaxOuter = 12;                  // refinement steps of a mixed-precision solve
constexpr int kMaxInner = 400;                 // FP32 iterations per refinement step

__device__ __forceinline__ void red_release_add(unsigned int *p, unsigned int v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned int ld_acquire(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Spins (thread 0) until *p >= target; false when the bound or another
// block's timeout ends the wait.
__device__ __forceinline__ bool spin_until(GridBarrier *gb, const unsigned int *p, unsigned int target, long limit) {
    volatile int *vto = &gb->timeout;
    long spins = 0;
    while (ld_acquire(p) < target) {
        if (++spins > limit || ((spins & 255) == 0 && *vto != 0)) {
            atomicExch(&gb->timeout, 1);
            return false;
        }
    }
    return true;
}

// Barrier number `epoch` (1, 2, ... in every block) among the nb blocks of
// one solve: the counter reaches epoch * nb once every block has arrived.
__device__ __forceinline__ bool grid_barrier(GridBarrier *gb, unsigned int epoch, int nb, long limit) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_add(&gb->count, 1u);
        ok = spin_until(gb, &gb->count, epoch * (unsigned)nb, limit);
    }
    __syncthreads();
    return ok != 0;
}

__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

// Sum of a float over the warp, carried as hi + lo (every level an error-free
// sum): exact but for terms 2^-48 below the total, at the FP32 rate
__device__ __forceinline__ float2 warp_sum_f2(float v) {
    float hi = v, lo = 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float b = __shfl_xor_sync(0xFFFFFFFFu, hi, o), bl = __shfl_xor_sync(0xFFFFFFFFu, lo, o);
        const float t = __fadd_rn(hi, b), z = __fsub_rn(t, hi);
        const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(b, z));
        lo = __fadd_rn(__fadd_rn(lo, bl), e);
        hi = t;
    }
    return make_float2(hi, lo);
}

__device__ __forceinline__ void sync_four_warps() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// Reduction of NS sums and one maximum (kept as bits) over the nb blocks of
// one solve at barrier number `epoch` (this block, of T threads, is number
// bid; its first `active` warps hold something), in a fixed order.  What it
// costs is FP64 instructions and round trips to L2: each of an SM's four
// schedulers issues one warp-wide FP64 instruction per 64 cycles (its result
// comes after ~80; a division takes ~550), and a round trip is ~800 cycles.  So
//  * per quantity one warp of the block, each on its own scheduler, adds the
//    threads' values through shared memory and leaves the block's partial
//    (sums in part[c * nb + block], the maximum's bits in part[NS * nb + block]);
//    FP32 values are first added within their warps, as pairs of floats;
//  * after ONE barrier (arrival counter, 1.2 us at 152 blocks, 2.2 us at 608)
//    the first four warps of every block add all blocks' partials themselves, a
//    quantity each, instead of waiting for a last block that combines and
//    publishes them (two more round trips);
//  * warps 0 and 1 then run scal(t, warp, lane), t[0..NS) the sums and t[NS]
//    the maximum: the solver's scalars are formed by one warp, independent
//    divisions in different lanes, its tests by the other, and handed to the
//    block in shared memory.  (Formed by every thread, three divisions an
//    iteration held the FP64 pipes for ~9 us.)
template <int NS, int T, typename V, typename Scal>
__device__ __forceinline__ bool grid_reduce(GridBarrier *gb, double *part, const V v[NS], unsigned long long mx,
                                            double *shv, unsigned long long *shm, unsigned int epoch, int nb, int bid,
                                            int active, long limit, Scal scal) {
    __shared__ int ok;
    __shared__ double res[NS + 1];
    constexpr bool kF32 = std::is_same<V, float>::value;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    static_assert(NS <= 4 && T / 32 > NS && T >= 128, "one warp per quantity");
    // two sets of partials by parity: the next reduction may begin in a fast
    // block while a slow one still reads this one's
    part += (size_t)(epoch & 1u) * 5 * nb;
    if (warp < active) {
        if constexpr (kF32) {
            float hi = 0.0f, lo = 0.0f;
#pragma unroll
            for (int c = 0; c < NS; c++) {
                const float2 t = warp_sum_f2(v[c]);
                hi = lane == c ? t.x : hi;
                lo = lane == c ? t.y : lo;
            }
            if (lane < NS) shv[lane * 32 + warp] = (double)hi + (double)lo;
        } else {
#pragma unroll
            for (int c = 0; c < NS; c++) shv[c * T + threadIdx.x] = v[c];
            shm[threadIdx.x] = mx;
        }
    }
    __syncthreads();
    if (warp < NS) {
        double sum;
        if constexpr (kF32) {
            sum = warp_sum_d(lane < active ? shv[warp * 32 + lane] : 0.0);
        } else {
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            for (int k = 0; k < active; k += 4) {
#pragma unroll
                for (int h = 0; h < 4; h++)
                    if (k + h < active) s[h] += shv[warp * T + lane + 32 * (k + h)];
            }
            sum = warp_sum_d((s[0] + s[1]) + (s[2] + s[3]));
        }
        if (lane == 0) part[warp * nb + bid] = sum;
    } else if (!kF32 && warp == NS) {
        unsigned long long m = 0;
        for (int k = 0; k < active; k++) m = max(m, shm[lane + 32 * k]);
        m = warp_max_u64(m);
        if (lane == 0) part[NS * nb + bid] = __longlong_as_double((long long)m);
    }
    __syncthreads();
    if (warp < 4) {
        if (threadIdx.x == 0) {
            red_release_add(&gb->count, 1u);
            ok = spin_until(gb, &gb->count, epoch * (unsigned)nb, limit);
        }
        sync_four_warps();
        int good = ok;
        if (good) {
            // raised by a block that lost a copy (stream.cuh): everybody leaves
            const int lost = *(volatile int *)&gb->timeout;
            constexpr int kU = 5;   // 152 blocks: one trip, every load issued before the first sum
            if (warp < NS) {
                double t = 0.0;
                for (int b0 = lane; b0 < nb; b0 += 32 * kU) {
                    double p[kU];
#pragma unroll
                    for (int k = 0; k < kU; k++) p[k] = b0 + 32 * k < nb ? __ldcg(part + warp * nb + b0 + 32 * k) : 0.0;
                    t += ((p[0] + p[1]) + (p[2] + p[3])) + p[4];
                }
                t = warp_sum_d(t);
                if (lane == 0) res[warp] = t;
            }
            if (warp == (NS < 4 ? NS : 3)) {
                unsigned long long m = 0;
                if constexpr (!kF32) {
                    const unsigned long long *pm = reinterpret_cast<const unsigned long long *>(part) + NS * nb;
                    for (int b0 = lane; b0 < nb; b0 += 32 * kU) {
#pragma unroll
                        for (int k = 0; k < kU; k++)
                            if (b0 + 32 * k < nb) m = max(m, __ldcg(pm + b0 + 32 * k));
                    }
                    m = warp_max_u64(m);
                }
                if (lane == 0) res[NS] = __longlong_as_double((long long)m);
            }
            good = lost == 0;
        }
        sync_four_warps();
        if (warp < 2) {
            if (good) {
                double t[NS + 1];
#pragma unroll
                for (int c = 0; c <= NS; c++) t[c] = res[c];
                scal(t, warp, lane);
            } else if (threadIdx.x == 0) {
                ok = 0;
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

// Several independent solves share one launch: run r owns the blocks
// [block0, block0 + blocks) and synchronises them with its own barrier.
template <int MAXR>
struct PcgBatch {
    int n_runs;
    PcgArgs run[MAXR];
};

// Scalars of an iteration, formed by one thread of the block
struct CgScalars {
    double alpha, ralpha, rgamma, beta;   // in this order (lanes 0..3); ralpha = 1 / alpha, rgamma = 1 / gamma
    double gamma, rr, bb, stop;           // stop: r.r at which the solve ends
    float alpha32, beta32;
    int iters, done, failed;
};

// first slice whose offset sp[] is at least `target` (all lanes of a warp;
// 32 probes a round)
__device__ __forceinline__ int find_slice(const int *__restrict__ sp, int ns, long target) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = ns;
    while (lo < hi) {
        const int step = (hi - lo + 31) >> 5, p = lo + lane * step;
        const bool reached = p >= hi || sp[p] >= target;
        const int f = __ffs(__ballot_sync(0xFFFFFFFFu, reached)) - 1;   // 0..32 (-1: none)
        const int last = f < 0 ? 31 : f - 1;                            // the last probe below the target
        if (f >= 0) hi = min(hi, lo + f * step);
        if (last >= 0) lo = lo + last * step + 1;
    }
    return lo;
}

extern __shared__ __align__(128) unsigned char s_ring[];   // dynamic shared memory of the persistent kernels

// Per-block context of one solve.  The slices are dealt to the run's warps in
// contiguous runs of equal numbers of entries; of the block's T / 32 warps,
// `warps` take part (all of them unless the system has fewer slices than the
// run has warps: a small system is spread over the run's blocks first, since
// its iterations are bound by the latency and the FP64 rate of each SM).
template <bool WIDE, int T, int RING>
struct SolveCtx {
    template <typename V>
    using S = Stream<V, WIDE, RING>;
    using S64 = S<double>;
    using S32 = S<float>;
    const PcgArgs *a;
    int nb, bid, lane, warp, active;
    int slice0;                  // first slice of the block
    bool cached;                 // its slices' widths are in shared memory
    const unsigned short *s_width;
    double *shv;
    unsigned long long *shm;
    CgScalars *sc;
    unsigned int epoch;
    WarpStream ws;
    __device__ __forceinline__ int width(int sl) const { return cached ? (int)s_width[sl - slice0] : a->sw[sl]; }
    // (a copy that does not arrive raises the run's timeout flag, which every
    // block sees after the next grid reduction)
    template <typename V, typename F>
    __device__ __forceinline__ void spmv(const unsigned char *recs, const V *v, bool more, F f) {
        if (!S<V>::pass(ws, recs, v, more, [&](int sl) { return width(sl); }, f) && lane == 0)
            atomicExch(&a->gb->timeout, 1);
    }
};

// 16 bytes of a vector: four FP32 or two FP64 consecutive rows of one lane
template <typename V>
struct Pack {
    static constexpr int n = 16 / (int)sizeof(V);
    V v[n];
    __device__ __forceinline__ void load(const V *p) {
        const int4 t = *reinterpret_cast<const int4 *>(p);
        memcpy(v, &t, 16);
    }
    __device__ __forceinline__ void store(V *p) const {
        int4 t;
        memcpy(&t, v, 16);
        *reinterpret_cast<int4 *>(p) = t;
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < n; k++) v[k] = 0;
    }
};

// Chronopoulos-Gear Jacobi-PCG on the context's matrix (records in precision
// V): x, r, u = D^-1 r, w = A u, p, s = A p.  With UNIT the matrix has a unit
// diagonal (a diagonally scaled system): u is r itself (the caller passes r
// for u), and neither D^-1 nor u is read or written.  Per-thread sums are kept
// in V and the block and grid reductions in FP64 (in FP32 the per-thread sums
// cover a few dozen rows, in four chains).  max|r| is tracked in FP64 only.
// The stream of the records is running (begun by the caller, which also ends
// it); the results are left in the context's scalars.  Returns false if a
// wait ran out.
template <typename V, bool UNIT, bool WIDE, int T, int RING>
__device__ __forceinline__ bool cg_core(SolveCtx<WIDE, T, RING> &c, const unsigned char *recs,
                                        const V *__restrict__ Dinv, const V *b, V *x, V *r, V *u, V *w, V *p, V *s,
                                        bool x_zero, double tol2, double abs_inf, int max_iters) {
    constexpr bool kF64 = std::is_same<V, double>::value;
    constexpr int E = Pack<V>::n;
    const PcgArgs &a = *c.a;
    CgScalars *sc = c.sc;
    const int row0 = 32 * c.ws.s0 + E * c.lane, row1 = 32 * c.ws.s1;   // the lane's packs: row0, row0 + 32 E, ...
    {
        V v[4] = {0, 0, 0, 0};   // gamma, rr, delta, bb
        unsigned long long mx = 0;
        auto init_row = [&](int i, V bi, V ri) {
            V ui;
            if constexpr (UNIT) ui = ri;
            else ui = Dinv[i] * ri;
            r[i] = ri;
            if constexpr (!UNIT) u[i] = ui;
            v[0] = fma(ri, ui, v[0]);
            v[1] = fma(ri, ri, v[1]);
            v[3] = fma(bi, bi, v[3]);
            if constexpr (kF64) mx = max(mx, abs_bits(ri));
        };
        if (x_zero) {
            for (int i = 32 * c.ws.s0 + c.lane; i < row1; i += 32) {
                const V bi = b[i];
                x[i] = 0;
                init_row(i, bi, bi);
            }
        } else {
            c.template spmv<V>(recs, x, true, [&](int i, V ax, V) {
                const V bi = b[i];
                init_row(i, bi, bi - ax);
            });
        }
        if (!grid_barrier(a.gb, ++c.epoch, c.nb, a.spin_limit)) return false;
        c.template spmv<V>(recs, u, true, [&](int i, V au, V ui) {
            w[i] = au;
            v[2] = fma(au, ui, v[2]);
        });
        if (!grid_reduce<4, T>(a.gb, a.part, v, mx, c.shv, c.shm, ++c.epoch, c.nb, c.bid, c.active, a.spin_limit,
                               [&](const double *t, int wp, int l) {
                                   if (wp == 0) {
                                       const double q = (l == 0 ? t[0] : l == 1 ? t[2] : 1.0) / (l == 0 ? t[2] : t[0]);
                                       if (l < 3) (&sc->alpha)[l] = q;
                                       if (l == 0) sc->alpha32 = (float)q;
                                   } else if (l == 0) {
                                       sc->beta = 0.0;
                                       sc->beta32 = 0.0f;
                                       sc->gamma = t[0];
                                       sc->rr = t[1];
                                       sc->bb = t[3];
                                       sc->stop = tol2 * t[3];
                                       sc->iters = 0;
                                       sc->failed = 0;
                                       sc->done = (t[3] == 0.0) || (t[1] <= sc->stop) || (t[4] <= abs_inf);
                                       if (!sc->done && max_iters <= 0) sc->done = sc->failed = 1;
                                   }
                               }))
            return false;
    }
    if (sc->bb == 0.0)
        for (int i = 32 * c.ws.s0 + c.lane; i < row1; i += 32) x[i] = 0;
    while (!sc->done) {
        const bool first = sc->iters == 0;
        V al, be;
        if constexpr (kF64) {
            al = sc->alpha;
            be = sc->beta;
        } else {
            al = sc->alpha32;
            be = sc->beta32;
        }
        // ---- p = u + beta p, s = w + beta s, x += alpha p, r -= alpha s, u = D^-1 r ----
        // 16 bytes a load, every load before the first store
        V vg[E], vr[E];   // gamma, rr: a chain per element of the pack
#pragma unroll
        for (int k = 0; k < E; k++) vg[k] = vr[k] = 0;
        unsigned long long mx = 0;
#pragma unroll 2
        for (int i = row0; i < row1; i += 32 * E) {
            Pack<V> qu, qw, qp, qs, qx, qr, qd;
            qw.load(w + i);
            qr.load(r + i);
            qx.load(x + i);
            qp.zero();
            qs.zero();
            if (!first) {
                qp.load(p + i);
                qs.load(s + i);
            }
            if constexpr (UNIT) {
                qu = qr;
            } else {
                qu.load(u + i);
                qd.load(Dinv + i);
            }
#pragma unroll
            for (int k = 0; k < E; k++) {
                const V pi = first ? qu.v[k] : fma(be, qp.v[k], qu.v[k]);
                const V si = first ? qw.v[k] : fma(be, qs.v[k], qw.v[k]);
                const V ri = fma(-al, si, qr.v[k]);
                V un;
                if constexpr (UNIT) un = ri;
                else un = qd.v[k] * ri;
                qp.v[k] = pi;
                qs.v[k] = si;
                qx.v[k] = fma(al, pi, qx.v[k]);
                qr.v[k] = ri;
                qu.v[k] = un;
                vg[k] = fma(ri, un, vg[k]);
                vr[k] = fma(ri, ri, vr[k]);
                if constexpr (kF64) mx = max(mx, abs_bits(ri));
            }
            qp.store(p + i);
            qs.store(s + i);
            qx.store(x + i);
            qr.store(r + i);
            if constexpr (!UNIT) qu.store(u + i);
        }
        if (!grid_barrier(a.gb, ++c.epoch, c.nb, a.spin_limit)) return false;
        // ---- w = A u ----
        V v2 = 0;   // delta
        c.template spmv<V>(recs, u, true, [&](int i, V au, V ui) {
            w[i] = au;
            v2 = fma(au, ui, v2);
        });
        V vd[3];
        if constexpr (UNIT) {   // u is r: gamma is rr
            vd[0] = (vg[0] + vg[1]) + (vg[2] + vg[3]);
            vd[1] = vd[0];
        } else {
            vd[0] = vg[0] + vg[1];
            vd[1] = vr[0] + vr[1];
        }
        vd[2] = v2;
        // beta = gamma'/gamma, alpha = gamma' / (delta - beta gamma' / alpha)
        if (!grid_reduce<3, T>(a.gb, a.part, vd, mx, c.shv, c.shm, ++c.epoch, c.nb, c.bid, c.active, a.spin_limit,
                               [&](const double *t, int wp, int l) {
                                   if (wp == 0) {
                                       const double be = t[0] * sc->rgamma, den = t[2] - be * t[0] * sc->ralpha;
                                       __syncwarp();
                                       const double q = (l == 0 ? t[0] : l == 1 ? den : 1.0) / (l == 0 ? den : t[0]);
                                       const double o = l == 3 ? be : q;
                                       if (l < 4) (&sc->alpha)[l] = o;
                                       const float f = (float)o;
                                       if (l == 0) sc->alpha32 = f;
                                       if (l == 3) sc->beta32 = f;
                                   } else if (l == 0) {
                                       sc->gamma = t[0];
                                       sc->rr = t[1];
                                       const int it = ++sc->iters;
                                       int done = (t[1] <= sc->stop) || (t[3] <= abs_inf);
                                       if (!done && it >= max_iters) done = sc->failed = 1;
                                       sc->done = done;
                                   }
                               }))
            return false;
    }
    return true;
}

// the whole solve, run by block `bid` (T threads) of the nb blocks that own
// it: FP64 PCG (REFINE false) or the MIXED refinement (REFINE true, a.refine
// set).  The two are separate kernels so that each gets the register
// allocation of its own loops.  ring: RING bytes of shared memory per warp.
template <bool REFINE, bool WIDE, int T, int RING>
__device__ __forceinline__ void pcg_body(const PcgArgs &a, const int nb, const int bid, unsigned char *ring, double *shv,
                                         unsigned long long *shm) {
    constexpr int W = T / 32;
    __shared__ unsigned short s_width[kSmemSlices];
    __shared__ __align__(8) unsigned long long s_bars[W][kStreamBars];
    __shared__ CgScalars scal;
    __shared__ int s_range[2];
    struct Refine {
        double rr, bb, sigma, inv;
        int stop, failed, total;
    };
    __shared__ Refine rf;
    using Ctx = SolveCtx<WIDE, T, RING>;
    Ctx c;
    c.a = &a;
    c.nb = nb;
    c.bid = bid;
    c.lane = threadIdx.x & 31;
    c.warp = threadIdx.x >> 5;
    c.shv = shv;
    c.shm = shm;
    c.sc = &scal;
    c.epoch = 0;
    {
        const int warps = min(W, (a.n_slices + nb - 1) / nb);   // the block's warps that take part
        const int gw = bid * warps + c.warp, total = nb * warps;
        const long cols = a.sp[a.n_slices] >> 5;
        c.active = warps;
        WarpStream &w = c.ws;
        w.s0 = w.s1 = w.rec0 = w.nrec = w.skip = w.stage = w.inflight = w.next = 0;
        w.parity = 0;
        if (c.warp < warps) {
            w.s0 = find_slice(a.sp, a.n_slices, cols * gw / total * 32);
            w.s1 = find_slice(a.sp, a.n_slices, cols * (gw + 1) / total * 32);
            if (w.s1 > w.s0) {
                const int k0 = a.sp[w.s0] >> 5, k1 = a.sp[w.s1] >> 5;
                w.rec0 = k0 / kCols;
                w.nrec = (k1 + kCols - 1) / kCols - w.rec0;
                w.skip = k0 - w.rec0 * kCols;
            }
        }
        w.ring = smem_u32(ring) + (uint32_t)(c.warp * RING);
        w.bars = smem_u32(&s_bars[c.warp][0]);
        w.policy = a.evict_first ? policy_evict_first() : policy_evict_normal();
        if (c.lane == 0 && c.warp == 0) s_range[0] = w.s0;
        if (c.lane == 0 && c.warp == warps - 1) s_range[1] = w.s1;
        __syncthreads();
        c.slice0 = s_range[0];
        c.cached = s_range[1] - s_range[0] <= kSmemSlices;
        c.s_width = s_width;
        if (c.cached)
            for (int sl = w.s0 + c.lane; sl < w.s1; sl += 32) s_width[sl - c.slice0] = (unsigned short)a.sw[sl];
        __syncwarp();
    }
    CgState *st = a.st;
    double abs_inf = a.abs_inf, tol2 = a.tol2;
    if (a.abs_src) {
        const double qv = *a.abs_src;
        if (qv > 0.0) abs_inf = a.abs_factor * qv;
        else tol2 = a.fallback_tol2;
    }
    int outer = 0;
    bool good = true;
    if constexpr (!REFINE) {
        Ctx::S64::begin(c.ws, a.rec, 1 << 30);
        good = cg_core<double, false, WIDE, T, RING>(c, a.rec, a.Dinv, a.b, a.x, a.r, a.u, a.w, a.p, a.s, a.x_zero != 0,
                                                     tol2, abs_inf, a.max_iters);
        good = Ctx::S64::end(c.ws) && good;
    } else {
        // Iterative refinement: the FP64 residual b - A x decides; each
        // correction A d = r / sigma is solved in FP32 (values and vectors) to
        // a relative residual of inner_tol, and x += sigma d in FP64.  The
        // correction solve is plain CG on the scaled system
        // (D^-1/2 A D^-1/2) dh = D^-1/2 r / sigma, d = D^-1/2 dh: the same
        // iterates as Jacobi-PCG on A without the D^-1 and u vectors.  sigma,
        // the RMS of the residual, keeps the FP32 vectors near 1: in SI units
        // the residuals are far below 1 and their squares would reach the
        // FP32 subnormal range.  (Stopping a correction solve at what the
        // stopping rule still asks saves FP32 iterations but leaves the
        // completion more to do, at a higher price per order of magnitude.)
        const int n = a.n, row0 = 32 * c.ws.s0 + c.lane, row1 = 32 * c.ws.s1;
        if (threadIdx.x == 0) {
            rf.failed = 0;
            rf.total = 0;
        }
        while (true) {
            Ctx::S64::begin(c.ws, a.rec, c.ws.nrec);   // on its way while the blocks meet
            if (outer > 0 && good) good = grid_barrier(a.gb, ++c.epoch, nb, a.spin_limit);   // x complete
            if (good) {
                double v2[2] = {0.0, 0.0};
                c.template spmv<double>(a.rec, a.x, false, [&](int i, double ax, double) {
                    const double bi = a.b[i], ri = bi - ax;
                    a.r[i] = ri;
                    v2[0] = fma(ri, ri, v2[0]);
                    v2[1] = fma(bi, bi, v2[1]);
                });
                good = grid_reduce<2, T>(a.gb, a.part, v2, 0ull, shv, shm, ++c.epoch, nb, bid, c.active, a.spin_limit,
                                         [&](const double *t, int wp, int l) {
                                             if (wp + l != 0) return;
                                             rf.rr = t[0];
                                             rf.bb = t[1];
                                             rf.stop = t[1] == 0.0 || t[0] <= tol2 * t[1];
                                             if (!rf.stop && (rf.total >= a.max_iters || outer >= kMaxOuter))
                                                 rf.stop = rf.failed = 1;
                                             rf.sigma = sqrt(t[0] / n);
                                             rf.inv = 1.0 / rf.sigma;
                                         });
            }
            good = Ctx::S64::end(c.ws) && good;
            if (!good || rf.stop) break;
            Ctx::S32::begin(c.ws, a.rec32, 1 << 30);
            const double sigma = rf.sigma, inv = rf.inv;
            for (int i = row0; i < row1; i += 32) a.b32[i] = (float)(a.r[i] * inv) * a.Dhalf32[i];
            good = cg_core<float, true, WIDE, T, RING>(c, a.rec32, a.Dhalf32, a.b32, a.d32, a.r32, a.r32, a.w32, a.p32,
                                                       a.s32, true, a.inner_tol2, -1.0,
                                                       min(kMaxInner, a.max_iters - rf.total));
            good = Ctx::S32::end(c.ws) && good;
            if (!good) break;
            outer++;
            for (int i = row0; i < row1; i += 32)
                a.x[i] = fma(sigma * (double)a.Dhalf32[i], (double)a.d32[i], a.x[i]);
            __syncthreads();   // every thread has read rf.total
            if (threadIdx.x == 0) rf.total += scal.iters;
        }
        if (good && rf.bb == 0.0)
            for (int i = row0; i < row1; i += 32) a.x[i] = 0.0;
    }
    if (bid == 0 && threadIdx.x == 0) {
        if (!good) {
            st->done = 1;
            st->failed = 1;
            atomicOr(a.status, (uint32_t)ST_BARRIER);
            return;
        }
        const int failed = REFINE ? rf.failed : scal.failed;
        st->iters = REFINE ? rf.total : scal.iters;
        st->outer = outer;
        st->rr = REFINE ? rf.rr : scal.rr;
        st->rz = REFINE ? 0.0 : scal.gamma;
        st->bb = REFINE ? rf.bb : scal.bb;
        st->done = 1;
        st->failed = failed;
        if (failed && !a.quiet) atomicOr(a.status, (uint32_t)ST_CG_NO_CONV);
    }
}

// ---------------------------------------------------------------------------
// FP64 PCG on a system small enough for one SELL slice per warp (the fields of
// small meshes, their node Laplacians).  Such an iteration is a chain of
// latencies: two meetings of the blocks, the FP64 instructions of the
// reduction and of the scalars, loads of vectors from L2.  So
//  * a lane keeps its row of every vector in registers and the warp its
//    slice's entries in shared memory for the whole solve; only the vector the
//    product gathers goes through L2;
//  * the recurrence is the pipelined one (Ghysels and Vanroose, "Hiding global
//    synchronization latency in the preconditioned Conjugate Gradient
//    algorithm", 2014): with m = D^-1 w and n = A m it needs one meeting of
//    the blocks per iteration, and n does not wait for the scalars, so the
//    product runs while four more warps of the block add the partials and form
//    the scalars;
//  * its rounding errors grow with the condition number where those of the
//    recurrence with two meetings (cg_core) do not: at 24^3 cells of sides
//    1 : 10 : 100 and a tolerance of 1e-13, or at 300 times the explicit time
//    step and 1e-10, its residual stops falling above the tolerance or parts from
//    b - A x.  So it ends when its residual has not fallen for kSmallStall
//    iterations (13 in a row at most in systems where it converged), a solution
//    that it ends with counts once b - A x itself meets the rule, and otherwise the
//    recurrence with two meetings goes on from there, with max_iters
//    iterations of its own.  Tolerances below kSmallTol2 (absolute ones
//    against the largest entry of b) take that one from the start.
// Per iteration, streamed form and this: 20^3 (52,460 rows) 12.2 and 7.5 us,
// 16^3 (26,416 rows) 10.7 and 7.1 us, 6^3 (1,206 rows) 9.6 and 6.2 us.
// ---------------------------------------------------------------------------
constexpr int kSmallWarps = 12;               // slices of a block; four more warps reduce
constexpr int kSmallThreads = 32 * (kSmallWarps + 4);
constexpr int kSmallWidth = 32;               // columns of a slice held in shared memory
constexpr int kSmallSlice = kSmallWidth * 32 * 12;
constexpr int kSmallStall = 32;
constexpr double kSmallAim2 = 0.96;           // the pipelined recurrence aims 2% below the tolerance (squared)
constexpr double kSmallTol2 = 0.9e-26;        // smallest relative tolerance (squared) of the pipelined recurrence
constexpr int kSmallBlocks = 160;             // partials a warp adds with five loads a lane

// the whole solve, run by block `bid` of the nb blocks that own it
__device__ __forceinline__ void small_body(const PcgArgs &a, const int nb, const int bid) {
    __shared__ double shv[3][kSmallWarps * 32];
    __shared__ unsigned long long shm[kSmallWarps * 32];
    __shared__ double res[4];
    struct Scalars {
        double alpha, ralpha, rgamma, beta;   // in this order (lanes 0..3)
        double gamma, rr, bb, stop, abs_inf, tol2, best;
        int iters, limit, since, fresh, plain, done, failed, ok;
    };
    __shared__ Scalars sc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (a.n_slices + nb - 1) / nb;              // slices of a block
    const int sl = bid * per + warp;
    const bool holds = warp < per && sl < a.n_slices;        // this warp has a slice
    const int active = min(per, a.n_slices - bid * per);     // warps of the block that have one
    const int i = sl * 32 + lane;
    double *sv = reinterpret_cast<double *>(s_ring + (size_t)warp * kSmallSlice);
    int *scol = reinterpret_cast<int *>(sv + kSmallWidth * 32);
    int width = 0;
    double x = 0, r = 0, u = 0, w = 0, m = 0, p = 0, s = 0, q = 0, z = 0, d = 0, b = 0;
    if (holds) {
        const int k0 = a.sp[sl];
        width = a.sw[sl];
        for (int j = 0; j < width; j++) {
            sv[32 * j + lane] = a.Av[k0 + 32 * j + lane];
            scol[32 * j + lane] = a.col[k0 + 32 * j + lane];
        }
        b = a.b[i];
        d = a.Dinv[i];
        if (!a.x_zero) x = a.x[i];
    }
    if (threadIdx.x == 0) {
        sc.abs_inf = a.abs_inf;
        sc.tol2 = a.tol2;
        if (a.abs_src) {
            const double qv = *a.abs_src;
            if (qv > 0.0) sc.abs_inf = a.abs_factor * qv;
            else sc.tol2 = a.fallback_tol2;
        }
        sc.iters = sc.done = sc.failed = sc.plain = 0;
        sc.limit = a.max_iters;
        sc.fresh = 1;
    }
    unsigned int epoch = 0;
    // row of A v: two chains, every gather of 24 columns in flight at once
    auto spmv = [&](const double *v) -> double {
        double s0 = 0, s1 = 0;
        for (int j0 = 0; j0 < width; j0 += 24) {
            double g[24];
#pragma unroll
            for (int j = 0; j < 24; j++) g[j] = j0 + j < width ? v[scol[32 * (j0 + j) + lane]] : 0.0;
#pragma unroll
            for (int j = 0; j < 24; j += 2) {
                if (j0 + j < width) s0 = fma(sv[32 * (j0 + j) + lane], g[j], s0);
                if (j0 + j + 1 < width) s1 = fma(sv[32 * (j0 + j + 1) + lane], g[j + 1], s1);
            }
        }
        return s0 + s1;
    };
    // meets the other blocks (all threads of the block; the reducing warps wait for them)
    auto meet = [&]() -> bool {
        __syncthreads();
        epoch++;
        if (threadIdx.x == 32 * kSmallWarps) {
            red_release_add(&a.gb->count, 1u);
            sc.ok = spin_until(a.gb, &a.gb->count, epoch * (unsigned)nb, a.spin_limit);
        }
        __syncthreads();
        return sc.ok != 0;
    };
    // meets the other blocks with three sums and a maximum; work() runs in the
    // slices' warps while the others add the partials and run scal(t, warp, lane)
    auto reduce = [&](double v0, double v1, double v2, double vm, auto work, auto scal) -> bool {
        if (warp < kSmallWarps) {
            const int t = threadIdx.x;
            shv[0][t] = v0;
            shv[1][t] = v1;
            shv[2][t] = v2;
            shm[t] = abs_bits(vm);
        }
        __syncthreads();
        epoch++;
        double *part = a.part + (size_t)(epoch & 1u) * 4 * nb;
        const int dw = warp - kSmallWarps;
        if (dw >= 0) {
            if (dw < 3) {
                double c[4] = {0, 0, 0, 0};
#pragma unroll
                for (int k = 0; k < kSmallWarps; k++)
                    if (k < active) c[k & 3] += shv[dw][32 * k + lane];
                const double t = warp_sum_d((c[0] + c[1]) + (c[2] + c[3]));
                if (lane == 0) part[dw * nb + bid] = t;
            } else {
                unsigned long long t = 0;
                for (int k = 0; k < active; k++) t = max(t, shm[32 * k + lane]);
                t = warp_max_u64(t);
                if (lane == 0) part[3 * nb + bid] = __longlong_as_double((long long)t);
            }
            sync_four_warps();
            if (threadIdx.x == 32 * kSmallWarps) {
                red_release_add(&a.gb->count, 1u);
                sc.ok = spin_until(a.gb, &a.gb->count, epoch * (unsigned)nb, a.spin_limit);
            }
            sync_four_warps();
        }
        __syncthreads();
        if (!sc.ok) return false;
        if (dw < 0) {
            work();
        } else {
            double c[5];
#pragma unroll
            for (int k = 0; k < 5; k++) c[k] = lane + 32 * k < nb ? __ldcg(part + dw * nb + lane + 32 * k) : 0.0;
            if (dw < 3) {
                const double t = warp_sum_d(((c[0] + c[1]) + (c[2] + c[3])) + c[4]);
                if (lane == 0) res[dw] = t;
            } else {
                unsigned long long t = 0;
#pragma unroll
                for (int k = 0; k < 5; k++) t = max(t, (unsigned long long)__double_as_longlong(c[k]));
                t = warp_max_u64(t);
                if (lane == 0) res[3] = __longlong_as_double((long long)t);
            }
            sync_four_warps();
            if (dw < 2) {
                const double t[4] = {res[0], res[1], res[2], res[3]};
                scal(t, dw, lane);
            }
        }
        __syncthreads();
        return true;
    };
    // meets with (r, u), |r|^2, (w, u) and max|r|: the next alpha and beta of
    // either recurrence, and its tests
    auto advance = [&](auto work) -> bool {
        return reduce(r * u, r * r, w * u, r, work, [&](const double *t, int wp, int l) {
            if (wp == 0) {
                const double be = sc.fresh ? 0.0 : t[0] * sc.rgamma;
                const double den = sc.fresh ? t[2] : t[2] - be * t[0] * sc.ralpha;
                __syncwarp();
                const double o = (l == 0 ? t[0] : l == 1 ? den : 1.0) / (l == 0 ? den : t[0]);
                if (l < 4) (&sc.alpha)[l] = l == 3 ? be : o;
            } else if (l == 0) {
                const double aim = sc.plain ? 1.0 : kSmallAim2, aim_inf = sc.plain ? 1.0 : 0.98;
                sc.gamma = t[0];
                sc.rr = t[1];
                int done = sc.bb == 0.0 || t[1] <= aim * sc.stop || t[3] <= aim_inf * sc.abs_inf;
                if (!done && sc.iters >= sc.limit) {
                    done = 1;
                    sc.failed = !(t[1] <= sc.stop || t[3] <= sc.abs_inf);
                }
                if (!done && !sc.plain) {
                    const bool falls = t[1] < sc.best;
                    sc.best = falls ? t[1] : sc.best;
                    sc.since = falls ? 0 : sc.since + 1;
                    done = sc.since >= kSmallStall;
                }
                sc.done = done;
            }
        });
    };
    double *buf[2] = {a.u, a.w};
    int turn = 0;
    bool good = true;
    const double x0 = x;
    // r = b - A x (x in memory, complete in every block)
    if (holds) r = a.x_zero ? b : b - spmv(a.x);
    while (true) {
        // from r: u = D^-1 r, w = A u, no directions yet
        u = d * r;
        p = s = q = z = 0;
        if (holds) buf[turn][i] = u;
        good = reduce(b * b, 0.0, 0.0, b, [&]() { if (holds) w = spmv(buf[turn]); },
                      [&](const double *t, int wp, int l) {
                          if (wp + l == 0) {
                              sc.bb = t[0];
                              sc.stop = sc.tol2 * t[0];
                              sc.best = 1.7976931348623157e308;
                              sc.since = 0;
                              if (sc.tol2 < kSmallTol2 && !(sc.abs_inf > 0.0 && sc.abs_inf * sc.abs_inf >= kSmallTol2 * t[3] * t[3]))
                                  sc.plain = 1;
                          }
                      });
        if (!good) break;
        turn ^= 1;
        const bool plain = sc.plain != 0;
        if (plain) good = advance([]() {});
        while (good) {
            double n = 0;
            if (plain) {
                if (sc.done) break;
            } else {
                m = d * w;
                if (holds) buf[turn][i] = m;
                good = advance([&]() { if (holds) n = spmv(buf[turn]); });
                if (!good || sc.done) break;
                turn ^= 1;
            }
            const double al = sc.alpha, be = sc.beta;
            s = fma(be, s, w);
            p = fma(be, p, u);
            x = fma(al, p, x);
            r = fma(-al, s, r);
            if (!plain) {
                z = fma(be, z, n);
                q = fma(be, q, m);
                u = fma(-al, q, u);
                w = fma(-al, z, w);
            }
            if (threadIdx.x == 0) {
                sc.iters++;
                sc.fresh = 0;
            }
            if (plain) {
                u = d * r;
                if (holds) buf[turn][i] = u;
                if (!(good = meet())) break;
                if (holds) w = spmv(buf[turn]);
                turn ^= 1;
                good = advance([]() {});
            }
        }
        if (!good) break;
        if (sc.bb == 0.0) x = 0.0;
        else if (!plain && !isfinite(sc.rr)) x = x0;   // broke down: from the start again
        if (holds) {
            a.x[i] = x;
            a.r[i] = r;
        }
        if (plain || sc.failed || sc.bb == 0.0) break;
        // the residual of x itself decides
        if (!(good = meet())) break;
        double t = 0;
        if (holds) t = b - spmv(a.x);
        good = reduce(t * t, 0.0, 0.0, t, []() {}, [&](const double *v, int wp, int l) {
            if (wp + l == 0) {
                sc.rr = v[0];
                sc.done = v[0] <= sc.stop || v[3] <= sc.abs_inf;
                sc.fresh = sc.plain = 1;
                sc.limit = a.max_iters < INT_MAX - sc.iters ? sc.iters + a.max_iters : INT_MAX;
            }
        });
        if (!good || sc.done) break;
        r = t;
    }
    if (bid == 0 && threadIdx.x == 0) {
        CgState *st = a.st;
        st->done = 1;
        st->failed = good ? sc.failed : 1;
        if (!good) {
            atomicOr(a.status, (uint32_t)ST_BARRIER);
            return;
        }
        st->iters = sc.iters;
        st->outer = 0;
        st->rr = sc.rr;
        st->rz = sc.gamma;
        st->bb = sc.bb;
        if (sc.failed && !a.quiet) atomicOr(a.status, (uint32_t)ST_CG_NO_CONV);
    }
}

// ---------------------------------------------------------------------------
// Completion preconditioned by multigrid.  Flexible PCG (Polak-Ribiere beta,
// since the preconditioner is applied in FP32) in FP64 on the node Laplacian
// L, with one V-cycle of the smoothed-aggregation hierarchy of multigrid.cpp
// as preconditioner: one damped-Jacobi sweep before and after the coarse
// correction on level 0, two Chebyshev steps before and after it on level 1,
// the dense inverse on level 2.  The V-cycle runs on the
// scaled operators s0 L in FP32 with the residual divided by its maximum
// (sigma), so z = sigma s0 V(r / sigma).  One persistent cooperative launch:
// every phase that reads other rows' values starts after a grid barrier, and
// the reductions have a fixed order (grid_reduce).  An iteration has twelve
// such phases, bound by the latency of dependent loads, so
//  * the row pointers of a block's level-0 slices and level-1 rows sit in
//    shared memory, a row's indices and values are loaded together before
//    its gathers, and what a phase gathers is one FP32 array: the update
//    leaves the scaled residual and its first Jacobi sweep w0 r (scaled by the
//    sigma of the iteration before; fac is the ratio to this one's), which the
//    next V-cycle's first pass used to form from r in FP64 per entry;
//  * L p is not formed: with w = L z and q = L p, (p', q') of p' = z + beta p
//    is (z, w) + 2 beta (z, q) + beta^2 (p, q), so that one reduction after w
//    gives beta and alpha, and p, q, x, r are updated in one pass.
// 48^3 Poisson solve 2.02 -> 1.72 ms, 40^3 completion 0.78 -> 0.70 ms, 64^3 1.44 ->
// 1.37 ms (there bound by its FP64 product and by streaming L: the hierarchy no
// longer fits in L2 beside the vectors).  Waits are bounded
// like those of the Jacobi-PCG (timeout status, no hang).
// ---------------------------------------------------------------------------
struct MgArgs {
    int n0, n1, n2, n_slices;
    const int *sp, *sw, *col;                 // SELL-32 of L on interior nodes
    const double *Lv;                         // FP64 values of L
    const float *L32;                         // FP32 values of s0 L
    const float *w0, *w1;                     // Jacobi weights 1 / (rho d_i)
    const int *p0p, *p0c;                     // P0 (fine rows)
    const float *p0v;
    const int *r0p, *r0c;                     // P0^T (coarse rows)
    const float *r0v;
    const int *l1p, *l1c;                     // L1
    const float *l1v;
    const int *agg1, *r1p, *r1c;              // level-1 aggregates and their members
    const float *l2inv;                       // n2 x n2
    double s0;
    const double *b;
    double *x, *r, *p, *q, *z, *zo;
    float *r32, *z0, *t0, *r1, *z1, *z1b, *t1, *d1, *r2, *z2;
    double *part;
    CgState *st;
    GridBarrier *gb;
    const double *abs_src;
    double abs_factor, fallback_tol2;
    uint32_t *status;
    int max_iters, spin_limit;
    int verify;                               // check the first solution against b - L x, and go on from it if need be
};

// Level-1 smoother: two steps of the Chebyshev iteration for D1^-1 L1 on
// [rho1 / 8, rho1], rho1 the (over)estimate behind w1 = 1 / (rho1 d1).  With
// theta, delta the centre and half-width of that interval (in units of rho1),
// sigma = theta / delta, c0 = 1 / sigma, c1 = 1 / (2 sigma - c0):
//   d = D^-1 res / theta = kCh1 w1 res,  z += d,  res -= L1 d,
//   d = c1 c0 d + (2 c1 / delta) D^-1 res = kCh2a d + kCh2b w1 res,  z += d.
// (A CPU prototype on the 64^3 mesh's Laplacian: 29 -> 20 PCG iterations
// against one damped-Jacobi sweep before and after.)
constexpr double kChTheta = (1.0 + 0.125) / 2.0, kChDelta = (1.0 - 0.125) / 2.0;
constexpr double kChSigma = kChTheta / kChDelta, kChC0 = 1.0 / kChSigma, kChC1 = 1.0 / (2.0 * kChSigma - kChC0);
constexpr float kCh1 = (float)(1.0 / kChTheta), kCh2a = (float)(kChC1 * kChC0), kCh2b = (float)(2.0 * kChC1 / kChDelta);

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Sums over two CSR rows (0 and 1) by a half warp, 16 lanes each row (the two
// halves of a warp take four rows at once), with every index and value of up
// to 48 entries of both loaded before the first gather: the phases are bound
// by the latency of these dependent loads, not by bandwidth.  val == nullptr
// means unit weights; get(c) is the gathered value of column c.
template <typename Get>
__device__ __forceinline__ float2 half_row_dots(int2 r0, int2 r1, const int *__restrict__ col,
                                                const float *__restrict__ val, int hl, Get get) {
    constexpr int kE = 3;
    float s[2] = {0.0f, 0.0f};
    while (r0.x < r0.y || r1.x < r1.y) {
        int c[2][kE];
        float v[2][kE];
#pragma unroll
        for (int u = 0; u < kE; u++) {
            const int k0 = r0.x + hl + 16 * u, k1 = r1.x + hl + 16 * u;
            c[0][u] = k0 < r0.y ? col[k0] : -1;
            c[1][u] = k1 < r1.y ? col[k1] : -1;
            v[0][u] = k0 < r0.y ? (val ? val[k0] : 1.0f) : 0.0f;
            v[1][u] = k1 < r1.y ? (val ? val[k1] : 1.0f) : 0.0f;
        }
#pragma unroll
        for (int h = 0; h < 2; h++)
#pragma unroll
            for (int u = 0; u < kE; u++)
                if (c[h][u] >= 0) s[h] = fmaf(v[h][u], get(c[h][u]), s[h]);
        r0.x += 16 * kE;
        r1.x += 16 * kE;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        s[0] += __shfl_xor_sync(0xFFFFFFFFu, s[0], o);
        s[1] += __shfl_xor_sync(0xFFFFFFFFu, s[1], o);
    }
    return make_float2(s[0], s[1]);
}

// the whole solve, run by block `bid` (T threads) of the nb blocks that own
// it; the scalars are formed by one thread per block (see grid_reduce)
template <int T>
__device__ __forceinline__ void mg_body(const MgArgs &a, const int nb, const int bid, double *shv,
                                        unsigned long long *shm) {
    struct Scalars {
        double thr, tol2, bb, rr, rz, pq, alpha, beta, zs, inv;
        float fac;
        int it, fresh, done, failed;
    };
    __shared__ Scalars sc;
    // the run's threads, warps and half warps, numbered across the blocks first:
    // what does not divide evenly (1.6 slices a warp, three coarse rows a half
    // warp on the 64^3 mesh) then spreads over all SMs instead of loading the
    // first blocks twice
    const int G = nb * T, lane = threadIdx.x & 31;
    const int nw = G >> 5, gw = (threadIdx.x >> 5) * nb + bid, gt = gw * 32 + lane;
    const long lim = a.spin_limit;
    unsigned int epoch = 0;
    // row pointers: the k-th slice of warp w (k * W + w) and the k-th coarse
    // row of half warp h (k * 2W + h), where the block has at most kPtrs of each
    constexpr int W = T / 32, kPtrs = 4;
    __shared__ int2 s_slice[kPtrs * W], s_l1[kPtrs * 2 * W], s_r0[kPtrs * 2 * W];
    {
        const int warp = threadIdx.x >> 5, half = threadIdx.x >> 4;
        for (int k = lane; k < kPtrs; k += 32) {
            const int sl = gw + k * nw;
            if (sl < a.n_slices) s_slice[k * W + warp] = make_int2(a.sp[sl], a.sw[sl]);
        }
        for (int k = threadIdx.x & 15; k < kPtrs; k += 16) {
            const int c = 2 * gw + (lane >> 4) + k * 2 * nw;
            if (c < a.n1) {
                s_l1[k * 2 * W + half] = make_int2(a.l1p[c], a.l1p[c + 1]);
                s_r0[k * 2 * W + half] = make_int2(a.r0p[c], a.r0p[c + 1]);
            }
        }
    }
    auto slice = [&](int k, int sl) { return k < kPtrs ? s_slice[k * W + (threadIdx.x >> 5)] : make_int2(a.sp[sl], a.sw[sl]); };
    auto coarse = [&](const int2 *sm, const int *ptr, int k, int c) {
        return c >= a.n1 ? make_int2(0, 0) : k < kPtrs ? sm[k * 2 * W + (threadIdx.x >> 4)] : make_int2(ptr[c], ptr[c + 1]);
    };
    // sum over a SELL row (lane's row of the slice at h): eight entries' columns
    // and values before their gathers
    auto sell_row = [&](int2 h, const auto *__restrict__ val, const auto *x) {
        using V = typename std::remove_cv<typename std::remove_reference<decltype(val[0])>::type>::type;
        V s = 0;
        const int kb = h.x + lane;
        for (int j0 = 0; j0 < h.y; j0 += 8) {
            int c[8];
            V v[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const bool in = j0 + u < h.y;
                c[u] = in ? a.col[kb + 32 * (j0 + u)] : 0;
                v[u] = in ? val[kb + 32 * (j0 + u)] : (V)0;
            }
#pragma unroll
            for (int u = 0; u < 8; u++)
                if (j0 + u < h.y) s = fma(v[u], x[c[u]], s);
        }
        return s;
    };
    __syncthreads();
    if (threadIdx.x == 0) {
        sc.thr = -1.0;
        sc.tol2 = a.fallback_tol2;
        if (a.abs_src) {
            const double qv = *a.abs_src;
            if (qv > 0.0) sc.thr = a.abs_factor * qv;
        }
        sc.it = 0;
        sc.fresh = 1;
        sc.failed = 0;
        sc.inv = 1.0;
    }
    // after a residual: |r|^2 = t[0], max|r| = t[1]; sigma scales the next V-cycle
    auto residual = [&](const double *t, int wp, int l) {
        if (wp + l != 0) return;
        sc.rr = t[0];
        int done = sc.bb == 0.0 || (sc.thr >= 0.0 ? t[1] <= sc.thr : t[0] <= sc.tol2 * sc.bb);
        if (!done && sc.it >= a.max_iters) done = sc.failed = 1;
        sc.done = done;
        const double sigma = t[1] > 0.0 ? t[1] : 1.0;
        const double inv = 1.0 / sigma;
        sc.fac = (float)(inv / sc.inv);
        sc.inv = inv;
        sc.zs = sigma * a.s0;
    };
    // x = 0, r = b; |b|^2 and max|r|
    {
        double v[1] = {0.0};
        unsigned long long mx = 0;
        for (int i = gt; i < a.n0; i += G) {
            const double bi = a.b[i];
            a.x[i] = 0.0;
            a.r[i] = bi;
            v[0] += bi * bi;
            mx = max(mx, abs_bits(bi));
        }
        if (!grid_reduce<1, T>(a.gb, a.part, v, mx, shv, shm, ++epoch, nb, bid, T / 32, lim, [&](const double *t, int wp, int l) {
                if (wp + l == 0) sc.bb = t[0];
                residual(t, wp, l);
            }))
            goto timeout;
    }
    {
        bool verify = a.verify != 0;
        while (true) {
            if (sc.done) {
                if (!verify || sc.failed || sc.bb == 0.0) break;
                // the residual of x itself, once: the recurrence's drifts from
                // it where the tolerance nears the rounding of L x
                verify = false;
                double v[1] = {0.0};
                unsigned long long mx = 0;
                for (int k = 0, sl = gw; sl < a.n_slices; k++, sl += nw) {
                    const int row = sl * 32 + lane;
                    const double s = sell_row(slice(k, sl), a.Lv, a.x);
                    if (row < a.n0) {
                        const double ri = a.b[row] - s;
                        a.r[row] = ri;
                        v[0] += ri * ri;
                        mx = max(mx, abs_bits(ri));
                    }
                }
                if (!grid_reduce<1, T>(a.gb, a.part, v, mx, shv, shm, ++epoch, nb, bid, T / 32, lim,
                                       [&](const double *t, int wp, int l) {
                                           if (wp + l == 0) sc.fresh = 1;
                                           residual(t, wp, l);
                                       }))
                    goto timeout;
                continue;
            }
            const bool first = sc.fresh != 0;
            float fac = sc.fac;
            if (first) {
                const double inv = sc.inv;
                for (int i = gt; i < a.n0; i += G) {
                    const float rs = (float)(a.r[i] * inv);
                    a.r32[i] = rs;
                    a.z0[i] = a.w0[i] * rs;
                }
                fac = 1.0f;
                if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            }
            // V1: t0 = r32 - L z0 with the first Jacobi sweep z0 = w0 r32
            for (int k = 0, sl = gw; sl < a.n_slices; k++, sl += nw) {
                const int row = sl * 32 + lane;
                const float s = sell_row(slice(k, sl), a.L32, a.z0);
                if (row < a.n0) a.t0[row] = fac * (a.r32[row] - s);
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // (coarse rows: half a warp takes two rows at once; the lanes 0 and 1
            // of the half finish one each, their operands loaded beforehand)
            const int hl = lane & 15, hw = 2 * gw + (lane >> 4), nhw = 2 * nw;
            const bool ends = hl < 2;
            // V2: r1 = P0^T t0, the first Chebyshev step z1 = kCh1 w1 r1
            for (int k = 0, c = hw; c - (hw & 1) < a.n1; k += 2, c += 2 * nhw) {
                const int cm = c + hl * nhw;   // the row this lane finishes
                const bool fin = ends && cm < a.n1;
                const float wm = fin ? a.w1[cm] : 0.0f;
                const float2 d = half_row_dots(coarse(s_r0, a.r0p, k, c), coarse(s_r0, a.r0p, k + 1, c + nhw), a.r0c,
                                               a.r0v, hl, [&](int q) { return a.t0[q]; });
                const float sum = hl ? d.y : d.x;
                if (fin) {
                    a.r1[cm] = sum;
                    a.z1[cm] = kCh1 * wm * sum;
                }
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V3: res = r1 - L1 z1 (into t1), the second step d1 = kCh2a z1 +
            // kCh2b w1 res, z1 + d1 (into z1b, since z1 is still read here)
            for (int k = 0, c = hw; c - (hw & 1) < a.n1; k += 2, c += 2 * nhw) {
                const int cm = c + hl * nhw;
                const bool fin = ends && cm < a.n1;
                const float wm = fin ? a.w1[cm] : 0.0f, rm = fin ? a.r1[cm] : 0.0f, zm = fin ? a.z1[cm] : 0.0f;
                const float2 d = half_row_dots(coarse(s_l1, a.l1p, k, c), coarse(s_l1, a.l1p, k + 1, c + nhw), a.l1c,
                                               a.l1v, hl, [&](int q) { return a.z1[q]; });
                if (fin) {
                    const float res = rm - (hl ? d.y : d.x);
                    const float dd = kCh2a * zm + kCh2b * wm * res;
                    a.t1[cm] = res;
                    a.d1[cm] = dd;
                    a.z1b[cm] = zm + dd;
                }
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V3b: the residual after the pre-smoothing, t1 = res - L1 d1
            for (int k = 0, c = hw; c - (hw & 1) < a.n1; k += 2, c += 2 * nhw) {
                const int cm = c + hl * nhw;
                const bool fin = ends && cm < a.n1;
                const float tm = fin ? a.t1[cm] : 0.0f;
                const float2 d = half_row_dots(coarse(s_l1, a.l1p, k, c), coarse(s_l1, a.l1p, k + 1, c + nhw), a.l1c,
                                               a.l1v, hl, [&](int q) { return a.d1[q]; });
                if (fin) a.t1[cm] = tm - (hl ? d.y : d.x);
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V4: r2 = sum of t1 over each level-2 aggregate
            for (int g = gw; g < a.n2; g += nw) {
                const int kb = a.r1p[g], ke = a.r1p[g + 1];
                float s = 0.0f;
#pragma unroll 4
                for (int k = kb + lane; k < ke; k += 32) s += a.t1[a.r1c[k]];
                s = warp_sum_f(s);
                if (lane == 0) a.r2[g] = s;
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V5: z2 = L2^-1 r2 (dense)
            for (int g = gw; g < a.n2; g += nw) {
                const float *row = a.l2inv + (size_t)g * a.n2;
                float s = 0.0f;
#pragma unroll 4
                for (int k = lane; k < a.n2; k += 32) s = fmaf(row[k], a.r2[k], s);
                s = warp_sum_f(s);
                if (lane == 0) a.z2[g] = s;
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V6: coarse correction and the first post-smoothing step in one
            // pass: zc = z1b + z2[agg] (the corrected neighbours formed on the
            // fly), res = r1 - L1 zc (into t1), d1 = kCh1 w1 res, zc + d1 (into z1)
            for (int k = 0, c = hw; c - (hw & 1) < a.n1; k += 2, c += 2 * nhw) {
                const int cm = c + hl * nhw;
                const bool fin = ends && cm < a.n1;
                const float wm = fin ? a.w1[cm] : 0.0f, rm = fin ? a.r1[cm] : 0.0f;
                const float zm = fin ? a.z1b[cm] + a.z2[a.agg1[cm]] : 0.0f;
                const float2 d = half_row_dots(coarse(s_l1, a.l1p, k, c), coarse(s_l1, a.l1p, k + 1, c + nhw), a.l1c,
                                               a.l1v, hl, [&](int q) { return a.z1b[q] + a.z2[a.agg1[q]]; });
                if (fin) {
                    const float res = rm - (hl ? d.y : d.x), dd = kCh1 * wm * res;
                    a.t1[cm] = res;
                    a.d1[cm] = dd;
                    a.z1[cm] = zm + dd;
                }
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V6b: the second post-smoothing step, res -= L1 d1,
            // z1b = z1 + kCh2a d1 + kCh2b w1 res
            for (int k = 0, c = hw; c - (hw & 1) < a.n1; k += 2, c += 2 * nhw) {
                const int cm = c + hl * nhw;
                const bool fin = ends && cm < a.n1;
                const float wm = fin ? a.w1[cm] : 0.0f, tm = fin ? a.t1[cm] : 0.0f, zm = fin ? a.z1[cm] : 0.0f,
                            dm = fin ? a.d1[cm] : 0.0f;
                const float2 d = half_row_dots(coarse(s_l1, a.l1p, k, c), coarse(s_l1, a.l1p, k + 1, c + nhw), a.l1c,
                                               a.l1v, hl, [&](int q) { return a.d1[q]; });
                if (fin) {
                    const float res = tm - (hl ? d.y : d.x);
                    a.z1b[cm] = zm + (kCh2a * dm + kCh2b * wm * res);
                }
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V7: coarse correction of level 0 (into t0, free now); the row's
            // indices and values (up to 8) are loaded before the gathers
            for (int i = gt; i < a.n0; i += G) {
                float s = fac * a.z0[i];
                const int kb = a.p0p[i], ke = a.p0p[i + 1];
                for (int k0 = kb; k0 < ke; k0 += 8) {
                    int c[8];
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; u++) {
                        const bool in = k0 + u < ke;
                        c[u] = in ? a.p0c[k0 + u] : 0;
                        v[u] = in ? a.p0v[k0 + u] : 0.0f;
                    }
#pragma unroll
                    for (int u = 0; u < 8; u++) s = fmaf(v[u], a.z1b[c[u]], s);
                }
                a.t0[i] = s;
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // V8: post-smoothing on level 0, z = sigma s0 z0 in FP64
            {
                const double zs = sc.zs;
                for (int k = 0, sl = gw; sl < a.n_slices; k++, sl += nw) {
                    const int row = sl * 32 + lane;
                    const float s = sell_row(slice(k, sl), a.L32, a.t0);
                    if (row < a.n0)
                        a.z[row] = zs * (double)(a.t0[row] + a.w0[row] * (fac * a.r32[row] - s));
                }
            }
            if (!grid_barrier(a.gb, ++epoch, nb, lim)) goto timeout;
            // w = L z (in z_old's place once (r, z_old) has read it), and
            // (r, z), (r, z_old), (z, w), (z, q)
            {
                double v[4] = {0.0, 0.0, 0.0, 0.0};
                for (int k = 0, sl = gw; sl < a.n_slices; k++, sl += nw) {
                    const int row = sl * 32 + lane;
                    const double s = sell_row(slice(k, sl), a.Lv, a.z);
                    if (row < a.n0) {
                        const double zi = a.z[row], ri = a.r[row];
                        v[0] = fma(ri, zi, v[0]);
                        if (!first) {   // z_old, q not read before set
                            v[1] = fma(ri, a.zo[row], v[1]);
                            v[3] = fma(zi, a.q[row], v[3]);
                        }
                        v[2] = fma(zi, s, v[2]);
                        a.zo[row] = s;
                    }
                }
                if (!grid_reduce<4, T>(a.gb, a.part, v, 0ull, shv, shm, ++epoch, nb, bid, T / 32, lim,
                                       [&](const double *t, int wp, int l) {
                                           if (wp + l != 0) return;
                                           const double be = sc.fresh ? 0.0 : (t[0] - t[1]) / sc.rz;
                                           const double pq = sc.fresh ? t[2] : t[2] + be * (2.0 * t[3] + be * sc.pq);
                                           sc.beta = be;
                                           sc.rz = t[0];
                                           sc.pq = pq;
                                           sc.alpha = t[0] / pq;
                                           sc.it++;
                                           sc.fresh = 0;
                                       }))
                    goto timeout;
            }
            // p = z + beta p, q = w + beta q, x += alpha p, r -= alpha q; |r|^2
            // and max|r|; the scaled residual and first sweep of the next V-cycle
            {
                const double alpha = sc.alpha, beta = sc.beta, inv = sc.inv;
                double v[1] = {0.0};
                unsigned long long mx = 0;
                for (int k = 0, sl = gw; sl < a.n_slices; k++, sl += nw) {
                    const int i = sl * 32 + lane;
                    if (i >= a.n0) continue;
                    const double zi = a.z[i], wi = a.zo[i];
                    const double pi = first ? zi : fma(beta, a.p[i], zi);
                    const double qi = first ? wi : fma(beta, a.q[i], wi);
                    const double ri = fma(-alpha, qi, a.r[i]);
                    a.p[i] = pi;
                    a.q[i] = qi;
                    a.zo[i] = zi;
                    a.x[i] = fma(alpha, pi, a.x[i]);
                    a.r[i] = ri;
                    const float rs = (float)(ri * inv);
                    a.r32[i] = rs;
                    a.z0[i] = a.w0[i] * rs;
                    v[0] += ri * ri;
                    mx = max(mx, abs_bits(ri));
                }
                if (!grid_reduce<1, T>(a.gb, a.part, v, mx, shv, shm, ++epoch, nb, bid, T / 32, lim, residual)) goto timeout;
            }
        }
        if (bid == 0 && threadIdx.x == 0) {
            a.st->iters = sc.it;
            a.st->rr = sc.rr;
            a.st->bb = sc.bb;
            a.st->done = 1;
            a.st->failed = sc.failed;
            if (sc.failed) atomicOr(a.status, (uint32_t)ST_CG_NO_CONV);
        }
        return;
    }
timeout:
    if (bid == 0 && threadIdx.x == 0) {
        a.st->done = 1;
        a.st->failed = 1;
        atomicOr(a.status, (uint32_t)ST_BARRIER);
    }
}

__global__ void __launch_bounds__(kMgThreads, 1) k_mg_pcg(const MgArgs a) {
    __shared__ double shv[4 * kMgThreads];
    __shared__ unsigned long long shm[kMgThreads];
    mg_body<kMgThreads>(a, gridDim.x, blockIdx.x, shv, shm);
}

// one solve per launch (its arguments passed by value), one block per SM
template <bool REFINE, bool WIDE>
__global__ void __launch_bounds__(PcgShape<REFINE, WIDE>::threads, 1) k_pcg_persistent(const PcgArgs a) {
    using P = PcgShape<REFINE, WIDE>;
    __shared__ double shv[4 * P::threads];
    __shared__ unsigned long long shm[P::threads];
    pcg_body<REFINE, WIDE, P::threads, P::ring>(a, gridDim.x, blockIdx.x, s_ring, shv, shm);
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_pcg_small(const PcgArgs a) {
    small_body(a, gridDim.x, blockIdx.x);
}
__global__ void __launch_bounds__(kSmallThreads, 1) k_pcg_small_batched(const __grid_constant__ PcgBatch<kMaxBatchRuns> B) {
    __shared__ PcgArgs sa;
    if (threadIdx.x == 0) {
        int ri = 0;
        while (ri + 1 < B.n_runs && (int)blockIdx.x >= B.run[ri + 1].block0) ri++;
        sa = B.run[ri];
    }
    __syncthreads();
    small_body(sa, sa.blocks, (int)blockIdx.x - sa.block0);
}

// several solves of one kind per launch: run r owns blocks [block0, block0 + blocks).
// Built for MINB = 4 blocks per SM (64 registers) and MINB = 3 (80); a batch's
// tuner picks.  ANYWIDE: some run's records are wide (the others' may be narrow).
template <bool REFINE, int MINB, bool ANYWIDE>
__global__ void __launch_bounds__(kThreads, MINB) k_pcg_batched(const __grid_constant__ PcgBatch<kMaxBatchRuns> B) {
    // the block's run, copied to shared memory: read through a dynamic index
    // in parameter space, the arguments made the solve half as fast again
    __shared__ PcgArgs sa;
    __shared__ double shv[4 * kThreads];
    __shared__ unsigned long long shm[kThreads];
    if (threadIdx.x == 0) {
        int ri = 0;
        while (ri + 1 < B.n_runs && (int)blockIdx.x >= B.run[ri + 1].block0) ri++;
        sa = B.run[ri];
    }
    __syncthreads();
    constexpr int kRing = ANYWIDE ? kBatchRingWide : kBatchRing;
    if (ANYWIDE && sa.wide)
        pcg_body<REFINE, true, kThreads, kBatchRingWide>(sa, sa.blocks, (int)blockIdx.x - sa.block0, s_ring, shv, shm);
    else
        pcg_body<REFINE, false, kThreads, kRing>(sa, sa.blocks, (int)blockIdx.x - sa.block0, s_ring, shv, shm);
}

int grid_for_elems(int n) { return std::max(1, std::min(kMaxBlocks, (n + kThreads - 1) / kThreads)); }

__global__ void k_recip_diag(int n, const double *__restrict__ d, double *__restrict__ dinv) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dinv[i] = 1.0 / d[i];
}

__global__ void k_axpby(int n, double a, const double *__restrict__ x, double b, const double *__restrict__ y,
                        double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = a * x[i] + b * y[i];
}

// The solvers' matrices as records (stream.cuh): the FP64 values as they are,
// or, with dinv, FP32 values of the diagonally scaled D^-1/2 A D^-1/2 (unit
// diagonal: Jacobi-PCG on A is plain CG on it, without the D^-1 and u vectors),
// which the MIXED corrections solve.  One warp a slice; the records past the
// last column were zeroed (value 0, an existing column).
template <typename V, bool WIDE>
__global__ void k_pack_records(int n, int n_slices, const int *__restrict__ sp, const int *__restrict__ sw,
                               const int *__restrict__ col, const int *__restrict__ base,
                               const unsigned char *__restrict__ off, const double *__restrict__ v,
                               const double *__restrict__ dinv, unsigned char *__restrict__ out) {
    using Rec = Record<V, WIDE>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int sl = t >> 5, lane = t & 31;
    if (sl >= n_slices) return;
    const int i = sl * 32 + lane, k0 = sp[sl] >> 5;
    const double di = dinv && i < n ? sqrt(dinv[i]) : 0.0;
    for (int j = 0; j < sw[sl]; j++) {
        const int k = k0 + j, c = k & (kCols - 1);
        const size_t e = 32 * (size_t)k + lane;
        unsigned char *rec = out + (size_t)(k / kCols) * Rec::bytes;
        double x = 0.0;
        if (i < n) x = dinv ? v[e] * di * sqrt(dinv[col[e]]) : v[e];
        *reinterpret_cast<V *>(rec + record_value_at<V>(c, lane)) = (V)x;
        if constexpr (WIDE) {
            *reinterpret_cast<int *>(rec + Rec::val + ((c >> 2) * 32 + lane) * 16 + (c & 3) * 4) = col[e];
        } else {
            rec[Rec::val + lane * kCols + c] = off[e];
            if (lane == 0) *reinterpret_cast<int *>(rec + Rec::val + Rec::idx + 4 * c) = base[k];
        }
    }
}

template <typename V>
int pack_records(const DevSell &A, const double *v, const double *dinv, DevBuf<unsigned char> &out) {
    const size_t cols = (size_t)(A.n_elems / 32), recs = (cols + kCols - 1) / kCols;
    const size_t bytes = recs * (A.narrow ? Record<V, false>::bytes : Record<V, true>::bytes);
    int rc = out.alloc(bytes);
    if (rc) return rc;
    if (!bytes) return PIC_OK;
    FP_CUDA(cudaMemset(out.p, 0, bytes));
    const unsigned blocks = (unsigned)((A.n_slices * 32 + 255) / 256);
    if (A.narrow) { k_pack_records<V, false><<<blocks, 256>>>(A.n_rows, A.n_slices, A.ptr.p, A.width.p, A.col.p, A.base.p, A.off.p, v, dinv, out.p); note_launch(); }
    else { k_pack_records<V, true><<<blocks, 256>>>(A.n_rows, A.n_slices, A.ptr.p, A.width.p, A.col.p, nullptr, nullptr, v, dinv, out.p); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

__global__ void k_sqrt_f32(int n, const double *__restrict__ dinv, float *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)sqrt(dinv[i]);
}


}  // namespace

int solver_alloc(Sim *s) {
    const Mesh *m = s->mesh;
    const int ne = m->n_edges, nf = m->n_faces, nn = m->n_nodes, ni = m->n_int_edges, nin = m->n_int_nodes;
    int rc;
    DevBuf<double> *edge_vecs[] = {&s->e, &s->e_prev, &s->x, &s->g, &s->g_prev, &s->g_new, &s->dg, &s->rhs};
    // the solvers' vectors are padded to whole slices, zeros past the rows
    auto padded = [](int n) { return (size_t)(std::max(n, 1) + 31) / 32 * 32; };
    for (auto *v : edge_vecs) {
        if ((rc = v->alloc(padded(ne)))) return rc;
        FP_CUDA(cudaMemset(v->p, 0, sizeof(double) * padded(ne)));
    }
    DevBuf<double> *face_vecs[] = {&s->b, &s->b_prev, &s->b_new, &s->hb};
    for (auto *v : face_vecs) {
        if ((rc = v->alloc(nf))) return rc;
        FP_CUDA(cudaMemset(v->p, 0, sizeof(double) * nf));
    }
    DevBuf<double> *node_vecs[] = {&s->rho, &s->rho_prev, &s->wall, &s->wall_prev, &s->rho_bg, &s->phi};
    for (auto *v : node_vecs) {
        if ((rc = v->alloc(nn))) return rc;
        FP_CUDA(cudaMemset(v->p, 0, sizeof(double) * nn));
    }
    DevBuf<double> *int_vecs[] = {&s->Dinv, &s->cg_r, &s->cg_z, &s->cg_p0, &s->cg_p1, &s->cg_q, &s->w_edge, &s->me, &s->ev};
    for (auto *v : int_vecs) {
        if ((rc = v->alloc(padded(ni)))) return rc;
        FP_CUDA(cudaMemset(v->p, 0, sizeof(double) * padded(ni)));
    }
    DevBuf<double> *lap_vecs[] = {&s->L_Dinv, &s->l_x, &s->l_b, &s->l_r, &s->l_z, &s->l_p0, &s->l_p1, &s->l_q};
    for (auto *v : lap_vecs) {
        if ((rc = v->alloc(padded(nin)))) return rc;
        FP_CUDA(cudaMemset(v->p, 0, sizeof(double) * padded(nin)));
    }
    if ((rc = s->cg_part.alloc(8 * kMaxBlocks)) || (rc = s->l_part.alloc(8 * kMaxBlocks)) ||
        (rc = s->diag_part.alloc(8 * kMaxBlocks)))
        return rc;
    // A = M + c4 K + ci I and the Jacobi preconditioners
    double c4, ci;
    system_coefficients(s, &c4, &ci);
    const long long nel = m->As.n_elems;
    if ((rc = s->A_val.alloc(std::max(nel, 1LL)))) return rc;
    if (nel > 0) {
        { k_axpby<<<(unsigned)((nel + 255) / 256), 256>>>((int)nel, 1.0, m->M_val.p, c4, m->K_val.p, s->A_val.p); note_launch(); }
        if (m->n_abs_faces > 0)
            { k_axpby<<<(unsigned)((nel + 255) / 256), 256>>>((int)nel, 1.0, s->A_val.p, ci, m->I_val.p, s->A_val.p); note_launch(); }
        { k_recip_diag_mk<<<(ni + 255) / 256, 256>>>(ni, m->M_diag.p, m->K_diag.p, c4,
                                                     m->n_abs_faces > 0 ? m->I_diag.p : nullptr, ci, s->Dinv.p); note_launch(); }
    }
    if (nin > 0) { k_recip_diag<<<(nin + 255) / 256, 256>>>(nin, m->L_diag.p, s->L_Dinv.p); note_launch(); }
    if (nel > 0 && (rc = pack_records<double>(m->As, s->A_val.p, nullptr, s->A_rec))) return rc;
    // (the node Laplacian is the mesh's own: packed by its first simulation)
    if (nin > 0 && !m->L_rec.p && (rc = pack_records<double>(m->Ls, m->Ls_val.p, nullptr, const_cast<Mesh *>(m)->L_rec)))
        return rc;
    // MIXED: the correction solves of the Newmark refinement run on the
    // diagonally scaled system in FP32
    if (s->mixed && nel > 0) {
        if ((rc = s->Dhalf32.alloc(padded(ni))) || (rc = s->cg32.alloc(6 * padded(ni)))) return rc;
        FP_CUDA(cudaMemset(s->Dhalf32.p, 0, sizeof(float) * padded(ni)));
        FP_CUDA(cudaMemset(s->cg32.p, 0, sizeof(float) * 6 * padded(ni)));
        if ((rc = pack_records<float>(m->As, s->A_val.p, s->Dinv.p, s->A_rec32))) return rc;
        { k_sqrt_f32<<<(unsigned)((ni + 255) / 256), 256>>>(ni, s->Dinv.p, s->Dhalf32.p); note_launch(); }
    }
    FP_CUDA(cudaGetLastError());
    FP_CUDA(cudaDeviceSynchronize());
    return PIC_OK;
}

// Coefficients of the system matrix A = M + c4 K + ci I of the field update:
// Newmark (gamma = 1/2, beta = 1/4), both forms: c4 = dt^2/4, ci = dt/(2c);
// backward difference: c4 = dt^2, ci = dt/c.
void system_coefficients(const Sim *s, double *c4, double *ci) {
    const double dt = s->cfg.dt;
    const bool bd = s->cfg.form == PIC_FORM_BD;
    *c4 = (bd ? 1.0 : 0.25) * dt * dt;
    *ci = (bd ? 1.0 : 0.5) * dt / kC0;
}

int newmark_rhs(Sim *s) {
    const Mesh *m = s->mesh;
    const int ni = m->n_int_edges;
    if (ni == 0) return PIC_OK;
    const double dt = s->cfg.dt, c4 = 0.25 * dt * dt;
    const DevSell &A = m->As;
    const int gs = grid_for_slices(A.n_slices);
    // the Newmark forms' predictor x = 2e - e' (also the initial guess of the
    // backward difference, whose right-hand side does not use it)
    { k_rhs_pre<<<(ni + 255) / 256, 256, 0, s->stream>>>(ni, s->e.p, s->e_prev.p, s->x.p, s->ev.p); note_launch(); }
    const int nr = m->I_row.n;
    if (s->cfg.form == PIC_FORM_WE) {
        { k_rhs_we_sell<<<gs, kThreads, 0, s->stream>>>(ni, A.n_slices, A.ptr.p, A.width.p, A.col.p, m->M_val.p, m->K_val.p, c4, s->x.p, s->ev.p, s->g_new.p, s->g.p, s->g_prev.p, s->rhs.p); note_launch(); }
        // the kernel above forms -(M + dt^2/4 K) e'; the absorbing walls add
        // the rest of -(M - dt/(2c) I + dt^2/4 K) e', i.e. + dt/(2c) I e'
        if (nr > 0)
            { k_rhs_impedance<<<(nr + 255) / 256, 256, 0, s->stream>>>(nr, m->I_row.p, m->Ir.rowptr.p, m->Ir.col.p, m->Ir_val.p, 0.5 * dt / kC0, s->e_prev.p, 0.0, nullptr, s->rhs.p); note_launch(); }
    } else if (s->cfg.form == PIC_FORM_MFEM) {
        { k_face_hb<false><<<grid_for_slices(m->Hs.n_slices), kThreads, 0, s->stream>>>(m->n_faces, m->Hs.n_slices, m->Hs.ptr.p, m->Hs.width.p, m->Hs.col.p, m->Hs_val.p, s->b.p, s->b_prev.p, s->hb.p); note_launch(); }
        { k_rhs_mfem_sell<<<gs, kThreads, 0, s->stream>>>(ni, A.n_slices, A.ptr.p, A.width.p, A.col.p, m->M_val.p, m->K_val.p, c4, dt, s->e_prev.p, s->ev.p, s->g_new.p, s->g_prev.p, m->e2f.rowptr.p, m->e2f.col.p, m->e2f_sgn.p, s->hb.p, s->rhs.p); note_launch(); }
        // the Ampere row's 2 dt/c I (e^{n+1}/4 + e^n/2 + e^{n-1}/4): the e^{n+1}
        // part is in A, - dt/c I (e^n + e^{n-1}/2) comes here
        if (nr > 0)
            { k_rhs_impedance<<<(nr + 255) / 256, 256, 0, s->stream>>>(nr, m->I_row.p, m->Ir.rowptr.p, m->Ir.col.p, m->Ir_val.p, -dt / kC0, s->e.p, -0.5 * dt / kC0, s->e_prev.p, s->rhs.p); note_launch(); }
    } else {
        { k_face_hb<true><<<grid_for_slices(m->Hs.n_slices), kThreads, 0, s->stream>>>(m->n_faces, m->Hs.n_slices, m->Hs.ptr.p, m->Hs.width.p, m->Hs.col.p, m->Hs_val.p, s->b.p, nullptr, s->hb.p); note_launch(); }
        { k_rhs_bd_sell<<<gs, kThreads, 0, s->stream>>>(ni, A.n_slices, A.ptr.p, A.width.p, A.col.p, m->M_val.p, dt, s->e.p, s->g_new.p, s->g.p, m->e2f.rowptr.p, m->e2f.col.p, m->e2f_sgn.p, s->hb.p, s->rhs.p); note_launch(); }
    }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

// A persistent kernel and its launch shape: co-resident blocks per SM (0: no
// cooperative launch on this device), queried once per device and kept (no
// runtime queries while a stream is being captured)
constexpr int kMaxDevices = 64;
struct CoopKernel {
    const void *fn;
    int threads, ring;            // dynamic shared memory: the warps' rings
    int cache[kMaxDevices];       // 0: not queried, -1: unavailable
    std::mutex lock;
    CoopKernel(const void *f, int t, int ring_per_warp) : fn(f), threads(t), ring(ring_per_warp * (t / 32)), cache{} {}
    int per_sm() {
        int dev = 0, coop = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
        std::lock_guard<std::mutex> hold(lock);
        if (cache[dev]) return std::max(cache[dev], 0);
        cache[dev] = -1;
        if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
        if (ring > 0 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, ring) != cudaSuccess) return 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, ring) != cudaSuccess) return 0;
        cache[dev] = n > 0 ? n : -1;
        return std::max(n, 0);
    }
    int launch(int blocks, void **args, cudaStream_t st) {
        FP_CUDA(cudaLaunchCooperativeKernel(fn, blocks, threads, args, ring, st));
        note_launch();
        return PIC_OK;
    }
};

template <bool REFINE, bool WIDE>
static CoopKernel &coop_single() {
    using P = PcgShape<REFINE, WIDE>;
    static CoopKernel k((const void *)k_pcg_persistent<REFINE, WIDE>, P::threads, P::ring);
    return k;
}
template <bool REFINE, int MINB, bool ANYWIDE>
static CoopKernel &coop_batched() {
    static CoopKernel k((const void *)k_pcg_batched<REFINE, MINB, ANYWIDE>, kThreads, ANYWIDE ? kBatchRingWide : kBatchRing);
    return k;
}
static CoopKernel &pcg_kernel(bool one, bool refine, bool wide, int build) {
    if (one) return refine ? (wide ? coop_single<true, true>() : coop_single<true, false>())
                           : (wide ? coop_single<false, true>() : coop_single<false, false>());
    if (wide) return refine ? coop_batched<true, 3, true>() : coop_batched<false, 3, true>();
    if (build == 1) return refine ? coop_batched<true, 3, false>() : coop_batched<false, 3, false>();
    return refine ? coop_batched<true, 4, false>() : coop_batched<false, 4, false>();
}

static int sm_count() {
    static int cache[kMaxDevices];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    if (cache[dev]) return cache[dev];
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    cache[dev] = sms;
    return sms;
}

__global__ void k_reset_gbar(GridBarrier *gb) {
    gb->count = 0;
    gb->timeout = 0;
}

__global__ void k_reset_barriers(PcgBatch<kMaxBatchRuns> B) {
    const int r = threadIdx.x;
    if (r < B.n_runs) {
        GridBarrier *gb = B.run[r].gb;
        gb->count = 0;
        gb->timeout = 0;
    }
}

// Splits a budget of co-resident blocks between the runs: each wants one
// warp per slice at most; when they want more than the budget, blocks go in
// proportion to the slices (at least one each).
static int assign_blocks(PcgArgs *runs, int n_runs, int budget) {
    if (n_runs > budget) {
        set_error("more batched solves than co-resident blocks");
        return PIC_ERR_INVALID_ARG;
    }
    long want_total = 0, slices = 0;
    std::vector<int> want(n_runs);
    for (int r = 0; r < n_runs; r++) {
        want[r] = std::max(1, std::min(kMaxPcgBlocks, (runs[r].n_slices + kSlicesPerPcgBlock - 1) / kSlicesPerPcgBlock));
        want_total += want[r];
        slices += std::max(runs[r].n_slices, 1);
    }
    std::vector<int> got(n_runs);
    long total = 0;
    for (int r = 0; r < n_runs; r++) {
        got[r] = want_total <= budget ? want[r]
                                      : std::max(1, std::min(want[r], (int)((double)budget * std::max(runs[r].n_slices, 1) / slices)));
        total += got[r];
    }
    while (total > budget) {
        int big = 0;
        for (int r = 1; r < n_runs; r++)
            if (got[r] > got[big]) big = r;
        got[big]--;
        total--;
    }
    int b0 = 0;
    for (int r = 0; r < n_runs; r++) {
        runs[r].block0 = b0;
        runs[r].blocks = got[r];
        b0 += got[r];
    }
    return PIC_OK;
}

// FP64 systems whose slices all find a warp (one block per SM): one slice a
// warp for the whole solve, whatever the launch shape asked for.  20^3 (52,460
// rows, 1,640 slices, 227 iterations) 2.77 -> 1.70 ms; systems beyond take the streamed
// form, whose iteration is bound by the FP64 pipes rather than by latency.  So
// do relative tolerances below 1e-13, which the pipelined recurrence does not
// reach (20^3 Laplacian, 1e-14: 3.0 ms with two restarts against 1.3 ms).  A run
// gets the same blocks alone and in a batch, so its results are the same bits
// there; where a run does not qualify or the runs' blocks exceed the SMs, all of
// them take the streamed form, and agree with their solves alone to the tolerance.
static int launch_small(PcgArgs *runs, int n_runs, cudaStream_t st, bool *launched) {
    const int most = std::min(sm_count(), kSmallBlocks);
    int G = 0;
    for (int r = 0; r < n_runs; r++) {
        PcgArgs &a = runs[r];
        if (a.max_width > kSmallWidth || a.n_slices > kSmallWarps * most || (!a.abs_src && a.tol2 < kSmallTol2))
            return PIC_OK;
        int blocks = std::min(most, std::max(1, (a.n_slices + kSlicesPerPcgBlock - 1) / kSlicesPerPcgBlock));
        const int per = (a.n_slices + blocks - 1) / blocks;
        blocks = (a.n_slices + per - 1) / per;   // no block without a slice
        a.block0 = G;
        a.blocks = blocks;
        G += blocks;
    }
    if (G > sm_count()) return PIC_OK;
    static CoopKernel one((const void *)k_pcg_small, kSmallThreads, kSmallSlice * kSmallWarps / (kSmallThreads / 32));
    static CoopKernel many((const void *)k_pcg_small_batched, kSmallThreads, kSmallSlice * kSmallWarps / (kSmallThreads / 32));
    CoopKernel &kernel = n_runs == 1 ? one : many;
    if (kernel.per_sm() <= 0) {
        set_error("the persistent PCG needs a device with cooperative launch");
        return PIC_ERR_CUDA;
    }
    PcgBatch<kMaxBatchRuns> all;
    all.n_runs = n_runs;
    for (int r = 0; r < n_runs; r++) all.run[r] = runs[r];
    { k_reset_barriers<<<1, kMaxBatchRuns, 0, st>>>(all); note_launch(); }
    void *args[] = {n_runs == 1 ? (void *)&all.run[0] : (void *)&all};
    *launched = true;
    return kernel.launch(G, args, st);
}

// One cooperative launch of the persistent PCG over n_runs solves on stream
// st.  Results and failures reach the host through each run's CgState and
// status word at the next synchronisation.
int launch_pcg_runs(PcgArgs *runs, int n_runs, int blocks_per_sm, cudaStream_t st, int build) {
    if (n_runs <= 0) return PIC_OK;
    if (n_runs > kMaxBatchRuns) {
        set_error("at most " + std::to_string(kMaxBatchRuns) + " solves per persistent launch");
        return PIC_ERR_INVALID_ARG;
    }
    const bool one = n_runs == 1, refine = runs[0].refine != 0;
    for (int r = 1; r < n_runs; r++)
        if ((runs[r].refine != 0) != refine) {
            set_error("the solves of one persistent launch must all be FP64 or all be refinements");
            return PIC_ERR_INVALID_ARG;
        }
    if (!refine) {
        bool launched = false;
        int rc = launch_small(runs, n_runs, st, &launched);
        if (rc || launched) return rc;
    }
    bool wide = false;
    for (int r = 0; r < n_runs; r++) wide = wide || runs[r].wide;
    CoopKernel &kernel = pcg_kernel(one, refine, wide, build);
    int per_sm = kernel.per_sm();
    if (per_sm <= 0) {
        set_error("the persistent PCG needs a device with cooperative launch");
        return PIC_ERR_CUDA;
    }
    if (blocks_per_sm > 0) per_sm = std::min(per_sm, blocks_per_sm);
    int rc = assign_blocks(runs, n_runs, per_sm * sm_count());
    if (rc) return rc;
    const int G = runs[n_runs - 1].block0 + runs[n_runs - 1].blocks;
    PcgBatch<kMaxBatchRuns> all;
    all.n_runs = n_runs;
    for (int r = 0; r < n_runs; r++) all.run[r] = runs[r];
    { k_reset_barriers<<<1, kMaxBatchRuns, 0, st>>>(all); note_launch(); }
    PcgArgs a1 = all.run[0];
    void *args[] = {one ? (void *)&a1 : (void *)&all};
    return kernel.launch(G, args, st);
}

static PcgArgs matrix_args(const DevSell &A, const double *Av, const DevBuf<unsigned char> &rec) {
    PcgArgs a{};
    a.col = A.col.p;
    a.Av = Av;
    a.max_width = A.max_width;
    a.n = A.n_rows;
    a.n_slices = A.n_slices;
    a.sp = A.ptr.p;
    a.sw = A.width.p;
    a.rec = rec.p;
    a.wide = !A.narrow;
    a.evict_first = rec.n > kKeepInL2;
    return a;
}

static PcgArgs make_args(Sim *s, const DevSell &A, const double *Av, const DevBuf<unsigned char> &rec, const double *Dinv, const double *b, double *x,
                         double *r, double *u, double *w, double *p, double *sv, double *part, CgState *st,
                         double tol, double fallback_tol, int max_iters, const double *abs_src, double abs_factor,
                         bool x_zero, bool quiet) {
    Control *dc = s->dctl.p;
    PcgArgs a = matrix_args(A, Av, rec);
    a.Dinv = Dinv;
    a.b = b;
    a.x = x;
    a.r = r;
    a.u = u;
    a.w = w;
    a.p = p;
    a.s = sv;
    a.part = part;
    a.st = st;
    a.gb = st == &dc->cg ? &dc->gbar : &dc->gbar2;
    a.abs_src = abs_src;
    a.abs_factor = abs_factor;
    a.tol2 = tol * tol;
    a.fallback_tol2 = fallback_tol * fallback_tol;
    a.abs_inf = -1.0;
    a.status = &dc->status;
    a.max_iters = max_iters;
    a.x_zero = x_zero ? 1 : 0;
    a.quiet = quiet ? 1 : 0;
    a.spin_limit = s->cfg.barrier_spin_limit > 0 ? s->cfg.barrier_spin_limit : (int)kSpinLimit;
    return a;
}

// Jacobi-PCG on the last Newmark system from x = 0, stopped after `iters`
// iterations without an error (training samples, solver timing)
PcgArgs pcg_args_truncated(Sim *s, int iters) {
    const Mesh *m = s->mesh;
    return make_args(s, m->As, s->A_val.p, s->A_rec, s->Dinv.p, s->rhs.p, s->x.p, s->cg_r.p, s->cg_z.p, s->cg_q.p, s->cg_p0.p,
                     s->cg_p1.p, s->cg_part.p, &s->dctl.p->cg, 0.0, 0.0, iters, nullptr, 0.0, true, true);
}

// The Newmark solve stopped after `iters` iterations (in MIXED, FP32
// correction iterations) without an error: a fixed amount of work for timing.
// It starts from the x it finds, so the caller zeroes x first.
PcgArgs pcg_args_newmark_truncated(Sim *s, int iters) {
    PcgArgs a = pcg_args_newmark(s);
    a.max_iters = iters;
    a.quiet = 1;
    a.x_zero = 1;
    return a;
}

// The Newmark solve.  MIXED refines in FP64 with FP32 correction solves
// (each to 1e-5 relative); the FP64 residual ||b - A x|| <= cg_tol ||b|| is
// the stopping rule in both precisions.
PcgArgs pcg_args_newmark(Sim *s) {
    const Mesh *m = s->mesh;
    PcgArgs a = make_args(s, m->As, s->A_val.p, s->A_rec, s->Dinv.p, s->rhs.p, s->x.p, s->cg_r.p, s->cg_z.p, s->cg_q.p,
                          s->cg_p0.p, s->cg_p1.p, s->cg_part.p, &s->dctl.p->cg, s->cfg.cg_tol, 0.0,
                          s->cfg.cg_max_iters, nullptr, 0.0, false, false);
    if (s->mixed && s->A_rec32.p) {
        const size_t ni = s->cg32.n / 6;
        float *v = s->cg32.p;
        a.refine = 1;
        a.inner_tol2 = 1e-10;
        a.rec32 = s->A_rec32.p;
        a.evict_first = s->A_rec32.n > kKeepInL2;
        a.Dhalf32 = s->Dhalf32.p;
        a.b32 = v;
        a.d32 = v + ni;
        a.r32 = v + 2 * ni;
        a.w32 = v + 3 * ni;
        a.p32 = v + 4 * ni;
        a.s32 = v + 5 * ni;
    }
    return a;
}

// the completion: defect in l_b, solution in l_x, stopping at
// max|d - L psi| <= completion_tol * max|rho + wall| (qmax, computed on the device)
PcgArgs pcg_args_completion(Sim *s) {
    const Mesh *m = s->mesh;
    // (in both precisions FP64: the completion is bound by the latency of its
    // iterations, not by their arithmetic, and FP32 corrections took more)
    return make_args(s, m->Ls, m->Ls_val.p, m->L_rec, s->L_Dinv.p, s->l_b.p, s->l_x.p, s->l_r.p, s->l_z.p, s->l_q.p,
                     s->l_p0.p, s->l_p1.p, s->l_part.p, &s->dctl.p->lap, 0.0, s->cfg.init_tol, 20000,
                     &s->dctl.p->qmax, s->cfg.completion_tol, true, false);
}

int pcg_newmark(Sim *s) {
    const Mesh *m = s->mesh;
    if (m->n_int_edges == 0) return PIC_OK;
    // the learned preconditioner takes over once it has weights; until then
    // (the steps whose systems it trains on) Jacobi-PCG runs
    if (s->cfg.preconditioner == PIC_PRECOND_GNN && s->gnn.trained) {
        int iters = 0, rc = fpcg_newmark(s, &iters);
        if (rc) return rc;
        s->gnn_iters = iters;
        FP_CUDA(cudaMemcpyAsync(&s->dctl.p->cg.iters, &s->gnn_iters, sizeof(int), cudaMemcpyHostToDevice, s->stream));
        return PIC_OK;
    }
    PcgArgs a = pcg_args_newmark(s);
    return launch_pcg_runs(&a, 1, s->cfg.solver_blocks_per_sm, s->stream);
}

// Residual of Jacobi-PCG on the last Newmark system (b = rhs) from x = 0
// after `iters` iterations, into r_out (device, interior edges); training
// samples of the learned preconditioner.  Overwrites the solver's scratch
// vectors and x (which holds no state between steps).
int newmark_truncated_residual(Sim *s, int iters, double *r_out) {
    const Mesh *m = s->mesh;
    const int n = m->n_int_edges;
    if (n == 0) return PIC_OK;
    PcgArgs a = pcg_args_truncated(s, iters);
    int rc = launch_pcg_runs(&a, 1, s->cfg.solver_blocks_per_sm, s->stream);
    if (rc) return rc;
    FP_CUDA(cudaMemcpyAsync(r_out, s->cg_r.p, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->stream));
    return PIC_OK;
}

// Node-Laplacian solve on interior nodes from x = 0.  Stops at
// ||r|| <= tol ||b||, or, with abs_src, at max|r| <= abs_factor * (*abs_src)
// (relative init_tol instead when *abs_src is 0).
int laplacian_solve(Sim *s, const double *rhs_int, double *x_int, double tol, const double *abs_src,
                    double abs_factor) {
    const Mesh *m = s->mesh;
    if (m->n_int_nodes == 0) return PIC_OK;
    PcgArgs a = make_args(s, m->Ls, m->Ls_val.p, m->L_rec, s->L_Dinv.p, rhs_int, x_int, s->l_r.p, s->l_z.p, s->l_q.p,
                          s->l_p0.p, s->l_p1.p, s->l_part.p, &s->dctl.p->lap, tol, s->cfg.init_tol, 20000, abs_src,
                          abs_factor, true, false);
    return launch_pcg_runs(&a, 1, s->cfg.solver_blocks_per_sm, s->stream);
}

// The multigrid solve's arguments: the hierarchy of mesh m, its vectors at v
// (b, x, r, p, q, z, z_old) and its FP32 scratch at f (mg_scratch floats)
static size_t mg_scratch(const Mesh *m) {
    return 3 * (size_t)m->n_int_nodes + 5 * (size_t)m->mg_n1 + 2 * (size_t)m->mg_n2;
}
static MgArgs mg_args(const Mesh *m, double *const v[7], float *f) {
    const int n0 = m->n_int_nodes, n1 = m->mg_n1, n2 = m->mg_n2;
    MgArgs a{};
    a.n0 = n0;
    a.n1 = n1;
    a.n2 = n2;
    a.n_slices = m->Ls.n_slices;
    a.sp = m->Ls.ptr.p;
    a.sw = m->Ls.width.p;
    a.col = m->Ls.col.p;
    a.Lv = m->Ls_val.p;
    a.L32 = m->mg_l0_32.p;
    a.w0 = m->mg_w0.p;
    a.w1 = m->mg_w1.p;
    a.p0p = m->mg_p0.rowptr.p;
    a.p0c = m->mg_p0.col.p;
    a.p0v = m->mg_p0v.p;
    a.r0p = m->mg_r0.rowptr.p;
    a.r0c = m->mg_r0.col.p;
    a.r0v = m->mg_r0v.p;
    a.l1p = m->mg_l1.rowptr.p;
    a.l1c = m->mg_l1.col.p;
    a.l1v = m->mg_l1v.p;
    a.agg1 = m->mg_agg1.p;
    a.r1p = m->mg_r1.rowptr.p;
    a.r1c = m->mg_r1.col.p;
    a.l2inv = m->mg_l2inv.p;
    a.s0 = m->mg_scale;
    a.b = v[0];
    a.x = v[1];
    a.r = v[2];
    a.p = v[3];
    a.q = v[4];
    a.z = v[5];
    a.zo = v[6];
    a.r32 = f;
    a.z0 = f + n0;
    a.t0 = f + 2 * (size_t)n0;
    a.r1 = f + 3 * (size_t)n0;
    a.z1 = a.r1 + n1;
    a.z1b = a.z1 + n1;
    a.t1 = a.z1b + n1;
    a.d1 = a.t1 + n1;
    a.r2 = a.d1 + n1;
    a.z2 = a.r2 + n2;
    a.max_iters = 2000;
    a.spin_limit = (int)kSpinLimit;
    return a;
}

// The completion's (defect in l_b, solution in l_x, the same stopping rule as
// the Jacobi-PCG); allocates the FP32 scratch on first use.
static int mg_args(Sim *s, MgArgs &a) {
    const Mesh *m = s->mesh;
    if (!s->mg32.p) {
        int rc = s->mg32.alloc(mg_scratch(m));
        if (rc) return rc;
    }
    double *const v[7] = {s->l_b.p, s->l_x.p, s->l_r.p, s->l_p0.p, s->l_q.p, s->l_z.p, s->l_p1.p};
    a = mg_args(m, v, s->mg32.p);
    Control *dc = s->dctl.p;
    a.part = s->l_part.p;
    a.st = &dc->lap;
    a.gb = &dc->gbar2;
    a.abs_src = &dc->qmax;
    a.abs_factor = s->cfg.completion_tol;
    a.fallback_tol2 = s->cfg.init_tol * s->cfg.init_tol;
    a.status = &dc->status;
    if (s->cfg.barrier_spin_limit > 0) a.spin_limit = s->cfg.barrier_spin_limit;
    return PIC_OK;
}

// launches a multigrid solve on `per_sm` blocks per SM (0: one)
static int launch_mg(MgArgs &a, int per_sm, cudaStream_t st) {
    static CoopKernel kernel((const void *)k_mg_pcg, kMgThreads, 0);
    const int fit = kernel.per_sm();
    if (fit <= 0) {
        set_error("the multigrid completion needs a device with cooperative launch");
        return PIC_ERR_CUDA;
    }
    { k_reset_gbar<<<1, 1, 0, st>>>(a.gb); note_launch(); }
    void *args[] = {&a};
    return kernel.launch(std::max(1, std::min(fit, std::max(per_sm, 1))) * sm_count(), args, st);
}

int mg_completion(Sim *s) {
    const int n0 = s->mesh->n_int_nodes;
    if (n0 == 0) return PIC_OK;
    MgArgs a;
    int rc = mg_args(s, a);
    if (rc) return rc;
    return launch_mg(a, s->cfg.solver_blocks_per_sm, s->stream);
}

// ---------------------------------------------------------------------------
// Completion solves of a batch in one cooperative launch: members whose mesh
// has a multigrid hierarchy run the multigrid-preconditioned PCG (as
// pic_step does), the others Jacobi-PCG; run r owns blocks [block0, block0 +
// blocks), its own grid barrier and partials.  The run records do not change
// from step to step (every pointer is a member's fixed buffer), so the table
// is written to device memory once, outside any stream capture, and the
// launches (also the captured ones) only read it.
// ---------------------------------------------------------------------------
struct CompletionRun {
    int kind;            // 1: multigrid, 0: Jacobi-PCG
    int block0, blocks, pad;
    PcgArgs pcg;
    MgArgs mg;
};
struct CompletionTable {
    int n_runs, total_blocks, any_wide, pad;
    CompletionRun run[kMaxBatchRuns];
};

template <bool ANYWIDE>
__global__ void __launch_bounds__(kThreads, ANYWIDE ? 3 : 4) k_completion_batched(const CompletionTable *__restrict__ T) {
    __shared__ double shv[4 * kThreads];
    __shared__ unsigned long long shm[kThreads];
    // the block's run record in shared memory (read through a dynamic index
    // from global memory, every use would be a load)
    __shared__ __align__(16) CompletionRun sr;
    __shared__ int s_ri;
    if (threadIdx.x == 0) {
        int ri = 0;
        while (ri + 1 < T->n_runs && (int)blockIdx.x >= T->run[ri + 1].block0) ri++;
        s_ri = ri;
    }
    __syncthreads();
    {
        const int *src = reinterpret_cast<const int *>(&T->run[s_ri]);
        int *dst = reinterpret_cast<int *>(&sr);
        for (int k = threadIdx.x; k < (int)(sizeof(CompletionRun) / sizeof(int)); k += blockDim.x) dst[k] = src[k];
    }
    __syncthreads();
    constexpr int kRing = ANYWIDE ? kBatchRingWide : kBatchRing;
    const int bid = (int)blockIdx.x - sr.block0;
    if (sr.kind) mg_body<kThreads>(sr.mg, sr.blocks, bid, shv, shm);
    else if (ANYWIDE && sr.pcg.wide) pcg_body<false, true, kThreads, kBatchRingWide>(sr.pcg, sr.blocks, bid, s_ring, shv, shm);
    else pcg_body<false, false, kThreads, kRing>(sr.pcg, sr.blocks, bid, s_ring, shv, shm);
}
static CoopKernel &completion_kernel(bool any_wide) {
    static CoopKernel narrow((const void *)k_completion_batched<false>, kThreads, kBatchRing);
    static CoopKernel wide((const void *)k_completion_batched<true>, kThreads, kBatchRingWide);
    return any_wide ? wide : narrow;
}

__global__ void k_reset_completion_barriers(const CompletionTable *__restrict__ T) {
    const int r = threadIdx.x;
    if (r < T->n_runs) {
        GridBarrier *gb = T->run[r].kind ? T->run[r].mg.gb : T->run[r].pcg.gb;
        gb->count = 0;
        gb->timeout = 0;
    }
}

size_t completion_table_bytes() { return sizeof(CompletionTable); }

bool completion_uses_multigrid(Sim *const *sims, int n) {
    for (int i = 0; i < n; i++)
        if (sims[i]->mesh->mg_levels > 0 && sims[i]->mesh->n_int_nodes > 0 && sims[i]->mesh->n_int_edges > 0) return true;
    return false;
}

// Fills and uploads the table for the members with a completion to solve
// (synchronously: call with nothing in flight that reads the table).  Blocks
// go to the runs in proportion to their interior nodes' slices, at most one
// warp per slice, up to blocks_per_sm (0: as many as fit) on every SM.
int prepare_completion_table(Sim *const *sims, int n, int blocks_per_sm, void *table_dev, int *n_runs,
                             int *total_blocks) {
    std::vector<CompletionTable> host(1);
    CompletionTable &T = host[0];
    std::memset(&T, 0, sizeof(T));
    std::vector<long> slices;
    for (int i = 0; i < n; i++) {
        Sim *s = sims[i];
        const Mesh *m = s->mesh;
        if (m->n_int_edges == 0 || m->n_int_nodes == 0) continue;
        CompletionRun &r = T.run[T.n_runs++];
        if (m->mg_levels > 0) {
            r.kind = 1;
            int rc = mg_args(s, r.mg);
            if (rc) return rc;
        } else {
            r.kind = 0;
            r.pcg = pcg_args_completion(s);
        }
        if (!r.kind && r.pcg.wide) T.any_wide = 1;
        slices.push_back(std::max(1, (m->n_int_nodes + 31) / 32));
    }
    const int fit = completion_kernel(T.any_wide != 0).per_sm();
    if (fit <= 0) {
        set_error("the batched completion needs a device with cooperative launch");
        return PIC_ERR_CUDA;
    }
    const int per_sm = blocks_per_sm > 0 ? std::min(fit, blocks_per_sm) : fit;
    const int budget = per_sm * sm_count();
    if (T.n_runs > budget) {
        set_error("more batched solves than co-resident blocks");
        return PIC_ERR_INVALID_ARG;
    }
    long want_total = 0, total_slices = 0;
    std::vector<int> want(T.n_runs), got(T.n_runs);
    for (int r = 0; r < T.n_runs; r++) {
        want[r] = (int)std::max(1L, std::min((long)kMaxPcgBlocks, (slices[r] + kSlicesPerBlock - 1) / kSlicesPerBlock));
        want_total += want[r];
        total_slices += slices[r];
    }
    long total = 0;
    for (int r = 0; r < T.n_runs; r++) {
        got[r] = want_total <= budget ? want[r]
                                      : std::max(1, std::min(want[r], (int)((double)budget * slices[r] / total_slices)));
        total += got[r];
    }
    while (total > budget) {
        int big = 0;
        for (int r = 1; r < T.n_runs; r++)
            if (got[r] > got[big]) big = r;
        got[big]--;
        total--;
    }
    int b0 = 0;
    for (int r = 0; r < T.n_runs; r++) {
        T.run[r].block0 = b0;
        T.run[r].blocks = got[r];
        b0 += got[r];
    }
    T.total_blocks = b0;
    FP_CUDA(cudaMemcpy(table_dev, &T, sizeof(T), cudaMemcpyHostToDevice));
    *n_runs = T.n_runs;
    *total_blocks = T.any_wide ? -T.total_blocks : T.total_blocks;
    return PIC_OK;
}

// One launch of the table's solves on st.  total_blocks: the table's block count,
// negative when a run's records are wide.
int launch_completion_table(const void *table_dev, int n_runs, int total_blocks, cudaStream_t st) {
    if (n_runs <= 0) return PIC_OK;
    const CompletionTable *T = static_cast<const CompletionTable *>(table_dev);
    { k_reset_completion_barriers<<<1, kMaxBatchRuns, 0, st>>>(T); note_launch(); }
    void *args[] = {&T};
    return completion_kernel(total_blocks < 0).launch(std::abs(total_blocks), args, st);
}

// Completion of the field solve on the gradient subspace: the part of the
// residual the discrete divergence sees, d = G_int^T (b - A x), equals (with
// G^T K = 0, G^T C^T = 0 and G_int^T I = 0, since no interior node touches a
// wall-face edge) G_int^T [M (2e - e' - x) - d2 Gbar] for the wave form,
// G_int^T [M (e' - x) - (Gbar^{n+1} - Gbar^{n-1})] for the Newmark Maxwell
// form and G_int^T [M (e - x) - (Gbar^{n+1} - Gbar^n)] for the backward
// difference.  Solving (G^T M G) psi = d and adding G psi removes it (A G = M G), so
// the Gauss residual does not drift with the CG tolerance (Sec. III.A notes
// that the linear solve is the only source of error).  The charge is not used.
int gc_prepare(Sim *s) {
    const Mesh *m = s->mesh;
    const int ni = m->n_int_edges, nin = m->n_int_nodes;
    if (ni == 0 || nin == 0) return PIC_OK;
    { k_gc_t<<<(ni + 255) / 256, 256, 0, s->stream>>>(ni, s->cfg.form, s->e.p, s->e_prev.p, s->x.p, s->ev.p); note_launch(); }
    { k_gc_w_sell<<<grid_for_slices(m->As.n_slices), kThreads, 0, s->stream>>>(ni, m->As.n_slices, m->As.ptr.p, m->As.width.p, m->As.col.p, m->M_val.p, s->cfg.form, s->ev.p, s->g_new.p, s->g.p, s->g_prev.p, s->w_edge.p); note_launch(); }
    { k_gc_d<<<(nin + 255) / 256, 256, 0, s->stream>>>(nin, m->int_node.p, m->n2e.rowptr.p, m->n2e.col.p, m->n2e_sgn.p,
                                                     ni, s->w_edge.p, s->l_b.p); note_launch(); }
    // stopping threshold: completion_tol * max_n |rho_n + wall_n| (charge at t^{n+1})
    { k_max_abs_sum<<<grid_for_elems(m->n_nodes), kThreads, 0, s->stream>>>(m->n_nodes, s->rho.p, s->wall.p, s->diag_part.p, &s->dctl.p->diag.count, &s->dctl.p->qmax); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

int gc_finish(Sim *s) {
    const Mesh *m = s->mesh;
    const int ni = m->n_int_edges, nin = m->n_int_nodes;
    if (ni == 0 || nin == 0) return PIC_OK;
    { k_gc_apply<<<(ni + 255) / 256, 256, 0, s->stream>>>(ni, m->edge_nodes.p, m->node_int.p, s->l_x.p, s->x.p); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

int faraday_update(Sim *s) {
    const Mesh *m = s->mesh;
    { k_faraday<<<(m->n_faces + 255) / 256, 256, 0, s->stream>>>(m->n_faces, m->f2e.p, s->cfg.form, s->cfg.dt, s->x.p,
                                                                s->e.p, s->e_prev.p, s->b.p, s->b_prev.p, s->b_new.p); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

// diagnostics of the state after a step (fields already rotated: e = e^{n+1})
int compute_diagnostics(Sim *s) {
    const Mesh *m = s->mesh;
    DiagDev *dg = &s->dctl.p->diag;
    const int ni = m->n_int_edges;
    DiagArgs a{};
    if (ni > 0) {
        system_coefficients(s, &a.c4, &a.ci);
        a.n = ni;
        a.n_slices = m->As.n_slices;
        a.sp = m->As.ptr.p, a.sw = m->As.width.p, a.col = m->As.col.p;
        a.Mv = m->M_val.p, a.Kv = m->K_val.p;
        a.x = s->e.p, a.rhs = s->rhs.p, a.me = s->me.p;
    }
    a.nt = m->n_tets, a.tf = m->tet_face.p, a.sign = m->tet_sign.p;
    a.nf = m->n_faces, a.f_slices = m->Hs.n_slices;
    a.fp = m->Hs.ptr.p, a.fw = m->Hs.width.p, a.fcol = m->Hs.col.p;
    a.Hv = m->Hs_val.p, a.b = s->b.p;
    a.n_ke = s->n_ke_parts, a.ke = s->ke_part.p;
    a.part = s->diag_part.p, a.dg = dg;
    const int grid = grid_for_slices(std::max(a.n_slices, a.f_slices));
    if (ni > 0 && m->n_abs_faces > 0) {
        a.Iv = m->I_val.p;
        { k_diag_fields<true><<<grid, kThreads, 0, s->stream>>>(a); note_launch(); }
    } else {
        a.ci = 0.0;
        { k_diag_fields<false><<<grid, kThreads, 0, s->stream>>>(a); note_launch(); }
    }
    { k_diag_nodes<<<grid_for_elems(m->n_nodes), kThreads, 0, s->stream>>>(
        m->n_nodes, m->n2e.rowptr.p, m->n2e.col.p, m->n2e_sgn.p, ni, s->dg.p, s->me.p, s->rho.p, s->rho_prev.p,
        s->wall.p, s->wall_prev.p, s->rho_bg.p, m->node_bnd.p, s->diag_part.p, dg); note_launch(); }
    FP_CUDA(cudaGetLastError());
    return PIC_OK;
}

// initial electrostatic field: (G^T M G) phi = rho + rho_bg on interior nodes, e = -G phi
int init_fields(Sim *s) {
    const Mesh *m = s->mesh;
    const int nin = m->n_int_nodes, ni = m->n_int_edges;
    if (nin > 0) {
        { k_node_to_int<<<(nin + 255) / 256, 256, 0, s->stream>>>(nin, m->int_node.p, s->rho.p, s->rho_bg.p, s->l_b.p); note_launch(); }
            int rc = laplacian_solve(s, s->l_b.p, s->l_x.p, s->cfg.init_tol, nullptr, 0.0);
        if (rc) return rc;
        FP_CUDA(cudaMemsetAsync(s->phi.p, 0, sizeof(double) * m->n_nodes, s->stream));
        { k_int_to_node<<<(nin + 255) / 256, 256, 0, s->stream>>>(nin, m->int_node.p, s->l_x.p, s->phi.p); note_launch(); }
        if (ni > 0)
            { k_minus_grad<<<(ni + 255) / 256, 256, 0, s->stream>>>(ni, m->edge_nodes.p, m->node_int.p, s->l_x.p, s->e.p,
                                                                  s->e_prev.p); note_launch(); }
        FP_CUDA(cudaGetLastError());
    }
    return PIC_OK;
}

int read_control(Sim *s) {
    FP_CUDA(cudaMemcpyAsync(s->hctl, s->dctl.p, sizeof(Control), cudaMemcpyDeviceToHost, s->stream));
    FP_CUDA(cudaStreamSynchronize(s->stream));
    return PIC_OK;
}


// ---------------------------------------------------------------------------
// Allocation-free electrostatic solve.
//
// Some callers cannot allocate device memory at the point where they need a
// solve: a host runtime that hands out all device memory from its own pool and
// forbids libraries to allocate, or a service whose memory budget was fixed
// when it started.  For them pic_electrostatic_solve_noalloc runs the node
// Laplacian's persistent solves, preconditioned by the mesh's multigrid
// hierarchy where it has one and by its diagonal otherwise, with the working
// vectors in the fixed array below instead of buffers it allocates.  One
// launch and one wait: 12.9 -> 2.0 ms on the 48^3 mesh (103,823 interior
// nodes, 1e-12) against the two launches an iteration and the wait every 16
// iterations of a Jacobi-PCG in separate kernels.
//
// The array is a file-scope device variable: every GPU on which this library's
// solver module is loaded holds its 37.9 MB until the process exits.  It
// bounds the problem to kNoAllocMaxNodes interior nodes.  All calls share it
// and it keeps the last call's contents; a call holds the device's lock until
// its work on the stream has ended, so calls from several threads or on several
// streams follow one another.
// ---------------------------------------------------------------------------
constexpr int kNoAllocMaxNodes = 524288;
// Multigrid iterations before the solve goes on with the diagonal as its
// preconditioner: meshes of ordinary shapes take 10 to 30, tangled ones (24^3,
// nodes moved by 0.6 of a cell: 160) are left to the cheaper iterations
constexpr int kNoAllocMgIters = 100;
constexpr size_t kNoAllocVectors = 9;   // b, x, r, p, q, z and z_old (or D^-1), then FP32 scratch
constexpr size_t kNoAllocDoubles = kNoAllocVectors * kNoAllocMaxNodes + 8 * (size_t)kMaxBlocks + 64;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];

// The call's return code for what its solve left: state flags and status word
int noalloc_outcome(int done, int failed, uint32_t status) {
    if (status & ST_BARRIER) {
        set_error("pic_electrostatic_solve_noalloc: a persistent solver kernel timed out at a grid barrier");
        return PIC_ERR_CUDA;
    }
    if (failed || !done) {
        set_error("pic_electrostatic_solve_noalloc: PCG did not reach the tolerance");
        return PIC_ERR_CG_NO_CONVERGENCE;
    }
    return PIC_OK;
}

namespace {
std::mutex g_noalloc_mutex;                            // of the address table
constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_busy[kNoAllocMaxDevices];         // of a device's array
double *g_noalloc_ptr[kNoAllocMaxDevices] = {};

// device address of the scratch array on the current device (looked up once
// per device)
int noalloc_scratch(double **out) {
    int dev = 0;
    FP_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kNoAllocMaxDevices) {
        set_error("pic_electrostatic_solve_noalloc: device index out of range");
        return PIC_ERR_INVALID_ARG;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        g_noalloc_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return PIC_OK;
}

// what a solve leaves, read back in one copy
struct NoAllocResult {
    CgState st;
    GridBarrier gb;
    uint32_t status;
};
static_assert(sizeof(NoAllocResult) <= 64 * sizeof(double), "behind the partials");

// the solve in the scratch array at base, which the caller holds
int noalloc_solve(const Mesh *m, const double *rho_nodes, double *phi_nodes, double tol, double *base,
                  cudaStream_t st) {
    const int nin = m->n_int_nodes;
    FP_CUDA(cudaMemsetAsync(phi_nodes, 0, sizeof(double) * m->n_nodes, st));
    int rc;
    double *v[7];
    for (size_t k = 0; k < 7; k++) v[k] = base + k * kNoAllocMaxNodes;
    float *scratch = reinterpret_cast<float *>(base + 7 * (size_t)kNoAllocMaxNodes);
    double *b = v[0], *x = v[1], *part = base + kNoAllocVectors * kNoAllocMaxNodes;
    NoAllocResult *res = reinterpret_cast<NoAllocResult *>(part + 8 * (size_t)kMaxBlocks);
    CgState *dst = &res->st;
    GridBarrier *gb = &res->gb;
    uint32_t *status = &res->status;
    // the vectors are padded to whole slices, zeros past the rows
    const size_t pad = (size_t)(nin + 31) / 32 * 32 * sizeof(double);
    for (size_t k = 0; k < 7; k++) FP_CUDA(cudaMemsetAsync(v[k], 0, pad, st));
    FP_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), st));
    { k_node_to_int<<<(nin + 255) / 256, 256, 0, st>>>(nin, m->int_node.p, rho_nodes, nullptr, b); note_launch(); }
    FP_CUDA(cudaGetLastError());
    // waits for a solve and reads back what it left
    NoAllocResult h{};
    auto finish = [&]() -> int {
        FP_CUDA(cudaMemcpyAsync(&h, res, sizeof(h), cudaMemcpyDeviceToHost, st));
        FP_CUDA(cudaStreamSynchronize(st));
        return PIC_OK;
    };
    bool solved = false;
    const bool hierarchy = m->mg_levels > 0 && mg_scratch(m) <= 4 * (size_t)kNoAllocMaxNodes;
    if (hierarchy) {
        MgArgs a = mg_args(m, v, scratch);
        a.part = part;
        a.st = dst;
        a.gb = gb;
        a.abs_src = nullptr;
        a.fallback_tol2 = tol * tol;
        a.status = status;
        a.max_iters = kNoAllocMgIters;
        a.verify = 1;
        if ((rc = launch_mg(a, 0, st)) || (rc = finish())) return rc;
        // (short of the tolerance here is not a failure of the call)
        if (h.status & ST_BARRIER) return noalloc_outcome(h.st.done, h.st.failed, h.status);
        solved = h.st.done && !h.st.failed;
    }
    if (!solved) {
        if (!m->L_rec.p) {
            set_error("pic_electrostatic_solve_noalloc: the mesh has no device copy yet (create a simulation on it first)");
            return PIC_ERR_STATE;
        }
        // after the multigrid solve: from its iterate, the other vectors cleared
        const bool x_zero = !hierarchy || !std::isfinite(h.st.rr);
        for (size_t k = x_zero ? 1 : 2; k < 7; k++) FP_CUDA(cudaMemsetAsync(v[k], 0, pad, st));
        FP_CUDA(cudaMemsetAsync(status, 0, sizeof(uint32_t), st));
        { k_recip_diag<<<(nin + 255) / 256, 256, 0, st>>>(nin, m->L_diag.p, v[6]); note_launch(); }
        PcgArgs a = matrix_args(m->Ls, m->Ls_val.p, m->L_rec);
        a.Dinv = v[6];
        a.b = b;
        a.x = x;
        a.r = v[2];
        a.u = v[5];
        a.w = reinterpret_cast<double *>(scratch);
        a.p = v[3];
        a.s = v[4];
        FP_CUDA(cudaMemsetAsync(a.w, 0, pad, st));
        a.part = part;
        a.st = dst;
        a.gb = gb;
        a.tol2 = tol * tol;
        a.abs_inf = -1.0;
        a.status = status;
        a.max_iters = 20000;
        a.x_zero = x_zero;
        a.spin_limit = (int)kSpinLimit;
        if ((rc = launch_pcg_runs(&a, 1, 0, st)) || (rc = finish()) ||
            (rc = noalloc_outcome(h.st.done, h.st.failed, h.status)))
            return rc;
    }
    { k_int_to_node<<<(nin + 255) / 256, 256, 0, st>>>(nin, m->int_node.p, x, phi_nodes); note_launch(); }
    FP_CUDA(cudaGetLastError());
    FP_CUDA(cudaStreamSynchronize(st));
    return PIC_OK;
}
}  // namespace

int electrostatic_solve_noalloc(const Mesh *m, const double *rho_nodes, double *phi_nodes, double tol,
                                cudaStream_t st) {
    const int nin = m->n_int_nodes;
    if (nin > kNoAllocMaxNodes) {
        set_error("pic_electrostatic_solve_noalloc: " + std::to_string(nin) + " interior nodes exceed the limit of " +
                  std::to_string(kNoAllocMaxNodes));
        return PIC_ERR_INVALID_ARG;
    }
    if (!m->uploaded) {
        set_error("pic_electrostatic_solve_noalloc: the mesh has no device copy yet (create a simulation on it first)");
        return PIC_ERR_STATE;
    }
    if (!(tol > 0) || !rho_nodes || !phi_nodes) {
        set_error("pic_electrostatic_solve_noalloc: needs tol > 0 and device arrays for rho and phi");
        return PIC_ERR_INVALID_ARG;
    }
    int dev = -1;
    FP_CUDA(cudaGetDevice(&dev));
    if (dev != m->device) {
        set_error("pic_electrostatic_solve_noalloc: the current device (" + std::to_string(dev) +
                  ") is not the device that holds the mesh (" + std::to_string(m->device) + ")");
        return PIC_ERR_INVALID_ARG;
    }
    // the result is read back and waited for below, which a stream under
    // capture does not allow
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    FP_CUDA(cudaStreamIsCapturing(st, &cap));
    if (cap != cudaStreamCaptureStatusNone) {
        set_error("pic_electrostatic_solve_noalloc: the stream is being captured; the call waits on the stream "
                  "for its result");
        return PIC_ERR_STATE;
    }
    double *base = nullptr;
    int rc = noalloc_scratch(&base);
    if (rc) return rc;
    if (nin == 0) {
        FP_CUDA(cudaMemsetAsync(phi_nodes, 0, sizeof(double) * m->n_nodes, st));
        return PIC_OK;
    }
    std::lock_guard<std::mutex> hold(g_noalloc_busy[dev]);
    rc = noalloc_solve(m, rho_nodes, phi_nodes, tol, base, st);
    if (rc) cudaStreamSynchronize(st);   // what was enqueued before the error leaves the array, too
    return rc;
}

}  // namespace fp
