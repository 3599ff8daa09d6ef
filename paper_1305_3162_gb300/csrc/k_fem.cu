// Kernels of the scalar potential (Alg. 1): phi_1 from the free subsystem of
// the P1 Dirichlet problem (Sec. 2.1), the boundary charges
// g = m.n - dphi_1/dn, and phi_1 + phi_2.
//
// The free subsystem S x = b is solved by iterative refinement: Jacobi-
// preconditioned conjugate gradients in FP32 reduce the residual of the
// current correction equation by FEM_INNER, the correction is added to the
// FP64 solution, and the residual b - S x is recomputed in FP64 (the FP64
// pipe of this GPU is a small fraction of its FP32 rate, while each
// correction needs only a few digits).  Per-thread FP64 work is confined to
// the load, the FP64 residual and the correction; the load and the residual
// form their scalars in their last block.
//
// The inner iteration is the conjugate-gradient recurrence with a single
// reduction per step (Chronopoulos and Gear): with u = D^-1 r and w = S u,
//   p_k = u_k + beta_k p_{k-1},  s_k = w_k + beta_k s_{k-1}  (s_k = S p_k),
//   x += alpha_k p_k,  r_{k+1} = r_k - alpha_k s_k,  u_{k+1} = D^-1 r_{k+1},
//   w_{k+1} = S u_{k+1},
//   gamma_{k+1} = r_{k+1} . u_{k+1},  delta_{k+1} = w_{k+1} . u_{k+1},
//   beta_{k+1} = gamma_{k+1} / gamma_k,
//   alpha_{k+1} = gamma_{k+1} / (delta_{k+1} - beta_{k+1} gamma_{k+1} / alpha_k),
// which needs both dot products at one point of the step.  Systems of up to
// SOLVE_THREADS 10 rows a block (0.78M free nodes) are solved in one launch
// (k_cg_solve, further down, with a better preconditioner); for larger ones a
// launch does a step: every vector update is per row, and u_{k+1} at the columns the
// product gathers is formed there from r_k, w_k and s_{k-1}, which a row
// keeps together with its 1 / diagonal in one 16-byte record (the step
// reads the records of one parity and writes those of the other).  A launch
// leaves its blocks' partial sums of gamma_{k+1}, delta_{k+1} and r.r; every
// block of the next launch adds them itself, in one fixed order, and derives
// alpha_{k+1} and beta_{k+1}, so all blocks hold the same scalars, no launch
// ends in a one-block tail, and the solve repeats bitwise.  An inner
// iteration starts with a set-up launch (the same kernel with alpha = beta =
// 0), which forms w_0 = S u_0 and the first partial sums.  The launches are
// chained by programmatic dependent launch: before its dependency wait a
// thread loads its row's first column indices and entries (plan data).  The
// inner steps give each row one thread over the matrix in slices of 32 rows
// (every lane busy with its own row's update, coalesced reads of the
// entries); the load uses groups of 8 lanes per row over CSR.  Launches
// after the inner stop return at once, so the rest of a pass of the solve
// graph's inner loop costs only empty launches.
#include <algorithm>
#include <cmath>

#include "dev_common.cuh"
#include "slp_fem.h"

namespace slp {
namespace {

constexpr int NT = FEM_THREADS;
constexpr int GROUP = 8;          // lanes per matrix row
constexpr int ROWS = NT / GROUP;  // rows per block and step

// Sum over the block in a fixed order (warp shuffles, then thread 0 adds
// the warps' sums); valid in thread 0 only.  The inner steps sum in FP32:
// this GPU's FP64 pipe is slow enough that a chain of FP64 operations in the
// last block's tail would cost more than the step's product.
template <typename V> __device__ V block_sum(V v, V *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();  // sh may still be read by a previous call
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    V t = V(0);
    if (threadIdx.x == 0)
        for (int w = 0; w < NT / 32; ++w) t += sh[w];
    return t;
}

// Sum over the GROUP lanes of a row group; the sum lands in the group's first lane.
template <typename V> __device__ V group_sum(V v) {
    for (int o = GROUP / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, GROUP);
    return v;
}

// True when the flag is set (read once per block, so that every thread of
// the block takes the same branch).
__device__ bool block_flag(const int *flag) {
    __shared__ int s_flag;
    if (threadIdx.x == 0) s_flag = *(volatile const int *)flag;
    __syncthreads();
    return s_flag != 0;
}

__device__ __forceinline__ double *partials(const FemDev &d, double) { return d.part; }

// Store this block's K partial sums (held by thread 0); returns true in the
// block that arrives last, after which that block may read every block's
// partials (and the arrival counter is reset for the next launch).
template <int K, typename V>
__device__ bool arrive(const FemDev &d, const V (&v)[K], unsigned *counter) {
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        V *part = partials(d, V(0));
        for (int k = 0; k < K; ++k) part[k * d.nblk_max + blockIdx.x] = v[k];
        __threadfence();
        const unsigned t = atomicAdd(counter, 1u);
        s_last = (t == gridDim.x - 1);
        if (s_last) *counter = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// Sums of the first n partials of rows 0..K-1 in the last block: every
// thread loads its strided share of all K rows before adding (the loads are
// independent, so they are in flight together: this tail runs while the
// rest of the GPU idles), then a fixed tree; valid in thread 0.
template <int K, typename V>
__device__ void sum_partials(const FemDev &d, int n, V (&out)[K], V *sh) {
    constexpr int PER = 8;  // partials per thread and row loaded at once
    const V *part = partials(d, V(0));
    V v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = V(0);
    for (int i0 = 0; i0 < n; i0 += NT * PER) {
        V buf[K][PER];
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int i = i0 + j * NT + threadIdx.x;
                buf[k][j] = i < n ? __ldcg(part + k * d.nblk_max + i) : V(0);
            }
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int j = 0; j < PER; ++j) v[k] += buf[k][j];
    }
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = block_sum(v[k], sh);
}

template <typename T> struct Vec4;
template <> struct Vec4<float> { typedef float4 t; };
template <> struct Vec4<double> { typedef double4 t; };

// The last block's bookkeeping of a new FP64 residual rho (|rho|^2 = hh):
// the scale of the next inner problem (its right-hand side is rho / scale,
// of unit mean square, so the FP32 inner sums neither underflow nor
// overflow whatever the units of m), and the outer stopping test.
__device__ __forceinline__ void new_residual(const FemDev &d, CgState &s, double hh) {
    s.rr_hi = hh;
    const double scale = sqrt(hh / (double)d.nf);
    s.scale = scale > 0.0 ? scale : 1.0;
    s.inv_scale = 1.0 / s.scale;
    s.bad = s.bad || !isfinite(hh);
    s.outer_done = s.bad || hh <= d.tol2 * s.bb || s.iter >= d.max_iter;
    s.done = s.outer_done;
}

// b(fn) = B m in the plan's precision from the differences m_col - m_row;
// x = 0 and the first residual is b.  The last block sets up the state.
template <typename T>
__global__ void __launch_bounds__(NT) k_fem_load(FemDev d, const T *__restrict__ m) {
    typedef typename Vec4<T>::t T4;
    __shared__ double sh[NT / 32];
    if (d.parts > 0) {  // no exchange has happened yet
        const int64_t step = (int64_t)gridDim.x * NT, i0 = (int64_t)blockIdx.x * NT + threadIdx.x;
        for (int64_t i = i0; i < d.nhalo; i += step) d.rec[0][i] = d.rec[1][i] = make_uint4(0, 0, 0, 0);
        for (int64_t i = i0; i < (int64_t)d.parts * d.parts; i += step)
            d.psum[0][i] = d.psum[1][i] = make_uint4(0, 0, 0, 0);
    }
    const int gl = threadIdx.x % GROUP;
    const T4 *__restrict__ bv = (const T4 *)d.b_val;
    double bb = 0.0;
    // the loop bound depends on the block only: every lane reaches the shuffles
    for (int64_t i0 = (int64_t)blockIdx.x * ROWS; i0 < d.nf; i0 += (int64_t)gridDim.x * ROWS) {
        const int64_t i = i0 + threadIdx.x / GROUP;
        T b = T(0);
        if (i < d.nf) {
            const int64_t self = d.fnode[i];
            const T mx = m[3 * self], my = m[3 * self + 1], mz = m[3 * self + 2];
            for (int64_t e = d.b_ptr[i] + gl; e < d.b_ptr[i + 1]; e += GROUP) {
                const T4 w = bv[e];
                const int64_t c = d.b_col[e];
                b += w.x * (m[3 * c] - mx) + w.y * (m[3 * c + 1] - my) + w.z * (m[3 * c + 2] - mz);
            }
        }
        b = group_sum(b);
        if (i < d.nf && gl == 0) {
            d.b[i] = (double)b;
            d.rho[i] = (double)b;
            d.x[i] = 0.0;
            bb += (double)b * (double)b;
        }
    }
    const double v[1] = {block_sum(bb, sh)};
    if (!arrive(d, v, &d.st->count[0])) return;
    double t[1];
    sum_partials(d, gridDim.x, t, sh);
    if (threadIdx.x == 0) {
        CgState &s = *d.st;
        s.bb = t[0];
        s.iter = 0;
        s.outer = 0;
        s.bad = 0;
        s.stalled = 0;
        new_residual(d, s, t[0]);
        if (t[0] == 0.0 || d.max_iter <= 0) s.outer_done = s.done = 1;
    }
}

// The FP64 residual rho = b - S x (one thread per row: no FP64 shuffles);
// the last block decides whether the solve is done.
__global__ void __launch_bounds__(NT) k_fem_residual(FemDev d) {
    __shared__ double sh[NT / 32];
    if (block_flag(&d.st->outer_done)) return;
    double hh = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < d.nf; i += (int64_t)gridDim.x * NT) {
        double sx = 0.0;
        for (int64_t e = d.s_ptr[i]; e < d.s_ptr[i + 1]; ++e) sx += d.s_val[e] * d.x[d.s_col[e]];
        const double rho = d.b[i] - sx;
        d.rho[i] = rho;
        hh += rho * rho;
    }
    const double v[1] = {block_sum(hh, sh)};
    if (!arrive(d, v, &d.st->count[1])) return;
    double t[1];
    sum_partials(d, gridDim.x, t, sh);
    if (threadIdx.x == 0) {
        CgState &s = *d.st;
        s.outer += 1;
        new_residual(d, s, t[0]);
    }
}

// Start of an inner iteration (per row): the parity-0 records
// {r_0 = rho / scale, w = 0, s = 0, 1 / diagonal}, correction and direction
// zero; the inner record 0 set for the set-up launch.
__global__ void __launch_bounds__(NT) k_cg_scale(FemDev d) {
    if (block_flag(&d.st->done)) return;
    const double inv = d.st->inv_scale;
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < d.nf; i += (int64_t)gridDim.x * NT) {
        d.xc[i] = 0.f;
        d.p[i] = 0.f;
        d.v[0][i] = make_float4((float)(d.rho[i] * inv), 0.f, 0.f, d.dinv[i]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        CgInner &o = d.st->in[0];
        o.gamma = o.alpha = o.rr0 = 0.f;
        o.mode = 0;
        o.iter = d.st->iter;
    }
}

// Sums over the block of K values, the same in every thread (a fixed order:
// shuffles down to lane 0, then the warps' sums in warp order).
template <int K> __device__ void block_sum_all(float (&v)[K], float (*sh)[NT / 32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) sh[k][warp] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) t += sh[k][w];
        v[k] = t;
    }
}

constexpr int CH = 8;  // matrix entries of a row loaded, and columns gathered, at once

// w += (S u)(row) over the row's entries [k0, width) of its slice (base: the
// lane's first entry), u at each column from its record, CH entries at a
// time; entries past the row's width read the row's own record with weight 0.
__device__ __forceinline__ void row_product(const FemDev &d, const float4 *__restrict__ v0, int64_t base, int width,
                                            int k0, int self, float alpha, float beta, float &w) {
    for (; k0 < width; k0 += CH) {
        int c[CH];
        float a[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            const bool ok = k0 + j < width;
            c[j] = ok ? d.sl_col[base + 32 * (k0 + j)] : self;
            a[j] = ok ? d.sl_val[base + 32 * (k0 + j)] : 0.f;
        }
        float4 g[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) g[j] = v0[c[j]];
#pragma unroll
        for (int j = 0; j < CH; ++j) w += a[j] * (g[j].w * (g[j].x - alpha * (g[j].y + beta * g[j].z)));
    }
}

// One inner launch of parity q (records and partial sums of parity q read,
// those of parity q ^ 1 written): the set-up launch (mode 0) or a step.
// Before the dependency wait a thread takes its row's first 2 CH entries
// (plan data): CH into registers, CH into shared memory.  After it, the
// loads that do not depend on the step's scalars go out together: the stop
// flag, the inner record, the previous launch's partial sums, the first CH
// gathered columns (their addresses are plan data) and the row's own record;
// alpha and beta are formed while they are in flight.
__global__ void __launch_bounds__(NT, 4) k_cg_step(FemDev d, int q) {
    __shared__ float sh_in[3][NT / 32], sh_out[3][NT / 32];
    __shared__ int s_col[CH][NT];
    __shared__ float s_val[CH][NT];
    __shared__ int s_done;
    const int lane = threadIdx.x & 31;
    const int64_t nsl = (d.nf + 31) >> 5, tstep = ((int64_t)gridDim.x * NT) >> 5;
    int64_t t = ((int64_t)blockIdx.x * NT + threadIdx.x) >> 5;
    int64_t base = 0;
    int width = 0;
    int self = 0;
    if (t < nsl) {
        base = d.sl_ptr[t] + lane;
        width = d.sl_w[t];
        self = (int)min(32 * t + lane, d.nf - 1);
    }
    int c[CH];
    float a[CH];
#pragma unroll
    for (int j = 0; j < 2 * CH; ++j) {
        const bool ok = j < width;
        const int cj = ok ? d.sl_col[base + 32 * j] : self;
        const float aj = ok ? d.sl_val[base + 32 * j] : 0.f;
        if (j < CH) {
            c[j] = cj;
            a[j] = aj;
        } else {
            s_col[j - CH][threadIdx.x] = cj;
            s_val[j - CH][threadIdx.x] = aj;
        }
    }
    pdl_wait();
    pdl_trigger();
    int flag = 0;
    if (threadIdx.x == 0) flag = *(volatile const int *)&d.st->done;
    const CgInner in = d.st->in[q];
    const float4 *__restrict__ v0 = d.v[q];
    float4 g[CH];
#pragma unroll
    for (int j = 0; j < CH; ++j) g[j] = v0[c[j]];
    // the previous launch's partial sums: gamma, delta and r.r of its result
    // (read whatever the mode; used only after a step)
    float v[3] = {0.f, 0.f, 0.f};
    {
        const float *part = d.part32 + (size_t)q * 3 * d.nblk_max;
        const int n = (int)gridDim.x;
        for (int i0 = 0; i0 < n; i0 += 2 * NT) {
            float b[3][2];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int ii = i0 + j * NT + threadIdx.x;
                    b[k][j] = ii < n ? __ldcg(part + k * d.nblk_max + ii) : 0.f;
                }
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int j = 0; j < 2; ++j) v[k] += b[k][j];
        }
    }
    if (threadIdx.x == 0) s_done = flag;
    block_sum_all(v, sh_in);  // its barrier also publishes s_done
    if (s_done) return;       // the same in every thread of the block
    float alpha = 0.f, beta = 0.f;
    if (in.mode > 0) {
        const float gm = v[0], dl = v[1], rr = v[2];
        float rr0 = in.rr0;
        if (in.mode == 1) {
            beta = 0.f;
            alpha = gm / dl;
            rr0 = rr;
        } else {
            beta = gm / in.gamma;
            alpha = gm / (dl - beta * gm / in.alpha);
        }
        // a residual that reached the stopping test (exactly zero included,
        // where the coefficients are 0/0) ends the inner iteration
        const bool conv = rr <= d.inner2 * rr0;
        const bool bad = !isfinite(rr) || (!conv && !(isfinite(alpha) && isfinite(beta)));
        const bool stop = bad || conv || in.iter >= d.max_iter;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            CgState &s = *d.st;
            s.gamma = gm;
            s.rr = rr;
            s.iter = stop ? in.iter : in.iter + 1;
            if (stop) {
                s.bad = s.bad || bad;
                s.done = 1;
            } else {
                CgInner &on = s.in[q ^ 1];
                on.gamma = gm;
                on.alpha = alpha;
                on.rr0 = rr0;
                on.mode = 2;
                on.iter = in.iter + 1;
            }
        }
        if (stop) return;  // the same decision in every block
    } else if (blockIdx.x == 0 && threadIdx.x == 0) {
        CgInner &on = d.st->in[q ^ 1];
        on.gamma = on.alpha = on.rr0 = 0.f;
        on.mode = 1;
        on.iter = in.iter;
    }
    float4 *__restrict__ v1 = d.v[q ^ 1];
    float gm = 0.f, dl = 0.f, rr = 0.f;
    // the row update from its own record and the product w of its row
    auto update = [&](int64_t r, float w, float4 rec, float p_old, float x_old) {
        const float p = rec.w * rec.x + beta * p_old;
        const float sn = rec.y + beta * rec.z;
        d.p[r] = p;
        d.xc[r] = x_old + alpha * p;
        const float rn = rec.x - alpha * sn;
        v1[r] = make_float4(rn, w, sn, rec.w);
        const float un = rec.w * rn;
        gm += rn * un;
        dl += w * un;
        rr += rn * rn;
    };
    int64_t i = 32 * t + lane;
    if (t < nsl) {
        // the row's own record and the second chunk's columns, in flight
        // while the first chunk is added
        const bool row = i < d.nf;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        float pold = 0.f, xold = 0.f;
        if (row) {
            o = v0[i];
            pold = d.p[i];
            xold = d.xc[i];
        }
        float4 h[CH];
        if (width > CH) {
#pragma unroll
            for (int j = 0; j < CH; ++j) h[j] = v0[s_col[j][threadIdx.x]];
        }
        // u_{k+1} at column c from r_k, w_k and s_{k-1}
        float w = 0.f;
#pragma unroll
        for (int j = 0; j < CH; ++j) w += a[j] * (g[j].w * (g[j].x - alpha * (g[j].y + beta * g[j].z)));
        if (width > CH) {
#pragma unroll
            for (int j = 0; j < CH; ++j)
                w += s_val[j][threadIdx.x] * (h[j].w * (h[j].x - alpha * (h[j].y + beta * h[j].z)));
        }
        if (width > 2 * CH) row_product(d, v0, base, width, 2 * CH, self, alpha, beta, w);
        if (row) update(i, w, o, pold, xold);
    }
    // further slices of the warp (meshes with more rows than one thread each)
    for (t += tstep; t < nsl; t += tstep) {
        base = d.sl_ptr[t] + lane;
        width = d.sl_w[t];
        i = 32 * t + lane;
        self = (int)min(i, d.nf - 1);
        float w = 0.f;
        row_product(d, v0, base, width, 0, self, alpha, beta, w);
        if (i < d.nf) update(i, w, v0[i], d.p[i], d.xc[i]);
    }
    float vo[3] = {gm, dl, rr};
    block_sum_all(vo, sh_out);
    if (threadIdx.x == 0) {
        float *out = d.part32 + (size_t)(q ^ 1) * 3 * d.nblk_max;
        out[blockIdx.x] = vo[0];
        out[d.nblk_max + blockIdx.x] = vo[1];
        out[2 * d.nblk_max + blockIdx.x] = vo[2];
    }
}

// The correction: x += scale xc (FP64), in its own launch so that the
// residual gathers a complete x.
__global__ void __launch_bounds__(NT) k_fem_correct(FemDev d) {
    if (block_flag(&d.st->outer_done)) return;
    const double scale = d.st->scale;
    for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < d.nf; i += (int64_t)gridDim.x * NT)
        d.x[i] += scale * (double)d.xc[i];
}

// Loop control of the solve graph: WHILE (corrections) { WHILE (inner) {
// FEM_CHUNK inner launches }, correction, residual, next inner start }.  One
// thread sets the handle (the only caller while the kernel runs).  Each loop
// also counts its passes on the device and ends at its bound whatever the
// state says, so both loops end: the corrections at FEM_MAX_OUTER, the inner
// passes (which end by themselves once max_iter steps are done) at a bound
// above that, where the solve is marked bad.
__global__ void k_loop_outer_start(FemDev d, cudaGraphConditionalHandle h) {
    d.st->loops_outer = 0;
    cudaGraphSetConditional(h, d.st->outer_done ? 0u : 1u);
}

__global__ void k_loop_outer_next(FemDev d, cudaGraphConditionalHandle h, int bound) {
    CgState &s = *d.st;
    const int n = ++s.loops_outer;
    cudaGraphSetConditional(h, (!s.outer_done && n < bound) ? 1u : 0u);
}

__global__ void k_loop_inner_start(FemDev d, cudaGraphConditionalHandle h) {
    d.st->loops_inner = 0;
    cudaGraphSetConditional(h, d.st->done ? 0u : 1u);
}

__global__ void k_loop_inner_next(FemDev d, cudaGraphConditionalHandle h, int bound) {
    CgState &s = *d.st;
    const int n = ++s.loops_inner;
    if (!s.done && n >= bound) {
        s.bad = 1;
        s.done = 1;
    }
    cudaGraphSetConditional(h, s.done ? 0u : 1u);
}

// ---------------------------------------------------------------- the solve in one launch
// The same iteration with the rows spread over one resident block per SM, in
// place of a launch per step.  A launch per step cost 7.1 us on the n = 32
// ball (128k rows) and 4.6 us on n = 16 (16k rows): the chained launch, 15.4 MB
// of matrix and 29 MB of gathered 16-byte records through L2 each time.  Here
// a block's rows keep their state (and, up to 16 off-diagonal entries and two
// rows a thread, their matrix rows) in registers, the gathered u of its own
// rows and its halo in shared memory, and a step moves only the halo records
// (about 600 of 16 bytes a block) and one record of partial sums per block.
//
// Exchange e: every block writes {r, w, s, e} of its rows into the halo lists
// of the blocks that need them, and {gamma, delta, Z^T w, e} of its sums into
// every block's list of sums, each list in two copies by the parity of e.  A
// 16-byte access is one access (ld/st .b128), so a reader that finds the
// number e has the record: no fence, no flag, one trip through L2 (560 cycles
// within a die, 900 across).  Only its owner reads a list: lines polled by
// several blocks while others write them cost more than the rest of the step,
// and so do polls by threads that wait for nothing (one record per row, read in
// place, and every thread polling: 5600 cycles an exchange; now 2500 to 4900).
// A block writes exchange e + 2 only after it has read every block's sums of
// e + 1, which that block wrote after it had read its records of e, so two
// copies suffice.  All blocks add the sums in one order and hold the same
// scalars.  The launch is cooperative (all blocks resident); every wait is
// bounded, all of a thread's waits in an exchange together, and a block that
// gives up sets `stalled` and leaves, after which the others' waits run out as
// well.
//
// The system is scaled by its diagonal (S_ij / sqrt(S_ii S_jj), unit
// diagonal).  The preconditioner adds to Jacobi's (the identity here) a coarse
// space of one constant per part: u = r + Z A^-1 Z^T r, Z the parts' indicator
// vectors times z_i = sqrt(S_ii), A = Z^T S Z inverted at set-up.  It removes
// the error modes longer than a part, which plain Jacobi needs most of its
// steps for (n = 32 ball: 289 steps with Jacobi alone, 145), and costs no exchange of its own: the
// sums carry Z^T w of each part, from which every block updates the whole
// coarse residual Z^T r as it does its rows' (s_c = w_c + beta s_c, r_c -=
// alpha s_c), and a block forms the corrections of its own and its halo's
// parts.  The inner iteration stops when r . u has fallen by 1e-8 (the
// residual by 1e-4 in the preconditioner's norm).
//
// Measured, phi_1 (load, solve and all corrections): ball n = 16 672 -> 281 us,
// n = 32 2155 -> 760 us (5.2 us a step: about 2.2 exchange, 0.9 product, the
// rest the coarse correction, sums and barriers), n = 48 7600 -> 5460 us (its
// matrix no longer fits the registers).  The line to the launch chain: a step is
// the slower here from n = 44 on (its matrix comes from L2 to half as many warps),
// but half as many steps are needed.  Chain and one launch, ms: n = 48 (436k
// rows) 8.2 and 5.8, n = 52 (555k) 10.0 and 7.9, n = 56 (693k, ten rows a
// thread) 15.1 and 13.4 to 14.3, n = 58 (771k) 16.2 and 14.0; with twelve rows a
// thread, which spill twice as much, 15 to 16.3 and 15.8 to 18.0, and 19.9 and
// 23.5 at n = 60 (853k).
constexpr int SNT = SOLVE_THREADS;
constexpr int SNW = SNT / 32;
constexpr int HB = 2;                  // halo records a thread reads at once
constexpr int WAIT_LIMIT = 1 << 21;    // polls of one exchange by a thread (about a second)

__device__ __forceinline__ uint4 ld_record(const uint4 *p) {
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}
__device__ __forceinline__ void st_record(uint4 *p, unsigned a, unsigned b, unsigned c, unsigned e) {
    const unsigned long long lo = (unsigned long long)a | (unsigned long long)b << 32,
                             hi = (unsigned long long)c | (unsigned long long)e << 32;
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}

// Waits until the record at q carries number e; false when `left`, the polls
// that the thread's waits of this exchange may still miss, runs out.
__device__ __forceinline__ bool wait_record(const uint4 *q, unsigned e, uint4 &v, int &left) {
    while (true) {
        v = ld_record(q);
        if (v.w == e) return true;
        if (--left <= 0) return false;
    }
}

// K sums over the block's first NW warps, the same in every thread: shuffles,
// then the warps' sums in order (NW a multiple of four: vector reads, as 16
// warps reading 48 values one by one took longer than the shuffles).  `stop`
// is or-ed over the block on the way.
template <int NW, int K, typename V> __device__ __forceinline__ bool solve_sum(V (&v)[K], V (*sh)[SNW], bool stop) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < NW) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; ++k) sh[k][warp] = v[k];
    }
    const bool any = __syncthreads_or(stop);
    typedef typename Vec4<V>::t V4;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        V t = V(0);
#pragma unroll
        for (int w = 0; w < NW / 4; ++w) {
            const V4 a = ((const V4 *)sh[k])[w];
            t += (a.x + a.y) + (a.z + a.w);
        }
        v[k] = t;
    }
    return any;
}

template <int RPT, bool REG> __global__ void __launch_bounds__(SNT, 1) k_cg_solve(FemDev d) {
    extern __shared__ __align__(16) double s_x[];  // x of the own rows and the halo; in the inner steps u, in FP32
    float *s_u = (float *)s_x;
    float *s_inv = (float *)(s_x + d.rp + d.hmax);  // coarse inverse, a row of P per listed part
    __shared__ __align__(32) float sh_in[2][SNW], sh_out[3][SNW];
    __shared__ float s_rc[SOLVE_PARTS], s_ec[SOLVE_PARTS];  // coarse residual; coarse correction of the listed parts
    __shared__ __align__(32) double sh_d[1][SNW], sh_e[1][SNW];
    const int part = blockIdx.x, P = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const CgState &st = *d.st;
    if (st.outer_done) return;  // the load's verdict, the same in every block
    const int r0 = d.part_row[part], nr = d.part_row[part + 1] - r0;
    const int h0 = d.halo_ptr[part], nh = d.halo_ptr[part + 1] - h0;
    const double bb = st.bb;
    double hh = st.rr_hi, scale = st.scale;
    long long iter = 0;
    int outer = 0;
    bool bad = false, done = false, stalled = false;

    float r[RPT], u[RPT], w[RPT], s[RPT], p[RPT], xc[RPT], z[RPT];
    double x[RPT], rho[RPT];
    int width[RPT], base[RPT];
    int out0[RPT], out1[RPT];  // the row's destinations: halo list entries dst[out0 .. out1)
    constexpr int W = SOLVE_REG_W;
    float av[REG ? RPT * W : 1];
    unsigned ac[REG ? RPT * W / 2 : 1];
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
        const int l = j * SNT + tid, slice = part * (d.rp / 32) + j * SNW + warp;
        const bool on = l < nr;
        base[j] = d.ps_ptr[slice] + lane;
        width[j] = d.ps_w[slice];
        x[j] = 0.0;
        rho[j] = on ? d.b[d.row_old[r0 + l]] : 0.0;
        z[j] = on ? d.pz[r0 + l] : 0.f;
        out0[j] = on ? d.dst_ptr[r0 + l] : 0;
        out1[j] = on ? d.dst_ptr[r0 + l + 1] : 0;
        if constexpr (REG) {
#pragma unroll
            for (int k = 0; k < W; k += 2) {
                const int a = base[j] + 32 * k;
                const unsigned c0 = k < width[j] ? d.pe_col[a] : l, c1 = k + 1 < width[j] ? d.pe_col[a + 32] : l;
                ac[j * (W / 2) + k / 2] = c0 | c1 << 16;
                av[j * W + k] = k < width[j] ? d.pe_val[a] : 0.f;
                av[j * W + k + 1] = k + 1 < width[j] ? d.pe_val[a + 32] : 0.f;
            }
        }
    }
    // the parts whose coarse correction the block needs: its own first, then its halo's
    const int a0 = d.near_ptr[part], na = d.near_ptr[part + 1] - a0;
    for (int i = tid; i < na * P; i += SNT) s_inv[i] = d.coarse_inv[(int64_t)d.near_part[a0 + i / P] * P + i % P];
    const int hid = SNT - 1 - tid;  // first halo entry of the thread
    uint4 *const rec0 = d.rec[0] + h0, *const rec1 = d.rec[1] + h0;  // the block's own lists
    uint4 *const in0 = d.psum[0] + part * P, *const in1 = d.psum[1] + part * P;
    uint4 *const to0 = d.psum[0] + (tid < P ? tid : part) * P + part;  // this block's place in part tid's list
    uint4 *const to1 = d.psum[1] + (tid < P ? tid : part) * P + part;
    unsigned e = 1;  // number of the current exchange
    while (!done && outer < FEM_MAX_OUTER) {
        // inner start: r = D^-1/2 rho / scale, everything else zero
        const double inv = 1.0 / scale;
        float inv_gamma = 0.f, inv_alpha = 0.f, gamma0 = 0.f;  // of the step before; of the first
        float rc = 0.f, sc = 0.f;                              // thread t: part t's coarse residual and S p
        uint4 *rec = e & 1 ? d.rec[1] : d.rec[0];
        float first[1] = {0.f};
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const int l = j * SNT + tid;
            r[j] = l < nr ? (float)(rho[j] * inv * d.pisd[r0 + l]) : 0.f;
            u[j] = w[j] = s[j] = p[j] = xc[j] = 0.f;
            first[0] += z[j] * r[j];
            for (int o = out0[j]; o < out1[j]; ++o) st_record(rec + d.dst[o], __float_as_uint(r[j]), 0u, 0u, e);
        }
        solve_sum<SNW>(first, sh_out, false);
        if (tid < P) st_record(e & 1 ? to1 : to0, 0u, 0u, __float_as_uint(first[0]), e);
        for (int mode = 0;; mode = min(mode + 1, 2), ++e) {
            const uint4 *mine = e & 1 ? rec1 : rec0;
            // the blocks' sums, then the first halo records (from the last thread
            // on, so that the warps without a sum to wait for take them first);
            // threads without a record of their own poll nothing
            uint4 sums, v[HB];
            bool lost = false;
            int left = WAIT_LIMIT;
            if (tid < P) lost = !wait_record((e & 1 ? in1 : in0) + tid, e, sums, left);
#pragma unroll
            for (int i = 0; i < HB; ++i)
                if (i * SNT + hid < nh) lost = !wait_record(mine + i * SNT + hid, e, v[i], left) || lost;
            float sum[2] = {0.f, 0.f}, wc = 0.f;
            if (tid < P) {
                sum[0] = __uint_as_float(sums.x);
                sum[1] = __uint_as_float(sums.y);
                wc = __uint_as_float(sums.z);
            }
            if (solve_sum<SOLVE_PARTS / 32>(sum, sh_in, lost)) {
                stalled = true;
                break;
            }
            float alpha = 0.f, beta = 0.f;
            if (mode > 0) {
                const float gm = sum[0], dl = sum[1];
                beta = gm * inv_gamma;  // zero in the first step
                alpha = __fdividef(gm, dl - beta * gm * inv_alpha);
                if (mode == 1) gamma0 = gm;
                // a residual that reached the stopping test (exactly zero included,
                // where the coefficients are 0/0) ends the inner iteration
                const bool conv = mode == 1 ? gm == 0.f : gm <= d.inner2 * gamma0;
                const bool nan = !isfinite(gm) || (!conv && !(isfinite(alpha) && isfinite(beta)));
                bad = bad || nan;
                if (nan || conv || iter >= d.max_iter) break;  // the same decision in every block
                ++iter;
                inv_gamma = __fdividef(1.f, gm);
                inv_alpha = __fdividef(1.f, alpha);
                sc = wc + beta * sc;
                rc -= alpha * sc;
            } else {
                rc = wc;
            }
            if (tid < P) s_rc[tid] = rc;
#pragma unroll
            for (int j = 0; j < RPT; ++j) {
                s[j] = w[j] + beta * s[j];
                p[j] = u[j] + beta * p[j];
                xc[j] += alpha * p[j];
                r[j] -= alpha * s[j];
            }
            __syncthreads();
            for (int a = warp; a < na; a += SNW) {
                float t = 0.f;
                for (int k = lane; k < P; k += 32) t += s_inv[a * P + k] * s_rc[k];
                t = warp_sum(t);
                if (lane == 0) s_ec[a] = t;
            }
            __syncthreads();
            // u = r + z e(part) of the own rows and, from r_k, w_k and s_{k-1}, of the halo
#pragma unroll
            for (int j = 0; j < RPT; ++j) {
                u[j] = r[j] + z[j] * s_ec[0];
                s_u[j * SNT + tid] = u[j];
            }
#pragma unroll
            for (int i = 0; i < HB; ++i) {
                const int h = i * SNT + hid;
                if (h < nh)
                    s_u[d.rp + h] = __uint_as_float(v[i].x) -
                                    alpha * (__uint_as_float(v[i].y) + beta * __uint_as_float(v[i].z)) +
                                    d.halo_z[h0 + h] * s_ec[d.halo_near[h0 + h]];
            }
            for (int h = HB * SNT + hid; h < nh; h += SNT) {
                uint4 vh;
                lost = !wait_record(mine + h, e, vh, left) || lost;
                s_u[d.rp + h] = __uint_as_float(vh.x) -
                                alpha * (__uint_as_float(vh.y) + beta * __uint_as_float(vh.z)) +
                                d.halo_z[h0 + h] * s_ec[d.halo_near[h0 + h]];
            }
            __syncthreads();
            rec = e & 1 ? d.rec[0] : d.rec[1];  // of exchange e + 1
            float out[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < RPT; ++j) {
                float t = u[j];
                if constexpr (REG) {
#pragma unroll
                    for (int k = 0; k < W; k += 2)
                        if (k < width[j]) {
                            const unsigned c = ac[j * (W / 2) + k / 2];
                            t += av[j * W + k] * s_u[c & 0xffffu];
                            t += av[j * W + k + 1] * s_u[c >> 16];
                        }
                } else {
#pragma unroll 8
                    for (int k = 0; k < width[j]; ++k)
                        t += __ldg(d.pe_val + base[j] + 32 * k) * s_u[__ldg(d.pe_col + base[j] + 32 * k)];
                }
                w[j] = t;
                for (int o = out0[j]; o < out1[j]; ++o)
                    st_record(rec + d.dst[o], __float_as_uint(r[j]), __float_as_uint(t), __float_as_uint(s[j]), e + 1);
                out[0] += r[j] * u[j];
                out[1] += t * u[j];
                out[2] += z[j] * t;
            }
            if (solve_sum<SNW>(out, sh_out, lost)) {
                stalled = true;
                break;
            }
            if (tid < P)
                st_record(e & 1 ? to0 : to1, __float_as_uint(out[0]), __float_as_uint(out[1]),
                          __float_as_uint(out[2]), e + 1);
        }
        if (stalled) break;
        // correction and FP64 residual (exchange e + 1 carries x)
        ++e;
        rec = e & 1 ? d.rec[1] : d.rec[0];
        __syncthreads();  // the last step's reads of u
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            if (j * SNT + tid < nr) x[j] += scale * d.pisd[r0 + j * SNT + tid] * (double)xc[j];
            s_x[j * SNT + tid] = x[j];
            const unsigned long long b = __double_as_longlong(x[j]);
            for (int o = out0[j]; o < out1[j]; ++o) st_record(rec + d.dst[o], (unsigned)b, (unsigned)(b >> 32), 0u, e);
        }
        bool lost = false;
        int left = WAIT_LIMIT;
        for (int h = tid; h < nh; h += SNT) {
            uint4 vh;
            lost = !wait_record((e & 1 ? rec1 : rec0) + h, e, vh, left) || lost;
            s_x[d.rp + h] = __longlong_as_double((long long)((unsigned long long)vh.x | (unsigned long long)vh.y << 32));
        }
        __syncthreads();
        double sq[1] = {0.0};
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const int l = j * SNT + tid;
            double t = 0.0;
            if (l < nr) {
                double sx = d.pdiag[r0 + l] * x[j];
#pragma unroll 4
                for (int k = 0; k < width[j]; ++k) sx += __ldg(d.pe_val64 + base[j] + 32 * k) * s_x[__ldg(d.pe_col + base[j] + 32 * k)];
                t = d.b[d.row_old[r0 + l]] - sx;
            }
            rho[j] = t;
            sq[0] += t * t;
        }
        if (solve_sum<SNW>(sq, sh_d, lost)) {
            stalled = true;
            break;
        }
        if (tid < P) {
            const unsigned long long b = __double_as_longlong(sq[0]);
            st_record(e & 1 ? to1 : to0, (unsigned)b, (unsigned)(b >> 32), 0u, e);
        }
        double tot[1] = {0.0};
        lost = false;
        if (tid < P) {
            uint4 vt;
            lost = !wait_record((e & 1 ? in1 : in0) + tid, e, vt, left);
            tot[0] = __longlong_as_double((long long)((unsigned long long)vt.x | (unsigned long long)vt.y << 32));
        }
        if (solve_sum<SNW>(tot, sh_e, lost)) {
            stalled = true;
            break;
        }
        ++e;
        ++outer;
        hh = tot[0];
        scale = sqrt(hh / (double)d.nf);
        if (!(scale > 0.0)) scale = 1.0;
        bad = bad || !isfinite(hh);
        done = bad || hh <= d.tol2 * bb || iter >= d.max_iter;
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
        const int l = j * SNT + tid;
        if (l < nr) d.x[d.row_old[r0 + l]] = x[j];
    }
    if (tid == 0 && (part == 0 || stalled)) {
        CgState &o = *d.st;
        if (stalled) o.stalled = 1;
        if (part == 0) {
            o.rr_hi = hh;
            o.iter = iter;
            o.outer = outer;
            o.bad = bad;
            o.outer_done = done;
        }
    }
}

// g_j = (mean of the nodal m over the triangle) . n_j + phi_1(opposite node) / h_j
// (dphi_1/dn = -phi_1(o)/h_j: the other three nodes are boundary nodes, phi_1 = 0)
template <typename T>
__global__ void __launch_bounds__(NT) k_fem_charges(FemDev d, const T *__restrict__ m, T *__restrict__ g) {
    const int64_t j = (int64_t)blockIdx.x * NT + threadIdx.x;
    if (j >= d.nfaces) return;
    const int4 f = d.face[j];
    const double4 n = d.face_n[j];
    double mx = 0.0, my = 0.0, mz = 0.0;
    const int v[3] = {f.x, f.y, f.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        mx += (double)m[3 * (int64_t)v[k]];
        my += (double)m[3 * (int64_t)v[k] + 1];
        mz += (double)m[3 * (int64_t)v[k] + 2];
    }
    double val = (mx * n.x + my * n.y + mz * n.z) / 3.0;
    if (f.w >= 0) val += d.x[f.w] * n.w;
    g[j] = (T)val;
}

template <typename T>
__global__ void __launch_bounds__(NT) k_fem_combine(FemDev d, const T *__restrict__ phi2_b,
                                                    const T *__restrict__ phi2_f, T *__restrict__ phi,
                                                    T *__restrict__ phi1) {
    const int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x;
    if (i >= d.nnodes) return;
    const int s = d.slot[i];
    double a = 0.0, b;
    if (s >= 0) {
        a = d.x[s];
        b = (double)phi2_f[s];
    } else {
        b = (double)phi2_b[-1 - s];
    }
    phi[i] = (T)(a + b);
    if (phi1) phi1[i] = (T)a;
}

unsigned blocks_of(int64_t n) { return (unsigned)((n + NT - 1) / NT); }

// blocks of the row-group kernels and of the element-wise kernels (at most nblk_max)
unsigned row_blocks(const FemDev &d) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((d.nf + ROWS - 1) / ROWS, d.nblk_max));
}
unsigned elem_blocks(const FemDev &d) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((d.nf + NT - 1) / NT, d.nblk_max));
}

}  // namespace

cudaError_t launch_fem_load(const FemDev &d, int prec, const void *m, cudaStream_t s) {
    if (prec == 64)
        k_fem_load<double><<<row_blocks(d), NT, 0, s>>>(d, (const double *)m);
    else
        k_fem_load<float><<<row_blocks(d), NT, 0, s>>>(d, (const float *)m);
    if (d.parts == 0) k_cg_scale<<<elem_blocks(d), NT, 0, s>>>(d);
    return cudaGetLastError();
}

namespace {
typedef void (*SolveKernel)(FemDev);
SolveKernel solve_kernel(const FemDev &d) {
    if (d.solve_reg) return d.rpt == 1 ? k_cg_solve<1, true> : k_cg_solve<2, true>;
    switch (d.rpt) {
        case 1: return k_cg_solve<1, false>;
        case 2: return k_cg_solve<2, false>;
        case 4: return k_cg_solve<4, false>;
        case 8: return k_cg_solve<8, false>;
        default: return k_cg_solve<10, false>;
    }
}
}  // namespace

size_t solve_smem(const FemDev &d) {
    return sizeof(double) * (size_t)(d.rp + d.hmax) + sizeof(float) * (size_t)d.near_max * d.parts;
}

cudaError_t solve_blocks(const FemDev &d, int *blocks) {
    int dev = 0, sms = 0, coop = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    // the limit belongs to the kernel, which every potential of the process that
    // runs it shares: always the same one, whatever this potential needs
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)solve_kernel(d), cudaFuncAttributeMaxDynamicSharedMemorySize, SOLVE_SMEM);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, solve_kernel(d), SNT, solve_smem(d));
    *blocks = coop ? sms * per : 0;
    return e;
}

cudaError_t launch_cg_solve(const FemDev &d, cudaStream_t s) {
    FemDev arg = d;
    void *args[] = {&arg};
    return cudaLaunchCooperativeKernel((const void *)solve_kernel(d), dim3(d.parts), dim3(SNT), args, solve_smem(d), s);
}

cudaError_t launch_cg_iteration(const FemDev &d, int parity, cudaStream_t s) {
    return launch_k(k_cg_step, dim3(elem_blocks(d)), NT, 0, s, d, parity);
}

cudaError_t launch_fem_correct(const FemDev &d, cudaStream_t s) {
    k_fem_correct<<<elem_blocks(d), NT, 0, s>>>(d);
    k_fem_residual<<<elem_blocks(d), NT, 0, s>>>(d);
    k_cg_scale<<<elem_blocks(d), NT, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_fem_loop(FemLoop which, const FemDev &d, cudaGraphConditionalHandle h, int bound, cudaStream_t s) {
    switch (which) {
        case LOOP_OUTER_START: k_loop_outer_start<<<1, 1, 0, s>>>(d, h); break;
        case LOOP_OUTER_NEXT: k_loop_outer_next<<<1, 1, 0, s>>>(d, h, bound); break;
        case LOOP_INNER_START: k_loop_inner_start<<<1, 1, 0, s>>>(d, h); break;
        case LOOP_INNER_NEXT: k_loop_inner_next<<<1, 1, 0, s>>>(d, h, bound); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_fem_charges(const FemDev &d, int prec, const void *m, void *g, cudaStream_t s) {
    if (d.nfaces == 0) return cudaSuccess;
    if (prec == 64)
        k_fem_charges<double><<<blocks_of(d.nfaces), NT, 0, s>>>(d, (const double *)m, (double *)g);
    else
        k_fem_charges<float><<<blocks_of(d.nfaces), NT, 0, s>>>(d, (const float *)m, (float *)g);
    return cudaGetLastError();
}

cudaError_t launch_fem_combine(const FemDev &d, int prec, const void *phi2_b, const void *phi2_f, void *phi,
                               void *phi1, cudaStream_t s) {
    if (d.nnodes == 0) return cudaSuccess;
    if (prec == 64)
        k_fem_combine<double><<<blocks_of(d.nnodes), NT, 0, s>>>(d, (const double *)phi2_b, (const double *)phi2_f,
                                                                 (double *)phi, (double *)phi1);
    else
        k_fem_combine<float><<<blocks_of(d.nnodes), NT, 0, s>>>(d, (const float *)phi2_b, (const float *)phi2_f,
                                                                (float *)phi, (float *)phi1);
    return cudaGetLastError();
}

}  // namespace slp
