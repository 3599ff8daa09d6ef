// Near-field correction (paper Sec. 3.4, Eq. (nfcorr)):
//
//   phi_i += sum_{k : |x_i - y_k| < eps} qk (N - N_s)(x_i - y_k),
//
// where N_s is the smooth kernel the far path actually applies:
//   RADIAL:    (N - N_s)(r) = erfc(r / (s sqrt 2)) / (4 pi r)  (r < eps);
//   SEPARABLE: (N - N_s)(d) = 1/(4 pi |d|) - A prod_q f_q(d_q / L_q), every pair;
//   EXPSUM:    (N - N_s)(r) = (1/r - sum_k w_k exp(-g_k r^2)) / (4 pi)  (r < eps,
//              the exponential sum of Sec. 3.3).
//
// One warp per work item: lanes t and t + 16 own target tbegin + t; the warp
// walks the item's source ranges 32 sources at a time, staging them in shared
// memory and broadcasting each to the lanes of one half, the halves taking
// sources in turn.  Pair distances are formed from the
// integer cell difference plus the fractional offsets, so they keep full
// precision however far the mesh sits from the origin.
//
// RADIAL plans (every FP32 plan and most FP64 ones) run k_near_radial32 and
// k_near_radial64, which write the kernel as
//   erfc(a r) / r = 1 / r - a E(a^2 r^2),  E(x) = erf(sqrt x) / sqrt x,
// E being smooth on [0, (a eps)^2]: one polynomial in r^2 in FP32, a table of
// short ones in FP64.  The general kernel k_near takes the other modes, and
// RADIAL plans whose a eps lies outside the fits' range.
#include <algorithm>
#include <climits>

#include "dev_common.cuh"

namespace slp {

constexpr int NEAR_WARPS = 8;

template <typename T> __device__ __forceinline__ T near_erfc(T x);
template <> __device__ __forceinline__ float near_erfc<float>(float x) { return erfcf(x); }
template <> __device__ __forceinline__ double near_erfc<double>(double x) { return erfc(x); }
__device__ __forceinline__ float near_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double near_rsqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float near_cospi(float x) { return cospif(x); }
__device__ __forceinline__ double near_cospi(double x) { return cospi(x); }
__device__ __forceinline__ float near_exp(float x) { return expf(x); }
__device__ __forceinline__ double near_exp(double x) { return exp(x); }

// sum_k w_k exp(-g_k r2) of the exp-sum kernel
template <typename T> __device__ __forceinline__ T expsum_value(const T *__restrict__ w, const T *__restrict__ g, int n, T r2) {
    T s = T(0);
    for (int k = 0; k < n; ++k) s += w[k] * near_exp(-g[k] * r2);
    return s;
}

// f(t) = h[0] + 2 sum_{l>=1} h[l] cos(2 pi l t), by Clenshaw's recurrence in x = cos(2 pi t).
template <typename T> __device__ __forceinline__ T sep_factor(const T *__restrict__ h, int nh, T t) {
    const T x = near_cospi(T(2) * t);
    T b1 = T(0), b2 = T(0);
    for (int l = nh - 1; l >= 1; --l) {
        const T b0 = T(2) * h[l] + T(2) * x * b1 - b2;
        b2 = b1;
        b1 = b0;
    }
    // sum_{l>=1} c_l T_l(x) = x b1 - b2 with c_l = 2 h[l]; plus c_0 = h[0]
    return h[0] + x * b1 - b2;
}

template <typename T, int MODE>
__global__ void __launch_bounds__(NEAR_WARPS * 32) k_near(DevPlan p) {
    pdl_wait();
    pdl_trigger();
    typedef typename VecT<T>::T4 T4;
    __shared__ T4 sg[NEAR_WARPS][32];
    __shared__ T sq[NEAR_WARPS][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.x * NEAR_WARPS + warp;
    if (item >= p.n_near) return;
    const NearItem it = p.near_items[item];
    const int half = lane / NEAR_TARGETS, tl = lane % NEAR_TARGETS;
    const bool active = tl < it.tcount;
    int ctx = 0, cty = 0, ctz = 0;
    T ftx = T(0), fty = T(0), ftz = T(0);
    if (active) {
        const T4 g = ((const T4 *)p.tgt_grid)[it.tbegin + tl];
        unpack_cell(packed_cell(g.w), ctx, cty, ctz);
        ftx = g.x;
        fty = g.y;
        ftz = g.z;
    }
    const T hx = (T)p.h[0], hy = (T)p.h[1], hz = (T)p.h[2];
    const T eps2 = (T)p.eps2;
    const T a = (T)p.inv_s_sqrt2;
    const T iLx = T(1) / T(p.L[0]), iLy = T(1) / T(p.L[1]), iLz = T(1) / T(p.L[2]);  // exact: powers of two
    const T4 *src = (const T4 *)p.src_grid;
    const T *qb = (const T *)p.qbuf;
    T acc = T(0);
    for (int r = it.rbegin; r < it.rend; ++r) {
        const int2 rg = p.near_ranges[r];
        for (int s0 = rg.x; s0 < rg.y; s0 += 32) {
            const int s = s0 + lane;
            if (s < rg.y) {
                sg[warp][lane] = src[s];
                sq[warp][lane] = qb[s];
            }
            __syncwarp();
            const int cnt = min(32, rg.y - s0);
            for (int j = half; j < cnt; j += 2) {
                const T4 g = sg[warp][j];
                int csx, csy, csz;
                unpack_cell(packed_cell(g.w), csx, csy, csz);
                const T dx = (T(ctx - csx) + (ftx - g.x)) * hx;
                const T dy = (T(cty - csy) + (fty - g.y)) * hy;
                const T dz = (T(ctz - csz) + (ftz - g.z)) * hz;
                const T r2 = dx * dx + dy * dy + dz * dz;
                if (MODE == 1) {
                    if (r2 < eps2) {
                        const T ri = near_rsqrt(r2);
                        acc += sq[warp][j] * near_erfc<T>(r2 * ri * a) * ri;
                    }
                } else if (MODE == 3) {
                    if (r2 < eps2)
                        acc += sq[warp][j] *
                               (near_rsqrt(r2) - expsum_value((const T *)p.es_w, (const T *)p.es_g, p.es_n, r2));
                } else {
                    const T ri = near_rsqrt(r2);
                    const T ux = (T(ctx - csx) + (ftx - g.x)) * iLx;
                    const T uy = (T(cty - csy) + (fty - g.y)) * iLy;
                    const T uz = (T(ctz - csz) + (ftz - g.z)) * iLz;
                    const T kn = sep_factor((const T *)p.sep_h[0], p.sep_nh[0], ux) *
                                 sep_factor((const T *)p.sep_h[1], p.sep_nh[1], uy) *
                                 sep_factor((const T *)p.sep_h[2], p.sep_nh[2], uz);
                    acc += sq[warp][j] * (ri - T(p.sep_A) * kn);
                }
            }
            __syncwarp();
        }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, NEAR_TARGETS);
    if (lane < it.tcount) {
        const T v = acc * T(0.079577471545947667884);  // 1 / (4 pi)
        if (p.deterministic)
            ((T *)p.phi_near)[(int64_t)item * 32 + lane] = v;
        else
            atomicAdd((T *)p.phi_part + it.tbegin + lane, v);
    }
}

// ---------------------------------------------------------------- RADIAL, fitted kernels
// What bounds both: arithmetic (sources and targets are read once per item
// and stay in L1/L2).  Both walk the sources of an item 32 at a time, one per
// lane, and first drop those farther than eps from the box around the warp's
// targets (the work list culls whole 2x2x2-cell bins only), so the inner loop
// runs over the kept ones, packed by ballot.  Positions are relative to the
// cell of the warp's first target: integer part and fraction separately in
// FP32, whose differences are exact; their sum in FP64.

// Keep this lane's source?  Distance from the targets' box, in cells of x, in
// FP32 with a margin far above its rounding.
__device__ __forceinline__ bool in_reach(const float (&lo)[3], const float (&hi)[3], float x, float y, float z,
                                         float ry, float rz, float reach2) {
    const float dx = fmaxf(0.f, fmaxf(lo[0] - x, x - hi[0]));
    const float dy = fmaxf(0.f, fmaxf(lo[1] - y, y - hi[1])) * ry;
    const float dz = fmaxf(0.f, fmaxf(lo[2] - z, z - hi[2])) * rz;
    return dx * dx + dy * dy + dz * dz <= reach2;
}
__device__ __forceinline__ void warp_box(float v, float &lo, float &hi) {
    lo = hi = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// FP32: a lane takes two sources per step in paired operations.  Per pair: 9 subtractions
// (integer and fractional parts), 5 operations for r^2, one reciprocal square
// root, the degree-14 polynomial of a E (15 multiply-adds, its argument's map
// included), 2 for the sum: 32 lane operations where erfcf, the integer
// conversions and the cell arithmetic per pair took about 180.  Level-5 sphere
// at 128^3 (118M lane pairs after the cull, 73M inside eps): 670 -> 164 us.
__global__ void __launch_bounds__(NEAR_WARPS * 32) k_near_radial32(DevPlan p) {
    __shared__ __align__(16) float2 st[NEAR_WARPS][16][10];  // per source pair: -H xyz, -f xyz, charge (80-byte
                                                             // rows: stores 2-way instead of 8-way on the banks)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.x * NEAR_WARPS + warp;
    pdl_wait();
    pdl_trigger();
    if (item >= p.n_near) return;
    const NearItem it = p.near_items[item];
    const int half = lane / NEAR_TARGETS;
    const float4 tg = ((const float4 *)p.tgt_grid)[it.tbegin + min(lane % NEAR_TARGETS, it.tcount - 1)];
    int cx, cy, cz;
    unpack_cell(packed_cell(tg.w), cx, cy, cz);
    const int c0x = __shfl_sync(0xffffffffu, cx, 0), c0y = __shfl_sync(0xffffffffu, cy, 0),
              c0z = __shfl_sync(0xffffffffu, cz, 0);
    const float Hx = (float)(cx - c0x), Hy = (float)(cy - c0y), Hz = (float)(cz - c0z);
    float lo[3], hi[3];
    warp_box(Hx + tg.x, lo[0], hi[0]);
    warp_box(Hy + tg.y, lo[1], hi[1]);
    warp_box(Hz + tg.z, lo[2], hi[2]);
    // lengths in cells of x
    const float ry = p.near_ryf, rz = p.near_rzf, eps2 = p.near_e2f, reach2 = eps2 * 1.001f;
    const float2 k1 = make_float2(p.near_k1f, p.near_k1f), m1 = make_float2(-1.f, -1.f);
    const float2 ry2 = make_float2(ry, ry), rz2 = make_float2(rz, rz);
    const float2 Hx2 = make_float2(Hx, Hx), Hy2 = make_float2(Hy, Hy), Hz2 = make_float2(Hz, Hz);
    const float2 fx2 = make_float2(tg.x, tg.x), fy2 = make_float2(tg.y, tg.y), fz2 = make_float2(tg.z, tg.z);
    float2 c[NEAR_DEG32 + 1];  // coefficients of -a E
#pragma unroll
    for (int k = 0; k <= NEAR_DEG32; ++k) c[k] = make_float2(p.near_c32[k], p.near_c32[k]);
    const float4 *src = (const float4 *)p.src_grid;
    const float *qb = (const float *)p.qbuf;
    float2 acc = make_float2(0.f, 0.f);
    for (int r = it.rbegin; r < it.rend; ++r) {
        const int2 rg = p.near_ranges[r];
        for (int s0 = rg.x; s0 < rg.y; s0 += 32) {
            const int s = min(s0 + lane, rg.y - 1);
            const float4 g = src[s];
            const float q = qb[s];
            int sx, sy, sz;
            unpack_cell(packed_cell(g.w), sx, sy, sz);
            const float Sx = (float)(sx - c0x), Sy = (float)(sy - c0y), Sz = (float)(sz - c0z);
            const bool keep = s0 + lane < rg.y && in_reach(lo, hi, Sx + g.x, Sy + g.y, Sz + g.z, ry, rz, reach2);
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            if (kept == 0) continue;
            const int cnt = __popc(kept);
            const int at = __popc(kept & ((1u << lane) - 1u));
            // a multiple of four: up to three lanes add their source once more, without charge
            const int npad = -cnt & 3;
            if (keep || lane < npad) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (e == 0 ? !keep : lane >= npad) continue;
                    const int k = e == 0 ? at : cnt + lane;
                    float *d = (float *)st[warp][k >> 1] + (k & 1);
                    d[0] = -Sx;
                    d[2] = -Sy;
                    d[4] = -Sz;
                    d[6] = -g.x;
                    d[8] = -g.y;
                    d[10] = -g.z;
                    d[12] = e == 0 ? q : 0.f;
                }
            }
            __syncwarp();
            for (int j = half; 2 * j < cnt; j += 2) {
                const float4 *v = (const float4 *)st[warp][j];
                const float4 v0 = v[0], v1 = v[1], v2 = v[2];
                const float2 qq = st[warp][j][6];
                float2 dx = __fadd2_rn(__fadd2_rn(Hx2, make_float2(v0.x, v0.y)), __fadd2_rn(fx2, make_float2(v1.z, v1.w)));
                float2 dy = __fadd2_rn(__fadd2_rn(Hy2, make_float2(v0.z, v0.w)), __fadd2_rn(fy2, make_float2(v2.x, v2.y)));
                float2 dz = __fadd2_rn(__fadd2_rn(Hz2, make_float2(v1.x, v1.y)), __fadd2_rn(fz2, make_float2(v2.z, v2.w)));
                dy = __fmul2_rn(dy, ry2);
                dz = __fmul2_rn(dz, rz2);
                const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
                const float2 u = __ffma2_rn(r2, k1, m1);
                float2 e = c[NEAR_DEG32];
#pragma unroll
                for (int k = NEAR_DEG32 - 1; k >= 0; --k) e = __ffma2_rn(e, u, c[k]);
                float2 w = __fadd2_rn(make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y)), e);
                w.x = r2.x < eps2 ? w.x : 0.f;
                w.y = r2.y < eps2 ? w.y : 0.f;
                acc = __ffma2_rn(qq, w, acc);
            }
            __syncwarp();
        }
    }
    float sum = acc.x + acc.y;
    sum += __shfl_xor_sync(0xffffffffu, sum, NEAR_TARGETS);
    if (lane < it.tcount) {
        const float v = sum * p.near_outf;
        if (p.deterministic)
            ((float *)p.phi_near)[(int64_t)item * 32 + lane] = v;
        else
            atomicAdd((float *)p.phi_part + it.tbegin + lane, v);
    }
}

// 1 / sqrt(x) in FP64: the FP32 value and one third-order step of Householder's
// iteration, y (1 + e/2 + 3 e^2 / 8) with e = 1 - x y^2 (e < 2^-21, so the
// remainder is below 2^-63).  The FP32 seed needs x in FP32's range; here x is
// a squared distance in grid cells.
__device__ __forceinline__ double rsqrt_refined(double x) {
    const double y = (double)rsqrt_approx((float)x);
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// -a E(a^2 r^2) from the table [k][ni] at x = r^2 iw, iw intervals per unit of
// r^2; false outside the table (r >= eps).  The interval is read off the low
// word of x - 1/2 + 1.5 2^52.
__device__ __forceinline__ bool table_value(const double *tab, int ni, double iw, double r2, double &e) {
    constexpr double MAGIC = 6755399441055744.0;  // 1.5 2^52
    const double t = fma(r2, iw, -0.5);            // interval i holds [i - 1/2, i + 1/2)
    const double tm = t + MAGIC;
    const int i = __double2loint(tm);
    const double u = t - (tm - MAGIC);
    const bool in = (unsigned)i < (unsigned)ni;
    const double *c = tab + (in ? i : 0);
    e = c[NEAR_DEG64 * ni];
#pragma unroll
    for (int k = NEAR_DEG64 - 1; k >= 0; --k) e = fma(e, u, c[k * ni]);
    return in;
}

// FP64: this GPU's FP64 pipe (2 lanes per SM) bounds it, so everything that is
// not the pair's own arithmetic is kept off it: about 27 FP64 operations per
// pair (3 subtractions, 5 for r^2, 5 for the reciprocal square root, 3 for the
// interval and its local coordinate, 9 of the degree-9 polynomial, 2 for the
// sum) where rsqrt, erfc and the conversions of the cell differences took over
// 100.
// Level-4 sphere at 128^3 (63M pairs listed): 129 -> 3.6 ms, level-3 20.4 ->
// 0.35 ms, both with the work list's full 16-target blocks.
__global__ void __launch_bounds__(NEAR_WARPS * 32) k_near_radial64(DevPlan p) {
    __shared__ __align__(16) double4 st[NEAR_WARPS][32];  // position, charge
    __shared__ double tab[(NEAR_DEG64 + 1) * NEAR_INT64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.x * NEAR_WARPS + warp;
    const int ni = p.near_ni64;
    for (int i = threadIdx.x; i < (NEAR_DEG64 + 1) * ni; i += blockDim.x) tab[i] = p.near_tab64[i];
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    if (item >= p.n_near) return;
    const NearItem it = p.near_items[item];
    const int half = lane / NEAR_TARGETS;
    const double4 tg = ((const double4 *)p.tgt_grid)[it.tbegin + min(lane % NEAR_TARGETS, it.tcount - 1)];
    int cx, cy, cz;
    unpack_cell(packed_cell(tg.w), cx, cy, cz);
    const int c0x = __shfl_sync(0xffffffffu, cx, 0), c0y = __shfl_sync(0xffffffffu, cy, 0),
              c0z = __shfl_sync(0xffffffffu, cz, 0);
    const double tx = (cx - c0x) + tg.x, ty = (cy - c0y) + tg.y, tz = (cz - c0z) + tg.z;
    float lo[3], hi[3];
    warp_box((float)tx, lo[0], hi[0]);
    warp_box((float)ty, lo[1], hi[1]);
    warp_box((float)tz, lo[2], hi[2]);
    const double ry = p.near_ry, rz = p.near_rz, iw = p.near_iw;
    const float reach2 = p.near_e2f * 1.001f, ryf = p.near_ryf, rzf = p.near_rzf;
    const double4 *src = (const double4 *)p.src_grid;
    const double *qb = (const double *)p.qbuf;
    double acc = 0.0;
    for (int r = it.rbegin; r < it.rend; ++r) {
        const int2 rg = p.near_ranges[r];
        for (int s0 = rg.x; s0 < rg.y; s0 += 32) {
            const int s = min(s0 + lane, rg.y - 1);
            const double4 g = src[s];
            const double q = qb[s];
            int sx, sy, sz;
            unpack_cell(packed_cell(g.w), sx, sy, sz);
            const double x = (sx - c0x) + g.x, y = (sy - c0y) + g.y, z = (sz - c0z) + g.z;
            const bool keep = s0 + lane < rg.y && in_reach(lo, hi, (float)x, (float)y, (float)z, ryf, rzf, reach2);
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            if (kept == 0) continue;
            if (keep) st[warp][__popc(kept & ((1u << lane) - 1u))] = make_double4(x, y, z, q);
            __syncwarp();
            const int cnt = __popc(kept);
            for (int j = half; j < cnt; j += 2) {
                const double4 v = st[warp][j];
                const double dx = tx - v.x, dy = (ty - v.y) * ry, dz = (tz - v.z) * rz;
                const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
                double e;
                const bool in = table_value(tab, ni, iw, r2, e);
                const double w = rsqrt_refined(r2) + e;
                acc = fma(in ? v.w : 0.0, w, acc);
            }
            __syncwarp();
        }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, NEAR_TARGETS);
    if (lane < it.tcount) {
        const double v = acc * p.near_out;
        if (p.deterministic)
            ((double *)p.phi_near)[(int64_t)item * 32 + lane] = v;
        else
            atomicAdd((double *)p.phi_part + it.tbegin + lane, v);
    }
}

// Deterministic mode: items of one target block are consecutive; add their
// partials in item order.  blk_items[b] = first item of block b (CSR).
template <typename T>
__global__ void k_near_reduce(DevPlan p, const int *__restrict__ blk_first, int nblk) {
    pdl_wait();
    pdl_trigger();
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= nblk) return;
    const int i0 = blk_first[b], i1 = blk_first[b + 1];
    const NearItem it0 = p.near_items[i0];
    if (lane >= it0.tcount) return;
    T s = T(0);
    for (int i = i0; i < i1; ++i) s += ((const T *)p.phi_near)[(int64_t)i * 32 + lane];
    ((T *)p.phi_part)[it0.tbegin + lane] = s;
}

template <typename T> static cudaError_t near_t(const DevPlan &p, cudaStream_t s) {
    if (p.n_near == 0) return cudaSuccess;
    const int nb = (p.n_near + NEAR_WARPS - 1) / NEAR_WARPS;
    if (p.near_fit)
        { const cudaError_t le = launch_k(sizeof(T) == 4 ? k_near_radial32 : k_near_radial64, nb, NEAR_WARPS * 32, 0, s, p); if (le != cudaSuccess) return le; }
    else if (p.kernel_mode == 2)
        { const cudaError_t le = launch_k(k_near<T, 2>, nb, NEAR_WARPS * 32, 0, s, p); if (le != cudaSuccess) return le; }
    else if (p.kernel_mode == 3)
        { const cudaError_t le = launch_k(k_near<T, 3>, nb, NEAR_WARPS * 32, 0, s, p); if (le != cudaSuccess) return le; }
    else
        { const cudaError_t le = launch_k(k_near<T, 1>, nb, NEAR_WARPS * 32, 0, s, p); if (le != cudaSuccess) return le; }
    return cudaGetLastError();
}

cudaError_t launch_near(const DevPlan &p, cudaStream_t s) {
    return p.prec == 64 ? near_t<double>(p, s) : near_t<float>(p, s);
}

cudaError_t launch_near_reduce(const DevPlan &p, const int *blk_first, int nblk, cudaStream_t s) {
    if (nblk == 0) return cudaSuccess;
    const int nb = (nblk + 7) / 8;
    if (p.prec == 64)
        { const cudaError_t le = launch_k(k_near_reduce<double>, nb, 256, 0, s, p, blk_first, nblk); if (le != cudaSuccess) return le; }
    else
        { const cudaError_t le = launch_k(k_near_reduce<float>, nb, 256, 0, s, p, blk_first, nblk); if (le != cudaSuccess) return le; }
    return cudaGetLastError();
}

}  // namespace slp

// =====================================================================
// Precomputed near-field operator for nodal magnetisation input.
//
// With sigma_k = m(y_k) . n_j and m interpolated linearly from the vertices
// (P1, Sec. 2.1), the near-field correction is linear in the nodal m:
//   phi_i += sum_v W_iv . m_v,
//   W_iv = sum_{k near x_i, v a vertex of tri(k)} w_k (N - N_s)(x_i - y_k) lambda_{s(k), a(v)} n_{j(k)}.
// The paper precomputes the near-field integrals in the set-up phase and
// applies them as a sparse matrix (Sec. 3.4); here W is assembled once per
// plan on the GPU in FP64 (two passes: count, fill) and stored by groups of
// four rows in sorted target order.  Each evaluation is then a sparse product
// streamed from HBM.
namespace slp {

__device__ __forceinline__ double nm_kernel(const NMBuild &b, const double *tab, double dx, double dy, double dz,
                                            double r2) {
    if (b.ni > 0) {
        double e;
        if (!table_value(tab, b.ni, b.iw, r2, e)) return 0.0;
        return fma(rsqrt_refined(r2 * b.iw), b.sqrt_iw, e) * 0.079577471545947667884;  // in range whatever the units
    }
    const double ri = rsqrt(r2);
    if (b.kernel_mode == 2) {
        const double kn = sep_factor(b.sep_h[0], b.sep_nh[0], dx / b.P[0]) *
                          sep_factor(b.sep_h[1], b.sep_nh[1], dy / b.P[1]) *
                          sep_factor(b.sep_h[2], b.sep_nh[2], dz / b.P[2]);
        return (ri - b.sep_A4pi * kn) * 0.079577471545947667884;
    }
    if (b.kernel_mode == 3) return (ri - expsum_value(b.es_w, b.es_g, b.es_n, r2)) * 0.079577471545947667884;
    return erfc(r2 * ri * b.inv_s_sqrt2) * ri * 0.079577471545947667884;
}

// b.parts warps per group of NM_ROWS consecutive sorted targets, which share its
// candidate vertices by consecutive batches of 32 (`batches`), a candidate per
// lane; counts and offsets are per part.  An entry is a vertex with a quadrature point of an adjacent
// triangle within eps of some target of the group; its weights are zero for the
// others.  pass 0: count the part's entries, its (target, vertex) pairs with a
// point inside and the near pairs; pass 1: fill.  The kernel is evaluated in
// FP64, three times per pair (once per vertex of the triangle), so the FP64 pipe
// bounds the fill: the table's 25 operations where erfc and rsqrt took over 100,
// no evaluation in the count, and vertices out of every target's reach passed
// over.  Plan of plate400 (319M pairs) 2.56 -> 0.83 s, of sphere5 at 128^3 (6M)
// 0.23 -> 0.09 s.  With one warp a group the 97 groups of the 8x8 cube are 13
// blocks, each with four rows' series to add up: plans with every pair near,
// FP64, 13.6 -> 2.9 ms (8x8 cube), 14.0 -> 2.7 (level-2 sphere, 7 points), 47.2 ->
// 10.3 (level 3); a radial one of the level-3 sphere 10.7 -> 7.0.
template <typename T4>
__global__ void __launch_bounds__(256) k_nm_build(NMBuild b, int pass, NMCount *__restrict__ counts,
                                                  const int64_t *__restrict__ offset, int *__restrict__ col,
                                                  T4 *__restrict__ val, int64_t stride) {
    constexpr int R = NM_ROWS;
    __shared__ double tab[(NEAR_DEG64 + 1) * NEAR_INT64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (pass == 1) {
        for (int i = threadIdx.x; i < (NEAR_DEG64 + 1) * b.ni; i += blockDim.x) tab[i] = b.tab[i];
        __syncthreads();
    }
    const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp, g = w / b.parts;
    const int part = (int)(w - g * b.parts);
    if (R * g >= b.N) return;
    const int nr = (int)min((int64_t)R, b.N - R * g);
    double4 x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = b.tgt[R * g + min(r, nr - 1)];
    const int blk = b.grp_block[g];
    int64_t out = pass == 1 ? offset[w] : 0;
    int64_t cnt = 0, npairs = 0, nnz = 0;
    int first = 0, last = INT_MAX, batch = 0;  // the part's batches of the group's candidates
    if (b.parts > 1) {
        int all = 0;
        for (int rr = b.blk_r0[blk]; rr < b.blk_r0[blk + 1]; ++rr) all += (b.ranges[rr].y - b.ranges[rr].x + 31) / 32;
        first = (int)((int64_t)all * part / b.parts);
        last = (int)((int64_t)all * (part + 1) / b.parts);
    }
    for (int rr = b.blk_r0[blk]; rr < b.blk_r0[blk + 1] && batch < last; ++rr) {
        const int2 rg = b.ranges[rr];
        for (int u0 = rg.x; u0 < rg.y; u0 += 32, ++batch) {
            if (batch < first || batch >= last) continue;
            const int u = u0 + lane;
            double wx[R], wy[R], wz[R];
#pragma unroll
            for (int r = 0; r < R; ++r) wx[r] = wy[r] = wz[r] = 0.0;
            unsigned reach = 0, hit = 0;  // targets: worth a look; with a point inside
            if (u < rg.y) {
                const double4 xv = b.vpos[u];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const double dx = x[r].x - xv.x, dy = x[r].y - xv.y, dz = x[r].z - xv.z;
                    if (r < nr && dx * dx + dy * dy + dz * dz <= b.reach2) reach |= 1u << r;
                }
            }
            if (reach) {
                const int v = b.tgt_perm[u];
                for (int e = b.vt_ptr[v]; e < b.vt_ptr[v + 1]; ++e) {
                    const int ent = b.vt_ent[e];
                    const int j = ent >> 2, a = ent & 3;
                    const double4 n = b.nrm[j];
                    double acc[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) acc[r] = 0.0;
                    for (int s = 0; s < b.q; ++s) {
                        const double4 y = b.src[(int64_t)j * b.q + s];
                        const double yw = pass == 1 ? y.w * b.lam[3 * s + a] : 0.0;
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const double dx = x[r].x - y.x, dy = x[r].y - y.y, dz = x[r].z - y.z;
                            const double r2 = dx * dx + dy * dy + dz * dz;
                            if ((reach >> r & 1) && r2 < b.eps2 && r2 > 0.0) {
                                hit |= 1u << r;
                                if (pass == 1) acc[r] += yw * nm_kernel(b, tab, dx, dy, dz, r2);
                                if (a == 0) ++npairs;
                            }
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        wx[r] += acc[r] * n.x;
                        wy[r] += acc[r] * n.y;
                        wz[r] += acc[r] * n.z;
                    }
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, hit != 0);
            if (pass == 1 && hit) {
                const int64_t at = out + cnt + __popc(bal & ((1u << lane) - 1u));
                T4 o;
                col[at] = u;  // vertex: sorted target position
                o.x = wx[0], o.y = wx[1], o.z = wx[2], o.w = wx[3];
                val[at] = o;
                o.x = wy[0], o.y = wy[1], o.z = wy[2], o.w = wy[3];
                val[at + stride] = o;
                o.x = wz[0], o.y = wz[1], o.z = wz[2], o.w = wz[3];
                val[at + 2 * stride] = o;
            }
            cnt += __popc(bal);
            nnz += __popc(hit);
        }
    }
    npairs = warp_sum((long long)npairs);
    nnz = warp_sum((long long)nnz);
    if (pass == 0 && lane == 0) counts[w] = {cnt, nnz, npairs};
}

// Warps per group: as many as give each of 152 SMs 16 warps, at most 32 (a
// candidate list is rarely longer than 32 batches where groups are so few).
int nm_build_parts(int64_t N) {
    const int64_t groups = (N + NM_ROWS - 1) / NM_ROWS;
    return (int)std::max<int64_t>(1, std::min<int64_t>(32, (152 * 16 + groups - 1) / groups));
}

cudaError_t launch_nm_build(const NMBuild &b, int pass, int prec, NMCount *counts, const int64_t *offset, int *col,
                            void *val, int64_t stride, cudaStream_t s) {
    const int64_t warps = (b.N + NM_ROWS - 1) / NM_ROWS * b.parts;
    const int wpb = warps >= 152 * 32 ? 8 : 2;  // few warps: small blocks, over all SMs
    const unsigned nb = (unsigned)((warps + wpb - 1) / wpb);
    if (prec == 64)
        k_nm_build<double4><<<nb, 32 * wpb, 0, s>>>(b, pass, counts, offset, col, (double4 *)val, stride);
    else
        k_nm_build<float4><<<nb, 32 * wpb, 0, s>>>(b, pass, counts, offset, col, (float4 *)val, stride);
    return cudaGetLastError();
}

// streaming (evict-first) loads of the operator, read once per evaluation
__device__ __forceinline__ float4 ld_stream(const float4 *p) { return __ldcs(p); }
__device__ __forceinline__ double4 ld_stream(const double4 *p) {
    const double2 a = __ldcs((const double2 *)p), b = __ldcs((const double2 *)p + 1);
    return make_double4(a.x, a.y, b.x, b.y);
}

// The product: one warp per group of four rows.  The rows of neighbouring
// targets have nearly the same columns, so the group keeps their union once: an
// entry is a column and 4 x 3 weights, in three streams of 4-vectors (the x, y
// and z weights of the four rows), and a gathered m serves four rows.  Bounds:
// HBM (52 bytes an entry against four of 16; 83 % of the weights are non-zero
// on the level-5 sphere at 128^3, 93 % on plate400, and 25 to 45 % for probes so
// scattered that neighbours share few vertices, where the product is no slower
// for it: level-6 sphere at 256^3 with 200, 2000 and 8000 probes 137.7, 142.0 and
// 149.5 us an evaluation, 143.7, 145.8 and 151.9 with a warp per row) and, with several states,
// the gathers through L1, which fall to a quarter.  Against one row per warp
// and 16-byte entries of their own: plate400 725 -> 650 us, cube200 371 -> 345,
// cube400 1392 -> 1240; evaluations with it beside the far field: sphere5 52.0
// -> 50.4 us, torus300 98.7 -> 90.4, eight states of torus400 786 -> 678.
//
// One batch: lane l takes entries j + l + 32 u (u < U), their loads issued
// before the gathered m; FULL batches need no predicates, the tail batch reads
// zero weights past the end.  The K sorted magnetisations are m4[k N + column];
// lane l adds its entries in order, and warps that share a group take chunks of
// 128 entries in turn whatever K, so a row's sums do not depend on K.
constexpr int CHUNK = 128;
template <typename T, int K, int U, bool FULL>
__device__ __forceinline__ void near_batch(const int *__restrict__ col, const typename VecT<T>::T4 *__restrict__ val,
                                           int64_t stride, int j, int n, int lane,
                                           const typename VecT<T>::T4 *__restrict__ m4, int64_t N, T (&acc)[K][NM_ROWS]) {
    typedef typename VecT<T>::T4 T4;
    T4 wx[U], wy[U], wz[U];
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (FULL || j + lane + 32 * u < n) {
            c[u] = __ldcs(col + j + 32 * u);
            wx[u] = ld_stream(val + j + 32 * u);
            wy[u] = ld_stream(val + stride + j + 32 * u);
            wz[u] = ld_stream(val + 2 * stride + j + 32 * u);
        } else {
            c[u] = 0;
            wx[u].x = wx[u].y = wx[u].z = wx[u].w = T(0);
            wy[u] = wz[u] = wx[u];
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const T4 m = m4[k * N + c[u]];
            acc[k][0] += wx[u].x * m.x + wy[u].x * m.y + wz[u].x * m.z;
            acc[k][1] += wx[u].y * m.x + wy[u].y * m.y + wz[u].y * m.z;
            acc[k][2] += wx[u].z * m.x + wy[u].z * m.y + wz[u].z * m.z;
            acc[k][3] += wx[u].w * m.x + wy[u].w * m.y + wz[u].w * m.z;
        }
}

// phi_part[k][t] = the rows of a group applied to K states with one pass over
// them.  `split` (1, 2 or 4) warps share a group, taking its chunks in turn,
// so that meshes with few groups fill the GPU; their sums are added in order.
template <typename T, int K> __global__ void __launch_bounds__(128) k_near_matrix(DevPlan p, int split) {
    typedef typename VecT<T>::T4 T4;
    // entries in flight per lane: a chunk in one batch, or for four and eight states
    // (registers) in two, unrolled.  With two a batch and a loop over batches,
    // torus400 with 2 to 8 states 287, 328, 382, 449, 500, 573, 642 us an evaluation;
    // so 260, 296, 365, 403, 472, 500, 570.  FP64, whose pipe the far field beside it
    // needs: two, or one from seven states on (a 10x10 cube with 4, 7 and 8 states
    // 469, 645 and 740 us with two, 486, 628 and 731 with one).
    constexpr int U = K == 1 ? 4 : sizeof(T) == 8 ? (K < 7 ? 2 : 1) : K == 4 || K == 8 ? 2 : 4;
    __shared__ T part[4][K * NM_ROWS];
    pdl_wait();
    pdl_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = warp & (split - 1);
    const int64_t g = (int64_t)blockIdx.x * (4 / split) + warp / split;
    const bool live = NM_ROWS * g < p.N;
    const T4 *m4 = (const T4 *)p.m4;  // sorted nodal m (k_nodal_prep), K copies
    T acc[K][NM_ROWS];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int r = 0; r < NM_ROWS; ++r) acc[k][r] = T(0);
    if (live) {
        const int64_t e0 = p.nm_gptr[g];
        const int n = (int)(p.nm_gptr[g + 1] - e0);  // a group holds < 2^31 entries
        const int *col = p.nm_col + e0 + lane;
        const T4 *val = (const T4 *)p.nm_val + e0 + lane;
        int j = CHUNK * sub;
        for (; j + CHUNK <= n; j += CHUNK * split)
#pragma unroll(sizeof(T) == 8 ? 1 : 2)
            for (int h = 0; h < CHUNK; h += 32 * U)
                near_batch<T, K, U, true>(col, val, p.nm_stride, j + h, n, lane, m4, p.N, acc);
        constexpr int UT = sizeof(T) == 4 && K == 2 ? 2 : U;  // two states, small meshes: 126 us in batches of two, 128 of four
#pragma unroll 1
        for (int h = 0; h < CHUNK && j + h < n; h += 32 * UT)
            near_batch<T, K, UT, false>(col, val, p.nm_stride, j + h, n, lane, m4, p.N, acc);
    }
    // lane r of the group's first warp ends up with row r
    T v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        v[k] = T(0);
#pragma unroll
        for (int r = 0; r < NM_ROWS; ++r) {
            const T a = warp_sum(acc[k][r]);
            if (lane == r) v[k] = a;
        }
    }
    if (split > 1) {
        if (lane < NM_ROWS)
#pragma unroll
            for (int k = 0; k < K; ++k) part[warp][k * NM_ROWS + lane] = v[k];
        __syncthreads();
        if (sub == 0 && lane < NM_ROWS)
#pragma unroll
            for (int k = 0; k < K; ++k)
                for (int w = 1; w < split; ++w) v[k] += part[warp + w][k * NM_ROWS + lane];
    }
    const int64_t t = NM_ROWS * g + lane;
    if (live && sub == 0 && lane < NM_ROWS && t < p.N)
#pragma unroll
        for (int k = 0; k < K; ++k) ((T *)p.phi_part)[k * p.N + t] = v[k];
}

// Warps per group: 48 or more warps for each of 152 SMs where two or four a
// group give them (sphere5 at 128^3, 2561 groups: the evaluation 51.8 us with
// one, 50.4 with two; sphere4 in FP64, 641 groups: the product 90 us with one,
// 49 with four).
static int near_split(const DevPlan &p) {
    const int64_t groups = (p.N + NM_ROWS - 1) / NM_ROWS;
    return groups >= 152 * 48 ? 1 : groups >= 152 * 12 ? 2 : 4;
}

template <typename T> static cudaError_t near_states_t(const DevPlan &p, int K, cudaStream_t s) {
    const int split = near_split(p), rows = NM_ROWS * 4 / split;  // rows of a block
    const unsigned nb = (unsigned)((p.N + rows - 1) / rows);
    switch (K) {
        case 1: return launch_k(k_near_matrix<T, 1>, nb, 128, 0, s, p, split);
        case 2: return launch_k(k_near_matrix<T, 2>, nb, 128, 0, s, p, split);
        case 3: return launch_k(k_near_matrix<T, 3>, nb, 128, 0, s, p, split);
        case 4: return launch_k(k_near_matrix<T, 4>, nb, 128, 0, s, p, split);
        case 5: return launch_k(k_near_matrix<T, 5>, nb, 128, 0, s, p, split);
        case 6: return launch_k(k_near_matrix<T, 6>, nb, 128, 0, s, p, split);
        case 7: return launch_k(k_near_matrix<T, 7>, nb, 128, 0, s, p, split);
        case 8: return launch_k(k_near_matrix<T, 8>, nb, 128, 0, s, p, split);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_near_matrix_states(const DevPlan &p, int K, cudaStream_t s) {
    if (p.N == 0 || K <= 0) return cudaSuccess;
    return p.prec == 64 ? near_states_t<double>(p, K, s) : near_states_t<float>(p, K, s);
}

cudaError_t launch_near_matrix(const DevPlan &p, const void *, cudaStream_t s) {
    return launch_near_matrix_states(p, 1, s);
}

}  // namespace slp
