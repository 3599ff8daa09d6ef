// Device data and launchers of the scalar potential phi = phi_1 + phi_2 on a
// tetrahedral mesh (Alg. 1, Sec. 2.1): the P1 load operator, the conjugate
// gradients for the Dirichlet problem of phi_1 (FP32 iterations refined by
// FP64 residuals), the boundary charges g = m.n - dphi_1/dn and the final sum.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace slp {

// Scalars an inner step carries to the next one.  A step of parity q reads
// record q and block 0 writes record q ^ 1, so no block reads what another
// block of the same launch writes.
struct CgInner {
    float gamma;     // gamma_k = r_k . D^-1 r_k of the step that wrote the record
    float alpha;     // alpha_k of that step
    float rr0;       // r . r at the start of the inner iteration
    int mode;        // 0: set-up launch (alpha = beta = 0), 1: first step, 2: later steps
    long long iter;  // inner steps so far, all corrections together
};

// Scalars of the solve.  The FP64 fields are written by the last block of the
// load and residual launches; the inner steps write `in` (above) and, from
// block 0, the fields the host reads (gamma, rr, iter, done, bad); the solve
// graph's loop-control kernels keep the loop counters.
struct CgState {
    CgInner in[2];
    float gamma;        // r . D^-1 r of the inner residual
    float rr;           // r . r of the inner residual at the last stopping test
    double bb;          // b . b
    double rr_hi;       // |b - S x|^2 (FP64 residual) after the last correction
    double scale;       // the inner problem's right-hand side is rho / scale
    double inv_scale;
    long long iter;     // inner steps, all corrections together
    long long outer;    // corrections (FP64 residuals) done
    int done;           // the inner iteration has stopped: later inner launches return at once
    int outer_done;     // |b - S x| <= tol |b|, out of iterations, or non-finite
    int bad;            // a non-finite scalar was seen
    unsigned count[2];  // arrival counters of the load and residual launches
    int stalled;        // a wait between the blocks of the one-launch solve gave up
    int loops_outer;    // passes of the solve graph's correction loop
    int loops_inner;    // passes of its inner loop in the current correction
};

struct FemDev {
    int64_t nf = 0;    // free nodes: the unknowns of the free subsystem
    int nblk_max = 1;  // most blocks of a launch, hence the row length of the partial sums
    // S(fn, fn): CSR over free rows and columns with FP64 values (the
    // residual), and the same matrix in FP32 in slices of 32 rows for the
    // inner steps (one thread per row: entry k of the slice's lane l at
    // sl_ptr[slice] + 32 k + l, sl_w[slice] entries per row, short rows
    // padded with zero entries at their own column); 1 / diagonal in FP32
    const int64_t *s_ptr = nullptr;
    const int *s_col = nullptr;
    const double *s_val = nullptr;
    const int64_t *sl_ptr = nullptr;
    const int *sl_w = nullptr;
    const int *sl_col = nullptr;
    const float *sl_val = nullptr;
    const float *dinv = nullptr;
    // load operator b(fn) = B m, CSR over free rows, columns are the other
    // nodes of the row's tetrahedra, entries |T|/4 grad eta_row summed over
    // them, applied to the differences m_col - m_row (every free row of B sums
    // to zero, so the row's own column drops out); float4 in FP32 plans,
    // double4 in FP64 plans
    const int *fnode = nullptr;  // node of each free row
    const int64_t *b_ptr = nullptr;
    const int *b_col = nullptr;
    const void *b_val = nullptr;
    double *b = nullptr, *x = nullptr, *rho = nullptr;  // FP64 load, solution and residual
    // the inner iteration (FP32): correction and direction, and per row
    // {r, w = S D^-1 r, s = S p, 1 / diagonal} in buffers of even and odd
    // steps (one 16-byte load gives a column everything the product needs)
    float *xc = nullptr, *p = nullptr;
    float4 *v[2] = {nullptr, nullptr};
    double *part = nullptr;   // [nblk_max] block partial sums, FP64 (load, residual)
    float *part32 = nullptr;  // [2][3][nblk_max] block partial sums of the inner steps, by parity
    CgState *st = nullptr;
    double tol2 = 0.0;    // outer stop: |b - S x|^2 <= tol2 |b|^2
    float inner2 = 0.f;   // inner stop: r.r <= inner2 r0.r0
    long long max_iter = 0;
    // The one-launch solve (parts > 0): the free rows cut into `parts` compact
    // sets of at most rp rows, one block each, renumbered part by part.  A
    // block's columns are its own rows (local index < rp) and its halo, the
    // other parts' rows its entries reach (rp + position in its halo list).
    int parts = 0, rpt = 0, rp = 0, hmax = 0;  // rpt: rows per thread, rp = SOLVE_THREADS rpt
    int solve_reg = 0;                         // 1: the matrix fits the threads' registers
    const int *part_row = nullptr;             // [parts + 1] first row of each part
    const int *row_old = nullptr;              // [nf] free index of a row
    const int *halo_ptr = nullptr;             // [parts + 1] the parts' halo lists, nhalo entries in all
    int64_t nhalo = 0;
    const int *dst_ptr = nullptr, *dst = nullptr;  // [nf + 1], the halo list entries that hold each row
    // off-diagonal entries in slices of 32 rows of a part (slice t of part k at
    // k rp / 32 + t, entry e of lane l at ps_ptr[slice] + 32 e + l): local
    // column, S_ij / sqrt(S_ii S_jj) in FP32, S_ij in FP64
    const int *ps_ptr = nullptr;
    const int *ps_w = nullptr;
    const unsigned short *pe_col = nullptr;
    const float *pe_val = nullptr;
    const double *pe_val64 = nullptr;
    const double *pdiag = nullptr, *pisd = nullptr;  // [nf] S_ii, 1 / sqrt(S_ii)
    const float *pz = nullptr;      // [nf] sqrt(S_ii)
    // coarse space: the parts each part needs the correction of (its own first),
    // at most near_max of them; each halo entry's z and its part's place in that
    // list; the inverse of the parts' matrix [parts][parts]
    const int *near_ptr = nullptr, *near_part = nullptr;
    int near_max = 0;
    const float *halo_z = nullptr;
    const unsigned char *halo_near = nullptr;
    const float *coarse_inv = nullptr;
    // exchanged between blocks, by parity of the exchange: a record per halo
    // list entry and a record of partial sums per pair of blocks (psum[reader parts + writer]),
    // each 16 bytes with its exchange number
    uint4 *rec[2] = {nullptr, nullptr}, *psum[2] = {nullptr, nullptr};
    // boundary triangles: nodes (a, b, c) wound outward and the free index of the
    // owning tetrahedron's fourth node (-1 when it lies on the boundary); unit
    // normal and 1/h, h the tetrahedron's height over the triangle
    int64_t nfaces = 0;
    const int4 *face = nullptr;
    const double4 *face_n = nullptr;
    // per node: free index (>= 0) or -1 - boundary index
    int64_t nnodes = 0;
    const int *slot = nullptr;
};

constexpr int FEM_THREADS = 256;
constexpr int SOLVE_THREADS = 512;  // threads of a block of the one-launch solve
constexpr int SOLVE_PARTS = 256;    // blocks at most (a thread reads one block's sums)
constexpr int SOLVE_RPT[] = {1, 2, 4, 8, 10};  // rows per thread it is compiled for
constexpr int SOLVE_SMEM = 200 * 1024;  // bytes of dynamic shared memory at most
constexpr int SOLVE_REG_W = 16;     // most off-diagonal entries of a row kept in registers (rpt <= 2)
constexpr int FEM_CHUNK = 16;       // inner launches per pass of the inner loop (even: parities repeat)
constexpr double FEM_INNER = 1e-4;  // each correction's inner steps cut its residual by this factor
constexpr int FEM_MAX_OUTER = 64;   // corrections at most

// Loop control of the solve graph (one thread each): the value of a WHILE
// node's handle, from the state.
enum FemLoop { LOOP_OUTER_START, LOOP_OUTER_NEXT, LOOP_INNER_START, LOOP_INNER_NEXT };

// b = B m and x = 0; the first inner iteration set up from r = b / scale
cudaError_t launch_fem_load(const FemDev &d, int prec, const void *m, cudaStream_t s);
// The whole solve in one cooperative launch of d.parts blocks (after
// launch_fem_load); solve_blocks: how many such blocks fit the device at once.
cudaError_t launch_cg_solve(const FemDev &d, cudaStream_t s);
cudaError_t solve_blocks(const FemDev &d, int *blocks);
size_t solve_smem(const FemDev &d);
// one inner launch (parity: the launch's index mod 2; each inner iteration
// starts at parity 0 with a set-up launch, then one step per launch)
cudaError_t launch_cg_iteration(const FemDev &d, int parity, cudaStream_t s);
// x += scale * correction, the FP64 residual, the next inner iteration set up from it
cudaError_t launch_fem_correct(const FemDev &d, cudaStream_t s);
// bound: LOOP_OUTER_NEXT the most corrections, LOOP_INNER_NEXT the most inner passes per correction
cudaError_t launch_fem_loop(FemLoop which, const FemDev &d, cudaGraphConditionalHandle h, int bound, cudaStream_t s);
cudaError_t launch_fem_charges(const FemDev &d, int prec, const void *m, void *g, cudaStream_t s);
cudaError_t launch_fem_combine(const FemDev &d, int prec, const void *phi2_b, const void *phi2_f, void *phi,
                               void *phi1, cudaStream_t s);

}  // namespace slp
