// Internal interface between the host runtime (igr_api.cu) and the kernel
// translation units (igr_kernels.cu, compiled once per storage type).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/igr.h"

namespace igr {

enum { BC_PERIODIC = 0, BC_OUTFLOW = 1, BC_INFLOW = 2 };

// Kernel classes for per-launch timing.
enum { KC_SOURCE = 0, KC_JACOBI = 1, KC_FLUX = 2, KC_OTHER = 3, KC_COUNT = 4 };

struct Geom {
    int nx, ny, nz;
    int bc[6];          // faces -x,+x,-y,+y,-z,+z
    long long plane;    // nx * ny
    long long n;        // nx * ny * nz
};

struct Phys {
    double dx, gamma, alpha, cfl;
    int order;   // face reconstruction: 5 or 3
    double mu, zeta;  // shear and bulk viscosity (0: Euler)
};

// Sigma sweep kinds (igr_config.sigma_solver)
enum { SOLVER_JACOBI = 0, SOLVER_RBGS = 1 };

// bits of Scalars::err
enum { ERRF_NONFINITE = 1, ERRF_FACE = 2 };

// Device-resident scalars of a context.
struct Scalars {
    double dt;          // time step of the current step
    double t;           // accumulated simulated time
    double speed;       // max_d(|u_d| + c) of the state at the start of the step
    int err;            // ERRF_NONFINITE: a non-finite value or dt; ERRF_FACE: a face with rho or p <= 0
    int pad;
};

// Inflow tables on the -z face, in the arithmetic type:
// W[j][i] = sum_n s_n, J[v][j][i] = sum_n s_n q_jet_n[v].
struct Inflow {
    const void *W;
    const void *J;
};

// Launch shapes chosen by the runtime.
struct Tiles {
    int zc_source;  // z-planes per block of the source kernel
    int zc_jacobi;  // z-planes per block of the Jacobi kernel
    int zc_flux;    // z-planes per block of the flux kernel
    int vec_source; // the source's and the sweeps' form: 0 pairs, 1 quads, -1 quads where
    int vec_jacobi; // rows are a multiple of 4 cells (igr_set_kernel_forms)
    int elem;       // 1: the source and the sweeps load element by element (pointers that are not
                    // aligned to 4 values)
    int z_begin;    // a flux launch covers planes [z_begin, z_end) only (z_begin a multiple
    int z_end;      // of zc_flux, z_end a multiple or nz); z_end = 0: all planes
};

// What igr_get_kernel_forms returns for the default setting: 1 where rows of nx
// cells fill blocks of 128 cells at least num / den times as well as blocks of 32,
// the rule by which kernels of one and four cells per thread were chosen. It
// chooses nothing now (igr_get_launch_forms says what is launched); callers
// compare the value.
inline int vec4_default(int nx, int num, int den)
{
    if (nx % 4) return 0;
    const long long t4 = (nx + 127LL) / 128 * 128, t1 = (nx + 31LL) / 32 * 32;
    return t1 * den >= t4 * num ? 1 : 0;  // nx / t4 >= (num / den) (nx / t1)
}
inline int vec4_default_source(int nx) { return vec4_default(nx, 80, 140); }
inline int vec4_default_jacobi(int nx) { return vec4_default(nx, 69, 79); }

// Tile of the source and sweep kernels: wq quads (four cells of a row) by
// rows rows, at most 256 threads, fitted to the plane so that rows of any
// length fill it: the row is cut into the fewest tiles of at most 32 quads,
// and the rows of the plane into tiles of equal height. On small grids lower
// tiles (down to 8 rows) make more blocks: every SM marching a few planes is
// what bounds them.
enum { QUAD_TILE = 1360 };  // cells of the largest plane tile with its halo, (rows + 2)(4 wq + 8)
struct QuadFit {
    int wq, rows, threads, gx, gy;
    bool full;  // 32 x 8 quads, every tile inside the grid
};
inline QuadFit quad_fit(const Geom &g)
{
    QuadFit f;
    const int nq = (g.nx + 3) / 4;
    f.gx = (nq + 31) / 32;
    f.wq = (nq + f.gx - 1) / f.gx;
    int rmax = 256 / f.wq < 32 ? 256 / f.wq : 32;
    while (rmax > 8 && (long long)f.gx * ((g.ny + rmax - 1) / rmax) * ((g.nz + 3) / 4) < 2 * 152) rmax = rmax / 2 < 8 ? 8 : rmax / 2;
    f.gy = (g.ny + rmax - 1) / rmax;
    f.rows = (g.ny + f.gy - 1) / f.gy;
    const int own = f.wq * f.rows, halo = 2 * f.wq + 2 * f.rows;  // a thread each
    f.threads = ((own > halo ? own : halo) + 31) / 32 * 32;
    f.full = g.nx % 128 == 0 && g.ny % 8 == 0 && f.rows == 8;
    return f;
}

// Alignment of caller device pointers. Every kernel reads and writes whole
// elements, so a pointer must be aligned to its element size. The source and
// the sweeps load and store 4 consecutive values at once on rows of a
// multiple of 4 cells (8 bytes at 16-bit storage, 16 bytes for FP32 and, as
// two 16-byte accesses, for FP64), so they need the field bases aligned to
// that; a call whose pointers are not takes element accesses (Tiles::elem),
// which give the same bits.
inline bool is_aligned(const void *p, size_t a) { return ((uintptr_t)p & (a - 1)) == 0; }
inline size_t vec4_align(int storage_bytes) { return storage_bytes * 4 > 16 ? 16 : (size_t)storage_bytes * 4; }

// Launches of a step's kernels (programmatic dependent launch). A kernel launched
// by `launch` may be placed on the SMs once every block of the kernel before it
// has begun, and waits in `launched`, its first statement, until that kernel has
// completed and its writes are visible to ordinary loads; so the order of all
// memory accesses is that of plain launches, and only the launch itself overlaps.
// Read-only loads (__ldg, const __restrict__) are not for such a kernel: the data
// change during its lifetime. A kernel without `launched` is launched plainly.
// The gap between two kernels was about 2 us, most of a small grid's step: ten
// steps at 32^3 (220 launches) 1671 us before, 1197 now; 254 x 201 x 130, 70
// launches a two-step run: 3958 and 3820.
__device__ __forceinline__ void launched()
{
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}
template <class... P, class... T>
cudaError_t launch(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, T &&...args)
{
    cudaLaunchAttribute overlap = {};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &overlap;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, kern, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // returned here, not left for a later call
    return e;
}

// Stage modes of the flux kernel.
enum { FLUX_RHS = 0, FLUX_STAGE1 = 1, FLUX_STAGE2 = 2, FLUX_STAGE3 = 3 };

// Kernel set of one storage type. Every entry enqueues on `st` and returns
// the launch error (cudaGetLastError) without synchronising.
struct Ops {
    int storage_bytes;  // bytes per stored value (Sigma, b; the increments of the increment modes)
    int compute_bytes;  // bytes per arithmetic value (8 for FP64, else 4)
    int state_bytes;    // bytes per value of the state q^n (the storage type; 4 in the increment modes)
    // b = alpha [tr(G^2) + tr(G)^2] from the stage state q (+ increments qd in the
    // increment modes, NULL in stage 1 and in every other mode); in the increment
    // modes rho_out gets the stage density in the storage type, which the sweeps
    // read as their q (NULL otherwise)
    cudaError_t (*source)(const Geom &, const Phys &, const Tiles &, const Inflow &,
                          const void *q, const void *qd, void *b, void *rho_out, cudaStream_t st);
    // one Jacobi sweep s_out <- (b + beta sum c s_in) / (1/rho + beta sum c) with
    // colour < 0; with colour 0 or 1 one red-black Gauss-Seidel half-sweep in
    // place (s_in == s_out), updating the cells with (i + j + k) % 2 == colour
    cudaError_t (*jacobi)(const Geom &, const Phys &, const Tiles &, const void *q,
                          const void *b, const void *s_in, void *s_out, int colour, cudaStream_t st);
    // flux divergence and RK stage (mode FLUX_STAGE*), or L(q; Sigma) into rhs (FLUX_RHS).
    // Stage 3 also writes the per-block maximum wave speed of its output to blockmax.
    // Stage 1 with base_out != NULL also copies its input qs there (the RK base of
    // stages 2 and 3 when it lives in host memory). In the increment modes the
    // stage input is qs (= q^n) plus the increments qd (stages 2 and 3; NULL in
    // stage 1 and in every other mode), stages 1 and 2 write increments to out
    // and stage 3 writes the FP32 state q^n+1 to out.
    cudaError_t (*flux)(const Geom &, const Phys &, const Tiles &, const Inflow &, int mode,
                        const void *qs, const void *qd, const void *sig, const void *qn, void *out,
                        void *rhs, void *base_out, const Scalars *sc, double *blockmax, int *err,
                        cudaStream_t st);
    // number of blocks of the flux launch (entries of blockmax it writes)
    long long (*flux_blocks)(const Geom &, const Tiles &);
    // per-block maximum wave speed of q; returns the block count in *nblocks
    cudaError_t (*speed)(const Geom &, const Phys &, const void *q, double *blockmax,
                         int *nblocks, cudaStream_t st);
    // out = qn + w ((qs - qn) + dt L) over n values, exactly as the flux
    // kernel's epilogue stores it (L in the arithmetic type; in the increment
    // modes the FP32 state update of stage 3 on FP32 arrays)
    cudaError_t (*rk_combine)(const void *qn, const void *qs, const void *L, void *out,
                              long long n, double dt, double w, cudaStream_t st);

    // ---- adjoint (all adjoint buffers in the arithmetic type) ----
    // reverse of the stage combination (weight w) and of L(qs; sig), from the adjoint
    // lout of the stage's output: lqs (5 n) = the adjoint of qs, lq0 += (1 - w) lout
    // (first: =), lsig += the adjoint of sig, lamJ += that of the inflow tables (5 x plane)
    cudaError_t (*adj_rhs)(const Geom &, const Phys &, const Inflow &, const void *qs, const void *sig,
                           const void *lout, void *lqs, void *lq0, void *lsig, void *lamJ, double w, double dt,
                           int first, cudaStream_t st);
    // r = 1 / rho, the diagonal of the sweeps and (FP64 only) its inverse
    cudaError_t (*adj_diag)(const Geom &, const Phys &, const void *q, void *r, void *diag, void *dinv,
                            cudaStream_t st);
    // one reversed Jacobi sweep s_k -> F: lsig (adjoint of F) -> nl (adjoint of s_k);
    // lb += mu, rb += d/d(1/rho) (first: =)
    cudaError_t (*adj_jacobi)(const Geom &, const Phys &, const void *r, const void *diag, const void *dinv,
                              const void *sk, const void *F, const void *lsig, void *nl, void *lb, void *rb,
                              int first, cudaStream_t st);
    // reverse of the IGR source and of 1 / rho: lb, rb -> lqs (rho, m), lamJ; grads: nine
    // scratch arrays of n values
    cudaError_t (*adj_source)(const Geom &, const Phys &, const Inflow &, const void *q, const void *r,
                              const void *lb, const void *rb, void *const grads[9], void *lqs, void *lamJ,
                              cudaStream_t st);
    // out = a + b (n values)
    cudaError_t (*adj_add)(const void *a, const void *b, void *out, long long n, cudaStream_t st);
    // gw[n] = sum over the inflow face of s_n (rho_n lamJ_mz + rho_n w_n lamJ_E); gw holds
    // njets (1 + ADJ_JET_BLOCKS) values, the sums and the blocks' shares
    cudaError_t (*adj_jets)(const Geom &, const Phys &, const double *jets, int njets,
                            const void *lamJ, double *gw, cudaStream_t st);
    // ---- the scatter forms of the faces' and the source's reverse (by atomics)
    // lq0 += (1 - w) lout; lqs = w lout; Lb = w dt lout   (5 n values)
    cudaError_t (*adj_rk)(const void *lout, void *lq0, void *lqs, void *Lb, long long n5, double w,
                          double dt, cudaStream_t st);
    // reverse of L(qs; sig): Lb -> lqs (5 fields), lsig, lamJ (5 x plane)
    cudaError_t (*adj_rhs_scatter)(const Geom &, const Phys &, const Inflow &, const void *qs,
                                   const void *sig, const void *Lb, void *lqs, void *lsig, void *lamJ,
                                   cudaStream_t st);
    // lqs[rho] -= rb / rho^2
    cudaError_t (*adj_rho)(const Geom &, const void *q, void *rb, void *lqs, cudaStream_t st);
    // reverse of the IGR source: lb -> lqs (rho, m), lamJ
    cudaError_t (*adj_source_scatter)(const Geom &, const Phys &, const Inflow &, const void *q,
                                      const void *lb, void *lqs, void *lamJ, cudaStream_t st);

    // ---- diagnostics (FP64) ----
    // per-block partials (DIAG_PARTS doubles each) of the state's totals,
    // extrema and the elliptic residual; *nblocks <= DIAG_MAXBLOCKS blocks
    cudaError_t (*diag)(const Geom &, const Phys &, const Inflow &, const void *q, const void *sig,
                        double *part, int *nblocks, cudaStream_t st);

    // ---- debug build (IGR_DEBUG_BOUNDS) ----
    // out-of-range indices counted by the forward kernels since the last clear
    // (~0 when the library is not a debug build); a self-test forming one
    // out-of-range index (checked, never dereferenced; sink is never written)
    unsigned long long (*bounds_hits)(int clear);
    cudaError_t (*bounds_selftest)(int *sink, cudaStream_t st);

    // ---- grouped launches over independent instances (batches) ----
    // One launch per kernel class covers every instance's blocks; each
    // instance keeps its own grid, launch shape and buffers, so its results
    // are bitwise those of its own launches. The launchers split the calls
    // into groups a single launch can take (the same kernel form, at most
    // kGroupMax instances).
    cudaError_t (*source_group)(const struct SourceCall *calls, int n, cudaStream_t st);
    cudaError_t (*jacobi_group)(const struct JacobiCall *calls, int n, int colour, cudaStream_t st);
    cudaError_t (*flux_group)(const struct FluxCall *calls, int n, int mode, cudaStream_t st);

    // blocks per plane of the source / of a sweep, and the blocks per SM that
    // their registers allow (for the choice of the z-chunks)
    // (source_form, sweep_form: 1 where the launch takes quads, 0 pairs)
    int (*source_form)(const Geom &, const Tiles &);
    int (*sweep_form)(const Geom &, const Tiles &);
    void (*source_shape)(const Geom &, long long *cols, int *resident);
    void (*jacobi_shape)(const Geom &, long long *cols, int *resident);
    // FP64 (NULL in the other modes): the sweeps' coefficients of the density q into
    // coefs (5 n scratch values), and a sweep with them; arguments and results as jacobi
    cudaError_t (*coefs)(const Geom &, const Phys &, const void *q, void *coefs, cudaStream_t st);
    cudaError_t (*sweep)(const Geom &, const void *coefs, const void *b, const void *s_in, void *s_out, int colour,
                         cudaStream_t st);
};

// One instance's arguments of a grouped launch (the same as the single
// launch's, see Ops::source, Ops::jacobi, Ops::flux).
struct SourceCall {
    Geom g;
    Phys p;
    Tiles t;
    Inflow in;
    const void *q, *qd;
    void *b, *rho_out;
};
struct JacobiCall {
    Geom g;
    Phys p;
    Tiles t;
    const void *q, *b, *s_in;
    void *s_out;
};
struct FluxCall {
    Geom g;
    Phys p;
    Tiles t;
    Inflow in;
    const void *qs, *qd, *sig, *qn;
    void *out;
    const Scalars *sc;
    double *blockmax;
    int *err;
};

// blocks per jet of the adjoint's sum over the inflow face
enum { ADJ_JET_BLOCKS = 32 };

// instances per grouped launch: their descriptors travel as one kernel
// parameter (at most 32 KB)
enum { kGroupMax = 64 };

// layout of one block's diagnostics partials: sums of rho, mx, my, mz, E,
// (A Sigma - b)^2, b^2; minima of rho and p; maximum |Sigma|
enum { DIAG_PARTS = 10, DIAG_BLOCKS_MAX = 152 * 8 };

extern const Ops ops_f64, ops_f32, ops_f16, ops_bf16, ops_f16inc, ops_bf16inc;

// shared by the host entry points (igr_api.cu, igr_noalloc.cu)
const Ops *ops_for(int precision);             // kernel set of an igr_precision
Tiles default_tiles(const Geom &g, const Ops *o);  // launch shapes for a grid
const char *validate_config(const igr_config *c);  // NULL when valid

}  // namespace igr
