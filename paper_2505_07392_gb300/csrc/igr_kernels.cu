// Stage kernels of the IGR Euler solver, compiled once per storage type
// (IGR_STORAGE = double | float | __half | __nv_bfloat16, exported as the
// kernel set IGR_OPS).
//
// Layout: structure of arrays, q[v][k][j][i] with x fastest, interior cells
// only; boundary conditions act by index mapping (periodic wrap, zero-
// gradient clamp, jet blend on the -z face), never through ghost storage.
//
// All three kernels are 2.5D: a block owns a TX x TY tile of (x, y) columns
// and marches up a chunk of z-planes, keeping the column's z-neighbours in
// registers and taking x/y neighbours from the plane just loaded.
//
//   k_source  grad u (2nd-order central) and the IGR source
//             b = alpha [tr(G^2) + tr(G)^2]            (Eq. igrelliptic)
//   k_jacobi  one Jacobi sweep of the 7-point operator
//             A s = s/rho - alpha div(grad s / rho)    (Eq. igrelliptic)
//   k_flux    5th-order face values of (rho, m, E, Sigma), local
//             Lax-Friedrichs flux with pressure p + Sigma
//             (Eqs. igrmabalance-igrenbalance, Sec. "Discretization"),
//             divergence, and the SSP-RK3 stage combination
//             out = qn + w [(qs - qn) + dt L]   (w = 1, 1/4, 2/3);
//             stage 3 also reduces max_d(|u_d| + c) of its output for the
//             next dt. No atomics on the data path: every face flux is
//             computed once per tile and the divergence sums in a fixed
//             order, so results are deterministic.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <stdio.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "igr_internal.h"

#ifndef IGR_STORAGE
#error "IGR_STORAGE must name the storage type"
#endif

namespace igr {
namespace {

using S = IGR_STORAGE;

// arithmetic type C and RK-combination type A of each storage type
template <typename T> struct Num;
template <> struct Num<double> { using C = double; using A = double; };
template <> struct Num<float> { using C = float; using A = float; };
template <> struct Num<__half> { using C = float; using A = double; };
template <> struct Num<__nv_bfloat16> { using C = float; using A = double; };
using C = Num<S>::C;
using A = Num<S>::A;

// Type of the conserved state q^n. It is the storage type, except in the
// increment modes (IGR_BASE=float, with 16-bit S): there q^n is kept in FP32
// and RK stages 1 and 2 store the 16-bit increments d_s = q_s - q^n, so a
// stage reads its input as q_s = RN32(q^n + d_s) and the RK accumulation of
// q^n never rounds to 16 bits. Sigma, b and the increments use S.
#ifdef IGR_BASE
using QB = IGR_BASE;
constexpr bool kInc = true;
#else
using QB = S;
constexpr bool kInc = false;
#endif

// Offsets inside one field are 32-bit (grids hold fewer than 2^32 cells);
// each field has its own base pointer, so an address is one 32x32->64 step.
using idx = unsigned;
// Index checks of the debug build (IGR_DEBUG_BOUNDS, a separate library):
// every global index the forward kernels form, and every shared-memory index
// that depends on more than the thread's position in its block (halo slots,
// the flux kernel's tile and face-buffer offsets), is compared with its
// array's length; an index out of range is counted and replaced by 0, so
// nothing is accessed out of bounds and the count is read on the host. In
// the normal build the checks compile to nothing.
#ifdef IGR_DEBUG_BOUNDS
static __device__ unsigned long long g_bounds_hits;
// element offset c of an array of n values (offsets are unsigned: a
// negative one wraps to a value >= n on the grids the checks run on)
__device__ __forceinline__ idx ck(idx c, long long n)
{
    if ((long long)c >= n) {
        atomicAdd(&g_bounds_hits, 1ull);
        return 0;
    }
    return c;
}
// pointer p to w consecutive values of the array of n values at base
template <class T>
__device__ __forceinline__ T *ckp(T *p, T *base, long long n, int w)
{
    const long long d = p - base;
    if (d < 0 || d + w > n) {
        atomicAdd(&g_bounds_hits, 1ull);
        return base;
    }
    return p;
}
// 64-bit element offset c of an array of n values
__device__ __forceinline__ size_t ckl(size_t c, long long n)
{
    if ((long long)c >= n) {
        atomicAdd(&g_bounds_hits, 1ull);
        return 0;
    }
    return c;
}
#define CKP(p, base, n) ckp((p), (base), (long long)(n), 1)
#define CKP4(p, base, n) ckp((p), (base), (long long)(n), 4)
// shared-memory element index c of a tile of n elements
__device__ __forceinline__ int cks(int c, int n)
{
    if (c < 0 || c >= n) {
        atomicAdd(&g_bounds_hits, 1ull);
        return 0;
    }
    return c;
}
// the first of 4 consecutive shared values of a vector access: in range and
// a multiple of 4 (16-byte aligned for 4-byte values)
__device__ __forceinline__ int cks4(int c, int n)
{
    if (c < 0 || c + 3 >= n || (c & 3)) {
        atomicAdd(&g_bounds_hits, 1ull);
        return 0;
    }
    return c;
}
#else
__device__ __forceinline__ idx ck(idx c, long long) { return c; }
__device__ __forceinline__ size_t ckl(size_t c, long long) { return c; }
#define CKP(p, base, n) (p)
#define CKP4(p, base, n) (p)
__device__ __forceinline__ int cks(int c, int) { return c; }
__device__ __forceinline__ int cks4(int c, int) { return c; }
#endif

template <int N> struct Fout { S *p[N]; };        // fields written
struct Frhs { C *p[5]; };
struct QBIn { const QB *p[5]; };                  // the state q^n (RK base)
struct QBOut { QB *p[5]; };                       // a new state q^n+1

// ------------------------------------------------------------ load/store
// Read-only (non-coherent) loads, for kernels that are launched plainly. A kernel
// that begins with launched() is resident while its predecessor writes, so it
// takes ordinary loads (ldv, ldr, ld4r, cp.async) and no __restrict__ pointers, and
// the writes that it waited for are visible to them. They cost next to nothing
// (plume 1024 x 1024 x 512, FP16 increments: 140.0 ms before, 139.7 now; two steps
// of 512 x 512 x 128: FP16 8.43 and 8.39 ms, FP32 9.58 and 9.64, BF16 8.42 and 8.78).
__device__ __forceinline__ double ldc(const double *p) { return __ldg(p); }
__device__ __forceinline__ float ldc(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ldc(const __half *p) { return __half2float(__ldg(p)); }
__device__ __forceinline__ float ldc(const __nv_bfloat16 *p) { return __bfloat162float(__ldg(p)); }

// Raw (ordinary) loads for prefetching: the value stays in its storage type until it is
// used, so no instruction waits on the load before then (a conversion right
// after the load would stall there and hide nothing).
// An ordinary load in the order of the source: the compiler may not move it over
// the wait, and the element loads of a plane stay together (as plain reads, which it
// moves between the stores, two FP16 steps of 512 x 512 x 128 took 8.51 ms against
// 8.39, the right-hand side with FP16 increments 818 us against 785).
__device__ __forceinline__ double ldv(const double *p) { return *p; }
__device__ __forceinline__ float ldv(const float *p)
{
    float r;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(r) : "l"(p));
    return r;
}
template <class H> __device__ __forceinline__ H ldv(const H *p)
{
    static_assert(sizeof(H) == 2, "16-bit types");
    unsigned short r;
    asm volatile("ld.global.b16 %0, [%1];" : "=h"(r) : "l"(p));
    return *reinterpret_cast<H *>(&r);
}
__device__ __forceinline__ S ldr(const S *p) { return ldv(p); }
__device__ __forceinline__ double cv(double v) { return v; }
__device__ __forceinline__ float cv(float v) { return v; }
__device__ __forceinline__ float cv(__half v) { return __half2float(v); }
__device__ __forceinline__ float cv(__nv_bfloat16 v) { return __bfloat162float(v); }

// Reading the state of a stage: the base fields b (type QB) plus, in the
// increment modes from stage 2 on, the increments d (type S). HASD says
// whether increments are read; without them the state is the base itself.
struct QIn {
    const QB *b[5];
    const S *d[5];
    size_t fs;  // values between consecutive fields of b and of d (the increment
                // modes address the fields from b[0] and d[0] with it)
};
struct QRawInc {  // one raw state value of the increment modes
    QB b;
    S d;
};
template <bool INC> struct StateIO;
template <> struct StateIO<false> {  // (used where the state has the storage type)
    using Raw = S;
    template <bool HASD> static __device__ __forceinline__ S ld(const QIn &q, int u, idx c)
    {
        return ldr(reinterpret_cast<const S *>(q.b[u]) + c);
    }
    template <bool HASD> static __device__ __forceinline__ C val(S r) { return cv(r); }
};
template <> struct StateIO<true> {
    using Raw = QRawInc;
    template <bool HASD> static __device__ __forceinline__ QRawInc ld(const QIn &q, int u, idx c)
    {
        QRawInc r;
        r.b = ldv(q.b[0] + u * q.fs + c);
        r.d = HASD ? ldr(q.d[0] + u * q.fs + c) : S(0.0f);
        return r;
    }
    // the stage value q_s = RN32(q^n + d_s) (q^n itself without increments)
    template <bool HASD> static __device__ __forceinline__ C val(const QRawInc &r)
    {
        return HASD ? C(__fadd_rn(float(cv(r.b)), float(cv(r.d)))) : C(cv(r.b));
    }
};
using QRaw = StateIO<kInc>::Raw;
template <bool HASD> __device__ __forceinline__ QRaw ldqr(const QIn &q, int u, idx c)
{
    return StateIO<kInc>::ld<HASD>(q, u, c);
}
template <bool HASD> __device__ __forceinline__ C cvq(const QRaw &r) { return StateIO<kInc>::val<HASD>(r); }
template <bool HASD> __device__ __forceinline__ C ldq(const QIn &q, int u, idx c)
{
    return cvq<HASD>(ldqr<HASD>(q, u, c));
}

// store v rounded to nearest even; returns the stored value in type C
__device__ __forceinline__ double stc(double *p, double v) { *p = v; return v; }
__device__ __forceinline__ float stc(float *p, float v) { *p = v; return v; }
__device__ __forceinline__ float stc(__half *p, double v)
{
    __half h = __double2half(v);
    *p = h;
    return __half2float(h);
}
__device__ __forceinline__ float stc(__half *p, float v)
{
    __half h = __float2half_rn(v);
    *p = h;
    return __half2float(h);
}
__device__ __forceinline__ float stc(__nv_bfloat16 *p, double v)
{
    __nv_bfloat16 h = __double2bfloat16(v);
    *p = h;
    return __bfloat162float(h);
}
__device__ __forceinline__ float stc(__nv_bfloat16 *p, float v)
{
    __nv_bfloat16 h = __float2bfloat16_rn(v);
    *p = h;
    return __bfloat162float(h);
}

// ------------------------------------------------------------ arithmetic
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double sqrt_c(double x) { return sqrt(x); }
__device__ __forceinline__ float sqrt_c(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// products that are never fused into a following add: velocities u = m/rho
// must round before they are differenced, so equal neighbours give an exact 0
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
// rounded operations that the compiler neither fuses nor reorders, for
// sequences that two kernel forms must evaluate identically
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// NaN-propagating maximum (a NaN wave speed must reach dt)
__device__ __forceinline__ double nanmax(double a, double b) { return (a > b || a != a) ? a : b; }

// Pairs of arithmetic values for packed FP32x2 operations (add.rn.f32x2,
// mul.rn.f32x2, fma.rn.f32x2 on sm_100 and later: each lane rounds exactly
// like the scalar operation); FP64 pairs take two scalar operations.
template <typename T> struct PairOf;
template <> struct PairOf<float> { using T = float2; };
template <> struct PairOf<double> { using T = double2; };
using C2 = typename PairOf<C>::T;

__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 pmul(double2 a, double2 b)
{
    return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y));
}
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c)
{
    return make_double2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
}
// a - b
__device__ __forceinline__ float2 psub(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n sub.rn.f32x2 rd, ra, rb;\n"
        " mov.b64 {%0, %1}, rd;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ double2 psub(double2 a, double2 b)
{
    return make_double2(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y));
}
__device__ __forceinline__ C2 pset(C x, C y)
{
    C2 r;
    r.x = x;
    r.y = y;
    return r;
}
__device__ __forceinline__ C2 bcast(C v) { return pset(v, v); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 padd(double2 a, double2 b)
{
    return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}

// ------------------------------------------------------------ indexing
__device__ __forceinline__ int wrap(int c, int n)
{
    c %= n;
    return c < 0 ? c + n : c;
}
// in-range index for coordinate c along an axis of n cells
__device__ __forceinline__ int map_axis(int c, int n, int bclo, int bchi)
{
    if (c < 0) return bclo == BC_PERIODIC ? wrap(c, n) : 0;
    if (c >= n) return bchi == BC_PERIODIC ? wrap(c, n) : n - 1;
    return c;
}

// 5th-order finite-volume face values at face i+1/2 from cell averages
// v[i-2..i+3]: the quartic through the five cell averages of the left-
// (resp. right-) biased stencil, evaluated at the face.
__device__ __forceinline__ C rec_left(C a, C b, C c, C d, C e)
{
    return C(2.0 / 60.0) * a - C(13.0 / 60.0) * b + C(47.0 / 60.0) * c + C(27.0 / 60.0) * d -
           C(3.0 / 60.0) * e;
}
__device__ __forceinline__ C rec_right(C b, C c, C d, C e, C f)
{
    return C(-3.0 / 60.0) * b + C(27.0 / 60.0) * c + C(47.0 / 60.0) * d - C(13.0 / 60.0) * e +
           C(2.0 / 60.0) * f;
}

// Doubled local Lax-Friedrichs flux along axis D from face states (rho, mx,
// my, mz, E, Sigma) on the left and right:
//   G = 2 F_hat = (F_L + F_R) - lam (q_R - q_L),
//   F = (m_D, m u_D + (p + Sigma) e_D, (E + p + Sigma) u_D),
//   p = (gamma - 1)(E - |m|^2 / (2 rho)), lam = max(|u_D| + c) over both sides,
//   c = sqrt(gamma p / rho).
// (The factor 1/2 is applied once, in the divergence.) Flags a non-positive
// face density or pressure.
// The warning flag of non-positive face states. In the 16-bit storage forms
// it is a running minimum of the face densities and pressures, tested once
// per block (fewer instructions per face: their flux kernel ran 2.4% faster
// at full size); FP32 and FP64 storage keep a boolean per face (the minimum
// measured 0.9% slower there). A face whose four values are all NaN sets
// the boolean and not the minimum; its outputs raise the non-finite error.
constexpr bool kFaceMin = sizeof(S) == 2;
using FaceFlag = std::conditional<kFaceMin, C, bool>::type;
__device__ __forceinline__ void flag_face(bool &f, C a, C b, C c, C d) { f |= !(fmin(fmin(a, b), fmin(c, d)) > C(0)); }
template <class T> __device__ __forceinline__ void flag_face(T &f, C a, C b, C c, C d)
{
    f = fmin(f, fmin(fmin(a, b), fmin(c, d)));
}
__device__ __forceinline__ bool flag_bad(bool f) { return f; }
template <class T> __device__ __forceinline__ bool flag_bad(T f) { return !(f > T(0)); }
// The five components of a flux: (rho, m_x), (m_y, m_z), E
struct Flux {
    C2 a, b;
    C e;
};
// gas constants of the flux: gamma and gamma - 1
struct Gas {
    C gamma, gm1;
};
template <int D>
__device__ __forceinline__ void lf_flux2(const C2 (&L)[3], const C2 (&R)[3], const Gas gas, Flux &G, FaceFlag &bad)
{
    const C mL = D == 0 ? L[0].y : D == 1 ? L[1].x : L[1].y, mR = D == 0 ? R[0].y : D == 1 ? R[1].x : R[1].y;
    const C rL = rcp(L[0].x), rR = rcp(R[0].x);
    const C uL = mL * rL, uR = mR * rR;
    const C pL = gas.gm1 * (L[2].x - C(0.5) * ((L[0].y * L[0].y + L[1].x * L[1].x + L[1].y * L[1].y) * rL));
    const C pR = gas.gm1 * (R[2].x - C(0.5) * ((R[0].y * R[0].y + R[1].x * R[1].x + R[1].y * R[1].y) * rR));
    flag_face(bad, L[0].x, R[0].x, pL, pR);
    const C aL = fabs(uL) + sqrt_c(gas.gamma * pL * rL);
    const C aR = fabs(uR) + sqrt_c(gas.gamma * pR * rR);
    const C lam = fmax(aL, aR);  // a NaN speed comes with a flagged face
    const C PL = pL + L[2].y, PR = pR + R[2].y;
    const C2 nl = bcast(-lam);
    C fx = L[0].y * uL + R[0].y * uR, fy = L[1].x * uL + R[1].x * uR, fz = L[1].y * uL + R[1].y * uR;
    if (D == 0) fx += PL + PR;
    if (D == 1) fy += PL + PR;
    if (D == 2) fz += PL + PR;
    G.a = pfma(nl, psub(R[0], L[0]), pset(mL + mR, fx));
    G.b = pfma(nl, psub(R[1], L[1]), pset(fy, fz));
    G.e = ((L[2].x + PL) * uL + (R[2].x + PR) * uR) - lam * (R[2].x - L[2].x);
}

// wave speed max_d |u_d| + c at a cell
__device__ __forceinline__ C cell_speed(C rho, C mx, C my, C mz, C E, C gamma, C gm1)
{
    C r = rcp(rho);
    C p = gm1 * (E - C(0.5) * (mx * mx + my * my + mz * mz) * r);
    C um = fmax(fabs(mx), fmax(fabs(my), fabs(mz))) * r;
    return um + sqrt_c(gamma * p * r);
}

// block-wide NaN-propagating max of v; thread 0 of the block gets the result
template <int NT>
__device__ __forceinline__ double block_max(double v)
{
    __shared__ double red[NT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = nanmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    int tid = threadIdx.x + threadIdx.y * blockDim.x;
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < NT / 32; w++) v = nanmax(v, red[w]);
    }
    return v;
}

// ------------------------------------------------ 16-bit RK combination
// The stage combination v = qn + w ((qs - qn) + dt L) is specified in FP64
// and then rounded to the 16-bit storage format. FP64 runs at a small
// fraction of the FP32 rate on this GPU, so it is evaluated in FP32 with a
// rigorous bound e on |v32 - v64|:
//   d = RN(qs - qn), p = RN(dt32 L + d), v = RN(w32 p + qn) with dt32, w32
//   the FP32 roundings of dt, w (w <= 1) gives, to first order,
//   |v32 - v64| <= 2^-24 (|v| + 3 |p| + 2 |d|) <= 2^-22 (|v| + |p| + |d|),
//   the slack covering the FP64 evaluation's own rounding and the FP32
//   evaluation of e; where a rounding result is an FP32 subnormal its error
//   is absolute (at most 2^-150), so e adds 2^-148 for the three roundings.
// So v64 lies in [RD(v32 - e), RU(v32 + e)] (directed FP32 roundings).
// Rounding to nearest-even is monotone: when both ends of that interval round
// to the same storage value (with -0 equal to +0), so does v64. Both ends are
// converted by one packed conversion and compared as a pair. Otherwise (for
// smooth data, about e / spacing of the values, well under one in a
// thousand) the combination is redone in FP64. The stored value therefore
// always equals the FP64 evaluation rounded to nearest-even, with zeros
// stored as +0.
template <typename T> struct Narrow;
template <> struct Narrow<__half> {
    using T2 = __half2;
    static __device__ __forceinline__ __half rn(double v) { return __double2half(v); }
    // (RN(a), RN(b)) in the low and high halves, one conversion
    static __device__ __forceinline__ __half2 rn2(float a, float b) { return __floats2half2_rn(a, b); }
    static __device__ __forceinline__ bool eq2(__half2 a, __half2 b) { return __hbeq2(a, b); }
    static __device__ __forceinline__ __half2 swap(__half2 a) { return __lowhigh2highlow(a); }
    static __device__ __forceinline__ __half lo(__half2 a) { return __low2half(a); }
    static __device__ __forceinline__ __half hi(__half2 a) { return __high2half(a); }
    // zeros are stored as +0 (-0 + +0 = +0 under round-to-nearest)
    static __device__ __forceinline__ __half canon(__half h) { return __hadd(h, __ushort_as_half(0)); }
    static __device__ __forceinline__ __half2 canon2(__half2 h)
    {
        return __hadd2(h, __halves2half2(__ushort_as_half(0), __ushort_as_half(0)));
    }
};
template <> struct Narrow<__nv_bfloat16> {
    using T2 = __nv_bfloat162;
    static __device__ __forceinline__ __nv_bfloat16 rn(double v) { return __double2bfloat16(v); }
    static __device__ __forceinline__ __nv_bfloat162 rn2(float a, float b) { return __floats2bfloat162_rn(a, b); }
    static __device__ __forceinline__ bool eq2(__nv_bfloat162 a, __nv_bfloat162 b) { return __hbeq2(a, b); }
    static __device__ __forceinline__ __nv_bfloat162 swap(__nv_bfloat162 a) { return __lowhigh2highlow(a); }
    static __device__ __forceinline__ __nv_bfloat16 lo(__nv_bfloat162 a) { return __low2bfloat16(a); }
    static __device__ __forceinline__ __nv_bfloat16 hi(__nv_bfloat162 a) { return __high2bfloat16(a); }
    static __device__ __forceinline__ __nv_bfloat16 canon(__nv_bfloat16 h)
    {
        return __hadd(h, __ushort_as_bfloat16(0));
    }
    static __device__ __forceinline__ __nv_bfloat162 canon2(__nv_bfloat162 h)
    {
        return __hadd2(h, __halves2bfloat162(__ushort_as_bfloat16(0), __ushort_as_bfloat16(0)));
    }
};

// FP64 evaluation, out of line so that only the rare lanes that need it run
// FP64 instructions
template <typename T>
__device__ __noinline__ T rk_fp64(float qn, float qs, float L, double dt, double w)
{
    double vd = __dadd_rn(double(qn),
                          __dmul_rn(w, __dadd_rn(__dsub_rn(double(qs), double(qn)),
                                                 __dmul_rn(dt, double(L)))));
    return Narrow<T>::canon(Narrow<T>::rn(vd));
}

// FP32 evaluation v of one combination and the bound e on |v - v64|
__device__ __forceinline__ float rk_eval32(float qn, float qs, float L, float dt32, float w32, float &e)
{
    float d = __fsub_rn(qs, qn);
    float pp = __fmaf_rn(dt32, L, d);
    float v = __fmaf_rn(w32, pp, qn);
    // relative rounding errors, plus 2^-148 for the three roundings whose
    // results may be FP32 subnormals (absolute error up to 2^-150 each)
    e = __fmaf_rn(fabsf(v) + fabsf(pp) + fabsf(d), 0x1p-22f, 0x1p-148f);
    return v;
}

// Two combinations rounded to the storage format (low, high); ok = false
// when either rounding could differ from the FP64 evaluation's
template <typename T>
__device__ __forceinline__ typename Narrow<T>::T2 rk_narrow_pair(float qn0, float qs0, float L0, float qn1,
                                                                 float qs1, float L1, float dt32, float w32,
                                                                 bool &ok)
{
    using NR = Narrow<T>;
    float e0, e1;
    const float v0 = rk_eval32(qn0, qs0, L0, dt32, w32, e0);
    const float v1 = rk_eval32(qn1, qs1, L1, dt32, w32, e1);
    const typename NR::T2 a = NR::rn2(__fsub_rd(v0, e0), __fsub_rd(v1, e1));
    const typename NR::T2 b = NR::rn2(__fadd_ru(v0, e0), __fadd_ru(v1, e1));
    ok = NR::eq2(a, b);
    return NR::canon2(b);
}

// One combination rounded to the storage format; ok as for the pair
template <typename T>
__device__ __forceinline__ T rk_narrow_one(float qn, float qs, float L, float dt32, float w32, bool &ok)
{
    using NR = Narrow<T>;
    float e;
    const float v = rk_eval32(qn, qs, L, dt32, w32, e);
    const typename NR::T2 x = NR::rn2(__fsub_rd(v, e), __fadd_ru(v, e));
    ok = NR::eq2(x, NR::swap(x));
    return NR::canon(NR::hi(x));
}

constexpr bool kNarrow = sizeof(S) == 2;

// The 16-bit stage combination of one cell's five values: two pairs and a
// single value, one branch per cell for the rare FP64 re-evaluations (a pair
// that failed is redone in FP64 for both of its values)
template <typename T>
__device__ __forceinline__ void rk_narrow5(const C qn[5], const C qs[5], const C L[5], C dt32, double dt,
                                           C w32, double w, T h[5])
{
    using NR = Narrow<T>;
    bool ok01, ok23, ok4;
    const typename NR::T2 h01 = rk_narrow_pair<T>(qn[0], qs[0], L[0], qn[1], qs[1], L[1], dt32, w32, ok01);
    const typename NR::T2 h23 = rk_narrow_pair<T>(qn[2], qs[2], L[2], qn[3], qs[3], L[3], dt32, w32, ok23);
    h[0] = NR::lo(h01);
    h[1] = NR::hi(h01);
    h[2] = NR::lo(h23);
    h[3] = NR::hi(h23);
    h[4] = rk_narrow_one<T>(qn[4], qs[4], L[4], dt32, w32, ok4);
    if (!(ok01 && ok23 && ok4)) {
#pragma unroll
        for (int u = 0; u < 5; u++)
            if (!(u < 2 ? ok01 : u < 4 ? ok23 : ok4)) h[u] = rk_fp64<T>(qn[u], qs[u], L[u], dt, w);
    }
}

// Stage combination of the five conserved values of one cell, stored at
// offset c of each output field; returns the stored values in type C.
__device__ __forceinline__ void rk_store5(const Fout<5> &out, idx c, const C qn[5], const C qs[5],
                                          const C L[5], C dt32, double dt, C w32, double w, C o[5])
{
    if constexpr (kNarrow) {
        S h[5];
        rk_narrow5<S>(qn, qs, L, dt32, dt, w32, w, h);
#pragma unroll
        for (int u = 0; u < 5; u++) {
            out.p[u][c] = h[u];
            o[u] = cv(h[u]);
        }
    } else {
#pragma unroll
        for (int u = 0; u < 5; u++) o[u] = stc(out.p[u] + c, qn[u] + w32 * ((qs[u] - qn[u]) + dt32 * L[u]));
    }
}

// Block coordinates of a stage kernel's body: those of the launch itself, or,
// in a grouped launch over several instances, the block's place in its own
// instance's grid.
struct BlockPos {
    int x, y, z, gx, gy;
    static __device__ __forceinline__ BlockPos of_launch()
    {
        return {(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, (int)gridDim.x, (int)gridDim.y};
    }
    // the l-th block of a grid of gx x gy x * blocks
    static __device__ __forceinline__ BlockPos of_index(int l, int gx, int gy)
    {
        return {l % gx, (l / gx) % gy, l / (gx * gy), gx, gy};
    }
};

// --------------------------------------------- tiles of the 7-point kernels
// Two forms of the source and of the sweeps, marching up a z-chunk:
//   quads  a thread has four consecutive cells of a row, one 4-wide load or
//          store per field (rows of a multiple of 4 cells, fields aligned to
//          4 values). A block owns wq quads x rows rows of the plane; quad_fit
//          (igr_internal.h) fits the tile to the grid, so short rows (48..96
//          cells) leave no lanes idle; grids that the largest tile (32 quads
//          x 8 rows) divides take it with its shape compiled in (FULL).
//   pairs  a thread has two cells, one above the other in y, loaded element by
//          element: any row length and alignment, coalesced, and the same
//          packed arithmetic. A block owns 32 x 16 cells of the plane.
// Both evaluate one sequence of rounded operations per cell: the same bits.
constexpr int VX = 4;
constexpr int FQ = 32, FR = 8, BT = FQ * FR;   // full tile: quads, rows, threads
constexpr int HXV = VX * FQ + 2 * VX;          // its row pitch (interior at column VX, 16-byte aligned)
constexpr int TILEV = QUAD_TILE;               // cells of one plane tile with its halo, any shape
static_assert((FR + 2) * HXV <= TILEV, "full tile");

// z-index of plane kk in [-1, nz]: periodic wrap or zero-gradient clamp
__device__ __forceinline__ int zmap(int kk, const Geom &g)
{
    return kk < 0 ? (g.bc[4] == BC_PERIODIC ? kk + g.nz : 0)
                  : (kk >= g.nz ? (g.bc[5] == BC_PERIODIC ? kk - g.nz : g.nz - 1) : kk);
}

// A thread's place in its tile. Threads 0..wq-1 also load the halo row below
// the tile, the next wq the row above (4-wide, under their own quad), and the
// next 2 rows threads the cells left and right of the rows. Everything is
// mapped once; lanes outside the grid load nothing.
struct Quad {
    int i0, j;            // first cell
    bool active;          // inside the grid
    int pitch, pos;       // row pitch of the plane tile, position of the first cell in it
    idx own;              // in-plane offset of the first cell
    bool yh, xh;          // halo tasks: a quad above or below, a cell left or right
    int hpos;             // position in the plane tile
    idx hoff;             // in-plane offset
    bool hdrop;           // the halo lies across a non-periodic boundary
};
template <bool FULL, int NR>
__device__ __forceinline__ Quad quad_of(const Geom &g, const BlockPos &bp, int wq, int rows)
{
    Quad t;
    if (FULL) {
        wq = FQ;
        rows = FR;
    }
    const int tid = threadIdx.x, row = tid / wq, qd = tid - row * wq, H = NR * rows;
    const int x0 = bp.x * VX * wq, y0 = bp.y * H;
    t.i0 = x0 + VX * qd;
    t.j = y0 + NR * row;
    t.active = FULL || (row < rows && t.i0 < g.nx && t.j < g.ny);
    t.pitch = VX * wq + 2 * VX;
    t.pos = (NR * row + 1) * t.pitch + VX + VX * qd;
    t.own = (idx)t.j * (idx)g.nx + (idx)t.i0;
    const int ye = FULL ? y0 + H : min(y0 + H, g.ny), xe = FULL ? x0 + VX * wq : min(x0 + VX * wq, g.nx);
    t.yh = row < 2 && (FULL || t.i0 < g.nx);
    t.xh = false;
    if (row < 2) {
        const int y = row ? ye : y0 - 1;
        t.hpos = (y - y0 + 1) * t.pitch + VX + VX * qd;
        t.hoff = (idx)map_axis(y, g.ny, g.bc[2], g.bc[3]) * (idx)g.nx + (idx)t.i0;
        t.hdrop = row ? y >= g.ny && g.bc[3] != BC_PERIODIC : y < 0 && g.bc[2] != BC_PERIODIC;
    } else {
        const int e = tid - 2 * wq, side = e / H, r = e - side * H;
        const int x = side ? xe : x0 - 1;
        t.xh = side < 2 && (FULL || y0 + r < g.ny);
        t.hpos = (r + 1) * t.pitch + VX + (x - x0);
        t.hoff = (idx)(y0 + r) * (idx)g.nx + (idx)map_axis(x, g.nx, g.bc[0], g.bc[1]);
        t.hdrop = side ? x >= g.nx && g.bc[1] != BC_PERIODIC : x < 0 && g.bc[0] != BC_PERIODIC;
    }
    return t;
}

// The pairs: lane tx, warp ty have cells (x0 + tx, y0 + 2 ty) and the one
// above; threads 0..95 each load one halo cell (32 below, 32 above, 16 left,
// 16 right). The tile's cells outside the grid hold the mapped cell next to
// it (the far halo of a tile that the grid's edge cuts).
constexpr int PX = 32, PWARPS = 8, PY = 2 * PWARPS, PPITCH = PX + 2, TILEP = (PY + 2) * PPITCH;
struct Pair {
    int i, j;             // lower cell
    bool in[2];           // the cells inside the grid
    bool need[2];         // the cells that are read (inside, or the first ones past the edge)
    bool drop[2];         // ... those across a non-periodic boundary
    int pos;              // position of the lower cell in the plane tile
    idx own[2];           // in-plane offsets, mapped
    bool h;               // a halo task
    int hpos;
    idx hoff;
    bool hdrop;
};
__device__ __forceinline__ Pair pair_of(const Geom &g, const BlockPos &bp)
{
    Pair t;
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int x0 = bp.x * PX, y0 = bp.y * PY;
    t.i = x0 + tx;
    t.j = y0 + 2 * ty;
    t.pos = (2 * ty + 1) * PPITCH + tx + 1;
    const idx mi = (idx)map_axis(t.i, g.nx, g.bc[0], g.bc[1]);
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const int j = t.j + c;
        t.in[c] = t.i < g.nx && j < g.ny;
        t.need[c] = t.i <= g.nx && j <= g.ny;
        t.drop[c] = (t.i >= g.nx && g.bc[1] != BC_PERIODIC) || (j >= g.ny && g.bc[3] != BC_PERIODIC);
        t.own[c] = (idx)map_axis(j, g.ny, g.bc[2], g.bc[3]) * (idx)g.nx + mi;
    }
    int lx, ly;  // halo cell in the tile
    if (tid < 2 * PX) {
        lx = 1 + tx;
        ly = ty ? PY + 1 : 0;
    } else {
        lx = tid - 2 * PX < PY ? 0 : PX + 1;
        ly = 1 + (tid & (PY - 1));
    }
    const int x = x0 + lx - 1, y = y0 + ly - 1;
    t.h = tid < 2 * PX + 2 * PY && x <= g.nx && y <= g.ny;
    t.hpos = ly * PPITCH + lx;
    t.hoff = (idx)map_axis(y, g.ny, g.bc[2], g.bc[3]) * (idx)g.nx + (idx)map_axis(x, g.nx, g.bc[0], g.bc[1]);
    t.hdrop = (x < 0 && g.bc[0] != BC_PERIODIC) || (x >= g.nx && g.bc[1] != BC_PERIODIC) ||
              (y < 0 && g.bc[2] != BC_PERIODIC) || (y >= g.ny && g.bc[3] != BC_PERIODIC);
    return t;
}

// ------------------------------------------- 4-wide loads, stores, shared rows
__device__ __forceinline__ void st4(double *p, const double v[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void st4(float *p, const float v[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(__half *p, const float v[4])
{
    __half2 a = __floats2half2_rn(v[0], v[1]), b = __floats2half2_rn(v[2], v[3]);
    uint2 u;
    u.x = *reinterpret_cast<unsigned *>(&a);
    u.y = *reinterpret_cast<unsigned *>(&b);
    *reinterpret_cast<uint2 *>(p) = u;
}
__device__ __forceinline__ void st4(__nv_bfloat16 *p, const float v[4])
{
    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    uint2 u;
    u.x = *reinterpret_cast<unsigned *>(&a);
    u.y = *reinterpret_cast<unsigned *>(&b);
    *reinterpret_cast<uint2 *>(p) = u;
}

// Four consecutive values as loaded: they stay raw until they are used, so
// that nothing waits on the load before then
template <typename T> struct Vec4;
template <> struct Vec4<double> { double2 a, b; };
template <> struct Vec4<float> { float4 a; };
template <> struct Vec4<__half> { uint2 a; };
template <> struct Vec4<__nv_bfloat16> { uint2 a; };
using V4 = Vec4<S>;

__device__ __forceinline__ Vec4<double> ld4r(const double *p)
{
    return {*reinterpret_cast<const double2 *>(p), reinterpret_cast<const double2 *>(p)[1]};
}
__device__ __forceinline__ Vec4<float> ld4r(const float *p) { return {*reinterpret_cast<const float4 *>(p)}; }
__device__ __forceinline__ Vec4<__half> ld4r(const __half *p) { return {*reinterpret_cast<const uint2 *>(p)}; }
__device__ __forceinline__ Vec4<__nv_bfloat16> ld4r(const __nv_bfloat16 *p)
{
    return {*reinterpret_cast<const uint2 *>(p)};
}
__device__ __forceinline__ void cv4(const Vec4<double> &v, double o[4])
{
    o[0] = v.a.x; o[1] = v.a.y; o[2] = v.b.x; o[3] = v.b.y;
}
__device__ __forceinline__ void cv4(const Vec4<float> &v, float o[4])
{
    o[0] = v.a.x; o[1] = v.a.y; o[2] = v.a.z; o[3] = v.a.w;
}
union H2U { unsigned u; __half2 h; };
union B2U { unsigned u; __nv_bfloat162 h; };
__device__ __forceinline__ void cv4(const Vec4<__half> &v, float o[4])
{
    H2U lo, hi;
    lo.u = v.a.x;
    hi.u = v.a.y;
    float2 a = __half22float2(lo.h), b = __half22float2(hi.h);
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void cv4(const Vec4<__nv_bfloat16> &v, float o[4])
{
    B2U lo, hi;
    lo.u = v.a.x;
    hi.u = v.a.y;
    float2 a = __bfloat1622float2(lo.h), b = __bfloat1622float2(hi.h);
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
// 4 consecutive values of a 16-byte aligned shared row (one 128-bit access
// for FP32, two for FP64; scalar accesses at stride 4 would conflict 4-way)
__device__ __forceinline__ void sh_st4(float *p, const float v[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void sh_st4(double *p, const double v[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void sh_ld4(const float *p, float v[4])
{
    float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void sh_ld4(const double *p, double v[4])
{
    double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// Asynchronous copies global -> shared of a quad and of a single value (at 16
// bits the aligned pair that holds it), and reading them back
__device__ __forceinline__ unsigned sh_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_quad(unsigned dst, const S *src)
{
    if constexpr (sizeof(S) == 2) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
    } else {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
        if constexpr (sizeof(S) == 8)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16), "l"(src + 2) : "memory");
    }
}
__device__ __forceinline__ void cp_one(unsigned dst, const S *src)
{
    if constexpr (sizeof(S) == 2)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"((size_t)src & ~(size_t)3) : "memory");
    else if constexpr (sizeof(S) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}

// --------------------------------------------------------------- Jacobi
// One sweep s_out = (b + beta sum_f c_f s_nb) / (1/rho + beta sum_f c_f),
// c_f = (1/rho_i + 1/rho_nb)/2; a face on a non-periodic boundary carries no
// term. 1/rho and sigma of plane k sit in a shared tile with a halo of 1;
// the z-neighbours stay in registers.
//
// The face factors c_f = hb (1/rho_i + 1/rho_nb), hb = beta / 2, take one
// constant: across a dropped face the neighbour's 1/rho is taken as -1/rho_i
// and its Sigma as 0, so that c_f is exactly 0. The z-face below a cell is the
// face above the cell of the last plane, kept from there.
//
// colour >= 0 makes it one half of a red-black Gauss-Seidel sweep, in place
// (s_in == s_out): only the cells with (i + j + k) % 2 == colour change.
// Their neighbours all have the other colour (periodic axes have even
// length), which no thread writes during the launch, so every updated value
// is the same whatever the order of execution; values read from cells of
// the updated colour feed only results that are discarded.

// The update of two cells: rc their 1/rho, bv their source; r*, s* the
// neighbours' 1/rho and Sigma in x and y; zm, zp the factors of the z-faces
// below and above, sm, sp Sigma there. Packed FP32x2 operations (FP64: two scalar ones).
__device__ __forceinline__ float2 pquot(float2 a, float2 b) { return pmul(a, make_float2(rcp(b.x), rcp(b.y))); }
__device__ __forceinline__ double2 pquot(double2 a, double2 b)
{
    return make_double2(__ddiv_rn(a.x, b.x), __ddiv_rn(a.y, b.y));
}
__device__ __forceinline__ C2 jacobi2(C2 rc, C2 rxm, C2 rxp, C2 rym, C2 ryp, C2 zm, C2 zp, C2 sxm, C2 sxp, C2 sym,
                                      C2 syp, C2 sm, C2 sp, C2 bv, C hb)
{
    const C2 h = bcast(hb);
    const C2 c0 = pmul(h, padd(rc, rxm)), c1 = pmul(h, padd(rc, rxp));
    const C2 c2 = pmul(h, padd(rc, rym)), c3 = pmul(h, padd(rc, ryp));
    const C2 diag = padd(padd(padd(padd(padd(padd(rc, c0), c1), c2), c3), zm), zp);
    C2 off = pmul(c0, sxm);
    off = pfma(c1, sxp, off);
    off = pfma(c2, sym, off);
    off = pfma(c3, syp, off);
    off = pfma(zm, sm, off);
    off = pfma(zp, sp, off);
    return pquot(padd(bv, off), diag);
}

// Raw values are copied to shared memory JRING - 1 planes ahead, each by the
// thread that uses it (so no barrier guards them): a plane's time is then not
// the latency of its loads. Register prefetch does not get there: loads of
// several planes in flight share a warp's six scoreboards, and a wait for
// the oldest waits for the youngest too. What bounds the 16-bit sweep next is
// instructions and shared-memory bandwidth: Sigma is exchanged in its storage
// type, the x-neighbours within a warp's row by shuffles, and on large grids
// a thread has two quads, one above the other (NR = 2): addresses, loop and
// barrier serve both, and they exchange in registers.
constexpr int JRING = sizeof(S) == 8 ? 2 : 4;
template <int NR> struct JShape {
    static constexpr int TILE = NR * QUAD_TILE;                      // cells of a plane tile with its halo
    static constexpr int HT = 96;                                    // threads that may have a halo task
    static constexpr int PLANE = VX * (3 * NR * BT + 2 * HT);        // values of one plane of the ring
    static constexpr int SMEM = JRING * PLANE * (int)sizeof(S) + 2 * TILE * (int)(sizeof(C) + sizeof(S));
};
template <bool FULL, bool RB, int NR>
__device__ __forceinline__ void jacobi_quads(const S *q, const S *b, const S *sin, S *sout, const Geom &g, C beta,
                                             int zc, int colour, const BlockPos &bp, int wq, int rows,
                                             unsigned char *smem)
{
    static_assert(FULL || NR == 1, "two rows per thread: full tiles");
    constexpr int JPLANE = JShape<NR>::PLANE, JTILE = JShape<NR>::TILE, HT = JShape<NR>::HT;
    S *ring = reinterpret_cast<S *>(smem);
    C *R2 = reinterpret_cast<C *>(ring + JRING * JPLANE);
    S *S2 = reinterpret_cast<S *>(R2 + 2 * JTILE);
    const Quad t = quad_of<FULL, NR>(g, bp, wq, rows);
    const int tid = threadIdx.x;
    const int k0 = bp.z * zc, k1 = min(g.nz, k0 + zc);
    const idx pl = (idx)g.plane;
    const C hb = C(0.5) * beta;
    idx own[NR];
#pragma unroll
    for (int r = 0; r < NR; r++) own[r] = t.own + (idx)r * (idx)g.nx;
    S *const mine = ring + VX * tid, *const minh = ring + VX * (3 * NR * BT + (tid < HT ? tid : 0));
    constexpr int F = VX * BT, FH = VX * HT;
    // start the copies of own density and Sigma of plane kk + 1, source and halo of plane kk
    auto load = [&](int kk) {
        const int at = ((kk - k0) & (JRING - 1)) * JPLANE;
        const unsigned d = sh_addr(mine + at), dh = sh_addr(minh + at);
        const idx pk = (idx)kk * pl, h = pk + t.hoff;
        if (FULL || t.active) {
            const idx pz = (idx)zmap(kk + 1, g) * pl;
#pragma unroll
            for (int r = 0; r < NR; r++) {
                cp_quad(d + (3 * r) * F * sizeof(S), CKP4(q + pz + own[r], q, g.n));
                cp_quad(d + (3 * r + 1) * F * sizeof(S), CKP4(sin + pz + own[r], sin, g.n));
                cp_quad(d + (3 * r + 2) * F * sizeof(S), CKP4(b + pk + own[r], b, g.n));
            }
        }
        if (t.yh) {
            cp_quad(dh, CKP4(q + h, q, g.n));
            cp_quad(dh + FH * sizeof(S), CKP4(sin + h, sin, g.n));
        } else if (t.xh) {
            cp_one(dh, CKP(q + h, q, g.n));
            cp_one(dh + FH * sizeof(S), CKP(sin + h, sin, g.n));
        }
    };
    auto conv = [&](const V4 &v, C (&r)[VX]) {
        cv4(v, r);
#pragma unroll
        for (int c = 0; c < VX; c++) r[c] = rcp(r[c]);
    };
    C sm[NR][VX], r0[NR][VX], s0[NR][VX];
    V4 s0r[NR];  // s0 as stored
    C2 zm[NR][2];
#pragma unroll
    for (int m = 0; m < JRING - 1; m++) {
        if (k0 + m < k1) load(k0 + m);
        cp_async_commit();
    }
    if (FULL || t.active) {
        const idx zb = (idx)zmap(k0 - 1, g) * pl, z0 = (idx)k0 * pl;
#pragma unroll
        for (int r = 0; r < NR; r++) {
            const V4 ar = ld4r(CKP4(q + zb + own[r], q, g.n));
            const V4 as = ld4r(CKP4(sin + zb + own[r], sin, g.n));
            const V4 or_ = ld4r(CKP4(q + z0 + own[r], q, g.n));
            s0r[r] = ld4r(CKP4(sin + z0 + own[r], sin, g.n));
            C rm[VX];
            conv(ar, rm);
            cv4(as, sm[r]);
            conv(or_, r0[r]);
            cv4(s0r[r], s0[r]);
#pragma unroll
            for (int h = 0; h < 2; h++)
                zm[r][h] = pmul(bcast(hb), padd(pset(r0[r][2 * h], r0[r][2 * h + 1]), pset(rm[2 * h], rm[2 * h + 1])));
            if (k0 == 0 && g.bc[4] != BC_PERIODIC) {
#pragma unroll
                for (int c = 0; c < VX; c++) sm[r][c] = C(0);
                zm[r][0] = zm[r][1] = bcast(C(0));
            }
        }
    }
    const int hodd = sizeof(S) == 2 ? (int)(t.hoff & 1) : 0;  // the halo cell in its pair (nx is even)
    for (int k = k0; k < k1; k++) {
        // two plane tiles, alternating: the buffer a plane writes was last
        // read two planes ago, before the barrier of the previous plane
        C *R = R2 + ((k - k0) & 1) * JTILE;
        S *SG = S2 + ((k - k0) & 1) * JTILE;
        const int at = ((k - k0) & (JRING - 1)) * JPLANE;
        C rp[NR][VX], sp[NR][VX], bv[NR][VX];
        V4 spr[NR];
        if (FULL || t.active) {
#pragma unroll
            for (int r = 0; r < NR; r++) {
                sh_st4(R + t.pos + r * t.pitch, r0[r]);
                *reinterpret_cast<V4 *>(SG + t.pos + r * t.pitch) = s0r[r];
            }
        }
        cp_async_wait<JRING - 2>();
        if (t.yh) {
            C w[VX];
            conv(*reinterpret_cast<const V4 *>(minh + at), w);
            if (t.hdrop) {
#pragma unroll
                for (int c = 0; c < VX; c++) w[c] = -w[c];
            }
            sh_st4(R + cks4(t.hpos, JTILE), w);
            V4 hs = *reinterpret_cast<const V4 *>(minh + at + FH);
            if (t.hdrop) hs = V4{};
            *reinterpret_cast<V4 *>(SG + cks4(t.hpos, JTILE)) = hs;
        } else if (t.xh) {
            const C w = rcp(C(cv(minh[at + hodd])));
            R[cks(t.hpos, JTILE)] = t.hdrop ? -w : w;
            SG[cks(t.hpos, JTILE)] = t.hdrop ? S(0.0f) : minh[at + FH + hodd];
        }
        if (FULL || t.active) {
#pragma unroll
            for (int r = 0; r < NR; r++) {
                conv(*reinterpret_cast<const V4 *>(mine + at + (3 * r) * F), rp[r]);
                spr[r] = *reinterpret_cast<const V4 *>(mine + at + (3 * r + 1) * F);
                cv4(spr[r], sp[r]);
                cv4(*reinterpret_cast<const V4 *>(mine + at + (3 * r + 2) * F), bv[r]);
            }
        }
        if (k + JRING - 1 < k1) load(k + JRING - 1);
        cp_async_commit();
        __syncthreads();
        if (FULL || t.active) {
            if (k == g.nz - 1 && g.bc[5] != BC_PERIODIC) {  // no face above the last plane
#pragma unroll
                for (int r = 0; r < NR; r++)
#pragma unroll
                    for (int c = 0; c < VX; c++) {
                        rp[r][c] = -r0[r][c];
                        sp[r][c] = C(0);
                    }
            }
            C rb[VX], ra[VX], sb[VX], sa[VX];  // rows below and above
            sh_ld4(R + t.pos - t.pitch, rb);
            sh_ld4(R + t.pos + NR * t.pitch, ra);
            cv4(*reinterpret_cast<const V4 *>(SG + t.pos - t.pitch), sb);
            cv4(*reinterpret_cast<const V4 *>(SG + t.pos + NR * t.pitch), sa);
#pragma unroll
            for (int r = 0; r < NR; r++) {
                const C (&ry0)[VX] = r ? r0[0] : rb, (&sy0)[VX] = r ? s0[0] : sb;
                const C (&ry1)[VX] = r + 1 < NR ? r0[NR - 1] : ra, (&sy1)[VX] = r + 1 < NR ? s0[NR - 1] : sa;
                const int pos = t.pos + r * t.pitch;
                C rl, rr, sl, sr;  // x-neighbours of the quad
                if (FULL) {        // a warp is a row: only its ends read the tile
                    const int lane = tid & 31;
                    rl = __shfl_up_sync(0xffffffffu, r0[r][3], 1);
                    sl = __shfl_up_sync(0xffffffffu, s0[r][3], 1);
                    rr = __shfl_down_sync(0xffffffffu, r0[r][0], 1);
                    sr = __shfl_down_sync(0xffffffffu, s0[r][0], 1);
                    if (lane == 0 || lane == 31) {
                        const int e = lane ? pos + VX : pos - 1;
                        const C re = R[e], se = C(cv(SG[e]));
                        if (lane) {
                            rr = re;
                            sr = se;
                        } else {
                            rl = re;
                            sl = se;
                        }
                    }
                } else {
                    rl = R[pos - 1];
                    rr = R[pos + VX];
                    sl = C(cv(SG[pos - 1]));
                    sr = C(cv(SG[pos + VX]));
                }
                const C rx[VX + 2] = {rl, r0[r][0], r0[r][1], r0[r][2], r0[r][3], rr};
                const C sx[VX + 2] = {sl, s0[r][0], s0[r][1], s0[r][2], s0[r][3], sr};
                C o[VX];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int c = 2 * h;
                    const C2 rc = pset(r0[r][c], r0[r][c + 1]);
                    const C2 zp = pmul(bcast(hb), padd(rc, pset(rp[r][c], rp[r][c + 1])));
                    const C2 v = jacobi2(rc, pset(rx[c], rx[c + 1]), pset(rx[c + 2], rx[c + 3]),
                                         pset(ry0[c], ry0[c + 1]), pset(ry1[c], ry1[c + 1]), zm[r][h], zp,
                                         pset(sx[c], sx[c + 1]), pset(sx[c + 2], sx[c + 3]),
                                         pset(sy0[c], sy0[c + 1]), pset(sy1[c], sy1[c + 1]),
                                         pset(sm[r][c], sm[r][c + 1]), pset(sp[r][c], sp[r][c + 1]),
                                         pset(bv[r][c], bv[r][c + 1]), hb);
                    o[c] = v.x;
                    o[c + 1] = v.y;
                    zm[r][h] = zp;
                }
                if (RB || (!FULL && colour >= 0)) {
#pragma unroll
                    for (int c = 0; c < VX; c++)
                        if (((t.i0 + c + t.j + r + k) & 1) != colour) o[c] = s0[r][c];
                }
                st4(CKP4(sout + (idx)k * pl + own[r], sout, g.n), o);
            }
#pragma unroll
            for (int r = 0; r < NR; r++) {
#pragma unroll
                for (int c = 0; c < VX; c++) {
                    sm[r][c] = s0[r][c];
                    r0[r][c] = rp[r][c];
                    s0[r][c] = sp[r][c];
                }
                s0r[r] = spr[r];
            }
        }
    }
}

// the pairs: one halo cell per thread of the first three warps, own values
// one plane ahead
__device__ __forceinline__ void jacobi_pairs(const S *q, const S *b, const S *sin, S *sout,
                                             const Geom &g, C beta, int zc, int colour, const BlockPos &bp, C *R2,
                                             C *S2)
{
    const Pair t = pair_of(g, bp);
    const int k0 = bp.z * zc, k1 = min(g.nz, k0 + zc);
    const idx pl = (idx)g.plane;
    const C hb = C(0.5) * beta;
    S nr[2] = {S(1.0f), S(1.0f)}, ns[2] = {S(0.0f), S(0.0f)}, nb[2] = {S(0.0f), S(0.0f)};
    S xr = S(1.0f), xs = S(0.0f);
    auto own = [&](int kk) {  // own cells of plane kk
        const idx pz = (idx)zmap(kk, g) * pl;
#pragma unroll
        for (int c = 0; c < 2; c++)
            if (t.need[c]) {
                nr[c] = ldr(CKP(q + pz + t.own[c], q, g.n));
                ns[c] = ldr(CKP(sin + pz + t.own[c], sin, g.n));
            }
    };
    auto rest = [&](int kk) {  // source and halo of plane kk
        const idx pk = (idx)kk * pl;
#pragma unroll
        for (int c = 0; c < 2; c++)
            if (t.in[c]) nb[c] = ldr(CKP(b + pk + t.own[c], b, g.n));
        if (t.h) {
            xr = ldr(CKP(q + pk + t.hoff, q, g.n));
            xs = ldr(CKP(sin + pk + t.hoff, sin, g.n));
        }
    };
    // a cell past a non-periodic edge stands for the dropped face's neighbour
    auto conv = [&](C2 &r, C2 &s) {
        const C a = rcp(C(cv(nr[0]))), e = rcp(C(cv(nr[1])));
        r = pset(t.drop[0] ? -a : a, t.drop[1] ? -e : e);
        s = pset(t.drop[0] ? C(0) : C(cv(ns[0])), t.drop[1] ? C(0) : C(cv(ns[1])));
    };
    C2 rm, sm, r0, s0, zm;
    own(k0 - 1);
    conv(rm, sm);
    own(k0);
    conv(r0, s0);
    own(k0 + 1);
    rest(k0);
    zm = pmul(bcast(hb), padd(r0, rm));
    if (k0 == 0 && g.bc[4] != BC_PERIODIC) zm = sm = bcast(C(0));
    for (int k = k0; k < k1; k++) {
        C *R = R2 + ((k - k0) & 1) * TILEP, *SG = S2 + ((k - k0) & 1) * TILEP;
        C2 rp, sp;
        R[t.pos] = r0.x;
        R[t.pos + PPITCH] = r0.y;
        SG[t.pos] = s0.x;
        SG[t.pos + PPITCH] = s0.y;
        if (t.h) {
            const C w = rcp(C(cv(xr)));
            R[cks(t.hpos, TILEP)] = t.hdrop ? -w : w;
            SG[cks(t.hpos, TILEP)] = t.hdrop ? C(0) : C(cv(xs));
        }
        conv(rp, sp);
        const C2 bv = pset(C(cv(nb[0])), C(cv(nb[1])));
        if (k + 1 < k1) {
            own(k + 2);
            rest(k + 1);
        }
        __syncthreads();
        if (k == g.nz - 1 && g.bc[5] != BC_PERIODIC) {  // no face above the last plane
            rp = pset(-r0.x, -r0.y);
            sp = bcast(C(0));
        }
        const C2 zp = pmul(bcast(hb), padd(r0, rp));
        const C *Rc = R + t.pos, *Sc = SG + t.pos;
        const C2 v = jacobi2(r0, pset(Rc[-1], Rc[PPITCH - 1]), pset(Rc[1], Rc[PPITCH + 1]),
                             pset(Rc[-PPITCH], r0.x), pset(r0.y, Rc[2 * PPITCH]), zm, zp,
                             pset(Sc[-1], Sc[PPITCH - 1]), pset(Sc[1], Sc[PPITCH + 1]),
                             pset(Sc[-PPITCH], s0.x), pset(s0.y, Sc[2 * PPITCH]), sm, sp, bv, hb);
        const int odd = (t.i + t.j + k) & 1;
        S *o = sout + (idx)k * pl;
        if (t.in[0] && (colour < 0 || odd == colour)) stc(CKP(o + t.own[0], sout, g.n), v.x);
        if (t.in[1] && (colour < 0 || odd != colour)) stc(CKP(o + t.own[1], sout, g.n), v.y);
        zm = zp;
        sm = s0;
        r0 = rp;
        s0 = sp;
    }
}
// resident blocks per SM that the registers are held to
template <int NR> constexpr int kJacobiBlocks = sizeof(S) == 8 ? 1 : sizeof(S) == 2 && NR == 1 ? 3 : 2;
constexpr int JACOBI_FIT_BLOCKS = sizeof(C) == 8 ? 1 : 2;
// four blocks of pairs (1022 x 255 x 255 FP32: 265 us; five: 252, six: 342; but
// 254 x 201 x 130: 34.7, 36.9 and 45.1)
constexpr int JACOBI_PAIR_BLOCKS = sizeof(C) == 8 ? 2 : 4;
template <bool RB, int NR>
__global__ void __launch_bounds__(BT, kJacobiBlocks<NR>) k_jacobi_full(const S *q, const S *b,
                                                                  const S *sin, S *sout, Geom g, C beta, int zc,
                                                                  int colour)
{
    launched();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    jacobi_quads<true, RB, NR>(q, b, sin, sout, g, beta, zc, colour, BlockPos::of_launch(), FQ, FR, smem_raw);
}
__global__ void __launch_bounds__(BT, JACOBI_FIT_BLOCKS) k_jacobi_fit(const S *q, const S *b,
                                                                     const S *sin, S *sout, Geom g, C beta, int zc,
                                                                     int colour, int wq, int rows)
{
    launched();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    jacobi_quads<false, false, 1>(q, b, sin, sout, g, beta, zc, colour, BlockPos::of_launch(), wq, rows, smem_raw);
}
__global__ void __launch_bounds__(BT, JACOBI_PAIR_BLOCKS) k_jacobi_pairs(const S *q,
                                                                        const S *b, const S *sin,
                                                                        S *sout, Geom g, C beta, int zc, int colour)
{
    launched();
    __shared__ C R[2 * TILEP];
    __shared__ C SG[2 * TILEP];
    jacobi_pairs(q, b, sin, sout, g, beta, zc, colour, BlockPos::of_launch(), R, SG);
}

// FP64 sweeps from stored coefficients. An FP64 instruction holds an SM's units
// for 16 cycles here, so the sweeps above are bound by the 40 or so that a cell
// takes (two divisions, 14 for the faces, 6 for the diagonal). None of these
// depend on Sigma, so where 5 n scratch values are free (a context's RK buffers)
// they are formed once per stage: the three low-face factors, the diagonal d and
// its inverse. That leaves 10: the sum and num / d (quot), so the results are those
// of the sweeps above. All else is free beside the FP64 units (64 bytes per cell
// from memory take half their time): one thread per cell, neighbours from L1, no
// alignment and no tile shape.
//
// num / d rounded to nearest from inv = 1 / d: v = num inv and one remainder step
// (Markstein, IBM J. R&D 34, 1990). The remainder is exact and inv normal where
// both num and v lie in [2^-500, 2^500) (tested on the exponents, by integer
// instructions); zero is 0 inv, and the rest (far smaller or larger, infinities,
// NaN) divides.
__device__ __forceinline__ bool mid_range(double x)
{
    return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 523u < 1000u;
}
__device__ __forceinline__ double quot(double num, double d, double inv)
{
    const double v = __dmul_rn(num, inv);
    if (mid_range(num) && mid_range(v)) return __fma_rn(__fma_rn(-d, v, num), inv, v);
    return num == 0.0 && mid_range(inv) ? v : __ddiv_rn(num, d);
}
template <class T> struct Coefs {
    T *cx, *cy, *cz, *d, *inv;
};
// a cell, its neighbours (wrapped) and whether the faces to them exist
struct Stencil {
    idx c, xl, xh, yl, yh, zl, zh;
    bool hxl, hxh, hyl, hyh, hzl, hzh;
};
__device__ __forceinline__ Stencil stencil_of(int i, int j, int k, const Geom &g)
{
    const bool px = g.bc[0] == BC_PERIODIC, py = g.bc[2] == BC_PERIODIC, pz = g.bc[4] == BC_PERIODIC;
    const idx nx = (idx)g.nx, pl = (idx)g.plane;
    Stencil t;
    t.c = (idx)k * pl + (idx)j * nx + (idx)i;
    t.xl = i > 0 ? t.c - 1 : t.c + (nx - 1);
    t.xh = i + 1 < g.nx ? t.c + 1 : t.c - (nx - 1);
    t.yl = j > 0 ? t.c - nx : t.c + (pl - nx);
    t.yh = j + 1 < g.ny ? t.c + nx : t.c - (pl - nx);
    t.zl = k > 0 ? t.c - pl : t.c + (idx)(g.nz - 1) * pl;
    t.zh = k + 1 < g.nz ? t.c + pl : t.c - (idx)(g.nz - 1) * pl;
    t.hxl = px || i > 0;
    t.hxh = px || i + 1 < g.nx;
    t.hyl = py || j > 0;
    t.hyh = py || j + 1 < g.ny;
    t.hzl = pz || k > 0;
    t.hzh = pz || k + 1 < g.nz;
    return t;
}
// fn(i, j, k) over the cells (colour >= 0: those of that colour), one per
// thread and plane: blocks of 256 along a plane (x), planes over y
template <class F> __device__ __forceinline__ void for_cells(const Geom &g, int colour, F fn)
{
    const unsigned w = colour < 0 ? g.nx : (g.nx + 1) / 2, p = blockIdx.x * 256u + threadIdx.x;
    const int j = (int)(p / w), h = (int)(p % w);
    if (j >= g.ny) return;
    for (int k = blockIdx.y; k < g.nz; k += gridDim.y) {
        const int i = colour < 0 ? h : 2 * h + ((colour + j + k) & 1);
        if (i < g.nx) fn(i, j, k);
    }
}
template <class T> __global__ void __launch_bounds__(256) k_coef_rcp(const T *q, T *r, Geom g)
{
    launched();
    for_cells(g, -1, [&](int i, int j, int k) {
        const idx c = ck((idx)k * (idx)g.plane + (idx)j * (idx)g.nx + (idx)i, g.n);
        r[c] = rcp(q[c]);
    });
}
// 1 / rho is in a.d
template <class T> __global__ void __launch_bounds__(256) k_coef_faces(Coefs<T> a, Geom g, T hb)
{
    launched();
    for_cells(g, -1, [&](int i, int j, int k) {
        const Stencil t = stencil_of(i, j, k, g);
        const idx c = ck(t.c, g.n);
        const T r = a.d[c];
        a.cx[c] = t.hxl ? mul_rn(hb, add_rn(r, a.d[ck(t.xl, g.n)])) : T(0);
        a.cy[c] = t.hyl ? mul_rn(hb, add_rn(r, a.d[ck(t.yl, g.n)])) : T(0);
        a.cz[c] = t.hzl ? mul_rn(hb, add_rn(r, a.d[ck(t.zl, g.n)])) : T(0);
    });
}
// the diagonal in place of 1 / rho, and its inverse (an outer face has the factor 0)
template <class T> __global__ void __launch_bounds__(256) k_coef_diag(Coefs<T> a, Geom g)
{
    launched();
    for_cells(g, -1, [&](int i, int j, int k) {
        const Stencil t = stencil_of(i, j, k, g);
        const idx c = ck(t.c, g.n);
        T d = add_rn(add_rn(a.d[c], a.cx[c]), a.cx[ck(t.xh, g.n)]);
        d = add_rn(add_rn(d, a.cy[c]), a.cy[ck(t.yh, g.n)]);
        d = add_rn(add_rn(d, a.cz[c]), a.cz[ck(t.zh, g.n)]);
        a.d[c] = d;
        a.inv[c] = rcp(d);
    });
}
// (RB: s_in == s_out; a launch reads the cells of the other colour)
template <class T>
__global__ void __launch_bounds__(256) k_sweep(Coefs<const T> a, const T *b, const T *sin, T *sout, Geom g,
                                              int colour)
{
    launched();
    for_cells(g, colour, [&](int i, int j, int k) {
        const Stencil t = stencil_of(i, j, k, g);
        const idx c = ck(t.c, g.n), xh = ck(t.xh, g.n), yh = ck(t.yh, g.n), zh = ck(t.zh, g.n);
        auto s = [&](bool face, idx at) { return face ? sin[ck(at, g.n)] : T(0); };
        T off = mul_rn(a.cx[c], s(t.hxl, t.xl));
        off = fma_rn(a.cx[xh], s(t.hxh, t.xh), off);
        off = fma_rn(a.cy[c], s(t.hyl, t.yl), off);
        off = fma_rn(a.cy[yh], s(t.hyh, t.yh), off);
        off = fma_rn(a.cz[c], s(t.hzl, t.zl), off);
        off = fma_rn(a.cz[zh], s(t.hzh, t.zh), off);
        sout[c] = quot(add_rn(b[c], off), a.d[c], a.inv[c]);
    });
}

// --------------------------------------------------------------- source
// b = alpha [tr(G^2) + tr(G)^2] (Eq. igrelliptic) from the undivided central
// differences D = 2 dx G of u, with alpha_s = alpha / (2 dx)^2:
//   b = alpha_s [sum_ab D_ab D_ba + (sum_a D_aa)^2],
// in one fixed order of rounded operations
__device__ __forceinline__ C source_b(const C (&D)[3][3], C alpha_s)
{
    const C tr = add_rn(add_rn(D[0][0], D[1][1]), D[2][2]);
    C sq = mul_rn(D[0][0], D[0][0]);
    sq = fma_rn(D[1][1], D[1][1], sq);
    sq = fma_rn(D[2][2], D[2][2], sq);
    C x = mul_rn(D[0][1], D[1][0]);
    x = fma_rn(D[0][2], D[2][0], x);
    x = fma_rn(D[1][2], D[2][1], x);
    const C tr2 = fma_rn(C(2), x, sq);  // sum_ab D_ab D_ba
    return mul_rn(alpha_s, fma_rn(tr, tr, tr2));
}

// Four raw state values and their stage values, as StateIO
struct QRaw4Inc {
    Vec4<QB> b;
    V4 d;
};
using QRaw4 = std::conditional<kInc, QRaw4Inc, V4>::type;
template <bool HASD, class R = QRaw4> __device__ __forceinline__ R ldq4(const QIn &q, int u, const Geom &g, idx off)
{
    if constexpr (std::is_same<R, QRaw4Inc>::value) {
        R r;
        r.b = ld4r(CKP4(q.b[0] + u * q.fs + off, q.b[0], 5 * g.n));
        if constexpr (HASD) r.d = ld4r(CKP4(q.d[0] + u * q.fs + off, q.d[0], 5 * g.n));
        return r;
    } else {
        const S *f = reinterpret_cast<const S *>(q.b[u]);
        return ld4r(CKP4(f + off, f, g.n));
    }
}
template <bool HASD, class R> __device__ __forceinline__ void cvq4(const R &r, C o[4])
{
    if constexpr (std::is_same<R, QRaw4Inc>::value) {
        cv4(r.b, o);
        if constexpr (HASD) {
            C d[4];
            cv4(r.d, d);
#pragma unroll
            for (int c = 0; c < 4; c++) o[c] = C(__fadd_rn(float(o[c]), float(d[c])));
        }
    } else {
        cv4(r, o);
    }
}

// grad u by central differences: u of plane k in a shared tile (x and y
// neighbours), the planes below and above in registers. In the increment
// modes the kernel also stores the stage's density rounded to the storage
// type (rho_out), which the sweeps of the stage read. 16-bit storage
// alternates two plane tiles (one barrier per plane); the others keep one.
constexpr int SOURCE_BUFS = sizeof(S) == 2 ? 2 : 1;
template <bool HASD, bool FULL>
__device__ __forceinline__ void source_quads(const QIn q, S *b, S *rho_out, const Geom &g,
                                            C alpha_s, const C *W, const C *J, int zc, const BlockPos &bp, int wq,
                                            int rows, C *U2)
{
    const Quad t = quad_of<FULL, 1>(g, bp, wq, rows);
    const int k0 = bp.z * zc, k1 = min(g.nz, k0 + zc);
    const idx pl = (idx)g.plane;
    // u = m / rho from raw values (products rounded before they are
    // differenced: equal neighbours give an exact 0)
    auto u4 = [&](const QRaw4 (&r)[4], C u[3][VX], C rho[VX]) {
        C m[VX], rr[VX];
        cvq4<HASD>(r[0], rho);
#pragma unroll
        for (int c = 0; c < VX; c++) rr[c] = rcp(rho[c]);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            cvq4<HASD>(r[1 + a], m);
#pragma unroll
            for (int c = 0; c < VX; c++) u[a][c] = mul_rn(m[c], rr[c]);
        }
    };
    // u of the own cells of plane kk (the jet blend below an inflow face);
    // rho gets their (unblended) densities
    auto own_u = [&](int kk, C u[3][VX], C rho[VX]) {
        const idx zb = (idx)zmap(kk, g) * pl + t.own;
        C v[4][VX];
#pragma unroll
        for (int f = 0; f < 4; f++) cvq4<HASD>(ldq4<HASD>(q, f, g, zb), v[f]);
#pragma unroll
        for (int c = 0; c < VX; c++) rho[c] = v[0][c];
        if (kk < 0 && g.bc[4] == BC_INFLOW) {
#pragma unroll
            for (int c = 0; c < VX; c++) {
                const idx fc = ck(t.own + (idx)c, g.plane);
                const C w = C(1) - W[fc];
#pragma unroll
                for (int f = 0; f < 4; f++) v[f][c] = fma_rn(w, v[f][c], J[(idx)f * pl + fc]);
            }
        }
#pragma unroll
        for (int c = 0; c < VX; c++) {
            const C r = rcp(v[0][c]);
#pragma unroll
            for (int a = 0; a < 3; a++) u[a][c] = mul_rn(v[1 + a][c], r);
        }
    };
    C um[3][VX], u0[3][VX], up[3][VX];
    C rho0[VX], rhop[VX];  // densities of the own cells at k and k + 1
    if (FULL || t.active) {
        own_u(k0 - 1, um, rhop);
        own_u(k0, u0, rho0);
    }
    // raw values one plane ahead: own cells at k + 1, halo at k (planes >= 0).
    // The increment modes' stages 2 and 3 (base and increments, 6 registers
    // per field and 4 cells) load the halo when it is used instead, which
    // keeps the registers under two blocks per SM with fewer spills.
    constexpr bool kHaloAhead = !(kInc && HASD);
    QRaw4 nc[4], nh[4];
    QRaw nxh[4];
    auto halo = [&](int kk) {
        if (t.yh) {
#pragma unroll
            for (int f = 0; f < 4; f++) nh[f] = ldq4<HASD>(q, f, g, (idx)kk * pl + t.hoff);
        } else if (t.xh) {
#pragma unroll
            for (int f = 0; f < 4; f++) nxh[f] = ldqr<HASD>(q, f, ck((idx)kk * pl + t.hoff, g.n));
        }
    };
    auto pre = [&](int kk) {
        if (FULL || t.active) {
            const idx pz = (idx)zmap(kk + 1, g) * pl + t.own;
#pragma unroll
            for (int f = 0; f < 4; f++) nc[f] = ldq4<HASD>(q, f, g, pz);
        }
        if (kHaloAhead) halo(kk);
    };
    pre(k0);
    for (int k = k0; k < k1; k++) {
        if (!kHaloAhead) halo(k);
        // two buffers: the one written here was last read two planes ago,
        // before the barrier of the previous plane
        C *U = U2 + (SOURCE_BUFS == 2 ? ((k - k0) & 1) * 3 * TILEV : 0);
        if (SOURCE_BUFS == 1) __syncthreads();  // readers of the previous plane are done
        if (FULL || t.active) {
#pragma unroll
            for (int a = 0; a < 3; a++) sh_st4(U + a * TILEV + t.pos, u0[a]);
        }
        if (t.yh) {
            C hu[3][VX], hrho[VX];
            u4(nh, hu, hrho);
#pragma unroll
            for (int a = 0; a < 3; a++) sh_st4(U + a * TILEV + cks4(t.hpos, TILEV), hu[a]);
        } else if (t.xh) {
            const C r = rcp(cvq<HASD>(nxh[0]));
#pragma unroll
            for (int a = 0; a < 3; a++) U[a * TILEV + cks(t.hpos, TILEV)] = mul_rn(cvq<HASD>(nxh[1 + a]), r);
        }
        if (FULL || t.active) u4(nc, up, rhop);
        if (k + 1 < k1) pre(k + 1);
        __syncthreads();
        if (FULL || t.active) {
            C ym[3][VX], yp[3][VX], o[VX], xl[3], xr[3];
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const C *T = U + a * TILEV + t.pos;
                sh_ld4(T - t.pitch, ym[a]);
                sh_ld4(T + t.pitch, yp[a]);
                xl[a] = T[-1];
                xr[a] = T[VX];
            }
#pragma unroll
            for (int c = 0; c < VX; c++) {
                C D[3][3];  // D[a][d]: undivided central difference of u_a along d
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    const C xm = c > 0 ? u0[a][c - 1] : xl[a];
                    const C xp = c < VX - 1 ? u0[a][c + 1] : xr[a];
                    D[a][0] = xp - xm;
                    D[a][1] = yp[a][c] - ym[a][c];
                    D[a][2] = up[a][c] - um[a][c];
                }
                o[c] = source_b(D, alpha_s);
            }
            const idx at = (idx)k * pl + t.own;
            st4(CKP4(b + at, b, g.n), o);
            if constexpr (kInc) st4(CKP4(rho_out + at, rho_out, g.n), rho0);
#pragma unroll
            for (int a = 0; a < 3; a++)
#pragma unroll
                for (int c = 0; c < VX; c++) {
                    um[a][c] = u0[a][c];
                    u0[a][c] = up[a][c];
                }
#pragma unroll
            for (int c = 0; c < VX; c++) rho0[c] = rhop[c];
        }
    }
}

// the pairs: u of a cell and the one above it, one halo cell per thread of
// the first three warps, raw values one plane ahead
template <bool HASD>
__device__ __forceinline__ void source_pairs(const QIn q, S *b, S *rho_out, const Geom &g,
                                             C alpha_s, const C *W, const C *J, int zc, const BlockPos &bp, C *U2)
{
    const Pair t = pair_of(g, bp);
    const int k0 = bp.z * zc, k1 = min(g.nz, k0 + zc);
    const idx pl = (idx)g.plane;
    QRaw nc[2][4], nh[4];
    auto load = [&](int kk) {  // own cells of plane kk
        const idx pz = (idx)zmap(kk, g) * pl;
#pragma unroll
        for (int c = 0; c < 2; c++)
            if (t.need[c]) {
#pragma unroll
                for (int f = 0; f < 4; f++) nc[c][f] = ldqr<HASD>(q, f, ck(pz + t.own[c], g.n));
            }
    };
    auto halo = [&](int kk) {
        if (t.h) {
#pragma unroll
            for (int f = 0; f < 4; f++) nh[f] = ldqr<HASD>(q, f, ck((idx)kk * pl + t.hoff, g.n));
        }
    };
    // u = m / rho (products rounded before they are differenced: equal
    // neighbours give an exact 0), with the jet blend below an inflow face
    auto conv = [&](int kk, C (&u)[2][3], C (&rho)[2]) {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (!t.need[c]) continue;
            C v[4];
#pragma unroll
            for (int f = 0; f < 4; f++) v[f] = cvq<HASD>(nc[c][f]);
            rho[c] = v[0];
            if (kk < 0 && g.bc[4] == BC_INFLOW) {
                const idx f0 = ck(t.own[c], g.plane);
                const C w = C(1) - W[f0];
#pragma unroll
                for (int f = 0; f < 4; f++) v[f] = fma_rn(w, v[f], J[(idx)f * pl + f0]);
            }
            const C r = rcp(v[0]);
#pragma unroll
            for (int a = 0; a < 3; a++) u[c][a] = mul_rn(v[1 + a], r);
        }
    };
    C um[2][3] = {}, u0[2][3] = {}, up[2][3] = {}, rho0[2] = {}, rhop[2] = {};
    load(k0 - 1);
    conv(k0 - 1, um, rhop);
    load(k0);
    conv(k0, u0, rho0);
    load(k0 + 1);
    halo(k0);
    for (int k = k0; k < k1; k++) {
        C *U = U2 + ((k - k0) & 1) * 3 * TILEP;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            U[a * TILEP + t.pos] = u0[0][a];
            U[a * TILEP + t.pos + PPITCH] = u0[1][a];
        }
        if (t.h) {
            const C r = rcp(cvq<HASD>(nh[0]));
#pragma unroll
            for (int a = 0; a < 3; a++) U[a * TILEP + cks(t.hpos, TILEP)] = mul_rn(cvq<HASD>(nh[1 + a]), r);
        }
        conv(k + 1, up, rhop);
        if (k + 1 < k1) {
            load(k + 2);
            halo(k + 1);
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (!t.in[c]) continue;
            C D[3][3];  // D[a][d]: undivided central difference of u_a along d
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const C *T = U + a * TILEP + t.pos + c * PPITCH;
                D[a][0] = T[1] - T[-1];
                D[a][1] = (c ? T[PPITCH] : u0[1][a]) - (c ? u0[0][a] : T[-PPITCH]);
                D[a][2] = up[c][a] - um[c][a];
            }
            const idx at = (idx)k * pl + t.own[c];
            stc(CKP(b + at, b, g.n), source_b(D, alpha_s));
            if constexpr (kInc) stc(CKP(rho_out + at, rho_out, g.n), rho0[c]);
        }
#pragma unroll
        for (int c = 0; c < 2; c++) {
#pragma unroll
            for (int a = 0; a < 3; a++) {
                um[c][a] = u0[c][a];
                u0[c][a] = up[c][a];
            }
            rho0[c] = rhop[c];
        }
    }
}

// Two blocks per SM (at most 128 registers): the kernel waits on load
// latency, and one block per SM, which a free register choice gives (about
// 156 registers), runs it 1.6x slower. The increment modes' form, which
// holds raw FP32 values and 16-bit increments one plane ahead, spills a few
// registers under this bound and still runs faster. FP64 keeps one block.
constexpr int SOURCE_BLOCKS = sizeof(C) == 8 ? 1 : 2;
template <bool HASD, bool FULL>
__global__ void __launch_bounds__(BT, SOURCE_BLOCKS) k_source(QIn q, S *b, S *rho_out, Geom g,
                                                              C alpha_s, const C *W, const C *J, int zc, int wq,
                                                              int rows)
{
    launched();
    __shared__ __align__(16) C U2[SOURCE_BUFS * 3 * TILEV];
    source_quads<HASD, FULL>(q, b, rho_out, g, alpha_s, W, J, zc, BlockPos::of_launch(), wq, rows, U2);
}
// The pairs wait on latency more (element loads, 24 per thread and plane in the
// increment modes): four blocks (64 registers, a few spilled) against three and
// two, 510 x 399 x 200: FP32 196, 221 and 262 us, BF16 increments 328, 378 and
// 448; only the smallest grids prefer fewer (33 x 35 x 37: 11.4, 10.5, 9.9).
constexpr int SOURCE_PAIR_BLOCKS = sizeof(C) == 8 ? 1 : 4;
template <bool HASD>
__global__ void __launch_bounds__(32 * PWARPS, SOURCE_PAIR_BLOCKS) k_source_pairs(QIn q, S *b, S *rho_out,
                                                                    Geom g, C alpha_s, const C *W, const C *J, int zc)
{
    launched();
    __shared__ C U2[2 * 3 * TILEP];
    source_pairs<HASD>(q, b, rho_out, g, alpha_s, W, J, zc, BlockPos::of_launch(), U2);
}


// ----------------------------------------------------------------- flux
// Block of TY + 1 warps over a TX x TY tile of columns. Warps 0..TY-1 own a
// row each: per plane a warp computes the x-face at the low side of each of
// its cells, the y-face below its row and, from its register queue, the
// z-face above; warp TY computes the y-faces above the last row and the
// x-faces at the high end of every row. Every warp thus does three face
// evaluations or fewer and the tile needs no face twice. The warp count is a
// multiple of 4 so that the four SM sub-partitions (16K registers each) hold
// equal shares: 16 warps of at most 128 registers in FP32 arithmetic, one
// block per SM, keep the stencil queue in registers.
constexpr int TX = 32, TY = sizeof(C) == 8 ? 7 : 15, NWARP = TY + 1, NT = 32 * NWARP;
constexpr int PW = TX + 6, PH = TY + 6;          // plane tile with a halo of 3
// tile cells that are read: the rows of the tile with the x-halo, the three
// rows above and below (no corner blocks), and the four cells diagonal to
// the interior's corners (the viscous faces' tangential neighbours)
constexpr int NPLANE = TY * PW + 6 * TX + 4;
constexpr int LPT = (NPLANE + NT - 1) / NT;      // tile cells loaded per thread
// every thread has a first tile cell (its test is dropped in the 16-bit
// forms, where that measured faster; FP32/FP64 keep it)
constexpr bool kR0 = sizeof(S) == 2 && NPLANE >= NT;

// The plane tiles keep the six face variables as three pairs, (rho, m_x),
// (m_y, m_z), (E, Sigma): a stencil point of a pair is one 8-byte (16-byte in
// FP64) shared load, and the reconstruction of a pair is one packed FP32x2
// multiply-add per term.

// 5th-order face values of a pair (weights as in rec_left / rec_right)
__device__ __forceinline__ C2 rec_left2(C2 a, C2 b, C2 c, C2 d, C2 e)
{
    C2 t = pmul(bcast(C(2.0 / 60.0)), a);
    t = pfma(bcast(C(-13.0 / 60.0)), b, t);
    t = pfma(bcast(C(47.0 / 60.0)), c, t);
    t = pfma(bcast(C(27.0 / 60.0)), d, t);
    return pfma(bcast(C(-3.0 / 60.0)), e, t);
}
__device__ __forceinline__ C2 rec_right2(C2 b, C2 c, C2 d, C2 e, C2 f)
{
    C2 t = pmul(bcast(C(-3.0 / 60.0)), b);
    t = pfma(bcast(C(27.0 / 60.0)), c, t);
    t = pfma(bcast(C(47.0 / 60.0)), d, t);
    t = pfma(bcast(C(-13.0 / 60.0)), e, t);
    return pfma(bcast(C(2.0 / 60.0)), f, t);
}

// 3rd-order face values of a pair: the quadratic through the three cell
// averages of the biased stencil (i-1..i+1 left, i..i+2 right) at the face
__device__ __forceinline__ C2 rec3_left2(C2 b, C2 c, C2 d)
{
    C2 t = pmul(bcast(C(-1.0 / 6.0)), b);
    t = pfma(bcast(C(5.0 / 6.0)), c, t);
    return pfma(bcast(C(2.0 / 6.0)), d, t);
}
__device__ __forceinline__ C2 rec3_right2(C2 c, C2 d, C2 e)
{
    C2 t = pmul(bcast(C(2.0 / 6.0)), c);
    t = pfma(bcast(C(5.0 / 6.0)), d, t);
    return pfma(bcast(C(-1.0 / 6.0)), e, t);
}

constexpr int TILE2 = 3 * PH * PW;  // pairs in one plane tile
// Layout of one plane tile: the pairs (rho, m_x) and (m_y, m_z) of a cell
// side by side, one 16-byte quad per cell (two in FP64) for cells 0..PH*PW-1,
// then the pairs (E, Sigma) of all cells. A stencil point is then one
// 16-byte shared load and one 8-byte load (FP32) instead of three 8-byte
// loads: the same shared-memory bandwidth in fewer instructions.
constexpr int QUADS = 2 * PH * PW;  // offset (in pairs) of the (E, Sigma) pairs
__device__ __forceinline__ int pair_at(int p, int e) { return p < 2 ? 2 * e + p : QUADS + e; }
// the pairs (rho, m_x), (m_y, m_z) of tile cell e
__device__ __forceinline__ void ld_quad(const float2 *T, int e, float2 &a, float2 &b)
{
    const float4 q = *reinterpret_cast<const float4 *>(T + 2 * e);
    a = make_float2(q.x, q.y);
    b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void ld_quad(const double2 *T, int e, double2 &a, double2 &b)
{
    a = T[2 * e];
    b = T[2 * e + 1];
}
__device__ __forceinline__ void st_quad(float2 *T, int e, float2 a, float2 b)
{
    *reinterpret_cast<float4 *>(T + 2 * e) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_quad(double2 *T, int e, double2 a, double2 b)
{
    T[2 * e] = a;
    T[2 * e + 1] = b;
}
// the three pairs of tile cell e
__device__ __forceinline__ void ld_cell(const C2 *T, int e, C2 &a, C2 &b, C2 &c)
{
    ld_quad(T, e, a, b);
    c = T[QUADS + e];
}
__device__ __forceinline__ void st_cell(C2 *T, int e, C2 a, C2 b, C2 c)
{
    st_quad(T, e, a, b);
    T[QUADS + e] = c;
}
// Face buffers of one parity: x-faces at w (TX + 1) + i, y-faces at w TX + i,
// each its two pairs side by side, then the E fluxes of all faces
constexpr int NFX = (TY * (TX + 1) + 3) / 4 * 4, NFY = (TY + 1) * TX, NFACE = 5 * (NFX + NFY);
__device__ __forceinline__ void ld_face(const C *B, int nf, int e, Flux &f)
{
    ld_quad(reinterpret_cast<const C2 *>(B), e, f.a, f.b);
    f.e = B[4 * nf + e];
}
__device__ __forceinline__ void st_face(C *B, int nf, int e, const Flux &f)
{
    st_quad(reinterpret_cast<C2 *>(B), e, f.a, f.b);
    B[4 * nf + e] = f.e;
}
// planes per turn of the march's loop: two in FP32 storage, where half the
// register rotations go (512 x 512 x 256, stages 1 to 3: 1.84 -> 1.78 ms per
// launch); the 16-bit forms, whose raw values are in flight in registers, and
// FP64 measured the same or slower (FP16 0.937 -> 0.965 ms, 512 x 512 x 128)
constexpr int kUnroll = sizeof(S) == 4 ? 2 : 1;
constexpr int RING = 7;             // plane tiles resident: k-2..k+3 and k+4 in flight

// Storage equal to the arithmetic type: plane tiles are copied global ->
// shared with cp.async (4- or 8-byte elements), which holds no registers.
constexpr bool kAsyncTile = sizeof(S) == sizeof(C);
__device__ __forceinline__ void cp_async_elem(C *dst, const S *src)
{
    unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(C) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// shared bytes: the ring of plane tiles (pairs), two sets of x- and y-face fluxes
__host__ __device__ constexpr size_t flux_smem_bytes()
{
    return RING * TILE2 * sizeof(C2) + 2 * NFACE * sizeof(C);
}

// tile cell e (0 <= e < NPLANE) -> position (lx, ly) in the PW x PH tile
__device__ __forceinline__ void plane_cell(int e, int &lx, int &ly)
{
    if (e < 3 * TX) { ly = e / TX; lx = 3 + e % TX; }
    else if (e < 3 * TX + TY * PW) { e -= 3 * TX; ly = 3 + e / PW; lx = e % PW; }
    else if (e < 6 * TX + TY * PW) { e -= 3 * TX + TY * PW; ly = TY + 3 + e / TX; lx = 3 + e % TX; }
    else { e -= 6 * TX + TY * PW; ly = (e & 2) ? TY + 3 : 2; lx = (e & 1) ? TX + 3 : 2; }
}

template <int D, int ORD>
__device__ __forceinline__ void face_from_stencil(const C2 (&s)[6][3], const Gas gas, Flux &F, FaceFlag &bad)
{
    C2 L[3], R[3];
#pragma unroll
    for (int p = 0; p < 3; p++) {
        L[p] = ORD == 3 ? rec3_left2(s[1][p], s[2][p], s[3][p])
                        : rec_left2(s[0][p], s[1][p], s[2][p], s[3][p], s[4][p]);
        R[p] = ORD == 3 ? rec3_right2(s[2][p], s[3][p], s[4][p])
                        : rec_right2(s[1][p], s[2][p], s[3][p], s[4][p], s[5][p]);
    }
    lf_flux2<D>(L, R, gas, F, bad);
}

// face along D (0, 1) from six consecutive cells of one plane tile starting
// at element `at`, `step` elements apart
template <int D, int ORD>
__device__ __forceinline__ void tile_face(const C2 *T, int at, int step, const Gas gas, Flux &F, FaceFlag &bad)
{
    C2 s[6][3];
#pragma unroll
    for (int m = 0; m < 6; m++) {
        if (ORD == 3 && (m == 0 || m == 5)) {
            s[m][0] = s[m][1] = s[m][2] = bcast(C(0));
        } else {
            ld_cell(T, cks(at + m * step, PH * PW), s[m][0], s[m][1], s[m][2]);
        }
    }
    face_from_stencil<D, ORD>(s, gas, F, bad);
}

// tile_face with the stencil's point 3 (the cell the face lies below / left of
// the row warp's own cell) given: the row warp holds it from its z-stencil
template <int D, int ORD>
__device__ __forceinline__ void tile_face_c(const C2 *T, int at, int step, const C2 (&c3)[3], const Gas gas, Flux &F,
                                            FaceFlag &bad)
{
    C2 s[6][3];
#pragma unroll
    for (int m = 0; m < 6; m++) {
        if (ORD == 3 && (m == 0 || m == 5)) {
            s[m][0] = s[m][1] = s[m][2] = bcast(C(0));
        } else if (m == 3) {
            s[m][0] = c3[0];
            s[m][1] = c3[1];
            s[m][2] = c3[2];
        } else {
            ld_cell(T, cks(at + m * step, PH * PW), s[m][0], s[m][1], s[m][2]);
        }
    }
    face_from_stencil<D, ORD>(s, gas, F, bad);
}

// ------------------------------------------------------- viscous stresses
// Velocity u = m / rho of the tile cell at pair offset `at`.
__device__ __forceinline__ void tvel(const C2 *T, int at, C u[3])
{
    C2 a, b;
    ld_quad(T, cks(at, PH * PW), a, b);
    C r = rcp(a.x);
    u[0] = a.y * r;
    u[1] = b.x * r;
    u[2] = b.y * r;
}

// Doubled viscous flux (like lf_flux2's 2 F_hat) through the face between
// cells A and B along axis D, added to G (Eqs. igrmobalance-igrenbalance with
// the stress of Eq. constitutive_law):
//   tau_aD = mu (du_a/dx_D + du_D/dx_a) + lam delta_aD div u, lam = zeta - 2 mu / 3,
//   G[1 + a] -= 2 tau_aD,  G[4] -= 2 sum_a ((u_a(A) + u_a(B)) / 2) tau_aD,
// with second-order face derivatives: normal (u(B) - u(A)) / dx, tangential
// along t the mean of the central differences at A and B. T1/T2 give the
// tangential axes t1 < t2 (the two axes other than D) as the cells on each
// side of A and B: a1m, a1p, b1m, b1p along t1 and a2m.. along t2.
template <int D>
__device__ __forceinline__ void visc_face(const C2 *TA, int a, const C2 *TB, int b, const C2 *T1Am,
                                          int a1m, const C2 *T1Ap, int a1p, const C2 *T1Bm, int b1m,
                                          const C2 *T1Bp, int b1p, const C2 *T2Am, int a2m,
                                          const C2 *T2Ap, int a2p, const C2 *T2Bm, int b2m,
                                          const C2 *T2Bp, int b2p, C mu, C lam, C inv_dx, Flux &G)
{
    constexpr int t1 = D == 0 ? 1 : 0, t2 = D == 2 ? 1 : 2;
    C uA[3], uB[3], p[3], m[3], q[3], r[3], Gr[3][3];
    tvel(TA, a, uA);
    tvel(TB, b, uB);
#pragma unroll
    for (int c = 0; c < 3; c++) Gr[c][D] = (uB[c] - uA[c]) * inv_dx;
    const C qd = C(0.25) * inv_dx;
    tvel(T1Ap, a1p, p); tvel(T1Am, a1m, m); tvel(T1Bp, b1p, q); tvel(T1Bm, b1m, r);
#pragma unroll
    for (int c = 0; c < 3; c++) Gr[c][t1] = ((p[c] - m[c]) + (q[c] - r[c])) * qd;
    tvel(T2Ap, a2p, p); tvel(T2Am, a2m, m); tvel(T2Bp, b2p, q); tvel(T2Bm, b2m, r);
#pragma unroll
    for (int c = 0; c < 3; c++) Gr[c][t2] = ((p[c] - m[c]) + (q[c] - r[c])) * qd;
    const C div = (Gr[0][0] + Gr[1][1]) + Gr[2][2];
    C work = C(0);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        C tau = mu * (Gr[c][D] + Gr[D][c]);
        if (c == D) tau += lam * div;
        (c == 0 ? G.a.y : c == 1 ? G.b.x : G.b.y) -= C(2) * tau;
        work += C(0.5) * (uA[c] + uB[c]) * tau;
    }
    G.e -= C(2) * work;
}

// registers per thread such that NWARP / 4 warps fit one sub-partition's 16K
constexpr int FLUX_MAXREG = sizeof(C) == 8 ? 224 : 128;

// The block keeps a ring of RING plane tiles (halo 3 in x and y) in shared
// memory: plane kk lives in slot (kk - k0 + 3) mod RING. Iteration k (from
// k0 - 1 to k1 - 1), one barrier each:
//   - start the copy of plane k + 4 into the slot of plane k - 3 (read for
//     the last time before the previous barrier);
//   - row warps: divergence and stage combination of plane k - 1 (face
//     buffers of parity k - 1), then the z-face k + 1/2 from planes
//     k - 2..k + 3 of the ring at the warp's own cells;
//   - all warps (k >= k0): the x- and y-faces of plane k into the face
//     buffers of parity k;
//   - complete the copy of plane k + 4, barrier.
// Planes k0 - 3..k0 + 2 are filled before the loop (with the boundary index
// mapping and, below an inflow face, the jet blend). Every plane is read from
// global memory once per block; nothing relies on the L1 cache.
//
// What bounds it is the latency of 16 warps' shared loads, MUFU operations
// and dependent arithmetic (issue slots 56-68% busy, no pipe above 35%): the face flux is packed by variable pairs and the
// face buffers hold quads (FP16 increments, stage 2: 695 -> 657 instructions
// per cell), and the prologue's planes are loaded three at a time. Per launch,
// stages 1 to 3: FP16 increments 1024 x 1024 x 256 7.26 -> 7.02 ms, FP32
// 512 x 512 x 256 1.96 -> 1.78 ms, 32^3 18.6 -> 16.8 us. Measured and not
// better: a split barrier with three face buffers (FP32 1.83 ms, FP16
// increments 7.9: the waits' polling costs issue slots), two rows per warp in
// eight warps of 255 registers (7.12 and 1.75 ms, FP16 6% slower).
//
// In the increment modes the input q_s is read as RN32(q^n + d_s) (d_s from
// stage 2 on), stages 1 and 2 store the 16-bit increment
// d_{s+1} = RN16(w [(q_s - q^n) + dt L]) into `out`, and stage 3 stores the
// FP32 state q^n + w [(q_s - q^n) + dt L] into `outb`.
template <int mode, int ORD, bool VISC>
__device__ __forceinline__ void flux_body(const QIn qin, const S *sig, const QBIn qn,
                                          const Fout<5> out, const QBOut outb, const Frhs rhs,
                                          const Fout<5> base_out, const Geom g, C gamma, C half_inv_dx,
                                          const Scalars *sc, double *blockmax, int *err, const C *W,
                                          const C *J, int zc, int cz0, C mu, C lamv, const BlockPos bp)
{
    constexpr bool HASD = kInc && (mode == FLUX_STAGE2 || mode == FLUX_STAGE3);
    // The five fields of every state buffer lie g.n values apart. In the
    // increment modes, which read and write more buffers, their addresses
    // come from the first field's pointer and that stride, so the kernel
    // holds one pointer per buffer: fewer constant-bank reloads of pointers
    // (9 against 26 per cell) for more 64-bit adds, 4.5% faster at full size;
    // the other forms keep a pointer per field (the same or 1% faster).
    const size_t fs = (size_t)g.n;
    const QB *const qb0 = qin.b[0];
    const S *const qd0 = qin.d[0];
    const QB *const qn0 = qn.p[0];
    S *const out0 = out.p[0];
    QB *const outb0 = outb.p[0];
    // raw state value u at offset c (StateIO's layout, one pointer per buffer)
    auto ldq_raw = [&](int u, idx c) -> QRaw {
        if constexpr (kInc) {
            QRawInc r;
            r.b = ldv(qb0 + u * fs + c);
            r.d = HASD ? ldr(qd0 + u * fs + c) : S(0.0f);
            return *reinterpret_cast<QRaw *>(&r);
        } else {
            return ldqr<HASD>(qin, u, c);
        }
    };
    // field u of the stored input (u < 5: q, 5: Sigma) where the state has the storage type
    auto fin = [&](int u) -> const S * { return u < 5 ? reinterpret_cast<const S *>(qin.b[u]) : sig; };
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *P = reinterpret_cast<C2 *>(smem_raw);        // [RING][3][PH][PW]
    C *FB = reinterpret_cast<C *>(P + RING * TILE2);  // [2][NFACE]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int x0 = bp.x * TX, y0 = bp.y * TY;
    const int cz = cz0 + bp.z;  // z-chunk (a launch may cover chunks cz0.. only)
    const int k0 = cz * zc, k1 = min(g.nz, k0 + zc);
    const bool rowwarp = w < TY;  // warp-uniform
    const int i = x0 + lane, j = y0 + (rowwarp ? w : 0);
    const bool active = rowwarp && i < g.nx && j < g.ny;
    const idx pl = (idx)g.plane;
    const idx own = (idx)(j * g.nx + i);
    const int tcell = (w + 3) * PW + lane + 3;  // this row-warp lane's cell in a tile
    const Gas gas = {gamma, gamma - C(1)};
    FaceFlag bad = FaceFlag(kFaceMin ? 1 : 0);  // face states with rho <= 0 or p <= 0 (warning)
    bool nonfinite = false; // a non-finite output (error)
    // ring slot offsets (in pairs) of planes k-2..k+4 in iteration k, rotated
    // once per plane: plane kk sits in slot (kk - k0 + 3) mod RING
    int ro[RING];
#pragma unroll
    for (int m = 0; m < RING; m++) ro[m] = m * TILE2;  // k = k0 - 1: planes k0-3.. in slots 0..


    // tile cells this thread loads each plane: shared and in-plane offsets
    int soff[LPT];
    idx goff[LPT];
#pragma unroll
    for (int r = 0; r < LPT; r++) {
        int e = tid + r * NT;
        soff[r] = -1;
        goff[r] = 0;
        if (e < NPLANE) {
            int lx, ly;
            plane_cell(e, lx, ly);
            soff[r] = ly * PW + lx;
            // Columns that no cell of the grid reads (past nx + 2) mirror the last ones
            // instead of repeating the last: a warp's cp.async copies of one address are
            // served one by one, which made the ragged blocks of an outflow edge twice as
            // long (right-hand side, FP32, 130 x 126 x 122: 138 us, 77 now; 75 periodic).
            int x = x0 + lx - 3;
            if (x > g.nx + 2 && g.bc[1] != BC_PERIODIC) x = max(2 * g.nx + 1 - x, 0);
            goff[r] = (idx)(map_axis(y0 + ly - 3, g.ny, g.bc[2], g.bc[3]) * g.nx + map_axis(x, g.nx, g.bc[0], g.bc[1]));
        }
    }

    // planes k0 - 3..k0 + 2, loaded (several planes' loads in flight: each
    // would cost a latency of its own) and stored directly, with the index
    // mapping in z and the jet blend below an inflow face
    constexpr int PLN = sizeof(C) == 8 ? 2 : 3;
#pragma unroll 1
    for (int kp = k0 - 3; kp < k0 + 3; kp += PLN) {
        QRaw v0[PLN][LPT][5];
        S v5[PLN][LPT];
#pragma unroll
        for (int m = 0; m < PLN; m++) {
            const idx zb = (idx)zmap(kp + m, g) * pl;
#pragma unroll
            for (int r = 0; r < LPT; r++)
                if ((kR0 && r == 0) || soff[r] >= 0) {
                    const idx c = ck(zb + goff[r], g.n);
#pragma unroll
                    for (int u = 0; u < 5; u++) v0[m][r][u] = ldq_raw(u, c);
                    v5[m][r] = ldr(sig + c);
                }
        }
#pragma unroll
        for (int m = 0; m < PLN; m++) {
            C2 *T = P + (kp + m - k0 + 3) * TILE2;
            const bool blend = kp + m < 0 && g.bc[4] == BC_INFLOW;
#pragma unroll
            for (int r = 0; r < LPT; r++)
                if ((kR0 && r == 0) || soff[r] >= 0) {
                    C v[5];
#pragma unroll
                    for (int u = 0; u < 5; u++) v[u] = cvq<HASD>(v0[m][r][u]);
                    if (blend) {
                        C wf = C(1) - W[ck(goff[r], g.plane)];
#pragma unroll
                        for (int u = 0; u < 5; u++) v[u] = wf * v[u] + J[(idx)u * pl + ck(goff[r], g.plane)];
                    }
                    st_cell(T, cks(soff[r], PH * PW), pset(v[0], v[1]), pset(v[2], v[3]), pset(v[4], C(cv(v5[m][r]))));
                }
        }
    }

    // plane kk >= k0 + 3 of the pipeline: FP32/FP64 storage copies with
    // cp.async; 16-bit storage loads raw values into registers at `fetch`
    // and converts and stores them at `land`
    S Rg[LPT][6];     // (unused with cp.async and in the increment modes)
    QRaw Rq[LPT][5];  // increment modes: raw q^n and d_s
    S Rs[LPT];        // increment modes: raw Sigma
    auto fetch = [&](int kk, C2 *T) {
        const idx zb = (idx)zmap(kk, g) * pl;
#pragma unroll
        for (int r = 0; r < LPT; r++)
            if ((kR0 && r == 0) || soff[r] >= 0) {
                if constexpr (kInc) {
                    const idx c = ck(zb + goff[r], g.n);
#pragma unroll
                    for (int u = 0; u < 5; u++) Rq[r][u] = ldq_raw(u, c);
                    Rs[r] = ldr(sig + c);
                } else {
#pragma unroll
                    for (int u = 0; u < 6; u++) {
                        if constexpr (kAsyncTile)
                            cp_async_elem(&T[pair_at(u >> 1, cks(soff[r], PH * PW))].x + (u & 1),
                                          CKP(fin(u) + zb + goff[r], fin(u), g.n));
                        else
                            Rg[r][u] = ldr(CKP(fin(u) + zb + goff[r], fin(u), g.n));
                    }
                }
            }
        if constexpr (kAsyncTile) cp_async_commit();
    };
    auto land = [&](C2 *T) {
        if constexpr (kAsyncTile) {
            cp_async_wait_all();
        } else if constexpr (kInc) {
#pragma unroll
            for (int r = 0; r < LPT; r++)
                if ((kR0 && r == 0) || soff[r] >= 0) {
                    st_cell(T, cks(soff[r], PH * PW), pset(cvq<HASD>(Rq[r][0]), cvq<HASD>(Rq[r][1])),
                            pset(cvq<HASD>(Rq[r][2]), cvq<HASD>(Rq[r][3])), pset(cvq<HASD>(Rq[r][4]), cv(Rs[r])));
                }
        } else {
#pragma unroll
            for (int r = 0; r < LPT; r++)
                if ((kR0 && r == 0) || soff[r] >= 0)
                    st_cell(T, cks(soff[r], PH * PW), pset(cv(Rg[r][0]), cv(Rg[r][1])), pset(cv(Rg[r][2]), cv(Rg[r][3])),
                            pset(cv(Rg[r][4]), cv(Rg[r][5])));
        }
    };
    __syncthreads();

    C dt32 = C(0), w32 = C(1);
    double dt = 0.0, wd = 1.0;
    if (mode != FLUX_RHS) {
        dt = sc->dt;
        wd = mode == FLUX_STAGE1 ? 1.0 : mode == FLUX_STAGE2 ? 0.25 : 2.0 / 3.0;
        dt32 = C(dt);
        w32 = C(wd);
    }
    C smax = C(0);  // running wave-speed maximum (FP32 here: FP64 is slow on this GPU)

    Flux Fzm, Fzp;
    // planes k and k + 1 at a row-warp lane's cell before iteration k: the
    // z-stencils of consecutive planes share them, so each iteration loads
    // four of its six points (shared loads are the flux kernel's most
    // contended resource; the copies are register moves). Not in the
    // viscous kernels, whose extra registers would spill.
    // this lane's x-face (at the low side of its cell) and y-face (below its
    // row) of the last plane: the divergence of that plane takes them from
    // registers and only the faces of its neighbours from the face buffers
    constexpr bool kOwnFaces = sizeof(C) == 4;
    Flux Fxo, Fyo;
    C2 zq[2][3];
    if (!VISC && rowwarp) {
        ld_cell(P + ro[2], cks(tcell, PH * PW), zq[0][0], zq[0][1], zq[0][2]);  // plane k0 - 1
        ld_cell(P + ro[3], cks(tcell, PH * PW), zq[1][0], zq[1][1], zq[1][2]);  // plane k0
    }
    QB qnv[5];  // q^n of plane k - 1 (stages 2 and 3), loaded one iteration ahead

    // divergence and stage combination of plane kk (face buffers of parity kk)
    // The three pairs of a row-warp lane's own cell in plane k, taken from its
    // z-stencil (the stencil's centre plane): they are point 3 of the lane's
    // x- and y-face stencils in plane k and the stage input the divergence of
    // plane k combines in the next iteration, so none is loaded twice.
    C2 cc[3];
    auto finish = [&](int kk) {
        const C *FX = FB + (kk & 1) * NFACE, *FY = FX + 5 * NFX;
        idx c = ck((idx)kk * pl + own, g.n);
        // the faces above and right of the cell from the buffers, the two
        // below and left of it computed by this lane (Fxo, Fyo; FP64
        // arithmetic reads them back, its extra registers would spill)
        Flux xr, yr, xl, yl;
        ld_face(FX, NFX, cks(w * (TX + 1) + lane + 1, NFX), xr);
        ld_face(FY, NFY, cks((w + 1) * TX + lane, NFY), yr);
        if (kOwnFaces) {
            xl = Fxo;
            yl = Fyo;
        } else {
            ld_face(FX, NFX, cks(w * (TX + 1) + lane, NFX), xl);
            ld_face(FY, NFY, cks(w * TX + lane, NFY), yl);
        }
        const C2 nh = bcast(-half_inv_dx);
        const C2 La = pmul(padd(padd(psub(xr.a, xl.a), psub(yr.a, yl.a)), psub(Fzp.a, Fzm.a)), nh);
        const C2 Lb = pmul(padd(padd(psub(xr.b, xl.b), psub(yr.b, yl.b)), psub(Fzp.b, Fzm.b)), nh);
        const C Lv[5] = {La.x, La.y, Lb.x, Lb.y, -(((xr.e - xl.e) + (yr.e - yl.e)) + (Fzp.e - Fzm.e)) * half_inv_dx};
        if (mode == FLUX_RHS) {
#pragma unroll
            for (int u = 0; u < 5; u++) rhs.p[u][c] = Lv[u];
            nonfinite |= !isfinite((Lv[0] + Lv[1]) + (Lv[2] + Lv[3]) + Lv[4]);
        } else {
            const C2 a = cc[0], b = cc[1], e = cc[2];  // plane kk at this cell
            const C qsv[5] = {a.x, a.y, b.x, b.y, e.x};
            if (mode == FLUX_STAGE1 && base_out.p[0]) {
                // the RK base q^n for stages 2 and 3 (exact: qsv holds stored values)
#pragma unroll
                for (int u = 0; u < 5; u++) stc(base_out.p[u] + c, qsv[u]);
            }
            C o[5], qb[5];
#pragma unroll
            for (int u = 0; u < 5; u++) qb[u] = mode == FLUX_STAGE1 ? qsv[u] : cv(qnv[u]);
            if constexpr (kInc) {
#pragma unroll
                for (int u = 0; u < 5; u++) {
                    const C inc = mode == FLUX_STAGE1 ? dt32 * Lv[u] : w32 * ((qsv[u] - qb[u]) + dt32 * Lv[u]);
                    if (mode == FLUX_STAGE3)
                        o[u] = stc(outb0 + u * fs + c, qb[u] + inc);  // q^n+1 in FP32
                    else
                        o[u] = stc(out0 + u * fs + c, inc);  // the increment d_s+1, rounded to 16 bits
                }
            } else {
                rk_store5(out, c, qb, qsv, Lv, dt32, dt, w32, wd, o);
            }
            nonfinite |= !isfinite((o[0] + o[1]) + (o[2] + o[3]) + o[4]);
            if (mode == FLUX_STAGE3) {
                C sp = cell_speed(o[0], o[1], o[2], o[3], o[4], gamma, gas.gm1);
                smax = (sp > smax || sp != sp) ? sp : smax;
            }
        }
    };

#pragma unroll kUnroll
    for (int k = k0 - 1; k < k1; k++) {
        const bool more = k + 4 <= k1 + 2;  // plane k + 4 feeds the z-faces
        if (more) fetch(k + 4, P + ro[6]);
        const C2 *T = P + ro[2];  // plane k
        C *FX = FB + (k & 1) * NFACE, *FY = FX + 5 * NFX;
        Flux F;
        const C2 *Tm = P + ro[1], *Tp = P + ro[3];  // planes k - 1, k + 1 (viscous terms)
        const C inv_dx = C(2) * half_inv_dx;
        // viscous x-face between tile cells a and a + 1 (same row)
        auto visc_x = [&](int a) {
            visc_face<0>(T, a, T, a + 1, T, a - PW, T, a + PW, T, a + 1 - PW, T, a + 1 + PW, Tm, a, Tp,
                         a, Tm, a + 1, Tp, a + 1, mu, lamv, inv_dx, F);
        };
        // viscous y-face between tile cells a and a + PW (same column)
        auto visc_y = [&](int a) {
            visc_face<1>(T, a, T, a + PW, T, a - 1, T, a + 1, T, a + PW - 1, T, a + PW + 1, Tm, a, Tp,
                         a, Tm, a + PW, Tp, a + PW, mu, lamv, inv_dx, F);
        };
        if (rowwarp) {
            if (active) {
                if (k > k0) finish(k - 1);
                if (k >= k0 && (mode == FLUX_STAGE2 || mode == FLUX_STAGE3)) {
                    idx c = ck((idx)k * pl + own, g.n);
#pragma unroll
                    for (int u = 0; u < 5; u++) qnv[u] = ldv(kInc ? qn0 + u * fs + c : qn.p[u] + c);
                }
            }
            Fzm = Fzp;
            C2 sz[6][3];  // z-stencil: planes k - 2..k + 3 at this cell
#pragma unroll
            for (int m = 0; m < 6; m++) {
                if (!VISC && (m == 2 || m == 3)) {  // planes k, k + 1: points 3, 4 of the previous z-stencil
#pragma unroll
                    for (int p = 0; p < 3; p++) sz[m][p] = zq[m - 2][p];
                } else {
                    ld_cell(P + ro[m], cks(tcell, PH * PW), sz[m][0], sz[m][1], sz[m][2]);
                }
            }
            if constexpr (!VISC) {
#pragma unroll
                for (int p = 0; p < 3; p++) {
                    zq[0][p] = sz[3][p];
                    zq[1][p] = sz[4][p];
                }
            }
            face_from_stencil<2, ORD>(sz, gas, Fzp, bad);  // z-face k + 1/2
            cc[0] = sz[2][0];  // plane k at this cell
            cc[1] = sz[2][1];
            cc[2] = sz[2][2];
            if constexpr (VISC) {
                const C2 *Ta = P + ro[2], *Tb = P + ro[3];  // planes k, k + 1
                visc_face<2>(Ta, tcell, Tb, tcell, Ta, tcell - 1, Ta, tcell + 1, Tb, tcell - 1, Tb,
                             tcell + 1, Ta, tcell - PW, Ta, tcell + PW, Tb, tcell - PW, Tb, tcell + PW,
                             mu, lamv, C(2) * half_inv_dx, Fzp);
            }
            if (k >= k0) {
                // x-face at the low side of cell `lane` of row w (tile cells lane-3..lane+2)
                tile_face_c<0, ORD>(T, (w + 3) * PW + lane, 1, cc, gas, F, bad);
                if constexpr (VISC) visc_x((w + 3) * PW + lane + 2);
                st_face(FX, NFX, cks(w * (TX + 1) + lane, NFX), F);
                if constexpr (kOwnFaces) Fxo = F;
                // y-face below row w in column lane (tile rows w-3..w+2)
                tile_face_c<1, ORD>(T, w * PW + lane + 3, PW, cc, gas, F, bad);
                if constexpr (VISC) visc_y((w + 2) * PW + lane + 3);
                st_face(FY, NFY, cks(w * TX + lane, NFY), F);
                if constexpr (kOwnFaces) Fyo = F;
            }
        } else if (k >= k0) {
            // y-face above the last row, column lane
            tile_face<1, ORD>(T, TY * PW + lane + 3, PW, gas, F, bad);
            if constexpr (VISC) visc_y((TY + 2) * PW + lane + 3);
            st_face(FY, NFY, cks(TY * TX + lane, NFY), F);
            if (lane < TY) {
                // x-face at the high end of row `lane`
                tile_face<0, ORD>(T, (lane + 3) * PW + TX, 1, gas, F, bad);
                if constexpr (VISC) visc_x((lane + 3) * PW + TX + 2);
                st_face(FX, NFX, cks(lane * (TX + 1) + TX, NFX), F);
            }
        }
        if (more) land(P + ro[6]);
        __syncthreads();
        const int r0 = ro[0];
#pragma unroll
        for (int m = 0; m + 1 < RING; m++) ro[m] = ro[m + 1];
        ro[RING - 1] = r0;
    }
    // the last plane (its faces are behind the final barrier; its cell's
    // values are in cc from the last z-stencil)
    if (active) finish(k1 - 1);
    const bool badf = flag_bad(bad);
    if (nonfinite || badf) atomicOr(err, (nonfinite ? ERRF_NONFINITE : 0) | (badf ? ERRF_FACE : 0));
    if (mode == FLUX_STAGE3) {
        double m = block_max<NT>(double(smax));
        if (tid == 0)
            blockmax[(cz * (long long)bp.gy + bp.y) * bp.gx + bp.x] = m;
    }
}
template <int mode, int ORD, bool VISC>
__global__ void __maxnreg__(FLUX_MAXREG)
    k_flux(QIn qin, const S *sig, QBIn qn, Fout<5> out, QBOut outb, Frhs rhs, Fout<5> base_out,
           Geom g, C gamma, C half_inv_dx, const Scalars *sc, double *blockmax, int *err, const C *W,
           const C *J, int zc, int cz0, C mu, C lamv)
{
    launched();
    flux_body<mode, ORD, VISC>(qin, sig, qn, out, outb, rhs, base_out, g, gamma, half_inv_dx, sc, blockmax, err,
                               W, J, zc, cz0, mu, lamv, BlockPos::of_launch());
}


// stand-alone stage combination (the flux kernel's epilogue) over n values;
// in the increment modes the FP32 state update of stage 3 on FP32 arrays
__global__ void k_rk_combine(const QB *__restrict__ qn, const QB *__restrict__ qs,
                             const C *__restrict__ L, QB *__restrict__ out, long long n, double dt,
                             double wd)
{
    C dt32 = C(dt), w32 = C(wd);
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x) {
        C a = cv(__ldg(qn + c)), b = cv(__ldg(qs + c)), l = L[c];
        if constexpr (kNarrow && !kInc) {
            bool ok;
            S h = rk_narrow_one<S>(a, b, l, dt32, w32, ok);
            if (!ok) h = rk_fp64<S>(a, b, l, dt, wd);
            reinterpret_cast<S *>(out)[c] = h;
        } else {
            out[c] = a + w32 * ((b - a) + dt32 * l);
        }
    }
}

// ---------------------------------------------------------- wave speed
// Memory-bound, five fields read once. The running maximum stays in the
// arithmetic type: one FP64 comparison per cell runs at a 64th of the FP32 rate
// and was what bounded the FP32 and 16-bit kernels. Four cells per load where
// the fields allow it. 67M cells in FP32: 416 us before, 207 us now (6.5 TB/s);
// 34M FP16 cells: 209 and 66 us.
constexpr int SPEED_NT = 256, SPEED_MAXBLOCKS = 152 * 8;

template <bool VEC>
__global__ void __launch_bounds__(SPEED_NT) k_speed(const QB *q, long long n, C gamma,
                                                     double *blockmax)
{
    launched();
    C m = C(0);
    const C gm1 = gamma - C(1);
    auto take = [&](C rho, C mx, C my, C mz, C E) {
        const C sp = cell_speed(rho, mx, my, mz, E, gamma, gm1);
        m = (sp > m || sp != sp) ? sp : m;  // a NaN stays (no later value exceeds it)
    };
    if constexpr (VEC) {
        for (long long c = blockIdx.x * (long long)SPEED_NT + threadIdx.x; c < n / 4; c += (long long)gridDim.x * SPEED_NT) {
            Vec4<QB> r[5];
            C v[5][4];
#pragma unroll
            for (int u = 0; u < 5; u++) r[u] = ld4r(q + u * n + 4 * c);
#pragma unroll
            for (int u = 0; u < 5; u++) cv4(r[u], v[u]);
#pragma unroll
            for (int x = 0; x < 4; x++) take(v[0][x], v[1][x], v[2][x], v[3][x], v[4][x]);
        }
    } else {
        for (long long c = blockIdx.x * (long long)SPEED_NT + threadIdx.x; c < n; c += (long long)gridDim.x * SPEED_NT)
            take(cv(q[c]), cv(q[n + c]), cv(q[2 * n + c]), cv(q[3 * n + c]), cv(q[4 * n + c]));
    }
    const double bm = block_max<SPEED_NT>(double(m));
    if (threadIdx.x == 0) blockmax[blockIdx.x] = bm;
}

// ------------------------------------------------------------ diagnostics
// FP64 evaluation of the state's totals, extrema and the residual of the
// elliptic equation (Eq. igrelliptic) for the stored Sigma:
//   (A s)_i = s_i (1/rho_i + beta sum_f c_f) - beta sum_f c_f s_nb,
//   c_f = (1/rho_i + 1/rho_nb) / 2, beta = alpha / dx^2, faces on a
//   non-periodic boundary dropped (the operator the Jacobi sweeps relax);
//   b_i = alpha [sum_ab G_ab G_ba + (sum_a G_aa)^2], G_ab the central
//   difference of u_a = m_a / rho along b (the source kernel's definition,
//   with the same boundary mapping and jet blend).
// Every stored value converts to double exactly, so the result is the FP64
// evaluation on the stored state. One thread per cell (grid-stride), per-block
// partial results in a fixed reduction order: deterministic.
constexpr int DIAG_NT = 256, DIAG_NV = DIAG_PARTS;

// conserved value u at (i, j, kk) through the boundary mapping, in FP64
__device__ __forceinline__ double dval(const QB *q, const Geom &g, const C *W, const C *J, int i,
                                       int j, int kk, int u)
{
    int mi = map_axis(i, g.nx, g.bc[0], g.bc[1]), mj = map_axis(j, g.ny, g.bc[2], g.bc[3]);
    int mk = map_axis(kk, g.nz, g.bc[4], g.bc[5]);
    idx f = (idx)(mj * g.nx + mi);
    double v = (double)cv(q[(size_t)u * (size_t)g.n + (size_t)mk * (size_t)g.plane + f]);
    if (kk < 0 && g.bc[4] == BC_INFLOW)
        v = (1.0 - (double)W[f]) * v + (double)J[(size_t)u * (size_t)g.plane + f];
    return v;
}

// velocity u_a at (i, j, kk), FP64
__device__ __forceinline__ void dvel(const QB *q, const Geom &g, const C *W, const C *J, int i, int j,
                                     int kk, double u[3])
{
    double rho = dval(q, g, W, J, i, j, kk, 0);
#pragma unroll
    for (int a = 0; a < 3; a++) u[a] = dval(q, g, W, J, i, j, kk, 1 + a) / rho;
}

__global__ void __launch_bounds__(DIAG_NT) k_diag(const QB *__restrict__ q, const S *__restrict__ sig,
                                                  Geom g, double gamma, double alpha, double dx,
                                                  const C *W, const C *J, double *part)
{
    // acc: sums of rho, mx, my, mz, E, (A s - b)^2, b^2; minima of rho, p; max |Sigma|
    double acc[DIAG_NV] = {0, 0, 0, 0, 0, 0, 0, INFINITY, INFINITY, 0};
    const double beta = alpha / (dx * dx), inv2dx = 0.5 / dx;
    for (long long c = blockIdx.x * (long long)DIAG_NT + threadIdx.x; c < g.n;
         c += (long long)gridDim.x * DIAG_NT) {
        int i = (int)(c % g.nx), j = (int)((c / g.nx) % g.ny), k = (int)(c / g.plane);
        double v[5];
#pragma unroll
        for (int u = 0; u < 5; u++) v[u] = (double)cv(q[(size_t)u * (size_t)g.n + (size_t)c]);
        double s0 = (double)cv(sig[c]);
#pragma unroll
        for (int u = 0; u < 5; u++) acc[u] += v[u];
        double p = (gamma - 1.0) * (v[4] - 0.5 * (v[1] * v[1] + v[2] * v[2] + v[3] * v[3]) / v[0]);
        acc[7] = fmin(acc[7], v[0]);
        acc[8] = fmin(acc[8], p);
        acc[9] = fmax(acc[9], fabs(s0));
        // b from central differences of u
        double G[3][3];
        const int di[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
#pragma unroll
        for (int b = 0; b < 3; b++) {
            double up[3], um[3];
            dvel(q, g, W, J, i + di[b][0], j + di[b][1], k + di[b][2], up);
            dvel(q, g, W, J, i - di[b][0], j - di[b][1], k - di[b][2], um);
#pragma unroll
            for (int a = 0; a < 3; a++) G[a][b] = (up[a] - um[a]) * inv2dx;
        }
        double tr = G[0][0] + G[1][1] + G[2][2], t2 = 0.0;
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) t2 += G[a][b] * G[b][a];
        double bv = alpha * (t2 + tr * tr);
        // A Sigma with the boundary faces of non-periodic sides dropped
        double r0 = 1.0 / v[0], diag = r0, off = 0.0;
        const int dir[6][3] = {{-1, 0, 0}, {1, 0, 0}, {0, -1, 0}, {0, 1, 0}, {0, 0, -1}, {0, 0, 1}};
        const int ext[3] = {g.nx, g.ny, g.nz}, pos[3] = {i, j, k};
#pragma unroll
        for (int f = 0; f < 6; f++) {
            int ax = f >> 1;
            int pn = pos[ax] + ((f & 1) ? 1 : -1);
            if ((pn < 0 || pn >= ext[ax]) && g.bc[f] != BC_PERIODIC) continue;
            int ni = map_axis(i + dir[f][0], g.nx, g.bc[0], g.bc[1]);
            int nj = map_axis(j + dir[f][1], g.ny, g.bc[2], g.bc[3]);
            int nk = map_axis(k + dir[f][2], g.nz, g.bc[4], g.bc[5]);
            size_t nc = (size_t)nk * (size_t)g.plane + (size_t)nj * g.nx + ni;
            double cf = 0.5 * beta * (r0 + 1.0 / (double)cv(q[nc]));
            diag += cf;
            off += cf * (double)cv(sig[nc]);
        }
        double res = diag * s0 - off - bv;
        acc[5] += res * res;
        acc[6] += bv * bv;
    }
    // block reduction in a fixed order
    __shared__ double red[DIAG_NT / 32][DIAG_NV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int t = 0; t < DIAG_NV; t++) {
        double x = acc[t];
        for (int o = 16; o > 0; o >>= 1) {
            double y = __shfl_down_sync(0xffffffffu, x, o);
            x = t < 7 ? x + y : (t < 9 ? fmin(x, y) : fmax(x, y));
        }
        if (lane == 0) red[w][t] = x;
    }
    __syncthreads();
    if (threadIdx.x < DIAG_NV) {
        int t = threadIdx.x;
        double x = red[0][t];
        for (int ww = 1; ww < DIAG_NT / 32; ww++)
            x = t < 7 ? x + red[ww][t] : (t < 9 ? fmin(x, red[ww][t]) : fmax(x, red[ww][t]));
        part[blockIdx.x * DIAG_NV + t] = x;
    }
}

// ---------------------------------------------------------------- adjoint
// Reverse of one stage (discrete adjoint with dt frozen). The faces and the
// source send their adjoints to the cells that they read in one of two ways
// (Ops::adj_rhs, Ops::adj_source and the scatter forms):
//   gather   a cell sums what the faces and cells that read it send back, in a
//            fixed order: deterministic, no atomics. Taken in FP64, and in
//            FP32 arithmetic without jets.
//   scatter  one thread per face or cell adds to the cells it read by atomics
//            (36 per face and 36 per cell of the source). Kept in FP32
//            arithmetic with jets, where it takes 9.3 ms for a step of 128^3
//            and four jets: its order of additions is not fixed, and dJ/dw, a
//            double summed from these FP32 values with cancellation, moves with
//            it, by 1e-8 to 1.3e-7 between two runs (median 3e-8) and by up to
//            8e-8 in the mean between two allocations of the same buffers. The
//            gather (2.6 ms) repeats its bits but moves dJ/dw by 0.6e-7 to
//            2.5e-7 and is less exact for some states (against FP64 3.3e-7 where
//            the scatter has 2.2e-7, 1.1e-7 where it has 0.5e-7).
// The reversed sweeps gather in both. Adjoint values are in the arithmetic
// type C. Non-smooth points follow the forward's branch: the LF speed
// max(aL, aR) sends its adjoint to the side the forward took (aR on a tie),
// |u| takes sign(u) with sign(0) = 0.

__device__ __forceinline__ void aadd(float *p, float v) { atomicAdd(p, v); }
__device__ __forceinline__ void aadd(double *p, double v) { atomicAdd(p, v); }

// forward value of field u (0..4 conserved, 5 Sigma) read at (i, j, kk):
// index mapping plus the jet blend of the -z inflow face
__device__ __forceinline__ C val_at(const S *q, const S *sig, const Geom &g, const C *W, const C *J,
                                    int i, int j, int kk, int u)
{
    int mi = map_axis(i, g.nx, g.bc[0], g.bc[1]), mj = map_axis(j, g.ny, g.bc[2], g.bc[3]);
    int mk = map_axis(kk, g.nz, g.bc[4], g.bc[5]);
    idx f = ck((idx)(mj * g.nx + mi), g.plane);
    idx c = ck((idx)mk * (idx)g.plane + f, g.n);
    if (u == 5) return ldc(sig + c);
    C v = ldc(q + ckl((size_t)u * (size_t)g.n + c, 5 * g.n));
    if (kk < 0 && g.bc[4] == BC_INFLOW)
        v = (C(1) - W[f]) * v + J[ckl((size_t)u * (size_t)g.plane + f, 5 * g.plane)];
    return v;
}

// adjoint of that read: scatter `a` back to the cell(s) the value came from
__device__ __forceinline__ void scatter_at(C *lq, C *lsig, C *lamJ, const Geom &g, const C *W, int i,
                                           int j, int kk, int u, C a)
{
    int mi = map_axis(i, g.nx, g.bc[0], g.bc[1]), mj = map_axis(j, g.ny, g.bc[2], g.bc[3]);
    int mk = map_axis(kk, g.nz, g.bc[4], g.bc[5]);
    idx f = ck((idx)(mj * g.nx + mi), g.plane);
    idx c = ck((idx)mk * (idx)g.plane + f, g.n);
    if (u == 5) {
        aadd(lsig + c, a);
        return;
    }
    const size_t qc = ckl((size_t)u * (size_t)g.n + c, 5 * g.n);
    if (kk < 0 && g.bc[4] == BC_INFLOW) {
        aadd(lq + qc, (C(1) - W[f]) * a);
        aadd(lamJ + ckl((size_t)u * (size_t)g.plane + f, 5 * g.plane), a);
        return;
    }
    aadd(lq + qc, a);
}

__global__ void k_adj_rk(const C *lout, C *lq0, C *lqs, C *Lb, long long n5, C w, C dt)
{
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n5;
         c += (long long)gridDim.x * blockDim.x) {
        C a = lout[c];
        lq0[c] += (C(1) - w) * a;
        lqs[c] = w * a;
        Lb[c] = w * dt * a;
    }
}

// reverse of the physical flux along D at a face state v = (rho, m, E) and
// Sigma s: Fb (adjoint of F) and ab (adjoint of |u_D| + c) into vb, sb
template <int D>
__device__ __forceinline__ void flux_rev_at(const C v[5], C s, const C Fb[5], C ab, C gamma, C vb[5], C &sb)
{
    C rho = v[0], E = v[4], r = C(1) / rho;
    C u[3] = {v[1] * r, v[2] * r, v[3] * r};
    C ke = C(0.5) * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    C p = (gamma - C(1)) * (E - ke);
    C P = p + s;
    C c = sqrt(gamma * p * r);
    C ub[3] = {C(0), C(0), C(0)}, rhob = C(0), Eb = C(0), Pb = C(0), pb = C(0);
    rhob += Fb[0] * u[D];
    ub[D] += Fb[0] * rho;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        vb[1 + a] += Fb[1 + a] * u[D];
        ub[D] += Fb[1 + a] * v[1 + a];
    }
    Pb += Fb[1 + D] + Fb[4] * u[D];
    Eb += Fb[4] * u[D];
    ub[D] += Fb[4] * (E + P);
    ub[D] += ab * (u[D] > C(0) ? C(1) : (u[D] < C(0) ? C(-1) : C(0)));
    pb += ab * gamma / (C(2) * c * rho);
    rhob -= ab * c / (C(2) * rho);
    pb += Pb;
    sb += Pb;
    Eb += (gamma - C(1)) * pb;
    C keb = -(gamma - C(1)) * pb;
    rhob += keb * C(0.5) * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
#pragma unroll
    for (int a = 0; a < 3; a++) ub[a] += keb * rho * u[a];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        vb[1 + a] += ub[a] * r;
        rhob -= ub[a] * u[a] * r;
    }
    vb[0] += rhob;
    vb[4] += Eb;
}

template <int D>
__device__ __forceinline__ C fwd_flux(const C v[5], C s, C gamma, C F[5])
{
    C rho = v[0], E = v[4], r = C(1) / rho;
    C u[3] = {v[1] * r, v[2] * r, v[3] * r};
    C p = (gamma - C(1)) * (E - C(0.5) * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
    C P = p + s;
    F[0] = rho * u[D];
#pragma unroll
    for (int a = 0; a < 3; a++) F[1 + a] = v[1 + a] * u[D] + (a == D ? P : C(0));
    F[4] = (E + P) * u[D];
    return fabs(u[D]) + sqrt(gamma * p * r);
}

// one thread per face normal to D: face f sits between cells f-1 and f
template <int D>
__global__ void k_adj_rhs_scatter(const S *q, const S *sig, const C *Lb, C *lq, C *lsig, C *lamJ, Geom g, C gamma,
                          C inv_dx, const C *W, const C *J)
{
    const int nf[3] = {g.nx + (D == 0), g.ny + (D == 1), g.nz + (D == 2)};
    const int nd = D == 0 ? g.nx : D == 1 ? g.ny : g.nz;
    const long long total = (long long)nf[0] * nf[1] * nf[2];
    const C cl[6] = {C(2.0 / 60), C(-13.0 / 60), C(47.0 / 60), C(27.0 / 60), C(-3.0 / 60), C(0)};
    const C cr[6] = {C(0), C(-3.0 / 60), C(27.0 / 60), C(47.0 / 60), C(-13.0 / 60), C(2.0 / 60)};
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        int c3[3];
        c3[0] = (int)(t % nf[0]);
        c3[1] = (int)((t / nf[0]) % nf[1]);
        c3[2] = (int)(t / ((long long)nf[0] * nf[1]));
        const int f = c3[D];
        C Fb[5];
#pragma unroll
        for (int u = 0; u < 5; u++) {
            C hi = C(0), lo = C(0);
            if (f < nd) hi = Lb[ckl((size_t)u * g.n + ((size_t)c3[2] * g.ny + c3[1]) * g.nx + c3[0], 5 * g.n)];
            if (f >= 1) {
                int cc[3] = {c3[0], c3[1], c3[2]};
                cc[D] = f - 1;
                lo = Lb[ckl((size_t)u * g.n + ((size_t)cc[2] * g.ny + cc[1]) * g.nx + cc[0], 5 * g.n)];
            }
            Fb[u] = (hi - lo) * inv_dx;
        }
        C sv[6][6];
#pragma unroll
        for (int m = 0; m < 6; m++) {
            int cc[3] = {c3[0], c3[1], c3[2]};
            cc[D] += m - 3;
#pragma unroll
            for (int u = 0; u < 6; u++) sv[m][u] = val_at(q, sig, g, W, J, cc[0], cc[1], cc[2], u);
        }
        C L[6], R[6];
#pragma unroll
        for (int u = 0; u < 6; u++) {
            L[u] = rec_left(sv[0][u], sv[1][u], sv[2][u], sv[3][u], sv[4][u]);
            R[u] = rec_right(sv[1][u], sv[2][u], sv[3][u], sv[4][u], sv[5][u]);
        }
        C FL[5], FR[5];
        C aL = fwd_flux<D>(L, L[5], gamma, FL);
        C aR = fwd_flux<D>(R, R[5], gamma, FR);
        C lam = aL > aR ? aL : aR;
        C Lbv[5] = {C(0), C(0), C(0), C(0), C(0)}, Rbv[5] = {C(0), C(0), C(0), C(0), C(0)};
        C FLb[5], FRb[5], lamb = C(0);
#pragma unroll
        for (int u = 0; u < 5; u++) {
            FLb[u] = C(0.5) * Fb[u];
            FRb[u] = C(0.5) * Fb[u];
            Lbv[u] += C(0.5) * lam * Fb[u];
            Rbv[u] -= C(0.5) * lam * Fb[u];
            lamb -= C(0.5) * (R[u] - L[u]) * Fb[u];
        }
        C sLb = C(0), sRb = C(0);
        flux_rev_at<D>(L, L[5], FLb, aL > aR ? lamb : C(0), gamma, Lbv, sLb);
        flux_rev_at<D>(R, R[5], FRb, aL > aR ? C(0) : lamb, gamma, Rbv, sRb);
#pragma unroll
        for (int m = 0; m < 6; m++) {
            int cc[3] = {c3[0], c3[1], c3[2]};
            cc[D] += m - 3;
#pragma unroll
            for (int u = 0; u < 5; u++) {
                C a = cl[m] * Lbv[u] + cr[m] * Rbv[u];
                if (a != C(0)) scatter_at(lq, lsig, lamJ, g, W, cc[0], cc[1], cc[2], u, a);
            }
            C a = cl[m] * sLb + cr[m] * sRb;
            if (a != C(0)) scatter_at(lq, lsig, lamJ, g, W, cc[0], cc[1], cc[2], 5, a);
        }
    }
}

__global__ void k_adj_rho(const S *q, C *rb, C *lqs, long long n)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        C rho = ldc(q + t);
        lqs[t] -= rb[t] / (rho * rho);
    }
}

// reverse of the source at one cell: lambda_b -> u at the 6 neighbours -> (rho, m) there
__global__ void k_adj_source_scatter(const S *q, const C *lb, C *lq, C *lamJ, Geom g, C alpha, C inv2dx, const C *W,
                             const C *J)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.n;
         t += (long long)gridDim.x * blockDim.x) {
        C bb = lb[t];
        if (bb == C(0)) continue;
        int i = (int)(t % g.nx), j = (int)((t / g.nx) % g.ny), k = (int)(t / g.plane);
        C rho[2][3], m[2][3][3], u[2][3][3];  // [+/-][direction][component]
        for (int c = 0; c < 3; c++)
            for (int sgn = 0; sgn < 2; sgn++) {
                int cc[3] = {i, j, k};
                cc[c] += sgn == 0 ? 1 : -1;
                rho[sgn][c] = val_at(q, nullptr, g, W, J, cc[0], cc[1], cc[2], 0);
                for (int a = 0; a < 3; a++) {
                    m[sgn][c][a] = val_at(q, nullptr, g, W, J, cc[0], cc[1], cc[2], 1 + a);
                    u[sgn][c][a] = m[sgn][c][a] / rho[sgn][c];
                }
            }
        C G[3][3];
        for (int a = 0; a < 3; a++)
            for (int c = 0; c < 3; c++) G[a][c] = (u[0][c][a] - u[1][c][a]) * inv2dx;
        C tr = G[0][0] + G[1][1] + G[2][2];
        for (int c = 0; c < 3; c++)
            for (int a = 0; a < 3; a++) {
                C Gb = alpha * (C(2) * G[c][a] + (a == c ? C(2) * tr : C(0))) * bb;
                C ub = Gb * inv2dx;
                for (int sgn = 0; sgn < 2; sgn++) {
                    C us = sgn == 0 ? ub : -ub;
                    int cc[3] = {i, j, k};
                    cc[c] += sgn == 0 ? 1 : -1;
                    C r = rho[sgn][c];
                    scatter_at(lq, nullptr, lamJ, g, W, cc[0], cc[1], cc[2], 1 + a, us / r);
                    scatter_at(lq, nullptr, lamJ, g, W, cc[0], cc[1], cc[2], 0, -us * m[sgn][c][a] / (r * r));
                }
            }
    }
}

// forward value of field u (0..4 conserved, 5 Sigma) at mapped in-plane
// offset f and plane kk: index mapping in z plus the jet blend of the -z
// inflow face
__device__ __forceinline__ C val_col(const S *q, const S *sig, const Geom &g, const C *W, const C *J, idx f, int kk,
                                     int u)
{
    const idx c = ck((idx)zmap(kk, g) * (idx)g.plane + f, g.n);
    if (u == 5) return ldc(sig + c);
    C v = ldc(q + ckl((size_t)u * (size_t)g.n + c, 5 * g.n));
    if (kk < 0 && g.bc[4] == BC_INFLOW)
        v = (C(1) - W[ck(f, g.plane)]) * v + J[ckl((size_t)u * (size_t)g.plane + f, 5 * g.plane)];
    return v;
}

// a face state's primitives: 1 / rho, u, p and the sound speed
struct Prim {
    C r, u[3], p, c;
};
__device__ __forceinline__ Prim prim_of(const C (&v)[6], C gamma)
{
    Prim w;
    w.r = C(1) / v[0];
    C ke = C(0);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        w.u[a] = v[1 + a] * w.r;
        ke += v[1 + a] * w.u[a];
    }
    w.p = (gamma - C(1)) * (v[4] - C(0.5) * ke);
    w.c = sqrt(gamma * w.p * w.r);
    return w;
}

// reverse of the physical flux along D at a face state v = (rho, m, E, Sigma)
// with primitives w: Fb (adjoint of F) and the adjoints pb, rhob, uDb that
// p, rho and u_D have besides (from the wave speed), added to vb
template <int D>
__device__ __forceinline__ void flux_rev(const C (&v)[6], const Prim &w, const C (&Fb)[5], C pb, C rhob, C uDb,
                                         C gamma, C (&vb)[6])
{
    C ub[3] = {C(0), C(0), C(0)};
    ub[D] = uDb + Fb[0] * v[0];
    rhob += Fb[0] * w.u[D];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        vb[1 + a] += Fb[1 + a] * w.u[D];
        ub[D] += Fb[1 + a] * v[1 + a];
    }
    const C Pb = Fb[1 + D] + Fb[4] * w.u[D];
    ub[D] += Fb[4] * (v[4] + (w.p + v[5]));
    pb += Pb;
    vb[5] += Pb;
    const C keb = -(gamma - C(1)) * pb;
    vb[4] += Fb[4] * w.u[D] - keb;
    C uu = C(0);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        ub[a] += keb * v[1 + a];
        uu += w.u[a] * w.u[a];
    }
    rhob += keb * C(0.5) * uu;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const C mb = ub[a] * w.r;
        vb[1 + a] += mb;
        rhob -= mb * w.u[a];
    }
    vb[0] += rhob;
}

// Reverse of one face along D: from the six cells s it reads (cell, field)
// and the adjoint Fb of its flux, the adjoints Lb, Rb of its two face values
template <int D>
__device__ __forceinline__ void face_rev(const C (&s)[6][6], const C (&Fb)[5], C gamma, C (&Lb)[6], C (&Rb)[6])
{
    C L[6], R[6];
#pragma unroll
    for (int u = 0; u < 6; u++) {
        L[u] = rec_left(s[0][u], s[1][u], s[2][u], s[3][u], s[4][u]);
        R[u] = rec_right(s[1][u], s[2][u], s[3][u], s[4][u], s[5][u]);
    }
    const Prim l = prim_of(L, gamma), r = prim_of(R, gamma);
    const C aL = fabs(l.u[D]) + l.c, aR = fabs(r.u[D]) + r.c;
    const bool left = aL > aR;
    const C lam = left ? aL : aR;
    C FLb[5], lamb = C(0);
#pragma unroll
    for (int u = 0; u < 5; u++) {
        FLb[u] = C(0.5) * Fb[u];
        Lb[u] = C(0.5) * lam * Fb[u];
        Rb[u] = -Lb[u];
        lamb -= C(0.5) * (R[u] - L[u]) * Fb[u];
    }
    Lb[5] = Rb[5] = C(0);
    // the wave speed's adjoint goes to the side it came from
    const C c = left ? l.c : r.c, ri = left ? l.r : r.r, uD = left ? l.u[D] : r.u[D];
    const C pb = lamb * gamma * ri / (C(2) * c), rhob = -lamb * c * ri * C(0.5);
    const C uDb = lamb * (uD > C(0) ? C(1) : (uD < C(0) ? C(-1) : C(0)));
    flux_rev<D>(L, l, FLb, left ? pb : C(0), left ? rhob : C(0), left ? uDb : C(0), gamma, Lb);
    flux_rev<D>(R, r, FLb, left ? C(0) : pb, left ? C(0) : rhob, left ? C(0) : uDb, gamma, Rb);
}
// weight of cell m (0..5) of a face's stencil in its left and right value
__device__ __forceinline__ C w_left(int m)
{
    return m == 0 ? C(2.0 / 60) : m == 1 ? C(-13.0 / 60) : m == 2 ? C(47.0 / 60) : m == 3 ? C(27.0 / 60) : m == 4 ? C(-3.0 / 60) : C(0);
}
__device__ __forceinline__ C w_right(int m) { return w_left(5 - m); }

// The stage combination's reverse and the x-faces': with lout the adjoint of
// the stage's output, lqs (the adjoint of its input) starts as w lout, lq0
// (of the step's input) gains (1 - w) lout, and L's adjoint is w dt lout
// (wdt = w dt); then every cell gathers from the six x-faces that read it. A
// warp takes 32 consecutive faces of a row (each loads its six cells; the
// next lanes' loads hit the same lines) and gathers by shuffles for the 27
// cells whose faces it has. Faces of a periodic row wrap; of another row
// there are faces 0..nx, and the three cells past each end, which stand for
// the end cell, are summed into it by the warp that has them all.
constexpr int XCELLS = 27, XWARPS = 4;
__global__ void __launch_bounds__(32 * XWARPS) k_adj_rhs_x(const S *q, const S *sig, const C *lout, C *lqs, C *lq0,
                                                           C *lsig, Geom g, C gamma, C inv_dx, C w, C wdt, int first,
                                                           int nseg)
{
    const unsigned wid = blockIdx.x * XWARPS + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31, seg = (int)(wid % nseg);
    const idx row = wid / nseg;
    if (row >= (idx)g.ny * (idx)g.nz) return;
    const idx base = row * (idx)g.nx;
    const int n = g.nx;
    const bool per = g.bc[0] == BC_PERIODIC;
    int c0, c1, fs;  // cells of this warp, its first face
    if (per) {
        c0 = XCELLS * seg;
        c1 = min(n, c0 + XCELLS);
        fs = c0 - 2;
    } else {
        const bool last = seg == nseg - 1;
        c0 = last ? min(XCELLS * seg - 3, n - 1) : XCELLS * seg - 3;
        c1 = last ? n + 3 : min(c0 + XCELLS, n - 1);
        fs = last ? n + 3 - XCELLS - 2 : c0 - 2;
        if (last && nseg == 1) c0 = -3;
    }
    const int f = fs + lane;
    C Lb[6], Rb[6];
#pragma unroll
    for (int u = 0; u < 6; u++) Lb[u] = Rb[u] = C(0);
    if (per || (f >= 0 && f <= n)) {
        C s[6][6], Fb[5];
#pragma unroll
        for (int m = 0; m < 6; m++) {
            const idx c = ck(base + (idx)map_axis(f - 3 + m, n, g.bc[0], g.bc[1]), g.n);
#pragma unroll
            for (int u = 0; u < 5; u++) s[m][u] = ldc(q + ckl((size_t)u * (size_t)g.n + c, 5 * g.n));
            s[m][5] = ldc(sig + c);
        }
        const idx ch = ck(base + (idx)map_axis(f, n, g.bc[0], g.bc[1]), g.n);
        const idx cl = ck(base + (idx)map_axis(f - 1, n, g.bc[0], g.bc[1]), g.n);
#pragma unroll
        for (int u = 0; u < 5; u++) {
            const C hi = per || f < n ? wdt * lout[ckl((size_t)u * (size_t)g.n + ch, 5 * g.n)] : C(0);
            const C lo = per || f >= 1 ? wdt * lout[ckl((size_t)u * (size_t)g.n + cl, 5 * g.n)] : C(0);
            Fb[u] = (hi - lo) * inv_dx;
        }
        face_rev<0>(s, Fb, gamma, Lb, Rb);
    }
    // lane l gathers for cell f = fs + l, on top of what the cell has: its
    // faces are those of lanes l + 3 .. l - 2
    const bool in = lane >= 2 && lane <= 28 && f >= max(c0, 0) && f < min(c1, n);
    const idx c = in ? ck(base + (idx)f, g.n) : 0;
    C v[6], a0[5];
#pragma unroll
    for (int u = 0; u < 5; u++) {
        a0[u] = in ? lout[ckl((size_t)u * (size_t)g.n + c, 5 * g.n)] : C(0);
        v[u] = w * a0[u];
    }
    v[5] = in ? lsig[c] : C(0);
#pragma unroll
    for (int m = 0; m < 6; m++)
#pragma unroll
        for (int u = 0; u < 6; u++)
            v[u] += w_left(m) * __shfl_sync(0xffffffffu, Lb[u], (lane + 3 - m) & 31) +
                    w_right(m) * __shfl_sync(0xffffffffu, Rb[u], (lane + 3 - m) & 31);
    if (!per && (seg == 0 || seg == nseg - 1)) {  // the cells past the ends
#pragma unroll
        for (int u = 0; u < 6; u++) {
            C lo = C(0), hi = C(0);
#pragma unroll
            for (int m = 1; m <= 3; m++) {
                lo += __shfl_sync(0xffffffffu, v[u], (lane - m) & 31);
                hi += __shfl_sync(0xffffffffu, v[u], (lane + m) & 31);
            }
            if (f == 0) v[u] += lo;
            if (f == n - 1) v[u] += hi;
        }
    }
    if (!in) return;
#pragma unroll
    for (int u = 0; u < 5; u++) {
        const size_t at = ckl((size_t)u * (size_t)g.n + c, 5 * g.n);
        lqs[at] = v[u];
        lq0[at] = first ? (C(1) - w) * a0[u] : lq0[at] + (C(1) - w) * a0[u];
    }
    lsig[c] = v[5];
}

// The y- and z-faces' reverse, and in FP64 the x-faces' of short rows: a thread
// marches along D over a chunk of cells of one line (lanes along x, then the next
// line; along D = 0 a row per lane), with the six cells of the face's stencil and
// the sums of the six cells it sends to; a cell is written when the last face that
// reads it is done. A chunk also evaluates the two faces before and after it that
// reach its cells. Ends as for the x-faces; the cells below an inflow face send to
// the cell above it (1 - W) and to the inflow tables (lamJ). Along x it does the
// stage combination's reverse as well. Not all of the sums are in registers: the
// ends' additions index them, so one 6 x 6 array and `below` are in local memory
// (stack frame: FP64 288 bytes along y, 656 along z; FP32 144 and 336).
template <int D>
__global__ void __launch_bounds__(128) k_adj_rhs_march(const S *q, const S *sig, const C *lout, C *lqs, C *lsig,
                                                       C *lq0, C *lamJ, Geom g, C gamma, C inv_dx, C w, C wdt,
                                                       int first, const C *W, const C *J, int chunk)
{
    const unsigned t = blockIdx.x * 128u + threadIdx.x, line = D == 0 ? t : t / (unsigned)g.nx,
                   i = D == 0 ? 0u : t - line * (unsigned)g.nx;
    if (line >= (unsigned)(D == 0 ? (idx)g.ny * (idx)g.nz : D == 1 ? g.nz : g.ny)) return;
    const int n = D == 0 ? g.nx : D == 1 ? g.ny : g.nz, blo = g.bc[2 * D], bhi = g.bc[2 * D + 1];
    const bool per = blo == BC_PERIODIC, jet = D == 2 && blo == BC_INFLOW;
    const idx step = D == 0 ? 1u : D == 1 ? (idx)g.nx : (idx)g.plane;
    const idx base = (idx)line * (D == 1 ? (idx)g.plane : (idx)g.nx) + (idx)i;
    const int c0 = blockIdx.y * chunk, c1 = min(n, c0 + chunk);
    const int f0 = per ? c0 - 2 : max(0, c0 - 2), f1 = per ? c1 + 2 : min(n, c1 + 2);
    auto cell = [&](int c) { return ck(base + (idx)map_axis(c, n, blo, bhi) * step, g.n); };
    auto value = [&](int c, C (&s)[6]) {
        const idx at = cell(c);
#pragma unroll
        for (int u = 0; u < 5; u++) s[u] = ldc(q + ckl((size_t)u * (size_t)g.n + at, 5 * g.n));
        s[5] = ldc(sig + at);
        if (jet && c < 0) {
            const C wf = C(1) - W[ck(base, g.plane)];
#pragma unroll
            for (int u = 0; u < 5; u++) s[u] = wf * s[u] + J[ckl((size_t)u * (size_t)g.plane + base, 5 * g.plane)];
        }
    };
    auto adjoint = [&](int c, C (&l)[5]) {
        const bool in = per || (c >= 0 && c < n);
        const idx at = cell(c);
#pragma unroll
        for (int u = 0; u < 5; u++) l[u] = in ? wdt * lout[ckl((size_t)u * (size_t)g.n + at, 5 * g.n)] : C(0);
    };
    // what the cell has so far (0 for one that this thread does not write)
    auto begin = [&](int c, C (&v)[6]) {
        const bool mine = c >= c0 && c < c1;
        const idx at = mine ? cell(c) : 0;
#pragma unroll
        for (int u = 0; u < 5; u++) {
            const size_t a = ckl((size_t)u * (size_t)g.n + at, 5 * g.n);
            v[u] = !mine ? C(0) : D == 0 ? w * lout[a] : lqs[a];
            if (D == 0 && mine) lq0[a] = first ? (C(1) - w) * lout[a] : lq0[a] + (C(1) - w) * lout[a];
        }
        v[5] = mine ? lsig[at] : C(0);
    };
    auto write = [&](int c, const C (&v)[6]) {
        if (c < c0 || c >= c1) return;
        const idx at = cell(c);
#pragma unroll
        for (int u = 0; u < 5; u++) lqs[ckl((size_t)u * (size_t)g.n + at, 5 * g.n)] = v[u];
        lsig[at] = v[5];
    };
    const C wf = jet ? C(1) - W[ck(base, g.plane)] : C(1);
    // From the last face down: a cell then gathers from the face three above
    // it first and the face two below it last, as from the x-faces.
    C s[6][6], acc[6][6], hi[5];
#pragma unroll
    for (int m = 1; m < 6; m++) {
        value(f1 - 3 + m, s[m]);
        begin(f1 - 3 + m, acc[m]);
    }
    adjoint(f1, hi);
    C below[3][3][5];  // what the faces 0..2 send below an inflow face's first cell
    for (int f = f1; f >= f0; f--) {
        C lo[5], Fb[5], Lb[6], Rb[6];
        value(f - 3, s[0]);
        begin(f - 3, acc[0]);
        adjoint(f - 1, lo);
#pragma unroll
        for (int u = 0; u < 5; u++) {
            Fb[u] = (hi[u] - lo[u]) * inv_dx;
            hi[u] = lo[u];
        }
        face_rev<D>(s, Fb, gamma, Lb, Rb);
        auto sent = [&](int m, int u) { return w_left(m) * Lb[u] + w_right(m) * Rb[u]; };
        if (!per && f < 3) {  // cells below the line's end: f - 3 .. -1, which stand for cell 0 = f - 3 + e
#pragma unroll
            for (int e = 1; e <= 3; e++)
                if (e == 3 - f) {
#pragma unroll
                    for (int m = 0; m < e; m++)
#pragma unroll
                        for (int u = 0; u < 6; u++) {
                            const C a = sent(m, u);
                            acc[e][u] += u < 5 ? wf * a : a;
                            if (jet && u < 5) below[3 - e][m][u] = a;
                        }
                }
        }
#pragma unroll
        for (int m = 0; m < 6; m++)
#pragma unroll
            for (int u = 0; u < 6; u++) acc[m][u] += sent(m, u);
        if (!per && f > n - 3) {  // cells past the end: n .. f + 2, which stand for cell n - 1 = f - 3 + e
#pragma unroll
            for (int e = 2; e <= 4; e++)
                if (e == n - 1 - f + 3) {
#pragma unroll
                    for (int m = e + 1; m < 6; m++)
#pragma unroll
                        for (int u = 0; u < 6; u++) acc[e][u] += sent(m, u);
                }
        }
        write(f + 2, acc[5]);  // no face below reads this cell
        if (f > f0) {
#pragma unroll
            for (int m = 5; m > 0; m--)
#pragma unroll
                for (int u = 0; u < 6; u++) {
                    s[m][u] = s[m - 1][u];
                    acc[m][u] = acc[m - 1][u];
                }
        }
    }
    if (!per && f0 == 0) {  // below the first face: cells 1 and 0
        write(1, acc[4]);
        write(0, acc[3]);
    }
    if (jet && c0 == 0) {
#pragma unroll
        for (int u = 0; u < 5; u++) {
            const size_t at = ckl((size_t)u * (size_t)g.plane + base, 5 * g.plane);
            C v = lamJ[at];
#pragma unroll
            for (int m = 0; m < 3; m++)
#pragma unroll
                for (int f = 0; f < 3 - m; f++) v += below[f][m][u];
            lamJ[at] = v;
        }
    }
}

// neighbour of the cell at (i, j, k) across face d (0: -x .. 5: +z); false on
// a non-periodic domain boundary (no face term there)
__device__ __forceinline__ bool nbr(const Geom &g, int i, int j, int k, int d, idx &out)
{
    int c[3] = {i, j, k}, n[3] = {g.nx, g.ny, g.nz};
    int ax = d >> 1;
    c[ax] += (d & 1) ? 1 : -1;
    if (c[ax] < 0 || c[ax] >= n[ax]) {
        if (g.bc[d] != BC_PERIODIC) return false;
        c[ax] = c[ax] < 0 ? c[ax] + n[ax] : c[ax] - n[ax];
    }
    out = ck(((idx)c[2] * (idx)g.ny + (idx)c[1]) * (idx)g.nx + (idx)c[0], g.n);
    return true;
}
// cell-wise kernels: 32 x 4 cells of a plane per block
constexpr int CBX = 32, CBY = 4;
__device__ __forceinline__ bool cell_of(const Geom &g, int &i, int &j, int &k, idx &t)
{
    const unsigned gx = ((unsigned)g.nx + CBX - 1) / CBX, gy = ((unsigned)g.ny + CBY - 1) / CBY;
    const unsigned rest = blockIdx.x / gx;
    i = (int)(blockIdx.x % gx) * CBX + (int)threadIdx.x;
    j = (int)(rest % gy) * CBY + (int)threadIdx.y;
    k = (int)(rest / gy);
    t = ((idx)k * (idx)g.ny + (idx)j) * (idx)g.nx + (idx)i;
    return i < g.nx && j < g.ny;
}

// r = 1 / rho, the diagonal D of the sweeps and, in FP64, its inverse, once per
// stage. mu = lsig / D is the division's rounding in both (quot): seven divisions
// per cell and sweep would hold the FP64 units.
__device__ __forceinline__ float mu_of(const float *l, const float *d, const float *, idx t) { return l[t] / d[t]; }
__device__ __forceinline__ double mu_of(const double *l, const double *d, const double *inv, idx t)
{
    return quot(l[t], d[t], inv[t]);
}
__global__ void __launch_bounds__(CBX *CBY) k_adj_diag(const S *q, C *r, C *dg, C *dinv, Geom g, C beta)
{
    int i, j, k;
    idx t;
    if (!cell_of(g, i, j, k, t)) return;
    const C ri = C(1) / ldc(q + t);
    C diag = ri;
#pragma unroll
    for (int d = 0; d < 6; d++) {
        idx m;
        if (nbr(g, i, j, k, d, m)) diag += beta * C(0.5) * (ri + C(1) / ldc(q + m));
    }
    r[t] = ri;
    dg[t] = diag;
    if (sizeof(C) == 8) dinv[t] = C(1) / diag;
}

// One reversed Jacobi sweep s_k -> F, gathered (the neighbour relation is
// symmetric): with mu = lsig / D (lsig the adjoint of F),
//   nl_m = sum_i beta c_im mu_i (the adjoint of s_k), lb_m += mu_m,
//   rb_m += mu_m (beta/2 sum s_nb - F_m (1 + beta nf/2)) + sum_i mu_i beta/2 (s_m - F_i);
// the neighbours' mu are formed again from lsig and D, which saves a pass.
__global__ void __launch_bounds__(CBX *CBY) k_adj_jacobi(const C *__restrict__ r, const C *__restrict__ dg,
                                                         const C *__restrict__ dinv, const S *__restrict__ sk, const S *__restrict__ F,
                                                         const C *__restrict__ lsig, C *nl, C *lb, C *rb, Geom g,
                                                         C beta, int first)
{
    int i, j, k;
    idx t;
    if (!cell_of(g, i, j, k, t)) return;
    const C rm = r[t], sm = ldc(sk + t), Fm = ldc(F + t), mum = mu_of(lsig, dg, dinv, t), hb = C(0.5) * beta;
    C acc = C(0), ssum = C(0), rbm = C(0);
    int nfc = 0;
#pragma unroll
    for (int d = 0; d < 6; d++) {
        idx n;
        if (!nbr(g, i, j, k, d, n)) continue;
        const C mun = mu_of(lsig, dg, dinv, n);
        acc += hb * (rm + r[n]) * mun;
        ssum += ldc(sk + n);
        nfc++;
        rbm += mun * hb * (sm - ldc(F + n));
    }
    rbm += mum * (hb * ssum - Fm * (C(1) + hb * C(nfc)));
    nl[t] = acc;
    lb[t] = first ? mum : lb[t] + mum;
    rb[t] = first ? rbm : rb[t] + rbm;
}

// Reverse of the source, first pass: the adjoints of the nine gradients of u
// at each cell, Gb[a][c] = alpha (2 G_ca + 2 delta_ac tr G) lb / (2 dx)
struct Grads {
    C *p[9];
};
__global__ void __launch_bounds__(CBX *CBY) k_adj_grad(const S *q, const C *__restrict__ r, const C *lb, Grads out,
                                                       Geom g, C alpha, C inv2dx, const C *W, const C *J)
{
    int i, j, k;
    idx t;
    if (!cell_of(g, i, j, k, t)) return;
    const C bb = lb[t];
    C G[3][3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        C u[2][3];
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int ii = i + (c == 0 ? 1 - 2 * s : 0), jj = j + (c == 1 ? 1 - 2 * s : 0),
                      kk = k + (c == 2 ? 1 - 2 * s : 0);
            const idx f = (idx)map_axis(jj, g.ny, g.bc[2], g.bc[3]) * (idx)g.nx + (idx)map_axis(ii, g.nx, g.bc[0], g.bc[1]);
            C ri;
            if (kk < 0 && g.bc[4] == BC_INFLOW)
                ri = C(1) / val_col(q, nullptr, g, W, J, f, kk, 0);
            else
                ri = r[ck((idx)zmap(kk, g) * (idx)g.plane + f, g.n)];
#pragma unroll
            for (int a = 0; a < 3; a++) u[s][a] = val_col(q, nullptr, g, W, J, f, kk, 1 + a) * ri;
        }
#pragma unroll
        for (int a = 0; a < 3; a++) G[a][c] = (u[0][a] - u[1][a]) * inv2dx;
    }
    const C tr = G[0][0] + G[1][1] + G[2][2], s = alpha * bb * inv2dx;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int c = 0; c < 3; c++) out.p[3 * a + c][t] = s * (C(2) * G[c][a] + (a == c ? C(2) * tr : C(0)));
}
// Second pass: a cell's u is the upper value of the gradient of the cell below
// it and the lower one of the cell above; at a boundary the cell's own
// gradient reads it (or, below an inflow face, the blend of it) as the ghost.
// Then u to (rho, m), and the sweeps' adjoint rb of 1/rho to rho.
__global__ void __launch_bounds__(CBX *CBY) k_adj_source(const S *q, const C *__restrict__ r, const C *rb, Grads G,
                                                         C *lq, C *lamJ, Geom g, const C *W, const C *J)
{
    int i, j, k;
    idx t;
    if (!cell_of(g, i, j, k, t)) return;
    const C ri = r[t];
    const bool jet = k == 0 && g.bc[4] == BC_INFLOW;
    C v[4], m[3], mg[3], rg = C(0), wf = C(0), lj[4];
#pragma unroll
    for (int f = 0; f < 4; f++) v[f] = lq[ckl((size_t)f * (size_t)g.n + t, 5 * g.n)];
#pragma unroll
    for (int a = 0; a < 3; a++) m[a] = ldc(q + ckl((size_t)(1 + a) * (size_t)g.n + t, 5 * g.n));
    if (jet) {
        rg = C(1) / val_col(q, nullptr, g, W, J, t, -1, 0);
        wf = C(1) - W[ck(t, g.plane)];
#pragma unroll
        for (int a = 0; a < 3; a++) mg[a] = val_col(q, nullptr, g, W, J, t, -1, 1 + a);
#pragma unroll
        for (int f = 0; f < 4; f++) lj[f] = lamJ[ckl((size_t)f * (size_t)g.plane + t, 5 * g.plane)];
    }
    v[0] -= rb[t] * ri * ri;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        idx lo = t, hi = t;
        const bool has_lo = nbr(g, i, j, k, 2 * c, lo), has_hi = nbr(g, i, j, k, 2 * c + 1, hi);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const C *p = G.p[3 * a + c];
            // adjoint us of this cell's u_a, added as that of (rho, m_a)
            auto add = [&](C us) {
                const C mb = us * ri;
                v[1 + a] += mb;
                v[0] -= mb * m[a] * ri;
            };
            add(has_hi ? -p[hi] : p[t]);
            if (c == 2 && jet) {
                const C mb = -p[t] * rg, rhob = -mb * mg[a] * rg;
                v[1 + a] += wf * mb;
                v[0] += wf * rhob;
                lj[1 + a] += mb;
                lj[0] += rhob;
            } else {
                add(has_lo ? p[lo] : -p[t]);
            }
        }
    }
#pragma unroll
    for (int f = 0; f < 4; f++) {
        lq[ckl((size_t)f * (size_t)g.n + t, 5 * g.n)] = v[f];
        if (jet) lamJ[ckl((size_t)f * (size_t)g.plane + t, 5 * g.plane)] = lj[f];
    }
}

// out = a + b over n values
__global__ void k_adj_add(const C *a, const C *b, C *out, long long n)
{
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        out[c] = a[c] + b[c];
}

// part[n][b] = block b's share of the sum over the inflow face of
// s_n (rho_n lamJ_mz + rho_n w_n lamJ_E), then gw[n] = the shares in order.
// Twenty edge widths outside a jet s_n is 0 to the last bit, so those cells
// skip the FP64 root and tanh (not the product: an infinity or a NaN in lamJ
// reaches the sum); one block per jet took 263 us on a 128^2 face.
__global__ void __launch_bounds__(256) k_adj_jets(const double *jets, const C *lamJ, double *part, int nx, int ny,
                                                  double dx)
{
    const double *jt = jets + 7 * blockIdx.x;
    const long long plane = (long long)nx * ny;
    const double reach = jt[2] + 20.0 * jt[6] * dx;
    double acc = 0.0;
    for (long long f = blockIdx.y * 256LL + threadIdx.x; f < plane; f += 256LL * gridDim.y) {
        const int i = (int)((unsigned)f % (unsigned)nx), j = (int)((unsigned)f / (unsigned)nx);
        const double x = (i + 0.5) * dx - jt[0], y = (j + 0.5) * dx - jt[1], r2 = x * x + y * y;
        const double sn = r2 > reach * reach ? 0.0 : 0.5 * (1.0 - tanh((sqrt(r2) - jt[2]) / (jt[6] * dx)));
        acc += sn * (jt[3] * double(lamJ[ckl(3 * plane + f, 5 * plane)]) +
                     jt[3] * jt[4] * double(lamJ[ckl(4 * plane + f, 5 * plane)]));
    }
    __shared__ double red[256];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x * gridDim.y + blockIdx.y] = red[0];
}
__global__ void k_adj_jets_sum(const double *part, double *gw, int njets, int nblk)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= njets) return;
    double s = 0.0;
    for (int b = 0; b < nblk; b++) s += part[n * nblk + b];
    gw[n] = s;
}

// ------------------------------------------------- grouped launches
// One launch covers the blocks of several independent instances: block b
// belongs to the instance whose first block blk0 is the largest <= b, and
// runs the instance's own body at its place in the instance's own grid.
struct SourceInst {
    QIn q;
    S *b, *rho_out;
    Geom g;
    C alpha_s;
    const C *W, *J;
    int zc, wq, rows, gx, gy, blk0;
};
struct JacobiInst {
    const S *q, *b, *sin;
    S *sout;
    Geom g;
    C beta;
    int zc, wq, rows, gx, gy, blk0;
};
struct FluxInst {
    QIn qin;
    const S *sig;
    QBIn qn;
    Fout<5> out;
    QBOut outb;
    Geom g;
    C gamma, half_inv_dx, mu, lamv;
    const Scalars *sc;
    double *blockmax;
    int *err;
    const C *W, *J;
    int zc, gx, gy, blk0;
};
template <class I> struct Group {
    int count;
    I d[kGroupMax];
};
static_assert(sizeof(Group<FluxInst>) <= 32000, "grouped launch descriptors exceed the kernel parameter space");

// index of the instance that owns block b (blk0 ascending, d[0].blk0 = 0)
template <class I> __device__ __forceinline__ int group_find(const Group<I> &a, int b)
{
    int lo = 0, hi = a.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.d[mid].blk0 <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <bool HASD, bool FULL>
__global__ void __launch_bounds__(BT, SOURCE_BLOCKS) k_source_group(const __grid_constant__ Group<SourceInst> a)
{
    launched();
    __shared__ __align__(16) C U2[SOURCE_BUFS * 3 * TILEV];
    const SourceInst &d = a.d[group_find(a, blockIdx.x)];
    source_quads<HASD, FULL>(d.q, d.b, d.rho_out, d.g, d.alpha_s, d.W, d.J, d.zc,
                             BlockPos::of_index(blockIdx.x - d.blk0, d.gx, d.gy), d.wq, d.rows, U2);
}
template <bool HASD>
__global__ void __launch_bounds__(32 * PWARPS, SOURCE_PAIR_BLOCKS) k_source_pairs_group(const __grid_constant__ Group<SourceInst> a)
{
    launched();
    __shared__ C U2[2 * 3 * TILEP];
    const SourceInst &d = a.d[group_find(a, blockIdx.x)];
    source_pairs<HASD>(d.q, d.b, d.rho_out, d.g, d.alpha_s, d.W, d.J, d.zc,
                       BlockPos::of_index(blockIdx.x - d.blk0, d.gx, d.gy), U2);
}
template <bool RB, int NR>
__global__ void __launch_bounds__(BT, kJacobiBlocks<NR>) k_jacobi_full_group(const __grid_constant__ Group<JacobiInst> a,
                                                                        int colour)
{
    launched();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const JacobiInst &d = a.d[group_find(a, blockIdx.x)];
    jacobi_quads<true, RB, NR>(d.q, d.b, d.sin, d.sout, d.g, d.beta, d.zc, colour,
                           BlockPos::of_index(blockIdx.x - d.blk0, d.gx, d.gy), FQ, FR, smem_raw);
}
__global__ void __launch_bounds__(BT, JACOBI_FIT_BLOCKS) k_jacobi_fit_group(const __grid_constant__ Group<JacobiInst> a,
                                                                           int colour)
{
    launched();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const JacobiInst &d = a.d[group_find(a, blockIdx.x)];
    jacobi_quads<false, false, 1>(d.q, d.b, d.sin, d.sout, d.g, d.beta, d.zc, colour,
                               BlockPos::of_index(blockIdx.x - d.blk0, d.gx, d.gy), d.wq, d.rows, smem_raw);
}
__global__ void __launch_bounds__(BT, JACOBI_PAIR_BLOCKS)
    k_jacobi_pairs_group(const __grid_constant__ Group<JacobiInst> a, int colour)
{
    launched();
    __shared__ C R[2 * TILEP];
    __shared__ C SG[2 * TILEP];
    const JacobiInst &d = a.d[group_find(a, blockIdx.x)];
    jacobi_pairs(d.q, d.b, d.sin, d.sout, d.g, d.beta, d.zc, colour,
                 BlockPos::of_index(blockIdx.x - d.blk0, d.gx, d.gy), R, SG);
}
template <int mode, int ORD, bool VISC>
__global__ void __maxnreg__(FLUX_MAXREG) k_flux_group(const __grid_constant__ Group<FluxInst> a)
{
    launched();
    const FluxInst &d = a.d[group_find(a, blockIdx.x)];
    const Frhs none_rhs = {};
    const Fout<5> none_base = {};
    flux_body<mode, ORD, VISC>(d.qin, d.sig, d.qn, d.out, d.outb, none_rhs, none_base, d.g, d.gamma,
                               d.half_inv_dx, d.sc, d.blockmax, d.err, d.W, d.J, d.zc, 0, d.mu, d.lamv,
                               BlockPos::of_index(blockIdx.x - d.blk0, d.gx, d.gy));
}

// ------------------------------------------------------------ launchers
dim3 grid_of(const Geom &g, int bx, int by, int zc)
{
    return dim3((g.nx + bx - 1) / bx, (g.ny + by - 1) / by, (g.nz + zc - 1) / zc);
}

// state input: base fields q (type QB) and increments qd (type S, or NULL)
QIn state_in(const void *q, const void *qd, long long n)
{
    QIn f;
    for (int u = 0; u < 5; u++) {
        f.b[u] = q ? (const QB *)q + u * n : nullptr;
        f.d[u] = qd ? (const S *)qd + u * n : nullptr;
    }
    f.fs = (size_t)n;
    return f;
}

template <class K> cudaError_t allow_smem(K kern, int bytes)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

constexpr int kRows = sizeof(S) == 2 ? 2 : 1;  // rows per thread of form 3
// Kernel form of a source or sweep launch: 2 full quad tiles, 1 fitted quad
// tiles, 0 pairs; a sweep's form 3: full tiles with two rows per thread
// (16-bit storage, from 2M cells, where the tiles of one row fill the SMs more than
// once; FP16, two rows against one: 128^3 7.0 and 7.3 us, 256 x 256 x 128 20.4 and
// 22.7, 256 x 256 x 192 29.4 and 32.6, 512 x 512 x 128 73 and 80, 512^3 262 and 295;
// 128 x 128 x 64 6.9 and 6.1). Its grid and block.
int quad_form(const Geom &g, const Tiles &t, int vec)
{
    if (t.elem || vec == 0 || g.nx % VX != 0) return 0;
    return quad_fit(g).full ? 2 : 1;
}
int source_form(const Geom &g, const Tiles &t) { return quad_form(g, t, t.vec_source); }
int sweep_form(const Geom &g, const Tiles &t)
{
    const int form = quad_form(g, t, t.vec_jacobi);
    return form == 2 && sizeof(S) == 2 && g.ny % (2 * FR) == 0 && g.n >= (1 << 21) ? 3 : form;
}
// the source takes the compiled-in tile in the 16-bit forms only (FP16, compiled in
// against shape at run time: 128^3 7.7 and 8.7 us, 512 x 512 x 128 114 and 164; FP32:
// 9.5 and 9.9, 171 and 138, 256 x 128 x 128 27.1 and 22.5)
bool source_full(int form) { return form == 2 && sizeof(S) == 2; }
dim3 quad_grid(const Geom &g, int form, int zc)
{
    if (!form) return grid_of(g, PX, PY, zc);
    const QuadFit f = quad_fit(g);
    return dim3(f.gx, form == 3 ? f.gy / 2 : f.gy, (g.nz + zc - 1) / zc);
}
int quad_threads(const Geom &g, int form) { return form ? quad_fit(g).threads : 32 * PWARPS; }
int takes_quads_source(const Geom &g, const Tiles &t) { return source_form(g, t) > 0; }
int takes_quads_sweep(const Geom &g, const Tiles &t) { return sweep_form(g, t) > 0; }
// blocks per plane and blocks per SM (Ops::source_shape, Ops::jacobi_shape), default forms
constexpr Tiles kDefaultForms = {0, 0, 0, -1, -1, 0, 0, 0};
void source_shape(const Geom &g, long long *cols, int *resident)
{
    const int form = source_form(g, kDefaultForms);
    const dim3 gr = quad_grid(g, form, g.nz);
    *cols = (long long)gr.x * gr.y;
    *resident = !form ? SOURCE_PAIR_BLOCKS : (sizeof(C) == 8 ? 256 : 512) / quad_threads(g, form);
}
void jacobi_shape(const Geom &g, long long *cols, int *resident)
{
    const int form = sweep_form(g, kDefaultForms);
    const dim3 gr = quad_grid(g, form, g.nz);
    *cols = (long long)gr.x * gr.y;
    const int blocks = form == 3 ? kJacobiBlocks<2> : form == 2 ? kJacobiBlocks<1> : form ? JACOBI_FIT_BLOCKS : JACOBI_PAIR_BLOCKS;
    // shared memory holds two blocks of fitted quads in FP32 and FP64, four at 16 bits,
    // however few threads they have (8 x 300 x 300, FP16: 54 us per five sweeps with
    // the chunk for 16 blocks, 42 for 4; 4 x 4 x 2000, FP32: 46 and 36)
    const int smem = form == 3 ? JShape<kRows>::SMEM : form ? JShape<1>::SMEM : 4 * TILEP * (int)sizeof(C);
    *resident = std::min(blocks * BT / quad_threads(g, form), 227 * 1024 / (smem + 1024));
}

cudaError_t launch_source(const Geom &g, const Phys &p, const Tiles &t, const Inflow &in,
                          const void *q, const void *qd, void *b, void *rho_out, cudaStream_t st)
{
    if (kInc != (rho_out != nullptr)) return cudaErrorInvalidValue;  // the stage density: increment modes only
    if (!kInc && qd) return cudaErrorInvalidValue;
    const QIn qi = state_in(q, qd, g.n);
    const C as = C(p.alpha * 0.25 / (p.dx * p.dx));
    const C *W = (const C *)in.W, *J = (const C *)in.J;
    const QuadFit f = quad_fit(g);
    const int form = source_form(g, t), threads = quad_threads(g, form);
    const dim3 gr = quad_grid(g, form, t.zc_source);
    if (form) {
        auto kern = source_full(form) ? (qd ? k_source<kInc, true> : k_source<false, true>)
                              : (qd ? k_source<kInc, false> : k_source<false, false>);
        return launch(kern, gr, threads, 0, st, qi, (S *)b, (S *)rho_out, g, as, W, J, t.zc_source, f.wq, f.rows);
    } else {
        auto kern = qd ? k_source_pairs<kInc> : k_source_pairs<false>;
        return launch(kern, gr, threads, 0, st, qi, (S *)b, (S *)rho_out, g, as, W, J, t.zc_source);
    }
}

template <int NR> auto full_sweep(int colour) { return colour < 0 ? k_jacobi_full<false, NR> : k_jacobi_full<true, NR>; }
template <int NR> auto full_sweep_group(int colour)
{
    return colour < 0 ? k_jacobi_full_group<false, NR> : k_jacobi_full_group<true, NR>;
}
cudaError_t launch_jacobi(const Geom &g, const Phys &p, const Tiles &t, const void *q,
                          const void *b, const void *s_in, void *s_out, int colour, cudaStream_t st)
{
    const QuadFit f = quad_fit(g);
    const int form = sweep_form(g, t), threads = quad_threads(g, form);
    const dim3 gr = quad_grid(g, form, t.zc_jacobi);
    const C beta = C(p.alpha / (p.dx * p.dx));
    const S *qs = (const S *)q, *bs = (const S *)b, *si = (const S *)s_in;
    if (form >= 2) {
        auto kern = form == 3 ? full_sweep<kRows>(colour) : full_sweep<1>(colour);
        const int smem = form == 3 ? JShape<kRows>::SMEM : JShape<1>::SMEM;
        cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return launch(kern, gr, threads, smem, st, qs, bs, si, (S *)s_out, g, beta, t.zc_jacobi, colour);
    } else if (form) {
        cudaError_t e = allow_smem(k_jacobi_fit, JShape<1>::SMEM);
        if (e != cudaSuccess) return e;
        return launch(k_jacobi_fit, gr, threads, JShape<1>::SMEM, st, qs, bs, si, (S *)s_out, g, beta, t.zc_jacobi,
                      colour, f.wq, f.rows);
    } else {
        return launch(k_jacobi_pairs, gr, threads, 0, st, qs, bs, si, (S *)s_out, g, beta, t.zc_jacobi, colour);
    }
}

template <class T> Coefs<T> coefs_at(void *p, long long n)
{
    T *a = (T *)p;
    return {a, a + n, a + 2 * n, a + 3 * n, a + 4 * n};
}
dim3 cells_grid(const Geom &g, int colour)
{
    const long long w = colour < 0 ? g.nx : (g.nx + 1) / 2;
    return dim3((unsigned)((w * g.ny + 255) / 256), (unsigned)std::min(g.nz, 65535));
}
template <class T>
cudaError_t launch_coefs(const Geom &g, const Phys &p, const void *q, void *coefs, cudaStream_t st)
{
    const Coefs<T> a = coefs_at<T>(coefs, g.n);
    const dim3 gr = cells_grid(g, -1);
    cudaError_t e = launch(k_coef_rcp<T>, gr, 256, 0, st, (const T *)q, a.d, g);
    if (e == cudaSuccess) e = launch(k_coef_faces<T>, gr, 256, 0, st, a, g, T(0.5) * T(p.alpha / (p.dx * p.dx)));
    return e == cudaSuccess ? launch(k_coef_diag<T>, gr, 256, 0, st, a, g) : e;
}
template <class T>
cudaError_t launch_sweep(const Geom &g, const void *coefs, const void *b, const void *s_in, void *s_out, int colour,
                         cudaStream_t st)
{
    const Coefs<T> a = coefs_at<T>((void *)coefs, g.n);
    const Coefs<const T> k = {a.cx, a.cy, a.cz, a.d, a.inv};
    return launch(k_sweep<T>, cells_grid(g, colour), 256, 0, st, k, (const T *)b, (const T *)s_in, (T *)s_out, g, colour);
}
// Ops::coefs and Ops::sweep: FP64 only
template <class T> constexpr auto coefs_op()
{
    if constexpr (sizeof(T) == 8) return &launch_coefs<T>;
    else return nullptr;
}
template <class T> constexpr auto sweep_op()
{
    if constexpr (sizeof(T) == 8) return &launch_sweep<T>;
    else return nullptr;
}

long long flux_blocks(const Geom &g, const Tiles &t)
{
    dim3 gr = grid_of(g, TX, TY, t.zc_flux);
    return (long long)gr.x * gr.y * gr.z;
}

cudaError_t launch_flux(const Geom &g, const Phys &p, const Tiles &t, const Inflow &in, int mode,
                        const void *qs, const void *qd, const void *sig, const void *qn, void *out, void *rhs,
                        void *base_out, const Scalars *sc, double *blockmax, int *err, cudaStream_t st)
{
    // increments are read from stage 2 on, and only in the increment modes
    if ((qd != nullptr) != (kInc && (mode == FLUX_STAGE2 || mode == FLUX_STAGE3))) return cudaErrorInvalidValue;
    if (kInc && base_out) return cudaErrorInvalidValue;
    size_t smem = flux_smem_bytes();
    auto go = [&](auto kern) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const QIn fi = state_in(qs, qd, g.n);
        QBIn fn;
        Fout<5> fo, fb;
        QBOut fob;
        Frhs fr;
        // the stage output: increments (S) for stages 1 and 2 of the increment
        // modes, the FP32 state for their stage 3, else the stored state (S)
        const bool out_is_state = !kInc || mode == FLUX_STAGE3;
        for (int u = 0; u < 5; u++) {
            fn.p[u] = qn ? (const QB *)qn + u * g.n : nullptr;
            fo.p[u] = out && !(kInc && out_is_state) ? (S *)out + u * g.n : nullptr;
            fob.p[u] = out && kInc && out_is_state ? (QB *)out + u * g.n : nullptr;
            fb.p[u] = base_out ? (S *)base_out + u * g.n : nullptr;
            fr.p[u] = rhs ? (C *)rhs + u * g.n : nullptr;
        }
        // the z-chunks of planes [z_begin, z_end) (all chunks when z_end = 0)
        dim3 gr = grid_of(g, TX, TY, t.zc_flux);
        const int cz0 = t.z_begin / t.zc_flux;
        if (t.z_end > 0) gr.z = (t.z_end - t.z_begin + t.zc_flux - 1) / t.zc_flux;
        e = launch(kern, gr, NT, smem, st, fi, (const S *)sig, fn, fo, fob, fr, fb, g, C(p.gamma), C(0.5 / p.dx), sc,
                                   blockmax, err, (const C *)in.W, (const C *)in.J, t.zc_flux, cz0, C(p.mu),
                                   C(p.zeta - 2.0 * p.mu / 3.0));
        if (e != cudaSuccess) {
            cudaFuncAttributes fa;
            if (cudaFuncGetAttributes(&fa, kern) == cudaSuccess)
                fprintf(stderr, "igr: flux launch failed (%s): block %d, regs %d, max threads %d, "
                                "static smem %zu, dynamic smem %zu, local %zu\n",
                        cudaGetErrorString(e), NT, fa.numRegs, fa.maxThreadsPerBlock,
                        fa.sharedSizeBytes, smem, fa.localSizeBytes);
        }
        return e;
    };
    auto by_mode = [&](auto k0, auto k1, auto k2, auto k3) {
        switch (mode) {
        case FLUX_RHS: return go(k0);
        case FLUX_STAGE1: return go(k1);
        case FLUX_STAGE2: return go(k2);
        default: return go(k3);
        }
    };
    const bool visc = p.mu != 0.0 || p.zeta != 0.0;
    if (p.order == 3) {
        if (visc)
            return by_mode(k_flux<FLUX_RHS, 3, true>, k_flux<FLUX_STAGE1, 3, true>,
                           k_flux<FLUX_STAGE2, 3, true>, k_flux<FLUX_STAGE3, 3, true>);
        return by_mode(k_flux<FLUX_RHS, 3, false>, k_flux<FLUX_STAGE1, 3, false>,
                       k_flux<FLUX_STAGE2, 3, false>, k_flux<FLUX_STAGE3, 3, false>);
    }
    if (visc)
        return by_mode(k_flux<FLUX_RHS, 5, true>, k_flux<FLUX_STAGE1, 5, true>,
                       k_flux<FLUX_STAGE2, 5, true>, k_flux<FLUX_STAGE3, 5, true>);
    return by_mode(k_flux<FLUX_RHS, 5, false>, k_flux<FLUX_STAGE1, 5, false>,
                   k_flux<FLUX_STAGE2, 5, false>, k_flux<FLUX_STAGE3, 5, false>);
}

// ---- grouped launches: calls are grouped by kernel form and in chunks of
// kGroupMax; each chunk is one launch over all its instances' blocks

// run fn(first, count) over the calls of each key(call), in their order
template <class T, class K, class F>
cudaError_t by_key(const T *calls, int n, K key, F fn)
{
    std::vector<T> sorted(calls, calls + n);
    std::stable_sort(sorted.begin(), sorted.end(), [&](const T &x, const T &y) { return key(x) < key(y); });
    for (int i = 0; i < n;) {
        int j = i + 1;
        while (j < n && j - i < kGroupMax && key(sorted[j]) == key(sorted[i])) j++;
        cudaError_t e = fn(sorted.data() + i, j - i);
        if (e != cudaSuccess) return e;
        i = j;
    }
    return cudaSuccess;
}

cudaError_t launch_source_group(const SourceCall *calls, int n, cudaStream_t st)
{
    for (int i = 0; i < n; i++)
        if ((kInc != (calls[i].rho_out != nullptr)) || (!kInc && calls[i].qd)) return cudaErrorInvalidValue;
    auto key = [](const SourceCall &c) { return 2 * source_form(c.g, c.t) + (c.qd ? 1 : 0); };
    return by_key(calls, n, key, [&](const SourceCall *cs, int m) {
        Group<SourceInst> a;
        a.count = m;
        int blk = 0, threads = 0;
        const int form = key(cs[0]) >> 1;
        for (int i = 0; i < m; i++) {
            const SourceCall &c = cs[i];
            const QuadFit f = quad_fit(c.g);
            SourceInst &d = a.d[i];
            d.q = state_in(c.q, c.qd, c.g.n);
            d.b = (S *)c.b;
            d.rho_out = (S *)c.rho_out;
            d.g = c.g;
            d.alpha_s = C(c.p.alpha * 0.25 / (c.p.dx * c.p.dx));
            d.W = (const C *)c.in.W;
            d.J = (const C *)c.in.J;
            d.zc = c.t.zc_source;
            d.wq = f.wq;
            d.rows = f.rows;
            const dim3 gr = quad_grid(c.g, form, d.zc);
            d.gx = (int)gr.x;
            d.gy = (int)gr.y;
            d.blk0 = blk;
            blk += (int)(gr.x * gr.y * gr.z);
            threads = std::max(threads, quad_threads(c.g, form));
        }
        auto kern = source_full(form) ? (cs[0].qd ? k_source_group<kInc, true> : k_source_group<false, true>)
                    : form ? (cs[0].qd ? k_source_group<kInc, false> : k_source_group<false, false>)
                           : (cs[0].qd ? k_source_pairs_group<kInc> : k_source_pairs_group<false>);
        return launch(kern, blk, threads, 0, st, a);
    });
}

cudaError_t launch_jacobi_group(const JacobiCall *calls, int n, int colour, cudaStream_t st)
{
    auto key = [](const JacobiCall &c) { return sweep_form(c.g, c.t); };
    return by_key(calls, n, key, [&](const JacobiCall *cs, int m) {
        Group<JacobiInst> a;
        a.count = m;
        int blk = 0, threads = 0;
        const int form = key(cs[0]);
        for (int i = 0; i < m; i++) {
            const JacobiCall &c = cs[i];
            const QuadFit f = quad_fit(c.g);
            JacobiInst &d = a.d[i];
            d.q = (const S *)c.q;
            d.b = (const S *)c.b;
            d.sin = (const S *)c.s_in;
            d.sout = (S *)c.s_out;
            d.g = c.g;
            d.beta = C(c.p.alpha / (c.p.dx * c.p.dx));
            d.zc = c.t.zc_jacobi;
            d.wq = f.wq;
            d.rows = f.rows;
            const dim3 gr = quad_grid(c.g, form, d.zc);
            d.gx = (int)gr.x;
            d.gy = (int)gr.y;
            d.blk0 = blk;
            blk += (int)(gr.x * gr.y * gr.z);
            threads = std::max(threads, quad_threads(c.g, form));
        }
        auto kern = form == 3 ? full_sweep_group<kRows>(colour)
                    : form == 2 ? full_sweep_group<1>(colour) : form ? k_jacobi_fit_group : k_jacobi_pairs_group;
        const int smem = form == 3 ? JShape<kRows>::SMEM : form ? JShape<1>::SMEM : 0;
        cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return launch(kern, blk, threads, smem, st, a, colour);
    });
}

cudaError_t launch_flux_group(const FluxCall *calls, int n, int mode, cudaStream_t st)
{
    if (mode == FLUX_RHS) return cudaErrorInvalidValue;
    for (int i = 0; i < n; i++)
        if ((calls[i].qd != nullptr) != (kInc && (mode == FLUX_STAGE2 || mode == FLUX_STAGE3)) ||
            calls[i].t.z_end != 0)
            return cudaErrorInvalidValue;
    auto kind = [](const FluxCall &c) {
        return 2 * (c.p.order == 3 ? 1 : 0) + (c.p.mu != 0.0 || c.p.zeta != 0.0 ? 1 : 0);
    };
    const size_t smem = flux_smem_bytes();
    return by_key(calls, n, kind, [&](const FluxCall *cs, int m) {
        Group<FluxInst> a;
        a.count = m;
        int blk = 0;
        const bool out_is_state = !kInc || mode == FLUX_STAGE3;
        for (int i = 0; i < m; i++) {
            const FluxCall &c = cs[i];
            FluxInst &d = a.d[i];
            d.qin = state_in(c.qs, c.qd, c.g.n);
            d.sig = (const S *)c.sig;
            for (int u = 0; u < 5; u++) {
                d.qn.p[u] = c.qn ? (const QB *)c.qn + u * c.g.n : nullptr;
                d.out.p[u] = c.out && !(kInc && out_is_state) ? (S *)c.out + u * c.g.n : nullptr;
                d.outb.p[u] = c.out && kInc && out_is_state ? (QB *)c.out + u * c.g.n : nullptr;
            }
            d.g = c.g;
            d.gamma = C(c.p.gamma);
            d.half_inv_dx = C(0.5 / c.p.dx);
            d.mu = C(c.p.mu);
            d.lamv = C(c.p.zeta - 2.0 * c.p.mu / 3.0);
            d.sc = c.sc;
            d.blockmax = c.blockmax;
            d.err = c.err;
            d.W = (const C *)c.in.W;
            d.J = (const C *)c.in.J;
            d.zc = c.t.zc_flux;
            const dim3 gr = grid_of(c.g, TX, TY, d.zc);
            d.gx = (int)gr.x;
            d.gy = (int)gr.y;
            d.blk0 = blk;
            blk += (int)(gr.x * gr.y * gr.z);
        }
        auto go = [&](auto kern) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            return launch(kern, blk, NT, smem, st, a);
        };
        auto by_mode = [&](auto k1, auto k2, auto k3) {
            return mode == FLUX_STAGE1 ? go(k1) : mode == FLUX_STAGE2 ? go(k2) : go(k3);
        };
        switch (kind(cs[0])) {
        case 0:
            return by_mode(k_flux_group<FLUX_STAGE1, 5, false>, k_flux_group<FLUX_STAGE2, 5, false>,
                           k_flux_group<FLUX_STAGE3, 5, false>);
        case 1:
            return by_mode(k_flux_group<FLUX_STAGE1, 5, true>, k_flux_group<FLUX_STAGE2, 5, true>,
                           k_flux_group<FLUX_STAGE3, 5, true>);
        case 2:
            return by_mode(k_flux_group<FLUX_STAGE1, 3, false>, k_flux_group<FLUX_STAGE2, 3, false>,
                           k_flux_group<FLUX_STAGE3, 3, false>);
        default:
            return by_mode(k_flux_group<FLUX_STAGE1, 3, true>, k_flux_group<FLUX_STAGE2, 3, true>,
                           k_flux_group<FLUX_STAGE3, 3, true>);
        }
    });
}

cudaError_t launch_speed(const Geom &g, const Phys &p, const void *q, double *blockmax,
                         int *nblocks, cudaStream_t st)
{
    const bool vec = g.n % 4 == 0 && (uintptr_t)q % (4 * sizeof(QB)) == 0;
    const long long want = (g.n / (vec ? 4 : 1) + SPEED_NT - 1) / SPEED_NT;
    const int nb = (int)std::min<long long>(want, SPEED_MAXBLOCKS);
    auto kern = vec ? k_speed<true> : k_speed<false>;
    *nblocks = nb;
    return launch(kern, nb, SPEED_NT, 0, st, (const QB *)q, g.n, C(p.gamma), blockmax);
}

cudaError_t launch_rk_combine(const void *qn, const void *qs, const void *L, void *out,
                              long long n, double dt, double w, cudaStream_t st)
{
    long long want = (n + 255) / 256;
    int nb = (int)(want < 152 * 16 ? (want > 0 ? want : 1) : 152 * 16);
    k_rk_combine<<<nb, 256, 0, st>>>((const QB *)qn, (const QB *)qs, (const C *)L, (QB *)out, n, dt, w);
    return cudaGetLastError();
}

// blocks of a grid-stride launch over n values
int flat_blocks(long long n)
{
    long long b = (n + 255) / 256;
    return (int)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}
unsigned cell_blocks(const Geom &g)
{
    return (unsigned)(((long long)g.nx + CBX - 1) / CBX * ((g.ny + CBY - 1) / CBY) * g.nz);
}
// cells per chunk of a march over n cells in `lines` blocks: a chunk evaluates
// five faces beyond its cells; three blocks fit an SM in FP32, and one fills
// its FP64 units (as choose_zc)
int march_chunk(long long lines, int n)
{
    int best = n;
    double tbest = 1e300;
    const long long slots = sizeof(C) == 8 ? 152 : 456;
    for (int m = (n + 65534) / 65535; m <= (n + 3) / 4; m++) {
        const int zc = (n + m - 1) / m;
        const long long blocks = lines * ((n + zc - 1) / zc);
        const double t = (zc + 5.0) * (double)((blocks + slots - 1) / slots);
        if (t < tbest * 0.999) {
            tbest = t;
            best = zc;
        }
        if (blocks > 16 * slots) break;
    }
    return best;
}

cudaError_t launch_adj_rhs(const Geom &g, const Phys &p, const Inflow &in, const void *qs, const void *sig,
                           const void *lout, void *lqs, void *lq0, void *lsig, void *lamJ, double w, double dt,
                           int first, cudaStream_t st)
{
    const C *W = (const C *)in.W, *J = (const C *)in.J, *lo = (const C *)lout;
    const S *q = (const S *)qs, *s = (const S *)sig;
    const C gamma = C(p.gamma), inv_dx = C(1.0 / p.dx), wdt = C(w) * C(dt);
    const long long rows = (long long)g.ny * g.nz;
    const int nseg = g.bc[0] == BC_PERIODIC ? (g.nx + XCELLS - 1) / XCELLS : (g.nx + 6 + XCELLS - 1) / XCELLS;
    // FP64 rows of up to 12 cells: a warp of the gather has 32 faces' worth of FP64
    // instructions for n + 1 (6 x 300 x 300, one step: 25.0 ms against 20.0 marching;
    // 12 x 200 x 200: 12.6 and 11.4; 20 x 200 x 200: 15.1 and 15.5; in FP32 the march
    // gains 6% at 6 cells and loses from 8)
    bool thin = false;
    if constexpr (sizeof(C) == 8) {
        thin = g.nx <= 12;
        if (thin)
            k_adj_rhs_march<0><<<(unsigned)((rows + 127) / 128), 128, 0, st>>>(
                q, s, lo, (C *)lqs, (C *)lsig, (C *)lq0, (C *)lamJ, g, gamma, inv_dx, C(w), wdt, first, W, J, g.nx);
    }
    if (!thin)
        k_adj_rhs_x<<<(unsigned)((rows * nseg + XWARPS - 1) / XWARPS), 32 * XWARPS, 0, st>>>(
            q, s, lo, (C *)lqs, (C *)lq0, (C *)lsig, g, gamma, inv_dx, C(w), wdt, first, nseg);
    const long long by = ((long long)g.nx * g.nz + 127) / 128, bz = (g.plane + 127) / 128;
    const int cy = march_chunk(by, g.ny), cz = march_chunk(bz, g.nz);
    k_adj_rhs_march<1><<<dim3((unsigned)by, (g.ny + cy - 1) / cy), 128, 0, st>>>(
        q, s, lo, (C *)lqs, (C *)lsig, (C *)lq0, (C *)lamJ, g, gamma, inv_dx, C(w), wdt, first, W, J, cy);
    k_adj_rhs_march<2><<<dim3((unsigned)bz, (g.nz + cz - 1) / cz), 128, 0, st>>>(
        q, s, lo, (C *)lqs, (C *)lsig, (C *)lq0, (C *)lamJ, g, gamma, inv_dx, C(w), wdt, first, W, J, cz);
    return cudaGetLastError();
}

cudaError_t launch_adj_rk(const void *lout, void *lq0, void *lqs, void *Lb, long long n5, double w,
                          double dt, cudaStream_t st)
{
    k_adj_rk<<<flat_blocks(n5), 256, 0, st>>>((const C *)lout, (C *)lq0, (C *)lqs, (C *)Lb, n5, C(w), C(dt));
    return cudaGetLastError();
}

cudaError_t launch_adj_rhs_scatter(const Geom &g, const Phys &p, const Inflow &in, const void *qs, const void *sig,
                           const void *Lb, void *lqs, void *lsig, void *lamJ, cudaStream_t st)
{
    long long nfx = (long long)(g.nx + 1) * g.ny * g.nz, nfy = (long long)g.nx * (g.ny + 1) * g.nz,
              nfz = (long long)g.nx * g.ny * (g.nz + 1);
    const C *W = (const C *)in.W, *J = (const C *)in.J;
    k_adj_rhs_scatter<0><<<flat_blocks(nfx), 256, 0, st>>>((const S *)qs, (const S *)sig, (const C *)Lb, (C *)lqs,
                                                   (C *)lsig, (C *)lamJ, g, C(p.gamma), C(1.0 / p.dx), W, J);
    k_adj_rhs_scatter<1><<<flat_blocks(nfy), 256, 0, st>>>((const S *)qs, (const S *)sig, (const C *)Lb, (C *)lqs,
                                                   (C *)lsig, (C *)lamJ, g, C(p.gamma), C(1.0 / p.dx), W, J);
    k_adj_rhs_scatter<2><<<flat_blocks(nfz), 256, 0, st>>>((const S *)qs, (const S *)sig, (const C *)Lb, (C *)lqs,
                                                   (C *)lsig, (C *)lamJ, g, C(p.gamma), C(1.0 / p.dx), W, J);
    return cudaGetLastError();
}

cudaError_t launch_adj_rho(const Geom &g, const void *q, void *rb, void *lqs, cudaStream_t st)
{
    k_adj_rho<<<flat_blocks(g.n), 256, 0, st>>>((const S *)q, (C *)rb, (C *)lqs, g.n);
    return cudaGetLastError();
}

cudaError_t launch_adj_source_scatter(const Geom &g, const Phys &p, const Inflow &in, const void *q, const void *lb,
                              void *lqs, void *lamJ, cudaStream_t st)
{
    k_adj_source_scatter<<<flat_blocks(g.n), 256, 0, st>>>((const S *)q, (const C *)lb, (C *)lqs, (C *)lamJ, g,
                                                   C(p.alpha), C(0.5 / p.dx), (const C *)in.W, (const C *)in.J);
    return cudaGetLastError();
}

cudaError_t launch_adj_diag(const Geom &g, const Phys &p, const void *q, void *r, void *diag, void *dinv,
                            cudaStream_t st)
{
    k_adj_diag<<<cell_blocks(g), dim3(CBX, CBY), 0, st>>>((const S *)q, (C *)r, (C *)diag, (C *)dinv, g,
                                                          C(p.alpha / (p.dx * p.dx)));
    return cudaGetLastError();
}

cudaError_t launch_adj_jacobi(const Geom &g, const Phys &p, const void *r, const void *diag, const void *dinv,
                              const void *sk, const void *F, const void *lsig, void *nl, void *lb, void *rb,
                              int first, cudaStream_t st)
{
    k_adj_jacobi<<<cell_blocks(g), dim3(CBX, CBY), 0, st>>>((const C *)r, (const C *)diag, (const C *)dinv,
                                                            (const S *)sk, (const S *)F, (const C *)lsig, (C *)nl,
                                                            (C *)lb, (C *)rb, g, C(p.alpha / (p.dx * p.dx)), first);
    return cudaGetLastError();
}

cudaError_t launch_adj_source(const Geom &g, const Phys &p, const Inflow &in, const void *q, const void *r,
                              const void *lb, const void *rb, void *const grads[9], void *lqs, void *lamJ,
                              cudaStream_t st)
{
    Grads G;
    for (int t = 0; t < 9; t++) G.p[t] = (C *)grads[t];
    const C *W = (const C *)in.W, *J = (const C *)in.J;
    k_adj_grad<<<cell_blocks(g), dim3(CBX, CBY), 0, st>>>((const S *)q, (const C *)r, (const C *)lb, G, g,
                                                          C(p.alpha), C(0.5 / p.dx), W, J);
    k_adj_source<<<cell_blocks(g), dim3(CBX, CBY), 0, st>>>((const S *)q, (const C *)r, (const C *)rb, G, (C *)lqs,
                                                            (C *)lamJ, g, W, J);
    return cudaGetLastError();
}

cudaError_t launch_adj_add(const void *a, const void *b, void *out, long long n, cudaStream_t st)
{
    k_adj_add<<<flat_blocks(n), 256, 0, st>>>((const C *)a, (const C *)b, (C *)out, n);
    return cudaGetLastError();
}

cudaError_t launch_adj_jets(const Geom &g, const Phys &p, const double *jets, int njets, const void *lamJ,
                            double *gw, cudaStream_t st)
{
    if (njets <= 0) return cudaSuccess;
    double *part = gw + njets;
    k_adj_jets<<<dim3(njets, ADJ_JET_BLOCKS), 256, 0, st>>>(jets, (const C *)lamJ, part, g.nx, g.ny, p.dx);
    k_adj_jets_sum<<<(njets + 31) / 32, 32, 0, st>>>(part, gw, njets, ADJ_JET_BLOCKS);
    return cudaGetLastError();
}

cudaError_t launch_diag(const Geom &g, const Phys &p, const Inflow &in, const void *q, const void *sig,
                        double *part, int *nblocks, cudaStream_t st)
{
    long long nb = (g.n + DIAG_NT - 1) / DIAG_NT;
    int blocks = (int)(nb < DIAG_BLOCKS_MAX ? nb : DIAG_BLOCKS_MAX);
    *nblocks = blocks;
    k_diag<<<blocks, DIAG_NT, 0, st>>>((const QB *)q, (const S *)sig, g, p.gamma, p.alpha, p.dx,
                                        (const C *)in.W, (const C *)in.J, part);
    return cudaGetLastError();
}

// debug build: read (and clear) the bounds-check counter; the self-test
// forms one index past the end of an array of n values (checked, not used)
__global__ void k_bounds_selftest(long long n, int *sink)
{
    idx c = ck((idx)(n + 5), n);
    if (c != 0) *sink = (int)c;  // never taken: the check returns 0
}

unsigned long long bounds_hits(int clear)
{
#ifdef IGR_DEBUG_BOUNDS
    unsigned long long h = 0;
    if (cudaMemcpyFromSymbol(&h, g_bounds_hits, sizeof h) != cudaSuccess) return ~0ull;
    if (clear) {
        unsigned long long z = 0;
        if (cudaMemcpyToSymbol(g_bounds_hits, &z, sizeof z) != cudaSuccess) return ~0ull;
    }
    return h;
#else
    (void)clear;
    return ~0ull;  // not a debug build
#endif
}

cudaError_t bounds_selftest(int *sink, cudaStream_t st)
{
    k_bounds_selftest<<<1, 1, 0, st>>>(1000, sink);
    return cudaGetLastError();
}

}  // namespace

extern const Ops IGR_OPS = {
    (int)sizeof(S), (int)sizeof(C), (int)sizeof(QB), launch_source, launch_jacobi, launch_flux, flux_blocks,
    launch_speed, launch_rk_combine, launch_adj_rhs, launch_adj_diag, launch_adj_jacobi, launch_adj_source,
    launch_adj_add, launch_adj_jets, launch_adj_rk, launch_adj_rhs_scatter, launch_adj_rho,
    launch_adj_source_scatter, launch_diag, bounds_hits, bounds_selftest,
    launch_source_group, launch_jacobi_group, launch_flux_group, takes_quads_source, takes_quads_sweep,
    source_shape, jacobi_shape,
    coefs_op<S>(), sweep_op<S>(),
};

}  // namespace igr
