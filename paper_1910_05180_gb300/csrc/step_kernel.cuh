// step_kernel.cuh -- z-marching 2.5D stencil kernel of one explicit SPFM / CF step.
//
// Data movement.  Every field buffer carries a one-cell ghost layer in HBM
// (spfm_internal.h), so a tile plus its halo is a set of plain, in-bounds,
// 16-byte-aligned rows.  One CTA owns an xy tile of TX*VX by TY cells
// (VX = cells per 16 bytes) and marches a chunk of z planes.  A producer warp
// brings each plane's tile plus halo into a ring of NS shared-memory stages
// with one TMA tensor copy (cp.async.bulk.tensor.3d over a tensor map of the
// ghosted buffer), or, where no map could be encoded, with one bulk copy per
// halo row (cp.async.bulk); both complete on the stage's "full" mbarrier by
// transaction count.  TX*TY consumer threads wait on "full", read the stage,
// and release it on its "empty" barrier.  There is no __syncthreads in the
// march, and NS-1 planes stay in flight per CTA.  Every wait is bounded: on
// timeout the thread sets the error word and leaves.
//
// Boundary conditions.  The kernel reads the ghost layer.  In general it
// writes interior cells only and a face kernel (boundary.cu) refreshes the
// ghosts of the new field after each step.  When every face is periodic and a
// row is a whole number of 32-byte sectors, the ghosts are plain periodic images:
// the thread that writes a cell next to a face also writes its image(s) on the
// far side (x images as whole 32-byte sectors of the row pads, two threads a
// sector), so no face kernel runs; where no face is periodic the producer warp
// builds the ghosts of the planes it stages.  The kernels of a call chain by
// programmatic dependent launch, each waiting for the one before in every tile.
//
// Arithmetic.  From each plane every thread forms, for its cells,
//   C  = phi at the cell,
//   F' = sum of the 4 in-plane face neighbours - 4 C,
//   E' = sum of the 4 in-plane diagonal neighbours - 4 C,
// kept in registers for the planes z-1, z, z+1 (the z loop is unrolled by
// three with rotating register roles).  The shell sums then follow:
//   S1 - 6 phi  = F'_z + t,             t = (C_{z-1} - phi) + (C_{z+1} - phi)
//   S2 - 12 phi = E'_z + F'_{z-1} + F'_{z+1} + 4 t
//   S3 - 8 phi  = E'_{z-1} + E'_{z+1} + 4 t
// Every term is a difference of neighbouring values, which keeps the drift far
// below that of a plain sum of neighbours.  FP32 runs on packed f32x2 pairs
// (FFMA2/FADD2/FMUL2 of sm_100+) of adjacent cells; FP64 on scalar doubles.
#pragma once

#include <cuda.h>   // CUtensorMap (the map is encoded on the host, see tma.cu)
#include <math.h>
#include <string.h>

#include <type_traits>

#include "spfm_internal.h"

namespace spfm {

constexpr long long kWaitCycles = 4000000000LL;   // ~2 s at 2 GHz per bounded wait

#ifndef SPFM_STAGES
#define SPFM_STAGES 6         // planes in flight per CTA
#endif
#ifndef SPFM_MIN_CTAS
#define SPFM_MIN_CTAS 3       // resident CTAs per SM the register budget is sized for
#endif

// ------------------------------------------------------------ pack arithmetic

template <class T> struct Pk;

// The FP32 packs run on the paired FP32 instructions.  The code generator
// fuses a paired multiply whose result feeds a paired add into one paired FMA,
// explicit rounding modifier or not, and decides per inlined copy; so the step
// code never adds or subtracts a product as a separate operation: where a
// product is summed the code writes the FMA.  Every unrolled copy of the
// z-march then computes the same expression, and a cell gets the same bits
// whichever CTA, z-chunk or kernel (single grid or batch) computes it.
template <> struct Pk<float> {
    using P = float2;
    static __device__ __forceinline__ P mk(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ float add1(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ P add(P a, P b) { return __fadd2_rn(a, b); }
    static __device__ __forceinline__ P mul(P a, P b) { return __fmul2_rn(a, b); }
    static __device__ __forceinline__ P fma(P a, P b, P c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ P sub(P a, P b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
    // a / b as a * rcp(b): two MUFU reciprocals (|rel. error| < 2^-22) and one
    // packed multiply, the accuracy of __fdividef without splitting the pack
    static __device__ __forceinline__ P div(P a, P b)
    {
        float2 r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(b.x));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(b.y));
        return __fmul2_rn(a, r);
    }
    static __device__ __forceinline__ P rsqrt(P a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }
    // v (1 - v)
    static __device__ __forceinline__ P bump(P v, P one) { return mul(v, sub(one, v)); }
    // a + b - 2 c as the sum of two differences
    static __device__ __forceinline__ P second(P a, P b, P c) { return add(sub(a, c), sub(b, c)); }
};

struct D2 { double x, y; };

template <> struct Pk<double> {
    using P = D2;
    static __device__ __forceinline__ P mk(double a, double b) { return {a, b}; }
    static __device__ __forceinline__ double add1(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ P add(P a, P b) { return {__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)}; }
    static __device__ __forceinline__ P mul(P a, P b) { return {__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)}; }
    static __device__ __forceinline__ P fma(P a, P b, P c)
    {
        return {__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y)};
    }
    static __device__ __forceinline__ P sub(P a, P b) { return {__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y)}; }
    // a / b in 7 instructions of the FP64 pipe, which bounds these kernels, where
    // a division takes some 14: the reciprocal r by one third-order Newton step
    // (Householder's iteration of order 2) from the hardware's approximation
    // (relative error e < 2^-18, then e^3), and Markstein's correction of the
    // quotient q by its remainder a - b q, which an FMA gives exactly (IBM J. Res.
    // Dev. 34, 1990): correctly rounded but for quotients within 2^-50 ulp of a tie.
    // The exponents of a and b keep the remainder and the reciprocal normal;
    // other operands (zeros, infinities, NaN, far too large or small) are divided.
    static __device__ __forceinline__ double quot(double a, double b)
    {
        constexpr uint32_t lo = (uint32_t)(1023 - 400) << 20, hi = (uint32_t)(1023 + 400) << 20;
        const uint32_t ea = (uint32_t)__double2hiint(a) & 0x7fffffffu, eb = (uint32_t)__double2hiint(b) & 0x7fffffffu;
        if (ea - lo >= hi - lo || eb - lo >= hi - lo) return divide(a, b);
        double r;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
        const double e = __fma_rn(-b, r, 1.0);
        r = __fma_rn(__fma_rn(e, e, e), r, r);
        const double q = __dmul_rn(a, r);
        return __fma_rn(__fma_rn(-b, q, a), r, q);
    }
    static __device__ __noinline__ double divide(double a, double b) { return __ddiv_rn(a, b); }
    static __device__ __forceinline__ P div(P a, P b) { return {quot(a.x, b.x), quot(a.y, b.y)}; }
    static __device__ __forceinline__ P rsqrt(P a) { return {::rsqrt(a.x), ::rsqrt(a.y)}; }
    // v - v^2, rounded once
    static __device__ __forceinline__ P bump(P v, P) { return {__fma_rn(-v.x, v.x, v.x), __fma_rn(-v.y, v.y, v.y)}; }
    // a + b - 2 c as the sum of two differences, exact where a and b are within a
    // factor of two of c (a + b first would round at the size of phi; one FP64
    // instruction less a cell, 2 %, but rms errors of a step 0.1 to 0.3 % larger)
    static __device__ __forceinline__ P second(P a, P b, P c) { return add(sub(a, c), sub(b, c)); }
};

template <class T> struct PackT;
template <> struct PackT<float> { using P = float2; static P splat(float v) { return make_float2(v, v); } };
template <> struct PackT<double> { using P = D2; static P splat(double v) { return {v, v}; } };

// Step coefficients pre-splatted into packs (kernel parameter space), with dt
// folded in: phi' = phi + c1 dt S1' + c2 dt S2' + c3 dt S3'
//                 + q (s (-dt) N(q) / D(q) - kmu dt)                    (TI)
//                 + q (s (-kappa dt) - kmu dt)                          (CF)
// with N(q) / D(q) = sum_k beta_k / (1 - A_k s^2) (potential.cu).
template <class T>
struct PackCoef {
    using P = typename PackT<T>::P;
    P one, m2, m4, c1, c2, c3, ct, nkmu, nkap;
    // coefficients of q^i in -dt N and in D, side by side (one 16- or 32-byte
    // load: a batch reads them from its warps' copies in shared memory)
    struct __align__(2 * sizeof(P)) Ratio {
        P num, den;
    };
    Ratio rat[kMaxTerms + 1];
    int deg;          // degree of D (0: the coupling groups are summed one by one)
    uint32_t guard;   // bits of the lowest q that N / D covers (potential.cu)
    // -A_k and -beta_k dt of the coupling groups, for the sum group by group
    struct __align__(2 * sizeof(P)) Pair {
        P nA, nbeta;
    };
    int nterms;
    Pair pair[kMaxTerms];
};

// the upper 32 bits of a value; for a negative limit l, bits(x) > bits(l) as
// unsigned numbers exactly where x < l (or x is a NaN with its sign set)
__host__ __device__ __forceinline__ uint32_t top_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t b;
    memcpy(&b, &x, 4);
    return b;
#endif
}
__host__ __device__ __forceinline__ uint32_t top_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2hiint(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return (uint32_t)(b >> 32);
#endif
}

template <class T>
inline PackCoef<T> make_pack_coef(const StepCoef<T> &c)
{
    using PT = PackT<T>;
    PackCoef<T> p;
    p.one = PT::splat(T(1));
    p.m2 = PT::splat(T(-2));
    p.m4 = PT::splat(T(-4));
    p.c1 = PT::splat(c.c1dt);
    p.c2 = PT::splat(c.c2dt);
    p.c3 = PT::splat(c.c3dt);
    p.ct = PT::splat(c.ctdt);
    p.nkmu = PT::splat(c.nkmudt);
    p.nkap = PT::splat(c.nkapdt);
    for (int k = 0; k < kMaxTerms; ++k) {
        p.pair[k].nA = PT::splat(-c.A[k]);
        p.pair[k].nbeta = PT::splat(c.nbetadt[k]);
    }
    p.nterms = c.nterms;
    for (int i = 0; i <= kMaxTerms; ++i) {
        p.rat[i].num = PT::splat(i < kMaxTerms ? c.rnum[i] : T(0));
        p.rat[i].den = PT::splat(c.rden[i]);
    }
    p.deg = c.deg;
    p.guard = top_bits(c.q_lo);
    return p;
}

// ------------------------------------------------------ storage <-> compute

template <class S, class T> struct Io;

template <> struct Io<float, float> {
    static constexpr int VX = 4;
    static __device__ __forceinline__ void lds(const float *p, float *v)   // 16 B of shared
    {
        const float4 r = *reinterpret_cast<const float4 *>(p);
        v[0] = r.x; v[1] = r.y; v[2] = r.z; v[3] = r.w;
    }
    static __device__ __forceinline__ void st(float *p, const float *v)
    {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
    static __device__ __forceinline__ float cvt_in(float s) { return s; }
    static __device__ __forceinline__ float cvt_out(float t) { return t; }
};

template <> struct Io<double, double> {
    static constexpr int VX = 2;
    static __device__ __forceinline__ void lds(const double *p, double *v)
    {
        const double2 r = *reinterpret_cast<const double2 *>(p);
        v[0] = r.x; v[1] = r.y;
    }
    static __device__ __forceinline__ void st(double *p, const double *v)
    {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
    }
    static __device__ __forceinline__ double cvt_in(double s) { return s; }
    static __device__ __forceinline__ double cvt_out(double t) { return t; }
};

template <> struct Io<__nv_bfloat16, float> {
    static constexpr int VX = 8;
    static __device__ __forceinline__ void lds(const __nv_bfloat16 *p, float *v)
    {
        const uint4 r = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ void st(__nv_bfloat16 *p, const float *v)
    {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<uint32_t *>(&h);
        }
        *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    static __device__ __forceinline__ float cvt_in(__nv_bfloat16 s) { return __bfloat162float(s); }
    static __device__ __forceinline__ __nv_bfloat16 cvt_out(float t) { return __float2bfloat16_rn(t); }
};

// --------------------------------------------------------------- mbarrier

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// One test of the phase; a thread whose phase is not complete is suspended in
// hardware for up to the hint (ns) instead of spinning on issue slots.
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(1000000u)
        : "memory");
    return ok != 0;
}

// One test of the phase that does not wait.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the barrier phase with the given parity; false after ~2 s.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > kWaitCycles) return false;
    return true;
}

// Bulk asynchronous copy global -> shared, completing bytes on bar.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Producer-side wait: polls with a nanosleep back-off so a waiting producer does
// not take issue slots from the consumers; false after ~2 s.
__device__ __forceinline__ bool mbar_wait_sleep(uint64_t *bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned ns = 32;
    while (!mbar_try_wait(bar, parity)) {
        __nanosleep(ns);
        ns = ns < 256 ? 2 * ns : 256;
        if (clock64() - t0 > kWaitCycles) return false;
    }
    return true;
}

// TMA tile copy of a 3D box (x, y, z start in elements) into shared memory.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// -------------------------------------------------------------------- tile

#ifndef SPFM_ROWS_PER_THREAD
#define SPFM_ROWS_PER_THREAD 2
#endif

template <class S, class T, int TX, int TY, int RPT_ = SPFM_ROWS_PER_THREAD>
struct TileShape {
    static constexpr int VX = Io<S, T>::VX;
    static constexpr int NP = VX / 2;
    static constexpr int RPT = RPT_;   // rows of the tile per consumer thread
    static constexpr int W = TX * VX;
    static constexpr int SW = W + 2 * VX;   // staged row: one 16-byte chunk of halo per side
    static constexpr int ROWS = TY + 2;
    static constexpr int BOX_BYTES = ROWS * SW * (int)sizeof(S);          // one TMA box
    static constexpr int STAGE = ((BOX_BYTES + 127) / 128 * 128) / (int)sizeof(S);   // 128-B aligned
    static constexpr int NS = SPFM_STAGES;  // pipeline depth (planes)
    static constexpr int NCONS = TX * TY / RPT;   // consumer threads
    static constexpr int NTHREADS = NCONS + 32;
};

// Per plane and pack: c = phi, h = c1 dt F' + c2 dt E' (the plane as the centre
// plane of an output), g = c2 dt F' + c3 dt E' (as the plane above or below);
// with 6 neighbours h = F', with 18 g = F' (their coefficients are applied in
// the update, by FMA).
template <class T, int NP>
struct PlaneQ {
    using P = typename Pk<T>::P;
    P c[NP], h[NP], g[NP];
    // TI_n only: 1 or 2 where phi is at or beyond the lower or upper clamp of the
    // profile inversion, else 0: at the row's own cells (own), and at those and
    // their in-plane face neighbours (level)
    int own, level;
};

// ----------------------------------------------------------------- TI_n

// Inversion of the ideal profile, psi = (lambda/2) artanh(1 - 2 phi)
// = (lambda/4) ln((1 - phi)/phi), with phi clamped to [eps, 1 - eps] (TI_n).
// Only its differences are needed: log-odds(a) - log-odds(b)
// = log((1 - a) b / (a (1 - b))), FP32 in log2 as the difference of the two
// products' logarithms, FP64 the natural logarithm of their quotient; the
// kernels scale it by StepCoef::psi_grad.  For a = b the products are the same
// number, so the difference is exactly zero (a clamped region keeps the CF
// fallback).
__device__ __forceinline__ float2 clamp_pack(float2 v, float eps)
{
    return make_float2(fminf(fmaxf(v.x, eps), 1.0f - eps), fminf(fmaxf(v.y, eps), 1.0f - eps));
}
__device__ __forceinline__ D2 clamp_pack(D2 v, double eps)
{
    return {fmin(fmax(v.x, eps), 1.0 - eps), fmin(fmax(v.y, eps), 1.0 - eps)};
}
__device__ __forceinline__ float2 log_ratio(float2 n, float2 d)
{
    return make_float2(__log2f(n.x) - __log2f(d.x), __log2f(n.y) - __log2f(d.y));
}
__device__ __forceinline__ D2 log_ratio(D2 n, D2 d) { return {log(n.x / d.x), log(n.y / d.y)}; }
// a and b clamped; na = 1 - a, nb = 1 - b
template <class P>
__device__ __forceinline__ P log_odds_diff(P a, P na, P b, P nb)
{
    using K = Pk<decltype(P().x)>;
    return log_ratio(K::mul(na, b), K::mul(a, nb));
}
// phi at or beyond the clamp, for a set of cells given by the largest and
// smallest of their upper 32 bits as signed integers: 1 all at or below eps, 2
// all at or above 1 - eps, else 0 (FP64 compares the upper words, which at a
// limit's own upper word says 0: such cells take the general form, as they may)
__device__ __forceinline__ int clamp_level(int hi, int lo, float eps)
{
    return hi <= __float_as_int(eps) ? 1 : (lo >= __float_as_int(1.0f - eps) ? 2 : 0);
}
__device__ __forceinline__ int clamp_level(int hi, int lo, double eps)
{
    return hi < __double2hiint(eps) ? 1 : (lo > __double2hiint(1.0 - eps) ? 2 : 0);
}
// tanh of a pack.  FP32: Lambert's continued fraction for tanh truncated
// after the term x^2/11, x (10395 + 1260 y + 21 y^2) / (10395 + 4725 y + 210 y^2 + y^3)
// with y = x^2 (|error| < 3.3e-10 for |x| <= 1, < 3e-8 for |x| <= 1.5), written
// as x - x y (3465 + 189 y + y^2) / den so that the result is an FMA and sums
// of tanh values fuse nothing; callers whose arguments can exceed 1.5 pass
// small = false and get tanhf.  FP64: tanh.
template <class T> struct TanhPk;
template <> struct TanhPk<float> {
    static __device__ __forceinline__ float2 eval(float2 x, bool small)
    {
        if (!small) return make_float2(tanhf(x.x), tanhf(x.y));
        const float2 y = __fmul2_rn(x, x);
        const float2 poly = __ffma2_rn(__ffma2_rn(x, x, make_float2(189.f, 189.f)), y, make_float2(3465.f, 3465.f));
        const float2 den = __ffma2_rn(__ffma2_rn(__ffma2_rn(x, x, make_float2(210.f, 210.f)), y,
                                                 make_float2(4725.f, 4725.f)),
                                      y, make_float2(10395.f, 10395.f));
        const float2 r = Pk<float>::div(__fmul2_rn(y, poly), den);
        return __ffma2_rn(r, __ffma2_rn(x, make_float2(-1.f, -1.f), make_float2(0.f, 0.f)), x);
    }
};
template <> struct TanhPk<double> {
    static __device__ __forceinline__ D2 eval(D2 x, bool) { return {tanh(x.x), tanh(x.y)}; }
};

// ---------------------------------------------------- stochastic rounding

// Stochastic rounding of the update phi + inc to the storage type S (FP32 or
// BF16): with a the largest value of S not above the exact sum and g the
// spacing of S above a, the stored value is a + g with probability
// (phi + inc - a) / g and a otherwise, so that its expectation is the exact
// update; an exactly representable sum (inc = 0 in particular) is stored as
// is.  It is computed as round-down(phi + (inc + u g)) with u uniform in
// [0, 1) on a 2^-16 grid (16 bits of h per cell): since inc + u g spans
// exactly one spacing above a, the round-down lands on a or a + g.  The
// rounding of inc + u g in FP32 (2^-24 of g) is far below the step.
template <class S> struct MantBits;
template <> struct MantBits<float> { static constexpr int v = 23; };
template <> struct MantBits<__nv_bfloat16> { static constexpr int v = 7; };

// the largest BF16 value not above v (an FP32 value): truncation, away from zero
// where v is negative
__device__ __forceinline__ float bf16_round_down(float v)
{
    const uint32_t b = __float_as_uint(v);
    uint32_t low;   // 0xffff where the sign bit is set (the top byte's sign, replicated)
    asm("prmt.b32 %0, %1, 0, 0x44bb;" : "=r"(low) : "r"(b));
    return __uint_as_float((b + low) & 0xffff0000u);
}

template <class S>
__device__ __forceinline__ float2 sr_update(float2 ph, float2 inc, uint32_t h)
{
    constexpr int mb = MantBits<S>::v;
    float2 a = __fadd2_rd(ph, inc);
    if constexpr (mb == 7) { a.x = bf16_round_down(a.x); a.y = bf16_round_down(a.y); }
    // the power of two of a; times u 2^-mb, u g of above (u 2^-mb is exact: its 16
    // bits in the mantissa of (1 + u) 2^-mb)
    const float2 p = make_float2(__uint_as_float(__float_as_uint(a.x) & 0x7f800000u),
                                 __uint_as_float(__float_as_uint(a.y) & 0x7f800000u));
    constexpr uint32_t one = (uint32_t)(127 - mb) << 23;   // 2^-mb
    const float2 u = __fadd2_rn(make_float2(__uint_as_float(one | ((h << 7) & 0x007fff80u)),
                                            __uint_as_float(one | ((h >> 9) & 0x007fff80u))),
                                make_float2(-__uint_as_float(one), -__uint_as_float(one)));
    float2 x = __fadd2_rd(ph, __ffma2_rn(u, p, inc));
    if constexpr (mb == 7) { x.x = bf16_round_down(x.x); x.y = bf16_round_down(x.y); }
    return x;
}

// TI_n factor w = -dt (potential / q + 4 M dF / (lambda Gamma)) of a pack of
// cells with s = 1 - 2 phi, u = s^2 and the profile-inversion gradient g
// (Sec. 2.1, TI_n): n = g / |g|, t_i = tanh(2 dx n_i / lambda), the 13
// couplings a = N / D from the tanh addition theorem, and the potential sum
// sum_k 4 c_k a_k^2 / (1 - a_k^2 s^2) = sum_k 4 c_k N^2 / (D^2 - N^2 s^2).
// c_k is one value per shell, so each shell's terms are summed as one running
// fraction and the three shells are joined with one reciprocal.  Where
// |g| < 1e-8 the normal is undefined and the cell takes the CF potential.
template <class T, int STENCIL>
__device__ __forceinline__ typename Pk<T>::P ti_local_w(const StepCoef<T> &C, typename Pk<T>::P sg,
                                                        typename Pk<T>::P u, typename Pk<T>::P gx,
                                                        typename Pk<T>::P gy, typename Pk<T>::P gz)
{
    using K = Pk<T>;
    using P = typename K::P;
    const P one = K::mk(T(1), T(1));
    const P zero = K::mk(T(0), T(0));
    const P neg_u = K::sub(zero, u);   // -s^2
    const P g2 = K::fma(gx, gx, K::fma(gy, gy, K::mul(gz, gz)));
    const P kin = K::mul(K::mk(C.two_dx_over_lam, C.two_dx_over_lam), K::rsqrt(g2));
    const bool small = C.two_dx_over_lam <= T(1.5);
    const P a = TanhPk<T>::eval(K::mul(gx, kin), small);
    const P b = TanhPk<T>::eval(K::mul(gy, kin), small);
    const P c = TanhPk<T>::eval(K::mul(gz, kin), small);
    // (num, den) += n / d as one fraction
    auto acc = [&](P &num, P &den, P n, P d) {
        num = K::fma(num, d, K::mul(n, den));
        den = K::mul(den, d);
    };
    // shell 1: N = t_i, D = 1
    const P a2 = K::mul(a, a), b2 = K::mul(b, b), c2 = K::mul(c, c);
    P n1 = a2, d1 = K::fma(a2, neg_u, one);
    acc(n1, d1, b2, K::fma(b2, neg_u, one));
    acc(n1, d1, c2, K::fma(c2, neg_u, one));
    P num = K::mul(K::mk(T(-4) * C.dt * C.ck[0], T(-4) * C.dt * C.ck[0]), n1), den = d1;
    // Shells 2 and 3 come in pairs of directions whose couplings are
    // N = x +- y, D = y' +- x' for one (x, y, x', y').  With S = x^2 + y^2,
    // B = x'^2 + y'^2 (S and B are the squares summed over the pair), R = 2 x y
    // (= 2 x' y'), P = B - S u and v = 1 - u, the pair's two terms
    // n/d = (S +- R) / (P +- R v) add up to 2 (S P - R^2 v) / (P^2 - R^2 v^2).
    const P v = K::fma(K::sub(zero, sg), sg, one);   // 1 - s^2
    const P m4 = K::mk(T(-4), T(-4));
    auto pair = [&](P &pn, P &pd, P S, P B, P r) {   // r = x^2 y^2 = R^2 / 4
        const P Pv = K::fma(S, neg_u, B);
        const P rv = K::mul(r, v);
        acc(pn, pd, K::fma(rv, m4, K::mul(S, Pv)), K::fma(K::mul(rv, v), m4, K::mul(Pv, Pv)));
    };
    if (STENCIL >= 18 && C.ck[3] != T(0)) {
        // shell 2: (1,+-1,0), (0,1,+-1), (1,0,+-1): x, y = t_i, t_j and x', y' = t_i t_j, 1
        P n2 = zero, d2 = one;
        const P ab = K::mul(a2, b2), bc = K::mul(b2, c2), ac = K::mul(a2, c2);
        pair(n2, d2, K::fma(a, a, b2), K::fma(a2, b2, one), ab);
        pair(n2, d2, K::fma(b, b, c2), K::fma(b2, c2, one), bc);
        pair(n2, d2, K::fma(a, a, c2), K::fma(a2, c2, one), ac);
        acc(num, den, K::mul(K::mk(T(-8) * C.dt * C.ck[3], T(-8) * C.dt * C.ck[3]), n2), d2);
    }
    if (STENCIL >= 26 && C.ck[9] != T(0)) {
        // shell 3: tanh(x + y + z) = (tx + ty + tz + tx ty tz) / (1 + tx ty + ty tz + tx tz).
        // (1,1,+-1): N = al +- tz be, D = be +- tz al with al = tx + ty, be = 1 + tx ty;
        // (-1,1,1), (1,-1,1): the same with al = ty - tx, be = 1 - tx ty.
        P n3 = zero, d3 = one;
        const P al1 = K::add(a, b), be1 = K::fma(a, b, one);
        const P al2 = K::sub(b, a), be2 = K::fma(K::sub(zero, a), b, one);
        const P A1 = K::mul(al1, al1), B1 = K::mul(be1, be1);
        const P A2 = K::mul(al2, al2), B2 = K::mul(be2, be2);
        pair(n3, d3, K::fma(c2, B1, A1), K::fma(c2, A1, B1), K::mul(K::mul(A1, B1), c2));
        pair(n3, d3, K::fma(c2, B2, A2), K::fma(c2, A2, B2), K::mul(K::mul(A2, B2), c2));
        acc(num, den, K::mul(K::mk(T(-8) * C.dt * C.ck[9], T(-8) * C.dt * C.ck[9]), n3), d3);
    }
    const P nkmu = K::mk(-C.dt * C.kmu, -C.dt * C.kmu);
    const P w = K::fma(sg, K::div(num, den), nkmu);
    const P wcf = K::fma(sg, K::mk(-C.dt * C.kappa, -C.dt * C.kappa), nkmu);
    const T lim = T(1e-16);
    return K::mk(g2.x >= lim ? w.x : wcf.x, g2.y >= lim ? w.y : wcf.y);
}

// One staged row around a thread's cells: v[0] the cell to their left, v[1..VX]
// the cells, v[VX + 1] the one to their right.
template <class S, class T, int VX>
__device__ __forceinline__ void get_row(const S *r, T *v)
{
    Io<S, T>::lds(r, v + 1);
    v[0] = Io<S, T>::cvt_in(r[-1]);
    v[VX + 1] = Io<S, T>::cvt_in(r[VX]);
}

// Periodic images across the z faces of the 16 bytes of new cells at
// (x.., y, z) of an all-periodic grid: z + nz on plane 0, z - nz on plane
// nz - 1, each also shifted by the cells' x and y images (edges, corners).
template <class S>
__device__ __forceinline__ void store_z_images(const GridGeom &g, S *dst, int x, int y, int z, uint4 v,
                                               int ximg, int yimg)
{
    const bool zu[2] = {z == 0, z == g.nz - 1};
    const int zs[2] = {g.nz, -g.nz};
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        if (!zu[c]) continue;
        S *p = dst + cell_index(g, x, y, z + zs[c]);
        *reinterpret_cast<uint4 *>(p) = v;
        if (ximg) *reinterpret_cast<uint4 *>(p + ximg) = v;
        if (yimg) *reinterpret_cast<uint4 *>(p + yimg) = v;
        if (ximg && yimg) *reinterpret_cast<uint4 *>(p + yimg + ximg) = v;
    }
}

// ------------------------------------------------ ghosts of non-periodic faces

// Ghost value of a non-periodic face from its source cell v: the
// contact-angle value of Eq. 7 with the face's signed coupling a,
// (1 - a) v / (1 - a (2 v - 1)) = k1 v / (k2 - k3 v), or a copy (no-flux).
// FP32 takes the approximate reciprocal (the face kernel divides exactly, so
// the two differ in the last unit; the ghosts are not kept in memory here).
template <class T> struct FaceMap {
    T k1, k2, k3;
    bool copy;
};
template <class T>
__device__ __forceinline__ FaceMap<T> face_map(int bc, T a)
{
    return FaceMap<T>{T(1) - a, T(1) + a, T(2) * a, bc != SPFM_CONTACT};
}
__device__ __forceinline__ float face_value(float v, const FaceMap<float> &m)
{
    if (m.copy) return v;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__fmaf_rn(-m.k3, v, m.k2)));
    return m.k1 * v * r;
}
__device__ __forceinline__ double face_value(double v, const FaceMap<double> &m)
{
    return m.copy ? v : m.k1 * v / (m.k2 - m.k3 * v);
}

// The staged plane st (ROWS x SW, the tile plus halo) of a grid whose faces
// are all non-periodic gets the ghost values of the faces it touches, from the
// interior cells next to them, in the face kernel's order: the x ghost columns
// of every row, then the y ghost rows (x ghosts included).  Run by the 32
// lanes of the producer warp; no face kernel then runs between steps.
template <class S, class T, int VX, int SW, int ROWS>
__device__ __forceinline__ void fix_xy(S *st, const GridGeom &g, const T *aface, int x0, int y0, int W, int TY,
                                       int lane)
{
    const bool xlo = x0 == 0;
    const int xhi = (g.nx - 1 >= x0 && g.nx - 1 < x0 + W) ? g.nx - x0 + VX : -1;   // column of x = nx
    const bool ylo = y0 == 0;
    const int yhi = (g.ny - 1 >= y0 && g.ny - 1 < y0 + TY) ? g.ny - y0 + 1 : -1;    // row of y = ny
    if (xlo || xhi >= 0) {
        const FaceMap<T> ml = face_map<T>(g.bc[0], aface[0]), mh = face_map<T>(g.bc[1], aface[1]);
        for (int k = lane; k < ROWS; k += 32) {
            S *row = st + k * SW;
            if (xlo) row[VX - 1] = Io<S, T>::cvt_out(face_value(Io<S, T>::cvt_in(row[VX]), ml));
            if (xhi >= 0) row[xhi] = Io<S, T>::cvt_out(face_value(Io<S, T>::cvt_in(row[xhi - 1]), mh));
        }
        __syncwarp();
    }
    if (ylo) {
        const FaceMap<T> m = face_map<T>(g.bc[2], aface[2]);
        for (int c = lane; c < SW; c += 32) st[c] = Io<S, T>::cvt_out(face_value(Io<S, T>::cvt_in(st[SW + c]), m));
    }
    if (yhi >= 0) {
        const FaceMap<T> m = face_map<T>(g.bc[3], aface[3]);
        for (int c = lane; c < SW; c += 32)
            st[yhi * SW + c] = Io<S, T>::cvt_out(face_value(Io<S, T>::cvt_in(st[(yhi - 1) * SW + c]), m));
    }
}

// A z ghost plane (plane -1 or nz) staged from its adjacent interior plane
// (already carrying its x and y ghosts): every value shifted by the z face.
template <class S, class T, int SW, int ROWS>
__device__ __forceinline__ void fix_z(S *dst, const S *src, const GridGeom &g, const T *aface, int face, int lane)
{
    const FaceMap<T> m = face_map<T>(g.bc[face], aface[face]);
    for (int i = lane; i < ROWS * SW; i += 32) dst[i] = Io<S, T>::cvt_out(face_value(Io<S, T>::cvt_in(src[i]), m));
}

// phi + dt (Laplacian part of Eq. 1) of a pack from its plane records: t the
// z-neighbour differences, h of the centre plane, g of the planes below and
// above (6 neighbours: h = F'; 18: g = F'; 26: h, g with their coefficients).
// SR: the increment alone (phi is added in sr_update).  Products are summed by
// FMAs only.
template <bool SR, int STENCIL, class P, class PCoef>
__device__ __forceinline__ P laplace_update(const PCoef &PC, P t, P ph, P h, P gm, P gp)
{
    using K = Pk<decltype(P().x)>;
    P acc;
    if constexpr (STENCIL == 6) acc = K::fma(PC.c1, h, SR ? K::mul(PC.ct, t) : K::fma(PC.ct, t, ph));
    else acc = SR ? K::fma(PC.ct, t, h) : K::add(K::fma(PC.ct, t, ph), h);
    if constexpr (STENCIL == 18) acc = K::fma(PC.c2, K::add(gm, gp), acc);
    if constexpr (STENCIL == 26) acc = K::add(acc, K::add(gm, gp));
    return acc;
}

// The potential's sum group by group as one running fraction num / den, u = s^2.
template <class T>
__device__ __forceinline__ void sum_groups(const typename PackCoef<T>::Pair *pair, int n, typename Pk<T>::P u,
                                           typename Pk<T>::P &num, typename Pk<T>::P &den)
{
    using K = Pk<T>;
    using P = typename K::P;
    const P one = K::mk(T(1), T(1));
    const typename PackCoef<T>::Pair t0 = pair[0];
    P nu = t0.nbeta, de = K::fma(t0.nA, u, one);
#pragma unroll 1
    for (int k = 1; k < n; ++k) {
        const typename PackCoef<T>::Pair t = pair[k];
        const P d = K::fma(t.nA, u, one);
        nu = K::fma(nu, d, K::mul(t.nbeta, de));
        de = K::mul(de, d);
    }
    num = nu;
    den = de;
}

// The same as a call: it is rare, and inlined in the batch kernel it holds
// registers that the plane loop spills for.
template <class T>
__device__ __noinline__ void call_sum_groups(const typename PackCoef<T>::Pair *pair, int n, typename Pk<T>::P u,
                                             typename Pk<T>::P &num, typename Pk<T>::P &den)
{
    sum_groups<T>(pair, n, u, num, den);
}

// Whether this thread lets the next launch start at the end of its CTA: the first
// thread of a CTA that triggers counts.  A consumer, after its last plane, since
// the producer warp ends up to a ring of planes before it (us a step, trigger by
// the warp that ends first -> by a consumer: FP64 96^3 periodic 142 -> 95, contact
// 158 -> 112; FP32 64^3 periodic 3.6 -> 3.1, 128^3 channel 8.5 -> 8.0).  In FP32 and
// BF16 grids whose ghosts the producer builds the planes are released one by
// one, and there the warp that ends first is as good or better (64^3 contact 4.79
// against 4.88, 96^3 7.04 against 7.28).
template <class T>
__device__ __forceinline__ bool ends_launch(bool fwd)
{
    return (fwd && sizeof(T) == 4) || threadIdx.x == 0;
}

// KIND: the potential (spfm_internal.h).  Degrees below the kernel's are padded
// with zero coefficients, which changes no bit.  IMM: the coefficients PC are in
// memory (a batch's), the constants 1, -2, -4 immediates.
// One tile (bx, by) of planes zc0..zc1-1.  The stage ring continues across the
// tiles a CTA processes: plane i of this tile is ring slot base + i.  The
// producer waits for its copies in flight before returning when drain is set.
// Returns false when a bounded wait gave up (the error word is set).
// SR: stochastic rounding of the update (FP32 compute only), random bits from
// sr_hash(padded cell index xor sr_key).
template <class S, class T, int STENCIL, int KIND, int TX, int TY, int RPT_, bool IMG = false, bool SR = false,
          bool IMM = false>
__device__ __forceinline__ bool step_tile(const StepCoef<T> &C, const PackCoef<T> &PC,
                                          const S *__restrict__ src, S *__restrict__ dst,
                                          int *__restrict__ err, const CUtensorMap *tmap, int bx,
                                          int by, int zc0, int zc1, S *__restrict__ stages,
                                          uint64_t *full, uint64_t *empty, int base, bool drain,
                                          int mode = 0, uint32_t sr_key = 0, uint64_t *ready = nullptr,
                                          bool fwd = false, bool wait = false)
{
    static_assert(!SR || sizeof(T) == 4, "stochastic rounding is for FP32 compute");
    using Sh = TileShape<S, T, TX, TY, RPT_>;
    using K = Pk<T>;
    using P = typename K::P;
    constexpr int VX = Sh::VX, NP = Sh::NP, W = Sh::W, SW = Sh::SW, ROWS = Sh::ROWS;
    constexpr int STAGE = Sh::STAGE, NS = Sh::NS;
    constexpr bool kGlobal = KIND != 0 && KIND != kKindLocal;
    constexpr bool kGuard = KIND > 4;                       // q below q_lo: group by group
    constexpr int DEG = KIND > kKindFew ? KIND - kKindFew : KIND;

    // one, -2, -4: from the parameters, or immediates (IMM: PC is in memory)
    const P k1 = IMM ? K::mk(T(1), T(1)) : PC.one, k2 = IMM ? K::mk(T(-2), T(-2)) : PC.m2,
            k4 = IMM ? K::mk(T(-4), T(-4)) : PC.m4;
    const GridGeom &g = C.g;
    const int tid = threadIdx.x;
    const int x0 = bx * W, y0 = by * TY;
    const int nplanes = zc1 - zc0 + 2;   // planes zc0-1 .. zc1
    // the planes this tile stages hold ghosts that the producer warp has to build
    const bool ghosts = fwd && (x0 == 0 || x0 + W >= g.nx || y0 == 0 || y0 + TY >= g.ny || zc0 == 0 || zc1 == g.nz);

    if (tid >= Sh::NCONS) {
        // ------------------------------------------------------- producer warp
        // ghosts (a tile that touches a face of a grid whose faces are all
        // non-periodic): the whole warp builds the ghosts of the faces a staged
        // plane touches (fix_xy, fix_z) and then releases it to the consumers on
        // its "ready" barrier; otherwise one lane issues the copies and the
        // consumers wait on "full".
        const int plane_lane = tid - Sh::NCONS;
        if (!ghosts && plane_lane != 0) return true;
        const bool lead = plane_lane == 0;
        // the kernel may start while the previous launch still runs (programmatic
        // dependent launch): every box waits for it
        if (lead && wait) asm volatile("griddepcontrol.wait;" ::: "memory");
        // kSkipCopy (a test of the bounded waits): the first CTA never fills the
        // stage of its plane 1, so its consumers' wait for that stage gives up
        const bool skip = (mode & kSkipCopy) && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
        const bool zlo = ghosts && zc0 == 0, zhi = ghosts && zc1 == g.nz;
        auto stage = [&](int j) { return stages + ((base + j) % NS) * STAGE; };
        // the copy of plane i into its (free) stage
        auto issue = [&](int i) {
            const int s = (base + i) % NS;
            // the ready barriers' phases go on with the ring, also where a tile of
            // a batch does without them
            if (fwd && !ghosts) mbar_arrive(&ready[s]);
            if (skip && i == 1) return;
            if (tmap) {
                mbar_expect_tx(&full[s], (uint32_t)Sh::BOX_BYTES);
                // one box: padded x from the 16-byte chunk left of the tile (x0 + off
                // - VX, 16-byte aligned), padded rows y0.., padded plane zc0 + i;
                // out-of-range parts are zero-filled, never used
                tma_load_3d(stages + s * STAGE, tmap, x0 + g.off - VX, y0, zc0 + i, &full[s]);
            } else {
                // row by row (no tensor map): the box's rows that lie in the buffer
                const long long row0 = (long long)(x0 + g.off - VX);
                const int bytes_row = (int)min((long long)SW, (long long)g.pitch - row0) * (int)sizeof(S);
                const int nrows = min(ROWS, g.ny + 2 - y0);
                mbar_expect_tx(&full[s], (uint32_t)(bytes_row * nrows));
                const S *plane = src + (long long)(zc0 + i) * g.plane + (long long)y0 * g.pitch + row0;
                S *st = stages + s * STAGE;
                for (int r = 0; r < nrows; ++r)
                    bulk_g2s(st + r * SW, plane + (long long)r * g.pitch, (uint32_t)bytes_row, &full[s]);
            }
        };
        // The lanes' ghost stores precede, through ready, the consumers and empty, a
        // later copy into the same stage by the asynchronous proxy, which the barriers
        // alone do not order after stores of the generic proxy.
        auto release = [&](int j) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lead) mbar_arrive(&ready[(base + j) % NS]);
        };
        int issued = 0;
        bool ok = true;
        if (!ghosts) {
            for (; issued < nplanes; ++issued) {
                const int I = base + issued;
                if (I >= NS && !mbar_wait_sleep(&empty[I % NS], ((I / NS) - 1) & 1)) {
                    ok = false;
                    break;
                }
                issue(issued);
            }
        } else {
            // Copies and releases go on independently, whichever can: a copy when its
            // stage is free, a plane's release when it has landed, in order (plane 0
            // of a z- face, which is built from plane 1, after that one).  A fixed
            // lag of the releases behind the copies left the consumers one plane of
            // slack.
            int done = 0;
            long long idle_since = 0;
            while (done < nplanes) {
                bool moved = false;
                if (issued < nplanes) {
                    const int I = base + issued;
                    if (I < NS || __all_sync(0xffffffffu, mbar_test(&empty[I % NS], ((I / NS) - 1) & 1))) {
                        if (lead) issue(issued);
                        ++issued;
                        moved = true;
                    }
                }
                const int j = zlo && done < 2 ? 1 - done : done;
                if (j < issued && __all_sync(0xffffffffu, mbar_test(&full[(base + j) % NS], ((base + j) / NS) & 1))) {
                    if (zlo && j == 0) fix_z<S, T, SW, ROWS>(stage(0), stage(1), g, C.aface, 4, plane_lane);
                    else if (zhi && j == nplanes - 1)
                        fix_z<S, T, SW, ROWS>(stage(j), stage(j - 1), g, C.aface, 5, plane_lane);
                    else fix_xy<S, T, VX, SW, ROWS>(stage(j), g, C.aface, x0, y0, W, TY, plane_lane);
                    release(j);
                    ++done;
                    moved = true;
                }
                if (moved) {
                    idle_since = 0;
                } else {
                    const long long now = clock64();
                    if (idle_since == 0) idle_since = now;
                    if (__any_sync(0xffffffffu, now - idle_since > kWaitCycles)) {
                        ok = false;
                        break;
                    }
                    __nanosleep(40);
                }
            }
        }
        if (!lead) return ok;
        if (!ok) atomicOr(err, 1);
        // never leave with copies in flight: wait for each stage's copy (a stage
        // whose wait gives up does not stop the waits for the others)
        if (drain || !ok)
            for (int I = max(0, base + issued - NS); I < base + issued; ++I)
                if (!mbar_wait_sleep(&full[I % NS], (I / NS) & 1)) atomicOr(err, 2);
        return ok;
    }

    // ------------------------------------------------------------- consumers
    constexpr int RPT = Sh::RPT;
    const int tx = tid % TX, ty = (tid / TX) * RPT;   // first of the thread's RPT rows
    const int lane = tid & 31;
    const int gx = x0 + tx * VX;
    const int gy = y0 + ty;
    const S *rbase = stages + (ty + 1) * SW + VX + tx * VX;   // first own row in a stage
    S *out = dst + cell_index(g, gx, gy, zc0);                // first own row of the output plane
    // Periodic images (IMG: all faces periodic, nx a multiple of 2 VX, nx >= 4 VX,
    // ny >= 2): a cell in the first two 16-byte chunks of a row also goes to the
    // sector right of the row (x + nx), one in the last two chunks to the sector
    // left of it (x - nx); the two threads of a sector store it in one request.
    // Rows 0 and ny - 1 also go to the ghost rows across (y -+ ny), with the x
    // image.  The offsets (elements, 0 where a cell has no image) are recomputed
    // where they are used, so that the plane loop keeps only the flag live.
    auto ximg = [&]() { return gx < 2 * VX ? g.nx : (gx >= g.nx - 2 * VX ? -g.nx : 0); };
    auto yimg = [&](int r) {
        return gy + r == 0 ? g.ny * g.pitch : (gy + r == g.ny - 1 ? -g.ny * g.pitch : 0);
    };
    bool img = false;
    if constexpr (IMG) img = gx < 2 * VX || gx >= g.nx - 2 * VX || gy == 0 || gy + RPT >= g.ny;

    const int rows = gx < g.nx ? min(RPT, g.ny - gy) : 0;   // own rows inside the grid
    const bool whole = gx + VX <= g.nx;
    bool ok = true;
    auto body = [&](int i, PlaneQ<T, NP> (&m)[RPT], PlaneQ<T, NP> (&z)[RPT],
                    PlaneQ<T, NP> (&p)[RPT]) -> bool {
        const int I = base + i, s = I % NS;
        // warp-uniform: every lane waits (acquire), the warp goes on only if all saw it
        if (!__all_sync(0xffffffffu, mbar_wait(ghosts ? &ready[s] : &full[s], (I / NS) & 1))) {
            if (lane == 0) atomicOr(err, 4);
            ok = false;
            return false;
        }
        {
            // rows ty-1 .. ty+RPT of the stage (north halo, own rows, south halo)
            const S *r0 = rbase + s * STAGE - SW;
            T v[RPT + 2][VX + 2];
#pragma unroll
            for (int r = 0; r < RPT + 2; ++r) get_row<S, T, VX>(r0 + r * SW, v[r]);
            // a pack of row r, and the sums W + E of its cells: the left and right
            // neighbours straddle register pairs, so they are added one by one
            // instead of being moved into packs (512^3 TI_<120> 194.9 -> 188.7 us,
            // 384^3 BF16 with stochastic rounding 139.7 -> 127.7)
            auto cell = [&](int r, int q) { return K::mk(v[r][2 * q + 1], v[r][2 * q + 2]); };
            auto side = [&](int r, int q) {
                return K::mk(K::add1(v[r][2 * q], v[r][2 * q + 2]), K::add1(v[r][2 * q + 1], v[r][2 * q + 3]));
            };
            // TI_n reads the plane's neighbours again when it is the centre plane, and
            // releases it then
            if constexpr (KIND != kKindLocal) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
            } else {
                int hi[RPT + 2], lo[RPT + 2];
#pragma unroll
                for (int r = 0; r < RPT + 2; ++r) {
                    hi[r] = lo[r] = (int)top_bits(v[r][1]);
#pragma unroll
                    for (int e = 2; e <= VX; ++e) {
                        const int b = (int)top_bits(v[r][e]);
                        hi[r] = max(hi[r], b);
                        lo[r] = min(lo[r], b);
                    }
                }
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    const int w = (int)top_bits(v[r + 1][0]), e = (int)top_bits(v[r + 1][VX + 1]);
                    p[r].own = clamp_level(hi[r + 1], lo[r + 1], C.eps);
                    p[r].level = clamp_level(max(max(max(hi[r], hi[r + 1]), hi[r + 2]), max(w, e)),
                                             min(min(min(lo[r], lo[r + 1]), lo[r + 2]), min(w, e)), C.eps);
                }
            }
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const P c = cell(r + 1, q);
                    p[r].c[q] = c;
                    // F' = (W + E + N + S) - 4C, E' = (NW + NE + SW + SE) - 4C
                    const P f = K::fma(k4, c, K::add(side(r + 1, q), K::add(cell(r, q), cell(r + 2, q))));
                    // 6 neighbours: h = F' (c1 applied in the update's FMA); 18: g = F'
                    // (c2 applied to the sum of the two planes' g in one FMA)
                    if (STENCIL == 6) {
                        p[r].h[q] = f;
                    } else {
                        const P e = K::fma(k4, c, K::add(side(r, q), side(r + 2, q)));
                        p[r].h[q] = K::fma(PC.c2, e, K::mul(PC.c1, f));
                        p[r].g[q] = STENCIL == 26 ? K::fma(PC.c3, e, K::mul(PC.c2, f)) : f;
                    }
                }
            }
        }
        if (i >= 2) {
            const int oz = zc0 - 2 + i;   // output plane
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                if (r >= rows) continue;
                T outv[VX];
                // padded index of the row's first cell (32-bit, wraps): the cell's
                // part of the stochastic-rounding hash
                const uint32_t sr_row = SR ? (uint32_t)cell_index(g, gx, gy + r, oz) : 0u;
                if constexpr (kGlobal) {
                    // w = s (-dt) N(q) / D(q) - kmu dt by Horner's rule (2 DEG - 1 FMAs; the
                    // running fraction it replaces took 4 operations a group: 512^3
                    // TI_<120> 211.6 -> 194.9 us a step, 13 groups at 150 x 133 x 117
                    // 19.6 -> 12.4, a 64-grid sweep step 156 -> 92); a thread with a cell
                    // below the guard (or a grid without N / D) sums its coupling groups
                    // one by one as that fraction
                    auto pack = [&](int q, auto by_group) -> P {
                        const P ph = z[r].c[q];
                        const P t = K::second(m[r].c[q], p[r].c[q], ph);
                        // SR: the increment alone, phi is added once in sr_update
                        const P acc = laplace_update<SR, STENCIL>(PC, t, ph, z[r].h[q], m[r].g[q], p[r].g[q]);
                        const P sg = K::fma(k2, ph, k1);
                        const P q1 = K::bump(ph, k1);
                        P num, den;
                        if constexpr (by_group.value) {
                            if constexpr (IMM) call_sum_groups<T>(PC.pair, PC.nterms, K::mul(sg, sg), num, den);
                            else sum_groups<T>(PC.pair, PC.nterms, K::mul(sg, sg), num, den);
                        } else if constexpr (KIND == kKindAny) {
                            const int n = PC.deg;
                            num = PC.rat[n - 1].num;
                            den = K::fma(PC.rat[n].den, q1, PC.rat[n - 1].den);
#pragma unroll 1
                            for (int i = n - 2; i >= 0; --i) {
                                const typename PackCoef<T>::Ratio c = PC.rat[i];
                                num = K::fma(num, q1, c.num);
                                den = K::fma(den, q1, c.den);
                            }
                        } else {
                            num = PC.rat[DEG - 1].num;
                            den = K::fma(PC.rat[DEG].den, q1, DEG == 1 ? k1 : PC.rat[DEG - 1].den);
#pragma unroll
                            for (int i = DEG - 2; i >= 0; --i) {
                                const typename PackCoef<T>::Ratio c = PC.rat[i];
                                num = K::fma(num, q1, c.num);
                                den = K::fma(den, q1, i == 0 ? k1 : c.den);
                            }
                        }
                        const P w = K::fma(sg, K::div(num, den), PC.nkmu);
                        P o = K::fma(q1, w, acc);
                        if constexpr (SR) o = sr_update<S>(ph, o, sr_hash((sr_row + 2 * q) ^ sr_key));
                        outv[2 * q] = o.x;
                        outv[2 * q + 1] = o.y;
                        return q1;
                    };
                    bool groups = KIND == kKindAny && PC.deg == 0;
                    if (!groups) {
                        uint32_t low = 0u;
#pragma unroll
                        for (int q = 0; q < NP; ++q) {
                            const P q1 = pack(q, std::false_type{});
                            if constexpr (kGuard) low = max(low, max(top_bits(q1.x), top_bits(q1.y)));
                        }
                        if constexpr (kGuard) groups = low > PC.guard;
                    }
                    if constexpr (kGuard) {
                        if (groups) {
#pragma unroll
                            for (int q = 0; q < NP; ++q) pack(q, std::true_type{});
                        }
                    }
                } else {
                    P wl[NP];   // TI_n: w of the row
                    if constexpr (KIND == kKindLocal) {
                        // Where every face neighbour sits in the same clamp the gradient is
                        // zero and ti_local_w falls back to the CF potential: the bulk
                        // phases take that alone.  Elsewhere the in-plane neighbours are
                        // read again from the centre plane's stage, which keeps the
                        // profile inversion out of the plane records.  320^3 grain:
                        // 258 -> 125 us a step (at two rows a thread and half the warps
                        // 200: a CTA's planes wait for the warps inside the band).
                        const bool bulk = z[r].level != 0 && m[r].own == z[r].level && p[r].own == z[r].level;
                        if (bulk) {
#pragma unroll
                            for (int q = 0; q < NP; ++q)
                                wl[q] = K::fma(K::fma(k2, z[r].c[q], k1),
                                               K::mk(-C.dt * C.kappa, -C.dt * C.kappa),
                                               K::mk(-C.dt * C.kmu, -C.dt * C.kmu));
                        } else {
                            const S *row = rbase + ((I + NS - 1) % NS) * STAGE + r * SW;
                            T x[VX + 2], n[VX], s[VX];
                            get_row<S, T, VX>(row, x);
                            Io<S, T>::lds(row - SW, n);
                            Io<S, T>::lds(row + SW, s);
                            const T ep = C.eps;
                            const P s2 = K::mk(C.psi_grad, C.psi_grad);
                            auto diff = [&](P a, P b) {
                                a = clamp_pack(a, ep);
                                b = clamp_pack(b, ep);
                                return K::mul(log_odds_diff(a, K::sub(k1, a), b, K::sub(k1, b)), s2);
                            };
#pragma unroll
                            for (int q = 0; q < NP; ++q) {
                                const P sg = K::fma(k2, z[r].c[q], k1);
                                wl[q] = ti_local_w<T, STENCIL>(
                                    C, sg, K::mul(sg, sg),
                                    diff(K::mk(x[2 * q + 2], x[2 * q + 3]), K::mk(x[2 * q], x[2 * q + 1])),
                                    diff(K::mk(s[2 * q], s[2 * q + 1]), K::mk(n[2 * q], n[2 * q + 1])),
                                    diff(p[r].c[q], m[r].c[q]));
                            }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < NP; ++q) {
                        const P ph = z[r].c[q];
                        const P t = K::second(m[r].c[q], p[r].c[q], ph);
                        // phi + dt * Laplacian (SR: the increment alone, phi is added in sr_update)
                        const P acc = laplace_update<SR, STENCIL>(PC, t, ph, z[r].h[q], m[r].g[q], p[r].g[q]);
                        const P sg = K::fma(k2, ph, k1);               // s = 1 - 2 phi
                        const P q1 = K::bump(ph, k1);                     // q = phi (1 - phi)
                        P w;   // -dt (potential / q + 4 M dF / (lambda Gamma))
                        if (KIND == 0) {
                            // driving term -dt pref dF h'(phi) = q (nkmu f): f = 1 for h3,
                            // 5 q for h5, 1/(3 (1 - 2q)^2) for h_Abel
                            P drive = PC.nkmu;
                            if (C.interp == 1) {
                                drive = K::mul(PC.nkmu, K::mul(K::mk(T(5), T(5)), q1));
                            } else if (C.interp == 2) {
                                const P d = K::fma(K::mk(T(-2), T(-2)), q1, k1);
                                drive = K::div(PC.nkmu, K::mul(K::mk(T(3), T(3)), K::mul(d, d)));
                            }
                            w = K::fma(sg, PC.nkap, drive);
                        } else {
                            w = wl[q];
                        }
                        P o = K::fma(q1, w, acc);
                        if constexpr (SR) o = sr_update<S>(ph, o, sr_hash((sr_row + 2 * q) ^ sr_key));
                        outv[2 * q] = o.x;
                        outv[2 * q + 1] = o.y;
                    }
                }
                S *optr = out + r * g.pitch;
                if (whole) {
                    Io<S, T>::st(optr, outv);
                    if (IMG && img) {
                        const int xo = ximg(), yo = yimg(r);
                        if (xo) Io<S, T>::st(optr + xo, outv);
                        if (yo) {
                            Io<S, T>::st(optr + yo, outv);
                            if (xo) Io<S, T>::st(optr + yo + xo, outv);
                        }
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < VX; ++e)
                        if (gx + e < g.nx) optr[e] = Io<S, T>::cvt_out(outv[e]);
                }
            }
        }
        if constexpr (KIND == kKindLocal) {
            if (i >= 1) {   // the plane before this one has been the centre plane
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[(I + NS - 1) % NS]);
            }
        }
        if (i >= 2) out += g.plane;
        return i + 1 < nplanes;
    };

    PlaneQ<T, NP> q0[RPT], q1[RPT], q2[RPT];
    for (int i = 0;; i += 3) {
        if (!body(i, q1, q2, q0)) break;
        if (!body(i + 1, q2, q0, q1)) break;
        if (!body(i + 2, q0, q1, q2)) break;
    }
    // Images across the z faces, after the march so that the plane loop stays
    // free of them: the threads of a tile holding plane 0 or nz - 1 read back
    // their own stores of that plane (program order) and copy them.
    if (IMG && ok && gx < g.nx && (zc0 == 0 || zc1 == g.nz)) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int oz = e == 0 ? 0 : g.nz - 1;
            if (oz < zc0 || oz >= zc1 || (e == 1 && oz == 0)) continue;
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                if (gy + r >= g.ny) continue;
                const uint4 v = *reinterpret_cast<const uint4 *>(dst + cell_index(g, gx, gy + r, oz));
                store_z_images<S>(g, dst, gx, gy + r, oz, v, ximg(), yimg(r));
            }
        }
    }
    return ok;
}

// Resident CTAs per SM the register budget is sized for: three by default;
// the single-grid FP32 kernels fit four (96 registers, no spills, 20 warps per
// SM: 2 % faster for TI_<120>, 3-6 % for CF at 512^3), while FP64 spills
// there, and the persistent batch kernel keeps three.
template <class S> struct MinBlocks { static constexpr int value = SPFM_MIN_CTAS; };
template <> struct MinBlocks<float> { static constexpr int value = 4; };

// (The potentials with the guard on q keep three CTAs per SM: at four their
// registers spill; 150 x 133 x 117 with a random normal 12.4 us a step at three,
// 12.6 at four, and the guard in the kernels of 1 to 4 groups, which do not need
// it, cost 18 % at 512^3.  The stochastic-rounding kernels keep three too: four
// fit without spills and gain at the largest sizes, 512^3 TI 234.0 -> 233.0 us,
// 256^3 CF contact 38.8 -> 35.8, but lose at the small ones, 128^3 7.8 -> 8.2,
// 32^3 3.2 -> 3.5; BF16 likewise, 512^3 241 -> 235, 128^3 7.5 -> 7.9.)
template <class S, class T, int STENCIL, int KIND, int TX, int TY, int RPT_, bool IMG, bool SR = false>
__global__ void __launch_bounds__(TileShape<S, T, TX, TY, RPT_>::NTHREADS,
                                  KIND == kKindLocal ? 2 : ((SR || KIND > 4) ? SPFM_MIN_CTAS : MinBlocks<S>::value))
    spfm_step_kernel(const StepCoef<T> C, const PackCoef<T> PC, const S *__restrict__ src,
                     S *__restrict__ dst, int *__restrict__ err, int zchunk,
                     const __grid_constant__ CUtensorMap tmap, int use_tmap, int mode)
{
    using Sh = TileShape<S, T, TX, TY, RPT_>;
    if (mode & kEarly) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ __align__(128) S stages[Sh::NS * Sh::STAGE];
    __shared__ __align__(8) uint64_t full[Sh::NS], empty[Sh::NS], ready[Sh::NS];
    if (threadIdx.x == 0) {
        for (int s = 0; s < Sh::NS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], Sh::NCONS / 32);
            mbar_init(&ready[s], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int zc0 = blockIdx.z * zchunk;
    const int zc1 = min(zc0 + zchunk, C.g.nz);
    // no periodic face: the producer warp stages the ghosts of the faces
    bool fwd = false;
    if constexpr (!IMG) {
        fwd = true;
#pragma unroll
        for (int f = 0; f < 6; ++f) fwd = fwd && C.g.bc[f] != SPFM_PERIODIC;
    }
    step_tile<S, T, STENCIL, KIND, TX, TY, RPT_, IMG, SR>(C, PC, src, dst, err, use_tmap ? &tmap : nullptr,
                                                     blockIdx.x, blockIdx.y, zc0, zc1, stages, full, empty, 0,
                                                     true, mode, C.sr_key, ready, fwd, true);
    if (!(mode & kEarly) && ends_launch<T>(fwd)) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------------------- batches

// One grid of a batch as the persistent kernel reads it from device memory.
template <class T>
struct BatchGrid {
    CUtensorMap map[2];     // TMA maps of the two buffers (when has_map)
    StepCoef<T> C;
    PackCoef<T> PC;
    void *field[2];
    int cur;                // buffer holding the field at parity 0
    int has_map;
    CUtensorMap map_sq[2];  // the same for the box of the square tile shape (when has_map_sq)
    int has_map_sq;
};

// Persistent kernel over a packed work-list of items of one tile shape (TX,
// TY): CTA b takes items start[b] .. start[b + 1] - 1 (batch.cu balances
// them).  Step `parity` reads buffer cur ^ parity.  Every thread waits for the
// launch before (programmatic dependent launch: the next step's CTAs take the
// slots that this one's leave).  SQ: the items use the square tile's TMA maps (map_sq).
// SR: stochastic rounding, the step key of grid i from sr_step_key(its seed,
// steps[i] + sub).  fwd: no grid of the batch has a periodic face (the
// producer warp stages the ghosts of the faces; no ghost kernel runs).
template <class S, class T, int STENCIL, int KIND, int TX, int TY, bool SQ, bool SR = false>
__global__ void __launch_bounds__(TileShape<S, T, TX, TY>::NTHREADS, kBatchCtasPerSm)
    spfm_batch_kernel(const BatchGrid<T> *__restrict__ grids, const BatchList list, int parity,
                      int *__restrict__ err, const long long *__restrict__ steps, int sub, int fwd)
{
    using Sh = TileShape<S, T, TX, TY>;
    __shared__ __align__(128) S stages[Sh::NS * Sh::STAGE];
    __shared__ __align__(8) uint64_t full[Sh::NS], empty[Sh::NS], ready[Sh::NS];
    if (threadIdx.x == 0) {
        for (int s = 0; s < Sh::NS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], Sh::NCONS / 32);
            mbar_init(&ready[s], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    __shared__ __align__(32) unsigned char s_raw[(Sh::NCONS / 32) * sizeof(PackCoef<T>)];
    PackCoef<T> *s_pc = reinterpret_cast<PackCoef<T> *>(s_raw);
    if (list.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int base = 0;
    const int end = list.start[blockIdx.x + 1];
    for (int w = list.start[blockIdx.x]; w < end; ++w) {
        const BatchItem it = list.work[w];
        const BatchGrid<T> &bg = grids[it.grid];
        const int cur = bg.cur ^ parity;
        const CUtensorMap *map =
            SQ ? (bg.has_map_sq ? &bg.map_sq[cur] : nullptr) : (bg.has_map ? &bg.map[cur] : nullptr);
        if (map && threadIdx.x == Sh::NCONS)
            asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
        const bool last = w + 1 == end;
        const uint32_t key = SR ? sr_step_key(bg.C.sr_seed, steps[it.grid] + sub) : 0u;
        const int warp = threadIdx.x >> 5;
        // each consumer warp reads the item's coefficients from a copy of its own in
        // shared memory: from the grid record in global memory every row waited for
        // them (long_scoreboard a third of the stalls; 64-grid sweep 89.7 -> 85.7 us
        // a step, served window 293.8 -> 274.1)
        if (warp < Sh::NCONS / 32) {
            __syncwarp();
            const uint32_t *from = reinterpret_cast<const uint32_t *>(&bg.PC);
            uint32_t *to = reinterpret_cast<uint32_t *>(&s_pc[warp]);
            for (int k = threadIdx.x & 31; k < (int)(sizeof(PackCoef<T>) / 4); k += 32) to[k] = from[k];
            __syncwarp();
        }
        const PackCoef<T> &pc = s_pc[warp < Sh::NCONS / 32 ? warp : 0];
        if (!step_tile<S, T, STENCIL, KIND, TX, TY, SPFM_ROWS_PER_THREAD, false, SR, true>(
                bg.C, pc, (const S *)bg.field[cur], (S *)bg.field[cur ^ 1], err, map, it.bx, it.by, it.zc0,
                it.zc1, stages, full, empty, base, last, 0, key, ready, fwd != 0))
            return;
        base += it.zc1 - it.zc0 + 2;
    }
    if (!list.early && ends_launch<T>(fwd != 0)) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Work-list entries of one grid for the tile shape (TX, TY) of the (S, T)
// kernel, marked with the item shape index `shape`.
template <class S, class T, int TX, int TY>
inline int batch_items_t(const GridGeom &g, int grid_index, int zchunk, BatchItem *out, int shape = 0)
{
    using Sh = TileShape<S, T, TX, TY>;
    const int gxn = (g.nx + Sh::W - 1) / Sh::W, gyn = (g.ny + TY - 1) / TY;
    int n = 0;
    for (int z = 0; z < g.nz; z += zchunk)
        for (int by = 0; by < gyn; ++by)
            for (int bx = 0; bx < gxn; ++bx) {
                if (out) out[n] = BatchItem{grid_index, bx, by, z, min(z + zchunk, g.nz), shape};
                ++n;
            }
    return n;
}

template <class S, class T, int TX, int TY, bool SQ = false, bool SR = false>
cudaError_t launch_batch_t(const void *grids, BatchList list, int parity, int *err,
                           int stencil, int kind, cudaStream_t st, const long long *steps = nullptr,
                           int sub = 0, int fwd = 0)
{
    using Sh = TileShape<S, T, TX, TY>;
    if (list.ctas < 1) return cudaSuccess;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(list.ctas);
    lc.blockDim = dim3(Sh::NTHREADS);
    lc.stream = st;
    lc.attrs = attr;
    lc.numAttrs = 1;
    cudaError_t le = cudaSuccess;
    const BatchGrid<T> *bg = (const BatchGrid<T> *)grids;
#define SPFM_BLAUNCH(ST, KD)                                                                                \
    le = cudaLaunchKernelEx(&lc, spfm_batch_kernel<S, T, ST, KD, TX, TY, SQ, SR>, bg, list, parity, err, steps, sub, \
                            fwd)
#define SPFM_BBY_KIND(ST)                      \
    do {                                       \
        if (kind == 0) SPFM_BLAUNCH(ST, 0);    \
        else if (kind <= kKindFew + 4) SPFM_BLAUNCH(ST, kKindFew + 4); \
        else if (kind <= kKindFew + 6) SPFM_BLAUNCH(ST, kKindFew + 6); \
        else SPFM_BLAUNCH(ST, kKindAny);       \
    } while (0)
    if (stencil == 6) SPFM_BBY_KIND(6);
    else if (stencil == 18) SPFM_BBY_KIND(18);
    else SPFM_BBY_KIND(26);
#undef SPFM_BBY_KIND
#undef SPFM_BLAUNCH
    if (le != cudaSuccess) return le;
    return cudaGetLastError();
}

// IMG: the kernels that write the periodic ghost images (cfg.mode has kImages)
// TI_n on the square tile LTX, LTY (tmap is then that tile's map)?  A warp of it
// covers 32 x 4 cells instead of 64 x 2, so fewer warps touch the interface
// band, whose cells cost several times those of the bulk; where the band fills
// much of the grid that gains nothing and the tile's wider x halo costs.  The
// line lies at an extent of 32 lambda, about 4.5 band widths (FP32 27-point, us a
// step, wide -> square: lambda = 3: 320^3 118.6 -> 112.1, 96^3 14.1 -> 12.2;
// lambda = 6: 256^3 88.0 -> 79.4, 192^3 55.8 -> 57.3, 128^3 23.3 -> 24.7).
template <class T>
inline bool local_square(const StepCoef<T> &c, int scheme)
{
    const int n = min(c.g.nx, min(c.g.ny, c.g.nz));
    return scheme == SPFM_TI_LOCAL && n * c.two_dx_over_lam >= T(64);
}

template <class S, class T, int TX, int TY, bool IMG, bool SR = false, int LTX = TX, int LTY = TY>
cudaError_t launch_step_t(const StepCoef<T> &c, const S *src, S *dst, int *err, LaunchCfg cfg,
                          const CUtensorMap *tmap, cudaStream_t st)
{
    using Lo = TileShape<S, T, LTX, LTY, 1>;
    const int kind = grid_kind(cfg.scheme, c.deg, isinf(c.q_lo));
    const bool square = LTX != TX && local_square(c, cfg.scheme);
    const int tw = square ? Lo::W : TileShape<S, T, TX, TY>::W, th = square ? LTY : TY;
    const int gxn = (c.g.nx + tw - 1) / tw, gyn = (c.g.ny + th - 1) / th;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int target = 6 * MinBlocks<S>::value * sms;
    const PackCoef<T> pc = make_pack_coef<T>(c);
    CUtensorMap map;
    if (tmap) map = *tmap;
    else memset(&map, 0, sizeof map);
    const int use = tmap ? 1 : 0;
    // Rows per thread: two, and one for BF16, whose threads take eight cells of a
    // row: with two a CTA had two consumer warps of 168 registers, six an SM
    // (384^3 TI_<120>, three CTAs per SM: 181 -> 140 us a step with stochastic
    // rounding, 97 -> 92 without; 64^3 8.6 -> 6.0)
    constexpr int R = sizeof(S) == 2 ? 1 : SPFM_ROWS_PER_THREAD;
    constexpr int NT1 = TileShape<S, T, TX, TY, 1>::NTHREADS;
    // programmatic dependent launch: the kernel may begin while the previous
    // kernel in the stream runs (griddepcontrol.wait)
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.dynamicSmemBytes = 0;
    lc.stream = st;
    lc.attrs = attr;
    lc.numAttrs = 1;
    int mode = cfg.mode;
    // z-chunk: the caller's, else the launch-shape model's for this kernel (a
    // grid dimension stays below 65536 chunks)
    auto go = [&](auto kern, int threads) {
        int zchunk = cfg.zchunk > 0 ? cfg.zchunk
                                    : pick_zchunk((const void *)kern, threads, gxn * gyn, c.g.nz, target,
                                                  kind == kKindLocal ? kUneven : sizeof(T) == 8 ? kFp64 : kStream);
        if (zchunk > c.g.nz) zchunk = c.g.nz;
        if (zchunk < (c.g.nz + 65534) / 65535) zchunk = (c.g.nz + 65534) / 65535;
        if (cfg.zchunk_used) *cfg.zchunk_used = zchunk;
        lc.gridDim = dim3(gxn, gyn, (c.g.nz + zchunk - 1) / zchunk);
        if ((long long)gxn * gyn * lc.gridDim.z >= 4LL * sms * MinBlocks<S>::value) mode |= kEarly;
        lc.blockDim = dim3(threads);
        return cudaLaunchKernelEx(&lc, kern, c, pc, src, dst, err, zchunk, map, use, mode);
    };
    cudaError_t le = cudaSuccess;
#define SPFM_LAUNCH(ST, KD) \
    le = go(spfm_step_kernel<S, T, ST, KD, TX, TY, R, IMG, SR>, TileShape<S, T, TX, TY, R>::NTHREADS)
#define SPFM_BY_KIND(ST)                        \
    do {                                        \
        if (kind == 0) SPFM_LAUNCH(ST, 0);      \
        else if (kind == 1) SPFM_LAUNCH(ST, 1); \
        else if (kind == 2) SPFM_LAUNCH(ST, 2); \
        else if (kind == 3) SPFM_LAUNCH(ST, 3); \
        else if (kind == 4) SPFM_LAUNCH(ST, 4); \
        else if (kind == kKindFew + 4) SPFM_LAUNCH(ST, kKindFew + 4); \
        else if (kind == kKindFew + 6) SPFM_LAUNCH(ST, kKindFew + 6); \
        else if (kind == kKindAny) SPFM_LAUNCH(ST, kKindAny); \
        else if (square) le = go(spfm_step_kernel<S, T, ST, kKindLocal, LTX, LTY, 1, IMG, SR>, Lo::NTHREADS); \
        else le = go(spfm_step_kernel<S, T, ST, kKindLocal, TX, TY, 1, IMG, SR>, NT1); \
    } while (0)
    if (cfg.stencil == 6) SPFM_BY_KIND(6);
    else if (cfg.stencil == 18) SPFM_BY_KIND(18);
    else SPFM_BY_KIND(26);
#undef SPFM_BY_KIND
#undef SPFM_LAUNCH
    if (le != cudaSuccess) return le;
    return cudaGetLastError();
}

}  // namespace spfm
