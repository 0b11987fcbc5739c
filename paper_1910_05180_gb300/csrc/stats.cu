// stats.cu -- ideal-profile initialisation and FP64 interface
// diagnostics on the ghosted field layout (spfm_internal.h).
//
// init: Eq. 3 (planar), its radial form, or a cube as the product of three 1D
// profiles (the start of the Sec. 3.3 shape relaxation), evaluated in FP64 per cell and
// rounded once to the storage type (the caller then fills the ghost layer).
//
// stats: one pass over the interior with sums per lane in a fixed order
// (double-float pairs for the band sums, FP64 otherwise, see below), then
// FP64 warp-shuffle and shared-memory block reductions into
// kStatsBlocks partials, then one CTA reducing the partials in a fixed order,
// so the result is bit-reproducible for a given grid size.  Sums over the band
// 1e-6 < phi < 1 - 1e-6 invert the ideal profile (Sec. 2.3):
//   position  c = sum q (p.n - (lambda/2) artanh(1-2phi)) / sum q
//   radius    R = sum q (|p - ctr| + (lambda/2) artanh(1-2phi)) / sum q
// The optional interface energy is Eq. 1 at dF = 0; its forward differences
// read the ghost layer.
#include <math.h>

#include <mutex>

#include "spfm_internal.h"

namespace spfm {

template <class S> __device__ __forceinline__ double rd(const S *f, long long i);
template <> __device__ __forceinline__ double rd<double>(const double *f, long long i) { return f[i]; }
template <> __device__ __forceinline__ double rd<float>(const float *f, long long i) { return (double)f[i]; }
template <> __device__ __forceinline__ double rd<__nv_bfloat16>(const __nv_bfloat16 *f, long long i)
{
    return (double)__bfloat162float(f[i]);
}

template <class S> __device__ __forceinline__ S wr(double v);
template <> __device__ __forceinline__ double wr<double>(double v) { return v; }
template <> __device__ __forceinline__ float wr<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ __nv_bfloat16 wr<__nv_bfloat16>(double v)
{
    return __float2bfloat16_rn((float)v);
}

template <class S>
__global__ void init_kernel(const InitArgs a, S *f)
{
    const long long rows = (long long)(a.g.ny + 2) * (a.g.nz + 2);
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
        const int j = (int)(row % (a.g.ny + 2)) - 1;
        const int k = (int)(row / (a.g.ny + 2)) - 1;
        S *r = f + row * a.g.pitch;
        const bool inner = j >= 0 && j < a.g.ny && k >= 0 && k < a.g.nz;
        for (int x = threadIdx.x; x < a.g.pitch; x += blockDim.x) {
            const int i = x - a.g.off;
            double v = 0.0;
            if (inner && i >= 0 && i < a.g.nx) {
                const double px = a.dx * i, py = a.dx * j, pz = a.dx * k;
                if (a.shape == 1) {
                    const double rx = px - a.ctr[0], ry = py - a.ctr[1], rz = pz - a.ctr[2];
                    const double rr = sqrt(rx * rx + ry * ry + rz * rz);
                    v = 0.5 * (1.0 - tanh(2.0 * (a.R - rr) / a.lambda));
                } else if (a.shape == 2) {
                    // cube: product of the three 1D particle fractions
                    const double d[3] = {px - a.ctr[0], py - a.ctr[1], pz - a.ctr[2]};
                    double inside = 1.0;
                    for (int ax = 0; ax < 3; ++ax) inside *= 0.5 * (1.0 - tanh(2.0 * (fabs(d[ax]) - a.half) / a.lambda));
                    v = 1.0 - inside;
                } else {
                    const double pn = px * a.n[0] + py * a.n[1] + pz * a.n[2];
                    v = 0.5 * (1.0 - tanh(2.0 * (pn - a.c) / a.lambda));
                }
            }
            r[x] = wr<S>(v);
        }
    }
}

cudaError_t launch_init(const InitArgs &a, void *field, cudaStream_t st)
{
    const long long rows = (long long)(a.g.ny + 2) * (a.g.nz + 2);
    const int blocks = (int)(rows < 8192 ? rows : 8192);
    if (a.dtype == SPFM_F64) init_kernel<double><<<blocks, 128, 0, st>>>(a, (double *)field);
    else if (a.dtype == SPFM_F32) init_kernel<float><<<blocks, 128, 0, st>>>(a, (float *)field);
    else init_kernel<__nv_bfloat16><<<blocks, 128, 0, st>>>(a, (__nv_bfloat16 *)field);
    return cudaGetLastError();
}

// Eq. 6 (TI) or the CF quartic per direction; lam2_r2 = lambda^2/|r_k|^2
__device__ __forceinline__ double potential(double phi, double a, double lam2_r2, int cf)
{
    const double q = phi * (1.0 - phi), s = 1.0 - 2.0 * phi;
    if (cf) return 8.0 * q * q / 3.0;
    const double A = a * a;
    if (A < 1e-8) return lam2_r2 * 2.0 * A * q * q;
    return lam2_r2 * (q + (1.0 - A) / (4.0 * A) * log((1.0 - A) / (1.0 - A * s * s)));
}

// One block's (256 threads) partial from the sums of its threads.  An FP64
// instruction of a warp holds the pipe 16 cycles for the whole SM, so the sums
// are added 8 values a lane from shared memory before they are shuffled (13
// instructions a sum, against 45 by shuffles in every warp), and the extrema
// and the count stay out of FP64.
template <class R>
__device__ __forceinline__ R fewest(R a, R b) { return b < a ? b : a; }
template <class R>
__device__ __forceinline__ R most(R a, R b) { return b > a ? b : a; }
constexpr int kSums = 5;   // volume, S_w, S_c, S_r, energy
__device__ __forceinline__ int sum_slot(int s) { return s < 4 ? s : 7; }   // of a partial
template <class R>
__device__ __forceinline__ void block_reduce_store(const double (&sum)[kSums], R mn, R mx, double count, double *out)
{
    __shared__ double sm[kSums][256];
    __shared__ R ext[2][8];
    __shared__ double cnt[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int s = 0; s < kSums; ++s) sm[s][threadIdx.x] = sum[s];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        mn = fewest(mn, __shfl_down_sync(0xffffffffu, mn, off));
        mx = most(mx, __shfl_down_sync(0xffffffffu, mx, off));
    }
    // counts are rare: a warp without one adds nothing
    if (__any_sync(0xffffffffu, count != 0.0))
        for (int off = 16; off > 0; off >>= 1) count += __shfl_down_sync(0xffffffffu, count, off);
    if (lane == 0) {
        ext[0][warp] = mn;
        ext[1][warp] = mx;
        cnt[warp] = count;
    }
    __syncthreads();
    if (warp < kSums) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += sm[warp][32 * w + lane];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) out[sum_slot(warp)] = v;
    } else if (warp == kSums && lane == 0) {
        R lo = ext[0][0], hi = ext[1][0];
        double n = cnt[0];
        for (int w = 1; w < 8; ++w) {
            lo = fewest(lo, ext[0][w]);
            hi = most(hi, ext[1][w]);
            n += cnt[w];
        }
        out[4] = (double)lo;
        out[5] = (double)hi;
        out[6] = n;
        for (int i = 8; i < kNStat; ++i) out[i] = 0.0;
    }
}

// Per-lane partials: [0] sum phi, [1] S_w, [2] S_c, [3] S_r, [4] min, [5] max,
// [6] non-finite count, [7] energy density sum, [8..11] unused.
//
// The pass is bound by the FP64 work of the band cells (GB300 issues FP64 at
// 1/64 of the FP32 rate), so everything else stays out of FP64:
//   - each warp walks whole rows with 16-byte loads; finiteness, min, max and
//     the band test run in the storage precision, where they are exact (the
//     band limits 1e-6 and 1 - 1e-6 are not floats, so the first float above
//     and the last float below them decide exactly the same cells);
//   - an FP32 field's volume is summed per lane and four sweeps as unevaluated
//     pairs (TwoSum, Knuth TAOCP vol. 2, 4.2.2), two chains on the paired FP32
//     instructions, carried in 2^-48 fixed point;
//   - a row of cells is taken as finite and tested for band cells as a whole (a
//     sum that is not finite has the lane look at its cells one by one; one
//     minimum of |phi - 1/2| over 16 cells says whether any may lie in the band),
//     so the cells of the bulk phases cost about 6 instructions each;
//   - band cells are queued per warp and evaluated 32 at a time, so the
//     inversion of the profile runs with every lane busy.
template <class S> struct Scr { using T = float; };
template <> struct Scr<double> { using T = double; };
template <class S> __device__ __forceinline__ typename Scr<S>::T scr(const S *f, long long i);
template <> __device__ __forceinline__ double scr<double>(const double *f, long long i) { return f[i]; }
template <> __device__ __forceinline__ float scr<float>(const float *f, long long i) { return f[i]; }
template <> __device__ __forceinline__ float scr<__nv_bfloat16>(const __nv_bfloat16 *f, long long i)
{
    return __bfloat162float(f[i]);
}

// 16 bytes of a row as storage elements, widened to the screening type
template <class S> struct Row16;
template <> struct Row16<float> {
    static constexpr int E = 4;
    static __device__ __forceinline__ float get(const uint4 &w, int e)
    {
        return __uint_as_float(e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w);
    }
};
template <> struct Row16<__nv_bfloat16> {
    static constexpr int E = 8;
    static __device__ __forceinline__ float get(const uint4 &w, int e)
    {
        const unsigned u = (e >> 1) == 0 ? w.x : (e >> 1) == 1 ? w.y : (e >> 1) == 2 ? w.z : w.w;
        return __uint_as_float((e & 1) ? (u & 0xffff0000u) : (u << 16));
    }
};
template <> struct Row16<double> {
    static constexpr int E = 2;
    static __device__ __forceinline__ double get(const uint4 &w, int e)
    {
        return e == 0 ? __hiloint2double((int)w.y, (int)w.x) : __hiloint2double((int)w.w, (int)w.z);
    }
};

// cell k of the storage elements in the words u
template <class S> __device__ __forceinline__ typename Scr<S>::T word_cell(const unsigned *u, int k);
template <> __device__ __forceinline__ float word_cell<float>(const unsigned *u, int k)
{
    return __uint_as_float(u[k]);
}
template <> __device__ __forceinline__ float word_cell<__nv_bfloat16>(const unsigned *u, int k)
{
    return __uint_as_float((k & 1) ? (u[k / 2] & 0xffff0000u) : (u[k / 2] << 16));
}
template <> __device__ __forceinline__ double word_cell<double>(const unsigned *u, int k)
{
    return __hiloint2double((int)u[2 * k + 1], (int)u[2 * k]);
}

// 1e-6 < x < 1 - 1e-6 for an FP32 x: the limits are not FP32 numbers, so the
// test compares with the first float above 1e-6 and the last float below
// 1 - 1e-6 (written out: a rounding conversion here would run on the FP64 pipe
// for every cell)
__device__ __forceinline__ bool in_band(float x)
{
    return x >= 0x1.0c6f7cp-20f && x <= 0x1.ffffdep-1f;
}
__device__ __forceinline__ bool in_band(double x) { return x > 1e-6 && x < 1.0 - 1e-6; }

// the upper words of 1e-6 and 1 - 1e-6 bound those of the band's cells
constexpr unsigned kBandLo = 0x3eb0c6f7u, kBandHi = 0x3feffffdu;
// a double's bits as a signed integer of the same order (-0 below +0), and back
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double key_value(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

// y * 2^48 truncated toward zero, for |y| < 2^14 (the bits below 2^-48 drop)
__device__ __forceinline__ long long fix48(float y)
{
    const unsigned b = __float_as_uint(y);
    const int E = (int)((b >> 23) & 0xffu);
    if (E < 78) return 0;   // |y| < 2^-49
    const long long m = (long long)((b & 0x7fffffu) | 0x800000u);   // |y| = m 2^(E - 150)
    const int sh = E - 102;
    const long long v = sh >= 0 ? (m << sh) : (m >> (-sh));
    return (b >> 31) ? -v : v;
}

// Volume of one lane.  FP32 values: unevaluated pairs s + c (TwoSum) over four
// sweeps, that is 64 cells a lane, then the pair in 2^-48 fixed point, carried
// into FP64 before the fixed point could overflow.  The sums s are exact but for
// what c takes; c is an FP32 sum of up to 32 such remainders a chain: for cells in
// [0, 1] each is at most 2^-20 and c at most 2^-15, so its roundings add up to
// 32 * 2^-40 = 3e-11 at the very most per four sweeps, typically 1e-14 (random
// profiles), beside the 2^-48 that the fixed point drops.  The count is of sweeps,
// not of rows, so that the chains stay that short where a row has more than one.
template <class R> struct VolSum;
template <> struct VolSum<float> {
    float2 s = {0.0f, 0.0f}, c = {0.0f, 0.0f};   // two chains
    long long fix = 0;
    double sum = 0.0;
    int sweeps = 0, flushes = 0;
    static __device__ __forceinline__ float2 sub(float2 a, float2 b)
    {
        return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
    }
    __device__ __forceinline__ void add(float2 x)
    {
        const float2 t = __fadd2_rn(s, x), z = sub(t, s);
        c = __fadd2_rn(c, __fadd2_rn(sub(s, sub(t, z)), sub(x, z)));
        s = t;
    }
    __device__ __forceinline__ void add(float x) { add(make_float2(x, 0.0f)); }
    __device__ __forceinline__ bool finite() const { return isfinite(s.x) && isfinite(s.y); }
    __device__ __forceinline__ float4 row() const { return make_float4(s.x, s.y, c.x, c.y); }
    __device__ __forceinline__ void set_row(float4 r)
    {
        s = make_float2(r.x, r.y);
        c = make_float2(r.z, r.w);
    }
    // the chains into fixed point
    __device__ __forceinline__ void flush()
    {
        const DF t = df_two_sum(s.x, s.y);
        const float lo = (c.x + c.y) + t.lo;
        if (fabsf(t.hi) < 256.0f && fabsf(lo) < 256.0f) fix += fix48(t.hi) + fix48(lo);
        else sum += (double)t.hi + (double)lo;
        set_row(make_float4(0.0f, 0.0f, 0.0f, 0.0f));
        if (++flushes == 32) {
            sum += (double)fix * 0x1p-48;
            fix = 0;
            flushes = 0;
        }
    }
    __device__ __forceinline__ void end_sweep()
    {
        if ((++sweeps & 3) == 0) flush();
    }
    __device__ __forceinline__ double total()
    {
        flush();
        return sum + (double)fix * 0x1p-48;
    }
};
template <> struct VolSum<double> {
    double sum = 0.0;
    __device__ __forceinline__ void add(double x) { sum += x; }
    __device__ __forceinline__ int row() const { return 0; }
    __device__ __forceinline__ void end_sweep() {}
    __device__ __forceinline__ double total() const { return sum; }
};

// Tables of the band evaluation, as double-float pairs written from FP64:
// g_ln_tab[j] = (ln F_j, 1/F_j) for F_j = 1 + j/256, g_kln2[k + 64] = k ln 2.
__device__ float4 g_ln_tab[256];
__device__ float2 g_kln2[128];

__global__ void ln_table_kernel()
{
    const int j = threadIdx.x;
    const double F = 1.0 + j / 256.0;
    const DF l = df_of(log(F)), r = df_of(1.0 / F);
    g_ln_tab[j] = make_float4(l.hi, l.lo, r.hi, r.lo);
    if (j < 128) {
        const DF k = df_of((double)(j - 64) * 0.69314718055994530942);
        g_kln2[j] = make_float2(k.hi, k.lo);
    }
}

// ln y for y = hi + lo in [2^-63, 2^63], table-driven (Tang, ACM TOMS 16, 1990):
// hi = 2^k m, m in [1, 2); F = 1 + j/256 takes the top 8 fraction bits of m, so
// f = (m - F) + lo 2^-k holds y 2^-k - F to double-float accuracy and u = f/F
// lies in (-2^-24, 2^-8).  ln(1 + u) is its Taylor series: u - u^2/2 in
// double-float, the terms u^3/3 - u^4/4 + u^5/5 (below 2e-8) in FP32,
// truncation below u^6/6 < 6e-16.  Returned as k, ln F and ln(1 + u).
struct LnParts {
    int k;
    DF lnF, s;
};
__device__ __forceinline__ LnParts ln_parts(DF y, const float4 *tab)
{
    const int bits = __float_as_int(y.hi);
    LnParts r;
    r.k = ((bits >> 23) & 0xff) - 127;
    const int j = (bits >> 15) & 0xff;
    const float m = __int_as_float((bits & 0x007fffff) | 0x3f800000);
    const float F = __int_as_float(0x3f800000 | (j << 15));
    const float lo = __fmul_rn(y.lo, __int_as_float((127 - r.k) << 23));   // lo 2^-k, exact
    const float4 t = tab[j];
    r.lnF = {t.x, t.y};
    const DF u = df_mul(df_two_sum(__fsub_rn(m, F), lo), DF{t.z, t.w});
    const DF u2 = df_mul(u, u);
    const float uh = u.hi;
    const float tail = uh * uh * uh * fmaf(uh, fmaf(uh, 0.2f, -0.25f), 1.0f / 3.0f);
    r.s = df_add(df_add(u, DF{-0.5f * u2.hi, -0.5f * u2.lo}), DF{tail, 0.0f});
    return r;
}

// one band cell waiting in its warp's queue: value, x index, and its row's
// share of p.n and of |p - ctr|^2
template <class R> struct BandCell {
    R phi;
    int i;
    DF pn_row, ryz2;
};

// Sec. 2.3 sums of one band cell, in double-float: q = phi(1 - phi),
// psi = (lambda/2) artanh(1 - 2 phi) = (lambda/4) ln((1 - phi) / phi), one
// logarithm of a double-float quotient, p = dx (i, j, k).  Absolute error of psi
// below about 1e-13.
template <class R> struct BandPhi;
template <> struct BandPhi<float> {   // FP32 and BF16 storage: phi exact, 1 - phi exact as a pair
    static __device__ __forceinline__ void get(float x, DF &ph, DF &om)
    {
        ph = {x, 0.0f};
        om = df_fast_sum(1.0f, -x);
    }
};
template <> struct BandPhi<double> {  // FP64 storage: 1 - phi in FP64, then both as pairs
    static __device__ __forceinline__ void get(double x, DF &ph, DF &om)
    {
        ph = df_of(x);
        om = df_of(1.0 - x);
    }
};
struct BandSums {
    DF w{0.0f, 0.0f}, c{0.0f, 0.0f}, r{0.0f, 0.0f};   // S_w, S_c, S_r
};
template <class R>
__device__ __forceinline__ void band_cell(const BandConst &bc, const BandCell<R> &c, const float4 *tab,
                                          const float2 *kln2, BandSums &acc)
{
    DF ph, om;
    BandPhi<R>::get(c.phi, ph, om);
    const DF q = df_mul(ph, om);
    const LnParts l = ln_parts(df_div(om, ph), tab);
    const float2 kl = kln2[l.k + 64];
    const DF d = df_add(df_add(DF{kl.x, kl.y}, l.lnF), l.s);
    const DF psi = df_mul(bc.quarter_lambda, d);
    const DF fi = df_of_int(c.i);
    const DF pn = df_add(c.pn_row, df_mul(bc.dxn0, fi));
    const DF rx = df_add(df_mul(bc.dx, fi), bc.neg_c0);
    const DF r = df_sqrt(df_add(df_mul(rx, rx), c.ryz2));
    acc.w = df_add_acc(acc.w, q);
    acc.c = df_add_acc(acc.c, df_mul(q, df_add(pn, df_neg(psi))));
    acc.r = df_add_acc(acc.r, df_mul(q, df_add(r, psi)));
}

// Partial sums of block b of nb (256 threads): rows ordered (j fastest, k) are
// dealt round-robin to the nb * 8 warps, so every block samples the whole
// grid and the band work (which sits in a few planes) is spread evenly.
template <class S>
__device__ __forceinline__ void stats_pass(const StatsArgs &a, const S *f, double *partial_out,
                                           long long blk, long long nblk)
{
    using R = typename Scr<S>::T;
    constexpr int E = Row16<S>::E;        // elements per 16-byte load
    constexpr int V = 16 / E;             // loads per lane and sweep
    constexpr int kWarps = 8;
    // Per warp: a ring of band cells (value, x index) with the slot of their
    // row's shares; a sweep is queued in four parts of at most 128 cells and
    // full warps of 32 are evaluated after each, so fewer than 32 wait between
    // parts and a part always fits.  Waiting cells come from fewer than 32 rows,
    // so 32 row slots, taken in turn, are never overwritten while referenced.
    constexpr int kRing = 256, kRowSlots = 32;
    __shared__ R ring_phi[kWarps][kRing];
    __shared__ int ring_i[kWarps][kRing];
    __shared__ unsigned char ring_slot[kWarps][kRing];
    __shared__ DF row_tab[kWarps][kRowSlots][2];
    const float4 *tab = g_ln_tab;
    const float2 *kln2 = g_kln2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    R mn = R(INFINITY), mx = R(-INFINITY);
    long long klo = order_key(INFINITY), khi = order_key(-INFINITY);   // FP64 extrema as order keys
    int nonfinite = 0;
    const BandConst &bconst = a.band;
    BandSums sums;
    int head = 0, tail = 0, band_rows = 0;   // ring positions and band rows so far (warp-uniform)
    // evaluate the waiting cell at ring position q (this lane's)
    auto eval_at = [&](int q) {
        const int r = q & (kRing - 1);
        BandCell<R> c;
        c.phi = ring_phi[warp][r];
        c.i = ring_i[warp][r];
        const int sl = ring_slot[warp][r];
        c.pn_row = row_tab[warp][sl][0];
        c.ryz2 = row_tab[warp][sl][1];
        band_cell<R>(bconst, c, tab, kln2, sums);
    };
    VolSum<R> vol;
    const long long rows = (long long)a.g.ny * a.g.nz;
    const int nvec = (a.g.nx + E - 1) / E, nwhole = a.g.nx / E;   // 16-byte pieces of a row, and whole ones
    // rows (j, k) dealt round-robin to the warps; ny nz < 2^30, and (j, k)
    // advance by the stride's split so that no row divides (64-bit division
    // is emulated in FP64, the slow pipe of this GPU)
    const long long row0 = blk * kWarps + warp, stride = nblk * kWarps;
    const int sj = (int)(stride % a.g.ny), sk = (int)(stride / a.g.ny);
    for (int j = (int)(row0 % a.g.ny), k = (int)(row0 / a.g.ny); k < a.g.nz;
         j += sj, k += sk, (j >= a.g.ny ? (j -= a.g.ny, ++k) : 0)) {
        bool row_known = false;   // the row's shares are in its slot
        int slot = 0;
        const uint4 *src = (const uint4 *)(f + cell_index(a.g, 0, j, k));
        for (int v0 = 0; v0 < nvec; v0 += 32 * V) {
            uint4 w[V];
            const auto before = vol.row();
#pragma unroll
            for (int t = 0; t < V; ++t) {
                const int vi = v0 + 32 * t + lane;
                w[t] = vi < nvec ? __ldg(src + vi) : make_uint4(0u, 0u, 0u, 0u);
            }
            // extrema and volume of the lane's whole pieces (a piece that a row's
            // end cuts goes cell by cell), and whether any cell may lie in the band
            unsigned parts = 0u;   // bit p: one of the lane's cells 4 p .. 4 p + 3 may lie in the band
            R lo = R(INFINITY), hi = R(-INFINITY);
            if constexpr (sizeof(R) == 4) {
#pragma unroll
                for (int t = 0; t < V; ++t) {
                    constexpr unsigned kPiece = (1u << (E / 4)) - 1u;   // its parts
                    const int vi = v0 + 32 * t + lane;
                    float far = 1.0f;   // the least |phi - 1/2|; band cells have less than 1/2 - 1e-6
                    if (vi < nwhole) {
#pragma unroll
                        for (int e = 0; e < E; e += 2) {
                            const float2 x = make_float2(Row16<S>::get(w[t], e), Row16<S>::get(w[t], e + 1));
                            vol.add(x);
                            lo = fminf(fminf(lo, x.x), x.y);
                            hi = fmaxf(fmaxf(hi, x.x), x.y);
                            const float2 d = __fadd2_rn(x, make_float2(-0.5f, -0.5f));
                            far = fminf(fminf(far, fabsf(d.x)), fabsf(d.y));
                        }
                    }
                    if (far < 0.5f - 0.5e-6f) parts |= kPiece << (t * E / 4);
                }
                // the piece that the row's end cuts, where the sweep holds it (a warp's
                // branch, so that other sweeps do not pass through this code)
                if (nwhole < nvec && nwhole >= v0 && nwhole < v0 + 32 * V) {
                    const int t = (nwhole - v0) / 32;
                    if (v0 + 32 * t + lane == nwhole) {
                        for (int i = nwhole * E; i < a.g.nx; ++i) {
                            const float x = scr<S>(reinterpret_cast<const S *>(src), i);
                            if (in_band(x)) parts |= 1u << ((t * E + i - nwhole * E) / 4);
                            vol.add(x);
                            lo = fminf(lo, x);
                            hi = fmaxf(hi, x);
                        }
                    }
                }
                if (!vol.finite()) {   // the sweep again, without the cells that are not
                    vol.set_row(before);
                    lo = R(INFINITY);
                    hi = R(-INFINITY);
#pragma unroll
                    for (int t = 0; t < V; ++t)
#pragma unroll
                        for (int e = 0; e < E; ++e)
                            if ((v0 + 32 * t + lane) * E + e < a.g.nx) {
                                const float x = Row16<S>::get(w[t], e);
                                if (!isfinite(x)) {
                                    ++nonfinite;
                                    continue;
                                }
                                vol.add(x);
                                lo = fminf(lo, x);
                                hi = fmaxf(hi, x);
                            }
                }
            } else {
                // FP64 cells: the one FP64 instruction each is the volume's add; the
                // rest compares integers (upper words for the tests)
#pragma unroll
                for (int t = 0; t < V; ++t)
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if ((v0 + 32 * t + lane) * E + e < a.g.nx) {
                            const R x = Row16<S>::get(w[t], e);
                            const unsigned h = (unsigned)__double2hiint(x);
                            if ((h & 0x7ff00000u) == 0x7ff00000u) {
                                ++nonfinite;
                                continue;
                            }
                            vol.add(x);
                            const long long k = order_key(x);
                            klo = k < klo ? k : klo;
                            khi = k > khi ? k : khi;
                            if (h - kBandLo <= kBandHi - kBandLo) parts |= 1u << ((t * E + e) / 4);
                        }
            }
            if constexpr (sizeof(R) == 4) {
                mn = fewest(mn, lo);
                mx = most(mx, hi);
            }
            parts = __reduce_or_sync(0xffffffffu, parts);   // of any lane
            if (parts != 0u) {
                // Queue the sweep's band cells in four parts of 4 cells a lane (a warp
                // prefix sum places each lane's), evaluating full warps after each.
                // The parts stay a loop, the sweep's words moving down by one part a
                // round: unrolled, four copies of the evaluation did not fit the
                // instruction cache (no_instruction the top stall).
                constexpr int kW = (int)sizeof(S);   // 32-bit words of 4 cells
                unsigned u[4 * V];
#pragma unroll
                for (int t = 0; t < V; ++t) {
                    u[4 * t] = w[t].x;
                    u[4 * t + 1] = w[t].y;
                    u[4 * t + 2] = w[t].z;
                    u[4 * t + 3] = w[t].w;
                }
#pragma unroll 1
                for (int part = 0; parts != 0u; ++part, parts >>= 1) {
                    unsigned m = 0u;   // the lane's band cells of the part
                    if (parts & 1u) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int b = 4 * part + k;   // cell of the lane's E * V
                            if (in_band(word_cell<S>(u, k)) && (v0 + 32 * (b / E) + lane) * E + b % E < a.g.nx)
                                m |= 1u << k;
                        }
                    }
                    if (__any_sync(0xffffffffu, m != 0u)) {
                        if (!row_known) {
                            // the row's shares of p.n and |p - ctr|^2, in double-float (FP64
                            // is the slow pipe of this GPU)
                            slot = band_rows++ & (kRowSlots - 1);
                            if (lane == 0) {
                                const DF fj = df_of_int(j), fk = df_of_int(k);
                                const DF ry = df_add(df_mul(bconst.dx, fj), bconst.neg_c1);
                                const DF rz = df_add(df_mul(bconst.dx, fk), bconst.neg_c2);
                                row_tab[warp][slot][0] = df_add(df_mul(bconst.dxn1, fj), df_mul(bconst.dxn2, fk));
                                row_tab[warp][slot][1] = df_add(df_mul(ry, ry), df_mul(rz, rz));
                            }
                            row_known = true;
                        }
                        const int c = __popc(m);
                        int incl = c;
#pragma unroll
                        for (int d = 1; d < 32; d <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, incl, d);
                            if (lane >= d) incl += y;
                        }
                        int pos = tail + incl - c;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (m & (1u << k)) {
                                const int r = pos & (kRing - 1);
                                const int b = 4 * part + k;
                                ring_phi[warp][r] = word_cell<S>(u, k);
                                ring_i[warp][r] = (v0 + 32 * (b / E) + lane) * E + b % E;
                                ring_slot[warp][r] = (unsigned char)slot;
                                ++pos;
                            }
                        }
                        tail += __shfl_sync(0xffffffffu, incl, 31);
                        __syncwarp();
                        for (; tail - head >= 32; head += 32) eval_at(head + lane);
                        __syncwarp();   // reads of evaluated cells before the next part's writes
                    }
#pragma unroll
                    for (int k = 0; k + kW < 4 * V; ++k) u[k] = u[k + kW];
                }
            }
            vol.end_sweep();
        }
    }
    if (lane < tail - head) eval_at(head + lane);
    double energy = 0.0;
    if (a.energy) {   // Eq. 1 at dF = 0, one cell per thread, contiguous rows per block
        const long long r0 = blk * rows / nblk, r1 = (blk + 1) * rows / nblk;
        const double e_pref = a.Gamma / (a.C_gamma * a.lambda);
        const int nd = a.stencil == 6 ? 3 : (a.stencil == 18 ? 9 : 13);
        for (long long row = r0; row < r1; ++row) {
            const int j = (int)(row % a.g.ny), k = (int)(row / a.g.ny);
            const long long rbase = cell_index(a.g, 0, j, k);
            for (int i = threadIdx.x; i < a.g.nx; i += blockDim.x) {
                const double ph = rd<S>(f, rbase + i);
                if (!isfinite(ph)) continue;
                double e = 0.0;
                for (int kk = 0; kk < nd; ++kk) {
                    const Dir d = grid_dir(kk);
                    const double r2 = (double)d.shell * a.dx * a.dx;
                    const double nb = rd<S>(f, cell_index(a.g, i + d.x, j + d.y, k + d.z));
                    const double dp = nb - ph;
                    e += a.w[kk] * (0.5 * a.lambda * a.lambda * dp * dp / r2 +
                                    potential(ph, a.a[kk], a.lambda * a.lambda / r2, is_fd_scheme(a.scheme)));
                }
                energy += e_pref * e;
            }
        }
    }
    const double total[kSums] = {vol.total(), df_to_double(sums.w), df_to_double(sums.c), df_to_double(sums.r),
                                 energy};
    if constexpr (sizeof(R) == 8) {
        mn = (R)key_value(klo);
        mx = (R)key_value(khi);
    }
    block_reduce_store<R>(total, mn, mx, (double)nonfinite, partial_out);
}

template <class S>
__global__ void __launch_bounds__(256, sizeof(S) == 8 ? 2 : 3)
    stats_kernel(const StatsArgs a, const S *f, double *partials)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    stats_pass<S>(a, f, partials + (long long)blockIdx.x * kNStat, blockIdx.x, gridDim.x);
}

// blockIdx.y selects the grid of the batch
template <class S>
__global__ void __launch_bounds__(256, 2) stats_batch_kernel(const StatsJob *jobs, double *partials)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const StatsJob &j = jobs[blockIdx.y];
    stats_pass<S>(j.a, (const S *)j.field[j.cur],
                  partials + ((long long)blockIdx.y * kBatchStatsBlocks + blockIdx.x) * kNStat,
                  blockIdx.x, gridDim.x);
}

// blockIdx.x selects a grid: reduce its nblocks partials into out[blockIdx.x]
__global__ void __launch_bounds__(256) stats_final_kernel(const double *partials, int nblocks, double *out)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");   // launched while the pass runs
    partials += (long long)blockIdx.x * nblocks * kNStat;
    out += (long long)blockIdx.x * kNStat;
    double sum[kSums] = {0.0, 0.0, 0.0, 0.0, 0.0}, mn = INFINITY, mx = -INFINITY, count = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        const double *p = partials + (long long)b * kNStat;
#pragma unroll
        for (int s = 0; s < kSums; ++s) sum[s] += p[sum_slot(s)];
        mn = fmin(mn, p[4]);
        mx = fmax(mx, p[5]);
        count += p[6];
    }
    block_reduce_store<double>(sum, mn, mx, count, out);
}

size_t stats_scratch_bytes()
{
    return sizeof(double) * (size_t)kNStat * (kStatsBlocks + 1);
}

size_t grid_scratch_bytes()
{
    return scratch_err_offset() + 16;
}

// The logarithm table of the band evaluation, written once per device by a
// kernel on the calling stream and waited for, so that calls on other streams
// can rely on it.  Inside a stream capture the writer is recorded into the
// graph instead (it cannot be waited for there) and the device stays unmarked.
static cudaError_t ensure_ln_table(cudaStream_t st)
{
    static std::mutex mu;
    static bool ready[128];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (ready[dev]) return cudaSuccess;
    ln_table_kernel<<<1, 256, 0, st>>>();
    e = cudaGetLastError();
    if (e != cudaSuccess || cs != cudaStreamCaptureStatusNone) return e;
    e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) ready[dev] = true;
    return e;
}

// One full wave of stats blocks on this device (at most kStatsBlocks): the
// band cells sit in a few planes and are spread over all warps, so a partial
// second wave would idle SMs.
template <class S> static int stats_blocks()
{
    static int cached[128];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return kStatsBlocks;
    if (!cached[dev]) {
        int per = 0, sms = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, stats_kernel<S>, 256, 0) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return kStatsBlocks;
        const int n = per * sms;
        cached[dev] = n < 1 ? 1 : (n > kStatsBlocks ? kStatsBlocks : n);
    }
    return cached[dev];
}

// the reduction of n grids' partials, which may launch while the pass before it runs
static cudaError_t launch_final(int n, const double *partials, int nblocks, double *out, cudaStream_t st)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(n);
    lc.blockDim = dim3(256);
    lc.stream = st;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, stats_final_kernel, partials, nblocks, out);
}

cudaError_t launch_stats(const StatsArgs &a, const void *field, double *partials, double *final_out,
                         cudaStream_t st)
{
    cudaError_t e = ensure_ln_table(st);
    if (e != cudaSuccess) return e;
    int nb;
    if (a.dtype == SPFM_F64) {
        nb = stats_blocks<double>();
        stats_kernel<double><<<nb, 256, 0, st>>>(a, (const double *)field, partials);
    } else if (a.dtype == SPFM_F32) {
        nb = stats_blocks<float>();
        stats_kernel<float><<<nb, 256, 0, st>>>(a, (const float *)field, partials);
    } else {
        nb = stats_blocks<__nv_bfloat16>();
        stats_kernel<__nv_bfloat16><<<nb, 256, 0, st>>>(a, (const __nv_bfloat16 *)field, partials);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_final(1, partials, nb, final_out, st);
}

cudaError_t launch_stats_batch(const StatsJob *jobs, int n, int dtype, double *partials, double *finals,
                               cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    cudaError_t e = ensure_ln_table(st);
    if (e != cudaSuccess) return e;
    const dim3 grid(kBatchStatsBlocks, n);
    if (dtype == SPFM_F64) stats_batch_kernel<double><<<grid, 256, 0, st>>>(jobs, partials);
    else if (dtype == SPFM_F32) stats_batch_kernel<float><<<grid, 256, 0, st>>>(jobs, partials);
    else stats_batch_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(jobs, partials);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_final(n, partials, kBatchStatsBlocks, finals, st);
}

}  // namespace spfm
