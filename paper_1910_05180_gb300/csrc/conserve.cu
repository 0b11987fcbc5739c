// conserve.cu -- the constant-volume correction of a step (Sec. 3.3).
//
// The shape relaxation of Sec. 3.3 keeps the particle volume fixed with a
// homogeneous, time-dependent driving force.  The driving term of one step is
// -dt (4 M dF / (lambda Gamma)) q(phi) per cell (q = phi (1 - phi), the h3
// term), so after the ordinary step at dF = 0 has written phi* = phi + dt R0,
// the dF that leaves sum_p phi_p unchanged subtracts alpha q(phi_p) from every
// cell with
//     alpha = sum_p (phi*_p - phi_p) / sum_p q(phi_p),
//     dF    = alpha lambda Gamma / (4 M dt).
// Pass 1 reduces the two sums (rows dealt round-robin to the warps, fixed order,
// so the result is reproducible); in pass 2 every block adds the partials in
// the same order, forms alpha, corrects its rows of phi* and writes the ghost
// cells whose source they hold, so that no face kernel follows.
//
// Both are bound by the FP64 pipe (a warp's FP64 instruction holds it 16 cycles
// for the whole SM) and by latency at the grids of this study (60^3: 0.9 MB a
// field).  So a warp takes a row in 16-byte loads; cells of FP32 and BF16 fields
// are summed by fours, whose terms and sums are exact but for 2^-70 (Sum3), and only
// those sums enter FP64; they are corrected in double-float pairs (48 bits against
// the 24 of a cell).  The block reduction adds 8 values a lane from shared memory
// before it shuffles.  The kernels of a step chain by programmatic dependent
// launch.  60^3 FP32, us a step: sums 10.9 -> 6.0 (6.8 with Sum3 in place of pairs),
// correction and ghosts 67.1 + 3.4 -> 6.9 (one thread added the 608 partials one by
// one); alpha formed once, by the last block of the sums, was slower (9.1 + 5.1).
// alpha of 28 fields of 40 to 97 cells a side against quadruple precision, in units
// of 2^-53: 3.8 on average and 9.3 at most with one FP64 sum a lane, 1.0 and 3.0 so.
#include "spfm_internal.h"

namespace spfm {

namespace {

// storage <-> compute (FP64, or FP32 for FP32 and BF16 storage)
template <class S> struct Cell {
    using T = float;
};
template <> struct Cell<double> {
    using T = double;
};
__device__ __forceinline__ double get(double v) { return v; }
__device__ __forceinline__ float get(float v) { return v; }
__device__ __forceinline__ float get(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void put(double &s, double v) { s = v; }
__device__ __forceinline__ void put(float &s, float v) { s = v; }
__device__ __forceinline__ void put(__nv_bfloat16 &s, float v) { s = __float2bfloat16_rn(v); }

// d - x and q(x) = x (1 - x) of the first n of a group of cells, added to the FP64 sums
__device__ __forceinline__ void add_cells(const double *x, const double *d, int n, double &dsum, double &qsum)
{
#pragma unroll
    for (int e = 0; e < 2; ++e)
        if (e < n) {
            dsum += d[e] - x[e];
            qsum += fma(-x[e], x[e], x[e]);
        }
}
__device__ __forceinline__ DF q_of(float x) { return df_mul_f(df_two_sum(1.0f, -x), x); }
// A sum of a few FP32 numbers as s + l + m: s the sum, l that of its remainders, m
// that of theirs, so that it is good to about 2^-70.  As pairs alone (2^-48 a cell) the
// sum of q came out 3e-16 too large, always to that side.
struct Sum3 {
    float s = 0.0f, l = 0.0f, m = 0.0f;
    __device__ __forceinline__ void low(float x)
    {
        const DF t = df_two_sum(l, x);
        l = t.hi;
        m = __fadd_rn(m, t.lo);
    }
    __device__ __forceinline__ void add(DF x)
    {
        const DF t = df_two_sum(s, x.hi);
        s = t.hi;
        low(t.lo);
        low(x.lo);
    }
    __device__ __forceinline__ double value() const { return (double)s + ((double)l + (double)m); }
};
__device__ __forceinline__ void add_cells(const float *x, const float *d, int n, double &dsum, double &qsum)
{
    Sum3 ds, qs;
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (e < n) {
            ds.add(df_two_sum(d[e], -x[e]));   // d - x exactly
            const DF xx = df_two_prod(x[e], x[e]);
            qs.add(df_two_sum(x[e], -xx.hi));   // x - x^2 exactly
            qs.low(-xx.lo);
        }
    dsum += ds.value();
    qsum += qs.value();
}

// d - alpha q(x), rounded once
__device__ __forceinline__ double corrected(double d, double x, double alpha, DF)
{
    return d - alpha * (x * (1.0 - x));
}
// alpha beyond the FP32 range (only minute cells take a correction then): as a
// call, since inlined its FP64 instructions took a relaxation step 21.2 -> 25.7 us
__device__ __noinline__ float corrected_wide(float d, float x, double alpha)
{
    return (float)((double)d - alpha * ((double)x * (1.0 - (double)x)));
}
__device__ __forceinline__ float corrected(float d, float x, double alpha, DF alpha2)
{
    if (!isfinite(alpha2.lo)) return corrected_wide(d, x, alpha);
    const DF t = df_mul(alpha2, q_of(x));
    const DF s = df_two_sum(d, -t.hi);
    return __fadd_rn(s.hi, __fsub_rn(s.lo, t.lo));
}

constexpr int kWarps = 8;   // per block

// sums of a and b over the block's threads, in a of threads 0 and 32
__device__ __forceinline__ void block_sum2(double &a, double b)
{
    __shared__ double s[2][32 * kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    s[0][threadIdx.x] = a;
    s[1][threadIdx.x] = b;
    __syncthreads();
    if (warp < 2) {
        a = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) a += s[warp][32 * w + lane];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
    }
}

// 16 bytes of a row as storage elements
template <class S> struct Vec {
    static constexpr int E = 16 / (int)sizeof(S);
    union {
        uint4 w;
        S v[E];
    };
    __device__ __forceinline__ Vec() {}
};

template <class S>
__global__ void __launch_bounds__(32 * kWarps) conserve_sums_kernel(const GridGeom g, const S *src, const S *dst,
                                                                    double *partials)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    using T = typename Cell<S>::T;
    constexpr int E = Vec<S>::E;
    const int lane = threadIdx.x & 31;
    double dsum = 0.0, qsum = 0.0;
    const int rows = g.ny * g.nz;   // a face of the grid is below 2^30 cells
    for (int row = blockIdx.x * kWarps + (threadIdx.x >> 5); row < rows; row += gridDim.x * kWarps) {
        const long long base = cell_index(g, 0, row % g.ny, row / g.ny);
        for (int i = lane * E; i < g.nx; i += 32 * E) {   // rows start on 32 bytes, the pitch covers the last 16
            Vec<S> p, d;
            p.w = *reinterpret_cast<const uint4 *>(src + base + i);
            d.w = *reinterpret_cast<const uint4 *>(dst + base + i);
            constexpr int G = E < 4 ? E : 4;   // cells of a group
#pragma unroll
            for (int e0 = 0; e0 < E; e0 += G) {
                T x[G], y[G];
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    x[e] = get(p.v[e0 + e]);
                    y[e] = get(d.v[e0 + e]);
                }
                if (i + e0 < g.nx) add_cells(x, y, g.nx - i - e0, dsum, qsum);
            }
        }
    }
    block_sum2(dsum, qsum);
    if (threadIdx.x == 0) partials[2 * blockIdx.x] = dsum;
    if (threadIdx.x == 32) partials[2 * blockIdx.x + 1] = dsum;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Boundary kinds of the faces as bits (an axis is periodic on both faces or on
// none) and the signed contact couplings.
template <class T>
struct Faces {
    unsigned periodic, contact;   // bit axis, bit face
    T a[6];
};

// The ghost coordinates whose source is c on an axis of n cells, the inverse of
// map_axis: image 0 is c itself, 1 and 2 the ghosts (kNone: c has none there).
constexpr int kNone = -2;
__device__ __forceinline__ int axis_image(int m, int c, int n, bool periodic)
{
    if (m == 0) return c;
    if (m == 1) return (periodic ? c == n - 1 : c == 0) ? -1 : kNone;
    return (periodic ? c == 0 : c == n - 1) ? n : kNone;
}

// E cells (i.., j, k) of a row with their stored values v, and the ghosts they
// are the source of, as the face kernel (boundary.cu) writes them: shifts along
// x, then y, then z in the compute type (CONTACT: some face has the shift of
// Eq. 7; without it the images are copies: 4 us less at 60^3).  The y and z images
// are the warp's, whole rows at a time; most rows have none.
template <class S, bool CONTACT, int E>
__device__ __forceinline__ void write_cells(const GridGeom &g, const Faces<typename Cell<S>::T> &fc, S *f,
                                            const Vec<S> &v, int i, int j, int k)
{
    using T = typename Cell<S>::T;
    auto image = [&](T x, int m, int axis) {
        const int face = 2 * axis + m - 1;
        return CONTACT && m > 0 && (fc.contact >> face & 1u) ? contact_shift_rn(x, fc.a[face]) : x;
    };
    const bool px = fc.periodic & 1u, py = fc.periodic & 2u, pz = fc.periodic & 4u;
    const bool edge = j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1;
#pragma unroll 1
    for (int mz = 0; mz < (edge ? 3 : 1); ++mz) {
        const int kk = axis_image(mz, k, g.nz, pz);
        if (kk == kNone) continue;
#pragma unroll 1
        for (int my = 0; my < (edge ? 3 : 1); ++my) {
            const int jj = axis_image(my, j, g.ny, py);
            if (jj == kNone) continue;
            auto yz = [&](T x) { return image(image(x, my, 1), mz, 2); };
            S *row = f + cell_index(g, 0, jj, kk);
            Vec<S> o;
            if (CONTACT) {
#pragma unroll
                for (int e = 0; e < E; ++e) put(o.v[e], yz(get(v.v[e])));
            } else {
                o.w = v.w;
            }
            if (i + E <= g.nx) {
                *reinterpret_cast<uint4 *>(row + i) = o.w;
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (i + e < g.nx) row[i + e] = o.v[e];
            }
            if (i == 0 || i + E >= g.nx) {   // x ghosts of the row's first and last cell
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int c = i + e;
                    if (c == 0) {
                        const int m = px ? 2 : 1;
                        put(row[px ? g.nx : -1], yz(image(get(v.v[e]), m, 0)));
                    }
                    if (c == g.nx - 1) {
                        const int m = px ? 1 : 2;
                        put(row[px ? -1 : g.nx], yz(image(get(v.v[e]), m, 0)));
                    }
                }
            }
        }
    }
}

template <class S, bool CONTACT>
__global__ void __launch_bounds__(32 * kWarps)
    conserve_apply_kernel(const GridGeom g, const __grid_constant__ Faces<typename Cell<S>::T> fc, const S *src,
                          S *dst, const double *partials, double *alpha_out)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    constexpr int E = Vec<S>::E;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = g.ny * g.nz;
    __shared__ double s_sum[2];
    __shared__ DF s_alpha;
    if (warp < 2) {   // warp 0 the differences, warp 1 the q; all loads under way at once
        constexpr int kLoads = (kStatsBlocks + 31) / 32;
        double x[kLoads], v = 0.0;
#pragma unroll
        for (int t = 0; t < kLoads; ++t)
            x[t] = lane + 32 * t < gridDim.x ? partials[2 * (lane + 32 * t) + warp] : 0.0;
#pragma unroll
        for (int t = 0; t < kLoads; ++t)
            if (32 * t < gridDim.x) v += x[t];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) s_sum[warp] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double al = s_sum[1] != 0.0 ? s_sum[0] / s_sum[1] : 0.0;
        s_alpha = df_of(al);
        s_sum[0] = al;
        if (blockIdx.x == 0) *alpha_out = al;
    }
    __syncthreads();
    const double alpha = s_sum[0];
    const DF alpha2 = s_alpha;
    for (int row = blockIdx.x * kWarps + warp; row < rows; row += gridDim.x * kWarps) {
        const int j = row % g.ny, k = row / g.ny;
        for (int i = lane * E; i < g.nx; i += 32 * E) {
            const long long at = cell_index(g, i, j, k);
            Vec<S> p, d;
            p.w = *reinterpret_cast<const uint4 *>(src + at);
            d.w = *reinterpret_cast<const uint4 *>(dst + at);
#pragma unroll
            for (int e = 0; e < E; ++e) put(d.v[e], corrected(get(d.v[e]), get(p.v[e]), alpha, alpha2));
            write_cells<S, CONTACT, E>(g, fc, dst, d, i, j, k);
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class S>
cudaError_t conserve(const GridGeom &g, const double aface[6], const S *src, S *dst, double *partials,
                     double *alpha_out, cudaStream_t st)
{
    const int rows = g.ny * g.nz, want = (rows + kWarps - 1) / kWarps;
    const int nblk = want < kStatsBlocks ? want : kStatsBlocks;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(nblk);
    lc.blockDim = dim3(32 * kWarps);
    lc.stream = st;
    lc.attrs = attr;
    lc.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&lc, conserve_sums_kernel<S>, g, src, (const S *)dst, partials);
    if (e != cudaSuccess) return e;
    using T = typename Cell<S>::T;
    Faces<T> fc = {0u, 0u, {}};
    for (int f = 0; f < 6; ++f) {
        if (g.bc[f] == SPFM_PERIODIC) fc.periodic |= 1u << (f / 2);
        if (g.bc[f] == SPFM_CONTACT) fc.contact |= 1u << f;
        fc.a[f] = (T)aface[f];
    }
    if (fc.contact)
        return cudaLaunchKernelEx(&lc, conserve_apply_kernel<S, true>, g, fc, src, dst,
                                  (const double *)partials, alpha_out);
    return cudaLaunchKernelEx(&lc, conserve_apply_kernel<S, false>, g, fc, src, dst,
                                  (const double *)partials, alpha_out);
}

}  // namespace

cudaError_t launch_conserve(const GridGeom &g, int dtype, const double aface[6], const void *src, void *dst,
                            double *partials, double *alpha_out, cudaStream_t st)
{
    if (dtype == SPFM_F64) return conserve(g, aface, (const double *)src, (double *)dst, partials, alpha_out, st);
    if (dtype == SPFM_F32) return conserve(g, aface, (const float *)src, (float *)dst, partials, alpha_out, st);
    return conserve(g, aface, (const __nv_bfloat16 *)src, (__nv_bfloat16 *)dst, partials, alpha_out, st);
}

}  // namespace spfm
