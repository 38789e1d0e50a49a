// Fixed-point forms of the double-precision passes (see fx_math.cuh): the
// same tiles, lines and exchanges as the passes of pass_kernels.cuh, with the
// transform on 64-bit integers.  A tile or line group that holds a line outside
// the conversions' range (non-finite values, exponents near the ends of the
// double range) runs the FP64 pass instead, from the same twiddle tables.
//
// Measured on GB300 in place (FP64 arithmetic -> fixed point): 1024^3 pair
// 190.3 -> 31.7 ms, 512^3 21.6 -> 3.58 ms; relative L2 error of one transform
// against extended precision, over line lengths, noise and single-spike lines:
// 1.6-2.8e-16 -> 0.5-1.8e-16.  The FP64 pass in place of it keeps the speed of
// kernels of FP64 arithmetic alone: 512^3 pair with one infinity 22.0 ms (21.6).
#pragma once

#include "pass_kernels.cuh"

namespace fft3d {

// Lengths transformed in fixed point; shorter ones have too few FP64
// operations per element to gain.
template <typename R, int L> __host__ __device__ constexpr bool col_fixed() { return sizeof(R) == 8 && L >= 8; }
template <typename R, int M> __host__ __device__ constexpr bool z_fixed() { return sizeof(R) == 8 && M >= 4; }

__device__ __forceinline__ fxtw fx_ldg(const fxtw *p)
{
    const int4 q = __ldg((const int4 *)p);
    return fxtw{q.x, q.y, q.z, q.w};
}

// A complex result: by integer operations, or where a component is below 2^32
// (2^-29 of the line's scale) or zero, by FP64 additions.
__device__ __forceinline__ double2 fx_out(fxc z, int e)
{
    int32_t big = -1;
    double2 r = cmake<double2>(fx_to_big(z.x, e, big), fx_to_big(z.y, e, big));
    if (big >= 0) r = cmake<double2>(fx_to(z.x, e), fx_to(z.y, e));
    return r;
}
// A thread's results v[i] 2^e, handed to f(i, value).  Small components are
// noticed on the way and all results handed over again by FP64 additions.
template <int E, class F> __device__ __forceinline__ void fx_out_all(const fxc *v, int e, const F &f)
{
    int32_t big = -1;
#pragma unroll
    for (int i = 0; i < E; ++i) f(i, cmake<double2>(fx_to_big(v[i].x, e, big), fx_to_big(v[i].y, e, big)));
    if (big >= 0) {
        fxc w[E];
#pragma unroll
        for (int i = 0; i < E; ++i) w[i] = v[i];
#pragma unroll 1
        for (int i = 0; i < E; ++i) f(i, cmake<double2>(fx_to(w[i].x, e), fx_to(w[i].y, e)));
    }
}

// z f, or z itself in the UNIT kernels, whose scales are 1 or (C2R) a power of
// two: a product costs an FP64 issue slot even where it is predicated off.
template <bool UNIT> __device__ __forceinline__ double2 fx_scale(double2 z, double f)
{
    if constexpr (UNIT) return z;
    else return cscale(z, f);
}

// A block lets the next pass be launched when only its stores are left.  From
// the start of the block instead, the next pass's blocks take the slots of the
// first SMs that run dry and crowd there (128^3 float pair 31.8 -> 40.1 us).
// The link-bound (max_blocks) kernels release nothing: a waiting block would
// keep another stream's passes off the SM for long.  64^3 double pair, each
// waited for: 78 -> 72 us.  The float passes release nothing either, as it
// costs every block: 16-thread tiles of short columns 23 -> 39 us at
// 4 x 1024 x 1024, where leaving it out costs the other grids nothing.
__device__ __forceinline__ void pass_release() { asm volatile("griddepcontrol.launch_dependents;\n"); }

// ------------------------------------------------------------ columns
// Load of a column entry, asking L2 for the whole 128-byte line: the tile beside
// it, run at the same time by another SM, wants the rest of it (512^3: y-pass
// 0.646 -> 0.636 ms).
__device__ __forceinline__ double2 fx_load(const double2 *p)
{
    double2 r;
    asm volatile("ld.global.L2::128B.v2.f64 {%0, %1}, [%2];\n" : "=d"(r.x), "=d"(r.y) : "l"(p) : "memory");
    return r;
}

template <int L, int E, int W, bool INV>
__device__ __noinline__ void col_tile_slow(const ColArgs &a, int64_t tile, unsigned char *smem, const fxtw *tw)
{
    col_tile<double, L, E, W, false, INV>(a, tile, smem, tw);
}

// Threads that are to share an SM: 64 registers each with 8 elements per
// thread, 168 with 24 in blocks of 128, else 128.
__host__ __device__ constexpr int fx_resident(int E, int block) { return E <= 8 ? 1024 : E == 24 && block <= 128 ? 384 : 512; }
__host__ __device__ constexpr int fx_min_blocks(int E, int block)
{
    const int n = fx_resident(E, block) / block;
    return n < 1 ? 1 : n > 32 ? 32 : n;
}

template <int L, int E, int W, bool INV>
__global__ void __launch_bounds__(W *(L / E), fx_min_blocks(E, W *(L / E)))
colpass_fx_kernel(const __grid_constant__ ColArgs a, const fxtw *__restrict__ tw)
{
    constexpr int NT = L / E;
    static_assert(W <= 32 && W * NT % 32 == 0, "a warp holds all columns of the tile");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pass_begin();
    int *code = (int *)(smem_raw + (size_t)L * W * sizeof(fxc));
    const int c = threadIdx.x % W;
    const int j = threadIdx.x / W;
    double2 *sp = nullptr, *dp = nullptr;
    int64_t ss = 0, ds = 0;
    const bool valid = col_decode<double2, W>(a, blockIdx.x, c, sp, ss, dp, ds);
    if (threadIdx.x < W) code[threadIdx.x] = 0;
    fxc v[E];
    int g;
    {
        double2 r[E];
        const double2 *sj = sp + (int64_t)j * ss;
        const int64_t sstep = (int64_t)NT * ss;
#pragma unroll
        for (int i = 0; i < E; ++i) r[i] = fx_load(sj + i * sstep);
        if constexpr (NT > 1) {
            g = fx_thread_code<E>(r);
            __syncthreads();
            if constexpr (W < 32) {
#pragma unroll
                for (int o = W; o < 32; o *= 2) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
                if ((threadIdx.x & 31) < W) atomicMax(code + c, g);
            } else {
                atomicMax(code + c, g);
            }
        } else {
            g = fx_thread_code<E>(r);
            code[c] = g;
        }
        __syncthreads();
        g = code[c];
        if (!__all_sync(0xffffffffu, fx_in_range(g))) {  // every warp holds every column of the tile
            if (__syncthreads_or(!fx_in_range(g) && fx_unfit<E>(g, r))) {
                col_tile_slow<L, E, W, INV>(a, blockIdx.x, smem_raw, tw);
                return;
            }
            g = g == 0 ? kFxZeroCode : g;
        }
#pragma unroll
        for (int i = 0; i < E; ++i)
            v[i] = fx_make(fx_from(INV ? r[i].y : r[i].x, g, kFxBits), fx_from(INV ? r[i].x : r[i].y, g, kFxBits));
    }
    ColEx<fxc, W> ex{(fxc *)smem_raw, c};
    line_fft<fx64, L, E>(v, j, tw, ex);
    pass_release();
    const int e = g - 1023 - kFxBits + fx_line_shift<L, E>();
    if (valid) {
        double2 *dj = dp + (int64_t)j * ds;
        // below 2^29 (128 rows of a 2048 x 2048 x 2048 grid): 32 bits spare the 8-element kernels a spilled register
        const uint32_t dstep = NT * (uint32_t)ds;
        fx_out_all<E>(v, e, [&](int i, double2 o) { dj[(uint32_t)i * (uint64_t)dstep] = INV ? cswap(o) : o; });
    }
}

// ------------------------------------------------------------ lines
// Largest scale code of a line (NT threads).
template <int NT, int LPB, class Ex> __device__ __forceinline__ int fx_line_max(int g, const Ex &ex)
{
#pragma unroll
    for (int o = (NT < 32 ? NT : 32) / 2; o > 0; o /= 2) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
    if constexpr (NT > 32) {
        constexpr int WPL = NT / 32;
        __shared__ int code[LPB * WPL];
        const int w = threadIdx.x / 32;
        if (threadIdx.x % 32 == 0) code[w] = g;
        ex.sync();
#pragma unroll
        for (int i = 0; i < WPL; ++i) g = max(g, code[w / WPL * WPL + i]);
    }
    return g;
}
// Whether the line of code g, of which the thread holds v, is transformed in fixed
// point; the threads that synchronise together agree.
template <int NT, int LPB, int N, class Ex> __device__ __forceinline__ bool fx_line_ok(int g, const double2 *v, const Ex &ex)
{
    if constexpr (NT > 32) {
        if (fx_in_range(g)) return true;
        ex.sync();  // every thread has read the code
        return fx_line_max<NT, LPB>(fx_unfit<N>(g, v), ex) == 0;
    } else {
        if (__all_sync(0xffffffffu, fx_in_range(g))) return true;
        return !__any_sync(0xffffffffu, !fx_in_range(g) && fx_unfit<N>(g, v));
    }
}

template <int M, int E, int LPB>
__device__ __noinline__ void zr2c_slow(const ZArgs &a, int64_t line0, unsigned char *smem, const fxtw *tw,
                                       const fxtw *rot)
{
    if constexpr (z_paired<double, M>()) zr2c_pairs<double, M, E, LPB>(a, line0, smem, tw);
    else zr2c_lines<double, M, E, LPB>(a, line0, smem, tw, rot);
}
template <int M, int E, int LPB>
__device__ __noinline__ void zc2r_slow(const ZArgs &a, int64_t line0, unsigned char *smem, const fxtw *tw,
                                       const fxtw *rot)
{
    if constexpr (z_paired<double, M>()) zc2r_pairs<double, M, E, LPB, false>(a, line0, smem, tw);
    else zc2r_lines<double, M, E, LPB, false>(a, line0, smem, tw, rot);
}

// zr2c_lines in fixed point: X[k] = (s - i r d) / 2 with s = Z[k] + conj Z[M - k],
// d = Z[k] - conj Z[M - k], formed as X / 2 = s / 4 - i (r / 4) d.
template <int M, int E, int LPB, bool UNIT>
__device__ __forceinline__ void zr2c_fx_lines(const ZArgs &a, int64_t line0, unsigned char *smem,
                                              const fxtw *__restrict__ tw, const fxtw *__restrict__ rot)
{
    constexpr int NT = M / E;
    constexpr int P = zline_pad<E>();
    const int lt = threadIdx.x / NT;
    const int j = threadIdx.x % NT;
    const int64_t line = line0 + lt;
    const bool active = line < a.nlines;
    LineEx<fxc, NT, P> ex{(fxc *)smem + lt * zline_smem_elems<M, E>(), line_bar<NT, LPB>(lt)};

    fxc v[E];
    int g;
    {
        const double2 *in = (const double2 *)((const double *)a.real + (active ? line : 0) * a.real_pitch);
        double2 r[E];
#pragma unroll
        for (int i = 0; i < E; ++i) r[i] = active ? in[j + i * NT] : cmake<double2>(0.0, 0.0);
        g = fx_line_max<NT, LPB>(fx_thread_code<E>(r), ex);
        if (!fx_line_ok<NT, LPB, E>(g, r, ex)) {
            zr2c_slow<M, E, LPB>(a, line0, smem, tw, rot);
            return;
        }
        g = g == 0 ? kFxZeroCode : g;
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = fx_make(fx_from(r[i].x, g, kFxBits), fx_from(r[i].y, g, kFxBits));
    }
    line_fft<fx64, M, E>(v, j, tw, ex);
    if (a.max_blocks == 0) pass_release();

    const int e = g - 1023 - kFxBits + fx_line_shift<M, E>();
    double2 *out = (double2 *)a.cplx.main + (active ? line : 0) * (M + 1);
    const double se = a.scale_edge, sm = a.scale_mid;
    auto emit = [&](int k, fxc z, fxc zm) {
        const fxc zc = cconj(zm);
        const fxc s = fx_shr<2>(cadd(z, zc));
        const fxc p = cmul(csub(z, zc), fx_ldg(rot + k));
        const double2 x = fx_out(fx_make(s.x + p.y, s.y - p.x), e + 1);
        if (active) store_out(out + k, fx_scale<UNIT>(x, k == 0 ? se : sm));
    };
    if constexpr (NT <= 32) {
        const int src = (NT - j) & (NT - 1);
        static_for<0, E>([&](auto II) {
            constexpr int i = decltype(II)::value;
            fxc zp;
            zp.x = __shfl_sync(0xffffffffu, (long long)v[E - 1 - i].x, src, NT);
            zp.y = __shfl_sync(0xffffffffu, (long long)v[E - 1 - i].y, src, NT);
            emit(j + i * NT, v[i], (j == 0) ? v[(E - i) % E] : zp);
        });
    } else {
        constexpr bool LR = pad_linear_reads<P>(NT);
        constexpr bool LREV = P < 0 || NT % (1 << P) == 0;
#pragma unroll
        for (int i = 0; i < E; ++i) ex.put(pad_row<P, LR>(j, i * NT), v[i]);
        ex.sync();
        static_for<0, E>([&](auto II) {
            constexpr int i = decltype(II)::value;
            emit(j + i * NT, v[i], (i == 0 && j == 0) ? v[0] : ex.get(pad_row<P, LREV>(M - j, -i * NT)));
        });
    }
    if (active && j == 0) {
        out[M] = fx_scale<UNIT>(cmake<double2>(fx_to(v[0].x - v[0].y, e), 0.0), se);
    }
}

// Output scale s of a C2R line as an exponent where it is a power of two (the
// factor left over is then 1; UNIT kernels run only then, see fx_unit_scale).
inline bool fx_unit_scale(double s)
{
    const uint64_t u = fx_bits(s);
    return (u & 0xfffffffffffffULL) == 0 && u >> 52 > 1023 - 100 && u >> 52 < 1023 + 100;
}
template <bool UNIT> __device__ __forceinline__ double fx_split_scale(double s, int &e)
{
    if constexpr (UNIT) {
        e += (int)(fx_bits(s) >> 52) - 1023;
        return 1.0;
    } else {
        return s;
    }
}

// zc2r_lines in fixed point.  The pre-process at most quadruples a thread's L1
// norm (its own entries and their mirror images, twice each), so the entries
// come in at 2^-2 of the usual scale; its rotation by r / 4 acts on 4 d.
template <int M, int E, int LPB, bool UNIT>
__device__ __forceinline__ void zc2r_fx_lines(const ZArgs &a, int64_t line0, unsigned char *smem,
                                              const fxtw *__restrict__ tw, const fxtw *__restrict__ rot)
{
    constexpr int NT = M / E;
    constexpr int P = zline_pad<E>();
    const int lt = threadIdx.x / NT;
    const int j = threadIdx.x % NT;
    const int64_t line = line0 + lt;
    const bool active = line < a.nlines;
    LineEx<fxc, NT, P> ex{(fxc *)smem + lt * zline_smem_elems<M, E>(), line_bar<NT, LPB>(lt)};

    const int64_t l = active ? line : 0;
    fxc v[E], xm;
    int g;
    {
        const double2 *src = (const double2 *)a.cplx.main + l * (a.cplx.split ? M : M + 1);
        const double2 *nyq = a.cplx.split ? (const double2 *)a.cplx.nyq + l : src + M;
        double2 r[E + 1];
#pragma unroll
        for (int i = 0; i < E; ++i) r[i] = active ? src[j + i * NT] : cmake<double2>(0.0, 0.0);
        r[E] = active && j == 0 ? *nyq : cmake<double2>(0.0, 0.0);
        if (j == 0) {
            // only the real parts of the k2 = 0 and k2 = M entries enter
            r[0] = cmake<double2>(a.scale_edge * r[0].x, 0.0);
            r[E] = cmake<double2>(a.scale_edge * r[E].x, 0.0);
        }
        g = fx_line_max<NT, LPB>(fx_thread_code<E + 1>(r), ex);
        if (!fx_line_ok<NT, LPB, E + 1>(g, r, ex)) {
            zc2r_slow<M, E, LPB>(a, line0, smem, tw, rot);
            return;
        }
        g = g == 0 ? kFxZeroCode : g;
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = fx_make(fx_from(r[i].x, g, kFxBits - 2), fx_from(r[i].y, g, kFxBits - 2));
        xm = fx_make(fx_from(r[E].x, g, kFxBits - 2), 0);
    }
    // conj(Z[k]) from x = X[k] and y = X[M - k]
    auto pre = [&](int k, fxc x, fxc y) -> fxc {
        const fxc yc = cconj(y);
        const fxc s = cadd(x, yc), d = csub(x, yc);
        const fxc o = cmulc(fx_make(d.x * 4, d.y * 4), fx_ldg(rot + k));
        return fx_make(s.x - o.y, -(s.y + o.x));
    };
    if constexpr (NT <= 32) {
        const int srcl = (NT - j) & (NT - 1);
        fxc up = xm;  // lane 0: the value that slot E - i held before its update
        static_for<0, (E + 1) / 2>([&](auto II) {
            constexpr int i = decltype(II)::value;
            constexpr int h = E - 1 - i;
            // slots i and h of lanes j and NT - j are each other's mirror images
            // (lane 0: slots i and E - i of its own)
            fxc pi, ph;
            pi.x = __shfl_sync(0xffffffffu, (long long)v[h].x, srcl, NT);
            pi.y = __shfl_sync(0xffffffffu, (long long)v[h].y, srcl, NT);
            ph.x = __shfl_sync(0xffffffffu, (long long)v[i].x, srcl, NT);
            ph.y = __shfl_sync(0xffffffffu, (long long)v[i].y, srcl, NT);
            if (j == 0) {
                pi = up;
                ph = v[i + 1 < E ? i + 1 : i];
                if constexpr (i == h) ph = pi;
            }
            up = v[h];
            const fxc nh = pre(j + h * NT, v[h], ph);
            if constexpr (i != h) {
                v[i] = pre(j + i * NT, v[i], pi);
                v[h] = nh;
            } else {
                v[h] = pre(j + h * NT, v[h], pi);
            }
        });
    } else {
        constexpr bool LR = pad_linear_reads<P>(NT);
        constexpr bool LREV = P < 0 || NT % (1 << P) == 0;
#pragma unroll
        for (int i = 0; i < E; ++i) ex.put(pad_row<P, LR>(j, i * NT), v[i]);
        if (j == 0) ex.put(pad_row<P, true>(M, 0), xm);
        ex.sync();
        static_for<0, E>([&](auto II) {
            constexpr int i = decltype(II)::value;
            v[i] = pre(j + i * NT, v[i], ex.get(pad_row<P, LREV>(M - j, -i * NT)));
        });
        ex.sync();
    }
    line_fft<fx64, M, E>(v, j, tw, ex);
    if (a.max_blocks == 0) pass_release();

    int e = g - 1023 - (kFxBits - 2) + fx_line_shift<M, E>();
    const double f = fx_split_scale<UNIT>(a.scale_mid, e);
    double2 *out = (double2 *)((double *)a.real_out + l * a.real_pitch);
    if (active)
        fx_out_all<E>(v, e, [&](int i, double2 o) { store_out(out + j + i * NT, fx_scale<UNIT>(cconj(o), f)); });
}

// zr2c_pairs in fixed point; the two lines share a scale, as they share the
// FP64 form's rounding errors.
template <int M, int E, int LPB, bool UNIT>
__device__ __forceinline__ void zr2c_fx_pairs(const ZArgs &a, int64_t line0, unsigned char *smem,
                                              const fxtw *__restrict__ tw)
{
    constexpr int N = 2 * M;
    constexpr int NT = N / E;
    constexpr int PPB = LPB / 2;
    constexpr int P = zline_pad<E>();
    static_assert(LPB % 2 == 0 && NT > 32, "pairs of lines");
    const int pt = threadIdx.x / NT;
    const int j = threadIdx.x % NT;
    const int64_t l0 = line0 + 2 * pt;
    const bool act0 = l0 < a.nlines, act1 = l0 + 1 < a.nlines;
    LineEx<fxc, NT, P> ex{(fxc *)smem + pt * zline_smem_elems<N, E>(), line_bar<NT, PPB>(pt)};

    fxc v[E];
    int g;
    {
        const double *in0 = (const double *)a.real + (act0 ? l0 : 0) * a.real_pitch;
        const double *in1 = (const double *)a.real + (act1 ? l0 + 1 : 0) * a.real_pitch;
        double2 r[E];
#pragma unroll
        for (int i = 0; i < E; ++i) r[i] = cmake<double2>(act0 ? in0[j + i * NT] : 0.0, act1 ? in1[j + i * NT] : 0.0);
        g = fx_line_max<NT, PPB>(fx_thread_code<E>(r), ex);
        if (!fx_line_ok<NT, PPB, E>(g, r, ex)) {
            zr2c_slow<M, E, LPB>(a, line0, smem, tw, nullptr);
            return;
        }
        g = g == 0 ? kFxZeroCode : g;
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = fx_make(fx_from(r[i].x, g, kFxBits), fx_from(r[i].y, g, kFxBits));
    }
    line_fft<fx64, N, E>(v, j, tw, ex);
    if (a.max_blocks == 0) pass_release();

    constexpr bool LR = pad_linear_reads<P>(NT);
    constexpr bool LREV = P < 0 || NT % (1 << P) == 0;
#pragma unroll
    for (int i = M / NT; i < E; ++i) ex.put(pad_row<P, LR>(j, i * NT), v[i]);  // only Z[N - k], k <= M, is read
    ex.sync();
    double2 *out0 = (double2 *)a.cplx.main + (act0 ? l0 : 0) * (M + 1);
    double2 *out1 = out0 + (M + 1);
    const int e = g - 1023 - kFxBits + fx_line_shift<N, E>() - 1;
    const double se = a.scale_edge, sm = a.scale_mid;
    static_for<0, M / NT + 1>([&](auto II) {
        constexpr int i = decltype(II)::value;
        if (i < M / NT || j == 0) {
            const int k = j + i * NT;
            const fxc z = v[i];
            const fxc zm = (k == 0 || k == M) ? z : ex.get(pad_row<P, LREV>(N - j, -i * NT));  // Z[N - k]
            const double2 x0 = fx_out(fx_make(z.x + zm.x, z.y - zm.y), e),
                          x1 = fx_out(fx_make(z.y + zm.y, zm.x - z.x), e);
            const double f = (k == 0 || k == M) ? se : sm;
            if (act0) store_out(out0 + k, fx_scale<UNIT>(x0, f));
            if (act1) store_out(out1 + k, fx_scale<UNIT>(x1, f));
        }
    });
}

// zc2r_pairs in fixed point.  Thread j converts the entries k = j + i NT < M of
// both lines once; they give Z[k] = x0 + i x1, its own, and Z[N - k] =
// conj x0 + i conj x1, which another thread of the pair owns.
template <int M, int E, int LPB, bool UNIT>
__device__ __forceinline__ void zc2r_fx_pairs(const ZArgs &a, int64_t line0, unsigned char *smem,
                                              const fxtw *__restrict__ tw)
{
    constexpr int N = 2 * M;
    constexpr int NT = N / E;
    constexpr int H = E / 2;
    constexpr int PPB = LPB / 2;
    constexpr int P = zline_pad<E>();
    static_assert(LPB % 2 == 0 && NT > 32 && H * NT == M, "pairs of lines");
    const int pt = threadIdx.x / NT;
    const int j = threadIdx.x % NT;
    const int64_t l0 = line0 + 2 * pt;
    const bool act0 = l0 < a.nlines, act1 = l0 + 1 < a.nlines;
    LineEx<fxc, NT, P> ex{(fxc *)smem + pt * zline_smem_elems<N, E>(), line_bar<NT, PPB>(pt)};
    constexpr bool LR = pad_linear_reads<P>(NT);
    constexpr bool LREV = P < 0 || NT % (1 << P) == 0;

    const int64_t la = act0 ? l0 : 0, lb = act1 ? l0 + 1 : 0;
    fxc v[E];
    int g;
    {
        const int64_t pitch = a.cplx.split ? M : M + 1;
        const double2 *src0 = (const double2 *)a.cplx.main + la * pitch;
        const double2 *src1 = (const double2 *)a.cplx.main + lb * pitch;
        const double2 zero = cmake<double2>(0.0, 0.0);
        double2 r[E + 1];  // line l: slots 0..H-1, line l + 1: slots H..E-1, the k2 = M pair last
#pragma unroll
        for (int i = 0; i < H; ++i) {
            r[i] = act0 ? src0[j + i * NT] : zero;
            r[H + i] = act1 ? src1[j + i * NT] : zero;
        }
        r[E] = zero;
        if (j == 0) {
            const double2 *nyq0 = a.cplx.split ? (const double2 *)a.cplx.nyq + la : src0 + M;
            const double2 *nyq1 = a.cplx.split ? (const double2 *)a.cplx.nyq + lb : src1 + M;
            const double we = a.scale_edge;
            r[0] = cmake<double2>(we * r[0].x, 0.0);
            r[H] = cmake<double2>(we * r[H].x, 0.0);
            r[E] = cmake<double2>(act0 ? we * nyq0->x : 0.0, act1 ? we * nyq1->x : 0.0);
        }
        // a thread's transform inputs have at most twice this L1 norm (its own entries and their mirror images)
        g = fx_line_max<NT, PPB>(fx_thread_code<E + 1>(r), ex);
        if (!fx_line_ok<NT, PPB, E + 1>(g, r, ex)) {
            zc2r_slow<M, E, LPB>(a, line0, smem, tw, nullptr);
            return;
        }
        g = g == 0 ? kFxZeroCode : g;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const fxc x0 = fx_make(fx_from(r[i].x, g, kFxBits - 1), fx_from(r[i].y, g, kFxBits - 1));
            const fxc x1 = fx_make(fx_from(r[H + i].x, g, kFxBits - 1), fx_from(r[H + i].y, g, kFxBits - 1));
            // inverse transform as swap(DFT(swap(Z)))
            v[i] = fx_make(x0.y + x1.x, x0.x - x1.y);
            const fxc m = fx_make(x1.x - x0.y, x0.x + x1.y);
            if (i > 0 || j > 0) ex.put(pad_row<P, LREV>(N - j, -i * NT), m);
        }
        if (j == 0) {
            const fxc x = fx_make(fx_from(r[E].x, g, kFxBits - 1), fx_from(r[E].y, g, kFxBits - 1));
            ex.put(pad_row<P, true>(M, 0), fx_make(x.y, x.x));
        }
        ex.sync();
#pragma unroll
        for (int i = H; i < E; ++i) v[i] = ex.get(pad_row<P, LR>(j, i * NT));
        ex.sync();
    }
    line_fft<fx64, N, E>(v, j, tw, ex);
    if (a.max_blocks == 0) pass_release();

    int e = g - 1023 - (kFxBits - 1) + fx_line_shift<N, E>();
    const double f = fx_split_scale<UNIT>(a.scale_mid, e);
    double *out0 = (double *)a.real_out + la * a.real_pitch;
    double *out1 = (double *)a.real_out + lb * a.real_pitch;
    fx_out_all<E>(v, e, [&](int i, double2 o) {  // x1 + i x0 at n = j + i NT
        const double2 z = fx_scale<UNIT>(o, f);
        if (act0) store_out(out0 + j + i * NT, z.y);
        if (act1) store_out(out1 + j + i * NT, z.x);
    });
}

// A group of LPB lines, by the form that serves the length.
template <int M, int E, int LPB, bool UNIT>
__device__ __forceinline__ void zr2c_fx_group(const ZArgs &a, int64_t line0, unsigned char *smem,
                                              const fxtw *__restrict__ tw, const fxtw *__restrict__ rot)
{
    if constexpr (z_paired<double, M>()) zr2c_fx_pairs<M, E, LPB, UNIT>(a, line0, smem, tw);
    else zr2c_fx_lines<M, E, LPB, UNIT>(a, line0, smem, tw, rot);
}
template <int M, int E, int LPB, bool UNIT>
__device__ __forceinline__ void zc2r_fx_group(const ZArgs &a, int64_t line0, unsigned char *smem,
                                              const fxtw *__restrict__ tw, const fxtw *__restrict__ rot)
{
    if constexpr (z_paired<double, M>()) zc2r_fx_pairs<M, E, LPB, UNIT>(a, line0, smem, tw);
    else zc2r_fx_lines<M, E, LPB, UNIT>(a, line0, smem, tw, rot);
}

// The z-passes in fixed point, blocks and LOOP as in zpass_r2c_kernel.  `a` is
// __grid_constant__ because the slow path takes its address (without, every
// thread copies it to local memory); the other z kernels are not: it costs
// them registers (float R2C lines of 512 points 64 -> 80, 768-point looping
// C2R ones 128 -> 159).
template <int M, int E, int LPB, bool LOOP, bool UNIT>
__global__ void __launch_bounds__(LPB *(M / E), fx_min_blocks(E, LPB *(M / E)))
zpass_r2c_fx_kernel(const __grid_constant__ ZArgs a, const fxtw *__restrict__ tw, const fxtw *__restrict__ rot)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pass_begin();
    if constexpr (LOOP) {
        for (int64_t blk = blockIdx.x; blk * LPB < a.nlines; blk += gridDim.x) {
            if (blk != blockIdx.x) __syncthreads();  // shared memory free for the next line group
            zr2c_fx_group<M, E, LPB, false>(a, blk * LPB, smem_raw, tw, rot);
        }
    } else {
        zr2c_fx_group<M, E, LPB, UNIT>(a, (int64_t)blockIdx.x * LPB, smem_raw, tw, rot);
    }
}

template <int M, int E, int LPB, bool LOOP, bool UNIT>
__global__ void __launch_bounds__(LPB *(M / E), fx_min_blocks(E, LPB *(M / E)))
zpass_c2r_fx_kernel(const __grid_constant__ ZArgs a, const fxtw *__restrict__ tw, const fxtw *__restrict__ rot)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pass_begin();
    if constexpr (LOOP) {
        for (int64_t blk = blockIdx.x; blk * LPB < a.nlines; blk += gridDim.x) {
            if (blk != blockIdx.x) __syncthreads();  // shared memory free for the next line group
            zc2r_fx_group<M, E, LPB, false>(a, blk * LPB, smem_raw, tw, rot);
        }
    } else {
        zc2r_fx_group<M, E, LPB, UNIT>(a, (int64_t)blockIdx.x * LPB, smem_raw, tw, rot);
    }
}

// ------------------------------------------------------------ twiddles
// Stage table of a line plan: entry (m - 1) * ns + k = exp(-2 pi i m k / (ns r)),
// computed in FP64 with sincospi after exact integer reduction of m k, then
// rounded once to the storage type.
template <typename R>
__global__ void twiddle_stage_kernel(typename cvec<R>::T *out, int ns, int r)
{
    typedef typename cvec<R>::T C;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (r - 1) * ns) return;
    const int m = i / ns + 1;
    const int k = i - (m - 1) * ns;
    const int64_t d = (int64_t)ns * r;
    const int64_t p = ((int64_t)m * k) % d;
    double s, c;
    sincospi(2.0 * (double)p / (double)d, &s, &c);
    out[i] = cmake<C>(R(c), R(-s));
}

// Fixed-point forms of the two tables, for double lines: entries of scale
// fx_stage_shift(r), rot[k] of scale kFxRotShift.
template <typename TW> __global__ void twiddle_stage_fx_kernel(TW *out, int ns, int r)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (r - 1) * ns) return;
    const int m = i / ns + 1;
    const int k = i - (m - 1) * ns;
    const uint32_t d = (uint32_t)ns * (uint32_t)r;
    out[i] = fx_twiddle((uint32_t)(m * k) % d, d, fx_stage_shift(r));
}
template <typename TW> __global__ void twiddle_rot_fx_kernel(TW *out, int n, int count)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < count) out[k] = fx_twiddle((uint32_t)k, (uint32_t)n, kFxRotShift);
}

// rot[k] = exp(-2 pi i k / n), k < count (FP64 sincospi, rounded once)
template <typename R>
__global__ void twiddle_rot_kernel(typename cvec<R>::T *out, int n, int count)
{
    typedef typename cvec<R>::T C;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    double s, c;
    sincospi(2.0 * (double)k / (double)n, &s, &c);
    out[k] = cmake<C>(R(c), R(-s));
}

}  // namespace fft3d
