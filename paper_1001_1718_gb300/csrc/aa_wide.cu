// Antialiased resampling with more taps per axis than the register-window
// forms hold: the single-image kernels of the vertical-first streaming form
// (aa_vs.cuh, vertical downscales) and of the tiled form (aa_wide.cuh, any
// ratio), for every storage dtype and for the fused pre-process's
// normalised planar output, and their host configuration.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "capi_internal.h"
#include "aa_wide.cuh"
#include "aa_vs.cuh"

// Compiled twice so both kernel sets build in parallel: AA_WIDE_PART 0 (the
// resize kernels, plus the configurations), 1 (the fused pre-process;
// aa_wide_norm.cu).
#ifndef AA_WIDE_PART
#define AA_WIDE_PART 0
#endif

namespace rs {

// (four blocks per SM: shared memory rarely lets more in, and without the bound
// the compiler kept to 32 registers a thread: FP32 RGBA 894 x 2591 -> 7 x 22
// bilinear 1540 us, with it 1307)
template <int C, typename T, typename TO, bool NORM>
__global__ void __launch_bounds__(kAwNT, 4)
k_aa_wide(const Geom g, const T* __restrict__ src, TO* __restrict__ dst, const AaWideCfg cfg, const NormOut no,
          unsigned int* fault)
{
    extern __shared__ __align__(16) float sm[];
    const int plane = blockIdx.z;
    aa_wide_body<C, T, TO, NORM>(g, src + g.sp.offset(plane), dst + g.dp.offset(plane), cfg, blockIdx.x, blockIdx.y,
                                 sm, fault, no);
}

template <int C, typename T, typename TO, bool NORM, int NA, bool AL>
__global__ void __launch_bounds__(kVsMaxNT, 2)
k_aa_vs(const Geom g, const T* __restrict__ src, TO* __restrict__ dst, const AaVsCfg cfg, const NormOut no,
        unsigned int* fault)
{
    extern __shared__ __align__(16) float sm[];
    const int plane = blockIdx.z;
    aa_vs_body<C, T, TO, NORM, NA, AL>(g, src + g.sp.offset(plane), dst + g.dp.offset(plane), cfg, blockIdx.x, blockIdx.y,
                                   sm, fault, no);
}

#if AA_WIDE_PART == 0

// Largest count and widest span of the antialias taps over the tiles of
// `tile` consecutive outputs along one axis.
static void aa_axis_bounds(int n, int m, int method, int tile, int& kmax, int& span)
{
    kmax = 1;
    span = 1;
    for (int j0 = 0; j0 < m; j0 += tile) {
        const int j1 = std::min(m, j0 + tile) - 1;
        int lo0, hi0, lo1, hi1;
        aa_range(j0, n, m, method, lo0, hi0);
        aa_range(j1, n, m, method, lo1, hi1);
        span = std::max(span, hi1 - lo0);
        for (int j = j0; j <= j1; ++j) {
            int lo, hi;
            aa_range(j, n, m, method, lo, hi);
            kmax = std::max(kmax, hi - lo);
        }
    }
}

bool aa_wide_config(const Geom& g, int method, AaWideCfg& c)
{
    if (method != M_BILINEAR && method != M_BICUBIC) return false;
    if (g.C < 1 || g.C > 4) return false;
    c.method = method;
    int fw = 0;
    aa_axis_bounds(g.W, g.Wo, method, kAwTW, c.KX, fw);
    c.fw = fw;
    for (int TH = 32; TH >= 1; TH /= 2) {
        int KY = 0, nr = 0;
        aa_axis_bounds(g.H, g.Ho, method, TH, KY, nr);
        for (int RG = 8; RG >= 1; RG /= 2) {
            c.TH = TH;
            c.KY = KY;
            c.nr = nr;
            c.RG = RG;
            const size_t tabs = sizeof(float) * ((size_t)kAwTW * c.KX + (size_t)TH * KY) +
                                sizeof(int) * (2 * (size_t)kAwTW + 2 * (size_t)TH);
            c.s_off = (int)((tabs + 15) / 16 * 4);   // in floats, 16-byte aligned
            c.smem = sizeof(float) * ((size_t)c.s_off + (size_t)RG * fw * g.C + (size_t)nr * kAwTW * g.C);
            if (c.smem <= max_smem_per_block()) return true;
        }
    }
    return false;
}

// Upper bound of the source samples that the taps of k consecutive outputs
// span on axis n -> m: floor(x + d) - floor(x) <= ceil(d).
static int aa_span_bound(int k, int n, int m, int method)
{
    const int64_t d = (int64_t)(k - 1) * n + 2 * (int64_t)(method == M_BILINEAR ? 1 : 2) * std::max(n, m);
    return (int)std::min<int64_t>(n, (d + m - 1) / m);
}

// The problems the form is held to whatever its tiles: what tiles of 8 to 256
// columns of at most 1024 elements and 8 rows took in its first layout (24
// bytes of weights a source row, eight finished rows, 40 KB of copies). Beyond
// them it takes what fits without more threads or single weights.
static bool aa_vs_range(const Geom& g, int method, int dtype)
{
    const size_t es = dtype_size(dtype), most = max_smem_per_block();
    const int nr = aa_span_bound(std::min(8, g.Ho), g.H, g.Ho, method);
    const auto bytes = [&](size_t elems, size_t tw, size_t kx, size_t rows) {
        const size_t row = ((elems * es + 15) / 16 + 2) * 16;
        size_t chunk = 8;
        while (chunk > 2 && 3 * chunk * row > 40 * 1024) chunk /= 2;
        return 3 * chunk * row + 32 * ((elems + 3) / 4 * 4) + 4 * tw * kx + 8 * tw + 24 * rows;
    };
    // most problems: bounds of all that it depends on
    const size_t kx = aa_span_bound(1, g.W, g.Wo, method);
    if (aa_span_bound(std::min(8, g.Wo), g.W, g.Wo, method) * g.C <= 1024 &&
        40 * 1024 + 32 * 1024 + 4 * 256 * kx + 8 * 256 + 24 * (size_t)nr <= most)
        return true;
    for (int tw = 256; tw >= 8; tw /= 2) {
        int k = 0, span = 0, ky = 0, rows = 0;
        aa_axis_bounds(g.W, g.Wo, method, tw, k, span);
        if ((int64_t)span * g.C > 1024) continue;
        aa_axis_bounds(g.H, g.Ho, method, 8, ky, rows);
        return bytes((size_t)span * g.C, tw, k, rows) <= most;
    }
    return false;
}

// The vertical-first form: output rows no more than source rows, and 8 output
// columns' footprint at most 1024 elements. Tiles: the fewest of equal width
// whose footprints fit a block (a partly filled tile would cost as much as a
// full one), with as few warps as hold them. Bands: blocks for whole waves of
// the resident ones, the count with the least rows per SM, counting the rows
// a band re-reads above it and its start-up (tables, first copies: ~20 rows);
// with fewer than three blocks on an SM its latencies show.
bool aa_vs_config(const Geom& g, int method, int dtype, AaVsCfg& c)
{
    if (method != M_BILINEAR && method != M_BICUBIC) return false;
    if (g.C < 1 || g.C > 4 || g.Ho > g.H) return false;
    const int es = (int)dtype_size(dtype), E = vs_elems(es);
    c.aligned = g.src_pitch % E == 0;
    c.method = method;
    c.NA = method == M_BILINEAR ? 2 : 4;
    int s8 = aa_span_bound(std::min(8, g.Wo), g.W, g.Wo, method);
    if (s8 * g.C > 1024) {
        int kx = 0;
        aa_axis_bounds(g.W, g.Wo, method, 8, kx, s8);
        if (s8 * g.C > 1024) return false;
    }
    c.KX = aa_span_bound(1, g.W, g.Wo, method);
    int slack = c.aligned ? E - 1 : 0;   // owned elements before the footprint
    int cap = kVsNT * E - slack;
    const bool range = aa_vs_range(g, method, dtype);
    if (c.KX * g.C > cap) {   // one column's footprint is wider: more threads (FP32), no element before it
        if (!range) return false;
        c.aligned = 0;
        slack = 0;
        cap = std::min(kVsMaxNT * E, 1024);
    }
    int tw = 1;
    while (tw < std::min(g.Wo, 1024) && aa_span_bound(tw + 1, g.W, g.Wo, method) * g.C <= cap) ++tw;
    const int tiles = (g.Wo + tw - 1) / tw;
    c.TW = (g.Wo + tiles - 1) / tiles;
    const int span = aa_span_bound(c.TW, g.W, g.Wo, method);
    if (span * g.C > cap) return false;
    const int elems = span * g.C + slack;
    c.ve = (elems + E - 1) / E * E;
    c.nt = std::min(kVsMaxNT, (c.ve / E + 31) / 32 * 32);
    c.raw_row = std::max((elems * es + 15) / 16 + 2, (15 + elems * es + 4 * vs_words(es) + 15) / 16) * 16;
    const int S = c.raw_row + (int)((g.src_pitch * es) & 15);
    const double f = (double)g.H / g.Ho, reach = 2.0 * (method == M_BILINEAR ? 1 : 2) * f + 20.0;
    const int64_t cols = (int64_t)((g.Wo + c.TW - 1) / c.TW) * g.planes;
    const double sms = num_sms();
    bool any = false;
    double best = 0.0;
    AaVsCfg fit = c;
    c.chunk = es == 1 ? 8 : 4;
    // Row weights as pairs (8 NA bytes a row), or where not even one output
    // row's fit (bicubic from ~5500 source rows on) once, 4 NA bytes: uint8 RGB
    // 8000 x 1200 -> 2 x 120 1157 us (the form before: 1970). With more threads
    // FP32 RGB 1000 x 200 -> 3 x 2 bilinear 103 us (278).
    for (c.single = 0; c.single < 1 + range && !any; ++c.single) {
        for (int k : {3, 4, 8, 12, 16}) {   // blocks per SM (4 are resident)
            const int64_t bands = std::max<int64_t>(1, k * (int64_t)sms / cols);
            AaVsCfg t = c;
            t.TH = (int)std::max<int64_t>(1, (g.Ho + bands - 1) / bands);
            for (;; t.TH = (t.TH + 1) / 2) {
                t.nr = aa_span_bound(t.TH, g.H, g.Ho, method);
                t.smem = 3 * (size_t)vs_rows_bytes(t.chunk, S) + sizeof(float2) * (2 * (size_t)t.ve + (size_t)(t.single ? t.chunk : t.nr) * t.NA) +
                         (t.single ? sizeof(float) * (size_t)t.nr * t.NA : 0) +
                         sizeof(float) * (size_t)t.TW * t.KX + sizeof(int) * (2 * (size_t)t.TW + t.TH);
                if (t.smem <= max_smem_per_block() || t.TH == 1) break;
            }
            if (t.smem > max_smem_per_block()) continue;
            const double per_sm = std::ceil(cols * ((g.Ho + t.TH - 1) / t.TH) / sms);
            const double resident = std::max(1.0, std::floor(224.0 * 1024 / (t.smem + 1024)));
            const double cost = per_sm * (t.TH * f + reach) * std::max(1.0, 3.0 / std::min(resident, per_sm));
            if (!any || cost < best) {
                fit = t;
                best = cost;
                any = true;
            }
        }
    }
    if (any) c = fit;
    return any;
}

#endif

template <typename T, typename TO, bool NORM, int NA, bool AL>
static void* aa_vs_func(int C)
{
    return C == 1 ? (void*)&k_aa_vs<1, T, TO, NORM, NA, AL> : C == 2 ? (void*)&k_aa_vs<2, T, TO, NORM, NA, AL>
         : C == 3 ? (void*)&k_aa_vs<3, T, TO, NORM, NA, AL> : (void*)&k_aa_vs<4, T, TO, NORM, NA, AL>;
}

template <typename T, typename TO, bool NORM>
static void* aa_vs_func_na(const AaVsCfg& c, int C)
{
    if (c.aligned) return c.NA == 2 ? aa_vs_func<T, TO, NORM, 2, true>(C) : aa_vs_func<T, TO, NORM, 4, true>(C);
    return c.NA == 2 ? aa_vs_func<T, TO, NORM, 2, false>(C) : aa_vs_func<T, TO, NORM, 4, false>(C);
}

static cudaError_t launch_aa_vs_common(const Geom& g, void* func, const void* src, void* dst, const AaVsCfg& c,
                                       const NormOut& no, cudaStream_t st)
{
    cudaError_t e = prepare_kernel(func, c.smem, c.nt, nullptr);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((g.Wo + c.TW - 1) / c.TW), (unsigned)((g.Ho + c.TH - 1) / c.TH), (unsigned)g.planes);
    unsigned int* fw = fault_word();
    void* args[] = {const_cast<Geom*>(&g), const_cast<void**>(&src), &dst, const_cast<AaVsCfg*>(&c),
                    const_cast<NormOut*>(&no), &fw};
    e = cudaLaunchKernel(func, grid, dim3(c.nt), args, c.smem, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

#if AA_WIDE_PART == 0

cudaError_t launch_aa_vs(const Geom& g, int dtype, const void* src, void* dst, const AaVsCfg& c, cudaStream_t st)
{
    void* func = dtype == DT_U8 ? aa_vs_func_na<uint8_t, uint8_t, false>(c, g.C)
               : dtype == DT_F16 ? aa_vs_func_na<__half, __half, false>(c, g.C)
               : dtype == DT_BF16 ? aa_vs_func_na<__nv_bfloat16, __nv_bfloat16, false>(c, g.C)
               : aa_vs_func_na<float, float, false>(c, g.C);
    return launch_aa_vs_common(g, func, src, dst, c, NormOut{}, st);
}

#else

cudaError_t launch_aa_vs_norm(const Geom& g, int out_dtype, const void* src, void* dst, const AaVsCfg& c,
                              const NormOut& no, cudaStream_t st)
{
    void* func = out_dtype == DT_F16 ? aa_vs_func_na<uint8_t, __half, true>(c, g.C)
               : out_dtype == DT_BF16 ? aa_vs_func_na<uint8_t, __nv_bfloat16, true>(c, g.C)
               : aa_vs_func_na<uint8_t, float, true>(c, g.C);
    return launch_aa_vs_common(g, func, src, dst, c, no, st);
}

#endif

template <typename T, typename TO, bool NORM>
static void* aa_wide_func(int C)
{
    return C == 1 ? (void*)&k_aa_wide<1, T, TO, NORM> : C == 2 ? (void*)&k_aa_wide<2, T, TO, NORM>
         : C == 3 ? (void*)&k_aa_wide<3, T, TO, NORM> : (void*)&k_aa_wide<4, T, TO, NORM>;
}

static cudaError_t launch_aa_wide_common(const Geom& g, void* func, const void* src, void* dst, const AaWideCfg& c,
                                         const NormOut& no, cudaStream_t st)
{
    cudaError_t e = prepare_kernel(func, c.smem, kAwNT, nullptr);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((g.Wo + kAwTW - 1) / kAwTW), (unsigned)((g.Ho + c.TH - 1) / c.TH), (unsigned)g.planes);
    unsigned int* fw = fault_word();
    void* args[] = {const_cast<Geom*>(&g), const_cast<void**>(&src), &dst, const_cast<AaWideCfg*>(&c),
                    const_cast<NormOut*>(&no), &fw};
    e = cudaLaunchKernel(func, grid, dim3(kAwNT), args, c.smem, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

#if AA_WIDE_PART == 0

cudaError_t launch_aa_wide(const Geom& g, int dtype, const void* src, void* dst, const AaWideCfg& c, cudaStream_t st)
{
    void* func = dtype == DT_U8 ? aa_wide_func<uint8_t, uint8_t, false>(g.C)
               : dtype == DT_F16 ? aa_wide_func<__half, __half, false>(g.C)
               : dtype == DT_BF16 ? aa_wide_func<__nv_bfloat16, __nv_bfloat16, false>(g.C)
               : aa_wide_func<float, float, false>(g.C);
    return launch_aa_wide_common(g, func, src, dst, c, NormOut{}, st);
}

#else

cudaError_t launch_aa_wide_norm(const Geom& g, int out_dtype, const void* src, void* dst, const AaWideCfg& c,
                                const NormOut& no, cudaStream_t st)
{
    void* func = out_dtype == DT_F16 ? aa_wide_func<uint8_t, __half, true>(g.C)
               : out_dtype == DT_BF16 ? aa_wide_func<uint8_t, __nv_bfloat16, true>(g.C)
               : aa_wide_func<uint8_t, float, true>(g.C);
    return launch_aa_wide_common(g, func, src, dst, c, no, st);
}

#endif

}  // namespace rs
