// The uint8 forms of the register-window kernel that read the source in place
// (win_raw.cuh): resize (k_win_raw) and the fused pre-process
// (k_win_raw_norm), one block per (strip of output pixels, band of output
// rows, plane).
#include <algorithm>
#include <climits>

#include "capi_internal.h"
#include "win_raw.cuh"

// Compiled in parts so the kernel sets build in parallel: WIN_RAW_PART 0
// (resize, bilinear, plus the configuration), 1 (resize, bicubic;
// win_raw_p1.cu), 2 and 3 (the fused pre-process, bilinear and bicubic;
// win_raw_p2.cu, win_raw_p3.cu).
#ifndef WIN_RAW_PART
#define WIN_RAW_PART 0
#endif

namespace rs {

// 128 threads: four blocks of at most 128 registers a thread per SM (RGB
// bicubic x1.7, 4096^2 -> 6964^2: 77.8 us; three blocks of up to 168
// registers: 79.9); the exact-x2 form five (4096^2 -> 8192^2: 55.4 us; four:
// 58.2, three: 60.6; the form on FP32 windows it replaces: 77.9).
// Four channels of whole bicubic runs need a few registers more.
template <int KT, int C, int PAT, int ST>
constexpr int raw_blocks() { return (PAT == kRawX2 ? 5 : PAT == 4 && KT == 4 && C > 2 ? 3 : 4) - (KT == 4 && C == 4 && ST == RAW_WORDS && PAT < 4); }

template <int KT, int C, int PAT, int ST>
__global__ void __launch_bounds__(kWinThreads, raw_blocks<KT, C, PAT, ST>())
k_win_raw(const Geom g, const uint8_t* __restrict__ src, uint8_t* __restrict__ dst, const WinCfg cfg,
          unsigned int* fault)
{
    extern __shared__ __align__(16) float sm[];
    const int plane = blockIdx.z;
    win_body_raw<KT, C, PAT, ST, uint8_t>(g, src + g.sp.offset(plane), dst + g.dp.offset(plane), cfg, blockIdx.x,
                                          blockIdx.y, sm, fault);
}

template <int KT, int C, int PAT, int ST, typename TO>
__global__ void __launch_bounds__(kWinThreads, raw_blocks<KT, C, PAT, ST>())
k_win_raw_norm(const Geom g, const uint8_t* __restrict__ src, TO* __restrict__ dst, const WinCfg cfg, const NormOut no,
               unsigned int* fault)
{
    extern __shared__ __align__(16) float sm[];
    const int img = blockIdx.z;
    win_body_raw<KT, C, PAT, ST, TO>(g, src + g.sp.offset(img), dst + g.dp.offset(img), cfg, blockIdx.x, blockIdx.y,
                                     sm, fault, no);
}

static constexpr int kRawKT = WIN_RAW_PART % 2 ? 4 : 2;

template <int C, int PAT>
static void* raw_func_s(int st)
{
    return st == RAW_WORDS ? (void*)&k_win_raw<kRawKT, C, PAT, RAW_WORDS> : (void*)&k_win_raw<kRawKT, C, PAT, RAW_ANY>;
}

// The fused pre-process: whole aligned runs, and for downscales (whose gain
// is the footprint) any alignment too: a thread's elements leave one by one
// there, 8 to 16 bytes apart in a warp, which costs upscales more than the
// form gains (9 x 1068 x 1171 -> 1473 x 1615 BF16 bicubic: 98 us, the general
// form's stores of neighbouring pixels 94).
template <int C, int PAT, typename TO>
static void* norm_func_t(int st)
{
    if constexpr (C == 3 && PAT == kRawX2 && sizeof(TO) == 4) return nullptr;   // win_raw_norm_ok
    else if (st == RAW_WORDS) return (void*)&k_win_raw_norm<kRawKT, C, PAT, RAW_WORDS, TO>;
    if constexpr (PAT == 2 || PAT == 4) return (void*)&k_win_raw_norm<kRawKT, C, PAT, RAW_ANY, TO>;
    return nullptr;
}

template <int C, int PAT>
static void* norm_func_s(int st, int out_dtype)
{
    return out_dtype == DT_F32 ? norm_func_t<C, PAT, float>(st) : out_dtype == DT_F16 ? norm_func_t<C, PAT, __half>(st)
                               : norm_func_t<C, PAT, __nv_bfloat16>(st);
}

template <int C>
static void* raw_func_p(int pat, int st, int out_dtype)
{
#if WIN_RAW_PART < 2
    (void)out_dtype;
    return pat == 0 ? raw_func_s<C, 0>(st) : pat == 1 ? raw_func_s<C, 1>(st) : pat == 2 ? raw_func_s<C, 2>(st)
         : pat == 4 ? raw_func_s<C, 4>(st) : raw_func_s<C, kRawX2>(st);
#else
    return pat == 0 ? norm_func_s<C, 0>(st, out_dtype) : pat == 1 ? norm_func_s<C, 1>(st, out_dtype)
         : pat == 2 ? norm_func_s<C, 2>(st, out_dtype) : pat == 4 ? norm_func_s<C, 4>(st, out_dtype)
                                                                  : norm_func_s<C, kRawX2>(st, out_dtype);
#endif
}

static void* raw_func(int C, int pat, int st, int out_dtype)
{
    switch (C) {
    case 1: return raw_func_p<1>(pat, st, out_dtype);
#if WIN_RAW_PART < 2
    case 2: return raw_func_p<2>(pat, st, out_dtype);
    case 4: return raw_func_p<4>(pat, st, out_dtype);
#endif
    case 3: return raw_func_p<3>(pat, st, out_dtype);
    default: return nullptr;   // excluded by the caller
    }
}

#if WIN_RAW_PART == 0

void* raw_kernel_bilinear(int C, int pat, int st) { return raw_func(C, pat, st, DT_U8); }
void* raw_kernel_bicubic(int C, int pat, int st);
void* raw_norm_bilinear(int C, int pat, int st, int out_dtype);
void* raw_norm_bicubic(int C, int pat, int st, int out_dtype);

// Threads per block for rows of Wo pixels: blocks of 1 to 4 warps of
// warp_px stored pixels, the count with the least to do counting the warps
// idle at the row's end (a warp of a narrower block, which shares the row
// tables, the copies' halo and the barriers among fewer, costs ~14% more per
// warp missing: RGB bicubic x1.7, 6963 wide, 88 us at 4 warps, 95 at 3).
int win_raw_threads(int Wo, int warp_px)
{
    const int warps = (Wo + warp_px - 1) / warp_px;
    int best = 4;
    double cost = 1e30;
    for (int nw = 4; nw >= 1; --nw) {
        const double c = (warps + nw - 1) / nw * nw * (1.0 + 0.14 * (4 - nw));
        if (c < cost) {
            cost = c;
            best = nw;
        }
    }
    return 32 * best;
}

// Strips of half the width beyond two source pixels per output pixel: their
// staged rows are as long as a full strip's at half the ratio.
int win_raw_block(const Geom& g, int warp_px)
{
    const int nt = win_raw_threads(g.Wo, warp_px);
    return (int64_t)g.W > 2 * (int64_t)g.Wo ? std::min(nt, 64) : nt;
}

// Two blocks per resident slot; one for outputs of at most 32 MB, whose bands
// would be hardly longer than the rows and copies a block starts with (exact
// x2, RGB 653 x 1148 bilinear, 9 MB: 5.7 us in one, 7.6 in two, and 6.6 on the
// form on FP32 windows that this one replaced; grey 32 x 485 x 171 -> 1570 x
// 553 bilinear, 28 MB: 26.0, 29.2 and 27.4). The two cross near 45 MB (exact
// x2, 16 planes of 356 x 2900, 66 MB: 28.6 in one, 25.5 in two). Two also
// where whole bands of many strips and planes fill one round of slots worse
// (512 planes of 407 x 22 doubled, 18 MB: 40.1, in one 48.5).
int win_raw_waves(const Geom& g, const WinCfg& c, int64_t out_bytes)
{
    if (out_bytes > (int64_t)32 << 20) return 2;
    const int64_t strip = raw_strip(c.nt, false), units = ((int64_t)g.Wo + strip - 1) / strip * g.planes;
    const int64_t by_regs = (c.pat == kRawX2 + 1 ? 5 : 4) * kWinThreads / c.nt, by_smem = 228 * 1024 / ((int64_t)c.smem + 1024);
    const int64_t slots = num_sms() * std::max<int64_t>(1, std::min(by_regs, by_smem));
    const auto filled = [&](int64_t n) { return (double)std::max<int64_t>(1, n / units) * units / n; };
    return filled(slots) < 0.95 * std::min(1.0, filled(2 * slots)) ? 2 : 1;
}

bool win_raw_config(const Geom& g, int method, int dtype, int nt, int band_cap, WinCfg& c, bool allow_x2)
{
    c.pat = 0;
    if (dtype != DT_U8 || (method != M_BILINEAR && method != M_BICUBIC) || g.C < 1 || g.C > 4) return false;
    const int KT = method_taps(method);
    if (c.chunk < KT || c.chunk % KT || c.chunk > 32 || nt < 32 || nt > kWinThreads || nt % 32) return false;
    int64_t an, am;
    coord_advance(g.W, g.Wo, g.coord, an, am);
    const int pat = allow_x2 && win_is_x2(g) ? kRawX2 : raw_pattern(an, am);
    if (pat < 0) return false;
    const int span = tap_span_bound(kRawP * nt, g.W, g.Wo, KT, g.coord) * g.C;
    const int fw = (pat == 0 ? RawPat<0>::hi(kRawP - 1) : pat == 1 ? RawPat<1>::hi(kRawP - 1)
                    : pat == 2 ? RawPat<2>::hi(kRawP - 1) : pat == 4 ? RawPat<4>::hi(kRawP - 1)
                    : RawPat<kRawX2>::hi(kRawP - 1)) + KT;
    const int nr = (fw * g.C + 3) / 4 + 1;   // words a thread reads of a row
    c.nt = nt;
    c.raw_row = std::max((span + 15) / 16 + 2, (15 + span + 4 * nr + 15) / 16) * 16;
    c.swe = 0;
    c.band_cap = std::min(std::min(kWinMaxBand, band_cap), g.Ho);
    c.pos_cap = tap_span_bound(c.band_cap, g.H, g.Ho, KT, g.coord);
    const int npos = (c.pos_cap + KT - 1) / KT * KT;
    const size_t tabs = sizeof(float2) * (size_t)c.band_cap * KT + sizeof(int) * ((size_t)c.band_cap + npos);
    c.tab_off = (int)((tabs + 15) & ~(size_t)15);   // the rows' waiting ends, then the staged rows
    const int ew = g.C == 1 ? raw_end_words<1>() : g.C == 4 ? raw_end_words<4>() : raw_end_words<3>();
    c.raw_off = c.tab_off + (int)(2 * sizeof(uint32_t) * ew * c.band_cap + 15) / 16 * 16;
    const int S = c.raw_row + (int)(g.src_pitch & 15);
    c.smem = (size_t)c.raw_off + raw_rows_bytes(KT - 1, S) + 3 * (size_t)raw_rows_bytes(c.chunk, S);
    if (c.smem > max_smem_per_block()) return false;
    c.pat = pat + 1;
    return true;
}

bool win_raw_default(const Geom& g, int method, int dtype, int nt, int band_cap, WinCfg& c, bool allow_x2)
{
    const int asked = c.chunk;
    c.pat = 0;
    for (int chunk : {asked ? asked : 8, asked ? 0 : 4}) {
        WinCfg t = c;
        t.chunk = chunk;
        if (!chunk || !win_raw_config(g, method, dtype, nt, band_cap, t, allow_x2)) continue;
        c = t;
        if (t.smem * (kWinThreads / nt) <= 56 * 1024) break;
    }
    return c.pat > 0;
}

// RAW_WORDS where every run is whole and aligned: widths of whole runs, and
// every row and plane on a boundary of `unit` bytes.
static int raw_store_mode(const Geom& g, const void* dst, size_t es, int unit, int64_t c_stride)
{
    const bool ok = g.Wo % kRawP == 0 && reinterpret_cast<uintptr_t>(dst) % unit == 0 && g.dst_pitch * es % unit == 0 &&
                    (g.planes == 1 || g.dp.n_stride * es % unit == 0) && (g.dp.cp == 1 || g.dp.c_stride * es % unit == 0) &&
                    c_stride * es % unit == 0;
    return ok ? RAW_WORDS : RAW_ANY;
}

static cudaError_t launch_raw(const Geom& g, void* func, int strip, const void* src, void* dst, WinCfg c,
                              const NormOut* no, cudaStream_t st)
{
    if (!func || c.pat < 1 || c.nt < 32 || c.nt > kWinThreads || c.nt % 32) return cudaErrorInvalidValue;
    int per_sm = 1;
    cudaError_t e = prepare_kernel(func, c.smem, c.nt, c.band_h <= 0 ? &per_sm : nullptr);
    if (e != cudaSuccess) return e;
    const int64_t strips = ((int64_t)g.Wo + strip - 1) / strip;
    if (c.band_h <= 0) {
        const int64_t resident = (int64_t)num_sms() * std::max(1, per_sm);
        const int64_t elems = (int64_t)g.Ho * g.Wo * g.C * g.planes;
        const int waves = c.waves > 0 ? c.waves : win_raw_waves(g, c, elems * (int64_t)(no ? dtype_size(no->dtype) : 1));
        // at most `waves` blocks per resident slot: a partial extra wave would run alone
        const int64_t bands = std::max<int64_t>(1, resident * waves / (strips * g.planes));
        c.band_h = (int)std::min<int64_t>(c.band_cap, std::max<int64_t>(1, (g.Ho + bands - 1) / bands));
    }
    if (c.pat == kRawX2 + 1 && c.band_h % 2) ++c.band_h;   // bands start on even rows (band_cap is even: Ho is)
    if (c.band_h > c.band_cap) return cudaErrorInvalidValue;
    dim3 grid((unsigned)strips, (unsigned)((g.Ho + c.band_h - 1) / c.band_h), (unsigned)g.planes);
    unsigned int* fw = fault_word();
    if (no) {
        void* args[] = {const_cast<Geom*>(&g), const_cast<void**>(&src), &dst, &c, const_cast<NormOut*>(no), &fw};
        e = cudaLaunchKernel(func, grid, dim3(c.nt), args, c.smem, st);
    } else {
        void* args[] = {const_cast<Geom*>(&g), const_cast<void**>(&src), &dst, &c, &fw};
        e = cudaLaunchKernel(func, grid, dim3(c.nt), args, c.smem, st);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_win_raw(const Geom& g, int method, const void* src, void* dst, WinCfg c, cudaStream_t st)
{
    const int mode = raw_store_mode(g, dst, 1, g.C == 3 ? 4 : 4 * g.C, 0);
    void* func = method == M_BILINEAR ? raw_kernel_bilinear(g.C, c.pat - 1, mode) : raw_kernel_bicubic(g.C, c.pat - 1, mode);
    return launch_raw(g, func, raw_strip(c.nt, raw_overlap(mode, 1)), src, dst, c, nullptr, st);
}

bool win_raw_norm_ok(const Geom& g, const void* dst, const WinCfg& c, const NormOut& no, const WinCfg& fp32)
{
    const bool x2 = c.pat == kRawX2 + 1;
    // three FP32 planes of an exact x2 are all stores: the form on consecutive
    // pairs keeps them a little faster (16 x 512^2 bicubic 38 us, here 39.5)
    if (x2 && no.dtype == DT_F32 && g.C == 3) return false;
    // Small outputs, whose shortest bands (one row; two of an exact x2) all run
    // at once on the FP32 forms: a block is all start-up, which takes longer
    // here (RGB 54 x 55 -> 27 x 28 bicubic 7.3 us, on FP32 rows 3.9; RGB exact
    // x2 to 152 x 340 bilinear 3.7 and 2.9).
    const int px = fp32.nt * win_pixels(g.C, DT_U8, x2);
    const int64_t blocks = ((int64_t)g.Wo + px - 1) / px * ((g.Ho + x2) / (x2 ? 2 : 1)) * g.planes;
    const int64_t per_sm = std::min<int64_t>(x2 ? 4 : 2, 228 * 1024 / ((int64_t)fp32.smem + 1024));
    if (blocks <= num_sms() * per_sm) return false;
    const size_t es = dtype_size(no.dtype);
    return c.pat == 2 + 1 || c.pat == 4 + 1 || raw_store_mode(g, dst, es, kRawP * (int)es, no.c_stride) == RAW_WORDS;
}

cudaError_t launch_win_raw_norm(const Geom& g, int method, const void* src, void* dst, WinCfg c, const NormOut& no,
                                cudaStream_t st)
{
    const size_t es = dtype_size(no.dtype);
    const int mode = raw_store_mode(g, dst, es, kRawP * (int)es, no.c_stride);
    void* func = method == M_BILINEAR ? raw_norm_bilinear(g.C, c.pat - 1, mode, no.dtype)
                                      : raw_norm_bicubic(g.C, c.pat - 1, mode, no.dtype);
    return launch_raw(g, func, raw_strip(c.nt, raw_overlap(mode, es)), src, dst, c, &no, st);
}

#elif WIN_RAW_PART == 1
void* raw_kernel_bicubic(int C, int pat, int st) { return raw_func(C, pat, st, DT_U8); }
#elif WIN_RAW_PART == 2
void* raw_norm_bilinear(int C, int pat, int st, int out_dtype) { return raw_func(C, pat, st, out_dtype); }
#else
void* raw_norm_bicubic(int C, int pat, int st, int out_dtype) { return raw_func(C, pat, st, out_dtype); }
#endif

}  // namespace rs
