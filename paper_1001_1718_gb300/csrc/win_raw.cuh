// Register-window resampling of uint8 sources read in place: the general
// form (any vertical ratio, horizontally at most three source pixels per
// output pixel) of the forward window kernel, the fused pre-process and the
// batch's window items.
//
// A block of nt threads owns a strip of output pixels (all C channels) and a
// band of output rows; every thread owns a run of 4 consecutive pixels of the
// strip for the whole band. Source rows are copied as bytes into a three-slot
// shared-memory ring (cp.async, one warp per row, two chunks ahead). Per
// source row a thread reads the words that hold its footprint (the source
// pixels its 4 pixels' taps reach), shifts them to the footprint's first
// byte, widens every byte once and interpolates its 4 pixels from registers.
// The last KT such rows stay in registers (rotated by renaming, the position
// loop is unrolled KT times) and every output row is blended from them, as in
// win_body.cuh.
//
// Which of the footprint's pixels are a pixel's taps depends on the
// coordinate: pixel k's first tap lies floor(k r) or ceil(k r) source pixels
// right of pixel 0's (r = source pixels per output pixel). A register cannot
// be indexed by a value, so each pixel sums over the whole range of its
// possible taps with weight 0 at the ones it does not have. Adding 0 * x to
// a sum of finite terms leaves it as it is, so every sum equals the general
// form's, in the same order, up to the sign of a zero (uint8 samples are
// always finite; the float dtypes keep win_body, where 0 * inf would not be
// 0). The ranges are compiled for four ratio ranges (RawPat).
//
// What bounds it: instruction issue (about 36 per output pixel and thread at
// RGB bicubic x1.7, ALU and FMA pipes at ~45% each, 65% of the issue slots
// used at 16 warps per SM). Against win_body's general form (FP32 rows staged
// channel-planar, one 4-byte shared load per tap and channel, one byte store
// per element) a thread's shared loads per source row fall from 48 to 7, the
// staging pass and one of two barriers per chunk go, and a row leaves as
// 32-bit words. The row's code has no branch before its stores: with a test
// of the row's alignment and of the strip's end in it, the same instruction
// count ran 25% longer.
#pragma once

#include "win_body.cuh"

namespace rs {


static constexpr int kRawP = 4;   // output pixels per thread

// Ratio ranges: first-tap offsets [lo(k), hi(k)] of pixel k against pixel 0.
// PAT 0: r <= 1/2, 1: 1/2 < r <= 1, 2: 1 < r <= 2, 4: 2 < r <= 3. PAT 3 is the
// exact x2 form (the asymmetric map, both axes exactly doubled): pixel 2u and
// row 2u have t = 0 and are the source samples and window rows themselves,
// pixel 2u + 1 and row 2u + 1 have t = 1/2 and the same weights for every u. A
// position yields two output rows, there are no row tables, and runs start at
// even pixels, bands at even rows.
static constexpr int kRawX2 = 3;
template <int PAT>
struct RawPat {
    static __host__ __device__ constexpr int lo(int k)
    {
        return PAT == 0 ? 0 : PAT == 1 ? (k < 2 ? 0 : 1) : PAT == 2 ? k : PAT == 4 ? 2 * k : k >> 1;
    }
    static __host__ __device__ constexpr int hi(int k)
    {
        return PAT == 0 ? (k == 0 ? 0 : k < 3 ? 1 : 2) : PAT == 1 ? k : PAT == 2 ? 2 * k : PAT == 4 ? 3 * k : k >> 1;
    }
};

// The ratio range of an axis advancing an / am source pixels per output
// pixel, or -1 beyond 3.
inline __host__ __device__ int raw_pattern(int64_t an, int64_t am)
{
    return 2 * an <= am ? 0 : an <= am ? 1 : an <= 2 * am ? 2 : an <= 3 * am ? 4 : -1;
}

// Source pixels of a thread's footprint, and the words read for it.
template <int KT, int PAT>
static __host__ __device__ constexpr int raw_fw() { return RawPat<PAT>::hi(kRawP - 1) + KT; }

// Shared memory of n rows lying S bytes apart from any 16-byte phase on.
inline __host__ __device__ constexpr int raw_rows_bytes(int n, int S) { return (n * S + 31) & ~15; }

// How a row leaves (chosen by the host from the output's alignment):
// RAW_WORDS: every run is whole and on a boundary of its own size (C = 3: of
// 4 bytes): vector stores. RAW_ANY: any output width and alignment; uint8
// runs leave as whole words all the same: warps overlap by one run, so each
// lane has its left neighbour's run and stores the aligned words that end in
// its own; a row's first and last run wait in shared memory and go out by
// bytes at the end of the band. Planar elements leave one by one.
enum { RAW_WORDS = 0, RAW_ANY = 1 };

// Words of a waiting run: the left neighbour's last word and the run's own.
template <int C>
__host__ __device__ constexpr int raw_end_words() { return C == 1 ? 2 : C == 4 ? 8 : 4; }

// Output pixels of a strip: 4 per thread; 31 of a warp's 32 runs where warps
// overlap.
inline __host__ __device__ constexpr bool raw_overlap(int st, size_t out_size) { return st == RAW_ANY && out_size == 1; }
inline __host__ __device__ constexpr int raw_strip(int nt, bool overlap) { return kRawP * (overlap ? 31 * (nt / 32) : nt); }

// The work of one block: strip bx and band by of one plane. TO = uint8_t, or
// the fused pre-process's planar output type.
template <int KT, int C, int PAT, int ST, typename TO>
__device__ __forceinline__ void win_body_raw(const Geom& g, const uint8_t* __restrict__ s, TO* __restrict__ d,
                                             const WinCfg& cfg, int bx, int by, float* sm, unsigned int* fault,
                                             const NormOut& no = NormOut{})
{
    constexpr bool NORM = sizeof(TO) > 1;
    constexpr bool OVL = raw_overlap(ST, sizeof(TO));
    constexpr bool X2 = PAT == kRawX2;
    constexpr int HK = KT / 2 - 1;                 // taps left of a pixel's own sample
    constexpr int P = kRawP;
    constexpr int E = P * C, NV = E / 2;           // elements, register pairs of a row
    constexpr int FW = raw_fw<KT, PAT>();          // footprint pixels
    constexpr int FPL = FW * C;                    // footprint bytes
    constexpr int NF = (FPL + 3) / 4, NR = NF + 1; // footprint words, words read
    using RP = RawPat<PAT>;
    const int tid = threadIdx.x, lane = tid & 31, NT = blockDim.x;

    const int strip = raw_strip(NT, OVL);
    const int j_lo = max(0, bx * strip - (OVL ? P : 0));      // first pixel of the footprint
    const int j_hi = min(g.Wo, bx * strip + strip) - 1;       // last pixel of the strip
    const int yb = by * cfg.band_h;
    const int ye = min(g.Ho, yb + cfg.band_h);
    const int nrows = ye - yb;

    // Footprint of the strip: source pixels [px_lo, px_hi], unclamped; the
    // raw copy of a row starts at byte base = px_lo C.
    const int px_lo = first_tap<KT>(j_lo, g.W, g.Wo, g.coord);
    const int px_hi = first_tap<KT>(j_hi, g.W, g.Wo, g.coord) + KT - 1;
    const int base = px_lo * C;
    const int span = (px_hi - px_lo + 1) * C;
    const int per = (span + 15) / 16 + 1;         // raw 16-byte blocks per row
    const int in_lo = max(0, -px_lo) * C;         // raw bytes [in_lo, in_hi) are in the image
    const int in_hi = (min(px_hi, g.W - 1) + 1) * C - base;
    if ((per + 1) * 16 > cfg.raw_row || 15 + span + 4 * NR > cfg.raw_row || nrows > cfg.band_cap ||
        (X2 && ((yb | nrows) & 1))) {
        if (tid == 0) report_fault(fault, FAULT_TILE_SRC_SPAN);   // uniform over the block
        return;
    }
    const int R = cfg.chunk;
    const int npos4 = (cfg.pos_cap + KT - 1) / KT * KT;
    float2* RW = reinterpret_cast<float2*>(sm);                          // [band_cap][KT] (w, w)
    int* NC = reinterpret_cast<int*>(RW + (size_t)cfg.band_cap * KT);    // [npos4] rows per position
    int* RF = NC + npos4;                                                // [band_cap] first taps
    constexpr int EW = raw_end_words<C>();
    uint32_t* ENDS = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(sm) + cfg.tab_off);   // [2][band_cap][EW] (OVL)
    unsigned char* RAW = reinterpret_cast<unsigned char*>(sm) + cfg.raw_off;   // [KT - 1 rows], [3][R rows]
    const bool edge = px_lo < 0 || px_hi >= g.W;                         // uniform over the block

    // ---- staging ----
    const int b_first = first_tap<KT>(yb, g.H, g.Ho, g.coord);
    const int b_last = first_tap<KT>(ye - 1, g.H, g.Ho, g.coord);   // positions of the band
    if (b_last - b_first + 1 > cfg.pos_cap) {   // uniform; the host bounds the positions
        if (tid == 0) report_fault(fault, FAULT_TILE_SRC_SPAN);
        return;
    }
    // Rows lie S bytes apart in shared memory, S = the source pitch mod 16, so
    // every row keeps its global address mod 16 and 16-byte blocks copy to
    // 16-byte blocks (rows past the image's top or bottom repeat the edge row
    // and are copied by bytes where that breaks).
    const int S = cfg.raw_row + (int)(g.src_pitch & 15);
    const uintptr_t plane_lo = reinterpret_cast<uintptr_t>(s);
    const uintptr_t plane_hi = reinterpret_cast<uintptr_t>(s + (int64_t)(g.H - 1) * g.src_pitch + (int64_t)g.W * C);
    const int r_first = b_first, r_end = b_last + KT;   // source rows [r_first, r_end)
    const int warp = tid >> 5, nwarps = NT >> 5;
    // the first footprint byte of row r in the slot at rb whose first row is r0
    auto row_at = [&](unsigned char* rb, int r0) {
        return rb + (int)((reinterpret_cast<uintptr_t>(s) + base + (int64_t)r0 * g.src_pitch) & 15);
    };
    auto copy_rows = [&](unsigned char* rb, int r0, int n) {
        const int nn = min(n, r_end - r0);
        unsigned char* rs = row_at(rb, r0);
        for (int k = warp; k < nn; k += nwarps) {
            const uint8_t* rp = s + (int64_t)clampi(r0 + k, g.H) * g.src_pitch + base;
            const uintptr_t ra = reinterpret_cast<uintptr_t>(rp);
            const uintptr_t blk = ra & ~(uintptr_t)15;
            unsigned char* dst = rs + k * S;
            const unsigned sdst = (unsigned)__cvta_generic_to_shared(dst);
            if (((sdst ^ (unsigned)ra) & 15) == 0 && blk >= plane_lo && blk + 16 * (uintptr_t)per <= plane_hi) {   // uniform over the warp
                for (int w = lane; w < per; w += 32)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((sdst & ~15u) + 16 * w),
                                 "l"(reinterpret_cast<const void*>(blk + 16 * w)) : "memory");
            } else {
                for (int e = in_lo + lane; e < in_hi; e += 32) dst[e] = rp[e];
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int slot_bytes = raw_rows_bytes(R, S);
    unsigned char* const RING = RAW + raw_rows_bytes(KT - 1, S);
    const int rc = r_first + KT - 1;    // chunk c: rows [rc + c R, rc + (c + 1) R)
    copy_rows(RAW, r_first, KT - 1);
    copy_rows(RING, rc, R);
    copy_rows(RING + slot_bytes, rc + R, R);

    // ---- row taps ----
    if constexpr (!X2)
    for (int i = tid; i < nrows; i += NT) {
        float w[KT];
        RF[i] = taps<KT>(yb + i, g.H, g.Ho, g.coord, g.a, w);
        #pragma unroll
        for (int q = 0; q < KT; ++q) RW[i * KT + q] = make_float2(w[q], w[q]);
    }
    if constexpr (!X2)
    for (int q = tid; q < npos4; q += NT) NC[q] = 0;

    // ---- this thread's pixels and their column weights over the ranges ----
    const int j0 = OVL ? bx * strip + P * (tid - (tid >> 5) - 1) : j_lo + P * tid;
    const int nact = j0 < 0 ? 0 : max(0, min(P, j_hi - j0 + 1));   // pixels of the run inside the image and strip
    constexpr int TW = KT + RP::hi(P - 1) - RP::lo(P - 1);   // widest range
    float wx[P][TW];
    float whalf[KT];   // X2: the t = 1/2 weights
    tap_weights<KT>(0.5f, g.a, whalf);
    int toff = 0;   // the footprint's first byte in the raw row, before the row's phase
    if constexpr (X2) {
        if (nact > 0) toff = (j0 / 2 - HK - px_lo) * C;
    } else {
        int f0 = 0;
        #pragma unroll
        for (int k = 0; k < P; ++k) {
            #pragma unroll
            for (int t = 0; t < TW; ++t) wx[k][t] = 0.0f;
            if (k < nact) {
                float w[KT];
                const int f = taps<KT>(j0 + k, g.W, g.Wo, g.coord, g.a, w);
                if (k == 0) f0 = f;
                const int d = f - f0 - RP::lo(k);   // 0 .. hi(k) - lo(k)
                if (d < 0 || d > RP::hi(k) - RP::lo(k)) report_fault(fault, FAULT_TILE_SRC_SPAN);
                #pragma unroll
                for (int t = 0; t < KT + RP::hi(k) - RP::lo(k); ++t)
                    #pragma unroll
                    for (int q = 0; q < KT; ++q)
                        if (t - q == d) wx[k][t] = w[q];
            }
        }
        if (nact > 0) toff = (f0 - px_lo) * C;
    }
    if constexpr (!X2) {
    __syncthreads();   // row taps visible, NC cleared
    for (int i0 = tid; i0 < nrows; i0 += NT) {   // rows per position (runs of equal first taps)
        if (i0 == 0 || RF[i0] != RF[i0 - 1]) {
            int len = 1;
            while (i0 + len < nrows && RF[i0 + len] == RF[i0]) ++len;
            NC[RF[i0] - b_first] = len;
        }
    }
    }
    // edge pads of landed rows: bytes outside [in_lo, in_hi) take the edge pixel
    auto padfix = [&](unsigned char* rb, int r0, int n) {
        const int nn = min(n, r_end - r0);
        const int npad = in_lo + (span - in_hi);
        unsigned char* rs = row_at(rb, r0);
        for (int u = tid; u < nn * npad; u += NT) {
            const int k = u / npad, q0 = u - k * npad;
            const int q = q0 < in_lo ? q0 : in_hi + (q0 - in_lo);
            const int src = (q < in_lo ? in_lo : in_hi - C) + q % C;
            rs[k * S + q] = rs[k * S + src];
        }
    };

    // Register pairs of a row of E values: C = 1: pixels (0, 1), (2, 3);
    // C = 2, 4: channel pairs of each pixel; C = 3: channels (0, 1) of each
    // pixel, then channel 2 of pixels (0, 1), (2, 3).
    auto get = [&](const float2 (&v)[NV], int k, int c) -> float {
        if constexpr (C == 1) return (k & 1) ? v[k >> 1].y : v[k >> 1].x;
        else if constexpr (C == 3) return c == 2 ? ((k & 1) ? v[4 + (k >> 1)].y : v[4 + (k >> 1)].x) : c ? v[k].y : v[k].x;
        else return (c & 1) ? v[k * (C / 2) + (c >> 1)].y : v[k * (C / 2) + (c >> 1)].x;
    };

    // ---- horizontal pass of a raw row in which this thread's footprint starts at byte p of shared memory ----
    const uint32_t* const words = reinterpret_cast<const uint32_t*>(sm);
    auto hrow = [&](int p, float2 (&h)[NV]) {
        uint32_t x[NR], y[NF];
        #pragma unroll
        for (int k = 0; k < NR; ++k) x[k] = words[(p >> 2) + k];
        const int sh = 8 * p;   // funnel shifts take it mod 32
        #pragma unroll
        for (int k = 0; k < NF; ++k) y[k] = __funnelshift_r(x[k], x[k + 1], sh);
        const float2 M = make_float2(-8388608.0f, -8388608.0f);
        auto magic = [&](int e) { return __int_as_float(__byte_perm(y[e >> 2], 0x4B000000u, 0x7650 + (e & 3))); };
        if constexpr (C == 1) {
            float F[FW + 1];
            #pragma unroll
            for (int e = 0; e < FW; e += 2) {
                const float2 f = __fadd2_rn(make_float2(magic(e), magic(e + 1 < FW ? e + 1 : e)), M);
                F[e] = f.x;
                F[e + 1] = f.y;
            }
            float a[P];
            #pragma unroll
            for (int k = 0; k < P; ++k) {
                if constexpr (X2) {
                    a[k] = F[RP::lo(k) + HK];
                    if (k & 1) {
                        a[k] = whalf[0] * F[RP::lo(k)];
                        #pragma unroll
                        for (int t = 1; t < KT; ++t) a[k] = fmaf(whalf[t], F[RP::lo(k) + t], a[k]);
                    }
                    continue;
                }
                a[k] = wx[k][0] * F[RP::lo(k)];
                #pragma unroll
                for (int t = 1; t < KT + RP::hi(k) - RP::lo(k); ++t) a[k] = fmaf(wx[k][t], F[RP::lo(k) + t], a[k]);
            }
            h[0] = make_float2(a[0], a[1]);
            h[1] = make_float2(a[2], a[3]);
        } else {
            constexpr int CP = C / 2;   // channel pairs per pixel
            float2 F[FW][CP];
            float B[FW + 1];
            #pragma unroll
            for (int f = 0; f < FW; ++f)
                #pragma unroll
                for (int c = 0; c < CP; ++c)
                    F[f][c] = __fadd2_rn(make_float2(magic(f * C + 2 * c), magic(f * C + 2 * c + 1)), M);
            if constexpr (C == 3) {
                #pragma unroll
                for (int f = 0; f < FW; f += 2) {
                    const float2 b = __fadd2_rn(make_float2(magic(f * C + 2), magic((f + 1 < FW ? f + 1 : f) * C + 2)), M);
                    B[f] = b.x;
                    B[f + 1] = b.y;
                }
            }
            float bb[P];
            #pragma unroll
            for (int k = 0; k < P; ++k) {
                float2 a[CP];
                if (X2 && !(k & 1)) {
                    #pragma unroll
                    for (int c = 0; c < CP; ++c) h[k * CP + c] = F[RP::lo(k) + HK][c];
                    if constexpr (C == 3) bb[k] = B[RP::lo(k) + HK];
                    continue;
                }
                #pragma unroll
                for (int t = 0; t < KT + RP::hi(k) - RP::lo(k); ++t) {
                    const float w = X2 ? whalf[t] : wx[k][t];
                    const float2 w2 = make_float2(w, w);
                    #pragma unroll
                    for (int c = 0; c < CP; ++c)
                        a[c] = t == 0 ? __fmul2_rn(w2, F[RP::lo(k)][c]) : __ffma2_rn(w2, F[RP::lo(k) + t][c], a[c]);
                    if constexpr (C == 3) bb[k] = t == 0 ? w * B[RP::lo(k)] : fmaf(w, B[RP::lo(k) + t], bb[k]);
                }
                #pragma unroll
                for (int c = 0; c < CP; ++c) h[k * CP + c] = a[c];
            }
            if constexpr (C == 3) {
                h[4] = make_float2(bb[0], bb[1]);
                h[5] = make_float2(bb[2], bb[3]);
            }
        }
    };

    // ---- output: the run's row at p ----
    const bool run = nact > 0;                                      // RAW_WORDS: whole runs only
    const bool rlast = lane > 0 && run && j0 + P >= g.Wo;           // OVL: the row's last run,
    const bool rfirst = lane > 0 && run && j0 == 0 && !rlast;       // its first
    const bool rmid = lane > 0 && run && !rlast && !rfirst;         // or another that this warp stores
    const bool rend = rfirst || rlast;
    uint32_t* ends = ENDS + (rlast ? cfg.band_cap * EW : 0);
    auto put = [&](TO* p, const float2 (&v)[NV]) {
        if constexpr (NORM) {
            #pragma unroll
            for (int c = 0; c < C; ++c) {
                float y[P];
                #pragma unroll
                for (int k = 0; k < P; ++k) y[k] = fmaf(get(v, k, c), no.scale[c], no.bias[c]);
                TO* pc = p + c * no.c_stride;
                if constexpr (ST == RAW_WORDS) {
                    uint32_t w[P * sizeof(TO) / 4];
                    win_pack_plane<P, TO>(y, w);
                    if (run) {
                        if constexpr (sizeof(TO) == 2) *reinterpret_cast<uint2*>(pc) = make_uint2(w[0], w[1]);
                        else *reinterpret_cast<uint4*>(pc) = make_uint4(w[0], w[1], w[P - 2], w[P - 1]);
                    }
                } else {
                    #pragma unroll
                    for (int k = 0; k < P; ++k)
                        if (k < nact) Store<TO>::put(pc + k, y[k]);
                }
            }
        } else {
            uint32_t w[C];
            #pragma unroll
            for (int q = 0; q < C; ++q) {
                uint32_t b[4];
                #pragma unroll
                for (int i = 0; i < 4; ++i) b[i] = win_u8(get(v, (4 * q + i) / C, (4 * q + i) % C));
                w[q] = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
            }
            if constexpr (ST == RAW_WORDS) {
                if (run) {
                    if constexpr (C == 4) *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
                    else if constexpr (C == 2) *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
                    else {
                        #pragma unroll
                        for (int q = 0; q < C; ++q) reinterpret_cast<uint32_t*>(p)[q] = w[q];
                    }
                }
            } else {
                const int ph = (int)(reinterpret_cast<uintptr_t>(p) & 3);   // the row's, in every lane
                const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, w[C - 1], 1);
                uint32_t* a = reinterpret_cast<uint32_t*>(p - ph);
                uint32_t x[C];   // aligned words, shifted outside the tests (predicated stores, no branch)
                x[0] = __funnelshift_l(prev, w[0], 8 * ph);
                #pragma unroll
                for (int q = 1; q < C; ++q) x[q] = __funnelshift_l(w[q - 1], w[q], 8 * ph);
                #pragma unroll
                for (int q = 0; q < C; ++q)
                    if (rmid) a[q] = x[q];
                if constexpr (C == 1) {
                    if (rend) *reinterpret_cast<uint2*>(ends) = make_uint2(prev, w[0]);
                } else {
                    if (rend) *reinterpret_cast<uint4*>(ends) = make_uint4(prev, w[0], w[1], w[C > 2 ? 2 : 1]);
                    if (C == 4 && rend) ends[4] = w[C - 1];
                }
                ends += EW;
            }
        }
    };

    float2 win[KT][NV];   // win[x]: source row b + x at position b (slots rotate)
    auto blend = [&](const float2* wrow, const int* slot, float2 (&v)[NV]) {
        float2 wr[KT];
        #pragma unroll
        for (int q = 0; X2 && q < KT; ++q) wr[q] = make_float2(whalf[q], whalf[q]);
        #pragma unroll
        for (int q = 0; !X2 && q < KT; q += 2) {
            const float4 w4 = *reinterpret_cast<const float4*>(wrow + q);
            wr[q] = make_float2(w4.x, w4.y);
            wr[q + 1] = make_float2(w4.z, w4.w);
        }
        #pragma unroll
        for (int e = 0; e < NV; ++e) v[e] = __fmul2_rn(wr[0], win[slot[0]][e]);
        #pragma unroll
        for (int q = 1; q < KT; ++q)
            #pragma unroll
            for (int e = 0; e < NV; ++e) v[e] = __ffma2_rn(wr[q], win[slot[q]][e], v[e]);
    };

    // ---- prologue: the first rows and chunks 0, 1, 2 in flight; the first rows and chunk 0 landed ----
    copy_rows(RING + 2 * slot_bytes, rc + 2 * R, R);
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncthreads();
    if (edge) {
        padfix(RAW, r_first, KT - 1);
        padfix(RING, rc, R);
        __syncthreads();
    }
    {
        int p = (int)(row_at(RAW, r_first) - reinterpret_cast<unsigned char*>(sm)) + toff;
        #pragma unroll
        for (int x = 0; x < KT - 1; ++x, p += S) hrow(p, win[x]);
    }
    const int npos = b_last - b_first + 1;
    const float2* wrow = RW;
    TO* out = d + (int64_t)yb * g.dst_pitch + (int64_t)j0 * (NORM ? 1 : C);   // this run's next row
    unsigned char* cur = RING;
    for (int c = 0, pos = 0; pos < npos; ++c) {
        if (c > 0) {
            unsigned char* freed = cur;
            cur = cur == RING + 2 * slot_bytes ? RING : cur + slot_bytes;
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();   // chunk c landed; every thread is done with chunk c - 1
            if (edge) {
                padfix(cur, rc + c * R, R);
                __syncthreads();
            }
            copy_rows(freed, rc + (c + 2) * R, R);
        }
        int p = (int)(row_at(cur, rc + c * R) - reinterpret_cast<unsigned char*>(sm)) + toff;
        const int pend = min(npos, pos + R);
        // KT positions at a time (past the band's last: rows that nothing is blended from)
        for (; pos < pend; pos += KT) {
            int nb[KT];
            if constexpr (X2) {
                #pragma unroll
                for (int u = 0; u < KT; ++u) nb[u] = pos + u < npos;
            } else if constexpr (KT == 4) {
                const int4 n4 = *reinterpret_cast<const int4*>(NC + pos);
                nb[0] = n4.x; nb[1] = n4.y; nb[2] = n4.z; nb[3] = n4.w;
            } else {
                const int2 n2 = *reinterpret_cast<const int2*>(NC + pos);
                nb[0] = n2.x; nb[1] = n2.y;
            }
            #pragma unroll
            for (int u = 0; u < KT; ++u, p += S) {
                hrow(p, win[(u + KT - 1) % KT]);
                int slot[KT];
                #pragma unroll
                for (int x = 0; x < KT; ++x) slot[x] = (u + x) % KT;
                if constexpr (X2) {
                    if (nb[u]) {   // rows 2u (the window row itself) and 2u + 1
                        float2 v[NV];
                        blend(wrow, slot, v);
                        put(out, win[slot[HK]]);
                        put(out + g.dst_pitch, v);
                        out += 2 * g.dst_pitch;
                    }
                    continue;
                }
                #pragma unroll 1
                for (int k = nb[u]; k > 0; --k) {
                    float2 v[NV];
                    blend(wrow, slot, v);
                    put(out, v);
                    wrow += KT;
                    out += g.dst_pitch;
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");   // nothing in flight when the block moves on
    if constexpr (OVL) {
        // the waiting runs: a row's first run up to the word its neighbour
        // stored, its last from the neighbour's tail on
        const int jl = (g.Wo - 1) / P * P;
        const bool has_last = bx == jl / strip, has_first = bx == 0 && jl > 0;
        if (!has_first && !has_last) return;   // uniform
        __syncthreads();
        for (int u = tid; u < 2 * nrows; u += NT) {
            const bool last = u >= nrows;
            const int i = last ? u - nrows : u;
            if (last ? !has_last : !has_first) continue;
            const int j = last ? jl : 0;
            unsigned char* p = reinterpret_cast<unsigned char*>(d + (int64_t)(yb + i) * g.dst_pitch + (int64_t)j * C);
            const int ph = (int)(reinterpret_cast<uintptr_t>(p) & 3);
            const uint32_t* w = ENDS + (last ? cfg.band_cap * EW : 0) + i * EW;
            const int lo = last && j > 0 ? -ph : 0, hi = last ? (g.Wo - j) * C : E - ph;
            for (int e = lo; e < hi; ++e) p[e] = (unsigned char)(w[(e + 4) >> 2] >> (8 * (e & 3)));
        }
    }
}

}  // namespace rs
