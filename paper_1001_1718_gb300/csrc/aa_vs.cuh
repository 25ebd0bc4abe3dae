// Antialiased resampling of vertical downscales, vertical pass first, with
// the source rows streamed once through a shared-memory copy ring and the
// vertical sums kept in registers (RS_FLAG_ANTIALIAS where the output rows
// are no more than the source rows and the window forms do not apply).
//
// One block of nt threads per output tile of TW columns x TH rows of one
// plane. The tile's source footprint (the source columns its TW outputs' x
// taps reach, times the channels: at most E elements per thread) is walked
// once, top to bottom. Rows are copied with 16-byte cp.async (one warp per
// row, rows lying the source pitch mod 16 apart so that every row keeps its
// address mod 16) into a three-slot ring of R-row chunks, two chunks ahead.
// Thread t owns footprint elements E t .. E t + E - 1: it reads them as words
// (AL: where the rows lie a whole number of E elements apart, in one aligned
// load, the ownership starting up to E - 1 elements before the footprint),
// widens them and adds the row, weighted, into NA sets of sums, one for every
// output row whose taps can include the row at once (2 bilinear, 4 bicubic:
// the stretched kernel is NA output steps long, and output row i + NA starts
// at or below row i's last tap). A per-row table holds the row's weight in
// each set, row i in set i mod NA, 0 elsewhere, as the pair that a packed FMA
// takes; where the pairs of one output row do not fit in shared memory the
// table holds the weights once and the pairs of one chunk at a time (single).
// The loop over output rows is unrolled four times, so the sets are registers
// with fixed roles: row i is complete where its taps end. Four complete rows
// go to shared memory as two interleaved pairs, and between two barriers the
// block blends them with the x taps (a thread per output column, two rows per
// packed FMA) and stores the outputs. Sums run over the taps in ascending
// order, y first, then x.
//
// What bounds it: instruction issue at 16 warps per SM (16 RGB 1080p frames to
// 455 x 256, bilinear: 34 M warp instructions, about half the issue slots; 36
// per source row and warp, a quarter of all in the blend, a tenth in a
// block's start-up). The form it replaces (4 elements per thread read byte by
// byte, sums in slots selected at run time, tiles of a power-of-two width)
// issued 134 M. Measured: 177 -> 59 us; on the way, against 62-65: the words
// read by funnel shifts at every pitch 70; five blocks of 96 registers per SM 67.
#pragma once

#include <type_traits>

#include "rs_common.cuh"

namespace rs {

static constexpr int kVsNT = 128;     // threads per block, at most
static constexpr int kVsMaxNT = 256;  // where one output column's footprint asks for more

// Footprint elements per thread: 8 bytes or halves, 4 floats.
constexpr __host__ __device__ int vs_elems(int es) { return es == 4 ? 4 : 8; }
// Words a thread reads of a row.
constexpr __host__ __device__ int vs_words(int es) { return vs_elems(es) * es / 4 + (es == 4 ? 0 : 1); }
// Shared memory of n rows lying S bytes apart from any 16-byte phase on.
constexpr __host__ __device__ int vs_rows_bytes(int n, int S) { return (n * S + 31) & ~15; }

template <int C, typename T, typename TO, bool NORM, int NA, bool AL>
__device__ __forceinline__ void aa_vs_body(const Geom& g, const T* __restrict__ s, TO* __restrict__ d,
                                           const AaVsCfg& cfg, int bx, int by, float* sm, unsigned int* fault,
                                           const NormOut& no)
{
    constexpr int ES = (int)sizeof(T), E = vs_elems(ES), NRD = vs_words(ES), NW = E * ES / 4;
    const int tid = threadIdx.x, lane = tid & 31, NT = blockDim.x;
    const int TW = cfg.TW, R = cfg.chunk;
    const int j0 = bx * TW, i0 = by * cfg.TH;
    const int nj = min(TW, g.Wo - j0), ni = min(cfg.TH, g.Ho - i0);
    const int m = cfg.method;

    int px_lo, px_hi, r_lo, r_hi, t0, t1;
    aa_range(j0, g.W, g.Wo, m, px_lo, t0);
    aa_range(j0 + nj - 1, g.W, g.Wo, m, t1, px_hi);   // exclusive
    aa_range(i0, g.H, g.Ho, m, r_lo, t0);
    aa_range(i0 + ni - 1, g.H, g.Ho, m, t1, r_hi);
    // AL: rows lie a thread's bytes apart (or a multiple), so owned elements
    // can start on their own boundary: sh elements before the footprint
    const int sh = AL ? (int)(reinterpret_cast<uintptr_t>(s + (int64_t)px_lo * C) % (E * ES)) / ES : 0;
    const int npx = px_hi - px_lo, nr = r_hi - r_lo, ne = npx * C + sh;
    const int per = (ne * ES + 15) / 16 + 1;   // 16-byte blocks around a row's footprint
    // a thread reads bytes [0, 15 + ne ES + 4 NRD) of a raw row
    if (ne > cfg.ve || ne > NT * E || nr > cfg.nr || (per + 1) * 16 > cfg.raw_row || 15 + ne * ES + 4 * NRD > cfg.raw_row ||
        npx < 1 || nr < 1) {
        if (tid == 0) report_fault(fault, FAULT_TILE_SRC_SPAN);   // uniform; bounded by the host
        return;
    }
    const int S = cfg.raw_row + (int)((g.src_pitch * ES) & 15);
    const int slot_bytes = vs_rows_bytes(R, S);
    unsigned char* RAW = reinterpret_cast<unsigned char*>(sm);                           // [3] slots
    float2* V = reinterpret_cast<float2*>(RAW + (size_t)3 * slot_bytes);                 // [2][ve] row pairs
    float2* YW = V + 2 * (size_t)cfg.ve;                                                 // [nr][NA] (w, w), or
    float* YS = reinterpret_cast<float*>(YW + (size_t)(cfg.single ? R : cfg.nr) * NA);   // the current chunk's and [nr][NA] w
    float* WX = YS + (cfg.single ? (size_t)cfg.nr * NA : 0);                             // [TW][KX]
    int* LX = reinterpret_cast<int*>(WX + (size_t)TW * cfg.KX);                          // [TW] first x tap - px_lo
    int* CX = LX + TW;                                                                   // [TW] x tap counts
    int* YH = CX + TW;                                                                   // [TH] last y tap + 1 - r_lo

    // ---- copies: rows [y0, y0 + n) of the footprint into the slot at rb ----
    const uintptr_t plane_lo = reinterpret_cast<uintptr_t>(s);
    const uintptr_t plane_hi = reinterpret_cast<uintptr_t>(s + (int64_t)(g.H - 1) * g.src_pitch + (int64_t)g.W * C);
    const T* const foot = s + (int64_t)r_lo * g.src_pitch + (int64_t)px_lo * C - sh;
    auto row_at = [&](unsigned char* rb, int y0) {
        return rb + (int)(reinterpret_cast<uintptr_t>(foot + (int64_t)y0 * g.src_pitch) & 15);
    };
    auto copy_rows = [&](unsigned char* rb, int y0) {
        const int nn = min(R, nr - y0);
        unsigned char* rs = row_at(rb, y0);
        for (int k = tid >> 5; k < nn; k += NT >> 5) {
            const T* rp = foot + (int64_t)(y0 + k) * g.src_pitch;
            const uintptr_t ra = reinterpret_cast<uintptr_t>(rp);
            const uintptr_t blk = ra & ~(uintptr_t)15;
            unsigned char* dst = rs + k * S;
            const unsigned sdst = (unsigned)__cvta_generic_to_shared(dst);
            if (blk >= plane_lo && blk + 16 * (uintptr_t)per <= plane_hi) {   // uniform over the warp
                for (int w = lane; w < per; w += 32)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((sdst & ~15u) + 16 * w),
                                 "l"(reinterpret_cast<const void*>(blk + 16 * w)) : "memory");
            } else {   // a block would reach outside the plane: element by element
                for (int e = sh + lane; e < ne; e += 32) reinterpret_cast<T*>(dst)[e] = rp[e];
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copy_rows(RAW, 0);
    copy_rows(RAW + slot_bytes, R);

    // ---- tap tables ----
    if (cfg.single)
        #pragma unroll 1
        for (int e = tid; e < nr * NA; e += NT) YS[e] = 0.0f;
    else
        for (int e = tid; e < nr * NA; e += NT) YW[e] = make_float2(0.0f, 0.0f);
    __syncthreads();
    for (int i = tid; i < ni + nj; i += NT) {
        if (i >= ni) {
            const int j = i - ni;
            int lo = 0;
            CX[j] = aa_taps_n(j0 + j, g.W, g.Wo, m, g.a, cfg.KX, lo, WX + j * cfg.KX, fault);
            LX[j] = (lo - px_lo) * C + sh;
            continue;
        }
        // tile row i: its renormalised y taps into its set's column
        int lo, hi;
        aa_range(i0 + i, g.H, g.Ho, m, lo, hi);
        const float inv2F = 1.0f / (2.0f * (float)max(g.H, g.Ho));
        const int step = cfg.single ? NA : 2 * NA;   // floats per row
        float* col = (cfg.single ? YS : reinterpret_cast<float*>(YW)) + (size_t)(lo - r_lo) * step + i % NA * (step / NA);
        float tot = 0.0f;
        for (int k = 0; k < hi - lo; ++k) {
            const float v = aa_kernel(lo + k, i0 + i, g.H, g.Ho, inv2F, m, g.a);
            col[(size_t)k * step] = v;
            tot += v;
        }
        const float inv = tot != 0.0f ? 1.0f / tot : 1.0f;
        for (int k = 0; k < hi - lo; ++k) {
            const float w = col[(size_t)k * step] * inv;
            if (cfg.single) col[(size_t)k * step] = w;
            else *reinterpret_cast<float2*>(col + (size_t)k * step) = make_float2(w, w);
        }
        YH[i] = hi - r_lo;
    }
    copy_rows(RAW + 2 * slot_bytes, 2 * R);
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncthreads();   // tables and chunk 0 visible

    // ---- vertical pass ----
    const int e0 = tid * E;
    const bool own = e0 < ne;
    const int eoff = own ? e0 * ES : 0;
    const uint32_t* const words = reinterpret_cast<const uint32_t*>(sm);
    float2 acc[NA][E / 2];
    #pragma unroll
    for (int q = 0; q < NA; ++q)
        #pragma unroll
        for (int k = 0; k < E / 2; ++k) acc[q][k] = make_float2(0.0f, 0.0f);
    float2 hold[E / 2];   // an even row, until the odd one is complete

    unsigned char* cur = RAW;
    int y = 0, y_end = min(R, nr), cidx = 0;   // next row, end of the current chunk
    int p = (int)(row_at(RAW, 0) - RAW) + eoff;   // the next row's first owned byte in shared memory
    const float2* yw = YW;
    auto pair_weights = [&]() {   // single: rows y .. y_end - 1 as pairs, between two barriers
        #pragma unroll 1
        for (int e = tid; e < (y_end - y) * NA; e += NT) {
            const float w = YS[y * NA + e];
            YW[e] = make_float2(w, w);
        }
        yw = YW;
        __syncthreads();
    };
    if (cfg.single) pair_weights();
    auto next_chunk = [&]() {
        ++cidx;
        unsigned char* freed = cur;
        cur = cur == RAW + 2 * slot_bytes ? RAW : cur + slot_bytes;
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();   // chunk cidx landed; every thread is done with chunk cidx - 1
        copy_rows(freed, (cidx + 2) * R);
        p = (int)(row_at(cur, y) - RAW) + eoff;
        y_end = min(y + R, nr);
        if (cfg.single) pair_weights();
    };
    // the row at p into every set
    auto add_row = [&]() {
        uint32_t x[NRD];
        if constexpr (AL && NW == 2) {
            const uint2 v = *reinterpret_cast<const uint2*>(reinterpret_cast<const unsigned char*>(sm) + p);
            x[0] = v.x; x[1] = v.y;
        } else if constexpr (AL) {
            const uint4 v = *reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(sm) + p);
            x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        } else {
            #pragma unroll
            for (int k = 0; k < NRD; ++k) x[k] = words[(p >> 2) + k];
        }
        float2 f[E / 2];
        if constexpr (ES == 4) {
            #pragma unroll
            for (int k = 0; k < E / 2; ++k) f[k] = make_float2(__uint_as_float(x[2 * k]), __uint_as_float(x[2 * k + 1]));
        } else {
            #pragma unroll
            for (int k = 0; k < NW; ++k) {
                const uint32_t w = AL ? x[k] : __funnelshift_r(x[k], x[k + 1], 8 * p);   // the shift counts mod 32
                if constexpr (ES == 1) {
                    const float2 M = make_float2(-8388608.0f, -8388608.0f);
                    f[2 * k] = __fadd2_rn(make_float2(__int_as_float(__byte_perm(w, 0x4B000000u, 0x7650)),
                                                      __int_as_float(__byte_perm(w, 0x4B000000u, 0x7651))), M);
                    f[2 * k + 1] = __fadd2_rn(make_float2(__int_as_float(__byte_perm(w, 0x4B000000u, 0x7652)),
                                                          __int_as_float(__byte_perm(w, 0x4B000000u, 0x7653))), M);
                } else if constexpr (std::is_same<T, __half>::value) {
                    f[k] = __half22float2(*reinterpret_cast<const __half2*>(&w));
                } else {
                    f[k] = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
                }
            }
        }
        float2 wy[NA];
        #pragma unroll
        for (int q = 0; q < NA; q += 2) {
            const float4 w4 = *reinterpret_cast<const float4*>(yw + q);
            wy[q] = make_float2(w4.x, w4.y);
            wy[q + 1] = make_float2(w4.z, w4.w);
        }
        #pragma unroll
        for (int q = 0; q < NA; ++q)
            #pragma unroll
            for (int k = 0; k < E / 2; ++k) acc[q][k] = __ffma2_rn(wy[q], f[k], acc[q][k]);
        p += S;
        yw += NA;
    };
    auto add_rows = [&](int to) {   // source rows y .. to - 1
        while (y < to) {
            if (y == y_end) next_chunk();   // uniform
            const int ys = min(to, y_end);
            for (; y < ys; ++y) add_row();
        }
    };
    // Sets 1 .. NA - 1 take in the tile's first rows before their own rows
    // begin, with weight 0: nothing, unless a row holds an infinity or a NaN
    // (further down a set's next row begins where its last one ended). So a
    // float set is cleared where its first row begins.
    if constexpr (ES > 1) {
        #pragma unroll 1
        for (int q = 1; q < min(NA, ni); ++q) {
            int lo, hi;
            aa_range(i0 + q, g.H, g.Ho, m, lo, hi);
            add_rows(lo - r_lo);
            #pragma unroll
            for (int t = 1; t < NA; ++t)
                if (t == q)
                    #pragma unroll
                    for (int k = 0; k < E / 2; ++k) acc[t][k] = make_float2(0.0f, 0.0f);
        }
    }
    for (int f0 = 0; f0 < ni; f0 += 4) {
        if (ni - f0 <= 2 && own) {   // no second pair: nothing to blend from it
            float4* v = reinterpret_cast<float4*>(V + cfg.ve + e0);
            #pragma unroll
            for (int k = 0; k < E / 2; ++k) v[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        #pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (f0 + u < ni) {   // uniform
                add_rows(YH[f0 + u]);
                float2 (&a)[E / 2] = acc[u % NA];
                if (u & 1) {
                    if (own) {
                        float4* v = reinterpret_cast<float4*>(V + (u >> 1) * (size_t)cfg.ve + e0);
                        #pragma unroll
                        for (int k = 0; k < E / 2; ++k) v[k] = make_float4(hold[k].x, a[k].x, hold[k].y, a[k].y);
                    }
                } else {
                    #pragma unroll
                    for (int k = 0; k < E / 2; ++k) hold[k] = a[k];
                    if (f0 + u == ni - 1 && own) {   // the tile's last row, alone in its pair
                        float4* v = reinterpret_cast<float4*>(V + (u >> 1) * (size_t)cfg.ve + e0);
                        #pragma unroll
                        for (int k = 0; k < E / 2; ++k) v[k] = make_float4(a[k].x, 0.0f, a[k].y, 0.0f);
                    }
                }
                #pragma unroll
                for (int k = 0; k < E / 2; ++k) a[k] = make_float2(0.0f, 0.0f);
            }
        }
        // ---- horizontal pass of rows f0 .. f0 + 3 (those the tile has), all channels of a column per thread ----
        __syncthreads();   // the row pairs complete
        const int nrow = min(4, ni - f0);
        for (int j = tid; j < nj; j += NT) {
            const float2* v0 = V + LX[j];
            const float2* v1 = v0 + cfg.ve;
            const float* w = WX + j * cfg.KX;
            const int cnt = CX[j];
            float2 a0[C], a1[C];
            #pragma unroll
            for (int c = 0; c < C; ++c) a0[c] = a1[c] = make_float2(0.0f, 0.0f);
            #pragma unroll 2
            for (int k = 0; k < cnt; ++k, v0 += C, v1 += C) {
                const float2 w2 = make_float2(w[k], w[k]);
                #pragma unroll
                for (int c = 0; c < C; ++c) {
                    a0[c] = __ffma2_rn(w2, v0[c], a0[c]);
                    a1[c] = __ffma2_rn(w2, v1[c], a1[c]);
                }
            }
            TO* o = d + (int64_t)(i0 + f0) * g.dst_pitch + (NORM ? j0 + j : (int64_t)(j0 + j) * C);
            #pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (r < nrow) {
                    #pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const float v = r == 0 ? a0[c].x : r == 1 ? a0[c].y : r == 2 ? a1[c].x : a1[c].y;
                        if constexpr (NORM) Store<TO>::put(o + c * no.c_stride, fmaf(v, no.scale[c], no.bias[c]));
                        else Store<TO>::put(o + c, v);
                    }
                    o += g.dst_pitch;
                }
            }
        }
        __syncthreads();   // the pairs free for the next four rows
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");   // nothing in flight when the block ends
}

}  // namespace rs
