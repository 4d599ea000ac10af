// Boxcar scan of finished dedispersion tiles inside the dedispersion CTA: the fused
// path of dd_dedisperse_boxcar (contiguous widths w0 .. w0 + nw - 1).  Integer plans
// (exact sums) first, then fp32 plans (the unfused fp32 scan's prefix chains).
// Included by dd_tile.cuh.
//
// A CTA walks its part of the launch's (trial block, time tile) items in order, a strip
// of consecutive tiles per trial block it touches.  After a tile's channel sum, each
// warp group writes its trial's outputs, minus the trial's offset o_d, into a shared-
// memory row behind the last C = wmax - 1 outputs of the previous tile (the carry), so
// that the row holds x[T0 - C .. T0 + L).  The tile then owns the window starts
// t in [T0 - C, T0 + L - C): every window of width <= wmax from such a start lies in
// the row.  The strip's first tile has no carry and starts at the strip start; its last
// tile also takes the starts up to the strip end, with windows cut off there; windows
// that cross a strip boundary are left to the seam pass (dd_fused.cu).
//
// Lane l of a warp owns the kRInt starts i0 = l * kRInt + s of a row segment and walks
// them for G widths at a time with a rotating register window of prefix sums: one
// subtract and one max per (start, width), in uint32 arithmetic whose differences are
// exact while every window sum of x - o fits int32 (checked per output against mlim;
// DD_ERR_OVERFLOW otherwise).  A warp reduction gives the tile's maximum per width;
// only where it beats (or ties from an earlier start) the merged maximum read from
// `key` is the earliest start searched -- the earliest segment holding the maximum
// writes its prefix values to the warp's scratch and the lanes test one start each --
// and (value, start) merged with one 64-bit atomicMax.
#pragma once

#include <cfloat>
#include <climits>

#include "dd_internal.h"

namespace dd {
namespace fused {
namespace {

constexpr int G = 16;  // widths per register window

// A warp's shared scratch for the earliest-start search (4-byte words): the prefix values
// P_0 .. P_30 of one segment, then P_{w0g} .. P_{w0g+45} (every P_s and P_{s+w} that a
// width of the group forms).  The packed row kernels' segments are 34 starts, of which 32 lanes
// make their 1088-output tile exactly: 35 (odd, so without the two-way bank conflicts) left one
// lane a partial segment, and its warp the masked scan beside the full one for every group
// (1500 low-band trials x 1024 channels x 35300 outputs, widths 1-256: 8.01 ms with 35, 5.94 with
// 34 and two starts per step; widths 1-64: 4.84 and 4.34).
constexpr int kSegPk = 34;
constexpr int kChainFloats = 2 * kSegPk + G - 1;

// Where the fused epilogue of a row kernel's tile (epilogue_pk, epilogue_f32) keeps what, in
// 4-byte words of the CTA's shared memory; the launch sizes it and the epilogues address it by
// this one table.  A row per trial, C + 48 words that the last row's reads may run into, then the
// warps' scratch.  one_row, where that is more than a CTA can have: a row per warp group, the
// scratch, then its other trials' waiting sums; reads past the last row run into those (what they
// return belongs to no window).  One row fits for every carry the call takes (1088- and 864-output
// tiles, 8 and 16 warps); it costs a copy and two barriers per further trial of a tile
// (packed, 1500 low-band trials x 1024 channels x 35300 outputs: widths 602-633 in two rows take 4.63 ms,
// 604-635 in one 4.63, 700-731 4.72; the tap kernel's scan of the last 21.8).
struct RowScan {
    int chain, wait, words;
    __host__ __device__ RowScan(int kind, int nw, int nch, int rowlen, int C, bool one_row) {
        const int nt = row_unit_trials(kind), rows = (one_row ? nw / nch : row_trials(kind, nw, nch)) * rowlen;
        chain = one_row ? rows : rows + C + 48;
        wait = chain + nw * kChainFloats;
        words = wait;
        if (one_row) {
            words += nw * (nt - 1) * row_warp_t(kind);
            if (words < rows + C + 48) words = rows + C + 48;
        }
    }
};

// S starts of one lane segment (x = row + i0) for widths w0g + j, j < G.
// q = sum_{k < w0g} x[k] on entry.  !FULL: starts outside [i_lo, i_hi) and windows
// ending past row index e_hi are left out.
template <bool FULL, int S>
__device__ __forceinline__ void scan_segment(const int* x, uint32_t q, int w0g, int i0, int i_lo,
                                             int i_hi, int e_hi, int (&seg)[G]) {
    uint32_t win[G];
    win[0] = q;
#pragma unroll
    for (int j = 1; j < G; ++j) win[j] = win[j - 1] + (uint32_t)x[w0g + j - 1];
    auto val = [&](uint32_t P, uint32_t p, int s, int j) {
        return FULL || (i0 + s >= i_lo && i0 + s < i_hi && i0 + s + w0g + j <= e_hi) ? (int)(P - p) : INT_MIN;
    };
    uint32_t p = 0;
    if constexpr (S % 2 == 0) {  // two starts per step, merged with one three-input maximum
#pragma unroll
        for (int s = 0; s < S; s += 2) {
            const uint32_t p1 = p + (uint32_t)x[s];
            const uint32_t next = win[(s + G - 1) % G] + (uint32_t)x[s + w0g + G - 1];
#pragma unroll
            for (int j = 0; j < G; ++j)
                seg[j] = __vimax3_s32(seg[j], val(win[(j + s) % G], p, s, j),
                                      val(j + 1 < G ? win[(j + s + 1) % G] : next, p1, s + 1, j));
            win[s % G] = next;
            p = p1 + (uint32_t)x[s + 1];
            win[(s + 1) % G] = next + (uint32_t)x[s + w0g + G];
        }
    } else {  // (the tap kernel's epilogue, which would spill more)
#pragma unroll
        for (int s = 0; s < S; ++s) {
#pragma unroll
            for (int j = 0; j < G; ++j) seg[j] = max(seg[j], val(win[(j + s) % G], p, s, j));
            p += (uint32_t)x[s];
            win[s % G] = win[(s + G - 1) % G] + (uint32_t)x[s + w0g + G - 1];
        }
    }
}

// Maximum over the warp of seg[j] for all j at once (each exchange level halves the
// values a lane keeps): lanes 2j and 2j + 1 return the maximum for j.
__device__ __forceinline__ int warp_max16(const int (&seg)[G], int lane) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    int v8[8], v4[4], v2[2];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v8[j] = max(b4 ? seg[j + 8] : seg[j], __shfl_xor_sync(0xffffffffu, b4 ? seg[j] : seg[j + 8], 16));
#pragma unroll
    for (int j = 0; j < 4; ++j)
        v4[j] = max(b3 ? v8[j + 4] : v8[j], __shfl_xor_sync(0xffffffffu, b3 ? v8[j] : v8[j + 4], 8));
#pragma unroll
    for (int j = 0; j < 2; ++j)
        v2[j] = max(b2 ? v4[j + 2] : v4[j], __shfl_xor_sync(0xffffffffu, b2 ? v4[j] : v4[j + 2], 4));
    int v = max(b1 ? v2[1] : v2[0], __shfl_xor_sync(0xffffffffu, b1 ? v2[0] : v2[1], 2));
    return max(v, __shfl_xor_sync(0xffffffffu, v, 1));
}

// Upper bound of every sum the FULL scan of one width group would form:
// max_{s, j} P[s + w0g + j] - min_s P[s] <= Q + Mrel, with P the prefix of the segment,
// Q = P[w0g] - min_s P[s] and Mrel = max(0, max_m sum_{k=w0g}^{w0g+m} x[k]), m < cnt + S - 2.
// Q is a window sum of at most wmax values and Mrel one of at most S + 14, so both are
// exact in int32 when wmax >= S + 15 (every such sum fits, by the overflow check).
template <int S>
__device__ __forceinline__ long long group_bound(const int* x, uint32_t q, uint32_t pmin, int w0g, int cnt) {
    int r = 0, mrel = 0;
    for (int m = 0; m < cnt + S - 2; ++m) {
        r += x[w0g + m];
        mrel = max(mrel, r);
    }
    return (long long)(int)(q - pmin) + mrel;
}

// Width groups from prune_w on skip the scan of segments whose group_bound is below
// the smallest merged maximum of the group (strictly: a tie from an earlier start could
// still win), which on noise-like series is most of them.  (Groups of 34-start segments
// from 49 on.)
template <int S>
__host__ __device__ constexpr int prune_w() { return S + 15 > 48 ? S + 15 : 48; }

// The search for the earliest start is latency in one warp of a CTA that waits for it at the tile's
// end, and common in the first tiles of a part: the holders of all widths are found in one pass
// and the holder's prefix values by warp scans from q (a lane walking from the segment's start,
// holders found width by width: 9.55 ms where this takes 8.01, widths 1-256 as above).

// In lanes 2 j and 2 j + 1: the earliest lane whose segment holds width j's maximum, which lane
// 2 j has in mx.
template <typename T>
__device__ __forceinline__ int holders(T mx, const T (&seg)[G], bool scan, int jl) {
    int hold = -1;
#pragma unroll
    for (int j = 0; j < G; ++j) {
        const T mj = __shfl_sync(0xffffffffu, mx, 2 * j);
        const int h = __ffs(__ballot_sync(0xffffffffu, scan && seg[j] == mj)) - 1;
        if (j == jl) hold = h;
    }
    return hold;
}

// out[k] = base + the first k values of x, k < N (a warp).
template <int N>
__device__ __forceinline__ void write_prefix(const int* x, uint32_t base, uint32_t* out, int lane) {
#pragma unroll
    for (int b = 0; b < N; b += 32) {
        const int k = b + lane;
        const uint32_t v = k < N - 1 ? (uint32_t)x[k] : 0u;
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (k < N) out[k] = base + incl - v;
        base += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// The scan of one row for one trial (warp-uniform arguments; see epilogue), S starts per lane.
template <int S>
__device__ __forceinline__ void scan_row(const FusedArgs& f, const int* row, uint32_t* chain,
                                      unsigned long long* keyrow, int64_t T0, int C, int chunk, int nch,
                                      int lane, int i_lo, int i_hi, int e_hi) {
    constexpr int R = S, TT = 32 * R;
    __builtin_assume(__isShared(row));
    const int ng = (f.nw + G - 1) / G;
    const int jl = lane >> 1;
    for (int k = chunk; k * TT < i_hi; k += nch) {
        const int i0 = k * TT + lane * R;
        const int* x = row + i0;
        const bool any = i0 + R > i_lo && i0 < i_hi;
        const bool inner = i0 >= i_lo && i0 + R <= i_hi;
        const int t_lo = (int)(T0 - C) + max(k * TT, i_lo);  // earliest start of the pass
        // lanes without a start here read nothing (their segment may lie past the row)
        uint32_t q = 0, pmin = 0;
        if (any) {
            for (int kk = 0; kk < f.w0; ++kk) q += (uint32_t)x[kk];
            if (inner) {  // min_s P[s] over the segment's starts (sums of < S values)
                int r = 0, mn = 0;
                for (int s = 0; s < R - 1; ++s) {
                    r += x[s];
                    mn = min(mn, r);
                }
                pmin = (uint32_t)mn;
            }
        }
        for (int g = 0; g < ng; ++g) {
            const int w0g = f.w0 + g * G;
            const int cnt = min(G, f.nw - g * G);
            unsigned long long bk = 0;
            if (!(lane & 1) && jl < cnt) bk = __ldcg(keyrow + g * G + jl);
            const int bv = (int)((uint32_t)(bk >> 32) ^ 0x80000000u);
            const int bt = (int)(0xffffffffu - (uint32_t)bk);
            const bool full = inner && i0 + R - 1 + w0g + cnt - 1 <= e_hi;
            bool scan = any;
            if (w0g >= prune_w<S>()) {
                // the smallest merged maximum over the group's widths
                int thr = (!(lane & 1) && jl < cnt) ? bv : INT_MAX;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) thr = min(thr, __shfl_xor_sync(0xffffffffu, thr, o));
                if (full && group_bound<S>(x, q, pmin, w0g, cnt) < (long long)thr) scan = false;
            }
            if (__any_sync(0xffffffffu, scan)) {
                int seg[G];
#pragma unroll
                for (int j = 0; j < G; ++j) seg[j] = INT_MIN;
                if (scan && full)
                    scan_segment<true, S>(x, q, w0g, i0, i_lo, i_hi, e_hi, seg);
                else if (scan)
                    scan_segment<false, S>(x, q, w0g, i0, i_lo, i_hi, e_hi, seg);
                const int mx = warp_max16(seg, lane);
                const bool better = !(lane & 1) && jl < cnt && mx > INT_MIN &&
                                    (mx > bv || (mx == bv && t_lo < bt));
                // widths whose maximum beats (or ties from an earlier start) the merged one:
                // the warp writes the prefix values of the earliest segment holding it to its
                // scratch, and the lanes test the starts for every such width that this
                // segment holds first
                unsigned need = __ballot_sync(0xffffffffu, better);
                if (need) {
                    const int hold = holders(mx, seg, scan, jl);
                    while (need) {  // warp-uniform
                        const int h = __shfl_sync(0xffffffffu, hold, __ffs(need) - 1);
                        const int ih = __shfl_sync(0xffffffffu, i0, h);
                        write_prefix<R>(row + ih, 0u, chain, lane);
                        write_prefix<R + G - 1>(row + ih + w0g, __shfl_sync(0xffffffffu, q, h), chain + R, lane);
                        __syncwarp();
                        const unsigned same = __ballot_sync(0xffffffffu, hold == h) & need;
                        for (unsigned rest = same; rest; rest &= rest - 1) {
                            const int hl = __ffs(rest) - 1;
                            const int j = hl >> 1;
                            const int mj = __shfl_sync(0xffffffffu, mx, hl);
                            int at = -1;  // the earliest start of the segment that reaches it
#pragma unroll
                            for (int s0 = 0; s0 < R; s0 += 32) {
                                const int sl = s0 + lane, i = ih + sl;
                                const bool eq = sl < R && i >= i_lo && i < i_hi && i + w0g + j <= e_hi &&
                                                (int)(chain[R + sl + j] - chain[sl]) == mj;
                                const unsigned st = __ballot_sync(0xffffffffu, eq);
                                if (at < 0 && st) at = s0 + __ffs(st) - 1;
                            }
                            if (lane == 0 && at >= 0)
                                atomicMax(keyrow + g * G + j, fused_key(mj, (int)(T0 - C) + ih + at));
                        }
                        need &= ~same;
                        __syncwarp();  // the scratch is rewritten for the next holder
                    }
                }
            }
            if (any)
#pragma unroll
                for (int kk = 0; kk < G; ++kk) q += (uint32_t)x[w0g + kk];
        }
    }
}

// Where a strip of one trial block starts and ends, and what its CTA carries and passes
// on.  seam_in / seam_out: the strip starts / ends inside the block, so its first /
// last C outputs go to that seam ([trial in block][2C], second / first half).
struct FusedTile {
    int64_t s1;         // end of the strip (exclusive), at most t_out
    bool first, last;   // first / last tile of the strip
    int32_t* carry;     // [trials per CTA][C]
    int32_t* seam_in;
    int32_t* seam_out;
};

// The fused epilogue of one tile (every thread of the CTA calls it).  NU trials per
// warp group (acc0, then accr[0 .. NU - 2]); d = the group's first trial, T0 = the
// tile's first output.

template <int NU, int NX>
__device__ __forceinline__ void epilogue(const DedispArgs& a, const FusedArgs& f, unsigned char* smem,
                                         int wu, int chunk, int lane, int d, int64_t T0,
                                         const FusedTile& ft,
                                         const int (&acc0)[kRInt], const int (&accr)[NX][kRInt]) {
    constexpr int R = kRInt, TT = 32 * R;
    const int L = TT * a.nch;
    const int C = f.C;
    int* row = (int*)smem + wu * f.rowlen;
    const int64_t S1 = ft.s1;
    const bool first = ft.first, last = ft.last;
    // row index i holds output T0 - C + i
    const int i_lo = first ? C : 0;             // first start owned by the tile
    const int e_hi = (int)(S1 - T0) + C;        // windows end at or before this index
    const int i_hi = last ? e_hi - f.w0 + 1 : L;  // starts below this index
    // the other trials' sums wait in shared memory behind the rows, so that no
    // accumulator stays live across a scan
    int* spill = (int*)smem + fused_rows_ints(kWarps / a.nch, f.rowlen, C) +
                 (threadIdx.x >> 5) * (NU - 1) * TT + lane * R;
#pragma unroll
    for (int u = 1; u < NU; ++u)
#pragma unroll
        for (int r = 0; r < R; ++r) spill[(u - 1) * TT + r] = accr[u - 1][r];
    // the warp's scratch for the earliest-start search lies behind the spilled sums
    uint32_t* chain = (uint32_t*)smem + fused_rows_ints(kWarps / a.nch, f.rowlen, C) + kWarps * (NU - 1) * TT +
                      (threadIdx.x >> 5) * kChainFloats;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        __syncthreads();  // the rows are free (stages consumed, or the previous trial scanned)
        const int du = d + u;
        const bool live = du < a.ndm;
        const int o = live ? (int)f.off[du] : 0;
        const int ib = C + chunk * TT + lane * R;
        const int64_t tb = T0 + chunk * TT + lane * R;
        int m = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int v = (u == 0 ? acc0[r] : spill[(u - 1) * TT + r]) - o;
            row[ib + r] = v;
            if (tb + r < S1) m = max(m, abs(v));
        }
        if (live && m > f.mlim) atomicExch(a.status, (int)DD_ERR_OVERFLOW);
        const int64_t cb = (int64_t)(wu * NU + u) * C;  // this trial's carry and seam rows
        if (live && chunk == 0 && !first)
            for (int k = lane; k < C; k += 32) row[k] = ft.carry[cb + k];
        __syncthreads();  // the row and its carry are complete
        if (!live) continue;
        if (chunk == 0) {
            if (!last)
                for (int k = lane; k < C; k += 32) ft.carry[cb + k] = row[L + k];
            if (first && ft.seam_in)
                for (int k = lane; k < C; k += 32) ft.seam_in[2 * cb + C + k] = row[C + k];
            if (last && ft.seam_out)
                for (int k = lane; k < C; k += 32) ft.seam_out[2 * cb + k] = row[e_hi - C + k];
        }
        scan_row<kRInt>(f, row, chain, f.key + (int64_t)du * f.nw, T0, C, chunk, a.nch, lane, i_lo, i_hi, e_hi);
    }
    // the next tile's bulk copies overwrite the rows
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
}

// The fused epilogue of one packed integer tile (dd_rows.cuh; every thread of the CTA
// calls it): the unit's two trials d, d + 1, one row each, s[u] = the lane's low sums
// (outputs lane * R + r of the warp's chunk), then its high ones (kPkHalf later).
// ONE_ROW: one row per warp group, the second trial's sums wait in shared memory (a kernel of its
// own: with a run-time switch, narrow lists took 2.5 % longer).
// Segments of 34 starts: 32 lanes cover the 1088-output tile.
template <int R, int NW, bool ONE_ROW>
__device__ __forceinline__ void epilogue_pk(const DedispArgs& a, const FusedArgs& f, unsigned char* smem,
                                            int wu, int chunk, int lane, int d, int64_t T0,
                                            const FusedTile& ft, const int (&s)[2][2 * R]) {
    constexpr int TT = 2 * kPkHalf;
    const int L = TT * a.nch;
    const int C = f.C;
    const RowScan lay(kRowsPk, NW, a.nch, f.rowlen, C, ONE_ROW);
    int* rows = (int*)smem + (ONE_ROW ? 1 : 2) * wu * f.rowlen;
    int* wait = (int*)smem + lay.wait + (int)(threadIdx.x >> 5) * TT + lane * R;  // (ONE_ROW)
    const int64_t S1 = ft.s1;
    const bool first = ft.first, last = ft.last;
    const int i_lo = first ? C : 0;
    const int e_hi = (int)(S1 - T0) + C;
    const int i_hi = last ? e_hi - f.w0 + 1 : L;
    uint32_t* chain = (uint32_t*)smem + lay.chain + (threadIdx.x >> 5) * kChainFloats;
    const int ib = C + chunk * TT + lane * R;
    const int64_t tb = T0 + chunk * TT + lane * R;
    // a trial's row behind its carry
    auto carry_in = [&](int u, int* row) {
        if (d + u < a.ndm && chunk == 0 && !first)
            for (int k = lane; k < C; k += 32) row[k] = ft.carry[(int64_t)(wu * 2 + u) * C + k];
    };
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const bool live = d + u < a.ndm, waits = u == 1 && ONE_ROW;
        const int o = live ? (int)f.off[d + u] : 0;
        int* row = rows + u * f.rowlen;
        int* at = waits ? wait : row + ib;
        int m = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int v0 = s[u][r] - o, v1 = s[u][R + r] - o;
            at[r] = v0;
            at[kPkHalf + r] = v1;
            if (tb + r < S1) m = max(m, abs(v0));
            if (tb + kPkHalf + r < S1) m = max(m, abs(v1));
        }
        if (live && m > f.mlim) atomicExch(a.status, (int)DD_ERR_OVERFLOW);
        if (!waits) carry_in(u, row);
    }
    __syncthreads();  // the rows and their carries are complete
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
        int* row = rows + (ONE_ROW ? 0 : u * f.rowlen);
        if (ONE_ROW && u) {
            __syncthreads();  // the row is free
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                row[ib + r] = wait[r];
                row[ib + kPkHalf + r] = wait[kPkHalf + r];
            }
            carry_in(u, row);
            __syncthreads();
        }
        if (d + u >= a.ndm) {
            if (ONE_ROW) continue;  // (every warp meets the barriers above)
            break;
        }
        const int64_t cb = (int64_t)(wu * 2 + u) * C;
        if (chunk == 0) {
            if (!last)
                for (int k = lane; k < C; k += 32) ft.carry[cb + k] = row[L + k];
            if (first && ft.seam_in)
                for (int k = lane; k < C; k += 32) ft.seam_in[2 * cb + C + k] = row[C + k];
            if (last && ft.seam_out)
                for (int k = lane; k < C; k += 32) ft.seam_out[2 * cb + k] = row[e_hi - C + k];
        }
        scan_row<kSegPk>(f, row, chain, f.key + (int64_t)(d + u) * f.nw, T0, C, chunk, a.nch, lane, i_lo, i_hi, e_hi);
    }
    // the next tile's bulk copies overwrite the rows
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
}

// ----------------------------------------------------------------------------- fp32 plans
//
// The unfused fp32 scan (k_boxcar_run) gives each thread kBoxSeg consecutive starts from
// a multiple of kBoxSeg and forms the segment's prefix chain P_0 = 0,
// P_{k+1} = P_k + x[k] (x = series - o_d in fp32), left to right; the window of width w
// at start s sums to P_{s+w} - P_s.  fp32 addition is deterministic, so a chain formed
// the same way anywhere gives the same sums bit for bit.  The fused scan therefore
// walks whole segments: a tile owns the segments whose first start lies in its start
// range, reads them from its shared-memory row (C = wmax + kBoxSeg - 2 outputs carried
// from the previous tile reach back to any such segment), and keeps the window ends
// that its strip holds; windows of a segment that begins before a strip boundary and
// ends past it go to the seam pass (dd_fused.cu).

// Segment at x (kBoxSeg starts) for widths w0g + j, j < G; q = P_{w0g}.  !FULL: windows
// ending past index e_rel are left out and no sample at or past it is read.  FULL
// reads up to 15 samples past the last window of the group's widths below cnt.
template <bool FULL>
__device__ __forceinline__ void scan_segment_f32(const float* x, float q, int w0g, int e_rel,
                                                 float (&seg)[G]) {
    constexpr int S = kBoxSeg;
    auto ld = [&](int k) { return (FULL || k < e_rel) ? x[k] : 0.f; };
    float win[G];
    win[0] = q;
#pragma unroll
    for (int j = 1; j < G; ++j) win[j] = win[j - 1] + ld(w0g + j - 1);
    float p = 0.f;
    // two starts per step, their sums merged with one three-input max
#pragma unroll
    for (int s = 0; s < S; s += 2) {
        float v0[G];
#pragma unroll
        for (int j = 0; j < G; ++j) {
            v0[j] = win[(j + s) % G] - p;
            if (!FULL) v0[j] = (s + w0g + j <= e_rel) ? v0[j] : -FLT_MAX;
        }
        if (s + 1 < S) {
            p += ld(s);
            win[s % G] = win[(s + G - 1) % G] + ld(s + w0g + G - 1);
#pragma unroll
            for (int j = 0; j < G; ++j) {
                float v = win[(j + s + 1) % G] - p;
                if (!FULL) v = (s + 1 + w0g + j <= e_rel) ? v : -FLT_MAX;
                seg[j] = max3(seg[j], v0[j], v);
            }
            if (s + 2 < S) {
                p += ld(s + 1);
                win[(s + 1) % G] = win[(s + G) % G] + ld(s + w0g + G);
            }
        } else {
#pragma unroll
            for (int j = 0; j < G; ++j) seg[j] = fmaxf(seg[j], v0[j]);
        }
    }
}

// warp_max16 for fp32 maxima (fmaxf, as the unfused scan).
__device__ __forceinline__ float warp_max16_f32(const float (&seg)[G], int lane) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    float v8[8], v4[4], v2[2];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v8[j] = fmaxf(b4 ? seg[j + 8] : seg[j], __shfl_xor_sync(0xffffffffu, b4 ? seg[j] : seg[j + 8], 16));
#pragma unroll
    for (int j = 0; j < 4; ++j)
        v4[j] = fmaxf(b3 ? v8[j + 4] : v8[j], __shfl_xor_sync(0xffffffffu, b3 ? v8[j] : v8[j + 4], 8));
#pragma unroll
    for (int j = 0; j < 2; ++j)
        v2[j] = fmaxf(b2 ? v4[j + 2] : v4[j], __shfl_xor_sync(0xffffffffu, b2 ? v4[j] : v4[j + 2], 4));
    const float v = fmaxf(b1 ? v2[1] : v2[0], __shfl_xor_sync(0xffffffffu, b1 ? v2[0] : v2[1], 2));
    return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
}

// The segments m_lo <= m < m_hi of one trial's row (row index of output t: t - base;
// windows end at or before row index e_hi), 32 per warp pass, passes shared by the
// nch warps of the trial's group.  Arguments are warp-uniform.
__device__ __forceinline__ void scan_row_f32(int w0, int nw, const float* row, float* chain,
                                             unsigned long long* keyrow, int64_t base, int chunk, int nch,
                                             int lane, int64_t m_lo, int64_t m_hi, int e_hi) {
    constexpr int S = kBoxSeg;
    __builtin_assume(__isShared(row));
    const int ng = (nw + G - 1) / G;
    const int jl = lane >> 1;
    for (int64_t mb = m_lo + (int64_t)chunk * 32; mb < m_hi; mb += (int64_t)nch * 32) {
        const int64_t m = mb + lane;
        const bool any = m < m_hi;
        const int i0 = any ? (int)(m * S - base) : 0;
        const float* x = row + i0;
        const int e_rel = e_hi - i0;
        const int t_first = (int)(mb * S);  // earliest start of the pass
        float q = 0.f;
        if (any)
            for (int k = 0; k < w0; ++k) q += k < e_rel ? x[k] : 0.f;
        for (int g = 0; g < ng; ++g) {
            const int w0g = w0 + g * G;
            const int cnt = min(G, nw - g * G);
            unsigned long long bk = 0;
            if (!(lane & 1) && jl < cnt) bk = __ldcg(keyrow + g * G + jl);
            const float bv = bk ? fused_key_value_f32(bk) : -INFINITY;
            const int bt = (int)(0xffffffffu - (uint32_t)bk);
            const bool full = any && S - 1 + w0g + cnt - 1 <= e_rel;
            float seg[G];
#pragma unroll
            for (int j = 0; j < G; ++j) seg[j] = -FLT_MAX;
            if (full)
                scan_segment_f32<true>(x, q, w0g, e_rel, seg);
            else if (any)
                scan_segment_f32<false>(x, q, w0g, e_rel, seg);
            const float mx = warp_max16_f32(seg, lane);
            const bool better = !(lane & 1) && jl < cnt && mx > -FLT_MAX &&
                                (mx > bv || (mx == bv && t_first < bt));
            // widths whose maximum beats the merged one: the chain of the earliest segment
            // holding it goes to the warp's scratch, and the lanes test one start each for
            // every such width that this segment holds first
            unsigned need = __ballot_sync(0xffffffffu, better);
            if (need) {
                const int hold = holders(mx, seg, any, jl);
                while (need) {  // warp-uniform
                    const int h = __shfl_sync(0xffffffffu, hold, __ffs(need) - 1);
                    const int ih = __shfl_sync(0xffffffffu, i0, h);
                    const int eh = __shfl_sync(0xffffffffu, e_rel, h);
                    const int th = __shfl_sync(0xffffffffu, (int)(m * S), h);
                    const float qh = __shfl_sync(0xffffffffu, q, h);
                    // one lane writes P_0.., another P_{w0g}.. (the chain's own value, q), each in order
                    if (lane < 2) {
                        const int k0 = lane ? w0g : 0, n = lane ? S + G - 1 : S;
                        const float* xh = row + ih + k0;
                        float* out = chain + (lane ? S : 0);
                        float P = lane ? qh : 0.f;
                        for (int k = 0; k < n; k += 8) {
                            float v[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) v[i] = k + i < n - 1 && k0 + k + i < eh ? xh[k + i] : 0.f;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                if (k + i < n) out[k + i] = P;
                                P += v[i];
                            }
                        }
                    }
                    __syncwarp();
                    const unsigned same = __ballot_sync(0xffffffffu, hold == h) & need;
                    for (unsigned rest = same; rest; rest &= rest - 1) {
                        const int hl = __ffs(rest) - 1;
                        const int j = hl >> 1;
                        const float mj = __shfl_sync(0xffffffffu, mx, hl);
                        const bool eq = lane < S && lane + w0g + j <= eh && chain[S + lane + j] - chain[lane] == mj;
                        const unsigned st = __ballot_sync(0xffffffffu, eq);
                        if (lane == 0 && st) atomicMax(keyrow + g * G + j, fused_key_f32(mj, th + __ffs(st) - 1));
                    }
                    need &= ~same;
                    __syncwarp();  // the scratch is rewritten for the next holder
                }
            }
            if (any)
#pragma unroll
                for (int kk = 0; kk < G; ++kk) q += w0g + kk < e_rel ? x[w0g + kk] : 0.f;
        }
    }
}

// Carries, seams and the scan of one trial's row (`sub` of the nsub warps that share it).
// Not inlined: its registers are then allocated apart from the channel sums', which
// keep the whole register file (the calls come once per tile and row).
__device__ __noinline__ void scan_trial_f32(float* row, float* chain, int w0, int nw, int C, int L,
                                            unsigned long long* keyrow, int64_t cb, int sub, int nsub, int lane,
                                            int64_t base, int64_t m_lo, int64_t m_hi, int e_hi, bool first,
                                            bool last, float* carry, float* seam_in, float* seam_out) {
    if (sub == 0) {
        if (!last)
            for (int k = lane; k < C; k += 32) carry[cb + k] = row[L + k];
        if (first && seam_in)
            for (int k = lane; k < C; k += 32) seam_in[2 * cb + C + k] = row[C + k];
        if (last && seam_out)
            for (int k = lane; k < C; k += 32) seam_out[2 * cb + k] = row[e_hi - C + k];
    }
    scan_row_f32(w0, nw, row, chain, keyrow, base, sub, nsub, lane, m_lo, m_hi, e_hi);
}

// The fused epilogue of one fp32 tile (every thread of the CTA calls it): the warp group's
// NT trials d .. d + NT - 1 (sums acc[u]), T0 = the tile's first output; one row per trial.
// The tile owns the segments whose first start lies in [T0 - C, T0 + L - C) (the strip's
// first tile: from T0; its last: up to the strip end S1, windows ending at or before S1).
// NW warps per CTA.  f.one_row: one row per warp group, its other trials' sums wait in
// shared memory.
template <int NT, int R, int NW = kWarps>
__device__ __forceinline__ void epilogue_f32(const DedispArgs& a, const FusedArgs& f, unsigned char* smem,
                                             int wu, int chunk, int lane, int d, int64_t T0,
                                             const FusedTile& ft, const float (&acc)[NT][R]) {
    constexpr int S = kBoxSeg, TT = 32 * R;
    const int L = TT * a.nch;
    const int C = f.C;
    const int64_t S1 = ft.s1;
    const bool first = ft.first, last = ft.last;
    const int64_t base = T0 - C;  // output of row index 0
    const int e_hi = (int)((last ? S1 : T0 + L) - base);
    const int64_t t_lo = first ? T0 : base, t_hi = last ? S1 : T0 + L - C;
    const int64_t m_lo = (t_lo + S - 1) / S, m_hi = (t_hi + S - 1) / S;
    float* carry = (float*)ft.carry;
    const int ib = C + chunk * TT + lane * R;
    const int warp = threadIdx.x >> 5;
    // a trial's row behind its carry
    auto carry_in = [&](int u, float* row) {
        if (d + u < a.ndm && chunk == 0 && !first)
            for (int k = lane; k < C; k += 32) row[k] = carry[(int64_t)(wu * NT + u) * C + k];
    };
    auto scan = [&](int u, float* row, float* chain) {
        if (d + u < a.ndm)
            scan_trial_f32(row, chain, f.w0, f.nw, C, L, f.key + (int64_t)(d + u) * f.nw, (int64_t)(wu * NT + u) * C,
                           chunk, a.nch, lane, base, m_lo, m_hi, e_hi, first, last, carry, (float*)ft.seam_in,
                           (float*)ft.seam_out);
    };
    auto off = [&](int u) { return d + u < a.ndm ? (float)f.off[d + u] : 0.f; };
    if (!f.one_row) {
        float* rows = (float*)smem + NT * wu * f.rowlen;
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const float o = off(u);
#pragma unroll
            for (int r = 0; r < R; ++r) rows[u * f.rowlen + ib + r] = acc[u][r] - o;
            carry_in(u, rows + u * f.rowlen);
        }
        __syncthreads();  // the rows and their carries are complete
        // (the row kernels' layout, RowScan, is this one too)
        float* chain = (float*)smem + fused_rows_ints(NT * NW / a.nch, f.rowlen, C) + warp * kChainFloats;
        for (int u = 0; u < NT; ++u) scan(u, rows + u * f.rowlen, chain);
    } else {
        const RowScan lay(kRowsFir, NW, a.nch, f.rowlen, C, true);
        float* row = (float*)smem + wu * f.rowlen;
        float* chain = (float*)smem + lay.chain + warp * kChainFloats;
        float* wait = (float*)smem + lay.wait + warp * (NT - 1) * TT + lane * R;
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const float o = off(u);
#pragma unroll
            for (int r = 0; r < R; ++r) *(u == 0 ? row + ib + r : wait + (u - 1) * TT + r) = acc[u][r] - o;
        }
        for (int u = 0; u < NT; ++u) {
            if (u) {
                __syncthreads();  // the row is free
                for (int r = 0; r < R; ++r) row[ib + r] = wait[(u - 1) * TT + r];
            }
            carry_in(u, row);
            __syncthreads();
            scan(u, row, chain);
        }
    }
    // the next tile's bulk copies overwrite the rows
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
}

}  // namespace
}  // namespace fused
}  // namespace dd
