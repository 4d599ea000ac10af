// Device side of the row kernels: dedispersion (eq. p_dedisp, Sec. 2.1) from tap sums that
// the trials of a CTA share.
//
//   out[d][t] = sum_c B_{c,q(d,c)}[t_offset + t + delta_dc],   B_{c,q}[i] = sum_k w_qk I[c][i+k]
//
// Neighbouring trials of a list have the same tap run (count and weights) on almost every
// channel and differ in its start only: a 16-trial block of the CRAFT-like list has 1.1
// distinct runs per channel.  A CTA therefore forms each distinct run's sums B_{c,q} once
// per tile, in shared memory (a "row"), and a trial costs one add per channel and output
// whatever its tap count, where the tap kernels (dd_tile.cuh) cost one multiply-add per tap.
// The kinds of rows (RowKind) and their units:
//
// kRowsFir: fp32 sums.  A warp unit is three trials x 864 outputs, lane l owning 27 consecutive ones (odd:
// lane-strided loads hit 32 banks).  Where each trial uses the row of the one before, at most
// two samples later (98 % on that list), each sample is loaded once for all three.
//
// Bound by shared-memory loads, 0.35 of a word per trial, channel and output where a
// window is shared (else 1), plus the rows' own building (a quad of outputs loads n / 4 + 1
// quads and stores one), against 1 + (n - 1) / 27 loads and n multiply-adds of the tap kernel.
// Measured on 4096 CRAFT-like trials x 336 channels x 60261 outputs: tap kernel 17.62 ms, rows
// 7.67 ms (1.08e13 trial-channel-samples/s); a launch of 512 trials takes 1.08 ms, 0.88 with
// the building skipped and 0.44 with the summing skipped.  Two trials per warp took 1.19 ms,
// four trials of 15 outputs with one switch per trial 2.40, 8-warp CTAs with two-trial warps
// 1.91; scalar instead of packed adds 1.24 (two trials).
//
// kRowsPk: exact sums of uint8 samples with unit weights, for runs of at most 257 taps (255 n <=
// 65535).  A row word holds two outputs, B[i] + (B[i + 544] << 16): one load and one 32-bit addition
// serve both, whatever the start's parity (consecutive outputs in a word would need a second copy
// of the row for odd starts).  A unit is two trials x 1088 outputs, lane l owning 17 consecutive
// words.  Rows come from packed prefix sums PW[i] = P[i] + (P[i + 544] << 16) in global memory
// (k_prefix_packed): B = PW[i + n] - PW[i], exact modulo 2^32.
// Where it pays (the host counts shared-memory words), two adjacent channels are one item: their
// trials share the relative delay and both runs in a few patterns (2.2 per pair and 32-trial block
// on the CRAFT-like lists, 3.2 on the low-band list), a row per pattern holds both channels' sums,
// and a trial reads one word for the two.
// Items go four at a time: their words are added up to the point where a half could pass 65535 (the
// host says: all four, two and two, or each), and those sums into a 32-bit sum of whole words and
// one of the high halves; low = whole - (high << 16), exact modulo 2^32.
// Bound by shared-memory loads: a quarter to half a word per trial, channel and output, and the
// rows' building.  Measured (trial-channel-samples/s): 1500 trials x 336 channels x 21364 outputs:
// tap kernel 4.1e12, rows from the staged samples in the CTA 1.11e13 (1.20e13 with patterns), from
// prefix sums 1.76e13; 2048 low-band trials x 1024 x 65536: 32-bit difference rows 5.5e12, packed
// rows 1.21e13, with patterns 1.54e13.
//
// Pipeline: channels stream in stages, as many channels each as their rows fit in a half of
// the row area.  All warps sum stage i from one half, then build the rows of stage i + 1 in
// the other from the raw samples that one buffer holds (bulk copies, one lane per channel);
// one CTA barrier per stage publishes the new rows and ends the reads of the old ones, and
// the raw buffer is refilled with stage i + 2 while stage i + 1 is summed.
//
// A CTA has NW = 16 warps (one CTA per SM) or 8 (two per SM): the
// rows of a stage cost the same however many trials read them, and a longer stage spreads
// its barrier over more channels; 8 where 16 would leave SMs without a tile.
#pragma once

#include "dd_tile.cuh"

namespace dd {
namespace {

// Staged element type; IN8: uint8 input (weighted uint8 plans).
template <int KIND, bool IN8>
struct RowIn {
    using T = typename std::conditional<KIND == kRowsPk, uint32_t, typename std::conditional<IN8, uint8_t, float>::type>::type;
};

// Four consecutive samples from a 16-byte (fp32) or 4-byte (uint8) aligned address.
__device__ __forceinline__ float4 ld_quad(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ float4 ld_quad(const uint8_t* p) {
    // byte b -> 2^23 + b as fp32 bits, minus 2^23: exact
    const uint32_t v = *(const uint32_t*)p;
    auto f = [&](uint32_t sel) { return __uint_as_float(__byte_perm(v, 0x4B000000u, sel)) - 8388608.f; };
    return make_float4(f(0x7540), f(0x7541), f(0x7542), f(0x7543));
}

// Weighted sums, two quads of outputs per lane (i and i + 128): o_j = sum_k w[k] x[j + k],
// taps in order from k = 0, exactly n of them (samples outside a run are never multiplied,
// so an infinity or NaN reaches only the outputs whose run holds it).
__device__ __forceinline__ void fir_tap(float4& o, float w, float a, float b, float c, float d) {
    o.x = fmaf(w, a, o.x);
    o.y = fmaf(w, b, o.y);
    o.z = fmaf(w, c, o.z);
    o.w = fmaf(w, d, o.w);
}
template <typename TIN>
__device__ __forceinline__ void build_fir(const TIN* x, const float* w, int n, int i, int len, float* dst) {
    __builtin_assume(__isShared(x));
    __builtin_assume(__isShared(w));
    __builtin_assume(__isShared(dst));
    const int i2 = i + 128;
    const bool two = i2 < len;
    if (i >= len) return;
    const TIN* p = x + i;
    const TIN* q = x + (two ? i2 : i);
    float4 a = ld_quad(p), c = ld_quad(q);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f), u = o;
    int k = 0;
#pragma unroll 1
    for (; k + 4 <= n; k += 4) {
        const float4 b = ld_quad(p + k + 4), d = ld_quad(q + k + 4);
        const float4 g = *(const float4*)(w + k);
        fir_tap(o, g.x, a.x, a.y, a.z, a.w);
        fir_tap(u, g.x, c.x, c.y, c.z, c.w);
        fir_tap(o, g.y, a.y, a.z, a.w, b.x);
        fir_tap(u, g.y, c.y, c.z, c.w, d.x);
        fir_tap(o, g.z, a.z, a.w, b.x, b.y);
        fir_tap(u, g.z, c.z, c.w, d.x, d.y);
        fir_tap(o, g.w, a.w, b.x, b.y, b.z);
        fir_tap(u, g.w, c.w, d.x, d.y, d.z);
        a = b;
        c = d;
    }
    if (k < n) {
        const float4 g = *(const float4*)(w + k);
        fir_tap(o, g.x, a.x, a.y, a.z, a.w);
        fir_tap(u, g.x, c.x, c.y, c.z, c.w);
        if (k + 1 < n) {
            const float4 b = ld_quad(p + k + 4), d = ld_quad(q + k + 4);
            fir_tap(o, g.y, a.y, a.z, a.w, b.x);
            fir_tap(u, g.y, c.y, c.z, c.w, d.x);
            if (k + 2 < n) {
                fir_tap(o, g.z, a.z, a.w, b.x, b.y);
                fir_tap(u, g.z, c.z, c.w, d.x, d.y);
            }
        }
    }
    *(float4*)(dst + i) = o;
    if (two) *(float4*)(dst + i2) = u;
}

// A trial's kRFir sums: packed pairs of consecutive outputs and the last one.
struct FirAcc {
    uint64_t v[kRFir / 2];
    float t;
};

// a += the samples v[S .. S + kRFir - 1]: one add.rn.f32x2 per two outputs, two scalar adds
// where an odd shift splits the register pairs.  The adds name the CASE they belong to, so
// that the compiler keeps the cases apart: merged, they cost a register move per sample.
template <int S, int CASE, int N>
__device__ __forceinline__ void fir_add(FirAcc& a, const float (&v)[N]) {
#pragma unroll
    for (int j = 0; j < kRFir / 2; ++j) {
        if constexpr (S % 2 == 0)
            asm("// case %2\n\tadd.rn.f32x2 %0, %0, %1;"
                : "+l"(a.v[j]) : "l"(pk2(v[2 * j + S], v[2 * j + 1 + S])), "n"(CASE));
        else
            asm("{ // case %3\n\t.reg .f32 x, y;\n\tmov.b64 {x, y}, %0;\n\tadd.f32 x, x, %1;\n\t"
                "add.f32 y, y, %2;\n\tmov.b64 %0, {x, y};\n\t}"
                : "+l"(a.v[j]) : "f"(v[2 * j + S]), "f"(v[2 * j + 1 + S]), "n"(CASE));
    }
    asm("// case %2\n\tadd.f32 %0, %0, %1;" : "+f"(a.t) : "f"(v[kRFir - 1 + S]), "n"(CASE));
}

// The unit's trials start in one row, S1 and S2 samples after the first: each sample of the
// row is loaded once.
template <int S1, int S2>
__device__ __forceinline__ void fir_shared(const float* p, FirAcc (&a)[3]) {
    constexpr int N = kRFir + S2, CASE = 10 * S1 + S2;
    float v[N];
#pragma unroll
    for (int r = 0; r < N; ++r) v[r] = p[r];
    fir_add<0, CASE>(a[0], v);
    fir_add<S1, CASE>(a[1], v);
    fir_add<S2, CASE>(a[2], v);
}
// The same for two trials (S < 0: one).
template <int S, int CASE>
__device__ __forceinline__ void fir_shared2(const float* p, FirAcc& a0, FirAcc& a1) {
    constexpr int N = kRFir + (S > 0 ? S : 0);
    float v[N];
#pragma unroll
    for (int r = 0; r < N; ++r) v[r] = p[r];
    fir_add<0, CASE>(a0, v);
    if constexpr (S >= 0) fir_add<S, CASE>(a1, v);
}

// One channel of a fp32 unit: entry (positions of trials 0 and 1 as half words, of trial 2).
__device__ __forceinline__ void fir_channel(const float* rows, int2 e, int lane_off, FirAcc (&a)[3]) {
    const int e0 = e.x & 0xffff, s1 = (int)((uint32_t)e.x >> 16) - e0, s2 = e.y - e0 - s1;
    const float* p = rows + e0 + lane_off;
    __builtin_assume(__isShared(p));
    if ((unsigned)s1 <= 2u && (unsigned)s2 <= 2u) {
        switch (3 * s1 + s2) {
            case 0: fir_shared<0, 0>(p, a); break;
            case 1: fir_shared<0, 1>(p, a); break;
            case 2: fir_shared<0, 2>(p, a); break;
            case 3: fir_shared<1, 1>(p, a); break;
            case 4: fir_shared<1, 2>(p, a); break;
            case 5: fir_shared<1, 3>(p, a); break;
            case 6: fir_shared<2, 2>(p, a); break;
            case 7: fir_shared<2, 3>(p, a); break;
            default: fir_shared<2, 4>(p, a);
        }
        return;
    }
    // trials further apart, or of different rows
    const float* q = p + s1;
    const float* z = q + s2;
    __builtin_assume(__isShared(q));
    __builtin_assume(__isShared(z));
    switch (s1) {
        case 0: fir_shared2<0, 100>(p, a[0], a[1]); break;
        case 1: fir_shared2<1, 101>(p, a[0], a[1]); break;
        case 2: fir_shared2<2, 102>(p, a[0], a[1]); break;
        case 3: fir_shared2<3, 103>(p, a[0], a[1]); break;
        default:
            fir_shared2<-1, 104>(p, a[0], a[0]);
            fir_shared2<-1, 105>(q, a[1], a[1]);
    }
    fir_shared2<-1, 106>(z, a[2], a[2]);
}

// 256 packed words from packed prefix sums, eight per lane: of one run (x, n taps), or of two
// channels' runs at once (z, m taps; m = 0: one run).
__device__ __forceinline__ void build_rl(const uint32_t* x, int n, const uint32_t* z, int m, int i, int len,
                                         uint32_t* dst) {
    __builtin_assume(__isShared(x));
    __builtin_assume(__isShared(z));
    __builtin_assume(__isShared(dst));
    const uint32_t *y = x + n, *u = z + m;
    __builtin_assume(__isShared(y));
    __builtin_assume(__isShared(u));
    if (i - (i & 31) + 256 <= len) {
        if (m) {
#pragma unroll
            for (int k = 0; k < 256; k += 32) dst[i + k] = (y[i + k] - x[i + k]) + (u[i + k] - z[i + k]);
        } else {
#pragma unroll
            for (int k = 0; k < 256; k += 32) dst[i + k] = y[i + k] - x[i + k];
        }
    } else {
        for (int k = 0; k < 256 && i + k < len; k += 32)
            dst[i + k] = (y[i + k] - x[i + k]) + (m ? u[i + k] - z[i + k] : 0u);
    }
}

// A trial's packed integer sums: whole words, and their high halves.
struct PkAcc {
    uint32_t whole[kRPk], hi[kRPk];
};

// Four channels of one trial: pos holds its four row positions as half words.  MODE: how many
// of the four words may be added before a half could pass 65535.
template <int MODE>
__device__ __forceinline__ void pk_channels(const uint32_t* rows, uint2 pos, PkAcc& a) {
    const uint32_t* p0 = rows + (pos.x & 0xffffu);
    const uint32_t* p1 = rows + (pos.x >> 16);
    const uint32_t* p2 = rows + (pos.y & 0xffffu);
    const uint32_t* p3 = rows + (pos.y >> 16);
    __builtin_assume(__isShared(p0));
    __builtin_assume(__isShared(p1));
    __builtin_assume(__isShared(p2));
    __builtin_assume(__isShared(p3));
#pragma unroll
    for (int r = 0; r < kRPk; ++r) {
        const uint32_t v0 = p0[r], v1 = p1[r], v2 = p2[r], v3 = p3[r];
        if constexpr (MODE == 4) {
            const uint32_t s = v0 + v1 + v2 + v3;
            a.whole[r] += s;
            a.hi[r] += s >> 16;
        } else if constexpr (MODE == 2) {
            const uint32_t s = v0 + v1, t = v2 + v3;
            a.whole[r] += s + t;
            a.hi[r] += s >> 16;
            a.hi[r] += t >> 16;
        } else {
            a.whole[r] += v0 + v1;
            a.whole[r] += v2 + v3;
            a.hi[r] += v0 >> 16;
            a.hi[r] += v1 >> 16;
            a.hi[r] += v2 >> 16;
            a.hi[r] += v3 >> 16;
        }
    }
}

struct RowSmem {
    unsigned char* raw;
    int* lo;         // the block's per-channel minimum delays, then its stages' first channels
    uint32_t* half;  // two halves: row area, then the stage's header and entries
    uint64_t* full;
    int* issued;
};

// Issues the bulk copies of stage `s` into the raw buffer (warp 0, one lane per channel, the
// last lane the record).  tail: some window of the CTA runs past the end of its row; the
// missing part is zeroed.
template <typename TIN>
__device__ __forceinline__ void issue_rows(const DedispArgs& a, const RowSmem& sm, const RowGeom& rg, int rec_off,
                                           int blk, int s, int64_t base, bool tail, int lane) {
    constexpr int Q = Elem<TIN>::Q;
    if (s == a.skip_stage) return;  // test hook: this stage is never filled
    const int c0 = sm.lo[a.nchan + 1 + s], csn = sm.lo[a.nchan + 2 + s] - c0;
    const unsigned char* rec = a.rec + ((int64_t)blk * a.nst + s) * rg.rec_bytes;
    int nin = 0;
    int64_t a0 = 0;
    if (lane < csn) {
        a0 = (base + sm.lo[c0 + lane]) & ~(int64_t)(Q - 1);
        nin = a.lcap;
        if (tail) {
            nin = (int)max((int64_t)0, min((int64_t)a.lcap, a.ld - a0));
            uint4* z = (uint4*)(sm.raw + ((int64_t)lane * a.lcap + nin) * sizeof(TIN));
            for (int k = 0; k < (int)((a.lcap - nin) * sizeof(TIN) / 16); ++k) z[k] = make_uint4(0, 0, 0, 0);
            fence_proxy_async();
        }
        if (!dbg_ok(a0 >= 0 && a0 + nin <= a.ld && c0 >= 0 && csn <= a.cs, a.status)) nin = 0;
    }
    int bytes = nin * (int)sizeof(TIN);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
    if (tail) __syncwarp();  // the lanes' zeros are written before lane 0 arrives on the barrier for them all
    if (lane == 0) {
        mbar_expect_tx(sm.full, (uint32_t)(bytes + rg.rec_bytes));
        *sm.issued += 1;
    }
    __syncwarp();  // and the barrier expects the copies before any lane issues one
    if (nin > 0)
        bulk_g2s(sm.raw + (int64_t)lane * a.lcap * sizeof(TIN), (const TIN*)a.in + (int64_t)(c0 + lane) * a.ld + a0,
                 (uint32_t)(nin * sizeof(TIN)), sm.full);
    if (lane == 31) bulk_g2s(sm.raw + rec_off, rec, (uint32_t)rg.rec_bytes, sm.full);
}

// One CTA tile: trial block `blk`, time tile `tx`.  MULTI, FUSED as dedisp_tile; ONE_ROW: the
// fused scan of packed rows in its form for wide lists.
template <int KIND, bool IN8, int NW, bool MULTI, bool FUSED, bool ONE_ROW = false>
__device__ __forceinline__ bool row_tile(const DedispArgs a, unsigned char* smem, int blk, int tx, TileState& ts,
                                         const FusedArgs* fa = nullptr, const fused::FusedTile* ft = nullptr) {
    using TIN = typename RowIn<KIND, IN8>::T;
    constexpr bool FIR = KIND == kRowsFir;
    constexpr int Q = Elem<TIN>::Q;
    constexpr int NT = row_unit_trials(KIND), R = FIR ? kRFir : kRPk;
    constexpr int TW = row_warp_t(KIND);  // outputs per warp
    const int cs = a.cs;
    const int wpg = a.nch;  // warps along time
    const int nu = NW / wpg;
    const RowGeom rg(KIND, cs, nu, a.rows_max, a.kpad);
    const int rec_off = cs * a.lcap * (int)sizeof(TIN);
    const int half_words = rg.half_words(a.blen);
    RowSmem sm;
    sm.raw = smem;
    sm.lo = (int*)(smem + ((rec_off + rg.rec_bytes + 127) & ~127));
    sm.half = (uint32_t*)((unsigned char*)sm.lo + ((4 * a.lo_ld + 15) & ~15));
    sm.full = (uint64_t*)pipeline_area(smem, a.smem_bytes, 1);
    sm.issued = (int*)(sm.full + 1) + 1;
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int wu = warp / wpg, chunk = warp - wu * wpg;
    const int d = (blk * nu + wu) * NT;                   // the unit's first trial
    const int64_t t0 = (int64_t)tx * TW * wpg;             // CTA time start
    const int64_t tw = t0 + (int64_t)chunk * TW;           // warp time start
    const int64_t base = a.t_offset + t0;

    int past_end = 0;
    for (int c = tid; c < a.lo_ld; c += NW * 32) {
        const int lo = a.blk_lo[(int64_t)blk * a.lo_ld + c];
        sm.lo[c] = lo;
        if (c < a.nchan) past_end |= (((base + lo) & ~(int64_t)(Q - 1)) + a.lcap > a.ld) ? 1 : 0;
    }
    if constexpr (!FIR)  // the row of zeros that channels past a stage's last read
        for (int k = tid; k < row_zero_words(KIND, a.nch); k += NW * 32) sm.half[k] = sm.half[half_words + k] = 0u;
    const bool tail = __syncthreads_or(past_end) != 0;
    const int nst = sm.lo[a.nchan];  // stages of this block
    if (warp == 0) issue_rows<TIN>(a, sm, rg, rec_off, blk, 0, base, tail, lane);

    const int bq = (int)(base & (Q - 1));
    const int lane_off = chunk * TW + lane * R;
    bool ok = true;
    typename std::conditional<FIR, FirAcc, PkAcc>::type sum[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
        if constexpr (FIR) {
#pragma unroll
            for (int j = 0; j < R / 2; ++j) sum[u].v[j] = 0ull;
            sum[u].t = 0.f;
        } else {
#pragma unroll
            for (int j = 0; j < R; ++j) sum[u].whole[j] = sum[u].hi[j] = 0u;
        }
    }

    auto build = [&](int i) {  // the rows of stage i, from the raw buffer
        const unsigned char* rec = smem + rec_off;
        const TIN* raw = (const TIN*)smem;
        uint32_t* half = sm.half + (i & 1) * half_words;
        const int c0 = sm.lo[a.nchan + 1 + i];
        const int4 hdr = *(const int4*)rec;
        // the misalignment of channel ci of the stage in the raw buffer
        auto shift = [&](int ci) { return (bq + sm.lo[c0 + ci]) & (Q - 1); };
        // the entries; fp32 ones moved by that (packed rows begin at their trials' starts)
        int* ed = (int*)(half + a.blen);
        if (tid == 0) *(int4*)ed = hdr;
        if constexpr (FIR) {
            const int2* es = (const int2*)(rec + rg.ent_off);
            for (int e = tid; e < nu * cs; e += NW * 32) {
                const int v = e % cs;
                if (v >= hdr.w) continue;
                const int sh = shift(v);
                const int2 q = es[e];
                ((int2*)(ed + 4))[e] = make_int2(q.x + sh + (sh << 16), q.y + sh);
            }
        } else {
            const int4* es = (const int4*)(rec + rg.ent_off);
            for (int e = tid; e < nu * (cs / 4); e += NW * 32) ((int4*)(ed + 4))[e] = es[e];
        }
        // tasks of 256 outputs or words of a row, one warp each
        const uint4* desc = (const uint4*)(rec + rg.desc_off);
        const int per = (hdr.z + 255) >> 8, dr = NW / per, dp = NW - dr * per;
        int r = warp / per, part = warp - r * per;
        for (; r < hdr.x; r += dr, part += dp, r += part >= per, part -= part >= per ? per : 0) {
            const uint4 q = desc[r];
            const int src = (int)(q.x & 0xffff), len = (int)(q.y >> 16), dst = (int)(q.y & 0xffff);
            const int n = (int)(q.z & 0xffff), m = (int)(q.z >> 16);
            if (!dbg_ok(n >= 1 && dst + ((len + 3) & ~3) <= a.blen && src + len + n <= cs * a.lcap &&
                            (int)(q.x >> 16) + (m ? len + m : 0) <= cs * a.lcap,
                        a.status))
                continue;
            if constexpr (FIR)
                build_fir<TIN>(raw + src, (const float*)(rec + rg.w_off) + q.w, n, part * 256 + 4 * lane, len, (float*)half + dst);
            else
                build_rl(raw + src, n, raw + (q.x >> 16), m, part * 256 + lane, len, half + dst);
        }
    };
    auto parity_of = [&](int i) { return (uint32_t)(((MULTI ? ts.uses[0] : 0) + i) & 1); };
    bool got = mbar_wait_bounded(sm.full, parity_of(0), a.wait_ns);
    if (got) build(0);
    if (__syncthreads_or(!got)) {
        if (tid == 0) atomicExch(a.status, (int)DD_ERR_TIMEOUT);
        ok = false;
    } else if (warp == 0 && 1 < nst) {
        issue_rows<TIN>(a, sm, rg, rec_off, blk, 1, base, tail, lane);
    }
    for (int i = 0; ok && i < nst; ++i) {
        const uint32_t* half = sm.half + (i & 1) * half_words;
        if (d < a.ndm) {
            const int nv = ((const int4*)(half + a.blen))->w;  // items
            if constexpr (FIR) {
                const int2* ent = (const int2*)(half + a.blen + 4) + wu * cs;
                __builtin_assume(__isShared(ent));
                int2 next = ent[0];
#pragma unroll 1
                for (int ci = 0; ci < nv; ++ci) {
                    const int2 e = next;
                    next = ent[ci + 1];
                    if (!dbg_ok(max(max(e.x & 0xffff, (int)((uint32_t)e.x >> 16)), e.y) + lane_off + R + 4 <= a.blen,
                                a.status))
                        continue;
                    fir_channel((const float*)half, e, lane_off, sum);
                }
            } else {
                const uint4* ent = (const uint4*)(half + a.blen + 4) + wu * (cs / 4);
                __builtin_assume(__isShared(ent));
                const uint32_t* rows = half + lane_off;
                int modes = ((const int4*)(half + a.blen))->y;
#pragma unroll 1
                for (int ci = 0; ci < nv; ci += 4, modes >>= 2) {
                    const uint4 e = ent[ci / 4];
                    if (!dbg_ok((int)max(max(max(e.x & 0xffffu, e.x >> 16), max(e.y & 0xffffu, e.y >> 16)),
                                         max(max(e.z & 0xffffu, e.z >> 16), max(e.w & 0xffffu, e.w >> 16))) +
                                        lane_off + R <= a.blen,
                                a.status))
                        continue;
                    if ((modes & 3) == 0) {
                        pk_channels<4>(rows, make_uint2(e.x, e.y), sum[0]);
                        pk_channels<4>(rows, make_uint2(e.z, e.w), sum[1]);
                    } else if ((modes & 3) == 1) {
                        pk_channels<2>(rows, make_uint2(e.x, e.y), sum[0]);
                        pk_channels<2>(rows, make_uint2(e.z, e.w), sum[1]);
                    } else {
                        pk_channels<1>(rows, make_uint2(e.x, e.y), sum[0]);
                        pk_channels<1>(rows, make_uint2(e.z, e.w), sum[1]);
                    }
                }
            }
        }
        if (i + 1 < nst) {
            got = mbar_wait_bounded(sm.full, parity_of(i + 1), a.wait_ns);
            if (got) build(i + 1);
        }
        if (__syncthreads_or(!got)) {
            if (tid == 0) atomicExch(a.status, (int)DD_ERR_TIMEOUT);
            ok = false;
            break;
        }
        if (warp == 0 && i + 2 < nst) issue_rows<TIN>(a, sm, rg, rec_off, blk, i + 2, base, tail, lane);
    }

    __syncthreads();
    if (!ok && tid == 0) {  // no copy may still be in flight when the CTA leaves
        if (*sm.issued > 0 && !mbar_wait_bounded(sm.full, (uint32_t)((*sm.issued - 1) & 1), a.wait_ns))
            atomicExch(a.status, (int)DD_ERR_TIMEOUT);
    }
    if (!__syncthreads_and(ok)) return false;
    if (MULTI && tid == 0) ts.uses[0] += nst;

    if constexpr (FIR) {
        float f[NT][R];
#pragma unroll
        for (int u = 0; u < NT; ++u) {
#pragma unroll
            for (int j = 0; j < R / 2; ++j) unpk(sum[u].v[j], f[u][2 * j], f[u][2 * j + 1]);
            f[u][R - 1] = sum[u].t;
        }
        if constexpr (FUSED) {
            fused::epilogue_f32<NT, R, NW>(a, *fa, smem, wu, chunk, lane, d, t0, *ft, f);
            return true;
        }
        float* out = (float*)a.out;
#pragma unroll
        for (int u = 0; u < NT; ++u)
            store_row<float, R>(smem, f[u], warp, lane, tw, a.t_out,
                                d + u < a.ndm ? out + (int64_t)(d + u) * a.out_ld : nullptr, a.out_ld, a.status);
    } else {
        // low and high sums: outputs tw + lane * R + r and kPkHalf later
        int s[NT][2 * R];
#pragma unroll
        for (int u = 0; u < NT; ++u)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                s[u][r] = (int)(sum[u].whole[r] - (sum[u].hi[r] << 16));
                s[u][R + r] = (int)sum[u].hi[r];
            }
        if constexpr (FUSED) {
            fused::epilogue_pk<R, NW, ONE_ROW>(a, *fa, smem, wu, chunk, lane, d, t0, *ft, s);
            return true;
        }
        int* st = (int*)smem + warp * TW;
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            if (d + u >= a.ndm) break;
            int* out = (int*)a.out + (int64_t)(d + u) * a.out_ld;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                st[lane * R + r] = s[u][r];
                st[kPkHalf + lane * R + r] = s[u][R + r];
            }
            __syncwarp();
#pragma unroll 4
            for (int j = 0; j < TW / 32; ++j) {
                const int64_t t = tw + j * 32 + lane;
                if (t < a.t_out && dbg_ok(t >= 0 && t < a.out_ld, a.status)) out[t] = st[j * 32 + lane];
            }
            __syncwarp();
        }
    }
    if (MULTI) __syncthreads();  // the staging area is the next tile's stage buffers
    return true;
}

}  // namespace
}  // namespace dd
