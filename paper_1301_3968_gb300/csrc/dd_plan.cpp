// Host side of the C ABI: band geometry, the default profile tables (Sec. 3), the
// trial-DM rule (eq. trial DMs, Sec. 6.3), argument checking and the dedispersion
// schedule (trial blocks and staged window lengths).
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstdio>
#include <cstdarg>
#include <cmath>
#include <cstring>
#include <exception>
#include <fstream>
#include <map>
#include <mutex>
#include <new>
#include <sstream>
#include <string>
#include <system_error>
#include <thread>

#include "dd_internal.h"
#include "dd_trace.h"

namespace {

constexpr double kDefaultKdm = 4.15;

double kdm_of(const dd_band& b) { return b.k_dm > 0 ? b.k_dm : kDefaultKdm; }

bool band_ok(const dd_band* b) {
    return b && b->nchan > 0 && b->f_lo_mhz > 0 && b->df_mhz > 0 && b->dt_ms > 0 &&
           b->nsamp >= 0 && (b->in_type == DD_U8 || b->in_type == DD_F32) &&
           b->f_lo_mhz > 0;
}

// nu_c: highest frequency of channel c in GHz (Sec. 3).
double chan_top_ghz(const dd_band& b, int c) {
    int j = b.descending ? (b.nchan - 1 - c) : c;
    return (b.f_lo_mhz + (j + 1) * b.df_mhz) / 1000.0;
}

double band_top_ghz(const dd_band& b) { return (b.f_lo_mhz + b.nchan * b.df_mhz) / 1000.0; }

// Sec. 6.2: [(1/C) sum_c nu_c^-3]^-1 (channel order does not matter).
double inv_mean_inv_cube(const dd_band& b) {
    double s = 0.0;
    for (int c = 0; c < b.nchan; ++c) {
        double nu = (b.f_lo_mhz + (c + 1) * b.df_mhz) / 1000.0;
        s += 1.0 / (nu * nu * nu);
    }
    return 1.0 / (s / b.nchan);
}

void build_trials(const dd_band& b, double dm0, double eps, int n, double extra2, double* out) {
    out[0] = dm0;
    double acc = 0.0;
    for (int i = 1; i < n; ++i) {
        acc += std::sqrt(out[i - 1] * out[i - 1] + extra2);
        out[i] = dm0 + 2.0 * eps / b.nchan * acc;
    }
}

// Runs fn(b) for the blocks 0 .. n - 1 on a few threads when there is enough work
// (entries: table entries touched); on this thread alone where threads cannot be had.  What fn
// throws (no memory for its tables) is thrown here, once all have returned.
template <typename F>
void for_blocks(int n, size_t entries, F fn) {
    // (a thread costs about what 6 x 10^4 entries do)
    const int nt = (int)std::min<size_t>(std::min<size_t>(8, std::max(1u, std::thread::hardware_concurrency())),
                                         std::max<size_t>(1, entries >> 16));
    std::vector<std::thread> th;
    std::vector<std::exception_ptr> thrown((size_t)nt);
    auto share = [&fn, &thrown, n, nt](int k) {
        try {
            for (int b = k; b < n; b += nt) fn(b);
        } catch (...) {
            thrown[k] = std::current_exception();
        }
    };
    int started = 1;
    if (nt > 1) {
        th.reserve(nt);
        try {
            for (; started < nt; ++started) th.emplace_back(share, started);
        } catch (const std::exception&) {  // (no thread, or no memory for its state)
        }
    }
    share(0);
    for (int k = started; k < nt; ++k) share(k);
    for (auto& t : th) t.join();
    for (auto& e : thrown)
        if (e) std::rethrow_exception(e);
}

// The largest fn(b) over the blocks (at least 0).
template <typename F>
int64_t max_blocks(int n, size_t entries, F fn) {
    std::vector<int64_t> m((size_t)n, 0);
    for_blocks(n, entries, [&](int b) { m[b] = fn(b); });
    int64_t r = 0;
    for (int64_t v : m) r = std::max(r, v);
    return r;
}

// Span of the staged window when `db` consecutive trials share a CTA: the largest
// max(delta + n) - min(delta) over blocks and channels.
int64_t block_span(const dd_plan_s* p, int db, std::vector<int32_t>* lo_out) {
    const int C = p->nchan;
    const int nblk = (p->ndm + db - 1) / db;
    if (lo_out) lo_out->assign((size_t)nblk * C, 0);
    return max_blocks(nblk, (size_t)p->ndm * C, [&](int b) {
        int64_t span = 0;
        for (int c = 0; c < C; ++c) {
            int64_t lo = INT64_MAX, hi = 0;
            for (int i = 0; i < db; ++i) {
                const int d = b * db + i;
                if (d >= p->ndm) break;
                const int64_t dl = p->delay[(size_t)d * C + c];
                lo = std::min(lo, dl);
                hi = std::max(hi, dl + p->taps[(size_t)d * C + c]);
            }
            if (lo_out) (*lo_out)[(size_t)b * C + c] = (int32_t)lo;
            span = std::max(span, hi - lo);
        }
        return span;
    });
}

// Trials per warp unit: two adjacent trials share one register window on the fp32
// path; the exact integer path sums one trial per unit.
int trials_per_unit(const dd_plan_s* p) { return p->pair ? 2 : 1; }

// Warp units per warp: a run-length warp keeps kRlUnits trials' sums (it needs no
// register window, so more trials share each staged prefix row).
int units_per_warp(const dd_plan_s* p) { return p->rl ? dd::kRlUnits : 1; }

// Buffers in the staging ring of the plan's path.
int stages_of(const dd_plan_s* p) {
    return p->rl ? dd::kStagesRl : (p->pair ? dd::kStagesPair : dd::kStagesInt);
}

// Staged element size and elements per 16-byte chunk: uint8 samples, fp32 samples, or
// uint32 prefix sums on the run-length path.
int stage_esz(const dd_plan_s* p) { return p->rl ? 4 : (p->band.in_type == DD_U8 ? 1 : 4); }

// Elements a CTA stages per channel: its outputs, the block's delay spread plus taps
// (plus the run's end point P[delta + n] on the run-length path), 16 bytes of
// alignment slack and the element that the register pipeline reads ahead.
int64_t staged_len(const dd_plan_s* p, int nch, int64_t span) {
    const int64_t q = 16 / stage_esz(p);
    int64_t need = (int64_t)nch * dd::chunk_t(p->pair) + span + (p->rl ? 1 : 0) + q + 2;
    return (need + q - 1) / q * q;
}

// Weight pairs per record entry on the pair path: the most taps of any warp unit on
// any channel, max(n0, n1) (each trial's tap k reads sample k of its own run).
int32_t pair_taps(const dd_plan_s* p) {
    const int C = p->nchan, tpw = trials_per_unit(p);
    int64_t u = 0;
    for (int d0 = 0; d0 < p->ndm; d0 += tpw)
        for (int c = 0; c < C; ++c)
            for (int i = 0; i < tpw && d0 + i < p->ndm; ++i)
                u = std::max<int64_t>(u, p->taps[(size_t)(d0 + i) * C + c]);
    return (int32_t)std::min<int64_t>(u, INT32_MAX);
}

// Weight pairs of the fullest stage record on the pair path for stages of cs channels:
// each entry holds max(n0, n1) pairs.
int32_t pair_record_pairs(const dd_plan_s* p, int db, int cs) {
    const int C = p->nchan;
    const int nblk = (p->ndm + db - 1) / db;
    const int64_t most = max_blocks(nblk, (size_t)p->ndm * C, [&](int b) {
        int64_t top = 0;
        for (int c0 = 0; c0 < C; c0 += cs) {
            int64_t tot = 0;
            for (int d0 = b * db; d0 < std::min(p->ndm, (b + 1) * db); d0 += 2)
                for (int c = c0; c < std::min(C, c0 + cs); ++c) {
                    const size_t a = (size_t)d0 * C + c;
                    int64_t n = p->taps[a];
                    if (d0 + 1 < p->ndm) n = std::max<int64_t>(n, p->taps[a + C]);
                    tot += n;
                }
            top = std::max(top, tot);
        }
        return top;
    });
    return (int32_t)std::min<int64_t>((most + 1) & ~(int64_t)1, INT32_MAX);
}

// Samples past the block minimum that a pair unit's register window reaches: each
// trial reads max(n0, n1) samples from its own start, so the shorter run's trial reads
// past its own window by |n0 - n1| (with zero weights).  The staged window must hold
// them.
int64_t pair_read_span(const dd_plan_s* p, int db) {
    const int C = p->nchan;
    const int nblk = (p->ndm + db - 1) / db;
    return max_blocks(nblk, (size_t)p->ndm * C, [&](int b) {
        int64_t span = 0;
        for (int c = 0; c < C; ++c) {
            int64_t lo = INT64_MAX;
            for (int d = b * db; d < std::min(p->ndm, (b + 1) * db); ++d)
                lo = std::min<int64_t>(lo, p->delay[(size_t)d * C + c]);
            for (int d0 = b * db; d0 < std::min(p->ndm, (b + 1) * db); d0 += 2) {
                const size_t a = (size_t)d0 * C + c;
                int64_t st = p->delay[a], n = p->taps[a];
                if (d0 + 1 < p->ndm) {
                    const size_t bb = (size_t)(d0 + 1) * C + c;
                    st = std::max<int64_t>(st, p->delay[bb]);
                    n = std::max<int64_t>(n, p->taps[bb]);
                }
                span = std::max(span, st + n - lo);
            }
        }
        return span;
    });
}

// Most distinct tap counts among one trial block's trials on any channel (run-length
// path): the CTA builds one difference row per distinct count, so at most two fit.
int max_distinct_taps(const dd_plan_s* p, int db) {
    const int C = p->nchan;
    int most = 0;
    for (int d0 = 0; d0 < p->ndm; d0 += db)
        for (int c = 0; c < C; ++c) {
            int a = -1, b = -1, n = 0;
            for (int d = d0; d < std::min(p->ndm, d0 + db); ++d) {
                const int t = p->taps[(size_t)d * C + c];
                if (t == a || t == b) continue;
                if (a < 0) a = t;
                else if (b < 0) b = t;
                ++n;
                if (n > 2) return n;
            }
            most = std::max(most, n);
        }
    return most;
}

// Length of one difference row (run-length path with shared rows) for tap count n on
// channel c of block b: its words are read up to the largest run start of the block's
// trials with that count (relative to the block minimum), plus the CTA's outputs, plus
// three words of 16-byte alignment slack.
int32_t brow_row_len(const dd_plan_s* p, int db, int nch, const std::vector<int32_t>& blk_lo, int b,
                     int c, int n) {
    const int C = p->nchan;
    const int64_t lo = blk_lo[(size_t)b * C + c];
    int64_t x = 0;
    for (int d = b * db; d < std::min(p->ndm, (b + 1) * db); ++d)
        if (p->taps[(size_t)d * C + c] == n) x = std::max<int64_t>(x, p->delay[(size_t)d * C + c] - lo);
    return (int32_t)(x + (int64_t)nch * dd::chunk_t(false) + 4);
}

// The stride of the difference rows: the longest row of any block and channel.
int32_t brow_stride(const dd_plan_s* p, int db, int nch) {
    const int C = p->nchan;
    const int nblk = (p->ndm + db - 1) / db;
    std::vector<int32_t> lo;
    block_span(p, db, &lo);
    int32_t len = 0;
    for (int b = 0; b < nblk; ++b)
        for (int c = 0; c < C; ++c) {
            int n0 = 0, n1 = 0;
            for (int d = b * db; d < std::min(p->ndm, (b + 1) * db); ++d) {
                const int t = p->taps[(size_t)d * C + c];
                if (n0 == 0) n0 = t;
                else if (t != n0 && n1 == 0) n1 = t;
            }
            len = std::max(len, brow_row_len(p, db, nch, lo, b, c, n0));
            if (n1) len = std::max(len, brow_row_len(p, db, nch, lo, b, c, n1));
        }
    return (len + 3) & ~3;
}

// Lays the profile tables out as the kernel stages them: one record per (trial block,
// channel stage).  Entry (unit j, channel ci) = (window start - block minimum, taps);
// on the pair path it is (trial 0's start - block minimum, max(n0, n1), trial 1's start
// - trial 0's, 0) and the weights are (w0, w1) pairs, zero past a trial's own taps.
void build_records(dd_plan_s* p) {
    const int C = p->nchan;
    const int tpw = trials_per_unit(p);
    const int nu = dd::kWarps / p->nch * units_per_warp(p);
    const int db = tpw * nu;
    const int nst = (C + p->cs - 1) / p->cs;
    const int kw = p->pair ? p->kw : 0;
    const dd::StageGeom g(stage_esz(p), p->pair, p->lcap, kw, p->cs, nu, p->rl_b, p->blen);
    p->rec_bytes = g.rec_bytes;
    // without the weights where a device copy of them follows
    p->rec_host = p->w_follows ? g.w_off : g.rec_bytes;
    p->rec.assign((size_t)p->nblk * nst * p->rec_host, 0);
    for_blocks(p->nblk, (size_t)p->ndm * C, [&](int b) {
        for (int st = 0; st < nst; ++st) {
            unsigned char* r = p->rec.data() + ((size_t)b * nst + st) * p->rec_host;
            int32_t* ent = (int32_t*)r;
            float* w = (float*)(r + g.w_off);
            // difference rows: (n0, n1, len0, len1) per channel
            int32_t* nlist = (int32_t*)(r + g.w_off);
            int32_t woff = 0;  // pair path: weight pairs used so far in this record
            if (p->rl_b)
                for (int ci = 0; ci < p->cs; ++ci) {
                    const int c = st * p->cs + ci;
                    if (c >= C) continue;
                    int a = 0, bb = 0;
                    for (int d = b * db; d < std::min(p->ndm, (b + 1) * db); ++d) {
                        const int t = p->taps[(size_t)d * C + c];
                        if (a == 0) a = t;
                        else if (t != a && bb == 0) bb = t;
                    }
                    nlist[4 * ci] = a;
                    nlist[4 * ci + 1] = bb;
                    nlist[4 * ci + 2] = a ? brow_row_len(p, db, p->nch, p->blk_lo, b, c, a) : 0;
                    nlist[4 * ci + 3] = bb ? brow_row_len(p, db, p->nch, p->blk_lo, b, c, bb) : 0;
                }
            for (int j = 0; j < nu; ++j)
                for (int ci = 0; ci < p->cs; ++ci) {
                    const int c = st * p->cs + ci;
                    const int d0 = b * db + j * tpw;
                    if (d0 >= p->ndm || c >= C) continue;
                    if (p->pair) {
                        // (trial 0's start, max(n0, n1), trial 1's start - trial 0's, offset of
                        // the entry's weights) and per tap k the pair (w0[k], w1[k]), zero past
                        // a trial's own taps; entries' weights follow one another
                        const int e = j * p->cs + ci;
                        const int64_t blo = p->blk_lo[(size_t)b * C + c];
                        const size_t a0 = (size_t)d0 * C + c;
                        const bool two = d0 + 1 < p->ndm;
                        const size_t a1 = two ? a0 + C : a0;
                        const int n = std::max(p->taps[a0], two ? p->taps[a1] : 0);
                        ent[4 * e] = (int32_t)(p->delay[a0] - blo);
                        ent[4 * e + 1] = n;
                        ent[4 * e + 2] = two ? p->delay[a1] - p->delay[a0] : 0;
                        ent[4 * e + 3] = woff;
                        for (int i = 0; i < 2 && !p->w_follows; ++i) {
                            if (i == 1 && !two) break;
                            const size_t dc = i ? a1 : a0;
                            for (int k = 0; k < p->taps[dc]; ++k)
                                w[((size_t)woff + k) * 2 + i] = p->unit ? 1.0f : p->w[dc * p->kpad + k];
                        }
                        woff += n;
                        continue;
                    }
                    int64_t lo = INT64_MAX, hi = 0;
                    for (int i = 0; i < tpw && d0 + i < p->ndm; ++i) {
                        const size_t dc = (size_t)(d0 + i) * C + c;
                        lo = std::min<int64_t>(lo, p->delay[dc]);
                        hi = std::max<int64_t>(hi, (int64_t)p->delay[dc] + p->taps[dc]);
                    }
                    const int e = j * p->cs + ci;
                    ent[2 * e] = (int32_t)(lo - p->blk_lo[(size_t)b * C + c]);
                    ent[2 * e + 1] = (int32_t)(hi - lo);
                    if (p->rl_b) ent[2 * e + 1] = (hi - lo) == nlist[4 * ci] ? 0 : 1;
                }
        }
    });
}

// ----------------------------------------------------------------------- row schedule

// One distinct tap run of a (trial block, channel): its taps and weights are those of
// `trial`; its trials start beg .. end samples past the block's minimum delay.
struct Row {
    int32_t n, trial, beg, end;
};
// A pair of adjacent channels of a block whose trials share (run, run, relative delay): a row
// per pattern holds both channels' sums.  a, b: the runs' rows (indexes in the block's rows);
// beg, end, beg1: the starts on the first channel, and of the earliest trial on the second.
struct Pattern {
    int32_t a, b, rel, beg, end, beg1;
};

// The plan's row kind, if its sums can be formed that way: fp32 sums with weights that the
// host knows, integer sums of runs that fit a half word.
int row_kind_of(const dd_plan_s* p) {
    if (p->no_rows) return dd::kRowsNone;
    if (p->pair) return p->w_dev || p->kmax > 0xffff ? dd::kRowsNone : dd::kRowsFir;
    if (p->kmax > dd::kPkMaxTaps) return dd::kRowsNone;
    // (the prefix sums of a direct plan live in a scratch that holds its longest delay)
    return p->rl || (double)p->nchan * (p->dmax + 16.0 * 2 * dd::kPkHalf) * 4.0 <= 16e9 ? dd::kRowsPk : dd::kRowsNone;
}

// Rows pay up to this many distinct runs per (trial, channel).
constexpr double kRowsMaxShare = 0.5;

// fp32 rows pay where a window often serves the next trial as well: the same run count, at most two
// samples later.  Elsewhere a trial reads a word per channel and output, which costs what seven or
// eight packed multiply-adds of the tap kernel do, and a block's spread of starts makes long rows:
// 92 trials over DM 0-1945 (0.16 of the pairs near) x 336 channels x 4433 samples took 542 us, with
// taps 178.  Lists with fewer near pairs than kRowsMinNear take the taps, fine lists (kRowsFine) the
// rows whatever their size, so that a list and its parts take one kernel; between, the plan's block
// decides by the estimate below.
constexpr double kRowsMinNear = 0.3, kRowsFine = 0.9;

// Estimated time (us) of a fp32 launch over the plan's block with rows and with taps, fitted to 779
// launches of either kernel: 64, 336 and 1024 channels, 40-2000 trials with 0.2-0.9 of their pairs
// near and 1-35 taps, 800-60000 outputs (and 531 with uint8 input, whose conversion makes the rows'
// building a quarter dearer).  A CTA's time per channel, times the rounds of CTAs that an
// SM works through; two at once take 1.6 (rows) and 1.2 (taps) times one.  Median errors 6 and 13 %,
// the larger ones where rows are long.  Rows are taken where taps would cost kRowsMargin times as much,
// and kRowsMarginWords more for each tile's length that a channel's rows are longer than one.  Of 747
// fp32 launches with at least kRowsMinNear five are then more than 3 % slower than with taps, four of
// them fine lists (0.82 the worst; without the estimate 128, down to 0.19), and they are 1.35 times as
// fast as with taps in the mean; uint8 input one of 531 (0.90) and 1.41.
constexpr double kRowsMargin = 1.05, kRowsMarginWords = 0.1;
double sm_rounds(int64_t ctas, double pair) {  // two CTAs per SM
    const int64_t rest = ctas % 304;
    return (double)(ctas / 304) * pair + (rest > 152 ? pair : rest > 0 ? 1.0 : 0.0);
}
// Per (trial block, channel): loads, words that a trial's lane reads; words and work, the rows' words
// and multiply-adds in units of a tile.
double rows_us(int nchan, int nw, int64_t ctas, bool one_wave, double loads, double words, double work) {
    if (nw == dd::kRowWarps)
        return 18.5 + nchan * (double)((ctas + 151) / 152) * (0.0143 * nw * loads + 0.006 * work + 0.2453 * words + 0.1438);
    return 18.5 + nchan * (one_wave ? 1.0 : sm_rounds(ctas, 1.6)) * (0.008 * nw * loads + 0.0204 * work + 0.2432 * words + 0.1323);
}
// taps: mean of the longer run of a pair.
double taps_us(const dd_plan_s* p, int nch, double taps) {
    const int64_t t_out = std::max<int64_t>(1, p->band.nsamp - p->dmax);
    if (dd::takes_units(p, t_out, nch)) return 11.4 + p->nchan * (0.0157 * taps + 0.508);
    const int64_t tile = (int64_t)dd::chunk_t(true) * nch, db = 2 * (dd::kWarps / nch);
    const int64_t ctas = (t_out + tile - 1) / tile * ((p->ndm + db - 1) / db);
    return 43.1 + p->nchan * sm_rounds(ctas, 1.2) * (0.1034 * taps + 0.382);
}

// Warps per CTA of the row kernels.  16 (one CTA per SM) form a stage's rows for twice the
// trials of 8 (two CTAs per SM), which measured 12 % faster on a long launch (CRAFT-like,
// 512 trials: 1.08 against 1.22 ms), but leave more of a short launch's last wave idle: the
// share of the waves' slots that the plan's block fills decides, on 152 SMs.
int row_warps_of(const dd_plan_s* p, int kind, int nch, bool* one_wave) {
    const int64_t tile = dd::row_tile_t(kind, nch);
    const int64_t tiles = (std::max<int64_t>(1, p->band.nsamp - p->dmax) + tile - 1) / tile;
    auto ctas = [&](int nw) {
        const int db = dd::row_trials(kind, nw, nch);
        return tiles * ((p->ndm + db - 1) / db);
    };
    // one CTA per SM or fewer: its own time counts, and it may have the SM's shared memory
    *one_wave = ctas(dd::kWarps) <= 152;
    if (ctas(dd::kWarps) <= 304) return dd::kWarps;
    auto fill = [&](int nw, int64_t slots) {
        const int db = dd::row_trials(kind, nw, nch);
        const int64_t n = ctas(nw);
        return (double)p->ndm / db * tiles / (double)((n + slots - 1) / slots * slots);
    };
    return 1.12 * fill(dd::kRowWarps, 152) >= fill(dd::kWarps, 304) ? dd::kRowWarps : dd::kWarps;
}

// The schedule and records of the row kernels (layout: RowGeom) for nch time chunks and at
// most cs_fixed channels per stage (0: what gives the fewest stages).  Leaves the plan as it
// is and returns false where rows do not fit or pay.
bool build_rows(dd_plan_s* p, int nch, int cs_fixed) {
    const int kind = row_kind_of(p);
    if (kind == dd::kRowsNone) return false;
    const double units = (double)p->ndm * p->nchan;
    const int C = p->nchan;
    bool one_wave = false;
    const int nw = row_warps_of(p, kind, nch, &one_wave);
    const int db = dd::row_trials(kind, nw, nch), nt = dd::row_unit_trials(kind), nu = db / nt;
    const int nblk = (p->ndm + db - 1) / db;
    const int esz = kind == dd::kRowsFir && p->band.in_type == DD_U8 ? 1 : 4, Q = 16 / esz;  // samples or prefix sums
    const int span = dd::row_span(kind, nch);
    const bool fir = kind == dd::kRowsFir;
    auto same = [&](size_t a, size_t b) {
        if (p->taps[a] != p->taps[b]) return false;
        return p->unit || std::memcmp(&p->w[a * p->kpad], &p->w[b * p->kpad], (size_t)p->taps[a] * sizeof(float)) == 0;
    };
    bool fine = true;
    if (fir && p->ndm > 1) {  // (over the list's own neighbours: no matter how blocks fall)
        constexpr int kPart = 96;
        std::vector<int64_t> nr((size_t)(p->ndm + kPart - 1) / kPart, 0);
        for_blocks((int)nr.size(), (size_t)p->ndm * C, [&](int k) {
            int64_t n = 0;
            for (size_t i = (size_t)std::max(1, k * kPart) * C; i < (size_t)std::min(p->ndm, (k + 1) * kPart) * C; ++i)
                n += p->taps[i] == p->taps[i - C] && (uint32_t)(p->delay[i] - p->delay[i - C]) <= 2u;
            nr[k] = n;
        });
        int64_t near = 0;
        for (int64_t n : nr) near += n;
        if ((double)near < kRowsMinNear * (units - C)) return false;
        fine = (double)near >= kRowsFine * (units - C);
    }
    // the distinct runs of every (block, channel), and each trial's
    std::vector<std::vector<Row>> rows(nblk);
    std::vector<std::vector<int32_t>> first(nblk);  // [C + 1] into rows[b]
    std::vector<uint8_t> rid((size_t)p->ndm * C);   // in its channel's rows, or pair's patterns
    std::vector<int32_t> lo((size_t)nblk * C);
    // the block's channels as items, each one channel or a pair (patterns i0 .. i1 of pats[b])
    struct Item {
        int32_t c, nc, i0, i1;
    };
    std::vector<std::vector<Item>> items(nblk);
    std::vector<std::vector<Pattern>> pats(nblk);
    for_blocks(nblk, (size_t)p->ndm * C, [&](int b) {
        const int d0 = b * db, d1 = std::min(p->ndm, d0 + db);
        first[b].resize(C + 1);
        rows[b].reserve((size_t)C * 2);
        for (int c = 0; c < C; ++c) {
            const size_t f = rows[b].size();
            first[b][c] = (int32_t)f;
            int32_t l = INT32_MAX;
            for (int d = d0; d < d1; ++d) l = std::min(l, p->delay[(size_t)d * C + c]);
            lo[(size_t)b * C + c] = l;
            size_t hint = f;
            for (int d = d0; d < d1; ++d) {
                const size_t dc = (size_t)d * C + c;
                size_t r = hint;
                if (r >= rows[b].size() || !same(dc, (size_t)rows[b][r].trial * C + c))
                    for (r = f; r < rows[b].size(); ++r)
                        if (r != hint && same(dc, (size_t)rows[b][r].trial * C + c)) break;
                const int32_t at = p->delay[dc] - l;
                if (r == rows[b].size()) rows[b].push_back({p->taps[dc], d, at, at});
                rows[b][r].beg = std::min(rows[b][r].beg, at);
                rows[b][r].end = std::max(rows[b][r].end, at);
                rid[dc] = (uint8_t)(r - f);
                hint = r;
            }
        }
        first[b][C] = (int32_t)rows[b].size();
        // Integer sums: pairs of channels whose trials share their patterns.  In shared-memory
        // words per trial-block tile a run's row of L words costs 3 L to build (two loads and a
        // store) and a pattern's 5 L; a trial reads `span` words per channel, or per pair.
        std::vector<Pattern> ps;
        std::vector<uint8_t> id((size_t)(d1 - d0));
        for (int c = 0; c < C;) {
            bool pair = !fir && c + 1 < C;
            if (pair) {
                ps.clear();
                int n0 = 0, n1 = 0;
                double single = 2.0 * (d1 - d0) * span, both = (double)(d1 - d0) * span;
                for (int k = c; k < c + 2; ++k)
                    for (int r = first[b][k]; r < first[b][k + 1]; ++r) {
                        const double L = (double)rows[b][r].end - rows[b][r].beg + span;
                        single += 3.0 * L;
                        (k == c ? n0 : n1) = std::max(k == c ? n0 : n1, rows[b][r].n);
                    }
                pair = n0 + n1 <= dd::kPkMaxTaps;
                for (int d = d0; d < d1 && pair; ++d) {
                    const size_t dc = (size_t)d * C + c;
                    const int32_t ra = first[b][c] + rid[dc], rb1 = first[b][c + 1] + rid[dc + 1];
                    const int32_t at = p->delay[dc] - lo[(size_t)b * C + c], at1 = p->delay[dc + 1] - lo[(size_t)b * C + c + 1];
                    size_t i = 0;
                    while (i < ps.size() && !(ps[i].a == ra && ps[i].b == rb1 && ps[i].rel == at1 - at)) ++i;
                    if (i == ps.size()) ps.push_back({ra, rb1, at1 - at, at, at, at1});
                    if (at < ps[i].beg) {
                        ps[i].beg = at;
                        ps[i].beg1 = at1;
                    }
                    ps[i].end = std::max(ps[i].end, at);
                    id[d - d0] = (uint8_t)i;
                }
                for (const Pattern& q : ps) both += 5.0 * ((double)q.end - q.beg + span);
                pair = pair && both < single;
            }
            const int32_t i0 = (int32_t)pats[b].size();
            if (pair) {
                pats[b].insert(pats[b].end(), ps.begin(), ps.end());
                for (int d = d0; d < d1; ++d) rid[(size_t)d * C + c] = id[d - d0];
            }
            items[b].push_back({c, pair ? 2 : 1, i0, (int32_t)pats[b].size()});
            c += pair ? 2 : 1;
        }
    });
    // Words of a row: fp32, a run's whole staged window (its start is aligned to the raw buffer's
    // quads); packed, what its own trials read.  (In 64 bits: a block's trials may start up to 2^31
    // samples apart.)
    auto whole_len = [&](const Row& r) { return ((int64_t)Q - 1 + r.end + span + 3) & ~(int64_t)3; };
    auto own_len = [&](int32_t beg, int32_t end) { return ((int64_t)end - beg + span + 3) & ~(int64_t)3; };
    auto low_bits = [&](int b, int c) { return lo[(size_t)b * C + c] & (Q - 1); };
    size_t total = 0;
    int64_t need = 0;
    // Stages are cut at multiples of `grain` items.  Of the grain from item v of block b:
    // channels, rows, weights (each row's padded to four) and words of the row area, and the most
    // of each.
    const int grain = fir ? 1 : 4;
    struct Need {
        int64_t c = 0, r = 0, w = 0, a = 0;
        void add(const Need& o) {
            c += o.c;
            r += o.r;
            w += o.w;
            a += o.a;
        }
        void top(const Need& o) {
            c = std::max(c, o.c);
            r = std::max(r, o.r);
            w = std::max(w, o.w);
            a = std::max(a, o.a);
        }
    };
    std::vector<std::vector<Need>> grains(nblk);  // of the items v, v + grain, ...
    auto count_grain = [&](int b, size_t v) {
        Need k;
        for (size_t i = v; i < std::min(items[b].size(), v + grain); ++i) {
            const Item& it = items[b][i];
            k.c += it.nc;
            if (it.nc == 2) {
                for (int q = it.i0; q < it.i1; ++q) k.a += own_len(pats[b][q].beg, pats[b][q].end);
                k.r += it.i1 - it.i0;
                continue;
            }
            for (int r = first[b][it.c]; r < first[b][it.c + 1]; ++r) {
                const Row& row = rows[b][r];
                k.r += 1;
                if (fir) k.w += (row.n + 3) & ~3;
                k.a += fir ? whole_len(row) : own_len(row.beg, row.end);
            }
        }
        return k;
    };
    Need one;
    for (int b = 0; b < nblk; ++b) {
        total += rows[b].size();
        for (int c = 0; c < C; ++c)
            for (int i = first[b][c]; i < first[b][c + 1]; ++i) {
                // samples that building the row reads (dd_rows.cuh)
                const Row& r = rows[b][i];
                need = std::max(need, fir ? whole_len(r) + (r.n & ~3) + 4
                                          : (int64_t)low_bits(b, c) + r.end + ((span + 3) & ~3) + 3 + r.n);
            }
        for (size_t v = 0; v < items[b].size(); v += grain) {
            const Need k = count_grain(b, v);
            grains[b].push_back(k);
            one.top(k);
        }
    }
    if ((double)total > kRowsMaxShare * units) return false;
    if (fir && !fine) {
        double words = 0, work = 0, loads = 0, taps = 0;
        for (int b = 0; b < nblk; ++b)
            for (const Row& r : rows[b]) {
                words += (double)whole_len(r);
                work += (double)whole_len(r) * r.n;
            }
        auto step = [&](size_t i) {  // a trial's start after that of the one before, in the same row (else far)
            return p->taps[i] == p->taps[i - C] ? (uint32_t)(p->delay[i] - p->delay[i - C]) : UINT32_MAX;
        };
        const int R = dd::kRFir;  // (fir_channel: all three trials from one window, the first two, or none)
        constexpr int kPart = 96;  // trials, whole units and pairs of them
        const int parts = (p->ndm + kPart - 1) / kPart;
        std::vector<int64_t> ld((size_t)parts, 0), tp((size_t)parts, 0);
        for_blocks(parts, (size_t)p->ndm * C, [&](int k) {
            const int end = std::min(p->ndm, (k + 1) * kPart);
            for (int d = k * kPart; d < end; d += nt)
                for (int c = 0; c < C; ++c) {
                    const size_t i = (size_t)d * C + c;
                    const uint32_t s1 = d + 1 < end ? step(i + C) : UINT32_MAX;
                    ld[k] += s1 <= 2u && d + 2 < end && step(i + 2 * C) <= 2u ? R + 2 : s1 <= 3u ? 2 * R + 2 : 3 * R;
                }
            for (int d = k * kPart; d < end; d += 2)
                for (int c = 0; c < C; ++c) {
                    const size_t i = (size_t)d * C + c;
                    tp[k] += std::max(p->taps[i], d + 1 < end ? p->taps[i + C] : 0);
                }
        });
        for (int k = 0; k < parts; ++k) {
            loads += (double)ld[k];
            taps += (double)tp[k];
        }
        const double per = (double)nblk * C, tile = dd::row_warp_t(kind);
        const int64_t t = dd::row_tile_t(kind, nch), t_out = std::max<int64_t>(1, p->band.nsamp - p->dmax);
        if (esz == 1) work *= 1.25;
        const double ru = rows_us(C, nw, (t_out + t - 1) / t * nblk, one_wave,
                                  loads / ((double)((p->ndm + nt - 1) / nt) * C * 3 * R), words / per / tile, work / per / tile);
        const double tu = taps_us(p, nch, taps / ((double)((p->ndm + 1) / 2) * C));
        dd::log_msg(1, "plan %d trials x %d channels: estimated %.0f us with shared rows, %.0f tap by tap", p->ndm, C, ru, tu);
        if (tu < (kRowsMargin + kRowsMarginWords * (words / per / tile - 1)) * ru) return false;
    }
    const int64_t lcap = (need + Q - 1) / Q * Q;
    if (lcap > 0xffff || one.w > 0xffff) return false;
    const int64_t zero = dd::row_zero_words(kind, nch);  // the area begins with a row of zeros
    // Stages: items in order, as many as the limits allow.
    struct Cut {
        int cs = 0, nst = 0;  // nst: most stages of a block
        int64_t total = 0;
        Need most;
        std::vector<std::vector<int32_t>> start;  // per block: first items, and the end
    };
    auto cut = [&](int cs, const Need& lim, bool keep) {
        Cut k;
        k.cs = cs;
        if (keep) k.start.resize(nblk);
        for (int b = 0; b < nblk; ++b) {
            int n = 0;
            Need in;
            for (size_t v = 0; v < items[b].size(); v += grain) {
                const Need& m = grains[b][v / grain];
                if (v == 0 || in.c + m.c > lim.c || in.r + m.r > lim.r || in.w + m.w > lim.w || in.a + m.a > lim.a) {
                    if (keep) k.start[b].push_back((int32_t)v);
                    ++n;
                    in = Need();
                }
                in.add(m);
                k.most.top(in);
            }
            if (keep) k.start[b].push_back((int32_t)items[b].size());
            k.nst = std::max(k.nst, n);
            k.total += n;
        }
        return k;
    };
    // (a fixed stage size that does not fit beside a second CTA may take the SM's shared memory)
    size_t budget = nw == dd::kRowWarps || (one_wave && !p->shares_sm) ? dd::kSmemBudgetOne : dd::kSmemBudget;
    auto smem_of = [&](int cs, const Need& m, int stages) {
        const dd::RowGeom g(kind, cs, nu, (int)m.r, (int)m.w);
        return dd::row_smem_bytes(g, 0, esz, (int)lcap, cs, C + stages + 2, (int)(zero + m.a) + 16);
    };
    // limits for at most cs channels; false where a single grain does not fit
    auto limits = [&](int cs, Need* lim) {
        lim->c = cs;
        if (one.c > cs || cs * lcap > 0xffff) return false;
        lim->r = std::max<int64_t>(one.r, 2 * cs);
        lim->w = fir ? std::min<int64_t>(0xffff, std::max<int64_t>(one.w, (int64_t)cs * ((p->kmax + 3) & ~3) * 5 / 4)) : 0;
        lim->a = 0;
        const size_t rest = smem_of(cs, *lim, C);
        if (rest >= budget) return false;
        lim->a = (int64_t)((budget - rest) / 8) & ~(int64_t)3;
        return lim->a >= one.a;
    };
    Cut best;
    Need lim;
    const int cs_hi = std::min(dd::kRowCsMax, cs_fixed > 0 ? (std::max<int>(cs_fixed, (int)one.c) + grain - 1) / grain * grain : dd::kRowCsMax);
    const int cs_lo = cs_fixed > 0 ? cs_hi : grain;
    for (int pass = 0; pass < 2 && best.cs == 0; ++pass) {
        if (pass == 1 && (cs_fixed == 0 || budget == dd::kSmemBudgetOne)) break;
        if (pass == 1) budget = dd::kSmemBudgetOne;
        for (int cs = cs_hi; cs >= cs_lo; cs -= grain) {
            if (!limits(cs, &lim)) continue;
            Cut k = cut(cs, lim, false);
            if (best.cs == 0 || k.total < best.total) best = k;
        }
    }
    if (best.cs == 0) return false;
    const int cs = best.cs;
    limits(cs, &lim);
    best = cut(cs, lim, true);
    const Need& most = best.most;
    const int nst = best.nst, lo_ld = C + nst + 2;
    const int32_t area = (int32_t)(zero + most.a) + 16;  // and what the last row's reads run past it
    if (area > 0xffff) return false;  // positions are half words
    const dd::RowGeom g(kind, cs, nu, (int)most.r, (int)most.w);
    std::vector<unsigned char> rec((size_t)nblk * nst * g.rec_bytes, 0);
    std::vector<int32_t> table((size_t)nblk * lo_ld, 0);
    for_blocks(nblk, (size_t)p->ndm * C, [&](int b) {
        int32_t* tb = table.data() + (size_t)b * lo_ld;
        const int ns = (int)best.start[b].size() - 1;
        std::copy(lo.begin() + (size_t)b * C, lo.begin() + (size_t)(b + 1) * C, tb);
        tb[C] = ns;
        for (int st = 0; st <= ns; ++st)  // first channels
            tb[C + 1 + st] = st < ns ? items[b][best.start[b][st]].c : C;
        std::vector<int32_t> at_row, at_pat;
        for (int st = 0; st < ns; ++st) {
            unsigned char* q = rec.data() + ((size_t)b * nst + st) * g.rec_bytes;
            int32_t* hdr = (int32_t*)q;
            uint32_t* ent = (uint32_t*)(q + g.ent_off);
            uint32_t* desc = (uint32_t*)(q + g.desc_off);
            float* w = (float*)(q + g.w_off);
            const int v0 = best.start[b][st], v1 = best.start[b][st + 1];
            const int c0 = tb[C + 1 + st];
            const int nv = v1 - v0;
            hdr[3] = nv;
            int32_t dst = (int32_t)zero, woff = 0;
            at_row.assign((size_t)(first[b][tb[C + 2 + st]] - first[b][c0]), 0);
            const int r0 = first[b][c0], q0 = items[b][v0].i0;
            at_pat.assign((size_t)(items[b][v1 - 1].i1 - q0), 0);
            auto emit = [&](int32_t src0, int32_t src1, int32_t len, int32_t n0, int32_t n1, int32_t wo) {
                uint32_t* ds = desc + 4 * (size_t)hdr[0]++;
                ds[0] = (uint32_t)src0 | (uint32_t)src1 << 16;
                ds[1] = (uint32_t)dst | (uint32_t)len << 16;
                ds[2] = (uint32_t)n0 | (uint32_t)n1 << 16;
                ds[3] = (uint32_t)wo;
                hdr[2] = std::max(hdr[2], len);
            };
            for (int v = v0; v < v1; ++v) {
                const Item& it = items[b][v];
                const int32_t raw = (it.c - c0) * (int32_t)lcap;
                for (int i = it.i0; i < it.i1; ++i) {
                    const Pattern& t = pats[b][i];
                    at_pat[i - q0] = dst;
                    emit(raw + low_bits(b, it.c) + t.beg, raw + (int32_t)lcap + low_bits(b, it.c + 1) + t.beg1,
                         t.end - t.beg + span, rows[b][t.a].n, rows[b][t.b].n, 0);
                    dst += (int32_t)own_len(t.beg, t.end);
                }
                if (it.nc == 2) continue;
                for (int r = first[b][it.c]; r < first[b][it.c + 1]; ++r) {
                    const Row& row = rows[b][r];
                    at_row[r - r0] = dst;
                    if (fir) {
                        emit(raw, 0, Q - 1 + row.end + span, row.n, 0, woff);
                        dst += (int32_t)whole_len(row);
                        const size_t dc = (size_t)row.trial * C + it.c;
                        for (int k = 0; k < row.n; ++k) w[woff + k] = p->unit ? 1.0f : p->w[dc * p->kpad + k];
                        woff += (row.n + 3) & ~3;
                    } else {
                        emit(raw + low_bits(b, it.c) + row.beg, 0, row.end - row.beg + span, row.n, 0, 0);
                        dst += (int32_t)own_len(row.beg, row.end);
                    }
                }
            }
            // a trial's position in the row area (fp32: before its channel's misalignment in the raw
            // buffer); trials past the list's end add what the last one does
            auto pos = [&](int d, int v) -> uint32_t {
                if (v >= v1) return 0;  // the zeros
                const Item& it = items[b][v];
                const size_t dc = (size_t)std::min(d, p->ndm - 1) * C + it.c;
                const int32_t start = p->delay[dc] - lo[(size_t)b * C + it.c];
                if (it.nc == 2) return (uint32_t)(at_pat[it.i0 - q0 + rid[dc]] + start - pats[b][it.i0 + rid[dc]].beg);
                const int r = first[b][it.c] + rid[dc];
                return (uint32_t)(at_row[r - r0] + start - (fir ? 0 : rows[b][r].beg));
            };
            for (int j = 0; j < nu && b * db + j * nt < p->ndm; ++j) {
                const int d0 = b * db + j * nt;
                if (fir) {
                    for (int v = v0; v < v1; ++v) {
                        uint32_t* e = ent + 2 * (size_t)(j * cs + v - v0);
                        e[0] = pos(d0, v) | pos(d0 + 1, v) << 16;
                        e[1] = pos(d0 + 2, v);
                    }
                } else {
                    for (int v = v0; v < v1; v += 4) {
                        uint32_t* e = ent + (size_t)(j * cs + v - v0);
                        for (int u = 0; u < 2; ++u) {
                            e[2 * u] = pos(d0 + u, v) | pos(d0 + u, v + 1) << 16;
                            e[2 * u + 1] = pos(d0 + u, v + 2) | pos(d0 + u, v + 3) << 16;
                        }
                    }
                }
            }
            if (!fir)
                for (int v = v0; v < v1; v += 4) {
                    int32_t m[4] = {0, 0, 0, 0};  // most taps in a word of each item
                    for (int i = 0; i < 4 && v + i < v1; ++i)
                        for (int c = items[b][v + i].c; c < items[b][v + i].c + items[b][v + i].nc; ++c) {
                            int32_t n = 0;
                            for (int r = first[b][c]; r < first[b][c + 1]; ++r) n = std::max(n, rows[b][r].n);
                            m[i] += n;
                        }
                    const int mode = m[0] + m[1] + m[2] + m[3] <= dd::kPkMaxTaps ? 0
                                     : std::max(m[0] + m[1], m[2] + m[3]) <= dd::kPkMaxTaps ? 1 : 2;
                    hdr[1] |= mode << ((v - v0) / 2);
                }
        }
    });
    p->rk = kind;
    p->row_warps = nw;
    p->nch = nch;
    p->cs = cs;
    p->kw = (int32_t)most.w;
    p->rows_max = (int32_t)most.r;
    p->blen = area;
    p->lcap = (int32_t)lcap;
    p->nblk = nblk;
    p->nst = nst;
    p->lo_ld = lo_ld;
    p->rec_bytes = p->rec_host = g.rec_bytes;
    p->blk_lo.swap(table);
    p->rec.swap(rec);
    p->dev_dirty = true;
    size_t npairs = 0, npats = 0;
    for (int b = 0; b < nblk; ++b) {
        npairs += C - items[b].size();
        npats += pats[b].size();
    }
    dd::log_msg(1, "plan %d trials x %d channels: %s, shared rows (%.3f per trial and channel; %zu channel pairs with "
                "%zu patterns), %d trials and %d warps per CTA, up to %d channels per stage (%.1f stages per block), staged rows of %d elements, row area of "
                "%d words, record %d bytes, %zu bytes of shared memory", p->ndm, C,
                fir ? "fp32 sums" : p->rl ? "run-length sums" : "exact integer sums", (double)total / units, npairs, npats, db, nw, cs,
                (double)best.total / nblk, p->lcap, p->blen, p->rec_bytes, dd::dedisp_smem_for(p));
    return true;
}

// Numbers every built schedule, every upload and every copy of weights, so that a batch sees when a
// plan has changed or its tables have moved and a caller when its weights are gone.
std::atomic<uint64_t> g_gen{0};

// Chooses the CTA shape of the dedispersion kernel (warp units x time chunks), the
// staged window length and the channels per pipeline stage.  The most trials per CTA
// (the most reuse of each staged sample) whose window still fits is taken.  Where shared
// rows fit that shape and pay, the row kernels take the plan.
dd_status build_schedule(dd_plan_s* p) {
    p->sched_id = ++g_gen;
    p->rk = dd::kRowsNone;
    p->own_schedule = true;
    const bool u8 = p->band.in_type == DD_U8;
    p->pair = !(u8 && p->unit);
    const double mean_taps = (double)p->ns_total / ((double)p->ndm * p->nchan);
    p->rl = u8 && p->unit &&
            (p->method == DD_METHOD_RUNLENGTH ||
             (p->method == DD_METHOD_AUTO && mean_taps >= dd::kRlMinMeanTaps));
    const int esz = stage_esz(p);
    const int cs_want = dd::kCsMax;
    const int nbuf = stages_of(p);
    const int tpw = trials_per_unit(p);
    // first pass: shared memory for two CTAs per SM and at least two channels per
    // stage; second pass: one CTA per SM, any stage size
    const int budgets[2] = {dd::kSmemBudget, dd::kSmemBudgetOne};
    const int min_cs[2] = {2, 1};
    for (int pass = 0; pass < 2; ++pass) {
        for (int nch = 1; nch <= dd::kWarps; nch *= 2) {
            const int nu = dd::kWarps / nch * units_per_warp(p);
            const int db = tpw * nu;
            int64_t span = block_span(p, db, nullptr);
            if (p->pair) span = std::max(span, pair_read_span(p, db));
            p->umax = p->pair ? pair_taps(p) : 0;
            p->rl_b = p->rl && max_distinct_taps(p, db) <= 2;
            const int64_t need = staged_len(p, nch, span);
            if (need > (1 << 22)) continue;
            p->blen = p->rl_b ? brow_stride(p, db, nch) : 0;
            auto fits = [&](int cs, int32_t kw) {
                return dd::dedisp_smem_bytes(dd::StageGeom(esz, p->pair, (int)need, kw, cs, nu, p->rl_b, p->blen),
                                             nbuf, p->nchan) <= budgets[pass];
            };
            if (!fits(min_cs[pass], p->pair ? pair_record_pairs(p, db, min_cs[pass]) : 0)) continue;
            if (build_rows(p, nch, 0)) return DD_OK;
            int cs = cs_want;
            int32_t kw = p->pair ? pair_record_pairs(p, db, cs) : 0;
            while (cs > min_cs[pass] && !fits(cs, kw)) {
                --cs;
                if (p->pair) kw = pair_record_pairs(p, db, cs);
            }
            p->nch = nch;
            p->cs = cs;
            p->kw = kw;
            p->lcap = (int32_t)need;
            p->nblk = (p->ndm + db - 1) / db;
            block_span(p, db, &p->blk_lo);
            build_records(p);
            p->dev_dirty = true;
            dd::log_msg(1, "plan %d trials x %d channels: %s, %d trials per CTA, %d channels per stage, "
                        "staged rows of %d elements, difference rows of %d, record %d bytes, %zu bytes "
                        "of shared memory",
                     p->ndm, p->nchan,
                     p->rl ? (p->rl_b ? "run-length sums with shared difference rows" : "run-length sums")
                           : (p->pair ? "fp32 pair units" : "exact integer sums"),
                     db, p->cs, p->lcap, p->blen, p->rec_bytes, dd::dedisp_smem_for(p));
            return DD_OK;
        }
    }
    dd::log_msg(1, "plan %d trials x %d channels: no CTA shape fits in shared memory", p->ndm, p->nchan);
    return DD_ERR_UNSUPPORTED;
}

// Fixed CTA shape (nch time chunks) and stage size (cs channels), if it fits.  tuned: the
// autotuner's, which may be a row schedule that the tap kernels have no shared memory for.
dd_status build_schedule_fixed(dd_plan_s* p, int nch, int cs, bool tuned = false) {
    if (nch < 1 || nch > dd::kWarps || (dd::kWarps % nch) != 0 || cs < 1 || cs > 32) return DD_ERR_ARG;
    auto done = [&] {
        p->sched_id = ++g_gen;
        p->own_schedule = false;
        return DD_OK;
    };
    if (tuned && build_rows(p, nch, cs)) return done();
    const int esz = stage_esz(p);
    const int nu = dd::kWarps / nch * units_per_warp(p);
    const int db = trials_per_unit(p) * nu;
    int64_t span = block_span(p, db, nullptr);
    if (p->pair) span = std::max(span, pair_read_span(p, db));
    p->umax = p->pair ? pair_taps(p) : 0;
    const bool rl_b = p->rl && max_distinct_taps(p, db) <= 2;
    const int32_t kw = p->pair ? pair_record_pairs(p, db, cs) : 0;
    const int64_t need = staged_len(p, nch, span);
    if (need > (1 << 22)) return DD_ERR_UNSUPPORTED;
    const int32_t blen = rl_b ? brow_stride(p, db, nch) : 0;
    if (dd::dedisp_smem_bytes(dd::StageGeom(esz, p->pair, (int)need, kw, cs, nu, rl_b, blen), stages_of(p),
                              p->nchan) > dd::kSmemBudgetOne)
        return DD_ERR_UNSUPPORTED;
    p->rk = dd::kRowsNone;
    p->rl_b = rl_b;
    if (build_rows(p, nch, cs)) return done();
    p->blen = blen;
    p->nch = nch;
    p->cs = cs;
    p->kw = kw;
    p->lcap = (int32_t)need;
    p->nblk = (p->ndm + db - 1) / db;
    block_span(p, db, &p->blk_lo);
    build_records(p);
    p->dev_dirty = true;
    return done();
}

dd_status finish_profiles(dd_plan_s* p) {
    const size_t n = (size_t)p->ndm * p->nchan;
    int32_t kmax = 1, dmax = 0;
    int64_t ns = 0, row_max = 0;
    for (int d = 0; d < p->ndm; ++d) {
        int64_t row = 0;
        for (int c = 0; c < p->nchan; ++c) {
            size_t i = (size_t)d * p->nchan + c;
            kmax = std::max(kmax, p->taps[i]);
            int64_t e = (int64_t)p->delay[i] + p->taps[i] - 1;
            if (e > INT32_MAX) return DD_ERR_OVERFLOW;
            dmax = std::max<int32_t>(dmax, (int32_t)e);
            ns += p->taps[i];
            row += p->taps[i];
        }
        row_max = std::max(row_max, row);
    }
    (void)n;
    p->kmax = kmax;
    p->dmax = dmax;
    p->ns_total = ns;
    p->out_int = p->unit && p->band.in_type == DD_U8;
    p->max_abs_row = row_max * 255;
    if (p->out_int && p->max_abs_row > INT32_MAX) return DD_ERR_OVERFLOW;
    p->adj_stale = true;
    p->adj_w_stale = true;
    int64_t bws = 0;  // (fp32 input only: the weight gradient's staging)
    for (int d0 = 0; d0 < (p->band.in_type == DD_F32 ? p->ndm : 0); d0 += 8)
        for (int c = 0; c < p->nchan; ++c) {
            int32_t lo = INT32_MAX, hi = 0;
            for (int d = d0; d < std::min(p->ndm, d0 + 8); ++d) {
                lo = std::min(lo, p->delay[(size_t)d * p->nchan + c]);
                hi = std::max(hi, p->delay[(size_t)d * p->nchan + c]);
            }
            bws = std::max<int64_t>(bws, (int64_t)hi - lo);
        }
    p->bw_span = (int32_t)std::min<int64_t>(bws, INT32_MAX);
    return build_schedule(p);
}

}  // namespace

namespace dd {

// The input gradient gI[c][tau] = sum_{d,k} w_dck g[d][tau - delta_dc - k] is a
// dedispersion with the roles swapped: output rows are channels, input rows are the
// trials' output gradients zero-padded by P = d_max on both sides, delays
// P - delta_dc - n_dc + 1 and the taps' weights reversed.  This builds that plan's
// tables on the host (its weights are filled on the device from the forward plan's).
dd_status build_adjoint_plan(dd_plan_s* p) {
    const int D = p->ndm, C = p->nchan;
    const int32_t P = p->dmax;
    if (p->adj) {
        destroy_plan(p->adj);
        p->adj = nullptr;
    }
    dd_plan_s* t = new (std::nothrow) dd_plan_s;
    if (!t) return DD_ERR_OOM;
    t->band = p->band;
    t->band.nchan = D;
    t->band.in_type = DD_F32;
    t->band.descending = 0;
    t->band.nsamp = 0;
    t->nchan = D;
    t->ndm = C;
    t->dms.assign(C, 0.0);
    t->delay.resize((size_t)C * D);
    t->taps.resize((size_t)C * D);
    for (int d = 0; d < D; ++d)
        for (int c = 0; c < C; ++c) {
            const size_t dc = (size_t)d * C + c, cd = (size_t)c * D + d;
            t->delay[cd] = P - p->delay[dc] - p->taps[dc] + 1;
            t->taps[cd] = p->taps[dc];
        }
    t->unit = false;
    t->w_dev = t->w_follows = true;  // filled on the device
    t->kpad = p->kpad;
    t->kuser = p->kuser;
    dd_status st = finish_profiles(t);
    if (st != DD_OK) {
        delete t;
        return st;
    }
    p->adj = t;
    p->adj_stale = false;
    p->adj_w_stale = true;
    return DD_OK;
}

int log_level() {
    static const int level = [] {
        const char* v = std::getenv("DD_LOG");
        return v ? std::atoi(v) : 0;
    }();
    return level;
}

void log_msg(int level, const char* fmt, ...) {
    if (log_level() < level) return;
    char line[512];
    va_list ap;
    va_start(ap, fmt);
    std::vsnprintf(line, sizeof line, fmt, ap);
    va_end(ap);
    std::fprintf(stderr, "[dd] %s\n", line);
}

dd_status cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return DD_OK;
    return e == cudaErrorMemoryAllocation ? DD_ERR_OOM : DD_ERR_CUDA;
}

// Frees the device tables, for new ones on device `to` (-1: none).
static void free_dev(dd_plan_s* p, int to) {
    if (p->dev.device < 0) return;
    int cur = -1;
    cudaGetDevice(&cur);
    if (cur != p->dev.device) cudaSetDevice(p->dev.device);
    for (uint32_t* q : p->prefix_old) cudaFree(q);  // (what was captured reads tables that go now)
    p->prefix_old.clear();
    if (to != p->dev.device) {
        cudaFree(p->d_prefix);
        p->d_prefix = nullptr;
        p->prefix_elems = 0;
    }
    if (p->prefix_done) cudaEventDestroy(p->prefix_done);
    p->prefix_done = nullptr;
    p->prefix_stream = 0;
    cudaFree(p->dev.slab);
    cudaFree(p->dev.mu);
    cudaFree(p->dev.isd);
    cudaFree(p->dev.widths);
    cudaFree(p->dev.narrow);
    if (cur >= 0 && cur != p->dev.device) cudaSetDevice(cur);
    p->dev = DevTables{};
    p->widths_on_dev.clear();
}

dd_plan_s* twin_of(dd_plan_s* p, Twin kind) {
    dd_plan_s* t = new (std::nothrow) dd_plan_s;
    if (!t) return nullptr;
    t->band = p->band;
    t->nchan = p->nchan;
    t->ndm = p->ndm;
    t->dms = p->dms;
    t->delay = p->delay;
    t->taps = p->taps;
    t->w = p->w;
    t->kpad = p->kpad;
    t->kuser = p->kuser;
    t->unit = p->unit;
    t->kmax = p->kmax;
    t->dmax = p->dmax;
    t->ns_total = p->ns_total;
    t->out_int = p->out_int;
    t->max_abs_row = p->max_abs_row;
    t->method = p->method;
    t->w_dev = p->w_dev;
    t->owner = p;
    t->shares_sm = kind == Twin::kSharesSm;
    t->no_rows = kind == Twin::kTaps;
    t->debug_fused_parts = p->debug_fused_parts;
    // (integer sums are the same from the tap kernels, which such a schedule may be; fp32 ones are not)
    if (build_schedule(t) == DD_OK && (!t->pair || t->rk == p->rk)) {
        // (the caller's shape, where the tap kernels have it)
        if (t->no_rows && !p->own_schedule) build_schedule_fixed(t, p->nch, p->cs);
        return t;
    }
    delete t;
    return nullptr;
}

dd_plan_s* tap_twin(dd_plan_s* p) {
    if (p->rl || p->rk != kRowsPk) return nullptr;
    std::lock_guard<std::mutex> lock(p->prefix_mu);
    if (p->tap && p->tap_id != p->sched_id) {
        destroy_plan(p->tap);
        p->tap = nullptr;
    }
    if (!p->tap) {
        log_msg(1, "plan %d trials x %d channels: no room for prefix sums, tap by tap", p->ndm, p->nchan);
        p->tap = twin_of(p, Twin::kTaps);
        p->tap_id = p->sched_id;
    }
    return p->tap;
}

void destroy_plan(dd_plan_s* p) {
    if (p->adj) destroy_plan(p->adj);
    if (p->tap) destroy_plan(p->tap);
    if (p->d_gpad) cudaFree(p->d_gpad);
    if (p->d_gsplit) cudaFree(p->d_gsplit);
    if (p->d_fkey) cudaFree(p->d_fkey);
    if (p->d_fcarry) cudaFree(p->d_fcarry);
    if (p->d_fseam) cudaFree(p->d_fseam);
    if (p->d_fstarts) cudaFree(p->d_fstarts);
    free_dev(p, -1);
    delete p;
}

dd_status upload_tables(dd_plan_s* p) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_status(e);
    if (!p->dev_dirty && p->dev.device == dev) return DD_OK;
    if (p->rec_host != p->rec_bytes && !p->w_follows) build_records(p);  // with the host's weights
    free_dev(p, dev);
    p->dev.device = dev;
    // one allocation for all tables
    const size_t n = (size_t)p->ndm * p->nchan;
    const size_t nrec = p->rec_host ? p->rec.size() / p->rec_host : 0;
    const size_t wlen = p->unit ? 0 : n * (size_t)p->kpad;
    size_t total = 0;
    auto room = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t at_delay = room(n * 4), at_taps = room(n * 4), at_lo = room(p->blk_lo.size() * 4),
                 at_rec = room(nrec * p->rec_bytes), at_w = room(wlen * sizeof(float)), at_status = room(4),
                 at_off = room((size_t)p->ndm * sizeof(double));
    e = cudaMalloc((void**)&p->dev.slab, total);
    if (e != cudaSuccess) return cuda_status(e);
    unsigned char* slab = p->dev.slab;
    p->dev.delay = (int32_t*)(slab + at_delay);
    p->dev.taps = (int32_t*)(slab + at_taps);
    p->dev.blk_lo = (int32_t*)(slab + at_lo);
    p->dev.rec = slab + at_rec;
    p->dev.w = p->unit ? nullptr : (float*)(slab + at_w);
    p->dev.status = (int32_t*)(slab + at_status);
    p->dev.off = (double*)(slab + at_off);
    const int32_t zero = 0;
    // small tables as one copy (a copy takes some 16 us whatever its size)
    std::vector<unsigned char> all(total <= ((size_t)1 << 20) && p->rec_host == p->rec_bytes ? total : 0);
    auto up = [&](void* dst, const void* src, size_t bytes) {
        if (e != cudaSuccess || !bytes) return;
        if (!all.empty()) std::memcpy(all.data() + ((unsigned char*)dst - slab), src, bytes);
        else e = cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice);
    };
    up(p->dev.delay, p->delay.data(), n * 4);
    up(p->dev.taps, p->taps.data(), n * 4);
    up(p->dev.blk_lo, p->blk_lo.data(), p->blk_lo.size() * 4);
    up(p->dev.status, &zero, 4);
    if (!p->w_follows) up(p->dev.w, p->w.data(), wlen * sizeof(float));
    if (p->rec_host == p->rec_bytes)
        up(p->dev.rec, p->rec.data(), p->rec.size());
    else if (e == cudaSuccess)
        e = cudaMemcpy2D(p->dev.rec, p->rec_bytes, p->rec.data(), p->rec_host, p->rec_host, nrec, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !all.empty()) e = cudaMemcpy(slab, all.data(), total, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_status(e);
    dd_status st;
    // place dd_boxcar_snr_noalloc's scratch array and kernels on this device now, so
    // that its calls allocate nothing (lazy module loading would do it at its first call)
    if ((st = noalloc_preload()) != DD_OK) return st;
    p->dev_dirty = false;
    p->dev_gen = p->w_id = ++g_gen;
    p->w_captured = false;  // (earlier captures read tables that are gone)
    return DD_OK;
}

}  // namespace dd

extern "C" {

const char* dd_status_str(dd_status s) {
    switch (s) {
        case DD_OK: return "ok";
        case DD_ERR_ARG: return "invalid argument";
        case DD_ERR_OVERFLOW: return "integer overflow";
        case DD_ERR_OOM: return "out of memory";
        case DD_ERR_CUDA: return "CUDA error";
        case DD_ERR_STATE: return "invalid state";
        case DD_ERR_TIMEOUT: return "device wait timed out";
        case DD_ERR_CAPACITY: return "capacity exceeded";
        case DD_ERR_UNSUPPORTED: return "unsupported";
    }
    return "unknown status";
}

int32_t dd_version(void) { return 100; }

dd_status dd_trial_dms(const dd_band* band, double dm0, double dm_max, int32_t n,
                       double tau_av_ms, int32_t smear_terms, double* dms_out,
                       double* eps_out) {
    if (!band_ok(band) || !dms_out || n < 2 || !(dm_max > dm0) || dm0 < 0 ||
        tau_av_ms < 0 || (smear_terms != 1 && smear_terms != 2))
        return DD_ERR_ARG;
    const dd_band& b = *band;
    const double k = kdm_of(b);
    const double dnu = b.df_mhz / 1000.0;
    const double geo = inv_mean_inv_cube(b);
    const double dm_diag = b.dt_ms / (2.0 * k * dnu) * geo;   // Sec. 6.2, kappa = 1/k
    const double dm_tau = tau_av_ms / (2.0 * k * dnu) * geo;  // eq. DM_tau
    const double extra2 = dm_diag * dm_diag + (smear_terms == 2 ? dm_tau * dm_tau : 0.0);
    std::vector<double> tmp(n);
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < 200; ++it) {
        build_trials(b, dm0, hi, n, extra2, tmp.data());
        if (tmp[n - 1] >= dm_max) break;
        hi *= 2.0;
    }
    for (int it = 0; it < 200; ++it) {
        double mid = 0.5 * (lo + hi);
        build_trials(b, dm0, mid, n, extra2, tmp.data());
        if (tmp[n - 1] < dm_max) lo = mid; else hi = mid;
    }
    const double eps = 0.5 * (lo + hi);
    build_trials(b, dm0, eps, n, extra2, dms_out);
    if (eps_out) *eps_out = eps;
    return DD_OK;
}

// The tables and schedule of a new plan.
static dd_status fill_plan(dd_plan_s* p, const dd_band* band, const double* dms, int32_t ndm) {
    p->band = *band;
    p->nchan = band->nchan;
    p->ndm = ndm;
    p->dms.assign(dms, dms + ndm);
    const size_t n = (size_t)ndm * band->nchan;
    p->delay.resize(n);
    p->taps.resize(n);
    const double k = kdm_of(*band);
    const double top = band_top_ghz(*band);
    const double dnu = band->df_mhz / 1000.0;
    // the channels' factors of DM, then the tables
    std::vector<double> fd(band->nchan), fn(band->nchan);
    for (int c = 0; c < band->nchan; ++c) {
        const double nu = chan_top_ghz(*band, c);
        const double lo = nu - dnu;
        fd[c] = 1.0 / (nu * nu) - 1.0 / (top * top);
        fn[c] = 1.0 / (lo * lo) - 1.0 / (nu * nu);
    }
    const int nblk = (ndm + 15) / 16;
    const int64_t far = max_blocks(nblk, n, [&](int b) -> int64_t {
        for (int d = 16 * b; d < std::min(ndm, 16 * b + 16); ++d) {
            const double kdm = k * dms[d];
            for (int c = 0; c < band->nchan; ++c) {
                const double raw_d = kdm * fd[c] / band->dt_ms;
                const double raw_n = kdm * fn[c] / band->dt_ms;
                if (!(raw_d < 2.0e9) || !(raw_n < 2.0e9)) return 1;
                p->delay[(size_t)d * band->nchan + c] = (int32_t)std::floor(raw_d);
                p->taps[(size_t)d * band->nchan + c] = std::max(1, (int32_t)std::ceil(raw_n));
            }
        }
        return 0;
    });
    return far ? DD_ERR_OVERFLOW : finish_profiles(p);
}

dd_status dd_plan_create(dd_plan_t* out, const dd_band* band, const double* dms, int32_t ndm) {
    if (!out || !band_ok(band) || !dms || ndm < 1) return DD_ERR_ARG;
    *out = nullptr;
    for (int d = 0; d < ndm; ++d)
        if (!(dms[d] >= 0.0) || !std::isfinite(dms[d])) return DD_ERR_ARG;
    dd_plan_s* p = new (std::nothrow) dd_plan_s;
    if (!p) return DD_ERR_OOM;
    dd_status st = DD_ERR_OOM;
    try {
        st = fill_plan(p, band, dms, ndm);
    } catch (const std::bad_alloc&) {
    }
    if (st == DD_OK) *out = p;
    else delete p;
    return st;
}

dd_status dd_set_profiles(dd_plan_t p, const int32_t* delay, const int32_t* ntaps,
                          const float* w, int32_t kmax) {
    if (!p) return DD_ERR_ARG;
    const size_t n = (size_t)p->ndm * p->nchan;
    if (w && kmax < 1) return DD_ERR_ARG;
    if (delay)
        for (size_t i = 0; i < n; ++i)
            if (delay[i] < 0) return DD_ERR_ARG;
    if (ntaps)
        for (size_t i = 0; i < n; ++i)
            if (ntaps[i] < 1) return DD_ERR_ARG;
    // keep the old state so that a rejected profile leaves the plan usable
    std::vector<int32_t> old_d = p->delay, old_t = p->taps;
    std::vector<float> old_w = p->w;
    int32_t old_kpad = p->kpad, old_kuser = p->kuser;
    bool old_unit = p->unit, old_w_dev = p->w_dev;
    if (delay) std::memcpy(p->delay.data(), delay, n * sizeof(int32_t));
    if (ntaps) std::memcpy(p->taps.data(), ntaps, n * sizeof(int32_t));
    if (w) {
        for (size_t i = 0; i < n; ++i)
            if (p->taps[i] > kmax) {
                p->delay = old_d;
                p->taps = old_t;
                return DD_ERR_ARG;
            }
        p->kpad = (kmax + 3) / 4 * 4;
        p->kuser = kmax;
        p->w.assign(n * (size_t)p->kpad, 0.0f);
        for (size_t i = 0; i < n; ++i)
            for (int k = 0; k < p->taps[i]; ++k) p->w[i * p->kpad + k] = w[i * (size_t)kmax + k];
        p->unit = false;
    } else {
        p->w.clear();
        p->kpad = 0;
        p->kuser = 0;
        p->unit = true;
    }
    p->w_dev = false;
    dd_status st = finish_profiles(p);
    if (st != DD_OK) {
        p->w_dev = old_w_dev;
        p->delay = old_d;
        p->taps = old_t;
        p->w = old_w;
        p->kpad = old_kpad;
        p->kuser = old_kuser;
        p->unit = old_unit;
        finish_profiles(p);
        return st;
    }
    p->dev_dirty = true;
    return DD_OK;
}

dd_status dd_set_weights_device(dd_plan_t p, const float* d_w, int32_t kmax, void* stream) {
    if (!p || !d_w || kmax < 1) return DD_ERR_ARG;
    if (p->kmax > kmax) return DD_ERR_ARG;
    const int32_t kpad = (kmax + 3) / 4 * 4;
    p->w_follows = true;  // tables built or uploaded here need no weights of the host's
    dd_status st = DD_OK;
    if (p->unit || p->kpad != kpad || p->kuser != kmax) {
        // switch the plan to weighted with this row length; host weights start at zero
        const size_t n = (size_t)p->ndm * p->nchan;
        p->w.assign(n * (size_t)kpad, 0.0f);
        p->kpad = kpad;
        p->kuser = kmax;
        p->unit = false;
        p->w_dev = true;
        st = finish_profiles(p);
    } else if (p->rk == dd::kRowsFir) {
        // the rows shared weights that the host knew: back to a record of every trial's own
        // (in the shape that a caller set, where there is one)
        p->w_dev = true;
        if (p->own_schedule || build_schedule_fixed(p, p->nch, p->cs) != DD_OK) st = build_schedule(p);
    }
    p->w_dev = true;
    if (st == DD_OK) st = dd::upload_tables(p);
    p->w_follows = false;
    if (st != DD_OK) return st;
    cudaError_t e = cudaMemcpy2DAsync(p->dev.w, (size_t)kpad * sizeof(float), d_w,
                                      (size_t)kmax * sizeof(float), (size_t)kmax * sizeof(float),
                                      (size_t)p->ndm * p->nchan, cudaMemcpyDeviceToDevice,
                                      (cudaStream_t)stream);
    if (e != cudaSuccess) return dd::cuda_status(e);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing((cudaStream_t)stream, &cap);
    if (e != cudaSuccess) return dd::cuda_status(e);
    if (cap != cudaStreamCaptureStatusNone) p->w_captured = true;
    p->w_id = ++g_gen;
    p->adj_w_stale = true;
    return dd::launch_repack(p, (cudaStream_t)stream);
}

uint64_t dd_plan_weights_id(dd_plan_t p) {
    int dev = -1;
    if (!p || p->dev_dirty || p->w_captured || cudaGetDevice(&dev) != cudaSuccess || p->dev.device != dev) return 0;
    return p->w_id;
}

dd_status dd_plan_info(dd_plan_t p, int64_t* t_out, int32_t* d_max, int32_t* kmax,
                       int64_t* ns_total, int32_t* out_is_int) {
    if (!p) return DD_ERR_ARG;
    if (t_out) *t_out = std::max<int64_t>(0, p->band.nsamp - p->dmax);
    if (d_max) *d_max = p->dmax;
    if (kmax) *kmax = p->kmax;
    if (ns_total) *ns_total = p->ns_total;
    if (out_is_int) *out_is_int = p->out_int ? 1 : 0;
    return DD_OK;
}

dd_status dd_get_tables(dd_plan_t p, int32_t* delay, int32_t* ntaps) {
    if (!p) return DD_ERR_ARG;
    const size_t n = (size_t)p->ndm * p->nchan;
    if (delay) std::memcpy(delay, p->delay.data(), n * sizeof(int32_t));
    if (ntaps) std::memcpy(ntaps, p->taps.data(), n * sizeof(int32_t));
    return DD_OK;
}

static bool aligned16(const void* ptr) { return ((uintptr_t)ptr & 15u) == 0; }

dd_status dd_dedisperse(dd_plan_t p, const void* in, int64_t in_ld, int64_t t_offset,
                        int64_t nsamp, void* out, int64_t out_ld, void* stream) {
    DD_TRACE("dd_dedisperse");
    dd::log_msg(2, "dd_dedisperse: %d trials, t_offset %lld, nsamp %lld", p ? p->ndm : 0, (long long)t_offset, (long long)nsamp);
    if (!p || !in || !out) return DD_ERR_ARG;
    const int64_t esz = p->band.in_type == DD_U8 ? 1 : 4;
    if (nsamp <= 0) nsamp = p->band.nsamp;
    if (t_offset < 0 || nsamp <= p->dmax || t_offset + nsamp > in_ld) return DD_ERR_ARG;
    if (!aligned16(in) || (in_ld * esz) % 16 != 0) return DD_ERR_ARG;
    const int64_t t_out = nsamp - p->dmax;
    if (out_ld < t_out) return DD_ERR_ARG;
    if (t_out > INT32_MAX - dd::chunk_t(false) * dd::kWarps || in_ld > (int64_t)1 << 40) return DD_ERR_OVERFLOW;
    if (p->rl && nsamp > ((int64_t)1 << 24)) return DD_ERR_UNSUPPORTED;
    dd_status st = dd::upload_tables(p);
    if (st != DD_OK) return st;
    if (p->rl) return dd::launch_dedisperse_rl(p, in, in_ld, t_offset, nsamp, out, out_ld, (cudaStream_t)stream);
    if (p->rk == dd::kRowsPk) {
        st = dd::launch_dedisperse_pk(p, in, in_ld, t_offset, nsamp, out, out_ld, (cudaStream_t)stream);
        dd_plan_s* t = st == DD_ERR_OOM ? dd::tap_twin(p) : nullptr;
        return t ? dd_dedisperse(t, in, in_ld, t_offset, nsamp, out, out_ld, stream) : st;
    }
    return dd::launch_dedisperse(p, in, in_ld, t_offset, t_out, out, out_ld, (cudaStream_t)stream);
}

dd_status dd_channel_stats(dd_plan_t p, const void* in, int64_t in_ld, int64_t t_offset,
                           int64_t nsamp, double* mean, double* sd, void* stream) {
    DD_TRACE("dd_channel_stats");
    if (!p || !in || !mean || !sd) return DD_ERR_ARG;
    if (nsamp <= 0) nsamp = p->band.nsamp;
    if (t_offset < 0 || nsamp < 1 || t_offset + nsamp > in_ld) return DD_ERR_ARG;
    dd_status st = dd::upload_tables(p);
    if (st != DD_OK) return st;
    return dd::launch_channel_stats(p, in, in_ld, t_offset, nsamp, mean, sd, (cudaStream_t)stream);
}

dd_status dd_boxcar_snr(dd_plan_t p, const void* x, int64_t ld, int64_t t_len,
                        const int32_t* widths, int32_t nw, const double* mean,
                        const double* sd, float* peak, int32_t* arg, float thresh,
                        dd_candidate* cands, int32_t cap, int32_t* ncands, void* stream) {
    DD_TRACE("dd_boxcar_snr");
    dd::log_msg(2, "dd_boxcar_snr: %d trials, %lld samples, %d widths", p ? p->ndm : 0, (long long)t_len, nw);
    if (!p || !x || !widths || nw < 1 || !mean || !sd || !peak || !arg) return DD_ERR_ARG;
    if (t_len < 1 || ld < t_len || t_len > INT32_MAX) return DD_ERR_ARG;
    if (cands && (!ncands || cap < 0)) return DD_ERR_ARG;
    for (int i = 0; i < nw; ++i) {
        if (widths[i] < 1 || widths[i] > t_len) return DD_ERR_ARG;
        if (i && widths[i] <= widths[i - 1]) return DD_ERR_ARG;
    }
    dd_status st = dd::upload_tables(p);
    if (st != DD_OK) return st;
    return dd::launch_boxcar(p, x, ld, t_len, widths, nw, mean, sd, peak, arg, thresh, cands,
                             cap, ncands, (cudaStream_t)stream);
}

dd_status dd_backward(dd_plan_t p, const float* in, int64_t in_ld, int64_t t_offset,
                      int64_t nsamp, const float* g, int64_t gld, float* gw, float* gin,
                      int64_t gin_ld, void* stream) {
    DD_TRACE("dd_backward");
    dd::log_msg(2, "dd_backward: %d trials, nsamp %lld, weight gradient %s, input gradient %s", p ? p->ndm : 0,
             (long long)nsamp, gw ? "yes" : "no", gin ? "yes" : "no");
    if (!p || !in || !g) return DD_ERR_ARG;
    if (p->band.in_type != DD_F32) return DD_ERR_UNSUPPORTED;
    if (nsamp <= 0) nsamp = p->band.nsamp;
    if (t_offset < 0 || nsamp <= p->dmax || t_offset + nsamp > in_ld) return DD_ERR_ARG;
    const int64_t t_out = nsamp - p->dmax;
    if (gld < t_out) return DD_ERR_ARG;
    if (gin && (gin_ld < t_offset + nsamp || (gin_ld * 4) % 16 != 0 || !aligned16(gin)))
        return DD_ERR_ARG;
    if (!aligned16(in) || (in_ld * 4) % 16 != 0) return DD_ERR_ARG;
    dd_status st = dd::upload_tables(p);
    if (st != DD_OK) return st;
    return dd::launch_backward(p, in, in_ld, t_offset, t_out, g, gld, gw, gin, gin_ld,
                               (cudaStream_t)stream);
}

static dd_status set_schedule(dd_plan_s* p, int nch, int cs, bool tuned) {
    const int old_nch = p->nch, old_cs = p->cs;
    dd_status st = build_schedule_fixed(p, nch, cs, tuned);
    if (st != DD_OK && (p->nch != old_nch || p->cs != old_cs)) build_schedule_fixed(p, old_nch, old_cs, true);
    return st;
}

dd_status dd_plan_set_schedule(dd_plan_t p, int32_t nch, int32_t cs) {
    if (!p) return DD_ERR_ARG;
    return set_schedule(p, nch, cs, false);
}

dd_status dd_plan_get_schedule(dd_plan_t p, int32_t* nch, int32_t* cs, int32_t* trials_per_cta) {
    if (!p) return DD_ERR_ARG;
    if (nch) *nch = p->nch;
    if (cs) *cs = p->cs;
    if (trials_per_cta) *trials_per_cta = dd::plan_trials(p);
    return DD_OK;
}

dd_status dd_plan_set_method(dd_plan_t p, int32_t method) {
    if (!p || method < DD_METHOD_AUTO || method > DD_METHOD_RUNLENGTH) return DD_ERR_ARG;
    if (method == DD_METHOD_RUNLENGTH && !(p->unit && p->band.in_type == DD_U8)) return DD_ERR_UNSUPPORTED;
    const int32_t old = p->method;
    p->method = method;
    dd_status st = build_schedule(p);
    if (st != DD_OK) {
        p->method = old;
        build_schedule(p);
    }
    return st;
}

dd_status dd_plan_get_method(dd_plan_t p, int32_t* method) {
    if (!p || !method) return DD_ERR_ARG;
    *method = p->rl ? DD_METHOD_RUNLENGTH : DD_METHOD_DIRECT;
    return DD_OK;
}

namespace {

std::mutex g_tune_mu;

// Schedule cache key: channel count, input type, path, and the trial-block delay
// spread and widest tap run in powers of two -- the quantities that decide which CTA
// shape and stage size fit and run best.
std::string tune_key(const dd_plan_s* p) {
    const int64_t span8 = block_span(p, 8, nullptr);
    const int sb = (int)std::floor(std::log2((double)span8 + 1.0));
    const int kb = (int)std::floor(std::log2((double)p->kmax + 1.0));
    std::ostringstream o;
    o << "C" << p->nchan << "_" << (p->band.in_type == DD_U8 ? "u8" : "f32") << "_"
      << (p->rk ? "rows" : "") << (p->pair ? "pair" : (p->rl ? "rl" : "int")) << "_s" << sb << "_k" << kb;
    return o.str();
}

std::map<std::string, std::pair<int, int>> read_cache(const char* path) {
    std::map<std::string, std::pair<int, int>> m;
    if (!path) return m;
    std::ifstream f(path);
    std::string key;
    int nch, cs;
    double ms;
    while (f >> key >> nch >> cs >> ms) m[key] = {nch, cs};
    return m;
}

}  // namespace

dd_status dd_plan_autotune(dd_plan_t p, const void* d_in, int64_t in_ld, void* d_out,
                           int64_t out_ld, const char* cache_path, float* best_ms, void* stream) {
    DD_TRACE("dd_plan_autotune");
    if (!p || !d_in || !d_out) return DD_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const std::string key = tune_key(p);
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto cache = read_cache(cache_path);
    auto hit = cache.find(key);
    if (hit != cache.end() && p->rk && hit->second.second == 0) {  // the plan's own schedule
        if (!p->own_schedule) {
            const dd_status st = build_schedule(p);
            if (st != DD_OK) return st;
        }
        if (best_ms) *best_ms = -1.0f;
        dd::log_msg(1, "autotune %s: cached: the plan's own schedule", key.c_str());
        return DD_OK;
    }
    if (hit != cache.end() && set_schedule(p, hit->second.first, hit->second.second, true) == DD_OK) {
        if (best_ms) *best_ms = -1.0f;
        dd::log_msg(1, "autotune %s: cached schedule (%d time chunks, %d channels per stage)", key.c_str(),
                 hit->second.first, hit->second.second);
        return DD_OK;
    }
    const int orig_nch = p->nch, orig_cs = p->cs, orig_rk = p->rk;
    const bool orig_own = p->own_schedule;
    std::vector<std::pair<int, int>> cand;  // (time chunks, channels per stage)
    if (orig_rk) cand.push_back({orig_nch, orig_cs});
    for (int nch = 1; nch <= 2; nch *= 2)
        for (int cs : orig_rk ? std::vector<int>{8, 16, 28}
                              : stage_esz(p) == 1 ? std::vector<int>{4, 8, 12, 16} : std::vector<int>{2, 3, 4, 6, 8})
            cand.push_back({nch, cs});
    int best_nch = orig_nch, best_cs = orig_cs;
    bool own = orig_own;  // the best is the plan's own schedule
    float best = 1e30f;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t ce = cudaEventCreate(&e0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e1);
    if (ce != cudaSuccess) return dd::cuda_status(ce);
    dd_status st = DD_OK;
    for (size_t i = 0; i < cand.size() && st == DD_OK; ++i) {
        // a row plan's first candidate is its schedule as it stands
        if (!(orig_rk && i == 0) && build_schedule_fixed(p, cand[i].first, cand[i].second, true) != DD_OK) continue;
        if (p->rk != orig_rk) continue;  // the same sums in every candidate
        st = dd_dedisperse(p, d_in, in_ld, 0, p->band.nsamp, d_out, out_ld, stream);
        if (st != DD_OK) break;
        float t = 1e30f;
        for (int rep = 0; rep < 2; ++rep) {
            cudaEventRecord(e0, s);
            st = dd_dedisperse(p, d_in, in_ld, 0, p->band.nsamp, d_out, out_ld, stream);
            cudaEventRecord(e1, s);
            if (st != DD_OK) break;
            ce = cudaEventSynchronize(e1);
            if (ce != cudaSuccess) {
                st = dd::cuda_status(ce);
                break;
            }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            t = std::min(t, ms);
        }
        if (st != DD_OK) break;
        // A row plan's own schedule fits its patterns and rows; another, which similar plans would
        // get too, has to be clearly faster (any lead: 36 small beams 13.6 ms, their own 12.4)
        if (t < (orig_rk && i > 0 ? 0.97f : 1.0f) * best) {
            best = t;
            own = orig_own && orig_rk && i == 0;
            best_nch = cand[i].first;
            best_cs = cand[i].second;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (own) build_schedule(p);
    else if (build_schedule_fixed(p, best_nch, best_cs, true) != DD_OK) build_schedule_fixed(p, orig_nch, orig_cs, true);
    if (st != DD_OK) return st;
    if (best_ms) *best_ms = best;
    dd::log_msg(1, "autotune %s: %d time chunks, %d channels per stage, %.3f ms (default %d, %d)", key.c_str(),
             best_nch, best_cs, best, orig_nch, orig_cs);
    if (cache_path) {
        std::ofstream f(cache_path, std::ios::app);
        if (f) f << key << " " << best_nch << " " << (own ? 0 : best_cs) << " " << best << "\n";
    }
    return DD_OK;
}

dd_status dd_get_device_status(dd_plan_t p, int32_t* code, void* stream) {
    if (!p || !code) return DD_ERR_ARG;
    *code = 0;
    if (p->dev.device < 0 || !p->dev.status) return DD_OK;
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    int32_t v = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&v, p->dev.status, sizeof(v), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && v != 0) e = cudaMemset(p->dev.status, 0, sizeof(int32_t));
    if (e != cudaSuccess) return dd::cuda_status(e);
    *code = v;
    return DD_OK;
}

dd_status dd_test_set_wait(dd_plan_t p, int32_t skip_stage, int64_t wait_ns) {
    if (!p || wait_ns < 0) return DD_ERR_ARG;
    p->debug_skip_stage = skip_stage;  // (a twin reads its owner's)
    p->wait_ns = wait_ns > 0 ? wait_ns : dd::kWaitNs;
    return DD_OK;
}

dd_status dd_test_set_scratch_limit(dd_plan_t p, int64_t bytes) {
    if (!p || bytes < 0) return DD_ERR_ARG;
    p->scratch_limit = bytes;
    return DD_OK;
}

dd_status dd_plan_destroy(dd_plan_t p) {
    if (!p) return DD_ERR_ARG;
    dd::destroy_plan(p);
    return DD_OK;
}

}  // extern "C"
