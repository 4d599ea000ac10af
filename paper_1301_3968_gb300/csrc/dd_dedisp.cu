// Profiled dedispersion, eq. p_dedisp (Sec. 2.1): the plain and batched kernels, the
// prefix pass of the run-length path and their launchers.  The tile itself (work
// decomposition, staging, sums) is in dd_tile.cuh.
#include "dd_tile.cuh"

namespace dd {
namespace {


// Order of the tiles.  Run-length path: trial blocks along x, time tiles along y, so that
// the CTAs resident together share time tiles and each tile's prefix rows come from L2
// for all trial blocks (instead of every trial block reading the whole prefix array from
// DRAM).  Other paths: the grid is (time tiles, trial blocks) and runs in groups of
// kGroupBlocks trial blocks, blocks fastest within a group and then time tiles, so that
// each group reads the input about once from DRAM (and its blocks' stage records from
// L2) instead of each trial block re-reading the input.
constexpr int kGroupBlocks = 16;
template <typename TIN, bool PAIR, int NBUF, int SHORT>
__global__ void __launch_bounds__(kWarps * 32, 2) k_dedisp(DedispArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TileState ts;
    if (threadIdx.x == 0) init_pipeline<NBUF>(pipeline_area(smem, a.smem_bytes, NBUF), ts);
    __syncthreads();
    if constexpr (std::is_same<TIN, uint32_t>::value) {
        dedisp_tile<TIN, PAIR, NBUF, false, SHORT>(a, smem, blockIdx.x, blockIdx.y, ts);
    } else {
        const int ntile = (int)gridDim.x, nblk = (int)gridDim.y;
        const int L = (int)blockIdx.y * ntile + (int)blockIdx.x;  // < 2^31: grid.y <= 65535
        const int g = L / (kGroupBlocks * ntile), r = L - g * kGroupBlocks * ntile;
        const int gb = min(kGroupBlocks, nblk - g * kGroupBlocks);
        dedisp_tile<TIN, PAIR, NBUF, false, SHORT>(a, smem, g * kGroupBlocks + r % gb, r / gb, ts);
    }
}

// Small launches (see run_unit): grid (time tiles of 8 x 32 kRSmall outputs, trial blocks, pair
// units of a block).
template <typename TIN, int NBUF>
__global__ void __launch_bounds__(kWarps * 32, 2) k_dedisp_unit(DedispArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TileState ts;
    if (threadIdx.x == 0) init_pipeline<NBUF>(pipeline_area(smem, a.smem_bytes, NBUF), ts);
    __syncthreads();
    dedisp_tile<TIN, true, NBUF, false, 0, false, true>(a, smem, blockIdx.y, blockIdx.x, ts);
}

// Batched form: one CTA per work item (beam, trial block, time tile) of the list, in list
// order (beams by decreasing cost, each in the plain grid's tile order); the hardware
// starts CTAs in index order as earlier ones finish, which balances uneven beams.
// Measured on 36 beams: a persistent form whose CTAs took items from an atomic counter
// was 3.6 % slower (and slower than separate launches).
template <typename TIN, bool PAIR, int NBUF, int SHORT>
__global__ void __launch_bounds__(kWarps * 32, 2) k_dedisp_batched(const DedispArgs* beams,
                                                                    const BatchItem* items,
                                                                    uint32_t smem_bytes) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TileState ts;
    __shared__ DedispArgs sa;
    if (threadIdx.x == 0) init_pipeline<NBUF>(pipeline_area(smem, smem_bytes, NBUF), ts);
    const BatchItem it = items[blockIdx.x];
    if (threadIdx.x == 0) {
        sa = beams[it.beam];
        sa.smem_bytes = smem_bytes;
    }
    __syncthreads();
    dedisp_tile<TIN, PAIR, NBUF, false, SHORT>(sa, smem, it.blk, it.tx, ts);
}

template <typename TIN, bool PAIR, int NBUF, int SHORT = 0>
dd_status run(DedispArgs a, cudaStream_t s) {
    const int nu = kWarps / a.nch * upw<TIN>();
    const size_t smem = smem_for<TIN, PAIR, NBUF>(a.lcap, a.kpad, a.cs, a.nch, a.nchan,
                                                  std::is_same<TIN, uint32_t>::value && SHORT != 0, a.blen);
    a.smem_bytes = (uint32_t)smem;
    auto kern = k_dedisp<TIN, PAIR, NBUF, SHORT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    const int64_t tile = (int64_t)chunk_t(PAIR) * a.nch;
    const int db = (PAIR ? 2 : 1) * nu;
    const unsigned ntile = (unsigned)((a.t_out + tile - 1) / tile), nblk = (unsigned)((a.ndm + db - 1) / db);
    const bool blk_x = std::is_same<TIN, uint32_t>::value;
    dim3 grid(blk_x ? nblk : ntile, blk_x ? ntile : nblk, (unsigned)a.nsplit);
    if (grid.y > 65535 || a.nsplit < 1 || a.nsplit > 64) return DD_ERR_UNSUPPORTED;
    if ((int64_t)grid.x * grid.y >= INT32_MAX) return DD_ERR_UNSUPPORTED;  // the tile index is int
    kern<<<grid, kWarps * 32, smem, s>>>(a);
    return cuda_status(cudaGetLastError());
}

// Small tap launches: one CTA per pair unit and 768 outputs instead of per eight units and 864.  A
// trial's outputs then run on eight warps of one SM, and the blocks' units on SMs of their own; each
// CTA stages the rows for itself.  One trial x 64 channels x 841 outputs x 32 taps: 36 us against 119.
// Up to a CTA per SM that pays whatever the taps are; long runs, which hide the staging, pay to four
// per SM.  64 and 336 channels, 1-600 trials, 300-9000 outputs, time of the full launch over this
// one's: up to 152 CTAs 0.96-2.2 with 2 taps, 1.06-2.5 with 6, 2.0-5.2 with 16, 2.6-5.1 with 32 and 48;
// 153-304 0.61-1.2, 0.87-1.4, 2.1-3.3, 2.4-3.0; 305-608 0.31-0.97, 0.45-1.2, 1.3-2.8, 1.4-2.8; 609-900
// 0.27-0.38, 0.38-0.46, 1.04-1.10, 0.97-1.11.
constexpr int64_t kUnitCtas = 152, kUnitCtasLong = 608;
constexpr double kUnitLongTaps = 16.0;  // mean taps of a run
struct UnitGrid {
    int64_t tiles, blocks, units;  // (the last block's units past the trial list have only copies to wait for)
};
UnitGrid unit_grid(int64_t t_out, int32_t ndm, int32_t nch) {
    const int nu = kWarps / nch, tile = kWarps * 32 * kRSmall;
    return {(t_out + tile - 1) / tile, (ndm + 2 * nu - 1) / (2 * nu), std::min(nu, (ndm + 1) / 2)};
}

template <typename TIN, int NBUF>
dd_status run_unit(DedispArgs a, cudaStream_t s) {
    const size_t smem = smem_for<TIN, true, NBUF>(a.lcap, a.kpad, a.cs, a.nch, a.nchan);
    a.smem_bytes = (uint32_t)smem;
    auto kern = k_dedisp_unit<TIN, NBUF>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    const UnitGrid g = unit_grid(a.t_out, a.ndm, a.nch);
    dim3 grid((unsigned)g.tiles, (unsigned)g.blocks, (unsigned)g.units);
    kern<<<grid, kWarps * 32, smem, s>>>(a);
    return cuda_status(cudaGetLastError());
}

template <typename TIN, bool PAIR, int NBUF, int SHORT = 0>
dd_status run_batched(const DedispArgs* d_args, const BatchItem* d_items, int32_t nitems, size_t smem,
                      cudaStream_t s) {
    auto kern = k_dedisp_batched<TIN, PAIR, NBUF, SHORT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    if (nitems < 1) return DD_OK;
    kern<<<(unsigned)nitems, kWarps * 32, smem, s>>>(d_args, d_items, (uint32_t)smem);
    return cuda_status(cudaGetLastError());
}

template <typename TIN, bool PAIR, int NBUF, int SHORT = 0>
int blocks_per_sm(size_t smem) {
    int n = 0;
    auto kern = k_dedisp_batched<TIN, PAIR, NBUF, SHORT>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kWarps * 32, smem) != cudaSuccess) return 0;
    return n;
}

// Builds the pair records' (w0, w1) weights from the device weights [d][c][kpad] and
// the tap table, at each entry's weight offset: tap k holds each trial's own tap k,
// zero past its taps (the entries themselves do not change).  One warp per entry.
__global__ void k_repack_w(const float* w, const int32_t* taps, unsigned char* rec, int32_t rec_bytes,
                           int32_t w_off, int32_t nchan, int32_t ndm, int32_t cs, int32_t nu,
                           int32_t kpad, int32_t nst) {
    const int rid = blockIdx.x;  // record = (block, stage)
    const int blk = rid / nst, st = rid - blk * nst;
    const int4* ent = (const int4*)(rec + (int64_t)rid * rec_bytes);
    float* dst = (float*)(rec + (int64_t)rid * rec_bytes + w_off);
    const int lane = threadIdx.x & 31;
    for (int e = threadIdx.x >> 5; e < nu * cs; e += blockDim.x >> 5) {
        const int j = e / cs, ci = e - j * cs;
        const int d0 = blk * 2 * nu + 2 * j, c = st * cs + ci;
        if (d0 >= ndm || c >= nchan) continue;
        const int4 q = ent[e];
        const int64_t dc0 = (int64_t)d0 * nchan + c, dc1 = dc0 + nchan;
        const int n0 = taps[dc0], n1 = d0 + 1 < ndm ? taps[dc1] : 0;
        for (int k = lane; k < q.y; k += 32) {
            dst[2 * (q.w + k)] = k < n0 ? w[dc0 * kpad + k] : 0.f;
            dst[2 * (q.w + k) + 1] = k < n1 ? w[dc1 * kpad + k] : 0.f;
        }
    }
}

// Run-length path, first step: per-channel prefix sums of the uint8 samples,
// P[c][i] = sum_{j<i} I[c][t_offset + j] for 0 <= i <= n (uint32; zero from n + 1 to
// the row's end).  One CTA per channel walks its row in blocks of 4096 samples: each
// thread sums 16 consecutive samples, a warp scan and a scan of the 8 warp totals
// place it, and the block total carries to the next block.
__global__ void __launch_bounds__(256) k_prefix(const uint8_t* in, int64_t ld, int64_t t_offset,
                                                int64_t n, uint32_t* P, int64_t ldp) {
    const int c = blockIdx.x;
    const uint8_t* row = in + (int64_t)c * ld + t_offset;
    uint32_t* prow = P + (int64_t)c * ldp;
    __shared__ uint32_t wsum[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool vec = (((uintptr_t)row) & 15) == 0;
    uint32_t carry = 0;
    int64_t end = 0;
    for (int64_t base = 0; base < n; base += 4096) {
        const int64_t i0 = base + 16 * tid;
        uint32_t v[16];
        if (vec && i0 + 16 <= n) {
            const uint4 q = *(const uint4*)(row + i0);
            const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = (w4[k >> 2] >> (8 * (k & 3))) & 0xffu;
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = i0 + k < n ? (uint32_t)row[i0 + k] : 0u;
        }
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t x = v[k];
            v[k] = sum;  // exclusive within the thread
            sum += x;
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const uint32_t x = wsum[w];
            before += w < warp ? x : 0u;
            total += x;
        }
        const uint32_t off = carry + before + incl - sum;
        if (i0 + 16 <= ldp) {
            uint4* dst = (uint4*)(prow + i0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint4 o4;
                o4.x = i0 + 4 * k + 0 <= n ? off + v[4 * k + 0] : 0u;
                o4.y = i0 + 4 * k + 1 <= n ? off + v[4 * k + 1] : 0u;
                o4.z = i0 + 4 * k + 2 <= n ? off + v[4 * k + 2] : 0u;
                o4.w = i0 + 4 * k + 3 <= n ? off + v[4 * k + 3] : 0u;
                dst[k] = o4;
            }
        } else {
            for (int k = 0; k < 16 && i0 + k < ldp; ++k) prow[i0 + k] = i0 + k <= n ? off + v[k] : 0u;
        }
        carry += total;
        end = base + 4096;
        __syncthreads();  // wsum is rewritten by the next block
    }
    // P[n] when no block reached it, and the zero tail of the row
    if (tid == 0)
        for (int64_t i = end > n ? end : n; i < ldp; ++i) prow[i] = i == n ? carry : 0u;
}

// The packed form for the row kernels: PW[c][i] = P[c][i] + (P[c][i + kPkHalf] << 16) modulo
// 2^32, with P constant past n.  As k_prefix; the block's P values and the kPkHalf before them
// stay in shared memory, so that a block writes the words that end in it.
__global__ void __launch_bounds__(256) k_prefix_packed(const uint8_t* in, int64_t ld, int64_t t_offset,
                                                       int64_t n, uint32_t* PW, int64_t ldp) {
    constexpr int H = kPkHalf, B = 4096;
    __shared__ __align__(16) uint32_t win[H + B];  // P[base - H .. base + B)
    __shared__ uint32_t wsum[8];
    const int c = blockIdx.x;
    const uint8_t* row = in + (int64_t)c * ld + t_offset;
    uint32_t* prow = PW + (int64_t)c * ldp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool vec = (((uintptr_t)row) & 15) == 0;
    uint32_t carry = 0;
    for (int64_t base = 0; base < ldp + H; base += B) {
        const int64_t i0 = base + 16 * tid;
        uint32_t v[16];
        if (vec && i0 + 16 <= n) {
            const uint4 q = *(const uint4*)(row + i0);
            const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = (w4[k >> 2] >> (8 * (k & 3))) & 0xffu;
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = i0 + k < n ? (uint32_t)row[i0 + k] : 0u;
        }
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t x = v[k];
            v[k] = sum;  // exclusive within the thread
            sum += x;
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const uint32_t x = wsum[w];
            before += w < warp ? x : 0u;
            total += x;
        }
        const uint32_t off = carry + before + incl - sum;
#pragma unroll
        for (int k = 0; k < 16; k += 4)
            *(uint4*)(win + H + 16 * tid + k) = make_uint4(off + v[k], off + v[k + 1], off + v[k + 2], off + v[k + 3]);
        carry += total;
        __syncthreads();
        // words base - H .. base + B - H (ldp is a multiple of four)
        for (int k = 4 * tid; k < B; k += 4 * 256) {
            const int64_t i = base - H + k;
            if (i < 0 || i >= ldp) continue;
            const uint4 lo = *(const uint4*)(win + k), hi = *(const uint4*)(win + H + k);
            *(uint4*)(prow + i) = make_uint4(lo.x + (hi.x << 16), lo.y + (hi.y << 16), lo.z + (hi.z << 16), lo.w + (hi.w << 16));
        }
        __syncthreads();
        for (int k = tid; k < H; k += 256) win[k] = win[B + k];
        __syncthreads();
    }
}

}  // namespace


dd_status launch_repack(dd_plan_s* p, cudaStream_t s) {
    if (!p->pair) return DD_OK;
    const int nu = kWarps / p->nch;
    const int nst = (p->nchan + p->cs - 1) / p->cs;
    const StageGeom g(p->band.in_type == DD_U8 ? 1 : 4, true, p->lcap, p->kw, p->cs, nu);
    k_repack_w<<<p->nblk * nst, 256, 0, s>>>(p->dev.w, p->dev.taps, p->dev.rec, g.rec_bytes, g.w_off,
                                              p->nchan, p->ndm, p->cs, nu, p->kpad, nst);
    return cuda_status(cudaGetLastError());
}

void fill_dedisp_args(const dd_plan_s* p, const void* in, int64_t ld, int64_t t_offset,
                      int64_t t_out, void* out, int64_t out_ld, DedispArgs* a) {
    a->in = in;
    a->ld = ld;
    a->t_offset = t_offset;
    a->out = out;
    a->out_ld = out_ld;
    a->t_out = (int32_t)t_out;
    a->rec = p->dev.rec;
    a->blk_lo = p->dev.blk_lo;
    a->nchan = p->nchan;
    a->ndm = p->ndm;
    a->lcap = p->lcap;
    a->blen = p->blen;
    a->cs = p->cs;
    a->nch = p->nch;
    a->kpad = p->pair || p->rk ? p->kw : 0;
    a->rows_max = p->rows_max;
    a->lo_ld = p->lo_ld;
    a->nst = p->nst;
    const dd_plan_s* own = p->owner ? p->owner : p;
    a->status = own->dev.status;
    a->skip_stage = own->debug_skip_stage;
    a->wait_ns = own->wait_ns;
    a->smem_bytes = (uint32_t)dedisp_smem_for(p);
    a->nsplit = 1;
    a->split_ld = 0;
}

size_t dedisp_smem_for(const dd_plan_s* p) {
    if (p->rk) return rows_smem_for(p);
    const int kp = p->pair ? p->kw : 0;
    if (p->rl) return smem_for<uint32_t, false, kStagesRl>(p->lcap, 0, p->cs, p->nch, p->nchan, p->rl_b, p->blen);
    if (!p->pair) return smem_for<uint8_t, false, kStagesInt>(p->lcap, kp, p->cs, p->nch, p->nchan);
    if (p->band.in_type == DD_U8) return smem_for<uint8_t, true, kStagesPair>(p->lcap, kp, p->cs, p->nch, p->nchan);
    return smem_for<float, true, kStagesPair>(p->lcap, kp, p->cs, p->nch, p->nchan);
}

bool takes_units(const dd_plan_s* p, int64_t t_out, int nch) {
    const UnitGrid g = unit_grid(t_out, p->ndm, nch);
    const bool long_taps = (double)p->ns_total >= kUnitLongTaps * p->ndm * p->nchan;
    return g.tiles * g.blocks * g.units <= (long_taps ? kUnitCtasLong : kUnitCtas);
}

dd_status launch_dedisperse(dd_plan_s* p, const void* in, int64_t ld, int64_t t_offset,
                            int64_t t_out, void* out, int64_t out_ld, cudaStream_t s, int nsplit,
                            int64_t split_ld) {
    DedispArgs a;
    fill_dedisp_args(p, in, ld, t_offset, t_out, out, out_ld, &a);
    if (p->rk) return nsplit == 1 ? launch_rows(p, a, s) : DD_ERR_UNSUPPORTED;
    a.nsplit = nsplit;
    a.split_ld = split_ld;
    const bool u8 = p->band.in_type == DD_U8;
    if (!p->pair)
        return p->kmax <= kRInt ? run<uint8_t, false, kStagesInt, 1>(a, s) : run<uint8_t, false, kStagesInt>(a, s);
    if (nsplit == 1 && takes_units(p, t_out, a.nch))
        return u8 ? run_unit<uint8_t, kStagesPair>(a, s) : run_unit<float, kStagesPair>(a, s);
    // union windows of at most R taps: one unrolled pass; at most 2R: two; longer: a loop
    const int passes = p->umax <= kRPair ? 1 : (p->umax <= 2 * kRPair ? 2 : 0);
    if (u8) {
        if (passes == 1) return run<uint8_t, true, kStagesPair, 1>(a, s);
        if (passes == 2) return run<uint8_t, true, kStagesPair, 2>(a, s);
        return run<uint8_t, true, kStagesPair>(a, s);
    }
    if (passes == 1) return run<float, true, kStagesPair, 1>(a, s);
    if (passes == 2) return run<float, true, kStagesPair, 2>(a, s);
    return run<float, true, kStagesPair>(a, s);
}

// Prefix sums of columns t_offset .. t_offset + nsamp - 1 into caller-owned P
// [nchan][ldp] (ldp >= nsamp + 1).
dd_status launch_prefix_into(const dd_plan_s* p, const void* in, int64_t ld, int64_t t_offset,
                             int64_t nsamp, uint32_t* P, int64_t ldp, cudaStream_t s) {
    if (p->rk == kRowsPk)
        k_prefix_packed<<<p->nchan, 256, 0, s>>>((const uint8_t*)in, ld, t_offset, nsamp, P, ldp);
    else
        k_prefix<<<p->nchan, 256, 0, s>>>((const uint8_t*)in, ld, t_offset, nsamp, P, ldp);
    return cuda_status(cudaGetLastError());
}

// A stream that is being captured is not ordered here (its events cannot leave the capture; the
// caller orders the replays).
// The legacy stream, which outlives every call, is recorded when another stream follows it.
PrefixUse::PrefixUse(dd_plan_s* plan, cudaStream_t stream) : p(plan), s(stream) {
    if (!p || p->rl) return;
    lock = std::unique_lock<std::mutex>(p->prefix_mu);
    if (s == nullptr || s == cudaStreamLegacy) {
        id = 1;
    } else {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
            cudaGetLastError();
            return;
        }
        err = cudaStreamGetId(s, &id);
        id += 2;
    }
    if (err != cudaSuccess || p->prefix_stream == 0 || p->prefix_stream == id) return;
    if (p->prefix_stream == 1) err = mark(cudaStreamLegacy);
    if (err == cudaSuccess) err = cudaStreamWaitEvent(s, p->prefix_done, 0);
}

cudaError_t PrefixUse::mark(cudaStream_t q) {
    cudaError_t e = cudaSuccess;
    if (!p->prefix_done) e = cudaEventCreateWithFlags(&p->prefix_done, cudaEventDisableTiming);
    return e == cudaSuccess ? cudaEventRecord(p->prefix_done, q) : e;
}

void PrefixUse::release() {
    if (id != 0 && err == cudaSuccess && (id == 1 || mark(s) == cudaSuccess)) p->prefix_stream = id;
    id = 0;
    if (lock.owns_lock()) lock.unlock();
}

// Room for `need` words of prefix sums (or DD_ERR_OOM, which leaves a direct plan what it has).  A
// run-length plan gives its old scratch back first.  A direct plan may get its scratch in a captured
// call, and keeps an old one for earlier captures until its tables change; the new one is twice as
// large (within `most`, where there is room), so that few are kept.
dd_status prefix_room(dd_plan_s* p, int64_t need, int64_t most = INT64_MAX) {
    if (need <= p->prefix_elems) return DD_OK;
    if (p->rl && p->d_prefix) {
        cudaFree(p->d_prefix);
        p->d_prefix = nullptr;
        p->prefix_elems = 0;
    }
    uint32_t* q = nullptr;
    const int64_t more = std::max(need, std::min(most, 2 * p->prefix_elems));
    cudaError_t e = cudaErrorMemoryAllocation;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (!p->rl) cudaThreadExchangeStreamCaptureMode(&mode);
    for (const int64_t n : {more, need}) {
        if (p->scratch_limit > 0 && n * (int64_t)sizeof(uint32_t) > p->scratch_limit) continue;
        e = cudaMalloc((void**)&q, (size_t)n * sizeof(uint32_t));
        if (e == cudaSuccess) {
            if (p->d_prefix) p->prefix_old.push_back(p->d_prefix);
            p->d_prefix = q;
            p->prefix_elems = n;
            break;
        }
        cudaGetLastError();
        if (e != cudaErrorMemoryAllocation || n == need) break;
    }
    if (!p->rl) cudaThreadExchangeStreamCaptureMode(&mode);
    return cuda_status(e);
}

// Run-length path: prefix sums of columns t_offset .. t_offset + nsamp - 1 into the
// plan's scratch, then the run-length sums over them.
dd_status launch_prefix(dd_plan_s* p, const void* in, int64_t ld, int64_t t_offset, int64_t nsamp,
                        int64_t* ldp_out, cudaStream_t s) {
    const int64_t ldp = (nsamp + 1 + 3) & ~(int64_t)3;
    *ldp_out = ldp;
    const dd_status st = prefix_room(p, ldp * p->nchan);
    if (st != DD_OK) return st;
    return launch_prefix_into(p, in, ld, t_offset, nsamp, p->d_prefix, ldp, s);
}

dd_status launch_dedisperse_rl(dd_plan_s* p, const void* in, int64_t ld, int64_t t_offset,
                               int64_t nsamp, void* out, int64_t out_ld, cudaStream_t s) {
    int64_t ldp = 0;
    const dd_status st = launch_prefix(p, in, ld, t_offset, nsamp, &ldp, s);
    if (st != DD_OK) return st;
    DedispArgs a;
    fill_dedisp_args(p, p->d_prefix, ldp, 0, nsamp - p->dmax, out, out_ld, &a);
    if (p->rk) return launch_rows(p, a, s);
    return p->rl_b ? run<uint32_t, false, kStagesRl, 1>(a, s) : run<uint32_t, false, kStagesRl>(a, s);
}

dd_status launch_dedisperse_pk(dd_plan_s* p, const void* in, int64_t ld, int64_t t_offset,
                               int64_t nsamp, void* out, int64_t out_ld, cudaStream_t s) {
    PrefixUse use(p, s);
    if (use.err != cudaSuccess) return cuda_status(use.err);
    // Columns of scratch: the call's, within 2 GiB or what the longest delay and two tiles need;
    // what there is, or that least, where no more is to be had.
    const int64_t tile = row_tile_t(kRowsPk, p->nch), t_out = nsamp - p->dmax;
    auto round4 = [](int64_t n) { return (n + 3) & ~(int64_t)3; };
    const int64_t least = round4((int64_t)p->dmax + 2 * tile + 1);
    const int64_t most = std::max(least, ((int64_t)1 << 29) / p->nchan & ~(int64_t)3);
    const int64_t want = std::min(round4(nsamp + 1), most);
    dd_status st = prefix_room(p, want * p->nchan, most * p->nchan);
    if (st == DD_ERR_OOM) st = prefix_room(p, std::min(want, least) * p->nchan);
    if (st != DD_OK) return st;
    // outputs per piece: whole tiles, as many as the scratch holds with the delays behind them
    const int64_t cols = p->prefix_elems / p->nchan & ~(int64_t)3;
    int64_t piece = std::min(cols - 1 - p->dmax, 65535 * tile);  // (grid y)
    if (piece < t_out) piece = piece / tile * tile;
    if (piece < 1) return DD_ERR_OOM;
    for (int64_t t0 = 0; t0 < t_out; t0 += piece) {
        const int64_t n = std::min(piece, t_out - t0) + p->dmax, ldp = (n + 1 + 3) & ~(int64_t)3;
        if ((st = launch_prefix_into(p, in, ld, t_offset + t0, n, p->d_prefix, ldp, s)) != DD_OK) return st;
        DedispArgs a;
        fill_dedisp_args(p, p->d_prefix, ldp, 0, n - p->dmax, (int32_t*)out + t0, out_ld, &a);
        if ((st = launch_rows(p, a, s)) != DD_OK) return st;
    }
    return DD_OK;
}

dd_status launch_dedisperse_batched(bool u8, bool pair, bool short_taps, const DedispArgs* d_args,
                                    const BatchItem* d_items, int32_t nitems, size_t smem, cudaStream_t s,
                                    bool rl) {
    if (rl)  // run-length beams: short_taps = difference rows shared by the CTA
        return short_taps ? run_batched<uint32_t, false, kStagesRl, 1>(d_args, d_items, nitems, smem, s)
                          : run_batched<uint32_t, false, kStagesRl>(d_args, d_items, nitems, smem, s);
    if (!pair)
        return short_taps ? run_batched<uint8_t, false, kStagesInt, 1>(d_args, d_items, nitems, smem, s)
                          : run_batched<uint8_t, false, kStagesInt>(d_args, d_items, nitems, smem, s);
    if (u8)
        return short_taps ? run_batched<uint8_t, true, kStagesPair, 1>(d_args, d_items, nitems, smem, s)
                          : run_batched<uint8_t, true, kStagesPair>(d_args, d_items, nitems, smem, s);
    return short_taps ? run_batched<float, true, kStagesPair, 1>(d_args, d_items, nitems, smem, s)
                      : run_batched<float, true, kStagesPair>(d_args, d_items, nitems, smem, s);
}

int dedisp_batched_blocks_per_sm(bool u8, bool pair, bool short_taps, size_t smem, bool rl) {
    if (rl) return short_taps ? blocks_per_sm<uint32_t, false, kStagesRl, 1>(smem) : blocks_per_sm<uint32_t, false, kStagesRl>(smem);
    if (!pair) return short_taps ? blocks_per_sm<uint8_t, false, kStagesInt, 1>(smem) : blocks_per_sm<uint8_t, false, kStagesInt>(smem);
    if (u8) return short_taps ? blocks_per_sm<uint8_t, true, kStagesPair, 1>(smem) : blocks_per_sm<uint8_t, true, kStagesPair>(smem);
    return short_taps ? blocks_per_sm<float, true, kStagesPair, 1>(smem) : blocks_per_sm<float, true, kStagesPair>(smem);
}

}  // namespace dd
