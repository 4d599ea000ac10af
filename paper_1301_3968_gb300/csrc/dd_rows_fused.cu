// Row kernels (dd_rows.cuh) with the boxcar scan of finished tiles in the CTA: the row form
// of k_dedisp_fused (dd_fused.cu), with the same parts, carries and seams.
#include "dd_rows.cuh"

namespace dd {
namespace {

// ONE_ROW: packed rows whose trials take turns in one row per warp group (FusedArgs::one_row; the
// fp32 rows read that at run time).
template <int KIND, bool IN8, int NW, bool ONE_ROW>
__global__ void __launch_bounds__(NW * 32, 16 / NW) k_rows_fused(DedispArgs a, const FusedArgs f) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TileState ts;
    if (threadIdx.x == 0) init_pipeline<1>(pipeline_area(smem, a.smem_bytes, 1), ts);
    __syncthreads();
    __shared__ fused::FusedTile ft;  // the tile's strip (as k_dedisp_fused)
    static_assert(sizeof(TileState) + sizeof(fused::FusedTile) + 64 <= kSmemStatic, "static shared memory");
    const int s = (int)f.order[blockIdx.x];
    const int i0 = (int)f.starts[s], i1 = (int)f.starts[s + 1];
    for (int it = i0; it < i1; ++it) {
        const int blk = it / f.tiles;
        const int tx = it - blk * f.tiles;
        if (threadIdx.x == 0) {
            const int L = row_tile_t(KIND, a.nch);
            const int tpc = row_trials(KIND, NW, a.nch);
            const int tx0 = it - tx <= i0 ? i0 - (it - tx) : 0;                    // strip start
            const int tx1 = i1 - (it - tx) < f.tiles ? i1 - (it - tx) : f.tiles;  // strip end
            ft.first = tx == tx0;
            ft.last = tx == tx1 - 1;
            ft.s1 = min((int64_t)tx1 * L, (int64_t)a.t_out);
            ft.carry = f.carry + (int64_t)s * tpc * f.C;
            ft.seam_in = tx0 > 0 ? f.seam + (int64_t)s * tpc * 2 * f.C : nullptr;
            ft.seam_out = tx1 < f.tiles ? f.seam + (int64_t)(s + 1) * tpc * 2 * f.C : nullptr;
        }
        if (!row_tile<KIND, IN8, NW, true, true, ONE_ROW>(a, smem, blk, tx, ts, &f, &ft)) break;
    }
}

template <int KIND, bool IN8, int NW>
dd_status run_fused(DedispArgs a, const FusedArgs& f, size_t smem, cudaStream_t s) {
    a.smem_bytes = (uint32_t)smem;
    auto kern = k_rows_fused<KIND, IN8, NW, false>;
    if constexpr (KIND == kRowsPk) {
        if (f.one_row) {  // (the rows of eight warps always fit)
            if constexpr (NW == kRowWarps) kern = k_rows_fused<KIND, IN8, NW, true>;
            else return DD_ERR_UNSUPPORTED;
        }
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    kern<<<(unsigned)f.nparts, NW * 32, smem, s>>>(a, f);
    return cuda_status(cudaGetLastError());
}

template <int KIND, bool IN8, int NW>
int fused_bps(size_t smem) {
    int n = 0;
    auto kern = k_rows_fused<KIND, IN8, NW, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, NW * 32, smem) != cudaSuccess) return 0;
    return n;
}

}  // namespace

#define DD_ROWS_NW(fn, kind, in8, nw, ...) \
    ((nw) == kRowWarps ? fn<kind, in8, kRowWarps>(__VA_ARGS__) : fn<kind, in8, kWarps>(__VA_ARGS__))
#define DD_ROWS(fn, p, ...)                                                                     \
    ((p)->rk == kRowsPk            ? DD_ROWS_NW(fn, kRowsPk, false, (p)->row_warps, __VA_ARGS__)  \
     : (p)->band.in_type == DD_U8 ? DD_ROWS_NW(fn, kRowsFir, true, (p)->row_warps, __VA_ARGS__)  \
                                  : DD_ROWS_NW(fn, kRowsFir, false, (p)->row_warps, __VA_ARGS__))

dd_status launch_rows_fused(const dd_plan_s* p, DedispArgs a, const FusedArgs& f, size_t smem, cudaStream_t s) {
    return DD_ROWS(run_fused, p, a, f, smem, s);
}

int rows_fused_blocks_per_sm(const dd_plan_s* p, size_t smem) { return DD_ROWS(fused_bps, p, smem); }

}  // namespace dd
