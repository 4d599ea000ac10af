// Row kernels (dd_rows.cuh): the plain and batched launches.
#include "dd_rows.cuh"

namespace dd {
namespace {

// Tile order as k_dedisp: packed rows with trial blocks along x (the resident CTAs share time
// tiles, whose prefix sums then come from L2), fp32 rows in groups of 16 blocks.
constexpr int kGroupBlocks = 16;

template <int KIND, bool IN8, int NW>
__global__ void __launch_bounds__(NW * 32, 16 / NW) k_rows(DedispArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TileState ts;
    if (threadIdx.x == 0) init_pipeline<1>(pipeline_area(smem, a.smem_bytes, 1), ts);
    __syncthreads();
    if constexpr (KIND == kRowsPk) {
        row_tile<KIND, IN8, NW, false, false>(a, smem, blockIdx.x, blockIdx.y, ts);
    } else {
        const int ntile = (int)gridDim.x, nblk = (int)gridDim.y;
        const int L = (int)blockIdx.y * ntile + (int)blockIdx.x;
        const int g = L / (kGroupBlocks * ntile), r = L - g * kGroupBlocks * ntile;
        const int gb = min(kGroupBlocks, nblk - g * kGroupBlocks);
        row_tile<KIND, IN8, NW, false, false>(a, smem, g * kGroupBlocks + r % gb, r / gb, ts);
    }
}

template <int KIND, bool IN8, int NW>
__global__ void __launch_bounds__(NW * 32, 16 / NW) k_rows_batched(const DedispArgs* beams, const BatchItem* items,
                                                                 uint32_t smem_bytes) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ TileState ts;
    __shared__ DedispArgs sa;
    if (threadIdx.x == 0) init_pipeline<1>(pipeline_area(smem, smem_bytes, 1), ts);
    const BatchItem it = items[blockIdx.x];
    if (threadIdx.x == 0) {
        sa = beams[it.beam];
        sa.smem_bytes = smem_bytes;
    }
    __syncthreads();
    row_tile<KIND, IN8, NW, false, false>(sa, smem, it.blk, it.tx, ts);
}

template <int KIND, bool IN8, int NW>
dd_status run(DedispArgs a, size_t smem, cudaStream_t s) {
    a.smem_bytes = (uint32_t)smem;
    auto kern = k_rows<KIND, IN8, NW>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    const int64_t tile = row_tile_t(KIND, a.nch);
    const int db = row_trials(KIND, NW, a.nch);
    const unsigned ntile = (unsigned)((a.t_out + tile - 1) / tile), nblk = (unsigned)((a.ndm + db - 1) / db);
    const bool blk_x = KIND == kRowsPk;
    dim3 grid(blk_x ? nblk : ntile, blk_x ? ntile : nblk);
    if (grid.y > 65535 || (int64_t)grid.x * grid.y >= INT32_MAX) return DD_ERR_UNSUPPORTED;
    kern<<<grid, NW * 32, smem, s>>>(a);
    return cuda_status(cudaGetLastError());
}

template <int KIND, bool IN8, int NW>
dd_status run_batched(const DedispArgs* d_args, const BatchItem* d_items, int32_t nitems, size_t smem,
                      cudaStream_t s) {
    auto kern = k_rows_batched<KIND, IN8, NW>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    if (nitems < 1) return DD_OK;
    kern<<<(unsigned)nitems, NW * 32, smem, s>>>(d_args, d_items, (uint32_t)smem);
    return cuda_status(cudaGetLastError());
}

template <int KIND, bool IN8, int NW>
int blocks_per_sm(size_t smem) {
    int n = 0;
    auto kern = k_rows_batched<KIND, IN8, NW>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, NW * 32, smem) != cudaSuccess) return 0;
    return n;
}

}  // namespace

size_t rows_smem_for(const dd_plan_s* p) {
    const RowGeom g(p->rk, p->cs, p->row_warps / p->nch, p->rows_max, p->kw);
    const int esz = p->rk == kRowsFir && p->band.in_type == DD_U8 ? 1 : 4;  // samples or prefix sums
    return row_smem_bytes(g, p->row_warps, esz, p->lcap, p->cs, p->lo_ld, p->blen);
}

// fn<kind, uint8 input, warps per CTA>(args) of a row plan
#define DD_ROWS_NW(fn, kind, in8, nw, ...) \
    ((nw) == kRowWarps ? fn<kind, in8, kRowWarps>(__VA_ARGS__) : fn<kind, in8, kWarps>(__VA_ARGS__))
#define DD_ROWS(fn, kind, in8, nw, ...)                                     \
    ((kind) == kRowsPk ? DD_ROWS_NW(fn, kRowsPk, false, nw, __VA_ARGS__)    \
     : (in8)           ? DD_ROWS_NW(fn, kRowsFir, true, nw, __VA_ARGS__)    \
                       : DD_ROWS_NW(fn, kRowsFir, false, nw, __VA_ARGS__))

dd_status launch_rows(const dd_plan_s* p, DedispArgs a, cudaStream_t s) {
    const size_t smem = rows_smem_for(p);
    return DD_ROWS(run, p->rk, p->band.in_type == DD_U8, p->row_warps, a, smem, s);
}

dd_status launch_rows_batched(int kind, bool in8, int nw, const DedispArgs* d_args, const BatchItem* d_items,
                              int32_t nitems, size_t smem, cudaStream_t s) {
    return DD_ROWS(run_batched, kind, in8, nw, d_args, d_items, nitems, smem, s);
}

int rows_batched_blocks_per_sm(int kind, bool in8, int nw, size_t smem) {
    return DD_ROWS(blocks_per_sm, kind, in8, nw, smem);
}

}  // namespace dd
