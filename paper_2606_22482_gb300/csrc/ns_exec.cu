// ns_exec.cu -- the persistent execute kernel (Sections 5.1 and 7 of arXiv 2606.22482).
//
// One launch, grid = resident CTAs on every SM.  CTAs pull work items from one atomic ticket in
// the plan's cost order (heaviest first, Section 7 "row window list migration" in GPU form):
//   * dense item    -- a row window: sum over its dense tiles of A_tile * B[cols, :] on the
//                      tensor cores (matrix-engine execution model, Section 5.1), then the rows'
//                      absorbed residual on the CUDA cores, then the rows are stored;
//   * residual item -- kExecWarps merge-path chunks of the residual CSR, one per warp: gather B
//                      rows by column index and accumulate into output rows (vector-engine
//                      execution model, Section 5.1), several B rows per warp step when K is
//                      narrow (Section 7 "vector tiles merging").
// A row assembled from several pieces (cut by a chunk boundary, or shared by a dense window and
// residual chunks) is combined without atomics on C: each piece writes a partial to its slot,
// the last piece to arrive sums the slots in piece order and stores the row.  The result is
// therefore deterministic.
//
// L2 policy (Section 6.2.1 hot-B staging in GPU form): A's arrays and C are streamed with an
// evict-first policy, B rows are loaded with evict-last so that reused B rows stay in L2.
#include "ns_internal.cuh"
#include "ns_mem.cuh"
#include "ns_ptx.cuh"

#include "ns_residual.cuh"
#include "ns_dense.cuh"
#include "ns_dense_tc.cuh"

namespace ns {

// ---------------------------------------------------------------------------------------------
// the persistent kernel
// ---------------------------------------------------------------------------------------------
// residual-only kernels are held to 128 registers (4 CTAs = 16 warps per SM, each with an 8-deep
// gather ring); kernels with the tensor-core item keep their registers for the accumulators
template <int L, int VPL, bool BF16, bool HINT, bool DENSE>
__global__ void __launch_bounds__(kExecThreads, DENSE ? 1 : 4) k_exec(const ExecDesc* __restrict__ descs,
                                                       const int32_t* __restrict__ queue,
                                                       const int32_t* __restrict__ queue_desc,
                                                       int64_t n_items, int32_t* ctrl,
                                                       const __grid_constant__ ExecDesc d0)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int32_t s_ticket;
    __shared__ int4 s_rowmeta[DENSE ? 64 : 1];  // a dense window's rows (TM <= 64)
    // BF16 plans with K <= 256 run their dense tiles on the 5th-generation tensor cores (tcgen05,
    // accumulator in tensor memory); other dense plans use the warp-level mma.sync item
    constexpr bool TC = DENSE && BF16 && VPL <= 2;
    __shared__ __align__(8) uint64_t s_tc_bars[TC ? kTcBars : 1];
    __shared__ uint32_t s_tc_tmem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Policies pol{0, 0};
    if (HINT) pol = make_policies();
    unsigned long long* const clk = descs ? nullptr : d0.class_clock;  // single-plan launches only
    if (clk && threadIdx.x == 0) atomicMin(clk, global_ns());
    if (DENSE) {
        TcState tcs{};
        if constexpr (TC) tc_setup(tcs, s_tc_bars, &s_tc_tmem);
        // phase 1: dense windows, one CTA each, taken in work-list order
        for (;;) {
            if (threadIdx.x == 0) s_ticket = atomicAdd(ctrl + 0, 1);
            __syncthreads();
            const int64_t t = s_ticket;
            __syncthreads();
            if (t >= n_items) break;
            const int32_t it = __ldg(queue + t);
            const ExecDesc& D = descs ? descs[queue_desc ? __ldg(queue_desc + t) : 0] : d0;
            if (it < D.n_dwin) {
                if constexpr (TC) {
                    const TcGeom G = tc_geom(D.K, D.TM, D.TK);
                    if (!tcs.ok) {
                        // an earlier bounded wait of this CTA gave up (status already set)
                    } else if (dynamic_smem_bytes() >= (uint32_t)G.total && tc_supported(D.K) && D.dtile_x &&
                               D.TM % 16 == 0 && D.TM <= 64 && D.TK % 16 == 0) {
                        const int32_t w = __ldg(D.dwin + it);
                        dense_row_meta<kExecWarps>(D, it, w, s_rowmeta);  // (read while the product runs)
                        if (tc_window_product<HINT>(D, w, smem_raw, G, tcs, pol))
                            dense_deliver_rows<L, VPL, BF16, HINT>(D, it, w, reinterpret_cast<float*>(smem_raw + G.off_c),
                                                                  G.cs_stride, s_rowmeta, pol);
                    } else if (threadIdx.x == 0) {
                        atomicOr(D.status, kStatusInternal);  // guard: launch without the tile buffers
                    }
                } else {
                    if (dynamic_smem_bytes() >= (uint32_t)dense_geom(D.K, D.TM, D.TK, BF16).total)
                        dense_item<L, VPL, BF16, HINT>(D, it, smem_raw, s_rowmeta, pol);
                    else if (threadIdx.x == 0)
                        atomicOr(D.status, kStatusInternal);  // guard: launch without the tile buffers
                }
                if (clk && threadIdx.x == 0) atomicMax(clk + 1, global_ns());
            }
        }
        if constexpr (TC) tc_teardown(tcs, descs ? descs[0].status : d0.status);
    }
    // phase 2: residual chunks
    residual_phase<L, VPL, BF16, HINT>(descs, queue, queue_desc, n_items, ctrl, d0, lane, warp, smem_raw, kExecWarps,
                                       pol, clk);
    end_launch(ctrl, d0, descs == nullptr);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
// the residual list is every row in order and A itself is the residual (no window pass ran):
// a chunk's nonzeros are one contiguous range of A and its rows are k0 .. kL
bool plan_contig(const Plan* P)
{
    return P->tune.tau_tile == kTauInf && P->st.n_dwin == 0 && P->st.n_rl == P->st.m;
}

// Column slices start every chunk once a slice, which costs more than they gain when a chunk is a few
// nonzeros (K 512 FP32, 2^16 nodes of 16, us by slices and by k_exec: W 128 197 and 225, 64 261 and 241, 32 385
// and 290, 16 653 and 389).
bool contig_form(const Plan* P, int K)
{
    return plan_contig(P) && !(contig_slices(K) > 1 && P->tune.chunk_nnz <= 32);
}

void fill_desc(const Plan* P, const void* B, int64_t ldb, float* C, int64_t ldc, ExecDesc* d)
{
    *d = ExecDesc{};
    d->res_rowptr = P->res_rowptr;
    d->res_col = P->res_col;
    d->res_val = P->res_val;
    d->rl_rows = P->rl_rows;
    d->rl_start = P->rl_start;
    d->chunk_b = P->chunk_b;
    d->chunk_k0 = P->chunk_k0;
    d->chunk_rec = P->chunk_rec;
    d->n_chunks = (int32_t)P->st.n_chunks;
    d->n_dwin = (int32_t)P->st.n_dwin;
    d->win_rows = P->win_rows;
    d->win_dptr = P->win_dptr;
    d->dwin = P->dwin;
    d->dwin_absorb = P->dwin_absorb;
    d->dtile_cols = P->dtile_cols;
    d->dtile_bits = P->dtile_bits;
    d->dtile_voff = P->dtile_voff;
    d->dtile_vals = P->dtile_vals;
    d->dtile_x = P->dtile_x;
    d->row_split = P->row_split;
    d->split_np = P->split_np;
    d->split_slot = P->split_slot;
    d->split_base = P->split_base;
    d->slots = P->slots;
    d->split_cnt = P->split_cnt;
    d->B = B;
    d->C = C;
    d->ldb = ldb;
    d->ldc = ldc;
    d->K = P->K;
    d->b_bf16 = P->dtype == NS_BF16;
    d->TM = P->tune.TM;
    d->TK = P->tune.TK;
    d->group = P->tune.group;
    d->l2_hints = P->tune.l2_hints;
    d->m = (int32_t)P->st.m;
    d->n = (int32_t)P->st.n;
    d->n_rl = (int32_t)P->st.n_rl;
    d->n_res = (int32_t)P->st.n_res;
    d->rl_all = plan_contig(P) ? 1 : 0;
    d->hot = P->hot_bits;
    d->chunk_nnz = P->tune.chunk_nnz;
    d->status = P->ctrl + 2;
    d->status_out = P->status_map;
    d->class_clock = P->class_clock;
}

typedef void (*ExecKernel)(const ExecDesc*, const int32_t*, const int32_t*, int64_t, int32_t*, ExecDesc);

template <bool BF16, bool HINT, bool DENSE>
static ExecKernel pick_kernel(int K)
{
    const int nv = K / 4;
    if (nv <= 2) return k_exec<2, 1, BF16, HINT, DENSE>;
    if (nv <= 4) return k_exec<4, 1, BF16, HINT, DENSE>;
    if (nv <= 8) return k_exec<8, 1, BF16, HINT, DENSE>;
    if (nv <= 16) return k_exec<16, 1, BF16, HINT, DENSE>;
    if (nv <= 32) return k_exec<32, 1, BF16, HINT, DENSE>;
    if (nv <= 64) return k_exec<32, 2, BF16, HINT, DENSE>;
    if (nv <= 128) return k_exec<32, 4, BF16, HINT, DENSE>;
    return k_exec<32, 8, BF16, HINT, DENSE>;
}

static ExecKernel select_kernel(int K, bool bf16, bool hint, bool dense)
{
    if (bf16) {
        if (hint) return dense ? pick_kernel<true, true, true>(K) : pick_kernel<true, true, false>(K);
        return dense ? pick_kernel<true, false, true>(K) : pick_kernel<true, false, false>(K);
    }
    if (hint) return dense ? pick_kernel<false, true, true>(K) : pick_kernel<false, true, false>(K);
    return dense ? pick_kernel<false, false, true>(K) : pick_kernel<false, false, false>(K);
}

int num_sms(int device)
{
    static int cached[64] = {0};
    if (device < 0 || device >= 64) return 148;
    if (!cached[device]) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || v <= 0) v = 148;
        cached[device] = v;
    }
    return cached[device];
}

int64_t l2_bytes(int device)
{
    static int64_t cached[64] = {0};
    if (device < 0 || device >= 64) return 126ll << 20;
    if (!cached[device]) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, device) != cudaSuccess || v <= 0) v = 126 << 20;
        cached[device] = v;
    }
    return cached[device];
}

// dynamic shared memory of one execute CTA: the dense item's tiles (phase 1) or the residual
// warps' staging rings (phase 2), whichever is larger
static size_t exec_smem_bytes(int K, int TM, int TK, bool bf16, bool dense, int W)
{
    // (L, VPL) exactly as pick_kernel chooses the instantiation
    const int nv = K / 4;
    const int L = nv <= 2 ? 2 : (nv <= 4 ? 4 : (nv <= 8 ? 8 : (nv <= 16 ? 16 : 32)));
    const int VPL = nv <= 32 ? 1 : (nv <= 64 ? 2 : (nv <= 128 ? 4 : 8));
    size_t b = staged_path(L, VPL) ? (size_t)kExecWarps * stage_geom(K, bf16, W).warp_bytes : 0;
    // (chunk_nnz <= 1024 keeps this within the 227 KB a CTA may use)
    if (dense) {
        // BF16 with K <= 256: the tensor-core (tcgen05) item's ring; otherwise the mma.sync item
        size_t d = (bf16 && VPL <= 2) ? (size_t)tc_geom(K, TM, TK).total : dense_smem_bytes(K, TM, TK, bf16);
        if (d > b) b = d;
    }
    return b;
}

// Kernel attributes and the persistent grid (resident CTAs on every SM, at most n_items).
// Must run outside stream capture.
ns_status_t exec_prepare(int64_t n_items, int K, int TM, int TK, bool bf16, bool hint, bool dense,
                         bool planes, int* grid_out, int W)
{
    if (dense && planes && K <= kF32TcMaxK) return f32_prepare(n_items, K, TM, TK, hint, W, grid_out);
    ExecKernel kern = select_kernel(K, bf16, hint, dense);
    const size_t smem = exec_smem_bytes(K, TM, TK, bf16, dense, W);
    if (smem > 48 * 1024) NS_TRY(dense_prepare(reinterpret_cast<const void*>(kern), smem));
    int per_sm = 0;
    NS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kExecThreads, smem));
    int dev = 0;
    NS_CUDA_TRY(cudaGetDevice(&dev));
    if (smem > 48 * 1024) {
        // The query may assume a smaller shared-memory carve-out than the SM has; the persistent
        // grid is sized from the SM's capacity (CTAs that do not fit simply start later).
        int sm_smem = 0, regs_sm = 0;
        cudaFuncAttributes fa{};
        NS_CUDA_TRY(cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
        NS_CUDA_TRY(cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev));
        NS_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
        const int by_smem = sm_smem / (int)(smem + fa.sharedSizeBytes + 1024);
        const int by_regs = fa.numRegs > 0 ? regs_sm / (fa.numRegs * kExecThreads) : by_smem;
        const int fit = by_smem < by_regs ? by_smem : by_regs;
        if (fit > per_sm) per_sm = fit;
    }
    // the tensor-core item allocates tensor memory per CTA: no more CTAs per SM than it holds
    if (dense && bf16 && tc_supported(K) && per_sm > kTcCtasPerSm) per_sm = kTcCtasPerSm;
    if (per_sm < 1) per_sm = 1;
    int64_t g = (int64_t)per_sm * num_sms(dev);
    if (g > n_items) g = n_items;
    *grid_out = (int)(g > 0 ? g : 1);
    return NS_OK;
}

// One persistent launch over `n_items` work items.  queue[t] is an item id of descriptor
// queue_desc[t] (descriptor 0 when queue_desc is NULL).  All descriptors share K, dtype and L2
// policy; `dense` selects the kernel with the tensor-core item compiled in, `planes` (every dense
// plan of an FP32 launch keeps its tiles' planes) the tcgen05 one up to kF32TcMaxK.  *grid_cache keeps
// the occupancy-derived grid between launches (0 = compute).
ns_status_t exec_launch(const ExecDesc* descs, const int32_t* queue, const int32_t* queue_desc,
                        int64_t n_items, int32_t* ctrl, int K, int TM, int TK, bool bf16, bool hint,
                        bool dense, bool planes, int* grid_cache, cudaStream_t s, const ExecDesc* d0, int W)
{
    if (dense && planes && K <= kF32TcMaxK)
        return f32_launch(descs, queue, queue_desc, n_items, ctrl, K, TM, TK, hint, W, grid_cache, s, d0);
    ExecKernel kern = select_kernel(K, bf16, hint, dense);
    const size_t smem = exec_smem_bytes(K, TM, TK, bf16, dense, W);
    int grid = grid_cache ? *grid_cache : 0;
    if (grid == 0) NS_TRY(exec_prepare(n_items, K, TM, TK, bf16, hint, dense, planes, &grid, W));
    if (grid_cache) *grid_cache = grid;
    if (n_items == 0) return NS_OK;
    ExecDesc dv{};
    if (d0) dv = *d0;
    kern<<<grid, kExecThreads, smem, s>>>(d0 ? nullptr : descs, queue, queue_desc, n_items, ctrl, dv);
    NS_LAUNCH_CHECK();
    return NS_OK;
}

// single plan: the descriptor travels as a kernel parameter (no upload per launch)
ns_status_t exec_launch_plan(Plan* P, cudaStream_t s)
{
    const int K = P->desc_host.K;  // the column slice of this launch
    const bool contig = contig_form(P, K);
    const bool any = contig && contig_any(P->desc_host.B, P->desc_host.ldb, P->dtype == NS_BF16);
    int* gc = K == P->K ? &P->exec_grid[any] : &P->exec_grid_slice[any];
    if (K != P->K && P->exec_grid_slice_K[any] != K) {
        P->exec_grid_slice[any] = 0;
        P->exec_grid_slice_K[any] = K;
    }
    if (contig) {
        ContigMode m;
        m.any = any;
        m.hot = P->hot_bits != nullptr;
        m.far = contig_far(P->st.n, K, P->dtype == NS_BF16, P->device);
        m.coop = contig_coop(P->st.n_chunks, P->device);
        return contig_launch(nullptr, P->queue, nullptr, P->st.n_items, P->ctrl, K, P->dtype == NS_BF16, m, gc, s,
                             &P->desc_host);
    }
    return exec_launch(nullptr, P->queue, nullptr, P->st.n_items, P->ctrl, K, P->tune.TM,
                       P->tune.TK, P->dtype == NS_BF16, P->tune.l2_hints != 0, P->st.n_dwin > 0,
                       plan_planes(P), gc, s, &P->desc_host, P->tune.chunk_nnz);
}

}  // namespace ns
