// ns_residual.cuh -- the CUDA-core side of the execute kernels: delivering rows and pieces of split
// rows, and the residual chunks of plans with dense windows.
#pragma once
#include "ns_internal.cuh"
#include "ns_mem.cuh"
#include "ns_ptx.cuh"

namespace ns {

// ---------------------------------------------------------------------------------------------
// delivering one piece of an output row
//   L lanes (lane < L) hold VPL float4 vectors each: vector v = lane + L*q covers columns 4v..4v+3
// ---------------------------------------------------------------------------------------------
// `split`: the row's split id when the caller has it (>= -1), else kSplitUnknown (loaded here)
constexpr int32_t kSplitUnknown = -2;
template <int L, int VPL, bool HINT>
__device__ __forceinline__ void deliver_row(const ExecDesc& D, int32_t row, int32_t piece_of_chunk,
                                            bool dense_piece, const float4 (&acc)[VPL], int lane,
                                            uint64_t pol_first, int32_t split = kSplitUnknown)
{
    const int nv = D.K >> 2;
    const int32_t s = split != kSplitUnknown ? split : __ldg(D.row_split + row);
    float* crow = D.C + (int64_t)row * D.ldc;
    if (s < 0) {
        if (lane < L) {
#pragma unroll
            for (int q = 0; q < VPL; ++q) {
                int v = lane + L * q;
                if (v < nv) st_c4<HINT>(crow + 4 * v, acc[q], pol_first);
            }
        }
        return;
    }
    const int32_t np = __ldg(D.split_np + s);
    const int32_t piece = dense_piece ? 0 : piece_of_chunk - __ldg(D.split_base + s);
    float* slot0 = D.slots + (int64_t)__ldg(D.split_slot + s) * D.K;
    if (lane < L) {
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            int v = lane + L * q;
            if (v < nv) __stcg(reinterpret_cast<float4*>(slot0 + (int64_t)piece * D.K + 4 * v), acc[q]);
        }
    }
    __threadfence();
    __syncwarp();
    int old = 0;
    if (lane == 0) old = atomicAdd(D.split_cnt + s, 1);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old != np - 1) return;  // not the last piece
    __threadfence();
    if (lane < L) {
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            int v = lane + L * q;
            if (v < nv) {
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int p = 0; p < np; ++p)
                    sum = f4_add(sum, __ldcg(reinterpret_cast<const float4*>(slot0 + (int64_t)p * D.K + 4 * v)));
                st_c4<HINT>(crow + 4 * v, sum, pol_first);
            }
        }
    }
    if (lane == 0) atomicExch(D.split_cnt + s, 0);  // ready for the next launch
}

// ---------------------------------------------------------------------------------------------
// residual: acc += sum_{z in [z0, z1)} val[z] * B[col[z], :]
//   the warp's 32 lanes form G = 32/L groups; group g handles nonzeros g, g+G, ... of each batch
//   of 32 (vector tiles merging when K < 128), then the groups are summed with shuffles.
// ---------------------------------------------------------------------------------------------
template <int L, int VPL, bool BF16, bool HINT>
__device__ __forceinline__ void gather_accumulate(const ExecDesc& D, int64_t z0, int64_t z1,
                                                  float4 (&acc)[VPL], int lane, const Policies& pol)
{
    constexpr int G = 32 / L;
    const int g = lane / L, li = lane % L;
    const int nv = D.K >> 2;
    for (int64_t zb = z0; zb < z1; zb += 32) {
        const int cnt = (int)(z1 - zb < 32 ? z1 - zb : 32);
        int32_t mc = 0;
        float mv = 0.f;
        if (lane < cnt) {
            mc = ld_stream_i32<HINT>(D.res_col + zb + lane, pol.first);
            mv = ld_stream_f32<HINT>(D.res_val + zb + lane, pol.first);
            if ((unsigned)mc >= (unsigned)D.n) {  // guard: never gather outside B
                atomicOr(D.status, kStatusInternal);
                mc = 0;
                mv = 0.f;
            }
        }
        // 4 independent B rows in flight per lane
        for (int j0 = 0; j0 < cnt; j0 += 4 * G) {
            int32_t col[4];
            float val[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int j = j0 + u * G + g;
                col[u] = __shfl_sync(0xffffffffu, mc, j & 31);
                val[u] = __shfl_sync(0xffffffffu, mv, j & 31);
                if (j >= cnt) val[u] = 0.f, col[u] = -1;
            }
            BRaw<BF16> b[4][VPL];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < VPL; ++q) {
                    const int v = li + L * q;
                    const int64_t off = (int64_t)col[u] * D.ldb + 4 * v;
                    b[u][q] = (col[u] >= 0 && v < nv)
                                  ? ld_braw<BF16, HINT>(static_cast<const unsigned char*>(D.B) +
                                                            off * (BF16 ? 2 : 4), pol.last)
                                  : braw_zero<BF16>();
                }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < VPL; ++q) acc[q] = f4_fma(val[u], widen(b[u][q]), acc[q]);
        }
    }
}

template <int L, int VPL>
__device__ __forceinline__ void group_reduce(float4 (&acc)[VPL])
{
#pragma unroll
    for (int o = L; o < 32; o <<= 1)
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, o);
            acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, o);
            acc[q].z += __shfl_xor_sync(0xffffffffu, acc[q].z, o);
            acc[q].w += __shfl_xor_sync(0xffffffffu, acc[q].w, o);
        }
}

// split-row delivery out of line (rare): keeps the inlined row flush of the stream path small
template <int VPL, bool HINT>
__device__ __noinline__ void deliver_split_row(const ExecDesc& D, int32_t row, int32_t s, int32_t c,
                                               float4 a0, float4 a1, int lane, uint64_t pol_first)
{
    const int nv = D.K >> 2;
    const int32_t np = __ldg(D.split_np + s);
    const int32_t piece = c - __ldg(D.split_base + s);
    float* slot0 = D.slots + (int64_t)__ldg(D.split_slot + s) * D.K;
    const int v0 = lane, v1 = lane + 32;
    if (v0 < nv) __stcg(reinterpret_cast<float4*>(slot0 + (int64_t)piece * D.K + 4 * v0), a0);
    if (VPL > 1 && v1 < nv) __stcg(reinterpret_cast<float4*>(slot0 + (int64_t)piece * D.K + 4 * v1), a1);
    __threadfence();
    __syncwarp();
    int old = 0;
    if (lane == 0) old = atomicAdd(D.split_cnt + s, 1);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old != np - 1) return;
    __threadfence();
    float* crow = D.C + (int64_t)row * D.ldc;
#pragma unroll
    for (int q = 0; q < VPL; ++q) {
        const int v = lane + 32 * q;
        if (v < nv) {
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int p = 0; p < np; ++p)
                sum = f4_add(sum, __ldcg(reinterpret_cast<const float4*>(slot0 + (int64_t)p * D.K + 4 * v)));
            st_c4<HINT>(crow + 4 * v, sum, pol_first);
        }
    }
    if (lane == 0) atomicExch(D.split_cnt + s, 0);
}

// ---------------------------------------------------------------------------------------------
// residual chunks with K <= 256: decoded chunk in shared memory, gathers through a register ring
// ---------------------------------------------------------------------------------------------
// A chunk holds at most 3W/2 merge items (boundaries snap by less than W/2), so its rows and its
// nonzero stream fit in `cap` entries.  Per warp, shared memory holds the decoded chunk: the
// nonzeros as (column, value) pairs (padded by the ring depth), and per row its id, split id,
// first and past-last stream positions and first residual index.
constexpr int kRing = 8;  // gathered rows in flight per warp (K <= 128; 4 for K <= 256)

struct StageGeom {
    int cap;         // capacity of the chunk's stream and of its row arrays
    int rows_off;    // byte offset of the row arrays (after cap + kRing (col, val) pairs)
    int warp_bytes;  // shared memory of one warp, a multiple of 128
};

__host__ __device__ inline StageGeom stage_geom(int K, bool bf16, int W)
{
    (void)K;
    (void)bf16;
    StageGeom g;
    g.cap = ((3 * W) / 2 + 32 + 31) & ~31;
    g.rows_off = 8 * (g.cap + kRing);
    g.warp_bytes = (g.rows_off + 16 * (g.cap + 1) + 8 * g.cap + 127) & ~127;
    return g;
}

// the staged stream path serves K <= 256 (at most two 4-column vectors per lane)
__host__ __device__ inline bool staged_path(int L, int VPL) { return VPL <= 2; }

__device__ __forceinline__ uint32_t dynamic_smem_bytes()
{
    uint32_t r;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
    return r;
}

// Row metadata of up to 32 consecutive residual-list rows of a chunk, one row per lane, with the
// rows' positions in the chunk's stream of nonzeros (rows clipped to the chunk's merge range).
struct RowWin {
    int64_t kb;     // first row of the window
    int64_t base;   // stream position of the window's first row
    int64_t total;  // stream position after the window
    int32_t row;    // original row id (-1 past the chunk's last row)
    int32_t split;  // split id of the row or -1
    int64_t zoff;   // residual index of the row's first nonzero inside the chunk
    int32_t n;      // nonzeros of the row inside the chunk
    int64_t cum;    // stream position of the row's first nonzero
};

__device__ __forceinline__ void load_win(const ExecDesc& D, RowWin& w, int64_t kb, int64_t base,
                                         int64_t kL, int64_t b0, int64_t b1, int lane)
{
    w.kb = kb;
    w.base = base;
    const int64_t k = kb + lane;
    int32_t n = 0;
    w.row = -1;
    w.split = -1;
    w.zoff = 0;
    if (k <= kL) {
        const int32_t i = __ldg(D.rl_rows + k);
        const int64_t s = __ldg(D.rl_start + k), e = __ldg(D.rl_start + k + 1);
        const int64_t xs = b0 > s ? b0 : s;
        const int64_t xe = b1 < e - 1 ? b1 : e - 1;
        n = xe > xs ? (int32_t)(xe - xs) : 0;
        if (i >= 0 && i < D.m) {
            w.row = i;
            w.split = __ldg(D.row_split + i);
            w.zoff = (int64_t)__ldg(D.res_rowptr + i) + (xs - s);
            if (w.zoff < 0 || w.zoff + n > D.n_res) n = 0, w.row = -2;  // guard: corrupt plan
        } else {
            w.row = -2;
        }
    }
    w.n = n;
    int32_t inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    w.cum = base + inc - n;
    w.total = base + __shfl_sync(0xffffffffu, inc, 31);
}

// The streamed inner loop.  FULL: every lane holds VPL whole vectors (K == 128 * VPL), so no
// per-lane width test; HOT: the planner's hot-row map picks each gather's L2 policy.
template <int VPL, bool BF16, bool HINT, bool FULL, bool HOT>
__device__ __forceinline__ void stream_rows(const ExecDesc& D, int32_t c, int lane, const int2* ent,
                                            int tot_pad, int nr, const int32_t* rrow,
                                            const int32_t* rsplit, const int32_t* rend,
                                            const Policies& pol)
{
    const int nv = D.K >> 2;
    constexpr int VB = BF16 ? 8 : 16;  // bytes of one 4-column vector
    const unsigned char* const Bl = reinterpret_cast<const unsigned char*>(D.B) + VB * lane;
    const uint64_t ldb_bytes = (uint64_t)D.ldb * (BF16 ? 2 : 4);
    float* const Cp = D.C;
    const int64_t ldc = D.ldc;

    float4 acc[VPL];
#pragma unroll
    for (int q = 0; q < VPL; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    int r = 0;
    int next_end = rend[0];
    auto flush = [&]() {  // deliver row r, move to row r + 1
        const int32_t i = rrow[r];
        const int32_t sp = rsplit[r];
        if (i >= 0) {
            if (sp < 0) {
                float* crow = Cp + (int64_t)i * ldc;
#pragma unroll
                for (int q = 0; q < VPL; ++q) {
                    const int v = lane + 32 * q;
                    if (FULL || v < nv) st_c4<HINT>(crow + 4 * v, acc[q], pol.first);
                }
            } else {
                deliver_split_row<VPL, HINT>(D, i, sp, c, acc[0], acc[VPL > 1 ? VPL - 1 : 0], lane, pol.first);
            }
        } else if (i == -2 && lane == 0) {
            atomicOr(D.status, kStatusInternal);
        }
#pragma unroll
        for (int q = 0; q < VPL; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        ++r;
        next_end = rend[r];
    };

    constexpr int U = VPL == 1 ? kRing : kRing / 2;
    BRaw<BF16> b[U][VPL];
    float w[U];
    auto gather = [&](int2 e, BRaw<BF16> (&dst)[VPL], float& wv) {
        // padding entries point at a real row with value 0: no test needed here.  With the hot
        // map, bit 31 of the column id marks a hot row (set when the chunk was decoded).
        const uint32_t col = HOT ? ((uint32_t)e.x & 0x7fffffffu) : (uint32_t)e.x;
        const unsigned char* row = Bl + (uint64_t)col * ldb_bytes;
        uint64_t pl = pol.last;
        if (HOT) pl = e.x < 0 ? pol.last : pol.first;
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            if (FULL || lane + 32 * q < nv) dst[q] = ld_braw<BF16, HINT>(row + 32 * VB * q, pl);
            else dst[q] = braw_zero<BF16>();
        }
        wv = __int_as_float(e.y);
    };
#pragma unroll
    for (int u = 0; u < U; ++u) gather(ent[u], b[u], w[u]);
    for (int j0 = 0; j0 < tot_pad; j0 += U) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int P = j0 + u;
            while (P >= next_end) flush();
            const int2 e = ent[P + U];
#pragma unroll
            for (int q = 0; q < VPL; ++q) acc[q] = f4_fma(w[u], widen(b[u][q]), acc[q]);
            gather(e, b[u], w[u]);
        }
    }
    while (r < nr) flush();  // rows ending at or after the last item (and the last row)
}

template <int VPL, bool BF16, bool HINT>
__device__ void residual_chunk_staged(const ExecDesc& D, int32_t c, int lane, unsigned char* wbase,
                                      const Policies& pol)
{
    const StageGeom G = stage_geom(D.K, BF16, D.chunk_nnz);
    const int64_t b0 = __ldg(D.chunk_b + c), b1 = __ldg(D.chunk_b + c + 1);
    const int64_t k0 = __ldg(D.chunk_k0 + c);
    // last row with a merge item in [b0, b1): the row holding b1 - 1
    int64_t kL = (c + 1 < D.n_chunks) ? (int64_t)__ldg(D.chunk_k0 + c + 1) : (int64_t)D.n_rl - 1;
    if (kL > k0 && (int64_t)__ldg(D.rl_start + kL) >= b1) --kL;
    const int nr = (int)(kL - k0 + 1);
    if (k0 < 0 || kL >= D.n_rl || kL < k0 || b1 <= b0 || nr > G.cap) {
        if (lane == 0) atomicOr(D.status, kStatusInternal);
        return;
    }
    int2* const ent = reinterpret_cast<int2*>(wbase);  // (col, value bits), cap + kRing
    int32_t* const rrow = reinterpret_cast<int32_t*>(wbase + G.rows_off);
    int32_t* const rsplit = rrow + (G.cap + 1);
    int32_t* const rbeg = rsplit + (G.cap + 1);
    int32_t* const rend = rbeg + (G.cap + 1);
    int64_t* const rzoff = reinterpret_cast<int64_t*>(rend + (G.cap + 1));

    // ---- decode the chunk's rows: ids, split ids, stream positions, first residual index ----
    int total = 0;
    {
        RowWin w;
        int64_t kb = k0, base = 0;
        for (;;) {
            load_win(D, w, kb, base, kL, b0, b1, lane);
            const int r = (int)(kb - k0) + lane;
            if (kb + lane <= kL) {
                rrow[r] = w.row;
                rsplit[r] = w.split;
                rbeg[r] = (int32_t)w.cum;
                rend[r] = (int32_t)(w.cum + w.n);
                rzoff[r] = w.zoff;
            }
            base = w.total;
            if (kb + 32 > kL) break;
            kb += 32;
        }
        total = (int)base;
        if (lane == 0) rend[nr] = 0x7fffffff;  // sentinel after the last row
    }
    if (total < 0 || total > G.cap) {
        if (lane == 0) atomicOr(D.status, kStatusInternal);
        return;
    }
    __syncwarp();
    // ---- the nonzero stream as (col, value) entries; every load issued before any store ----
    const int tot_pad = (total + kRing - 1) / kRing * kRing;
    int32_t last_col = 0;
    for (int P0 = 0; P0 < total; P0 += 128) {
        int32_t cc[4];
        float vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int P = P0 + 32 * u + lane;
            cc[u] = 0;
            vv[u] = 0.f;
            if (P < total) {
                int lo = 0, hi = nr;  // the row holding P: largest r with rbeg[r] <= P
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (rbeg[mid] <= P) lo = mid;
                    else hi = mid;
                }
                const int64_t z = rzoff[lo] + (P - rbeg[lo]);
                if (z >= 0 && z < D.n_res) {
                    cc[u] = ld_stream_i32<HINT>(D.res_col + z, pol.first);
                    vv[u] = ld_stream_f32<HINT>(D.res_val + z, pol.first);
                } else {
                    atomicOr(D.status, kStatusInternal);
                }
            }
        }
        uint32_t hw[4];  // hot-map words of the columns (independent loads as well)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int P = P0 + 32 * u + lane;
            if ((unsigned)cc[u] >= (unsigned)D.n) {  // guard: never gather outside B
                if (P < total) atomicOr(D.status, kStatusInternal);
                cc[u] = 0;
                vv[u] = 0.f;
            }
            hw[u] = (D.hot && P < total) ? __ldg(D.hot + (cc[u] >> 5)) : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int P = P0 + 32 * u + lane;
            if (P < total) {
                const int32_t hotbit = (D.hot && ((hw[u] >> (cc[u] & 31)) & 1u)) ? (int32_t)0x80000000 : 0;
                ent[P] = make_int2(cc[u] | hotbit, __float_as_int(vv[u]));
            }
        }
    }
    __syncwarp();
    if (total > 0) last_col = ent[total - 1].x;
    // padding: the last real row again with value 0 (a cached load, no branch in the loop)
    for (int P = total + lane; P < tot_pad + kRing; P += 32) ent[P] = make_int2(last_col, 0);
    __syncwarp();

    const bool full = D.K == 128 * VPL;
    if (D.hot) {
        if (full) stream_rows<VPL, BF16, HINT, true, true>(D, c, lane, ent, tot_pad, nr, rrow, rsplit, rend, pol);
        else stream_rows<VPL, BF16, HINT, false, true>(D, c, lane, ent, tot_pad, nr, rrow, rsplit, rend, pol);
    } else {
        if (full) stream_rows<VPL, BF16, HINT, true, false>(D, c, lane, ent, tot_pad, nr, rrow, rsplit, rend, pol);
        else stream_rows<VPL, BF16, HINT, false, false>(D, c, lane, ent, tot_pad, nr, rrow, rsplit, rend, pol);
    }
}

// one merge-path chunk c of the residual (one warp)
template <int L, int VPL, bool BF16, bool HINT>
__device__ void residual_chunk(const ExecDesc& D, int32_t c, int lane, const Policies& pol)
{
    const int64_t b0 = __ldg(D.chunk_b + c), b1 = __ldg(D.chunk_b + c + 1);
    int64_t k = __ldg(D.chunk_k0 + c);
    int64_t x = b0;
    while (x < b1) {
        // guards: a corrupt plan sets the status word and stops instead of faulting
        if (k < 0 || k >= D.n_rl) {
            if (lane == 0) atomicOr(D.status, kStatusInternal);
            return;
        }
        const int32_t i = __ldg(D.rl_rows + k);
        const int64_t s = __ldg(D.rl_start + k), e = __ldg(D.rl_start + k + 1);
        const int64_t zrow = (i >= 0 && i < D.m) ? __ldg(D.res_rowptr + i) : -1;
        const int64_t xe = b1 < e - 1 ? b1 : e - 1;  // nonzero merge items of this row in chunk
        if (zrow < 0 || x < s || e <= s || zrow + (xe - s) > D.n_res) {
            if (lane == 0) atomicOr(D.status, kStatusInternal);
            return;
        }
        float4 acc[VPL];
#pragma unroll
        for (int q = 0; q < VPL; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        gather_accumulate<L, VPL, BF16, HINT>(D, zrow + (x - s), zrow + (xe - s), acc, lane, pol);
        group_reduce<L, VPL>(acc);
        deliver_row<L, VPL, HINT>(D, i, c, false, acc, lane, pol.first);
        if (e - 1 < b1) {  // the row's end item is in this chunk: move on
            x = e;
            ++k;
        } else {
            x = b1;
        }
    }
}


__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Residual chunks in work-list order, one per warp (no CTA barrier); with K <= 256 each of the CTA's
// `warps` calling warps has a staging area in smem_raw.
template <int L, int VPL, bool BF16, bool HINT>
__device__ __forceinline__ void residual_phase(const ExecDesc* descs, const int32_t* queue, const int32_t* queue_desc,
                                               int64_t n_items, int32_t* ctrl, const ExecDesc& d0, int lane,
                                               int warp, unsigned char* smem_raw, int warps, const Policies& pol,
                                               unsigned long long* clk)
{
    for (;;) {
        int64_t u = 0;
        if (lane == 0) u = atomicAdd(ctrl + 3, 1);
        u = __shfl_sync(0xffffffffu, u, 0);
        const int64_t t = u / kExecWarps;
        if (t >= n_items) break;
        const int32_t it = __ldg(queue + t);
        const ExecDesc& D = descs ? descs[queue_desc ? __ldg(queue_desc + t) : 0] : d0;
        if (it < D.n_dwin) continue;
        const int64_t c = (int64_t)(it - D.n_dwin) * kExecWarps + (u % kExecWarps);
        if (c >= D.n_chunks) continue;
        // K <= 256: the streamed path, which needs the shared memory the host sized for it; this
        // warp's slice follows the descriptor's chunk geometry (plans of one batched launch may
        // differ in W; nothing in it outlives a chunk)
        if constexpr (VPL <= 2) {
            const StageGeom SG = stage_geom(D.K, BF16, D.chunk_nnz);
            if (dynamic_smem_bytes() < (uint32_t)(warps * SG.warp_bytes)) {
                if (lane == 0) atomicOr(D.status, kStatusInternal);  // guard: misconfigured launch
                continue;
            }
            residual_chunk_staged<(VPL <= 2 ? VPL : 2), BF16, HINT>(D, (int32_t)c, lane,
                                                                    smem_raw + warp * SG.warp_bytes, pol);
        } else {
            residual_chunk<L, VPL, BF16, HINT>(D, (int32_t)c, lane, pol);
        }
        if (clk && lane == 0) atomicMax(clk + 2, global_ns());
    }
}

}  // namespace ns
