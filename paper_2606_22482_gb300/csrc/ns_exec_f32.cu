// ns_exec_f32.cu -- the persistent kernel of FP32 plans that keep their dense tiles' planes (K <= 256): the
// dense item on the 5th-generation tensor cores.
//
// FP32 operands run as three BF16 pieces each, x = x0 + x1 + x2 (x0 by truncation, so that it never
// overflows; x1 and x2 rounded to nearest; 24 bits in all), and the product keeps the six largest
// terms (what is left out is below 2^-22 of |a b|: a truncated x0 leaves x1 up to 2^-7 of x): a0 b0 | a0 b1 + a1 b0 | a1 b1 + a0 b2 + a2 b0, in three accumulators X0 | X1 | X2 by
// size.  The tensor pipe's FP32 accumulation is not round-to-nearest, so a tile's a0 b0 starts a
// fresh X0 (two alternate), which is added to the window's sum in registers with an ordinary FP32
// add; X1 and X2, 2^-8 and 2^-16 of the result, accumulate over the window.
//
// The MMA is posed transposed, D (features x TM rows) += B[cols, :]^T (features x TK) * A_tile^T:
//   * the gathered B rows are the first operand and live in tensor memory, one feature per lane: a
//     producer warp copies its 32 features (128 bytes) of the tile's TK rows into shared memory with
//     cp.async, and each lane splits its feature's values in registers and writes the pieces with
//     tcgen05.st;
//   * the A tile's three planes were laid out at plan time in the K-major layout of the second
//     operand (dtile_x) and come as one bulk copy of 6 TM TK bytes, four tiles ahead.  Planes are
//     stacked along N, so b0 meets a1 and a2, and b1 meets a0 and a1, in one MMA each: eight MMAs a
//     tile instead of twelve of N = 64.
// One CTA per SM: warps 0-3 add X0 to the window sums (32 features a warp), warps 4-7 and 8-11 produce
// every other tile (two tiles of copies in flight each, four tiles in tensor memory), warp 12
// issues the MMAs.  The sums then meet the rows' absorbed residual in a shared TM x K tile and the
// rows are delivered as in the other items.
//
// What bounds it (attention mask 32768, TM 64, TK 32, K 128: 834 -> 131 us an execute against the
// mma.sync item with a three-term TF32 split; error against 64 bits 2.7e-7 -> 1.3e-7): 512 windows
// on 152 SMs are 3.4 rounds of about 33 us; a tile takes about 0.8 us, its eight small MMAs and the
// producers' splits about half of that each way, and a window's delivery adds 4 us.  Traffic (240 MB
// of planes from HBM) and the tensor pipe (31 GFLOP of pieces) would each allow about 35 us.
// Other widths and tiles, against the mma.sync item (us an execute): mask 8192, TM 16, TK 16, K 8 127 -> 86,
// K 32 126 -> 86, K 256 258 -> 149; TM 64, TK 32, K 8 102 -> 29, K 64 160 -> 29; RMAT 2^15, TM 16, TK 16, tau 32,
// K 8 to 32, where the residual decides, 148 on both sides: nowhere slower, so K alone is the rule.
// Also tried: all operands of an MMA computed by the issuing lane alone (100 cycles an MMA), loads of
// one feature a lane (32 instructions a tile and warp, 90 cycles each): 213 to 276 us.
//
// Every wait is bounded: one that gives up sets the plan's timeout status and the CTA takes no more
// dense items; its copies and MMAs are waited for (again bounded) before tensor memory is freed.
#include "ns_internal.cuh"
#include "ns_mem.cuh"
#include "ns_ptx.cuh"

#include "ns_residual.cuh"
#include "ns_dense.cuh"
#include "ns_dense_tc.cuh"

namespace ns {

constexpr int kTsWarps = 13;                 // warps 0-3 drain, 4-11 produce, 12 issues the MMAs; all deliver
constexpr int kTsThreads = kTsWarps * 32;
constexpr int kTsRing = 8;                   // A-tile stages in shared memory (copies run four tiles ahead)
constexpr int kTsOps = 4;                    // first-operand stages in tensor memory
constexpr int kTsTmemCols = 512;
constexpr int kTsX1 = 128;                   // X0: two accumulators of TM <= 64 columns; then X1, X2 side by side
constexpr int kTsOperandCol = 256;           // kTsOps stages of three pieces of TK / 2 <= 16 columns
// barriers: full_a[8] (a plane copy landed), full_b[4] (four producer warps stored a tile), empty[4] (a
// tile's MMAs completed), acc_full[2], acc_empty[2] (four drain warps), drain
constexpr int kTsFullA = 0, kTsFullB = 8, kTsEmpty = 12, kTsAccFull = 16, kTsAccEmpty = 18, kTsDrain = 20, kTsBars = 21;

struct TsGeom {
    int FB;          // feature blocks of 128, one after another
    int plane;       // bytes of one plane of an A tile
    int off_b;       // gathered B rows as they come (FP32): two groups x two stages of TK x 128 features
    int off_c;       // TM x cs_stride FP32 result tile
    int cs_stride;
    int total;
};

__host__ __device__ inline TsGeom ts_geom(int K, int TM, int TK)
{
    TsGeom g;
    g.FB = (K + 127) / 128;
    g.plane = TM * TK * 2;
    g.cs_stride = K + 4;
    const int ring = kTsRing * 3 * g.plane, cs = TM * g.cs_stride * 4;
    g.off_b = ring;
    g.off_c = ring + 4 * TK * 512;
    g.total = g.off_c + cs;
    return g;
}

struct TsState {
    uint64_t* bars;
    uint32_t* copies;  // plane copies issued to each ring stage (shared memory)
    uint32_t tmem;
    uint32_t g;  // tiles this CTA has multiplied (a tile counts once per feature block)
    bool ok;     // false once a bounded wait gave up
};

// The four MMAs of 16 compacted columns (first operand in tensor memory, second in shared memory),
// issued by one elected lane of a converged warp.  The whole warp computes the operands: code of one
// lane alone makes the compiler broadcast every descriptor through the uniform registers, at about
// 100 cycles an MMA.
__device__ __forceinline__ void ts_mma4(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t b0, uint32_t b1, uint32_t b2,
                                        uint64_t a0, uint64_t a1, uint32_t i1, uint32_t i2, uint32_t more_x, uint32_t more_0)
{
    asm volatile("{\n\t.reg .pred e, px, p0, one;\n\telect.sync _|e, 0xffffffff;\n\t"
                 "setp.ne.b32 px, %10, 0;\n\tsetp.ne.b32 p0, %11, 0;\n\tsetp.eq.b32 one, %8, %8;\n\t"
                 "@e tcgen05.mma.cta_group::1.kind::f16 [%1], [%3], %7, %9, px;\n\t"   // X1 += a1 b0, X2 += a2 b0
                 "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%3], %6, %8, p0;\n\t"   // X0  = a0 b0 of this tile
                 "@e tcgen05.mma.cta_group::1.kind::f16 [%1], [%4], %6, %9, one;\n\t"  // X1 += a0 b1, X2 += a1 b1
                 "@e tcgen05.mma.cta_group::1.kind::f16 [%2], [%5], %6, %8, one;\n\t}" // X2 += a0 b2
                 :: "r"(x0), "r"(x1), "r"(x2), "r"(b0), "r"(b1), "r"(b2), "l"(a0), "l"(a1), "r"(i1), "r"(i2), "r"(more_x),
                    "r"(more_0) : "memory");
}

// arrive on both barriers when every MMA that the elected lane issued before has completed
__device__ __forceinline__ void ts_commit2(uint32_t bar0, uint32_t bar1)
{
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
                 "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
                 "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%1];\n\t}"
                 :: "r"(bar0), "r"(bar1) : "memory");
}

// 8 columns of this lane's row of tensor memory
__device__ __forceinline__ void ts_st8(uint32_t taddr, const uint32_t (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

__device__ __forceinline__ void ts_bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

template <bool HINT>
__device__ bool ts_window_product(const ExecDesc& D, int32_t w, unsigned char* smem, const TsGeom& G, TsState& S,
                                  const Policies& pol)
{
    const int TM = D.TM, TK = D.TK;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t t0 = __ldg(D.win_dptr + w);
    const int T = __ldg(D.win_dptr + w + 1) - t0;
    uint64_t* const bars = S.bars;
    float* const Cs = reinterpret_cast<float*>(smem + G.off_c);
    if (T <= 0) {  // a dense window holds at least one tile; guard against a corrupt plan
        if (threadIdx.x == 0) atomicOr(D.status, kStatusInternal);
        for (int q = threadIdx.x; q < TM * G.cs_stride; q += kTsThreads) Cs[q] = 0.f;
        __syncthreads();
        return true;
    }
    const int J = G.FB * T;  // tiles to multiply, feature block by feature block
    const uint32_t g0 = S.g;
    const uint32_t a_bytes = 3u * (uint32_t)G.plane;
    const int acols = TK / 2;  // tensor-memory columns of one piece of a tile
    bool ok = true;
    if (warp >= 4 && warp < 12) {
        // ---- producers: group 0 (warps 4-7) takes the even tiles, group 1 the odd ones ----
        const int grp = (warp - 4) >> 2, pw = warp & 3;
        const uint32_t lanes = (uint32_t)(32 * pw) << 16;
        const bool leader = pw == 0 && lane == 0;
        // (the descriptor's fields once: the loop's memory clobbers would read them again each time)
        const int32_t n = D.n, K = D.K;
        int32_t* const status = D.status;
        const int64_t ldb_bytes = D.ldb * 4;
        const unsigned char* const Bw = reinterpret_cast<const unsigned char*>(D.B) + 128 * pw + 16 * (lane & 7);
        // this warp's 32 features of a stage: [column][feature]
        float* const raw = reinterpret_cast<float*>(smem + G.off_b + grp * 2 * TK * 512 + pw * TK * 128);
        const int32_t* const cols = D.dtile_cols + (int64_t)t0 * TK + lane;
        const unsigned char* const tiles = reinterpret_cast<const unsigned char*>(D.dtile_x) + (int64_t)t0 * a_bytes;
        auto copy_a = [&](int j) {
            const uint32_t g = g0 + (uint32_t)j;
            const int tile = j < T ? j : j - T;  // (at most two feature blocks)
            ts_bulk_copy(smem + (g % kTsRing) * a_bytes, tiles + (int64_t)tile * a_bytes, a_bytes,
                         bars + kTsFullA + g % kTsRing);
            S.copies[g % kTsRing] = g / kTsRing + 1;
        };
        if (leader) {
            if (grp < J) copy_a(grp);
            if (grp + 2 < J) copy_a(grp + 2);
        }
        auto ids = [&](int j) -> int32_t {
            int32_t id = -1;  // (in place, two tiles before its use: a plain load would be moved down to it)
            asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q ld.global.nc.s32 %0, [%1];\n\t}"
                         : "+r"(id) : "l"(cols + (int64_t)(j < T ? j : j - T) * TK), "r"((int)(j < J && lane < TK)));
            return id;
        };
        // Tile j's B rows into stage b by 16-byte copies: lane l copies piece l % 8 of the warp's 128
        // bytes of columns l / 8, l / 8 + 4, ...; columns past the window's last and features past the
        // width become zeros.  (Loads of one feature a lane would be 32 instructions a tile and warp,
        // and that many cannot be in flight: 90 cycles each.)
        auto load = [&](int j, int32_t id, int b) {
            if (id >= n) atomicOr(status, kStatusInternal);  // guard: corrupt plan (no copy is made)
            const int32_t col = id >= 0 && id < n ? id : -1;
            const bool in = j < J && (j < T ? 0 : 128) + 32 * pw + 4 * (lane & 7) < K;
            const unsigned char* const src = Bw + (j < T ? 0 : 512);
            float* const dst = raw + b * TK * 128 + (lane >> 3) * 32 + 4 * (lane & 7);
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                const int32_t cc = __shfl_sync(0xffffffffu, col, c + (lane >> 3));
                if (c < TK) {
                    const bool on = in && cc >= 0;
                    cp_async16<HINT>(dst + c * 32, src + (on ? (int64_t)cc * ldb_bytes : 0), on, pol.last);
                }
            }
            cp_async_commit();
        };
        auto store = [&](int j, int b) {
            const uint32_t g = g0 + (uint32_t)j, s = g % kTsOps;
            if (ok && g >= kTsOps && !mbar_wait(bars + kTsEmpty + s, (g / kTsOps - 1u) & 1u)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            // the wait above also freed the A stage of tile j - 4, which tile j + 4 takes
            if (leader && ok && j + 4 < J) copy_a(j + 4);
            cp_async_wait<1>();  // this stage's copies have landed (the other's may be under way)
            __syncwarp();
            tc_fence_after();
            const float* const v = raw + b * TK * 128 + lane;
            const uint32_t base = S.tmem + lanes + kTsOperandCol + s * (uint32_t)(3 * acols);
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                if (16 * ks < TK) {
                    float x[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) x[q] = v[(16 * ks + q) * 32];
                    uint32_t p0[8], p1[8], p2[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) split3(x[2 * q], x[2 * q + 1], p0[q], p1[q], p2[q]);
                    ts_st8(base + 8 * ks, p0);
                    ts_st8(base + acols + 8 * ks, p1);
                    ts_st8(base + 2 * acols + 8 * ks, p2);
                }
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();  // (the stage is read: its next copies may be issued)
            if (lane == 0) mbar_arrive(bars + kTsFullB + s);
        };
        int32_t ia = ids(grp), ib = ids(grp + 2);
        load(grp, ia, 0);
        load(grp + 2, ib, 1);
        ia = ids(grp + 4);
        ib = ids(grp + 6);
        for (int j = grp; j < J; j += 4) {
            store(j, 0);
            load(j + 4, ia, 0);
            ia = ids(j + 8);
            if (j + 2 < J) {
                store(j + 2, 1);
                load(j + 6, ib, 1);
                ib = ids(j + 10);
            }
        }
        cp_async_wait<0>();
        ok = __all_sync(0xffffffffu, ok);
    } else if (warp == 12) {
        // ---- MMAs ----
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);  // + (N / 8) << 17
        const uint32_t n1 = (uint32_t)(TM >> 3) << 17, n2 = (uint32_t)(TM >> 2) << 17;
        const uint32_t tmem = __shfl_sync(0xffffffffu, S.tmem, 0), ring = smem_u32(smem), bar = smem_u32(bars);
        for (int j = 0; j < J; ++j) {
            const uint32_t g = g0 + (uint32_t)j, s = g & 1u, o = g % kTsOps;
            if (ok && !mbar_wait(bars + kTsFullA + g % kTsRing, (g / kTsRing) & 1u)) ok = false;
            if (ok && !mbar_wait(bars + kTsFullB + o, (g / kTsOps) & 1u)) ok = false;
            if (ok && g >= 2 && !mbar_wait(bars + kTsAccEmpty + s, ((g >> 1) - 1u) & 1u)) ok = false;
            // X1 and X2 of the feature block before have been read
            if (ok && j == T && !mbar_wait(bars + kTsAccEmpty + (s ^ 1u), ((g - 1u) >> 1) & 1u)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            if (ok) {
                const uint32_t first = j == 0 || j == T ? 1u : 0u;  // of a feature block
                const uint32_t tb = tmem + kTsOperandCol + o * (uint32_t)(3 * acols);
                const uint32_t x0 = tmem + s * (uint32_t)TM, x1 = tmem + kTsX1;
                const uint64_t a0 = tc_desc(ring + (g % kTsRing) * a_bytes, 128, TK * 16);
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    if (16 * ks < TK) {  // (addresses in a descriptor count 16 bytes)
                        const uint64_t ak = a0 + 16 * ks;
                        const uint32_t b0 = tb + 8 * ks;
                        ts_mma4(x0, x1, x1 + (uint32_t)TM, b0, b0 + acols, b0 + 2 * acols, ak,
                                ak + (uint64_t)(G.plane >> 4), idesc | n1, idesc | n2, ks > 0 || !first, ks > 0);
                    }
                }
            }
            ts_commit2(bar + 8 * (kTsEmpty + o), bar + 8 * (kTsAccFull + s));
            __syncwarp();
        }
    } else {
        // ---- the window's sums ----
        float acc[64];
#pragma unroll
        for (int q = 0; q < 64; ++q) acc[q] = 0.f;
        const uint32_t lanes = (uint32_t)(32 * warp) << 16;
        const int32_t Kw = D.K;
        for (int j = 1; j <= J; ++j) {
            const uint32_t g = g0 + (uint32_t)(j - 1), s = g & 1u;
            if (ok && !mbar_wait(bars + kTsAccFull + s, (g >> 1) & 1u)) ok = false;
            __syncwarp();
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 16) {
                if (c0 < TM) {
                    uint32_t r[16];
                    tc_ld16(S.tmem + lanes + s * (uint32_t)TM + c0, r);
#pragma unroll
                    for (int q = 0; q < 16; ++q) acc[c0 + q] += __uint_as_float(r[q]);
                }
            }
            if (j == T || j == J) {  // a feature block is complete (with it X1 and X2)
#pragma unroll
                for (int c0 = 0; c0 < 64; c0 += 16) {
                    if (c0 < TM) {
                        uint32_t r[16], q2[16];
                        tc_ld16(S.tmem + lanes + kTsX1 + TM + c0, q2);
                        tc_ld16(S.tmem + lanes + kTsX1 + c0, r);
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            acc[c0 + q] += __uint_as_float(r[q]) + __uint_as_float(q2[q]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + kTsAccEmpty + s);
            if (j == T || j == J) {
                const int f = (j == T ? 0 : 128) + 32 * warp + lane;
#pragma unroll
                for (int q = 0; q < 64; ++q) {
                    if (q < TM && f < Kw) Cs[q * G.cs_stride + f] = acc[q];
                    acc[q] = 0.f;
                }
            }
        }
    }
    S.g = g0 + (uint32_t)J;
    const int all_ok = __syncthreads_and(ok ? 1 : 0);
    if (!all_ok) {
        if (threadIdx.x == 0) atomicOr(D.status, kStatusTimeout);
        S.ok = false;
        return false;
    }
    return true;
}

template <int VPL, bool HINT>
__global__ void __launch_bounds__(kTsThreads, 1) k_exec_f32(const ExecDesc* __restrict__ descs,
                                                                      const int32_t* __restrict__ queue,
                                                                      const int32_t* __restrict__ queue_desc,
                                                                      int64_t n_items, int32_t* ctrl, int32_t res_warps,
                                                                      const __grid_constant__ ExecDesc d0)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int32_t s_ticket;
    __shared__ int4 s_rowmeta[64];  // a dense window's rows (TM <= 64)
    __shared__ __align__(8) uint64_t s_bars[kTsBars];
    __shared__ uint32_t s_tmem, s_copies[kTsRing];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Policies pol{0, 0};
    if (HINT) pol = make_policies();
    unsigned long long* const clk = descs ? nullptr : d0.class_clock;  // single-plan launches only
    if (clk && threadIdx.x == 0) atomicMin(clk, global_ns());
    int32_t* const status0 = descs ? descs[0].status : d0.status;
    // ---- barriers and tensor memory ----
    TsState S;
    S.bars = s_bars;
    S.copies = s_copies;
    S.g = 0;
    S.ok = true;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kTsRing; ++i) s_copies[i] = 0;
        for (int i = 0; i < kTsBars; ++i)
            mbar_init(s_bars + i, i >= kTsFullB && i < kTsEmpty ? 4 : (i >= kTsAccEmpty && i < kTsDrain ? 4 : 1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&s_tmem)), "r"(kTsTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    S.tmem = s_tmem;
    // ---- phase 1: dense windows, one CTA each, taken in work-list order ----
    for (;;) {
        if (threadIdx.x == 0) s_ticket = atomicAdd(ctrl + 0, 1);
        __syncthreads();
        const int64_t t = s_ticket;
        __syncthreads();
        if (t >= n_items) break;
        const int32_t it = __ldg(queue + t);
        const ExecDesc& D = descs ? descs[queue_desc ? __ldg(queue_desc + t) : 0] : d0;
        if (it >= D.n_dwin || !S.ok) continue;
        const TsGeom G = ts_geom(D.K, D.TM, D.TK);
        if (dynamic_smem_bytes() < (uint32_t)G.total || D.K > 256 || !D.dtile_x || D.TM % 16 || D.TM > 64 ||
            (D.TK != 16 && D.TK != 32)) {
            if (threadIdx.x == 0) atomicOr(D.status, kStatusInternal);  // guard: launch without the tile buffers
            continue;
        }
        const int32_t w = __ldg(D.dwin + it);
        dense_row_meta<kTsWarps>(D, it, w, s_rowmeta);  // (read while the product runs)
        if (ts_window_product<HINT>(D, w, smem_raw, G, S, pol))
            dense_deliver_rows<32, VPL, false, HINT, kTsWarps>(D, it, w, reinterpret_cast<float*>(smem_raw + G.off_c),
                                                              G.cs_stride, s_rowmeta, pol);
        if (clk && threadIdx.x == 0) atomicMax(clk + 1, global_ns());
    }
    // ---- the CTA's copies and MMAs have completed; tensor memory is freed ----
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && S.g > 0) {
        // (after a wait that gave up, plane copies may still be under way: at most one per stage)
        for (int i = 0; i < kTsRing; ++i)
            if (s_copies[i] > 0 && !mbar_wait(s_bars + kTsFullA + i, (s_copies[i] - 1u) & 1u) && status0)
                atomicOr(status0, kStatusTimeout);
    }
    __syncwarp();
    if (warp == 12 && S.g > 0) {  // the lane that issued the MMAs
        asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
                     "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
                     :: "r"(smem_u32(s_bars + kTsDrain)) : "memory");
        if (!mbar_wait(s_bars + kTsDrain, 0) && status0) atomicOr(status0, kStatusTimeout);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(S.tmem), "r"(kTsTmemCols) : "memory");
    // ---- phase 2: residual chunks ----
    if (warp < res_warps)
        residual_phase<32, VPL, false, HINT>(descs, queue, queue_desc, n_items, ctrl, d0, lane, warp, smem_raw, res_warps,
                                             pol, clk);
    end_launch(ctrl, d0, descs == nullptr);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
typedef void (*F32Kernel)(const ExecDesc*, const int32_t*, const int32_t*, int64_t, int32_t*, int32_t, ExecDesc);

static F32Kernel pick_f32(int K, bool hint)
{
    if (K <= 128) return hint ? k_exec_f32<1, true> : k_exec_f32<1, false>;
    return hint ? k_exec_f32<2, true> : k_exec_f32<2, false>;
}

// Dynamic shared memory, and the warps of a CTA that take residual chunks: all of them
// while their staging areas fit, never fewer than the four that always do.
static size_t f32_smem(int K, int TM, int TK, int W, int* res_warps)
{
    const int wb = stage_geom(K, false, W).warp_bytes;
    int rw = kTsWarps;
    while (rw > kExecWarps && (size_t)rw * wb > 216 * 1024) --rw;
    *res_warps = rw;
    const size_t d = (size_t)ts_geom(K, TM, TK).total, r = (size_t)rw * wb;
    return d > r ? d : r;
}

ns_status_t f32_prepare(int64_t n_items, int K, int TM, int TK, bool hint, int W, int* grid_out)
{
    F32Kernel kern = pick_f32(K, hint);
    int rw = 0, dev = 0;
    const size_t smem = f32_smem(K, TM, TK, W, &rw);
    NS_TRY(dense_prepare(reinterpret_cast<const void*>(kern), smem));
    NS_CUDA_TRY(cudaGetDevice(&dev));
    int64_t g = num_sms(dev);  // one CTA per SM (tensor memory)
    if (g > n_items) g = n_items;
    *grid_out = (int)(g > 0 ? g : 1);
    return NS_OK;
}

ns_status_t f32_launch(const ExecDesc* descs, const int32_t* queue, const int32_t* queue_desc, int64_t n_items,
                       int32_t* ctrl, int K, int TM, int TK, bool hint, int W, int* grid_cache, cudaStream_t s,
                       const ExecDesc* d0)
{
    int grid = grid_cache ? *grid_cache : 0;
    if (grid == 0) NS_TRY(f32_prepare(n_items, K, TM, TK, hint, W, &grid));
    if (grid_cache) *grid_cache = grid;
    if (n_items == 0) return NS_OK;
    int rw = 0;
    const size_t smem = f32_smem(K, TM, TK, W, &rw);
    ExecDesc dv{};
    if (d0) dv = *d0;
    pick_f32(K, hint)<<<grid, kTsThreads, smem, s>>>(d0 ? nullptr : descs, queue, queue_desc, n_items, ctrl, rw, dv);
    NS_LAUNCH_CHECK();
    return NS_OK;
}

}  // namespace ns
