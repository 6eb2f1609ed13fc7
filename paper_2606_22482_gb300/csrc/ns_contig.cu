// ns_contig.cu -- residual-only plans: the contiguous-stream execute kernel (arXiv 2606.22482
// Sections 5.1 and 7).
//
// With tau_tile = inf the residual is A itself and the residual list is every row in order, so a
// merge-path chunk's nonzeros are one contiguous range of A and its rows are k0 .. kL.
//
// What bounds it: every nonzero gathers one B row (4 K or 2 K bytes) from L2 into an SM.  A kernel
// that only gathers the same column streams moves 21 TB/s (power-law graph of 2^20 nodes, 512-byte
// rows, 0.39 ms).  This one moves 12.8 TB/s there: the rest of the time goes to instructions around
// the gathers (53 per step of two nonzeros; row ends take most of what is not the product itself)
// and to the starts of chunks (about 10 us each, a chain of dependent loads).
//
// Split of the work: a lane owns 8 adjacent columns (32 bytes of FP32 in one 256-bit load, or 16
// bytes of BF16; FP32 off the 32-byte boundaries: 4 in each half of the row), so G = K / 8 lanes cover a row and the warp holds EPS = 32 / G lane groups.
// Each group is a stream of its own: the chunk's nonzeros are divided equally among the groups,
// each group walks its share in order and stores its own rows, so a row end costs no sum over the
// warp.  A row that straddles shares is put together at the end of the chunk: every share but the
// first one of such a row parks its part in shared memory and the row's first share adds the parts
// in order.  Sums therefore have a fixed order that depends only on the plan and K (a graph of a batch:
// and on how many chunks the graphs of its width have together, contig_coop).  Gathers run
// DEPTH steps ahead in a register ring, so a row crosses the L1 data pipe once; products are packed
// two columns to an instruction (fma.rn.f32x2, the same rounding as two fmaf).
//
// Measured against the kernel before it (one nonzero per warp step, 16-byte lanes, an 8-deep ring
// in shared memory at K = 128; lane groups summed by shuffles at every row end below that):
//   power-law 2^20, K 128 FP32     0.705 -> 0.679 ms      512 graphs, K 64 FP32   2.93 -> 2.40 ms
//   300007 nodes, K 96 BF16        0.210 -> 0.184 ms      100003 nodes, K 512     0.313 -> 0.222 ms
// Where that first form of it was slower, and what it takes now (us before it, then, now; RMAT of 16 a row, W 256):
//   2^20 nodes, K 32 FP32   339  446  338    batches and a ring half as long for 4-lane groups, one more CTA
//   2^16 nodes, K 128 FP32   62   74   63    5 CTAs an SM without spills while B is within L2
//   rows of 700 pieces, K 32 BF16  89  188   50    all lane groups add a split row's pieces
//   2^17 nodes, K 256 FP32, B on a 16-byte boundary  172  269  154    4 columns of a lane in each half of the row
//
// Cooperative form (contig_coop): when a launch has so few chunks that most warps would get none, the
// four warps of a CTA share one chunk (4 EPS streams) and the straddling rows meet in shared memory.
// 4096 rows of 16, K 32: 25.5 -> 13.5 us per call (9.2 since launches report their status themselves).
#include "ns_internal.cuh"
#include "ns_mem.cuh"

#include <type_traits>

namespace ns {

constexpr int kFormF32 = 0;      // B rows 32-byte aligned: one 32-byte load per lane
constexpr int kFormF32Any = 1;   // B rows 16-byte aligned, any distance apart: two 16-byte loads
constexpr int kFormBf16 = 2;     // one 16-byte load of 8 BF16
constexpr int kFormBf16Any = 3;  // ... of rows any distance apart
// (the other forms keep the distance in 32 bits of bytes: one multiply an address, and a register less)
constexpr bool form_bf16(int form) { return form >= kFormBf16; }
constexpr bool form_any(int form) { return form == kFormF32Any || form == kFormBf16Any; }

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float lo, float hi)
{
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(u64 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c)
{
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b)
{
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// the raw form of 8 columns of a gathered row
struct GatheredF32 {
    u64 v[4];
};
struct GatheredBf16 {
    uint4 v;
};
template <int FORM>
using Gathered = std::conditional_t<form_bf16(FORM), GatheredBf16, GatheredF32>;

// Loads under a predicate that lives inside the instruction: the destination is read-write, so a
// skipped load leaves the slot as it was, and no select or copy after the load waits for its data.
template <int FORM, int G>
__device__ __forceinline__ void gather8(Gathered<FORM>& r, const unsigned char* p, uint64_t pol, bool on, bool on1)
{
    if constexpr (FORM == kFormF32)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %6, 0;\n\t"
                     "@q ld.global.nc.L1::no_allocate.L2::cache_hint.v4.b64 {%0,%1,%2,%3}, [%4], %5;\n\t}"
                     : "+l"(r.v[0]), "+l"(r.v[1]), "+l"(r.v[2]), "+l"(r.v[3]) : "l"(p), "l"(pol), "r"((int)on));
    else if constexpr (FORM == kFormF32Any)
        asm volatile("{\n\t.reg .pred q, q1;\n\tsetp.ne.s32 q, %6, 0;\n\tsetp.ne.s32 q1, %7, 0;\n\t"
                     "@q ld.global.nc.L1::no_allocate.L2::cache_hint.v2.b64 {%0,%1}, [%4], %5;\n\t"
                     "@q1 ld.global.nc.L1::no_allocate.L2::cache_hint.v2.b64 {%2,%3}, [%4 + %8], %5;\n\t}"
                     : "+l"(r.v[0]), "+l"(r.v[1]), "+l"(r.v[2]), "+l"(r.v[3])
                     : "l"(p), "l"(pol), "r"((int)on), "r"((int)on1), "n"(16 * G));
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %6, 0;\n\t"
                     "@q ld.global.nc.L1::no_allocate.L2::cache_hint.v4.b32 {%0,%1,%2,%3}, [%4], %5;\n\t}"
                     : "+r"(r.v.x), "+r"(r.v.y), "+r"(r.v.z), "+r"(r.v.w) : "l"(p), "l"(pol), "r"((int)on));
}
// one (column, value) pair of A's streams
__device__ __forceinline__ void stream_pair(int32_t& c, float& v, const int32_t* cp, const float* vp, uint64_t pol,
                                            bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %5, 0;\n\t"
                 "@q ld.global.nc.L2::cache_hint.b32 %0, [%2], %4;\n\t"
                 "@q ld.global.nc.L2::cache_hint.f32 %1, [%3], %4;\n\t}"
                 : "+r"(c), "+f"(v) : "l"(cp), "l"(vp), "l"(pol), "r"((int)on));
}

template <int FORM>
__device__ __forceinline__ void accumulate(u64 (&acc)[4], float w, const Gathered<FORM>& r)
{
    const u64 ww = pack2(w, w);
    if constexpr (!form_bf16(FORM)) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fma2(ww, r.v[q], acc[q]);
    } else {
        const uint32_t x[4] = {r.v.x, r.v.y, r.v.z, r.v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)  // BF16 is the high half of an FP32
            acc[q] = fma2(ww, pack2(__uint_as_float(x[q] << 16), __uint_as_float(x[q] & 0xffff0000u)), acc[q]);
    }
}

// a lane's two times 4 columns, HI apart, where they exist (both or none of 8 in a row)
template <int HI>
__device__ __forceinline__ void store8(float* p, bool act, bool act1, const u64 (&a)[4], uint64_t pol)
{
    const float2 x = unpack2(a[0]), y = unpack2(a[1]), z = unpack2(a[2]), w = unpack2(a[3]);
    if (act) {
        st_c4<true>(p, make_float4(x.x, x.y, y.x, y.y), pol);
        if (HI == 4) st_c4<true>(p + 4, make_float4(z.x, z.y, w.x, w.y), pol);
    }
    if (HI != 4 && act1) st_c4<true>(p + HI, make_float4(z.x, z.y, w.x, w.y), pol);
}

// One piece of a row that several chunks share (out of line: at most two per chunk).  The lanes
// with `mine` set hold the piece; the whole warp calls, each lane with the columns that its place in
// a group of G lanes stands for: 4 from `col` where `act` and 4 from col + HI where `act1`.  The piece that
// arrives last sums the pieces and stores the row: lane group j adds pieces j, j + 32 / G, ... in order,
// kAhead of them on their way at a time, then the groups' sums are added in order.
template <int G, int HI, int kAhead>
__device__ __noinline__ void deliver_piece(const ExecDesc& D, int32_t row, int32_t c, bool mine, bool act, bool act1,
                                           int col, u64 a0, u64 a1, u64 a2, u64 a3, int nsl, int slice,
                                           uint64_t pol)
{
    constexpr int EPS = 32 / G;
    const int lane = threadIdx.x & 31;
    const unsigned who = __ballot_sync(0xffffffffu, mine);
    if (who == 0u) return;
    const int leader = __ffs(who) - 1;
    row = __shfl_sync(0xffffffffu, row, leader);
    const int32_t s = __ldg(D.row_split + row);
    int32_t np = 0, piece = -1;
    float* slot0 = D.slots;
    if (s >= 0) {
        np = __ldg(D.split_np + s);
        piece = c - __ldg(D.split_base + s);
        slot0 += (int64_t)__ldg(D.split_slot + s) * D.K + col;
    }
    if (piece < 0 || piece >= np) {  // guard: a cut row that the plan does not list as split
        if (lane == 0) atomicOr(D.status, kStatusInternal);
        return;
    }
    if (mine) {
        float* p = slot0 + (int64_t)piece * D.K;
        const float2 x = unpack2(a0), y = unpack2(a1), z = unpack2(a2), w = unpack2(a3);
        if (act) __stcg(reinterpret_cast<float4*>(p), make_float4(x.x, x.y, y.x, y.y));
        if (act1) __stcg(reinterpret_cast<float4*>(p + HI), make_float4(z.x, z.y, w.x, w.y));
    }
    __threadfence();
    __syncwarp();
    int32_t* const cnt = D.split_cnt + (int64_t)s * nsl + slice;
    int old = 0;
    if (lane == 0) old = atomicAdd(cnt, 1);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old != np - 1) return;  // not the last piece
    __threadfence();
    u64 sum[4] = {0ull, 0ull, 0ull, 0ull};
    for (int q0 = lane / G; q0 < np; q0 += kAhead * EPS) {
        float4 x[kAhead], y[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const float* p = slot0 + (int64_t)(q0 + u * EPS) * D.K;
            const bool in = q0 + u * EPS < np;
            x[u] = y[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (in && act) x[u] = __ldcg(reinterpret_cast<const float4*>(p));
            if (in && act1) y[u] = __ldcg(reinterpret_cast<const float4*>(p + HI));
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            sum[0] = add2(sum[0], pack2(x[u].x, x[u].y));
            sum[1] = add2(sum[1], pack2(x[u].z, x[u].w));
            sum[2] = add2(sum[2], pack2(y[u].x, y[u].y));
            sum[3] = add2(sum[3], pack2(y[u].z, y[u].w));
        }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const u64 own = sum[q];
#pragma unroll
        for (int j = 1; j < EPS; ++j) sum[q] = add2(sum[q], __shfl_sync(0xffffffffu, own, (lane + j * G) & 31));
    }
    if (lane < G) store8<HI>(D.C + (int64_t)row * D.ldc + col, act, act1, sum, pol);
    if (lane == 0) atomicExch(cnt, 0);  // ready for the next launch
}

struct ContigPolicies {
    uint64_t first, last;
};

// A's streams and C evict first, B rows evict last; without hints everything evicts normally
__device__ __forceinline__ ContigPolicies contig_policies(bool hint)
{
    ContigPolicies p;
    if (hint) {
        const Policies q = make_policies();
        p.first = q.first;
        p.last = q.last;
    } else {
        asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p.first));
        p.last = p.first;
    }
    return p;
}

template <int G, int FORM>
struct ContigShape {
    static constexpr int EPS = 32 / G;                       // streams per warp
    // gathers in flight per stream (8 at 4 or 5 CTAs per SM: 0.85-0.89 ms on the power-law graph)
    static constexpr int DEPTH = G == 4 ? 2 : 4;             // (4 lanes: see contig_ctas)
    static constexpr int BE = G == 4 ? 8 : G < 16 ? 16 : G;  // entries per batch of a stream
    static constexpr int NB = BE / G;                        // entries a lane loads per batch
    // a lane's columns: two times 4, HI apart, CW from lane to lane (8 in a row, or, so that lanes of 16-byte
    // loads read whole lines, 4 in each half of the row)
    static constexpr int CW = FORM == kFormF32Any ? 4 : 8, HI = FORM == kFormF32Any ? 4 * G : 4;
    static_assert(BE % DEPTH == 0 && DEPTH <= BE, "batches start on a group of DEPTH steps, entries reach DEPTH ahead");
};

// What the streaming loop needs only at row ends and batch ends, kept in shared memory (one per
// warp) and read there each time: the loop's registers go to the gather ring.
struct ContigCold {
    const int32_t* col;   // the chunk's first column id
    const float* val;     // ... and value
    const int32_t* ends;  // rl_start + k0 + 1
    float* C;             // C + k0 * ldc (the chunk's first row), at the slice's first column
    int64_t ldc;
    const uint32_t* hot;
    int32_t* status;
    int32_t n, b0, nend;  // columns of A; the chunk's first merge item; rows that end in the chunk
    int32_t total;
};

__device__ __forceinline__ int32_t cold32(const int32_t& x) { return *const_cast<const volatile int32_t*>(&x); }
template <class T>
__device__ __forceinline__ T* coldp(T* const& x)
{
    return (T*)*reinterpret_cast<const volatile u64*>(&x);
}
__device__ __forceinline__ int64_t cold64(const int64_t& x) { return *const_cast<const volatile int64_t*>(&x); }

// HOT: the planner's hot-row map picks each gather's L2 policy; its bit travels as bit 31 of the
// column id.
template <int G, int FORM, bool HOT, bool FAR>
__device__ __forceinline__ void contig_chunk(const ExecDesc* Dp, int32_t c, int slice, int nsl, int lgU, int lane,
                                             int warp, const ContigPolicies& pol, float4* park0, int2* bat,
                                             int32_t* through0, ContigCold* cold)
{
    using Sh = ContigShape<G, FORM>;
    constexpr int EPS = Sh::EPS, DEPTH = Sh::DEPTH, BE = Sh::BE, NB = Sh::NB, MASK = 2 * BE - 1;
    constexpr int ES = form_bf16(FORM) ? 2 : 4;
    constexpr int lgE = EPS == 1 ? 0 : EPS == 2 ? 1 : EPS == 4 ? 2 : 3;
    const int g = lane / G, li = lane % G;
    // pieces of a split row on their way at a time (what the call saves counts in this kernel's registers:
    // power-law 2^20, K 128, 676 us with 4, 675 with 2, 670 with 1; 2^20 nodes, K 64 467 with 4, 456 with 2)
    constexpr int AHEAD = FAR ? 1 : G < 32 ? 2 : 4;
    const bool coop = lgU != lgE;  // the CTA's four warps share the chunk
    const int U = 1 << lgU;        // shares (streams) of the chunk
    const int u0 = warp * EPS;     // this warp's first share (warp is 0 in the one-warp form)
    const int my = u0 + g;
    auto sync = [&]() {
        if (coop) __syncthreads();
        else __syncwarp();
    };
    // nonzeros of the chunk before row k0 + q ends
    auto row_end = [&](int q) -> int32_t {
        return __ldg(coldp(cold->ends) + q) - 1 - cold32(cold->b0) - q;
    };

    // ------------------------------- the chunk and its shares -------------------------------
    unsigned char const* Bl;
    std::conditional_t<form_any(FORM), uint64_t, uint32_t> ldb_bytes;
    bool act, act1;      // this lane's first and second 4 columns exist
    int S, Smin;         // every share has Smin or S nonzeros
    int cnt;             // this share's nonzeros
    int k, k1;           // the next row to store and the first one this share does not store, less k0
    bool open, tail;     // the share starts inside row k; it holds a part of row k1
    int32_t cr[NB];
    float vr[NB];
    Gathered<FORM> b[DEPTH];
    const int2* const batg = bat + g;  // entry P of this share: batg[(P & MASK) * EPS]

    // the stream's (column, value) pairs, in batches of BE through shared memory
    auto fetch = [&](int e0, int32_t (&cc)[NB], float (&vv)[NB]) {
        const int p0 = (cold32(cold->total) * my) >> lgU;
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int e = e0 + li + G * q;
            cc[q] = 0;
            vv[q] = 0.f;
            stream_pair(cc[q], vv[q], coldp(cold->col) + (p0 + e), coldp(cold->val) + (p0 + e), pol.first, e < cnt);
        }
    };
    auto put = [&](int e0, int32_t (&cc)[NB], float (&vv)[NB]) {
        const int32_t n = cold32(cold->n);
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            if ((unsigned)cc[q] >= (unsigned)n) {  // guard: never gather outside B
                if (e0 + li + G * q < cnt) atomicOr(coldp(cold->status), kStatusInternal);
                cc[q] = 0;
                vv[q] = 0.f;
            }
            if (HOT) cc[q] |= (int32_t)(((__ldg(coldp(cold->hot) + (cc[q] >> 5)) >> (cc[q] & 31)) & 1u) << 31);
            bat[((e0 + li + G * q) & MASK) * EPS + g] = make_int2(cc[q], __float_as_int(vv[q]));
        }
    };
    // the column id of an entry (bit 31: hot row) gathered into slot u, when `on`
    auto gather = [&](int32_t e, int u, bool on, bool on1) {
        const uint32_t col = HOT ? ((uint32_t)e & 0x7fffffffu) : (uint32_t)e;
        gather8<FORM, G>(b[u], Bl + (size_t)col * ldb_bytes, HOT && e >= 0 ? pol.first : pol.last, on, on1);
    };
    {
        const ExecDesc& D = *Dp;
        const int4 h0 = __ldg(reinterpret_cast<const int4*>(D.chunk_rec + c));
        const int4 h1 = __ldg(reinterpret_cast<const int4*>(D.chunk_rec + c) + 1);
        const int32_t b0 = h0.x, b1 = h0.y, k0 = h0.z, kL = h0.w, z0 = h1.x, total = h1.y;
        const int nr = kL - k0 + 1;
        if (k0 < 0 || kL >= D.n_rl || kL < k0 || b1 <= b0 || total < 0 || total > 4096 || z0 < 0 ||
            (int64_t)z0 + total > D.n_res) {
            if (lane == 0) atomicOr(D.status, kStatusInternal);  // guard: corrupt plan
            return;                                              // (the same for every warp of a CTA)
        }
        const int sw = ((D.K + nsl - 1) / nsl + 7) & ~7;
        const int col0 = slice * sw + Sh::CW * li;
        act = Sh::CW * li < sw && col0 < D.K;
        act1 = FORM == kFormF32Any ? Sh::CW * li + Sh::HI < sw && col0 + Sh::HI < D.K : act;
        Bl = reinterpret_cast<const unsigned char*>(D.B) + (int64_t)col0 * ES;
        ldb_bytes = (decltype(ldb_bytes))(D.ldb * ES);
        const int p0 = (total * my) >> lgU, p1 = (total * (my + 1)) >> lgU;
        cnt = p1 - p0;
        S = (total + U - 1) >> lgU;
        Smin = total >> lgU;
        // a row that does not end in the chunk (only kL can) is not among the `nend` rows that do
        const int nend = (h1.z & kChunkTailCut) ? nr - 1 : nr;
        if (lane == 0) {
            cold->col = D.res_col + z0;
            cold->val = D.res_val + z0;
            cold->ends = D.rl_start + k0 + 1;
            cold->C = D.C + (int64_t)k0 * D.ldc + slice * sw;
            cold->ldc = D.ldc;
            cold->hot = D.hot;
            cold->status = D.status;
            cold->n = D.n;
            cold->b0 = b0;
            cold->nend = nend;
            cold->total = total;
        }
        __syncwarp();
        int32_t ca[NB];
        float va[NB];
        fetch(0, ca, va);
        fetch(BE, cr, vr);
        const int32_t e_first = lane < nend ? row_end(lane) : 0x7fffffff;
        put(0, ca, va);
        put(BE, cr, vr);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            b[u] = Gathered<FORM>{};  // inactive lanes hold zeros
            gather(batg[u * EPS].x, u, act && u < cnt, act1 && u < cnt);
        }
        fetch(2 * BE, cr, vr);  // stored when batch 1 starts
        // the rows of this share: those that end after p0 (from the chunk's start on, for the
        // first share) and at or before p1
        k = k1 = 0;
        for (int base = 0; base < nend; base += 32) {
            const int32_t e = base == 0 ? e_first : (base + lane < nend ? row_end(base + lane) : 0x7fffffff);
#pragma unroll
            for (int j = 0; j <= EPS; ++j) {
                const int n = __popc(__ballot_sync(0xffffffffu, e <= ((total * (u0 + j)) >> lgU)));
                if (g == j) k += n;
                if (g + 1 == j) k1 += n;
            }
        }
        if (my == 0) k = 0;
        if (my == U - 1) k1 = nend;
        const int start0 = (h1.z & kChunkHeadCut) ? -1 : 0;
        open = (k > 0 ? row_end(k - 1) : start0) < p0;
        tail = my == U - 1 ? nend < nr : (k1 > 0 ? row_end(k1 - 1) : start0) < p1;
    }

    // -------------------------------------- the stream --------------------------------------
    u64 acc[4] = {0ull, 0ull, 0ull, 0ull};
    int32_t wend;  // lane li: the end of row (k rounded down to G) + li, less the share's start
    auto load_ends = [&]() {
        const int q = (k & ~(G - 1)) + li;
        wend = q < k1 ? row_end(q) - ((cold32(cold->total) * my) >> lgU) : 0x7fffffff;
    };
    load_ends();
    int32_t next_end = __shfl_sync(0xffffffffu, wend, k & (G - 1), G);
    int32_t min_end = __reduce_min_sync(0xffffffffu, next_end);
    float4* const park = park0 + (warp * 32 + lane) * 2;
    auto park_acc = [&]() {
        const float2 x = unpack2(acc[0]), y = unpack2(acc[1]), z = unpack2(acc[2]), v = unpack2(acc[3]);
        park[0] = make_float4(x.x, x.y, y.x, y.y);
        park[1] = make_float4(z.x, z.y, v.x, v.y);
    };
    auto crow = [&](int q) { return coldp(cold->C) + (int64_t)q * cold64(cold->ldc) + Sh::CW * li; };
    // every row that ends at or before entry P, one per share and turn
    auto flush = [&](int P) {
        do {
            if (next_end <= P) {
                if (open) {
                    park_acc();
                    open = false;
                } else {
                    store8<Sh::HI>(crow(k), act, act1, acc, pol.first);
                }
                acc[0] = acc[1] = acc[2] = acc[3] = 0ull;
                ++k;
                if ((k & (G - 1)) == 0) load_ends();
            }
            __syncwarp();
            next_end = __shfl_sync(0xffffffffu, wend, k & (G - 1), G);
            min_end = __reduce_min_sync(0xffffffffu, next_end);
        } while (min_end <= P);
    };

    int P = 0;
    for (; P + DEPTH <= Smin; P += DEPTH) {
        if ((P & (BE - 1)) == 0 && P > 0) {  // batch P + BE into the ring, batch P + 2 BE requested
            __syncwarp();
            put(P + BE, cr, vr);
            __syncwarp();
            fetch(P + 2 * BE, cr, vr);
        }
        const int2* const e0 = batg + (P & MASK) * EPS;
        const int2* const e1 = batg + ((P + DEPTH) & MASK) * EPS;
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            if (P + u >= min_end) flush(P + u);
            accumulate<FORM>(acc, __int_as_float(e0[u * EPS].y), b[u]);
            gather(e1[u * EPS].x, u, act && P + u + DEPTH < cnt, act1 && P + u + DEPTH < cnt);
        }
    }
    {
        const int2* const e0 = batg + (P & MASK) * EPS;  // the last DEPTH entries or fewer, all gathered
#pragma unroll
        for (int u = 0; u < DEPTH; ++u) {
            if (P + u < S) {
                if (P + u >= min_end) flush(P + u);
                if (P + u < cnt) accumulate<FORM>(acc, __int_as_float(e0[u * EPS].y), b[u]);
            }
        }
    }
    if (min_end <= S) flush(S);

    // ------------------------------ rows that straddle shares -------------------------------
    asm volatile("" : "+l"(Dp));  // nothing of the descriptor is kept in registers through the stream
    const ExecDesc& D = *Dp;
    const bool through = open;  // the share lies inside one row
    if (through) park_acc();
    if (li == 0) through0[my] = through ? 1 : 0;
    sync();
    // adds the parts of shares my + 1, ... of one row; true when the row ends in one of them
    auto chain = [&](u64 (&a)[4]) -> bool {
        for (int v = my + 1; v < U; ++v) {
            const float4* pp = park0 + ((v * G) + li) * 2;  // share v = lanes v G .. v G + G - 1
            const float4 x = pp[0], y = pp[1];
            a[0] = add2(a[0], pack2(x.x, x.y));
            a[1] = add2(a[1], pack2(x.z, x.w));
            a[2] = add2(a[2], pack2(y.x, y.y));
            a[3] = add2(a[3], pack2(y.z, y.w));
            if (!through0[v]) return true;
        }
        return false;
    };
    bool cut = false;  // the share's last row goes on in the next chunk
    if (tail && !through) {
        const bool ended = chain(acc);
        cut = !ended;
        if (ended) store8<Sh::HI>(crow(k1), act, act1, acc, pol.first);
    }
    __syncwarp();
    const int32_t k0 = __ldg(&D.chunk_rec[c].k0);
    const int sw = ((D.K + nsl - 1) / nsl + 7) & ~7;
    const int col0 = slice * sw + Sh::CW * li;
    if (__any_sync(0xffffffffu, cut))
        deliver_piece<G, Sh::HI, AHEAD>(D, k0 + k1, c, cut, act, act1, col0, acc[0], acc[1], acc[2], acc[3], nsl, slice, pol.first);
    // the chunk starts inside row k0: its part is the first share's
    const bool head = my == 0 && (__ldg(&D.chunk_rec[c].flags) & kChunkHeadCut);
    if (__any_sync(0xffffffffu, head)) {
        if (head) {
            const float4 x = park[0], y = park[1];
            acc[0] = pack2(x.x, x.y);
            acc[1] = pack2(x.z, x.w);
            acc[2] = pack2(y.x, y.y);
            acc[3] = pack2(y.z, y.w);
            if (through) chain(acc);
        }
        __syncwarp();
        deliver_piece<G, Sh::HI, AHEAD>(D, k0, c, head, act, act1, col0, acc[0], acc[1], acc[2], acc[3], nsl, slice, pol.first);
    }
    sync();  // the parked parts and the batch ring are reused by the next chunk
}

// CTAs per SM, by what is left of the registers for the gather ring (each side measured with the next
// number up and down):
//   FP32, 32-byte B, 16 lanes: 5, and 7 where B is past L2 (FAR) and more warps hide HBM's latency, although
//     7 spill (2^16 / 2^20 nodes of 16, K 128, W 256: 63 / 743 us at 5, 73 / 686 at 7; W 512 58 / 710, 70 / 667)
//   4 lanes: 6, BF16 7, with a ring of 2 (2^20 nodes, K 32: 338 us; 388 at 5; 446 at 5 with a ring of 4 and
//     batches of 16)
//   other FP32 widths 5 (512 graphs, K 64: 2.35 ms; 2.39 at 7), BF16 6 (300007 nodes, K 96: 0.184 ms; 0.203 at 5)
constexpr int contig_ctas(int G, int form, bool far)
{
    return form_bf16(form) ? (G == 4 ? 7 : 6) : G == 4 ? 6 : G == 16 && far ? 7 : 5;
}
template <int G, int FORM, bool HOT, bool FAR>
__global__ void __launch_bounds__(kExecThreads, contig_ctas(G, FORM, FAR)) k_exec_contig(
    const ExecDesc* __restrict__ descs, const int32_t* __restrict__ queue,
    const int32_t* __restrict__ queue_desc, int64_t n_items, int32_t* ctrl, int32_t nsl, int32_t coop,
    const __grid_constant__ ExecDesc d0)
{
    using Sh = ContigShape<G, FORM>;
    constexpr int lgE = Sh::EPS == 1 ? 0 : Sh::EPS == 2 ? 1 : Sh::EPS == 4 ? 2 : 3;
    static_assert(kExecWarps == 4, "the cooperative form divides a chunk among four warps");
    __shared__ float4 s_park[kExecWarps * 32 * 2];  // per lane: its part of a straddling row
    __shared__ int2 s_bat[kExecWarps][2 * Sh::BE * Sh::EPS];
    __shared__ int32_t s_through[kExecWarps * Sh::EPS];
    __shared__ ContigCold s_cold[kExecWarps];
    __shared__ u64 s_ticket;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const ContigPolicies pol = contig_policies((descs ? descs[0].l2_hints : d0.l2_hints) != 0);
    // per-warp areas of the one-warp form; the cooperative form numbers the CTA's shares through
    float4* const park0 = coop ? s_park : s_park + warp * 64;
    int32_t* const through0 = coop ? s_through : s_through + warp * Sh::EPS;
    // chunk tickets in work-list order: the first one is the warp's (CTA's) own number, the next
    // is drawn while a chunk is in work
    u64* const ticket = reinterpret_cast<u64*>(ctrl + 4);
    const int64_t first = coop ? gridDim.x : (int64_t)gridDim.x * kExecWarps;
    int64_t u = coop ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * kExecWarps + warp;
    for (;;) {
        int64_t t = u / kExecWarps;
        if (t >= n_items * nsl) break;
        u64 next = 0;
        if (lane == 0 && (!coop || warp == 0)) next = atomicAdd(ticket, 1ull);
        const int slice = nsl > 1 ? (int)(t / n_items) : 0;
        if (nsl > 1) t -= (int64_t)slice * n_items;
        const int32_t it = __ldg(queue + t);
        const ExecDesc& D = descs ? descs[queue_desc ? __ldg(queue_desc + t) : 0] : d0;
        const int64_t c = (int64_t)(it - D.n_dwin) * kExecWarps + (u % kExecWarps);
        if (!D.rl_all) {  // guard: launched for a plan without a contiguous residual stream
            if (lane == 0) atomicOr(D.status, kStatusInternal);
        } else if (c >= 0 && c < D.n_chunks) {
            contig_chunk<G, FORM, HOT, FAR>(&D, (int32_t)c, slice, nsl, coop ? lgE + 2 : lgE, lane, coop ? warp : 0, pol,
                                       park0, s_bat[warp], through0, s_cold + warp);
        }
        if (coop) {
            if (threadIdx.x == 0) s_ticket = next;
            __syncthreads();
            next = s_ticket;
            __syncthreads();
        } else {
            next = __shfl_sync(0xffffffffu, next, 0);
        }
        u = first + (int64_t)next;
    }
    end_launch(ctrl, d0, descs == nullptr);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
typedef void (*ContigKernel)(const ExecDesc*, const int32_t*, const int32_t*, int64_t, int32_t*, int32_t, int32_t,
                             ExecDesc);

template <int FORM, bool HOT>
static ContigKernel pick_lanes(int width, bool far = false)
{
    if (width <= 32) return k_exec_contig<4, FORM, HOT, false>;
    if (width <= 64) return k_exec_contig<8, FORM, HOT, false>;
    if (width <= 128) {
        if constexpr (FORM == kFormF32)
            if (far) return k_exec_contig<16, FORM, HOT, true>;
        return k_exec_contig<16, FORM, HOT, false>;
    }
    return k_exec_contig<32, FORM, HOT, false>;
}

static ContigKernel pick_contig(int K, bool bf16, const ContigMode& m)
{
    const int nsl = contig_slices(K);
    const int width = ((K + nsl - 1) / nsl + 7) & ~7;
    if (m.any)  // (the hot map is only a cache hint)
        return bf16 ? pick_lanes<kFormBf16Any, false>(width) : pick_lanes<kFormF32Any, false>(width);
    if (bf16) return m.hot ? pick_lanes<kFormBf16, true>(width) : pick_lanes<kFormBf16, false>(width);
    return m.hot ? pick_lanes<kFormF32, true>(width, m.far) : pick_lanes<kFormF32, false>(width, m.far);
}

const void* contig_kernel(int K, bool bf16, const ContigMode& m)
{
    return reinterpret_cast<const void*>(pick_contig(K, bf16, m));
}

// Past L2 (K 128 FP32, us at 5 and at 7 CTAs an SM: 2^17 nodes, 67 MB, W 256 97 and 109; 2^18 nodes, 134 MB,
// 180 and 185; 2^19 nodes, 268 MB, 361 and 350; 2^20 nodes 741 and 692).
bool contig_far(int64_t n, int K, bool bf16, int device)
{
    return n * ((K + contig_slices(K) - 1) / contig_slices(K)) * (bf16 ? 2 : 4) > l2_bytes(device);
}

// At most 8 chunks per SM, while the launch has 20 to 28 warps there: with one chunk a warp most
// warps would have none, and sharing a chunk among four shortens its chain of steps (4096 rows of
// 16, 272 chunks: 25.5 -> 13.5 us a call).  For a plan it depends on the plan alone, so that a
// request sums its rows in the same order whatever shares its launch; a batch decides for all of its graphs
// of a width together.
bool contig_coop(int64_t n_chunks, int device) { return n_chunks <= 8 * (int64_t)num_sms(device); }

// the persistent grid: resident CTAs on every SM, at most one per unit of work
ns_status_t contig_prepare(int64_t n_items, int K, bool bf16, const ContigMode& m, int* grid_out)
{
    int per_sm = 0, dev = 0;
    NS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pick_contig(K, bf16, m), kExecThreads, 0));
    NS_CUDA_TRY(cudaGetDevice(&dev));
    int64_t g = (int64_t)(per_sm > 0 ? per_sm : 1) * num_sms(dev);
    const int64_t units = n_items * contig_slices(K) * (m.coop ? kExecWarps : 1);
    if (g > units) g = units;
    *grid_out = (int)(g > 0 ? g : 1);
    return NS_OK;
}

ns_status_t contig_launch(const ExecDesc* descs, const int32_t* queue, const int32_t* queue_desc, int64_t n_items,
                          int32_t* ctrl, int K, bool bf16, const ContigMode& m, int* grid_cache, cudaStream_t s,
                          const ExecDesc* d0)
{
    int grid = grid_cache ? *grid_cache : 0;
    if (grid == 0) NS_TRY(contig_prepare(n_items, K, bf16, m, &grid));
    if (grid_cache) *grid_cache = grid;
    if (n_items == 0) return NS_OK;
    ExecDesc dv{};
    if (d0) dv = *d0;
    pick_contig(K, bf16, m)<<<grid, kExecThreads, 0, s>>>(d0 ? nullptr : descs, queue, queue_desc, n_items, ctrl,
                                                           contig_slices(K), m.coop ? 1 : 0, dv);
    NS_LAUNCH_CHECK();
    return NS_OK;
}

}  // namespace ns
