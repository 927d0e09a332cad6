// vsd_gemm2.cuh -- the tensor-core GEMM of the draft LM head and its backward
// on CTA pairs (tcgen05 cta_group::2): C[M][N] = A . B with bf16 operands and
// fp32 accumulation in tensor memory.
//
// A cluster of two CTAs (one SM each) computes 256 x 256 output tiles: CTA 0
// holds rows 0 .. 127 of the tile's A and of its accumulator, CTA 1 rows
// 128 .. 255, and each holds half of the tile's B columns, which the pair's
// MMA reads from both.  So a K block of 64 brings 32 KB into each CTA's shared
// memory for 2.1 MMAC of its tensor core, where a single CTA with a 128 x 256
// tile needs 48 KB; shared-memory bandwidth, which bounded that kernel, is
// used a third less, and six stages fit where four did.
//   warp 0      TMA producer (in each CTA): its rows of A, its half of B;
//   warp 1      MMA issuer (CTA 0): tcgen05.mma M = 256, N = 256, K = 16 into
//               one of two accumulators of 256 TMEM columns;
//   warps 2-5   epilogue (in each CTA): tcgen05.ld of its 128 rows, stores.
// The epilogue of one tile overlaps the main loop of the next.
//
// Measured at R = 4096, H = 4096, V = 32000 (1.07 TFLOP a product, one launch
// alone): logits 572 us (655 with one CTA per 128 x 256 tile), d_hidden 547 and
// d_weight 555 from a gradient in memory plus 70 to write it (962 and 1205 with
// the gradient made on chip for every tile): 1.88 to 1.96 PFLOP/s; cuBLAS ran at
// 1.91 on this pool.  The tensor pipe bounds it.
//
// Every wait is bounded; a wait that runs out sets VSD_STATUS_TIMEOUT in the
// status word, and the pair winds down: it waits (again bounded) for its MMAs
// and copies in flight, then frees its tensor memory.  In every case a CTA
// leaves only when the arrivals of all commits onto its barriers have landed:
// they come from the tensor core, after the thread that committed went on, and
// its shared memory may be another block's as soon as it has left.
#pragma once

#include "vsd_tc.cuh"

namespace vsd_g2 {

using namespace vsd_lm;

constexpr int BM = 128;        // rows per CTA (256 per pair)
constexpr int BN = 256;        // tile columns
constexpr int BH = BN / 2;     // columns of B held by each CTA
constexpr int BK = 64;
constexpr int kStages = 6;
constexpr int kThreads = 192;
constexpr int kABytes = BM * BK * 2;  // 16 KB
constexpr int kBBytes = BH * BK * 2;  // 16 KB
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kTmemCols = 512;

struct Bars {
    uint64_t full[kStages];   // CTA 0: both CTAs' TMA bytes of stage s landed
    uint64_t empty[kStages];  // the MMAs reading stage s are done (in both CTAs)
    uint64_t acc_full[2];     // accumulator b holds a finished tile (in both CTAs)
    uint64_t acc_empty[2];    // CTA 0: both epilogues have read accumulator b (8 arrivals)
    uint64_t drain;           // CTA 0: the last MMAs are done
    uint64_t timeout_ns;
    uint32_t tmem_base;
    int err;
    uint32_t peer_it;         // CTA 0: stages the other CTA's producer issued
    uint32_t freed, filled;   // commits the issuer made onto empty[] and acc_full[]
};
// [alignment][stages][the epilogue's staging][barriers]
template <class Epi> constexpr size_t smem_bytes() {
    static_assert(1024 + kStages * kStageBytes + Epi::kStaging + sizeof(Bars) <= 232448,
                  "227 KB of shared memory per block");
    return 1024 + kStages * kStageBytes + Epi::kStaging + sizeof(Bars);
}

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of p's counterpart in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(const void* p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
// 2-D TMA load into this CTA's shared memory, completion counted on the
// barrier at the cluster address `bar` (of either CTA of the pair).
__device__ __forceinline__ void tma_load_pair(void* dst, const CUtensorMap* map, int x, int y,
                                              uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];"
        :: "r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :: "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on `bar` in both CTAs once every MMA this thread issued is done.
__device__ __forceinline__ void commit_pair(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
        " [%0], %1;"
        :: "r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void commit_one(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];"
        :: "r"(smem_u32(bar)) : "memory");
}
// Arrive on a barrier of either CTA.  What it hands over is tensor memory, which
// the tcgen05 fences order; a release at cluster scope would make the warp wait
// for its global stores too, about a microsecond a tile (M = 4096, N = 128256,
// K = 256: 583 us with it, 474 now).
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void store_cluster(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait (as wait_phase_err) that also orders the other CTA's arrivals.
__device__ __forceinline__ bool wait_pair(uint64_t* bar, uint32_t parity, Bars* sb, int* status) {
    if (try_wait_cluster(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    for (;;) {
        if (try_wait_cluster(bar, parity)) return true;
        if (*(volatile int*)&sb->err) return false;
        if (global_timer_ns() - t0 > sb->timeout_ns) {
            sb->err = 1;
            atomicOr(status, VSD_STATUS_TIMEOUT);
            return false;
        }
    }
}
__device__ __forceinline__ bool wait_pair_warp(uint64_t* bar, uint32_t parity, Bars* sb,
                                               int* status) {
    return __all_sync(0xffffffffu, wait_pair(bar, parity, sb, status));
}

// ---------------------------------------------------------------- work
// One output tile, K blocks kb0 .. kb1 - 1.  part: the tile's other K blocks
// are another pair's, and both add into the zeroed output.
struct Work {
    int m0, n0, kb0, kb1;
    bool part;
    bool first, last;  // the first / last tile of a 1024-column chunk (chunk order)
};

// Chunk order: pairs take units of one 256-row M tile by one 1024-column chunk
// (per = kPerChunk tiles in turn), M tile fastest, so that an epilogue thread can
// carry its row's statistics over the chunk; without statistics a unit is one
// tile (per = 1), which spreads few units over the pairs (M = 256, K = 4096: N =
// 8000, 8 units of four tiles on 76 pairs 89 us, 32 of one 36; N = 128256 218, 204).
struct ChunkOrder {
    int mt, ntn, nk, nunits, u, nt, step, per;
    static constexpr int kPerChunk = 1024 / BN;
    __host__ __device__ static long long units(int M, int N, int per) {
        const int ntn = (N + BN - 1) / BN;
        return (long long)((M + 2 * BM - 1) / (2 * BM)) * ((ntn + per - 1) / per);
    }
    __device__ ChunkOrder(int M, int N, int K, int c, int nc, int per_) {
        mt = (M + 2 * BM - 1) / (2 * BM);
        ntn = (N + BN - 1) / BN;
        nk = (K + BK - 1) / BK;
        per = per_;
        nunits = (int)units(M, N, per);
        u = c;
        nt = 0;
        step = nc;
    }
    __device__ bool next(Work& w) {
        if (u >= nunits) return false;
        const int t0 = (u / mt) * per, t1 = min(t0 + per, ntn);
        w.m0 = (u % mt) * 2 * BM;
        w.n0 = (t0 + nt) * BN;
        w.kb0 = 0;
        w.kb1 = nk;
        w.part = false;
        w.first = nt == 0;
        w.last = t0 + nt + 1 == t1;
        if (w.last) {
            nt = 0;
            u += step;
        } else {
            ++nt;
        }
        return true;
    }
};

// Split order: whole tiles (N fastest, so that the pairs at work share their
// rows of A and walk B's K blocks together), then the tiles of an incomplete
// last round.  If those are at most half as many as there are pairs, two
// pairs share each, half of its K blocks each.
struct SplitOrder {
    int ntn, nk, whole, tiles, half, i, step, items;
    __host__ __device__ static int whole_tiles(long long tiles, int nc) {
        const int rem = (int)(tiles % nc);
        return (int)tiles - (2 * rem <= nc ? rem : 0);
    }
    __device__ SplitOrder(int M, int N, int K, int c, int nc) {
        ntn = (N + BN - 1) / BN;
        tiles = (M + 2 * BM - 1) / (2 * BM) * ntn;
        nk = (K + BK - 1) / BK;
        whole = nk > 1 ? whole_tiles(tiles, nc) : tiles;
        half = (nk + 1) / 2;
        items = whole + 2 * (tiles - whole);
        i = c;
        step = nc;
    }
    __device__ bool next(Work& w) {
        if (i >= items) return false;
        const int j = i - whole, t = j < 0 ? i : whole + (j >> 1);
        w.m0 = t / ntn * 2 * BM;
        w.n0 = t % ntn * BN;
        w.part = j >= 0;
        w.kb0 = j >= 0 && (j & 1) ? half : 0;
        w.kb1 = j >= 0 && !(j & 1) ? half : nk;
        i += step;
        return true;
    }
};

// ---------------------------------------------------------------- epilogues
// fp32 output, row-major [M][N] (N a multiple of 4); a part of a tile is added.
// Each warp stages 32 rows x 32 columns in shared memory (128-byte swizzle, two
// buffers) and stores them by TMA: a thread's own stores, 16 bytes of a row
// each, kept the epilogue at about 9 us a tile, longer than the main loop of a
// small K (d_weight at R = 672, H = 2888, V = 32000: 193 us with them, 114 now).
struct StoreF32 {
    using Order = SplitOrder;
    __device__ Order order(int M, int N, int K, int c, int nc) const {
        return SplitOrder(M, N, K, c, nc);
    }
    static constexpr int kStaging = 4 * 2 * 4096;
    CUtensorMap map;  // boxes of 32 x 32
    int M, N;
    struct State {
        unsigned char* buf;  // this warp's two buffers
        int n;               // stores issued
    };
    __device__ void init(State& st, unsigned char* staging, int q) const {
        st.buf = staging + q * 2 * 4096;
        st.n = 0;
    }
    __device__ void begin(State&, const Work&) const {}
    // (row: this lane's; the warp's first row is row - lane)
    __device__ void columns(State& st, const Work& w, int row, int col, uint32_t (&r)[32]) const {
        const int lane = threadIdx.x & 31, row0 = row - lane;
        if (row0 >= M || col >= N) return;
        unsigned char* b = st.buf + (st.n & 1) * 4096;
        if (lane == 0)  // the store before the last has read its buffer
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        __syncwarp();
#pragma unroll
        for (int v = 0; v < 8; ++v)
            *reinterpret_cast<uint4*>(b + lane * 128 + ((v ^ (lane & 7)) << 4)) =
                make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
        vsd::fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
            const uint64_t m = reinterpret_cast<uint64_t>(&map);
            if (w.part)
                asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group"
                             " [%0, {%1, %2}], [%3];"
                             :: "l"(m), "r"(col), "r"(row0), "r"(smem_u32(b)) : "memory");
            else
                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group"
                             " [%0, {%1, %2}], [%3];"
                             :: "l"(m), "r"(col), "r"(row0), "r"(smem_u32(b)) : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
        ++st.n;
    }
    __device__ void end(State&, const Work&, int) const {}
    __device__ void finish(State&) const {  // the buffers outlive the stores
        if ((threadIdx.x & 31) == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }
};

// bf16 output, row-major [M][N] (N a multiple of 8), and, with tab, each row's
// statistics of its rounded logits per 1024-column chunk for the E-step (a1 of
// the hot path): tab[row * stride + chunk].xy = (max, sum 2^{(x - max) c}).
struct StoreLogits {
    using Order = ChunkOrder;
    __host__ __device__ static int per_unit(bool stats) {
        return stats ? ChunkOrder::kPerChunk : 1;
    }
    __device__ Order order(int M, int N, int K, int c, int nc) const {
        return ChunkOrder(M, N, K, c, nc, per_unit(tab != nullptr));
    }
    static constexpr int kStaging = 0;
    __nv_bfloat16* out;
    int M, N;
    float4* tab;  // null: none
    int stride;   // float4 entries per row
    float c;
    struct State {
        float m, s;
    };
    __device__ void init(State&, unsigned char*, int) const {}
    __device__ void finish(State&) const {}
    __device__ void begin(State& st, const Work& w) const {
        if (w.first) {
            st.m = -INFINITY;
            st.s = 0.f;
        }
    }
    __device__ void columns(State& st, const Work&, int row, int col, uint32_t (&r)[32]) const {
        if (row >= M || col >= N) return;
        __nv_bfloat16* o = out + (size_t)row * N + col;
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = pack_bf16(r[2 * i], r[2 * i + 1]);
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (col + 8 * v < N)
                *reinterpret_cast<uint4*>(o + 8 * v) =
                    make_uint4(w[4 * v], w[4 * v + 1], w[4 * v + 2], w[4 * v + 3]);
        if (!tab) return;
        // the rounded logits of the group, then the running (max, sum)
        // rescaled to the new maximum
        float f[32];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
        float gm = -INFINITY;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (col + i < N) gm = fmaxf(gm, f[i]);
        const float nm = fmaxf(st.m, gm);
        if (nm > -INFINITY) {
            // (column col < N: the first term, and the carried sum in one rounding)
            float acc = fmaf(st.s, vsd::ex2((st.m - nm) * c), vsd::ex2((f[0] - nm) * c));
#pragma unroll
            for (int i = 1; i < 32; ++i)
                if (col + i < N) acc += vsd::ex2((f[i] - nm) * c);
            st.s = acc;
            st.m = nm;
        }
    }
    __device__ void end(State& st, const Work& w, int row) const {
        if (tab && w.last && row < M)
            reinterpret_cast<float2*>(tab + (size_t)row * stride + w.n0 / 1024)[0] =
                make_float2(st.m, st.s);
    }
};

// ---------------------------------------------------------------- the kernel
// AMN / BMN: the operand is stored with its M (N) index contiguous, [K][M]
// ([K][N]): MN-major in the tensor cores' terms, 64-column boxes of 64 K rows;
// otherwise K is contiguous, one box of 64 K columns by 128 rows.
template <bool AMN, bool BMN, class Epi>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_gemm2(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
            int M, int N, int K, const __grid_constant__ Epi epi, int* status,
            uint64_t timeout_ns) {
    extern __shared__ unsigned char dsm_raw[];
    // (the same offsets in both CTAs: the dynamic shared memory starts alike)
    unsigned char* dsm = dsm_raw + ((1024u - (smem_u32(dsm_raw) & 1023u)) & 1023u);
    unsigned char* staging = dsm + kStages * kStageBytes;
    Bars* sb = reinterpret_cast<Bars*>(staging + Epi::kStaging);
    constexpr uint32_t kIdesc =
        idesc_bf16(2 * BM, BN) | (AMN ? (1u << 15) : 0u) | (BMN ? (1u << 16) : 0u);
    constexpr int kBox = 64 * BK * 2;  // one MN-major box: 8 KB
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int c = blockIdx.x >> 1, nc = gridDim.x >> 1;
    // (a dependent E-step takes up the SMs that run out of tiles)
    vsd::grid_launch_next();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sb->full[s], 1);
            mbar_init(&sb->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sb->acc_full[b], 1);
            mbar_init(&sb->acc_empty[b], 8);
        }
        mbar_init(&sb->drain, 1);
        sb->err = 0;
        sb->peer_it = 0;
        sb->freed = sb->filled = 0;
        sb->timeout_ns = timeout_ns;
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&sb->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers are ready before either signals the other
    tc_fence_after();
    const uint32_t tmem = sb->tmem_base;
    uint32_t issued = 0;  // producer: stages issued

    if (warp == 0) {
        // ------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            typename Epi::Order order = epi.order(M, N, K, c, nc);
            Work w;
            while (ok && !*(volatile int*)&sb->err && order.next(w)) {
                const int m0 = w.m0 + (int)rank * BM, n0 = w.n0 + (int)rank * BH;
                for (int kb = w.kb0; kb < w.kb1; ++kb) {
                    const int s = (int)(it % kStages);
                    const uint32_t round = it / kStages;
                    if (round > 0 && !wait_pair(&sb->empty[s], (round - 1) & 1u, sb, status)) {
                        ok = false;
                        break;
                    }
                    unsigned char* a = dsm + s * kStageBytes;
                    unsigned char* b = a + kABytes;
                    const uint32_t bar = map_rank(&sb->full[s], 0);
                    const int k0 = kb * BK;
                    // CTA 0 expects the bytes of both
                    if (rank == 0) mbar_expect_tx(&sb->full[s], 2 * kStageBytes);
                    if (AMN) {
                        tma_load_pair(a, &tmA, m0, k0, bar);
                        tma_load_pair(a + kBox, &tmA, m0 + 64, k0, bar);
                    } else {
                        tma_load_pair(a, &tmA, k0, m0, bar);
                    }
                    if (BMN) {
                        tma_load_pair(b, &tmB, n0, k0, bar);
                        tma_load_pair(b + kBox, &tmB, n0 + 64, k0, bar);
                    } else {
                        tma_load_pair(b, &tmB, k0, n0, bar);
                    }
                    ++it;
                }
            }
            issued = it;
            if (rank == 1) store_cluster(map_rank(&sb->peer_it, 0), it);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------ MMA issuer
        if (rank == 0 && lane == 0) {
            uint32_t it = 0;
            int lt = 0;
            bool ok = true;
            typename Epi::Order order = epi.order(M, N, K, c, nc);
            Work w;
            for (; ok && !*(volatile int*)&sb->err && order.next(w); ++lt) {
                const int buf = lt & 1;
                const uint32_t use = (uint32_t)lt >> 1;
                if (use > 0 && !wait_pair(&sb->acc_empty[buf], (use - 1) & 1u, sb, status)) break;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(buf * BN);
                for (int kb = w.kb0; kb < w.kb1; ++kb) {
                    const int s = (int)(it % kStages);
                    if (!wait_pair(&sb->full[s], (it / kStages) & 1u, sb, status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = smem_u32(dsm + s * kStageBytes), b = a + kABytes;
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        // K step of 16: 32 bytes along a K-major row, or two
                        // 8-row K groups (2048 bytes) of an MN-major tile
                        const uint64_t ad = AMN ? sdesc_mn_sw128(a + 2048u * k, kBox)
                                                : sdesc_sw128(a + 32u * k);
                        const uint64_t bd = BMN ? sdesc_mn_sw128(b + 2048u * k, kBox)
                                                : sdesc_sw128(b + 32u * k);
                        mma_pair(d, ad, bd, kIdesc, (kb != w.kb0 || k != 0) ? 1u : 0u);
                    }
                    commit_pair(&sb->empty[s]);  // frees the stage in both CTAs
                    ++it;
                }
                if (!ok) break;
                commit_pair(&sb->acc_full[buf]);
            }
            commit_one(&sb->drain);
            wait_phase_drain(&sb->drain, 0, timeout_ns);
            for (uint32_t r = 0; r < 2; ++r) {  // (lt: tiles whose accumulator was committed)
                store_cluster(map_rank(&sb->freed, r), it);
                store_cluster(map_rank(&sb->filled, r), (uint32_t)lt);
            }
        }
    } else {
        // ------------------------------------------------------ epilogue
        const int q = warp & 3;  // TMEM lanes 32q .. 32q + 31
        int lt = 0;
        typename Epi::Order order = epi.order(M, N, K, c, nc);
        typename Epi::State st;
        epi.init(st, staging, q);
        Work w;
        for (; order.next(w); ++lt) {
            const int buf = lt & 1;
            const uint32_t use = (uint32_t)lt >> 1;
            if (!wait_pair_warp(&sb->acc_full[buf], use & 1u, sb, status)) break;
            tc_fence_after();
            const int row = w.m0 + (int)rank * BM + 32 * q + lane;
            const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * BN);
            epi.begin(st, w);
#pragma unroll 1
            for (int cc = 0; cc < BN / 32; ++cc) {
                uint32_t r[32];
                __syncwarp();  // (lanes beyond M do not store)
                tmem_ld32(taddr + 32u * cc, r);
                epi.columns(st, w, row, w.n0 + 32 * cc, r);
            }
            epi.end(st, w, row);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_cluster(map_rank(&sb->acc_empty[buf], 0));
        }
        epi.finish(st);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // no MMA is in flight any more, nothing more is issued
    if (threadIdx.x == 0) {
        // the arrivals of the commits onto this CTA's barriers have landed (the
        // last phase of each barrier; the earlier ones have been waited for)
        const uint32_t freed = *(volatile uint32_t*)&sb->freed;
        const uint32_t filled = *(volatile uint32_t*)&sb->filled;
        for (uint32_t j = freed > (uint32_t)kStages ? freed - kStages : 0; j < freed; ++j)
            wait_phase_drain(&sb->empty[j % kStages], (j / kStages) & 1u, timeout_ns);
        for (uint32_t j = filled > 2u ? filled - 2u : 0; j < filled; ++j)
            wait_phase_drain(&sb->acc_full[j & 1u], (j >> 1) & 1u, timeout_ns);
    }
    if (rank == 0 && threadIdx.x == 0) {
        // The copies of the last stages have landed.  (Always so unless a wait
        // ran out; the two producers may then have stopped at different
        // stages, and what one of them never issued is made up for.)
        const uint32_t other = *(volatile uint32_t*)&sb->peer_it;
        const uint32_t top = issued > other ? issued : other;
        const uint32_t low = issued < other ? issued : other;
        for (uint32_t j = top > (uint32_t)kStages ? top - kStages : 0; j < top; ++j) {
            uint64_t* bar = &sb->full[j % kStages];
            if (j >= low) {
                if (issued > other)
                    asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cta.b64 [%0], %1;"
                                 :: "r"(smem_u32(bar)), "r"((uint32_t)kStageBytes) : "memory");
                else
                    mbar_expect_tx(bar, kStageBytes);
            }
            wait_phase_drain(bar, (j / kStages) & 1u, timeout_ns);
        }
    }
    __syncthreads();
    cluster_sync();  // the other CTA's copies too, before either leaves
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;"
                     :: "r"(tmem), "r"(kTmemCols) : "memory");
    }
}

}  // namespace vsd_g2
