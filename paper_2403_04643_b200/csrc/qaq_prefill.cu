// Score window after a prefill (Section 4.2 of the paper, "Attention score prediction": the
// predicted score of a token is the maximum over the scores of the preceding n queries).  Right
// after a prefill of T tokens those are the attention rows of its last n queries on the
// unquantized binary16 keys:
//   row of query i (position T-n+i):  softmax over the tokens t <= T-n+i of  scale * q_i . k_t.
// Rows are written newest first (row r = query n-1-r), so that the rows in which token t exists
// are 0..nvalid[t]-1 with nvalid[t] = min(n, T-t); entries of tokens a query cannot see are 0.
//
// This is the one dense contraction on the path ([n x D] x [D x T] per (b,h)); with n <= 64 rows it is bound by reading K once, and by
// the exponentials and stores of the rows.  The logits of 128 tokens are one accumulator of the fifth-generation tensor cores
// (tcgen05.mma, binary16 in, binary32 sums in tensor memory: a token a lane, a query a column), so neither the keys nor the
// logits pass through registers on their way there, and a row's 32 consecutive tokens are one store of a warp.  What the keys
// wait for in the meantime decides between three ways:
//   window_short_kernel   few tiles in all (64 of a (b,h) at most): the logits in registers, several CTAs per SM.
//   window_kernel         one pass: resident CTAs, the logits of a (b,h) in the tensor memory of a cluster until the statistics of its
//                         rows are known; K is read once and the rows written once.
//                         Two passes, (b,h) longer than that (8192 tokens with 64 rows, 16384 with 32, 32768 with 16) or too few to keep
//                         the SMs busy in clusters: statistics per chunk of tokens, then the logits again and the rows.
// Before (mma.sync fragments from global memory, logits in shared memory; beyond 4096 tokens two passes), now: 256 (b,h) of 4096
// tokens, 32 rows 129 and 70 us, with 64 rows 345 and 115; 160 of 8192, 64 rows 321 and 152; 32 of 32768, 32 rows 187 and 118; 32 of 333
// 8.3 and 5.5; 256 of 300 11.9 and 9.2; with head_dim 32 and 5 rows 64 of 2048 tokens 7.0 and 7.1, 192 of 600 (head_dim 64) 13.6 and 7.8.
#include <cuda.h>

#include "qaq_internal.cuh"

namespace {

constexpr int PW_CHUNK = 512;          // tokens per entry of the workspace's statistics at least
constexpr int PW_MAXQ = 64;            // rows (queries) at most
constexpr int PW_TILE = 128;           // tokens per accumulator: rows of the tensor-core instruction
constexpr int PW_CLUSTER = 8;          // CTAs of a cluster at most
constexpr int PW_SMEM = 227 * 1024;    // all of it: a CTA has its SM, and the SM's tensor memory, to itself
constexpr int PW_WORKERS = 16;         // warps that look at the logits: groups of four, up to 32 columns of a tile each
constexpr int PW_THREADS = 32 * (2 + PW_WORKERS);

struct PrefillArgs {
    const __half* Q;     // [BH][n][D]
    int H, BH, T, n;
    float scale;
    float* ring;         // [BH][n][T]
    uint8_t* nvalid;     // [BH][T]
    float* qnorm2;       // [BH][n] or null
    float2* part;        // [BH][nchunk][n] (reference, sum of powers of two relative to it) of the visible logits of a chunk
    int nchunk, tiles;   // chunks of a (b,h); tiles of a chunk, or of a CTA of a cluster
    int each_head, each_batch;   // 1, or 0 where all heads (batch elements) share their keys
};

// ONE_PASS: the CTAs of a cluster share a (b,h) and keep its logits in tensor memory until they have the statistics of its rows.
// STATS, ROWS: two passes over chunks of any length.
enum { ONE_PASS, STATS, ROWS };

// Operands in shared memory: rows of 64 channels (head_dim 128: two such regions) or 32, their 16-byte pieces swizzled.
template <int D, int NC, int MODE>
struct Window {
    static constexpr int ROW_BYTES = D >= 64 ? 128 : 64, REGIONS = (D + 63) / 64;
    static constexpr uint32_t TILE_BYTES = PW_TILE * D * 2, QUERY_BYTES = NC * D * 2;
    static constexpr int SLOTS = 512 / NC;                   // accumulators in tensor memory
    static constexpr bool SPLIT = MODE == ONE_PASS && NC <= 32;                                         // statistics and rows by warps of their own
    static constexpr int TEAM = SPLIT ? PW_WORKERS / 2 : PW_WORKERS;                                    // warps with the same job
    static constexpr int CW = NC < 32 ? NC : 32, PARTS = NC / CW, GROUPS = TEAM / 4 / PARTS;            // columns of a warp; groups that share a tile; tiles at a time
    struct Shared {
        unsigned long long full[8], empty[8];                // stages of the keys
        unsigned long long there[SLOTS], taken[SLOTS];       // accumulators
        unsigned long long q_free[2], stats[2], used[2];     // queries; statistics of the cluster's CTAs: there, no longer needed by any
        alignas(16) float ref[2][TEAM][CW], sum[2][TEAM][CW];      // of a warp: reference and sum of every row over its tokens
        alignas(16) float2 all[2][PW_CLUSTER][NC];           // the same of every CTA of the cluster, which all write here
        alignas(16) float2 row[2][NC];                        // what the rows are normalised with: reference, 1 / sum
        uint32_t tmem, failed;                               // a wait ran out
        int stopped;                                         // the first of the CTA's items whose statistics it has not taken, then; else -1
    };
    static constexpr int FIT = (PW_SMEM - 1024 - 2 * (int)QUERY_BYTES - (int)sizeof(Shared)) / (int)TILE_BYTES, STAGES = FIT < 8 ? FIT : 8;
    static_assert(STAGES >= 4, "stages");
};

__device__ __forceinline__ void bulk_tile(uint32_t dst, const CUtensorMap* map, int x, int t, int h, int b, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(t), "r"(h), "r"(b) : "memory");
}
__device__ __forceinline__ void bulk_rows(uint32_t dst, const CUtensorMap* map, int x, int row, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(row) : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t arrivals) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(arrivals) : "memory"); }
__device__ __forceinline__ void bar_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
// for what other CTAs of the cluster have done
__device__ __forceinline__ bool bar_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t done = 0;
#pragma unroll 1
    for (int i = 0; i < (1 << 14) && !done; ++i)
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
__device__ __forceinline__ void tensor_done(uint32_t bar) {           // arrives when what this thread has asked of the tensor cores is done
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
template <int ROW_BYTES>
__device__ __forceinline__ uint64_t operand(uint32_t addr) {          // K-major, swizzled over its row length, eight rows and then the next eight
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(8 * ROW_BYTES / 16) << 32) | (1ull << 46) | ((uint64_t)(ROW_BYTES == 128 ? 2 : 4) << 61);
}
// accumulator (128 lanes x NC columns of tensor memory) = tile . queries; by one thread
template <int D, int NC>
__device__ __forceinline__ void multiply(uint32_t acc, uint32_t tile, uint32_t queries) {
    constexpr uint32_t kind = (1u << 4) | (NC / 8) << 17 | (PW_TILE / 16) << 24;           // binary32 sums of binary16 products
    constexpr int RB = Window<D, NC, STATS>::ROW_BYTES, PER = RB / 32;                            // steps of 16 channels per region
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        const uint64_t x = operand<RB>(tile + (ks / PER) * (PW_TILE * RB) + (ks % PER) * 32), y = operand<RB>(queries + (ks / PER) * (NC * RB) + (ks % PER) * 32);
        asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                     ::"r"(acc), "l"(x), "l"(y), "r"(kind), "r"(ks) : "memory");
    }
}
// the columns of an accumulator from `at` on, for the thread's token
__device__ __forceinline__ void load_acc(uint32_t at, float (&x)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7]), "=f"(x[8]), "=f"(x[9]), "=f"(x[10]),
          "=f"(x[11]), "=f"(x[12]), "=f"(x[13]), "=f"(x[14]), "=f"(x[15]), "=f"(x[16]), "=f"(x[17]), "=f"(x[18]), "=f"(x[19]), "=f"(x[20]),
          "=f"(x[21]), "=f"(x[22]), "=f"(x[23]), "=f"(x[24]), "=f"(x[25]), "=f"(x[26]), "=f"(x[27]), "=f"(x[28]), "=f"(x[29]), "=f"(x[30]), "=f"(x[31])
        : "r"(at)
        : "memory");
}
__device__ __forceinline__ void load_acc(uint32_t at, float (&x)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7]), "=f"(x[8]), "=f"(x[9]), "=f"(x[10]),
          "=f"(x[11]), "=f"(x[12]), "=f"(x[13]), "=f"(x[14]), "=f"(x[15])
        : "r"(at)
        : "memory");
}
__device__ __forceinline__ void tmem_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int THREADS>
__device__ __forceinline__ void team_sync(int team) { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(THREADS) : "memory"); }

__device__ __forceinline__ float pow2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// (reference, sum of 2^(logit - reference)); a sum of 0 says that there was nothing (a reference of -inf does not: it may be logits that
// are no numbers, and a sum that is none)
__device__ __forceinline__ void fold_stats(float2& to, const float2& p) {
    const float m = fmaxf(to.x, p.x);
    to.y = (to.y == 0.f ? 0.f : to.y * pow2(to.x - m)) + (p.y == 0.f ? 0.f : p.y * pow2(p.x - m));
    to.x = m;
}
// Sums of eight columns over the lanes of the warp: lane 4k (and the three behind it) gets that of column k.
__device__ __forceinline__ float sum8(const float (&v)[8], int lane) {
    float a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = ((lane & 16) ? v[k + 4] : v[k]) + __shfl_xor_sync(0xFFFFFFFFu, (lane & 16) ? v[k] : v[k + 4], 16);
    float b[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) b[k] = ((lane & 8) ? a[k + 2] : a[k]) + __shfl_xor_sync(0xFFFFFFFFu, (lane & 8) ? a[k] : a[k + 2], 8);
    float c = ((lane & 4) ? b[1] : b[0]) + __shfl_xor_sync(0xFFFFFFFFu, (lane & 4) ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xFFFFFFFFu, c, 2);
    return c + __shfl_xor_sync(0xFFFFFFFFu, c, 1);
}

template <int D>
__device__ __forceinline__ void query_norm(const PrefillArgs& a, int bh, int i) {
    const __half* q = a.Q + ((size_t)bh * a.n + i) * D;
    float s = 0.f;
    for (int d = 0; d < D; ++d) { const float f = a.scale * __half2float(q[d]); s = fmaf(f, f, s); }
    a.qnorm2[(size_t)bh * a.n + i] = s;
}

// `tokens` entries of n rows, T apart, by a whole CTA
__device__ __noinline__ void lose_rows(float* row, int n, int T, int tokens) {
    for (; n > 0; --n, row += T)
        for (int t = threadIdx.x; t < tokens; t += blockDim.x) row[t] = __uint_as_float(QAQ_SCORE_LOST);
}

// One CTA per SM, which goes through its share of the work: a warp asks for the keys (tiles of 128 tokens, a ring of stages), a
// warp multiplies them, sixteen look at the accumulators.  Row t of an accumulator is a token, a thread's; column i a query.
// The reference of a row is a warp's largest logit of its first tile that has one above -inf (keys that are not finite); it is raised
// where a later logit exceeds it by 2^64.
// A wait that runs out of tries (a copy or a peer that never came) ends the CTA's waiting.  It then sends no more statistics, so that the
// other CTAs of the (b,h) run out of tries as well, or leaves a mark in place of those of its chunk, and in the end QAQ_SCORE_LOST
// in all rows of its tokens.
// Where the accumulators of two (b,h) have room (up to 32 rows) half of the sixteen warps take the statistics of the next one while
// the others write the rows of the last (256 (b,h) of 4096 tokens, 32 rows: 70 us, 82 with all of them at one job after the other, 78
// with eight warps); with 64 rows the tensor memory is full and the halves wait for each other (160 of 8192: 222 us, 152 together).
template <int D, int NC, int MODE>
__global__ void __launch_bounds__(PW_THREADS, 1) window_kernel(const __grid_constant__ CUtensorMap keys, const __grid_constant__ CUtensorMap queries, const PrefillArgs a) {
    using W = Window<D, NC, MODE>;
    constexpr int STAGES = W::STAGES, SLOTS = W::SLOTS;
    const float NEG = __int_as_float(0xff800000);
    extern __shared__ unsigned char s_dyn[];
    const uint32_t base = (smem_addr(s_dyn) + 1023u) & ~1023u, s_q = base + STAGES * W::TILE_BYTES;
    typename W::Shared& sm = *reinterpret_cast<typename W::Shared*>(s_dyn + (s_q + 2 * W::QUERY_BYTES - smem_addr(s_dyn)));
    const uint32_t full = smem_addr(sm.full), empty = smem_addr(sm.empty), there = smem_addr(sm.there), taken = smem_addr(sm.taken), q_free = smem_addr(sm.q_free), stats = smem_addr(sm.stats), used = smem_addr(sm.used);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // items: (b,h), or chunks of them; of an item the CTA has the tiles from tile0(item) on
    const int ncta = MODE == ONE_PASS ? (a.tiles ? ((a.T + PW_TILE - 1) / PW_TILE + a.tiles - 1) / a.tiles : 1) : 1;
    const int rank = MODE == ONE_PASS ? blockIdx.x % ncta : 0, step = gridDim.x / ncta, items = MODE == ONE_PASS ? a.BH : a.BH * a.nchunk;
    const int all_tiles = (a.T + PW_TILE - 1) / PW_TILE;
    struct Item { int bh, chunk, tile, n; };
    auto item_of = [&](int i) {
        Item o;
        if (MODE == ROWS) i = items - 1 - i;                 // backwards: the keys the first pass has read last are still in L2
        o.bh = MODE == ONE_PASS ? i : i / a.nchunk;
        o.chunk = MODE == ONE_PASS ? rank : i - o.bh * a.nchunk;
        o.tile = o.chunk * a.tiles;
        o.n = min(a.tiles, all_tiles - o.tile);
        return o;
    };
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) { bar_init(full + 8 * i, 1); bar_init(empty + 8 * i, 1); }
        for (int i = 0; i < SLOTS; ++i) { bar_init(there + 8 * i, 1); bar_init(taken + 8 * i, 4 * W::PARTS); }
        for (int i = 0; i < 2; ++i) { bar_init(q_free + 8 * i, 1); bar_init(stats + 8 * i, 1); bar_init(used + 8 * i, ncta); }
        sm.failed = 0; sm.stopped = -1;
        asm volatile("fence.mbarrier_init.release.cluster;\nfence.proxy.async.shared::cta;" ::: "memory");
    }
    qaq_dependency();
    if (warp == 1)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\ntcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::"r"(smem_addr(&sm.tmem)) : "memory");
    tmem_before_sync();
    if (MODE == ONE_PASS) cluster_barrier(); else __syncthreads();
    tmem_after_sync();
    const uint32_t acc = *(volatile uint32_t*)&sm.tmem;
    volatile uint32_t& failed = sm.failed;
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t g = 0;
            int it = 0;
            for (int i = blockIdx.x / ncta; i < items && ok; i += step, ++it) {
                const Item o = item_of(i);
                ok = bar_wait(q_free + 8 * (it & 1), ((uint32_t)(it >> 1) & 1u) ^ 1u);
                for (int k = 0; k < o.n && ok; ++k, ++g) {
                    const uint32_t st = g % STAGES, bar = full + 8 * st;
                    ok = bar_wait(empty + 8 * st, ((g / STAGES) & 1u) ^ 1u);
                    if (!ok) break;
                    bar_expect(bar, W::TILE_BYTES + (k == 0 ? W::QUERY_BYTES : 0u));
#pragma unroll
                    for (int r = 0; r < W::REGIONS; ++r) {
                        if (k == 0) bulk_rows(s_q + (it & 1) * W::QUERY_BYTES + r * (NC * W::ROW_BYTES), &queries, 64 * r, o.bh * a.n, bar);
                        bulk_tile(base + st * W::TILE_BYTES + r * (PW_TILE * W::ROW_BYTES), &keys, 64 * r, (o.tile + k) * PW_TILE, o.bh % a.H * a.each_head, o.bh / a.H * a.each_batch, bar);
                    }
                }
            }
            if (!ok) failed = 1;
            // what is on its way arrives before the CTA leaves (which takes no time but where something has failed)
            for (uint32_t j = g > STAGES ? g - STAGES : 0; j < g; ++j) bar_wait(full + 8 * (j % STAGES), (j / STAGES) & 1u);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t g = 0;
            int it = 0;
            for (int i = blockIdx.x / ncta; i < items && ok; i += step, ++it) {
                const Item o = item_of(i);
                for (int k = 0; k < o.n && ok; ++k, ++g) {
                    const uint32_t st = g % STAGES, slot = g % SLOTS;
                    ok = bar_wait(full + 8 * st, (g / STAGES) & 1u) && bar_wait(taken + 8 * slot, ((g / SLOTS) & 1u) ^ 1u);
                    if (!ok) break;
                    tmem_after_sync();
                    multiply<D, NC>(acc + slot * NC, base + st * W::TILE_BYTES, s_q + (it & 1) * W::QUERY_BYTES);
                    tensor_done(empty + 8 * st);
                    tensor_done(there + 8 * slot);
                }
                tensor_done(q_free + 8 * (it & 1));
            }
            if (!ok) failed = 1;
            if (it) bar_wait(q_free + 8 * ((it - 1) & 1), (uint32_t)((it - 1) >> 1) & 1u);              // likewise
        }
    } else {
        constexpr int CW = W::CW, GROUPS = W::GROUPS, TEAM = W::TEAM;
        // a warp reads the lanes of its quarter of a tile, columns h to h + CW - 1
        const int team = (warp - 2) / TEAM, w = (warp - 2) % TEAM, e = 32 * w + lane, quarter = warp & 3, group = (w >> 2) / W::PARTS, h = (w >> 2) % W::PARTS * CW;
        const float sc = a.scale * 1.4426950408889634f;
        const uint32_t lanes = acc + ((uint32_t)(32 * quarter) << 16) + h;
        auto wait_for = [&](uint32_t g) {
            ok = __all_sync(0xFFFFFFFFu, ok && bar_wait(there + 8 * (g % SLOTS), (g / SLOTS) & 1u));
            tmem_after_sync();
        };
        auto release = [&](uint32_t g) {
            tmem_before_sync();
            __syncwarp();
            if (lane == 0) bar_arrive(taken + 8 * (g % SLOTS));
        };
        uint32_t g0 = 0;
        int it = 0, bh_was = -1, buf = 0;
        for (int i = blockIdx.x / ncta; i < items; i += step, ++it) {
            const Item o = item_of(i);
            const int t0 = o.tile * PW_TILE + 32 * quarter + lane;          // the thread's token of the first tile
            // ---- statistics of the rows.  Query i sees token t if t <= T - n + i, that is from column t - (T - n) on.
            if (MODE != ROWS && (!W::SPLIT || team == 0)) {
                float sum[CW];
#pragma unroll
                for (int c = 0; c < CW; ++c) sum[c] = 0.f;
                float* const ref = sm.ref[it & 1][w];
                float* const top = sm.sum[it & 1][w];            // (until the sums are there: largest logits)
                bool none = true;                                // the row of the lane's column has no reference yet, 0 stands in: its logits are -inf
#pragma unroll 1
                for (int k = group; k < o.n; k += GROUPS) {
                    const uint32_t g = g0 + k;
                    wait_for(g);
                    const int hidden = t0 + k * PW_TILE - (a.T - a.n) - h;
                    const bool part_hidden = hidden - lane + 31 > 0;
                    float x[CW];
                    load_acc(lanes + (g % SLOTS) * NC, x);
                    if (MODE == STATS) release(g);
                    if (__any_sync(0xFFFFFFFFu, none)) {
#pragma unroll
                        for (int c = 0; c < CW; c += 4) {
                            float m[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) m[j] = warp_max(c + j < hidden ? NEG : x[c + j] * sc);
                            if (lane == 0) *reinterpret_cast<float4*>(top + c) = make_float4(m[0], m[1], m[2], m[3]);
                        }
                        __syncwarp();
                        if (none) {
                            const float m = top[lane % CW];
                            none = m == NEG;
                            ref[lane % CW] = none ? 0.f : m;
                        }
                        __syncwarp();
                    }
#pragma unroll
                    for (int c = 0; c < CW; c += 4) {
                        const float4 r = *reinterpret_cast<const float4*>(ref + c);
                        x[c] = fmaf(x[c], sc, -r.x); x[c + 1] = fmaf(x[c + 1], sc, -r.y); x[c + 2] = fmaf(x[c + 2], sc, -r.z); x[c + 3] = fmaf(x[c + 3], sc, -r.w);
                    }
                    if (part_hidden)
#pragma unroll
                        for (int c = 0; c < CW; ++c) if (c < hidden) x[c] = NEG;
                    float most = NEG;
#pragma unroll
                    for (int c = 0; c < CW; c += 2) most = fmaxf(most, fmaxf(x[c], x[c + 1]));
                    if (__any_sync(0xFFFFFFFFu, most > 64.0f)) {
                        __syncwarp();
#pragma unroll
                        for (int c = 0; c < CW; ++c) {
                            const float up = fmaxf(warp_max(x[c]), 0.f);
                            if (up > 0.f) { x[c] -= up; sum[c] *= pow2(-up); }
                            if (lane == 0) ref[c] += up;
                        }
                        __syncwarp();
                    }
#pragma unroll
                    for (int c = 0; c < CW; ++c) sum[c] += pow2(x[c]);
                }
                __syncwarp();
#pragma unroll
                for (int c0 = 0; c0 < CW; c0 += 8) {
                    float v[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) v[c] = sum[c0 + c];
                    const float s = sum8(v, lane);
                    if ((lane & 3) == 0) sm.sum[it & 1][w][c0 + (lane >> 2)] = s;
                }
                if (group >= o.n && lane < CW) { ref[lane] = NEG; sm.sum[it & 1][w][lane] = 0.f; }      // no tile for the group
                if (!ok) failed = 1;
                team_sync<32 * TEAM>(0);
                ok = !failed;              // whatever warp of the team has waited in vain so far
                const int c = e % NC;
                float2 st = make_float2(NEG, 0.f);
                if (c < a.n)
#pragma unroll
                    for (int j = 0; j < 4 * GROUPS; ++j) {
                        const int from = ((j >> 2) * W::PARTS + c / CW) * 4 + (j & 3);
                        if (!(sm.sum[it & 1][from][c % CW] == 0.f)) fold_stats(st, make_float2(sm.ref[it & 1][from][c % CW], sm.sum[it & 1][from][c % CW]));
                    }
                if (MODE == STATS) {
                    if (e < a.n) a.part[((size_t)o.bh * a.nchunk + o.chunk) * a.n + e] = ok ? st : make_float2(0.f, -1.0f);      // (no sum is negative)
                } else {
                    // every CTA of the (b,h) gets the statistics of all of them, as soon as all have used those of two items before.
                    // (A launch without clusters knows no asynchronous stores to a CTA of the cluster, its own included.)
                    const uint32_t bar = stats + 8 * (it & 1);
                    // Only warps that send wait: one that does not could come so late that the phase is over, and the one after.
                    if ((e & ~31) < ncta * NC) ok = __all_sync(0xFFFFFFFFu, ok && bar_wait_cluster(used + 8 * (it & 1), ((uint32_t)(it >> 1) & 1u) ^ 1u));
                    if (!ok) failed = 1;
                    if (ncta == 1) {
                        if (e < a.n) sm.all[it & 1][0][e] = st;
                        team_sync<32 * TEAM>(0);
                        if (e == 0 && !failed) bar_arrive(bar);
                    } else if (ok) {
                    if (e == 0) bar_expect(bar, (uint32_t)(ncta * a.n) * 8u);
                    if (c < a.n)
                        for (int r = e / NC; r < ncta; r += 32 * TEAM / NC)
                            asm volatile("{\n.reg .u32 p, m;\nmapa.shared::cluster.u32 p, %0, %2;\nmapa.shared::cluster.u32 m, %1, %2;\n"
                                         "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [p], {%3, %4}, [m];\n}"
                                         ::"r"(smem_addr(&sm.all[it & 1][rank][c])), "r"(bar), "r"(r), "f"(st.x), "f"(st.y) : "memory");
                    }
                }
                if (a.qnorm2 && o.chunk == 0 && e < a.n) query_norm<D>(a, o.bh, e);
            }
            // ---- normalised rows, newest first, written once; rows-per-token counts
            if (MODE != STATS && (!W::SPLIT || team == 1)) {
                if constexpr (MODE == ONE_PASS) {
                    buf = it & 1;
                    ok = __all_sync(0xFFFFFFFFu, ok && bar_wait_cluster(stats + 8 * buf, (uint32_t)(it >> 1) & 1u));
                    if (e < a.n) {
                        float2 st = make_float2(NEG, 0.f);
                        for (int r = 0; r < ncta; ++r) fold_stats(st, sm.all[buf][r][e]);
                        sm.row[buf][e] = make_float2(st.x, st.y > 0.f ? 1.0f / st.y : 0.f);
                    }
                    team_sync<32 * TEAM>(1);
                    if (!ok) {
                        if (e == 0 && sm.stopped < 0) sm.stopped = it;
                    } else if (ncta == 1) {
                        if (e == 0) bar_arrive(used + 8 * buf);
                    } else if (e < ncta)
                        asm volatile("{\n.reg .u32 m;\nmapa.shared::cluster.u32 m, %0, %1;\nmbarrier.arrive.release.cluster.shared::cluster.b64 _, [m];\n}" ::"r"(used + 8 * buf), "r"(e) : "memory");
                } else if (o.bh != bh_was) {           // merged statistics of the chunks
                    bh_was = o.bh;
                    buf ^= 1;
                    constexpr int EACH = 8;
                    float2 st = make_float2(NEG, 0.f);
                    static_assert(EACH <= PW_CLUSTER && EACH * NC <= 32 * TEAM, "parts");
                    if (e < EACH * NC) {
                        if (e % NC < a.n)
                            for (int ch = e / NC; ch < a.nchunk; ch += EACH) {
                                const float2 p = a.part[((size_t)o.bh * a.nchunk + ch) * a.n + e % NC];
                                if (p.y < 0.f) failed = 1;
                                fold_stats(st, p);
                            }
                        sm.all[buf][e / NC][e % NC] = st;
                    }
                    team_sync<32 * TEAM>(1);
                    if (e < a.n) {
                        for (int j = 1; j < EACH; ++j) fold_stats(st, sm.all[buf][j][e]);
                        sm.row[buf][e] = make_float2(st.x, st.y > 0.f ? 1.0f / st.y : 0.f);
                    }
                    team_sync<32 * TEAM>(1);
                }
                float* row0 = a.ring + ((size_t)o.bh * a.n + (a.n - 1 - h)) * a.T + t0;
#pragma unroll 1
                for (int k = group; k < o.n; k += GROUPS) {
                    const uint32_t g = g0 + k;
                    wait_for(g);
                    const int t = t0 + k * PW_TILE, hidden = t - (a.T - a.n) - h;
                    const bool part_hidden = hidden - lane + 31 > 0;
                    float* row = row0 + k * PW_TILE;
                    float x[CW];
                    load_acc(lanes + (g % SLOTS) * NC, x);
                    release(g);
#pragma unroll
                    for (int c = 0; c < CW; c += 2) {
                        const float4 r = *reinterpret_cast<const float4*>(&sm.row[buf][h + c]);
                        x[c] = pow2(fmaf(x[c], sc, -r.x)) * r.y;
                        x[c + 1] = pow2(fmaf(x[c + 1], sc, -r.z)) * r.w;
                    }
                    if (part_hidden)
#pragma unroll
                        for (int c = 0; c < CW; ++c) x[c] = c < hidden ? 0.f : x[c];
                    if (t < a.T) {
                        if (a.n - h >= CW) {
#pragma unroll
                            for (int c = 0; c < CW; ++c) { *row = x[c]; row -= a.T; }
                        } else {
#pragma unroll
                            for (int c = 0; c < CW; ++c) { if (h + c < a.n) *row = x[c]; row -= a.T; }
                        }
                        if (h == 0) a.nvalid[(size_t)o.bh * a.T + t] = (uint8_t)min(a.n, a.T - t);
                    }
                }
            }
            g0 += o.n;
        }
        if (!ok) failed = 1;
    }
    __syncwarp();
    tmem_before_sync();
    if (MODE == ONE_PASS) cluster_barrier(); else __syncthreads();       // nobody leaves while somebody may write to its shared memory
    if (warp == 1) { tmem_after_sync(); asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(acc) : "memory"); }
    if (MODE != STATS && failed) {
        // Statistics that are on their way arrive before the CTA leaves.  Those of an item are sent when all CTAs of the cluster have
        // taken the ones of two items before, so they can only be those of the first item that this CTA has not taken, and of the next;
        // all that will be sent has been sent before the barrier above.
        if (MODE == ONE_PASS && ncta > 1 && tid == 0 && sm.stopped >= 0)
            for (int it = sm.stopped; it < sm.stopped + 2 && blockIdx.x / ncta + it * step < items; ++it) bar_wait_cluster(stats + 8 * (it & 1), (uint32_t)(it >> 1) & 1u);
        for (int i = blockIdx.x / ncta; i < items; i += step) {
            const Item o = item_of(i);
            lose_rows(a.ring + (size_t)o.bh * a.n * a.T + o.tile * PW_TILE, a.n, a.T, min(o.n * PW_TILE, a.T - o.tile * PW_TILE));
        }
    }
}

// ---- few tiles in all: a thread keeps the logits of its token (up to 16 rows: or of two) in registers, a CTA is one group of four warps to
// four, a tile (or two) each, and the CTAs of a (b,h) form a cluster where it has more than one.  No warp waits for another's work but at
// barriers, several CTAs share an SM, keys come by plain asynchronous copies.  Tensor memory is given back before the CTAs of a cluster
// wait for each other, so that nobody waits for it who is waited for.  32 (b,h) of 333 tokens, 32 rows: 5.6 us, the kernel above 7.8 us; of 2048 tokens 10.7 and 12.8;
// of 4096 tokens, head_dim 32, 5 rows 7.2 us with two tiles to a group, 10.2 with one, 11.7.
constexpr int PS_GROUPS = 4;           // groups of four warps of a CTA at most
template <int ROW_BYTES, int ROWS>     // rows of a [.][D] operand on their way to shared memory, by four warps; what lies beyond `rows` is not touched
__device__ __forceinline__ void fetch_rows(uint32_t dst, const __half* src, long stride, int rows, int D, int thread) {
    const int PR = D / 8, row = thread / PR, c = thread % PR, step = 128 / PR;           // 16-byte pieces of a row; rows at a time, a multiple of 8
    constexpr int IN = ROW_BYTES / 16;
    dst += (c / IN) * (ROWS * ROW_BYTES) + row * ROW_BYTES + (((c % IN) ^ (ROW_BYTES == 128 ? row & 7 : (row >> 1) & 3)) << 4);
    src += (ptrdiff_t)row * stride + 8 * c;
#pragma unroll 16
    for (int r = row; r < ROWS; r += step, src += step * stride, dst += step * ROW_BYTES)
        if (r < rows) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
constexpr int short_ctas(int NC) { return NC <= 32 ? 2 : 1; }          // of PS_GROUPS groups to an SM, for their registers
// TP: tokens of a thread, tiles of a group of four warps.
template <int D, int NC, int TP>
__global__ void __launch_bounds__(128 * PS_GROUPS, short_ctas(NC)) window_short_kernel(const PrefillArgs a, const __half* K, long sb, long sh, long st) {
    using W = Window<D, NC, STATS>;
    constexpr int RB = W::ROW_BYTES, CW = NC < 32 ? NC : 32;
    const float NEG = __int_as_float(0xff800000), LOWEST = __int_as_float(0xff7fffff), sc = a.scale * 1.4426950408889634f;
    extern __shared__ unsigned char s_dyn[];
    __shared__ alignas(8) unsigned long long s_bar[PS_GROUPS];
    __shared__ uint32_t s_tmem, s_failed;                    // s_failed: a wait ran out
    __shared__ alignas(16) float s_max[4 * PS_GROUPS][NC], s_sum[4 * PS_GROUPS][NC];       // of a warp: reference and sum of every row over its tokens
    __shared__ float2 s_all[PW_CLUSTER][NC];                 // the same of every CTA of the cluster, which all write here
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, group = warp >> 2, groups = blockDim.x >> 7, warps = 4 * groups;
    const int bh = blockIdx.y, rank = blockIdx.x, ncta = gridDim.x;
    const uint32_t base = (smem_addr(s_dyn) + 1023u) & ~1023u, tile = base + group * TP * W::TILE_BYTES, queries = base + groups * TP * W::TILE_BYTES, bar = smem_addr(s_bar) + 8 * group;
    const uint32_t columns = max(32, 1 << (32 - __clz(groups * TP * NC - 1)));                // (a power of two)
    if (tid == 0) {
        for (int i = 0; i < PS_GROUPS; ++i) bar_init(smem_addr(s_bar) + 8 * i, 1);
        s_failed = 0;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    qaq_dependency();
    // first half of a cluster barrier: by the time the row statistics are exchanged every CTA of the cluster is known
    // to be running (its shared memory may be written)
    if (ncta > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const int t_group = (rank * groups + group) * TP * PW_TILE;
#pragma unroll
    for (int i = 0; i < TP; ++i) {
        const int t0 = t_group + i * PW_TILE;
        fetch_rows<RB, PW_TILE>(tile + i * W::TILE_BYTES, K + (size_t)(bh / a.H) * sb + (size_t)(bh % a.H) * sh + (ptrdiff_t)t0 * st, st, a.T - t0, D, tid & 127);
    }
    if (group == 0) fetch_rows<RB, NC>(queries, a.Q + (size_t)bh * a.n * D, D, a.n, D, tid);      // (columns of rows that are not there are not looked at)
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\ntcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::"r"(smem_addr(&s_tmem)), "r"(columns) : "memory");
    if (a.qnorm2 && rank == 0 && tid < a.n) query_norm<D>(a, bh, tid);
    asm volatile("cp.async.wait_all;\nfence.proxy.async.shared::cta;" ::: "memory");
    tmem_before_sync();
    __syncthreads();
    tmem_after_sync();
    const uint32_t acc = *(volatile uint32_t*)&s_tmem;
    if ((tid & 127) == 0) {
#pragma unroll
        for (int i = 0; i < TP; ++i) multiply<D, NC>(acc + (group * TP + i) * NC, tile + i * W::TILE_BYTES, queries);
        tensor_done(bar);
    }
    __syncwarp();
    if (!bar_wait(bar, 0u)) s_failed = 1;
    __syncwarp();
    tmem_after_sync();
    float x[TP][NC];
#pragma unroll
    for (int i = 0; i < TP; ++i)
#pragma unroll
        for (int h = 0; h < NC; h += CW) {
            float v[CW];
            load_acc(acc + ((uint32_t)(32 * (warp & 3)) << 16) + (group * TP + i) * NC + h, v);
#pragma unroll
            for (int c = 0; c < CW; ++c) x[i][h + c] = v[c];
        }
    // ---- per warp: maximum of every row over its tokens, the logits become powers of two relative to it (0 where the query cannot
    //      see the token), and their sum
    const int t = t_group + 32 * (warp & 3) + lane, hidden = t - (a.T - a.n);
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 8) {
        if (c0 >= a.n) break;
        float m[8], sum[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float top = NEG;
#pragma unroll
            for (int i = 0; i < TP; ++i) top = fmaxf(top, c0 + c >= hidden + i * PW_TILE ? x[i][c0 + c] * sc : NEG);
            m[c] = warp_max(top);
            sum[c] = 0.f;
#pragma unroll
            for (int i = 0; i < TP; ++i)
                sum[c] += x[i][c0 + c] = c0 + c >= hidden + i * PW_TILE ? pow2(fmaf(x[i][c0 + c], sc, -fmaxf(m[c], LOWEST))) : 0.f;      // (a maximum of -inf: zeros)
        }
        if (lane == 0) {
            *reinterpret_cast<float4*>(&s_max[warp][c0]) = make_float4(m[0], m[1], m[2], m[3]);
            *reinterpret_cast<float4*>(&s_max[warp][c0 + 4]) = make_float4(m[4], m[5], m[6], m[7]);
        }
        const float s = sum8(sum, lane);
        if ((lane & 3) == 0) s_sum[warp][c0 + (lane >> 2)] = s;
    }
    tmem_before_sync();
    __syncthreads();
    if (warp == 0) { tmem_after_sync(); asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(acc), "r"(columns) : "memory"); }
    bool lost = *(volatile uint32_t*)&s_failed != 0;
    if (ncta > 1) {
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");              // second half of the barrier begun at the start
        if (const int c = tid % NC; c < a.n) {
            float2 own = make_float2(NEG, 0.f);
            for (int w = 0; w < warps; ++w) fold_stats(own, make_float2(s_max[w][c], s_sum[w][c]));
            if (lost) own.y = -1.0f;                         // (no sum is negative)
            for (int r = tid / NC; r < ncta; r += blockDim.x / NC)
                asm volatile("{\n.reg .u32 p;\nmapa.shared::cluster.u32 p, %0, %1;\nst.shared::cluster.v2.f32 [p], {%2, %3};\n}"
                             ::"r"(smem_addr(&s_all[rank][c])), "r"(r), "f"(own.x), "f"(own.y) : "memory");
        }
        // every CTA has the statistics of all of them (the stores are complete at the barrier, and nothing is written to or read
        // from another CTA afterwards)
        cluster_barrier();
    }
    // ---- what the warp's powers are multiplied by, a row per lane; normalised rows, newest first, written once; rows-per-token counts
    float f[NC / CW];
#pragma unroll
    for (int h = 0; h < NC / CW; ++h) {
        const int c = CW * h + lane % CW;
        float2 all = make_float2(NEG, 0.f);
        if (c < a.n) {
            if (ncta > 1) for (int r = 0; r < ncta; ++r) { lost = lost || s_all[r][c].y < 0.f; fold_stats(all, s_all[r][c]); }
            else for (int w = 0; w < warps; ++w) fold_stats(all, make_float2(s_max[w][c], s_sum[w][c]));
        }
        const float own = c < a.n ? s_max[warp][c] : NEG;
        f[h] = all.y > 0.f && own != NEG ? pow2(own - all.x) / all.y : 0.f;
    }
    float* row = a.ring + ((size_t)bh * a.n + (a.n - 1)) * a.T + t;
    if (__any_sync(0xFFFFFFFFu, lost)) {                     // the tokens of the CTA, by all of its warps alike
        for (int c = 0; c < a.n; ++c, row -= a.T)
            for (int i = 0; i < TP; ++i)
                if (t + i * PW_TILE < a.T) row[i * PW_TILE] = __uint_as_float(QAQ_SCORE_LOST);
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (c >= a.n) break;
            const float y = __shfl_sync(0xFFFFFFFFu, f[c / CW], c % CW);
#pragma unroll
            for (int i = 0; i < TP; ++i)
                if (t + i * PW_TILE < a.T) row[i * PW_TILE] = x[i][c] * y;
            row -= a.T;
        }
    }
#pragma unroll
    for (int i = 0; i < TP; ++i)
        if (t + i * PW_TILE < a.T) a.nvalid[(size_t)bh * a.T + t + i * PW_TILE] = (uint8_t)min(a.n, a.T - t - i * PW_TILE);
}

// Descriptions of K ([batch][head][token][channel] with the caller's strides) and of the queries for the copies of tiles.
typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
cudaError_t describe(CUtensorMap* map, const void* at, int rank, const cuuint64_t* size, const cuuint64_t* stride, const cuuint32_t* box, int D) {
    static std::atomic<void*> known;                         // once it is found
    void* f = known.load(std::memory_order_acquire);
    if (!f) {
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &found);
        if (e != cudaSuccess) return e;
        if (found != cudaDriverEntryPointSuccess || !f) return cudaErrorSymbolNotFound;
        known.store(f, std::memory_order_release);
    }
    const cuuint32_t each[4] = {1, 1, 1, 1};
    const CUresult r = ((EncodeTiled)f)(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, rank, const_cast<void*>(at), size, stride, box, each, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                        D >= 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : r == CUDA_ERROR_INVALID_VALUE ? cudaErrorInvalidValue : cudaErrorUnknown;
}

// Which way: the one whose time, estimated from the work of the fullest SM, is the least.  The figures (us) are fitted to some 1300 sizes
// from 4 to 320 (b,h), 100 to 8192 tokens, measured each way: off by 11, 8 and 7 % (window_short_kernel, by rows), 6, 5 and 4 % (one pass).
struct Costs {
    float start, cluster, cta, group[2], turn; // window_short_kernel: a launch, one of clusters, every CTA of an SM, every group of warps of them (of one tile, of
                                               // two), every time that CTAs wait for others to end (for clusters 1 + D / 64 times that)
    float resident, item, tile, bytes;         // window_kernel: a launch, every (b,h) of a CTA, every tile, its bytes with head_dim 128
};
constexpr Costs costs_of(int NC) {
    return NC == 16 ? Costs{1.74f, 1.18f, 0.86f, {0.45f, 0.64f}, 3.f, 6.1f, 0.79f, 0.35f, 0.54f}
         : NC == 32 ? Costs{2.53f, 1.13f, 0.87f, {0.79f, 0.f}, 2.5f, 6.25f, 1.06f, 0.49f, 0.52f}
                    : Costs{4.2f, 1.22f, 0.82f, {1.14f, 0.f}, 5.f, 4.65f, 2.66f, 1.05f, 0.46f};
}
struct ShortPlan { float time; int tp, groups, ncta; };
template <int D, int NC, int TP>
constexpr int short_smem(int groups) { return 1024 + groups * TP * Window<D, NC, STATS>::TILE_BYTES + Window<D, NC, STATS>::QUERY_BYTES; }
// The best plan with TP tiles to a group, if it is better than `best` (alone[k]: so many clusters of k CTAs have an SM for every CTA).
template <int D, int NC, int TP>
void plan_short(int BH, int tiles, const int* alone, ShortPlan& best) {
    constexpr Costs cost = costs_of(NC);
    for (int g = 1; g <= PS_GROUPS && (g - 1) * TP < tiles; ++g) {
        const int k = (tiles + g * TP - 1) / (g * TP), smem = short_smem<D, NC, TP>(g) + NC * 200 + 1024;         // (200 bytes a row: the statistics)
        if (k > PW_CLUSTER || alone[k] < 1 || smem > PW_SMEM) continue;
        const int ctas = (BH + alone[k] - 1) / alone[k], at_once = min(short_ctas(NC) * PS_GROUPS / g, (PW_SMEM + 1024) / smem);
        const float time = cost.start + (k > 1 ? cost.cluster : 0.f) + (float)ctas * (cost.cta + (float)g * cost.group[TP - 1]) +
                           (float)((ctas - 1) / at_once) * (k > 1 ? 1.f + D / 64.f : 1.f) * cost.turn;
        if (time < best.time) best = {time, TP, g, k};
    }
}
template <int D, int NC, int TP>
qaq_status run_short(const PrefillArgs& a, const void* K, long sb, long sh, long st, const ShortPlan& p, cudaStream_t s) {
    constexpr int most = PW_SMEM - NC * 200 - 1024, all = short_smem<D, NC, TP>(PS_GROUPS);
    static SmemSeen seen;
    QAQ_CUDA_TRY(qaq_allow_smem((const void*)window_short_kernel<D, NC, TP>, all < most ? all : most, seen));
    QAQ_CUDA_TRY(qaq_launch_cluster(window_short_kernel<D, NC, TP>, dim3((unsigned)p.ncta, (unsigned)a.BH), dim3(128u * p.groups), p.ncta, short_smem<D, NC, TP>(p.groups), s,
                                    a, (const __half*)K, sb, sh, st));
    return QAQ_OK;
}

template <int D, int NC>
qaq_status run_window(PrefillArgs a, const void* K, long sb, long sh, long st, int batch, cudaStream_t s) {
    using W = Window<D, NC, ONE_PASS>;
    constexpr Costs cost = costs_of(NC);
    constexpr float per_tile = cost.tile + cost.bytes * D / 128.f;
    const int tiles = (a.T + PW_TILE - 1) / PW_TILE;
    static SmemSeen seen[3];
    static ClusterRoom room;
    const ContextName context;
    QAQ_CUDA_TRY(qaq_allow_smem((const void*)window_kernel<D, NC, ONE_PASS>, PW_SMEM, seen[0]));
    // two passes: chunks of at least PW_CHUNK tokens (the workspace's), as long as every SM gets eight
    const int chunk = max(PW_CHUNK / PW_TILE, (int)((long long)tiles * a.BH / (8 * 148)));
    const long long chunks = (long long)a.BH * ((tiles + chunk - 1) / chunk);
    float least = cost.resident + 2.f * (float)((chunks + 147) / 148 * chunk) * per_tile;
    // one pass: the size of the cluster; one that leaves no accumulators for a second (b,h) has to be that much better
    int alone[PW_CLUSTER + 1] = {}, best = 0, each = 0;
    float one_pass = 0.f;
    for (int k = 1; k <= PW_CLUSTER && k <= tiles; ++k) {
        const int n = (tiles + k - 1) / k;
        alone[k] = clusters_at_once(window_kernel<D, NC, ONE_PASS>, PW_THREADS, PW_SMEM, k, room, context);
        if (n > W::SLOTS || (tiles + n - 1) / n != k || alone[k] < 1) continue;
        const int items = (a.BH + alone[k] - 1) / alone[k];
        const float time = cost.resident + (float)items * cost.item + (float)items * (float)n * per_tile, chosen_by = time * (2 * n > W::SLOTS ? 1.08f : 1.f);
        if (time < least && (!best || chosen_by < one_pass)) { best = k; one_pass = chosen_by; each = n; }
    }
    if (best) least = one_pass;
    // few tiles
    if (tiles <= PW_CLUSTER * PS_GROUPS * 2) {
        ShortPlan plan = {least, 0, 0, 0};
        plan_short<D, NC, 1>(a.BH, tiles, alone, plan);
        if constexpr (NC == 16) {
            plan_short<D, NC, 2>(a.BH, tiles, alone, plan);
            if (plan.tp == 2) return run_short<D, NC, 2>(a, K, sb, sh, st, plan, s);
        }
        if (plan.tp == 1) return run_short<D, NC, 1>(a, K, sb, sh, st, plan, s);
    }
    CUtensorMap keys, queries;
    const cuuint32_t inner = D >= 64 ? 64 : 32;
    // (a stride of zero is a dimension of one in the description; the stride of such a dimension is never used)
    a.each_head = sh && a.H > 1; a.each_batch = sb && batch > 1;
    const cuuint64_t ksize[4] = {(cuuint64_t)D, (cuuint64_t)a.T, (cuuint64_t)(a.each_head ? a.H : 1), (cuuint64_t)(a.each_batch ? batch : 1)};
    const cuuint64_t kstride[3] = {2ull * st, 2ull * (a.each_head ? sh : st), 2ull * (a.each_batch ? sb : st)};
    const cuuint64_t qsize[2] = {(cuuint64_t)D, (cuuint64_t)a.BH * a.n}, qstride[1] = {2ull * D};
    const cuuint32_t kbox[4] = {inner, PW_TILE, 1, 1}, qbox[2] = {inner, NC};
    QAQ_CUDA_TRY(describe(&keys, K, 4, ksize, kstride, kbox, D));
    QAQ_CUDA_TRY(describe(&queries, a.Q, 2, qsize, qstride, qbox, D));
    if (best) {
        a.tiles = each;
        QAQ_CUDA_TRY(qaq_launch_cluster(window_kernel<D, NC, ONE_PASS>, dim3((unsigned)(min(a.BH, alone[best]) * best)), dim3(PW_THREADS), best, PW_SMEM, s, keys, queries, a));
        return QAQ_OK;
    }
    QAQ_CUDA_TRY(qaq_allow_smem((const void*)window_kernel<D, NC, STATS>, PW_SMEM, seen[1]));
    QAQ_CUDA_TRY(qaq_allow_smem((const void*)window_kernel<D, NC, ROWS>, PW_SMEM, seen[2]));
    a.tiles = chunk;
    a.nchunk = (tiles + chunk - 1) / chunk;
    const dim3 grid((unsigned)min(148, a.BH * a.nchunk));
    QAQ_CUDA_TRY(qaq_launch(window_kernel<D, NC, STATS>, grid, dim3(PW_THREADS), PW_SMEM, s, keys, queries, a));
    QAQ_CUDA_TRY(qaq_launch(window_kernel<D, NC, ROWS>, grid, dim3(PW_THREADS), PW_SMEM, s, keys, queries, a));
    return QAQ_OK;
}

template <int D>
qaq_status pick_window(const PrefillArgs& a, const void* K, long sb, long sh, long st, int batch, cudaStream_t s) {
    return a.n <= 16 ? run_window<D, 16>(a, K, sb, sh, st, batch, s) : a.n <= 32 ? run_window<D, 32>(a, K, sb, sh, st, batch, s) : run_window<D, 64>(a, K, sb, sh, st, batch, s);
}

// Upper quantile of a list of binary32 values (the squared query norms): exact 4 x 8-bit radix select on
// order-preserving keys by one CTA.  NaNs are not counted.
constexpr int QS_THREADS = 1024;
__device__ __forceinline__ uint32_t order_key(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__global__ void __launch_bounds__(QS_THREADS) quantile_kernel(const float* __restrict__ v, long n, double upper_frac, float* out) {
    __shared__ unsigned int hist[256];
    __shared__ unsigned long long s_count;
    __shared__ uint32_t s_prefix;
    __shared__ unsigned long long s_rank;
    const int tid = threadIdx.x;
    if (tid == 0) s_count = 0;
    __syncthreads();
    unsigned long long mine = 0;
    for (long i = tid; i < n; i += QS_THREADS) mine += (v[i] == v[i]) ? 1ull : 0ull;
    atomicAdd(&s_count, mine);
    __syncthreads();
    const unsigned long long N = s_count;
    if (N == 0) { if (tid == 0) *out = 0.f; return; }
    if (tid == 0) {
        unsigned long long k = (unsigned long long)floor(upper_frac * (double)N);
        if (k > N - 1) k = N - 1;
        s_rank = N - 1 - k;          // ascending rank of the answer
        s_prefix = 0;
    }
    __syncthreads();
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        const uint32_t prefix = s_prefix, pmask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
        if (tid < 256) hist[tid] = 0;
        __syncthreads();
        for (long i = tid; i < n; i += QS_THREADS) {
            const float f = v[i];
            if (f == f) {
                const uint32_t key = order_key(f);
                if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 0xFF], 1u);
            }
        }
        __syncthreads();
        if (tid == 0) {
            unsigned long long r = s_rank;
            int b = 0;
            for (; b < 255; ++b) {
                if (r < hist[b]) break;
                r -= hist[b];
            }
            s_rank = r;
            s_prefix = prefix | ((uint32_t)b << shift);
        }
        __syncthreads();
    }
    if (tid == 0) {
        const uint32_t key = s_prefix;
        const uint32_t u = (key & 0x80000000u) ? (key & 0x7FFFFFFFu) : ~key;
        *out = __uint_as_float(u);
    }
}

}  // namespace

extern "C" qaq_status qaq_prefill_window_workspace_bytes(const qaq_config* cfg, int n_tokens, size_t* host_out) {
    if (!cfg || !host_out || n_tokens < 1 || cfg->batch < 1 || cfg->heads < 1 || cfg->window < 1) return QAQ_ERR_INVALID_ARG;
    const size_t nchunk = ((size_t)n_tokens + PW_CHUNK - 1) / PW_CHUNK;
    *host_out = (size_t)cfg->batch * cfg->heads * nchunk * (size_t)cfg->window * sizeof(float2);
    return QAQ_OK;
}

extern "C" qaq_status qaq_prefill_window(const qaq_config* cfg, const void* Q, const void* K, long stride_b, long stride_h,
                                         long stride_t, int n_tokens, float softmax_scale, float* score_ring,
                                         uint8_t* nvalid, float* qnorm2, void* ws, size_t ws_bytes, void* stream) {
    if (!cfg || !Q || !K || !score_ring || !nvalid || !ws || n_tokens < 1) return QAQ_ERR_INVALID_ARG;
    if (!qaq_dim_ok(cfg->head_dim) || cfg->window < 1 || cfg->window > PW_MAXQ) return QAQ_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)K & 15) || ((uintptr_t)Q & 15) || (stride_b & 7) || (stride_h & 7) || (stride_t & 7) ||
        stride_t < cfg->head_dim || stride_b < 0 || stride_h < 0)
        return QAQ_ERR_INVALID_ARG;
    size_t need = 0;
    qaq_prefill_window_workspace_bytes(cfg, n_tokens, &need);
    if (ws_bytes < need || ((uintptr_t)ws & 7)) return QAQ_ERR_WORKSPACE;
    PrefillArgs a;
    a.Q = (const __half*)Q; a.H = cfg->heads; a.BH = cfg->batch * cfg->heads; a.T = n_tokens; a.n = cfg->window; a.scale = softmax_scale;
    a.ring = score_ring; a.nvalid = nvalid; a.qnorm2 = qnorm2; a.part = (float2*)ws;
    a.nchunk = a.tiles = 0;
    cudaStream_t s = (cudaStream_t)stream;
    switch (cfg->head_dim) {
        case 32: return pick_window<32>(a, K, stride_b, stride_h, stride_t, cfg->batch, s);
        case 64: return pick_window<64>(a, K, stride_b, stride_h, stride_t, cfg->batch, s);
        case 128: return pick_window<128>(a, K, stride_b, stride_h, stride_t, cfg->batch, s);
    }
    return QAQ_ERR_UNSUPPORTED_SHAPE;
}

extern "C" qaq_status qaq_qnorm2_quantile(const float* values, long n, double upper_frac, float* out, void* stream) {
    if (!values || !out || n < 1 || !(upper_frac >= 0.0 && upper_frac < 1.0)) return QAQ_ERR_INVALID_ARG;
    quantile_kernel<<<1, QS_THREADS, 0, (cudaStream_t)stream>>>(values, n, upper_frac, out);
    QAQ_CUDA_TRY(cudaGetLastError());
    return QAQ_OK;
}
