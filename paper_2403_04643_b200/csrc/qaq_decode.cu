// S4+S5: decode attention over the packed cache (Section 2.1 / Figure 1 of the paper):
//   S = Softmax(scale * q Khat^T),  X = S Vhat,  xhat = min + (code + 1/2) * step,
// outliers restored from the sparse side list, split over the sequence with a
// log-sum-exp merge of the split partials; one, two or four queries per (b,h) and pass (Section 4.2,
// "Integration in text generation process": the packed cache is what every query reads).
//
// The affine map is factored out of the inner loops so they work on raw codes:
//   q . Khat_t = step_t * sum_d q_d c_td + (min_t + step_t/2) * sum_d q_d
//   X_d        = sum_t (p_t step_t) c_td + sum_t p_t (min_t + step_t/2)
// and a token's outliers add  q_ch * (x - (min_t + step_t/2))  resp.  p_t * (v - ...)
// because their code slot holds 0.
//
// Both sums over codes run on the integer tensor-core instruction mma.sync (u8 operands, s32 sums).  The cache stores
// the codes so that a loaded word is one mask (for some widths a shift) away from an operand register
// (qaq_codec.cuh), so a decode step - a GEMV, whose cost here is taking bit fields apart, not multiplying - spends one
// tensor-core instruction per 512 (keys) or 256 (values) code-times-weight products.  The exact integer sums make the
// result independent of any accumulation order.
//   q.K:  m16n8k32, rows = 16 tokens of one width, k = channels; B = q in 16-bit fixed point per (b,h), split into two
//         signed byte digits in two columns per query (q_d ~ qscale * (256 * hi_d + lo_d)).
//   S.V:  m16n8k16, rows = 16 channels, k = 16 slots of one width; B = the per-token weights p_t * step_t in 28-bit
//         fixed point, four byte digits in four columns per query.  The sums of consecutive tiles stay in the integer
//         accumulators while they share the reference of the exponentials and the size of a unit.
//
// One CTA = one run of consecutive tiles of the flattened (b,h, tile) sequence (runs of equal length, so every SM
// gets the same amount of work), cut once more into one piece per warp; each warp works through its tiles (QAQ_TILE
// tokens) on its own, with its own running sums and no CTA barrier; warps are merged once at the end.  (With the tiles
// of a (b,h) dealt out to the warps in turn, warps waited for each other at every (b,h) boundary: 11 % of a 7B layer at
// batch 8.)  Lane l looks after tokens 2l and
// 2l + 1 of the tile (logit, softmax weight, value weight); the tokens of a tile are stored sorted by width, so the
// section loops run one extraction routine over full row blocks, write dot products and read weights by slot, and a
// token finds its own through the slot in its metadata.
// The packed bytes and the outlier list of a tile come to the warp's shared-memory buffer by bulk copies (one per piece,
// completion on a transaction barrier): the next keys to the front while the values are worked on, the values to the back
// while the keys are.  The buffer holds both for typical tiles; what does not fit beside its neighbour is copied later,
// when the neighbour has been used.
//
// Outlier corrections are summed in fixed point with 32-bit integer atomics in shared memory, so the result does not
// depend on the order in which lanes arrive.
//
// The partials of a (b,h) that was split over several CTAs are merged by the last of these CTAs to finish, in the
// same launch (see merge_split).
#include <chrono>
#include <mutex>

#include "qaq_codec.cuh"
#include "qaq_internal.cuh"

namespace {


// ------------------------------------------------------------------------------------------ instructions
// D(16x8, s32) += A(16x32, u8, row) * B(32x8, s8, col).  Lane = 4*g + t holds
//   a0: row g, k 4t..4t+3   a1: row g+8, k 4t..4t+3   a2: row g, k 16+4t..   a3: row g+8, k 16+4t..   (one k per byte)
//   b0: k 4t..4t+3, column g   b1: k 16+4t.., column g
//   d0, d1: row g, columns 2t, 2t+1   d2, d3: row g+8, columns 2t, 2t+1
__device__ __forceinline__ void mma_k32(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// D(16x8, s32) += A(16x16, u8, row) * B(16x8, u8, col): a0, a1 and b0 as above
__device__ __forceinline__ void mma_k16(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(b0));
}
// the same two with a zero third operand
__device__ __forceinline__ void mma_k32_first(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
}
// W words from shared memory (aligned to the widest access taken: 16 bytes for four words, 8 for two, else 4)
template <int W>
__device__ __forceinline__ void lds_words(uint32_t addr, uint32_t (&x)[W]) {
    if constexpr (W == 4) asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(addr));
    else if constexpr (W == 2) asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(x[0]), "=r"(x[1]) : "r"(addr));
    else {
#pragma unroll
        for (int i = 0; i < W; ++i) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x[i]) : "r"(addr + 4 * i));
    }
}
__device__ __forceinline__ void sts_word(uint32_t addr, int v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

// Loads that stay where they are written: the metadata of the next tile is fetched long before its use.
__device__ __forceinline__ uint4 ldg_now4(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ldg_now2(const void* p) {
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ldg_now1(const void* p) {
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// bulk copies into shared memory, completion on a transaction barrier
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    return x;
}

// ------------------------------------------------------------------------------------------ shapes
// Warps per CTA and CTAs per SM by queries per pass: 16 warps per SM for one query (128 registers each), 12 for four
// (168 registers: four times the accumulators on the value side).
template <int NQ> struct Shape {
    static constexpr int WARPS = NQ == 4 ? 4 : 8, CTAS_PER_SM = NQ == 4 ? 3 : 2, THREADS = 32 * WARPS, SLOTS = 148 * CTAS_PER_SM;
};
constexpr int SCORES_FUSED_TOKENS = 8192;          // up to here the CTA that merges a (b,h) normalises its score row too
constexpr uint32_t LIST_STAGED = 1024;             // outlier entries per tile and tensor that come through shared memory at most; more are read in place
// Tiles whose value sums may stay in the 32-bit accumulators.  The row blocks of high nibbles add most: bytes up to 240 times
// digits up to 255, 64 tokens, once for the low four bits of a code (digits of the weight) and once for those above (digits of
// 16 times the weight).  (Up to 500 tiles, the bound of one of the two, sums of 6- to 8-bit codes wrapped where weights were equal.)
constexpr int HELD_TILES = 256;
static_assert(2LL * QAQ_TILE * 255 * 240 * HELD_TILES < (1LL << 31), "sums of the held tiles");
constexpr uint32_t SMALL_MAX = 0x5800u;            // 128 as binary16: up to here outlier terms are summed in one 32-bit word

struct DecArgs {
    TensorStore k, v;
    size_t pool_bytes;
    uint32_t ocap;
    int tmax_pad, ntiles_max;
    int T;
    const int* d_count;          // counted kernels only: the token count in device memory (T, run and ncta are then derived from it)
    const __half* q;
    long q_stride, out_stride;   // elements between the rows of consecutive (b,h) in q and in out (queries of a (b,h) are D apart)
    float scale;
    float* part;       // [ncta][2][NQ][D+4]: accumulators, reference of the exponentials, sum of p
    unsigned long long* done;    // [BH]: tag of the call | partials that are complete (see merge_split)
    unsigned long long tag;      // of this call; the low 12 bits are zero
    float* ml;         // [BH][2]   merged (max, sum) for the normalisation of long score rows, or null
    int BH, run, ncta; // (b,h) count; tiles per CTA of the flattened (b,h, tile) sequence; CTAs
    int cluster;       // CTAs per (b,h), a thread-block cluster, or 0: runs of the flattened sequence
    int nq, groups;    // queries of the launch and groups of NQ of them; blockIdx.y is the group (the last one may be short of queries)
    float* out;
    float* scores;     // [BH][scores_stride] or null (one query only)
    long scores_stride;
    int* status;       // device status of the cache (a copy that never completed)
};

// The flattened sequence of BH * ntiles tiles is cut into runs of `run` consecutive tiles, one CTA
// each, and a run into pieces of ceil(run / warps), one warp each: as few tiles per warp as fill every SM evenly, and
// never more than one (b,h) boundary inside a run.
struct DecPlan { int run, ncta; };
// Groups of queries share the chip.
template <int NQ>
__host__ __device__ inline DecPlan plan_decode(int BH, int ntiles, int groups) {
    using S = Shape<NQ>;
    const long long total = (long long)BH * ntiles, warps = (long long)(S::SLOTS / groups) * S::WARPS;
    long long run = (total + warps - 1) / warps * S::WARPS;
    if (run > ntiles) run = ntiles;
    DecPlan p;
    p.run = (int)run;
    p.ncta = (int)((total + run - 1) / run);
    return p;
}

// What the CTAs of a group of queries work on.
template <int D, int NQ>
struct Group {
    const __half* q;
    float *out, *part;
    unsigned long long* done;
    int nq;
    __device__ __forceinline__ explicit Group(const DecArgs& a) : q(a.q), out(a.out), part(a.part), done(a.done), nq(NQ) {
        if (NQ == 1) return;
        const int g = blockIdx.y;
        q += g * NQ * D;
        out += g * NQ * D;
        part += (size_t)g * 2 * (Shape<NQ>::SLOTS / a.groups) * NQ * (D + 4);
        done += (size_t)g * a.BH;
        nq = min(NQ, a.nq - g * NQ);
    }
};

// Short sequences: the CTAs of a (b,h) are a thread-block cluster, with as many tiles each, and their results meet in shared
// memory.  (Through memory - partials stored, CTAs counted by an atomic, partials loaded by the last one - a split costs 3 to
// 4 us: 32 (b,h) of 8 tiles, one CTA each, 8.3 us, of 9 tiles 12.4.)  Taken where a portable cluster makes no warp do
// more tiles than the flattened sequence would and the clusters all run at once: fits(k) says how many of k CTAs can (a cluster
// stays inside a part of the chip, so that 96 of three are fewer than 296 places promise: 96 (b,h) of 20975 tokens took 113 us in
// clusters of three, 74 as a flattened sequence).  Returns the size of the cluster, 0: the flattened sequence.
template <int NQ, class F>
inline int plan_cluster(int BH, int ntiles, int groups, F&& fits) {
    using S = Shape<NQ>;
    const int places = S::SLOTS / groups / BH;               // CTAs a (b,h) can have at once
    const int run = plan_decode<NQ>(BH, ntiles, groups).run;
    for (int k = min(min(8, places), (ntiles + S::WARPS - 1) / S::WARPS); k >= 2; --k) {
        const int crun = (ntiles + k - 1) / k;
        if ((crun + S::WARPS - 1) / S::WARPS > (run + S::WARPS - 1) / S::WARPS) return 0;
        if (BH * groups <= fits(k)) return k;
    }
    return 0;
}

// ------------------------------------------------------------------------------------------ shared memory
// per-warp scratch for the tile a warp is working on
template <int D, int NQ>
struct WarpScratch {
    static constexpr int STAGE = (NQ == 1 ? 84 : 72) * D;      // bytes of the staging buffer; any tile of one tensor fits alone
    static constexpr int DOTS = QAQ_TILE + 16;                 // the last row block of a list may store up to 15 rows too many
    static constexpr int WROW = QAQ_TILE + 4;                  // digit rows are spread over the banks
    static constexpr int VC = NQ < 2 ? 2 : NQ;
    static_assert(STAGE % 16 == 0 && STAGE >= qaqc::tile_bytes_max(D), "staging buffer");
    alignas(16) uint8_t buf[STAGE];           // keys (tile, outlier list) from the front, values to the back
    union alignas(16) {                       // used one after the other: key phase (until the logits are taken), value lists, value outliers
        int dot[2][DOTS][NQ];                 // integer q . (low 4 bits of the code), q . (the bits above) by slot
        uint8_t wts[2][NQ][4][WROW];          // the four byte digits (highest first) of the value weights, and of 16 times them, by slot
        int vcorr[VC][D];                     // fixed-point sums of the value-outlier corrections per channel
    };
    union alignas(16) {                       // likewise
        int kcorr[NQ][2][QAQ_TILE];           // fixed-point sums of the key-outlier corrections per token (second word: the low part)
        float2 tok[NQ][QAQ_TILE];             // p, p * (min + step/2) of the values
    };
    alignas(8) float mid[QAQ_TILE];           // min + step/2 of the keys
    alignas(16) float macc[NQ][D];            // weighted sums of the values, as far as they have left the integer accumulators
    alignas(8) unsigned long long bar[2];     // transaction barriers of the keys and of the values
};

template <int D, int NQ>
struct DecSmem {
    static constexpr int W = Shape<NQ>::WARPS;
    WarpScratch<D, NQ> ws[W];
    // the queries of the run's two (b,h); several: each over a power of two (its largest entry below 2), which is behind them
    alignas(16) float qf[2][D + (NQ > 1)][NQ];
    alignas(16) uint32_t qw[2][2][32][D / 32];// operand words of q per lane: low nibbles of its words, high nibbles
    float qscale[2][NQ], qsum[2][NQ];
    // results of the warps; the warp that meets the (b,h) boundary leaves what it has of the first one in entry W
    union {
        float cross[NQ][D];
        float from_sum[8][D];                 // clusters, where no warp meets a boundary: what the CTAs send (see merge_cluster), and nothing else
    };
    float mm[W + 1][NQ], ml[W + 1][NQ], cs[W + 1][NQ];
    int seg[W + 1];                           // which of the two (b,h) an entry belongs to, -1: none
    float2 from_ml[NQ][8];                    // likewise
    int last[2];
};

// ------------------------------------------------------------------------------------------ lists of rows
// The nibble words of a key row a lane works with: of the four of its unit those of its channels (at head_dim 128 all
// four, at 64 two, at 32 one, by t).
template <int D, int W>
__device__ __forceinline__ void key_words(uint32_t addr, int t, uint32_t (&v)[D / 32]) {
    uint32_t x[W], a[4];
    lds_words<W>(addr, x);
    qaqc::nibble_words<W>(x, a);
    if (D == 128) {
#pragma unroll
        for (int u = 0; u < D / 32; ++u) v[u] = a[u];
    } else if (D == 64) {
#pragma unroll
        for (int u = 0; u < D / 32; ++u) v[u] = (t & 1) ? a[2 + u] : a[u];
    } else {
        const uint32_t lo = (t & 1) ? a[1] : a[0], hi = (t & 1) ? a[3] : a[2];
        v[0] = (t & 2) ? hi : lo;
    }
}

// q . code for a list of n rows of W-bit codes of the keys: 16 rows per block, lane 4g+t holds the channels of q operand
// (t, u) of rows g and g+8.  The last block reads past the list (at most 15 rows, inside the warp's scratch) and
// stores what the next list or nobody writes over it.  A nibble word gives two operand registers: the low nibbles
// as they are, the high nibbles sixteen times too large, which is taken out of the exact sums.
template <int D, int W, int NQ>
__device__ __forceinline__ void k_list(uint32_t addr, int n, uint32_t dots, const uint32_t (&qa)[D / 32], const uint32_t (&qb)[D / 32], int g, int t) {
    constexpr int P = D / 32;
    constexpr uint32_t MA = 0x01010101u * ((1u << W) - 1u), MB = MA << 4;
    addr += (g * P + (t * P >> 2)) * 4 * W;
    dots += (g * NQ + t) * 4;
#pragma unroll 1
    for (; n > 0; n -= 16, addr += 64 * P * W, dots += 64 * NQ) {
        uint32_t v0[P], v1[P];
        key_words<D, W>(addr, t, v0);
        key_words<D, W>(addr + 32 * P * W, t, v1);
        int s0, s1;
        if constexpr (P == 1) {
            int a[4];
            mma_k32_first(a, v0[0] & MA, v1[0] & MA, (v0[0] >> 4) & MA, (v1[0] >> 4) & MA, qa[0], qb[0]);
            s0 = a[0] * 256 + a[1];
            s1 = a[2] * 256 + a[3];
        } else {
            int a[4], b[4];
            mma_k32_first(a, v0[0] & MA, v1[0] & MA, v0[1] & MA, v1[1] & MA, qa[0], qa[1]);
            mma_k32_first(b, v0[0] & MB, v1[0] & MB, v0[1] & MB, v1[1] & MB, qb[0], qb[1]);
            if constexpr (P == 4) {
                mma_k32(a, v0[2] & MA, v1[2] & MA, v0[3] & MA, v1[3] & MA, qa[2], qa[3]);
                mma_k32(b, v0[2] & MB, v1[2] & MB, v0[3] & MB, v1[3] & MB, qb[2], qb[3]);
            }
            s0 = a[0] * 256 + a[1] + ((b[0] * 256 + b[1]) >> 4);
            s1 = a[2] * 256 + a[3] + ((b[2] * 256 + b[3]) >> 4);
        }
        if (t < NQ) { sts_word(dots, s0); sts_word(dots + 32 * NQ, s1); }       // columns 2t, 2t+1: the digits of query t
    }
}

// Weighted sums over a list of n rows (groups of four slots) of W-bit codes of the values: 4 rows per instruction, lane
// 4g+t holds the channels of units g (and g + 8 at head_dim 128) of row t.  wt: the lane's digits at the list's first
// row, pair of queries by pair (`pair` bytes apart).  Rows past the list are read (inside shared memory) with weight
// zero.  The sums of the high nibbles come out sixteen times too large.
template <int D, int W, int NQ>
__device__ __forceinline__ void v_list(uint32_t addr, int n, uint32_t wt, bool use, int (&acc)[(NQ + 1) / 2][D / 16][4], int g, int t) {
    constexpr int NH = D == 128 ? 2 : 1, NP = (NQ + 1) / 2, PAIR = 8 * WarpScratch<D, NQ>::WROW;
    constexpr uint32_t MA = 0x01010101u * ((1u << W) - 1u), MB = MA << 4;
    const int e = D == 32 ? (g & 3) : g;
#pragma unroll 1
    for (; n > 0; n -= 4, addr += (D / 2) * 4 * W, wt += 16) {
        const int m = min(4, n);
        uint32_t wgt[NP];
#pragma unroll
        for (int pr = 0; pr < NP; ++pr) {
            uint32_t x[1] = {0};
            if (use && t < m) lds_words<1>(wt + pr * PAIR, x);
            wgt[pr] = x[0];
        }
        const uint32_t at = addr + (e * m + t) * 4 * W;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            uint32_t x[W], v[4];
            lds_words<W>(at + h * 32 * W * m, x);
            qaqc::nibble_words<W>(x, v);
            // row block 4h + 2 * nibble + u/2: rows g and g+8 are the channels of words u, u+1
#pragma unroll
            for (int pr = 0; pr < NP; ++pr) {
                if constexpr (D == 32) {
                    const uint32_t u0 = g >= 4 ? v[2] : v[0], u1 = g >= 4 ? v[3] : v[1];
                    mma_k16(acc[pr][0], u0 & MA, u1 & MA, wgt[pr]);
                    mma_k16(acc[pr][1], u0 & MB, u1 & MB, wgt[pr]);
                } else {
                    mma_k16(acc[pr][4 * h], v[0] & MA, v[1] & MA, wgt[pr]);
                    mma_k16(acc[pr][4 * h + 1], v[2] & MA, v[3] & MA, wgt[pr]);
                    mma_k16(acc[pr][4 * h + 2], v[0] & MB, v[1] & MB, wgt[pr]);
                    mma_k16(acc[pr][4 * h + 3], v[2] & MB, v[3] & MB, wgt[pr]);
                }
            }
        }
    }
}

// The lists of a tile with U units per row, from its header: pass 0 the main parts (4, 3, 2, 1 bits; rows in slot order),
// pass 1 the high parts (widths 8, 7, 6, 5; rows in slot order).  o: byte offset, n: rows.
struct Lists { uint32_t o4, o3, o2, o1; int n4, n3, n2, n1; };
template <int U>
__device__ __forceinline__ Lists lists_of(const uint4& h, int pass) {
    const uint32_t n7 = (h.y >> 16) & 0xFF, n6 = (h.y >> 8) & 0xFF, n5 = h.y & 0xFF, n3 = (h.x >> 16) & 0xFF;
    const uint32_t z2 = h.z >> 16, z13 = h.w & 0xFFFFu, m3 = z13 + n7 * U * 12, h5 = m3 + n3 * U * 12;
    Lists l;
    if (pass == 0) {
        l.o4 = qaqc::QAQ_TILE_HDR; l.n4 = (int)__dp4a(h.y, 0x01010101u, h.x >> 24);
        l.o3 = m3; l.n3 = (int)n3;
        l.o2 = z2 + n6 * U * 8; l.n2 = (int)((h.x >> 8) & 0xFF);
        l.o1 = h5 + n5 * U * 4; l.n1 = (int)(h.x & 0xFF);
    } else {
        l.o4 = h.z & 0xFFFFu; l.n4 = (int)(h.y >> 24);
        l.o3 = z13; l.n3 = (int)n7;
        l.o2 = z2; l.n2 = (int)n6;
        l.o1 = h5; l.n1 = (int)n5;
    }
    return l;
}
// channel of row g + 8s of value row block mb (blocks of high nibbles: v_high)
template <int D>
__device__ __forceinline__ constexpr bool v_high(int mb) { return D == 32 ? mb == 1 : ((mb >> 1) & 1) == 1; }
template <int D>
__device__ __forceinline__ int v_channel(int mb, int g, int s) {
    if (D == 32) return 8 * (2 * (g >> 2) + s) + 4 * mb + (g & 3);
    const int e = g + 8 * (mb >> 2), u = 2 * (mb & 1) + s;
    return 32 * (e >> 2) + 8 * u + 4 * ((mb >> 1) & 1) + (e & 3);
}

// ------------------------------------------------------------------------------------------ outlier sums
// Outlier terms are summed in fixed point.  Where all values of a tile are small (up to 128) one word is enough: a unit
// is 2^-24 of a bound on the largest term, so that a channel's 64 terms stay inside 32 bits, and a token's 127 (128 have half
// of the bound: without an inlier the minimum is 0).  The bound of a query's terms is its own, whatever queries share the pass.
// (The largest value of a tile is in its header.)  Otherwise a term is a high part in units of 2^-4 and the exact remainder in units of 2^-28; terms of 2^18 or more (and
// non-finite ones) are left out.
constexpr float OC_LIMIT = 262144.0f;
__device__ __forceinline__ void wide_add(int* hi_cell, int* lo_cell, float tm) {
    if (fabsf(tm) < OC_LIMIT) {
        const float hi = rintf(tm * 16.0f);
        const float rem = fmaf(hi, -0.0625f, tm);              // exact, |rem| <= 2^-5
        atomicAdd(hi_cell, (int)hi);
        atomicAdd(lo_cell, __float2int_rn(rem * 268435456.0f));
    }
}
__device__ __forceinline__ float wide_sum(int hi, int lo) { return fmaf((float)lo, 1.0f / 268435456.0f, (float)hi * 0.0625f); }
// 2^24 over a power of two above x (x > 0, normal), and its inverse
__device__ __forceinline__ void fixed_unit(float x, float& inv, float& unit) {
    const int ex = min(max((__float_as_int(x) >> 23) & 0xFF, 40), 240);
    inv = __int_as_float((254 - ex - 1 + 24) << 23);
    unit = __int_as_float((ex + 1 - 24) << 23);
}

// What of a tile's outlier list did not fit into the staging buffer (entries from..to, dense wide tiles only), read in
// place with four loads in flight.  Such lists are summed in two words: their largest value is not known.  (Read twice,
// for one word where the values allow it, 96 (b,h) of 1783 tokens with 8-bit codes and 5 % take 44 instead of 50 us for
// three queries, but the code costs every other case 1 to 3 %: 131072 tokens 171.7 instead of 167.6 us.)
template <class F>
__device__ __forceinline__ void unstaged(const uint32_t* list, uint32_t from, uint32_t to, F&& each) {
#pragma unroll 1
    for (uint32_t i = from + (threadIdx.x & 31); i < to; i += 128) {
        uint32_t e[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = ldg_now1(list + min(i + 32u * k, to - 1));
#pragma unroll
        for (int k = 0; k < 4; ++k) if (i + 32u * k < to) each(e[k]);
    }
}

// The score row of one (b,h), normalised in place by the whole CTA.
template <int THREADS>
__device__ __forceinline__ void normalise_scores(float* row, int T, float M, float L) {
    const float inv = L > 0.f ? 1.0f / L : 0.f;
    int t = threadIdx.x;
    for (; t + 7 * THREADS < T; t += 8 * THREADS) {
        float x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = __ldcg(row + t + u * THREADS);
#pragma unroll
        for (int u = 0; u < 8; ++u) row[t + u * THREADS] = __expf(x[u] - M) * inv;
    }
    for (; t < T; t += THREADS) row[t] = __expf(__ldcg(row + t) - M) * inv;
}

// The CTA that completes the partials of a (b,h) merges them (log-sum-exp), in CTA order, so the result does not depend
// on which one it is.
//
// The CTAs are counted in a word of the workspace, which comes uninitialised: the count carries the tag of the call, a
// number no other call uses.  Every CTA sees to it when it begins that the word carries the tag (with a count of zero, if
// nobody has put it there yet), so that being counted at the end is one atomic addition; with the tag checked there, in
// a compare-and-swap loop, eight CTAs took up to 5 us to be counted.  The last CTA clears the word, so that a replay of
// the same launch (a CUDA graph carries the same tag) starts anew.
__device__ __forceinline__ void open_count(unsigned long long* word, unsigned long long tag) {
    unsigned long long cur = *(volatile unsigned long long*)word;
    while (((cur ^ tag) >> 12) != 0) {       // a failed exchange means that another CTA has put the tag there: two rounds at most
        const unsigned long long was = atomicCAS(word, cur, tag);
        if (was == cur) break;
        cur = was;
    }
}
__device__ __forceinline__ bool count_partial(unsigned long long* word, int n) {
    unsigned long long was;
    asm volatile("fence.acq_rel.gpu;\natom.add.relaxed.gpu.global.u64 %0, [%1], 1;\nfence.acq_rel.gpu;" : "=l"(was) : "l"(word) : "memory");
    const bool last = (int)(was & 0xFFF) + 1 == n;
    if (last) *word = 0ull;
    return last;
}

// The CTAs whose runs meet a (b,h): the first of them and how many; only the first can have begun in the (b,h) before
// (then the partial is that of its second segment).
__device__ __forceinline__ void split_of(int bh, int ntiles, int run, int& first, int& n) {
    first = (bh * ntiles) / run;
    n = ((bh + 1) * ntiles - 1) / run - first + 1;
}

// log-sum-exp merge of the partials of a (b,h), by the whole CTA: D/4 threads take a partial, four channels each, every
// group of D/4 threads its share of the partials with the next four on their way; the groups meet in shared memory
template <int D, int NQ>
__device__ void merge_split(const DecArgs& a, DecSmem<D, NQ>& sm, int bh, int ntiles, int run, int T) {
    using S = Shape<NQ>;
    int c_lo, n;
    split_of(bh, ntiles, run, c_lo, n);
    const int first_slot = 2 * c_lo + (c_lo * run < bh * ntiles ? 1 : 0);
    constexpr int PS = D + 4, CT = D / 4, G = S::THREADS / CT, AHEAD = 4;
    const float NEG = __int_as_float(0xff800000);
    const int tid = threadIdx.x, d4 = tid % CT, grp = tid / CT;
    const Group<D, NQ> gr(a);
    struct Part { float4 x; float m, l; };
    Part* s_part = reinterpret_cast<Part*>(sm.ws[0].buf);          // [G][CT], then the group's reference and sum beside each
    static_assert(S::THREADS * sizeof(Part) <= sizeof(sm.ws), "scratch of the merge");
    auto fold = [&](Part& to, const Part& p) {
        const float m = fmaxf(to.m, p.m);
        const float wa = to.m == NEG ? 0.f : __expf(to.m - m), wb = p.m == NEG ? 0.f : __expf(p.m - m);
        to.x.x = fmaf(wb, p.x.x, wa * to.x.x); to.x.y = fmaf(wb, p.x.y, wa * to.x.y);
        to.x.z = fmaf(wb, p.x.z, wa * to.x.z); to.x.w = fmaf(wb, p.x.w, wa * to.x.w);
        to.l = fmaf(wb, p.l, wa * to.l);
        to.m = m;
    };
    for (int j = 0; j < gr.nq; ++j) {
        Part mine;
        mine.x = make_float4(0.f, 0.f, 0.f, 0.f); mine.m = NEG; mine.l = 0.f;
        for (int i0 = grp; i0 < n; i0 += AHEAD * G) {
            Part p[AHEAD];
#pragma unroll
            for (int k = 0; k < AHEAD; ++k) {
                const int i = min(i0 + k * G, n - 1);
                const float* src = gr.part + ((size_t)(i == 0 ? first_slot : 2 * (c_lo + i)) * NQ + j) * PS;
                p[k].x = __ldcg(reinterpret_cast<const float4*>(src) + d4);
                const float2 ml = __ldcg(reinterpret_cast<const float2*>(src + D));
                p[k].m = ml.x; p[k].l = ml.y;
            }
#pragma unroll
            for (int k = 0; k < AHEAD; ++k) if (i0 + k * G < n) fold(mine, p[k]);
        }
        s_part[tid] = mine;
        __syncthreads();
        // whole warps only from here to the barrier: those that hold channels, all of them where a score row is normalised
        if (tid < (CT > 32 ? CT : 32) || (NQ == 1 && a.scores)) {
            float M = NEG;
#pragma unroll 8
            for (int g = 0; g < G; ++g) M = fmaxf(M, s_part[g * CT + d4].m);
            mine.x = make_float4(0.f, 0.f, 0.f, 0.f); mine.m = M; mine.l = 0.f;
#pragma unroll 8
            for (int g = 0; g < G; ++g) {
                const Part p = s_part[g * CT + d4];
                const float w = p.m == NEG ? 0.f : __expf(p.m - M);
                mine.x.x = fmaf(w, p.x.x, mine.x.x); mine.x.y = fmaf(w, p.x.y, mine.x.y);
                mine.x.z = fmaf(w, p.x.z, mine.x.z); mine.x.w = fmaf(w, p.x.w, mine.x.w);
                mine.l = fmaf(w, p.l, mine.l);
            }
            if (tid < CT) {
                const float inv = mine.l > 0.f ? 1.0f / mine.l : 0.f;
                float* o = gr.out + (size_t)bh * a.out_stride + j * D + 4 * d4;
                const bool any = inv > 0.f;           // (a sum that is zero or not a number: zeros, as where nothing is merged)
                o[0] = any ? mine.x.x * inv : 0.f; o[1] = any ? mine.x.y * inv : 0.f; o[2] = any ? mine.x.z * inv : 0.f; o[3] = any ? mine.x.w * inv : 0.f;
            }
            if (NQ == 1) {
                if (a.ml && tid == 0) { a.ml[2 * bh] = mine.m; a.ml[2 * bh + 1] = mine.l; }
                if (a.scores && !a.ml) normalise_scores<S::THREADS>(a.scores + (size_t)bh * a.scores_stride, T, mine.m, mine.l);
            }
        }
        __syncthreads();
    }
}

// The same for the CTAs of a cluster, which send their results to each other's shared memory before they meet at the cluster barrier:
// query j is put together by CTA j mod cluster, which gets its sums; (max, sum of p) go to all.  After the barrier everything is local,
// and a CTA can leave without waiting for the others.  (Results left in place, read by the peers after the barrier, a second barrier before anybody
// leaves, operands of two (b,h) prepared: 32 (b,h) of 4096 tokens 11.4 us, this way 10.8.)  Every CTA normalises its share of the scores.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void peer_store(const float* p, int rank, float x) {
    asm volatile("{\n.reg .u32 a;\nmapa.shared::cluster.u32 a, %0, %1;\nst.shared::cluster.f32 [a], %2;\n}" ::"r"(smem_addr(p)), "r"(rank), "f"(x) : "memory");
}
__device__ __forceinline__ void peer_store(const float2* p, int rank, float x, float y) {
    asm volatile("{\n.reg .u32 a;\nmapa.shared::cluster.u32 a, %0, %1;\nst.shared::cluster.v2.f32 [a], {%2, %3};\n}" ::"r"(smem_addr(p)), "r"(rank), "f"(x), "f"(y) : "memory");
}
template <int D, int NQ>
__device__ __forceinline__ void merge_cluster(const DecArgs& a, DecSmem<D, NQ>& sm, const Group<D, NQ>& gr, int bh, int rank, int T, bool kept) {
    using S = Shape<NQ>;
    const float NEG = __int_as_float(0xff800000);
    const int tid = threadIdx.x, lane = tid & 31, ncl = a.cluster;
    float M = NEG, L = 0.f;
    cluster_arrive();
    cluster_wait();
#pragma unroll 1
    for (int j = 0; j < gr.nq; ++j) {
        if (j % ncl != rank && !(NQ == 1 && (a.scores || a.ml))) continue;
        float m = NEG, l = 0.f;
        if (lane < ncl) { const float2 ml = sm.from_ml[j][lane]; m = ml.x; l = ml.y; }
        M = warp_max(m);
        const float w = m == NEG ? 0.f : __expf(m - M);
        L = warp_sum(w * l);
        if (j % ncl == rank) {
            float x[8], sum = 0.f;
            const int d = tid < D ? tid : 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = i < ncl ? sm.from_sum[j / ncl * ncl + i][d] : 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) sum = fmaf(__shfl_sync(0xFFFFFFFFu, w, i), x[i], sum);
            if (tid < D) gr.out[(size_t)bh * a.out_stride + j * D + tid] = L > 0.f ? sum / L : 0.f;
            if (NQ == 1 && a.ml && tid == 0) { a.ml[2 * bh] = M; a.ml[2 * bh + 1] = L; }
        }
    }
    if (NQ == 1 && a.scores && !a.ml) {
        float* row = a.scores + (size_t)bh * a.scores_stride;
        const int t = (rank + ncl * (tid >> 5)) * QAQ_TILE + 2 * lane;
        if (!kept) {                    // a piece of the row, whoever wrote it
            const int each = (T + ncl - 1) / ncl, lo = min(rank * each, T);
            normalise_scores<S::THREADS>(row + lo, min(each, T - lo), M, L);
        } else {
            const float2 lg = *reinterpret_cast<const float2*>(&sm.ws[tid >> 5].mid[2 * lane]);
            const float inv = L > 0.f ? 1.0f / L : 0.f;
            if (t < T) row[t] = __expf(lg.x - M) * inv;
            if (t + 1 < T) row[t + 1] = __expf(lg.y - M) * inv;
        }
    }
}

// A CTA's run meets one or two (b,h); it leaves one partial for each, or the result where a (b,h) is one CTA's alone.
// In the loops over lists lane 4g+t is lane (g, t) of the tensor-core fragments.
// COUNTED: the token count is read from device memory and the split derived from it here (the grid is then the
// largest one any count needs; CTAs beyond the split find no tiles and leave).
// CLUSTER: the CTAs of a (b,h) are a cluster (a kernel of its own: decided at run time, 256 (b,h) of 4096 tokens took
// 52.7 us instead of 50.4).
template <int D, int NQ, bool COUNTED, bool CLUSTER>
__global__ void __launch_bounds__(Shape<NQ>::THREADS, Shape<NQ>::CTAS_PER_SM) decode_kernel(const DecArgs a) {
    using S = Shape<NQ>;
    using WS = WarpScratch<D, NQ>;
    constexpr int P = D / 32;        // nibble words of a key row per lane
    constexpr int MB = D / 16;       // 16-channel row blocks of the value side
    constexpr int NP = (NQ + 1) / 2; // pairs of queries that share an instruction on the value side
    constexpr int CPL = D / 32;      // channels per lane in the outlier sums of the values
    constexpr int TWO = NQ < 4 ? 2 : 1;      // outlier entries of a lane at a time: their chains of dependent loads run beside each other (four queries: spills)
    constexpr uint32_t STAGE = WS::STAGE;
    const float NEG = __int_as_float(0xff800000);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DecSmem<D, NQ>& sm = *reinterpret_cast<DecSmem<D, NQ>*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int fg = lane >> 2, ft = lane & 3;
    WS& ws = sm.ws[warp];
    if (lane == 0) { bar_init(smem_addr(ws.bar)); bar_init(smem_addr(ws.bar) + 8); asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
    const Group<D, NQ> gr(a);
    qaq_dependency();
    // Clusters: the warps of a (b,h) take its tiles in turn, so that a warp knows its first tile before it knows how many there are
    // (counted: their table entries and the count are one wait, not two).
    const int ncl = CLUSTER ? a.cluster : 1, rank = CLUSTER ? blockIdx.x % ncl : 0, stride = CLUSTER ? ncl * S::WARPS : 1;
    int T = a.T;
    if (COUNTED) T = (int)ldg_now1(a.d_count);
    uint4 tk, tv;
    struct Toks { uint2 mm; uint32_t b; };      // min | max << 16; width | slot << 8 of two tokens
    Toks kt;
    auto tab_at = [&](const uint4* tab, uint32_t place) { return ldg_now4(tab + place); };
    auto toks_at = [&](const TensorStore& ts, uint32_t place) {
        const size_t t0 = (size_t)place * QAQ_TILE + 2 * lane;
        Toks t;
        t.mm = ldg_now2(ts.mnmx + t0);
        t.b = ldg_now1(ts.bs + t0);
        return t;
    };
    if (CLUSTER) {
        const uint32_t place = (uint32_t)(blockIdx.x / ncl) * (uint32_t)a.ntiles_max + (uint32_t)min(rank + ncl * warp, a.ntiles_max - 1);
        tk = tab_at(a.k.tile, place); tv = tab_at(a.v.tile, place); kt = toks_at(a.k, place);
    }
    if (COUNTED && T < 1) {          // nothing cached: zeros
        for (int bh = blockIdx.x; bh < a.BH; bh += gridDim.x)
            if (tid < D) a.out[(size_t)bh * a.out_stride + tid] = 0.f;
        return;
    }
    __syncwarp();
    if (CLUSTER) cluster_arrive();
    // this CTA's run of the flattened (b,h, tile) sequence: it begins in bh0 and may reach into bh0 + 1, which begins at f_bound;
    // in a cluster the CTA has one (b,h)
    const int ntiles = (T + QAQ_TILE - 1) / QAQ_TILE;
    const int run = CLUSTER ? (ntiles + ncl - 1) / ncl : COUNTED ? plan_decode<NQ>(a.BH, ntiles, 1).run : a.run;
    const int flat_lo = CLUSTER ? 0 : blockIdx.x * run;
    if (!CLUSTER && flat_lo >= a.BH * ntiles) return;
    const int bh0 = CLUSTER ? blockIdx.x / ncl : flat_lo / ntiles;
    const int f_bound = CLUSTER ? ntiles : (bh0 + 1) * ntiles, flat_hi = CLUSTER ? ntiles : min(a.BH * ntiles, flat_lo + run);
    const int nseg = !CLUSTER && flat_hi > f_bound ? 2 : 1;
    // a warp that has one tile at most keeps its logits until they can be normalised: they need not come back from memory
    const bool kept = CLUSTER && NQ == 1 && a.scores && !a.ml && run <= S::WARPS;
    // this warp's piece of it
    const int piece = (run + S::WARPS - 1) / S::WARPS;
    int f = CLUSTER ? rank + ncl * warp : flat_lo + warp * piece;
    const int f_end = CLUSTER ? ntiles : min(f + piece, flat_hi), f_last = min(f_end, flat_hi) - 1;
    auto bh_of = [&](int i) { return bh0 + (!CLUSTER && i >= f_bound ? 1 : 0); };
    const uint32_t buf = smem_addr(ws.buf), bar = smem_addr(ws.bar);

    // ---- tile metadata: the table words (offset and length of the bytes, first entry and length of the outlier list),
    //      min/max, widths and slots of tokens 2*lane, 2*lane+1; fetched as late as their latency allows
    //      (a piece that has no tile i fetches its last one again: a load behind a condition would be waited for on the spot)
    auto place_of = [&](int i) {
        i = min(i, f_last);
        const int b = bh_of(i);
        return (uint32_t)(CLUSTER ? b * a.ntiles_max + i : b * a.ntiles_max + (i - b * ntiles));
    };
    auto fetch_tab = [&](const uint4* tab, int i) { return tab_at(tab, place_of(i)); };
    auto fetch_toks = [&](const TensorStore& ts, int i) { return toks_at(ts, place_of(i)); };
    // how a tile lies in the buffer: bytes of the tile and of the piece of the outlier list that comes with it (from the
    // 16-byte boundary before its first entry; what lies behind its last one belongs to the read-ahead margin of the
    // list's capacity), both multiples of 16
    struct Lay { uint32_t nb, lb; };
    auto layout = [&](const uint4& tb) {
        Lay l;
        l.nb = (tb.y + 15u) & ~15u;
        l.lb = tb.w ? (((tb.z & 3u) + min(tb.w, LIST_STAGED)) * 4u + 15u) & ~15u : 0u;
        l.lb = min(l.lb, STAGE - l.nb);
        return l;
    };
    auto stage = [&](uint32_t dst, const Lay& l, const TensorStore& ts, int b, const uint4& tb, int x) {
        if (lane == 0) {
            bar_expect(bar + 8 * x, l.nb + l.lb);
            if (l.nb) bulk_copy(dst, ts.codes + (size_t)b * a.pool_bytes + tb.x, l.nb, bar + 8 * x);
            if (l.lb) bulk_copy(dst + l.nb, ts.outl + (size_t)b * a.ocap + (tb.z & ~3u), l.lb, bar + 8 * x);
        }
    };

    if (!CLUSTER) { tk = fetch_tab(a.k.tile, f); tv = fetch_tab(a.v.tile, f); kt = fetch_toks(a.k, f); }
    // ---- queries of the run's (b,h), by all warps alike: four channels per lane of every query, and the four channels whose
    //      operand word the thread makes; all loads first
    constexpr int SEGS = CLUSTER ? 1 : 2;
    constexpr int WORDS = 64 * P, PER = (SEGS * WORDS + S::THREADS - 1) / S::THREADS;   // operand words of a (b,h); words per thread
    uint2 qrow[SEGS][NQ], qword[PER];
    const bool q_aligned = ((uintptr_t)a.q & 7) == 0 && (a.q_stride & 3) == 0;
    auto load4 = [&](const __half* p) {
        if (q_aligned) return *reinterpret_cast<const uint2*>(p);
        const unsigned short* h = reinterpret_cast<const unsigned short*>(p);
        return make_uint2(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16);
    };
#pragma unroll
    for (int sg = 0; sg < SEGS; ++sg)
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            qrow[sg][j] = make_uint2(0u, 0u);
            if (sg < nseg && 4 * lane < D && j < gr.nq) qrow[sg][j] = load4(gr.q + (size_t)(bh0 + sg) * a.q_stride + j * D + 4 * lane);
        }
    // word idx: nibble word r / 2 of lane ln of (b,h) sg, its low (even r) or high nibbles; column ln / 4: the high (even) or
    // low (odd) digit of query ln / 8; first channel: unit p = lt * P / 4, word (lt * P mod 4) + r / 2 of it
    auto word_of = [&](int idx, int& sg, int& ln, int& r, int& ch) {
        sg = idx / WORDS; ln = idx / (2 * P) % 32; r = idx % (2 * P);
        ch = 32 * ((ln & 3) * P >> 2) + 8 * (((ln & 3) * P & 3) + (r >> 1)) + 4 * (r & 1);
    };
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int sg, ln, r, ch;
        word_of(tid + k * S::THREADS, sg, ln, r, ch);
        qword[k] = make_uint2(0u, 0u);
        if (sg < nseg && ln < 8 * gr.nq) qword[k] = load4(gr.q + (size_t)(bh0 + sg) * a.q_stride + (ln >> 3) * D + ch);
    }
    __syncwarp();
    if (f < f_end) stage(buf, layout(tk), a.k, bh_of(f), tk, 0);
    if (lane == 0 && warp < nseg && !CLUSTER) {
        int first, n;
        split_of(bh0 + warp, ntiles, run, first, n);
        if (n > 1) open_count(gr.done + bh0 + warp, a.tag);
    }
    for (int i = 4 * lane; i < NQ * D; i += 128) *reinterpret_cast<float4*>(&ws.macc[0][0] + i) = make_float4(0.f, 0.f, 0.f, 0.f);
    auto half_at = [](const uint2& v, int i) { return __half2float(__ushort_as_half((unsigned short)((i < 2 ? v.x : v.y) >> (16 * (i & 1))))); };
    float qsc[SEGS][NQ];
#pragma unroll
    for (int sg = 0; sg < SEGS; ++sg)
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            float qmax = 0.f, qs = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) { const float x = half_at(qrow[sg][j], i); qmax = fmaxf(qmax, fabsf(x)); qs += x; }
            qsc[sg][j] = warp_max(qmax) / 32639.0f;             // |q| <= 32639 units: both byte digits of 256 * hi + lo stay signed bytes
            if (warp == (sg * NQ + j) % S::WARPS && sg < nseg) {
                qs = warp_sum(qs);
                if (lane == 0) { sm.qscale[sg][j] = qsc[sg][j]; sm.qsum[sg][j] = qs; }
                float over = 1.0f;
                if constexpr (NQ > 1) {
                    const int e = __float_as_int(qsc[sg][j]) >> 23, ex = e == 0 || e == 255 ? 127 : e + 15;       // 32639 < 2^15; zero and infinity have no power of two
                    over = __int_as_float((254 - ex) << 23);
                    if (lane == 0) sm.qf[sg][D][j] = __int_as_float(ex << 23);
                }
                if (4 * lane < D)
#pragma unroll
                    for (int i = 0; i < 4; ++i) sm.qf[sg][4 * lane + i][j] = half_at(qrow[sg][j], i) * over;
            }
        }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int sg, ln, r, ch;
        word_of(tid + k * S::THREADS, sg, ln, r, ch);
        float sc = 0.f;
#pragma unroll
        for (int j = 0; j < NQ; ++j) if ((ln >> 3) == j) sc = sg ? qsc[SEGS - 1][j] : qsc[0][j];
        const float qinv = sc > 0.f ? 1.0f / sc : 0.f;
        uint32_t v = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int qi = __float2int_rn(half_at(qword[k], i) * qinv);
            qi = max(-32639, min(32639, qi));
            const int dg = ((ln >> 2) & 1) == 0 ? ((qi + 128) >> 8) : qi;     // 256 * hi + lo with lo in [-128, 127]
            v |= (uint32_t)(dg & 0xFF) << (8 * i);
        }
        if (sg < nseg) sm.qw[sg][r & 1][ln][r >> 1] = v;
    }
    if (tid == 0) sm.seg[S::WARPS] = -1;
    if (!CLUSTER)
        for (int i = tid; i < NQ * D; i += S::THREADS) (&sm.cross[0][0])[i] = 0.f;
    __syncthreads();

    // digit rows of the value weights this lane feeds: columns 0..3 of the first query of a pair, 4..7 of the second
    const bool wuse = NQ > 1 || fg < 4;
    const uint32_t wrow = smem_addr(&ws.wts[0][NQ > 1 ? fg >> 2 : 0][fg & 3][4 * ft]);
    uint32_t phase = 0;          // of the warp's two transaction barriers

    // The value sums of several tiles stay in integer accumulators (exact) as long as the tiles agree on the reference
    // of the exponentials and on the size of one fixed-point unit; they are added to ws.macc when one of the two changes.
    int acc[NP][MB][4];
#pragma unroll
    for (int pr = 0; pr < NP; ++pr)
#pragma unroll
        for (int mb = 0; mb < MB; ++mb) { acc[pr][mb][0] = 0; acc[pr][mb][1] = 0; acc[pr][mb][2] = 0; acc[pr][mb][3] = 0; }
    int held = 0;                // tiles in the accumulators, at most HELD_TILES
    float m_ref[NQ], wunit[NQ];  // exponentials are taken relative to this logit; weight of one fixed-point unit, a power of two
    float l_run[NQ], c_run[NQ];  // over this lane's tokens: sum of p, of p * (min + step/2) of the values
    auto flush = [&]() {
        // digits 2^24, 2^16, 2^8, 1: columns 0..3 (lanes ft = 0, 1) are the first query of a pair, columns 4..7 the second
        const float d0 = (ft & 1) ? 256.0f : 16777216.0f, d1 = (ft & 1) ? 1.0f : 65536.0f;
        __syncwarp();
#pragma unroll
        for (int pr = 0; pr < NP; ++pr) {
            float un = wunit[2 * pr];
            if constexpr (NQ > 1) { if (ft >= 2) un = wunit[2 * pr + 1]; }
            float* row = ws.macc[NQ > 1 ? 2 * pr + (ft >> 1) : 0];
#pragma unroll
            for (int mb = 0; mb < MB; ++mb)
#pragma unroll
                for (int s2 = 0; s2 < 2; ++s2) {
                    float v = fmaf((float)acc[pr][mb][2 * s2], d0, (float)acc[pr][mb][2 * s2 + 1] * d1);
                    v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                    if ((ft & 1) == 0 && (NQ > 1 || ft == 0)) row[v_channel<D>(mb, fg, s2)] += v * (v_high<D>(mb) ? 0.0625f * un : un);
                    acc[pr][mb][2 * s2] = 0; acc[pr][mb][2 * s2 + 1] = 0;
                }
        }
        held = 0;
        __syncwarp();
    };

    if (f >= f_end && lane == 0) sm.seg[warp] = -1;
#pragma unroll 1
    while (f < f_end) {          // once per (b,h) of the warp's piece: one or two times
    const int bh = bh_of(f), seg = bh - bh0, f_stop = CLUSTER || seg ? f_end : min(f_end, f_bound);
    float qscale[NQ], qsum[NQ], qtop = NQ == 1 ? 0.f : 2.0f;       // qtop: a bound on the entries of the queries as they are kept
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        qscale[j] = sm.qscale[seg][j];
        qsum[j] = sm.qsum[seg][j];
        if (NQ == 1) qtop = fmaxf(qtop, qscale[j] * 32639.0f);
        m_ref[j] = NEG; wunit[j] = 0.f; l_run[j] = 0.f; c_run[j] = 0.f;
    }
#pragma unroll 1
    for (; f < f_stop; f += stride) {
        const Lay lk = layout(tk), lv = layout(tv);
        const uint32_t tV = buf + STAGE - lv.nb - lv.lb;
        // the tile before is done with: this tile's values come in behind its keys, if there is room
        const bool besideV = lk.nb + lk.lb + lv.nb + lv.lb <= STAGE;
        if (besideV) stage(tV, lv, a.v, bh, tv, 1);
        const uint4 tk_next = fetch_tab(a.k.tile, f + stride);
        const Toks vt = fetch_toks(a.v, f);
        const bool has_next = f + stride < f_end;
        const int t0 = (CLUSTER ? f : f - bh * ntiles) * QAQ_TILE + 2 * lane;              // this lane's tokens: t0 and t0 + 1
        const bool val[2] = {t0 < T, t0 + 1 < T};
        int B[2], sl[2];             // width; slot (tokens that are not there: a place nobody reads)
        float step[2], mid[2];
        auto scalars = [&](const Toks& tt) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t mm = i ? tt.mm.y : tt.mm.x, bs = tt.b >> (16 * i);
                B[i] = val[i] ? (int)(bs & 15u) : 0;
                sl[i] = B[i] ? (int)((bs >> 8) & (QAQ_TILE - 1)) : QAQ_TILE;
                const float mn = __half2float(__ushort_as_half((unsigned short)(mm & 0xFFFF))), mx = __half2float(__ushort_as_half((unsigned short)(mm >> 16)));
                step[i] = val[i] ? qaqc::step_of(mn, mx, B[i]) : 0.f;
                mid[i] = val[i] ? fmaf(0.5f, step[i], mn) : 0.f;
            }
        };
        scalars(kt);
        *reinterpret_cast<float2*>(&ws.mid[2 * lane]) = make_float2(mid[0], mid[1]);
#pragma unroll
        for (int i = 0; i < NQ; ++i) *reinterpret_cast<uint4*>(&ws.kcorr[i][0][4 * lane]) = make_uint4(0u, 0u, 0u, 0u);
        bool landed = bar_wait(bar, phase & 1u);
        __syncwarp();

        // ---- K: integer dot products, list by list
        {
            uint32_t qa[P], qb[P];
            lds_words<P>(smem_addr(sm.qw[seg][0][lane]), qa);
            lds_words<P>(smem_addr(sm.qw[seg][1][lane]), qb);
            uint4 h = *reinterpret_cast<const uint4*>(ws.buf);
            if (!tk.y || !landed) h = make_uint4(0u, 0u, 0u, 0u);
            uint32_t dots = smem_addr(&ws.dot[0][0][0]);
#pragma unroll 1
            for (int pass = 0;; ++pass) {
                const Lists l = lists_of<P>(h, pass);
                k_list<D, 4, NQ>(buf + l.o4, l.n4, dots, qa, qb, fg, ft);
                k_list<D, 3, NQ>(buf + l.o3, l.n3, dots + l.n4 * 4 * NQ, qa, qb, fg, ft);
                k_list<D, 2, NQ>(buf + l.o2, l.n2, dots + (l.n4 + l.n3) * 4 * NQ, qa, qb, fg, ft);
                k_list<D, 1, NQ>(buf + l.o1, l.n1, dots + (l.n4 + l.n3 + l.n2) * 4 * NQ, qa, qb, fg, ft);
                if (pass || !h.y) break;
                dots += WS::DOTS * 4 * NQ;
            }
        }
        // ---- key outliers: q_ch * (x - mid) per token; up to 128 entries stay in registers between the two looks at them
        float kunit = 0.f;          // > 0: the corrections are one word in this unit (of a query over its power of two); < 0: two words
        if (tk.w && landed) {
            const uint32_t oc = tk.w, sc = min(min(oc, LIST_STAGED), lk.lb / 4 - (tk.z & 3u));       // entries, of which staged
            const uint32_t* list = reinterpret_cast<const uint32_t*>(ws.buf + lk.nb) + (tk.z & 3u);
            auto term = [&](uint32_t v, float inv, int& tok, float (&tm)[NQ]) {
                tok = (v >> 24) & (QAQ_TILE - 1);
                const float dx = (__half2float(__ushort_as_half((unsigned short)(v & 0xFFFF))) - ws.mid[tok]) * inv;
                const float* qv = &sm.qf[seg][(v >> 16) & (D - 1)][0];
#pragma unroll
                for (int j = 0; j < NQ; ++j) tm[j] = qv[j] * dx;
            };
            const uint32_t* all = a.k.outl + (size_t)bh * a.ocap + tk.z;
            const uint32_t top = sc == oc ? reinterpret_cast<const uint4*>(ws.buf)->w >> 16 : SMALL_MAX + 1;
            if (top <= SMALL_MAX) {
                float inv;
                fixed_unit(qtop * 2.0f * __half2float(__ushort_as_half((unsigned short)top)), inv, kunit);        // |x - mid| <= 2 top
                auto add = [&](const uint32_t* v, uint32_t i) {
                    int tok[TWO]; float tm[TWO][NQ];
#pragma unroll
                    for (int k = 0; k < TWO; ++k) term(v[k], inv, tok[k], tm[k]);
#pragma unroll
                    for (int k = 0; k < TWO; ++k)
#pragma unroll
                        for (int j = 0; j < NQ; ++j) if (i + 32u * k < sc) atomicAdd(&ws.kcorr[j][0][tok[k]], __float2int_rn(tm[k][j]));
                };
#pragma unroll 1
                for (uint32_t i = lane; i - lane < sc; i += 32 * TWO) {
                    uint32_t e[TWO];
#pragma unroll
                    for (int k = 0; k < TWO; ++k) e[k] = list[min(i + 32u * k, sc - 1)];
                    add(e, i);
                }
            } else {
                kunit = -1.0f;
                auto add = [&](uint32_t v) {
                    int tok; float tm[NQ];
                    term(v, 1.0f, tok, tm);
#pragma unroll
                    for (int j = 0; j < NQ; ++j) wide_add(&ws.kcorr[j][0][tok], &ws.kcorr[j][1][tok], tm[j] * (NQ == 1 ? 1.0f : sm.qf[seg][D][j]));
                };
#pragma unroll 1
                for (uint32_t i = lane; i < sc; i += 32) add(list[i]);
                if (sc < oc) unstaged(all, sc, oc, add);
            }
        }
        __syncwarp();
        // ---- logits of this lane's tokens
        float lg[NQ][2];
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const int2 k0 = *reinterpret_cast<const int2*>(&ws.kcorr[j][0][2 * lane]);
            const float ku = NQ == 1 ? kunit : kunit * sm.qf[seg][D][j];
            float kc[2] = {(float)k0.x * ku, (float)k0.y * ku};
            if (kunit < 0.f) {
                const int2 k1 = *reinterpret_cast<const int2*>(&ws.kcorr[j][1][2 * lane]);
                kc[0] = wide_sum(k0.x, k1.x); kc[1] = wide_sum(k0.y, k1.y);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int lo = ws.dot[0][sl[i]][j], hi = ws.dot[1][sl[i]][j];
                const int dot = lo + (B[i] > 4 ? hi << 4 : 0);       // a token that is not there has step 0
                const float qk = fmaf(qscale[j] * step[i], (float)dot, fmaf(mid[i], qsum[j], kc[i]));
                lg[j][i] = val[i] ? a.scale * qk : NEG;
                if (NQ == 1 && a.scores && !kept && val[i]) a.scores[(size_t)bh * a.scores_stride + t0 + i] = lg[j][i];
            }
            if (NQ == 1 && kept) *reinterpret_cast<float2*>(&ws.mid[2 * lane]) = make_float2(lg[j][0], lg[j][1]);
        }
        __syncwarp();
        // ---- the front of the buffer is free: start the copy of the next tile's keys (beside this tile's values)
        if (!besideV) stage(tV, lv, a.v, bh, tv, 1);
        const Lay ln = layout(tk_next);
        const bool besideK = ln.nb + ln.lb + lv.nb + lv.lb <= STAGE;
        if (has_next && besideK) stage(buf, ln, a.k, bh_of(f + stride), tk_next, 0);
        const uint4 tv_next = fetch_tab(a.v.tile, f + stride);
        kt = fetch_toks(a.k, f + stride);

        // ---- p relative to a reference somewhat above the largest logit, which is moved only when a logit exceeds it (so
        //      p never exceeds 1), and value weights p * step as fixed point of up to 28 bits.  (A token's step falls with
        //      its width, so next to a 2-bit token an 8-bit token of the same p has a weight 64 times smaller.)  The largest
        //      weight of every tile takes 21 bits or more: the unit stays while it takes between 2^21 and 2^28 units, and is
        //      set so that it takes 2^24 to 2^25.
        scalars(vt);
        float alpha[NQ], wnew[NQ];
        bool wok[NQ], any_w = false, change = held == HELD_TILES;
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const float m = warp_max(fmaxf(lg[j][0], lg[j][1]));
            alpha[j] = 1.0f;
            if (m > m_ref[j]) {
                alpha[j] = __expf(m_ref[j] - (m + 3.0f));       // 0 on the first tile
                m_ref[j] = m + 3.0f;
                change = true;
            }
            // from here on: p (0 for slots beyond T, and for a token whose logit is not a number: one with an infinite range)
            lg[j][0] = fmaxf(__expf(lg[j][0] - m_ref[j]), 0.f);
            lg[j][1] = fmaxf(__expf(lg[j][1] - m_ref[j]), 0.f);
            const float wmax = warp_max(fmaxf(lg[j][0] * step[0], lg[j][1] * step[1]));
            const int wex = (__float_as_int(wmax) >> 23) & 0xFF;
            wok[j] = wex > 28 && wex < 255 && tv.y;             // zero, tiny or non-finite weights: the codes add nothing
            any_w = any_w || wok[j];
            wnew[j] = wunit[j];
            if (wok[j] && !(wmax >= 2097152.0f * wunit[j] && wmax < 268435440.0f * wunit[j])) {
                wnew[j] = __int_as_float((wex - 24) << 23);
                change = true;
            }
        }
        if (change) {
            if (held) flush();
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                wunit[j] = wnew[j];
                if (alpha[j] != 1.0f) {
#pragma unroll
                    for (int k = 0; k < CPL; ++k) ws.macc[j][lane + 32 * k] *= alpha[j];
                    c_run[j] *= alpha[j]; l_run[j] *= alpha[j];
                }
            }
        }
        const bool wide = __any_sync(0xFFFFFFFFu, max(B[0], B[1]) > 4);
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const float winv = wok[j] ? __int_as_float((254 << 23) - __float_as_int(wunit[j])) : 0.f;       // 1 / wunit
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t iw = __float2uint_rn(lg[j][i] * step[i] * winv);
                uint8_t* gp = &ws.wts[0][j][0][sl[i]];
                gp[0] = (uint8_t)(iw >> 24);
                gp[WS::WROW] = (uint8_t)(iw >> 16);
                gp[2 * WS::WROW] = (uint8_t)(iw >> 8);
                gp[3 * WS::WROW] = (uint8_t)iw;
                if (wide) {                          // 16 times the weight, for the bits above the low four
                    gp += 4 * NQ * WS::WROW;
                    gp[0] = (uint8_t)(iw >> 20);
                    gp[WS::WROW] = (uint8_t)(iw >> 12);
                    gp[2 * WS::WROW] = (uint8_t)(iw >> 4);
                    gp[3 * WS::WROW] = (uint8_t)(iw << 4);
                }
            }
            const float c0 = lg[j][0] * mid[0], c1 = lg[j][1] * mid[1];
            c_run[j] += c0 + c1;
            l_run[j] += lg[j][0] + lg[j][1];
            *reinterpret_cast<float4*>(&ws.tok[j][2 * lane]) = make_float4(lg[j][0], c0, lg[j][1], c1);
        }
        landed = bar_wait(bar + 8, phase & 1u) && landed;     // this tile's values are there
        __syncwarp();

        // ---- V: integer weighted sums, list by list
        if (any_w && landed) {
            const uint4 h = *reinterpret_cast<const uint4*>(ws.buf + STAGE - lv.nb - lv.lb);
            uint32_t wt = wrow;
#pragma unroll 1
            for (int pass = 0;; ++pass) {
                const Lists l = lists_of<D / 8>(h, pass);
                v_list<D, 4, NQ>(tV + l.o4, l.n4, wt, wuse, acc, fg, ft);
                v_list<D, 3, NQ>(tV + l.o3, l.n3, wt + 4 * l.n4, wuse, acc, fg, ft);
                v_list<D, 2, NQ>(tV + l.o2, l.n2, wt + 4 * (l.n4 + l.n3), wuse, acc, fg, ft);
                v_list<D, 1, NQ>(tV + l.o1, l.n1, wt + 4 * (l.n4 + l.n3 + l.n2), wuse, acc, fg, ft);
                if (pass || !h.y) break;
                wt += 4 * NQ * WS::WROW;
            }
            ++held;
        }
        // ---- value outliers: p_t * (v - mid) per channel
        if (tv.w && landed) {
            const uint32_t oc = tv.w, sc = min(min(oc, LIST_STAGED), lv.lb / 4 - (tv.z & 3u));
            const uint32_t* list = reinterpret_cast<const uint32_t*>(ws.buf + STAGE - lv.lb) + (tv.z & 3u);
            auto term = [&](uint32_t v, int j) {
                const float2 pm = ws.tok[j][(v >> 24) & (QAQ_TILE - 1)];
                return fmaf(__half2float(__ushort_as_half((unsigned short)(v & 0xFFFF))), pm.x, -pm.y);
            };
            auto clear_vcorr = [&](int rows) {
                for (int i = 4 * lane; i < rows * D; i += 128) *reinterpret_cast<uint4*>(&ws.vcorr[0][0] + i) = make_uint4(0u, 0u, 0u, 0u);
            };
            const uint32_t* all = a.v.outl + (size_t)bh * a.ocap + tv.z;
            const uint32_t top = sc == oc ? reinterpret_cast<const uint4*>(ws.buf + STAGE - lv.nb - lv.lb)->w >> 16 : SMALL_MAX + 1;
            if (top <= SMALL_MAX) {
                float inv[NQ], unit[NQ];
                __syncwarp();
                clear_vcorr(NQ);
#pragma unroll
                for (int j = 0; j < NQ; ++j)
                    fixed_unit(warp_max(fmaxf(lg[j][0], lg[j][1])) * 2.5f * __half2float(__ushort_as_half((unsigned short)top)), inv[j], unit[j]);
                __syncwarp();
                auto add = [&](const uint32_t* v, uint32_t i) {
                    int x[TWO][NQ];
#pragma unroll
                    for (int k = 0; k < TWO; ++k)
#pragma unroll
                        for (int j = 0; j < NQ; ++j) x[k][j] = __float2int_rn(term(v[k], j) * inv[j]);
#pragma unroll
                    for (int k = 0; k < TWO; ++k)
#pragma unroll
                        for (int j = 0; j < NQ; ++j) if (i + 32u * k < sc) atomicAdd(&ws.vcorr[j][(v[k] >> 16) & (D - 1)], x[k][j]);
                };
#pragma unroll 1
                for (uint32_t i = lane; i - lane < sc; i += 32 * TWO) {
                    uint32_t e[TWO];
#pragma unroll
                    for (int k = 0; k < TWO; ++k) e[k] = list[min(i + 32u * k, sc - 1)];
                    add(e, i);
                }
                __syncwarp();
#pragma unroll
                for (int j = 0; j < NQ; ++j)
#pragma unroll
                    for (int k = 0; k < CPL; ++k) {
                        const int d = lane + 32 * k;
                        ws.macc[j][d] += (float)ws.vcorr[j][d] * unit[j];
                    }
            } else {
                constexpr int TOGETHER = NQ == 4 ? 2 : 1;             // queries whose two words have room
#pragma unroll 1
                for (int j = 0; j < NQ; j += TOGETHER) {
                    __syncwarp();
                    clear_vcorr(2 * TOGETHER);
                    __syncwarp();
                    auto add = [&](uint32_t v) {
                        const int ch = (v >> 16) & (D - 1);
#pragma unroll
                        for (int i = 0; i < TOGETHER; ++i) wide_add(&ws.vcorr[2 * i][ch], &ws.vcorr[2 * i + 1][ch], term(v, j + i));
                    };
#pragma unroll 1
                    for (uint32_t i = lane; i < sc; i += 32) add(list[i]);
                    if (sc < oc) unstaged(all, sc, oc, add);
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < TOGETHER; ++i)
#pragma unroll
                        for (int k = 0; k < CPL; ++k) {
                            const int d = lane + 32 * k;
                            ws.macc[j + i][d] += wide_sum(ws.vcorr[2 * i][d], ws.vcorr[2 * i + 1][d]);
                        }
                }
            }
        }
        __syncwarp();
        if (has_next && !besideK) stage(buf, ln, a.k, bh_of(f + stride), tk_next, 0);
        if (!landed) atomicMax(a.status, (int)QAQ_ERR_CUDA);
        phase ^= 1u;
        tk = tk_next;
        tv = tv_next;
    }
    if (held) flush();
    // ---- what the warp has of this (b,h)
    const bool cross = !CLUSTER && f < f_end;                     // it goes on in the next one
    const int entry = cross ? S::WARPS : warp;
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        const float l = warp_sum(l_run[j]), cs = warp_sum(c_run[j]);
        if (lane == 0) { sm.mm[entry][j] = m_ref[j]; sm.ml[entry][j] = l; sm.cs[entry][j] = cs; }
        if (cross) {
#pragma unroll
            for (int k = 0; k < CPL; ++k) { sm.cross[j][lane + 32 * k] = ws.macc[j][lane + 32 * k]; ws.macc[j][lane + 32 * k] = 0.f; }
        }
    }
    if (lane == 0) sm.seg[entry] = seg;
    __syncwarp();
    }
    __syncthreads();
    if (CLUSTER) cluster_wait();         // (all CTAs of the cluster run: what follows writes to them)
    // ---- merge the warps (log-sum-exp) into the partials of the (b,h): lane i knows the weight of entry i
#pragma unroll 1
    for (int seg = 0; seg < nseg; ++seg) {
        const int bh = bh0 + seg;
        const bool alone = !CLUSTER && min(flat_hi, (bh + 1) * ntiles) - max(flat_lo, bh * ntiles) == ntiles;        // nothing to merge with
        const bool mine = lane <= S::WARPS && sm.seg[min(lane, S::WARPS)] == seg;
#pragma unroll 1
        for (int j = 0; j < gr.nq; ++j) {
            const float m = mine ? sm.mm[lane][j] : NEG, M = warp_max(m);
            const float wgt = m == NEG ? 0.f : __expf(m - M);
            const float L = warp_sum(mine ? wgt * sm.ml[lane][j] : 0.f);
            float x = warp_sum(mine ? wgt * sm.cs[lane][j] : 0.f);
            const int d = tid < D ? tid : 0;
#pragma unroll
            for (int i = 0; i < S::WARPS; ++i) x = fmaf(__shfl_sync(0xFFFFFFFFu, wgt, i), sm.ws[i].macc[j][d], x);
            if (!CLUSTER) x = fmaf(__shfl_sync(0xFFFFFFFFu, wgt, S::WARPS), sm.cross[j][d], x);
            float* dst = gr.part + ((size_t)(2 * blockIdx.x + seg) * NQ + j) * (D + 4);
            if (alone) {
                if (tid < D) gr.out[(size_t)bh * a.out_stride + j * D + tid] = L > 0.f ? x / L : 0.f;
                if (NQ == 1) {
                    if (a.ml && tid == 0) { a.ml[2 * bh] = M; a.ml[2 * bh + 1] = L; }
                    if (a.scores && !a.ml) normalise_scores<S::THREADS>(a.scores + (size_t)bh * a.scores_stride, T, M, L);
                }
            } else if (CLUSTER) {
                if (tid < D) peer_store(&sm.from_sum[j / ncl * ncl + rank][tid], j % ncl, x);
                if (tid < ncl) peer_store(&sm.from_ml[j][rank], tid, M, L);
            } else {
                if (tid < D) __stcg(dst + tid, x);
                if (tid == 0) __stcg(reinterpret_cast<float2*>(dst + D), make_float2(M, L));
            }
        }
    }
    if (CLUSTER) {
        merge_cluster<D, NQ>(a, sm, gr, bh0, rank, T, kept);
        return;
    }
    __syncthreads();
    if (lane == 0 && warp < nseg) {
        int first, n;
        split_of(bh0 + warp, ntiles, run, first, n);
        sm.last[warp] = n > 1 && count_partial(gr.done + bh0 + warp, n);
    }
    __syncthreads();
#pragma unroll 1
    for (int seg = 0; seg < nseg; ++seg)
        if (sm.last[seg]) merge_split<D, NQ>(a, sm, bh0 + seg, ntiles, run, T);
}

// Score rows too long for one CTA to normalise on the side.
__global__ void scores_kernel(float* scores, long stride, const float* ml, int T, const int* d_count) {
    qaq_dependency();
    const int bh = blockIdx.y;
    if (d_count) T = *d_count;
    const float M = ml[2 * bh], L = ml[2 * bh + 1];
    const float inv = L > 0.f ? 1.0f / L : 0.f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
        float* s = scores + (size_t)bh * stride + t;
        *s = __expf(*s - M) * inv;
    }
}

// bytes of workspace: the partials of split (b,h) (two slots per CTA; a grid of more than SLOTS CTAs splits none), the
// counting words, the merged (max, sum) pairs
template <int NQ>
size_t decode_ws_bytes(int BH, int D, int groups) {
    return (size_t)2 * Shape<NQ>::SLOTS * NQ * (D + 4) * sizeof(float) + (size_t)BH * (groups * sizeof(unsigned long long) + 2 * sizeof(float));
}

// a number no other call of this process uses (splitmix64 of a counter that starts at the clock), the low 12 bits zero
unsigned long long call_tag() {
    static std::atomic<unsigned long long> next{(unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count()};
    unsigned long long z = next.fetch_add(1, std::memory_order_relaxed) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = (z ^ (z >> 31)) & ~0xFFFull;
    return z ? z : 0x1000ull;
}

template <int D, int NQ, bool COUNTED>
qaq_status launch_decode(DecArgs a, cudaStream_t s) {
    const size_t smem = sizeof(DecSmem<D, NQ>);
    static_assert(sizeof(DecSmem<D, NQ>) + 1024 <= 227 * 1024 / Shape<NQ>::CTAS_PER_SM, "shared memory of the CTAs of an SM");
    static SmemSeen seen[2];
    static ClusterRoom room;
    QAQ_CUDA_TRY(qaq_allow_smem((const void*)decode_kernel<D, NQ, COUNTED, true>, smem, seen[1]));
    a.cluster = plan_cluster<NQ>(a.BH, (a.T + QAQ_TILE - 1) / QAQ_TILE, a.groups, [&](int k) {
        return clusters_at_once(decode_kernel<D, NQ, COUNTED, true>, Shape<NQ>::THREADS, smem, k, room);
    });
    if (a.cluster) a.ncta = a.BH * a.cluster;
    const dim3 grid(a.ncta, a.groups), block(Shape<NQ>::THREADS);
    if (a.cluster) {
        QAQ_CUDA_TRY(qaq_launch_cluster(decode_kernel<D, NQ, COUNTED, true>, grid, block, a.cluster, smem, s, a));
    } else {
        QAQ_CUDA_TRY(qaq_allow_smem((const void*)decode_kernel<D, NQ, COUNTED, false>, smem, seen[0]));
        QAQ_CUDA_TRY(qaq_launch(decode_kernel<D, NQ, COUNTED, false>, grid, block, smem, s, a));
    }
    if (NQ == 1 && a.ml) {
        int gx = (a.T + 1023) / 1024;     // counted: a.T holds the capacity
        if (gx > 64) gx = 64;
        QAQ_CUDA_TRY(qaq_launch(scores_kernel, dim3(gx, a.BH), dim3(256), 0, s, a.scores, a.scores_stride, a.ml, a.T, COUNTED ? a.d_count : nullptr));
    }
    return QAQ_OK;
}

// nq queries per (b,h), NQ to a CTA (D elements apart inside a row of q and of out; rows of consecutive (b,h) lie q_stride /
// out_stride elements apart); counted: the token count is taken from device memory
template <int NQ, bool COUNTED>
qaq_status decode(const qaq_cache* c, const void* q, long q_stride, float softmax_scale, float* out, long out_stride, float* scores,
                  long scores_stride, void* ws, cudaStream_t s, int nq = NQ) {
    const int D = c->cfg.head_dim, BH = c->BH;
    DecArgs a;
    a.k = c->t[0]; a.v = c->t[1]; a.pool_bytes = c->pool_bytes; a.ocap = c->ocap;
    a.tmax_pad = c->tmax_pad; a.ntiles_max = c->ntiles;
    a.T = COUNTED ? (int)c->cfg.max_tokens : (int)c->tokens;
    a.d_count = COUNTED ? qaq_d_count(c) : nullptr;
    a.q = (const __half*)q; a.q_stride = q_stride; a.scale = softmax_scale;
    a.out = out; a.out_stride = out_stride; a.scores = scores; a.scores_stride = scores_stride; a.status = c->d_status;
    a.nq = nq;
    a.groups = (nq + NQ - 1) / NQ;
    const DecPlan plan = plan_decode<NQ>(BH, (a.T + QAQ_TILE - 1) / QAQ_TILE, a.groups);
    a.BH = BH;
    a.run = COUNTED ? 0 : plan.run;
    a.ncta = COUNTED ? (BH > Shape<NQ>::SLOTS ? BH : Shape<NQ>::SLOTS) : plan.ncta;   // counted: the largest grid any count needs
    a.cluster = 0;               // (launch_decode)
    // nothing in the workspace is read before it is written (the counting words: see merge_split)
    a.part = (float*)ws;
    a.done = (unsigned long long*)(a.part + (size_t)(BH > Shape<NQ>::SLOTS ? 0 : 2 * Shape<NQ>::SLOTS) * NQ * (D + 4));
    a.tag = call_tag();
    a.ml = scores && a.T > SCORES_FUSED_TOKENS ? (float*)(a.done + BH) : nullptr;
    switch (D) {
        case 32: return launch_decode<32, NQ, COUNTED>(a, s);
        case 64: return launch_decode<64, NQ, COUNTED>(a, s);
        case 128: return launch_decode<128, NQ, COUNTED>(a, s);
    }
    return QAQ_ERR_UNSUPPORTED_SHAPE;
}

}  // namespace

extern "C" qaq_status qaq_decode_workspace_bytes(const qaq_cache* c, size_t* host_out) {
    if (!c || !host_out) return QAQ_ERR_INVALID_ARG;
    *host_out = decode_ws_bytes<1>(c->BH, c->cfg.head_dim, 1);
    return QAQ_OK;
}

extern "C" qaq_status qaq_decode_attention(const qaq_cache* c, const void* q, float softmax_scale, float* out,
                                           float* scores_out, void* ws, size_t ws_bytes, void* stream) {
    if (!c || !q || !out || !ws) return QAQ_ERR_INVALID_ARG;
    if (c->tokens < 1) return QAQ_ERR_INVALID_ARG;
    size_t need = 0;
    qaq_decode_workspace_bytes(c, &need);
    if (ws_bytes < need || ((uintptr_t)ws & 15)) return QAQ_ERR_WORKSPACE;
    return decode<1, false>(c, q, c->cfg.head_dim, softmax_scale, out, c->cfg.head_dim, scores_out, c->tokens, ws, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------------------
// Several queries per (b,h): one, two, or three and four (one launch: at 256 (b,h) of 4096 tokens 110 us against 114 us for
// three queries as two and one, at 40 of 380 tokens 20 against 23 us).  Five to eight are two groups of up to four, either side
// by side in one launch or one after the other (a second group of one or two queries as what it is): the first has one
// start and one end and cuts finer (16 (b,h) of 10175 tokens, five queries: 41 against 59 us; 24 of 2000 tokens: 21 against
// 30 us), the other does not read every code with four queries' instructions for the sake of one or two (256 (b,h) of 4096
// tokens: 161 against 262 us) and is needed where half of the chip has fewer places than there are (b,h).
static bool side_by_side(int BH, int ntiles, int n) {
    const DecPlan both = plan_decode<4>(BH, ntiles, 2), four = plan_decode<4>(BH, ntiles, 1), few = plan_decode<1>(BH, ntiles, 1);
    if (both.ncta > Shape<4>::SLOTS / 2) return false;
    // tiles per warp; a tile takes a warp about 11 us with four queries, half of that with one or two; a launch costs as much again
    auto tiles = [](int run, int warps) { return (run + warps - 1) / warps; };
    const int w4 = tiles(four.run, Shape<4>::WARPS);
    return 2 * tiles(both.run, Shape<4>::WARPS) <= 2 * w4 + (n > 6 ? 2 * w4 : tiles(few.run, Shape<1>::WARPS)) + 2;
}

// Where many entries are outliers, their sums are most of the time, and four queries take longer for them than twice two: three,
// five and six queries are taken two at a time from 10 % on, four from 20 % (32 (b,h) of 4096 tokens, 8 bits, 10 %: three 70 us
// at once and 59 as two and one, five 118 and 94, four 70 and 71, eight 120 and 142; 4 bits, 50 %: three 381 and 279, four 381
// and 361).
static bool in_twos(double outlier_frac, int left) {
    return left <= 6 && outlier_frac >= (left == 4 ? 0.2 : 0.1);
}

extern "C" qaq_status qaq_decode_multi_workspace_bytes(const qaq_cache* c, size_t* host_out) {
    if (!c || !host_out) return QAQ_ERR_INVALID_ARG;
    const int D = c->cfg.head_dim, BH = c->BH;       // the passes of a call reuse the space
    const size_t b1 = decode_ws_bytes<1>(BH, D, 1), b2 = decode_ws_bytes<2>(BH, D, 1), b4 = decode_ws_bytes<4>(BH, D, 2);
    *host_out = b1 > b2 ? (b1 > b4 ? b1 : b4) : (b2 > b4 ? b2 : b4);
    return QAQ_OK;
}

extern "C" qaq_status qaq_decode_attention_multi(const qaq_cache* c, const void* q, int n_q, float softmax_scale, float* out,
                                                 void* ws, size_t ws_bytes, void* stream) {
    if (!c || !q || !out || !ws || n_q < 1 || n_q > 8) return QAQ_ERR_INVALID_ARG;
    if (c->tokens < 1) return QAQ_ERR_INVALID_ARG;
    size_t need = 0;
    qaq_decode_multi_workspace_bytes(c, &need);
    if (ws_bytes < need || ((uintptr_t)ws & 15)) return QAQ_ERR_WORKSPACE;
    const int D = c->cfg.head_dim;
    const long row = (long)n_q * D;
    cudaStream_t s = (cudaStream_t)stream;
    const int ntiles = (int)((c->tokens + QAQ_TILE - 1) / QAQ_TILE);
    for (int q0 = 0; q0 < n_q;) {
        const int left = n_q - q0;
        const __half* qp = (const __half*)q + (size_t)q0 * D;
        float* op = out + (size_t)q0 * D;
        const int n = in_twos(c->cfg.outlier_frac, left) ? (left < 2 ? left : 2) : left > 4 && !side_by_side(c->BH, ntiles, left) ? 4 : left;
        const qaq_status st = n >= 3 ? decode<4, false>(c, qp, row, softmax_scale, op, row, nullptr, 0, ws, s, n)
                              : n == 2 ? decode<2, false>(c, qp, row, softmax_scale, op, row, nullptr, 0, ws, s)
                                       : decode<1, false>(c, qp, row, softmax_scale, op, row, nullptr, 0, ws, s);
        if (st != QAQ_OK) return st;
        q0 += n;
    }
    return QAQ_OK;
}

// ---------------------------------------------------------------------------------------
// Decode attention for callers that have no way to hand over a workspace.
//
// The split partials of the decode kernel need a few hundred KB of global scratch.  The
// regular entry point takes it from the caller; this one keeps it in a fixed array that
// is part of the library image, so the call itself never asks the CUDA allocator (or any
// other allocator) for memory.
#define QAQ_STATIC_SCRATCH_BYTES (4u << 20)
static __device__ __align__(256) unsigned char g_decode_scratch[QAQ_STATIC_SCRATCH_BYTES];

static std::mutex g_scratch_mutex;
static void* g_scratch_addr[64];  // device address of g_decode_scratch, per device ordinal

// the documented limit: what two partials per CTA of a split into at most 592 (or one per (b,h)) and a pair of words
// per (b,h) would take; decode_ws_bytes<1> never needs more than 4 MiB within it
static bool static_scratch_fits(int BH, long tokens, int D) {
    const long ntiles = (tokens + QAQ_TILE - 1) / QAQ_TILE;
    const long long total = (long long)BH * ntiles, floor_run = ntiles < 4 ? ntiles : 4;
    long long run = (total + 591) / 592;
    run = run < floor_run ? floor_run : (run > ntiles ? ntiles : run);
    const long long ncta = (total + run - 1) / run;
    return ((size_t)2 * ncta * (D + 3) + (size_t)BH * 2) * sizeof(float) <= QAQ_STATIC_SCRATCH_BYTES;
}

extern "C" qaq_status qaq_decode_attention_static(const qaq_cache* c, const void* q, float softmax_scale,
                                                  float* out, void* stream) {
    if (!c || !q || !out) return QAQ_ERR_INVALID_ARG;
    if (c->tokens < 1) return QAQ_ERR_INVALID_ARG;
    const int D = c->cfg.head_dim;
    if (!static_scratch_fits(c->BH, c->tokens, D)) return QAQ_ERR_WORKSPACE;  // shape too large for the built-in scratch

    int dev = -1;
    QAQ_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return QAQ_ERR_UNSUPPORTED_SHAPE;
    void* scratch = nullptr;
    {
        // In host code the array's name is only a handle; the device address has to be
        // looked up, once per device, with that device current.
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        if (!g_scratch_addr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_decode_scratch) != cudaSuccess || !p) {
                (void)cudaGetLastError();
                return QAQ_ERR_CUDA;
            }
            g_scratch_addr[dev] = p;
        }
        scratch = g_scratch_addr[dev];
    }
    return decode<1, false>(c, q, D, softmax_scale, out, D, nullptr, 0, scratch, (cudaStream_t)stream);
}

// Decode attention over as many tokens as the device-side count says (qaq_stream_begin / qaq_stream_append): the
// split over CTAs is derived from the count inside the kernels, the grid is the largest any count needs, and nothing
// on the host is read or changed, so the call can be captured in a CUDA graph and replayed while the cache grows.
extern "C" qaq_status qaq_stream_decode(const qaq_cache* c, const void* q, float softmax_scale, float* out,
                                        float* scores_out, long scores_stride, void* ws, size_t ws_bytes, void* stream) {
    if (!c || !q || !out || !ws) return QAQ_ERR_INVALID_ARG;
    if (scores_out && scores_stride < c->cfg.max_tokens) return QAQ_ERR_INVALID_ARG;
    size_t need = 0;
    qaq_decode_workspace_bytes(c, &need);
    if (ws_bytes < need || ((uintptr_t)ws & 15)) return QAQ_ERR_WORKSPACE;
    return decode<1, true>(c, q, c->cfg.head_dim, softmax_scale, out, c->cfg.head_dim, scores_out, scores_stride, ws, (cudaStream_t)stream);
}
