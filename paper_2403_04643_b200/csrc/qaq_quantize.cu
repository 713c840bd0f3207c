// S1-S3: bit-width selection, outlier split, uniform quantization and bit-packing.
//
// One CTA handles one tile (QAQ_TILE consecutive tokens) of one (b,h) and tensor; K and V are read from HBM once.
//   loads    the tokens' rows to shared memory; the attention-window maximum of a token by its thread (Section 4.2)
//   pass 1   outlier masks and min/max of the non-outliers in binary16 pair arithmetic (exact: the inputs are
//            binary16); the outliers listed; width from the exponents (Section 4.1)
//   order    the tokens sorted by width, sections and size of the tile, space taken from the (b,h) pools
//   pass 2   codes (binary32: one sub, one mul, round down), packed words to the section layout of qaq_codec.cuh;
//            outlier entries, per-token metadata, the tile's table entry
// A tile that is continued (an append behind a partly filled tile) is built anew: the words of its old tokens come
// from the tile as it is stored and go to their new places without becoming codes.
#include "qaq_codec.cuh"
#include "qaq_internal.cuh"

namespace {

struct QuantArgs {
    const __half* K;
    const __half* V;
    long sb, sh, st;       // element strides of K/V (batch, head, token)
    int H;                 // heads
    int n_new;             // tokens per (b,h) in K/V (and in bits/ring/nvalid rows)
    int t_old;             // tokens already cached (0 for selection only)
    int tok_lo, tok_hi;    // new-token index range handled by this launch
    int first_tile;        // absolute index of the first tile touched by this launch
    const uint8_t* bitsK;  // given widths [BH][n_new] or null
    const uint8_t* bitsV;
    const float* ring;     // [BH][W][n_new]
    const uint8_t* nvalid; // [BH][n_new]
    int W;
    const float* thr;      // [BH][4]
    float cK, cV;
    int bmin, bmax;
    TensorStore k, v;
    size_t pool_bytes;
    uint32_t ocap;
    int tmax_pad, ntiles;
    int* status;
    int* d_count;          // null, or the token count kept in device memory: read instead of t_old / first_tile and
    unsigned* d_ticket;    //   advanced by the last CTA of the launch to have read it (one-token appends)
    int max_tokens;
    uint8_t* out_bitsK;    // selection only
    uint8_t* out_bitsV;
    uint32_t k64 = 65536, k16 = 16;      // multipliers that the compiler is not to know (see code_pair)
};

using qaqc::ladder;

__device__ __forceinline__ __half2 as_h2(uint32_t x) { return *reinterpret_cast<__half2*>(&x); }
__device__ __forceinline__ uint32_t as_u32(__half2 x) { return *reinterpret_cast<uint32_t*>(&x); }
// Space for a whole tile from a (b,h) pool: a rounded-up amount in one atomic.  `taken` is what the pool end moved by (to be
// given back if the space turns out not to fit: pool_give_back).  full: the pool end already lay beyond the pool when the
// CTA began; nothing is taken, so that the end cannot run away.
__device__ __forceinline__ uint32_t pool_take(uint32_t* pool, uint32_t amount, uint32_t unit_mask, bool full, uint32_t& taken) {
    taken = full ? 0u : (amount + unit_mask) & ~unit_mask;
    return full ? 0xFFFF0000u : atomicAdd(pool, taken);
}

// ------------------------------------------------------------------------------------------ whole tiles, two warps each
// A tile of one tensor comes to shared memory by asynchronous copies and is gone through twice: tokens in order for the
// ranges and the outliers, then, with the widths known, tokens in the order they are stored in for the codes, which go
// straight to their places (a round's lanes mostly have the same width, so they seldom part at the stores; four tokens of
// a group of values swap bytes by shuffles).  What is done once per tile - the order, the sections, the space from the
// pools - is done for 64 tokens by 64 threads.
//
// What bounds it: instructions (70 % of the issue slots, 60 % of the integer unit's cycles at 7B, batch 8).  A kernel with
// 256 threads per tile, a lane per 32 channels of a token throughout and an image of the tile in shared memory took
// 7300 (keys) and 9100 (values) warp instructions per tile, this one 4400 on average.  4096 tokens, 256 (b,h), head_dim
// 128: 173 us for keys and values, against 323 us; one warp per tile 231 us (as many tiles in flight per SM, for their
// shared memory); rounds unrolled by two 7 % slower, by four 20 % (the code of one round is what the instruction cache
// holds); the window in batches of 16 loads 3 % slower, eleven CTAs per SM 3 %.  32 (b,h) of one tile 7.0 against 7.7 us, of 16 tiles 10.5 against 17.2 us.
// A one-token append is a chain of memory latencies (token count; table and metadata; the tile) and of instructions: eight
// warps share pass 2, a round each, and nothing but the tile itself waits for the table.  32 (b,h), a tile of 1 to 64
// tokens, captured: 5.5 us, 5.8 with four warps; where not all CTAs of eight warps run at once (96 registers: two to an SM) four are
// better: 148 (b,h) 7.1 and 7.4, 160 9.6 and 7.5, 256 10.3 and 7.7, 512 18.8 and 12.0.
// The integer unit limits this kernel (compares, minima, byte shuffles and selects all run there, at half rate), so sums,
// shifts and packing are put where the multipliers are.
__device__ __forceinline__ uint64_t pair_of(float a, float b) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ uint32_t mad(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
struct Scale {                 // of a token: code = min(floor((x - mn) * inv), 2^B - 1)
    float mn;
    uint64_t inv;              // the reciprocal of the step, twice; 0 for a constant token
    uint32_t top;              // 2^B - 1 in the low half, that and the bits of 2^23 in the high half
    uint32_t k64;              // 65536, kept from the compiler, which would take a byte shuffle
};
// Codes of a binary16 pair: the first in the low byte, the second in byte 2 (byte 3 is not clean).  2^23 + floor(t) has
// the code in its low bits; an outlier's place holds the minimum, which has code 0.
__device__ __forceinline__ uint32_t code_pair(uint32_t v, const Scale& s) {
    float x0, x1;
    asm("{\n.reg .b16 h0, h1;\nmov.b32 {h0, h1}, %2;\nsub.rn.f32.f16 %0, h0, %3;\nsub.rn.f32.f16 %1, h1, %3;\n}" : "=f"(x0), "=f"(x1) : "r"(v), "f"(s.mn));
    uint64_t t;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(pair_of(x0, x1)), "l"(s.inv));
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(t) : "l"(t), "l"(pair_of(8388608.0f, 8388608.0f)));
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(mad((uint32_t)(t >> 32), s.k64, (uint32_t)t)), "r"(s.top));
    return d;
}
constexpr uint32_t GONE = 0xFFFFu;      // in the place of an outlier of a token whose range is not finite: not a number

// What a warp keeps of its tile in shared memory.  The 16-byte pieces of the rows are stored swizzled (piece U at U ^ (U/8
// mod 4)), so that lanes that read 64 bytes each do not meet in the banks.
template <int D>
struct TileScratch {
    alignas(64) uint8_t data[QAQ_TILE * D * 2];
    union {                            // one after the other
        alignas(16) uint32_t out[QAQ_TILE * D / 32];   // by token and 32 channels: which are outliers
        uint4 slot[QAQ_TILE];          // by slot: minimum, 1 / step, byte offsets of the parts, what else a lane has to know
    };
    uint32_t range[QAQ_TILE];          // by token: min | max << 16
    alignas(8) uint32_t count[2][2];   // by half of the tile: tokens of every width, a byte each
    uint32_t nout[2], top[2], base[2]; // outliers of the halves, largest magnitudes of their new tokens; space taken for the tile and for its outlier list
    int skip;
};
__device__ __forceinline__ uint4 lds4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void load_row(uint32_t addr, uint32_t (&v)[16]) {     // a lane's 64 bytes of a swizzled row
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 x = lds4(addr ^ (16 * i));
        v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
    }
}
// Range of the inliers of 32 channels and, in channel order, which of them are outliers.
__device__ __forceinline__ uint32_t outliers_and_range(const uint32_t (&v)[16], __half2 lo2, __half2 hi2, __half2& mn2, __half2& mx2) {
    __half2 mn = as_h2(0x7C007C00u), mx = as_h2(0xFC00FC00u);
    int out[4] = {255, 255, 255, 255};     // eight channels each; an inlier (all ones, -1) takes its bit away
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t m = __hge2_mask(as_h2(v[k]), lo2) & __hle2_mask(as_h2(v[k]), hi2);
        const __half2 x = as_h2(v[k] | ~m);                // not a number: passed over by both
        mn = __hmin2(mn, x);
        mx = __hmax2(mx, x);
        asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(out[k >> 2]) : "r"(m), "r"(0x00020001u << (2 * (k & 3))));
    }
    mn2 = mn; mx2 = mx;
    return qaqc::prmt(qaqc::prmt((uint32_t)out[0], (uint32_t)out[1], 0x0040u), qaqc::prmt((uint32_t)out[2], (uint32_t)out[3], 0x0040u), 0x5410u);
}
// of a token, from those of its P lanes: min | max << 16; 0, 0 where there is no inlier
template <int P>
__device__ __forceinline__ uint32_t range_of_token(__half2 mn2, __half2 mx2) {
    __half2 pk = __halves2half2(__hmin(__low2half(mn2), __high2half(mn2)), __hneg(__hmax(__low2half(mx2), __high2half(mx2))));
#pragma unroll
    for (int o = 1; o < P; o <<= 1) pk = __hmin2(pk, as_h2(__shfl_xor_sync(0xFFFFFFFFu, as_u32(pk), o)));
    return __hgt(__low2half(pk), __hneg(__high2half(pk))) ? 0u : as_u32(pk) ^ 0x80000000u;
}
// exclusive prefix over the lanes, and the sum
__device__ __forceinline__ uint32_t prefix(uint32_t x, int lane, uint32_t& sum) {
    uint32_t inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += o;
    }
    sum = __shfl_sync(0xFFFFFFFFu, inc, 31);
    return inc - x;
}
constexpr uint32_t STORED = 1u << 30;   // of a slot's last word: the token is taken from the stored tile

// One tile of one tensor, by two warps: half of its tokens each until the widths are known, half of the slots each from there.
// By NW warps.  OPEN: a tile that is begun, continued or closed, the only one of its (b,h) in the
// launch: its tokens up to s_lo are cached already (and come from the tile as it is stored), those from s_lo to s_hi are new.
template <int D, bool IS_V, bool OPEN, int NW>
__device__ __forceinline__ void quantize_tile(const QuantArgs& a, TileScratch<D>& sm, uint8_t* stored_tile, uint32_t* list, const uint32_t cap) {
    constexpr int P = D / 32, TPI = 32 / P, IT = QAQ_TILE / 2 / TPI;  // lanes per token, tokens of a warp at a time, rounds
    constexpr int PR = D / 8;                                         // 16-byte pieces of a row
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane / P, p = lane % P;
    const bool counted = OPEN && a.d_count;
    const int t_old = counted ? *a.d_count : a.t_old;
    if (counted && t_old + a.tok_hi > a.max_tokens) {       // no room: nothing is stored, the count stays
        if (tid == 0) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
        return;
    }
    const int tile = (counted ? t_old / QAQ_TILE : a.first_tile) + blockIdx.x, bh = blockIdx.y, tn0 = tile * QAQ_TILE - t_old;
    const int s_lo = OPEN ? max(0, a.tok_lo - tn0) : 0, s_hi = OPEN ? min(QAQ_TILE, a.tok_hi - tn0) : QAQ_TILE;
    const bool old = OPEN && tid < s_lo, fresh = !OPEN || (tid >= s_lo && tid < s_hi);      // this thread's token
    const TensorStore& ts = IS_V ? a.v : a.k;
    const bool main = !OPEN || warp < 2;                   // the threads of the 64 tokens; the others of an open tile help with the codes
    const size_t mt = (size_t)bh * a.tmax_pad + (size_t)tile * QAQ_TILE + tid;
    uint4* const tab = ts.tile + (size_t)bh * a.ntiles + tile;
    const __half* X = (IS_V ? a.V : a.K) + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh + (ptrdiff_t)tn0 * a.st;
    const uint32_t data = (uint32_t)__cvta_generic_to_shared(sm.data);
    // ---- all loads that wait for nothing else
    uint4 tw = make_uint4(0u, 0u, 0u, 0u);
    uint32_t bs_old = 0;
    if (OPEN && s_lo > 0) tw = *tab;
    if (OPEN && old) bs_old = ts.bs[mt];
    const float* thr = a.thr + (size_t)bh * 4 + (IS_V ? 2 : 0);
    const float thr_lo = thr[0], thr_hi = thr[1];
    uint32_t* const pool = (lane ? ts.opool_end : ts.pool_end) + bh;
    uint32_t pool_now = 0;
    if (tid < 2) pool_now = *pool;
    const bool given = a.bitsK != nullptr;
    const int col = OPEN ? min(max(tn0 + tid, 0), a.n_new - 1) : tn0 + tid;       // whole warps read; not every thread has a new token
    int b = 0, nv = 0;
    if (main) {
        if (given) b = (IS_V ? a.bitsV : a.bitsK)[(size_t)bh * a.n_new + col];
        else if (IS_V) nv = a.nvalid[(size_t)bh * a.n_new + col];
        const int row = 32 * warp + lane / PR;
        const __half* src = X + (ptrdiff_t)row * a.st + 8 * (lane % PR);
        const uint32_t dst = data + warp * (QAQ_TILE * D) + 16 * (lane ^ ((lane >> 3) & 3));
#pragma unroll
        for (int i = 0; i < PR; ++i, src += (32 / PR) * a.st)
            if (!OPEN || (row + i * (32 / PR) >= s_lo && row + i * (32 / PR) < s_hi))
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * i), "l"(src) : "memory");
    }
    // ---- attention window of this thread's token
    float shat = __int_as_float(0xff800000);
    if (IS_V && !given && main) {
        nv = min(nv, a.W);
        const float* scores = a.ring + (size_t)bh * a.W * a.n_new + col;
        shat = OPEN ? qaqc::window_max_one_loop<32>(scores, a.W, a.n_new, nv) : qaqc::window_max<32>(scores, a.W, a.n_new, nv);
    }
    if (OPEN) {                        // the tile as it is stored follows on its own: it is needed later
        asm volatile("cp.async.commit_group;" ::: "memory");
        const uint8_t* src = ts.codes + (size_t)bh * a.pool_bytes + tw.x;
        for (uint32_t o = tid * 16; o < min(tw.y, (uint32_t)qaqc::tile_bytes_max(D)); o += 64 * NW / 2 * 16)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(stored_tile + o)), "l"(src + o) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // thresholds as binary16 bounds that decide exactly like the binary32 ones on binary16 data
    const __half2 lo2 = __half2half2(__float2half_ru(thr_lo)), hi2 = __half2half2(__float2half_rd(thr_hi));
    if (OPEN) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();

    // ---- ranges and outliers, tokens in order: an outlier goes to the warp's list, its place is marked
    list += warp * cap;
#pragma unroll 1
    for (int it = 0; it < IT; ++it) {
        if (OPEN && !main) break;
        if (OPEN && (32 * warp + it * TPI >= s_hi || 32 * warp + (it + 1) * TPI <= s_lo)) continue;        // no new token among them
        const int tok = 32 * warp + it * TPI + g, U = tok * PR + 4 * p;
        const uint32_t at = data + 16 * (U ^ ((U >> 3) & 3));
        uint32_t v[16];
        load_row(at, v);
        __half2 mn2, mx2;
        uint32_t ob = outliers_and_range(v, lo2, hi2, mn2, mx2);
        const uint32_t range = range_of_token<P>(mn2, mx2);
        if (p == 0) sm.range[tok] = range;
        sm.out[tok * P + p] = ob;
    }
    __syncwarp();
    // ---- the outliers go to the warp's list, a token per lane, their places are marked
    uint32_t nout = 0, top = 0;
    if (main) {
        uint32_t ob[P], cnt = 0;
        if constexpr (P == 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(&sm.out[tid * P]);
            ob[0] = x.x; ob[1] = x.y; ob[2] = x.z; ob[3] = x.w;
        } else {
#pragma unroll
            for (int k = 0; k < P; ++k) ob[k] = sm.out[tid * P + k];
        }
#pragma unroll
        for (int k = 0; k < P; ++k) {
            if (!fresh) ob[k] = 0;
            cnt += (uint32_t)__popc(ob[k]);
        }
        uint32_t pos = prefix(cnt, lane, nout);
        const uint32_t r = sm.range[tid], fill = ((r & 0x7C00u) == 0x7C00u || (r >> 16 & 0x7C00u) == 0x7C00u) ? GONE : r & 0xFFFFu;
#pragma unroll
        for (int k = 0; k < P; ++k)
            while (ob[k]) {
                const uint32_t c = 32 * k + (uint32_t)__ffs(ob[k]) - 1u, U = tid * PR + (c >> 3);
                ob[k] &= ob[k] - 1;
                unsigned short* where = reinterpret_cast<unsigned short*>(sm.data + 16 * (U ^ ((U >> 3) & 3))) + (c & 7);
                const uint32_t x = *where;
                if (pos < cap) list[pos] = ((uint32_t)tid << 24) | (c << 16) | x;
                top = max(top, x & 0x7FFFu);
                *where = (unsigned short)fill;
                ++pos;
            }
    }

    // ---- widths; which tokens have which
    const uint32_t range = sm.range[tid & (QAQ_TILE - 1)];
    const float mn = __low2float(as_h2(range)), mx = __high2float(as_h2(range));
    {
        const float r = __fsub_rn(mx, mn);
        if (given) b = b < 1 ? 1 : (b > 8 ? 8 : b);
        else if (!IS_V) b = ladder(r, a.cK, a.bmin, a.bmax);
        else b = nv == 0 ? a.bmax : ladder(__fmul_rn(r, shat), a.cV, a.bmin, a.bmax);
        if (IS_V && __float_as_uint(shat) == QAQ_SCORE_LOST) atomicMax(a.status, (int)QAQ_ERR_CUDA);
        if (OPEN && !fresh) b = old ? min((int)(bs_old & 0xFFu), 8) : 0;
    }
    uint32_t alike = 0;
    if (main) {
        alike = qaqc::count_half(b, lane, sm.count[warp]);
        top = __reduce_max_sync(0xFFFFFFFFu, fresh ? max(top, qaqc::top_of(range)) : 0u);
        if (lane == 0) { sm.nout[warp] = nout; sm.top[warp] = top; }
    }
    if (OPEN) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // the CTA that is the last to have read the token count moves it on
    if (counted && tid == 0) {
        const unsigned n = gridDim.x * gridDim.y * gridDim.z;
        if (atomicInc(a.d_ticket, n - 1) == n - 1) *a.d_count = t_old + a.tok_hi;
    }
    // ---- order and sections, by both warps alike; space from the pools
    int slot;
    const qaqc::TileRows rows = qaqc::rows_of_counts<IS_V>(sm.count, b, alike, warp, lane, slot);
    const uint32_t total = qaqc::tile_total<D, IS_V>(rows);
    const uint32_t nout0 = sm.nout[0], nall = nout0 + sm.nout[1];
    uint32_t base = 0, taken = 0;
    if (!OPEN && tid < 2) base = pool_take(pool, lane ? nall : total, lane ? 3u : 15u, pool_now > (lane ? a.ocap : a.pool_bytes), taken);
    if (!OPEN || b) {
        const int row = IS_V ? slot >> 2 : slot, row_w = IS_V ? qaqc::width_of_row(rows, row) : b;
        const qaqc::RowPlace pl = qaqc::place_row<D, IS_V>(rows, row, row_w);
        const float step = qaqc::step_of(mn, mx, b), inv = step > 0.f ? __fdiv_rn(1.0f, step) : 0.f;
        const bool endless = ((range & 0x7C00u) == 0x7C00u || (range >> 16 & 0x7C00u) == 0x7C00u);
        uint4 q = make_uint4(__float_as_uint(mn), __float_as_uint(inv), pl.main | (pl.high << 16),
                             (uint32_t)tid | ((uint32_t)b << 8) | ((uint32_t)row_w << 16) | (pl.mm << 20) | (pl.mh << 24) | (endless ? 0x80000000u : 0u));
        if (OPEN && old) {             // where it is in the tile as it is stored, instead of the range
            const int oslot = (int)((bs_old >> 8) & (QAQ_TILE - 1));
            uint4 h = *reinterpret_cast<const uint4*>(stored_tile);
            if (!tw.y) h = make_uint4(0u, 0u, 0u, 0u);
            const qaqc::TileRows orows = qaqc::rows_of_header(h.x, h.y);
            const int orow = IS_V ? oslot >> 2 : oslot, ow = IS_V ? max(1, min(8, qaqc::width_of_row(orows, orow))) : b;
            const qaqc::RowPlace o = qaqc::place_row<D, IS_V>(orows, orow, ow);
            q.x = o.main | (o.high << 16);
            q.y = (uint32_t)ow | (o.mm << 4) | (o.mh << 8) | ((uint32_t)(oslot & 3) << 12);
            q.w = (q.w & 0x7FFFFFFFu) | STORED;
        }
        sm.slot[slot] = q;
    }
    // ---- a pool without room: the space is given back (or not taken), nothing about the tile is published; the device
    //      status reports the lost tokens
    if (warp == 0) {
        bool fail;
        if (OPEN) {
            // nobody else is at these pools: a tile that is begun goes to the end, one that is continued has to be the last
            // thing before it (an open tile that re-quantization could not keep there, in a full pool, cannot grow); what is
            // closed takes a rounded amount, and one that would have been closed leaves the end where the next tile can begin
            const uint32_t pool_end = __shfl_sync(0xFFFFFFFFu, pool_now, 0), opool_end = __shfl_sync(0xFFFFFFFFu, pool_now, 1);
            const uint32_t next = (pool_end + 15u) & ~15u;
            const uint32_t off = s_lo ? tw.x : next, end = s_hi == QAQ_TILE ? (off + total + 15u) & ~15u : off + total;
            fail = pool_end > a.pool_bytes || (size_t)end + 16 > a.pool_bytes || (s_lo && pool_end != tw.x + tw.y);
            const bool full = opool_end > a.ocap;
            base = lane == 0 ? off : (full ? 0xFFFF0000u : opool_end);
            if (lane == 0 && (!fail || s_hi == QAQ_TILE)) *pool = fail ? next : end;
            if (lane == 1 && !fail && !full) *pool = s_hi == QAQ_TILE ? (opool_end + nall + 3u) & ~3u : opool_end + nall;
        } else {
            const uint32_t off = __shfl_sync(0xFFFFFFFFu, base, 0);
            fail = (size_t)off + __shfl_sync(0xFFFFFFFFu, taken, 0) + 16 > a.pool_bytes || (size_t)off + total + 16 > a.pool_bytes;
            if (fail && lane < 2) pool_give_back(pool, base, taken);
        }
        if (lane < 2) sm.base[lane] = base;
        if (lane == 0) {
            sm.skip = fail;
            if (fail) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
        }
    }
    __syncthreads();
    if (sm.skip) return;
    const uint32_t off = sm.base[0], obase = sm.base[1];
    const uint32_t room = (size_t)obase + 8 < a.ocap ? a.ocap - 8 - obase : 0;         // 8 entries of read-ahead margin
    const uint32_t stored = min(nall, room);
    uint8_t* const dst = ts.codes + (size_t)bh * a.pool_bytes + off;
    uint32_t* const outl = ts.outl + (size_t)bh * a.ocap + obase;
    if (tid == 0) {
        if (stored < nall) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
        *tab = s_lo ? make_uint4(off, total, tw.z, tw.w + stored) : make_uint4(off, total, obase, stored);
        top = max(sm.top[0], sm.top[1]);
        if (OPEN && s_lo && tw.y) top = max(top, reinterpret_cast<const uint4*>(stored_tile)->w >> 16);
        *reinterpret_cast<uint4*>(dst) = qaqc::header_of<D, IS_V>(rows, top);
    }
    if (!OPEN || b) ts.bs[mt] = (unsigned short)(b | (slot << 8));
    if (fresh) ts.mnmx[mt] = range;
    const uint32_t first = warp ? nout0 : 0u;
    for (uint32_t i = lane; i < min(nout, cap); i += 32)          // (none beyond the first two warps)
        if (first + i < stored) outl[first + i] = list[i];
    if (nout > cap) {                  // more outliers than were listed: the rest is found once more in the input
        uint32_t seen = 0;
#pragma unroll 1
        for (int it = 0; it < IT; ++it) {
            const int tok = 32 * warp + it * TPI + g;
            const bool there = !OPEN || (tok >= s_lo && tok < s_hi);
            const __half* row = X + (ptrdiff_t)(there ? tok : s_lo) * a.st + 32 * p;
            uint32_t v[16];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 x = *reinterpret_cast<const uint4*>(row + 8 * i);
                v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
            }
            __half2 mn2, mx2;
            uint32_t ob = outliers_and_range(v, lo2, hi2, mn2, mx2);
            if (!there) ob = 0;
            uint32_t sum, pos = seen + prefix((uint32_t)__popc(ob), lane, sum);
            seen += sum;
            for (; ob; ob &= ob - 1, ++pos) {
                const uint32_t c = (uint32_t)__ffs(ob) - 1u;
                if (pos >= cap && first + pos < stored)
                    outl[first + pos] = ((uint32_t)tok << 24) | ((uint32_t)(32 * p + c) << 16) | __half_as_ushort(row[c]);
            }
        }
    }

    // ---- codes, tokens by slot
    Scale sc;
    sc.k64 = a.k64;
    const int nt = OPEN ? (int)(((sm.count[0][0] + sm.count[1][0]) * qaqc::ONES >> 24) + ((sm.count[0][1] + sm.count[1][1]) * qaqc::ONES >> 24)) : QAQ_TILE;
#pragma unroll 1
    for (int s0 = warp * TPI; s0 < nt; s0 += NW * TPI) {
        const int sl = s0 + g;
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (!OPEN || sl < nt) q = sm.slot[sl];
        const int U = (int)(q.w & 63u) * PR + 4 * p, B = (int)((q.w >> 8) & 15u);
        const int w = OPEN && IS_V ? ((sl & ~3) < nt ? (int)((sm.slot[sl & ~3].w >> 16) & 15u) : 0) : (int)((q.w >> 16) & 15u);
        uint32_t lo[4], hi[4];
        const bool wide = __any_sync(0xFFFFFFFFu, w > 4);
        if (!OPEN || __any_sync(0xFFFFFFFFu, sl < nt && !(q.w & STORED))) {
        uint32_t v[16], c[16];
        load_row(data + 16 * (U ^ ((U >> 3) & 3)), v);
        sc.mn = __uint_as_float(q.x);
        sc.inv = pair_of(__uint_as_float(q.y), __uint_as_float(q.y));
        sc.top = ((1u << B) - 1u) * 0x00010001u + 0x4B000000u;
#pragma unroll
        for (int k = 0; k < 16; ++k) c[k] = code_pair(v[k], sc);
        if (__any_sync(0xFFFFFFFFu, q.w >> 31)) {
            if (q.w >> 31) {           // a range that is not finite: marks become -inf, which the plain arithmetic takes to code 0
                uint32_t creg[8];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    if ((v[k] & 0xFFFFu) == GONE) v[k] = (v[k] & 0xFFFF0000u) | 0xFC00u;
                    if ((v[k] >> 16) == GONE) v[k] = (v[k] & 0xFFFFu) | 0xFC000000u;
                }
                const __half2 mm = as_h2(sm.range[q.w & 63u]);
                qaqc::codes32(v, __low2float(mm), __high2float(mm), B, creg);
#pragma unroll
                for (int j = 0; j < 8; ++j) { c[2 * j] = qaqc::prmt(creg[j], 0u, 0x4140u); c[2 * j + 1] = qaqc::prmt(creg[j], 0u, 0x4342u); }
            }
            __syncwarp();
        }
        if (wide) {
            uint32_t creg[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) creg[j] = qaqc::prmt(c[2 * j], c[2 * j + 1], 0x6420u);
            qaqc::nibbles_of(creg, 0, lo);
            qaqc::nibbles_of(creg, 4, hi);
        } else {                       // codes of up to 4 bits
#pragma unroll
            for (int u = 0; u < 4; ++u) lo[u] = qaqc::prmt(mad(c[4 * u + 2], a.k16, c[4 * u]), mad(c[4 * u + 3], a.k16, c[4 * u + 1]), 0x6420u);
        }
        }
        if (OPEN) {
            if ((q.w & STORED) || sl >= nt) {
#pragma unroll
                for (int u = 0; u < 4; ++u) lo[u] = hi[u] = 0;
                if (sl < nt) qaqc::take_token<D, IS_V>(stored_tile, qaqc::tile_bytes_max(D) + 16, q.x & 0xFFFFu, q.x >> 16, (int)(q.y & 15u), (q.y >> 4) & 15u,
                                                       (q.y >> 8) & 15u, (int)((q.y >> 12) & 3u), p, lo, hi);
            }
            __syncwarp();
            if (IS_V && (sl & ~3) < nt) q = sm.slot[sl & ~3];       // empty slots of the last group have its row
        }
        if (IS_V) qaqc::transpose4<P>(lo, g & 3);
        const int e = IS_V ? 4 * p + (g & 3) : p;
        const int wm = min(w, 4);
        if (!OPEN || w) qaqc::store_nibbles(dst + (q.z & 0xFFFFu) + (IS_V ? e * (int)((q.w >> 20) & 7u) : e) * 4 * wm, wm, lo);
        if (wide) {
            if (IS_V) qaqc::transpose4<P>(hi, g & 3);
            if (w > 4) qaqc::store_nibbles(dst + (q.z >> 16) + (IS_V ? e * (int)((q.w >> 24) & 7u) : e) * 4 * (w - 4), w - 4, hi);
        }
    }
}

// dynamic shared memory: the scratch, the tile as it is stored (OPEN), the warps' lists of outliers
template <int D, bool OPEN, int NW>
__global__ void __launch_bounds__(32 * NW, OPEN ? 16 / NW : 12) quant_tiles_kernel(const QuantArgs a, uint32_t cap) {
    extern __shared__ __align__(64) unsigned char tiles_smem[];
    TileScratch<D>& sm = *reinterpret_cast<TileScratch<D>*>(tiles_smem);
    uint8_t* stored_tile = tiles_smem + sizeof(TileScratch<D>);
    uint32_t* list = reinterpret_cast<uint32_t*>(stored_tile + (OPEN ? qaqc::tile_bytes_max(D) + 16 : 0));
    qaq_dependency();
    if (blockIdx.z == 0) quantize_tile<D, false, OPEN, NW>(a, sm, stored_tile, list, cap);
    else quantize_tile<D, true, OPEN, NW>(a, sm, stored_tile, list, cap);
}

// tiles.x tiles of every (b,h), all whole, or one that is not (or may not be)
template <int D, bool OPEN, int NW>
qaq_status launch_tiles(int tiles, int BH, const QuantArgs& a, double alpha, cudaStream_t s) {
    // the lists hold a tenth more than the share of outliers asked for gives a tile, and some (twelve CTAs per SM at 1 %)
    const uint32_t want = (uint32_t)(alpha * (QAQ_TILE * D) * 1.1) + 60, cap = (want < 2048 ? want : 2048) / 2;
    const size_t smem = sizeof(TileScratch<D>) + (OPEN ? qaqc::tile_bytes_max(D) + 16 : 0) + 2 * cap * sizeof(uint32_t);
    static_assert(sizeof(TileScratch<D>) + qaqc::tile_bytes_max(D) + 16 + 2048 * sizeof(uint32_t) <= 48 * 1024, "shared memory that needs no attribute");
    QAQ_CUDA_TRY(qaq_launch(quant_tiles_kernel<D, OPEN, NW>, dim3((unsigned)tiles, (unsigned)BH, 2), dim3(32 * NW), smem, s, a, cap));
    return QAQ_OK;
}
template <bool OPEN, int NW>
qaq_status launch(int D, int tiles, int BH, const QuantArgs& a, double alpha, cudaStream_t s) {
    switch (D) {
        case 32: return launch_tiles<32, OPEN, NW>(tiles, BH, a, alpha, s);
        case 64: return launch_tiles<64, OPEN, NW>(tiles, BH, a, alpha, s);
        case 128: return launch_tiles<128, OPEN, NW>(tiles, BH, a, alpha, s);
    }
    return QAQ_ERR_UNSUPPORTED_SHAPE;
}
// eight warps while all CTAs run at once, else four (figures at the top)
qaq_status launch_open(int D, int BH, const QuantArgs& a, double alpha, cudaStream_t s) {
    return 2 * BH <= 2 * 148 ? launch<true, 8>(D, 1, BH, a, alpha, s) : launch<true, 4>(D, 1, BH, a, alpha, s);
}

// Widths alone: one CTA = 64 tokens of one (b,h); P = D/32 lanes own a token, each lane 32 consecutive channels (64 bytes) of
// K and of V.
template <int D>
__global__ void __launch_bounds__(2 * D) select_kernel(const QuantArgs a) {
    constexpr int P = D / 32;
    qaq_dependency();
    const int bh = blockIdx.y, tn = blockIdx.x * QAQ_TILE + threadIdx.x / P, p = threadIdx.x % P;
    const bool valid = tn < a.n_new;
    const float* thr = a.thr + (size_t)bh * 4;
    uint32_t v[2][16];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const __half* row = (x ? a.V : a.K) + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh + (size_t)(valid ? tn : 0) * a.st + 32 * p;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint4 y = *reinterpret_cast<const uint4*>(row + 8 * i);
            v[x][4 * i] = y.x; v[x][4 * i + 1] = y.y; v[x][4 * i + 2] = y.z; v[x][4 * i + 3] = y.w;
        }
    }
    // the P lanes of a token take rows p, p+P, ... of its window
    float shat = __int_as_float(0xff800000);
    int nv = 0;
    if (valid) {
        nv = min((int)a.nvalid[(size_t)bh * a.n_new + tn], a.W);
        const float* r = a.ring + (size_t)bh * a.W * a.n_new + tn;
        for (int i = p; i < nv; i += P) shat = fmaxf(shat, r[(size_t)i * a.n_new]);
    }
#pragma unroll
    for (int o = 1; o < P; o <<= 1) shat = fmaxf(shat, __shfl_xor_sync(0xFFFFFFFFu, shat, o));
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const __half2 lo2 = __half2half2(__float2half_ru(thr[2 * x])), hi2 = __half2half2(__float2half_rd(thr[2 * x + 1]));
        __half2 mn2, mx2;
        outliers_and_range(v[x], lo2, hi2, mn2, mx2);
        const uint32_t range = range_of_token<P>(mn2, mx2);
        const float r = __fsub_rn(__high2float(as_h2(range)), __low2float(as_h2(range)));
        if (valid && p == 0) {
            const int b = x == 0 ? ladder(r, a.cK, a.bmin, a.bmax) : (nv == 0 ? a.bmax : ladder(__fmul_rn(r, shat), a.cV, a.bmin, a.bmax));
            (x ? a.out_bitsV : a.out_bitsK)[(size_t)bh * a.n_new + tn] = (uint8_t)b;
        }
    }
}

qaq_status check_dense(const void* K, const void* V, long sb, long sh, long st, int D) {
    if (!K || !V) return QAQ_ERR_INVALID_ARG;
    if (((uintptr_t)K & 15) || ((uintptr_t)V & 15)) return QAQ_ERR_INVALID_ARG;  // 16-byte vector loads
    if (st < D || (sb & 7) || (sh & 7) || (st & 7) || sb < 0 || sh < 0) return QAQ_ERR_INVALID_ARG;
    return QAQ_OK;
}

}  // namespace

qaq_status qaq_launch_select(const qaq_config* cfg, const qaq_policy* pol, const void* K, const void* V, long sb,
                             long sh, long st, int n, const float* ring, const uint8_t* nvalid, const float* thr,
                             uint8_t* bitsK, uint8_t* bitsV, cudaStream_t s) {
    QuantArgs a{};
    a.K = (const __half*)K; a.V = (const __half*)V; a.sb = sb; a.sh = sh; a.st = st;
    a.H = cfg->heads; a.n_new = n; a.t_old = 0; a.tok_lo = 0; a.tok_hi = n; a.first_tile = 0;
    a.ring = ring; a.nvalid = nvalid; a.W = cfg->window; a.thr = thr;
    a.cK = pol->cK; a.cV = pol->cV; a.bmin = cfg->bits_min; a.bmax = cfg->bits_max;
    a.out_bitsK = bitsK; a.out_bitsV = bitsV;
    const dim3 grid((n + QAQ_TILE - 1) / QAQ_TILE, cfg->batch * cfg->heads);
    switch (cfg->head_dim) {
        case 32: QAQ_CUDA_TRY(qaq_launch(select_kernel<32>, grid, dim3(64), 0, s, a)); break;
        case 64: QAQ_CUDA_TRY(qaq_launch(select_kernel<64>, grid, dim3(128), 0, s, a)); break;
        case 128: QAQ_CUDA_TRY(qaq_launch(select_kernel<128>, grid, dim3(256), 0, s, a)); break;
        default: return QAQ_ERR_UNSUPPORTED_SHAPE;
    }
    return QAQ_OK;
}

qaq_status qaq_launch_append(qaq_cache* c, const void* K, const void* V, long sb, long sh, long st, int n_new,
                             const uint8_t* bitsK, const uint8_t* bitsV, const qaq_policy* pol, const float* ring,
                             const uint8_t* nvalid, const float* thr, cudaStream_t s) {
    QuantArgs a{};
    a.K = (const __half*)K; a.V = (const __half*)V; a.sb = sb; a.sh = sh; a.st = st;
    a.H = c->cfg.heads; a.n_new = n_new; a.t_old = (int)c->tokens;
    a.bitsK = bitsK; a.bitsV = bitsV; a.ring = ring; a.nvalid = nvalid; a.W = c->cfg.window; a.thr = thr;
    a.cK = pol ? pol->cK : 0.f; a.cV = pol ? pol->cV : 0.f; a.bmin = c->cfg.bits_min; a.bmax = c->cfg.bits_max;
    a.k = c->t[0]; a.v = c->t[1]; a.pool_bytes = c->pool_bytes; a.ocap = c->ocap;
    a.tmax_pad = c->tmax_pad; a.ntiles = c->ntiles; a.status = c->d_status;
    const int D = c->cfg.head_dim, BH = c->BH;
    // Tiles are placed by atomic bump allocation, so a tile that stays open (partly filled)
    // must be the last thing allocated in its pool: the head of the range (completing an
    // open tile), the whole tiles, and a trailing partial tile go in separate launches.
    const int t0 = (int)c->tokens, t1 = t0 + n_new;
    int cur = t0;
    qaq_status stt;
    if (cur % QAQ_TILE != 0) {  // head: finish (or extend) the open tile
        const int end = min(t1, (cur / QAQ_TILE + 1) * QAQ_TILE);
        a.tok_lo = cur - t0; a.tok_hi = end - t0; a.first_tile = cur / QAQ_TILE;
        if ((stt = launch_open(D, BH, a, c->cfg.outlier_frac, s)) != QAQ_OK) return stt;
        cur = end;
    }
    const int full_end = t1 / QAQ_TILE * QAQ_TILE;
    if (cur < full_end) {       // body: whole tiles
        a.tok_lo = cur - t0; a.tok_hi = full_end - t0; a.first_tile = cur / QAQ_TILE;
        if ((stt = launch<false, 2>(D, (full_end - cur) / QAQ_TILE, BH, a, c->cfg.outlier_frac, s)) != QAQ_OK) return stt;
        cur = full_end;
    }
    if (cur < t1) {             // tail: a new, partly filled tile
        a.tok_lo = cur - t0; a.tok_hi = t1 - t0; a.first_tile = cur / QAQ_TILE;
        if ((stt = launch_open(D, BH, a, c->cfg.outlier_frac, s)) != QAQ_OK) return stt;
    }
    c->tokens = t1;
    return QAQ_OK;
}

extern "C" qaq_status qaq_select_bits(const qaq_config* cfg, const qaq_policy* policy, const void* K, const void* V,
                                      long stride_b, long stride_h, long stride_t, int n_tokens,
                                      const float* score_ring, const uint8_t* nvalid, const float* thr,
                                      uint8_t* bitsK, uint8_t* bitsV, void* stream) {
    if (!cfg || !policy || !score_ring || !nvalid || !thr || !bitsK || !bitsV || n_tokens < 0) return QAQ_ERR_INVALID_ARG;
    if (!qaq_dim_ok(cfg->head_dim)) return QAQ_ERR_UNSUPPORTED_SHAPE;
    if (cfg->bits_min < 1 || cfg->bits_max > 8 || cfg->bits_min > cfg->bits_max || cfg->window < 1) return QAQ_ERR_UNSUPPORTED_SHAPE;
    qaq_status st = check_dense(K, V, stride_b, stride_h, stride_t, cfg->head_dim);
    if (st != QAQ_OK) return st;
    if (n_tokens == 0) return QAQ_OK;
    return qaq_launch_select(cfg, policy, K, V, stride_b, stride_h, stride_t, n_tokens, score_ring, nvalid, thr, bitsK,
                             bitsV, (cudaStream_t)stream);
}

extern "C" qaq_status qaq_quantize_append(qaq_cache* c, const void* K_new, const void* V_new, long stride_b,
                                          long stride_h, long stride_t, int n_new, const uint8_t* bitsK,
                                          const uint8_t* bitsV, const qaq_policy* policy, const float* score_ring,
                                          const uint8_t* nvalid, const float* thr, void* stream) {
    if (!c || !thr || n_new < 0) return QAQ_ERR_INVALID_ARG;
    if ((bitsK == nullptr) != (bitsV == nullptr)) return QAQ_ERR_INVALID_ARG;
    if (!bitsK && (!policy || !score_ring || !nvalid)) return QAQ_ERR_INVALID_ARG;
    qaq_status st = check_dense(K_new, V_new, stride_b, stride_h, stride_t, c->cfg.head_dim);
    if (st != QAQ_OK) return st;
    if (c->tokens + n_new > c->cfg.max_tokens) return QAQ_ERR_CAPACITY;
    if (n_new == 0) return QAQ_OK;
    return qaq_launch_append(c, K_new, V_new, stride_b, stride_h, stride_t, n_new, bitsK, bitsV, policy, score_ring,
                             nvalid, thr, (cudaStream_t)stream);
}

// One new token per (b,h) with the token count taken from (and advanced in) device memory: the open tile (or a new one)
// of every (b,h) is rebuilt by one CTA, as in the head / tail launch of qaq_launch_append.  Nothing on the host changes,
// so the call can be captured in a CUDA graph and replayed.
extern "C" qaq_status qaq_stream_append(qaq_cache* c, const void* k_new, const void* v_new, long stride_b, long stride_h,
                                        const uint8_t* bitK, const uint8_t* bitV, const qaq_policy* policy,
                                        const float* score_col, const uint8_t* nvalid, const float* thr, void* stream) {
    if (!c || !thr) return QAQ_ERR_INVALID_ARG;
    if ((bitK == nullptr) != (bitV == nullptr)) return QAQ_ERR_INVALID_ARG;
    if (!bitK && (!policy || !score_col || !nvalid)) return QAQ_ERR_INVALID_ARG;
    const int D = c->cfg.head_dim;
    qaq_status st = check_dense(k_new, v_new, stride_b, stride_h, D, D);
    if (st != QAQ_OK) return st;
    QuantArgs a{};
    a.K = (const __half*)k_new; a.V = (const __half*)v_new; a.sb = stride_b; a.sh = stride_h; a.st = D;
    a.H = c->cfg.heads; a.n_new = 1; a.tok_lo = 0; a.tok_hi = 1;
    a.bitsK = bitK; a.bitsV = bitV; a.ring = score_col; a.nvalid = nvalid; a.W = c->cfg.window; a.thr = thr;
    a.cK = policy ? policy->cK : 0.f; a.cV = policy ? policy->cV : 0.f; a.bmin = c->cfg.bits_min; a.bmax = c->cfg.bits_max;
    a.k = c->t[0]; a.v = c->t[1]; a.pool_bytes = c->pool_bytes; a.ocap = c->ocap;
    a.tmax_pad = c->tmax_pad; a.ntiles = c->ntiles; a.status = c->d_status;
    a.d_count = qaq_d_count(c); a.d_ticket = qaq_d_ticket(c); a.max_tokens = (int)c->cfg.max_tokens;
    return launch_open(D, c->BH, a, c->cfg.outlier_frac, (cudaStream_t)stream);
}
