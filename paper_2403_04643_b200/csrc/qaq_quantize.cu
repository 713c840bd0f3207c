// S1-S3: bit-width selection, outlier split, uniform quantization and bit-packing.
//
// Two kernels: whole tiles, which is all of a prompt but its last tokens, by two warps per tile and tensor
// (quant_tiles_kernel, further down); partly filled tiles, tiles that are continued, the launches that take the token count
// from device memory, and the selection of widths alone by a CTA per tile (quant_kernel):
//
// One CTA handles one tile (QAQ_TILE consecutive tokens) of one (b,h); head_dim/32 lanes
// own one token, each lane 32 consecutive channels of K and of V (64 bytes each), held in
// registers from the min/max pass to the packing pass, so K and V are read from HBM once.
//   phase 0  attention-window maximum of the score rows (Section 4.2)
//   phase 1  outlier masks and min/max of the non-outliers in binary16 pair arithmetic
//            (exact: the inputs are binary16), width from the exponents (Section 4.1)
//   phase 2  warp 0: the tokens sorted by width (ballots), sections and size of the tile,
//            exclusive scan of the outlier counts, space taken from the (b,h) pools by atomicAdd
//   phase 3  codes (binary32: one sub, one mul, round down), packed words written into a shared-memory
//            image of the tile in the section layout of qaq_codec.cuh (values token by token, which
//            the copy-out transposes into rows of four tokens), vector stores; outlier
//            entries placed by popc ranks
// A tile that is continued (an append behind a partly filled tile) is built anew: the codes of
// its old tokens are read back from the pool, the image of old and new tokens replaces it.
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
    unsigned* d_ticket;    //   advanced by the last CTA of the launch to finish (small appends only)
    int max_tokens;
    uint8_t* out_bitsK;    // selection only
    uint8_t* out_bitsV;
    uint32_t k64 = 65536, k16 = 16;      // multipliers that the compiler is not to know (see code_pair)
};

using qaqc::ladder;

__device__ __forceinline__ uint32_t lop3_sel(uint32_t a, uint32_t m, uint32_t c) {  // (a & m) | (c & ~m)
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xE2;" : "=r"(d) : "r"(a), "r"(m), "r"(c));
    return d;
}
__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t b, uint32_t c) {  // (a & b) | c
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ __half2 as_h2(uint32_t x) { return *reinterpret_cast<__half2*>(&x); }
__device__ __forceinline__ uint32_t as_u32(__half2 x) { return *reinterpret_cast<uint32_t*>(&x); }
// One lane's 32 channels of one token and tensor: outlier masks, masked min / max.
//   v[k] holds channels 2k, 2k+1 (binary16 pairs).  On return every outlier entry of v has
//   been replaced by -inf: in the code computation that yields code byte 0 without a mask
//   (the outlier's own value is re-read from memory when its list entry is written).
//   inl : bit k = channel 2k is an inlier, bit 16+k = channel 2k+1 is an inlier
__device__ __forceinline__ void analyze32(uint32_t (&v)[16], __half2 lo2, __half2 hi2, uint32_t& inl, __half2& mn2,
                                          __half2& mx2) {
    uint32_t mnacc = 0x7C007C00u, mxacc = 0xFC00FC00u, bits = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const __half2 x = as_h2(v[k]);
        const uint32_t m = __hge2_mask(x, lo2) & __hle2_mask(x, hi2);
        mnacc = as_u32(__hmin2(as_h2(mnacc), as_h2(lop3_sel(v[k], m, 0x7C007C00u))));
        v[k] = lop3_sel(v[k], m, 0xFC00FC00u);
        mxacc = as_u32(__hmax2(as_h2(mxacc), as_h2(v[k])));
        bits = lop3_and_or(m, 0x00010001u << k, bits);
    }
    inl = bits;
    mn2 = as_h2(mnacc);
    mx2 = as_h2(mxacc);
}

// space from a (b,h) pool: `whole` tiles take a rounded-up amount in one atomic; a tile that is
// being continued takes the exact amount and is padded to the unit when it closes.  `taken` is
// what the pool end moved by (to be given back if the space turns out not to fit: pool_give_back).
// full: the pool end already lay beyond the pool when the CTA began; nothing is taken, so that the end cannot run away.
__device__ __forceinline__ uint32_t pool_take(uint32_t* pool, uint32_t amount, uint32_t unit_mask, bool whole, bool closes, bool full,
                                              uint32_t& taken) {
    uint32_t base;
    if (full) {
        taken = 0;
        base = 0xFFFF0000u;
    } else if (whole) {
        taken = (amount + unit_mask) & ~unit_mask;
        base = atomicAdd(pool, taken);
    } else {
        base = atomicAdd(pool, amount);
        taken = amount;
        if (closes) {
            const uint32_t pad = (0u - (base + amount)) & unit_mask;
            if (pad) atomicAdd(pool, pad);
            taken += pad;
        }
    }
    return base;
}

// One CTA = one tile of 64 tokens of one (b,h); P = D/32 lanes own a token, each lane 32
// consecutive channels (64 bytes) of K and of V, kept in registers across all phases.
// Order of work (barriers in brackets): loads, attention window, outlier masks and ranges,
// widths [A] warp 0 sorts the tile's tokens by width and sizes its sections, warp 1 scans the outlier counts and takes pool
// space with four atomics in flight at once while every warp computes its codes [B] words into a
// shared-memory image of the tile [C] the image goes out with 16-byte stores; outlier entries and
// per-token metadata follow.  Slots below the first new token of a continued tile hold the tile's
// old tokens: their widths come from the metadata, their codes from the tile as it is stored.
template <int D, bool SELECT_ONLY>
__global__ void __launch_bounds__(2 * D, D == 128 ? 3 : 4) quant_kernel(const QuantArgs a) {
    constexpr int P = D / 32;            // lanes per token
    constexpr int NT = 2 * D;            // threads
    constexpr int IMG = qaqc::tile_bytes_max(D);
    constexpr bool COUNTED = !SELECT_ONLY;   // the launches that may take the token count from device memory
    const int bh = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int slot = tid / P, p = tid % P;
    qaq_dependency();
    int t_old = a.t_old, first_tile = a.first_tile;
    if (COUNTED && a.d_count) {
        t_old = *a.d_count;                // the same value in every thread of the launch: it is written only by tick()
        first_tile = t_old / QAQ_TILE;
        if (t_old + a.tok_hi > a.max_tokens) {             // no room: nothing is stored, the count stays
            if (tid == 0) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
            return;
        }
    }
    const int tile = first_tile + blockIdx.x;
    // counted launches: the last CTA to get here moves the count on.  Every thread of every CTA has used the count it
    // read by then (the barrier), and nothing else of the launch reads it afterwards.
    auto tick = [&]() {
        if (COUNTED && a.d_count) {
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                const unsigned n = gridDim.x * gridDim.y;
                if (atomicInc(a.d_ticket, n - 1) == n - 1) *a.d_count = t_old + a.tok_hi;
            }
        }
    };

    const int abs_lo = max(tile * QAQ_TILE, t_old + a.tok_lo);
    const int abs_hi = min((tile + 1) * QAQ_TILE, t_old + a.tok_hi);
    const int s_lo = abs_lo - tile * QAQ_TILE, s_hi = abs_hi - tile * QAQ_TILE;
    const bool valid = slot >= s_lo && slot < s_hi;       // a new token
    const bool old = !SELECT_ONLY && slot < s_lo;         // a token the tile already holds
    const int tn = tile * QAQ_TILE + slot - t_old;        // index among the new tokens

    __shared__ uint8_t s_bits[2][QAQ_TILE];   // widths of the tile's slots (0: empty)
    __shared__ uint32_t s_cnt[2][QAQ_TILE];   // outlier counts of the new tokens, then exclusive offsets
    __shared__ qaqc::Section s_tab[2][9], s_otab[2][9];   // sections of the tile by width, and of the tile as it was (continued tiles)
    __shared__ unsigned short s_place[2][QAQ_TILE];       // slot of every token in the sorted order | width of its row << 8
    __shared__ uint8_t s_sorted[2][QAQ_TILE], s_orow[2][QAQ_TILE / 4];   // width of every slot; width of the stored rows of values
    __shared__ uint32_t s_tot[2], s_base[2], s_obase[2], s_olimit[2], s_otot[2];
    constexpr uint32_t OUT_STAGE = 4 * D;      // outliers of a tile whose (slot, channel) are listed on chip in entry order; more go out one by one
    __shared__ unsigned short s_work[SELECT_ONLY ? 1 : 2][SELECT_ONLY ? 1 : OUT_STAGE];
    __shared__ int s_skip;
    __shared__ __align__(16) uint8_t s_img[SELECT_ONLY ? 1 : 2][SELECT_ONLY ? 16 : IMG];  // the tile as it will be stored

    const float* thr = a.thr + (size_t)bh * 4;
    const bool given = a.bitsK != nullptr;
    const size_t ti = (size_t)bh * a.ntiles + tile;
    const size_t mt = (size_t)bh * a.tmax_pad + (size_t)tile * QAQ_TILE + slot;

    // ---- loads first (independent of everything else)
    const int b_idx = bh / a.H, h_idx = bh % a.H;
    uint32_t vk[16], vv[16];
    {
        const __half* Kr = a.K + (size_t)b_idx * a.sb + (size_t)h_idx * a.sh + (size_t)(valid ? tn : 0) * a.st + 32 * p;
        const __half* Vr = a.V + (size_t)b_idx * a.sb + (size_t)h_idx * a.sh + (size_t)(valid ? tn : 0) * a.st + 32 * p;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint4 x = make_uint4(0, 0, 0, 0), y = make_uint4(0, 0, 0, 0);
            if (valid) {
                x = *reinterpret_cast<const uint4*>(Kr + 8 * i);
                y = *reinterpret_cast<const uint4*>(Vr + 8 * i);
            }
            vk[4 * i] = x.x; vk[4 * i + 1] = x.y; vk[4 * i + 2] = x.z; vk[4 * i + 3] = x.w;
            vv[4 * i] = y.x; vv[4 * i + 1] = y.y; vv[4 * i + 2] = y.z; vv[4 * i + 3] = y.w;
        }
    }
    uint32_t pool_now = 0;          // in the lanes that take space further down
    if (!SELECT_ONLY && warp < 2 && lane < 4 && (lane & 1) == warp)
        pool_now = (warp ? ((lane >> 1) ? a.v : a.k).opool_end : ((lane >> 1) ? a.v : a.k).pool_end)[bh];
    // a continued tile: its sections as they are stored (warp x for tensor x; used behind the first barrier)
    if (!SELECT_ONLY && s_lo > 0) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            if (warp != x) continue;
            const TensorStore& ts = x ? a.v : a.k;
            uint2 h = make_uint2(0u, 0u);
            if (ts.tile[ti].y) h = *reinterpret_cast<const uint2*>(ts.codes + (size_t)bh * a.pool_bytes + ts.tile[ti].x);
            int n[9];
            qaqc::counts_of(h.x, h.y, n);
            if (lane == 0) {
                if (x) qaqc::make_sections<qaqc::UNITS<D, true>>(n, s_otab[x], nullptr);
                else qaqc::make_sections<qaqc::UNITS<D, false>>(n, s_otab[x], nullptr);
            }
            if (x && lane < QAQ_TILE / 4) {
                int w = 0, end = 0;
#pragma unroll
                for (int k = 8; k >= 1; --k) {
                    if (lane >= end && lane < end + n[k]) w = k;
                    end += n[k];
                }
                s_orow[x][lane] = (uint8_t)w;
            }
        }
    }
    // empty slots of the value groups have to read as zero
    if (!SELECT_ONLY) {
        uint4* z = reinterpret_cast<uint4*>(s_img[1]);
        for (int o = tid; o < IMG / 16; o += NT) z[o] = make_uint4(0, 0, 0, 0);
    }

    // ---- attention window: the P lanes of a token take its rows p, p+P, ... and combine by shuffles
    float shat = __int_as_float(0xff800000);
    int nv_tok = 0;
    {
        if (!given && valid) {
            nv_tok = a.nvalid[(size_t)bh * a.n_new + tn];
            nv_tok = nv_tok < a.W ? nv_tok : a.W;
            // every row of the window is read (the ring is allocated in full), rows the token has no score in are
            // left out of the maximum: the loads then depend on nothing and go out together
            const float* r = a.ring + (size_t)bh * a.W * a.n_new + tn;
            int i = p;
            for (; i + 7 * P < a.W; i += 8 * P) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = r[(size_t)(i + u * P) * a.n_new];
#pragma unroll
                for (int u = 0; u < 8; ++u) if (i + u * P < nv_tok) shat = fmaxf(shat, v[u]);
            }
            for (; i < a.W; i += P) {
                const float v = r[(size_t)i * a.n_new];
                if (i < nv_tok) shat = fmaxf(shat, v);
            }
        }
#pragma unroll
        for (int o = 1; o < P; o <<= 1) shat = fmaxf(shat, __shfl_xor_sync(0xFFFFFFFFu, shat, o));
    }

    // ---- outlier masks and range of the rest (register work, needs nothing from shared memory)
    uint32_t inl[2], cntx[2];
    float mnf[2], mxf[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        // thresholds as binary16 bounds that decide exactly like the binary32 ones on binary16 data
        const __half lo = __float2half_ru(thr[2 * x]), hi = __float2half_rd(thr[2 * x + 1]);
        __half2 mn2, mx2;
        analyze32(x ? vv : vk, __half2half2(lo), __half2half2(hi), inl[x], mn2, mx2);
        const __half lmin = __hmin(__low2half(mn2), __high2half(mn2));
        const __half lmax = __hmax(__low2half(mx2), __high2half(mx2));
        __half2 pk = __halves2half2(lmin, __hneg(lmax));
#pragma unroll
        for (int o = 1; o < P; o <<= 1) pk = __hmin2(pk, as_h2(__shfl_xor_sync(0xFFFFFFFFu, as_u32(pk), o)));
        float mn = __low2float(pk), mx = -__high2float(pk);
        if (mn > mx) { mn = 0.f; mx = 0.f; }   // no entry inside [lo, hi]
        uint32_t cnt = 32u - (uint32_t)__popc(inl[x]);
#pragma unroll
        for (int o = 1; o < P; o <<= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
        mnf[x] = mn; mxf[x] = mx; cntx[x] = cnt;
    }

    // ---- widths
    int Bx[2], oslot[2] = {0, 0};      // oslot: where an old token lies in the tile as it is stored
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        int B;
        if (given) {
            B = valid ? (x ? a.bitsV : a.bitsK)[(size_t)bh * a.n_new + tn] : 0;
            B = B < 1 ? 1 : (B > 8 ? 8 : B);
        } else {
            const float r = __fsub_rn(mxf[x], mnf[x]);
            if (x == 0) {
                B = ladder(r, a.cK, a.bmin, a.bmax);
            } else {
                B = (nv_tok == 0) ? a.bmax : ladder(__fmul_rn(r, shat), a.cV, a.bmin, a.bmax);
            }
        }
        Bx[x] = valid ? B : 0;
        if (old) {
            const uint32_t bs = (x ? a.v : a.k).bs[mt];
            Bx[x] = min((int)(bs & 0xFFu), 8);
            oslot[x] = (int)(bs >> 8);
        }
        if (p == 0) {                                   // every slot of the tile is written: empty ones count nothing
            s_bits[x][slot] = (uint8_t)Bx[x];
            s_cnt[x][slot] = valid ? cntx[x] : 0u;
            if (SELECT_ONLY && valid) (x ? a.out_bitsV : a.out_bitsK)[(size_t)bh * a.n_new + tn] = (uint8_t)B;
        }
    }
    if (SELECT_ONLY) return;
    __syncthreads();   // [A] widths and outlier counts visible

    // ---- warp 0: tokens sorted by width, sections and header of the tile, space for the bytes; warp 1: scan of the
    //      outlier counts, space for the entries (the two halves do not depend on each other; the atomics - lane 2x of
    //      warp 0 and lane 2x + 1 of warp 1 for tensor x - stay in flight while every warp computes its codes)
    const bool starts = (s_lo == 0), closes = (s_hi == QAQ_TILE), whole = starts && closes;
    uint32_t my_base = 0, my_amount = 0, my_taken = 0;
    if (warp == 0) {
        uint32_t amount[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int b0 = s_bits[x][lane], b1 = s_bits[x][lane + 32];
            int n[9];
            const qaqc::Sorted so = x ? qaqc::sort_tile<true>(lane, b0, b1, n, s_sorted[x]) : qaqc::sort_tile<false>(lane, b0, b1, n, s_sorted[x]);
            s_place[x][lane] = (unsigned short)(so.slot[0] | (so.row_w[0] << 8));
            s_place[x][lane + 32] = (unsigned short)(so.slot[1] | (so.row_w[1] << 8));
            uint32_t total = 0;
            if (lane == 0) {
                uint32_t* head = reinterpret_cast<uint32_t*>(s_img[x]);
                total = x ? qaqc::make_sections<qaqc::UNITS<D, true>>(n, s_tab[x], head) : qaqc::make_sections<qaqc::UNITS<D, false>>(n, s_tab[x], head);
                s_tot[x] = total;
            }
            total = __shfl_sync(0xFFFFFFFFu, total, 0);
            // a continued tile stays where it is and takes only what it grows by behind its end
            const uint32_t old_nb = starts ? 0u : (x ? a.v : a.k).tile[ti].y;
            amount[x] = total - old_nb;
        }
        if (!(lane & 1) && lane < 4) {
            const int x = lane >> 1;
            my_amount = x ? amount[1] : amount[0];
            my_base = pool_take(&(x ? a.v : a.k).pool_end[bh], my_amount, 15u, whole, closes, pool_now > a.pool_bytes, my_taken);
        }
    } else if (warp == 1) {
        uint32_t amount[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const uint32_t c0 = s_cnt[x][lane], c1 = s_cnt[x][lane + 32];
            uint32_t ic0 = c0, ic1 = c1;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t u0 = __shfl_up_sync(0xFFFFFFFFu, ic0, d), u1 = __shfl_up_sync(0xFFFFFFFFu, ic1, d);
                if (lane >= d) { ic0 += u0; ic1 += u1; }
            }
            const uint32_t ctot0 = __shfl_sync(0xFFFFFFFFu, ic0, 31), ctot1 = __shfl_sync(0xFFFFFFFFu, ic1, 31);
            s_cnt[x][lane] = ic0 - c0; s_cnt[x][lane + 32] = ctot0 + ic1 - c1;
            amount[x] = ctot0 + ctot1;
            if (lane == 0) s_otot[x] = ctot0 + ctot1;
        }
        if ((lane & 1) && lane < 4) {
            const int x = lane >> 1;
            my_amount = x ? amount[1] : amount[0];
            my_base = pool_take(&(x ? a.v : a.k).opool_end[bh], my_amount, 3u, whole, closes, pool_now > a.ocap, my_taken);
        }
    }

    // ---- codes of the new tokens (every warp; needs only registers): channels 4j..4j+3 in the byte lanes of creg[j]
    uint32_t cregs[2][8];
#pragma unroll
    for (int x = 0; x < 2; ++x) qaqc::codes32(x ? vv : vk, mnf[x], mxf[x], Bx[x], cregs[x]);
    // old tokens of a continued tile: their codes from the tile as it is stored (read before anything is written)
    if (!starts) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            if (!old) continue;
            const TensorStore& ts = x ? a.v : a.k;
            const uint8_t* src = ts.codes + (size_t)bh * a.pool_bytes + ts.tile[ti].x;
            const int w = x ? (int)s_orow[x][(oslot[x] >> 2) & (QAQ_TILE / 4 - 1)] : Bx[x];
            if (!Bx[x]) continue;                       // never stored (the pool was full)
            if (x == 0) qaqc::read_token<D, false>(src, s_otab[x][w], oslot[x], w, p, cregs[x]);
            else        qaqc::read_token<D, true>(src, s_otab[x][w], oslot[x], w, p, cregs[x]);
        }
    }
    __syncthreads();   // [B] sections visible

    // ---- packed words into the shared-memory image of the tile (the values token by token: the copy to global memory
    //      turns them into rows of four tokens)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const uint32_t pl = s_place[x][slot & (QAQ_TILE - 1)];
        const int w = (int)(pl >> 8);
        if ((valid || old) && w) qaqc::write_token<D>(s_img[x], s_tab[x][w], x == 1, (int)(pl & 0xFFu), w, p, cregs[x]);
    }
    // ---- where the outliers of the new tokens are: (slot, channel) in (token, channel) order - entries of lanes
    //      p' < p of a token come first - listed in shared memory; their place needs only the scan of the counts.
    //      The values are fetched and the entries written afterwards by all threads, one entry each.
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        uint32_t ob = valid ? ~inl[x] : 0u;
        const uint32_t mine = (uint32_t)__popc(ob);
        uint32_t before = 0;
#pragma unroll
        for (int d = 1; d < P; ++d) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, mine, d);
            if (p >= d) before += o;
        }
        if (ob) {
            const uint32_t all = ob;
            const uint32_t lp0 = s_cnt[x][slot & (QAQ_TILE - 1)] + before;
            while (ob) {
                const int bit = __ffs(ob) - 1;
                ob &= ob - 1;
                const int k = bit & 15, hi = bit >> 4;
                const int c = 2 * k + hi;                                   // channel inside the lane's 32
                // entries of lower channels: pairs k' < k, plus channel 2k when this is 2k+1
                const uint32_t lower = (((1u << k) - 1u) * 0x00010001u) | (hi ? (1u << k) : 0u);
                const uint32_t lp = lp0 + (uint32_t)__popc(all & lower);
                if (lp < OUT_STAGE) s_work[x][lp] = (unsigned short)(((slot & (QAQ_TILE - 1)) << 8) | (32 * p + c));
            }
        }
    }
    // ---- allocation results (the atomics were issued before the codes were computed).  A pool without room:
    //      the space is given back, nothing about the tile is published and the CTA stops; the device status
    //      reports the lost tokens.
    if (warp == 0) {          // the byte pools
        bool fail = false;
        const bool mine = !(lane & 1) && lane < 4;
        const int x = lane >> 1;
        const TensorStore& ts = x ? a.v : a.k;
        if (mine) {
            const uint32_t off = starts ? my_base : ts.tile[ti].x;
            fail = (size_t)my_base + my_taken + 16 > a.pool_bytes || (size_t)off + s_tot[x] + 16 > a.pool_bytes;
            // a continued tile grows into what lies behind it: that has to be the space just taken (an open tile that
            // re-quantization could not keep the last thing in a full pool cannot grow)
            if (!starts && my_base != off + ts.tile[ti].y) fail = true;
            s_base[x] = off;
        }
        const bool any_fail = __any_sync(0xFFFFFFFFu, fail);
        if (mine) {
            if (any_fail) {
                pool_give_back(&ts.pool_end[bh], my_base, my_taken);
            } else {
                if (starts) ts.tile[ti].x = my_base;
                ts.tile[ti].y = s_tot[x];
            }
        }
        if (lane == 0) {
            s_skip = any_fail ? 1 : 0;
            if (any_fail) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
        }
    } else if (warp == 1) {   // the outlier lists: what fits is known now, the table is written once the byte pools have answered
        if ((lane & 1) && lane < 4) {
            const int x = lane >> 1;
            const uint32_t room = (size_t)my_base + 8 < a.ocap ? a.ocap - 8 - my_base : 0;  // 8 entries of read-ahead margin
            const uint32_t stored = my_amount < room ? my_amount : room;
            if (stored < my_amount) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
            s_obase[x] = my_base;
            s_olimit[x] = my_base + stored;
        }
    }
    __syncthreads();   // [C] image complete, pool positions known, every old byte of the tile has been read
    if (warp == 1 && (lane & 1) && lane < 4) {
        const int x = lane >> 1;
        const TensorStore& ts = x ? a.v : a.k;
        if (s_skip) {
            pool_give_back(&ts.opool_end[bh], my_base, my_taken);
        } else {
            const uint32_t stored = s_olimit[x] - s_obase[x];
            if (starts) { ts.tile[ti].z = my_base; ts.tile[ti].w = stored; }
            else ts.tile[ti].w += stored;
        }
    }
    if (s_skip) { tick(); return; }

    // ---- the image goes out with vector stores; outlier list; per-token metadata
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const TensorStore& ts = x ? a.v : a.k;
        uint8_t* dst = ts.codes + (size_t)bh * a.pool_bytes + s_base[x];
        const uint32_t nb = (s_tot[x] + 15u) & ~15u;     // tiles start 16-byte aligned and own a rounded amount
        // the value of the first listed outlier of this thread is on its way (read again from the input: the
        // registers hold -inf in its place) while the image goes out
        const uint32_t ntot = s_otot[x], nst = ntot < OUT_STAGE ? ntot : OUT_STAGE;
        const __half* X = (x ? a.V : a.K) + (size_t)b_idx * a.sb + (size_t)h_idx * a.sh;
        uint32_t w_first = 0;
        unsigned short v_first = 0;
        if ((uint32_t)tid < nst) {
            w_first = s_work[x][tid];
            v_first = __half_as_ushort(X[(size_t)(tile * QAQ_TILE + (int)(w_first >> 8) - t_old) * a.st + (w_first & 0xFFu)]);
        }
        if (x == 0) {
            for (uint32_t o = tid * 16; o < nb; o += NT * 16)
                *reinterpret_cast<uint4*>(dst + o) = *reinterpret_cast<const uint4*>(s_img[x] + o);
        } else {
            // one unit per thread, the four rows that are interleaved side by side
            const int row = (tid / (16 * P)) * 4 + (tid & 3), e = (tid >> 2) % (4 * P);
            if (row < s_tab[x][1].start + s_tab[x][1].n) {
                const int w = s_sorted[x][4 * row];
                qaqc::group_out<D>(s_img[x], dst, s_tab[x][w], w, row, e);
            }
            if (tid == 0) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(s_img[x]);
        }
        // outlier entries: one listed outlier per thread (value read again from the input: the registers hold -inf in
        // its place), stores next to each other; a tile with more outliers than are listed writes the rest one by one
        {
            if ((uint32_t)tid < nst) {
                const uint32_t pos = s_obase[x] + tid;
                if (pos < s_olimit[x]) ts.outl[(size_t)bh * a.ocap + pos] = (uint32_t)v_first | ((w_first & 0xFFu) << 16) | ((w_first >> 8) << 24);
            }
            for (uint32_t i = tid + NT; i < nst; i += NT) {
                const uint32_t w = s_work[x][i], sl = w >> 8, ch = w & 0xFFu;
                const uint32_t pos = s_obase[x] + i;
                if (pos < s_olimit[x])
                    ts.outl[(size_t)bh * a.ocap + pos] = (uint32_t)__half_as_ushort(X[(size_t)(tile * QAQ_TILE + (int)sl - t_old) * a.st + ch]) |
                                                          (ch << 16) | (sl << 24);
            }
            if (ntot > OUT_STAGE) {
                // rare.  Nothing of the listing pass is kept in registers for this: the lane reads its 32 channels
                // again and repeats the outlier test (same bounds, same bit order as analyze32)
                const __half2 lo2 = __half2half2(__float2half_ru(thr[2 * x])), hi2 = __half2half2(__float2half_rd(thr[2 * x + 1]));
                const __half* row = X + (size_t)(valid ? tn : 0) * a.st + 32 * p;
                uint32_t ob = 0;
                if (valid) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const __half2 v = as_h2(reinterpret_cast<const uint32_t*>(row)[k]);
                        ob |= (~(__hge2_mask(v, lo2) & __hle2_mask(v, hi2)) & 0x00010001u) << k;
                    }
                }
                const uint32_t mine = (uint32_t)__popc(ob);
                uint32_t lp0 = s_cnt[x][slot & (QAQ_TILE - 1)];
#pragma unroll
                for (int d = 1; d < P; ++d) {
                    const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, mine, d);
                    if (p >= d) lp0 += o;
                }
                const uint32_t all = ob;
                while (ob) {
                    const int bit = __ffs(ob) - 1;
                    ob &= ob - 1;
                    const int k = bit & 15, hi = bit >> 4;
                    const int c = 2 * k + hi;
                    const uint32_t lower = (((1u << k) - 1u) * 0x00010001u) | (hi ? (1u << k) : 0u);
                    const uint32_t lp = lp0 + (uint32_t)__popc(all & lower);
                    if (lp >= OUT_STAGE && s_obase[x] + lp < s_olimit[x])
                        ts.outl[(size_t)bh * a.ocap + s_obase[x] + lp] = (uint32_t)__half_as_ushort(row[c]) | ((uint32_t)(32 * p + c) << 16) |
                                                                           ((uint32_t)(slot & (QAQ_TILE - 1)) << 24);
                }
            }
        }
        if ((valid || old) && p == 0) ts.bs[mt] = (unsigned short)(Bx[x] | ((s_place[x][slot & (QAQ_TILE - 1)] & 0xFFu) << 8));
        if (valid && p == 0) {
            ts.mnmx[mt] = (uint32_t)__half_as_ushort(__float2half_rn(mnf[x])) | ((uint32_t)__half_as_ushort(__float2half_rn(mxf[x])) << 16);
        }
    }
    tick();
}


// ------------------------------------------------------------------------------------------ whole tiles, two warps each
// A tile of one tensor comes to shared memory by asynchronous copies and is gone through twice: tokens in order for the
// ranges and the outliers, then, with the widths known, tokens in the order they are stored in for the codes, which go
// straight to their places (a round's lanes mostly have the same width, so they seldom part at the stores; four tokens of
// a group of values swap bytes by shuffles).  What is done once per tile - the order, the sections, the space from the
// pools - is done for 64 tokens by 64 threads.
//
// What bounds it: instructions (70 % of the issue slots, 60 % of the integer unit's cycles at 7B, batch 8).  The kernel for
// any tile takes 7300 (keys) and 9100 (values) warp instructions per tile, this one 4200 on average.  4096 tokens, 256
// (b,h), head_dim 128: 188 us for keys and values, against 323 us for the other kernel in a launch for each; one warp per
// tile 231 us (11 tiles in flight per SM either way, for their shared memory); rounds unrolled by two 200 us, by four
// 226 us (the code of one round is what the instruction cache holds).  It is the faster one down to the smallest launch:
// 32 (b,h) of one tile 7.0 against 7.7 us, of 16 tiles 10.5 against 17.2 us.
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
struct Scale {                 // of a token: code = min(floor(sat((x - mn) * inv) * 2^B), 2^B - 1)
    float mn, inv;             // 1 / (max - min), which is 2^-B times the reciprocal of the step; 0 for a constant token
    uint64_t levels;           // 2^B, twice
    uint32_t top;              // 2^B - 1 in the low half, that and the bits of 2^23 in the high half
    uint32_t k64;              // 65536, kept from the compiler, which would take a byte shuffle
};
// Codes of a binary16 pair: the first in the low byte, the second in byte 2 (byte 3 is not clean).  2^23 + floor(t) has
// the code in its low bits; an outlier's place holds a number that is none, which saturates to 0.
__device__ __forceinline__ uint32_t code_pair(uint32_t v, const Scale& s) {
    float x0, x1, u0, u1;
    asm("{\n.reg .b16 h0, h1;\nmov.b32 {h0, h1}, %2;\nsub.rn.f32.f16 %0, h0, %3;\nsub.rn.f32.f16 %1, h1, %3;\n}" : "=f"(x0), "=f"(x1) : "r"(v), "f"(s.mn));
    asm("mul.rn.sat.f32 %0, %1, %2;" : "=f"(u0) : "f"(x0), "f"(s.inv));
    asm("mul.rn.sat.f32 %0, %1, %2;" : "=f"(u1) : "f"(x1), "f"(s.inv));
    uint64_t t;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(t) : "l"(pair_of(u0, u1)), "l"(s.levels), "l"(pair_of(8388608.0f, 8388608.0f)));
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(mad((uint32_t)(t >> 32), s.k64, (uint32_t)t)), "r"(s.top));
    return d;
}
constexpr uint32_t GONE = 0xFFFFu;      // in the place of an outlier: not a number

// What a warp keeps of its tile in shared memory.  The 16-byte pieces of the rows are stored swizzled (piece U at U ^ (U/8
// mod 4)), so that lanes that read 64 bytes each do not meet in the banks.
template <int D>
struct TileScratch {
    alignas(64) uint8_t data[QAQ_TILE * D * 2];
    uint4 slot[QAQ_TILE];              // by slot: minimum, 1 / step, byte offsets of the parts, what else a lane has to know
    uint32_t range[QAQ_TILE];          // by token: min | max << 16
    alignas(16) uint32_t out[QAQ_TILE * D / 32];  // by token and 32 channels: which are outliers
    alignas(8) uint32_t count[2][2];   // by half of the tile: tokens of every width, a byte each
    uint32_t nout[2], base[2];         // outliers of the halves; space taken for the tile and for its outlier list
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
// One tile of one tensor, by two warps: half of its tokens each until the widths are known, half of the slots each from there.
template <int D, bool IS_V>
__device__ __forceinline__ void quantize_tile(const QuantArgs& a, TileScratch<D>& sm, uint32_t* list, const uint32_t cap) {
    constexpr int P = D / 32, TPI = 32 / P, IT = QAQ_TILE / 2 / TPI;  // lanes per token, tokens of a warp at a time, rounds
    constexpr int PR = D / 8;                                         // 16-byte pieces of a row
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane / P, p = lane % P;
    const int tile = a.first_tile + blockIdx.x, bh = blockIdx.y, tn0 = tile * QAQ_TILE - a.t_old;
    const TensorStore& ts = IS_V ? a.v : a.k;
    const __half* X = (IS_V ? a.V : a.K) + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh + (size_t)tn0 * a.st;
    const uint32_t data = (uint32_t)__cvta_generic_to_shared(sm.data);
    {
        const __half* src = X + (size_t)(32 * warp + lane / PR) * a.st + 8 * (lane % PR);
        const uint32_t dst = data + warp * (QAQ_TILE * D) + 16 * (lane ^ ((lane >> 3) & 3));
#pragma unroll
        for (int i = 0; i < PR; ++i, src += (32 / PR) * a.st)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 * i), "l"(src) : "memory");
    }
    const float* thr = a.thr + (size_t)bh * 4 + (IS_V ? 2 : 0);
    // thresholds as binary16 bounds that decide exactly like the binary32 ones on binary16 data
    const __half2 lo2 = __half2half2(__float2half_ru(thr[0])), hi2 = __half2half2(__float2half_rd(thr[1]));
    uint32_t* const pool = (lane ? ts.opool_end : ts.pool_end) + bh;
    uint32_t pool_now = 0;
    if (tid < 2) pool_now = *pool;
    // ---- attention window of this thread's token
    const bool given = a.bitsK != nullptr;
    int b = 0, nv = 0;
    float shat = __int_as_float(0xff800000);
    if (given) {
        b = (IS_V ? a.bitsV : a.bitsK)[(size_t)bh * a.n_new + tn0 + tid];
    } else if (IS_V) {
        nv = min((int)a.nvalid[(size_t)bh * a.n_new + tn0 + tid], a.W);
        shat = qaqc::window_max(a.ring + (size_t)bh * a.W * a.n_new + tn0 + tid, a.W, a.n_new, nv);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();

    // ---- ranges and outliers, tokens in order: an outlier goes to the warp's list, its place is marked
    list += warp * cap;
#pragma unroll 1
    for (int it = 0; it < IT; ++it) {
        const int tok = 32 * warp + it * TPI + g, U = tok * PR + 4 * p;
        const uint32_t at = data + 16 * (U ^ ((U >> 3) & 3));
        uint32_t v[16];
        load_row(at, v);
        __half2 mn2, mx2;
        uint32_t ob = outliers_and_range(v, lo2, hi2, mn2, mx2);
        __half2 pk = __halves2half2(__hmin(__low2half(mn2), __high2half(mn2)), __hneg(__hmax(__low2half(mx2), __high2half(mx2))));
#pragma unroll
        for (int o = 1; o < P; o <<= 1) pk = __hmin2(pk, as_h2(__shfl_xor_sync(0xFFFFFFFFu, as_u32(pk), o)));
        if (p == 0) sm.range[tok] = __hgt(__low2half(pk), __hneg(__high2half(pk))) ? 0u : as_u32(pk) ^ 0x80000000u;    // 0, 0: no inlier
        sm.out[tok * P + p] = ob;
    }
    __syncwarp();
    // ---- the outliers go to the warp's list, a token per lane, their places are marked
    uint32_t nout;
    {
        uint32_t ob[P], cnt = 0;
        if constexpr (P == 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(&sm.out[tid * P]);
            ob[0] = x.x; ob[1] = x.y; ob[2] = x.z; ob[3] = x.w;
        } else {
#pragma unroll
            for (int k = 0; k < P; ++k) ob[k] = sm.out[tid * P + k];
        }
#pragma unroll
        for (int k = 0; k < P; ++k) cnt += (uint32_t)__popc(ob[k]);
        uint32_t pos = prefix(cnt, lane, nout);
#pragma unroll
        for (int k = 0; k < P; ++k)
            while (ob[k]) {
                const uint32_t c = 32 * k + (uint32_t)__ffs(ob[k]) - 1u, U = tid * PR + (c >> 3);
                ob[k] &= ob[k] - 1;
                unsigned short* where = reinterpret_cast<unsigned short*>(sm.data + 16 * (U ^ ((U >> 3) & 3))) + (c & 7);
                if (pos < cap) list[pos] = ((uint32_t)tid << 24) | (c << 16) | *where;
                *where = GONE;
                ++pos;
            }
    }

    // ---- widths; which tokens have which
    const uint32_t range = sm.range[tid];
    const float mn = __low2float(as_h2(range)), mx = __high2float(as_h2(range));
    {
        const float r = __fsub_rn(mx, mn);
        if (given) b = b < 1 ? 1 : (b > 8 ? 8 : b);
        else if (!IS_V) b = ladder(r, a.cK, a.bmin, a.bmax);
        else b = nv == 0 ? a.bmax : ladder(__fmul_rn(r, shat), a.cV, a.bmin, a.bmax);
    }
    const uint32_t alike = qaqc::count_half(b, lane, sm.count[warp]);
    if (lane == 0) sm.nout[warp] = nout;
    __syncthreads();
    // ---- order and sections, by both warps alike; space from the pools
    int slot;
    const qaqc::TileRows rows = qaqc::rows_of_counts<IS_V>(sm.count, b, alike, warp, lane, slot);
    const uint32_t total = qaqc::tile_total<D, IS_V>(rows);
    const uint32_t nout0 = sm.nout[0], nall = nout0 + sm.nout[1];
    uint32_t base = 0, taken = 0;
    if (tid < 2) base = pool_take(pool, lane ? nall : total, lane ? 3u : 15u, true, true, pool_now > (lane ? a.ocap : a.pool_bytes), taken);
    {
        const int row = IS_V ? slot >> 2 : slot, row_w = IS_V ? qaqc::width_of_row(rows, row) : b;
        const qaqc::RowPlace pl = qaqc::place_row<D, IS_V>(rows, row, row_w);
        // the reciprocal of the step without its power of two (the range of binary16 numbers is nowhere near the ends of
        // binary32: both are the same number but for the exponent)
        const float len = __fsub_rn(mx, mn), inv = len > 0.f ? __fdiv_rn(1.0f, len) : 0.f;
        const bool endless = len > 0.f && inv == 0.f;         // a range that is not finite
        sm.slot[slot] = make_uint4(__float_as_uint(mn), __float_as_uint(inv), pl.main | (pl.high << 16),
                                   (uint32_t)tid | ((uint32_t)b << 8) | ((uint32_t)row_w << 16) | (pl.mm << 20) | (pl.mh << 24) | (endless ? 0x80000000u : 0u));
    }
    // ---- a pool without room: the space is given back, nothing about the tile is published; the device status reports
    //      the lost tokens
    if (warp == 0) {
        const uint32_t off = __shfl_sync(0xFFFFFFFFu, base, 0);
        const bool fail = (size_t)off + __shfl_sync(0xFFFFFFFFu, taken, 0) + 16 > a.pool_bytes || (size_t)off + total + 16 > a.pool_bytes;
        if (fail && lane < 2) pool_give_back(pool, base, taken);
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
        ts.tile[(size_t)bh * a.ntiles + tile] = make_uint4(off, total, obase, stored);
        *reinterpret_cast<uint4*>(dst) = qaqc::header_of<D, IS_V>(rows);
    }
    {
        const size_t mt = (size_t)bh * a.tmax_pad + (size_t)tile * QAQ_TILE + tid;
        ts.bs[mt] = (unsigned short)(b | (slot << 8));
        ts.mnmx[mt] = range;
    }
    const uint32_t first = warp ? nout0 : 0u;
    for (uint32_t i = lane; i < min(nout, cap); i += 32)
        if (first + i < stored) outl[first + i] = list[i];
    if (nout > cap) {                  // more outliers than were listed: the rest is found once more in the input
        uint32_t seen = 0;
#pragma unroll 1
        for (int it = 0; it < IT; ++it) {
            const int tok = 32 * warp + it * TPI + g;
            const __half* row = X + (size_t)tok * a.st + 32 * p;
            uint32_t v[16];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 x = *reinterpret_cast<const uint4*>(row + 8 * i);
                v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
            }
            __half2 mn2, mx2;
            uint32_t ob = outliers_and_range(v, lo2, hi2, mn2, mx2);
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
#pragma unroll 1
    for (int it = 0; it < IT; ++it) {
        const uint4 q = sm.slot[32 * warp + it * TPI + g];
        const int U = (int)(q.w & 63u) * PR + 4 * p, B = (int)((q.w >> 8) & 15u), w = (int)((q.w >> 16) & 15u);
        uint32_t v[16], c[16], lo[4], hi[4];
        load_row(data + 16 * (U ^ ((U >> 3) & 3)), v);
        sc.mn = __uint_as_float(q.x);
        sc.inv = __uint_as_float(q.y);
        const float levels = __int_as_float((127 + B) << 23);
        sc.levels = pair_of(levels, levels);
        sc.top = ((1u << B) - 1u) * 0x00010001u + 0x4B000000u;
#pragma unroll
        for (int k = 0; k < 16; ++k) c[k] = code_pair(v[k], sc);
        if (__any_sync(0xFFFFFFFFu, q.w >> 31)) {
            if (q.w >> 31) {           // marks become -inf, which the plain arithmetic takes to code 0
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
        const bool wide = __any_sync(0xFFFFFFFFu, w > 4);
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
        if (IS_V) qaqc::transpose4<P>(lo, g & 3);
        const int e = IS_V ? 4 * p + (g & 3) : p;
        const int wm = min(w, 4);
        qaqc::store_nibbles(dst + (q.z & 0xFFFFu) + (IS_V ? e * (int)((q.w >> 20) & 7u) : e) * 4 * wm, wm, lo);
        if (wide) {
            if (IS_V) qaqc::transpose4<P>(hi, g & 3);
            if (w > 4) qaqc::store_nibbles(dst + (q.z >> 16) + (IS_V ? e * (int)((q.w >> 24) & 7u) : e) * 4 * (w - 4), w - 4, hi);
        }
    }
}

template <int D>
__global__ void __launch_bounds__(64, D == 128 ? 11 : 12) quant_tiles_kernel(const QuantArgs a, uint32_t cap) {
    extern __shared__ __align__(64) unsigned char tiles_smem[];
    TileScratch<D>& sm = *reinterpret_cast<TileScratch<D>*>(tiles_smem);
    uint32_t* list = reinterpret_cast<uint32_t*>(tiles_smem + sizeof(TileScratch<D>));
    qaq_dependency();
    if (blockIdx.z == 0) quantize_tile<D, false>(a, sm, list, cap);
    else quantize_tile<D, true>(a, sm, list, cap);
}

template <int D>
qaq_status launch_tiles(dim3 grid, const QuantArgs& a, double alpha, cudaStream_t s) {
    // the list holds a third more than the share of outliers asked for gives a tile, and some
    const uint32_t want = (uint32_t)(alpha * (QAQ_TILE * D) * 1.34) + 96, cap = (want < 2048 ? want : 2048) / 2;
    QAQ_CUDA_TRY(qaq_launch(quant_tiles_kernel<D>, grid, dim3(64), sizeof(TileScratch<D>) + 2 * cap * sizeof(uint32_t), s, a, cap));
    return QAQ_OK;
}

template <bool SELECT_ONLY>
qaq_status launch(int D, dim3 grid, const QuantArgs& a, cudaStream_t s) {
    switch (D) {
        case 32: QAQ_CUDA_TRY(qaq_launch(quant_kernel<32, SELECT_ONLY>, grid, dim3(64), 0, s, a)); break;
        case 64: QAQ_CUDA_TRY(qaq_launch(quant_kernel<64, SELECT_ONLY>, grid, dim3(128), 0, s, a)); break;
        case 128: QAQ_CUDA_TRY(qaq_launch(quant_kernel<128, SELECT_ONLY>, grid, dim3(256), 0, s, a)); break;
        default: return QAQ_ERR_UNSUPPORTED_SHAPE;
    }
    return QAQ_OK;
}

// whole tiles
qaq_status launch_whole(int D, dim3 grid, const QuantArgs& a, double alpha, cudaStream_t s) {
    grid.z = 2;
    switch (D) {
        case 32: return launch_tiles<32>(grid, a, alpha, s);
        case 64: return launch_tiles<64>(grid, a, alpha, s);
        case 128: return launch_tiles<128>(grid, a, alpha, s);
    }
    return QAQ_ERR_UNSUPPORTED_SHAPE;
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
    dim3 grid((n + QAQ_TILE - 1) / QAQ_TILE, cfg->batch * cfg->heads);
    return launch<true>(cfg->head_dim, grid, a, s);
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
        if ((stt = launch<false>(D, dim3(1, BH), a, s)) != QAQ_OK) return stt;
        cur = end;
    }
    const int full_end = t1 / QAQ_TILE * QAQ_TILE;
    if (cur < full_end) {       // body: whole tiles
        a.tok_lo = cur - t0; a.tok_hi = full_end - t0; a.first_tile = cur / QAQ_TILE;
        if ((stt = launch_whole(D, dim3((full_end - cur) / QAQ_TILE, BH), a, c->cfg.outlier_frac, s)) != QAQ_OK) return stt;
        cur = full_end;
    }
    if (cur < t1) {             // tail: a new, partly filled tile
        a.tok_lo = cur - t0; a.tok_hi = t1 - t0; a.first_tile = cur / QAQ_TILE;
        if ((stt = launch<false>(D, dim3(1, BH), a, s)) != QAQ_OK) return stt;
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
    st = launch<false>(D, dim3(1, c->BH), a, (cudaStream_t)stream);
    return st;
}
