// Re-quantization of cached tokens (Section 4.2 of the paper, "Integration in text generation
// process"): in every generation step the widths of all cached tokens are computed again.
//   lower width:  the token is quantized further.  The quantizer is nested (min and range kept,
//                 the B'-bit code is the B-bit code without its low B-B' bits), so this needs
//                 nothing but the packed cache:  code >>= (B - B').
//   higher width: the paper takes the unquantized values from a copy kept in CPU memory and
//                 quantizes them again.  Here the caller passes that copy (any memory the GPU can
//                 read, e.g. mapped pinned host memory: only the rows of the raised tokens are
//                 touched); min, max and the outliers of the token stay what they were, the codes
//                 are computed as at append time.  Without a copy, widths are only lowered.
// The new widths come from the caller or from the rules of Section 4.1 applied to the stored
// range (max - min of the token's metadata) with the current score window and policy scalars.
//
// Two warps = one tile (QAQ_TILE tokens) of one (b,h) and tensor.  A thread finds the new width of one token; a CTA whose
// widths stay as they are leaves.  Otherwise the tile's bytes come to shared memory, and the tokens are gone through in
// their new order, head_dim/32 lanes to a token: words of the old tile, low bits dropped in the nibbles (or codes from
// the unquantized row), words of the new tile straight to where they belong, which is where the tile was, unless it grows.
// A closed tile that grows takes a new place at the end of its pool (the
// old bytes stay unused); the open (last, partly filled) tile is then handled in a launch of its own
// after the closed ones and is kept - or made again - the last thing in its pool, so that later
// appends continue right behind it.  Lowered widths never make a tile grow.
//
// What bounds it: instructions, and where few tiles change the latency of the metadata and of the window.  With a thread per
// 32 channels from the start, every tile of changed widths decoded to codes, encoded to an image and copied out, lowering
// a 4096-token layer at batch 4 took 120 us and raising it again 170; as it is now 55 and 103.  With a step's few changes
// (2048 tokens, batch 4) 29.6 us became 15.9.
#include "qaq_codec.cuh"
#include "qaq_internal.cuh"

namespace {

struct RequantArgs {
    TensorStore k, v;
    size_t pool_bytes;
    int tmax_pad, ntiles;
    int H, T;                // heads; cached tokens
    long ncols;              // row length of bitsK/bitsV/ring/nvalid (>= T)
    const uint8_t* bitsK;    // requested widths [BH][ncols] or null
    const uint8_t* bitsV;
    const float* ring;       // [BH][W][ncols]
    const uint8_t* nvalid;   // [BH][ncols]
    int W;
    float cK, cV;
    int bmin, bmax;
    // raising widths: the unquantized values [B,H,T,D] (element strides), the thresholds, the tile to start at
    const __half* Ks;
    const __half* Vs;
    long sb, sh, st;
    const float* thr;        // [BH][4]
    int first_tile;
    int* status;
};

using qaqc::ladder;

// Codes of one lane's 32 channels computed from the unquantized row, as at append time:
// code = min(2^B - 1, floor((x - min) * (1/step))) in binary32, 0 for an outlier (outside [lo, hi]).
__device__ __forceinline__ void fresh_codes(const __half* row, float lo, float hi, float mn, float mx, int B, uint32_t (&creg)[8]) {
    uint32_t v[16];
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
        const uint4 raw = *reinterpret_cast<const uint4*>(row + 8 * q4);
        v[4 * q4] = raw.x; v[4 * q4 + 1] = raw.y; v[4 * q4 + 2] = raw.z; v[4 * q4 + 3] = raw.w;
    }
    qaqc::mask_outliers32(v, __half2half2(__float2half_ru(lo)), __half2half2(__float2half_rd(hi)));
    qaqc::codes32(v, mn, mx, B, creg);
}

// 32 codes, one per nibble pair of lo and hi (bits 0..3 and 4..7 of the codes, in nibble words), without their low d bits
__device__ __forceinline__ void drop_bits(uint32_t (&lo)[4], uint32_t (&hi)[4], int d) {
    if (d >= 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) { lo[u] = hi[u]; hi[u] = 0; }
        d -= 4;
    }
    const uint32_t keep = 0x11111111u * (0xFu >> d);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        lo[u] = ((lo[u] >> d) & keep) | ((hi[u] << (4 - d)) & ~keep);
        hi[u] = (hi[u] >> d) & keep;
    }
}
// What the CTA keeps of its tile.
template <int D>
struct RequantScratch {
    alignas(16) uint8_t old[qaqc::tile_bytes_max(D) + 16];
    // by new slot: byte offsets of the row's parts before | and after << 16 (main, high); token, widths before and after, row
    // widths before and after; for values the distances of the units and the old slot's place in its group
    alignas(16) uint4 slot[QAQ_TILE];
    uint32_t range[QAQ_TILE];
    alignas(8) uint32_t count[2][2];
    uint32_t off;
    int skip;
};

// One tile of one tensor.  UP: widths may be raised (the unquantized copy is there).
template <int D, bool UP, bool IS_V>
__device__ __forceinline__ void requantize_tile(const RequantArgs& a, RequantScratch<D>& sm) {
    constexpr int P = D / 32, TPI = 32 / P, IT = QAQ_TILE / 2 / TPI;      // lanes per token, tokens of a warp at a time, rounds
    const int tile = a.first_tile + blockIdx.x, bh = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane / P, p = lane % P;
    const int tok = tile * QAQ_TILE + tid;
    const bool valid = tok < a.T;
    const TensorStore& ts = IS_V ? a.v : a.k;
    const size_t ti = (size_t)bh * a.ntiles + tile;

    // ---- current width and range of this thread's token, its new width: the rule's (or the caller's) width; without the
    //      unquantized copy only where it is lower
    const size_t mt = (size_t)bh * a.tmax_pad + tok;
    const uint4 tw = ts.tile[ti];
    const uint32_t pool_end = ts.pool_end[bh];
    int Bo = 0, oslot = 0, Bn = 0;
    uint32_t range = 0;
    if (valid) {
        const uint32_t bs = ts.bs[mt];
        range = ts.mnmx[mt];
        Bo = min((int)(bs & 0xFFu), 8);
        oslot = (int)((bs >> 8) & (QAQ_TILE - 1));
    }
    const float rng = __fsub_rn(__half2float(__ushort_as_half((unsigned short)(range >> 16))), __half2float(__ushort_as_half((unsigned short)(range & 0xFFFF))));
    {
        int B = 0;
        if (a.bitsK) {
            if (valid) B = (IS_V ? a.bitsV : a.bitsK)[(size_t)bh * a.ncols + tok];
            B = B < 1 ? 1 : (B > 8 ? 8 : B);
        } else if (!IS_V) {
            B = ladder(rng, a.cK, a.bmin, a.bmax);
        } else {
            const long col = (long)min(tok, a.T - 1);           // whole warps read the window; columns beyond the last are not used
            const int nv = min((int)a.nvalid[(size_t)bh * a.ncols + col], a.W);
            const float sh = qaqc::window_max<16, true>(a.ring + (size_t)bh * a.W * a.ncols + col, a.W, a.ncols, nv);
            if (__float_as_uint(sh) == QAQ_SCORE_LOST) atomicMax(a.status, (int)QAQ_ERR_CUDA);
            B = nv == 0 ? a.bmax : ladder(__fmul_rn(rng, sh), a.cV, a.bmin, a.bmax);
        }
        if (valid) Bn = (UP || B < Bo) ? B : Bo;
    }
    // a raised token's row is on its way to L2 while the tile's order is found
    if (UP && Bn > Bo) {
        const __half* row = (IS_V ? a.Vs : a.Ks) + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh + (size_t)tok * a.st;
#pragma unroll
        for (int i = 0; i < D; i += 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + i));
    }
    const uint32_t alike = qaqc::count_half(Bn, lane, sm.count[warp]);
    bool changed = __syncthreads_or(Bn != Bo) != 0;          // also makes the counts visible
    // An open tile has to be the last thing in its pool.  If closed tiles of this (b,h) have just been moved
    // behind it, it moves to the end as well, whether its own tokens change or not.
    const bool open = tile == a.T / QAQ_TILE && (a.T % QAQ_TILE) != 0;
    const bool relocate = open && tw.x + tw.y != pool_end;
    changed = changed || relocate;
    if (!changed) return;

    // ---- the stored bytes come to shared memory; order, size and place of the new tile
    const uint8_t* src = ts.codes + (size_t)bh * a.pool_bytes + tw.x;
    const uint32_t old_nb = min(tw.y, (uint32_t)qaqc::tile_bytes_max(D));
    for (uint32_t o = tid * 16; o < old_nb; o += 64 * 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(sm.old + o)), "l"(src + o) : "memory");
    int slot;
    const qaqc::TileRows rows = qaqc::rows_of_counts<IS_V>(sm.count, Bn, alike, warp, lane, slot);
    const uint32_t nb = qaqc::tile_total<D, IS_V>(rows);
    sm.range[tid] = range;
    if (tid == 0) {
        // where the new tile goes: in place unless it grows
        const uint32_t off = tw.x;
        const uint32_t old_own = open ? old_nb : ((old_nb + 15u) & ~15u);   // closed tiles own a rounded amount
        uint32_t noff = off;
        int skip = 0;
        if (nb > old_own || relocate) {
            if (open && off + old_nb == pool_end) {
                // still the last thing in its pool: it grows where it is
                if ((size_t)off + nb + 16 > a.pool_bytes) skip = 1;
                else ts.pool_end[bh] = off + nb;
            } else if (open) {
                // behind everything else, 16-byte aligned, and exactly as long as its bytes: the last thing
                // in the pool again (one CTA per pool does this, and nobody else touches the pool in its launch)
                noff = (pool_end + 15u) & ~15u;
                if ((size_t)noff + nb + 16 > a.pool_bytes) skip = 1;
                ts.pool_end[bh] = skip ? noff : noff + nb;         // (without room: where whole tiles can begin)
            } else {
                // the end of the pool need not be aligned while a tile is open: take 16 bytes more and align;
                // space that does not fit is given back
                const uint32_t take = ((nb + 15u) & ~15u) + 16u;
                const bool full = *(volatile uint32_t*)&ts.pool_end[bh] > a.pool_bytes;      // takes nothing: the end must not run away
                const uint32_t at = full ? 0u : atomicAdd(&ts.pool_end[bh], take);
                noff = (at + 15u) & ~15u;
                if (full) skip = 1;
                else if ((size_t)at + take + 16 > a.pool_bytes) { skip = 1; pool_give_back(&ts.pool_end[bh], at, take); }
            }
            if (skip) atomicMax(a.status, (int)QAQ_ERR_CAPACITY);
        }
        sm.off = noff; sm.skip = skip;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (sm.skip) return;                 // no room in the pool: the tile stays as it is
    const uint32_t noff = sm.off;
    if (valid && Bn) {
        uint4 h = *reinterpret_cast<const uint4*>(sm.old);
        if (!tw.y) h = make_uint4(0u, 0u, 0u, 0u);
        const qaqc::TileRows orows = qaqc::rows_of_header(h.x, h.y);
        const int orow = IS_V ? oslot >> 2 : oslot, ow = IS_V ? max(1, min(8, qaqc::width_of_row(orows, orow))) : max(Bo, 1);
        const qaqc::RowPlace o = qaqc::place_row<D, IS_V>(orows, orow, ow);
        const int row = IS_V ? slot >> 2 : slot, w = IS_V ? qaqc::width_of_row(rows, row) : Bn;
        const qaqc::RowPlace n = qaqc::place_row<D, IS_V>(rows, row, w);
        sm.slot[slot] = make_uint4(o.main | (n.main << 16), o.high | (n.high << 16),
                                   (uint32_t)tid | ((uint32_t)Bo << 8) | ((uint32_t)Bn << 12) | ((uint32_t)ow << 16) | ((uint32_t)w << 20),
                                   o.mm | (o.mh << 4) | (n.mm << 8) | (n.mh << 12) | ((uint32_t)(oslot & 3) << 16));
    }
    __syncthreads();

    uint8_t* dst = ts.codes + (size_t)bh * a.pool_bytes + noff;
    const int nt = (int)(((sm.count[0][0] + sm.count[1][0]) * qaqc::ONES >> 24) + ((sm.count[0][1] + sm.count[1][1]) * qaqc::ONES >> 24));     // slots in use
#pragma unroll 1
    for (int it = 0; it < IT; ++it) {
        const int sl = 32 * warp + it * TPI + g;
        uint32_t lo[4] = {0, 0, 0, 0}, hi[4] = {0, 0, 0, 0};
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (sl < nt) {
            q = sm.slot[sl];
            const int t = (int)(q.z & 63u), bo = (int)((q.z >> 8) & 15u), bn = (int)((q.z >> 12) & 15u), ow = (int)((q.z >> 16) & 15u);
            if (UP && bn > bo) {
                // raised: with the token's stored min / max and the thresholds
                const uint32_t mm = sm.range[t];
                const float mn = __half2float(__ushort_as_half((unsigned short)(mm & 0xFFFF))), mx = __half2float(__ushort_as_half((unsigned short)(mm >> 16)));
                const __half* row = (IS_V ? a.Vs : a.Ks) + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh + (size_t)(tile * QAQ_TILE + t) * a.st + 32 * p;
                uint32_t creg[8];
                fresh_codes(row, a.thr[(size_t)bh * 4 + 2 * IS_V], a.thr[(size_t)bh * 4 + 2 * IS_V + 1], mn, mx, bn, creg);
                qaqc::nibbles_of(creg, 0, lo);
                qaqc::nibbles_of(creg, 4, hi);
            } else {
                qaqc::take_token<D, IS_V>(sm.old, sizeof(sm.old), q.x & 0xFFFFu, q.y & 0xFFFFu, ow, q.w & 15u, (q.w >> 4) & 15u, (int)((q.w >> 16) & 3u), p, lo, hi);
                drop_bits(lo, hi, bo - bn);
            }
        }
        __syncwarp();
        if (IS_V) {                    // the group's row: that of its first slot
            const int first = sl & ~3;
            if (first < nt) q = sm.slot[first];
        }
        const int w = (int)((q.z >> 20) & 15u);
        const bool wide = __any_sync(0xFFFFFFFFu, w > 4);
        if (IS_V) qaqc::transpose4<P>(lo, g & 3);
        if (IS_V && wide) qaqc::transpose4<P>(hi, g & 3);
        const int e = IS_V ? 4 * p + (g & 3) : p;
        if (w) {
            const int wm = min(w, 4);
            qaqc::store_nibbles(dst + (q.x >> 16) + (IS_V ? e * (int)((q.w >> 8) & 15u) : e) * 4 * wm, wm, lo);
            if (w > 4) qaqc::store_nibbles(dst + (q.y >> 16) + (IS_V ? e * (int)((q.w >> 12) & 15u) : e) * 4 * (w - 4), w - 4, hi);
        }
    }
    if (valid && Bn) ts.bs[mt] = (unsigned short)(Bn | (slot << 8));
    if (tid == 0) {
        *reinterpret_cast<uint4*>(dst) = qaqc::header_of<D, IS_V>(rows, tw.y ? reinterpret_cast<const uint4*>(sm.old)->w >> 16 : 0u);
        // an open tile that is still the last thing in its pool gives back what it no longer needs:
        // appends continue right behind its bytes
        if (open && noff == tw.x && nb < tw.y && tw.x + tw.y == pool_end) ts.pool_end[bh] = noff + nb;
        ts.tile[ti].x = noff;
        ts.tile[ti].y = nb;
    }
}

// blockIdx.z: keys or values.  64 registers, 16 CTAs per SM: with 80 and 12 lowering a 4096-token layer at batch 4 takes 61
// instead of 55 us, raising it 111 instead of 103; 51 and 20 are no better.
template <int D, bool UP>
__global__ void __launch_bounds__(64, 16) requant_kernel(const RequantArgs a) {
    __shared__ RequantScratch<D> sm;
    qaq_dependency();
    if (blockIdx.z == 0) requantize_tile<D, UP, false>(a, sm);
    else requantize_tile<D, UP, true>(a, sm);
}

template <bool UP>
qaq_status launch_requant(int D, dim3 grid, const RequantArgs& a, cudaStream_t s) {
    switch (D) {
        case 32: QAQ_CUDA_TRY(qaq_launch(requant_kernel<32, UP>, grid, dim3(64), 0, s, a)); break;
        case 64: QAQ_CUDA_TRY(qaq_launch(requant_kernel<64, UP>, grid, dim3(64), 0, s, a)); break;
        case 128: QAQ_CUDA_TRY(qaq_launch(requant_kernel<128, UP>, grid, dim3(64), 0, s, a)); break;
        default: return QAQ_ERR_UNSUPPORTED_SHAPE;
    }
    return QAQ_OK;
}

// a pointer the GPU can read: device memory, managed memory or mapped (pinned) host memory
const void* device_view(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { (void)cudaGetLastError(); return nullptr; }
    if (at.type == cudaMemoryTypeUnregistered) return nullptr;   // pageable host memory
    return at.devicePointer;
}

}  // namespace

extern "C" qaq_status qaq_requantize(qaq_cache* c, const void* K_full, const void* V_full, long stride_b, long stride_h,
                                     long stride_t, const float* thr, const uint8_t* bitsK, const uint8_t* bitsV,
                                     const qaq_policy* policy, const float* score_ring, const uint8_t* nvalid,
                                     long n_cols, void* stream) {
    if (!c) return QAQ_ERR_INVALID_ARG;
    if ((bitsK == nullptr) != (bitsV == nullptr)) return QAQ_ERR_INVALID_ARG;
    if (!bitsK && (!policy || !score_ring || !nvalid)) return QAQ_ERR_INVALID_ARG;
    if ((K_full == nullptr) != (V_full == nullptr)) return QAQ_ERR_INVALID_ARG;
    const bool up = K_full != nullptr;
    if (c->tokens == 0) return QAQ_OK;
    if (n_cols < c->tokens) return QAQ_ERR_INVALID_ARG;
    RequantArgs a{};
    a.k = c->t[0]; a.v = c->t[1]; a.pool_bytes = c->pool_bytes; a.tmax_pad = c->tmax_pad; a.ntiles = c->ntiles;
    a.H = c->cfg.heads; a.T = (int)c->tokens; a.ncols = n_cols;
    a.bitsK = bitsK; a.bitsV = bitsV; a.ring = score_ring; a.nvalid = nvalid; a.W = c->cfg.window;
    a.cK = policy ? policy->cK : 0.f; a.cV = policy ? policy->cV : 0.f;
    a.bmin = c->cfg.bits_min; a.bmax = c->cfg.bits_max;
    a.status = c->d_status;
    cudaStream_t s = (cudaStream_t)stream;
    const int D = c->cfg.head_dim;
    const int ntile = (int)((c->tokens + QAQ_TILE - 1) / QAQ_TILE);
    if (up) {
        if (!thr) return QAQ_ERR_INVALID_ARG;
        if (stride_t < D || (stride_b & 7) || (stride_h & 7) || (stride_t & 7) || stride_b < 0 || stride_h < 0) return QAQ_ERR_INVALID_ARG;
        a.Ks = (const __half*)device_view(K_full); a.Vs = (const __half*)device_view(V_full);
        if (!a.Ks || !a.Vs || ((uintptr_t)a.Ks & 15) || ((uintptr_t)a.Vs & 15)) return QAQ_ERR_INVALID_ARG;
        a.sb = stride_b; a.sh = stride_h; a.st = stride_t; a.thr = thr;
    }
    // Where widths may be raised, closed tiles come first (a tile that grows moves to the end of its pool), then the open
    // tile, which has to be the last thing in its pool when this call is over.  Lowered widths move nothing: one launch.
    const int closed = (int)(c->tokens / QAQ_TILE);
    if (!up) {
        a.first_tile = 0;
        return launch_requant<false>(D, dim3((unsigned)ntile, (unsigned)c->BH, 2), a, s);
    }
    qaq_status st = QAQ_OK;
    if (closed > 0) {
        a.first_tile = 0;
        if ((st = launch_requant<true>(D, dim3((unsigned)closed, (unsigned)c->BH, 2), a, s)) != QAQ_OK) return st;
    }
    if (closed < ntile) {
        a.first_tile = closed;
        st = launch_requant<true>(D, dim3(1, (unsigned)c->BH, 2), a, s);
    }
    return st;
}

extern "C" qaq_status qaq_requantize_down(qaq_cache* c, const uint8_t* bitsK, const uint8_t* bitsV,
                                          const qaq_policy* policy, const float* score_ring, const uint8_t* nvalid,
                                          long n_cols, void* stream) {
    return qaq_requantize(c, nullptr, nullptr, 0, 0, 0, nullptr, bitsK, bitsV, policy, score_ring, nvalid, n_cols, stream);
}

// ---------------------------------------------------------------------------------------
// Compaction of the code pools.  Tiles that grew in qaq_requantize were placed anew at the end
// of their pool and left their old bytes behind; this closes the gaps again: the tiles of a
// (b,h) pool are moved down, in the order in which they lie in memory, until they are
// contiguous (16-byte aligned each), the open tile last.  One CTA per (b,h) and tensor: offsets sorted, new offsets
// by a prefix sum, then the pool is written front to back in rounds of 64 KB, whatever tiles the bytes
// belong to.  All loads of a round come before its first store; a byte moves to a lower address or
// stays, so what a round overwrites no later round reads.  (128 (b,h) of 4096 tokens whose tiles have all moved, 67 MB:
// 25 us.  In rounds of 32 KB, every piece's tile found by bisection and the offsets summed by every thread for itself it
// took 40 us, moved tile by tile in pieces of 4 KB 94.)
namespace {

constexpr int COMPACT_MAX_TILES = 4096;
constexpr int COMPACT_REGS = 8;           // 16-byte pieces per thread and round

struct CompactArgs {
    TensorStore t[2];
    size_t pool_bytes;
    int ntiles, T, n2;       // n2: tiles per (b,h), rounded up to a power of two
};

// dynamic shared memory: n2 keys of 8 bytes, n2 + 1 new offsets, one partial sum per warp
template <int COMPACT_THREADS>
__global__ void __launch_bounds__(COMPACT_THREADS) compact_kernel(const CompactArgs a) {
    qaq_dependency();
    const int bh = blockIdx.x, tid = threadIdx.x;
    const TensorStore& ts = a.t[blockIdx.y];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long* s_key = reinterpret_cast<unsigned long long*>(smem_raw);      // current offset << 32 | tile index
    uint32_t* s_dst = reinterpret_cast<uint32_t*>(s_key + a.n2);                      // new offset of the tile of every rank, end
    uint32_t* s_sum = s_dst + a.n2 + 1;
    const int nt = (a.T + QAQ_TILE - 1) / QAQ_TILE;
    uint4* tab = ts.tile + (size_t)bh * a.ntiles;
    for (int i = tid; i < a.n2; i += COMPACT_THREADS)
        s_key[i] = i < nt ? ((unsigned long long)tab[i].x << 32) | (unsigned)i : ~0ull;
    __syncthreads();
    // bitonic sort by current offset
    for (int k = 2; k <= a.n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < a.n2; i += COMPACT_THREADS) {
                const int l = i ^ j;
                if (l > i) {
                    const unsigned long long x = s_key[i], y = s_key[l];
                    const bool up = (i & k) == 0;
                    if ((x > y) == up) { s_key[i] = y; s_key[l] = x; }
                }
            }
            __syncthreads();
        }
    // new offsets: closed tiles own a 16-byte rounded amount; the open tile, if it is the last one, its exact bytes
    const int per = (nt + COMPACT_THREADS - 1) / COMPACT_THREADS, lo = min(nt, tid * per), hi = min(nt, lo + per);
    uint32_t sum = 0;
    for (int i = lo; i < hi; ++i) {
        const uint32_t n = tab[(uint32_t)s_key[i]].y;
        s_dst[i] = sum;
        sum += (i == nt - 1 && (a.T % QAQ_TILE) != 0 && (int)(uint32_t)s_key[i] == a.T / QAQ_TILE) ? n : (n + 15u) & ~15u;
    }
    uint32_t inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if ((tid & 31) >= d) inc += o;
    }
    if ((tid & 31) == 31) s_sum[tid >> 5] = inc;
    __syncthreads();
    uint32_t before = inc - sum;
    for (int w = 0; w < tid >> 5; ++w) before += s_sum[w];
    for (int i = lo; i < hi; ++i) s_dst[i] += before;
    if (tid == COMPACT_THREADS - 1) s_dst[nt] = before + sum;
    __syncthreads();
    // the bytes
    uint8_t* pool = ts.codes + (size_t)bh * a.pool_bytes;
    const uint32_t end = s_dst[nt];
    int first = 0;                                 // tiles before this one are where they belong
    while (first < nt && (uint32_t)(s_key[first] >> 32) == s_dst[first]) ++first;
    int l = first;                                 // the last tile whose new offset is at most that of the thread's piece: moves on with it
    if (first < nt)
        for (uint32_t base = s_dst[first]; base < end; base += COMPACT_THREADS * COMPACT_REGS * 16) {
            uint4 v[COMPACT_REGS];
#pragma unroll
            for (int r = 0; r < COMPACT_REGS; ++r) {
                const uint32_t o = base + (uint32_t)(r * COMPACT_THREADS + tid) * 16;
                if (o >= end) continue;
                while (s_dst[l + 1] <= o) ++l;     // (o < end = s_dst[nt])
                v[r] = *reinterpret_cast<const uint4*>(pool + (uint32_t)(s_key[l] >> 32) + (o - s_dst[l]));
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < COMPACT_REGS; ++r) {
                const uint32_t o = base + (uint32_t)(r * COMPACT_THREADS + tid) * 16;
                if (o < end) *reinterpret_cast<uint4*>(pool + o) = v[r];
            }
            __syncthreads();
        }
    for (int i = tid; i < nt; i += COMPACT_THREADS) tab[(uint32_t)s_key[i]].x = s_dst[i];
    if (tid == 0) ts.pool_end[bh] = end;
}

// (a pool end can stand beyond the pool's capacity when takers that found no room could not give their space back)
__global__ void pool_use_kernel(TensorStore tk, TensorStore tv, int BH, unsigned int cap, unsigned int* out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < BH; i += gridDim.x * blockDim.x) {
        atomicMax(&out[0], min(tk.pool_end[i], cap));
        atomicMax(&out[1], min(tv.pool_end[i], cap));
    }
}

}  // namespace

extern "C" qaq_status qaq_cache_compact(qaq_cache* c, void* stream) {
    if (!c) return QAQ_ERR_INVALID_ARG;
    if (c->tokens == 0) return QAQ_OK;
    const long nt = (c->tokens + QAQ_TILE - 1) / QAQ_TILE;
    if (nt > COMPACT_MAX_TILES) return QAQ_ERR_UNSUPPORTED_SHAPE;
    CompactArgs a;
    a.t[0] = c->t[0]; a.t[1] = c->t[1]; a.pool_bytes = c->pool_bytes; a.ntiles = c->ntiles; a.T = (int)c->tokens;
    a.n2 = 1;
    while (a.n2 < nt) a.n2 <<= 1;
    // 512 threads while all pools are worked on at once (two to an SM), else 256 (256 (b,h) of 4096 tokens, one tile moved: 21.5
    // us with 512, 14.3 with 256, all tiles moved 50 and 44)
    auto launch = [&](auto kernel, int threads, SmemSeen& seen) {
        auto smem_for = [](int n2) { return (size_t)n2 * 8 + (size_t)(n2 + 1) * 4 + 16 * 4; };
        QAQ_CUDA_TRY(qaq_allow_smem((const void*)kernel, smem_for(COMPACT_MAX_TILES), seen));
        QAQ_CUDA_TRY(qaq_launch(kernel, dim3((unsigned)c->BH, 2), dim3((unsigned)threads), smem_for(a.n2), (cudaStream_t)stream, a));
        return QAQ_OK;
    };
    static SmemSeen seen[2];
    return 2 * c->BH <= 2 * 148 ? launch(compact_kernel<512>, 512, seen[0]) : launch(compact_kernel<256>, 256, seen[1]);
}

extern "C" qaq_status qaq_cache_pool_use(const qaq_cache* c, long* host_used, long* host_capacity, void* stream) {
    if (!c || !host_used) return QAQ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    unsigned int* d = qaq_d_pool_use(c);
    QAQ_CUDA_TRY(cudaMemsetAsync(d, 0, 8, s));
    pool_use_kernel<<<32, 256, 0, s>>>(c->t[0], c->t[1], c->BH, (unsigned)c->pool_bytes, d);
    QAQ_CUDA_TRY(cudaGetLastError());
    unsigned int h[2] = {0, 0};
    QAQ_CUDA_TRY(cudaMemcpyAsync(h, d, 8, cudaMemcpyDeviceToHost, s));
    QAQ_CUDA_TRY(cudaStreamSynchronize(s));
    host_used[0] = (long)h[0]; host_used[1] = (long)h[1];
    if (host_capacity) *host_capacity = (long)c->pool_bytes;
    return QAQ_OK;
}
