// S2a: exact outlier thresholds (order statistics) per (b,h) and tensor, in one read of the data.
//
// Wanted: lo = k-th smallest and hi = k-th largest of the N non-NaN values, k = floor(alpha*N/2).
// Only the two tails matter, so the bulk of the data is never histogrammed:
//   1. thr_sample_kernel   a few tokens spread over the sequence give a bracket per tail: a value
//                          below (above) which somewhat more than the wanted tail mass lies.
//   2. thr_scan_kernel     the one pass over all values: entries beyond the brackets ("candidates",
//                          a few per cent) are compacted into per-problem lists (shared-memory lists
//                          per CTA, one global reservation per CTA; what a CTA's list does not hold goes to
//                          the problem's directly), NaNs are counted.
//   3. thr_select_kernel   exact radix select of rank k inside the candidate lists.  If a bracket
//                          turned out too tight (fewer than k+1 candidates) or a problem's list overflowed, the
//                          problem is redone exactly by a two-pass radix select over its data, so the
//                          result is always the exact order statistic.
// Short sequences take one kernel (thr_short_kernel; a tile or less of many (b,h) the first one above, whose sample is then everything).
// binary16 patterns are mapped to 16-bit keys that sort like the values.
#include "qaq_internal.cuh"

namespace {

constexpr int SAMPLE_TOKENS = 64;
constexpr int SCAN_TOKENS_MAX = 1024; // tokens per CTA of the scan (fewer where alpha is large: see scan_tokens_for)
constexpr int WARP_FLAGS = 192;      // 16-byte pieces a warp of the scan can set aside before it has to look at them
constexpr int CTA_LIST = 8192;       // candidates a scan CTA can hold (see scan_tokens_for)
constexpr int SELECT_KEYS = 16384;   // candidates the select kernel keeps in shared memory

__device__ __forceinline__ uint32_t key_of(unsigned short h) { return (h & 0x8000u) ? (uint32_t)(~h & 0xFFFFu) : (uint32_t)(h | 0x8000u); }
__device__ __forceinline__ unsigned short half_of_key(uint32_t k) { return (k & 0x8000u) ? (unsigned short)(k & 0x7FFFu) : (unsigned short)(~k & 0xFFFFu); }
__device__ __forceinline__ __half2 h2_of(uint32_t x) { return *reinterpret_cast<__half2*>(&x); }
__device__ __forceinline__ float float_of_key(uint32_t k) { return __half2float(__ushort_as_half(half_of_key(k))); }

struct Problem {          // per (b,h,tensor), in the workspace
    uint32_t klo, khi;    // bracket keys: candidates are keys < klo and keys > khi
    uint32_t cnt[2];      // candidates found below and above (their sum may exceed the capacity: then the list is incomplete)
    uint32_t nan;         // NaN entries seen by the scan
    uint32_t n;           // places taken in the list
    uint32_t pad[2];
};

struct ThrArgs {
    const __half* X[2];
    long sb, sh, st;
    int H, T, D;
    double alpha;
    Problem* prob;        // [BH*2]
    unsigned short* list; // [BH*2][cap]: candidates of both tails in any order (every lower one is below every upper one)
    uint32_t cap;
    int scan_tokens;      // tokens per CTA of the scan
    float* thr;           // [BH][4]
};

// Rank select over n 16-bit keys, eight at a time (load(i): the i-th eight), for two 0-based ranks at once; all THREADS of the
// CTA call it; hist: 2048 words of shared memory, s_tmp: 4.  Two passes of a radix select: the upper 11 bits of the key
// first, then the lower 5.  binary16 data piles up in a few exponents, so a histogram of the upper byte alone would send most
// lanes of a warp to the same handful of counters; 11 bits spread them over 32 bins per octave.  In the first pass every
// thread sums its bins and a CTA-wide prefix sum finds the bins holding the wanted ranks; in the second each rank has 32 bins,
// one per lane of a warp.
// NaNs sort below -inf (sign set) or above +inf.  SKIP_NAN: they do not count (the data itself); else a caller whose ranks are meant among
// the non-NaN values adds the number of negative NaNs.  AHEAD pieces of a thread are on their way at once.
constexpr uint32_t KEY_MINUS_INF = 0x03FF, KEY_PLUS_INF = 0xFC00;
template <int THREADS, bool SKIP_NAN, int AHEAD, typename Load>
__device__ void cta_select(Load load, uint32_t n, uint32_t wantA, uint32_t wantB, uint32_t* hist, uint32_t* s_tmp, uint32_t& outA, uint32_t& outB) {
    constexpr int BINS = 2048 / THREADS;                     // of a thread
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t n8 = (n + 7) / 8;
    auto for_keys = [&](auto each) {
        for (uint32_t i = threadIdx.x; i < n8; i += AHEAD * THREADS) {
            uint4 r[AHEAD];
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) r[u] = load(AHEAD > 1 ? min(i + u * THREADS, n8 - 1) : i);
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                const uint32_t w[4] = {r[u].x, r[u].y, r[u].z, r[u].w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t k = (w[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
                    if (8 * (i + u * THREADS) + j < n && (!SKIP_NAN || (k >= KEY_MINUS_INF && k <= KEY_PLUS_INF))) each(k);
                }
            }
        }
    };
    for (int i = threadIdx.x; i < 2048; i += blockDim.x) hist[i] = 0;
    if (threadIdx.x < 4) s_tmp[threadIdx.x] = 0;
    __syncthreads();
    for_keys([&](uint32_t k) { atomicAdd(&hist[k >> 5], 1u); });
    __syncthreads();
    uint32_t c[BINS], tot = 0;
#pragma unroll
    for (int j = 0; j < BINS; ++j) { c[j] = hist[BINS * threadIdx.x + j]; tot += c[j]; }
    uint32_t inc = tot;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += t;
    }
    __syncthreads();
    if (lane == 31) hist[warp] = inc;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        const uint32_t v = hist[w];
        if (w < warp) before += v;
        all += v;
    }
    const uint32_t first = before + inc - tot;               // keys in the bins before this thread's
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const uint32_t want = r ? wantB : wantA;
        const uint32_t w2 = want < all ? want : (all ? all - 1 : 0);
        if (tot > 0 && w2 >= first && w2 < first + tot) {    // exactly one thread per rank
            uint32_t acc = first;
            int bsel = 0;
#pragma unroll
            for (int j = 0; j < BINS; ++j) {
                if (w2 >= acc + c[j] && j < BINS - 1) { acc += c[j]; bsel = j + 1; }
                else break;
            }
            s_tmp[2 * r] = (uint32_t)(BINS * threadIdx.x + bsel);
            s_tmp[2 * r + 1] = w2 - acc;
        }
    }
    __syncthreads();
    const uint32_t prefA = s_tmp[0], want1A = s_tmp[1], prefB = s_tmp[2], want1B = s_tmp[3];
    if (threadIdx.x < 64) hist[threadIdx.x] = 0;
    __syncthreads();
    for_keys([&](uint32_t k) {
        if ((k >> 5) == prefA) atomicAdd(&hist[k & 31], 1u);
        if ((k >> 5) == prefB) atomicAdd(&hist[32 + (k & 31)], 1u);
    });
    __syncthreads();
    if (warp < 2) {                                          // warp 0: rank A, warp 1: rank B
        const uint32_t v = hist[32 * warp + lane];
        uint32_t in2 = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, in2, d);
            if (lane >= d) in2 += t;
        }
        const uint32_t all2 = __shfl_sync(0xFFFFFFFFu, in2, 31);
        const uint32_t want1 = warp ? want1B : want1A;
        const uint32_t w3 = want1 < all2 ? want1 : (all2 ? all2 - 1 : 0);
        if (all2 == 0 && lane == 0) s_tmp[2 * warp] = 0;
        if (v > 0 && w3 >= in2 - v && w3 < in2) s_tmp[2 * warp] = (uint32_t)lane;
    }
    __syncthreads();
    outA = (prefA << 5) | s_tmp[0];
    outB = (prefB << 5) | s_tmp[2];
    __syncthreads();
}

// keys that sit in shared memory (AHEAD 1) or global memory (16-byte aligned)
template <int THREADS, int AHEAD = 1>
__device__ __forceinline__ void cta_select_keys(const unsigned short* keys, uint32_t n, uint32_t wantA, uint32_t wantB, uint32_t* hist, uint32_t* s_tmp, uint32_t& outA, uint32_t& outB) {
    cta_select<THREADS, false, AHEAD>([&](uint32_t i) { return reinterpret_cast<const uint4*>(keys)[i]; }, n, wantA, wantB, hist, s_tmp, outA, outB);
}

__device__ __forceinline__ unsigned long long rank_k(double alpha, unsigned long long N) {
    unsigned long long k = (unsigned long long)floor(alpha * (double)N / 2.0);
    if (N > 0 && k > (N - 1) / 2) k = (N - 1) / 2;
    return k;
}

// binary16 pair -> pair of keys (a set sign flips all 16 bits, a clear one only the sign bit)
__device__ __forceinline__ uint32_t keys_of(uint32_t w) { return w ^ (((w >> 15) & 0x00010001u) * 0xFFFFu | 0x80008000u); }
// the same; NaNs are counted, negative ones once more
__device__ __forceinline__ uint32_t keys_of(uint32_t w, uint32_t& nn, uint32_t& nneg) {
    const uint32_t mag = w & 0x7FFF7FFFu;
    const uint32_t nan_lo = (mag & 0xFFFFu) > 0x7C00u, nan_hi = (mag >> 16) > 0x7C00u;
    nn += nan_lo + nan_hi;
    nneg += (nan_lo & (w >> 15)) + (nan_hi & (w >> 31));
    return keys_of(w);
}
// Rank of 1.25 times the wanted tail mass plus four standard deviations of the count in a sample of M (a wider bracket
// makes the scan set aside more pieces: 2.0 times costs 7 % more time on stationary data; a bracket that
// turns out too tight only sends that problem to the exact two-pass select).
__device__ __forceinline__ uint32_t bracket_rank(double alpha, uint32_t M) {
    const double f2 = 1.25 * 0.5 * alpha * (double)M;
    const uint32_t r = (uint32_t)ceil(f2 + 4.0 * sqrt(f2 + 1.0) + 2.0);
    return r > (M - 1) / 2 ? (M - 1) / 2 : r;
}

// ---- 1. sample: brackets.  WHOLE: up to SAMPLE_TOKENS tokens, which are all looked at: the answer.
template <int THREADS, bool WHOLE>
__global__ void __launch_bounds__(THREADS) thr_sample_kernel(const ThrArgs a) {
    constexpr int PIECES = SAMPLE_TOKENS * 128 / 8 / THREADS;            // 16-byte pieces of a thread at most
    qaq_dependency();
    const int bhx = blockIdx.x, bh = bhx >> 1, x = bhx & 1;
    __shared__ __align__(16) unsigned short s_keys[SAMPLE_TOKENS * 128];
    __shared__ uint32_t hist[2048], s_tmp[4], s_cnt[2];
    const int b_idx = bh / a.H, h_idx = bh % a.H;
    const __half* X = a.X[x] + (size_t)b_idx * a.sb + (size_t)h_idx * a.sh;
    const int ns = WHOLE ? a.T : SAMPLE_TOKENS;
    const int M = ns * a.D;
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    uint32_t nn = 0, nneg = 0;                                  // NaNs, NaNs with the sign set
    // all 16-byte pieces of a thread are on their way before the first is looked at
    uint4 raw[PIECES];
#pragma unroll
    for (int k = 0; k < PIECES; ++k) {
        const int i = min((int)threadIdx.x + THREADS * k, M / 8 - 1);
        const int sp = (i * 8) / a.D, c = (i * 8) % a.D;
        const long t = (long)sp * a.T / ns;                       // tokens spread over the sequence
        raw[k] = *reinterpret_cast<const uint4*>(X + (size_t)t * a.st + c);
    }
#pragma unroll
    for (int k = 0; k < PIECES; ++k) {
        const int i = threadIdx.x + THREADS * k;
        if (i >= M / 8) break;
        uint32_t w[4] = {raw[k].x, raw[k].y, raw[k].z, raw[k].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = keys_of(w[j], nn, nneg);
        *reinterpret_cast<uint4*>(&s_keys[8 * i]) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (nn) { atomicAdd(&s_cnt[0], nn); atomicAdd(&s_cnt[1], nneg); }
    __syncthreads();
    const uint32_t Mv = (uint32_t)M - s_cnt[0];                    // non-NaN sample values
    const uint32_t n_neg_nan = s_cnt[1];
    Problem* pr = a.prob + bhx;
    float* const thr = a.thr + (size_t)bh * 4 + 2 * x;
    if (Mv == 0) {
        if (WHOLE) { if (threadIdx.x < 2) thr[threadIdx.x] = 0.f; }
        else if (threadIdx.x == 0) { pr->klo = 0; pr->khi = 0xFFFF; pr->cnt[0] = pr->cnt[1] = 0; pr->nan = 0; pr->n = 0; }
        return;
    }
    const uint32_t r = WHOLE ? (uint32_t)rank_k(a.alpha, Mv) : bracket_rank(a.alpha, Mv);
    uint32_t klo, khi;
    cta_select_keys<THREADS>(s_keys, (uint32_t)M, r + n_neg_nan, Mv - 1 - r + n_neg_nan, hist, s_tmp, klo, khi);
    if (WHOLE) { if (threadIdx.x < 2) thr[threadIdx.x] = float_of_key(threadIdx.x ? khi : klo); }
    else if (threadIdx.x == 0) { pr->klo = klo; pr->khi = khi; pr->cnt[0] = pr->cnt[1] = 0; pr->nan = 0; pr->n = 0; }
}

// ---- 2. the one pass over the data: compaction of the tail candidates.
// Almost all entries are inside [lo, hi], so the pass is a cheap filter first: a 16-byte piece whose smallest entry is
// at least lo and whose largest is at most hi (NaN-propagating min / max, so a NaN fails both) is dropped; the others
// (about one in ten at alpha = 1 %) are set aside in a buffer of the warp's own, and when enough of them have come
// together the warp looks at them entry by entry with all lanes busy.  Nothing in the loop needs the other warps:
// no CTA barrier, one shared-memory reservation per warp and batch of set-aside pieces; the candidates of both tails share a
// list, which the select takes apart by rank.
// What bounds it: memory where outliers are few (256 (b,h) of 4096 tokens, alpha = 1 %: 105 us, 5.1 TB/s; 124 us without
// the next pieces on their way while four are looked at, and with 512 tokens per CTA), the extraction where they are many
// (160 (b,h) of 8192 tokens, 5 %: 204 us; 215 with a loop over the candidates of a piece).  60 registers, four
// CTAs per SM: held to five it takes 114 us, to six 169.
__global__ void __launch_bounds__(256) thr_scan_kernel(const ThrArgs a) {
    qaq_dependency();
    const int bhx = blockIdx.y, bh = bhx >> 1, x = bhx & 1;
    Problem* pr = a.prob + bhx;
    __shared__ unsigned short s_list[CTA_LIST];
    __shared__ uint4 s_flag[8][WARP_FLAGS];                   // per warp: pieces with something outside [lo, hi]
    __shared__ uint32_t s_n, s_low, s_base, s_nan;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    if (threadIdx.x == 0) { s_n = 0; s_low = 0; s_nan = 0; }
    __syncthreads();
    const uint32_t klo = pr->klo;
    const float flo = float_of_key(klo), fhi = float_of_key(pr->khi);
    const __half2 lo2 = __float2half2_rn(flo), hi2 = __float2half2_rn(fhi);   // exact: both are binary16 values
    const int b_idx = bh / a.H, h_idx = bh % a.H;
    const int t0 = blockIdx.x * a.scan_tokens, ntok = min(a.T, t0 + a.scan_tokens) - t0;
    const int tok_shift = 31 - __clz(a.D / 8);                   // 16-byte pieces per token is a power of two (4, 8, 16)
    // thread tid looks at piece (tid mod pieces per token) of tokens tid >> tok_shift, + 256 >> tok_shift, ...
    int tok = (int)threadIdx.x >> tok_shift;
    const int tok_step = 256 >> tok_shift;
    const __half* ptr = (x ? a.X[1] : a.X[0]) + (size_t)b_idx * a.sb + (size_t)h_idx * a.sh + (size_t)(t0 + tok) * a.st +
                        (((int)threadIdx.x & ((1 << tok_shift) - 1)) << 3);
    const size_t ptr_step = (size_t)tok_step * a.st;
    unsigned short* const dst = a.list + (size_t)bhx * a.cap;
    uint4* wflag = s_flag[warp];
    uint32_t nflag = 0;      // pieces set aside by this warp (the same in all its lanes)
    uint32_t nnan = 0, nlow = 0;

    // four independent 16-byte loads per thread, the next four on their way while these are looked at
    uint4 next[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        next[u] = make_uint4(0, 0, 0, 0);
        if (tok + u * tok_step < ntok) next[u] = *reinterpret_cast<const uint4*>(ptr + u * ptr_step);
    }
    for (int c0 = 0; c0 < ntok; c0 += 4 * tok_step) {
        uint4 raw[4];
        bool in_range[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { in_range[u] = tok + u * tok_step < ntok; raw[u] = next[u]; }
        tok += 4 * tok_step;
        ptr += 4 * ptr_step;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (tok + u * tok_step < ntok) next[u] = *reinterpret_cast<const uint4*>(ptr + u * ptr_step);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const __half2 v0 = h2_of(raw[u].x), v1 = h2_of(raw[u].y), v2 = h2_of(raw[u].z), v3 = h2_of(raw[u].w);
            const __half2 mn = __hmin2_nan(__hmin2_nan(v0, v1), __hmin2_nan(v2, v3));
            const __half2 mx = __hmax2_nan(__hmax2_nan(v0, v1), __hmax2_nan(v2, v3));
            const bool flag = in_range[u] && !(__hbge2(mn, lo2) && __hble2(mx, hi2));
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, flag);
            if (flag) wflag[nflag + __popc(bal & lt)] = raw[u];
            nflag += (uint32_t)__popc(bal);
        }
        __syncwarp();
        // the next round may set aside 128 more; the last round empties the buffer
        const bool last_round = c0 + 4 * tok_step >= ntok;
        if (!(nflag > (uint32_t)(WARP_FLAGS - 128) || last_round)) continue;
        // whole batches of 32 only (every lane busy); what is left over stays in the buffer for the next time,
        // except in the last round
        const uint32_t ntake = last_round ? nflag : (nflag & ~31u);
        // the warp's set-aside pieces entry by entry: per lane the entries below lo, above hi and NaN; one reservation
        // per tail for the whole batch, then every lane writes its keys
        for (uint32_t i0 = 0; i0 < ntake; i0 += 32) {
            const bool have = i0 + lane < ntake;
            const uint4 r = have ? wflag[i0 + lane] : make_uint4(0, 0, 0, 0);
            const uint32_t w[4] = {r.x, r.y, r.z, r.w};
            uint32_t m = 0, numbers = 0;                          // bit j / 16 + j: low / high half of word j
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __half2 v = h2_of(w[j]);
                m |= (__hlt2_mask(v, lo2) | __hgt2_mask(v, hi2)) & (0x00010001u << j);       // a NaN is neither
                numbers |= __heq2_mask(v, v) & (0x00010001u << j);
            }
            if (!have) m = 0;
            else nnan += 8u - (uint32_t)__popc(numbers);
            const uint32_t mine = (uint32_t)__popc(m);            // at most 8
            uint32_t inc = mine;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                if (lane >= d) inc += t;
            }
            uint32_t b0 = 0, g0 = 0;
            if (lane == 31 && inc) {
                b0 = atomicAdd(&s_n, inc);
                // beyond the CTA's list: entry `pos` goes to place g0 + pos of the problem's
                const uint32_t from = max(b0, (uint32_t)CTA_LIST);
                if (b0 + inc > from) g0 = atomicAdd(&pr->n, b0 + inc - from) - from;
            }
            uint32_t pos = __shfl_sync(0xFFFFFFFFu, b0, 31) + inc - mine;
            if (__all_sync(0xFFFFFFFFu, pos + mine <= (uint32_t)CTA_LIST)) {
                // entry by entry without a loop over the set bits (whose address and selection took more than half of the batch)
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (m & (1u << ((j >> 1) + 16 * (j & 1)))) s_list[pos++] = (unsigned short)(w[j >> 1] >> (16 * (j & 1)));
            } else {
                g0 = __shfl_sync(0xFFFFFFFFu, g0, 31);
                while (m) {
                    const int bit = __ffs(m) - 1;
                    m &= m - 1;
                    const int j = bit & 3;
                    const uint32_t wj = (j & 2) ? ((j & 1) ? w[3] : w[2]) : ((j & 1) ? w[1] : w[0]);
                    const unsigned short h = (unsigned short)((bit >> 4) ? (wj >> 16) : (wj & 0xFFFFu));
                    if (pos < (uint32_t)CTA_LIST) s_list[pos] = h;
                    else {
                        const uint32_t key = key_of(h);
                        if (key < klo) ++nlow;
                        if (g0 + pos < a.cap) dst[g0 + pos] = (unsigned short)key;
                    }
                    ++pos;
                }
                __syncwarp();
            }
        }
        const uint32_t left = nflag - ntake;           // fewer than 32
        uint4 keep = make_uint4(0, 0, 0, 0);
        if ((uint32_t)lane < left) keep = wflag[ntake + lane];
        __syncwarp();
        if ((uint32_t)lane < left) wflag[lane] = keep;
        nflag = left;
        __syncwarp();     // the rest of the buffer is free again
    }
    nnan = __reduce_add_sync(0xFFFFFFFFu, nnan);
    if (lane == 0 && nnan) atomicAdd(&s_nan, nnan);
    __syncthreads();
    const uint32_t cnt = min(s_n, (uint32_t)CTA_LIST);
    if (threadIdx.x == 0) s_base = cnt ? atomicAdd(&pr->n, cnt) : 0u;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < cnt; i += blockDim.x) {
        const uint32_t pos = s_base + i, key = key_of(s_list[i]);
        if (key < klo) ++nlow;
        if (pos < a.cap) dst[pos] = (unsigned short)key;
    }
    nlow = __reduce_add_sync(0xFFFFFFFFu, nlow);
    if (lane == 0 && nlow) atomicAdd(&s_low, nlow);
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t low = s_low;
        if (low) atomicAdd(&pr->cnt[0], low);
        if (s_n > low) atomicAdd(&pr->cnt[1], s_n - low);
        if (s_nan) atomicAdd(&pr->nan, s_nan);
    }
}

// ---- 3. exact select among the candidates, exact fallback over the data when that is not possible.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) thr_select_kernel(const ThrArgs a) {
    qaq_dependency();
    const int bhx = blockIdx.x, bh = bhx >> 1, x = bhx & 1;
    Problem* pr = a.prob + bhx;
    __shared__ uint32_t hist[2048], s_tmp[4];
    __shared__ __align__(16) unsigned short s_keys[SELECT_KEYS];
    const unsigned long long total = (unsigned long long)a.T * a.D;
    const unsigned long long N = total - pr->nan;
    float res[2] = {0.f, 0.f};
    if (N > 0) {
        const unsigned long long k = rank_k(a.alpha, N);
        const uint32_t c0 = pr->cnt[0], c1 = pr->cnt[1], c = c0 + c1;
        if (c0 > k && c1 > k && c <= a.cap) {
            // rank k from below and rank k from above
            const unsigned short* l = a.list + (size_t)bhx * a.cap;                // 16-byte aligned
            uint32_t lo, hi;
            if (c <= (uint32_t)SELECT_KEYS) {
                // the usual case: the list fits in shared memory; bring it in with independent wide loads
                for (uint32_t i = threadIdx.x; i < (c + 7) / 8; i += THREADS)
                    reinterpret_cast<uint4*>(s_keys)[i] = reinterpret_cast<const uint4*>(l)[i];
                __syncthreads();
                cta_select_keys<THREADS>(s_keys, c, (uint32_t)k, (uint32_t)(c - 1 - k), hist, s_tmp, lo, hi);
            } else {
                // a longer list is read twice where it lies, four times eight keys at a time (160 (b,h) of 8192 tokens at 5 %, the whole
                // search: eight 261 us, four times eight 258; one at a time the select alone took 124)
                cta_select_keys<THREADS, 4>(l, c, (uint32_t)k, (uint32_t)(c - 1 - k), hist, s_tmp, lo, hi);
            }
            res[0] = float_of_key(lo); res[1] = float_of_key(hi);
        } else {
            // bracket too tight or list overflow: two-pass radix select over this problem's data, for both ranks at once, eight
            // entries at a time (each rank for itself, entry by entry: 32 (b,h) of 4096 tokens 2090 us, this way 268)
            const __half* X = a.X[x] + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh;
            const int shift = 31 - __clz(a.D / 8);                 // 16-byte pieces per token
            auto load = [&](uint32_t i) {
                const uint4 r = *reinterpret_cast<const uint4*>(X + (size_t)(i >> shift) * a.st + ((i & ((1u << shift) - 1)) << 3));
                return make_uint4(keys_of(r.x), keys_of(r.y), keys_of(r.z), keys_of(r.w));
            };
            uint32_t lo, hi;
            cta_select<THREADS, true, 4>(load, (uint32_t)total, (uint32_t)k, (uint32_t)(N - 1 - k), hist, s_tmp, lo, hi);
            res[0] = float_of_key(lo); res[1] = float_of_key(hi);
        }
    }
    if (threadIdx.x < 2) a.thr[(size_t)bh * 4 + 2 * x + threadIdx.x] = threadIdx.x ? res[1] : res[0];
}

// ---- short sequences: one launch, a CTA per problem, its keys in registers.
// A key among the k + 1 smallest is not above the (k + 1)-th smallest of the pieces' minima (a piece: eight keys), so the minima
// and the maxima give a bin of 32 keys for either tail; the keys up to the one and from the other on are counted by bins, which
// gives the bin of each rank, and a second count, of the keys inside these two bins, the keys themselves.  Nothing is guessed, there
// is no other path to fall back to.  What bounds it: one step after the other, by 16 warps.  32 (b,h) of 100 tokens 13.2 us with a sample,
// brackets from it and lists of candidates, 7.8 with every key tested against the bins in both counts, 6.0 with a mask of what lies in
// them; 256 of 100 tokens 22.5, 21.4, 16.0; 64 of 400, head_dim 64, 15.5, 10.9, 7.3.  (The keys of a problem spread over a thread-block
// cluster, whose counts meet in distributed shared memory: 32 (b,h) of 1000 tokens 25 to 36 us, the three kernels above 19.)
constexpr int SHORT_THREADS = 512;
template <int PIECES>                                                            // of a thread
__global__ void __launch_bounds__(SHORT_THREADS, PIECES > 8 ? 1 : 2) thr_short_kernel(const ThrArgs a) {
    constexpr int THREADS = SHORT_THREADS;
    static_assert(PIECES <= 16, "eight bits for each");
    constexpr int PER = 2048 / THREADS;                                          // bins of a thread
    __shared__ uint32_t s_lo[2048], s_hi[2048];                                  // counts by the upper 11 bits of the key: minima, maxima; then s_lo: keys
    __shared__ uint32_t s_fine[64], s_nan, s_part[2][32], s_found[4];            // counts by the lower 5 bits; NaNs
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, bhx = blockIdx.x, bh = bhx >> 1, x = bhx & 1;
    for (int i = tid; i < 2048; i += THREADS) { s_lo[i] = 0; s_hi[i] = 0; }
    if (tid < 64) s_fine[tid] = 0;
    if (tid == 0) { s_nan = 0; s_found[0] = 2047; s_found[2] = 0; }              // (fewer pieces than the rank: all keys are counted)
    __syncthreads();
    qaq_dependency();
    const int shift = 31 - __clz(a.D / 8);                                       // pieces of a token
    const uint32_t total = (uint32_t)a.T * (uint32_t)a.D, n8 = total / 8;
    const __half* X = (x ? a.X[1] : a.X[0]) + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh;
    uint4 raw[PIECES];
#pragma unroll
    for (int u = 0; u < PIECES; ++u) {
        const uint32_t i = tid + THREADS * u;
        raw[u] = make_uint4(0x7FFF7FFFu, 0x7FFF7FFFu, 0x7FFF7FFFu, 0x7FFF7FFFu);            // not numbers where there is no piece
        if (i < n8) raw[u] = *reinterpret_cast<const uint4*>(X + (size_t)(i >> shift) * a.st + ((i & ((1u << shift) - 1)) << 3));
    }
    uint32_t nan = 0;
#pragma unroll
    for (int u = 0; u < PIECES; ++u) {
        if (THREADS * u >= n8) break;
        const __half2 v0 = h2_of(raw[u].x), v1 = h2_of(raw[u].y), v2 = h2_of(raw[u].z), v3 = h2_of(raw[u].w);
        const __half2 mn = __hmin2(__hmin2(v0, v1), __hmin2(v2, v3)), mx = __hmax2(__hmax2(v0, v1), __hmax2(v2, v3));
        const __half m = __hmin(__low2half(mn), __high2half(mn)), M = __hmax(__low2half(mx), __high2half(mx));
        if (m == m) {                                                            // (a piece without a number counts as none)
            atomicAdd(&s_lo[key_of(__half_as_ushort(m)) >> 5], 1u);
            atomicAdd(&s_hi[key_of(__half_as_ushort(M)) >> 5], 1u);
        }
        const __half2 sum = __hmin2_nan(__hmin2_nan(v0, v1), __hmin2_nan(v2, v3));
        if (!__hbeq2(sum, sum) && tid + THREADS * u < n8) {                      // a NaN among them
            uint32_t neg = 0;
            (void)keys_of(raw[u].x, nan, neg); (void)keys_of(raw[u].y, nan, neg); (void)keys_of(raw[u].z, nan, neg); (void)keys_of(raw[u].w, nan, neg);
        }
    }
    nan = __reduce_add_sync(0xFFFFFFFFu, nan);
    if (lane == 0 && nan) atomicAdd(&s_nan, nan);
    __syncthreads();
    // the bins of two 0-based ranks, each among counts of its own, PER to a thread
    auto bins_of = [&](const uint32_t* countsA, const uint32_t* countsB, auto rankA, auto rankB) {
        uint32_t cA[PER], cB[PER], totA = 0, totB = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) { cA[j] = countsA[PER * tid + j]; cB[j] = countsB[PER * tid + j]; totA += cA[j]; totB += cB[j]; }
        uint32_t incA = totA, incB = totB;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t oA = __shfl_up_sync(0xFFFFFFFFu, incA, d), oB = __shfl_up_sync(0xFFFFFFFFu, incB, d);
            if (lane >= d) { incA += oA; incB += oB; }
        }
        if (lane == 31) { s_part[0][warp] = incA; s_part[1][warp] = incB; }
        __syncthreads();
        uint32_t beforeA = 0, beforeB = 0, allA = 0, allB = 0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) {
            const uint32_t pA = s_part[0][w], pB = s_part[1][w];
            if (w < warp) { beforeA += pA; beforeB += pB; }
            allA += pA; allB += pB;
        }
        auto place = [&](const uint32_t (&c)[PER], uint32_t at, uint32_t tot, uint32_t want, uint32_t* found) {
            if (tot == 0 || want < at || want >= at + tot) return;               // one thread, or none where the rank does not exist
            int j = 0;
#pragma unroll
            for (; j < PER - 1; ++j) { if (want < at + c[j]) break; at += c[j]; }
            found[0] = (uint32_t)(PER * tid + j); found[1] = want - at;
        };
        place(cA, beforeA + incA - totA, totA, rankA(allA), &s_found[0]);
        place(cB, beforeB + incB - totB, totB, rankB(allB), &s_found[2]);
        __syncthreads();
    };
    const uint32_t most = (uint32_t)rank_k(a.alpha, total);                      // not less than the rank among the numbers
    bins_of(s_lo, s_hi, [&](uint32_t) { return most; }, [&](uint32_t all) { return all > most ? all - 1 - most : 0xFFFFFFFFu; });
    const uint32_t lo = s_found[0], hi = s_found[2];
    for (int i = tid; i < 2048; i += THREADS) s_lo[i] = 0;
    __syncthreads();
    // what lies in these bins or beyond, as values (NaNs compare false; a zero of the other sign may come along, which changes no rank)
    const __half2 lo2 = __half2half2(__ushort_as_half(half_of_key(min((lo << 5) | 31u, KEY_PLUS_INF)))), hi2 = __half2half2(__ushort_as_half(half_of_key(max(hi << 5, KEY_MINUS_INF))));
    uint32_t set[(PIECES + 3) / 4];                                              // eight bits a piece: bit 2j + h is half h of word j
#pragma unroll
    for (int i = 0; i < (PIECES + 3) / 4; ++i) set[i] = 0;
#pragma unroll
    for (int u = 0; u < PIECES; ++u) {
        if (THREADS * u >= n8) break;
        const uint32_t w[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
        uint32_t m = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t out = __hle2_mask(h2_of(w[j]), lo2) | __hge2_mask(h2_of(w[j]), hi2);
            m |= (out & 0x00010001u) << (2 * j);
        }
        set[u >> 2] |= ((m | (m >> 15)) & 0xFFu) << (8 * (u & 3));
    }
    auto for_set = [&](auto each) {
#pragma unroll
        for (int u = 0; u < PIECES; ++u) {
            if (THREADS * u >= n8) break;
            uint32_t m = (set[u >> 2] >> (8 * (u & 3))) & 0xFFu;
            while (m) {
                const int bit = __ffs(m) - 1;
                m &= m - 1;
                const uint32_t a01 = (bit & 2) ? raw[u].y : raw[u].x, a23 = (bit & 2) ? raw[u].w : raw[u].z, w = (bit & 4) ? a23 : a01;
                each(key_of((unsigned short)((bit & 1) ? w >> 16 : w & 0xFFFFu)));
            }
        }
    };
    for_set([&](uint32_t k) { atomicAdd(&s_lo[k >> 5], 1u); });
    __syncthreads();
    const uint32_t N = total - s_nan, k = (uint32_t)rank_k(a.alpha, N);
    bins_of(s_lo, s_lo, [&](uint32_t) { return k; }, [&](uint32_t all) { return all > k ? all - 1 - k : 0xFFFFFFFFu; });
    const uint32_t binA = s_found[0], binB = s_found[2];
    for_set([&](uint32_t key) {
        if ((key >> 5) == binA) atomicAdd(&s_fine[key & 31], 1u);
        if ((key >> 5) == binB) atomicAdd(&s_fine[32 + (key & 31)], 1u);
    });
    __syncthreads();
    if (warp < 2) {                                                              // warp 0: rank k, warp 1: rank N - 1 - k
        const uint32_t v = s_fine[32 * warp + lane], want = s_found[2 * warp + 1];
        uint32_t inc = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += t;
        }
        float* out = a.thr + (size_t)bh * 4 + 2 * x + warp;
        if (N == 0) { if (lane == 0) *out = 0.f; }
        else if (v > 0 && want >= inc - v && want < inc) *out = float_of_key((s_found[2 * warp] << 5) | (uint32_t)lane);
    }
}

// Tokens per CTA of the scan: as many as keep the expected number of candidates (1.25 times the tail mass
// plus the bracket's slack, of both tails) inside the CTA's list.  Where tails are not spread evenly over the sequence a CTA
// finds more; those go to the problem's list batch by batch (a tail in the first quarter of 256 (b,h) x 4096 tokens: 151 us,
// 132 where it is spread evenly; as an overflow that sends the problem to the exact select over its data it took 4390).
// Fewer too while the launch does not fill the chip: a thread's loads then come one round after the other for nothing
// (32 (b,h) of 333 tokens: one CTA for each and tensor 8.5 us, six 4.9).
int scan_tokens_for(double alpha, int D, int BH, int T) {
    const double per_token = 2.0 * (0.625 * alpha + 0.004) * D;
    int tokens = SCAN_TOKENS_MAX;
    while (tokens > 64 && per_token * tokens > 0.6 * CTA_LIST) tokens /= 2;
    while (tokens > 64 && (long long)BH * 2 * ((T + tokens - 1) / tokens) < 4 * 148) tokens /= 2;
    return tokens;
}

uint32_t list_capacity(const qaq_config* cfg, int n_tokens) {
    // expected candidates per tail: (alpha + margin) * N; keep three times that, at least 4096
    const double N = (double)n_tokens * cfg->head_dim;
    double want = 3.0 * (cfg->outlier_frac * N + 8.0 * sqrt(cfg->outlier_frac * N + 64.0) + 64.0) + 4096.0;
    if (want > N) want = N;
    uint32_t cap = (uint32_t)want;
    return (cap + 63u) & ~63u;
}

}  // namespace

extern "C" qaq_status qaq_thresholds_workspace_bytes(const qaq_config* cfg, size_t* host_out) {
    if (!cfg || !host_out || cfg->batch < 1 || cfg->heads < 1 || cfg->max_tokens < 1) return QAQ_ERR_INVALID_ARG;
    const size_t P = (size_t)cfg->batch * cfg->heads * 2;
    *host_out = P * sizeof(Problem) + P * 2 * (size_t)list_capacity(cfg, cfg->max_tokens) * sizeof(unsigned short) + 256;
    return QAQ_OK;
}

extern "C" qaq_status qaq_outlier_thresholds(const qaq_config* cfg, const void* K, const void* V, long stride_b,
                                             long stride_h, long stride_t, int n_tokens, float* thr, void* ws,
                                             size_t ws_bytes, void* stream) {
    if (!cfg || !K || !V || !thr || !ws || n_tokens < 1) return QAQ_ERR_INVALID_ARG;
    if (!qaq_dim_ok(cfg->head_dim)) return QAQ_ERR_UNSUPPORTED_SHAPE;
    if (!(cfg->outlier_frac >= 0.0 && cfg->outlier_frac <= 1.0)) return QAQ_ERR_INVALID_ARG;
    if ((double)n_tokens * cfg->head_dim >= 4.0e9) return QAQ_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)K & 15) || ((uintptr_t)V & 15) || (stride_b & 7) || (stride_h & 7) || (stride_t & 7) ||
        stride_t < cfg->head_dim)
        return QAQ_ERR_INVALID_ARG;
    size_t need = 0;
    qaq_thresholds_workspace_bytes(cfg, &need);
    if (ws_bytes < need || ((uintptr_t)ws & 15)) return QAQ_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    const int BH = cfg->batch * cfg->heads;
    ThrArgs a;
    a.X[0] = (const __half*)K; a.X[1] = (const __half*)V;
    a.sb = stride_b; a.sh = stride_h; a.st = stride_t;
    a.H = cfg->heads; a.T = n_tokens; a.D = cfg->head_dim; a.alpha = cfg->outlier_frac;
    a.prob = (Problem*)ws;
    // the candidate lists take whatever the workspace offers beyond the problem records
    const size_t head = ((size_t)BH * 2 * sizeof(Problem) + 255) / 256 * 256;
    const size_t per_list = (ws_bytes - head) / ((size_t)BH * 2 * sizeof(unsigned short));
    a.cap = (uint32_t)(per_list > 0x3FFFFFC0u ? 0x3FFFFFC0u : per_list) & ~63u;
    if (a.cap < 64) return QAQ_ERR_WORKSPACE;
    a.list = (unsigned short*)((char*)ws + head);
    a.thr = thr;
    a.scan_tokens = SCAN_TOKENS_MAX;
    const size_t keys = (size_t)n_tokens * cfg->head_dim;
    // a tile or less of so many (b,h) that the CTAs of 512 threads come in turns (two to an SM): 160 (b,h) of 40 tokens, head_dim 32, 6.4 us,
    // 9.0 by the kernel for short sequences, 320 of them 8.5 and 13.7 (head_dim 128: 13.0 and 16.1); 148 6.4 and 6.5
    if (n_tokens <= SAMPLE_TOKENS && BH * 2 > 2 * 148) {
        QAQ_CUDA_TRY(qaq_launch(thr_sample_kernel<256, true>, dim3(BH * 2), dim3(256), 0, s, a));
        return QAQ_OK;
    }
    // 32768 keys; twice as many while every problem has an SM to itself (32 (b,h) of 333 tokens 10.4 us, 13.4 by the kernels below;
    // 256 of them 38.7 and 31.0), not quite where these would spread few problems over all SMs (one (b,h) of 800 tokens, head_dim 64, 11.3 and
    // 11.5, of 1024 13.0 and 11.7; 12 of 1024 13.0 and 12.9)
    if (keys <= SHORT_THREADS * 8 * 8) {
        QAQ_CUDA_TRY(qaq_launch(thr_short_kernel<8>, dim3(BH * 2), dim3(SHORT_THREADS), 0, s, a));
        return QAQ_OK;
    }
    if (keys <= (size_t)SHORT_THREADS * 8 * (BH < 8 ? 12 : 16) && BH * 2 <= 148) {
        QAQ_CUDA_TRY(qaq_launch(thr_short_kernel<16>, dim3(BH * 2), dim3(SHORT_THREADS), 0, s, a));
        return QAQ_OK;
    }
    // 512 threads while a problem has an SM to itself or shares it with one (32 (b,h): 6.4 against 7.9 us), else 256 (256
    // (b,h): 14.4 against 15.6)
    if (BH * 2 <= 2 * 148) QAQ_CUDA_TRY(qaq_launch(thr_sample_kernel<512, false>, dim3(BH * 2), dim3(512), 0, s, a));
    else QAQ_CUDA_TRY(qaq_launch(thr_sample_kernel<256, false>, dim3(BH * 2), dim3(256), 0, s, a));
    a.scan_tokens = scan_tokens_for(cfg->outlier_frac, cfg->head_dim, BH, n_tokens);
    dim3 grid((n_tokens + a.scan_tokens - 1) / a.scan_tokens, BH * 2);
    QAQ_CUDA_TRY(qaq_launch(thr_scan_kernel, grid, dim3(256), 0, s, a));
    // lists that stay in shared memory are a matter of latency (256 (b,h) of 4096 tokens, alpha = 1 %: 14.6 us with 256
    // threads, 19.1 with 512), longer ones of throughput (160 of 8192 tokens, 5 %: 68.3 and 48.7 us, 46 with four loads ahead)
    if (1.25 * cfg->outlier_frac * (double)keys <= SELECT_KEYS) QAQ_CUDA_TRY(qaq_launch(thr_select_kernel<256>, dim3(BH * 2), dim3(256), 0, s, a));
    else QAQ_CUDA_TRY(qaq_launch(thr_select_kernel<512>, dim3(BH * 2), dim3(512), 0, s, a));
    return QAQ_OK;
}
