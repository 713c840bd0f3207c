// Score window after a prefill (Section 4.2 of the paper, "Attention score prediction": the
// predicted score of a token is the maximum over the scores of the preceding n queries).  Right
// after a prefill of T tokens those are the attention rows of its last n queries on the
// unquantized binary16 keys:
//   row of query i (position T-n+i):  softmax over the tokens t <= T-n+i of  scale * q_i . k_t.
// Rows are written newest first (row r = query n-1-r), so that the rows in which token t exists
// are 0..nvalid[t]-1 with nvalid[t] = min(n, T-t); entries of tokens a query cannot see are 0.
//
// This is the one dense contraction on the path ([n x D] x [D x T] per (b,h)), so the logits run
// on the tensor cores (mma.sync m16n8k16, binary16 in, binary32 accumulate); with n <= 64 rows it is
// bound by reading K once.  Sequences of up to 4096 tokens take one kernel whose CTAs form a
// thread-block cluster per (b,h) (logits stay in shared memory, row statistics travel through
// distributed shared memory, the ring is written once); longer ones take two passes of one kernel: the first
// leaves (max, sum of exponentials) of every row per chunk of tokens, the second computes the logits again
// and writes the rows normalised with the merged statistics.
#include <cooperative_groups.h>

#include "qaq_internal.cuh"

namespace {

constexpr int PW_WARPS = 8;            // three CTAs per SM (80 registers per thread)
constexpr int PW_CHUNK = 512;          // tokens per CTA: 64 per warp, 16 at a time
constexpr int PW_MAXQ = 64;            // rows (queries) at most

struct PrefillArgs {
    const __half* Q;     // [BH][n][D]
    const __half* K;
    long sb, sh, st;
    int H, T, n;
    float scale;
    float* ring;         // [BH][n][T]
    uint8_t* nvalid;     // [BH][T]
    float* qnorm2;       // [BH][n] or null
    float2* part;        // [BH][nchunk][n] (max, sum of exp) of the visible logits of a chunk
    int nchunk;
};

__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The queries as A-operand fragments in shared memory, one uint4 per (16-row tile, k step, lane): every warp reads the
// same ones.  The contraction index is permuted the same way in both operands: lane (., c) of k step ks takes words
// 2 (ks mod 2), + 1 of the 16-byte piece 4 (ks / 2) + c of a row.
template <int D>
__device__ __forceinline__ void lay_out_queries(uint4* s_q, const __half* Qb, int n) {
    constexpr int KS = D / 16;
    const int ntile = 2 * ((n + 31) / 32);
    for (int idx = threadIdx.x; idx < ntile * KS * 32; idx += blockDim.x) {
        const int ln = idx & 31, ks = (idx >> 5) % KS, tile = idx / (32 * KS);
        const int r0 = tile * 16 + (ln >> 2), r1 = r0 + 8, cc = ln & 3;
        const int w0 = 4 * (4 * (ks >> 1) + cc) + 2 * (ks & 1);
        const uint32_t* q0 = reinterpret_cast<const uint32_t*>(Qb + (size_t)r0 * D) + w0;
        const uint32_t* q1 = reinterpret_cast<const uint32_t*>(Qb + (size_t)r1 * D) + w0;
        uint4 f;
        f.x = r0 < n ? q0[0] : 0u;
        f.y = r1 < n ? q1[0] : 0u;
        f.z = r0 < n ? q0[1] : 0u;
        f.w = r1 < n ? q1[1] : 0u;
        s_q[idx] = f;
    }
}

template <int D>
__device__ __forceinline__ void query_norms(const PrefillArgs& a, int bh) {
    const __half* Qb = a.Q + (size_t)bh * a.n * D;
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) {
        float s = 0.f;
        for (int d = 0; d < D; ++d) { const float f = a.scale * __half2float(Qb[(size_t)i * D + d]); s = fmaf(f, f, s); }
        a.qnorm2[(size_t)bh * a.n + i] = s;
    }
}

__device__ __forceinline__ void fold_stats(float2& to, const float2& p) {          // (max, sum of exponentials)
    const float NEG = __int_as_float(0xff800000), m = fmaxf(to.x, p.x);
    to.y = (to.x == NEG ? 0.f : to.y * __expf(to.x - m)) + (p.x == NEG ? 0.f : p.y * __expf(p.x - m));
    to.x = m;
}

// Sequences of more than a cluster of CTAs.  What bounds it is memory: the keys are read twice and the rows written once.
// (Logits written by the first pass and normalised in place by a second kernel - the keys read once, the rows written
// twice and read once - took 374 + 217 us for 160 (b,h) x 8192 tokens and 64 rows.)  A warp takes 16 tokens per
// step; column g of its two 8-token operands is token 4 (g / 2) + (g mod 2) resp. that + 2, so that a lane ends up with
// four consecutive tokens of a row.  STATS: the first pass.
template <int D, bool STATS>
__global__ void __launch_bounds__(PW_WARPS * 32, 3) window_long_kernel(const PrefillArgs a) {
    constexpr int WPL = D / 8;          // 32-bit words per lane and token
    constexpr int KS = D / 16;          // k-steps
    extern __shared__ __align__(16) float s_dyn[];
    uint4* s_q = reinterpret_cast<uint4*>(s_dyn);
    __shared__ float2 s_part[PW_WARPS][PW_MAXQ];             // STATS: per warp; else entry 0: what the rows are normalised with
    qaq_dependency();
    const int bh = blockIdx.y, chunk = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, c = lane & 3;
    const float NEG = __int_as_float(0xff800000);
    const __half* Kb = a.K + (size_t)(bh / a.H) * a.sb + (size_t)(bh % a.H) * a.sh;
    const int t_warp = chunk * PW_CHUNK + warp * (PW_CHUNK / PW_WARPS);
    // this warp's keys are on their way to L2 while the queries are laid out
    constexpr int LPT = D >= 64 ? D / 64 : 1;                                    // 128-byte lines per token
    for (int ln = lane; ln < (PW_CHUNK / PW_WARPS) * LPT; ln += 32) {
        const int t = t_warp + ln / LPT;
        if (t < a.T) asm volatile("prefetch.global.L2 [%0];" ::"l"(Kb + (size_t)t * a.st + (ln % LPT) * 64));
    }
    if (STATS && a.qnorm2 && chunk == 0) query_norms<D>(a, bh);
    lay_out_queries<D>(s_q, a.Q + (size_t)bh * a.n * D, a.n);
    if (!STATS) {      // merged statistics of the rows: four threads per row
        const int i = threadIdx.x >> 2, part = threadIdx.x & 3;
        float2 st = make_float2(NEG, 0.f);
        if (i < a.n)
            for (int ch = part; ch < a.nchunk; ch += 4) fold_stats(st, a.part[((size_t)bh * a.nchunk + ch) * a.n + i]);
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) fold_stats(st, make_float2(__shfl_xor_sync(0xFFFFFFFFu, st.x, o), __shfl_xor_sync(0xFFFFFFFFu, st.y, o)));
        if (i < a.n && part == 0) s_part[0][i] = make_float2(st.x, st.y > 0.f ? 1.0f / st.y : 0.f);
        for (int k = threadIdx.x; k < PW_CHUNK; k += blockDim.x) {
            const int t = chunk * PW_CHUNK + k;
            if (t < a.T) a.nvalid[(size_t)bh * a.T + t] = (uint8_t)min(a.n, a.T - t);
        }
    }
    __syncthreads();
    const bool vec_ok = (a.T & 3) == 0 && ((uintptr_t)a.ring & 15) == 0;      // rows start 16-byte aligned, no ragged end

    {
        constexpr int MT = PW_MAXQ / 16;                // 16-row tiles of queries: a warp's keys are read once for all of them
        float2 st[MT][2];               // rows g, g + 8 of the tiles over the tokens this lane sees
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) st[mt][0] = st[mt][1] = make_float2(NEG, 0.f);
#pragma unroll 1
        for (int step = 0; step < PW_CHUNK / PW_WARPS / 16; ++step) {
            const int t0 = t_warp + 16 * step;
            if (t0 >= a.T) break;
            uint32_t bw[2][WPL];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = t0 + 4 * (g >> 1) + (g & 1) + 2 * h;
                const uint4* src = reinterpret_cast<const uint4*>(Kb + (size_t)(t < a.T ? t : 0) * a.st) + c;
#pragma unroll
                for (int i = 0; i < WPL / 4; ++i) {
                    uint4 v = make_uint4(0, 0, 0, 0);
                    if (t < a.T) v = src[4 * i];
                    bw[h][4 * i] = v.x; bw[h][4 * i + 1] = v.y; bw[h][4 * i + 2] = v.z; bw[h][4 * i + 3] = v.w;
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                if (mt * 16 >= a.n) break;
                float acc[2][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) { acc[0][i] = 0.f; acc[1][i] = 0.f; }
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    const uint4 f = s_q[(mt * KS + ks) * 32 + lane];
                    const uint32_t fr[4] = {f.x, f.y, f.z, f.w};
                    mma_16816(acc[0], fr, bw[0][2 * ks], bw[0][2 * ks + 1]);
                    mma_16816(acc[1], fr, bw[1][2 * ks], bw[1][2 * ks + 1]);
                }
                // acc[h][2 hr], acc[h][2 hr + 1]: row g + 8 hr, tokens t0 + 4c + 2h, + 1
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    const int i = mt * 16 + g + 8 * hr;          // query
                    if (i >= a.n) continue;
                    const int t = t0 + 4 * c, left = a.T - a.n + i - t + 1; // how many of the lane's tokens the query sees (or more)
                    const float l[4] = {a.scale * acc[0][2 * hr], a.scale * acc[0][2 * hr + 1], a.scale * acc[1][2 * hr], a.scale * acc[1][2 * hr + 1]};
                    if (STATS) {
                        float m = NEG;
#pragma unroll
                        for (int e = 0; e < 4; ++e) if (e < left) m = fmaxf(m, l[e]);
                        float sum = 0.f;
#pragma unroll
                        for (int e = 0; e < 4; ++e) if (e < left) sum += __expf(l[e] - m);
                        fold_stats(st[mt][hr], make_float2(m, sum));
                    } else {
                        const float2 mi = s_part[0][i];
                        float4 o;
                        o.x = left > 0 ? __expf(l[0] - mi.x) * mi.y : 0.f;
                        o.y = left > 1 ? __expf(l[1] - mi.x) * mi.y : 0.f;
                        o.z = left > 2 ? __expf(l[2] - mi.x) * mi.y : 0.f;
                        o.w = left > 3 ? __expf(l[3] - mi.x) * mi.y : 0.f;
                        float* row = a.ring + ((size_t)bh * a.n + (a.n - 1 - i)) * a.T + t;
                        if (vec_ok) { if (t < a.T) *reinterpret_cast<float4*>(row) = o; }
                        else {
                            if (t < a.T) row[0] = o.x;
                            if (t + 1 < a.T) row[1] = o.y;
                            if (t + 2 < a.T) row[2] = o.z;
                            if (t + 3 < a.T) row[3] = o.w;
                        }
                    }
                }
            }
        }
        if (STATS) {      // merge the four lanes of a row
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    float2 v = st[mt][hr];
                    fold_stats(v, make_float2(__shfl_xor_sync(0xFFFFFFFFu, v.x, 1), __shfl_xor_sync(0xFFFFFFFFu, v.y, 1)));
                    fold_stats(v, make_float2(__shfl_xor_sync(0xFFFFFFFFu, v.x, 2), __shfl_xor_sync(0xFFFFFFFFu, v.y, 2)));
                    if (c == 0) s_part[warp][mt * 16 + g + 8 * hr] = v;
                }
        }
    }
    if (STATS) {          // then the warps
        __syncthreads();
        if ((int)threadIdx.x < a.n) {
            float2 v = make_float2(NEG, 0.f);
#pragma unroll
            for (int w = 0; w < PW_WARPS; ++w) fold_stats(v, s_part[w][threadIdx.x]);
            a.part[((size_t)bh * a.nchunk + chunk) * a.n + threadIdx.x] = v;
        }
    }
}

// ---- one pass: the CTAs of one (b,h) form a thread-block cluster.  Each keeps the logits of its 512 tokens in
// shared memory, the per-row (max, sum) of the CTAs are exchanged through distributed shared memory, and the
// normalised rows are written once: K is read once and the ring written once (no logits in global memory, no
// workspace).  Used while a (b,h) fits a portable cluster (up to 8 x 512 tokens); longer sequences take the two
// kernels above.
constexpr int PC_WARPS = 16;            // 32 tokens per warp
constexpr int PC_MINCTA = 2;            // two CTAs per SM (64 registers per thread)
constexpr int PC_CHUNK = 512;           // tokens per CTA
constexpr int PC_MAXCTA = 8;            // portable cluster size
constexpr int PC_PITCH = PC_CHUNK + 8;  // row pitch of the logits tile in floats (spreads the rows of a fragment over the banks)

template <int D>
__global__ void __launch_bounds__(PC_WARPS * 32, PC_MINCTA) window_cluster_kernel(const PrefillArgs a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int WPL = D / 8;
    constexpr int KS = D / 16;
    extern __shared__ __align__(16) float s_l[];            // [n][PC_PITCH] logits of this CTA's tokens, then the queries
    // the queries as A-operand fragments, one uint4 per (16-row tile, k step, lane): every warp reads the same ones
    uint4* s_q = reinterpret_cast<uint4*>(s_l + (size_t)a.n * PC_PITCH);
    __shared__ float s_part[PC_WARPS][32];                   // per warp: maximum of every row of the current 32 over its tokens
    __shared__ float s_mcta[PW_MAXQ];                        // maximum of every row over this CTA's tokens
    __shared__ float2 s_all[PC_MAXCTA][PW_MAXQ];             // (max, sum of exponentials) of every row over the tokens of every CTA
                                                             // of the cluster: each CTA writes its entries into all the copies
    __shared__ float s_inv[PW_MAXQ];
    qaq_dependency();
    const int bh = blockIdx.y, chunk = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, c = lane & 3;
    const int b_idx = bh / a.H, h_idx = bh % a.H;
    const __half* Kb = a.K + (size_t)b_idx * a.sb + (size_t)h_idx * a.sh;
    const __half* Qb = a.Q + (size_t)bh * a.n * D;
    const float NEG = __int_as_float(0xff800000);

    if (a.qnorm2 && chunk == 0) query_norms<D>(a, bh);
    const int t_cta = chunk * PC_CHUNK;
    const int t_warp = t_cta + warp * (PC_CHUNK / PC_WARPS);
    // this warp's keys are on their way to L2 while the queries are laid out
    constexpr int LPT = D >= 64 ? D / 64 : 1;                                    // 128-byte lines per token
    for (int ln = lane; ln < (PC_CHUNK / PC_WARPS) * LPT; ln += 32) {
        const int t = t_warp + ln / LPT;
        if (t < a.T) asm volatile("prefetch.global.L2 [%0];" ::"l"(Kb + (size_t)t * a.st + (ln % LPT) * 64));
    }
    // first half of a cluster barrier: by the time the row statistics are exchanged every CTA of the cluster is known
    // to be running (its shared memory may be written)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

    lay_out_queries<D>(s_q, Qb, a.n);
    __syncthreads();

    for (int mp = 0; mp * 32 < a.n; ++mp) {            // two 16-row tiles of queries at a time
        float rm[2][2];                 // running maximum of rows g, g + 8 of the two tiles over the tokens this lane sees
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) rm[mt][0] = rm[mt][1] = NEG;

#pragma unroll 1
        for (int step = 0; step < PC_CHUNK / PC_WARPS / 8; step += 2) {    // two groups of 8 tokens per set of query fragments
            const int t0 = t_warp + 8 * step;
            if (t0 >= a.T) break;
            // lane (g, c) holds, of token t0 + g (and t0 + 8 + g), the 16-byte pieces c, c + 4, ...: the four lanes of a
            // token read 64 consecutive bytes at a time, and the words of piece 4i + c are the B operands of k steps
            // 2i and 2i + 1 (the queries are laid out to match)
            uint32_t bw[2][WPL];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = t0 + 8 * h + g;
                const uint4* src = reinterpret_cast<const uint4*>(Kb + (size_t)(t < a.T ? t : 0) * a.st) + c;
#pragma unroll
                for (int i = 0; i < WPL / 4; ++i) {
                    uint4 v = make_uint4(0, 0, 0, 0);
                    if (t < a.T) v = src[4 * i];
                    bw[h][4 * i] = v.x; bw[h][4 * i + 1] = v.y; bw[h][4 * i + 2] = v.z; bw[h][4 * i + 3] = v.w;
                }
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                float acc[2][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) { acc[0][i] = 0.f; acc[1][i] = 0.f; }
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    const uint4 f = s_q[((2 * mp + mt) * KS + ks) * 32 + lane];
                    const uint32_t fr[4] = {f.x, f.y, f.z, f.w};
                    mma_16816(acc[0], fr, bw[0][2 * ks], bw[0][2 * ks + 1]);
                    mma_16816(acc[1], fr, bw[1][2 * ks], bw[1][2 * ks + 1]);
                }
                // acc[h][0..1]: row g, tokens t0+8h+2c, +1;  acc[h][2..3]: row g+8
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    const int i = mp * 32 + mt * 16 + g + 8 * hr;          // query
                    if (i >= a.n) continue;
                    const int last = a.T - a.n + i;                         // last token the query sees
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int t = t0 + 8 * h + 2 * c;
                        const float l0 = a.scale * acc[h][2 * hr], l1 = a.scale * acc[h][2 * hr + 1];
                        *reinterpret_cast<float2*>(&s_l[(size_t)i * PC_PITCH + (t - t_cta)]) = make_float2(l0, l1);
                        if (t <= last) rm[mt][hr] = fmaxf(rm[mt][hr], l0);       // last < T: one bound does for both
                        if (t + 1 <= last) rm[mt][hr] = fmaxf(rm[mt][hr], l1);
                    }
                }
            }
        }
        // merge the four lanes of a row, then the warps, into this CTA's maximum of the row
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                float m = rm[mt][hr];
                m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
                m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, 2));
                if (c == 0) s_part[warp][mt * 16 + g + 8 * hr] = m;
            }
        __syncthreads();
        if (threadIdx.x < 32 && mp * 32 + (int)threadIdx.x < a.n) {
            float m = NEG;
#pragma unroll
            for (int w = 0; w < PC_WARPS; ++w) m = fmaxf(m, s_part[w][threadIdx.x]);
            s_mcta[mp * 32 + threadIdx.x] = m;
        }
        __syncthreads();
    }
    // ---- the logits become exponentials relative to the CTA's row maximum, in place (one exponential per entry in
    //      all; entries a query cannot see become 0), and every row gets its sum over this CTA's tokens
    const int nt = min(PC_CHUNK, a.T - t_cta);
    const unsigned ncta = cluster.num_blocks(), rank = cluster.block_rank();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // second half of the barrier begun at the start
    for (int i = warp; i < a.n; i += PC_WARPS) {
        const int last = a.T - a.n + i;
        const float m = s_mcta[i];
        float* rowl = s_l + (size_t)i * PC_PITCH;
        float sum = 0.f;
        for (int k = 4 * lane; k < nt; k += 128) {       // the pitch covers the four of a ragged end; what is there is not used
            const float4 l = *reinterpret_cast<const float4*>(rowl + k);
            float4 e;
            e.x = (t_cta + k <= last) ? __expf(l.x - m) : 0.f;
            e.y = (t_cta + k + 1 <= last) ? __expf(l.y - m) : 0.f;
            e.z = (t_cta + k + 2 <= last) ? __expf(l.z - m) : 0.f;
            e.w = (t_cta + k + 3 <= last) ? __expf(l.w - m) : 0.f;
            *reinterpret_cast<float4*>(rowl + k) = e;
            sum += (e.x + e.y) + (e.z + e.w);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (lane < (int)ncta) *cluster.map_shared_rank(&s_all[rank][i], lane) = make_float2(m, sum);
    }
    // ---- every CTA of the (b,h) has the row statistics of all of them (the remote stores are complete at the cluster
    //      barrier, and nothing is read from or written to another CTA afterwards): merge them
    cluster.sync();
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) {
        float m = NEG, s = 0.f;
        for (unsigned r = 0; r < ncta; ++r) {
            const float2 p = s_all[r][i];
            const float mn = fmaxf(m, p.x);
            s = (m == NEG ? 0.f : s * __expf(m - mn)) + (p.x == NEG ? 0.f : p.y * __expf(p.x - mn));
            m = mn;
        }
        // what this CTA's exponentials are multiplied by: exp(own maximum - maximum of the row) / sum of the row
        const float own = s_mcta[i];
        s_inv[i] = (s > 0.f && own != NEG) ? __expf(own - m) / s : 0.f;
    }
    __syncthreads();
    // ---- normalised rows, newest first, written once; rows-per-token counts
    const bool vec_ok = (a.T & 3) == 0 && ((uintptr_t)a.ring & 15) == 0;      // rows start 16-byte aligned, no ragged end
    for (int r = warp; r < a.n; r += PC_WARPS) {
        const int i = a.n - 1 - r;
        const float f = s_inv[i];
        float* row = a.ring + ((size_t)bh * a.n + r) * a.T + t_cta;
        const float* src = s_l + (size_t)i * PC_PITCH;
        if (vec_ok) {     // four tokens per lane and store
            for (int k = 4 * lane; k < nt; k += 128) {
                float4 o = *reinterpret_cast<const float4*>(src + k);
                o.x *= f; o.y *= f; o.z *= f; o.w *= f;
                *reinterpret_cast<float4*>(row + k) = o;
            }
        } else {
            for (int k = lane; k < nt; k += 32) row[k] = src[k] * f;
        }
    }
    for (int k = threadIdx.x; k < nt; k += blockDim.x) a.nvalid[(size_t)bh * a.T + t_cta + k] = (uint8_t)min(a.n, a.T - (t_cta + k));
}

template <int D>
qaq_status run_cluster(const PrefillArgs& a, int BH, int ncl, size_t smem, cudaStream_t s) {
    static SmemSeen seen;
    const size_t most = (size_t)PW_MAXQ * PC_PITCH * sizeof(float) + 4 * (D / 16) * 32 * sizeof(uint4);
    QAQ_CUDA_TRY(qaq_allow_smem((const void*)window_cluster_kernel<D>, most, seen));
    QAQ_CUDA_TRY(qaq_launch_cluster(window_cluster_kernel<D>, dim3((unsigned)ncl, (unsigned)BH), dim3(PC_WARPS * 32), ncl, smem, s, a));
    return QAQ_OK;
}

template <int D>
qaq_status run_long(const PrefillArgs& a, int BH, cudaStream_t s) {
    const dim3 grid((unsigned)a.nchunk, (unsigned)BH);
    const size_t smem = (size_t)(2 * ((a.n + 31) / 32)) * (D / 16) * 32 * sizeof(uint4);       // at most 16 KB
    QAQ_CUDA_TRY(qaq_launch(window_long_kernel<D, true>, grid, dim3(PW_WARPS * 32), smem, s, a));
    QAQ_CUDA_TRY(qaq_launch(window_long_kernel<D, false>, grid, dim3(PW_WARPS * 32), smem, s, a));
    return QAQ_OK;
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
    a.Q = (const __half*)Q; a.K = (const __half*)K; a.sb = stride_b; a.sh = stride_h; a.st = stride_t;
    a.H = cfg->heads; a.T = n_tokens; a.n = cfg->window; a.scale = softmax_scale;
    a.ring = score_ring; a.nvalid = nvalid; a.qnorm2 = qnorm2; a.part = (float2*)ws;
    a.nchunk = (n_tokens + PW_CHUNK - 1) / PW_CHUNK;
    cudaStream_t s = (cudaStream_t)stream;
    const int ncl = (n_tokens + PC_CHUNK - 1) / PC_CHUNK;
    if (ncl <= PC_MAXCTA) {
        // one pass: the CTAs of a (b,h) are one cluster
        const size_t smem = (size_t)cfg->window * PC_PITCH * sizeof(float) +
                            (size_t)(2 * ((cfg->window + 31) / 32)) * (cfg->head_dim / 16) * 32 * sizeof(uint4);   // logits, query fragments
        const int BH = cfg->batch * cfg->heads;
        switch (cfg->head_dim) {
            case 32: return run_cluster<32>(a, BH, ncl, smem, s);
            case 64: return run_cluster<64>(a, BH, ncl, smem, s);
            case 128: return run_cluster<128>(a, BH, ncl, smem, s);
        }
        return QAQ_ERR_UNSUPPORTED_SHAPE;
    }
    switch (cfg->head_dim) {
        case 32: return run_long<32>(a, cfg->batch * cfg->heads, s);
        case 64: return run_long<64>(a, cfg->batch * cfg->heads, s);
        case 128: return run_long<128>(a, cfg->batch * cfg->heads, s);
    }
    return QAQ_ERR_UNSUPPORTED_SHAPE;
}

extern "C" qaq_status qaq_qnorm2_quantile(const float* values, long n, double upper_frac, float* out, void* stream) {
    if (!values || !out || n < 1 || !(upper_frac >= 0.0 && upper_frac < 1.0)) return QAQ_ERR_INVALID_ARG;
    quantile_kernel<<<1, QS_THREADS, 0, (cudaStream_t)stream>>>(values, n, upper_frac, out);
    QAQ_CUDA_TRY(cudaGetLastError());
    return QAQ_OK;
}
