// Internal definitions shared by the libqaq translation units (not part of the ABI).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "qaq.h"

#define QAQ_TILE QAQ_TILE_TOKENS

// Device storage of one tensor (K or V) of the cache.  Tokens are grouped in tiles of
// QAQ_TILE consecutive tokens; a tile's packed codes are contiguous, sorted by width, and
// start 16-byte aligned somewhere in the (b,h) pool (tiles are placed by a bump allocator,
// so their order in memory is not the token order).  Per-token metadata is 6 bytes: the width, the
// token's place in the tile (qaq_codec.cuh) and the binary16 min and max of the non-outlier entries
// (step = (max-min)*2^-B is recomputed where needed).  Outliers of a tile are contiguous 32-bit entries
//   value(binary16) | channel << 16 | token-in-tile << 24,  sorted by (token, channel).
struct TensorStore {
    uint8_t* codes;         // [BH][pool_bytes]
    unsigned short* bs;     // [BH][tmax_pad]  width | slot << 8
    uint32_t* mnmx;         // [BH][tmax_pad]  half(min) | half(max) << 16
    uint4* tile;            // [BH][ntiles]    byte offset of the tile in its pool, bytes, first outlier entry, outlier entries
    uint32_t* outl;         // [BH][ocap]
    uint32_t* pool_end;     // [BH] bump pointer, bytes; a multiple of 16 unless the last thing before it is the open tile
    uint32_t* opool_end;    // [BH] bump pointer, entries
};

struct qaq_cache {
    qaq_config cfg;
    int BH;
    int tmax_pad;       // max_tokens rounded up to a tile
    int ntiles;         // tmax_pad / QAQ_TILE
    size_t pool_bytes;  // per (b,h)
    uint32_t ocap;      // outlier entries per (b,h)
    TensorStore t[2];
    int* d_status;      // sticky device-side status; the words behind it: qaq_d_count, qaq_d_ticket, qaq_d_pool_use
    void* slab;         // the one allocation everything above lives in
    size_t slab_bytes;
    size_t reset_off, reset_bytes;   // the range of the slab that qaq_cache_reset clears
    long tokens;        // host counter
    // lazily sized staging for the *_host entry points
    void* stage[8];
    size_t stage_bytes[8];
};

// the CUDA error behind the most recent QAQ_ERR_CUDA of this process (qaq_last_cuda_error)
extern int g_qaq_last_cuda_error;

#define QAQ_CUDA_TRY(expr)                                  \
    do {                                                    \
        cudaError_t _e = (expr);                            \
        if (_e != cudaSuccess) { g_qaq_last_cuda_error = (int)_e; (void)cudaGetLastError(); return QAQ_ERR_CUDA; } \
    } while (0)

// the token count in device memory that the qaq_stream_* calls work with (valid between qaq_stream_begin and
// qaq_stream_end), and the arrival counter of the kernel that advances it (zero between launches)
static inline int* qaq_d_count(const qaq_cache* c) { return c->d_status + 1; }
static inline unsigned* qaq_d_ticket(const qaq_cache* c) { return (unsigned*)(c->d_status + 2); }
// two words for what qaq_cache_pool_use finds
static inline unsigned* qaq_d_pool_use(const qaq_cache* c) { return (unsigned*)(c->d_status + 4); }

#ifdef __CUDACC__
// Kernels of this library are launched with programmatic dependent launch: the launch of a kernel is prepared while the
// one before runs, its CTAs begin as the last ones of the one before leave, and wait there (qaq_dependency) until all
// writes of the one before are visible.  Every kernel launched with qaq_launch calls qaq_dependency first thing in every
// CTA; so a kernel that has got past it has everything before it in the stream behind it.  Such a kernel must not use
// non-coherent loads (__ldg) for what its predecessor writes.  Letting the successor begin earlier
// (griddepcontrol.launch_dependents) was slower: its waiting CTAs take room (a captured step of four layers: 24.1 us per
// layer without, 26.7 with it at the start of the kernels, 24.4 without dependent launch; a 333-token prefill 58, 64, 75).
__device__ __forceinline__ void qaq_dependency() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// transaction barriers in shared memory, for one arrival
__device__ __forceinline__ void bar_init(uint32_t bar) { asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// false if the phase did not complete within the limit (a copy takes microseconds; every try waits for a while itself)
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    uint32_t done = 0;
#pragma unroll 1
    for (int i = 0; i < (1 << 14) && !done; ++i)
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
__device__ __forceinline__ float warp_max(float x) {
    float r;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
    return r;
}
// cluster: CTAs (consecutive in x) that form a thread-block cluster
template <typename... P, typename... A>
static inline cudaError_t qaq_launch_cluster(void (*kernel)(P...), dim3 grid, dim3 block, int cluster, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = grid; lc.blockDim = block; lc.dynamicSmemBytes = smem; lc.stream = s; lc.attrs = at; lc.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&lc, kernel, P(args)...);
}
template <typename... P, typename... A>
static inline cudaError_t qaq_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    return qaq_launch_cluster(kernel, grid, block, 1, smem, s, args...);
}
// Shared memory beyond 48 KB has to be allowed once per kernel and context.  `seen` (one per kernel) remembers contexts by their
// ids, which are not used again; where a context has no id yet, or another one has taken its place, the kernel is allowed once more.
struct SmemSeen { std::atomic<unsigned long long> id[8]; };
// the id of the current context; false where there is none
static inline bool qaq_context_id(unsigned long long& id) {
    typedef int (*GetId)(void* context, unsigned long long* id);          // cuCtxGetId; null: the current context
    static const GetId get_id = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &found);
        if (e != cudaSuccess) (void)cudaGetLastError();
        return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? (GetId)f : (GetId) nullptr;
    }();
    return get_id && get_id(nullptr, &id) == 0;
}
static inline cudaError_t qaq_allow_smem(const void* kernel, size_t smem, SmemSeen& seen) {
    unsigned long long id = 0;
    const bool known = qaq_context_id(id);
    // (an entry holds the id plus one: zero is an empty one)
    if (known && seen.id[id % 8].load(std::memory_order_acquire) == id + 1) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && known) seen.id[id % 8].store(id + 1, std::memory_order_release);
    return e;
}
// How many clusters of k CTAs of a kernel run at once: asked once per kernel, k and context (whose id goes with the answer).
struct ClusterRoom { std::atomic<unsigned long long> known[9]; };
struct ContextName {                             // (who asks for several sizes looks it up once)
    unsigned long long id = 0;
    bool named;
    ContextName() { named = qaq_context_id(id); }
};
template <class K>
int clusters_at_once(K kernel, int threads, size_t smem, int k, ClusterRoom& room, const ContextName& context = ContextName()) {
    const unsigned long long id = context.id;
    const bool named = context.named;
    const unsigned long long was = room.known[k].load(std::memory_order_acquire);
    if (named && (was >> 16) == id + 1) return (int)(was & 0xFFFFu);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)k; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)k); lc.blockDim = dim3((unsigned)threads); lc.dynamicSmemBytes = smem; lc.attrs = &at; lc.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &lc) != cudaSuccess) { (void)cudaGetLastError(); return 0; }
    n = n < 0 ? 0 : n > 0xFFFF ? 0xFFFF : n;
    if (named) room.known[k].store((id + 1) << 16 | (unsigned)n, std::memory_order_release);
    return n;
}

// Space taken from a pool that turned out not to fit is given back only while nothing has been taken behind it: with a
// plain subtraction a later taker could be handed space that somebody else holds.  Otherwise it stays taken until
// qaq_cache_compact or qaq_cache_reset.
__device__ __forceinline__ void pool_give_back(uint32_t* pool_end, uint32_t base, uint32_t taken) {
    if (taken) atomicCAS(pool_end, base + taken, base);
}
#endif

static inline bool qaq_dim_ok(int D) { return D == 32 || D == 64 || D == 128; }

// launchers implemented in the kernel translation units
qaq_status qaq_launch_select(const qaq_config* cfg, const qaq_policy* pol, const void* K, const void* V, long sb,
                             long sh, long st, int n, const float* ring, const uint8_t* nvalid, const float* thr,
                             uint8_t* bitsK, uint8_t* bitsV, cudaStream_t s);
qaq_status qaq_launch_append(qaq_cache* c, const void* K, const void* V, long sb, long sh, long st, int n_new,
                             const uint8_t* bitsK, const uint8_t* bitsV, const qaq_policy* pol, const float* ring,
                             const uint8_t* nvalid, const float* thr, cudaStream_t s);
