// Shared device/host helpers of the carnator library (workspace layout, status word, small math).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stdio.h>
#include <atomic>

#include "carnator.h"

namespace carnator {

constexpr int kMaxKeyBlocksBuilder = 4096;   // rows above 1024 blocks are sorted in shared memory (mass) or held 128 keys a lane (top-k)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr unsigned long long kDefaultWaitNs = 2000000000ull;   // limit of a bounded device-side wait unless the header says otherwise

// First 256 bytes of every workspace.
struct WsHeader {
    int32_t status;              // carnator_status set by kernels (0 = ok); first error wins
    int32_t info[3];             // where a bounded wait gave up / which check failed
    unsigned long long tiles;    // evaluated (query block, key block) pairs, written by carnator_compacted_tiles
    int32_t work[4];             // work-item counters of persistent kernels (zeroed with the header)
    unsigned long long wait_limit_ns;   // 0: the default limit of every bounded device-side wait; tests set a short one
    int32_t debug_withhold;      // 0 except in the test of the time-out path: the K producer withholds one copy
    int32_t pad[51];
};
static_assert(sizeof(WsHeader) == 256, "header is 256 bytes");

__host__ __device__ inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
__host__ __device__ inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Layout of the attention workspace: header | counts | order | lists.
struct AttnWs {
    WsHeader* hdr;
    int32_t* counts;   // [B,H,nqb]   number of listed key blocks of each query block
    int32_t* order;    // [B,H,nqb]   query blocks of a head, longest list first; of 64 tokens: pairs, longest pair first
    int32_t* lists;    // [B,H,nqb,nkb] ascending key-block indices, first counts[...] entries valid
    size_t bytes;
};

inline AttnWs attn_ws_layout(void* base, int B, int H, int nqb, int nkb) {
    AttnWs w;
    char* p = static_cast<char*>(base);
    size_t off = 0;
    w.hdr = reinterpret_cast<WsHeader*>(p + off);           off += align256(sizeof(WsHeader));
    size_t rows = size_t(B) * H * nqb;
    w.counts = reinterpret_cast<int32_t*>(p + off);         off += align256(rows * 4);
    w.order = reinterpret_cast<int32_t*>(p + off);          off += align256(rows * 4);
    w.lists = reinterpret_cast<int32_t*>(p + off);          off += align256(rows * size_t(nkb) * 4);
    w.bytes = off;
    return w;
}

// Layout of the builder workspace: header | pooled-blocks counters | qbar | kbar | scores | three-term means of Q, of K.
struct BuildWs {
    WsHeader* hdr;
    int32_t* done;   // [B,H]  pooled blocks of each head written so far (fused builder; zeroed together with the header)
    float* qbar;     // [B,H,nqb,D]
    float* kbar;     // [B,H,nkb,D]
    float* scores;   // [B,H,nqb,nkb]
    __nv_bfloat16* qsplit;   // [3][B*H*nqb][D]  block means of Q as three bf16 terms (fused builder)
    __nv_bfloat16* ksplit;   // [3][B*H*nkb][D]
    size_t bytes;
};

inline BuildWs build_ws_layout(void* base, int B, int H, int nqb, int nkb, int D) {
    BuildWs w;
    char* p = static_cast<char*>(base);
    size_t off = 0;
    w.hdr = reinterpret_cast<WsHeader*>(p + off);           off += align256(sizeof(WsHeader));
    w.done = reinterpret_cast<int32_t*>(p + off);           off += align256(size_t(B) * H * 4);
    w.qbar = reinterpret_cast<float*>(p + off);             off += align256(size_t(B) * H * nqb * D * 4);
    w.kbar = reinterpret_cast<float*>(p + off);             off += align256(size_t(B) * H * nkb * D * 4);
    w.scores = reinterpret_cast<float*>(p + off);           off += align256(size_t(B) * H * nqb * size_t(nkb) * 4);
    w.qsplit = reinterpret_cast<__nv_bfloat16*>(p + off);   off += align256(size_t(3) * B * H * nqb * D * 2);
    w.ksplit = reinterpret_cast<__nv_bfloat16*>(p + off);   off += align256(size_t(3) * B * H * nkb * D * 2);
    w.bytes = off;
    return w;
}

__device__ inline void set_status(WsHeader* hdr, int32_t code, int32_t i0, int32_t i1, int32_t i2) {
    if (atomicCAS(&hdr->status, 0, code) == 0) {
        hdr->info[0] = i0; hdr->info[1] = i1; hdr->info[2] = i2;
    }
}

__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Token geometry used by the always-kept rule of the builder.
struct Geometry {
    int N, n_text, hw, T, bq, bk, window, text_dense;
};

// Programmatic dependent launch: the next kernel of a call starts while this one drains, and waits here for its results.
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Notes a failed runtime call and takes it out of the runtime's record of the last error: it is reported here, and the next
// call's launch check must not find it again.
inline carnator_status cuda_error(cudaError_t e, const char* where, char* err, size_t errlen) {
    snprintf(err, errlen, "%s: %s", where, cudaGetErrorString(e));
    cudaGetLastError();
    return CARNATOR_ERR_CUDA;
}

// Number of the current CUDA context, unique for the life of the process (a reset of the device makes a new one); 0 if there
// is none yet.
inline unsigned long long context_id() {
    typedef int (*CtxGetIdFn)(void*, unsigned long long*);
    static const CtxGetIdFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<CtxGetIdFn>(p);
        cudaGetLastError();
        return CtxGetIdFn(nullptr);
    }();
    unsigned long long id = 0;
    return fn && fn(nullptr, &id) == 0 ? id : 0;
}

// Contexts in which a kernel has been allowed the dynamic shared memory of its largest launch (an attribute of the kernel in
// each context): asking the runtime on every call costs about a microsecond.  One static object per kernel, at the place that
// launches it.  A context that is not in its slot is asked for again.
struct SmemAllowed {
    static constexpr int kSlots = 16;
    std::atomic<unsigned long long> ctx[kSlots];
    bool has(unsigned long long id) const { return id != 0 && ctx[id % kSlots].load(std::memory_order_acquire) == id; }
    void add(unsigned long long id) { if (id != 0) ctx[id % kSlots].store(id, std::memory_order_release); }
};

// Launch that may begin before the kernel ahead of it in the stream has ended (that kernel calls grid_launch_dependents,
// this one grid_wait before it reads anything of it).
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace carnator
