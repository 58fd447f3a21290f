// Connectivity builder kernels: block pooling (HBM-bound), pooled-score tile product (fp32 FFMA),
// per-row selection (top-k or cumulative softmax mass) with the always-kept blocks.
// Paper: Appendix "Reuse-Scope Implementation Details" (per head and query block, the smallest set of
// key blocks covering a fixed fraction of the attention mass), in the pooled-score form.
#pragma once
#include "common.cuh"

namespace carnator {

// ----------------------------------------------------------------------------------------------
// M1: block means of Q and K.  One CTA per (tensor, b, h, block); reads block x D bf16 once.
// ----------------------------------------------------------------------------------------------
struct PoolArgs {
    const __nv_bfloat16* X[2];
    int64_t stride[2][3];
    int block[2];
    int nb[2];
    float* out[2];     // [B,H,nb,D]
    int N, H;
    WsHeader* hdr;
};

__device__ __forceinline__ uint4 ld_stream16(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// A CTA takes 32 KB of consecutive tokens, one block at D = 128 and two at D = 64, with all eight 16-byte loads of a thread
// in flight at once (with four loads, and 16 KB per CTA at D = 64, 218 MB took 46 us).
// The first CTA clears the workspace header for the kernels behind it.
template <int D>
__global__ void __launch_bounds__(256) pool_kernel(PoolArgs a) {
    constexpr int TPR = D / 8;          // threads per token row (16 B each)
    constexpr int TPB = 2 * D;          // threads per block of tokens
    constexpr int RPP = TPB / TPR;      // token rows per pass (16)
    constexpr int BPC = 256 / TPB;      // blocks per CTA
    constexpr int U = 128 / RPP;        // passes of a 128-token block
    grid_launch_dependents();
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x < sizeof(WsHeader) / 4)
        reinterpret_cast<int32_t*>(a.hdr)[threadIdx.x] = 0;
    const int which = blockIdx.z & 1;
    const int b = blockIdx.z >> 1;
    const int h = blockIdx.y;
    const int part = threadIdx.x / TPB, t = threadIdx.x % TPB;
    const int I = blockIdx.x * BPC + part;
    // select with ternaries: dynamic indexing of the argument struct would force a local copy
    const int nb = which ? a.nb[1] : a.nb[0];
    if (int(blockIdx.x) * BPC >= nb) return;
    const int block = which ? a.block[1] : a.block[0];
    const __nv_bfloat16* X = which ? a.X[1] : a.X[0];
    float* out = which ? a.out[1] : a.out[0];
    const int64_t sb = which ? a.stride[1][0] : a.stride[0][0];
    const int64_t sh = which ? a.stride[1][1] : a.stride[0][1];
    const int64_t sn = which ? a.stride[1][2] : a.stride[0][2];
    const int tok0 = I * block;
    const int nvalid = I < nb ? min(block, a.N - tok0) : 0;
    const int r = t / TPR, c = t % TPR;
    const __nv_bfloat16* base = X + b * sb + h * sh + int64_t(tok0) * sn + c * 8;

    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int row = r + u * RPP;
        v[u] = (row < nvalid) ? ld_stream16(base + int64_t(row) * sn) : make_uint4(0, 0, 0, 0);
    }
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            acc[2 * e]     += __uint_as_float(w[e] << 16);
            acc[2 * e + 1] += __uint_as_float(w[e] & 0xFFFF0000u);
        }
    }

    __shared__ float red[BPC][RPP][D + 4];
#pragma unroll
    for (int e = 0; e < 8; ++e) red[part][r][c * 8 + e] = acc[e];
    __syncthreads();
    if (t < D && I < nb) {
        float s = 0.f;
#pragma unroll
        for (int rr = 0; rr < RPP; ++rr) s += red[part][rr][t];
        out[((int64_t(b) * a.H + h) * nb + I) * D + t] = s / float(nvalid);
    }
}

// ----------------------------------------------------------------------------------------------
// M2: S[I,J] = scale * <qbar_I, kbar_J>, plain fp32 FFMA (no tensor-core rounding), 64x64 tile per CTA.
// ----------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(256) score_kernel(const float* __restrict__ qbar, const float* __restrict__ kbar,
                                                    float* __restrict__ scores, int nqb, int nkb, float scale) {
    constexpr int TM = 64, TN = 64, TK = 16;
    __shared__ float As[TK][TM + 4];
    __shared__ float Bs[TK][TN + 4];
    const int bh = blockIdx.z;
    const int i0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    const float* A = qbar + int64_t(bh) * nqb * D;
    const float* Bm = kbar + int64_t(bh) * nkb * D;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    // loader mapping: 256 threads move a 64 x 16 slab (float4 per thread)
    const int lrow = threadIdx.x / 4, lcol = (threadIdx.x % 4) * 4;
    for (int k0 = 0; k0 < D; k0 += TK) {
        float4 va = make_float4(0, 0, 0, 0), vb = make_float4(0, 0, 0, 0);
        if (i0 + lrow < nqb) va = *reinterpret_cast<const float4*>(A + int64_t(i0 + lrow) * D + k0 + lcol);
        if (j0 + lrow < nkb) vb = *reinterpret_cast<const float4*>(Bm + int64_t(j0 + lrow) * D + k0 + lcol);
        As[lcol + 0][lrow] = va.x; As[lcol + 1][lrow] = va.y; As[lcol + 2][lrow] = va.z; As[lcol + 3][lrow] = va.w;
        Bs[lcol + 0][lrow] = vb.x; Bs[lcol + 1][lrow] = vb.y; Bs[lcol + 2][lrow] = vb.z; Bs[lcol + 3][lrow] = vb.w;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TK; ++k) {
            float av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) av[i] = As[k][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = Bs[k][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        int I = i0 + ty * 4 + i;
        if (I >= nqb) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int J = j0 + tx * 4 + j;
            if (J < nkb) scores[(int64_t(bh) * nqb + I) * nkb + J] = scale * acc[i][j];
        }
    }
}

// ----------------------------------------------------------------------------------------------
// M3: per-row selection.
// ----------------------------------------------------------------------------------------------
__device__ __forceinline__ bool forced_block(int I, int J, const Geometry& g) {
    if (g.text_dense && g.n_text > 0 && (I * g.bq < g.n_text || J * g.bk < g.n_text)) return true;
    if (g.window >= 0) {
        int q_lo = max(I * g.bq, g.n_text), q_hi = min(g.N, (I + 1) * g.bq) - 1;
        int k_lo = max(J * g.bk, g.n_text), k_hi = min(g.N, (J + 1) * g.bk) - 1;
        if (q_hi >= q_lo && k_hi >= k_lo) {
            int f_lo = max(0, (q_lo - g.n_text) / g.hw - g.window);
            int f_hi = min(g.T - 1, (q_hi - g.n_text) / g.hw + g.window);
            int kf_lo = (k_lo - g.n_text) / g.hw, kf_hi = (k_hi - g.n_text) / g.hw;
            if (kf_lo <= f_hi && kf_hi >= f_lo) return true;
        }
    }
    return false;
}

__device__ __forceinline__ uint32_t ordered_bits(float s) {
    uint32_t u = __float_as_uint(s);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ int topk_count_dev(float ratio, int n) {
    if (n <= 0) return 0;
    double x = __dsub_rn(__dmul_rn(double(ratio), double(n)), 1e-6);
    int k = int(ceil(x));
    return max(1, min(n, k));
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T* scratch /* >= 8 */) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    T t = 0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) t += scratch[w];
    return t;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct SelectArgs {
    const float* scores;   // [B,H,nqb,nkb]
    uint8_t* mask;         // [B,H,nqb,nkb]
    int nqb, nkb, npad, H;
    int mode;
    float keep_ratio, mass;
    int count_includes_forced;
    int k_all;             // top-k count over all nkb blocks (host computed)
    int values_are_mass;   // cumulative-mass mode on non-negative block masses: p = value / sum instead of a softmax
    Geometry g;
};

// One CTA (256 threads) per (b,h,I).  Dynamic shared memory: npad uint64 sort keys + nkb keep bytes
// (+ npad doubles for the cumulative-mass mode).  Cumulative-mass rows of more than 1024 key blocks.
__global__ void __launch_bounds__(256) select_kernel(SelectArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem_raw);
    double* pm = reinterpret_cast<double*>(smem_raw + size_t(a.npad) * 8);                 // only in cumulative-mass mode
    uint8_t* keep = smem_raw + size_t(a.npad) * 8 * (a.mode == CARNATOR_MODE_CUMMASS ? 2 : 1);
    __shared__ double dscratch[8];
    __shared__ int iscratch[8];
    __shared__ float fscratch[8];

    const int I = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int64_t row = ((int64_t(b) * a.H + h) * a.nqb + I) * a.nkb;
    const float* s = a.scores + row;
    const int tid = threadIdx.x, nt = blockDim.x;

    // keys: score-ordered bits, ties -> lower J first.  Always-kept and padding entries get key 0 (sort last).
    int my_forced = 0;
    float my_max = -INFINITY;
    for (int J = tid; J < a.npad; J += nt) {
        unsigned long long key = 0ull;
        if (J < a.nkb) {
            bool f = forced_block(I, J, a.g);
            float v = s[J];
            my_max = fmaxf(my_max, v);
            keep[J] = f ? 1 : 0;
            my_forced += f ? 1 : 0;
            if (!f) key = (static_cast<unsigned long long>(ordered_bits(v)) << 32) | (0xFFFFFFFFu - uint32_t(J));
        }
        keys[J] = key;
    }
    const int nforced = block_sum<int>(my_forced, iscratch);
    const int nfree = a.nkb - nforced;

    // bitonic sort, descending
    for (int k = 2; k <= a.npad; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (int i = tid; i < a.npad; i += nt) {
                int ixj = i ^ j;
                if (ixj > i) {
                    unsigned long long x = keys[i], y = keys[ixj];
                    bool desc = ((i & k) == 0);
                    if (desc ? (x < y) : (x > y)) { keys[i] = y; keys[ixj] = x; }
                }
            }
        }
    }
    __syncthreads();

    int n_admit = 0;
    if (a.mode == CARNATOR_MODE_TOPK) {
        n_admit = a.count_includes_forced ? max(0, a.k_all - nforced) : topk_count_dev(a.keep_ratio, nfree);
        n_admit = min(n_admit, nfree);
    } else {
        // row max (block reduce), softmax mass in fp64
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) my_max = fmaxf(my_max, __shfl_xor_sync(0xffffffffu, my_max, o));
        if ((tid & 31) == 0) fscratch[tid >> 5] = my_max;
        __syncthreads();
        float rmax = fscratch[0];
        for (int w = 1; w < (nt >> 5); ++w) rmax = fmaxf(rmax, fscratch[w]);
        double my_all = 0.0, my_fm = 0.0;
        for (int J = tid; J < a.nkb; J += nt) {
            double e = a.values_are_mass ? double(s[J]) : exp(double(s[J]) - double(rmax));
            my_all += e;
            if (keep[J]) my_fm += e;
        }
        const double total = block_sum<double>(my_all, dscratch);
        const double forced_mass = block_sum<double>(my_fm, dscratch) / total;
        // p of the sorted free blocks, then an exclusive prefix sum in sorted order
        const int per = a.npad / nt > 0 ? a.npad / nt : 1;
        for (int t = tid; t < a.npad; t += nt) {
            double p = 0.0;
            if (t < nfree) {
                int J = int(0xFFFFFFFFu - uint32_t(keys[t] & 0xFFFFFFFFull));
                p = (a.values_are_mass ? double(s[J]) : exp(double(s[J]) - double(rmax))) / total;
            }
            pm[t] = p;
        }
        __syncthreads();
        // chunked scan: thread t owns [t*per, (t+1)*per)
        double chunk = 0.0;
        const int c0 = tid * per;
        if (c0 < a.npad) for (int t = c0; t < c0 + per && t < a.npad; ++t) chunk += pm[t];
        __shared__ double chunk_sums[256];
        chunk_sums[tid] = chunk;
        __syncthreads();
        double before = forced_mass;
        for (int t = 0; t < tid; ++t) before += chunk_sums[t];
        // admitted iff the mass kept before this block is still below the target
        int my_admit = 0;
        const double target = double(a.mass);
        if (c0 < a.npad) {
            double run = before;
            for (int t = c0; t < c0 + per && t < a.npad; ++t) {
                if (t < nfree && run < target) my_admit++;
                run += pm[t];
            }
        }
        n_admit = block_sum<int>(my_admit, iscratch);
    }

    for (int t = tid; t < n_admit; t += nt) {
        int J = int(0xFFFFFFFFu - uint32_t(keys[t] & 0xFFFFFFFFull));
        keep[J] = 1;
    }
    __syncthreads();
    for (int J = tid; J < a.nkb; J += nt) a.mask[row + J] = keep[J];
}

// Selection of one row by one warp, the row's scores at `s` (shared or global memory), without a sort: each lane keeps the
// order-preserving keys of the blocks J = lane, lane + 32, ... in registers and the warp searches the threshold key bit by bit.
//   top-k: the largest T that at least n_admit keys reach; equal keys are admitted in ascending block order.
//   cumulative mass: blocks are admitted in descending order as long as the mass kept before them is below the target, so T
//   is the largest key for which the forced mass plus the mass of the keys >= T reaches the target.  The masses are fp64, as
//   in select_kernel.
template <int NPL>   // keys per lane: nkb <= 32 * NPL
__device__ __forceinline__ void select_row(const SelectArgs& a, const float* s, int I, uint8_t* mask_row) {
    const int lane = threadIdx.x & 31;
    const Geometry& g = a.g;
    const int nkb = a.nkb;
    const int text_cols = (g.text_dense && g.n_text > 0) ? (g.n_text + g.bk - 1) / g.bk : 0;
    // Always-kept key blocks of the frame window: blocks are runs of consecutive tokens, so the blocks that touch frames
    // [f_lo, f_hi] are the interval of blocks that touch tokens [n_text + f_lo hw, n_text + (f_hi + 1) hw).
    int j_lo = 1, j_hi = 0;
    if (g.window >= 0) {
        const int q_lo = max(I * g.bq, g.n_text), q_hi = min(g.N, (I + 1) * g.bq) - 1;
        if (q_hi >= q_lo) {
            const int f_lo = max(0, (q_lo - g.n_text) / g.hw - g.window);
            const int f_hi = min(g.T - 1, (q_hi - g.n_text) / g.hw + g.window);
            j_lo = (g.n_text + f_lo * g.hw) / g.bk;
            j_hi = (min(g.N, g.n_text + (f_hi + 1) * g.hw) - 1) / g.bk;
        }
    }
    if (g.text_dense && g.n_text > 0 && I * g.bq < g.n_text) { j_lo = 0; j_hi = nkb - 1; }

    uint32_t key[NPL], forced = 0u;      // bit q: block q * 32 + lane is always kept (its key is 0 and never competes)
    static_assert(NPL <= 32, "one word of always-kept bits per lane");
    float smax = -INFINITY;
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
        const int J = q * 32 + lane;
        key[q] = 0u;
        if (J < nkb) {
            const float v = s[J];
            smax = fmaxf(smax, v);
            if (J < text_cols || (J >= j_lo && J <= j_hi)) forced |= 1u << q;
            else key[q] = ordered_bits(v);
        }
    }
    const int nforced = __reduce_add_sync(0xffffffffu, __popc(forced));
    const int nfree = nkb - nforced;

    // bits above the first one in which two competing keys differ are the same in every such key
    uint32_t k_or = 0u, k_and = 0xFFFFFFFFu;
#pragma unroll
    for (int q = 0; q < NPL; ++q) { k_or |= key[q]; k_and &= key[q] ? key[q] : 0xFFFFFFFFu; }
    k_or = __reduce_or_sync(0xffffffffu, k_or);
    k_and = __reduce_and_sync(0xffffffffu, k_and);
    const int top = 31 - __clz(int((k_or ^ k_and) | 1u));
    uint32_t T = (top >= 31) ? 0u : (k_and & ~((2u << top) - 1u));

    int need_eq = 0;                     // blocks with key == T that are admitted, lowest index first
    bool any = true;                     // false: nothing is admitted by score
    if (a.mode == CARNATOR_MODE_TOPK) {
        int n_admit = a.count_includes_forced ? max(0, a.k_all - nforced) : topk_count_dev(a.keep_ratio, nfree);
        n_admit = min(n_admit, nfree);
        any = n_admit > 0;
        bool exact = !any;               // a threshold that exactly n_admit keys reach: no tie to break
#pragma unroll 1
        for (int bit = top; bit >= 0 && !exact; --bit) {
            const uint32_t cand = T | (1u << bit);
            int c = 0;
#pragma unroll
            for (int q = 0; q < NPL; ++q) c += (key[q] >= cand) ? 1 : 0;
            c = __reduce_add_sync(0xffffffffu, c);
            if (c >= n_admit) { T = cand; exact = c == n_admit; }
        }
        if (exact) need_eq = nkb;        // every key >= T
        else {
            int gt = 0;
#pragma unroll
            for (int q = 0; q < NPL; ++q) gt += (key[q] > T) ? 1 : 0;
            need_eq = n_admit - __reduce_add_sync(0xffffffffu, gt);
        }
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        double e[NPL], all = 0.0, kept = 0.0;
#pragma unroll
        for (int q = 0; q < NPL; ++q) {
            const int J = q * 32 + lane;
            e[q] = 0.0;
            if (J < nkb) {
                e[q] = a.values_are_mass ? double(s[J]) : exp(double(s[J]) - double(smax));
                all += e[q];
                if ((forced >> q) & 1u) kept += e[q];
            }
        }
        all = warp_sum(all);
        const double inv = 1.0 / all;
        kept = warp_sum(kept) * inv;
#pragma unroll
        for (int q = 0; q < NPL; ++q) e[q] *= inv;
        const double target = double(a.mass);
        // mass kept once the blocks with keys >= c are in; comparisons are written so that a NaN reads as "target reached"
        auto mass_from = [&](uint32_t c) {
            double m = 0.0;
#pragma unroll
            for (int q = 0; q < NPL; ++q) m += (key[q] >= c && key[q] != 0u) ? e[q] : 0.0;
            return kept + warp_sum(m);
        };
        any = nfree > 0 && kept < target;
        if (any) {
            // First on masses in integer units, with the count of the keys above them in the same word, so that one warp sum gives
            // both: as soon as one key is left between the bounds, it is the threshold (about 13 steps for 139 random scores, 32
            // down to the last bit).  The count takes the bits that a row of this form needs, the masses the rest: a row of up to
            // 64 blocks has units of 2^-24, one of 1024 of 2^-20.
            constexpr int kMassBits = NPL <= 2 ? 25 : NPL <= 5 ? 24 : NPL <= 8 ? 23 : NPL <= 20 ? 22 : 21;
            constexpr uint32_t kUnits = 1u << (kMassBits - 1), kMass = (1u << kMassBits) - 1u;
            static_assert((uint64_t(32 * NPL) << kMassBits) + kUnits + 16 * NPL <= 0xFFFFFFFFull && 16 * NPL < int(kUnits), "count and mass of a full row fit the word");
            const uint32_t T0 = T;
            const uint32_t goal = uint32_t(fmax(1.0, ceil((target - kept) * double(kUnits))));
            uint32_t fine[NPL];
#pragma unroll
            for (int q = 0; q < NPL; ++q) fine[q] = key[q] != 0u ? (1u << kMassBits) + uint32_t(e[q] * double(kUnits) + 0.5) : 0u;
            int n_lo = nfree, n_hi = 0;                    // keys >= T, keys above the interval that is left
#pragma unroll 1
            for (int bit = top; bit >= 0; --bit) {
                const uint32_t cand = T | (1u << bit);
                uint32_t m = 0u;
#pragma unroll
                for (int q = 0; q < NPL; ++q) m += key[q] >= cand ? fine[q] : 0u;
                m = __reduce_add_sync(0xffffffffu, m);
                if ((m & kMass) >= goal) { T = cand; n_lo = int(m >> kMassBits); } else n_hi = int(m >> kMassBits);
                if (n_lo - n_hi <= 1) {
                    const uint32_t last = T + ((1u << bit) - 1u);
                    uint32_t k = 0u;
#pragma unroll
                    for (int q = 0; q < NPL; ++q) k = max(k, key[q] <= last ? key[q] : 0u);
                    T = max(T, __reduce_max_sync(0xffffffffu, k));
                    break;
                }
            }
            double over, with;                             // mass kept with the keys > T, with the keys >= T
            auto both_masses = [&] {
                double gt = 0.0, eq = 0.0;
#pragma unroll
                for (int q = 0; q < NPL; ++q) {
                    if (key[q] > T) gt += e[q];
                    if (key[q] == T && key[q] != 0u) eq += e[q];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) { gt += __shfl_xor_sync(0xffffffffu, gt, o); eq += __shfl_xor_sync(0xffffffffu, eq, o); }
                over = kept + gt; with = kept + (gt + eq);
            };
            both_masses();
            // The outcome is checked in fp64.  Rounded masses can miss the threshold by a few keys, most often where the target lies
            // among many small ones (1000 blocks, target 0.999: half of the rows), so the keys next to it are tried in turn.  With
            // the search on the fp64 masses (up to 32 of their sums) for every such row, 16 heads of 1000 blocks, D = 64, took
            // 422 us at 0.999 and 321 at 0.5; now 332 and 319.
            bool all_in = false;                           // no key is left below T, and the target is still out of reach
            bool wrong = !(over < target) || with < target;
#pragma unroll 1
            for (int hop = 0; hop < 8 && wrong; ++hop) {
                const bool down = with < target;
                uint32_t k = 0u;                           // next key below T, or the complement of the next one above
                if (down) {
#pragma unroll
                    for (int q = 0; q < NPL; ++q) k = max(k, key[q] < T ? key[q] : 0u);
                } else {
#pragma unroll
                    for (int q = 0; q < NPL; ++q) k = max(k, key[q] > T ? ~key[q] : 0u);
                }
                k = __reduce_max_sync(0xffffffffu, k);
                if (k == 0u) { all_in = down; break; }     // (none above: masses that are NaN)
                T = down ? k : ~k;
                both_masses();
                wrong = !(over < target) || with < target;
            }
            if (wrong && !all_in) {                        // the same search on the masses themselves
                T = T0;
                for (int bit = top; bit >= 0; --bit)
                    if (!(mass_from(T | (1u << bit)) < target)) T |= 1u << bit;
                both_masses();
            }
            if (with < target) need_eq = nkb;                      // even all of them fall short: all are admitted (T is at most the lowest key)
            else {
                // the blocks with the threshold's key are admitted one by one, as long as the mass before them is short
                int ties = 0;
                double p = 0.0;
#pragma unroll
                for (int q = 0; q < NPL; ++q) if (key[q] == T && key[q] != 0u) { ++ties; p = e[q]; }
                ties = __reduce_add_sync(0xffffffffu, ties);
                need_eq = 1;
                if (ties > 1) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) p = fmax(p, __shfl_xor_sync(0xffffffffu, p, o));
                    for (double run = over + p; run < target && need_eq < ties; run += p) ++need_eq;
                }
            }
        }
    }
    int seen = 0;
#pragma unroll
    for (int q = 0; q < NPL; ++q) {
        const int J = q * 32 + lane;
        const bool eq = any && key[q] == T && key[q] != 0u;
        const unsigned bal = __ballot_sync(0xffffffffu, eq);
        const bool keep = ((forced >> q) & 1u) || (any && key[q] > T) || (eq && seen + __popc(bal & ((1u << lane) - 1u)) < need_eq);
        seen += __popc(bal);
        if (J < nkb) mask_row[J] = keep ? 1 : 0;
    }
}

// Rows whose scores lie in global memory (the exact builder's masses): one warp per (b,h,I).
template <int NPL>
__global__ void __launch_bounds__(256) select_rows_kernel(SelectArgs a, int rows) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp >= rows) return;
    select_row<NPL>(a, a.scores + int64_t(warp) * a.nkb, warp % a.nqb, a.mask + int64_t(warp) * a.nkb);
}

// M2 + M3 for layers of up to 1024 key blocks: a CTA takes R query blocks of a head, computes their scores in fp32 (the
// same sequence of FFMAs over the head dimension as score_kernel) into shared memory, and each of its R warps selects one
// row there.  A thread takes RG rows of one key block, so that a key-block mean read from shared memory serves RG products and a
// query-block mean (one address for the warp) 32: the product is bound by those reads.  The key-block means come a tile of
// key blocks at a time, 32 or 64 elements of the head dimension per step, through two cp.async buffers; rows of 36 or 68 floats
// keep the 16-byte reads free of bank conflicts.  The tile is what a row of this form has, up to 256.  What this saves against score_kernel and
// a selection kernel is a launch and the scores' way through memory.  Whole calls, against those: 12 heads, 61 blocks,
// top-k 34.1 -> 18.5 us; 48 heads, 139 blocks, cumulative mass 209 -> 53.3 us (the sort of every row took 153; tiles of 128 key
// blocks with four rows a thread and a search down to the last bit 59.7: this kernel alone 31.2 -> 24.6 us).
template <int D, int R, int NPL>
struct ScoreSelect {
    // key blocks per tile.  Eight rows of 129 to 160 key blocks: two tiles of 128, whose threads take four rows, are done sooner than one of
    // 160 while an SM has one such CTA (9 heads of 139 blocks, D = 128, cumulative mass, 20.7 and 26.2 us; 24 heads 41.9 and 37.9).
    // Sixteen rows: one tile of 160, of whose 512 threads 320 take eight rows each (48 heads 63.5 us, two tiles of 128 66.7).
    static constexpr int kKeys = R == 8 && NPL == 5 ? 128 : (32 * NPL < 256 ? 32 * NPL : 256);
    // Rows per thread.  Four also where a row has up to 64 key blocks, although half of the threads are then left out of the product: with two
    // (GPU time of whole builds) 12 heads of 61 blocks, D = 128, top-k, took 16.1 us against 15.3, 24 of 26 blocks 12.3 against 11.9, and 4
    // heads of 13 blocks 5.8 against 5.9; only D = 64 with up to 26 blocks gained (24 heads of 13 blocks, cumulative mass, 8.9 against 9.7).
    static constexpr int RG = kKeys <= 128 ? 4 : 8;
    static constexpr int kSlab = kKeys <= 128 ? 64 : 32, kLd = kSlab + 4;    // elements of the head dimension per step
    // CTAs that an SM is to hold, where that has to be said (0: the compiler's choice).  It has given sixteen rows of 161 to 256 blocks 64
    // registers or 76, and with 76 an SM holds one CTA instead of two: 48 heads of 256 blocks, D = 64, mass 0.9, 88.5 and 101.2 us.
    static constexpr int kCtas = R == 16 && NPL == 8 ? 2 : 0;
    static_assert(kKeys * (R / RG) <= 32 * R && R % RG == 0, "a thread per key block and row group");
    static constexpr size_t smem(int nkb) { return size_t(2 * kKeys * kLd + R * D) * 4 + size_t(R) * ((nkb + 3) & ~3) * 4; }
};
__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
template <int D, int R, int NPL>
__global__ void __launch_bounds__(R * 32, ScoreSelect<D, R, NPL>::kCtas) score_select_kernel(const float* __restrict__ qbar, const float* __restrict__ kbar,
                                                              float* __restrict__ scores_out, float scale, SelectArgs a) {
    using S = ScoreSelect<D, R, NPL>;
    extern __shared__ __align__(16) float ssm[];
    constexpr int NT = R * 32, RG = S::RG, kKeys = S::kKeys, kLd = S::kLd, kSlab = S::kSlab, kSlabs = D / kSlab;
    float* const sK = ssm;                                             // [2][kKeys][kLd]
    float* const sQ = sK + 2 * kKeys * kLd;                            // [R][D]
    float* const sS = sQ + R * D;                                      // [R][nkb_pad]
    const int nkb = a.nkb, nkb_pad = (nkb + 3) & ~3;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int I0 = blockIdx.x * R;
    const int64_t bh = int64_t(blockIdx.z) * a.H + blockIdx.y;
    const float* K = kbar + bh * nkb * D;
    const int steps = ((nkb + kKeys - 1) / kKeys) * kSlabs;
    auto load = [&](int st) {
        const int j0 = (st / kSlabs) * kKeys, d0 = (st % kSlabs) * kSlab, n = min(kKeys, nkb - j0);
        for (int i = tid; i < n * (kSlab / 4); i += NT) {
            const int j = i / (kSlab / 4), c = (i % (kSlab / 4)) * 4;
            cp16(sK + ((st & 1) * kKeys + j) * kLd + c, K + int64_t(j0 + j) * D + d0 + c, true);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    grid_wait();                                                       // the means are complete
    for (int i = tid; i < R * (D / 4); i += NT) {
        const int r = i / (D / 4), c = (i % (D / 4)) * 4;
        cp16(sQ + r * D + c, qbar + (bh * a.nqb + min(I0 + r, a.nqb - 1)) * D + c, true);
    }
    load(0);
    float acc[RG];
    const int key = tid % kKeys, r0 = (tid / kKeys) * RG;              // threads past the last row group only load and select
    for (int st = 0; st < steps; ++st) {
        if (st + 1 < steps) { load(st + 1); asm volatile("cp.async.wait_group 1;" ::: "memory"); }
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const int d0 = (st % kSlabs) * kSlab, J = (st / kSlabs) * kKeys + key;
        if (r0 < R && J < nkb) {
            if (d0 == 0) {
#pragma unroll
                for (int r = 0; r < RG; ++r) acc[r] = 0.f;
            }
            const float* kr = sK + ((st & 1) * kKeys + key) * kLd;
            const float* qr = sQ + r0 * D + d0;
#pragma unroll 4
            for (int d = 0; d < kSlab; d += 4) {
                const float4 k4 = *reinterpret_cast<const float4*>(kr + d);
#pragma unroll
                for (int r = 0; r < RG; ++r) {
                    const float4 q4 = *reinterpret_cast<const float4*>(qr + r * D + d);
                    acc[r] = fmaf(q4.x, k4.x, acc[r]); acc[r] = fmaf(q4.y, k4.y, acc[r]);
                    acc[r] = fmaf(q4.z, k4.z, acc[r]); acc[r] = fmaf(q4.w, k4.w, acc[r]);
                }
            }
            if (d0 + kSlab == D) {
#pragma unroll
                for (int r = 0; r < RG; ++r) sS[(r0 + r) * nkb_pad + J] = scale * acc[r];
            }
        }
        __syncthreads();
    }
    const int I = I0 + warp;
    if (I >= a.nqb) return;
    const float* row = sS + warp * nkb_pad;
    if (scores_out)
        for (int J = lane; J < nkb; J += 32) scores_out[(bh * a.nqb + I) * nkb + J] = row[J];
    select_row<NPL>(a, row, I, a.mask + (bh * a.nqb + I) * nkb);
}

// Top-k rows of more than 1024 key blocks.  One warp per (b,h,I).  Each lane keeps the order-preserving keys of the
// blocks J = lane, lane+32, ... in registers; the k-th largest key is found bit by bit (largest T with
// #(key >= T) >= k), then equal keys are admitted in ascending block order until k is reached.
template <int NPL>   // keys per lane: nkb <= 32 * NPL
__global__ void __launch_bounds__(256) select_topk_kernel(SelectArgs a, int rows) {
    // frame span of every key block, computed once per CTA (two integer divisions per block)
    extern __shared__ int2 kframes[];
    const Geometry g = a.g;
    for (int J = threadIdx.x; J < a.nkb; J += blockDim.x) {
        const int k_lo = max(J * g.bk, g.n_text), k_hi = min(g.N, (J + 1) * g.bk) - 1;
        kframes[J] = (k_hi >= k_lo) ? make_int2((k_lo - g.n_text) / g.hw, (k_hi - g.n_text) / g.hw) : make_int2(1, 0);
    }
    __syncthreads();
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= rows) return;
    const int I = warp % a.nqb;
    const int64_t row = int64_t(warp) * a.nkb;
    const float* s = a.scores + row;

    // the query block's side of the always-kept rule
    const bool text_row = g.text_dense && g.n_text > 0 && I * g.bq < g.n_text;
    const int text_cols = (g.text_dense && g.n_text > 0) ? (g.n_text + g.bk - 1) / g.bk : 0;   // key blocks holding text
    int f_lo = 0, f_hi = 0;
    bool has_window = false;                   // the query block holds video tokens and a window is asked for
    if (g.window >= 0) {
        const int q_lo = max(I * g.bq, g.n_text), q_hi = min(g.N, (I + 1) * g.bq) - 1;
        if (q_hi >= q_lo) {
            has_window = true;
            f_lo = max(0, (q_lo - g.n_text) / g.hw - g.window);
            f_hi = min(g.T - 1, (q_hi - g.n_text) / g.hw + g.window);
        }
    }

    uint32_t key[NPL];
    uint32_t forced_bits[(NPL + 31) / 32];
#pragma unroll
    for (int w = 0; w < (NPL + 31) / 32; ++w) forced_bits[w] = 0u;
    int my_forced = 0;
#pragma unroll
    for (int t = 0; t < NPL; ++t) {
        const int J = t * 32 + lane;
        uint32_t k = 0u;                       // always-kept and out-of-range entries never compete
        if (J < a.nkb) {
            const int2 kf = kframes[J];
            const bool forced = text_row || J < text_cols || (has_window && kf.x <= kf.y && kf.x <= f_hi && kf.y >= f_lo);
            if (forced) { forced_bits[t >> 5] |= 1u << (t & 31); ++my_forced; }
            else k = ordered_bits(s[J]);
        }
        key[t] = k;
    }
    int nforced = my_forced;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nforced += __shfl_xor_sync(0xffffffffu, nforced, o);
    const int nfree = a.nkb - nforced;
    int n_admit = a.count_includes_forced ? max(0, a.k_all - nforced) : topk_count_dev(a.keep_ratio, nfree);
    n_admit = min(n_admit, nfree);

    uint32_t T = 0xFFFFFFFFu;                  // nothing admitted by score
    int need_eq = 0;
    if (n_admit > 0) {
        T = 0u;
        for (int bit = 31; bit >= 0; --bit) {
            const uint32_t cand = T | (1u << bit);
            int c = 0;
#pragma unroll
            for (int t = 0; t < NPL; ++t) c += (key[t] >= cand) ? 1 : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            if (c >= n_admit) T = cand;
        }
        int gt = 0;
#pragma unroll
        for (int t = 0; t < NPL; ++t) gt += (key[t] > T) ? 1 : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gt += __shfl_xor_sync(0xffffffffu, gt, o);
        need_eq = n_admit - gt;                // >= 1 blocks with key == T, lowest block index first
    }
    int seen_eq = 0;
#pragma unroll
    for (int t = 0; t < NPL; ++t) {
        const int J = t * 32 + lane;
        const bool eq = (n_admit > 0) && key[t] == T;
        const unsigned bal = __ballot_sync(0xffffffffu, eq);
        const int rank = seen_eq + __popc(bal & ((1u << lane) - 1u));
        seen_eq += __popc(bal);
        const bool keep = ((forced_bits[t >> 5] >> (t & 31)) & 1u) || (n_admit > 0 && key[t] > T) || (eq && rank < need_eq);
        if (J < a.nkb) a.mask[row + J] = keep ? 1 : 0;
    }
}


}  // namespace carnator
