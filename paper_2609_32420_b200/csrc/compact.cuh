// C1: block mask (+ recompute rows) -> per-row ascending key-block lists, counts, and a per-head
// execution order (longest list first), so the attention kernel never fetches an empty tile.
// Paper: Appendix "Reuse-Scope Implementation Details" (connectivity is restricted before sparse
// execution) and "Latency Accounting" (in-loop mask / index lookups).
#pragma once
#include "common.cuh"

namespace carnator {

constexpr int kCompactThreads = 1024;         // at most; 512 or 256 where there are many heads
constexpr int kCompactPairsPerCta = 4096;
constexpr int kMaxQueryBlocks = 12000;       // a head's sort keys in shared memory; also keeps key and index in one word

struct CompactArgs {
    const uint8_t *mask, *recompute, *active_q, *context_k;     // the last three may be null
    int32_t *counts, *lists, *order;
    WsHeader* hdr;
    int H, nqb, nkb, ctas;                   // ctas: CTAs (one cluster) per head
};

// Lists, counts and order of one head by one cluster: a warp per row compacts with ballots, 128 bytes of the mask in flight,
// then the cluster meets and every CTA ranks its share of the rows.  The cluster has 1 to 8 CTAs by the size of the head's
// mask (4 K block pairs per CTA) and by the number of heads (see the launch): one kernel where a clear and two kernels ran.  2
// heads of 16 rows: whole attention call 24.8 -> 21.5 us; 12 heads of 256 rows, region form: 12.1 us and a clear -> 10.2 us.
// Two CTAs of 1024 threads have to fit an SM: with the next 128 bytes fetched ahead (38 registers and more) 40 heads of 592
// rows took 46 to 61 us instead of 41.
//   order: longest list first (stable), so that the longest CTAs of the attention kernel start first.
//   kPairs (64-token query blocks): consecutive entries 2x, 2x+1 share a tile, so rows with like lists should meet: rows that
//   list everything first, then the others, each by index (neighbours in the video), then the empty and skipped ones; the
//   pairs are then put longest first.
template <bool kPairs>
__global__ void __launch_bounds__(kCompactThreads, 2) compact_order_kernel(CompactArgs a) {
    extern __shared__ __align__(16) int32_t csm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bh = blockIdx.x / a.ctas, rank_cta = blockIdx.x % a.ctas;
    const int nqb = a.nqb, nkb = a.nkb, b = bh / a.H;
    const int share = (nqb + a.ctas - 1) / a.ctas, i_lo = min(nqb, rank_cta * share), i_hi = min(nqb, i_lo + share);
    grid_launch_dependents();
    grid_wait();
    if (blockIdx.x == 0 && tid < int(sizeof(WsHeader) / 4)) reinterpret_cast<int32_t*>(a.hdr)[tid] = 0;
    const uint8_t* ctx = a.context_k ? a.context_k + int64_t(b) * nkb : nullptr;
    unsigned active = ~0u, recomp = 0u;          // flags of this warp's next 32 rows, fetched together
    const int nt = blockDim.x, nw = nt >> 5;
    for (int I = i_lo + warp, n_row = 0; I < i_hi; I += nw, ++n_row) {
        const int64_t row = int64_t(bh) * nqb + I;
        if ((n_row & 31) == 0) {
            const int mine = I + lane * nw;
            const int64_t at = int64_t(b) * nqb + mine;
            const bool f_act = !a.active_q || (mine < i_hi && a.active_q[at] != 0);
            const bool f_rec = a.recompute && mine < i_hi && a.recompute[at] != 0;
            active = __ballot_sync(0xffffffffu, f_act);
            recomp = __ballot_sync(0xffffffffu, f_rec);
        }
        // region-restricted form: a query block that is not active is skipped altogether (count -1: the attention
        // kernels leave its output rows untouched); listed key blocks must also be context blocks
        if (!((active >> (n_row & 31)) & 1u)) {
            if (lane == 0) a.counts[row] = -1;
            continue;
        }
        const bool dense = (recomp >> (n_row & 31)) & 1u;
        const uint8_t* m = a.mask + row * nkb;
        int32_t* out = a.lists + row * nkb;
        int n = 0;
        for (int J0 = 0; J0 < nkb; J0 += 128) {
            bool on[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int J = J0 + u * 32 + lane;
                on[u] = J < nkb && (dense || m[J] != 0) && (ctx == nullptr || ctx[J] != 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned bal = __ballot_sync(0xffffffffu, on[u]);
                if (on[u]) out[n + __popc(bal & ((1u << lane) - 1u))] = J0 + u * 32 + lane;
                n += __popc(bal);
            }
        }
        if (lane == 0) a.counts[row] = n;
    }
    if (a.ctas > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else __syncthreads();

    // sort keys, larger first: value in the high bits, lower index wins among equals (16384 > kMaxQueryBlocks)
    const int nq4 = (nqb + 3) & ~3;
    int32_t* const cnt = csm;                                          // counts
    int32_t* const key = csm + nq4;                                    // sort keys
    auto rank_of = [&](int k, int n4) {                                // how many keys are larger
        int r = 0;
        const int4* p = reinterpret_cast<const int4*>(key);
        for (int j = 0; j < n4 / 4; ++j) {
            const int4 v = p[j];
            r += (v.x > k) + (v.y > k) + (v.z > k) + (v.w > k);
        }
        return r;
    };
    for (int i = tid; i < nq4; i += nt) {
        const int c = i < nqb ? __ldcg(a.counts + int64_t(bh) * nqb + i) : 0;
        cnt[i] = c;
        if (!kPairs) key[i] = i < nqb ? c * 16384 + 16383 - i : INT32_MIN;
    }
    __syncthreads();
    int32_t* order = a.order + int64_t(bh) * nqb;
    if (!kPairs) {
        for (int i = i_lo + tid; i < i_hi; i += nt) order[rank_of(key[i], nq4)] = i;
        return;
    }
    uint16_t* const at = reinterpret_cast<uint16_t*>(csm + 2 * nq4);   // rows in pairing order
    {   // Three classes, each by index: a thread counts those of its run of rows, a scan over the threads places them.  Ranked
        // against all rows instead, in every CTA, 1 head of 12000 rows took 6.44 ms against 4.51, 12 heads of 512 rows 27.4 us against 19.3.
        __shared__ uint32_t warp_sum[kCompactThreads / 32];
        const int run = (nqb + nt - 1) / nt, r0 = min(nqb, tid * run), r1 = min(nqb, r0 + run);
        auto bump = [&](int c) -> uint32_t { return c == nkb ? 1u << 16 : (c > 0 ? 1u : 0u); };      // full rows | other listed rows
        uint32_t mine = 0u;
        for (int i = r0; i < r1; ++i) mine += bump(cnt[i]);
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        uint32_t before = incl - mine, total = 0u;
        for (int w = 0; w < nw; ++w) {
            if (w < warp) before += warp_sum[w];
            total += warp_sum[w];
        }
        const int full = int(total >> 16), listed = int(total & 0xFFFFu);
        int f = int(before >> 16), l = full + int(before & 0xFFFFu), e = full + listed + r0 - f - int(before & 0xFFFFu);
        for (int i = r0; i < r1; ++i) {
            const uint32_t b = bump(cnt[i]);
            at[b >> 16 ? f++ : (b ? l++ : e++)] = uint16_t(i);
        }
    }
    __syncthreads();
    const int np = (nqb + 1) / 2, np4 = (np + 3) & ~3;
    for (int p = tid; p < np4; p += nt) {
        // a row left without a partner stays last: entries 2x, 2x + 1 have to remain pairs
        const int w = p >= np ? 0 : (2 * p + 1 < nqb ? max(cnt[at[2 * p]], cnt[at[2 * p + 1]]) : -2);
        key[p] = p < np ? w * 16384 + 16383 - p : INT32_MIN;
    }
    __syncthreads();
    for (int p = rank_cta * nt + tid; p < np; p += a.ctas * nt) {
        const int r = rank_of(key[p], np4);
        order[2 * r] = at[2 * p];
        if (2 * p + 1 < nqb) order[2 * r + 1] = at[2 * p + 1];
    }
}
inline size_t compact_smem(int nqb, bool pairs) { return size_t((nqb + 3) & ~3) * (pairs ? 10 : 8); }

// Listed tiles of a compacted workspace, into its header (on request only: the sum over all heads is no business of the
// compaction).  `counts` is aligned to 256 bytes: four counts a load, four loads in flight.
__global__ void __launch_bounds__(1024) count_tiles_kernel(const int32_t* __restrict__ counts, int64_t rows, WsHeader* hdr) {
    __shared__ unsigned long long part[32];
    unsigned long long n = 0;
    const int4* four = reinterpret_cast<const int4*>(counts);
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < rows / 4; i += 1024) {
        const int4 c = four[i];
        n += (unsigned long long)max(c.x, 0) + max(c.y, 0) + max(c.z, 0) + max(c.w, 0);
    }
    if (threadIdx.x < (rows & 3)) n += (unsigned long long)max(counts[(rows & ~int64_t(3)) + threadIdx.x], 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 32; ++w) n += part[w];
        hdr->tiles = n;
    }
}

}  // namespace carnator
