// Work items handed out dynamically by cluster launch control, and a warp's look at a head's retained list for an item of 128
// consecutive queries.  Both are what the load warps of the prefill kernels (prefill_tc.cu, prefill_tc_pair.cu) and of the backward
// (bwd_tc.cu) do at an item's start.
#pragma once
#include "tc_common.cuh"

namespace lte {
namespace tc {

// The grid has a block per item, but a block that has run out of work takes over the next block that has not started instead of
// leaving, so items are handed out in order to whoever is free.
// Asks for a block of this grid that has not started (the answer, 16 bytes, arrives on the barrier).
__device__ __forceinline__ void ask_for_block(uint32_t answer, uint32_t bar) {
    mbar_expect_tx(bar, 16);
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(answer), "r"(bar) : "memory");
}
__device__ __forceinline__ int block_from(uint32_t answer) {   // its index, or -1
    uint32_t ok, x;
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b128 h;\n\tld.shared.b128 h, [%2];\n\tclusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\tmov.u32 %1, 0;\n\t@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, _, _, _}, h;\n\t}"
                 : "=r"(ok), "=r"(x) : "r"(answer) : "memory");
    return ok ? (int)x : -1;
}
// The items of one block (used by one whole warp): the block's own, then what its requests bring.  A request reserves the item it
// brings, so it is made only kAskTiles tiles before the current item's loads end: blocks that are behind would otherwise sit on
// items that others could have started.  (Prefill at d = 64, asking at an item's start and searching the list step by step: 64 heads
// x 4,096, W = R = 128, the whole call 72.2 us, so 71.3; eight chunks of 512 114.3 and 113.6; 1,024 x 4,096, W = 768 2,141 and 2,148.)
constexpr int kAskTiles = 4;
struct ItemQueue {
    uint32_t answer, bar, asked = 0;
    int lane;
    __device__ __forceinline__ ItemQueue(uint32_t answer_, uint32_t bar_, int lane_) : answer(answer_), bar(bar_), lane(lane_) {}
    __device__ __forceinline__ void ask() {
        fence_proxy_async();                                   // the last answer has been read before this one is written
        __syncwarp();
        if (lane == 0) ask_for_block(answer, bar);
        ++asked;
    }
    // the answer to the last request; -1: there is no further item, or the launch is lost (the wait gave up)
    __device__ __forceinline__ int take(int code, StatusWord* st) {
        bool ok = false;
        for (uint32_t i = 0; i < kSpinLimit && !ok; ++i) {
            ok = mbar_try_wait(bar, (asked - 1) & 1);
            if (!ok && (i & 1023u) == 1023u && launch_aborted(st)) break;
        }
        if (!ok) wait_gave_up(st, code);
        return __all_sync(0xffffffffu, ok) ? block_from(answer) : -1;
    }
};

// Row x (0 .. 127) sees before[x / 32] list entries and those of bits[x / 32] below bit x % 32; `all`: what the last row sees.
struct ListView { uint32_t before[4], bits[4]; int all; };
// Rows 0 .. last see the entries of the ascending list id[0, n) up to lim0, .., lim0 + last (whole warp; R: the list's capacity, n is
// read here).  Two dependent loads for R <= 1024: probes at fixed places beside the count, then the rest of the search and the
// entries between the limits in one go.
__device__ __forceinline__ ListView view_list(const int32_t* id, const int32_t* cnt, int R, int lim0, int last, int lane)
{
    ListView f;
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    int lo = 0, n = 0;
    if (R > 0) {
        int step = (R + 31) >> 5;
        const int probe = id[min((lane + 1) * step - 1, R - 1)];
        n = *cnt;
        const int m = lim0 + last < 0 ? 0 : n;                 // nothing is visible before position 0
        lo = min(m, step * __popc(__ballot_sync(0xffffffffu, (lane + 1) * step - 1 < m && probe <= lim0)));   // entries before lo are <= lim0
        while (step > 32) {                                    // the first entry > lim0 is within `step` of lo
            const int sub = (step + 31) >> 5, at = lo + (lane + 1) * sub - 1;
            lo = min(m, lo + sub * __popc(__ballot_sync(0xffffffffu, (lane + 1) * sub - 1 < step && at < m && id[min(at, R - 1)] <= lim0)));
            step = sub;
        }
        int v[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) v[u] = lo + u * 32 + lane < m ? id[lo + u * 32 + lane] : 0x7fffffff;
        lo += __popc(__ballot_sync(0xffffffffu, v[0] <= lim0));
#pragma unroll
        for (int u = 0; u < 5; ++u) {                          // at most 127 entries lie in (lim0, lim0 + 127]
            const int x = v[u] == 0x7fffffff ? 128 : v[u] - lim0 - 1;
            const uint32_t bit = x >= 0 && x < last ? 1u << (x & 31) : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] |= (x >> 5) == k ? bit : 0u;
        }
    }
    uint32_t sum = (uint32_t)lo;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        f.bits[k] = __reduce_or_sync(0xffffffffu, w[k]);
        f.before[k] = sum;
        sum += __popc(f.bits[k]);
    }
    f.all = (int)sum;
    return f;
}

}  // namespace tc
}  // namespace lte
