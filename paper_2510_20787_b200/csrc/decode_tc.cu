// Decode step on the tensor cores (bf16, d = 64, W + R <= 256): Fig. 3's cache, Section 3.1.3's decoding paragraph.
//
// The per-head cache block stores its key and value rows with the 128-byte swizzle, so that once cp.async.bulk has
// copied the block into shared memory it is a valid tcgen05 operand as it stands:
//   logits   S^T[256 keys] = K[256 x 64] q[64]:  two MMAs-groups M = 128 (keys), N = 16 (row 0 of B is q, the rest 0),
//            K = 64; the logit of key j lands in TMEM lane j mod 128, and the thread owning that lane masks it
//            (ring / pool validity after the replacement decision), takes part in the block max / sum and writes
//            p_j = exp(s_j - max) as bf16 into a small B tile;
//   output   O[64] = sum_j p_j V_j:  one MMA chain M = 128 = two stacked halves of 64 channels (A = the value block as
//            MN-major operand: group 0 = rows 0..127, group 1 = rows 128..255), N = 16 (B row 0 = p[0..127],
//            row 1 = p[128..255]), K = 128 keys; channel c is D[c][0] + D[64+c][1].
// Persistent CTAs walk consecutive heads; a control lane issues the bulk copies (next head's keys as soon as this
// head's logits are taken, next values after the PV chain, the logits and positions a head ahead) and every tcgen05.mma; the replacement
// decision, the scorer tap sums and the write-back stay as in the ALU kernel.  Every wait is bounded.
//
// Bound by memory only as far as the chain of a head (copy, logits, softmax, output: some 4 us) is short enough for the CTAs that fit
// on an SM to keep it busy.  So only rows that exist are copied, the worst pool entry and the maximum are found by warp-wide
// reductions of one instruction, the next head's inputs are asked for under this head's output, and one barrier per head is left.
// Measured (B200, a step in a CUDA graph of steps, before -> now): 2,048 heads x 256 rows 29.1 -> 26.0 us (137 MB: 5.3 TB/s; 28.3 with
// R = 196, of which two blocks fit an SM), 1,024 x 256 15.0 -> 12.8, 4,096 x 128 53.8 -> 27.6, 16 x 256 4.9 -> 4.4.  Asking for the next head in L2 ahead: 31.2 -> 33.3; two stages of 128
// rows each instead of five CTAs: 37.9.
#include <type_traits>

#include "tc_common.cuh"

namespace lte {

__device__ StatusWord g_decode_tc_status = LTE_STATUS_INIT;

namespace {

using namespace tc;
// NC compute threads (thread j owns cache row j): 256, or 128 where there are no more rows.  Half the threads and half the shared memory
// then let five CTAs share an SM instead of three, which counts because every head costs its CTA a chain of some 4 us.
template <int NC> constexpr int kThreads = NC + 32;            // + control warp
template <int NC> constexpr int kPerSm = NC == 256 ? 3 : 5;
constexpr int D = 64;
constexpr uint32_t TMEM_COLS = 64;         // S^T: [0,16) keys 0..127, [16,32) keys 128..255;  O halves: [32,48)

__device__ __forceinline__ void dwait(uint32_t bar, uint32_t parity, int code) { mbar_wait_s(bar, parity, code, &g_decode_tc_status); }
__device__ __forceinline__ float redux_max(float x) {
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
// Loads that stay where they are written (the compiler would move them to their first use, behind the waits).
__device__ __forceinline__ uint32_t load32(const void* p) {
    uint32_t x;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ uint4 load128(const void* p) {
    uint4 x;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ float2 bf16_pair(uint32_t x) { return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
template <int NC> __device__ __forceinline__ void csync() { asm volatile("bar.sync 1, %0;" ::"n"(NC) : "memory"); }
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

struct Plan { uint32_t off_v, off_k, off_tail, tail_bytes, off_q, off_p, off_bar, total; };
template <int NC> __host__ __device__ inline Plan plan_of(const CacheLayout& L) {
    Plan P;
    // V block [NC][64] bf16, then K block: the output product reads 256 rows from the value block on (its upper half is used with
    // NC = 256 only), which have to be there
    P.off_v = 0;
    P.off_k = NC * 128;
    P.off_q = 2 * NC * 128;                            // B operand of the logits: [16][64] bf16 (2 KB)
    P.off_p = P.off_q + 2048;                          // B operand of the PV chain: [2][16][64] bf16 (4 KB)
    P.off_tail = P.off_p + 4096;                       // two tail buffers
    P.tail_bytes = (uint32_t)(L.stride - L.off_z);
    P.off_bar = (P.off_tail + 2 * P.tail_bytes + 15) & ~15u;
    P.total = P.off_bar + 128;
    return P;
}
// The most a plan takes: NC rows, of which one is the ring's and the others the pool's (a logit each, a position for those).
template <int NC> constexpr int kMostSmem = 2 * NC * 128 + 2048 + 4096 + 2 * ((4 * NC + 4 * (NC - 1) + 16 + 255) / 256 * 256) + 128;

template <int NC, bool TURN>
__global__ void __launch_bounds__(kThreads<NC>, kPerSm<NC>) decode_tc_kernel(unsigned char* __restrict__ cache, CacheLayout L,
                                                         const __nv_bfloat16* __restrict__ q1,
                                                         const __nv_bfloat16* __restrict__ k1,
                                                         const __nv_bfloat16* __restrict__ v1,
                                                         __nv_bfloat16* __restrict__ o1, float* __restrict__ lse1,
                                                         const float* __restrict__ cw, const float* __restrict__ cbias,
                                                         int BH, int H, int W, int R, int sink, int K,
                                                         float zthr, float scale)
{
    extern __shared__ __align__(1024) unsigned char dsm[];
    constexpr int NW = NC / 32, NTHR = kThreads<NC>, TAPS = (kMaxTaps + NW - 1) / NW;
    const Plan P = plan_of<NC>(L);
    const uint32_t base = smem_u32(dsm);
    if ((base & 1023u) != 0) { if (threadIdx.x == 0) atomicExch(&g_decode_tc_status.code, 9); return; }
    const uint32_t sK = base + P.off_k, sV = base + P.off_v, sT = base + P.off_tail, sQ = base + P.off_q, sP = base + P.off_p;
    const uint32_t bar_k = base + P.off_bar, bar_v = bar_k + 8, bar_t0 = bar_k + 16;     // bar_t0, bar_t0 + 8
    const uint32_t bar_q = bar_k + 32, bar_s = bar_k + 40, bar_p = bar_k + 48, bar_o = bar_k + 56, tmem_slot = bar_k + 64;
    volatile uint32_t* tmem_slot_gen = reinterpret_cast<volatile uint32_t*>(dsm + P.off_bar + 64);
    __shared__ float s_part[NW], s_sum[NW], s_tap[2][kMaxTaps], s_o[D];

    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rows = W + R, half = K / 2;
    const int bh_begin = (int)((long long)blockIdx.x * BH / gridDim.x), bh_end = (int)((long long)(blockIdx.x + 1) * BH / gridDim.x);
    const uint32_t blk_bytes = rows * 128;                     // only the rows that there are

    if (tid == 0) {
        mbar_init(bar_k, 1); mbar_init(bar_v, 1); mbar_init(bar_t0, 1); mbar_init(bar_t0 + 8, 1);
        mbar_init(bar_q, 8); mbar_init(bar_s, 1); mbar_init(bar_p, NC); mbar_init(bar_o, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the two small B tiles start as zeros (only row 0 of the q tile and rows 0, 1 of the p tile are ever written)
    for (int e = tid; e < (2048 + 4096) / 16; e += NTHR)
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sQ + e * 16), "r"(0u) : "memory");
    // rows that there are not are zeros (their logits are masked, but the values enter the product with weight 0)
    for (int e = tid + rows * 8; e < NC * 8; e += NTHR) {
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sK + e * 16), "r"(0u) : "memory");
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sV + e * 16), "r"(0u) : "memory");
    }
    if (wid == NW) tmem_alloc(tmem_slot, TMEM_COLS);
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_gen;
    // (asked for in L2 while the step before may still be at work, so that the copies below wait less for the direction)
    const int32_t* counter = reinterpret_cast<const int32_t*>(cache + L.header + (size_t)bh_begin * L.stride + L.off_meta);
    if (TURN && tid == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(counter));
    pdl_launch_dependents();
    pdl_wait();                                                // the previous step (or whatever wrote the cache and the inputs) has completed

    // TURN: the block's heads from the last to the first in every other step (see decode_turns; all threads read the counter before any of
    // them can have come to its write-back, which lies behind barriers of the compute threads and behind the control lane's copies)
    const int n_heads = bh_end - bh_begin;
    const bool back = TURN && (*counter & 1) != 0;
    const int first = back ? bh_end - 1 : bh_begin, step = back ? -1 : 1;

    if (wid == NW) {
        // ======================================== control lane ==================================================
        if (lane == 0) {
            constexpr uint32_t IDESC_S = instr_desc(128, 16, false);
            constexpr uint32_t IDESC_O = instr_desc(128, 16, false, true);        // A (values) MN-major, B (p) K-major
            const uint32_t k_lo = desc_lo(sK, 16), q_lo = desc_lo(sQ, 16), vmn_lo = desc_lo(sV, 16384), p_lo = desc_lo(sP, 16);
            const unsigned char* g0 = cache + L.header + (size_t)first * L.stride;
            bulk_load(sT, g0 + L.off_z, P.tail_bytes, bar_t0);
            bulk_load(sK, g0 + L.off_k, blk_bytes, bar_k);
            bulk_load(sV, g0 + L.off_v, blk_bytes, bar_v);
            for (int it = 0, bh = first; it < n_heads; ++it, bh += step) {
                const unsigned char* gnext = cache + L.header + (size_t)(bh + step) * L.stride;
                dwait(bar_k, it & 1, 1);
                dwait(bar_q, it & 1, 2);                       // q of this head is in the B tile (and the tail of the head before has been used)
                if (it + 1 < n_heads) bulk_load(sT + ((it & 1) ^ 1) * P.tail_bytes, gnext + L.off_z, P.tail_bytes, bar_t0 + 8 * ((it & 1) ^ 1));
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < NC / 128; ++g)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        umma(tmem + g * 16, desc64(k_lo + g * 1024 + kk * 2, kDescHi), desc64(q_lo + kk * 2, kDescHi), IDESC_S, kk > 0);
                umma_commit(bar_s);
                dwait(bar_p, it & 1, 3);                       // p is in its B tile; the key block is no longer read by anyone
                if (it + 1 < n_heads) bulk_load(sK, gnext + L.off_k, blk_bytes, bar_k);
                dwait(bar_v, it & 1, 4);
                tc_fence_after();
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)                 // 128 keys per half, 16 per instruction (NC = 128: the lower half only)
                    umma(tmem + 32, desc64(vmn_lo + kk * 128, kDescHi), desc64(p_lo + (kk >> 2) * 128 + (kk & 3) * 2, kDescHi),
                         IDESC_O, kk > 0);
                umma_commit(bar_o);
                if (it + 1 < n_heads) {
                    dwait(bar_o, it & 1, 5);                   // the value block has been consumed
                    bulk_load(sV, gnext + L.off_v, blk_bytes, bar_v);
                }
            }
        }
    } else {
        // ======================================== compute threads ===============================================
        // Warp-per-row pieces: a lane has channels 2 lane, 2 lane + 1.  The inputs of a head are fetched under the head before.
        const uint32_t lane_base = ((uint32_t)((wid & 3) * 32)) << 16;
        uint32_t k1r, v1r, q1r, wk[TAPS][2], wv[TAPS][2], bias = 0u;   // (converted where they are used: fetching them waits for nothing)
        uint4 kv_new = make_uint4(0, 0, 0, 0), q_chunk = make_uint4(0, 0, 0, 0);
        uint32_t v1_pair = 0u;
        auto pair = [&](const __nv_bfloat16* x) { return load32(x + 2 * lane); };
        auto fetch_inputs = [&](int bh) {
            const int h = bh % H;
            k1r = pair(k1 + (size_t)bh * D); v1r = pair(v1 + (size_t)bh * D); q1r = pair(q1 + (size_t)bh * D);
#pragma unroll
            for (int u = 0; u < TAPS; ++u) {
                const float* w = cw + ((size_t)h * K + wid + u * NW) * 2 * D + 2 * lane;   // (4-byte aligned)
                if (wid + u * NW < K) { wk[u][0] = load32(w); wk[u][1] = load32(w + 1); wv[u][0] = load32(w + D); wv[u][1] = load32(w + D + 1); }
            }
            if (cbias) bias = load32(cbias + h);
            if (tid < D) v1_pair = load32(v1 + (size_t)bh * D + (tid & ~1));
            if (tid < 8) q_chunk = load128(q1 + (size_t)bh * D + tid * 8);
            if (tid >= 64 && tid < 80) {
                const int t2 = tid - 64;
                kv_new = load128((t2 < 8 ? k1 : v1) + (size_t)bh * D + (t2 & 7) * 8);
            }
        };
        fetch_inputs(first);

        for (int it = 0, bh = first; it < n_heads; ++it, bh += step) {
            const int tb = it & 1;
            unsigned char* gblk = cache + L.header + (size_t)bh * L.stride;
            // q -> row 0 of the logits' B tile (row 0 of a swizzled tile is stored in order)
            if (tid < 8) {
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sQ + tid * 16), "r"(q_chunk.x), "r"(q_chunk.y),
                             "r"(q_chunk.z), "r"(q_chunk.w) : "memory");
                fence_proxy_async();
                mbar_arrive(bar_q);
            }
            dwait(bar_t0 + 8 * tb, (it >> 1) & 1, 6);
            const unsigned char* tail = dsm + P.off_tail + (size_t)tb * P.tail_bytes;
            const float* zc = reinterpret_cast<const float*>(tail);
            const int32_t* pidx = reinterpret_cast<const int32_t*>(tail + (L.off_pidx - L.off_z));
            const int32_t* meta = reinterpret_cast<const int32_t*>(tail + (L.off_meta - L.off_z));
            const int n = meta[0], cnt_old = meta[1];
            const int slot = n % W;

            // ---- pool decision, taken redundantly by every warp so that the row masks are known early -----------
            int dst = -1, cnt_new = cnt_old;
            const int p = n - W;
            const float zp = zc[slot];
            if (p >= 0 && R > 0 && (p < sink || zp > zthr)) {
                if (cnt_old < R) { dst = cnt_old; cnt_new = cnt_old + 1; }
                else if (p >= sink) {
                    // worst entry: lowest logit, the youngest among equals, never a sink entry
                    uint32_t key = 0xffffffffu;
                    int wpos = -1, wslot = -1;
                    for (int m = lane; m < cnt_old; m += 32) {
                        const int pos = pidx[m];
                        const uint32_t k = order_key(zc[W + m] + 0.f);
                        if (pos >= sink && (k < key || (k == key && pos > wpos))) { key = k; wpos = pos; wslot = m; }
                    }
                    const uint32_t kmin = __reduce_min_sync(0xffffffffu, key);
                    const int pmax = __reduce_max_sync(0xffffffffu, key == kmin ? wpos : -1);
                    const unsigned who = __ballot_sync(0xffffffffu, key == kmin && wpos == pmax);
                    wslot = __shfl_sync(0xffffffffu, wslot, __ffs(who) - 1);
                    if (wslot >= 0 && order_key(zp + 0.f) > kmin) dst = wslot;
                }
            }
            // ---- direct reads of the key / value blocks: scorer taps and the popped row ----------------------
            dwait(bar_k, it & 1, 7);
            dwait(bar_v, it & 1, 8);
            const float2 k1f = bf16_pair(k1r), q1f = bf16_pair(q1r);
            const int jsc = K > 0 ? n - half : -1;   // K = 0: the scorer runs outside (lte_cache_score)
            if (jsc >= 0) {
#pragma unroll
                for (int u = 0; u < TAPS; ++u) {
                    const int t = wid + u * NW;
                    if (t >= K) continue;
                    const int pos = jsc + t - half;
                    float2 x = k1f, y = bf16_pair(v1r);
                    if (pos != n) {                            // row of the ring (W >= K); channel -> swizzled place within the row
                        const int back = slot - (n - pos), rr = back < 0 ? back + W : back;
                        const int el = rr * D + ((((lane >> 2) ^ (rr & 7)) << 3) | ((2 * lane) & 7));
                        x = bf16_pair(*reinterpret_cast<const uint32_t*>(reinterpret_cast<const __nv_bfloat16*>(dsm + P.off_k) + el));
                        y = bf16_pair(*reinterpret_cast<const uint32_t*>(reinterpret_cast<const __nv_bfloat16*>(dsm + P.off_v) + el));
                    }
                    float a = pos < 0 ? 0.f : __uint_as_float(wk[u][0]) * x.x + __uint_as_float(wk[u][1]) * x.y + __uint_as_float(wv[u][0]) * y.x + __uint_as_float(wv[u][1]) * y.y;
                    a = warp_sum(a);
                    if (lane == 0) s_tap[tb][t] = a;
                }
            }
            // the popped row doubles as the new pool entry: logical chunk c of row `slot`, kept in a register
            uint4 mv = make_uint4(0, 0, 0, 0);
            if (tid < 16)
                mv = reinterpret_cast<const uint4*>(dsm + (tid < 8 ? P.off_k : P.off_v))[(size_t)slot * 8 + ((tid & 7) ^ (slot & 7))];
            const float s_new = warp_sum(q1f.x * k1f.x + q1f.y * k1f.y) * scale;   // logit of the incoming token (every warp computes it)

            // ---- logits from TMEM, masks, softmax --------------------------------------------------------------
            dwait(bar_s, it & 1, 9);
            tc_fence_after();
            uint32_t sraw;
            tmem_ld1(tmem + lane_base + (tid >> 7) * 16, sraw);
            tmem_wait_ld();
            const int row = tid;
            bool ok;
            if (row >= rows) ok = false;
            else if (row < W) ok = (n >= W) ? (row != slot || dst >= 0) : (row < n);
            else ok = (row - W) < cnt_old && (row - W) != dst;
            const float sl = ok ? __uint_as_float(sraw) * scale : -INFINITY;
            float mx = redux_max(fmaxf(sl, s_new));
            if (lane == 0) s_part[wid] = mx;
            csync<NC>();
            mx = s_part[0];
#pragma unroll
            for (int w2 = 1; w2 < NW; ++w2) mx = fmaxf(mx, s_part[w2]);
            // p rounded to bf16: the same rounded values enter the product and the normalisation
            const __nv_bfloat16 pb = __float2bfloat16_rn(__expf(sl - mx));
            {
                const int rr = row >> 7, col = row & 127, c64 = col & 63;
                const uint32_t off = (col >> 6) * 2048 + rr * 128 + ((((c64 >> 3) ^ (rr & 7))) << 4) + (c64 & 7) * 2;
                asm volatile("st.shared.b16 [%0], %1;" ::"r"(sP + off), "h"(*reinterpret_cast<const unsigned short*>(&pb)) : "memory");
            }
            float lsum = warp_sum(__bfloat162float(pb));
            if (lane == 0) s_sum[wid] = lsum;
            fence_proxy_async();
            tc_fence_before();
            mbar_arrive(bar_p);
            // what the rest of this head needs, and the next head's inputs
            const uint4 kv = kv_new;
            const float bias_now = __uint_as_float(bias), v_now = __uint_as_float(tid & 1 ? v1_pair & 0xffff0000u : v1_pair << 16);
            if (it + 1 < n_heads) fetch_inputs(bh + step);

            // ---- output ----------------------------------------------------------------------------------------
            dwait(bar_o, it & 1, 10);
            tc_fence_after();
            const float p_new = __expf(s_new - mx);
            float sum = p_new;
#pragma unroll
            for (int w2 = 0; w2 < NW; ++w2) sum += s_sum[w2];
            float o_mine = 0.f;
            if (tid < NC / 2) {                                // lanes 0..63: column 0, and for rows 128..255 lanes 64..127: column 1
                uint32_t oraw;
                tmem_ld1(tmem + lane_base + 32 + (tid >> 6), oraw);
                tmem_wait_ld();
                o_mine = __uint_as_float(oraw);
                if (NC == 256) {
                    if (tid >= D) s_o[tid - D] = o_mine;
                    asm volatile("bar.sync 2, 128;" ::: "memory");
                    if (tid < D) o_mine += s_o[tid];
                }
            }
            tc_fence_before();
            if (tid < D) {
                const float o = o_mine + p_new * v_now;
                o1[(size_t)bh * D + tid] = __float2bfloat16_rn(o / sum);
            }
            if (tid == 0) lse1[bh] = mx + logf(sum);

            // ---- write-back: only what changed goes to HBM (rows are stored swizzled) ----------------------------
            uint4* Kw = reinterpret_cast<uint4*>(gblk + L.off_k);
            uint4* Vw = reinterpret_cast<uint4*>(gblk + L.off_v);
            float* zw = reinterpret_cast<float*>(gblk + L.off_z);
            int32_t* pw = reinterpret_cast<int32_t*>(gblk + L.off_pidx);
            int32_t* mw = reinterpret_cast<int32_t*>(gblk + L.off_meta);
            if (dst >= 0 && tid < 16) {
                const int rr = W + dst;
                (tid < 8 ? Kw : Vw)[(size_t)rr * 8 + ((tid & 7) ^ (rr & 7))] = mv;
            }
            if (tid >= 64 && tid < 80) {
                const int t2 = tid - 64;
                (t2 < 8 ? Kw : Vw)[(size_t)slot * 8 + ((t2 & 7) ^ (slot & 7))] = kv;
            }
            if (tid == NC / 2 + 32) {                          // (a warp with nothing else to write)
                if (dst >= 0) { zw[W + dst] = zp; pw[dst] = p; }
                float znew = -INFINITY;
                if (jsc >= 0) {
                    znew = bias_now;
                    for (int t = 0; t < K; ++t) znew += s_tap[tb][t];
                }
                zw[slot] = -INFINITY;
                if (jsc >= 0) zw[jsc % W] = znew;
                mw[0] = n + 1;
                mw[1] = cnt_new;
            }
            // (shared scratch: s_part, s_sum, s_o are written again only after a barrier of the next head that every reader of this
            // one has reached; the taps alternate between two sets)
        }
    }
    tc_fence_before();
    __syncthreads();
    if (wid == NW) tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace

int launch_decode_tc(const Params& p, void* cache, const void* q1, const void* k1, const void* v1, void* o1, float* lse1,
                     cudaStream_t st)
{
    const CacheLayout L = cache_layout(p.d, p.W, p.R, p.dtype);
    if (!L.swz || p.G > 1) return LTE_ERR_UNSUPPORTED;
    int n_sm = 0;
    if (int e = device_sm_count(&n_sm)) return e;
    const int BH = p.B * p.H;
    bool turn = false;
    if (int e = decode_turns(p, &turn)) return e;
    auto go = [&](auto nc, auto kern, PerDeviceOnce& attr) {
        constexpr int NC = decltype(nc)::value;
        const Plan P = plan_of<NC>(L);
        if (int e = attr.run([=] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem<NC>); })) return e;
        if (P.total > (uint32_t)kMostSmem<NC>) return (int)LTE_ERR_UNSUPPORTED;
        // As many CTAs as are resident at once, each with an equal share of the heads (+- 1).  Pools of which W + 2 R > 444 have two
        // longer tail buffers (logits and positions), and with 256 rows two CTAs then fit an SM in place of three.
        const int fit = 227 * 1024 / (int)(P.total + 2048), slots = (fit < kPerSm<NC> ? fit : kPerSm<NC>) * n_sm;
        const int n_cta = BH < slots ? BH : slots;
        return cuda_status(launch_pdl(kern, dim3(n_cta), dim3(kThreads<NC>), P.total, st, (unsigned char*)cache, L, (const __nv_bfloat16*)q1,
                                      (const __nv_bfloat16*)k1, (const __nv_bfloat16*)v1, (__nv_bfloat16*)o1, lse1, p.w, p.bias, BH, p.H, p.W, p.R,
                                      p.sink, p.K, p.zthr, p.scale));
    };
    static PerDeviceOnce attr256, attr128, attr256t, attr128t;
    if (turn && p.W + p.R > 128) return go(std::integral_constant<int, 256>{}, decode_tc_kernel<256, true>, attr256t);
    if (turn) return go(std::integral_constant<int, 128>{}, decode_tc_kernel<128, true>, attr128t);
    if (p.W + p.R > 128) return go(std::integral_constant<int, 256>{}, decode_tc_kernel<256, false>, attr256);
    return go(std::integral_constant<int, 128>{}, decode_tc_kernel<128, false>, attr128);
}

int decode_tc_status_fetch_and_clear() { return status_fetch_and_clear(g_decode_tc_status); }

}  // namespace lte
