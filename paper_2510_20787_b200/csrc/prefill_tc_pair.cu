// Prefill attention at d = 128 on the 5th-generation tensor cores (Section 3.1.3): pairs of 128-query tiles that share their key and
// value tiles.
//   S = Q K^T      tcgen05.mma (kind::f16, bf16 in, fp32 out) into TMEM, tiles of 64 keys
//   softmax        eight warps per query tile, two threads per row (32 of a tile's 64 keys each); P goes back into one of two TMEM
//                  buffers as bf16
//   O += P V       tcgen05.mma with P as the TMEM A operand
// Bound by the exponentials (512 cycles of their unit for 128 x 64) and the tensor core (about 600), so both have to run all the time:
// S of the next tile is computed as soon as this one's is in registers, P V of the last ones runs meanwhile, and there are two query
// tiles (O, S, P of both: all 512 TMEM columns).  One CTA of two query tiles per SM instead of two independent ones, because K and V
// then come through L2 once for 256 queries.  Two warps issue the products, one per query tile (a warp issues one every 54 cycles).
// Items (256 queries of one head) are handed out dynamically, the longest first.
// The two halves of a row do not wait for each other's maximum: the exponentials' reference is the maximum of the first tile that the row
// sees part of and moves only when a later logit is far above it (the arguments stay <= kFar, so that weights, O and the sum keep within a
// factor of 2^8 of the values and the largest weights stay near 1), which is asked once the exponentials are done.  (kFar = 64 is not
// faster: 364.0 and 363.6 us for the whole case of the first line below.)
// Every mbarrier wait is bounded; a wait that runs out records a status word and the kernel still terminates.
// Measured (B200, us, compaction included, back to back in a CUDA graph, where the clock moves by some 5 % from run to run; before: a CTA
// per 128-query tile, two CTAs per SM, prefill_tc_long.cu):
//   16 heads x 32,768, W = R = 512      254 - 276 (769 TFLOP/s), before 283 - 294
//   16 heads x 8,192, W = R = 512       88 - 91, before 92 - 98    32 heads x 8,192, W = R = 64         63 - 68, before 70 - 72
//   64 heads x 4,096, W = R = 128       72 - 77, before 82 - 86    256 heads x 2,000 in fours, W 300    166 - 176, before 188 - 192
// What was slower in the first line: S of 128 keys with P in its place (264 to 271: the chain P, PV, S is exposed), two S buffers and
// groups of warps taking turns at the tiles (283), a product warp whose control flow the compiler takes for divergent (276), one
// commit per tile and plain arrivals for what it implies (269: stages come free too late for short items).
#include "tile_items.cuh"

namespace lte {

__device__ StatusWord g_prefill_pair_status = LTE_STATUS_INIT; // 0 = fine; otherwise the code of the wait that gave up

namespace {

using namespace tc;
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, int code) { mbar_wait_call(bar, parity, code, &g_prefill_pair_status); }

__device__ __forceinline__ void mbar_wait_u(uint32_t bar, uint32_t parity, int code) { mbar_wait_uni_call(bar, parity, code, &g_prefill_pair_status); }

constexpr int D = 128, BM = 128, BN = 64, ST = 5;              // query tile, key tile, stages (of K, and as many of V)
constexpr int W_MMA = 16, W_LOAD = 18, NTHREADS = 19 * 32;     // 16 softmax warps, an MMA warp per query tile, a load warp
constexpr int QTILE = BM * D * 2, TILE = BN * D * 2;           // a tile is two 64-column sub-tiles
constexpr int OFF_Q = 0, OFF_K = 2 * QTILE, OFF_V = OFF_K + ST * TILE, OFF_BAR = OFF_V + ST * TILE, OFF_INFO = OFF_BAR + 512, OFF_X = OFF_INFO + 4 * 96;
constexpr int SMEM_BYTES = OFF_X + 2 * 2 * BM * 4;             // X[query tile][half][row]: maxima, then sums, on their way to the other half
static_assert(SMEM_BYTES <= 232448, "shared memory");
constexpr float kFar = 8.f;                                   // (log2) how far above the reference a logit may lie
constexpr uint32_t S_COL = 0, P_COL = 64, O_COL = 256;         // + 128 for the second query tile;  P: two buffers of 32 columns

struct Args { int n_qt, n_bh, Tlen, W, R, G, qoff; float scale; };
// Row x of query tile q (0, 1) sees before[q][x / 32] list entries and those of bits[q][x / 32] below bit x % 32; all[q]: what its last
// row sees.  bh = -1: there is no further item.
struct Info { uint32_t before[2][4], bits[2][4]; int all[2], bh, bhk, i0; };

// Tiles of an item: n_win window tiles from key j_start on, then list tiles.  Of them query tile q takes window tiles [w0, w1) and
// the first nl list tiles (it may have no rows at all: none).
struct Item { int bh, bhk, i0, j_start, n_win; };
struct Part { int w0, w1, nl, n_tiles, n; };                   // n_tiles: of the item;  n: of this query tile
__device__ __forceinline__ Item item_at(const Args& a, int bh, int bhk, int i0)
{
    Item it;
    it.bh = bh; it.bhk = bhk; it.i0 = i0;
    it.j_start = max(i0 - a.W + 1, 0);
    it.n_win = (min(i0 + 2 * BM - 1, a.Tlen - 1) - it.j_start) / BN + 1;
    return it;
}
__device__ __forceinline__ Item item_of(const Args& a, int item)
{
    const int r = item / a.n_bh, bh = item - r * a.n_bh;       // from the last query tile of every head down to the first
    return item_at(a, bh, bh / a.G, a.qoff + (a.n_qt - 1 - r) * 2 * BM);
}
__device__ __forceinline__ Part part_of(const Args& a, const Item& it, int q, int all0, int all1)
{
    Part p;
    const int r0 = it.i0 + q * BM, r1 = min(r0 + BM - 1, a.Tlen - 1);
    p.n_tiles = it.n_win + (max(all0, all1) + BN - 1) / BN;
    p.w0 = p.w1 = p.nl = 0;
    if (r0 < a.Tlen) {
        p.w0 = (max(r0 - a.W + 1, 0) - it.j_start) / BN;
        p.w1 = (r1 - it.j_start) / BN + 1;
        p.nl = ((q ? all1 : all0) + BN - 1) / BN;
    }
    p.n = p.w1 - p.w0 + p.nl;
    return p;
}
__device__ __forceinline__ bool takes(const Item& it, const Part& p, int t) { return t < it.n_win ? t >= p.w0 && t < p.w1 : t - it.n_win < p.nl; }

// Barriers (n = item number within the CTA; g = tile number; a = tile number and e = item number counted over what the query tile takes
// part in; b = a & 1):
//   bar_k[s], bar_v[s]       K, V of tile g are in stage s = g % ST (TMA)          phase g / ST
//   bar_ke[s], bar_ve[s] (2) both query tiles are done with them (commit)
//   bar_q, bar_qf (2)        Q of item n is there / both query tiles' last S are complete (commit)
//   bar_s[q]     (commit)    S of tile a is in TMEM; PV of tile a-2 is complete     phase a
//   bar_sf[q]    (8)         it is in registers
//   bar_p[q][b]  (8)         P of tile a is in buffer b                             phase a >> 1
//   bar_l[q]     (commit)    PV of an item's last tile but one is complete          phase: items of at least two tiles
__global__ void __launch_bounds__(NTHREADS, 1)
prefill_pair_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const __grid_constant__ CUtensorMap tmKc, const __grid_constant__ CUtensorMap tmVc, const Args args,
                    const int32_t* __restrict__ idx, const int32_t* __restrict__ cnt, __nv_bfloat16* __restrict__ og, float* __restrict__ lse)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0) { if (threadIdx.x == 0) atomicExch(&g_prefill_pair_status.code, 9); return; }   // the swizzled tiles need it
    const uint32_t sQ = base + OFF_Q, sK = base + OFF_K, sV = base + OFF_V, bars = base + OFF_BAR;
    const uint32_t bar_k = bars, bar_v = bars + 40, bar_ke = bars + 80, bar_ve = bars + 120, bar_q = bars + 160, bar_qf = bars + 168, bar_s = bars + 176,
                   bar_sf = bars + 192, bar_p = bars + 208, bar_l = bars + 240, bar_o = bars + 272, bar_of = bars + 288, bar_i = bars + 304,
                   bar_c = bars + 336, tmem_slot = bars + 344, answer = bars + 352;
    auto slot = [&](int n) { return reinterpret_cast<volatile Info*>(smem_raw + OFF_INFO + (n & 3) * 96); };
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < ST; ++s) { mbar_init(bar_k + 8 * s, 1); mbar_init(bar_v + 8 * s, 1); mbar_init(bar_ke + 8 * s, 2); mbar_init(bar_ve + 8 * s, 2); }
#pragma unroll
        for (int s = 0; s < 2; ++s) { mbar_init(bar_s + 8 * s, 1); mbar_init(bar_sf + 8 * s, 8); mbar_init(bar_l + 8 * s, 1); mbar_init(bar_o + 8 * s, 1); mbar_init(bar_of + 8 * s, 8); }
#pragma unroll
        for (int s = 0; s < 4; ++s) { mbar_init(bar_p + 8 * s, 8); mbar_init(bar_i + 8 * s, 1); }
        mbar_init(bar_q, 1); mbar_init(bar_qf, 2); mbar_init(bar_c, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem_raw + OFF_BAR + 344);
    pdl_launch_dependents();
    pdl_wait();                                                // everything above ran beside the previous kernel's tail

    auto enter = [&](int n) {                                  // the n-th item out of the ring (whole warp)
        const volatile Info* f = slot(n);
        const int bh = __shfl_sync(0xffffffffu, f->bh, 0), bhk = __shfl_sync(0xffffffffu, f->bhk, 0), i0 = __shfl_sync(0xffffffffu, f->i0, 0);
        return item_at(args, bh, bhk, i0);
    };

    if (warp == W_LOAD) {
        // ================================= load warp (lane 0 issues) ==============================================
        ItemQueue queue(answer, bar_c, lane);
        uint32_t s = 0, lap = 0;                               // stage of the next tile, how often the ring has been round
        for (int n = 0;; ++n) {
            const int item = n == 0 ? (int)blockIdx.x : queue.take(17, &g_prefill_pair_status);
            if (item < 0) {
                if (lane == 0) { slot(n)->bh = -1; mbar_arrive(bar_i + 8 * (n & 3)); }
                break;
            }
            const Item it = item_of(args, item);
            int n_tiles = it.n_win;                            // until the list has been looked at
            for (int t = 0; t < n_tiles; ++t) {
                const bool win = t < it.n_win;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const uint32_t full = (v ? bar_v : bar_k) + 8 * s, dst = (v ? sV : sK) + s * TILE;
                    if (lap > 0) mbar_wait((v ? bar_ve : bar_ke) + 8 * s, (lap - 1) & 1u, 6);
                    if (lane == 0) {
                        const CUtensorMap* tm = v ? (win ? &tmV : &tmVc) : (win ? &tmK : &tmKc);
                        mbar_expect_tx(full, TILE);
#pragma unroll
                        for (int sb = 0; sb < 2; ++sb)
                            tma_load_3d(dst + sb * (TILE / 2), tm, sb * 64, win ? it.j_start + t * BN : (t - it.n_win) * BN, it.bhk, full);
                    }
                }
                if (++s == ST) { s = 0; ++lap; }
                if (t == 0) {                                  // tile 0 is a window tile; the list is looked up while it is on its way
                    const int32_t* id = idx + (size_t)it.bhk * args.R;
                    const int last = args.Tlen - 1 - it.i0;
                    const ListView a = view_list(id, cnt + it.bhk, args.R, it.i0 - args.W, min(last, BM - 1), lane);
                    const ListView b = view_list(id, cnt + it.bhk, args.R, it.i0 + BM - args.W, max(min(last - BM, BM - 1), 0), lane);
                    const int all1 = last >= BM ? b.all : 0;
                    n_tiles = it.n_win + (max(a.all, all1) + BN - 1) / BN;
                    if (lane == 0) {
                        volatile Info* o = slot(n);
#pragma unroll
                        for (int k = 0; k < 4; ++k) { o->before[0][k] = a.before[k]; o->bits[0][k] = a.bits[k]; o->before[1][k] = b.before[k]; o->bits[1][k] = b.bits[k]; }
                        o->all[0] = a.all; o->all[1] = all1; o->bh = it.bh; o->bhk = it.bhk; o->i0 = it.i0;
                        mbar_arrive(bar_i + 8 * (n & 3));
                    }
                    if (n > 0) mbar_wait(bar_qf, (n - 1) & 1, 12);
                    if (lane == 0) {
                        mbar_expect_tx(bar_q, 2 * QTILE);
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            tma_load_3d(sQ + x * (QTILE / 2), &tmQ, (x & 1) * 64, it.i0 - args.qoff + (x >> 1) * BM, it.bh, bar_q);
                    }
                }
                if (t == max(n_tiles - kAskTiles, 0)) queue.ask();
            }
        }
        __syncwarp();
    } else if (warp >= W_MMA) {
        // ================================= MMA warps (an elected thread issues; the whole warp walks the loop) ======
        constexpr uint32_t IDESC_S = instr_desc(BM, BN, false), IDESC_O = instr_desc(BM, D, true);
        const int q = warp - W_MMA;
        const uint32_t q_lo = desc_lo(sQ + q * QTILE, 16), k_lo = desc_lo(sK, 16), v_lo = desc_lo(sV, TILE / 2);
        const uint32_t s_tm = tmem + S_COL + q * 128, o_tm = tmem + O_COL + q * 128;
        struct Ring { uint32_t s = 0, lap = 0; __device__ __forceinline__ void next() { const bool w = uni(++s == ST); s = w ? 0 : s; lap += w; } } rk, rv;
        uint32_t as = 0, ap = 0, e = 0;                        // tiles: S issued, P V issued
        for (int n = 0;; ++n) {
            mbar_wait_u(bar_i + 8 * (n & 3), (n >> 2) & 1, 9);
            const Item it = enter(n);
            if (uni(it.bh < 0)) break;
            const Part p = part_of(args, it, q, __shfl_sync(0xffffffffu, slot(n)->all[0], 0), __shfl_sync(0xffffffffu, slot(n)->all[1], 0));
            mbar_wait_u(bar_q, n & 1, 1);
            if (p.n == 0 && lane == 0) mbar_arrive(bar_qf);
            int tk = 0, tv = 0, left = p.n;
            auto skip_one = [&](Ring& r, uint32_t full, uint32_t free) {   // a tile of the other query tile alone
                mbar_wait_u(full + 8 * r.s, r.lap & 1u, 10);
                if (lane == 0) mbar_arrive(free + 8 * r.s);
                r.next();
            };
            auto mma_s = [&]() {
                for (; uni(!takes(it, p, tk)); ++tk) skip_one(rk, bar_k, bar_ke);   // (at most two at a time)
                if (uni(as > 0)) mbar_wait_u(bar_sf + 8 * q, (as - 1) & 1, 3);   // the previous tile's S is in registers
                mbar_wait_u(bar_k + 8 * rk.s, rk.lap & 1u, 2);
                tc_fence_after();
                --left;
                if (elect_one()) {
                    const uint32_t kd = k_lo + rk.s * (TILE >> 4);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        umma(s_tm, desc64(q_lo + (kk >> 2) * (QTILE >> 5) + (kk & 3) * 2, kDescHi),
                             desc64(kd + (kk >> 2) * (TILE >> 5) + (kk & 3) * 2, kDescHi), IDESC_S, kk > 0);
                    umma_commit(bar_s + 8 * q);
                    umma_commit(bar_ke + 8 * rk.s);
                    if (left == 0) umma_commit(bar_qf);
                }
                __syncwarp();
                ++as; ++tk; rk.next();
            };
            if (uni(left > 0)) mma_s();
            for (int k = 0; uni(k < p.n); ++k, ++ap) {
                if (uni(left > 0)) mma_s();                         // S of the next tile before PV of this one
                for (; uni(!takes(it, p, tv)); ++tv) skip_one(rv, bar_v, bar_ve);
                mbar_wait_u(bar_v + 8 * rv.s, rv.lap & 1u, 4);
                if (uni(k == 0 && e > 0)) mbar_wait_u(bar_of + 8 * q, (e - 1) & 1, 13);   // the previous item's O has been read out
                mbar_wait_u(bar_p + 16 * q + 8 * (ap & 1), (ap >> 1) & 1u, 7);
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t vd = v_lo + rv.s * (TILE >> 4);
#pragma unroll
                    for (int kk = 0; kk < BN / 16; ++kk)
                        umma_ts(o_tm, s_tm + P_COL + (ap & 1) * 32 + kk * 8, desc64(vd + kk * 128, kDescHi), IDESC_O, (k > 0 || kk > 0) ? 1u : 0u);
                    umma_commit(bar_ve + 8 * rv.s);
                    if (k >= p.n - 2) umma_commit(k == p.n - 1 ? bar_o + 8 * q : bar_l + 8 * q);   // (no S of this item follows that would tell)
                }
                __syncwarp();
                ++tv; rv.next();
            }
            // the remaining tiles are the other query tile's, K and V in the order in which they come (stages of one wait for the other's)
            while (uni(tv < p.n_tiles)) {
                if (uni(tk == tv)) { skip_one(rk, bar_k, bar_ke); ++tk; }
                skip_one(rv, bar_v, bar_ve); ++tv;
            }
            if (p.n > 0) ++e;
        }
    } else {
        // =================================== softmax warps ==================================================
        // Two threads per row: of query tile q = warp / 8, warps 0-3 take columns [0, 32) of every tile, warps 4-7 columns [32, 64).
        const int q = warp >> 3, hf = (warp >> 2) & 1, wq = warp & 3, row = wq * 32 + lane, c0 = hf * 32;
        const int W = args.W, Tlen = args.Tlen;
        const float c2 = args.scale * 1.4426950408889634f;     // logits are handled in the log2 domain: x = s * c2
        const uint64_t c2_2 = pack2(c2, c2);
        const uint32_t trow = tmem + ((uint32_t)(wq * 32) << 16) + q * 128;   // this warp's TMEM lanes
        const uint32_t s_col = trow + S_COL + c0, p_col = trow + P_COL + hf * 16, o_col = trow + O_COL + hf * 64;
        volatile float* x_mine = reinterpret_cast<volatile float*>(smem_raw + OFF_X) + (q * 2 + hf) * BM + row;
        volatile float* x_other = reinterpret_cast<volatile float*>(smem_raw + OFF_X) + (q * 2 + (hf ^ 1)) * BM + row;
        auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + q * 4 + wq) : "memory"); };   // the two warps of these rows
        auto pair_any = [&](bool mine) {                       // ... meeting, and asking whether any of their threads says so
            uint32_t any;
            asm volatile("{\n\t.reg .pred p, r;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred r, %2, 64, p;\n\tselp.u32 %0, 1, 0, r;\n\t}"
                         : "=r"(any) : "r"(mine ? 1u : 0u), "r"(1 + q * 4 + wq) : "memory");
            return any != 0u;
        };
        uint32_t a = 0, e = 0, el = 0;
        for (int n = 0;; ++n) {
            mbar_wait(bar_i + 8 * (n & 3), (n >> 2) & 1, 15);
            const Item it = enter(n);
            if (it.bh < 0) break;
            const volatile Info* f = slot(n);
            const Part p = part_of(args, it, q, __shfl_sync(0xffffffffu, f->all[0], 0), __shfl_sync(0xffffffffu, f->all[1], 0));
            if (p.n == 0) continue;                            // (no rows)
            const int i0 = it.i0 + q * BM, ia = i0 + wq * 32, i = ia + lane;   // the tile's, the warp's first query row, this thread's
            const int x_row = min(i, Tlen - 1) - i0;           // (rows past the end repeat the last one)
            const int nvis = (int)(f->before[q][x_row >> 5] + __popc(f->bits[q][x_row >> 5] & ((1u << (x_row & 31)) - 1u)));
            const int nvis_first = __shfl_sync(0xffffffffu, nvis, 0);
            float m_run = -INFINITY;                           // the row's reference (log2 domain), the same in both halves; -inf: none yet
            uint64_t ls[2] = {0ull, 0ull};                     // sum of this half of the row, two packed pairs
            for (int k = 0; k < p.n; ++k, ++a) {
                const int t = k < p.w1 - p.w0 ? p.w0 + k : it.n_win + k - (p.w1 - p.w0);
                // columns (of this half) the row may see in the tile; `full`: every row of the warp (the bounds grow with the row) sees all
                int c_lo, c_hi;
                bool full;
                if (t < it.n_win) {
                    const int jt0 = it.j_start + t * BN + c0;
                    c_lo = max(i - W + 1, 0) - jt0; c_hi = i - jt0;
                    full = max(ia + 31 - W + 1, 0) <= jt0 && ia - jt0 >= 31;
                } else {
                    const int e0 = (t - it.n_win) * BN + c0;
                    c_lo = 0; c_hi = nvis - e0 - 1;
                    full = nvis_first - e0 - 1 >= 31;
                }
                uint32_t vm = 0xffffffffu;
                bool act = true;                               // any row of the warp sees anything
                if (!full) {
                    const int lo = min(max(c_lo, 0), 32), hi = min(max(c_hi + 1, 0), 32);
                    const uint32_t below_hi = hi >= 32 ? 0xffffffffu : ((1u << hi) - 1u), below_lo = lo >= 32 ? 0xffffffffu : ((1u << lo) - 1u);
                    vm = hi > lo ? (below_hi & ~below_lo) : 0u;
                    act = __any_sync(0xffffffffu, vm != 0u);
                }
                uint32_t x[32], pk[16];                        // logits; P, two columns per word
                mbar_wait(bar_s + 8 * q, a & 1, 5);
                tc_fence_after();
                tmem_ld32(s_col, x);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_sf + 8 * q);    // S of the next tile may overwrite it
                if (!full) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) x[c] = (vm & (1u << c)) ? x[c] : 0xff800000u;   // -inf
                }
                float mr[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int c = 0; c < 32; c += 2) mr[(c >> 1) & 3] = max3(mr[(c >> 1) & 3], __uint_as_float(x[c]), __uint_as_float(x[c + 1]));
                const float m_mine = fmaxf(fmaxf(mr[0], mr[1]), fmaxf(mr[2], mr[3])) * c2;
                auto move_reference = [&]() {                  // (both halves of the rows)
                    *x_mine = m_mine;
                    pair_sync();
                    const float m_tile = fmaxf(m_mine, *x_other);
                    float alpha = 1.f;
                    bool rescale = false;
                    if (m_run == -INFINITY) m_run = m_tile;    // nothing accumulated yet for this row: its O is 0
                    else if (m_tile > m_run + kFar) { alpha = fast_exp2(m_run - m_tile); m_run = m_tile; rescale = true; }
                    if (k > 0 && __any_sync(0xffffffffu, rescale)) {   // (then PV of the tile before has to be complete)
                        if (k < p.n - 1) mbar_wait(bar_s + 8 * q, (a + 1) & 1, 19);   // (issued behind it)
                        else mbar_wait(bar_l + 8 * q, el & 1, 18);
                        tc_fence_after();
#pragma unroll 1
                        for (int cb = 0; cb < 4; ++cb) {
                            uint32_t o[16];
                            tmem_ld16(o_col + cb * 16, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int c = 0; c < 16; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                            tmem_st16(o_col + cb * 16, o);
                        }
                        tmem_wait_st();
                    }
                    const uint64_t a2 = pack2(alpha, alpha);
                    ls[0] = mul2(ls[0], a2); ls[1] = mul2(ls[1], a2);
                    pair_sync();                               // (both have read)
                };
                bool asked = false;
                if (__any_sync(0xffffffffu, m_run == -INFINITY)) { move_reference(); asked = true; }   // (the same in both halves) an item's first tiles
                const uint64_t l0 = ls[0], l1 = ls[1];
                for (;;) {
                    if (act) {
                        const float neg_m = m_run == -INFINITY ? 0.f : -m_run;
                        const uint64_t neg_m2 = pack2(neg_m, neg_m);
#pragma unroll
                        for (int c = 0; c < 32; c += 2) {
                            // masked entries hold -inf: fma gives -inf and exp2(-inf) = 0
                            float p0, p1;                      // two columns per packed fp32 instruction
                            unpack2(fma2(pack2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), c2_2, neg_m2), p0, p1);
                            p0 = fast_exp2(p0); p1 = fast_exp2(p1);
                            ls[(c >> 1) & 1] = add2(ls[(c >> 1) & 1], pack2(p0, p1));
                            const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
                            pk[c >> 1] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; ++c) pk[c] = 0u;
                    }
                    if (asked || !pair_any(m_mine > m_run + kFar)) break;
                    ls[0] = l0; ls[1] = l1;                    // (rare) once more, with another reference
                    move_reference();
                    asked = true;
                }
                tmem_st16(p_col + (a & 1) * 32, pk);           // (PV of tile a-2 was complete with this S)
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p + 16 * q + 8 * (a & 1));
            }
            // the item's output (64 columns each); the next item's first S is computed meanwhile
            float l, lb;
            unpack2(add2(ls[0], ls[1]), l, lb);
            l += lb;
            mbar_wait(bar_o + 8 * q, e & 1, 14);
            tc_fence_after();
            uint32_t o[2][32];
            tmem_ld32(o_col, o[0]);
            tmem_ld32(o_col + 32, o[1]);
            *x_mine = l;
            pair_sync();
            l += *x_other;
            tmem_wait_ld();
            tc_fence_before();
            pair_sync();
            const float inv = 1.f / l;
            if (lane == 0) mbar_arrive(bar_of + 8 * q);        // the accumulator may take the next item
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                uint32_t w[4][4];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(o[cb][2 * c]) * inv, __uint_as_float(o[cb][2 * c + 1]) * inv);
                    w[c >> 2][c & 3] = *reinterpret_cast<const uint32_t*>(&h);
                }
                // four lanes transpose their four 16-byte pieces, so that a store covers 64 bytes of 8 rows instead of 16 of 32
#pragma unroll
                for (int m = 1; m <= 2; m <<= 1)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c & m) continue;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {          // my piece for the partner: c ^ m if I am the lower lane, else c
                            const bool up = (lane & m) != 0;
                            const uint32_t r = __shfl_xor_sync(0xffffffffu, up ? w[c][k] : w[c ^ m][k], m);
                            if (up) w[c][k] = r; else w[c ^ m][k] = r;
                        }
                    }
#pragma unroll
                for (int c = 0; c < 4; ++c) {                  // now piece lane & 3 of row (lane & ~3) + c
                    const int r = ia + (lane & ~3) + c;
                    if (r < Tlen)
                        *reinterpret_cast<uint4*>(og + ((size_t)it.bh * (Tlen - args.qoff) + r - args.qoff) * D + hf * 64 + cb * 32 + (lane & 3) * 8) =
                            make_uint4(w[c][0], w[c][1], w[c][2], w[c][3]);
                }
            }
            if (hf == 0 && i < Tlen) lse[(size_t)it.bh * (Tlen - args.qoff) + i - args.qoff] = m_run * 0.6931471805599453f + logf(l);
            ++e;
            if (p.n > 1) ++el;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == W_MMA) tmem_dealloc(tmem, 512);
}

}  // namespace

// with a workspace of `half` bytes each for the compacted keys and values (prefill_compact_bytes)
int launch_prefill_tc_pair(const Params& p, const void* q, const void* k, const void* v, const int32_t* idx, const int32_t* cnt, void* o,
                           float* lse, void* ws, size_t half, cudaStream_t st)
{
    CUtensorMap tq, tk, tv, tkc, tvc;
    const int BHK = p.B * p.H, BH = BHK * p.G, Tq = p.T - p.qoff;   // key/value heads, query heads, query rows
    char* kc = (char*)ws; char* vc = kc + half;
    if (!make_map(&tq, q, BH, Tq, D, BM) || !make_map(&tk, k, BHK, p.T, D, BN) || !make_map(&tv, v, BHK, p.T, D, BN) ||
        !make_map(&tkc, kc, BHK, p.R, D, BN) || !make_map(&tvc, vc, BHK, p.R, D, BN)) return LTE_ERR_CUDA;
    if (int e = launch_prefill_compact(p, k, v, idx, cnt, kc, vc, st)) return e;
    static PerDeviceOnce attr;
    if (int e = attr.run([] { return cudaFuncSetAttribute(prefill_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES); })) return e;
    Args a;
    a.n_qt = (Tq + 2 * BM - 1) / (2 * BM); a.n_bh = BH; a.Tlen = p.T; a.W = p.W; a.R = p.R; a.G = p.G; a.qoff = p.qoff; a.scale = p.scale;
    return cuda_status(launch_pdl(prefill_pair_kernel, dim3(a.n_qt * BH), dim3(NTHREADS), SMEM_BYTES, st, tq, tk, tv, tkc, tvc, a, idx, cnt,
                                  (__nv_bfloat16*)o, lse));
}

int prefill_pair_status_fetch_and_clear() { return status_fetch_and_clear(g_prefill_pair_status); }

}  // namespace lte
