// Prefill attention on the 5th-generation tensor cores for bf16, d = 64 and d = 32 (Section 3.1.3, "Cached prefilling and
// decoding").
//
// Bound by the instruction stream of the softmax warps and the latencies between them (no pipe is full: with items of nine tiles issue
// 60 %, exponential unit 55 %, tensor pipe 31 %; with items of four 55, 37, 27), so work is paid once per 128 keys, spread over 16
// warps per SM, and nothing waits that need not:
//   work      Two CTAs per SM; an item is a 128-query tile of one head.  Key/value tiles of 128 rows come by TMA, first the window
//             span, then the head's retained rows that any of the item's rows may see (compacted beforehand where the caller
//             brought a workspace; otherwise the load warp gathers them row by row into the same swizzled layout).  Eight softmax
//             warps (two threads per row, 64 columns each), one warp issuing the products, one issuing the loads.
//   S(g) = Q K^T    one buffer: the softmax has taken all of S(g) when half of its exponentials are done, and S(g+1) is computed
//             under the other half (P has columns of its own, so nothing else holds the buffer).  TMEM: S [0,128), P [128,192),
//             O [192,256)
//   softmax   mask from positions (32-column chunks are skipped or taken unmasked where the warp's rows allow); the row maximum
//             of the two halves is exchanged through shared memory; the reference follows it only when it grew by 2^8 (lazy
//             rescale); exp2 with the scale folded in; P as bf16 into TMEM.  O is divided by the sum of P, so that its rounding
//             cancels as far as it is common to the row, and lse is the logarithm of the sum of the weights themselves (the two
//             sums against one: 3 % of the time; with the weights' sum alone O's error is 2 % larger, with P's alone lse's 1e-3)
//   O += P V  P as the TMEM A operand, V as the MN-major shared-memory operand; O is read and stored under the next item's first tile
// How many retained entries a row sees: the load warp finds an item's place in the list (a 32-way search) and hands out, one
// item ahead, a bit map of the entries that fall between the limits of the item's first and last row.
// Tiles are numbered through all items of a CTA (g); stage, buffer and barrier phase follow from that number, and the loads
// and products of the next item run under the current one.  Every mbarrier wait is bounded; one that runs out records a
// status word and the kernel still terminates.
//
// Measured (B200, the call with a workspace, back to back in a CUDA graph; before: four warps with 64-key tiles, items dealt out):
//   1,024 query heads x 4,096, W = 768, R = 512 half used   1.67 ms (515 TFLOP/s), before 2.09
//   32 x 4,096 of it                                       198 us (542), before 285
//   64 heads x 4,096, W = R = 128                          54 us, before 62      128 x 2,048, W = R = 64   44 us, before 50
// The steps, at an eighth of the first shape and with one sum per row: four warps with 64-key tiles 275 us; one thread per row, 128-key
// tiles 242; two threads per row 223; dynamic items 203; O stored under the next item 190.  Tried there and slower: rolled
// 32-column loops (214), column bounds carried from tile to tile and a vote in place of the exchange of maxima (209), one thread
// per row with dynamic items (213), the two streams of an SM taking turns at the exponential unit (328), a quarter of the
// exponentials as polynomials on the multiply-add pipe (207).
//
// d = 32 runs the same kernel: the tensor maps describe 32-column rows with a 64-column box, the copy engine fills the upper
// half of every tile row with zeros, and only the first 32 output columns are stored.
#include "tile_items.cuh"

namespace lte {

__device__ StatusWord g_prefill_status = LTE_STATUS_INIT;         // 0 = fine; otherwise the code of the wait that gave up

namespace {

constexpr int BM = 128, BN = 128, D = 64, NTHREADS = 320;         // warps 0-7 softmax, 8 products, 9 loads
using namespace tc;
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, int code) { mbar_wait_call(bar, parity, code, &g_prefill_status); }
__device__ __forceinline__ void mbar_wait_u(uint32_t bar, uint32_t parity, int code) { mbar_wait_uni_call(bar, parity, code, &g_prefill_status); }

template <bool STREAM> struct Smem {
    static constexpr int TILE = 128 * D * 2;                  // [128][64] bf16: Q, K and V tiles alike
    static constexpr int QST = 2, KST = 2, VST = 2;
    static constexpr int OFF_Q = 0, OFF_K = QST * TILE, OFF_V = OFF_K + KST * TILE;
    static constexpr int OFF_BAR = OFF_V + VST * TILE;
    static constexpr int OFF_INFO = OFF_BAR + 256;            // ring of four items' Info
    static constexpr int OFF_X = OFF_INFO + 4 * 64;           // row maxima on their way to the other half (by tile parity), [2][2][128]
    static constexpr int OFF_L = OFF_X + 2 * 2 * BM * 4;      // row sums of the two halves (by item parity), [2][2][128] pairs
    static constexpr int OFF_LV = OFF_L + 2 * 2 * BM * 8;     // STREAM: the leave times of a retained tile, [8 warps][64]
    static constexpr int BYTES = OFF_LV + (STREAM ? 8 * 64 * 4 : 0);
};
constexpr uint32_t TMEM_COLS = 256, S_COL = 0, P_COL = 128, O_COL = 192;

// An item: a 128-query tile of one (b,h).  Items are numbered from the last query tile of every head down to the first: later
// tiles see more retained rows and cost more.  The grid has a block per item, but a block that has run out of work takes the
// next block that has not started (cluster launch control) instead of leaving, so items are handed out in order, largest
// first, to whoever is free: dealt out beforehand, the blocks finished up to 30 % apart (159 to 219 us).
struct Item { int bh, bhk, i0, j_start, n_win, n_tiles, item; };   // bh: query head (b, h, g); bhk: its key/value head (b, h)
struct Args { int n_items, n_qt, n_bh, Tlen, W, G, qoff; };
// What the load warp tells the others about an item.  Row x of the item (0 .. 127) sees before[x / 32] entries and those of
// bits[x / 32] below bit x % 32.
struct Info { uint32_t before[4], bits[4]; int n_tiles, item; };   // item = -1: there is none

__device__ __forceinline__ Item item_of(const Args& a, int item)
{
    Item it;
    const int r = item / a.n_bh;
    it.item = item;
    it.bh = item - r * a.n_bh;
    it.bhk = it.bh / a.G;
    it.i0 = a.qoff + (a.n_qt - 1 - r) * BM;                    // positions; the query tensors start at position qoff
    const int i_hi = min(it.i0 + BM - 1, a.Tlen - 1);
    it.j_start = max(it.i0 - a.W + 1, 0);
    it.n_win = (i_hi - it.j_start + BN) / BN;
    it.n_tiles = it.n_win;                                     // until the item's Info is there
    return it;
}
// Walks a CTA's tiles in order: tile t of its n-th item is tile g.
struct Cursor {
    Item it;
    int n = 0, t = 0;
    uint32_t g = 0;
    bool live = true;
    __device__ __forceinline__ void advance() { ++g; if (++t == it.n_tiles) { t = 0; ++n; } }
};
__device__ __forceinline__ void add_bf16x2(float& a, float& b, uint32_t x) {   // a += the lower, b += the upper half of x
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.rn.f32.bf16 %0, l, %0;\n\tadd.rn.f32.bf16 %1, h, %1;\n\t}" : "+f"(a), "+f"(b) : "r"(x));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr) : "memory");
}

// Barriers (g = tile number, n = item number within the CTA):
//   bar_q[b], bar_qf[b]   Q of item n has landed in buffer b = n & 1 (TMA) / the item's last S is complete (commit)    phase n >> 1
//   bar_k[s], bar_v[s]    TMA of tile g into stage s = g % stages                                                       phase g / stages
//   bar_kf[s], bar_vf[s]  (commit) the product that read the stage's tile is complete                                   phase g / stages
//   bar_s    (commit)     S(g) is in TMEM                   bar_sf (8 arrivals)  S(g) is in registers                   phase g
//   bar_p    (8 arrivals) P(g) is in TMEM, and PV(g-1) has been awaited               bar_pv (commit)  PV(g) is complete  phase g
//   bar_of   (8 arrivals) O of item n has been read out                                                                phase n
//   bar_i[n & 3]          Info of item n is in the ring (1 arrival): a slot is written again only after the last S of item n + 2
//                         is complete, by when every warp is past item n                                       phase n >> 2
//   bar_c                 the answer to the n-th request for a block                                           phase n
//   GATHER: bar_gk[s], bar_gv[s] (32 arrivals, by cp.async completion) a gathered tile is in stage s; the TMA barriers then only
//           count the window tiles (their phases are followed by toggling)
// STREAM: the list is every entry that is retained at some query of a chunk, and entry e is gone from query leave[e] on (the
// streaming reading of a chunk): retained tiles take one more mask, leave > query position.
template <bool GATHER, bool STREAM>
__global__ void __launch_bounds__(NTHREADS, 2)
prefill_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                  const __grid_constant__ CUtensorMap tmKc, const __grid_constant__ CUtensorMap tmVc, const Args args,
                  const __nv_bfloat16* __restrict__ kg, const __nv_bfloat16* __restrict__ vg, const int32_t* __restrict__ idx,
                  const int32_t* __restrict__ cnt, __nv_bfloat16* __restrict__ og, float* __restrict__ lse,
                  const int32_t* __restrict__ leave, int R, float scale, int dg)
{
    using S = Smem<STREAM>;
    constexpr int KST = S::KST, VST = S::VST, TILE = S::TILE;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0) {                                 // the swizzled tiles need 1024-byte alignment
        if (threadIdx.x == 0) atomicExch(&g_prefill_status.code, 9);
        return;
    }
    const uint32_t sQ = base + S::OFF_Q, sK = base + S::OFF_K, sV = base + S::OFF_V;
    const uint32_t bar_q = base + S::OFF_BAR, bar_qf = bar_q + 16, bar_k = bar_q + 32, bar_kf = bar_q + 48, bar_v = bar_q + 64, bar_vf = bar_q + 80;
    const uint32_t bar_s = bar_q + 96, bar_sf = bar_q + 104, bar_p = bar_q + 112, bar_pv = bar_q + 120, bar_of = bar_q + 128, bar_c = bar_q + 136;
    const uint32_t bar_i = bar_q + 144, bar_gk = bar_q + 176, bar_gv = bar_q + 192, tmem_slot = bar_q + 208, answer = bar_q + 224;   // (answer: 16 bytes)
    auto slot = [&](int n) { return reinterpret_cast<volatile Info*>(smem_raw + S::OFF_INFO + (n & 3) * 64); };
    volatile uint32_t* tmem_slot_gen = reinterpret_cast<volatile uint32_t*>(smem_raw + S::OFF_BAR + 208);
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (so the compiler knows warp is uniform)

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_q + 8 * s, 1); mbar_init(bar_qf + 8 * s, 1);
            mbar_init(bar_k + 8 * s, 1); mbar_init(bar_kf + 8 * s, 1);
            mbar_init(bar_v + 8 * s, 1); mbar_init(bar_vf + 8 * s, 1);
            mbar_init(bar_gk + 8 * s, 32); mbar_init(bar_gv + 8 * s, 32);
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) mbar_init(bar_i + 8 * s, 1);
        mbar_init(bar_c, 1);
        mbar_init(bar_s, 1); mbar_init(bar_sf, 8); mbar_init(bar_p, 8); mbar_init(bar_pv, 1); mbar_init(bar_of, 8);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 8) tmem_alloc(tmem_slot, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_gen;
    pdl_launch_dependents();
    pdl_wait();                                                // everything above ran beside the previous kernel's tail

    if (warp == 9) {
        // ================================= load warp ========================================================
        // Keys run one tile ahead of values: K(g+1) is wanted at the start of softmax g, V(g) at its end.  The whole warp walks
        // the loop, lane 0 issues the copies.
        Cursor ck, cv;
        ItemQueue queue(answer, bar_c, lane);
        int pos_k[4], pos_v[4];                                // GATHER: positions of the rows of the key cursor's tile, of the tile before it
        auto fetch_positions = [&]() {                         // (of a retained tile)
            const int e0 = (ck.t - ck.it.n_win) * BN, n = cnt[ck.it.bhk];
            const int32_t* id = idx + (size_t)ck.it.bhk * R;
#pragma unroll
            for (int u = 0; u < 4; ++u) pos_k[u] = e0 + u * 32 + lane < n ? id[e0 + u * 32 + lane] : -1;
        };
        auto load = [&](const Cursor& c, bool is_v, uint32_t dst, uint32_t bar, uint32_t gbar) {
            const bool win = c.t < c.it.n_win;
            if (!GATHER || win) {
                if (lane == 0) {
                    mbar_expect_tx(bar, TILE);
                    tma_load_3d(dst, is_v ? (win ? &tmV : &tmVc) : (win ? &tmK : &tmKc), 0, win ? c.it.j_start + c.t * BN : (c.t - c.it.n_win) * BN, c.it.bhk, bar);
                }
            } else {                                           // 8 lanes per row copy its 16-byte pieces; rows past the list are zero
                const __nv_bfloat16* src = (is_v ? vg : kg) + (size_t)c.it.bhk * args.Tlen * dg;
                const int sub = lane & 7;
#pragma unroll
                for (int ps = 0; ps < 32; ++ps) {
                    const int row = ps * 4 + (lane >> 3), at = __shfl_sync(0xffffffffu, is_v ? pos_v[ps >> 3] : pos_k[ps >> 3], row & 31);
                    const bool real = at >= 0 && sub * 8 < dg; // (columns past the head dimension are zero-filled)
                    cp_async16(dst + row * 128 + ((sub ^ (row & 7)) << 4), src + (real ? (size_t)at * dg + sub * 8 : 0), real ? 16u : 0u);
                }
                cp_async_arrive(gbar);
            }
        };
        auto load_k = [&]() {
            const bool first = ck.t == 0;
            if (first) {
                // the item: this block's own, then whatever the last request brought
                const int item = ck.n > 0 ? queue.take(17, &g_prefill_status) : (int)blockIdx.x;
                const uint32_t b = ck.n & 1;
                if (ck.n >= 2) mbar_wait(bar_qf + 8 * b, ((ck.n >> 1) - 1) & 1, 12);
                if (item < 0) {
                    ck.live = false;
                    if (lane == 0) { slot(ck.n)->item = -1; mbar_arrive(bar_i + 8 * (ck.n & 3)); }
                    return;
                }
                ck.it = item_of(args, item);
                if (lane == 0) {
                    mbar_expect_tx(bar_q + 8 * b, TILE);
                    tma_load_3d(sQ + b * TILE, &tmQ, 0, ck.it.i0 - args.qoff, ck.it.bh, bar_q + 8 * b);
                }
            }
            if (GATHER && ck.t >= ck.it.n_win) fetch_positions();   // (never tile 0)
            const uint32_t s = ck.g % KST;
            if (ck.g >= (uint32_t)KST) mbar_wait(bar_kf + 8 * s, (ck.g / KST - 1) & 1u, 6);
            load(ck, false, sK + s * TILE, bar_k + 8 * s, bar_gk + 8 * s);
            if (first) {                                       // tile 0 is a window tile; the list is looked up while it is on its way
                const int last = min(ck.it.i0 + BM - 1, args.Tlen - 1) - ck.it.i0;   // rows 0 .. last see positions up to i0 - W .. i0 - W + last
                const ListView f = view_list(idx + (size_t)ck.it.bhk * R, cnt + ck.it.bhk, R, ck.it.i0 - args.W, last, lane);
                ck.it.n_tiles = ck.it.n_win + (f.all + BN - 1) / BN;
                if (lane == 0) {
                    volatile Info* o = slot(ck.n);
#pragma unroll
                    for (int k = 0; k < 4; ++k) { o->before[k] = f.before[k]; o->bits[k] = f.bits[k]; }
                    o->n_tiles = ck.it.n_tiles; o->item = ck.it.item;
                    mbar_arrive(bar_i + 8 * (ck.n & 3));
                }
            }
            if (ck.t == max(ck.it.n_tiles - kAskTiles, 0)) queue.ask();
            ck.advance();
        };
        load_k();
        for (;;) {
            if (GATHER) {
#pragma unroll
                for (int u = 0; u < 4; ++u) pos_v[u] = pos_k[u];
            }
            if (ck.live) load_k();
            if (cv.t == 0) {                                   // (written by this warp's lane 0: the key cursor is in or past this item)
                __syncwarp();
                const int item = slot(cv.n)->item;
                if (item < 0) break;
                cv.it = item_of(args, item);
                cv.it.n_tiles = slot(cv.n)->n_tiles;
            }
            const uint32_t s = cv.g % VST;
            if (cv.g >= (uint32_t)VST) mbar_wait(bar_vf + 8 * s, (cv.g / VST - 1) & 1u, 8);
            load(cv, true, sV + s * TILE, bar_v + 8 * s, bar_gv + 8 * s);
            cv.advance();
        }
        __syncwarp();
    } else if (warp == 8) {
        // ================================= MMA warp (an elected thread issues; the whole warp walks the loop) ====
        constexpr uint32_t IDESC_S = instr_desc(BM, BN, false), IDESC_O = instr_desc(BM, D, true);
        const uint32_t q_lo = desc_lo(sQ, 16), k_lo = desc_lo(sK, 16), v_lo = desc_lo(sV, 16);
        Cursor cs, cp;
        uint32_t par = 0;                                      // GATHER: parities of bar_k (bits 0, 1), bar_gk (2, 3), bar_v (4, 5), bar_gv (6, 7)
        auto landed = [&](uint32_t bar, uint32_t gbar, bool win, uint32_t s, uint32_t phase, int bit, int gbit, int code) {
            if (!GATHER) { mbar_wait_u(bar + 8 * s, phase, code); return; }
            const int at = (win ? bit : gbit) + (int)s;
            mbar_wait_u((win ? bar : gbar) + 8 * s, (par >> at) & 1u, code);
            par ^= 1u << at;
            if (!win) fence_proxy_async();                     // the copies were generic-proxy writes
        };
        auto enter = [&](Cursor& c) {                          // the cursor's next item out of the ring
            const int item = __shfl_sync(0xffffffffu, slot(c.n)->item, 0);
            c.live = item >= 0;
            if (!c.live) return;
            c.it = item_of(args, item);
            c.it.n_tiles = __shfl_sync(0xffffffffu, slot(c.n)->n_tiles, 0);
        };
        auto mma_s = [&]() {
            const uint32_t s = cs.g % KST, b = cs.n & 1;
            if (uni(cs.t == 0)) {
                mbar_wait_u(bar_i + 8 * (cs.n & 3), (cs.n >> 2) & 1, 9);
                enter(cs);
                if (uni(!cs.live)) return;
                mbar_wait_u(bar_q + 8 * b, (cs.n >> 1) & 1, 1);
            }
            landed(bar_k, bar_gk, cs.t < cs.it.n_win, s, (cs.g / KST) & 1u, 0, 2, 2);
            if (uni(cs.g > 0)) mbar_wait_u(bar_sf, (cs.g - 1) & 1, 3);    // the previous tile's S is in registers
            tc_fence_after();
            if (elect_one()) {
                const uint32_t qd = q_lo + b * (TILE >> 4), kd = k_lo + s * (TILE >> 4);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) umma(tmem + S_COL, desc64(qd + kk * 2, kDescHi), desc64(kd + kk * 2, kDescHi), IDESC_S, kk > 0);
                umma_commit(bar_s);
                umma_commit(bar_kf + 8 * s);
                if (cs.t == cs.it.n_tiles - 1) umma_commit(bar_qf + 8 * b);
            }
            __syncwarp();
            cs.advance();
        };
        mma_s();
        for (;;) {
            if (uni(cs.live)) mma_s();
            if (uni(cp.t == 0)) { enter(cp); if (uni(!cp.live)) break; }
            const uint32_t s = cp.g % VST;
            landed(bar_v, bar_gv, cp.t < cp.it.n_win, s, (cp.g / VST) & 1u, 4, 6, 4);
            if (uni(cp.t == 0 && cp.n > 0)) mbar_wait_u(bar_of, (cp.n - 1) & 1, 13);   // the previous item's O has been read out
            mbar_wait_u(bar_p, cp.g & 1, 7);
            tc_fence_after();
            if (elect_one()) {
                const uint32_t vd = v_lo + s * (TILE >> 4);
#pragma unroll
                for (int kk = 0; kk < BN / 16; ++kk)
                    umma_ts(tmem + O_COL, tmem + P_COL + kk * 8, desc64(vd + kk * 128, kDescHi), IDESC_O, (cp.t > 0 || kk > 0) ? 1u : 0u);
                umma_commit(bar_pv);
                umma_commit(bar_vf + 8 * s);
            }
            __syncwarp();
            cp.advance();
        }
    } else {
        // =================================== softmax warps ==================================================
        // Two threads per row: thread r of warps 0-3 takes columns [0, 64) of every tile, thread r of warps 4-7 columns [64, 128).
        const int hf = warp >> 2, row = tid & 127, c0 = hf * 64;
        const float c2 = scale * 1.4426950408889634f;          // logits are handled in the log2 domain: x = s * c2
        const uint64_t c2_2 = pack2(c2, c2);
        const uint32_t trow = tmem + (((uint32_t)((warp & 3) * 32)) << 16);   // this warp's TMEM lanes
        const uint32_t s_col = trow + S_COL + c0, p_col = trow + P_COL + hf * 32, o_col = trow + O_COL + hf * 32;
        float* x_mine = reinterpret_cast<float*>(smem_raw + S::OFF_X) + hf * BM + row;
        const float* x_other = reinterpret_cast<float*>(smem_raw + S::OFF_X) + (hf ^ 1) * BM + row;
        auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp & 3)) : "memory"); };   // the two warps of these rows
        uint32_t g = 0;
        int n = 0;
        // A row's output is read and stored while the next item's first tile is under way (its PV has then long completed).
        float last_m = 0.f;
        int last_row = -1;                                     // row of o and lse (-1: none)
        auto epilogue = [&](int item_no) {
            const float2* lsum = reinterpret_cast<const float2*>(smem_raw + S::OFF_L) + (item_no & 1) * 2 * BM + row;
            const float l = lsum[0].x + lsum[BM].x, inv = 1.f / (lsum[0].y + lsum[BM].y);
            __nv_bfloat16* orow = og + (size_t)last_row * dg + hf * 32;   // 64 contiguous bytes of the row
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                uint32_t o[16], x[8];
                tmem_ld16(o_col + cb * 16, o);
                tmem_wait_ld();
                if (cb == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_of);        // the accumulator may take the next item
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(o[2 * c]) * inv, __uint_as_float(o[2 * c + 1]) * inv);
                    x[c] = *reinterpret_cast<const uint32_t*>(&h);
                }
                if (last_row >= 0 && hf * 32 + cb * 16 < dg) {
                    *reinterpret_cast<uint4*>(orow + cb * 16) = make_uint4(x[0], x[1], x[2], x[3]);
                    *reinterpret_cast<uint4*>(orow + cb * 16 + 8) = make_uint4(x[4], x[5], x[6], x[7]);
                }
            }
            if (last_row >= 0 && hf == 0) lse[last_row] = last_m * 0.6931471805599453f + logf(l);
        };
        for (;; ++n) {
            mbar_wait(bar_i + 8 * (n & 3), (n >> 2) & 1, 15);
            const int item = __shfl_sync(0xffffffffu, slot(n)->item, 0);
            if (item < 0) break;
            const Item w = item_of(args, item);
            const int W = args.W, Tlen = args.Tlen;
            const int ia = w.i0 + (warp & 3) * 32, i = ia + lane;   // the warp's first query row, this thread's
            int nvis, n_tiles;                                 // retained entries this row sees (a prefix of the list), tiles of the item
            {
                const volatile Info* f = slot(n);
                const int x = min(i, Tlen - 1) - w.i0;
                nvis = (int)(f->before[x >> 5] + __popc(f->bits[x >> 5] & ((1u << (x & 31)) - 1u)));
                n_tiles = f->n_tiles;
            }
            n_tiles = __shfl_sync(0xffffffffu, n_tiles, 0);
            const int nvis_first = __shfl_sync(0xffffffffu, nvis, 0), nvis_last = __shfl_sync(0xffffffffu, nvis, 31);
            float m_run = -INFINITY;                           // reference (log2 domain), the same in both halves
            uint64_t ls = 0ull;                                // sums of this half of the row, even and odd columns: of the weights ...
            float lr[2] = {0.f, 0.f};                          // ... and of P, which is the weights in bf16

            for (int t = 0; t < n_tiles; ++t, ++g) {
                // columns (of this half) the row may see in the tile, and (the bounds grow with the row, so the warp's first and
                // last row give them) the columns any row and every row of the warp may see
                int c_lo, c_hi, u_lo, u_hi, n_lo, n_hi;
                if (t < w.n_win) {
                    const int jt0 = w.j_start + t * BN + c0;
                    c_lo = max(i - W + 1, 0) - jt0; c_hi = i - jt0;
                    u_lo = max(ia - W + 1, 0) - jt0; n_lo = max(ia + 31 - W + 1, 0) - jt0;
                    n_hi = ia - jt0; u_hi = ia + 31 - jt0;
                } else {
                    const int e0 = (t - w.n_win) * BN + c0;
                    c_lo = u_lo = n_lo = 0;
                    c_hi = nvis - e0 - 1; n_hi = nvis_first - e0 - 1; u_hi = nvis_last - e0 - 1;
                }
                const bool timed = STREAM && t >= w.n_win;
                if (timed) {                                   // the leave times of this half of the tile go through a per-warp scratch
                    int* slv = reinterpret_cast<int*>(smem_raw + S::OFF_LV) + warp * 64;
                    const int e0 = (t - w.n_win) * BN + c0;
                    const int32_t* lvp = leave + (size_t)w.bhk * R;
                    __syncwarp();                              // the previous tile's readers are done
#pragma unroll
                    for (int u = 0; u < 2; ++u) slv[u * 32 + lane] = e0 + u * 32 + lane < R ? lvp[e0 + u * 32 + lane] : 0;
                    __syncwarp();
                }
                bool act[2], plain[2];
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    act[cb] = cb * 32 <= u_hi && cb * 32 + 31 >= u_lo;
                    plain[cb] = cb * 32 >= n_lo && cb * 32 + 31 <= n_hi && !timed;
                }
                auto mask_of = [&](int cb) {                   // this row's columns of a chunk that needs a mask
                    const int a = min(max(c_lo - cb * 32, 0), 32), b = min(max(c_hi - cb * 32 + 1, 0), 32);
                    const uint32_t below_b = b >= 32 ? 0xffffffffu : ((1u << b) - 1u), below_a = a >= 32 ? 0xffffffffu : ((1u << a) - 1u);
                    uint32_t vm = b > a ? (below_b & ~below_a) : 0u;
                    if (timed) {
                        const int* slv = reinterpret_cast<const int*>(smem_raw + S::OFF_LV) + warp * 64 + cb * 32;
                        uint32_t m = 0;
#pragma unroll
                        for (int c = 0; c < 32; c += 4) {
                            const int4 l4 = *reinterpret_cast<const int4*>(slv + c);
                            m |= (l4.x > i ? 1u : 0u) << c; m |= (l4.y > i ? 2u : 0u) << c;
                            m |= (l4.z > i ? 4u : 0u) << c; m |= (l4.w > i ? 8u : 0u) << c;
                        }
                        vm &= m;
                    }
                    return vm;
                };
                auto apply = [&](uint32_t (&x)[32], uint32_t vm) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) x[c] = (vm & (1u << c)) ? x[c] : 0xff800000u;   // -inf
                };
                float mr[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                auto max_of = [&](const uint32_t (&x)[32]) {
#pragma unroll
                    for (int c = 0; c < 32; c += 2) mr[(c >> 1) & 3] = max3(mr[(c >> 1) & 3], __uint_as_float(x[c]), __uint_as_float(x[c + 1]));
                };
                mbar_wait(bar_s, g & 1, 5);
                tc_fence_after();
                // Chunk 0 passes through for the maximum and is fetched again after the exponentials of chunk 1 (32 logits at a time
                // and the loop's state are what fits in the 96 registers there are).
                uint32_t x[32], vm0 = 0xffffffffu;
                if (act[0]) {
                    tmem_ld32(s_col, x);
                    tmem_wait_ld();
                    if (!plain[0]) { vm0 = mask_of(0); apply(x, vm0); }
                    max_of(x);
                }
                if (act[1]) {
                    tmem_ld32(s_col + 32, x);
                    tmem_wait_ld();
                    if (!plain[1]) apply(x, mask_of(1));
                    max_of(x);
                }
                float m_tile = fmaxf(fmaxf(mr[0], mr[1]), fmaxf(mr[2], mr[3])) * c2;
                x_mine[(g & 1) * 2 * BM] = m_tile;
                pair_sync();
                m_tile = fmaxf(m_tile, x_other[(g & 1) * 2 * BM]);
                // lazy rescale: the reference only moves when the maximum is far above it (exp2 arguments stay <= 8)
                float alpha = 1.f;
                bool need = false;
                if (m_run == -INFINITY) m_run = m_tile;        // nothing accumulated yet for this row: its O is 0
                else if (m_tile > m_run + 8.f) { alpha = fast_exp2(m_run - m_tile); m_run = m_tile; need = true; }
                if (__any_sync(0xffffffffu, need)) {
                    if (t > 0) {                               // PV of the previous tile must be done before O is rescaled
                        mbar_wait(bar_pv, (g - 1) & 1, 10);
                        tc_fence_after();
#pragma unroll 1
                        for (int cb = 0; cb < 2; ++cb) {       // (rolled, in small pieces: rarely taken, and S holds the registers)
                            uint32_t q4[16];
                            tmem_ld16(o_col + cb * 16, q4);
                            tmem_wait_ld();
#pragma unroll
                            for (int c = 0; c < 16; ++c) q4[c] = __float_as_uint(__uint_as_float(q4[c]) * alpha);
                            tmem_st16(o_col + cb * 16, q4);
                        }
                        tmem_wait_st();
                    }
                    const uint64_t a2 = pack2(alpha, alpha);
                    ls = mul2(ls, a2); lr[0] *= alpha; lr[1] *= alpha;
                }
                const float neg_m = m_run == -INFINITY ? 0.f : -m_run;
                const uint64_t neg_m2 = pack2(neg_m, neg_m);
                auto exps = [&](const uint32_t (&x)[32], uint32_t (&pk)[16]) {
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        // masked entries hold -inf: fma gives -inf and exp2(-inf) = 0
                        float x0, x1;                          // two columns per packed fp32 instruction
                        unpack2(fma2(pack2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), c2_2, neg_m2), x0, x1);
                        const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        ls = add2(ls, pack2(p0, p1));
                        const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
                        pk[c >> 1] = *reinterpret_cast<const uint32_t*>(&h);
                        add_bf16x2(lr[0], lr[1], pk[c >> 1]);
                    }
                };
                uint32_t pk[16];                               // 32 columns of the row of P, two per word
                if (act[1]) exps(x, pk);
                else
#pragma unroll
                    for (int c = 0; c < 16; ++c) pk[c] = 0u;
                if (act[0]) tmem_ld32(s_col, x);
                // P(g) takes the place of P(g-1), whose product has normally completed long ago; every phase is awaited in turn
                if (g > 0) { mbar_wait(bar_pv, (g - 1) & 1, 11); tc_fence_after(); }
                tmem_st16(p_col + 16, pk);
                if (t == 0 && n > 0) epilogue(n - 1);          // the previous item's
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_sf);            // S(g+1) may overwrite the buffer
                if (act[0]) {
                    if (!plain[0]) apply(x, vm0);
                    exps(x, pk);
                } else {
#pragma unroll
                    for (int c = 0; c < 16; ++c) pk[c] = 0u;
                }
                tmem_st16(p_col, pk);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p);
            }
            float l0, l1;
            unpack2(ls, l0, l1);
            // (read after the pair's next barrier; written again two items on)
            reinterpret_cast<float2*>(smem_raw + S::OFF_L)[(n & 1) * 2 * BM + hf * BM + row] = make_float2(l0 + l1, lr[0] + lr[1]);
            last_m = m_run;
            last_row = i < Tlen ? w.bh * (Tlen - args.qoff) + (i - args.qoff) : -1;
        }
        pair_sync();
        mbar_wait(bar_pv, (g - 1) & 1, 14);
        tc_fence_after();
        epilogue(n - 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace

static int launch_d64(const Params& p, const void* q, const void* k, const void* v, const int32_t* idx, const int32_t* cnt, void* o,
                      float* lse, void* ws, size_t ws_bytes, cudaStream_t st, const int32_t* leave)
{
    // with a workspace the retained rows are compacted first and every tile is a TMA box
    const size_t half = prefill_compact_bytes(p) / 2;
    const bool compact = ws != nullptr && half > 0 && ws_bytes >= 2 * half && ((uintptr_t)ws & 127u) == 0;
    if (leave && !compact) return LTE_ERR_UNSUPPORTED;
    CUtensorMap tq, tk, tv, tkc, tvc;
    const int BHK = p.B * p.H, BH = BHK * p.G, Tq = p.T - p.qoff;   // key/value heads, query heads, query rows
    if (!make_map(&tq, q, BH, Tq, p.d, BM) || !make_map(&tk, k, BHK, p.T, p.d, BN) || !make_map(&tv, v, BHK, p.T, p.d, BN)) return LTE_ERR_CUDA;
    tkc = tk; tvc = tv;
    if (compact) {
        char* kc = (char*)ws; char* vc = kc + half;
        if (int e = launch_prefill_compact(p, k, v, idx, cnt, kc, vc, st)) return e;
        if (!make_map(&tkc, kc, BHK, p.R, p.d, BN) || !make_map(&tvc, vc, BHK, p.R, p.d, BN)) return LTE_ERR_CUDA;
    }
    static PerDeviceOnce attr;
    if (int e = attr.run([] {
            cudaError_t a = cudaFuncSetAttribute(prefill_tc_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<false>::BYTES);
            if (a == cudaSuccess) a = cudaFuncSetAttribute(prefill_tc_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<false>::BYTES);
            return a != cudaSuccess ? a : cudaFuncSetAttribute(prefill_tc_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<true>::BYTES);
        })) return e;
    Args a;
    a.n_qt = (Tq + BM - 1) / BM; a.n_bh = BH; a.n_items = a.n_qt * BH; a.Tlen = p.T; a.W = p.W; a.G = p.G; a.qoff = p.qoff;
    auto go = [&](auto kern, int smem) {
        return cuda_status(launch_pdl(kern, dim3(a.n_items), dim3(NTHREADS), smem, st, tq, tk, tv, tkc, tvc, a, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v,
                                      idx, cnt, (__nv_bfloat16*)o, lse, leave, p.R, p.scale, p.d));
    };
    if (leave) return go(prefill_tc_kernel<false, true>, Smem<true>::BYTES);
    return compact ? go(prefill_tc_kernel<false, false>, Smem<false>::BYTES) : go(prefill_tc_kernel<true, false>, Smem<false>::BYTES);
}

// leave: null, or the streaming reading's per-entry leave times (with a workspace the tiled kernels; otherwise the row-by-row
// kernel)
int launch_prefill_tc(const Params& p, const void* q, const void* k, const void* v, const int32_t* idx,
                      const int32_t* cnt, void* o, float* lse, void* ws, size_t ws_bytes, cudaStream_t st, const int32_t* leave)
{
    int e = LTE_ERR_UNSUPPORTED;
    if (p.d == 64 || p.d == 32) e = launch_d64(p, q, k, v, idx, cnt, o, lse, ws, ws_bytes, st, leave);
    else if (p.d == 128) e = launch_prefill_tc_long(p, q, k, v, idx, cnt, o, lse, ws, ws_bytes, st, leave);
    return e != LTE_ERR_UNSUPPORTED ? e : launch_prefill_simt(p, q, k, v, idx, cnt, o, lse, st, leave);
}

int prefill_status_fetch_and_clear()
{
    const int h = status_fetch_and_clear(g_prefill_status), h2 = prefill_long_status_fetch_and_clear(), h3 = prefill_pair_status_fetch_and_clear();
    return h != 0 ? h : h2 != 0 ? h2 : h3;
}

}  // namespace lte
