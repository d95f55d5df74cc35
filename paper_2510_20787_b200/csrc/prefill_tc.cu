// Prefill attention on the 5th-generation tensor cores for bf16, d = 64 and d = 32 (Section 3.1.3, "Cached prefilling and
// decoding").
//
// Bound by the latencies of the softmax warps' chain (load, maximum, exponentials, store) and by their instructions (7 a weight, of which
// the arithmetic is 4; with items of ten window tiles and up to three of the list issue 51 %, exponential unit 60 %, tensor pipe 36 %), so a row belongs to one thread, which
// waits for no other, and nothing waits that need not:
//   work      Two CTAs per SM; an item is a 128-query tile of one head.  Key/value tiles of 96 rows come by TMA, first the window
//             span, then the head's retained rows that any of the item's rows may see (compacted beforehand where the caller
//             brought a workspace; otherwise the load warp gathers them row by row into the same swizzled layout).  Four softmax
//             warps (a thread per row), one warp issuing the products, one issuing the loads.
//   S(g) = Q K^T    two buffers, and P(g) takes the place of S(g): S(g+2) is issued when P V of tile g is complete (products of different
//             accumulators need not keep their order; the wait costs 0.3 % at the first shape below, nothing at the others), so S(g+1) is
//             there when a warp comes to it.  96 columns because two such buffers and O fill the 256 TMEM columns of a CTA: S [0,96), [96,192), O [192,256)
//   softmax   mask from positions.  A tile that all of the warp's rows see is taken whole (its 96 logits in registers, one vote); others
//             go in chunks of 32 columns, which are skipped where no row sees any, twice: for the tile's maximum and for the weights.  The
//             reference is the maximum of the first tile seen and moves to a later tile's that is more than 2^4 above it (in an item's
//             first tiles 2); exp2 with the scale folded in.  O is divided by the sum of P, so that its rounding cancels as far as it is
//             common to the row, and lse is the logarithm of the sum of the weights themselves (with the weights' sum alone O's error is
//             2 % larger, with P's alone lse's 1e-3).
//   O += P V  P as the TMEM A operand, V as the MN-major shared-memory operand; O is read and stored under the next item's first tile
// How many retained entries a row sees: the load warp finds an item's place in the list (a 32-way search) and hands out, one
// item ahead, a bit map of the entries that fall between the limits of the item's first and last row.
// Tiles are numbered through all items of a CTA (g); stage, buffer and barrier phase follow from that number, and the loads
// and products of the next item run under the current one.  Every mbarrier wait is bounded; one that runs out records a
// status word and the kernel still terminates.
//
// Measured (B200, the call with a workspace, back to back in a CUDA graph; before: two threads per row, 128-key tiles, one S buffer), logits of
// N(0,1/64) / N(0,1) / N(0,4), which move the reference the more often the wider they are:
//   128 query heads x 4,096, W = 768, R = 512 half used     176 / 181 / 191 us (611 TFLOP/s), before 196 / 196 / 199
//   64 heads x 4,096, W = R = 128                          45 / 46 / 48 us, before 49 / 49 / 50
//   128 x 2,048, W = R = 64                                37 / 37 / 38 us, before 44 / 44 / 47
//   48 x 3,001, W = 300, R = 200                           39 / 40 / 41 us, before 44 / 44 / 45
// O's error against 64 bits, logits of N(0,1) rising by 0 to 1 per key, W = 64 to 768: 0.962 to 0.9995 times what it was, 1.000 to 1.022 times
// that of weights rounded beside each row's own maximum (tests/test_gpu_prefill_rounding.py).  A reference that follows from 2^2 on makes
// that 0.945 to 0.998 and 1.006, the first line 176 / 194 / 202 us.  Without the look at a partial tile's maximum, chunk by chunk, with
// a reference that moves within a tile from 2^8 on and what is there of P rescaled (rounded a second time): 177 / 188 / 188, 45 / 53 / 54,
// 37 / 42 / 42, and O's error up to 1.04 times what it was.  The maximum in a pass of its own, all chunks fetched again: 183, 49, 40, 41;
// partial tiles' chunks all in registers, on one path with whole tiles: 190, 45, 36, 40.
// Tried and slower, the first line unless said otherwise: every tile in rolled chunks (192 us; the small windows 43 and 35), every tile
// whole (183; 48 and 39), the next tile's logits fetched ahead (194), the maximum asked only behind the exponentials (193), tiles of 80
// keys with the sum of P as sixteen columns more of the product (188), four CTAs per SM with one S buffer and 64-key tiles (181; 44 and 38),
// the sums of P by mma.sync (10 % more: it contends with tcgen05).  A longer loop costs more than it saves: the warps of an SM run different
// code and wait for instructions (the exponentials written out twice, 296 us).
//
// d = 32 runs the same kernel: the tensor maps describe 32-column rows with a 64-column box, the copy engine fills the upper
// half of every tile row with zeros, and only the first 32 output columns are stored.
#include "tile_items.cuh"

namespace lte {

__device__ StatusWord g_prefill_status = LTE_STATUS_INIT;         // 0 = fine; otherwise the code of the wait that gave up

namespace {

constexpr int BM = 128, BN = 96, D = 64, NTHREADS = 192;          // warps 0-3 softmax, 4 products, 5 loads
constexpr int W_MMA = 4, W_LOAD = 5, CHUNKS = BN / 32;
using namespace tc;
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, int code) { mbar_wait_call(bar, parity, code, &g_prefill_status); }
__device__ __forceinline__ void mbar_wait_u(uint32_t bar, uint32_t parity, int code) { mbar_wait_uni_call(bar, parity, code, &g_prefill_status); }

constexpr int QTILE = BM * D * 2, TILE = BN * D * 2;               // [128][64], [96][64] bf16
constexpr int QST = 2, KST = 3, VST = 3;                           // buffers of Q (by item), stages of K and V
constexpr int OFF_Q = 0, OFF_K = QST * QTILE, OFF_V = OFF_K + KST * TILE, OFF_BAR = OFF_V + VST * TILE;
constexpr int OFF_INFO = OFF_BAR + 320;                            // ring of four items' Info
constexpr int OFF_LV = OFF_INFO + 4 * 64;                          // STREAM: the leave times of a retained tile, [4 warps][96]
constexpr int smem_bytes(bool stream) { return OFF_LV + (stream ? 4 * BN * 4 : 0); }
constexpr uint32_t TMEM_COLS = 256, S_COL = 0, O_COL = 2 * BN, P_AT = BN / 2;   // two S buffers, P in the second half of its S

// An item: a 128-query tile of one (b,h).  Items are numbered from the last query tile of every head down to the first: later
// tiles see more retained rows and cost more.  The grid has a block per item, but a block that has run out of work takes the
// next block that has not started (cluster launch control) instead of leaving, so items are handed out in order, largest
// first, to whoever is free: dealt out beforehand, the blocks finished up to 30 % apart (159 to 219 us).
struct Item { int bh, bhk, i0, j_start, n_win, n_tiles; };   // bh: query head (b, h, g); bhk: its key/value head (b, h)
struct Args { int n_items, n_qt, n_bh, Tlen, W, G, qoff; };
// What the load warp tells the others about an item.  Row x of the item (0 .. 127) sees before[x / 32] entries and those of
// bits[x / 32] below bit x % 32.
struct Info { uint32_t before[4], bits[4]; int n_tiles, n_win, bh, bhk, i0, j_start; };   // n_tiles = 0: there is no item

__device__ __forceinline__ Item item_of(const Args& a, int item)
{
    Item it;
    const int r = item / a.n_bh;
    it.bh = item - r * a.n_bh;
    it.bhk = it.bh / a.G;
    it.i0 = a.qoff + (a.n_qt - 1 - r) * BM;                    // positions; the query tensors start at position qoff
    const int i_hi = min(it.i0 + BM - 1, a.Tlen - 1);
    it.j_start = max(it.i0 - a.W + 1, 0);
    it.n_win = (i_hi - it.j_start + BN) / BN;
    it.n_tiles = it.n_win;                                     // until the item's Info is there
    return it;
}
struct Ring {                                                  // a stage and the parity of its laps
    uint32_t s, lap;
    template <int N> __device__ __forceinline__ void next() { if (++s == (uint32_t)N) { s = 0; lap ^= 1u; } }
};
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

// Barriers (g = tile number, n = item number within the CTA):
//   bar_q[b], bar_qf[b]   Q of item n has landed in buffer b = n & 1 (TMA) / the item's last S is complete (commit)    phase n >> 1
//   bar_k[s], bar_v[s]    TMA of tile g into stage s = g % stages                                                       phase g / stages
//   bar_kf[s], bar_vf[s]  (commit) the product that read the stage's tile is complete                                   phase g / stages
//   bar_s[b] (commit)     S(g) is in TMEM buffer b = g & 1  bar_p[b] (4 arrivals)  P(g) has taken its place              phase g >> 1
//   bar_pv[b] (commit)    PV(g) is complete, b = g & 1: awaited by who has seen S(g + 1), behind PV(g - 1), or S(g), behind PV(g - 2)   phase g >> 1
//   bar_of   (4 arrivals) O of item n has been read out                                                                phase n
//   bar_i[n & 3]          Info of item n is in the ring (1 arrival): a slot is written again only after the last S of item n + 2
//                         is complete; that S is issued behind the product of the tile two before it, which belongs to item n or a
//                         later one, so every warp has read the slot by then   phase n >> 2
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
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0) {                                 // the swizzled tiles need 1024-byte alignment
        if (threadIdx.x == 0) atomicExch(&g_prefill_status.code, 9);
        return;
    }
    const uint32_t sQ = base + OFF_Q, sK = base + OFF_K, sV = base + OFF_V, bars = base + OFF_BAR;
    const uint32_t bar_q = bars, bar_qf = bars + 16, bar_k = bars + 32, bar_kf = bars + 56, bar_v = bars + 80, bar_vf = bars + 104;
    const uint32_t bar_gk = bars + 128, bar_gv = bars + 152, bar_s = bars + 176, bar_p = bars + 192, bar_i = bars + 208;
    const uint32_t bar_pv = bars + 240, bar_of = bars + 256, bar_c = bars + 264, tmem_slot = bars + 272, answer = bars + 288;   // (answer: 16 bytes)
    auto slot = [&](int n) { return reinterpret_cast<volatile Info*>(smem_raw + OFF_INFO + (n & 3) * 64); };
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (so the compiler knows warp is uniform)

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_q + 8 * s, 1); mbar_init(bar_qf + 8 * s, 1);
            mbar_init(bar_s + 8 * s, 1); mbar_init(bar_p + 8 * s, 4);
        }
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            mbar_init(bar_k + 8 * s, 1); mbar_init(bar_kf + 8 * s, 1);
            mbar_init(bar_v + 8 * s, 1); mbar_init(bar_vf + 8 * s, 1);
            mbar_init(bar_gk + 8 * s, 32); mbar_init(bar_gv + 8 * s, 32);
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) mbar_init(bar_i + 8 * s, 1);
        mbar_init(bar_c, 1); mbar_init(bar_pv, 1); mbar_init(bar_pv + 8, 1); mbar_init(bar_of, 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) tmem_alloc(tmem_slot, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem_raw + OFF_BAR + 272);
    pdl_launch_dependents();
    pdl_wait();                                                // everything above ran beside the previous kernel's tail

    if (warp == W_LOAD) {
        // ================================= load warp ========================================================
        // Keys run two tiles ahead of values: S(g+2) is computed right behind P V of tile g.  The whole warp walks the loop, lane 0
        // issues the copies.
        Cursor ck, cv;
        Ring rk{}, rv{};
        ItemQueue queue(answer, bar_c, lane);
        int pos_k[CHUNKS], pos_n[CHUNKS], pos_v[CHUNKS];       // GATHER: positions of the rows of the key cursor's tile, of the two tiles before it
        auto fetch_positions = [&]() {                         // (of a retained tile)
            const int e0 = (ck.t - ck.it.n_win) * BN, n = cnt[ck.it.bhk];
            const int32_t* id = idx + (size_t)ck.it.bhk * R;
#pragma unroll
            for (int u = 0; u < CHUNKS; ++u) pos_k[u] = e0 + u * 32 + lane < n ? id[e0 + u * 32 + lane] : -1;
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
                for (int ps = 0; ps < BN / 4; ++ps) {
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
                    if (lane == 0) { slot(ck.n)->n_tiles = 0; mbar_arrive(bar_i + 8 * (ck.n & 3)); }
                    return;
                }
                ck.it = item_of(args, item);
                if (lane == 0) {
                    mbar_expect_tx(bar_q + 8 * b, QTILE);
                    tma_load_3d(sQ + b * QTILE, &tmQ, 0, ck.it.i0 - args.qoff, ck.it.bh, bar_q + 8 * b);
                }
            }
            if (GATHER && ck.t >= ck.it.n_win) fetch_positions();   // (never tile 0)
            const uint32_t s = rk.s;
            if (ck.g >= (uint32_t)KST) mbar_wait(bar_kf + 8 * s, rk.lap ^ 1u, 6);
            rk.next<KST>();
            load(ck, false, sK + s * TILE, bar_k + 8 * s, bar_gk + 8 * s);
            if (first) {                                       // tile 0 is a window tile; the list is looked up while it is on its way
                const int last = min(ck.it.i0 + BM - 1, args.Tlen - 1) - ck.it.i0;   // rows 0 .. last see positions up to i0 - W .. i0 - W + last
                const ListView f = view_list(idx + (size_t)ck.it.bhk * R, cnt + ck.it.bhk, R, ck.it.i0 - args.W, last, lane);
                ck.it.n_tiles = ck.it.n_win + (f.all + BN - 1) / BN;
                if (lane == 0) {
                    volatile Info* o = slot(ck.n);
#pragma unroll
                    for (int k = 0; k < 4; ++k) { o->before[k] = f.before[k]; o->bits[k] = f.bits[k]; }
                    o->n_tiles = ck.it.n_tiles; o->n_win = ck.it.n_win; o->bh = ck.it.bh; o->bhk = ck.it.bhk; o->i0 = ck.it.i0; o->j_start = ck.it.j_start;
                    mbar_arrive(bar_i + 8 * (ck.n & 3));
                }
            }
            if (ck.t == max(ck.it.n_tiles - kAskTiles, 0)) queue.ask();
            ck.advance();
        };
        auto next_positions = [&]() {
            if (GATHER) {
#pragma unroll
                for (int u = 0; u < CHUNKS; ++u) { pos_v[u] = pos_n[u]; pos_n[u] = pos_k[u]; }
            }
        };
        load_k();
        next_positions();
        load_k();
        for (;;) {
            next_positions();
            if (ck.live) load_k();
            if (cv.t == 0) {                                   // (written by this warp's lane 0: the key cursor is in or past this item)
                __syncwarp();
                const volatile Info* f = slot(cv.n);
                cv.it.n_tiles = f->n_tiles; cv.it.n_win = f->n_win; cv.it.bhk = f->bhk; cv.it.j_start = f->j_start;
                if (cv.it.n_tiles == 0) break;
            }
            const uint32_t s = rv.s;
            if (cv.g >= (uint32_t)VST) mbar_wait(bar_vf + 8 * s, rv.lap ^ 1u, 8);
            rv.next<VST>();
            load(cv, true, sV + s * TILE, bar_v + 8 * s, bar_gv + 8 * s);
            cv.advance();
        }
        __syncwarp();
    } else if (warp == W_MMA) {
        // ================================= MMA warp (an elected thread issues; the whole warp walks the loop) ====
        constexpr uint32_t IDESC_S = instr_desc(BM, BN, false), IDESC_O = instr_desc(BM, D, true);
        const uint32_t q_lo = desc_lo(sQ, 16), k_lo = desc_lo(sK, 16), v_lo = desc_lo(sV, 16);
        uint32_t par = 0;                                      // GATHER: parities of bar_k (bits 0-2), bar_gk (3-5), bar_v (6-8), bar_gv (9-11)
        auto landed = [&](uint32_t bar, uint32_t gbar, bool win, const Ring& r, int bit, int gbit, int code) {
            if (!GATHER) { mbar_wait_u(bar + 8 * r.s, r.lap, code); return; }
            const int at = (win ? bit : gbit) + (int)r.s;
            mbar_wait_u((win ? bar : gbar) + 8 * r.s, (par >> at) & 1u, code);
            par ^= 1u << at;
            if (!win) fence_proxy_async();                     // the copies were generic-proxy writes
        };
        struct Walk { Ring r; int n, t, n_tiles, n_win; uint32_t g; } ws{}, wp{};   // S and P V: stage, item, tile of the item, its tiles
        auto enter = [&](Walk& c) {                            // the next item out of the ring
            c.t = 0;
            c.n_tiles = __shfl_sync(0xffffffffu, slot(c.n)->n_tiles, 0);
            if (GATHER) c.n_win = __shfl_sync(0xffffffffu, slot(c.n)->n_win, 0);
        };
        auto mma_s = [&]() {                                   // false: there is no further tile
            if (uni(ws.t == ws.n_tiles)) {
                if (ws.g > 0) ++ws.n;
                mbar_wait_u(bar_i + 8 * (ws.n & 3), (ws.n >> 2) & 1, 9);
                enter(ws);
                if (uni(ws.n_tiles == 0)) return false;
                mbar_wait_u(bar_q + 8 * (ws.n & 1), (ws.n >> 1) & 1, 1);
            }
            landed(bar_k, bar_gk, ws.t < ws.n_win, ws.r, 0, 3, 2);
            ++ws.t;
            tc_fence_after();
            const uint32_t s_tm = tmem + S_COL + (ws.g & 1) * BN;    // P of the tile two before, which lay there, has been multiplied
            if (elect_one()) {
                const uint32_t qd = q_lo + (ws.n & 1) * (QTILE >> 4), kd = k_lo + ws.r.s * (TILE >> 4);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) umma(s_tm, desc64(qd + kk * 2, kDescHi), desc64(kd + kk * 2, kDescHi), IDESC_S, kk > 0);
                umma_commit(bar_s + 8 * (ws.g & 1));
                umma_commit(bar_kf + 8 * ws.r.s);
                if (ws.t == ws.n_tiles) umma_commit(bar_qf + 8 * (ws.n & 1));
            }
            __syncwarp();
            ++ws.g; ws.r.next<KST>();
            return true;
        };
        mma_s();
        bool more = mma_s();
        for (;;) {
            if (uni(wp.t == wp.n_tiles)) {
                if (wp.g > 0) ++wp.n;
                enter(wp);
                if (uni(wp.n_tiles == 0)) break;
                if (uni(wp.n > 0)) mbar_wait_u(bar_of, (wp.n - 1) & 1, 13);   // the previous item's O has been read out
            }
            landed(bar_v, bar_gv, wp.t < wp.n_win, wp.r, 6, 9, 4);
            mbar_wait_u(bar_p + 8 * (wp.g & 1), (wp.g >> 1) & 1u, 7);
            tc_fence_after();
            if (elect_one()) {
                const uint32_t vd = v_lo + wp.r.s * (TILE >> 4), p_tm = tmem + S_COL + (wp.g & 1) * BN + P_AT;
#pragma unroll
                for (int kk = 0; kk < BN / 16; ++kk)
                    umma_ts(tmem + O_COL, p_tm + kk * 8, desc64(vd + kk * 128, kDescHi), IDESC_O, (wp.t > 0 || kk > 0) ? 1u : 0u);
                umma_commit(bar_pv + 8 * (wp.g & 1));
                umma_commit(bar_vf + 8 * wp.r.s);
            }
            __syncwarp();
            if (uni(more)) {                                   // the next S but one takes the place of the P that this product reads
                mbar_wait_u(bar_pv + 8 * (wp.g & 1), (wp.g >> 1) & 1, 3);
                more = mma_s();
            }
            ++wp.t; ++wp.g; wp.r.next<VST>();
        }
    } else {
        // =================================== softmax warps ==================================================
        // Thread r takes row r of every tile.
        const float c2 = scale * 1.4426950408889634f;          // logits are handled in the log2 domain: x = s * c2
        const uint64_t c2_2 = pack2(c2, c2);
        const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16), o_col = trow + O_COL;   // this warp's TMEM lanes
        uint32_t g = 0;
        int n = 0;
        // A row's output is read and stored while the next item's first tile is under way (its PV has then long completed).
        float last_m = 0.f, last_l = 0.f, last_r = 1.f;
        int last_row = -1;                                     // row of o and lse (-1: none)
        auto epilogue = [&]() {
            const float inv = 1.f / last_r;
            __nv_bfloat16* orow = og + (size_t)last_row * dg;
#pragma unroll 1
            for (int cb = 0; cb < 4; ++cb) {
                uint32_t o[16], x[8];
                tmem_ld16(o_col + cb * 16, o);
                tmem_wait_ld();
                if (cb == 3) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_of);        // the accumulator may take the next item
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(o[2 * c]) * inv, __uint_as_float(o[2 * c + 1]) * inv);
                    x[c] = *reinterpret_cast<const uint32_t*>(&h);
                }
                if (last_row >= 0 && cb * 16 < dg) {
                    *reinterpret_cast<uint4*>(orow + cb * 16) = make_uint4(x[0], x[1], x[2], x[3]);
                    *reinterpret_cast<uint4*>(orow + cb * 16 + 8) = make_uint4(x[4], x[5], x[6], x[7]);
                }
            }
            if (last_row >= 0) lse[last_row] = last_m * 0.6931471805599453f + logf(last_l);
        };
        for (;; ++n) {
            mbar_wait(bar_i + 8 * (n & 3), (n >> 2) & 1, 15);
            const volatile Info* f = slot(n);
            const int n_tiles = __shfl_sync(0xffffffffu, f->n_tiles, 0);
            if (n_tiles == 0) break;
            Item w;
            w.bh = __shfl_sync(0xffffffffu, f->bh, 0); w.bhk = __shfl_sync(0xffffffffu, f->bhk, 0); w.i0 = __shfl_sync(0xffffffffu, f->i0, 0);
            w.j_start = __shfl_sync(0xffffffffu, f->j_start, 0); w.n_win = __shfl_sync(0xffffffffu, f->n_win, 0);
            const int W = args.W, Tlen = args.Tlen;
            const int ia = w.i0 + warp * 32, i = ia + lane;    // the warp's first query row, this thread's
            const int x_row = min(i, Tlen - 1) - w.i0;
            const int nvis = (int)(f->before[x_row >> 5] + __popc(f->bits[x_row >> 5] & ((1u << (x_row & 31)) - 1u)));   // retained entries this row sees (a prefix of the list)
            const int nvis_first = __shfl_sync(0xffffffffu, nvis, 0), nvis_last = __shfl_sync(0xffffffffu, nvis, 31);
            float m_run = -INFINITY;                           // reference (log2 domain); -inf: the row has seen nothing yet
            uint64_t ls[2] = {0ull, 0ull};                     // sums of the row, a quarter of the columns each: of the weights ...
            float lr[2] = {0.f, 0.f};                          // ... and of P, which is the weights in bf16

            for (int t = 0; t < n_tiles; ++t, ++g) {
                // columns the row may see in the tile, and (the bounds grow with the row, so the warp's first and last row give them)
                // the columns any row and every row of the warp may see
                int c_lo, c_hi, u_lo, u_hi, n_lo, n_hi;
                if (t < w.n_win) {
                    const int jt0 = w.j_start + t * BN;
                    c_lo = max(i - W + 1, 0) - jt0; c_hi = i - jt0;
                    u_lo = max(ia - W + 1, 0) - jt0; n_lo = max(ia + 31 - W + 1, 0) - jt0;
                    n_hi = ia - jt0; u_hi = ia + 31 - jt0;
                } else {
                    const int e0 = (t - w.n_win) * BN;
                    c_lo = u_lo = n_lo = 0;
                    c_hi = nvis - e0 - 1; n_hi = nvis_first - e0 - 1; u_hi = nvis_last - e0 - 1;
                }
                const bool timed = STREAM && t >= w.n_win;
                int* slv = reinterpret_cast<int*>(smem_raw + OFF_LV) + warp * BN;
                if (timed) {                                   // the leave times of the tile go through a per-warp scratch
                    const int e0 = (t - w.n_win) * BN;
                    const int32_t* lvp = leave + (size_t)w.bhk * R;
                    __syncwarp();                              // the previous tile's readers are done
#pragma unroll
                    for (int u = 0; u < CHUNKS; ++u) slv[u * 32 + lane] = e0 + u * 32 + lane < R ? lvp[e0 + u * 32 + lane] : 0;
                    __syncwarp();
                }
                const uint32_t s_col = trow + S_COL + (g & 1) * BN;
                // The reference is the maximum of the first tile that the row sees and moves to a later tile's that is more than 2^4 above it (in
                // an item's first tiles 2): the nearer it is to the largest logit, the smaller P's rounding beside the large weights, whose
                // largest has none at the reference.  Then what has been added up is rescaled.
                auto follow = [&](float m_here) {
                    const bool up = m_here > m_run + (t < 2 ? 1.f : 4.f);
                    if (!__any_sync(0xffffffffu, up)) return;
                    const float alpha = up && m_run != -INFINITY ? fast_exp2(m_run - m_here) : 1.f;   // (1: nothing has been added up for this row)
                    if (up) m_run = m_here;
                    if (__any_sync(0xffffffffu, alpha != 1.f)) {
                        if (t > 0) {                           // PV of the previous tile must be done before O is rescaled
                            mbar_wait(bar_pv + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1, 10);
                            tc_fence_after();
#pragma unroll 1
                            for (int c4 = 0; c4 < 4; ++c4) {
                                uint32_t q4[16];
                                tmem_ld16(o_col + c4 * 16, q4);
                                tmem_wait_ld();
#pragma unroll
                                for (int c = 0; c < 16; ++c) q4[c] = __float_as_uint(__uint_as_float(q4[c]) * alpha);
                                tmem_st16(o_col + c4 * 16, q4);
                            }
                        }
                        tmem_wait_st();
                        ls[0] = mul2(ls[0], pack2(alpha, alpha)); ls[1] = mul2(ls[1], pack2(alpha, alpha)); lr[0] *= alpha; lr[1] *= alpha;
                    }
                };
                auto weigh = [&](const uint32_t (&x)[32], uint32_t (&pk)[16], uint64_t neg_m2) {   // P of 32 columns, two per word
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        // masked entries hold -inf: fma gives -inf and exp2(-inf) = 0
                        float x0, x1;                          // two columns per packed fp32 instruction
                        unpack2(fma2(pack2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), c2_2, neg_m2), x0, x1);
                        const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        ls[(c >> 1) & 1] = add2(ls[(c >> 1) & 1], pack2(p0, p1));
                        const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
                        pk[c >> 1] = *reinterpret_cast<const uint32_t*>(&h);
                        add_bf16x2(lr[0], lr[1], pk[c >> 1]);
                    }
                };
                mbar_wait(bar_s + 8 * (g & 1), (g >> 1) & 1, 5);
                tc_fence_after();
                if (!timed && n_lo <= 0 && n_hi >= BN - 1) {   // every row of the warp sees all of the tile
                    uint32_t x0[32], x1[32], x2[32], pk[16];
                    tmem_ld32(s_col, x0);
                    tmem_ld32(s_col + 32, x1);
                    tmem_ld32(s_col + 64, x2);
                    tmem_wait_ld();
                    float mr[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) mr[c] = max3(__uint_as_float(x0[c]), __uint_as_float(x1[c]), __uint_as_float(x2[c]));
#pragma unroll
                    for (int c = 8; c < 32; c += 2) {
                        mr[(c >> 1) & 7] = max3(mr[(c >> 1) & 7], __uint_as_float(x0[c]), __uint_as_float(x0[c + 1]));
                        mr[((c >> 1) + 3) & 7] = max3(mr[((c >> 1) + 3) & 7], __uint_as_float(x1[c]), __uint_as_float(x1[c + 1]));
                        mr[((c >> 1) + 6) & 7] = max3(mr[((c >> 1) + 6) & 7], __uint_as_float(x2[c]), __uint_as_float(x2[c + 1]));
                    }
                    follow(max3(max3(mr[0], mr[1], mr[2]), max3(mr[3], mr[4], mr[5]), fmaxf(mr[6], mr[7])) * c2);
                    const float neg_m = m_run == -INFINITY ? 0.f : -m_run;
                    const uint64_t neg_m2 = pack2(neg_m, neg_m);
                    weigh(x0, pk, neg_m2);
                    tmem_st16(s_col + P_AT, pk);               // (over columns of S that have been taken)
                    weigh(x1, pk, neg_m2);
                    tmem_st16(s_col + P_AT + 16, pk);
                    weigh(x2, pk, neg_m2);
                    tmem_st16(s_col + P_AT + 32, pk);
                } else {
                    // The chunks that any row sees: up to the last one for the maximum, then down again for the weights, the last one's logits
                    // being there still and the others fetched again (P has the columns from P_AT on, so that on the way down it
                    // lies over chunks that have been taken).
                    uint32_t pk[16];
                    const int first = max(u_lo, 0) & ~31, last = min(u_hi, BN - 1) & ~31;
                    float mr[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                    uint64_t neg_m2 = 0ull;
                    int at = first;
                    bool down = false;
#pragma unroll 1
                    while (u_hi >= 0 && u_lo < BN) {
                        uint32_t x[32];
                        tmem_ld32(s_col + at, x);
                        tmem_wait_ld();
                        if (timed || at < n_lo || at + 31 > n_hi) {   // some row does not see all of it
                            const int a = min(max(c_lo - at, 0), 32), b = min(max(c_hi - at + 1, 0), 32);
                            const uint32_t below_b = b >= 32 ? 0xffffffffu : ((1u << b) - 1u), below_a = a >= 32 ? 0xffffffffu : ((1u << a) - 1u);
                            uint32_t vm = b > a ? (below_b & ~below_a) : 0u;
                            if (timed) {
                                uint32_t m = 0;
#pragma unroll
                                for (int c = 0; c < 32; c += 4) {
                                    const int4 l4 = *reinterpret_cast<const int4*>(slv + at + c);
                                    m |= (l4.x > i ? 1u : 0u) << c; m |= (l4.y > i ? 2u : 0u) << c;
                                    m |= (l4.z > i ? 4u : 0u) << c; m |= (l4.w > i ? 8u : 0u) << c;
                                }
                                vm &= m;
                            }
#pragma unroll
                            for (int c = 0; c < 32; ++c) x[c] = (vm & (1u << c)) ? x[c] : 0xff800000u;   // -inf
                        }
                        if (!down) {
#pragma unroll
                            for (int c = 0; c < 32; c += 2) mr[(c >> 1) & 3] = max3(mr[(c >> 1) & 3], __uint_as_float(x[c]), __uint_as_float(x[c + 1]));
                            if (at < last) { at += 32; continue; }
                            follow(fmaxf(fmaxf(mr[0], mr[1]), fmaxf(mr[2], mr[3])) * c2);
                            const float neg_m = m_run == -INFINITY ? 0.f : -m_run;
                            neg_m2 = pack2(neg_m, neg_m);
                            down = true;
                        }
                        weigh(x, pk, neg_m2);
                        tmem_st16(s_col + P_AT + at / 2, pk);  // (over columns of S that have been taken)
                        if (at == first) break;
                        at -= 32;
                    }
#pragma unroll
                    for (int c = 0; c < 16; ++c) pk[c] = 0u;
#pragma unroll
                    for (int cb = 0; cb < CHUNKS; ++cb)
                        if (cb * 32 > u_hi || cb * 32 + 31 < u_lo) tmem_st16(s_col + P_AT + cb * 16, pk);
                }
                if (t == 0 && n > 0) {                         // the previous item's output
                    mbar_wait(bar_pv + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1, 11);
                    tc_fence_after();
                    epilogue();
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p + 8 * (g & 1));
            }
            float l0, l1;
            unpack2(add2(ls[0], ls[1]), l0, l1);
            last_l = l0 + l1;
            last_r = lr[0] + lr[1];
            last_m = m_run;
            last_row = i < Tlen ? w.bh * (Tlen - args.qoff) + (i - args.qoff) : -1;
        }
        mbar_wait(bar_pv + 8 * ((g - 1) & 1), ((g - 1) >> 1) & 1, 14);
        tc_fence_after();
        epilogue();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == W_MMA) tmem_dealloc(tmem, TMEM_COLS);
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
            cudaError_t a = cudaFuncSetAttribute(prefill_tc_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(false));
            if (a == cudaSuccess) a = cudaFuncSetAttribute(prefill_tc_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(false));
            return a != cudaSuccess ? a : cudaFuncSetAttribute(prefill_tc_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(true));
        })) return e;
    Args a;
    a.n_qt = (Tq + BM - 1) / BM; a.n_bh = BH; a.n_items = a.n_qt * BH; a.Tlen = p.T; a.W = p.W; a.G = p.G; a.qoff = p.qoff;
    auto go = [&](auto kern, int smem) {
        return cuda_status(launch_pdl(kern, dim3(a.n_items), dim3(NTHREADS), smem, st, tq, tk, tv, tkc, tvc, a, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v,
                                      idx, cnt, (__nv_bfloat16*)o, lse, leave, p.R, p.scale, p.d));
    };
    if (leave) return go(prefill_tc_kernel<false, true>, smem_bytes(true));
    return compact ? go(prefill_tc_kernel<false, false>, smem_bytes(false)) : go(prefill_tc_kernel<true, false>, smem_bytes(false));
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
