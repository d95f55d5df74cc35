// Backward of the LTE prefill attention on the tcgen05 tensor cores (Section 3.1.2), bf16, d = 128, 64 and 32.
//
// Two passes of one kernel, both in gather form (no floating-point atomics, deterministic).  A pass keeps 128 rows (operands
// A1, A2) and walks tiles of BN rows (operands B1, B2):
//            rows        A1, A2     tiles          B1, B2     X = A1 B1^T   Y = A2 B2^T    accumulated
//   dq       queries     Q,  dO     keys           K, V       S             dP             dQ += dS K
//   dkv      keys        K,  V      queries        Q, dO      S^T           dP^T           dK += dS^T Q,  dV += P^T dO
// with P = exp2(S c2 - L2_i) (the forward's logsumexp fixes the normalisation) and dS = P (dP - delta_i) scale,
// delta_i = <dO_i, O_i>.  dq rows see the window keys and then the retained list (rows gathered); dkv rows are the 128 keys of a
// window tile, or 128 entries of the retained list (gathered once), whose tiles are the query blocks that can see them, of
// every query head of the group.  dkv also takes Eq. 6's inner product <v_j, dV_j> = sum_i P_ij dP_ij on the way; window tiles write
// dK, dV of their keys, list tiles write their share to scratch, which the last pass adds row by row (a fixed order).
//
// Bound by the exponentials and the operand reads of the products about equally (a 128 x 128 tile: 1,024 cycles of the exponential
// unit; at d = 64 dkv 24 products of 50-60 cycles), so both have to run all the time:
//   - One CTA per SM with 16 row warps (four threads per row, BN/4 columns each): what two CTAs of four warps had in flight, but
//     with wide tiles, and all of tensor memory for one set of buffers: X, Y, P, dS, accumulators side by side.
//   - X, Y of tile g+1 are computed while the row warps work on tile g (X, Y are free as soon as they are in registers) and the
//     accumulation of tile g runs under tile g+1; the two kinds of product are issued by two warps (one warp issues a product
//     every 54 cycles at best).  P and dS are TMEM A operands: no trip through shared memory.
//   - At d = 64 the halves of a tile's columns go their own way (X, Y of a half are issued when its eight row warps have the last
//     tile's in registers, its share of the accumulation when its P, dS are there), so the products of one run under the
//     exponentials of the other: dq + dkv and tail at the second shape below 570 -> 561, 64 x 3,000 with W = 300, R = 200 196 -> 192, the first
//     190 -> 186.  At d = 128 a half would be 32 or 64 columns of products that read 256 of A.
//   - Items are handed out dynamically, the longest (list tiles) first; a finished item's accumulators are read and stored
//     under the next item's first tile.
//   - dq at d = 128 has room for two 64 KB tiles, and dQ's product holds K: three stages of K and one of V (free once Y is computed, before
//     the tile's exponentials) instead of two of both, 16 heads x 8,192 255 -> 246 for the call (at d = 64, with three stages of both, the
//     barriers more cost 2 %).
// One warp loads (TMA; cp.async for gathered rows).  dq forms delta at an item's start, each thread from its part of the row, and writes
// it for the dkv pass, where another warp prepares the constants -L2, -delta scale of every tile.  Every wait is bounded.
// Slower: two threads per row in place of four with the halves (64 columns each in two chunks: dkv 2 % at the second shape, 1 % faster at the
// first), taking turns at the exponential unit, two of a scheduler's four row warps at a time (2 to 7 %), a barrier per half for the end
// of the accumulation in place of one (1 %).
// Measured (B200, us for dq + dkv; four warps a CTA, two CTAs an SM, items dealt out beforehand; then one CTA of 16 row warps, both in a CUDA graph;
// then with the halves and the stages of K, launches under ncu; exponential unit and tensor pipe active there):
//   128 heads x 2,048, d = 64, W = R = 64                        74 + 96     60 + 78     62 + 77     dq 17 %, 31 %;  dkv 14 %, 33 %
//   128 heads of 4-head groups x 4,096, d = 64, W 768, R 512   364 + 455   243 + 298   259 + 271     dq 42 %, 36 %;  dkv 41 %, 48 %
//   16 heads x 8,192, d = 128, W = R = 512                     185 + 195   101 + 107    88 + 117     dq 32 %, 56 %;  dkv 25 %, 58 %
#include "tile_items.cuh"

namespace lte {

__device__ StatusWord g_bwd_status = LTE_STATUS_INIT;

namespace {

using namespace tc;
__device__ __forceinline__ void bwait(uint32_t bar, uint32_t parity, int code) { mbar_wait_s(bar, parity, code, &g_bwd_status); }

__device__ __forceinline__ void bwait_u(uint32_t bar, uint32_t parity, int code) { mbar_wait_uni(bar, parity, code, &g_bwd_status); }

constexpr int BM = 128, NRW = 16;                              // rows per item, row warps
constexpr int W_LOAD = NRW, W_XY = NRW + 1, W_ACC = NRW + 2, NTHREADS = (NRW + 4) * 32;   // the last warp prepares constants
constexpr float kLog2e = 1.4426950408889634f;

// Stages are what shared memory holds (192 KB of tiles, and O beside them).
template <int D, bool DKV> struct Cfg {
    static constexpr int BN = D == 128 && DKV ? 64 : 128;      // d = 128 dkv: two accumulators of 128 columns leave room for 64-wide tiles
    static constexpr int PARTS = D == 128 ? 1 : 2;             // halves of a tile's columns that go their own way
    static constexpr int AST = D == 128 ? 1 : 3, ATILE = BM * D * 2;
    static constexpr bool SPLIT = D == 128 && !DKV;            // K (needed twice) and V (needed once) in stages of their own
    static constexpr int BST = D == 128 && DKV ? 4 : 3, VST = 1, BTILE = BN * D * 2;   // stages of B1 and B2; SPLIT: of B1, of B2
    static constexpr int OFF_A = 0, OFF_B = AST * 2 * ATILE, OFF_O = OFF_B + (SPLIT ? BST + VST : 2 * BST) * BTILE;   // dq: the item's O, for delta
    static constexpr int OFF_BAR = OFF_O + (DKV ? 0 : ATILE);
    static constexpr int OFF_INFO = OFF_BAR + 512;             // ring of eight items' Info, 64 bytes apart
    static constexpr int OFF_C = OFF_INFO + 512;               // dkv: constants [2][2][128];  dq: lse [2][128]
    static constexpr int OFF_DR = OFF_C + 2 * (DKV ? 2 : 1) * 128 * 4;   // dkv: the four parts of a row's <v, dV> [2][4][128]
    static constexpr int BYTES = OFF_DR + (DKV ? 2 * 4 * 128 * 4 : 0);
    // tensor memory
    static constexpr uint32_t X = 0, Y = BN, DS = 2 * BN, P = DS + BN / 2, ACC0 = DKV ? P + BN / 2 : P, ACC1 = ACC0 + D;
    static_assert(BYTES <= 232448, "shared memory");
    static_assert((DKV ? ACC1 + D : ACC1) <= 512, "tensor memory");
};

struct Args {
    const __nv_bfloat16 *k, *v;
    const float* lse;
    float* delta;
    const int32_t *idx, *cnt;
    __nv_bfloat16 *dq, *dk, *dv;
    float *dr_win, *dk_ret, *dv_ret, *dr_ret;
    int n_rows, n_bh;                                          // dq: query tiles, query heads;  dkv: window tiles, key/value heads
    int n_list;                                                // dkv: list tiles per head
    int Tlen, W, R, G, dg;
    float scale;
};
// dq: row x (0 .. 127) sees before[x / 32] list entries and those of bits[x / 32] below bit x % 32.  dkv: a, b = first query, blocks
// per query head.  item = -1: there is none.
struct Info { uint32_t before[4], bits[4]; int n_tiles, item, a, b; };

struct Item {
    int item, bh, bhk, row0, n_win, j_start, n_tiles;          // dq: query head, its key/value head, first query, window tiles and their first key
    int list, a, b;                                            // dkv: bh = key/value head, row0 = first key or list entry, list tile or not
};
template <bool DKV, int BN> __device__ __forceinline__ Item item_of(const Args& g, int item)
{
    Item it;
    it.item = item;
    it.list = 0; it.a = it.b = 0; it.n_win = it.j_start = 0;
    if (!DKV) {                                                // from the last query tile of every head down to the first
        const int r = item / g.n_bh;
        it.bh = item - r * g.n_bh;
        it.bhk = it.bh / g.G;
        it.row0 = (g.n_rows - 1 - r) * BM;
        const int i_hi = min(it.row0 + BM - 1, g.Tlen - 1);
        it.j_start = max(it.row0 - g.W + 1, 0);
        it.n_win = (i_hi - it.j_start + BN) / BN;
        it.n_tiles = it.n_win;                                 // until the item's Info is there
    } else {                                                   // the list tiles first: they walk many more query blocks
        it.list = item < g.n_list * g.n_bh;
        const int x = it.list ? item : item - g.n_list * g.n_bh;
        const int tile = x / g.n_bh;
        it.bh = it.bhk = x - tile * g.n_bh;
        it.row0 = tile * BM;
        it.a = it.row0;
        it.b = (min(g.Tlen - 1, it.row0 + BM - 1 + g.W - 1) - it.row0) / BN + 1;
        it.n_tiles = it.b * g.G;                               // (window tile)
    }
    return it;
}
template <int N> struct Tmem;                                  // N consecutive columns of the warp's lanes
template <> struct Tmem<32> { static __device__ __forceinline__ void ld(uint32_t a, uint32_t (&r)[32]) { tmem_ld32(a, r); } };
template <> struct Tmem<16> {
    static __device__ __forceinline__ void ld(uint32_t a, uint32_t (&r)[16]) { tmem_ld16(a, r); }
    static __device__ __forceinline__ void st(uint32_t a, const uint32_t (&r)[16]) { tmem_st16(a, r); }
};
template <> struct Tmem<8> {
    static __device__ __forceinline__ void st(uint32_t a, const uint32_t (&r)[8]) {
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
    }
};
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ uint32_t bf16x2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Barriers (g = tile number, n = item number within the CTA):
//   bar_a[b], bar_ga[b]  rows of item n are in buffer b = n % AST: by TMA / gathered (dkv list tiles; 32 arrivals by cp.async completion)
//   bar_af[b]  (commit)  the item's last X, Y are complete                                                     phase n / AST
//   bar_o, bar_od (16)   dq: O (TMA) and lse (32 arrivals by cp.async) of item n are in shared memory / have been read   phase n
//   bar_b[s]             tile g (SPLIT: its K) is in stage s = g % BST                                          phase g / BST
//   bar_v[s], bar_vf[s]  SPLIT: V of tile g is in stage s = g % VST / (commit) X, Y of the tile are complete      phase g / VST
//   bar_bf[s]  (commit)  the accumulation of the stage's tile is complete                                       phase g / BST
//   bar_x[h]  (commit) X, Y of part h of tile g are in TMEM      bar_xf[h] (row warps of the part) they are in registers   phase g
//   bar_p[h]  (row warps of the part) its P, dS are in TMEM and the accumulation of tile g-1 has been awaited                  phase g
//   bar_acc   (commit) the accumulation of tile g is complete                                                              phase g
//   bar_es[b] (4)  STAGED: the outputs of item n have left its A buffer                                           phase n / AST
//   bar_of (16) the accumulators of item n have been read out                                                    phase n
//   bar_i[n & 7]         Info of item n is in the ring                                                           phase n >> 3
//   bar_cc[b], bar_cf[b] (16) dkv: the constants of tile g are in buffer b = g & 1 / have been read                phase g >> 1
//   bar_c                the answer to the request for a block
template <int D, bool DKV>
__global__ void __launch_bounds__(NTHREADS, 1)
bwd_tc_kernel(const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB1,
              const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmL1,
              const __grid_constant__ CUtensorMap tmL2, const __grid_constant__ CUtensorMap tmS1, const __grid_constant__ CUtensorMap tmS2, const Args args)
{
    using C = Cfg<D, DKV>;
    constexpr int BN = C::BN, SUB = D / 64, CW = BN / 4, AST = C::AST, BST = C::BST, VST = C::VST, BPITCH = (C::SPLIT ? 1 : 2) * C::BTILE, ATILE = C::ATILE, BTILE = C::BTILE;
    constexpr int PARTS = C::PARTS, PN = BN / PARTS, PW = NRW / PARTS;   // columns and row warps of a part
    constexpr bool STAGED = D == 64;                           // outputs leave through the item's A buffers as tiles
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0) { if (threadIdx.x == 0) atomicExch(&g_bwd_status.code, 9); return; }
    const uint32_t sA = base + C::OFF_A, sB = base + C::OFF_B, bars = base + C::OFF_BAR;
    const uint32_t bar_a = bars, bar_ga = bars + 32, bar_af = bars + 64, bar_b = bars + 96, bar_bf = bars + 128, bar_i = bars + 160;   // 4 slots each, bar_i 8
    const uint32_t bar_x = bars + 224, bar_xf = bars + 376, bar_p = bars + 392, bar_acc = bars + 248, bar_of = bars + 256, bar_c = bars + 264;
    const uint32_t bar_cc = bars + 272, bar_cf = bars + 288, bar_o = bars + 304, bar_od = bars + 312, bar_es = bars + 320, tmem_slot = bars + 352, answer = bars + 416, bar_v = bars + 432, bar_vf = bars + 464;   // bar_es, bar_v, bar_vf 4, bar_x, bar_xf, bar_p 2
    auto slot = [&](int n) { return reinterpret_cast<volatile Info*>(smem_raw + C::OFF_INFO + (n & 7) * 64); };
    float* const consts = reinterpret_cast<float*>(smem_raw + C::OFF_C);
    volatile uint32_t* tmem_slot_gen = reinterpret_cast<volatile uint32_t*>(smem_raw + C::OFF_BAR + 352);
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (so the compiler knows warp is uniform)

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < 2; ++s) { mbar_init(bar_cc + 8 * s, 1); mbar_init(bar_cf + 8 * s, NRW); }
#pragma unroll
        for (int s = 0; s < PARTS; ++s) { mbar_init(bar_x + 8 * s, 1); mbar_init(bar_xf + 8 * s, PW); mbar_init(bar_p + 8 * s, PW); }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            mbar_init(bar_a + 8 * s, 1); mbar_init(bar_ga + 8 * s, 32); mbar_init(bar_af + 8 * s, 1);
            mbar_init(bar_b + 8 * s, 1); mbar_init(bar_bf + 8 * s, 1); mbar_init(bar_es + 8 * s, 4);
            mbar_init(bar_v + 8 * s, 1); mbar_init(bar_vf + 8 * s, 1);
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) mbar_init(bar_i + 8 * s, 1);
        mbar_init(bar_acc, 1); mbar_init(bar_of, NRW); mbar_init(bar_c, 1);
        mbar_init(bar_o, 33); mbar_init(bar_od, NRW);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_XY) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_gen;
    pdl_launch_dependents();
    pdl_wait();                                                // everything above ran beside the previous kernel's tail (see launch_pdl)

    // the n-th item out of the ring (whole warp); false: there is none
    auto enter = [&](int n, Item& it) {
        bwait(bar_i + 8 * (n & 7), (n >> 3) & 1, 9);
        const int item = __shfl_sync(0xffffffffu, slot(n)->item, 0);
        if (item < 0) return false;
        it = item_of<DKV, BN>(args, item);
        it.n_tiles = __shfl_sync(0xffffffffu, slot(n)->n_tiles, 0);
        if (DKV) { it.a = __shfl_sync(0xffffffffu, slot(n)->a, 0); it.b = __shfl_sync(0xffffffffu, slot(n)->b, 0); }
        return true;
    };

    if (warp == W_LOAD) {
        // ================================= load warp (lane 0 issues the TMA loads) ==============================
        // gathers the k and v rows at pos (-1: zeros): 8 lanes per row copy their 16-byte pieces
        auto gather = [&](uint32_t dst1, uint32_t dst2, int bhk, const int (&pos)[4], uint32_t bar) {
            const size_t head = (size_t)bhk * args.Tlen * args.dg;
            const int sub = lane & 7;
#pragma unroll
            for (int ps = 0; ps < 32; ++ps) {
                const int row = ps * 4 + (lane >> 3), at = __shfl_sync(0xffffffffu, pos[ps >> 3], row & 31);
#pragma unroll
                for (int sb = 0; sb < SUB; ++sb) {
                    const int c = sb * 8 + sub;
                    const bool real = at >= 0 && c * 8 < args.dg;   // (columns past the head dimension are zero-filled)
                    const size_t off = real ? head + (size_t)at * args.dg + c * 8 : 0;
                    const uint32_t to = sb * 16384 + row * 128 + ((sub ^ (row & 7)) << 4);
                    cp_async16(dst1 + to, args.k + off, real ? 16u : 0u);
                    cp_async16(dst2 + to, args.v + off, real ? 16u : 0u);
                }
            }
            cp_async_arrive(bar);
        };
        uint32_t g = 0;
        ItemQueue queue(answer, bar_c, lane);
        for (int n = 0;; ++n) {
            Item it;
            int pos[4] = {-1, -1, -1, -1};                     // dkv list tiles: the positions of their rows
            for (bool own = n == 0;; own = false) {
                it.item = own ? (int)blockIdx.x : queue.take(17, &g_bwd_status);
                if (it.item < 0) break;
                it = item_of<DKV, BN>(args, it.item);
                if (!it.list) break;
                const int n_ret = args.cnt[it.bhk];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int e = it.row0 + u * 32 + lane, at = e < args.R ? args.idx[(size_t)it.bhk * args.R + e] : -1;
                    pos[u] = e < n_ret ? at : -1;
                }
                if (it.row0 < n_ret) break;
                queue.ask();                                   // nothing is retained in this part of the list
            }
            const bool brief = it.item >= 0 && !DKV && it.n_win <= 2;   // (the answer is wanted soon)
            if (brief) queue.ask();
            volatile Info* o = slot(n);
            auto publish = [&]() {
                if (lane == 0) {
                    o->item = it.item; o->n_tiles = it.n_tiles; o->a = it.a; o->b = it.b;
                    mbar_arrive(bar_i + 8 * (n & 7));
                }
            };
            const uint32_t ab = n % AST, a1 = sA + ab * 2 * ATILE, a2 = a1 + ATILE;
            if (n >= AST) bwait(bar_af + 8 * ab, (n / AST - 1) & 1, 12);
            if (it.item < 0) { publish(); break; }
            if (STAGED && n >= AST) bwait(bar_es + 8 * ab, (n / AST - 1) & 1, 22);   // the item's outputs have left the buffer
            if (!DKV && n >= 1) bwait(bar_od, (n - 1) & 1, 19);   // (O and lse of the item before have been read)
            if (!it.list) {
                if (lane == 0) {
                    mbar_expect_tx(bar_a + 8 * ab, 2 * ATILE);
#pragma unroll
                    for (int sb = 0; sb < SUB; ++sb) {
                        tma_load_3d(a1 + sb * 16384, &tmA1, sb * 64, it.row0, it.bh, bar_a + 8 * ab);
                        tma_load_3d(a2 + sb * 16384, &tmA2, sb * 64, it.row0, it.bh, bar_a + 8 * ab);
                    }
                    if (!DKV) {
                        mbar_expect_tx(bar_o, ATILE);
#pragma unroll
                        for (int sb = 0; sb < SUB; ++sb) tma_load_3d(base + C::OFF_O + sb * 16384, &tmO, sb * 64, it.row0, it.bh, bar_o);
                    }
                }
                if (!DKV) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int r = u * 32 + lane;
                        cp_async4(base + C::OFF_C + (n & 1) * 512 + r * 4, args.lse + (size_t)it.bh * args.Tlen + min(it.row0 + r, args.Tlen - 1));
                    }
                    cp_async_arrive(bar_o);
                }
            } else {
                gather(a1, a2, it.bhk, pos, bar_ga + 8 * ab);
                // queries from the oldest entry's first far query on (at least one block, whose columns the masks then take out)
                const int first = min(__shfl_sync(0xffffffffu, pos[0], 0) + args.W, args.Tlen - 1);
                it.a = first / BN * BN;
                it.b = (args.Tlen - 1 - it.a) / BN + 1;
                it.n_tiles = it.b * args.G;
            }
            if (DKV) publish();
            int blk = 0, h = DKV ? it.bh * args.G : it.bhk;    // dkv: block of the query head, query head
            for (int t = 0; t < it.n_tiles; ++t, ++g) {
                const uint32_t s = g % BST, sv = g % VST, b1 = sB + s * BPITCH, b2 = C::SPLIT ? sB + (BST + sv) * BTILE : b1 + BTILE;
                const uint32_t bar2 = C::SPLIT ? bar_v + 8 * sv : bar_b + 8 * s;
                const bool list = !DKV && t >= it.n_win;
                const int y = DKV ? it.a + blk * BN : list ? (t - it.n_win) * BN : it.j_start + t * BN;
                if (g >= (uint32_t)BST) bwait(bar_bf + 8 * s, (g / BST - 1) & 1u, 6);
                if (lane == 0) {
                    mbar_expect_tx(bar_b + 8 * s, BPITCH);
#pragma unroll
                    for (int sb = 0; sb < SUB; ++sb) tma_load_3d(b1 + sb * BN * 128, list ? &tmL1 : &tmB1, sb * 64, y, h, bar_b + 8 * s);
                }
                if (C::SPLIT && g >= (uint32_t)VST) bwait(bar_vf + 8 * sv, (g / VST - 1) & 1u, 24);
                if (lane == 0) {
                    if (C::SPLIT) mbar_expect_tx(bar2, BTILE);
#pragma unroll
                    for (int sb = 0; sb < SUB; ++sb) tma_load_3d(b2 + sb * BN * 128, list ? &tmL2 : &tmB2, sb * 64, y, h, bar2);
                }
                if (!DKV && t == 0) {                          // tile 0 is a window tile; the list is looked up while it is on its way
                    const int last = min(it.row0 + BM - 1, args.Tlen - 1) - it.row0;
                    const ListView f = view_list(args.idx + (size_t)it.bhk * args.R, args.cnt + it.bhk, args.R, it.row0 - args.W, last, lane);
                    it.n_tiles = it.n_win + (f.all + BN - 1) / BN;
                    if (lane == 0) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) { o->before[k] = f.before[k]; o->bits[k] = f.bits[k]; }
                    }
                    publish();
                }
                if (!brief && t == max(it.n_tiles - kAskTiles, 0)) queue.ask();
                if (DKV && ++blk == it.b) { blk = 0; ++h; }
            }
        }
        __syncwarp();
    } else if (warp == W_XY) {
        // ================================= X, Y products (an elected thread issues; the whole warp walks the loop) =
        constexpr uint32_t IDESC = instr_desc(BM, PN, false);
        const uint32_t a_lo = desc_lo(sA, 16), b_lo = desc_lo(sB, 16);
        uint32_t g = 0, par_a = 0;                             // parities of bar_a (bits 0 .. 3), bar_ga (4 .. 7)
        Item it;
        for (int n = 0; uni(enter(n, it)); ++n) {
            const uint32_t ab = n % AST, at = (it.list ? 4 : 0) + ab;
            bwait_u((it.list ? bar_ga : bar_a) + 8 * ab, (par_a >> at) & 1u, 1);
            par_a ^= 1u << at;
            if (uni(it.list)) fence_proxy_async();                  // (gathered rows are generic-proxy writes)
            for (int t = 0; uni(t < it.n_tiles); ++t, ++g) {
                const uint32_t s = g % BST;
                bwait_u(bar_b + 8 * s, (g / BST) & 1u, 2);
#pragma unroll
                for (int h = 0; h < PARTS; ++h) {
                    if (uni(g > 0)) bwait_u(bar_xf + 8 * h, (g - 1) & 1, 3);   // the previous tile's X, Y are in registers
                    tc_fence_after();
                    const uint32_t a1 = a_lo + ab * (2 * ATILE >> 4), hb = h * (PN * 8), sv = g % VST;
                    const uint32_t b1 = b_lo + s * (BPITCH >> 4), b2 = C::SPLIT ? b_lo + (BST + sv) * (BTILE >> 4) : b1 + (BTILE >> 4);
                    auto product = [&](uint32_t d, uint32_t a, uint32_t b) {
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)
                            umma(d + h * PN, desc64(a + (kk >> 2) * 1024 + (kk & 3) * 2, kDescHi), desc64(b + hb + (kk >> 2) * (BN * 8) + (kk & 3) * 2, kDescHi), IDESC, kk > 0);
                    };
                    if (C::SPLIT) {
                        if (elect_one()) product(tmem + C::X, a1, b1);
                        __syncwarp();
                        if (h == 0) { bwait_u(bar_v + 8 * sv, (g / VST) & 1u, 25); tc_fence_after(); }
                    }
                    if (elect_one()) {
                        if (!C::SPLIT) product(tmem + C::X, a1, b1);
                        product(tmem + C::Y, a1 + (ATILE >> 4), b2);
                        umma_commit(bar_x + 8 * h);
                        if (C::SPLIT && h == PARTS - 1) umma_commit(bar_vf + 8 * sv);
                        if (h == PARTS - 1 && t == it.n_tiles - 1) umma_commit(bar_af + 8 * ab);
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp == W_ACC) {
        // ================================= accumulation ==========================================================
        constexpr uint32_t IDESC = instr_desc(BM, D, true);
        const uint32_t b_lo = desc_lo(sB, BN * 128);
        uint32_t g = 0;
        Item it;
        for (int n = 0; uni(enter(n, it)); ++n) {
            for (int t = 0; uni(t < it.n_tiles); ++t, ++g) {
                const uint32_t s = g % BST;
                if (uni(t == 0 && n > 0)) bwait_u(bar_of, (n - 1) & 1, 13);   // the previous item's accumulators have been read out
#pragma unroll
                for (int h = 0; h < PARTS; ++h) {
                    constexpr int KP = PN / 16;
                    bwait_u(bar_p + 8 * h, g & 1, 7);
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t b1 = b_lo + s * (BPITCH >> 4);
                        if (DKV) {
#pragma unroll
                            for (int kk = h * KP; kk < h * KP + KP; ++kk)
                                umma_ts(tmem + C::ACC1, tmem + C::P + kk * 8, desc64(b1 + (BTILE >> 4) + kk * 128, kDescHi), IDESC, (t > 0 || kk > 0) ? 1u : 0u);
                        }
#pragma unroll
                        for (int kk = h * KP; kk < h * KP + KP; ++kk)
                            umma_ts(tmem + C::ACC0, tmem + C::DS + kk * 8, desc64(b1 + kk * 128, kDescHi), IDESC, (t > 0 || kk > 0) ? 1u : 0u);
                        if (h == PARTS - 1) {
                            umma_commit(bar_acc);
                            umma_commit(bar_bf + 8 * s);
                        }
                    }
                    __syncwarp();
                }
            }
        }
    } else if (warp >= NRW) {
        // ================================= constants (dkv) =======================================================
        // per tile: -L2 and -delta scale of its BN queries (queries past the end are masked by the rows)
        Item it;
        uint32_t g = 0;
        for (int n = 0; DKV && enter(n, it); ++n) {
            int i0 = it.a;
            size_t head = (size_t)it.bh * args.G * args.Tlen;
            for (int t = 0, blk = 0; t < it.n_tiles; ++t, ++g) {
                float l[BN / 32], dl[BN / 32];
#pragma unroll
                for (int u = 0; u < BN / 32; ++u) {
                    const int i = min(i0 + u * 32 + lane, args.Tlen - 1);
                    l[u] = args.lse[head + i]; dl[u] = args.delta[head + i];
                }
                if (g >= 2) bwait(bar_cf + 8 * (g & 1), ((g >> 1) - 1) & 1, 14);
                float* c = consts + (g & 1) * 256;
#pragma unroll
                for (int u = 0; u < BN / 32; ++u) { c[u * 32 + lane] = -l[u] * kLog2e; c[128 + u * 32 + lane] = -dl[u] * args.scale; }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_cc + 8 * (g & 1));
                i0 += BN;
                if (++blk == it.b) { blk = 0; i0 = it.a; head += args.Tlen; }
            }
        }
    } else {
        // ================================= row warps ==============================================================
        // Four threads per row: thread `row` of warps 4 q .. 4 q + 3 takes columns [q CW, q CW + CW) of every tile.
        const int quarter = warp & 3, q = warp >> 2, row = quarter * 32 + lane, c0 = q * CW, part8 = q / (4 / PARTS) * 8;
        const float c2 = args.scale * kLog2e;
        const uint64_t c2_2 = pack2(c2, c2), scale_2 = pack2(args.scale, args.scale);
        const uint32_t trow = tmem + (((uint32_t)(quarter * 32)) << 16);   // this warp's TMEM lanes
        const int Tlen = args.Tlen, W = args.W, dg = args.dg;
        uint32_t g = 0;
        // The accumulators of a finished item: D/4 columns per thread, read and stored under the next item's first tile.
        uint64_t l_dr = 0ull, dr2 = 0ull;                      // dkv: Eq. 6's <v_j, dV_j> = sum_i P_ij dP_ij over this thread's columns
        int l_list = 0, l_bh = 0, l_row = -1, l_pos = -1;      // its kind, head, list entry or row, position (-1: none)
        auto epilogue = [&](int n) {
            constexpr int EC = D / 4;
            const int e0 = q * EC;
            const bool live = l_pos >= 0 && e0 < dg, tiles = STAGED && !l_list;
            const size_t out = ((size_t)l_bh * (l_list ? args.R : Tlen) + l_row) * dg + e0;
            const uint32_t stage = sA + (n % AST) * 2 * ATILE;
#pragma unroll
            for (int a = DKV ? 1 : 0; a >= 0; --a) {           // dkv: dV (1), then dK (0);  dq: dQ
                uint32_t x[EC];
                Tmem<EC>::ld(trow + (a ? C::ACC1 : C::ACC0) + e0, x);
                tmem_wait_ld();
                if (a == 0) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_of);
                }
                if (DKV && l_list) {
                    float* dst = (a ? args.dv_ret : args.dk_ret) + out;
                    if (live)
#pragma unroll
                        for (int c = 0; c < EC; c += 4)
                            *reinterpret_cast<float4*>(dst + c) = make_float4(__uint_as_float(x[c]), __uint_as_float(x[c + 1]), __uint_as_float(x[c + 2]), __uint_as_float(x[c + 3]));
                } else if constexpr (!STAGED) {
                    // four lanes transpose their four 16-byte pieces, so that a store covers 64 bytes of 8 rows instead of 16 of 32
                    uint32_t w[4][4];
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int e = 0; e < 4; ++e) w[c][e] = bf16x2(__uint_as_float(x[c * 8 + 2 * e]), __uint_as_float(x[c * 8 + 2 * e + 1]));
#pragma unroll
                    for (int m = 1; m <= 2; m <<= 1)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            if (c & m) continue;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {      // my piece for the partner: c ^ m if I am the lower lane, else c
                                const bool up = (lane & m) != 0;
                                const uint32_t r = __shfl_xor_sync(0xffffffffu, up ? w[c][e] : w[c ^ m][e], m);
                                if (up) w[c][e] = r; else w[c ^ m][e] = r;
                            }
                        }
                    __nv_bfloat16* dst = (DKV ? (a ? args.dv : args.dk) : args.dq);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {              // now piece lane & 3 of row (lane & ~3) + c
                        const int r = l_row - lane + (lane & ~3) + c;
                        if (r < Tlen) *reinterpret_cast<uint4*>(dst + ((size_t)l_bh * Tlen + r) * D + e0 + (lane & 3) * 8) = make_uint4(w[c][0], w[c][1], w[c][2], w[c][3]);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < EC; c += 8) {
                        uint32_t w4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) w4[e] = bf16x2(__uint_as_float(x[c + 2 * e]), __uint_as_float(x[c + 2 * e + 1]));
                        const uint32_t to = stage + a * ATILE + row * 128 + ((((e0 + c) >> 3) ^ (row & 7)) << 4);   // (leave as tiles)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(w4[0]), "r"(w4[1]), "r"(w4[2]), "r"(w4[3]) : "memory");
                    }
                }
            }
            float* s = reinterpret_cast<float*>(smem_raw + C::OFF_DR) + (n & 1) * 512;
            if (DKV) {                                         // the row's four parts meet (rewritten two items, so two barriers, on)
                float d0, d1;
                unpack2(l_dr, d0, d1);
                s[q * 128 + row] = d0 + d1;
            }
            if (tiles) fence_proxy_async();
            if (DKV || STAGED) asm volatile("bar.sync %0, 128;" ::"r"(1 + quarter) : "memory");
            if (q != 0) return;
            if (STAGED && lane == 0) {
                const int r0 = l_row;                          // (lane 0: the first of the quarter's 32 rows)
                if (tiles && r0 < Tlen) {
                    tma_store_3d(&tmS1, stage + quarter * 4096, 0, r0, l_bh);
                    if (DKV) tma_store_3d(&tmS2, stage + ATILE + quarter * 4096, 0, r0, l_bh);
                    bulk_commit();
                    bulk_wait_read0();
                }
                mbar_arrive(bar_es + 8 * (n % AST));
            }
            if (DKV && l_pos >= 0) {
                const float sum = (s[row] + s[128 + row]) + (s[256 + row] + s[384 + row]);
                if (l_list) args.dr_ret[(size_t)l_bh * args.R + l_row] = sum;
                else args.dr_win[(size_t)l_bh * Tlen + l_row] = sum;
            }
        };
        Item it;
        int n = 0;
        for (; enter(n, it); ++n) {
            const int r_abs = it.row0 + row;                   // query, key, or list entry
            int pos = r_abs, nvis = 0, key_lo = 0, key_hi = 0;
            uint64_t nl2 = 0ull, ndls = 0ull;
            if (DKV) {
                if (it.list) pos = r_abs < args.cnt[it.bh] ? args.idx[(size_t)it.bh * args.R + r_abs] : -1;
                else if (r_abs >= Tlen) pos = -1;
                key_lo = it.list ? pos + W : pos;              // queries that see the key
                key_hi = pos < 0 ? -1 - BN * it.b - it.a : min(it.list ? Tlen - 1 : pos + W - 1, Tlen - 1);
            } else {
                const volatile Info* f = slot(n);
                const int x = min(r_abs, Tlen - 1) - it.row0;
                nvis = (int)(f->before[x >> 5] + __popc(f->bits[x >> 5] & ((1u << (x & 31)) - 1u)));
                // delta = <dO, O>: this thread's quarter of the channels, then the four parts (chunk c of row r is at c ^ (r & 7))
                bwait(bar_a + 8 * (n % AST), (n / AST) & 1, 20);
                bwait(bar_o, n & 1, 21);
                const uint32_t so = base + C::OFF_O, sdo = sA + (n % AST) * 2 * ATILE + ATILE;
                float d0 = 0.f, d1 = 0.f;
#pragma unroll
                for (int u = 0; u < D / 32; ++u) {
                    const int ch = q * (D / 32) + u;
                    const uint32_t off = (ch >> 3) * 16384 + row * 128 + (((ch & 7) ^ (row & 7)) << 4);
                    uint32_t aw[4], bw[4];
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(aw[0]), "=r"(aw[1]), "=r"(aw[2]), "=r"(aw[3]) : "r"(so + off));
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(bw[0]), "=r"(bw[1]), "=r"(bw[2]), "=r"(bw[3]) : "r"(sdo + off));
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        d0 = fmaf(__uint_as_float(aw[e] << 16), __uint_as_float(bw[e] << 16), d0);
                        d1 = fmaf(__uint_as_float(aw[e] & 0xffff0000u), __uint_as_float(bw[e] & 0xffff0000u), d1);
                    }
                }
                auto part = [&](int k) {                       // part k replaces the first of the chunks that it was formed from
                    const int ch = k * (D / 32);
                    return reinterpret_cast<float*>(smem_raw + C::OFF_O + (ch >> 3) * 16384 + row * 128 + (((ch & 7) ^ (row & 7)) << 4));
                };
                *part(q) = d0 + d1;
                const float nl = -consts[(n & 1) * 128 + row] * kLog2e;
                asm volatile("bar.sync %0, 128;" ::"r"(5 + quarter) : "memory");
                const float d = (*part(0) + *part(1)) + (*part(2) + *part(3));
                fence_proxy_async();                           // (TMA writes the next item's O there)
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_od);
                if (q == 0 && r_abs < Tlen) args.delta[(size_t)it.bh * Tlen + r_abs] = d;
                nl2 = pack2(nl, nl); ndls = pack2(-d * args.scale, -d * args.scale);
            }
            int i_blk = it.a + c0, blk = 0;                    // dkv: first query of this thread's columns, block of the query head
            for (int t = 0; t < it.n_tiles; ++t, ++g) {
                // columns of this thread's part that the row may see
                int c_lo, c_hi;
                if (!DKV) {
                    if (t < it.n_win) { const int j = it.j_start + t * BN + c0; c_lo = max(r_abs - W + 1, 0) - j; c_hi = r_abs - j; }
                    else { c_lo = 0; c_hi = nvis - (t - it.n_win) * BN - c0 - 1; }
                } else {
                    c_lo = key_lo - i_blk; c_hi = key_hi - i_blk;
                    i_blk += BN;
                    if (++blk == it.b) { blk = 0; i_blk = it.a + c0; }
                }
                const int a = min(max(c_lo, 0), CW), b = min(max(c_hi + 1, 0), CW);
                const uint32_t below_b = b >= 32 ? 0xffffffffu : ((1u << b) - 1u), below_a = a >= 32 ? 0xffffffffu : ((1u << a) - 1u);
                const uint32_t vm = below_b & ~below_a;
                const bool some = __any_sync(0xffffffffu, vm != 0u), plain = __all_sync(0xffffffffu, a == 0 && b == CW);
                uint32_t ds[CW / 2], pp[CW / 2];
                const float* col = consts + (g & 1) * 256 + c0;
                if (DKV) bwait(bar_cc + 8 * (g & 1), (g >> 1) & 1, 16);
                bwait(bar_x + part8, g & 1, 5);
                tc_fence_after();
                if (some) {
                    uint32_t x[CW], y[CW];
                    Tmem<CW>::ld(trow + C::X + c0, x);
                    Tmem<CW>::ld(trow + C::Y + c0, y);
                    tmem_wait_ld();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_xf + part8);   // X, Y of tile g+1 may overwrite the buffers
                    if (!plain) {
#pragma unroll
                        for (int c = 0; c < CW; ++c) x[c] = (vm & (1u << c)) ? x[c] : 0xff800000u;   // -inf: P = 0
                    }
#pragma unroll
                    for (int c = 0; c < CW; c += 4) {          // packed fp32 pairs
                        uint64_t nl_a = nl2, nl_b = nl2, nd_a = ndls, nd_b = ndls;
                        if (DKV) {
                            const float4 l4 = *reinterpret_cast<const float4*>(col + c), d4 = *reinterpret_cast<const float4*>(col + 128 + c);
                            nl_a = pack2(l4.x, l4.y); nl_b = pack2(l4.z, l4.w); nd_a = pack2(d4.x, d4.y); nd_b = pack2(d4.z, d4.w);
                        }
                        float e[4], s[4];
                        unpack2(fma2(pack2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), c2_2, nl_a), e[0], e[1]);
                        unpack2(fma2(pack2(__uint_as_float(x[c + 2]), __uint_as_float(x[c + 3])), c2_2, nl_b), e[2], e[3]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) e[u] = fast_exp2(e[u]);
                        if (DKV) {
                            dr2 = fma2(pack2(e[0], e[1]), pack2(__uint_as_float(y[c]), __uint_as_float(y[c + 1])), dr2);
                            dr2 = fma2(pack2(e[2], e[3]), pack2(__uint_as_float(y[c + 2]), __uint_as_float(y[c + 3])), dr2);
                        }
                        unpack2(mul2(pack2(e[0], e[1]), fma2(pack2(__uint_as_float(y[c]), __uint_as_float(y[c + 1])), scale_2, nd_a)), s[0], s[1]);
                        unpack2(mul2(pack2(e[2], e[3]), fma2(pack2(__uint_as_float(y[c + 2]), __uint_as_float(y[c + 3])), scale_2, nd_b)), s[2], s[3]);
                        ds[c / 2] = bf16x2(s[0], s[1]); ds[c / 2 + 1] = bf16x2(s[2], s[3]);
                        if (DKV) { pp[c / 2] = bf16x2(e[0], e[1]); pp[c / 2 + 1] = bf16x2(e[2], e[3]); }
                    }
                } else {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_xf + part8);
#pragma unroll
                    for (int c = 0; c < CW / 2; ++c) { ds[c] = 0u; pp[c] = 0u; }
                }
                // P(g), dS(g) take the place of tile g-1's, whose accumulation has normally completed; every phase is awaited in turn
                if (g > 0) { bwait(bar_acc, (g - 1) & 1, 11); tc_fence_after(); }
                if (t == 0 && n > 0) epilogue(n - 1);
                Tmem<CW / 2>::st(trow + C::DS + c0 / 2, ds);
                if (DKV) Tmem<CW / 2>::st(trow + C::P + c0 / 2, pp);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { mbar_arrive(bar_p + part8); if (DKV) mbar_arrive(bar_cf + 8 * (g & 1)); }
            }
            l_list = it.list; l_bh = it.bh; l_row = r_abs;
            l_dr = dr2; dr2 = 0ull;
            l_pos = DKV ? pos : r_abs < Tlen ? r_abs : -1;
        }
        if (n > 0) {
            bwait(bar_acc, (g - 1) & 1, 18);
            tc_fence_after();
            epilogue(n - 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == W_XY) tmem_dealloc(tmem, 512);
}

// Far-query share of the retained keys added onto their rows (each key appears once in the list: fixed order).  Four channels per thread,
// 1,024 / D rows per block (4 x 8 heads, 512 rows: 5.8 us; a block of 64 threads per row 15.7).
__global__ void __launch_bounds__(256) bwd_merge_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ cnt,
                                 const float* __restrict__ dk_ret, const float* __restrict__ dv_ret,
                                 const float* __restrict__ dr_ret, __nv_bfloat16* __restrict__ dk,
                                 __nv_bfloat16* __restrict__ dv, float* __restrict__ dr_win, int Tlen, int R, int D)
{
    pdl_launch_dependents();
    pdl_wait();                                                // see launch_pdl: earlier kernels of the stream have completed
    const int tpr = D / 4, bh = blockIdx.y, e = blockIdx.x * (256 / tpr) + threadIdx.x / tpr, c = threadIdx.x % tpr * 4;
    if (e >= cnt[bh]) return;
    const int j = idx[(size_t)bh * R + e];
    const size_t src = ((size_t)bh * R + e) * D + c, dst = ((size_t)bh * Tlen + j) * D + c;
    auto add = [](__nv_bfloat16* x, const float* y) {
        const uint2 u = *reinterpret_cast<const uint2*>(x);
        const float4 f = *reinterpret_cast<const float4*>(y);
        *reinterpret_cast<uint2*>(x) = make_uint2(bf16x2(__uint_as_float(u.x << 16) + f.x, __uint_as_float(u.x & 0xffff0000u) + f.y),
                                                  bf16x2(__uint_as_float(u.y << 16) + f.z, __uint_as_float(u.y & 0xffff0000u) + f.w));
    };
    add(dk + dst, dk_ret + src);
    add(dv + dst, dv_ret + src);
    if (c == 0) dr_win[(size_t)bh * Tlen + j] += dr_ret[(size_t)bh * R + e];
}

// dr -> dz in place: Eq. 6 (+ Eq. 7's lambda term) through the sigmoid, for scored tokens only.
__global__ void bwd_dz_kernel(float* __restrict__ dz, const float* __restrict__ z, const float* __restrict__ lambda, int H,
                              int Tlen, int half, float zthr)
{
    pdl_launch_dependents();
    pdl_wait();                                                // see launch_pdl: earlier kernels of the stream have completed
    const int bh = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= Tlen) return;
    float g = 0.f;
    if (j + half <= Tlen - 1) {
        const float zz = z[(size_t)bh * Tlen + j];
        const float r = 1.f / (1.f + expf(-zz));
        float dr = dz[(size_t)bh * Tlen + j];
        if (lambda && zz > zthr) dr += lambda[bh % H];
        g = dr * r * (1.f - r);
    }
    dz[(size_t)bh * Tlen + j] = g;
}

template <int D, bool DKV> int launch_pass(const CUtensorMap& a1, const CUtensorMap& a2, const CUtensorMap& b1, const CUtensorMap& b2, const CUtensorMap& o,
                                           const CUtensorMap& l1, const CUtensorMap& l2, const CUtensorMap& s1, const CUtensorMap& s2, const Args& a, int items, cudaStream_t st)
{
    using C = Cfg<D, DKV>;
    static PerDeviceOnce attr;
    if (int e = attr.run([] { return cudaFuncSetAttribute(bwd_tc_kernel<D, DKV>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::BYTES); })) return e;
    return cuda_status(launch_pdl(bwd_tc_kernel<D, DKV>, dim3(items), dim3(NTHREADS), C::BYTES, st, a1, a2, b1, b2, o, l1, l2, s1, s2, a));
}

}  // namespace

size_t bwd_tc_ret_bytes(const Params& p)
{
    const size_t n = (size_t)p.B * p.H * (p.R > 0 ? p.R : 1);
    return ((2 * n * p.d + n) * 4 + 255) / 256 * 256;
}

// dq (and delta) on the tensor cores.  Returns LTE_OK or an error; the caller runs the remaining stages.  `ret_ws` (the dkv pass's
// scratch, not in use yet) takes the retained rows of k and v in list order, so that list tiles are TMA boxes.
int launch_bwd_dq_tc(const Params& p, const void* q, const void* k, const void* v, const void* o, const float* lse,
                     const void* dO, const int32_t* idx, const int32_t* cnt, void* dq, float* delta, void* ret_ws, cudaStream_t st)
{
    const int BHK = p.B * p.H, BH = BHK * p.G;                 // key/value heads, query heads
    CUtensorMap tq, tdo, tk, tv, to, tdq, tlk, tlv;
    constexpr int bn = Cfg<64, false>::BN;
    static_assert(bn == Cfg<128, false>::BN, "");
    if (!make_map(&tq, q, BH, p.T, p.d, BM) || !make_map(&tdo, dO, BH, p.T, p.d, BM) || !make_map(&to, o, BH, p.T, p.d, BM) ||
        !make_map(&tdq, dq, BH, p.T, p.d, 32) || !make_map(&tk, k, BHK, p.T, p.d, bn) || !make_map(&tv, v, BHK, p.T, p.d, bn)) return LTE_ERR_CUDA;
    tlk = tk; tlv = tv;
    if (p.R > 0) {
        char* kc = (char*)ret_ws; char* vc = kc + (size_t)BHK * p.R * p.d * 4;   // (each of the two fp32 tensors has room for a bf16 one)
        if (int e = launch_prefill_compact(p, k, v, idx, cnt, kc, vc, st)) return e;
        if (!make_map(&tlk, kc, BHK, p.R, p.d, bn) || !make_map(&tlv, vc, BHK, p.R, p.d, bn)) return LTE_ERR_CUDA;
    }
    Args a = {};
    a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
    a.lse = lse; a.delta = delta; a.idx = idx; a.cnt = cnt; a.dq = (__nv_bfloat16*)dq;
    a.n_rows = (p.T + BM - 1) / BM; a.n_bh = BH;
    a.Tlen = p.T; a.W = p.W; a.R = p.R; a.G = p.G; a.dg = p.d; a.scale = p.scale;
    const int items = a.n_rows * BH;
    if (p.d == 64 || p.d == 32) return launch_pass<64, false>(tq, tdo, tk, tv, to, tlk, tlv, tdq, tdq, a, items, st);
    return p.d == 128 ? launch_pass<128, false>(tq, tdo, tk, tv, to, tlk, tlv, tdq, tdq, a, items, st) : LTE_ERR_UNSUPPORTED;
}

// dk, dv, dz on the tensor cores.  `ret_ws` holds dk_ret, dv_ret [B,H,R,d] and dr_ret [B,H,R] (fp32).
int launch_bwd_dkv_tc(const Params& p, const void* q, const void* k, const void* v, const float* lse, const void* dO,
                      const float* delta, const float* z, const int32_t* idx, const int32_t* cnt, const float* lambda,
                      void* dk, void* dv, float* dz, void* ret_ws, bool merge_here, cudaStream_t st)
{
    const int BH = p.B * p.H, bn = p.d == 128 ? Cfg<128, true>::BN : Cfg<64, true>::BN;
    CUtensorMap tk, tv, tq, tdo, tdk, tdv;
    if (!make_map(&tk, k, BH, p.T, p.d, BM) || !make_map(&tv, v, BH, p.T, p.d, BM) ||
        !make_map(&tq, q, BH * p.G, p.T, p.d, bn) || !make_map(&tdo, dO, BH * p.G, p.T, p.d, bn) ||
        !make_map(&tdk, dk, BH, p.T, p.d, 32) || !make_map(&tdv, dv, BH, p.T, p.d, 32)) return LTE_ERR_CUDA;
    const size_t n = (size_t)BH * (p.R > 0 ? p.R : 1);
    float* dk_ret = (float*)ret_ws;
    float* dv_ret = dk_ret + n * p.d;
    float* dr_ret = dv_ret + n * p.d;
    Args a = {};
    a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
    a.lse = lse; a.delta = const_cast<float*>(delta); a.idx = idx; a.cnt = cnt;
    a.dk = (__nv_bfloat16*)dk; a.dv = (__nv_bfloat16*)dv; a.dr_win = dz; a.dk_ret = dk_ret; a.dv_ret = dv_ret; a.dr_ret = dr_ret;
    a.n_rows = (p.T + BM - 1) / BM; a.n_bh = BH; a.n_list = (p.R + BM - 1) / BM;
    a.Tlen = p.T; a.W = p.W; a.R = p.R; a.G = p.G; a.dg = p.d; a.scale = p.scale;
    const int items = (a.n_rows + a.n_list) * BH;
    int e = LTE_ERR_UNSUPPORTED;
    if (p.d == 64 || p.d == 32) e = launch_pass<64, true>(tk, tv, tq, tdo, tq, tq, tq, tdk, tdv, a, items, st);
    else if (p.d == 128) e = launch_pass<128, true>(tk, tv, tq, tdo, tq, tq, tq, tdk, tdv, a, items, st);
    // merge_here = false: the caller's last pass adds the retained shares and turns dr into dz itself
    if (e || !merge_here) return e;
    if (p.R > 0) {
        if (int e2 = cuda_status(launch_pdl(bwd_merge_kernel, dim3((p.R * p.d + 1023) / 1024, BH), dim3(256), 0, st, idx, cnt, dk_ret, dv_ret, dr_ret,
                                            (__nv_bfloat16*)dk, (__nv_bfloat16*)dv, dz, p.T, p.R, p.d))) return e2;
    }
    return cuda_status(launch_pdl(bwd_dz_kernel, dim3((p.T + 255) / 256, BH), dim3(256), 0, st, dz, z, lambda, p.H, p.T, p.half, p.zthr));
}

int bwd_status_fetch_and_clear() { return status_fetch_and_clear(g_bwd_status); }

}  // namespace lte
