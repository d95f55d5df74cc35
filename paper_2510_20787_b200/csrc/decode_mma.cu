// Decode step for bf16 caches (Fig. 3; Section 3.1.3, decoding paragraph) whose rows go from memory straight into
// tensor-core operands: every query head of a group at once, heads split over a thread-block cluster where there are few.
//
// Bound by memory: the step reads a head's rows once and does almost nothing with them, so what counts is that enough of
// them are in flight from the first moment on, and few instructions per row.  Every warp walks spans of 16 rows (interleaved
// over the warps of all blocks that share the head) with two spans in flight, keeps its own reference, sum and output, and
// meets the others once at the end; the replacement decision runs beside the first loads and only turns into row masks.
//
// The products are mma.sync m16n8k16, not tcgen05: N = 8 query heads and 16 rows at a time need no shared memory at all.
// The contraction index of a product may be permuted freely, so a lane's operand registers are the 16-byte pieces it loaded:
//   logits   S^T[16 rows][8 queries] = K q^T:  lane (g, t) = (lane / 4, lane % 4) holds pieces t, t + 4, .. of rows g and g + 8
//            as A and the same pieces of query g as B (products of bf16 values are exact, the scale is applied in fp32 after: to
//            the distance from the reference, which is held unscaled, so that the largest logit's weight is exact however large
//            it is and the scale's rounding does not grow with the logits);
//   output   O^T[16 channels][8 queries] += V^T P^T:  lane (g, t) holds piece g (and g + 8) of rows 2t, 2t+1, 2t+8, 2t+9; a
//            byte permute pairs two rows' words into A.  P comes out of the logits' registers through movmatrix, split
//            into two bf16 terms: 16 bits of mantissa, below what the output's rounding shows (o against 64 bits over 35,000 random
//            steps: 1.53e-3, the same to four digits as with fp32 weights).
//
// Measured (B200, a step in a CUDA graph of steps, full pools; before: a block per head on the fp32 ALUs):
//   256 heads x 1,280 rows, four query heads each, d = 64    17.7 us (84 MB: 4.8 TB/s), before 29.9; with 1,160 rows 15.4
//   512 heads x 1,280 rows, d = 64                           34.0 us (4.9 TB/s), before 43.1
//   512 heads x 1,024 rows, d = 128                          49.1 us (5.5 TB/s), before 63.6
//   16 heads x 1,024 rows, d = 128                            7.5 us in clusters of 8, before 16.5; six of it are the chain launch,
//                                                            counters, rows, combination, and stay when there are fewer rows
// With row-by-row address arithmetic (600 instead of 130 instructions a span) the first line was a quarter slower; asking for the
// ring's rows in L2 ahead of the grid dependency made the large shapes slower (4 and 13 %).
#include <cooperative_groups.h>

#include "common.cuh"

namespace lte {
namespace cg = cooperative_groups;
namespace {

constexpr int MQ = 8;                                          // query heads per pass
constexpr float M_NONE = -1e30f;                                // a reference before the first row (finite: no inf - inf)
// Resident warps per SM the registers are budgeted for (128 and 255 a thread), and warps per block at most.
__host__ __device__ constexpr int warps_per_sm(int d) { return d == 128 ? 8 : 16; }
__host__ __device__ constexpr int max_warps(int d) { return d == 128 ? 4 : 8; }
constexpr int MAX_SPLIT = 8;                                   // blocks per head

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t word(const uint4& u, int i) { return i == 0 ? u.x : i == 1 ? u.y : i == 2 ? u.z : u.w; }

// Up to 16 consecutive rows of the ring or of the pool, or the incoming token alone (row = -1).
struct Span { int row, n; };
// A head's rows as a list of spans: ring, pool, incoming token.
struct Rows {
    const unsigned char *K, *V, *k1, *v1;
    int n_ring, cnt, W, ring_spans, spans;
    __device__ __forceinline__ Span span(int i) const {
        const bool ring = i < ring_spans;
        const int at = (ring ? i : i - ring_spans) << 4;
        Span s = {ring ? at : W + at, min(16, (ring ? n_ring : cnt) - at)};
        if (i == spans - 1) s = {-1, 1};
        return s;
    }
};

template <int D, bool SWZ> struct Group {                      // what a lane holds of a span's 16 rows
    static constexpr int KP = D / 32, VB = D / 16, PITCH = D * 2;   // 16-byte key pieces and 4-byte value words per row
    uint4 k[2][KP];
    uint32_t v[4][VB];
    // Rows past the end of a span repeat its last row with weight zero, and so do the row that leaves and the entry that is replaced
    // in this step.  (Zero times an infinite value is NaN, but those two have been part of every step up to this one.  Clearing
    // their values cost 2.5 % of a step with grouped queries.)
    __device__ __forceinline__ void load_k(const Rows& R, const Span& s, int g, int t) {
        const unsigned char* base = s.row >= 0 ? R.K + (size_t)s.row * PITCH : R.k1;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = s.n == 16 ? g + 8 * i : min(g + 8 * i, s.n - 1);
            const unsigned char* p = base + r * PITCH;
            const int sw = SWZ && s.row >= 0 ? (s.row + r) & 7 : 0;
#pragma unroll
            for (int j = 0; j < KP; ++j) k[i][j] = *reinterpret_cast<const uint4*>(p + (((t + 4 * j) ^ sw) << 4));
        }
    }
    __device__ __forceinline__ void load_v(const Rows& R, const Span& s, int g, int t) {
        const unsigned char* base = s.row >= 0 ? R.V + (size_t)s.row * PITCH : R.v1;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int ri = 2 * t + (i & 1) + 8 * (i >> 1), r = s.n == 16 ? ri : min(ri, s.n - 1);
            const unsigned char* p = base + r * PITCH;
            const int sw = SWZ && s.row >= 0 ? (s.row + r) & 7 : 0;
            if constexpr (D == 32) {
                const uint2 u = *reinterpret_cast<const uint2*>(p + (g << 3));
                v[i][0] = u.x; v[i][1] = u.y;
            } else {
#pragma unroll
                for (int j = 0; j < D / 64; ++j) {
                    const uint4 u = *reinterpret_cast<const uint4*>(p + (((g + 8 * j) ^ sw) << 4));
#pragma unroll
                    for (int w = 0; w < 4; ++w) v[i][4 * j + w] = word(u, w);
                }
            }
        }
    }
};

// BACK: in every other step the spans come from the last to the first (see decode_turns; a variant of its own, since the sign of the
// stride costs up to 3 % of a step that takes its rows from L2, which is where `turn` is off).
template <int D, int NW, bool SWZ, bool BACK>
__global__ void __launch_bounds__(NW * 32, warps_per_sm(D) / NW) decode_mma_kernel(
    unsigned char* __restrict__ cache, CacheLayout L, const __nv_bfloat16* __restrict__ q1, const __nv_bfloat16* __restrict__ k1,
    const __nv_bfloat16* __restrict__ v1, __nv_bfloat16* __restrict__ o1, float* __restrict__ lse1, const float* __restrict__ cw,
    const float* __restrict__ cbias, int H, int W, int R, int sink, int K, float zthr, float scale, int G)
{
    constexpr int NT = NW * 32, KP = D / 32, MT = D / 16, PITCH = D + 8, PIECES = D / 8, CPL = D / 32;
    constexpr int NBUF = 2;                                    // spans in flight per warp
    __shared__ __align__(16) float s_acc[NW][MQ][PITCH];
    __shared__ float s_m[NW][MQ], s_l[NW][MQ];
    constexpr int SPLIT = NW == max_warps(D) ? MAX_SPLIT : 1;  // (only the largest blocks come in clusters)
    __shared__ float s_in[2][SPLIT > 1 ? MQ * D : 1];
    __shared__ __align__(16) float s_ml[2][SPLIT][MQ][2];  // the cluster's shares of this block's output elements (by pass parity)
    __shared__ float s_tap[kMaxTaps];
    __shared__ uint32_t s_wkey[NW];
    __shared__ int s_wpos[NW], s_wslot[NW];
    cg::cluster_group cluster = cg::this_cluster();
    const int nsplit = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int bh = blockIdx.x / nsplit, h = bh % H;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
    unsigned char* blk = cache + L.header + (size_t)bh * L.stride;
    float* zc = reinterpret_cast<float*>(blk + L.off_z);
    int32_t* pidx = reinterpret_cast<int32_t*>(blk + L.off_pidx);
    int32_t* meta = reinterpret_cast<int32_t*>(blk + L.off_meta);
    const bool shared_head = SPLIT > 1 && nsplit > 1;          // (uniform in the cluster)
    if (shared_head) cluster.barrier_arrive();                 // (awaited before the first store into another block's shared memory)
    pdl_launch_dependents();
    pdl_wait();

    // Everything whose address is known is asked for at once, then everything that needs the counters: two memory latencies
    // stand before the first product, whatever the shape.
    const int n = meta[0], cnt_old = meta[1];
    uint4 qf[KP];                                              // pieces t, t + 4, .. of query head g (of the first pass)
    auto load_q = [&](int g0) {
#pragma unroll
        for (int j = 0; j < KP; ++j)
            qf[j] = g0 + g < G ? reinterpret_cast<const uint4*>(q1 + ((size_t)bh * G + g0 + g) * D)[t + 4 * j] : make_uint4(0, 0, 0, 0);
    };
    load_q(0);
    // the pool's logits and positions, before it is known whether the decision needs them
    constexpr int PRE = NT < 256 ? 4 : 2;
    float pz[PRE];
    int pp[PRE];
#pragma unroll
    for (int u = 0; u < PRE; ++u) {
        const int m = tid + u * NT;
        pz[u] = m < R ? zc[W + m] : INFINITY;
        pp[u] = m < R ? pidx[m] : -1;
    }
    float wk[CPL], wv[CPL];                                    // scorer weights of tap `wid` (the first block scores)
    const bool taps = rank == 0 && wid < K;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        wk[c] = taps ? cw[((size_t)h * K + wid) * 2 * D + lane + 32 * c] : 0.f;
        wv[c] = taps ? cw[((size_t)h * K + wid) * 2 * D + D + lane + 32 * c] : 0.f;
    }
    const int slot = n % W, p = n - W, half = K / 2;
    Rows rows;
    rows.K = blk + L.off_k; rows.V = blk + L.off_v;
    rows.k1 = reinterpret_cast<const unsigned char*>(k1 + (size_t)bh * D);
    rows.v1 = reinterpret_cast<const unsigned char*>(v1 + (size_t)bh * D);
    rows.W = W; rows.cnt = cnt_old;
    rows.n_ring = n < W ? n : W;
    rows.ring_spans = (rows.n_ring + 15) >> 4;
    rows.spans = rows.ring_spans + ((cnt_old + 15) >> 4) + 1;
    const bool back = BACK && (n & 1);
    const int step = back ? -NW * nsplit : NW * nsplit, first = back ? rows.spans - 1 - wid * nsplit - rank : wid * nsplit + rank;
    auto has = [&](int i) { return BACK ? (unsigned)i < (unsigned)rows.spans : i < rows.spans; };
    Group<D, SWZ> buf[NBUF];
    const float zp = p >= 0 && R > 0 ? zc[slot] : 0.f;
    if (has(first)) { const Span sp = rows.span(first); buf[0].load_k(rows, sp, g, t); buf[0].load_v(rows, sp, g, t); }
    const int jsc = K > 0 ? n - half : -1;                     // K = 0: the scorer runs outside (lte_cache_score)
    auto tap_rows = [&](int tap, float (&kx)[CPL], float (&vx)[CPL]) {   // channels lane, lane + 32, .. of the row under a tap
        const int pos = jsc + tap - half, r = pos < 0 ? 0 : pos % W;
        const bool ring = pos != n;
        const __nv_bfloat16* kr = reinterpret_cast<const __nv_bfloat16*>(ring ? rows.K : rows.k1) + (ring ? (size_t)r * D : 0);
        const __nv_bfloat16* vr = reinterpret_cast<const __nv_bfloat16*>(ring ? rows.V : rows.v1) + (ring ? (size_t)r * D : 0);
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int ch = lane + 32 * c, el = ring ? (cache_chunk_pos(L, r, ch >> 3) << 3) | (ch & 7) : ch;
            kx[c] = pos < 0 ? 0.f : __bfloat162float(kr[el]);
            vx[c] = pos < 0 ? 0.f : __bfloat162float(vr[el]);
        }
    };
    float kx[CPL], vx[CPL];
    if (taps && jsc >= 0) tap_rows(wid, kx, vx);
    if (NBUF == 2 && has(first + step)) { const Span sp = rows.span(first + step); buf[NBUF - 1].load_k(rows, sp, g, t); buf[NBUF - 1].load_v(rows, sp, g, t); }

    // ---- what happens to the token leaving the window ------------------------------------------------------------
    int dst = -1, cnt_new = cnt_old;
    if (p >= 0 && R > 0 && (p < sink || zp > zthr)) {
        if (cnt_old < R) { dst = cnt_old; cnt_new = cnt_old + 1; }
        else if (p >= sink) {
            // worst entry: lowest logit, the youngest among equals, never a sink entry
            uint32_t key = 0xffffffffu;                        // (order_key of a number; -0 counts as 0)
            int wpos = -1, wslot = -1;
            auto offer = [&](float z, int pos, int m) {
                const uint32_t k = order_key(z + 0.f);
                if (m < cnt_old && pos >= sink && (k < key || (k == key && pos > wpos))) { key = k; wpos = pos; wslot = m; }
            };
#pragma unroll
            for (int u = 0; u < PRE; ++u) offer(pz[u], pp[u], tid + u * NT);
            for (int m = tid + PRE * NT; m < cnt_old; m += NT) offer(zc[W + m], pidx[m], m);
            auto worst = [&]() {                               // over the warp; every lane then has it
                const uint32_t kmin = __reduce_min_sync(0xffffffffu, key);
                const int pmax = __reduce_max_sync(0xffffffffu, key == kmin ? wpos : -1);
                const unsigned who = __ballot_sync(0xffffffffu, key == kmin && wpos == pmax);
                wslot = __shfl_sync(0xffffffffu, wslot, __ffs(who) - 1);
                key = kmin; wpos = pmax;
            };
            worst();
            if (NW > 1) {
                if (lane == 0) { s_wkey[wid] = key; s_wpos[wid] = wpos; s_wslot[wid] = wslot; }
                __syncthreads();
                key = lane < NW ? s_wkey[lane] : 0xffffffffu; wpos = lane < NW ? s_wpos[lane] : -1; wslot = lane < NW ? s_wslot[lane] : -1;
                worst();
            }
            if (wslot >= 0 && order_key(zp + 0.f) > key) dst = wslot;
        }
    }
    const int masked_ring = p >= 0 && dst < 0 ? slot : -2;     // the popped row counts iff the pool takes it ...
    const int masked_pool = dst >= 0 && dst < cnt_old ? W + dst : -2;   // ... and then the entry it replaces does not

    // ---- the first block: logit of the newest token whose receptive field is complete -----------------------------
    if (rank == 0 && jsc >= 0) {
        for (int tap = wid; tap < K; tap += NW) {
            if (tap >= NW) {
                tap_rows(tap, kx, vx);
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    wk[c] = cw[((size_t)h * K + tap) * 2 * D + lane + 32 * c];
                    wv[c] = cw[((size_t)h * K + tap) * 2 * D + D + lane + 32 * c];
                }
            }
            float a = 0.f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) a += wk[c] * kx[c] + wv[c] * vx[c];
            a = warp_sum(a);
            if (lane == 0) s_tap[tap] = a;
        }
    }

    const int mover = NT - 1 - tid;                            // threads that move rows (not the warps that write the output, where there are several)
    uint4 mv = make_uint4(0, 0, 0, 0), nw = mv;                // a piece of the popped row, of the incoming one
    const float scale2 = scale * 1.44269504088896340736f, jump = 8.f / scale2;   // jump: a factor of 2^8 between weights, unscaled
    for (int g0 = 0; g0 < G; g0 += MQ) {
        const int nq = min(MQ, G - g0);
        if (g0 > 0) {                                          // further query heads read the rows again
            load_q(g0);
#pragma unroll
            for (int b = 0; b < NBUF; ++b)
                if (has(first + b * step)) { const Span sp = rows.span(first + b * step); buf[b].load_k(rows, sp, g, t); buf[b].load_v(rows, sp, g, t); }
        }
        float acc[MT][4], m0 = M_NONE, m1 = M_NONE, l0 = 0.f, l1 = 0.f;
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;

        // one span; its registers are refilled with the warp's span NBUF steps ahead as soon as a product has taken them
        auto compute = [&](Group<D, SWZ>& u, int i) {
            const Span cur = rows.span(i), nxt = rows.span(i + NBUF * step);
            const bool more = has(i + NBUF * step);
            // A product rounds its running sum towards zero, so every one starts from zero and the parts are added to the nearest
            // (NS sums side by side where the registers allow it: at d = 64 that costs 5 %).  With one running sum lse's error was 1.7
            // and 2.5 times what it is in plain fp32 (d = 64, 128; logits of 5), so it is 0.9 to 1.1 times.
            constexpr int NS = D == 128 ? 2 * KP : 1;
            float cs[NS][4];
#pragma unroll
            for (int i = 0; i < 2 * KP; ++i) {
                const int j = i >> 1, s = 2 * (i & 1);
                float part[4] = {0.f, 0.f, 0.f, 0.f};
                mma16816(part, word(u.k[0][j], s), word(u.k[1][j], s), word(u.k[0][j], s + 1), word(u.k[1][j], s + 1), word(qf[j], s), word(qf[j], s + 1));
#pragma unroll
                for (int e = 0; e < 4; ++e) cs[i % NS][e] = i < NS ? part[e] : cs[i % NS][e] + part[e];
            }
#pragma unroll
            for (int w = NS / 2; w > 0; w >>= 1)
#pragma unroll
                for (int j = 0; j < w; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) cs[j][e] += cs[j + w][e];
            float (&c)[4] = cs[0];
            if (more) u.load_k(rows, nxt, g, t);
            // c: rows g (0, 1) and g + 8 (2, 3), queries 2t and 2t + 1
            if (cur.n < 16 || (unsigned)(masked_ring - cur.row) < 16u || (unsigned)(masked_pool - cur.row) < 16u) {
                const int ra = cur.row + g, rb = ra + 8;
                if (g >= cur.n || ra == masked_ring || ra == masked_pool) c[0] = c[1] = -INFINITY;
                if (g + 8 >= cur.n || rb == masked_ring || rb == masked_pool) c[2] = c[3] = -INFINITY;
            }
            // The reference m follows the maximum only when that has grown by 2^8 (weights stay below 2^8, in fp32): a vote per
            // span instead of a reduction over its rows.
            const float x0 = fmaxf(c[0], c[2]), x1 = fmaxf(c[1], c[3]);
            if (__any_sync(0xffffffffu, x0 > m0 + jump || x1 > m1 + jump)) {
                float y0 = x0, y1 = x1;
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    y0 = fmaxf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
                    y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
                }
                y0 = fmaxf(y0, m0); y1 = fmaxf(y1, m1);
                const float f0 = exp2_fast((m0 - y0) * scale2), f1 = exp2_fast((m1 - y1) * scale2);
                m0 = y0; m1 = y1;
                l0 *= f0; l1 *= f1;
#pragma unroll
                for (int m = 0; m < MT; ++m) { acc[m][0] *= f0; acc[m][1] *= f1; acc[m][2] *= f0; acc[m][3] *= f1; }
            }
            const float p0 = exp2_fast((c[0] - m0) * scale2), p1 = exp2_fast((c[1] - m1) * scale2);
            const float p2 = exp2_fast((c[2] - m0) * scale2), p3 = exp2_fast((c[3] - m1) * scale2);
            l0 += p0 + p2; l1 += p1 + p3;
            const uint32_t hi0 = pack_bf16(p0, p1), hi1 = pack_bf16(p2, p3);
            const uint32_t lo0 = pack_bf16(p0 - __uint_as_float(hi0 << 16), p1 - __uint_as_float(hi0 & 0xffff0000u));
            const uint32_t lo1 = pack_bf16(p2 - __uint_as_float(hi1 << 16), p3 - __uint_as_float(hi1 & 0xffff0000u));
            const uint32_t h0 = movmatrix_trans(hi0), h1 = movmatrix_trans(hi1), e0 = movmatrix_trans(lo0), e1 = movmatrix_trans(lo1);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint32_t a0v = __byte_perm(u.v[0][m], u.v[1][m], 0x5410), a1v = __byte_perm(u.v[0][m], u.v[1][m], 0x7632);
                const uint32_t a2v = __byte_perm(u.v[2][m], u.v[3][m], 0x5410), a3v = __byte_perm(u.v[2][m], u.v[3][m], 0x7632);
                mma16816(acc[m], a0v, a1v, a2v, a3v, h0, h1);
                mma16816(acc[m], a0v, a1v, a2v, a3v, e0, e1);
            }
            if (more) u.load_v(rows, nxt, g, t);
        };
        for (int i = first; has(i); i += NBUF * step) {
            compute(buf[0], i);
            if (NBUF == 2 && has(i + step)) compute(buf[NBUF - 1], i + step);
        }
        if (rank == 0 && g0 + MQ >= G && mover < 2 * PIECES) {  // (back by the time the write-back needs them)
            mv = reinterpret_cast<const uint4*>(mover < PIECES ? rows.K : rows.V)[(size_t)slot * PIECES + cache_chunk_pos(L, slot, mover % PIECES)];
            nw = reinterpret_cast<const uint4*>(mover < PIECES ? rows.k1 : rows.v1)[mover % PIECES];
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) { l0 += __shfl_xor_sync(0xffffffffu, l0, o); l1 += __shfl_xor_sync(0xffffffffu, l1, o); }
        if (g0 > 0) __syncthreads();                           // the previous pass has been combined
        if (g == 0) { s_m[wid][2 * t] = m0; s_m[wid][2 * t + 1] = m1; s_l[wid][2 * t] = l0; s_l[wid][2 * t + 1] = l1; }
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            const int ch = D == 32 ? g * 4 + 2 * i : (i >> 2) * 64 + g * 8 + 2 * (i & 3);
            if (2 * t < nq) *reinterpret_cast<float2*>(&s_acc[wid][2 * t][ch]) = make_float2(acc[i][0], acc[i][2]);
            if (2 * t + 1 < nq) *reinterpret_cast<float2*>(&s_acc[wid][2 * t + 1][ch]) = make_float2(acc[i][1], acc[i][3]);
        }
        __syncthreads();
        if (shared_head && g0 == 0) cluster.barrier_wait();    // every block of the cluster has started: its shared memory is there
        const int per = nq * D / nsplit, par = (g0 / MQ) & 1;  // output elements each block of the cluster finishes
        for (int e = tid; e < nq * D; e += NT) {
            const int u = e / D, ch = e - u * D;
            float m = s_m[0][u];
#pragma unroll
            for (int w2 = 1; w2 < NW; ++w2) m = fmaxf(m, s_m[w2][u]);
            float tot = 0.f, o = 0.f;
#pragma unroll
            for (int w2 = 0; w2 < NW; ++w2) {
                const float f = exp2_fast((s_m[w2][u] - m) * scale2);   // a warp without rows: 0
                tot = fmaf(f, s_l[w2][u], tot);
                o = fmaf(f, s_acc[w2][u][ch], o);
            }
            if (!shared_head) {
                o1[((size_t)bh * G + g0 + u) * D + ch] = __float2bfloat16_rn(o / tot);
                if (ch == 0) lse1[(size_t)bh * G + g0 + u] = m * scale + logf(tot);
            } else {                                           // into the shared memory of the block that finishes this element
                const int own = e / per;
                *cluster.map_shared_rank(&s_in[par][rank * per + (e - own * per)], own) = o;
                if (ch < nsplit) *reinterpret_cast<float2*>(cluster.map_shared_rank(&s_ml[par][rank][u][0], ch)) = make_float2(m, tot);
            }
        }
        if (shared_head) {
            cluster.sync();                                    // all shares have arrived, and every row has been read
            for (int e = tid; e < per; e += NT) {
                const int el = rank * per + e, u = el / D, ch = el - u * D;
                float2 ml[SPLIT];
                float m = -INFINITY, tot = 0.f, o = 0.f;
#pragma unroll
                for (int r2 = 0; r2 < SPLIT; ++r2) {
                    ml[r2] = r2 < nsplit ? make_float2(s_ml[par][r2][u][0], s_ml[par][r2][u][1]) : make_float2(M_NONE, 0.f);
                    m = fmaxf(m, ml[r2].x);
                }
#pragma unroll
                for (int r2 = 0; r2 < SPLIT; ++r2) {
                    const float f = exp2_fast((ml[r2].x - m) * scale2);
                    tot = fmaf(f, ml[r2].y, tot);
                    if (r2 < nsplit) o = fmaf(f, s_in[par][r2 * per + e], o);
                }
                o1[((size_t)bh * G + g0 + u) * D + ch] = __float2bfloat16_rn(o / tot);
                if (ch == 0) lse1[(size_t)bh * G + g0 + u] = m * scale + logf(tot);
            }
        }
    }

    // ---- write-back: only what changed; every read of the old block lies before the barriers above ------------------
    if (rank != 0) return;
    if (mover < 2 * PIECES) {
        uint4* rowp = reinterpret_cast<uint4*>(const_cast<unsigned char*>(mover < PIECES ? rows.K : rows.V));
        const int pc = mover % PIECES;
        if (dst >= 0) rowp[(size_t)(W + dst) * PIECES + cache_chunk_pos(L, W + dst, pc)] = mv;
        rowp[(size_t)slot * PIECES + cache_chunk_pos(L, slot, pc)] = nw;
    }
    if (tid == (NW > 2 ? 32 : 0)) {
        if (dst >= 0) { zc[W + dst] = zp; pidx[dst] = p; }
        float znew = -INFINITY;
        if (jsc >= 0) {
            znew = cbias ? cbias[h] : 0.f;
            for (int tap = 0; tap < K; ++tap) znew += s_tap[tap];
        }
        zc[slot] = -INFINITY;                                  // the incoming token is not scored yet ...
        if (jsc >= 0) zc[jsc % W] = znew;                      // ... unless half == 0 (then jsc == n)
        meta[0] = n + 1;
        meta[1] = cnt_new;
    }
}

}  // namespace

// How many warps share a head: all warps of the launch are resident at once (16 per SM), so that the fixed parts of the
// heads (the counters, the combination, the write-back: about 4 us) run side by side instead of in waves.  Many heads: one
// warp each; fewer: up to eight, and beyond that a cluster of up to eight such blocks, while every warp has a group of rows.
int launch_decode_mma(const Params& p, void* cache, const void* q1, const void* k1, const void* v1, void* o1, float* lse1,
                      cudaStream_t st)
{
    const CacheLayout L = cache_layout(p.d, p.W, p.R, p.dtype);
    int n_sm = 0;
    if (int e = device_sm_count(&n_sm)) return e;
    const int BH = p.B * p.H;
    bool turn = false;
    if (int e = decode_turns(p, &turn)) return e;
    const int warps = warps_per_sm(p.d) * n_sm, most = max_warps(p.d);
    int nw = 1, nsplit = 1;
    for (int c : {2, 3, 4, 8})
        if (c <= most && BH <= n_sm * (warps_per_sm(p.d) / c) && (p.W + p.R) / c >= 16) nw = c;
    if (nw == most)
        while (nsplit < MAX_SPLIT && BH * nw * nsplit * 2 <= warps && (p.W + p.R) / (nw * nsplit * 2) >= 8) nsplit *= 2;
    // The direction is that of a head's rows: with more heads than run at once a step ends with the last heads and the next one begins
    // with the first, whose rows are gone either way (4,096 heads x 400 rows at d = 32: 57.7 us alternating, 56.3 forwards; 1,696 x 725 at d = 128,
    // four query heads each, 134.8 and 134.2).  With as many as run at once 2,368 x 300 at d = 64 takes 38.6 and 41.8, 1,184 x 725 at d = 128 71.1 and 74.6.
    turn = turn && (long long)BH * nw * nsplit <= warps;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(BH * nsplit); cfg.blockDim = dim3(nw * 32); cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = nsplit; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = nsplit > 1 ? 2 : 1;
    auto go = [&](auto kern) {
        return cudaLaunchKernelEx(&cfg, kern, (unsigned char*)cache, L, (const __nv_bfloat16*)q1, (const __nv_bfloat16*)k1,
                                  (const __nv_bfloat16*)v1, (__nv_bfloat16*)o1, lse1, p.w, p.bias, p.H, p.W, p.R, p.sink, p.K, p.zthr, p.scale, p.G);
    };
#define LTE_GO2(D, S, T) (nw == 8 ? go(decode_mma_kernel<D, max_warps(D), S, T>) : nw == 4 ? go(decode_mma_kernel<D, 4, S, T>) : \
                          nw == 3 ? go(decode_mma_kernel<D, 3, S, T>) : nw == 2 ? go(decode_mma_kernel<D, 2, S, T>) : go(decode_mma_kernel<D, 1, S, T>))
    // (256 swizzled rows pass the line of decode_turns from 1,400 heads on, which have a warp each)
#define LTE_GO(D, S) (!turn ? LTE_GO2(D, S, false) : !S ? LTE_GO2(D, false, true) : nw == 1 ? go(decode_mma_kernel<D, 1, S, true>) : LTE_GO2(D, S, false))
    cudaError_t e;
    switch (p.d) {
        case 32: e = LTE_GO(32, false); break;
        case 64: e = L.swz ? LTE_GO(64, true) : LTE_GO(64, false); break;
        case 128: e = LTE_GO(128, false); break;
        default: return LTE_ERR_UNSUPPORTED;
    }
#undef LTE_GO
#undef LTE_GO2
    return cuda_status(e);
}

}  // namespace lte
