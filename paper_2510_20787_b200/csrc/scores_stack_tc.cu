// The paper's scorer stack on the tcgen05 tensor cores (Section 3.1.1, hyper-parameters of Appendix A), bf16 inputs,
// d = 64: three dilated conv layers (kernel 3, dilation 2) over x = [k ; v], channels 128 -> 64 -> 32 -> 16, Swish
// after each, then a per-head linear map to one logit; the logit of token j is the stack's output at time j + 6.
//
// The keep decision z > logit(tau) has to agree with an fp64 evaluation to a few 1e-5 on z, so every product is
// exact: fp32 weights and fp32 hidden activations are split into three bf16 pieces (hi + mid + lo, 24 bits), and the
// pieces whose product matters (orders hi*hi, hi*mid, mid*hi, mid*mid, hi*lo, lo*hi) are accumulated in fp32 by the
// tensor core.  The pieces of a weight sit side by side along N (one MMA of N = 3 C_out covers hi, mid and lo at
// once; the epilogue adds the three column blocks), so an input tile is read from shared memory once per K step.
//
// Products of different widths accumulate in the same columns of the second and third layer.  One thread issues them and the chip runs them in
// that order (the logits agree with 64 bits to rounding wherever they have been compared), though only products of one shape are
// promised to keep it.
//
// A layer is a sum over its three taps of a [128 rows x C_in] x [C_in x C_out] product whose A operand is the
// previous layer's tile shifted down by 4, 2 or 0 rows.  Operands are kept in the unswizzled canonical layout (a
// column of 16-byte chunks per 8 channels, rows 16 bytes apart), where a row shift is a 16-byte-aligned change of the
// start address.  Row m of a tile is time tb - 8 + m: the input tile carries 4 more rows above, the first 4 rows of
// the second layer and the first 8 of the third are not used, so a tile yields 120 logits.
//
// One CTA per SM walks consecutive tiles of (head, batch) rows.  Four warps bring the input rows, by 16-byte asynchronous copies into
// their chunk columns (rows before time 0 zero-filled); one the first layer's weights, 64 input channels of a tap at a time,
// through a ring of three slots (their split image, 144 KB per head, does not fit beside the rest), and the small layers'
// weights once per head; two issue the MMAs.  Sixteen are the epilogues of the first two layers: TMEM -> bias, Swish -> three
// bf16 pieces -> the next layer's operand in shared memory; four take the third layer's dot product with the output vector.
// The weight image is built by a small kernel per call into caller-provided workspace.
//
// Bound by shared memory (per tile about 540 KB of MMA operands, 147 KB of weights and 140 KB of rows written and read: 6,500 cycles at
// 128 B a cycle, of about 7,700) and by a tile's chain (first epilogue, second layer's products, second epilogue), so what is not in that
// chain runs beside it: input rows half a tile ahead (the keys' columns are free while the values are multiplied), the first
// layer a tile ahead, the third layer and the output map behind (h1 has its own columns, so the next tile's h0 may be
// written meanwhile), and the second layer starts on the first 32 channels of h0 while the epilogue works on the others.
// Measured (weight image and scorer in a CUDA graph, us; before: one warp for rows and weights, whole taps in a ring of two, h1 in the place of
// h0, eight epilogue warps): 256 heads x 4,096 337 -> 271 64 x 4,096 101 -> 83, 32 x 4,096 59 -> 48,
// 256 x 768 84 -> 68, 8 x 1,000 16.4 -> 13.5; mean error against 64 bits 1.5e-6 -> 1.3e-6.  The row warps gave 337 -> 282, sixteen epilogue
// warps in place of eight 275, the image by chunks and the wait for it behind the set-up the rest (4 us a call).
#include "tc_common.cuh"

#include <type_traits>

namespace lte {

__device__ StatusWord g_stack_tc_status = LTE_STATUS_INIT;

namespace {

using namespace tc;

constexpr int ST_D = 64, ST_C0 = 128, ST_C1 = 64, ST_C2 = 32, ST_C3 = 16;
constexpr int ST_ROWS = 132;                                   // rows of a chunk column (132 input rows; 4 + 128 hidden rows)
constexpr int ST_COL = ST_ROWS * 16;                           // bytes of a chunk column
constexpr int ST_XROWS = 132;                                  // input rows per tile: times tb-12 .. tb+119
constexpr int ST_VALID = 120;                                  // logits per tile
constexpr int ST_HALF = 6;
constexpr int W_EPI = 16, W_MMA0 = W_EPI, W_WEIGHTS = W_MMA0 + 1, W_MMA1 = W_MMA0 + 2, W_OUT = W_MMA0 + 3, W_X = W_OUT + 4, X_WARPS = 4;
constexpr int ST_THREADS = (W_X + X_WARPS) * 32;

// per-head image in the workspace (bytes): first-layer weights per tap, then what stays resident for the head
constexpr int IMG_W0_TAP = 16 * 192 * 16;                      // [chunk 16][n = piece * 64 + c_out][8 channels] bf16
constexpr int IMG_W0 = 3 * IMG_W0_TAP;
constexpr int IMG_W1 = 3 * 8 * 96 * 16;                        // [tap][chunk 8][n = piece * 32 + c_out][8]
constexpr int IMG_W2 = 3 * 4 * 48 * 16;                        // [tap][chunk 4][n = piece * 16 + c_out][8]
constexpr int IMG_PAR = 640;                                   // floats: b0[64] b1[32] b2[16] wout[16] bout
constexpr int IMG_RES = IMG_W1 + IMG_W2 + IMG_PAR;             // resident part, one bulk copy
constexpr int IMG_HEAD = IMG_W0 + IMG_RES;

// shared memory map (every offset a multiple of 128)
constexpr int RING = 3, W0_PART = IMG_W0_TAP / 2, PARTS = 6;   // a slot holds 64 input channels of a tap; parts of a tile: keys (taps 0, 1, 2), values
__device__ __forceinline__ int part_of(int j) { return j < 3 ? 2 * j : 2 * (j - 3) + 1; }   // its place in the image
constexpr int OFF_RING = 0;
constexpr int OFF_X = OFF_RING + RING * W0_PART;               // input tile: 16 chunk columns
constexpr int OFF_H0 = OFF_X + 16 * ST_COL;                    // 3 x 8 columns of h0
constexpr int OFF_H1 = OFF_H0 + 24 * ST_COL;                   // 3 x 4 columns of h1
constexpr int OFF_W1 = OFF_H1 + 12 * ST_COL;
constexpr int OFF_W2 = OFF_W1 + IMG_W1;
constexpr int OFF_PAR = OFF_W2 + IMG_W2;
constexpr int OFF_BAR = OFF_PAR + IMG_PAR;
constexpr int ST_SMEM = OFF_BAR + 256;
static_assert(ST_SMEM <= 232448, "shared memory");
// two first-layer accumulators of 192 columns, the second layer's (96), the third's (32: the products with a weight's low piece go to the
// columns of its middle piece, beside which they are as small as beside their own sum)
constexpr uint32_t D0_COL = 0, D1_COL = 384, D2_COL = 480, ST_TMEM = 512;

// unswizzled K-major descriptor: 8 rows x 16 bytes per core matrix, SBO = 128 bytes between 8-row groups, LBO = the
// distance between the two 8-channel chunk columns of a K = 16 step
constexpr uint32_t kDescHiFlat = (128u >> 4) | (1u << 14);

__device__ __forceinline__ void swait(uint32_t bar, uint32_t parity, int code) { mbar_wait_long(bar, parity, code, &g_stack_tc_status); }
__device__ __forceinline__ void swait_uni(uint32_t bar, uint32_t parity, int code) { mbar_wait_uni_long(bar, parity, code, &g_stack_tc_status); }
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Swish with the fast exponential and division: their error (a few 1e-7 relative) is below that of the tensor core's
// fp32 accumulation, which bounds the accuracy of the logits here (about 1e-5 absolute at |z| of a few units)
__device__ __forceinline__ float swish(float y) { return __fdividef(y, 1.f + __expf(-y)); }

// three bf16 pieces of two floats, packed (low half = a)
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    hi = *reinterpret_cast<uint32_t*>(&h);
    a -= __uint_as_float(hi << 16); b -= __uint_as_float(hi & 0xffff0000u);
    h = __floats2bfloat162_rn(a, b);
    mid = *reinterpret_cast<uint32_t*>(&h);
    a -= __uint_as_float(mid << 16); b -= __uint_as_float(mid & 0xffff0000u);
    h = __floats2bfloat162_rn(a, b);
    lo = *reinterpret_cast<uint32_t*>(&h);
}

// ---- weight image -------------------------------------------------------------------------------------------------
// blockIdx.x = head, the blocks along y share its elements, eight input channels a thread (an element a thread and a loop: 4 to 5 us more).  wpack = wl0 | wl1 | wl2 | wout with wl[l] [H][c_out][3][c_in]; bpack = bl0 | bl1 | bl2 | bout or null.
// dg = the head dimension of the data, 64 or 32.  d = 32 runs the d = 64 kernel on a padded problem: channels [dg, 64) of the
// key and value halves of the input, and the upper half of every hidden layer, carry zero weights (and zero biases, so the
// padded activations are Swish(0) = 0); the image below is the d = 64 layout with those zeros written in.
constexpr int IMG_N0 = 3 * ST_C0 / 8 * ST_C1, IMG_N1 = 3 * ST_C1 / 8 * ST_C2, IMG_N2 = 3 * ST_C2 / 8 * ST_C3;   // items of the three layers
constexpr int IMG_THREADS = 256, IMG_BLOCKS = (IMG_N0 + IMG_N1 + IMG_N2 + IMG_PAR / 4 + IMG_THREADS - 1) / IMG_THREADS;
__global__ void __launch_bounds__(IMG_THREADS) stack_image_kernel(const float* __restrict__ wpack, const float* __restrict__ bpack, uint8_t* __restrict__ img, int H, int dg)
{
    pdl_launch_dependents();
    pdl_wait();
    const int h = blockIdx.x, item = blockIdx.y * IMG_THREADS + threadIdx.x;
    uint8_t* out = img + (size_t)h * IMG_HEAD;
    const int c0 = 2 * dg, c1 = dg, c2 = dg / 2, c3 = dg / 4;   // the real channel plan
    const float* g0 = wpack + (size_t)h * c1 * 3 * c0;
    const float* g1 = wpack + (size_t)H * c1 * 3 * c0 + (size_t)h * c2 * 3 * c1;
    const float* g2 = wpack + (size_t)H * (c1 * 3 * c0 + c2 * 3 * c1) + (size_t)h * c3 * 3 * c2;
    const float* go = wpack + (size_t)H * (c1 * 3 * c0 + c2 * 3 * c1 + c3 * 3 * c2) + (size_t)h * c3;
    // Eight input channels of one output channel and tap in their three pieces.  Padded dims CIN x COUT, real dims cin_r x cout_r;
    // the first layer's input channels are two halves (key, value), each with its real channels first.  A chunk of
    // eight channels is real or padding as a whole.
    auto fill = [&](uint8_t* dst, const float* g, auto cin, auto cout, int cin_r, int cout_r, bool split, int e) {
        constexpr int CIN = decltype(cin)::value, COUT = decltype(cout)::value;
        // dst [tap][chunk CIN/8][n = piece * COUT + o][8] ; g [o][tap][cin_r]
        const int c = e % (CIN / 8), o = e / (CIN / 8) % COUT, tau = e / (CIN / 8 * COUT), ch = c * 8;
        const int cr = !split ? (ch < cin_r ? ch : -1) : ch % (CIN / 2) < cin_r / 2 ? ch / (CIN / 2) * (cin_r / 2) + ch % (CIN / 2) : -1;
        uint32_t pc[3][4] = {};
        if (o < cout_r && cr >= 0) {
            const float* src = g + ((size_t)o * 3 + tau) * cin_r + cr;
#pragma unroll
            for (int u = 0; u < 4; ++u) split3(src[2 * u], src[2 * u + 1], pc[0][u], pc[1][u], pc[2][u]);
        }
#pragma unroll
        for (int u = 0; u < 3; ++u)
            *reinterpret_cast<uint4*>(dst + ((size_t)(tau * (CIN / 8) + c) * 3 * COUT + u * COUT + o) * 16) = make_uint4(pc[u][0], pc[u][1], pc[u][2], pc[u][3]);
    };
    using std::integral_constant;
    if (item < IMG_N0) fill(out, g0, integral_constant<int, ST_C0>{}, integral_constant<int, ST_C1>{}, c0, c1, true, item);
    else if (item < IMG_N0 + IMG_N1) fill(out + IMG_W0, g1, integral_constant<int, ST_C1>{}, integral_constant<int, ST_C2>{}, c1, c2, false, item - IMG_N0);
    else if (item < IMG_N0 + IMG_N1 + IMG_N2)
        fill(out + IMG_W0 + IMG_W1, g2, integral_constant<int, ST_C2>{}, integral_constant<int, ST_C3>{}, c2, c3, false, item - IMG_N0 - IMG_N1);
    else if (const int e = item - IMG_N0 - IMG_N1 - IMG_N2; e < IMG_PAR / 4) {
        float x = 0.f;
        if (e < 64) x = (bpack && e < c1) ? bpack[(size_t)h * c1 + e] : 0.f;
        else if (e < 96) x = (bpack && e - 64 < c2) ? bpack[(size_t)H * c1 + (size_t)h * c2 + (e - 64)] : 0.f;
        else if (e < 112) x = (bpack && e - 96 < c3) ? bpack[(size_t)H * (c1 + c2) + (size_t)h * c3 + (e - 96)] : 0.f;
        else if (e < 128) x = e - 112 < c3 ? go[e - 112] : 0.f;
        else if (e == 128) x = bpack ? bpack[(size_t)H * (c1 + c2 + c3) + h] : 0.f;
        reinterpret_cast<float*>(out + IMG_W0 + IMG_W1 + IMG_W2)[e] = x;
    }
}

// ---- main kernel --------------------------------------------------------------------------------------------------
struct StackWork { int h, bh, tb; };
__device__ __forceinline__ StackWork stack_work(int f, int n_t, int B, int H) {
    const int hb = f / n_t, tile = f - hb * n_t, h = hb / B, b = hb - h * B;
    return StackWork{h, b * H + h, ST_HALF + tile * ST_VALID};
}

__global__ void __launch_bounds__(ST_THREADS, 1)
scores_stack_tc_kernel(const __nv_bfloat16* __restrict__ kg, const __nv_bfloat16* __restrict__ vg,
                       const uint8_t* __restrict__ img, float* __restrict__ z, float* __restrict__ r_out, int B, int H,
                       int Tlen, int n_t, int n_flat, int per_cta, int dg)
{
    pdl_launch_dependents();
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 127u) != 0) { if (threadIdx.x == 0) atomicExch(&g_stack_tc_status.code, 9); return; }
    const uint32_t sRing = base + OFF_RING, sX = base + OFF_X, sH0 = base + OFF_H0, sH1 = base + OFF_H1, sW1 = base + OFF_W1, sW2 = base + OFF_W2;
    const float* par = reinterpret_cast<const float*>(smem_raw + OFF_PAR);
    // Barriers (it: tile of this CTA's walk; n: part of the first layer's weights, PARTS per tile):
    //   bar_x[2], bar_xe[2]   the tile's keys / values are in (2 arrivals) / have been read
    //   bar_rf[n % 3], bar_re[n % 3]   part n has landed / been read
    //   bar_d0[it & 1], bar_f0[it & 1]   the first layer's accumulator is complete / has been loaded (16 arrivals)
    //   bar_h0[2]        (16 arrivals) channels 0-31 / 32-63 of h0 are in     bar_d1   the second layer is complete
    //   bar_h1           (16 arrivals) h1 is in, the second accumulator free  bar_d2   the third layer is complete, h1's columns free
    //   bar_f2           (4 arrivals) the third accumulator has been loaded  bar_ed4[it & 3]  (4 arrivals) the tile's logits are out
    //   bar_w            the head's resident weights are in
    const uint32_t bar0 = base + OFF_BAR;
    const uint32_t bar_x = bar0 + 184, bar_xe = bar0 + 200, bar_w = bar0 + 8, bar_rf = bar0 + 16, bar_re = bar0 + 40, bar_d0 = bar0 + 64, bar_f0 = bar0 + 80, bar_h0 = bar0 + 96;
    const uint32_t bar_d1 = bar0 + 112, bar_h1 = bar0 + 120, bar_d2 = bar0 + 128, bar_f2 = bar0 + 136, bar_ed4 = bar0 + 144, tmem_slot = bar0 + 176;
    volatile uint32_t* tmem_slot_gen = reinterpret_cast<volatile uint32_t*>(smem_raw + OFF_BAR + 176);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int f_begin = blockIdx.x * per_cta, f_end = min(f_begin + per_cta, n_flat);
    const int n_my = f_end - f_begin;

    // hidden-activation columns start out as zeros (their first rows are read by shifted operands before anything
    // meaningful is written there; what those rows produce is never used, but it should be finite)
    for (int e = tid; e < (36 * ST_COL) / 16; e += ST_THREADS)
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sH0 + e * 16), "r"(0u) : "memory");
    if (tid == 0) {
        mbar_init(bar_w, 1);
#pragma unroll
        for (int e = 0; e < RING; ++e) { mbar_init(bar_rf + 8 * e, 1); mbar_init(bar_re + 8 * e, 1); }
#pragma unroll
        for (int e = 0; e < 2; ++e) { mbar_init(bar_d0 + 8 * e, 1); mbar_init(bar_f0 + 8 * e, W_EPI); mbar_init(bar_h0 + 8 * e, W_EPI); mbar_init(bar_x + 8 * e, X_WARPS / 2); mbar_init(bar_xe + 8 * e, 1); }
        mbar_init(bar_d1, 1); mbar_init(bar_h1, W_EPI); mbar_init(bar_d2, 1); mbar_init(bar_f2, 4);
#pragma unroll
        for (int e = 0; e < 4; ++e) mbar_init(bar_ed4 + 8 * e, 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA0) tmem_alloc(tmem_slot, ST_TMEM);
    fence_proxy_async();                                       // the zero fill is visible to the TMA writes and MMA reads that follow
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_gen;
    pdl_wait();                                                // the weight image is written by the preceding kernel

    if (warp == W_WEIGHTS) {
        // =================================== producer ======================================================
        const bool leader = lane == 0;
        auto load_part = [&](int n, int h) {
            if (leader) {
                const uint32_t bar = bar_rf + 8 * (n % RING);
                mbar_expect_tx(bar, W0_PART);
                bulk_g2s(sRing + (n % RING) * W0_PART, img + (size_t)h * IMG_HEAD + (size_t)part_of(n % PARTS) * W0_PART, W0_PART, bar);
            }
        };
        auto load_head = [&](int h) {
            if (leader) {
                mbar_expect_tx(bar_w, IMG_RES);
                bulk_g2s(sW1, img + (size_t)h * IMG_HEAD + IMG_W0, IMG_RES, bar_w);
            }
        };
        if (n_my > 0) {
            StackWork w = stack_work(f_begin, n_t, B, H);
            int h_loaded = w.h;
            load_head(w.h);
            for (int n = 0; n < RING; ++n) load_part(n, w.h);
            for (int it = 0; it < n_my; ++it) {
                const bool more = it + 1 < n_my;
                const StackWork wn = more ? stack_work(f_begin + it + 1, n_t, B, H) : w;
#pragma unroll 1
                for (int j = 0; j < PARTS; ++j) {              // every part is awaited once, in order; its slot takes the part three later
                    const int n = PARTS * it + j;
                    swait(bar_re + 8 * (n % RING), (n / RING) & 1, 20);
                    if (j + RING < PARTS) load_part(n + RING, w.h);
                    else if (more) load_part(n + RING, wn.h);
                }
                // The resident weights change with the head, once every reader of the old ones is done with the previous tile; a
                // head's first tile waits for the new ones.  The ends of the tiles are awaited two tiles late, where that does not hold
                // up the loads above.  While this warp waits for the end of tile it-2, the others can get as far as the end of tile it (of tile
                // it+1 only the keys' parts are there), so the barrier is one of four by tile number: with two, a late waiter would
                // take the later completion for the one it wants.
                if (it >= 2) swait(bar_ed4 + 8 * ((it - 2) & 3), ((it - 2) >> 2) & 1, 22);
                if (more && wn.h != h_loaded) {
                    swait(bar_ed4 + 8 * (it & 3), (it >> 2) & 1, 23);
                    load_head(wn.h);
                    h_loaded = wn.h;
                }
                w = wn;
            }
        }
    } else if (warp >= W_X) {
        // =================================== input rows ====================================================
        // Two warps load the keys' half of the tile, two the values', 16 bytes per copy: a lane takes row (l & 7) of a block of 8
        // rows and one of 4 chunks, so a quarter warp writes 128 contiguous bytes and reads full 32-byte sectors.  Rows outside
        // [0, T) are zero-filled.  (Tensor-map copies with 16-byte boxes needed about 3,600 cycles per tile, one warp for everything
        // 4,900, which the first layer waited for.)
        const int part = (warp - W_X) >> 1, sub = (warp - W_X) & 1, r_in = lane & 7, cq = lane >> 3;
        for (int it = 0; it < n_my; ++it) {
            const StackWork w = stack_work(f_begin + it, n_t, B, H);
            const __nv_bfloat16* rows = (part ? vg : kg) + (size_t)w.bh * Tlen * dg;
            const int t0 = w.tb - 12;
            if (it > 0) swait(bar_xe + 8 * part, (it - 1) & 1, 24);
#pragma unroll 3
            for (int rb = sub; rb < (ST_XROWS + 7) / 8; rb += 2) {
                const int r = rb * 8 + r_in, t = t0 + r;
                const bool ok = t >= 0 && t < Tlen;
                if (r < ST_XROWS) {
#pragma unroll
                    for (int cg = 0; cg < 2; ++cg) {
                        const int c = cg * 4 + cq;
                        const bool real = ok && c * 8 < dg;    // channels past the head dimension are zero-filled
                        cp_async16(sX + (part * 8 + c) * ST_COL + r * 16, rows + (size_t)(real ? t : 0) * dg + (real ? c * 8 : 0), real ? 16u : 0u);
                    }
                }
            }
            cp_async_commit();
            cp_async_wait<0>();
            fence_proxy_async();                               // the tensor core reads these rows through the async proxy
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_x + 8 * part);
        }
    } else if (warp == W_MMA0) {
        // =================================== MMA issue, first layer ========================================
        // Two warps issue MMAs: this one the first layer, one tile ahead of the epilogues and into the other of two accumulators;
        // another warp the second and third layers.  The whole warp walks the schedule, an elected thread issues.
        constexpr uint32_t LBO_X = ST_COL, LBO_W0 = 192 * 16;
        for (int it = 0; it < n_my; ++it) {
            // this accumulator was last used by tile it-2: its epilogue has loaded it.  (Barriers per accumulator: this
            // warp runs up to two tiles ahead of the epilogues, and a barrier must never get two phases ahead of a waiter.)
            if (uni(it >= 2)) swait_uni(bar_f0 + 8 * (it & 1), ((it >> 1) - 1) & 1, 6);
            const uint32_t d = tmem + D0_COL + (it & 1) * 192;
#pragma unroll 1
            for (int j = 0; j < PARTS; ++j) {                  // the keys' half, taps 0, 1, 2, then the values'
                const int n = PARTS * it + j, hv = j >= 3, tau = j - 3 * hv;
                if (uni(tau == 0)) swait_uni(bar_x + 8 * hv, it & 1, 1);
                swait_uni(bar_rf + 8 * (n % RING), (n / RING) & 1, 2);
                tc_fence_after();
                const uint32_t a0 = desc_lo(sX + hv * 8 * ST_COL + 2 * tau * 16, LBO_X), b0 = desc_lo(sRing + (n % RING) * W0_PART, LBO_W0);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        umma(d, desc64(a0 + ((2 * kk * ST_COL) >> 4), kDescHiFlat), desc64(b0 + ((2 * kk * 192 * 16) >> 4), kDescHiFlat),
                             instr_desc(128, 192, false), (j > 0 || kk > 0) ? 1u : 0u);
                    umma_commit(bar_re + 8 * (n % RING));
                    if (tau == 2) umma_commit(bar_xe + 8 * hv);
                    if (j == PARTS - 1) umma_commit(bar_d0 + 8 * (it & 1));
                }
                __syncwarp();
            }
        }
    } else if (warp == W_MMA1) {
        // =================================== MMA issue, second and third layers ============================
        constexpr uint32_t LBO_X = ST_COL, LBO_W1 = 96 * 16, LBO_W2 = 48 * 16;
        int heads_seen = 0, h_prev = -1;
        for (int it = 0; it < n_my; ++it) {
            const StackWork w = stack_work(f_begin + it, n_t, B, H);
            if (uni(w.h != h_prev)) { swait_uni(bar_w, heads_seen & 1, 3); ++heads_seen; h_prev = w.h; }   // this head's small layers are in
            // ---- layer 1: halves of h0 as they come, taps x activation pieces (N = 96, 64, 32: the weight pieces each one meets) x 2 K steps ----
#pragma unroll
            for (int hv = 0; hv < 2; ++hv) {
                swait_uni(bar_h0 + 8 * hv, it & 1, 4);
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int s = 0; s < 18; ++s) {
                        const int tau = s / 6, p = s / 2 % 3, kk = 2 * hv + (s & 1);
                        const uint32_t a1 = desc_lo(sH0 + p * 8 * ST_COL + 2 * tau * 16, LBO_X), b1 = desc_lo(sW1 + tau * 8 * 96 * 16, LBO_W1);
                        const uint32_t idesc = p == 0 ? instr_desc(128, 96, false) : p == 1 ? instr_desc(128, 64, false) : instr_desc(128, 32, false);
                        umma(tmem + D1_COL, desc64(a1 + ((2 * kk * ST_COL) >> 4), kDescHiFlat), desc64(b1 + ((2 * kk * 96 * 16) >> 4), kDescHiFlat), idesc,
                             (hv > 0 || s > 0) ? 1u : 0u);
                    }
                    if (hv == 1) umma_commit(bar_d1);
                }
                __syncwarp();
            }
            // ---- layer 2: 2 K steps; activation pieces hi, mid, lo meet the weight pieces hi and mid (N = 32), the same, hi (N = 16);
            // hi meets lo (N = 16) in the middle pieces' columns ----
            swait_uni(bar_h1, it & 1, 5);
            if (uni(it > 0)) swait_uni(bar_f2, (it - 1) & 1, 7);
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
                for (int s = 0; s < 24; ++s) {
                    const int tau = s / 8, p = s / 2 % 4, kk = s & 1;      // (p = 3: hi with lo)
                    const uint32_t a2 = desc_lo(sH1 + (p % 3) * 4 * ST_COL + 2 * tau * 16, LBO_X);
                    const uint32_t b2 = desc_lo(sW2 + tau * 4 * 48 * 16 + (p == 3 ? 32 * 16 : 0), LBO_W2);
                    const uint32_t idesc = p < 2 ? instr_desc(128, 32, false) : instr_desc(128, 16, false);
                    umma(tmem + D2_COL + (p == 3 ? 16 : 0), desc64(a2 + ((2 * kk * ST_COL) >> 4), kDescHiFlat),
                         desc64(b2 + ((2 * kk * 48 * 16) >> 4), kDescHiFlat), idesc, s > 0 ? 1u : 0u);
                }
                umma_commit(bar_d2);
            }
            __syncwarp();
        }
    } else if (warp < W_EPI) {
        // =================================== epilogue warps, first and second layer ========================
        // warp w owns TMEM lanes 32 (w & 3) .. +31 (row m of the tile) and 8 of every 32 channels.  (Sixteen warps: the work is a chain of
        // latencies.  Eight took 5,100 cycles a tile.)
        const int q = warp & 3, c4 = warp >> 2;
        const int m = q * 32 + lane;
        const uint32_t lane_base = ((uint32_t)(q * 32)) << 16;
        const uint32_t row_off = (uint32_t)(4 + m) * 16;       // hidden rows sit 4 rows down their columns
        auto store_chunk = [](uint32_t dst, const uint32_t (&wv)[4]) {
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(wv[0]), "r"(wv[1]), "r"(wv[2]), "r"(wv[3]) : "memory");
        };
        // chunk ch of 8 channels: the three column blocks of a layer's accumulator, `step` columns apart -> the next layer's
        // operand, three pieces `next` bytes apart
        auto load_chunk = [&](uint32_t col, uint32_t step, int ch, uint32_t (&a)[3][8]) {
#pragma unroll
            for (int s = 0; s < 3; ++s) tmem_ld8(tmem + lane_base + col + s * step + ch * 8, a[s]);
            tmem_wait_ld();
        };
        auto hidden = [&](const uint32_t (&a)[3][8], const float* bias, uint32_t dst0, uint32_t next, int ch, uint32_t live_mask) {
            float bv[8];
            *reinterpret_cast<float4*>(&bv[0]) = *reinterpret_cast<const float4*>(bias + ch * 8);
            *reinterpret_cast<float4*>(&bv[4]) = *reinterpret_cast<const float4*>(bias + ch * 8 + 4);
            uint32_t hi[4], mid[4], lo[4];
            auto two = [&](int s, int e) { return pack2(__uint_as_float(a[s][2 * e]), __uint_as_float(a[s][2 * e + 1])); };
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float y0, y1;
                unpack2(add2(add2(add2(two(0, e), two(1, e)), two(2, e)), pack2(bv[2 * e], bv[2 * e + 1])), y0, y1);
                y0 = __uint_as_float(__float_as_uint(swish(y0)) & live_mask);
                y1 = __uint_as_float(__float_as_uint(swish(y1)) & live_mask);
                split3(y0, y1, hi[e], mid[e], lo[e]);
            }
            const uint32_t dst = dst0 + (uint32_t)ch * ST_COL + row_off;
            store_chunk(dst, hi); store_chunk(dst + next, mid); store_chunk(dst + 2 * next, lo);
        };
        auto publish = [&](uint32_t bar) {
            fence_proxy_async();                               // the tensor core reads these rows through the async proxy
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        int heads_seen = 0, h_prev = -1;
        for (int it = 0; it < n_my; ++it) {
            const StackWork w = stack_work(f_begin + it, n_t, B, H);
            // every layer's output is zero at negative times (a mask, not a branch: the channels' chains must interleave)
            const uint32_t live_mask = w.tb - 8 + m >= 0 ? 0xffffffffu : 0u;
            if (w.h != h_prev) { swait(bar_w, heads_seen & 1, 10); ++heads_seen; h_prev = w.h; }

            // ---- layer 0 -> h0, 32 channels at a time ----
            swait(bar_d0 + 8 * (it & 1), (it >> 1) & 1, 11);
            tc_fence_after();
#pragma unroll
            for (int hv = 0; hv < 2; ++hv) {
                uint32_t a[3][8];
                load_chunk(D0_COL + (it & 1) * 192, 64, 4 * hv + c4, a);
                if (hv == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_f0 + 8 * (it & 1));   // the accumulator may take tile it + 2
                }
                hidden(a, par, sH0, 8 * ST_COL, 4 * hv + c4, live_mask);
                publish(bar_h0 + 8 * hv);
            }

            // ---- layer 1 -> h1 ----
            swait(bar_d1, it & 1, 12);
            tc_fence_after();
            uint32_t a[3][8];
            load_chunk(D1_COL, 32, c4, a);
            if (it > 0) swait(bar_d2, (it - 1) & 1, 13);       // the third layer has read the previous tile's h1
            hidden(a, par + 64, sH1, 4 * ST_COL, c4, live_mask);
            publish(bar_h1);
        }
    } else {
        // =================================== output warps: third layer and the output map, one logit per row =
        const int q = warp & 3, m = q * 32 + lane;
        const uint32_t lane_base = ((uint32_t)(q * 32)) << 16;
        auto f = [](uint32_t u) { return __uint_as_float(u); };
        int heads_seen = 0, h_prev = -1;
        for (int it = 0; it < n_my; ++it) {
            const int ff = f_begin + it;
            const StackWork w = stack_work(ff, n_t, B, H);
            const int time = w.tb - 8 + m;
            const uint32_t live_mask = time >= 0 ? 0xffffffffu : 0u;
            if (w.h != h_prev) { swait(bar_w, heads_seen & 1, 14); ++heads_seen; h_prev = w.h; }
            swait(bar_d2, it & 1, 15);
            tc_fence_after();
            uint32_t a[16], b[16];
            tmem_ld16(tmem + lane_base + D2_COL, a);
            tmem_ld16(tmem + lane_base + D2_COL + 16, b);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_f2);                // the accumulator may take the next tile
            float pv[32];                                      // b2[16] | wout[16]
#pragma unroll
            for (int e = 0; e < 8; ++e) *reinterpret_cast<float4*>(&pv[4 * e]) = *reinterpret_cast<const float4*>(par + 96 + 4 * e);
            float zq[4] = {par[128], 0.f, 0.f, 0.f};
#pragma unroll
            for (int c0 = 0; c0 < 16; ++c0) {
                float y = (f(a[c0]) + f(b[c0])) + pv[c0];
                y = __uint_as_float(__float_as_uint(swish(y)) & live_mask);
                zq[c0 & 3] = fmaf(pv[16 + c0], y, zq[c0 & 3]);
            }
            const float zz = (zq[0] + zq[1]) + (zq[2] + zq[3]);
            const int j = time - ST_HALF;                      // the logit of token j is the output at time j + 6
            if (m >= 8 && time < Tlen) {
                z[(size_t)w.bh * Tlen + j] = zz;
                if (r_out) r_out[(size_t)w.bh * Tlen + j] = 1.f / (1.f + expf(-zz));
            }
            // the last tile of a row also marks the six tokens whose right context does not exist yet
            if ((ff + 1) % n_t == 0 && q == 0 && lane < ST_HALF && Tlen - ST_HALF + lane >= 0) {
                z[(size_t)w.bh * Tlen + Tlen - ST_HALF + lane] = -INFINITY;
                if (r_out) r_out[(size_t)w.bh * Tlen + Tlen - ST_HALF + lane] = 0.f;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_ed4 + 8 * (it & 3));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == W_MMA0) tmem_dealloc(tmem, ST_TMEM);
}

}  // namespace

int stack_tc_status_fetch_and_clear() { return status_fetch_and_clear(g_stack_tc_status); }

// Workspace of the tensor-core stack scorer (the split weight image), 0 where that path does not apply.
size_t scores_stack_tc_workspace(const Params& p)
{
    if (p.dtype != LTE_BF16 || (p.d != ST_D && p.d != 32) || p.T <= 2 * ST_HALF) return 0;
    return (size_t)p.H * IMG_HEAD;
}

// LTE_ERR_UNSUPPORTED where the path does not apply or the workspace is too small (the caller then runs the fp32 kernel).
int launch_scores_stack_tc(const Params& p, const void* k, const void* v, float* z, float* r, void* ws, size_t ws_bytes,
                           cudaStream_t st)
{
    const size_t need = scores_stack_tc_workspace(p);
    if (need == 0 || !ws || ws_bytes < need || ((uintptr_t)ws & 127u) != 0) return LTE_ERR_UNSUPPORTED;
    static PerDeviceOnce attr;
    if (int e = attr.run([] { return cudaFuncSetAttribute(scores_stack_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ST_SMEM); })) return e;
    int n_sm = 0;
    if (int e = device_sm_count(&n_sm)) return e;
    const int BH = p.B * p.H;
    if (int e = cuda_status(launch_pdl(stack_image_kernel, dim3(p.H, IMG_BLOCKS), dim3(IMG_THREADS), 0, st, p.w, p.bias, (uint8_t*)ws, p.H, p.d))) return e;
    const int n_t = (p.T - ST_HALF + ST_VALID - 1) / ST_VALID;
    const long long n_flat = (long long)BH * n_t;
    if (n_flat > 0x7fffffffLL) return LTE_ERR_UNSUPPORTED;
    const int grid = (int)(n_flat < n_sm ? n_flat : n_sm);
    const int per = (int)((n_flat + grid - 1) / grid);
    const int n_cta = (int)((n_flat + per - 1) / per);
    return cuda_status(launch_pdl(scores_stack_tc_kernel, dim3(n_cta), dim3(ST_THREADS), ST_SMEM, st, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v,
                                  (const uint8_t*)ws, z, r, p.B, p.H, p.T, n_t, (int)n_flat, per, p.d));
}

}  // namespace lte
