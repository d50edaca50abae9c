// The two-sided transform (Eq. 4-5 literally) with one weight scale per output channel, widths 128
// and 256, in one kernel per forward.
//
// The layer output is z = H_M (s_w s_x acc) + b with acc = q_W q_x.  The rotation of the outputs acts on
// numbers that are no longer integers times one scale, so it cannot be taken on the accumulators (as
// the fused kernel does with one scale per tensor), and an fp32 butterfly of them would cost 1e-7 per
// radian of phase.  But it is linear, and everything but q_x is known at prepare time:
//
//     z = s_x (G q_x) + b,     G = H_M diag(s_w) q_W   (real, M x K; formed in fp64)
//
// A row of G is held as 32-bit fixed point relative to its largest entry, in four signed base-256
// digits, and G q_x is four int8 products with exact int32 sums - the same product for every order of
// summation, so this kernel and the layer-by-layer one (layer_kernel) give the same bits.  What is
// lost against fp64 is 2^-32 of the row's largest entry per weight.
//
// Layout: one tile of 128 coordinates at a time, 16 epilogue warps; a token is a tensor-memory lane
// and the four threads of a row own a chunk of W/4 features each.  The outputs come in blocks of 64:
// block b holds 16 features of every chunk, so that all warps work on every block, in two halves whose sums
// (32 outputs by four digits) have a set of 128 columns each; activations wait in columns 256-511 until the
// whole row is there and the rotation of the next layer's input can run through it (stages 1, 2, 4 inside a
// block, 8 .. W/8 in a thread's chunk, W/4 and W/2 across chunks).  The weights stream from L2 in pieces of 16 KB.
//
// What bounds it: issue slots of the epilogue, about 29 per element (7 of them the phase, carried as if in
// fp64: digit_phase_pair), beside 8 x 67 cycles of MMAs per half block of 32 outputs (N = 128, all four
// digits' rows in one MMA; digit by digit with N = 64 the same outputs took 16 x 51, because operands leave shared
// memory at 128 B per cycle).  Two sets of sums: one half's MMAs run while the other's sums are read and worked on;
// the first half block's MMAs and the stages across chunks are exposed (activations fill the rest of tensor memory).
// Measured: 2 -> 256 x 5 -> 3, per-channel / per-token, 262,144 coordinates 535 us (two sets of sums and one MMA for all digits
// against one set of 4 x 64 and an MMA per digit, both with MMAs issued by one lane: 604 against 667; 9.79 ms with one dp4a
// pass and an fp64 butterfly per layer).
#include "dhq_fused.cuh"

namespace dhq {

constexpr int kDBlock = 64;          // outputs per block
constexpr int kDActCol = 256;        // first tensor-memory column of the activations
constexpr int kDThreads = 18 * 32;   // 16 epilogue warps, MMA, weight copies
constexpr int kDMaxStages = 12;

// Feature of position `i` (0..15) of thread `sub` in block b, chunks of CH = W/4 features: positions 2p and
// 2p+1 are the features p and p + CH/2 of the chunk, so that a register pair goes through the stages
// below CH/2 as one packed value.
__host__ __device__ inline int digit_feature(int W, int b, int sub, int i)
{
    const int ch = W / 4;
    return sub * ch + b * 8 + (i >> 1) + (i & 1) * (ch / 2);
}

// Place of weight digit d of output m at input k in a layer's image.  Hidden layers: [block][half][K/16][128][16], a half block's
// rows being 32 of each digit (8 per thread of a row), so that one MMA with N = 128 takes all four digits; last
// layer: [K/16][16][16], row 4 d + m.
__host__ __device__ inline size_t digit_image_offset(int W, bool last, int m, int k, int d)
{
    if (last) return (size_t)(k >> 4) * 256 + (4 * d + m) * 16 + (k & 15);
    const int ch = W / 4, sub = m / ch, q = m % ch, pos = q % (ch / 2), b = pos / 8, i = 2 * (pos % 8) + q / (ch / 2);
    return ((size_t)(b * 2 + (i >> 3)) * (W / 16) + (k >> 4)) * 2048 + (d * 32 + sub * 8 + (i & 7)) * 16 + (k & 15);
}

struct DigitLayer {
    const uint8_t *img;              // see digit_image_offset
    const float *c, *c_lo, *cb, *cb_lo, *cn; // per output: see digit_phase
    const float *act;
};
struct DigitParams {
    const float *coords;
    float *out;
    long long n, n_tiles;
    int L, d_L, n_stages;
    int skip_last_weights;           // test hook: see dhq_debug_stall_next_forward
    float qmaxf;
    float2 one2;                     // {1, 1}: see code_bits2
    double gabor_c;                  // see digit_envelope; 0 for the sine
    int *status;
    unsigned long long wait_limit_ns;
    DigitLayer layer[kMaxLayers];
    const uint32_t *l1w;             // [4 digits][M] words of four k
    const double *last_scale;        // [4]
    const float *last_bias;
};

struct DigitMap {
    uint32_t a, ring, last_w, consts, amax, w_full, w_empty, codes_full, acc_full, acc_empty, acc_last, last_full, quad_sync, drain, holder, abort_flag, total;
};
__host__ __device__ inline DigitMap digit_map(int W, int n_stages, int L)
{
    DigitMap m;
    uint32_t off = 0;
    m.a = off; off += kTile * W;
    m.ring = off; off += (uint32_t)n_stages * kDBlock * W;
    m.last_w = off; off += 16 * W;
    m.consts = off; off += (uint32_t)(5 * (L - 1) + 4) * W * 4; // per layer c | c_lo | cb | cb_lo | cn in block order; then layer 1's digits
    m.amax = off; off += 4 * kTile * 4;
    m.w_full = off; off += 8 * kDMaxStages;
    m.w_empty = off; off += 8 * kDMaxStages;
    m.codes_full = off; off += 8;
    m.acc_full = off; off += 16;
    m.acc_empty = off; off += 16;
    m.acc_last = off; off += 8;
    m.last_full = off; off += 8;
    m.quad_sync = off; off += 8 * 4;
    m.drain = off; off += 8;
    m.holder = off; off += 8;
    m.abort_flag = off; off += 16;
    m.total = off;
    return m;
}

// digit_phase of dhq_math.cuh for two outputs: the same operations, packed, and the same bits (one value at a time: width
// 256, 262,144 coordinates, 5 layers, per-channel / per-token 757 us, packed 667).
__device__ __forceinline__ f32x2 digit_phase_pair(f32x2 f0, f32x2 f1, f32x2 c_hi, f32x2 c_lo, f32x2 cb, f32x2 cb_lo, f32x2 &s, f32x2 &lo)
{
    const f32x2 two_pi = pack2(6.2831853071795865f, 6.2831853071795865f), two_pi_lo = pack2(-1.7484555e-07f, -1.7484555e-07f);
    const f32x2 grid = pack2(6144.0f, 6144.0f), magic = pack2(12582912.0f, 12582912.0f);
    const f32x2 nq = sub2(grid, fma2(f0, c_hi, grid)); // minus the product's part on the grid
    s = sub2(cb, nq);
    lo = add2(fma2(f0, c_hi, nq), fma2(f0, c_lo, fma2(f1, c_hi, cb_lo)));
    const f32x2 t = sub2(s, sub2(add2(add2(s, lo), magic), magic));
    return fma2(t, two_pi, fma2(lo, two_pi, mul2(t, two_pi_lo)));
}

// Rotated activations of this thread's quarter of the row -> codes (and, per token, their scale).
// Chunks of CH columns; the thread takes CH/4 positions of every chunk.
template <int W, bool PER_TOKEN>
__device__ __forceinline__ bool digit_finish(SlotCtx &c, float static_s, float static_inv, float &s_out)
{
    constexpr int CH = W / 4, G = CH / 4;
    uint32_t u[4][G];
    ptx::tmem_wait_st();
    ptx::tc_fence_before();
    if (!slot_barrier<true>(c)) return false;
    ptx::tc_fence_after();
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) tmem_ld<G>(c.taddr + ch * CH + c.sub * G, u[ch]);
    ptx::tmem_wait_ld();
#pragma unroll
    for (int h = 1; h < 4; h <<= 1) {
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
            if ((ch & h) == 0) {
#pragma unroll
                for (int i = 0; i < G; i += 2) {
                    f32x2 a = pack2u(u[ch][i], u[ch][i + 1]), b = pack2u(u[ch + h][i], u[ch + h][i + 1]);
                    bfly2(a, b);
                    unpack2u(a, u[ch][i], u[ch][i + 1]);
                    unpack2u(b, u[ch + h][i], u[ch + h][i + 1]);
                }
            }
        }
    }
    float inv = static_inv;
    s_out = static_s;
    if (PER_TOKEN) {
        float amax = 0.f;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
#pragma unroll
            for (int i = 0; i < G; i += 2) amax = max_abs(amax, __uint_as_float(u[ch][i]), __uint_as_float(u[ch][i + 1]));
        }
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(c.amax_addr + (c.sub * kTile + c.row) * 4), "f"(amax) : "memory");
        if (!slot_barrier<true>(c)) return false;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float o;
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(o) : "r"(c.amax_addr + (r * kTile + c.row) * 4));
            amax = fmaxf(amax, o);
        }
        scales_of(amax, c.qmaxf, s_out, inv);
    }
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) quantize_store<G, !PER_TOKEN>(c.a_tile, c.row, ch * CH + c.sub * G, u[ch], inv, c.qmaxf, c.one2);
    ptx::fence_proxy_async();
    ptx::tc_fence_before();
    ptx::mbar_arrive(c.bar_codes);
    return true;
}

template <int W, bool PER_TOKEN, bool GABOR>
__device__ void digit_epilogue(const DigitParams &p, const DigitMap &sm, uint32_t base, int warp, int lane, uint32_t tmem, volatile int *abort_flag)
{
    constexpr int CH = W / 4, NB = W / kDBlock;
    const int quad = warp & 3, sub = warp >> 2;
    SlotCtx c;
    c.row = quad * 32 + lane;
    c.sub = sub;
    c.taddr = tmem + kDActCol + ((uint32_t)(quad * 32) << 16);
    c.a_tile = base + sm.a;
    c.bar_sync = base + sm.quad_sync + 8 * quad;
    c.bar_codes = base + sm.codes_full;
    c.amax_addr = base + sm.amax;
    c.sync_parity = 0;
    c.qmaxf = p.qmaxf;
    c.one2 = pack2(p.one2.x, p.one2.y);
    c.abort_flag = abort_flag;
    c.status = p.status;
    const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + sub * 8;
    uint32_t use = 0, last_parity = 0;
    float s_x = 1.0f;

    // four outputs' sums, and constants from shared memory, -> activations
    auto activations4 = [&](const float *f0, const float *f1, uint32_t at, float *y) {
        const float4 ca = lds128(at), cl = lds128(at + W * 4), cb = lds128(at + 2 * W * 4), cbl = lds128(at + 3 * W * 4);
        float4 cn = make_float4(0.f, 0.f, 0.f, 0.f);
        if (GABOR) cn = lds128(at + 4 * W * 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            f32x2 c_hi = h ? pack2(ca.z, ca.w) : pack2(ca.x, ca.y), c_lo = h ? pack2(cl.z, cl.w) : pack2(cl.x, cl.y);
            if (PER_TOKEN) token_const2(c_hi, c_lo, pack2(s_x, s_x), pack2(-s_x, -s_x), c_hi, c_lo);
            f32x2 s, lo;
            const f32x2 x = digit_phase_pair(pack2(f0[2 * h], f0[2 * h + 1]), pack2(f1[2 * h], f1[2 * h + 1]), c_hi, c_lo,
                                             h ? pack2(cb.z, cb.w) : pack2(cb.x, cb.y), h ? pack2(cbl.z, cbl.w) : pack2(cbl.x, cbl.y), s, lo);
            unpack2(sine2(x), y[2 * h], y[2 * h + 1]);
            if constexpr (GABOR) {
                float sv[2], lv[2];
                unpack2(s, sv[0], sv[1]);
                unpack2(lo, lv[0], lv[1]);
#pragma unroll
                for (int e = 0; e < 2; ++e) y[2 * h + e] = __fmul_rn(y[2 * h + e], digit_envelope(sv[e], lv[e], h ? (e ? cn.w : cn.z) : (e ? cn.y : cn.x), p.gabor_c));
            }
        }
    };
    // stages 1, 2, 4 of 16 finished activations, and into the row's columns
    auto put_block = [&](int b, const float (&y)[16]) {
        f32x2 P[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) P[i] = pack2(y[2 * i], y[2 * i + 1]);
#pragma unroll
        for (int h = 1; h < 8; h <<= 1) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if ((i & h) == 0) bfly2(P[i], P[i + h]);
        }
        uint32_t v[16];
#pragma unroll
        for (int i = 0; i < 8; ++i) unpack2u(P[i], v[2 * i], v[2 * i + 1]);
        ptx::tmem_st16(c.taddr + sub * CH + b * 16, v);
    };
    // stages 8 .. CH/2 of the thread's own chunk, which is then in feature order
    auto chunk_stages = [&]() {
        uint32_t v[CH];
        ptx::tmem_wait_st();
        tmem_ld<CH>(c.taddr + sub * CH, v);
        ptx::tmem_wait_ld();
        f32x2 P[CH / 2];
#pragma unroll
        for (int i = 0; i < CH / 2; ++i) P[i] = pack2u(v[2 * i], v[2 * i + 1]);
#pragma unroll
        for (int h = 8; h < CH / 2; h <<= 1) {
#pragma unroll
            for (int i = 0; i < CH / 2; ++i)
                if ((i & h) == 0) bfly2(P[i], P[i + h]);
        }
#pragma unroll
        for (int i = 0; i < CH / 2; ++i) {
            float a, b;
            unpack2(P[i], a, b);
            v[i] = __float_as_uint(__fadd_rn(a, b));
            v[i + CH / 2] = __float_as_uint(__fsub_rn(a, b));
        }
        tmem_st<CH>(c.taddr + sub * CH, v);
    };

    ptx::wait_for_previous_kernels(); // coordinates and result
    for (long long tile = blockIdx.x; tile < p.n_tiles; tile += gridDim.x) {
        const long long tok = tile * kTile + c.row;
        const bool valid = tok < p.n;
        float x = 0.f, yc = 0.f;
        if (valid) { const float2 xy = load_coords(p.coords, tok); x = xy.x; yc = xy.y; }
        // layer 1: the rotated padded coordinate is [x+y, x-y, x+y, x-y]
        const float e0 = __fadd_rn(__fadd_rn(x, yc), 0.f), e1 = __fadd_rn(__fsub_rn(x, yc), 0.f);
        float inv_x;
        if (PER_TOKEN) {
            scales_of(fmaxf(fabsf(e0), fabsf(e1)), p.qmaxf, s_x, inv_x);
        } else {
            s_x = 1.0f; // the constants hold it
            inv_x = __ldg(p.layer[0].act + 2);
        }
        const uint32_t b0 = code_bits<true>(e0, inv_x, p.qmaxf), b1 = code_bits<true>(e1, inv_x, p.qmaxf);
        const int qx = (int)pack4(b0, b1, b0, b1);
        for (int l = 1; l < p.L; ++l) {
            const uint32_t cbase = base + sm.consts + (uint32_t)((l - 1) * 5 * W * 4);
            float static_inv = 0.f;
            if (!PER_TOKEN) static_inv = __ldg(p.layer[l].act + 2);
#pragma unroll 1
            for (int b = 0; b < NB; ++b) {
                const uint32_t at = cbase + (uint32_t)(b * kDBlock + sub * 16) * 4;
                float f0[16], f1[16];
                if (l == 1) {
                    const uint32_t dg = base + sm.consts + (uint32_t)((5 * (p.L - 1) * W + b * kDBlock + sub * 16) * 4);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 w0 = lds128(dg + q * 16), w1 = lds128(dg + W * 4 + q * 16), w2 = lds128(dg + 2 * W * 4 + q * 16), w3 = lds128(dg + 3 * W * 4 + q * 16);
                        const float wv[4][4] = {{w0.x, w0.y, w0.z, w0.w}, {w1.x, w1.y, w1.z, w1.w}, {w2.x, w2.y, w2.z, w2.w}, {w3.x, w3.y, w3.z, w3.w}};
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            digit_sums(__dp4a(qx, (int)__float_as_uint(wv[0][e]), 0), __dp4a(qx, (int)__float_as_uint(wv[1][e]), 0),
                                       __dp4a(qx, (int)__float_as_uint(wv[2][e]), 0), __dp4a(qx, (int)__float_as_uint(wv[3][e]), 0), f0[4 * q + e], f1[4 * q + e]);
                    }
                } else {
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        if (!wait_bar_warp<true>(base + sm.acc_full + 8 * hf, use & 1, abort_flag, p.status)) return;
                        ptx::tc_fence_after();
                        uint32_t D[4][8];
#pragma unroll
                        for (int d = 0; d < 4; ++d) ptx::tmem_ld8(acc + hf * 128 + d * 32, D[d]);
                        ptx::tmem_wait_ld();
                        ptx::tc_fence_before();
                        ptx::mbar_arrive(base + sm.acc_empty + 8 * hf); // the sums are free for the next block
#pragma unroll
                        for (int i = 0; i < 8; ++i) digit_sums((int)D[0][i], (int)D[1][i], (int)D[2][i], (int)D[3][i], f0[hf * 8 + i], f1[hf * 8 + i]);
                    }
                    ++use;
                }
                float y[16];
#pragma unroll
                for (int q = 0; q < 4; ++q) activations4(f0 + 4 * q, f1 + 4 * q, at + q * 16, y + 4 * q);
                put_block(b, y);
            }
            chunk_stages();
            if (!digit_finish<W, PER_TOKEN>(c, 1.0f, static_inv, s_x)) return;
        }
        // last layer: the sums of digit d of output m in column 4 d + m
        if (!wait_bar_warp<true>(base + sm.acc_last, last_parity, abort_flag, p.status)) return;
        last_parity ^= 1;
        ptx::tc_fence_after();
        if (sub == 0) {
            uint32_t u[16];
            ptx::tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16), u);
            ptx::tmem_wait_ld();
            if (valid) {
                const double st = PER_TOKEN ? (double)s_x : (double)__ldg(p.layer[p.L - 1].act + 1);
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    if (m < p.d_L) p.out[tok * p.d_L + m] = digit_last((int)u[m], (int)u[4 + m], (int)u[8 + m], (int)u[12 + m], __ldg(p.last_scale + m), st, __ldg(p.last_bias + m));
            }
        }
        ptx::tc_fence_before();
    }
}

template <int W>
__device__ void digit_mma(const DigitParams &p, const DigitMap &sm, uint32_t base, uint32_t tmem, volatile int *abort_flag)
{
    constexpr int NB = W / kDBlock, PIECE = kDBlock * W;
    ptx::wait_for_previous_kernels(); // before the first bounded wait
    const uint32_t idesc = ptx::idesc_i8(kTile, 128), idesc_last = ptx::idesc_i8(kTile, 16);
    constexpr uint32_t kDescHi = (128u >> 4) | (1u << 14);
    const uint32_t a0 = ((base + sm.a) >> 4) | ((kTile * 16u >> 4) << 16), b0 = ((base + sm.ring) >> 4) | ((128 * 16u >> 4) << 16);
    const uint32_t l0 = ((base + sm.last_w) >> 4) | ((16u * 16u >> 4) << 16);
    uint32_t use = 0, codes = 0, wpar = 0;
    int stage = 0;
    bool ok = true;
    for (long long tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x) {
        for (int l = 2; l < p.L && ok; ++l) {
            ok = wait_bar_warp<true>(base + sm.codes_full, codes & 1, abort_flag, p.status);
            ++codes;
            for (int hb = 0; hb < 2 * NB && ok; ++hb, ++use) { // half blocks; set hb & 1 of the sums
                const uint32_t set = hb & 1;
                if (!wait_bar_warp<true>(base + sm.acc_empty + 8 * set, ((use >> 1) & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
                ptx::tc_fence_after();
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    if (!wait_bar_warp<true>(base + sm.w_full + 8 * stage, wpar, abort_flag, p.status)) { ok = false; break; }
                    const uint32_t bk = b0 + (uint32_t)stage * (PIECE >> 4);
#pragma unroll
                    for (int ks = 0; ks < W / 64; ++ks)
                        ptx::mma_i8_words(tmem + set * 128, a0 + ((q * (W / 64) + ks) * 2 * kTile * 16 >> 4), bk + (ks * 2 * 128 * 16 >> 4), kDescHi, idesc, q > 0 || ks > 0 ? 1u : 0u);
                    ptx::mma_commit(base + sm.w_empty + 8 * stage);
                    if (++stage == p.n_stages) { stage = 0; wpar ^= 1; }
                }
                if (ok) ptx::mma_commit(base + sm.acc_full + 8 * set);
            }
        }
        if (!ok) break;
        if (!wait_bar_warp<true>(base + sm.last_full, 0, abort_flag, p.status) ||
            !wait_bar_warp<true>(base + sm.codes_full, codes & 1, abort_flag, p.status)) { ok = false; break; }
        ++codes;
        ptx::tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < W / 32; ++ks)
            ptx::mma_i8_words(tmem, a0 + (ks * 2 * kTile * 16 >> 4), l0 + (ks * 2 * 16 * 16 >> 4), kDescHi, idesc_last, ks > 0 ? 1u : 0u);
        ptx::mma_commit(base + sm.acc_last);
    }
    if (!ok) { // give the MMAs already issued a bounded time to finish before tensor memory is released
        ptx::mma_commit(base + sm.drain);
        const unsigned long long t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(base + sm.drain, 0) && ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
    }
}

template <int W>
__device__ void digit_load(const DigitParams &p, const DigitMap &sm, uint32_t base, volatile int *abort_flag)
{
    constexpr int PIECE = kDBlock * W, PIECES = W / kDBlock * 4;
    if (!p.skip_last_weights) {
        ptx::mbar_expect_tx_warp(base + sm.last_full, 16 * W);
        ptx::bulk_g2s_warp(base + sm.last_w, p.layer[p.L - 1].img, 16 * W, base + sm.last_full);
    }
    int stage = 0;
    uint32_t par = 1, issued = 0;
    bool ok = true;
    for (long long tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x) {
        for (int l = 2; l < p.L && ok; ++l) {
            for (int i = 0; i < PIECES; ++i) {
                if (issued == (uint32_t)p.n_stages) ptx::wait_for_previous_kernels();
                if (!wait_bar_warp<true>(base + sm.w_empty + 8 * stage, par, abort_flag, p.status)) { ok = false; break; }
                ptx::mbar_expect_tx_warp(base + sm.w_full + 8 * stage, PIECE);
                ptx::bulk_g2s_warp(base + sm.ring + (uint32_t)stage * PIECE, p.layer[l - 1].img + (size_t)i * PIECE, PIECE, base + sm.w_full + 8 * stage);
                ++issued;
                if (++stage == p.n_stages) { stage = 0; par ^= 1; }
            }
        }
    }
    if (!ok || *abort_flag) { // let copies in flight land before the CTA may exit
        const unsigned long long t0 = ptx::globaltimer();
        const uint32_t n = (uint32_t)p.n_stages;
        for (uint32_t i = issued > n ? issued - n : 0; i < issued; ++i)
            while (!ptx::mbar_try_wait(base + sm.w_full + 8 * (i % n), (i / n) & 1) && ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
        while (!p.skip_last_weights && !ptx::mbar_try_wait(base + sm.last_full, 0) && ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
    }
}

template <int W, bool PER_TOKEN, bool GABOR>
__global__ void __launch_bounds__(kDThreads, 1) digit_kernel(const __grid_constant__ DigitParams p)
{
    constexpr int NB = W / kDBlock;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - raw);
    const DigitMap sm = digit_map(W, p.n_stages, p.L);
    const int warp = ptx::uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gen + sm.abort_flag);
    ptx::launch_dependents();
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        *reinterpret_cast<volatile unsigned long long *>(abort_flag + 2) = p.wait_limit_ns;
        for (int i = 0; i < kDMaxStages; ++i) {
            ptx::mbar_init(base + sm.w_full + 8 * i, 1);
            ptx::mbar_init(base + sm.w_empty + 8 * i, 1);
        }
        ptx::mbar_init(base + sm.codes_full, kEpiWarps * 32);
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(base + sm.acc_full + 8 * i, 1);
            ptx::mbar_init(base + sm.acc_empty + 8 * i, kEpiWarps * 32);
        }
        ptx::mbar_init(base + sm.acc_last, 1);
        ptx::mbar_init(base + sm.last_full, 1);
        for (int i = 0; i < 4; ++i) ptx::mbar_init(base + sm.quad_sync + 8 * i, 128);
        ptx::mbar_init(base + sm.drain, 1);
        ptx::fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        ptx::tmem_alloc(base + sm.holder, 512);
        ptx::tmem_relinquish();
    }
    float *consts = reinterpret_cast<float *>(gen + sm.consts);
    for (int i = threadIdx.x; i < W; i += kDThreads) { // i: position in block order, m: its feature
        const int b = i / kDBlock, m = digit_feature(W, b, (i % kDBlock) >> 4, i & 15);
        for (int l = 0; l < p.L - 1; ++l) {
            float *d = consts + l * 5 * W + i;
            d[0] = __ldg(p.layer[l].c + m);
            d[W] = __ldg(p.layer[l].c_lo + m);
            d[2 * W] = __ldg(p.layer[l].cb + m);
            d[3 * W] = __ldg(p.layer[l].cb_lo + m);
            d[4 * W] = __ldg(p.layer[l].cn + m);
        }
        for (int d = 0; d < 4; ++d) reinterpret_cast<uint32_t *>(consts)[(5 * (p.L - 1) + d) * W + i] = __ldg(p.l1w + d * W + m);
    }
    static_assert(NB * kDBlock == W, "whole blocks");
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ptx::uniform(*reinterpret_cast<volatile uint32_t *>(gen + sm.holder));
    if (warp < kEpiWarps) digit_epilogue<W, PER_TOKEN, GABOR>(p, sm, base, warp, lane, tmem, abort_flag);
    else if (warp == kMmaWarp) digit_mma<W>(p, sm, base, tmem, abort_flag);
    else digit_load<W>(p, sm, base, abort_flag);
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        ptx::tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------- weight side, once per network

// G = H_M diag(s_w) q_W, one block per column k of a layer, in fp64 (a 24-bit scale times a 7-bit code,
// sums of up to 256 of them: exact but for rows whose scales lie more than 2^14 apart).
__global__ void prep_digit_cols_kernel(const __grid_constant__ DigitPrep a)
{
    extern __shared__ double gcol[];
    const int l = (int)blockIdx.x < 4 ? 0 : 1 + ((int)blockIdx.x - 4) / a.w; // 4 columns, then w per layer
    const int k = l == 0 ? (int)blockIdx.x : ((int)blockIdx.x - 4) % a.w;
    const LayerDev &dev = a.dev[l];
    const int K = dev.K, M = dev.M;
    for (int m = threadIdx.x; m < M; m += blockDim.x) gcol[m] = (double)dev.s_w[m] * (double)dev.qw[(size_t)m * K + k];
    for (int h = 1; h < M; h <<= 1) {
        __syncthreads();
        for (int p = threadIdx.x; p < M / 2; p += blockDim.x) {
            const int i = ((p & ~(h - 1)) << 1) | (p & (h - 1));
            const double x = gcol[i], y = gcol[i + h];
            gcol[i] = x + y;
            gcol[i + h] = x - y;
        }
    }
    __syncthreads();
    for (int m = threadIdx.x; m < M; m += blockDim.x) a.g[l][(size_t)m * K + k] = gcol[m];
}

// One block per row: 32-bit fixed point relative to the largest entry, four signed base-256 digits in both
// layouts, and the row's scale (per unit of the integer; hidden layers in turns of the phase, times
// 2^24 because the first digit's sum is the unit there).
__global__ void __launch_bounds__(128) prep_digit_rows_kernel(const __grid_constant__ DigitPrep a)
{
    __shared__ double red[4];
    const int l = min((int)blockIdx.x / a.w, a.L - 1), m = (int)blockIdx.x - l * a.w, tid = threadIdx.x;
    const LayerDev &dev = a.dev[l];
    const int K = dev.K, M = dev.M;
    const double *row = a.g[l] + (size_t)m * K;
    double g = 0.0;
    for (int k = tid; k < K; k += 128) g = fmax(g, fabs(row[k]));
    for (int o = 16; o; o >>= 1) g = fmax(g, __shfl_xor_sync(0xffffffffu, g, o));
    if ((tid & 31) == 0) red[tid >> 5] = g;
    __syncthreads();
    g = fmax(fmax(red[0], red[1]), fmax(red[2], red[3]));
    const double f = g > 0.0 ? 2139062143.0 / g : 0.0; // 127 in every digit
    for (int k = tid; k < K; k += 128) {
        const uint32_t v = (uint32_t)((long long)rint(row[k] * f) + 0x80808080ll) ^ 0x80808080u;
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const uint8_t byte = (uint8_t)(v >> (24 - 8 * d));
            reinterpret_cast<uint8_t *>(dev.gd_k4m)[(size_t)d * M * K + ((size_t)(k >> 2) * M + m) * 4 + (k & 3)] = byte;
            if (l > 0) dev.gd_img[digit_image_offset(a.w, l == a.L - 1, m, k, d)] = byte;
        }
    }
    if (tid == 0) {
        const bool sine = l < a.L - 1;
        dev.g_scale[m] = f > 0.0 ? (sine ? a.omega0 * 0.15915494309189533576888 * 16777216.0 : 1.0) / f : 0.0;
        if (a.finalize) finalize_row(dev, m, 1.0f, 0.f, sine, a.omega0);
    }
}

// The image again from the digits in [4][K/4][M] words: a block saved by an earlier build holds it in another order.
__global__ void __launch_bounds__(256) repack_digits_kernel(LayerDev dev, int w, int last)
{
    const int K = dev.K, M = dev.M, words = M * K; // four digits of M K / 4 words
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= words) return;
    const int d = i / (words / 4), r = i % (words / 4), k = r / M * 4, m = r % M;
    *reinterpret_cast<uint32_t *>(dev.gd_img + digit_image_offset(w, last != 0, m, k, d)) = dev.gd_k4m[i];
}
cudaError_t launch_repack_digits(const LayerDev &dev, int w, bool last, cudaStream_t st, int64_t *launches)
{
    repack_digits_kernel<<<(dev.M * dev.K + 255) / 256, 256, 0, st>>>(dev, w, last ? 1 : 0);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_prep_digits(const DigitPrep &a, cudaStream_t st, int64_t *launches)
{
    prep_digit_cols_kernel<<<4 + (a.L - 1) * a.w, 128, a.w * sizeof(double), st>>>(a);
    prep_digit_rows_kernel<<<(a.L - 1) * a.w + 4, 128, 0, st>>>(a);
    *launches += 2;
    return cudaGetLastError();
}

// ------------------------------------------------------------------- host side

struct DigitState {
    DigitParams p;
    size_t smem_bytes;
    int sm_count;
};

typedef void (*digit_fn)(const DigitParams);
template <int W> static digit_fn pick_digit(bool per_token, bool gabor)
{
    if (gabor) return per_token ? digit_kernel<W, true, true> : digit_kernel<W, false, true>;
    return per_token ? digit_kernel<W, true, false> : digit_kernel<W, false, false>;
}
static digit_fn digit_kernel_of(const dhq_handle_s *h)
{
    const bool per_token = h->cfg.a_gran == DHQ_GRAN_CHANNEL_OR_TOKEN, gabor = h->gabor_s0 > 0.0;
    return h->w == 256 ? pick_digit<256>(per_token, gabor) : h->w == 128 ? pick_digit<128>(per_token, gabor) : nullptr;
}

dhq_status_t digit_create(dhq_handle_s *h)
{
    DigitState *ds = new (std::nothrow) DigitState();
    if (!ds) return DHQ_ERR_ALLOC;
    memset(ds, 0, sizeof(*ds));
    h->digit_state = ds;
    int max_optin = 0;
    if (cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&ds->sm_count, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess)
        return DHQ_ERR_CUDA;
    DigitParams &p = ds->p;
    p.L = h->L; p.d_L = h->d_L;
    p.qmaxf = (float)((1 << (h->cfg.a_bits - 1)) - 1);
    p.one2 = make_float2(1.0f, 1.0f);
    p.gabor_c = digit_gabor_c(h->gabor_s0, (double)h->cfg.omega0);
    p.status = h->d_status;
    for (int l = 0; l < h->L; ++l) {
        const LayerDev &d = h->layer[l];
        p.layer[l].img = d.gd_img;
        p.layer[l].c = d.cA; p.layer[l].c_lo = d.cA_lo; p.layer[l].cb = d.cB; p.layer[l].cb_lo = d.cB_lo; p.layer[l].cn = d.cN;
        p.layer[l].act = d.act;
    }
    p.l1w = reinterpret_cast<const uint32_t *>(h->layer[0].gd_k4m);
    p.last_scale = h->layer[h->L - 1].g_scale;
    p.last_bias = h->layer[h->L - 1].bias;
    const size_t piece = (size_t)kDBlock * h->w, fixed = digit_map(h->w, 0, h->L).total + 1024;
    if (fixed + piece > (size_t)max_optin) return DHQ_ERR_UNSUPPORTED;
    int stages = (int)(((size_t)max_optin - fixed) / piece);
    p.n_stages = stages < kDMaxStages ? stages : kDMaxStages;
    ds->smem_bytes = digit_map(h->w, p.n_stages, h->L).total + 1024;
    if (ds->smem_bytes < (size_t)kMinSmem) ds->smem_bytes = kMinSmem;
    return allow_smem((const void *)digit_kernel_of(h), h->device, max_optin) ? DHQ_OK : DHQ_ERR_CUDA;
}

void digit_destroy(dhq_handle_s *h)
{
    delete static_cast<DigitState *>(h->digit_state);
    h->digit_state = nullptr;
}

dhq_status_t digit_forward(dhq_handle_s *h, const float *coords, int64_t n, float *out, cudaStream_t st)
{
    DigitState *ds = static_cast<DigitState *>(h->digit_state);
    DigitParams p = ds->p;
    p.coords = coords; p.out = out; p.n = n;
    p.n_tiles = (n + kTile - 1) / kTile;
    p.wait_limit_ns = h->wait_limit_ns;
    if (h->stall_next_forward) { // test hook, one launch only
        p.skip_last_weights = 1;
        h->stall_next_forward = false;
    }
    const int grid = (int)(p.n_tiles < ds->sm_count ? p.n_tiles : ds->sm_count);
    const cudaError_t e = launch_after(h, (const void *)digit_kernel_of(h), grid, kDThreads, ds->smem_bytes, st, &p);
    h->launches++;
    return e == cudaSuccess ? DHQ_OK : DHQ_ERR_CUDA;
}

} // namespace dhq
