// The two comparison datapaths of the paper's hardware table (Table 2) and motivation figure
// (Section I): W8A32 - weights folded and quantized exactly as for DHQ, activations kept in fp32 -
// and W32A32 - the plain fp32 sinusoidal network.
//
//   W8A32:  z = s_w[m] * sum_k q_w[m][k] (H_K x)_k + b[m]  =  s_w[m] * sum_j (q_w H_K)[m][j] x_j + b[m]
//   W32A32: z = sum_k W[m][k] x_k + b[m]
//   y = sin(omega0 z) for hidden layers, z for the last layer.
//
// q_w H_K is an integer matrix (|.| <= 127 K) formed once at prepare time, so both datapaths are the
// same computation: a real matrix times activations that lie in [-1, 1].
//
// One persistent kernel, tiles of 128 coordinates, all layers of a tile one after the other.  The
// hidden layers run on the int8 tensor cores in fixed point: an activation is a 24-bit integer held
// as three signed base-256 digits X_0 X_1 X_2, a weight row has a scale of its own and two or three
// digits W_0 W_1 (W_2); digit products of equal weight 256^-(i+j) share one int32 accumulator, which
// is exact, and the three accumulators of an output meet in fp32 in the epilogue.  Products with
// i + j > 2 are left out (they are below 2^-23 of the largest product).  The error of an output is
// that of rounding x and W to 24 bits of their range, which does not grow along the sum the way a
// chain of K fp32 additions does, and the phase is reduced modulo one turn before it is rounded.  Networks whose
// activations or weights use little of that range go to dhq_float_layers.cu (fixed_point_serves).
//
// What bounds it.  The digits of a tile of 128 activations stay in shared memory for a whole layer
// (128 KB and a quarter of tensor memory at width 512; below that from layer to layer), the weights stream past them from L2.  An MMA takes
// 67 cycles at N = 128 and 51 at N = 64 (operands leave shared memory at 128 B per cycle), hence blocks of 128 outputs
// and a single set of 3 x 128 accumulator columns: the epilogue releases it as soon as the phases
// are in registers and computes sines and digits beside the next block's MMAs.  The sines
// and digits of a block take as long as the next block's MMAs or longer.
// Measured: 2 -> 256 x 3 -> 3, fp32, 65,536 coordinates 940 -> 65 us (88 with the digits through L2); 2 -> 512 x 4 -> 3, 8-bit
// weights, 262,144 coordinates 17.2 -> 0.94 ms (one fp32 CUDA-core pass per layer before).  Blocks of 64 outputs with the weight
// digits stacked in one operand and two sets of accumulators were slower (70.6 against 67.9 us, 1.16 against 1.10 ms, both
// before the warp's number was a uniform value): fewer outputs at a time hide less of the epilogue's latency.
#include "dhq_fused.cuh"

namespace dhq {

__host__ __device__ constexpr int float_block(int W) { return W < 128 ? W : 128; } // outputs per accumulator set, three times as many columns
__host__ __device__ constexpr int float_kc(int W) { return W == 256 || W == 128 ? 128 : 64; }   // k per weight piece (4 to 16 KB)
constexpr int kFPartCol = 3 * 128;           // first tensor-memory column of the last layer's partial sums: two sets of 16 columns
constexpr int kFLoaders = 2;                 // warps that copy weights, see float_load_weights
constexpr int kFThreads = (18 + kFLoaders) * 32; // 16 epilogue warps, MMA, weight copies, activation copies
constexpr int kFMaxStages = 16;
constexpr float kFXScale = 8355711.0f;       // 127 * (65536 + 256 + 1): the largest three-digit integer

struct FloatParams {
    const float *coords;
    float *out;
    long long n, n_tiles;
    int L, d_L, n_stages;
    int skip_first_weights;                  // test hook: see dhq_debug_stall_next_forward
    int *status;
    unsigned long long wait_limit_ns;
    uint8_t *x;                              // [gridDim.x][3][W/16][128][16]: the digits of a tile's activations
    const uint8_t *wimg[kMaxLayers];         // hidden layers: weight digits, see float_image_offset
    const float *c0[kMaxLayers], *c0_lo[kMaxLayers], *cb[kMaxLayers];
    const float4 *l1;                        // first layer: per output the two weights and the bias in turns of the phase
    const float4 *wl;                        // fp32 weights of the last layer, [K/4][4]
    const float *sl, *bl;
    float *dX[kMaxLayers], *dY[kMaxLayers];  // dumps (DUMP instantiation)
};

// Below width 512 the activations' digits never leave shared memory.  The operand area is cut into parts of KC
// features (the outputs of one block), one more than a layer has: part k of the t-th tensor-core layer of the
// CTA lies in buffer (t NB + k) mod (NB + 1).  Block 0's outputs go to the buffer that this layer does not
// read, block 1's (the last) to the one of this layer's part 0, whose MMAs have all completed with that block's
// sums.  So the next layer's MMAs begin on part 0 while block 1's outputs are still being formed.  At width 512 one layer's
// digits take 128 KB of shared memory and 128 tensor-memory columns, which leaves no room beside them: they go through L2.
__host__ __device__ constexpr bool float_x_in_smem(int W) { return W < 512; }
// Width 512: the third digit, which meets the first weight digit only, is an operand in tensor memory (columns 384-511,
// four consecutive k to a column) instead of shared memory.  That leaves room for the epilogue constants, which were read
// through an L1 cache of a few KB, and for seven weight pieces in flight instead of four: 262,144 coordinates, 5 layers, 8-bit
// weights 1,011 -> 940 us (the third digit alone, without the constants: no gain).
constexpr int kFX2Col = 3 * 128;
__host__ __device__ constexpr int float_smem_digits(int W) { return W == 512 ? 2 : 3; }
__host__ __device__ constexpr uint32_t float_part_bytes(int W) { return 3u * kTile * (W < 128 ? W : 128); }

// At width 512 there is room for the first layer's epilogue constants and those of two hidden layers: a layer's three arrays
// are brought by bulk copies while the layer before is worked on.
__host__ __device__ constexpr bool float_consts_resident(int W) { return W < 512; }
__host__ __device__ constexpr int float_areas(int W) { return W <= 128 ? 4 : 3; } // per hidden layer, see digit_phase2

struct FloatMap {
    uint32_t a, ring, consts, part, w_full, w_empty, a_full, x_ready, x2_ready, c_full, acc_full, acc_empty, quad_sync, drain, holder, abort_flag, total;
};
__host__ __device__ inline FloatMap float_map(int W, int n_stages, int L)
{
    FloatMap m;
    uint32_t off = 0;
    m.a = off; off += float_x_in_smem(W) ? (uint32_t)(W / float_block(W) + 1) * float_part_bytes(W) : (uint32_t)float_smem_digits(W) * kTile * W;
    m.ring = off; off += (uint32_t)n_stages * float_block(W) * float_kc(W);
    m.consts = off; off += (uint32_t)(4 + float_areas(W) * (float_consts_resident(W) ? L - 2 : 2)) * W * 4; // first layer, then c0 | c0_lo | cb (| cb_lo) per hidden layer
    m.part = off; off += float_x_in_smem(W) ? 0 : 2 * 4 * kTile * 16; // width 512: the last layer's partial sums
    m.w_full = off; off += 8 * kFMaxStages;
    m.w_empty = off; off += 8 * kFMaxStages;
    m.a_full = off; off += 8 * 8;
    m.x_ready = off; off += 8;
    m.x2_ready = off; off += 8;
    m.c_full = off; off += 8 * 2;
    m.acc_full = off; off += 8;
    m.acc_empty = off; off += 8;
    m.quad_sync = off; off += 8 * 4;
    m.drain = off; off += 8;
    m.holder = off; off += 8;
    m.abort_flag = off; off += 16;
    m.total = off;
    return m;
}

// Sixteen activations of one token, consecutive features starting at a multiple of 16, as base-256
// digits: I = rint(y * 8355711) = 65536 X_0 + 256 X_1 + X_2 with digits in [-128, 127].  Adding
// 0x808080 makes the digits' carries ordinary ones, and flipping each byte's top bit takes the
// offset of 128 out again.
struct Digits16 { uint32_t w[3][4]; };
__device__ __forceinline__ void digits4(const float (&y)[4], int j, Digits16 &d)
{
    uint32_t v[4];
    float t[4];
    unpack2(mul2(pack2(y[0], y[1]), pack2(kFXScale, kFXScale)), t[0], t[1]);
    unpack2(mul2(pack2(y[2], y[3]), pack2(kFXScale, kFXScale)), t[2], t[3]);
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = (uint32_t)(min(__float2int_rn(t[e]), 8355711) + 0x808080); // sin.approx may pass 1 by an ulp
    const uint32_t a = __byte_perm(v[0], v[1], 0x5140), b = __byte_perm(v[2], v[3], 0x5140);
    const uint32_t c = __byte_perm(v[0], v[1], 0x0062), e = __byte_perm(v[2], v[3], 0x0062);
    d.w[0][j] = __byte_perm(c, e, 0x5410) ^ 0x80808080u;
    d.w[1][j] = __byte_perm(a, b, 0x7632) ^ 0x80808080u;
    d.w[2][j] = __byte_perm(a, b, 0x5410) ^ 0x80808080u;
}

// The phases of two hidden outputs in radians, less whole turns: 2 pi (c0 (D0 + D1 / 256 + D2 / 65536) + cb) with
// c0 = fl32 value plus remainder c0_lo, cb = omega0 b / (2 pi) modulo 1.  The integer is taken off inside an fma, before
// anything is rounded, so that the error does not grow with the phase, and it is the one nearest to the whole phase: the
// hardware sine rounds its argument twice as coarsely beyond pi.  Up to width 128, where the fp32 sums of few
// products are themselves exact to 1.5e-7, the phase is rounded only once, as digit_phase of dhq_math.cuh does it (cb is
// the part on its 2^-11 grid, cb_lo the rest).
// Error of the hidden outputs of the second layer against fp64, rms relative to theirs, default initialisation, widths 64 and 256:
// with fp32 multiply-adds 2.1e-7 and 3.3e-7; here 1.9e-7 and 2.0e-7.
__host__ __device__ constexpr bool float_rounds_once(int W) { return W <= 128; }
template <int W>
__device__ __forceinline__ f32x2 digit_phase2(const uint32_t *D0, const uint32_t *D1, const uint32_t *D2, f32x2 c0, f32x2 c0_lo, f32x2 cb, f32x2 cb_lo)
{
    const f32x2 magic = pack2(12582912.0f, 12582912.0f), two_pi = pack2(6.2831853071795865f, 6.2831853071795865f);
    const f32x2 f0 = pack2((float)(int)D0[0], (float)(int)D0[1]); // |D0| < 2^24: exact
    // (D1 < 2^24 at width 512: 256 times that and D2 are still an int32 at width 256)
    constexpr int S = W == 512 ? 1 : 0;
    const f32x2 f1 = mul2(pack2((float)((int)D1[0] * (256 >> S) + ((int)D2[0] >> S)), (float)((int)D1[1] * (256 >> S) + ((int)D2[1] >> S))),
                          pack2(S ? 0x1p-15f : 0x1p-16f, S ? 0x1p-15f : 0x1p-16f));
    if constexpr (float_rounds_once(W)) {
        const f32x2 grid = pack2(6144.0f, 6144.0f), two_pi_lo = pack2(-1.7484555e-07f, -1.7484555e-07f);
        const f32x2 nq = sub2(grid, fma2(f0, c0, grid)), s = sub2(cb, nq); // minus the product's part on the grid
        const f32x2 lo = add2(fma2(f0, c0, nq), fma2(f0, c0_lo, fma2(f1, c0, cb_lo)));
        const f32x2 t = sub2(s, sub2(add2(add2(s, lo), magic), magic));
        return fma2(t, two_pi, fma2(lo, two_pi, mul2(t, two_pi_lo)));
    } else {
        const f32x2 w = fma2(f0, c0_lo, fma2(f1, c0, cb));
        const f32x2 k = sub2(magic, add2(fma2(f0, c0, w), magic)); // minus the nearest integer
        return mul2(add2(fma2(f0, c0, k), w), two_pi);
    }
}
__device__ __forceinline__ float sine_of_turns(float r) { return sin_approx(__fmul_rn(r, 6.2831853071795865f)); }

template <int W, int WL, bool DUMP>
__device__ void float_epilogue(const FloatParams &p, const FloatMap &sm, uint32_t base, int warp, int lane, uint32_t tmem,
                               volatile int *abort_flag)
{
    constexpr int FB = float_block(W), NB = W / FB, GPB = FB / 64; // GPB groups of 16 outputs per thread and block
    constexpr bool XS = float_x_in_smem(W);
    uint32_t tlayer = 0, x_addr = 0; // tensor-core layers so far; where the block's digits go (XS)
    const int quad = warp & 3, sub = warp >> 2, row = quad * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16);
    uint8_t *xrow = p.x + (size_t)blockIdx.x * (3 * kTile * W) + row * 16;
    uint32_t use = 0, qpar = 0;
    float part[4];
    // what happens to 16 finished activations: features k0 .. k0+15 of layer l (1-based)
    auto emit = [&](int l, int k0, const float (&y)[16], long long tok, bool valid) {
        if constexpr (DUMP) {
            if (valid) {
                // (one float at a time: the caller's buffers are 4-byte aligned and no more)
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (p.dY[l - 1]) p.dY[l - 1][tok * W + k0 + j] = y[j];
                    if (p.dX[l]) p.dX[l][tok * W + k0 + j] = y[j];
                }
            }
        }
        if (l < p.L - 1) {
            Digits16 d;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float v[4] = {y[4 * j], y[4 * j + 1], y[4 * j + 2], y[4 * j + 3]};
                digits4(v, j, d);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if constexpr (XS)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(x_addr + (uint32_t)(i * kTile * FB + (k0 % FB) * kTile + row * 16)),
                                 "r"(d.w[i][0]), "r"(d.w[i][1]), "r"(d.w[i][2]), "r"(d.w[i][3]) : "memory");
                else *reinterpret_cast<uint4 *>(xrow + i * (kTile * W) + (k0 / 16) * (kTile * 16)) = make_uint4(d.w[i][0], d.w[i][1], d.w[i][2], d.w[i][3]);
            }
        } else {
            // last layer (at most four outputs): fp32 multiply-adds here, this thread's share of the K products
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                if (m >= p.d_L) break;
                float s = part[m];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 w = __ldg(p.wl + (k0 / 4 + j) * 4 + m);
                    s = __fmaf_rn(w.w, y[4 * j + 3], __fmaf_rn(w.z, y[4 * j + 2], __fmaf_rn(w.y, y[4 * j + 1], __fmaf_rn(w.x, y[4 * j], s))));
                }
                part[m] = s;
            }
        }
    };
    auto coords_of = [&](long long tile, float &x, float &yc) {
        const long long tok = tile * kTile + row;
        x = yc = 0.f;
        if (tile < p.n_tiles && tok < p.n) { x = p.coords[2 * tok]; yc = p.coords[2 * tok + 1]; } // plain loads: see load_coords (dhq_forward_debug takes any 4-byte aligned coords)
    };
    // block b of the outputs is about to be formed / is complete: the inputs of tensor-core layer t
    auto begin_part = [&](uint32_t t, int b) {
        if constexpr (XS) x_addr = base + sm.a + (t * NB + b) % (NB + 1) * float_part_bytes(W);
    };
    auto end_part = [&](int b) {
        if constexpr (XS) {
            ptx::fence_proxy_async();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(base + sm.a_full + 8 * b);
        }
    };
    // layer 1, two products per output: block b of a tile
    auto first_layer = [&](int b, float x, float yc, long long tok, bool valid) {
#pragma unroll
        for (int g = 0; g < GPB; ++g) {
            const int k0 = b * FB + (sub * GPB + g) * 16;
            float y[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float4 w = lds128(base + sm.consts + (k0 + j) * 16);
                const float t = __fmaf_rn(x, w.x, __fmaf_rn(yc, w.y, w.z));
                y[j] = sine_of_turns(__fsub_rn(t, __fsub_rn(__fadd_rn(t, 12582912.0f), 12582912.0f)));
            }
            emit(1, k0, y, tok, valid);
        }
    };
    float x, yc;
    ptx::wait_for_previous_kernels(); // coordinates, result and the scratch activations
    coords_of(blockIdx.x, x, yc);
    for (long long tile = blockIdx.x; tile < p.n_tiles; tile += gridDim.x) {
        const long long tok = tile * kTile + row;
        const bool valid = tok < p.n;
        if constexpr (DUMP) {
            if (valid && sub == 0 && p.dX[0]) {
                float *q = p.dX[0] + tok * 4;
                q[0] = x; q[1] = yc; q[2] = 0.f; q[3] = 0.f;
            }
        }
        // (NaN where a coordinate is not finite: digits cannot carry it to the result)
        const float zero = __fadd_rn(fabsf(__fmul_rn(x, 0.f)), fabsf(__fmul_rn(yc, 0.f)));
#pragma unroll
        for (int m = 0; m < 4; ++m) part[m] = zero;
        // (with hidden layers, the first layer of every tile but the first was done beside the tile before)
        if (tile == blockIdx.x || p.L == 2) {
#pragma unroll 1
            for (int b = 0; b < NB; ++b) {
                begin_part(tlayer, b);
                first_layer(b, x, yc, tok, valid);
                if (p.L > 2) end_part(b);
            }
        }
        coords_of(tile + gridDim.x, x, yc);
        for (int l = 2; l < p.L; ++l) {
            ++tlayer;
            const uint32_t cbase = base + sm.consts + (uint32_t)((4 + float_areas(W) * (float_consts_resident(W) ? (uint32_t)(l - 2) : (tlayer - 1) & 1)) * W * 4);
            if constexpr (!XS) {
                // the activations in device memory become visible to the bulk copies of this CTA
                asm volatile("fence.proxy.async;" ::: "memory");
                ptx::mbar_arrive(base + sm.x_ready);
                // this thread's part of the third digit to tensor memory: the MMAs of the layer before, which read that
                // operand, completed with its last block's sums
                uint4 v[2 * NB];
#pragma unroll
                for (int q = 0; q < 2 * NB; ++q) v[q] = __ldcg(reinterpret_cast<const uint4 *>(xrow + 2 * (kTile * W) + (q / 2 * 8 + sub * 2 + q % 2) * (kTile * 16)));
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const uint32_t u[8] = {v[2 * b].x, v[2 * b].y, v[2 * b].z, v[2 * b].w, v[2 * b + 1].x, v[2 * b + 1].y, v[2 * b + 1].z, v[2 * b + 1].w};
                    ptx::tmem_st8(taddr + kFX2Col + (b * 8 + sub * 2) * 4, u);
                }
                ptx::tmem_wait_st();
                ptx::tc_fence_before();
                ptx::mbar_arrive(base + sm.x2_ready);
                if (!wait_bar_warp<true>(base + sm.c_full + 8 * ((tlayer - 1) & 1), ((tlayer - 1) >> 1) & 1, abort_flag, p.status)) return;
            }
#pragma unroll 1
            for (int b = 0; b < NB; ++b, ++use) {
                const int k0 = b * FB + sub * GPB * 16;
                const uint32_t t = taddr + sub * GPB * 16;
                if (!wait_bar_warp<true>(base + sm.acc_full, use & 1, abort_flag, p.status)) return;
                ptx::tc_fence_after();
                begin_part(tlayer, b);
                f32x2 r[GPB * 8];
#pragma unroll
                for (int g = 0; g < GPB; ++g) {
                    uint32_t D[3][16];
#pragma unroll
                    for (int d = 0; d < 3; ++d) ptx::tmem_ld16(t + d * FB + g * 16, D[d]);
                    ptx::tmem_wait_ld();
                    if (g == GPB - 1) { // the accumulators are free for the next block
                        ptx::tc_fence_before();
                        ptx::mbar_arrive(base + sm.acc_empty);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float4 c, e, o, ol = make_float4(0.f, 0.f, 0.f, 0.f);
                        const uint32_t at = cbase + (uint32_t)((k0 + g * 16 + 4 * q) * 4);
                        c = lds128(at); e = lds128(at + W * 4); o = lds128(at + 2 * W * 4);
                        if constexpr (float_rounds_once(W)) ol = lds128(at + 3 * W * 4);
                        r[g * 8 + 2 * q] = digit_phase2<W>(&D[0][4 * q], &D[1][4 * q], &D[2][4 * q], pack2(c.x, c.y), pack2(e.x, e.y), pack2(o.x, o.y), pack2(ol.x, ol.y));
                        r[g * 8 + 2 * q + 1] = digit_phase2<W>(&D[0][4 * q + 2], &D[1][4 * q + 2], &D[2][4 * q + 2], pack2(c.z, c.w), pack2(e.z, e.w), pack2(o.z, o.w), pack2(ol.z, ol.w));
                    }
                }
#pragma unroll
                for (int g = 0; g < GPB; ++g) {
                    float y[16];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float u, v;
                        unpack2(r[g * 8 + q], u, v);
                        y[2 * q] = sin_approx(u);
                        y[2 * q + 1] = sin_approx(v);
                    }
                    emit(l, k0 + g * 16, y, tok, valid);
                }
                // Beside the last tensor-core layer, which writes no activations: the first layer of the CTA's next
                // tile, whose digits go where this tile's were.  At width 512 the first two digits have all been copied to
                // shared memory by now (this block's sums needed every copy), and each thread read its part of the third,
                // which it is about to overwrite, at the start of the layer.
                if (l == p.L - 1 && tile + gridDim.x < p.n_tiles)
                    first_layer(b, x, yc, tok + gridDim.x * (long long)kTile, (tok + gridDim.x * (long long)kTile) < p.n);
                if (l < p.L - 1 || tile + gridDim.x < p.n_tiles) end_part(b);
            }
        }
        // last layer: the four threads of a row exchange their partial sums through tensor memory.  Tiles use two sets of
        // columns in turn: a thread may write the next tile's sums while a slower one still reads this tile's (with three
        // layers and one block of outputs nothing else orders the two), but to come back to this set it has to pass the
        // next tile's barrier, where the reader arrives after its reads.
        {
            const uint32_t u[4] = {__float_as_uint(part[0]), __float_as_uint(part[1]), __float_as_uint(part[2]), __float_as_uint(part[3])};
            const uint32_t part_col = taddr + kFPartCol + 16 * qpar;
            const uint32_t part_at = base + sm.part + qpar * (4 * kTile * 16) + row * 16; // (width 512: in shared memory)
            if constexpr (XS) {
                ptx::tmem_st4(part_col + 4 * sub, u);
                ptx::tmem_wait_st();
                ptx::tc_fence_before();
            } else {
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(part_at + sub * (kTile * 16)), "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]) : "memory");
            }
            ptx::mbar_arrive(base + sm.quad_sync + 8 * quad);
            if (!wait_bar_warp<true>(base + sm.quad_sync + 8 * quad, qpar, abort_flag, p.status)) return;
            qpar ^= 1;
            ptx::tc_fence_after();
            if (sub == 0) {
                uint32_t v[16];
                if constexpr (XS) {
                    ptx::tmem_ld16(part_col, v);
                    ptx::tmem_wait_ld();
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 f = lds128(part_at + q * (kTile * 16));
                        v[4 * q] = __float_as_uint(f.x); v[4 * q + 1] = __float_as_uint(f.y); v[4 * q + 2] = __float_as_uint(f.z); v[4 * q + 3] = __float_as_uint(f.w);
                    }
                }
                if (valid) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const float s = __fadd_rn(__fadd_rn(__uint_as_float(v[m]), __uint_as_float(v[4 + m])),
                                                  __fadd_rn(__uint_as_float(v[8 + m]), __uint_as_float(v[12 + m])));
                        const float z = __fmaf_rn(s, __ldg(p.sl + m), __ldg(p.bl + m));
                        if (m < p.d_L && (!DUMP || p.out)) p.out[tok * p.d_L + m] = z;
                        if constexpr (DUMP) {
                            if (p.dY[p.L - 1]) p.dY[p.L - 1][tok * 4 + m] = z;
                        }
                    }
                }
                ptx::tc_fence_before();
            }
        }
    }
}

// One warp issues the MMAs and has about 67 cycles for each, so the descriptors are kept as 32-bit
// words to which constants are added: the low word holds the operand's address in units of 16 bytes and
// the distance of core matrices along K, the high word is the same for every operand here.
template <int W, int WL>
__device__ void float_mma(const FloatParams &p, const FloatMap &sm, uint32_t base, uint32_t tmem, volatile int *abort_flag)
{
    constexpr int FB = float_block(W), KC = float_kc(W), NB = W / FB, NKC = W / KC, PIECE = FB * KC;
    ptx::wait_for_previous_kernels(); // before the first bounded wait
    const uint32_t idesc = ptx::idesc_i8(kTile, FB);
    constexpr uint32_t kDescHi = (128u >> 4) | (1u << 14);
    constexpr bool XS = float_x_in_smem(W);
    constexpr int DIGIT = kTile * (XS ? FB : W); // bytes between the digits of an activation
    const uint32_t a0 = ((base + sm.a) >> 4) | ((kTile * 16u >> 4) << 16), b0 = ((base + sm.ring) >> 4) | ((FB * 16u >> 4) << 16);
    uint32_t use = 0, layers = 0;
    int stage = 0;
    uint32_t wpar = 0;
    bool ok = true;
    for (long long tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x) {
        for (int l = 2; l < p.L && ok; ++l, ++layers) {
            for (int b = 0; b < NB && ok; ++b, ++use) {
                if (!wait_bar_warp<true>(base + sm.acc_empty, (use & 1) ^ 1, abort_flag, p.status)) { ok = false; break; }
                ptx::tc_fence_after();
                uint32_t ak = a0;
                for (int kc = 0; kc < NKC; ++kc, ak += (KC / 16) * (kTile * 16) >> 4) {
                    if constexpr (XS) {
                        static_assert(KC == FB && NB <= 2, "a part is a weight piece's k range; see float_x_in_smem");
                        ak = a0 + (((layers * NB + kc) % (NB + 1) * float_part_bytes(W)) >> 4);
                        if (b == 0) ok = wait_bar_warp<true>(base + sm.a_full + 8 * kc, layers & 1, abort_flag, p.status);
                        if (b == 0 && ok) ptx::tc_fence_after();
                    } else
                    for (int c = 0; b == 0 && c < KC / 64 && ok; ++c)
                        ok = wait_bar_warp<true>(base + sm.a_full + 8 * (kc * (KC / 64) + c), layers & 1, abort_flag, p.status);
                    if (!ok) break;
#pragma unroll
                    for (int j = 0; j < WL; ++j) {
                        if (!wait_bar_warp<true>(base + sm.w_full + 8 * stage, wpar, abort_flag, p.status)) { ok = false; break; }
                        const uint32_t bk = b0 + (uint32_t)stage * (PIECE >> 4);
#pragma unroll
                        for (int i = 0; i + j < 3; ++i) {
                            if (!XS && i == 2 && b == 0 && kc == 0) { // the third digit is in tensor memory
                                ok = wait_bar_warp<true>(base + sm.x2_ready, layers & 1, abort_flag, p.status);
                                if (!ok) break;
                                ptx::tc_fence_after();
                            }
#pragma unroll
                            for (int ks = 0; ks < KC / 32; ++ks) {
                                if constexpr (!XS) {
                                    if (i == 2) {
                                        ptx::mma_i8_tmem(tmem + (uint32_t)(i + j) * FB, tmem + kFX2Col + (uint32_t)((kc * (KC / 32) + ks) * 8), bk + (ks * 2 * FB * 16 >> 4), kDescHi, idesc, (j > 0 || ks > 0) ? 1u : (uint32_t)kc);
                                        continue;
                                    }
                                }
                                ptx::mma_i8_words(tmem + (uint32_t)(i + j) * FB, ak + ((i * DIGIT + ks * 2 * kTile * 16) >> 4), bk + (ks * 2 * FB * 16 >> 4),
                                                  kDescHi, idesc, (j > 0 || ks > 0) ? 1u : (uint32_t)kc);
                            }
                        }
                        if (!ok) break;
                        ptx::mma_commit(base + sm.w_empty + 8 * stage);
                        if (++stage == p.n_stages) { stage = 0; wpar ^= 1; }
                    }
                    if (!ok) break;
                }
                if (ok) ptx::mma_commit(base + sm.acc_full);
            }
        }
    }
    if (!ok) { // give the MMAs already issued a bounded time to finish before tensor memory is released
        ptx::mma_commit(base + sm.drain);
        const unsigned long long t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(base + sm.drain, 0) && ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
    }
}

// kFLoaders warps take the pieces in turn: waiting for a stage, arming its barrier and issuing the copy take one
// warp longer than a piece's MMAs.
template <int W, int WL>
__device__ void float_load_weights(const FloatParams &p, const FloatMap &sm, uint32_t base, int which, volatile int *abort_flag)
{
    constexpr int FB = float_block(W), KC = float_kc(W), PIECE = FB * KC, PIECES = (W / FB) * (W / KC) * WL;
    uint32_t i = 0, mine = 0, issued = 0; // pieces so far; the last one of this warp; how many it issued
    bool ok = true;
    for (long long tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x) {
        for (int l = 2; l < p.L && ok; ++l) {
            for (int q = 0; q < PIECES; ++q, ++i) {
                if ((int)(i % kFLoaders) != which || (p.skip_first_weights && i == 0)) continue;
                if (i >= (uint32_t)p.n_stages && i < (uint32_t)p.n_stages + kFLoaders) ptx::wait_for_previous_kernels();
                const uint32_t stage = i % (uint32_t)p.n_stages, par = ((i / (uint32_t)p.n_stages) & 1) ^ 1;
                if (!wait_bar_warp<true>(base + sm.w_empty + 8 * stage, par, abort_flag, p.status)) { ok = false; break; }
                ptx::mbar_expect_tx_warp(base + sm.w_full + 8 * stage, PIECE);
                ptx::bulk_g2s_warp(base + sm.ring + stage * PIECE, p.wimg[l - 1] + (size_t)q * PIECE, PIECE, base + sm.w_full + 8 * stage);
                mine = i;
                ++issued;
            }
        }
    }
    if (!ok || *abort_flag) { // let copies in flight land before the CTA may exit
        const unsigned long long t0 = ptx::globaltimer();
        for (int k = 0; k < p.n_stages && issued > 0; ++k, --issued, mine -= kFLoaders)
            while (!ptx::mbar_try_wait(base + sm.w_full + 8 * (mine % (uint32_t)p.n_stages), (mine / (uint32_t)p.n_stages) & 1) &&
                   ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
    }
}

// The activations of the next layer, written by this CTA's epilogue warps, back into shared memory:
// 64 features (8 KB of each digit) per barrier, so that the MMAs start with the first of them.  When all
// epilogue threads have arrived on x_ready they have read every accumulator of the layer before, so
// its MMAs are done with the operand area.
template <int W>
__device__ void float_load_x(const FloatParams &p, const FloatMap &sm, uint32_t base, volatile int *abort_flag)
{
    const uint8_t *src = p.x + (size_t)blockIdx.x * (3 * kTile * W);
    // the constants of layer l for the CTA's t-th tensor-core layer, into set t & 1
    uint32_t asked = 0;
    auto load_consts = [&](int l, uint32_t t) {
        asked = t + 1;
        const uint32_t at = base + sm.consts + (4 + 3 * (t & 1)) * W * 4, bar = base + sm.c_full + 8 * (t & 1);
        ptx::mbar_expect_tx_warp(bar, 3 * W * 4);
        ptx::bulk_g2s_warp(at, p.c0[l - 1], W * 4, bar);
        ptx::bulk_g2s_warp(at + W * 4, p.c0_lo[l - 1], W * 4, bar);
        ptx::bulk_g2s_warp(at + 2 * W * 4, p.cb[l - 1], W * 4, bar);
    };
    if (p.L > 2) load_consts(2, 0);
    ptx::wait_for_previous_kernels();
    uint32_t layers = 0;
    bool ok = true;
    for (long long tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x) {
        for (int l = 2; l < p.L; ++l, ++layers) {
            if (!wait_bar_warp<true>(base + sm.x_ready, layers & 1, abort_flag, p.status)) { ok = false; break; }
            asm volatile("fence.proxy.async;" ::: "memory");
            for (int c = 0; c < W / 64; ++c) {
                ptx::mbar_expect_tx_warp(base + sm.a_full + 8 * c, float_smem_digits(W) * 64 * kTile);
                for (int i = 0; i < float_smem_digits(W); ++i) {
                    const uint32_t off = (uint32_t)(i * kTile * W + c * 64 * kTile);
                    ptx::bulk_g2s_warp(base + sm.a + off, src + off, 64 * kTile, base + sm.a_full + 8 * c);
                }
            }
            // all threads are done with the layer before: the next one's constants take the place of that one's
            if (l + 1 < p.L || tile + gridDim.x < p.n_tiles) load_consts(l + 1 < p.L ? l + 1 : 2, layers + 1);
        }
    }
    if (!ok || *abort_flag) { // let copies in flight land before the CTA may exit
        const unsigned long long t0 = ptx::globaltimer();
        // (set t & 1 holds the constants of layer t; the last copies were those for `asked` - 1 and the one before)
        for (uint32_t t = asked > 2 ? asked - 2 : 0; t < asked; ++t)
            while (!ptx::mbar_try_wait(base + sm.c_full + 8 * (t & 1), (t >> 1) & 1) && ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
        for (int c = 0; layers > 0 && c < W / 64; ++c)
            while (!ptx::mbar_try_wait(base + sm.a_full + 8 * c, (layers - 1) & 1) && ptx::globaltimer() - t0 < wait_limit_of(abort_flag)) {}
    }
}

template <int W, int WL, bool DUMP>
__global__ void __launch_bounds__(kFThreads, 1) float_kernel(const __grid_constant__ FloatParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - raw);
    const FloatMap sm = float_map(W, p.n_stages, p.L);
    const int warp = ptx::uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gen + sm.abort_flag);
    ptx::launch_dependents();
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        *reinterpret_cast<volatile unsigned long long *>(abort_flag + 2) = p.wait_limit_ns;
        for (int i = 0; i < kFMaxStages; ++i) {
            ptx::mbar_init(base + sm.w_full + 8 * i, 1);
            ptx::mbar_init(base + sm.w_empty + 8 * i, 1);
        }
        for (int i = 0; i < 8; ++i) ptx::mbar_init(base + sm.a_full + 8 * i, float_x_in_smem(W) ? kEpiWarps : 1);
        ptx::mbar_init(base + sm.x_ready, kEpiWarps * 32);
        ptx::mbar_init(base + sm.x2_ready, kEpiWarps * 32);
        for (int i = 0; i < 2; ++i) ptx::mbar_init(base + sm.c_full + 8 * i, 1);
        ptx::mbar_init(base + sm.acc_full, 1);
        ptx::mbar_init(base + sm.acc_empty, kEpiWarps * 32);
        for (int i = 0; i < 4; ++i) ptx::mbar_init(base + sm.quad_sync + 8 * i, 128);
        ptx::mbar_init(base + sm.drain, 1);
        ptx::fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        ptx::tmem_alloc(base + sm.holder, 512);
        ptx::tmem_relinquish();
    }
    {
        float4 *dst = reinterpret_cast<float4 *>(gen + sm.consts);
        for (int i = threadIdx.x; i < W; i += kFThreads) dst[i] = __ldg(p.l1 + i);
        for (int l = 1; float_consts_resident(W) && l < p.L - 1; ++l) {
            float *c = reinterpret_cast<float *>(dst) + (4 + float_areas(W) * (l - 1)) * W;
            for (int i = threadIdx.x; i < W; i += kFThreads) {
                c[i] = __ldg(p.c0[l] + i);
                c[W + i] = __ldg(p.c0_lo[l] + i);
                const float b = __ldg(p.cb[l] + i), on_grid = float_rounds_once(W) ? __fsub_rn(__fadd_rn(b, 6144.0f), 6144.0f) : b;
                c[2 * W + i] = on_grid;
                if constexpr (float_rounds_once(W)) c[3 * W + i] = __fsub_rn(b, on_grid);
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ptx::uniform(*reinterpret_cast<volatile uint32_t *>(gen + sm.holder));
    if (warp < kEpiWarps) ptx::take_registers<kEpiRegs>(); // see splits_registers
    else ptx::give_registers<kRoleRegs>();
    if (warp < kEpiWarps) float_epilogue<W, WL, DUMP>(p, sm, base, warp, lane, tmem, abort_flag);
    else if (warp == kMmaWarp) float_mma<W, WL>(p, sm, base, tmem, abort_flag);
    else if (warp < kLoadWarp + kFLoaders) float_load_weights<W, WL>(p, sm, base, warp - kLoadWarp, abort_flag);
    else if constexpr (!float_x_in_smem(W)) float_load_x<W>(p, sm, base, abort_flag);
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        ptx::tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------- weight side, once per network

// One block per output row of a layer.  w8: the integer row q_w (H_K), else the fp32 row.
// Hidden layers: the row as base-256 digits in the order the MMAs take them - pieces of FB rows x KC k of
// one digit, ordered (block of FB rows, KC-slice, digit) - and the epilogue constants.  First layer: weights and
// bias in turns of the phase.  Last layer: the row as fp32 values, [K/4][M] float4.
__global__ void prep_float_kernel(FloatPrepArgs a)
{
    extern __shared__ int vi[];
    __shared__ double red[32];
    const int m = blockIdx.x, K = a.K, M = a.M, tid = threadIdx.x;
    const bool live = m < a.d_out;
    if (a.w8) {
        for (int k = tid; k < K; k += blockDim.x) vi[k] = a.dev.qw[(size_t)m * K + k];
        for (int h = 1; h < (a.rotate ? K : 1); h <<= 1) {
            __syncthreads();
            for (int q = tid; q < K / 2; q += blockDim.x) {
                const int i = ((q & ~(h - 1)) << 1) | (q & (h - 1));
                const int x = vi[i], y = vi[i + h];
                vi[i] = x + y;
                vi[i + h] = x - y;
            }
        }
        __syncthreads();
    }
    auto value = [&](int k) -> double {
        if (a.w8) return (double)vi[k];
        return live && k < a.d_in ? (double)a.W[(size_t)m * a.d_in + k] : 0.0;
    };
    const float row_scale = a.w8 ? a.dev.s_w[m] : 1.0f;
    const double turns = a.omega0 * 0.15915494309189533576888;
    if (a.first) {
        const double b = turns * (double)a.dev.bias[m];
        if (tid == 0)
            reinterpret_cast<float4 *>(a.dev.w_f32)[m] = make_float4((float)(turns * (double)row_scale * value(0)), (float)(turns * (double)row_scale * value(1)),
                                                                     (float)(b - rint(b)), 0.f); // whole turns would cost the bias bits
        return;
    }
    if (!a.hidden) {
        for (int k = tid; k < K; k += blockDim.x)
            reinterpret_cast<float *>(a.dev.w_f32)[((size_t)(k >> 2) * M + m) * 4 + (k & 3)] = (float)value(k);
        if (tid == 0) a.dev.f_scale[m] = row_scale;
        return;
    }
    double g = 0.0;
    for (int k = tid; k < K; k += blockDim.x) g = fmax(g, fabs(value(k)));
    for (int o = 16; o; o >>= 1) g = fmax(g, __shfl_xor_sync(0xffffffffu, g, o));
    if ((tid & 31) == 0) red[tid >> 5] = g;
    __syncthreads();
    for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) g = fmax(g, red[i]);
    if (a.digits == 0) { // measuring pass
        double sq = 0.0;
        for (int k = tid; k < K; k += blockDim.x) sq += value(k) * value(k);
        for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        __syncthreads();
        if ((tid & 31) == 0) red[tid >> 5] = sq;
        __syncthreads();
        if (tid == 0) {
            sq = 0.0;
            for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) sq += red[i];
            a.dev.cA[m] = (float)(sq * (double)row_scale * (double)row_scale);
            a.dev.cA_lo[m] = (float)(g * g * (double)row_scale * (double)row_scale);
            if (a.w8) atomicMax(a.row_max, (unsigned int)g);
        }
        return;
    }
    const double top = a.digits == 2 ? 32639.0 : 8355711.0; // 127 in every digit
    double f = 1.0;                                         // integers per unit of the row's values
    if (a.w8) while (g > 0.0 && g * f * 2.0 <= top) f *= 2.0; // integer rows stay integers
    else f = g > 0.0 ? top / g : 0.0;
    const int FB = float_block(K), KC = float_kc(K), piece = FB * KC;
    uint8_t *row = a.dev.wdig + (size_t)(m / FB) * (K / KC) * a.digits * piece + (m % FB) * 16;
    for (int k = tid; k < K; k += blockDim.x) {
        const int I = (int)rint(value(k) * f);
        const uint32_t v = (uint32_t)(I + (a.digits == 2 ? 0x8080 : 0x808080)) ^ (a.digits == 2 ? 0x8080u : 0x808080u);
        for (int j = 0; j < a.digits; ++j)
            row[(size_t)((k / KC) * a.digits + j) * piece + ((k % KC) >> 4) * (FB * 16) + (k & 15)] = (uint8_t)(v >> (8 * (a.digits - 1 - j)));
    }
    if (tid == 0) {
        const double c = f > 0.0 ? turns * (double)row_scale / f / 8355711.0 * (a.digits == 2 ? 16777216.0 : 4294967296.0) : 0.0;
        const float hi = (float)c;
        a.dev.cA[m] = hi;
        a.dev.cA_lo[m] = (float)(c - (double)hi);
        const double b = turns * (double)a.dev.bias[m];
        a.dev.cB[m] = (float)(b - rint(b));
    }
}

// One block for the network, so that the sums, and what is decided by them, do not depend on an order of arrival.
struct FloatSumsArgs { int L; double omega0; PrepSums *sums; LayerDev dev[kMaxLayers]; };
__global__ void __launch_bounds__(256) prep_float_sums_kernel(const __grid_constant__ FloatSumsArgs a)
{
    __shared__ double red[8][4];
    __shared__ int bad;
    const int tid = threadIdx.x;
    if (tid == 0) bad = 0;
    for (int l = 0; l < a.L; ++l) {
        const LayerDev &d = a.dev[l];
        const bool hidden = l > 0 && l < a.L - 1;
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        int nonfinite = 0;
        for (int m = tid; m < d.M; m += 256) {
            if (!isfinite(d.row_l1[m]) || !isfinite(d.s_w[m])) nonfinite = 1; // sum |W_mk| + |b_m|
            if (l < a.L - 1) v[2] += cos(2.0 * a.omega0 * (double)d.bias[m]);
            if (hidden) {
                const double sq = (double)d.cA[m], top = (double)d.cA_lo[m];
                v[0] += sq;
                v[1] += top;
                if (sq > 0.0) v[3] = fmax(v[3], top / sq);
            }
        }
        __syncthreads(); // (the words of the layer before have been read)
        for (int i = 0; i < 4; ++i) {
            for (int o = 16; o; o >>= 1) {
                const double u = __shfl_xor_sync(0xffffffffu, v[i], o);
                v[i] = i == 3 ? fmax(v[i], u) : v[i] + u;
            }
            if ((tid & 31) == 0) red[tid >> 5][i] = v[i];
        }
        if (nonfinite) bad = 1;
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < 8; ++w)
                for (int i = 0; i < 4; ++i) v[i] = i == 3 ? fmax(v[i], red[w][i]) : v[i] + red[w][i];
            a.sums->row_sq[l] = v[0];
            a.sums->row_top[l] = v[1];
            a.sums->cos_bias[l] = v[2];
            a.sums->worst_top[l] = v[3];
            if (l == a.L - 1) a.sums->finite = !bad;
        }
    }
}
cudaError_t launch_prep_float_sums(int L, double omega0, const LayerDev *layers, PrepSums *sums, cudaStream_t st, int64_t *launches)
{
    FloatSumsArgs a;
    a.L = L; a.omega0 = omega0; a.sums = sums;
    for (int l = 0; l < L; ++l) a.dev[l] = layers[l];
    prep_float_sums_kernel<<<1, 256, 0, st>>>(a);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_prep_float(const FloatPrepArgs &a, cudaStream_t st, int64_t *launches)
{
    prep_float_kernel<<<a.M, 128, a.K * sizeof(int), st>>>(a);
    *launches += 1;
    return cudaGetLastError();
}

// ------------------------------------------------------------------- host side

// One tile's activations per SM.
size_t float_scratch_bytes(const dhq_handle_s *h)
{
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess) sms = 148;
    return float_x_in_smem(h->w) || h->float_digits == 0 ? 0 : (size_t)sms * 3 * kTile * h->w;
}

struct FloatState {
    FloatParams p;
    size_t smem_bytes;
    int sm_count;
};

typedef void (*float_fn)(const FloatParams);
template <bool DUMP> static float_fn pick_float(int W, int digits)
{
    switch (W) {
    case 64: return digits == 2 ? float_kernel<64, 2, DUMP> : float_kernel<64, 3, DUMP>;
    case 128: return digits == 2 ? float_kernel<128, 2, DUMP> : float_kernel<128, 3, DUMP>;
    case 256: return digits == 2 ? float_kernel<256, 2, DUMP> : float_kernel<256, 3, DUMP>;
    case 512: return digits == 2 ? float_kernel<512, 2, DUMP> : float_kernel<512, 3, DUMP>;
    }
    return nullptr;
}

dhq_status_t float_create(dhq_handle_s *h)
{
    FloatState *fs = new (std::nothrow) FloatState();
    if (!fs) return DHQ_ERR_ALLOC;
    memset(fs, 0, sizeof(*fs));
    h->float_state = fs;
    const int dev = h->device;
    int max_optin = 0;
    if (cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&fs->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return DHQ_ERR_CUDA;
    FloatParams &p = fs->p;
    p.L = h->L; p.d_L = h->d_L;
    p.status = h->d_status;
    for (int l = 0; l < h->L; ++l) {
        const LayerDev &d = h->layer[l];
        p.wimg[l] = d.wdig;
        p.c0[l] = d.cA; p.c0_lo[l] = d.cA_lo; p.cb[l] = d.cB;
    }
    const LayerDev &d1 = h->layer[0], &dl = h->layer[h->L - 1];
    p.l1 = reinterpret_cast<const float4 *>(d1.w_f32);
    p.wl = reinterpret_cast<const float4 *>(dl.w_f32); p.sl = dl.f_scale; p.bl = dl.bias;
    // as many weight pieces in flight as fit beside the activations
    const size_t piece = (size_t)float_block(h->w) * float_kc(h->w);
    const size_t fixed = float_map(h->w, 0, h->L).total + 1024;
    int stages = (int)(((size_t)max_optin - fixed) / piece);
    if (stages > kFMaxStages) stages = kFMaxStages;
    if (fixed > (size_t)max_optin || stages < 1) return DHQ_ERR_UNSUPPORTED;
    p.n_stages = stages;
    fs->smem_bytes = float_map(h->w, stages, h->L).total + 1024;
    if (fs->smem_bytes < (size_t)kMinSmem) fs->smem_bytes = kMinSmem;
    p.x = h->x_scratch;
    float_fn fns[2] = {pick_float<false>(h->w, h->float_digits), pick_float<true>(h->w, h->float_digits)};
    for (float_fn f : fns)
        if (!allow_smem((const void *)f, dev, max_optin, kLaunchRegs)) return DHQ_ERR_CUDA;
    return DHQ_OK;
}

void float_destroy(dhq_handle_s *h)
{
    delete static_cast<FloatState *>(h->float_state);
    h->float_state = nullptr;
}

dhq_status_t float_forward(dhq_handle_s *h, const float *coords, int64_t n, float *out, const dhq_debug_bufs_t *bufs, cudaStream_t st)
{
    FloatState *fs = static_cast<FloatState *>(h->float_state);
    if (!fs) return DHQ_ERR_INVALID_ARG;
    FloatParams p = fs->p;
    p.coords = coords; p.out = out; p.n = n;
    p.n_tiles = (n + kTile - 1) / kTile;
    p.wait_limit_ns = h->wait_limit_ns;
    if (!bufs && h->stall_next_forward) { // test hook, one launch only
        p.skip_first_weights = 1;
        h->stall_next_forward = false;
    }
    bool dump = !out;
    if (bufs) {
        for (int l = 0; l < h->L; ++l) {
            if (bufs->X && bufs->X[l]) { p.dX[l] = bufs->X[l]; dump = true; }
            if (bufs->Y && bufs->Y[l]) { p.dY[l] = bufs->Y[l]; dump = true; }
        }
    }
    const int grid = (int)(p.n_tiles < fs->sm_count ? p.n_tiles : fs->sm_count);
    const float_fn fn = dump ? pick_float<true>(h->w, h->float_digits) : pick_float<false>(h->w, h->float_digits);
    const cudaError_t e = launch_after(h, (const void *)fn, grid, kFThreads, fs->smem_bytes, st, &p);
    h->launches++;
    return e == cudaSuccess ? DHQ_OK : DHQ_ERR_CUDA;
}

} // namespace dhq
