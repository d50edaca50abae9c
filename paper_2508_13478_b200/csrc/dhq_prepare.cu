// Weight side of DHQ (Eq. 4-5 of the paper, the factor acting on the input dimension, and the
// quantizer of Section III-B), run once per network on the device:
//   pad -> rotate each row by H_K (fp32 butterfly, strides 1, 2, ..., K/2) -> scale by 1/K
//   -> absmax per tensor or per row -> quantize -> write the codes in three layouts.
// Each kernel covers the rows of all layers at once: the layers do not depend on one another, and a
// network of a few layers is launch-bound here (two launches in place of four to six per layer).
#include "dhq_internal.cuh"
#include "dhq_finalize.cuh"

namespace dhq {

// Block index -> layer (0-based) and row: w rows for each layer but the last, which has `last_rows`.
__device__ __forceinline__ void row_of_block(const PrepNet &a, int &l, int &m)
{
    l = min((int)blockIdx.x / a.w, a.L - 1);
    m = (int)blockIdx.x - l * a.w;
}

// One block per padded output row; K/2 threads, one butterfly pair each per stage.
__global__ void prep_rotate_kernel(const __grid_constant__ PrepNet a)
{
    extern __shared__ float row[];
    int l, m;
    row_of_block(a, l, m);
    const LayerDev &dev = a.dev[l];
    const int K = dev.K;
    for (int k = threadIdx.x; k < K; k += blockDim.x)
        row[k] = (m < dev.d_out && k < dev.d_in) ? a.W[l][(size_t)m * dev.d_in + k] : 0.0f;
    // phase bound of this row: sum_k |W_mk| + |b_m| (inputs of hidden layers lie in [-1, 1])
    __shared__ float red[32];
    float part = 0.f;
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) part += fabsf(row[k]);
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int i = 0; i < (blockDim.x + 31) / 32; ++i) s += red[i];
        const float b = m < dev.d_out ? a.b[l][m] : 0.0f;
        dev.row_l1[m] = s + fabsf(b); // |W_m . x + b_m| <= this for inputs in [-1, 1]
        dev.bias[m] = b;
    }
    for (int h = 1; h < (a.rotate ? K : 1); h <<= 1) {
        __syncthreads();
        for (int p = threadIdx.x; p < K / 2; p += blockDim.x) {
            int i = ((p & ~(h - 1)) << 1) | (p & (h - 1));
            float x = row[i], y = row[i + h];
            row[i] = __fadd_rn(x, y);
            row[i + h] = __fsub_rn(x, y);
        }
    }
    __syncthreads();
    const float invK = a.rotate ? 1.0f / (float)K : 1.0f; // power of two: exact
    float amax = 0.f;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        float v = __fmul_rn(row[k], invK);
        dev.w_rot[(size_t)m * K + k] = v;
        amax = fmaxf(amax, fabsf(v));
    }
    for (int o = 16; o; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x == 0) {
        float r = 0.f;
        for (int i = 0; i < (blockDim.x + 31) / 32; ++i) r = fmaxf(r, red[i]);
        dev.row_absmax[m] = r;
    }
}

// DHQ_ROT_BOTH, output-side factor of Eq. 4: one block per column k; the column of the row-rotated
// weights goes through the same fp32 butterfly over the M rows and is scaled by the exact 1/M.
__global__ void prep_rotate_cols_kernel(const __grid_constant__ PrepNet a)
{
    extern __shared__ float col[];
    const int l = (int)blockIdx.x < 4 ? 0 : 1 + ((int)blockIdx.x - 4) / a.w; // 4 columns, then w per layer
    const int k = l == 0 ? (int)blockIdx.x : ((int)blockIdx.x - 4) % a.w;
    const LayerDev &dev = a.dev[l];
    const int K = dev.K, M = dev.M;
    for (int m = threadIdx.x; m < M; m += blockDim.x) col[m] = dev.w_rot[(size_t)m * K + k];
    for (int h = 1; h < M; h <<= 1) {
        __syncthreads();
        for (int p = threadIdx.x; p < M / 2; p += blockDim.x) {
            int i = ((p & ~(h - 1)) << 1) | (p & (h - 1));
            float x = col[i], y = col[i + h];
            col[i] = __fadd_rn(x, y);
            col[i + h] = __fsub_rn(x, y);
        }
    }
    __syncthreads();
    const float invM = 1.0f / (float)M; // power of two: exact
    for (int m = threadIdx.x; m < M; m += blockDim.x) dev.w_rot[(size_t)m * K + k] = __fmul_rn(col[m], invM);
}

// Row absmax of the final rotated weights (after the column pass).
__global__ void prep_row_absmax_kernel(const __grid_constant__ PrepNet a)
{
    __shared__ float red[32];
    int l, m;
    row_of_block(a, l, m);
    const LayerDev &dev = a.dev[l];
    const int K = dev.K;
    float amax = 0.f;
    for (int k = threadIdx.x; k < K; k += blockDim.x) amax = fmaxf(amax, fabsf(dev.w_rot[(size_t)m * K + k]));
    for (int o = 16; o; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x == 0) {
        float r = 0.f;
        for (int i = 0; i < (blockDim.x + 31) / 32; ++i) r = fmaxf(r, red[i]);
        dev.row_absmax[m] = r;
    }
}

// One block per row of the tensor-core image (the last layer has 16 rows, of which 4 are the padded
// layer's): scales of the row, its codes in the three layouts, and its share of the phase bound.
//
// Bound of the phase omega0 (s_w s_x acc + b) that the epilogue of a hidden layer sees, over all
// inputs in [-1, 1]^K whose codes do not saturate: the unquantized bound sum_k |W_mk| + |b_m|
// plus what the two quantizers can add.  With s_x q_x = x~ + e_x, |e_x| <= s_x / 2 and
// s_w q_w = w~ + e_w, |e_w| <= s_w / 2:
//   s_w s_x acc = W x + sum_k e_w x~_k + sum_k s_w q_w e_x
//   |sum e_w x~|    <= (s_w / 2) * sum_k |x~_k|,  sum |x~_k| <= K sqrt(K) rotated (||x~||_2 = sqrt(K) ||x||_2), K unrotated
//   |sum s_w q_w e_x| <= (s_x / 2) * s_w * sum_k |q_w[m][k]|,  s_x <= max |x~| / qmax <= K / qmax rotated, 1 / qmax unrotated.
// The maximum over the rows decides between the fast and the wide sine.
__global__ void __launch_bounds__(128) prep_quant_kernel(const __grid_constant__ PrepNet a)
{
    __shared__ float red[4];
    __shared__ unsigned int red_q[4];
    int l, m;
    row_of_block(a, l, m);
    const LayerDev &dev = a.dev[l];
    const int K = dev.K, M = dev.M, tid = threadIdx.x, warp = tid >> 5;
    const bool live = m < M;
    const float qmaxf = qmax_of(a.bits);
    float s = 0.f, inv = 0.f;
    if (a.per_channel) {
        if (live) scales_of(dev.row_absmax[m], qmaxf, s, inv);
    } else {
        float r = 0.f;
        for (int i = tid; i < M; i += 128) r = fmaxf(r, dev.row_absmax[i]);
        for (int o = 16; o; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
        if ((tid & 31) == 0) red[warp] = r;
        __syncthreads();
        scales_of(fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3])), qmaxf, s, inv);
    }
    unsigned int qsum = 0;
    const int row = (l > 0 && l < a.L - 1) ? fused_column(m, M) : m; // hidden layers: tensor-memory column order
    for (int k = tid; k < K; k += 128) {
        int q = 0;
        if (live) {
            q = quantize(dev.w_rot[(size_t)m * K + k], inv, qmaxf);
            dev.qw[(size_t)m * K + k] = (int8_t)q;
            ((int8_t *)dev.qw_k4m)[((size_t)(k >> 2) * M + m) * 4 + (k & 3)] = (int8_t)q;
            qsum += (unsigned int)(q < 0 ? -q : q);
        }
        dev.qw_umma[umma_offset(row, k, dev.Mt, dev.slab_k)] = (uint8_t)(int8_t)q;
    }
    if (!live) return;
    qsum = __reduce_add_sync(0xffffffffu, qsum);
    if ((tid & 31) == 0) red_q[warp] = qsum;
    __syncthreads();
    if (tid != 0) return;
    qsum = red_q[0] + red_q[1] + red_q[2] + red_q[3]; // at most 512 * 127: exact in fp32 too
    dev.s_w[m] = s;
    dev.inv_w[m] = inv;
    const float xsum = a.rotate ? (float)K * sqrtf((float)K) : (float)K;
    const float sx_max = (a.rotate ? (float)K : 1.0f) / qmax_of(a.a_bits);
    const float slack = 0.5f * s * xsum + 0.5f * sx_max * s * (float)qsum;
    const float bound = (float)a.omega0 * (dev.row_l1[m] + slack) * 1.0001f;
    if (bound > 0.f) atomicMax(reinterpret_cast<unsigned int *>(&a.sums->phase_bound[l]), __float_as_uint(bound));
    atomicAdd(&a.sums->code_l1[l], (unsigned long long)qsum);
    if (a.finalize && !dev.has_digits) finalize_row(dev, m, 1.0f, s, l < a.L - 1, a.omega0);
}

// Two-sided transform, layer 1 (K = 4): the rotated padded coordinate has the codes [qs, qd, qs, qd],
// so acc_m = qs u_m + qd v_m with u_m = q[m][0] + q[m][2], v_m = q[m][1] + q[m][3], and the rotated
// accumulators are acc'_j = qs (H_M u)_j + qd (H_M v)_j.  One block computes H_M u and H_M v.
__global__ void prep_l1_both_kernel(LayerDev dev)
{
    extern __shared__ int uv[]; // [2][M]
    const int M = dev.M;
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        const int8_t *q = dev.qw + (size_t)m * 4;
        uv[m] = (int)q[0] + (int)q[2];
        uv[M + m] = (int)q[1] + (int)q[3];
    }
    for (int h = 1; h < M; h <<= 1) {
        __syncthreads();
        for (int p = threadIdx.x; p < M; p += blockDim.x) { // M/2 pairs for each of the two vectors
            const int which = p / (M / 2), j = p % (M / 2);
            const int i = which * M + (((j & ~(h - 1)) << 1) | (j & (h - 1)));
            const int x = uv[i], y = uv[i + h];
            uv[i] = x + y;
            uv[i + h] = x - y;
        }
    }
    __syncthreads();
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        dev.l1U[m] = uv[m];
        dev.l1V[m] = uv[M + m];
    }
}

__global__ void finalize_kernel(LayerDev dev, int a_bits, int per_token, int sine, double omega0)
{
    finalize_layer(dev, a_bits, per_token, sine, omega0, threadIdx.x, blockDim.x);
}

cudaError_t launch_prepare(const PrepNet &a, cudaStream_t st, int64_t *launches)
{
    const int rows = (a.L - 1) * a.w, threads = a.w / 2;
    prep_rotate_kernel<<<rows + 4, threads, a.w * sizeof(float), st>>>(a);
    if (a.rotate == 2) {
        prep_rotate_cols_kernel<<<4 + (a.L - 1) * a.w, threads, a.w * sizeof(float), st>>>(a);
        prep_row_absmax_kernel<<<rows + 4, 128, 0, st>>>(a);
        *launches += 2;
    }
    prep_quant_kernel<<<rows + 16, 128, 0, st>>>(a);
    *launches += 2;
    if (a.rotate == 2) {
        prep_l1_both_kernel<<<1, 256, 2 * a.w * sizeof(int), st>>>(a.dev[0]);
        *launches += 1;
    }
    return cudaGetLastError();
}

cudaError_t launch_finalize(const LayerDev &dev, int a_bits, int per_token, int sine, double omega0,
                            cudaStream_t st, int64_t *launches)
{
    finalize_kernel<<<1, 256, 0, st>>>(dev, a_bits, per_token, sine, omega0);
    *launches += 1;
    return cudaGetLastError();
}

} // namespace dhq
