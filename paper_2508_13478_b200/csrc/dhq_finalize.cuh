// Epilogue constants of a layer once its scales are known.
#pragma once
#include "dhq_internal.cuh"

namespace dhq {

// One output row, in fp64, rounded once: cA = fl32(A), cA_lo = fl32(A - cA) with A = f * s_w * s_x (s_x = 1
// when the activation scale is per token), cB = fl32(f * b), f = omega0 for sine layers and 1 for the
// last layer.
__device__ __forceinline__ double finalize_row(const LayerDev &dev, int m, float s_x, float s_w, int sine, double omega0)
{
    if (dev.has_digits) { // phases in turns, the bias modulo one turn
        const double A = dev.g_scale[m] * (double)s_x, b = omega0 * (double)dev.bias[m] * 0.15915494309189533576888, n = rint(b);
        const float hi = (float)A;
        dev.cA[m] = hi;
        dev.cA_lo[m] = (float)(A - (double)hi);
        const double hi_b = rint((b - n) * 2048.0) * (1.0 / 2048.0); // see digit_phase
        dev.cB[m] = (float)hi_b;
        dev.cB_lo[m] = (float)(b - n - hi_b);
        dev.cN[m] = (float)n; // the wavelet's envelope needs the whole bias
        return A;
    }
    const double f = sine ? omega0 : 1.0;
    const double A = f * (double)s_w * (double)s_x;
    const float hi = (float)A;
    dev.cA[m] = hi;
    dev.cA_lo[m] = (float)(A - (double)hi);
    dev.cB[m] = (float)(f * (double)dev.bias[m]);
    return A;
}

// A whole layer by `threads` threads of one block.  Per-tensor activation scales: s_x and inv come
// from the frozen absmax in act[0].
__device__ __forceinline__ void finalize_layer(const LayerDev &dev, int a_bits, int per_token, int sine, double omega0, int tid, int threads)
{
    float s = 1.0f;
    if (!per_token) {
        float inv;
        scales_of(__ldcg(dev.act), qmax_of(a_bits), s, inv);
        if (tid == 0) {
            dev.act[1] = s;
            dev.act[2] = inv;
        }
    }
    for (int m = tid; m < dev.M; m += threads) {
        const double A = finalize_row(dev, m, s, dev.s_w[m], sine, omega0);
        if (dev.epi_mode == EPI_SINE_FIXED) {
            const double inv_two_pi = 0.15915494309189533576888;
            const int8_t *q = dev.qw + (size_t)m * 4;   // layer 1: K = 4
            double u = (double)((int)q[0] + (int)q[2]), v = (double)((int)q[1] + (int)q[3]);
            if (dev.has_uv) { // two-sided transform: the phase of output j comes from the rotated sums
                u = (double)dev.l1U[m];
                v = (double)dev.l1V[m];
            }
            auto to_fix = [](double turns) { return (uint32_t)(unsigned long long)llrint(turns * 4294967296.0); };
            dev.fxP[m] = to_fix(A * u * inv_two_pi);
            dev.fxQ[m] = to_fix(A * v * inv_two_pi);
            dev.fxB[m] = to_fix((sine ? omega0 : 1.0) * (double)dev.bias[m] * inv_two_pi);
        }
    }
}

// The last block of a calibration kernel to get here freezes the layer: act[0] then holds the maximum
// of all blocks.  act[3] counts the blocks (zero at the launch).  Called by all threads of a block;
// `last` is a word of shared memory.
__device__ __forceinline__ void freeze_by_last_block(const LayerDev &dev, int a_bits, int sine, double omega0, volatile int *last)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        *last = atomicAdd(reinterpret_cast<unsigned int *>(dev.act) + 3, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!*last) return;
    __threadfence();
    finalize_layer(dev, a_bits, 0, sine, omega0, threadIdx.x, blockDim.x);
}

} // namespace dhq
