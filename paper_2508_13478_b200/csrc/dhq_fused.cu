// Host side of the fused forward (kernels: dhq_fused.cuh, instantiated per width in
// dhq_fused_w*.cu): the parameter block of a handle, the choice of the instantiation and the
// launch; and the kernel's per-element loops run in isolation (micro-benchmark).
#include <mutex>
#include "dhq_fused.cuh"

namespace dhq {

// spread: the tile-to-CTA mapping for launches smaller than one tile per slot of every SM (tile_index);
// ahead: coordinates of the next tile copied to shared memory early (device memory only; width 512
// gained nothing from it and has no such variant)
static fused_fn pick_kernel(int W, bool per_token, bool rot, bool spread, bool ahead)
{
    switch (W) {
    case 64: return fused_pick_64(per_token, rot, spread, ahead);
    case 128: return fused_pick_128(per_token, rot, spread, ahead);
    case 256: return fused_pick_256(per_token, rot, spread, ahead);
    case 512: return fused_pick_512(per_token, rot, spread, ahead);
    }
    return nullptr;
}

static fused_fn pick_gabor_kernel(int W, bool per_token, bool rot)
{
    switch (W) {
    case 64: return fused_pick_gabor_64(per_token, rot);
    case 128: return fused_pick_gabor_128(per_token, rot);
    case 256: return fused_pick_gabor_256(per_token, rot);
    case 512: return fused_pick_gabor_512(per_token, rot);
    }
    return nullptr;
}
static fused_calib_fn pick_calib_kernel(int W, bool rot, bool gabor, bool both)
{
    switch (W) {
    case 64: return fused_pick_calib_64(rot, gabor, both);
    case 128: return fused_pick_calib_128(rot, gabor, both);
    case 256: return fused_pick_calib_256(rot, gabor, both);
    case 512: return fused_pick_calib_512(rot, gabor, both);
    }
    return nullptr;
}
static fused_fn pick_both_kernel(int W, bool per_token)
{
    switch (W) {
    case 64: return fused_pick_both_64(per_token);
    case 128: return fused_pick_both_128(per_token);
    case 256: return fused_pick_both_256(per_token);
    case 512: return fused_pick_both_512(per_token);
    }
    return nullptr;
}
static fused_dump_fn pick_both_dump_kernel(int W, bool per_token)
{
    switch (W) {
    case 64: return fused_pick_both_dump_64(per_token);
    case 128: return fused_pick_both_dump_128(per_token);
    case 256: return fused_pick_both_dump_256(per_token);
    case 512: return fused_pick_both_dump_512(per_token);
    }
    return nullptr;
}
static fused_fn pick_gabor_both_kernel(int W, bool per_token)
{
    switch (W) {
    case 64: return fused_pick_gabor_both_64(per_token);
    case 128: return fused_pick_gabor_both_128(per_token);
    case 256: return fused_pick_gabor_both_256(per_token);
    case 512: return fused_pick_gabor_both_512(per_token);
    }
    return nullptr;
}

static fused_dump_fn pick_gabor_both_dump_kernel(int W, bool per_token)
{
    switch (W) {
    case 64: return fused_pick_gabor_both_dump_64(per_token);
    case 128: return fused_pick_gabor_both_dump_128(per_token);
    case 256: return fused_pick_gabor_both_dump_256(per_token);
    case 512: return fused_pick_gabor_both_dump_512(per_token);
    }
    return nullptr;
}

static fused_dump_fn pick_gabor_dump_kernel(int W, bool per_token, bool rot)
{
    switch (W) {
    case 64: return fused_pick_gabor_dump_64(per_token, rot);
    case 128: return fused_pick_gabor_dump_128(per_token, rot);
    case 256: return fused_pick_gabor_dump_256(per_token, rot);
    case 512: return fused_pick_gabor_dump_512(per_token, rot);
    }
    return nullptr;
}

static fused_dump_fn pick_dump_kernel(int W, bool per_token, bool rot)
{
    switch (W) {
    case 64: return fused_pick_dump_64(per_token, rot);
    case 128: return fused_pick_dump_128(per_token, rot);
    case 256: return fused_pick_dump_256(per_token, rot);
    case 512: return fused_pick_dump_512(per_token, rot);
    }
    return nullptr;
}

static fused_fn pick_mixed_kernel(int W, bool rot, bool ahead)
{
    switch (W) {
    case 64: return fused_pick_mixed_64(rot, ahead);
    case 128: return fused_pick_mixed_128(rot, ahead);
    case 256: return fused_pick_mixed_256(rot, ahead);
    case 512: return fused_pick_mixed_512(rot, ahead);
    }
    return nullptr;
}

static fused_dump_fn pick_mixed_dump_kernel(int W, bool rot)
{
    switch (W) {
    case 64: return fused_pick_mixed_dump_64(rot);
    case 128: return fused_pick_mixed_dump_128(rot);
    case 256: return fused_pick_mixed_dump_256(rot);
    case 512: return fused_pick_mixed_dump_512(rot);
    }
    return nullptr;
}

// Per-token scales, one-sided or no rotation, sine, and a hidden layer under EPI_SINE_MIXED: the handle
// runs the instantiations that carry that variant.
static bool runs_mixed(const dhq_handle_s *h)
{
    if (h->cfg.a_gran != DHQ_GRAN_CHANNEL_OR_TOKEN || h->cfg.rotation == DHQ_ROT_BOTH || h->gabor_s0 > 0.0) return false;
    for (int l = 0; l < h->L; ++l)
        if (h->layer[l].epi_mode == EPI_SINE_MIXED) return true;
    return false;
}

static int threads_for(const dhq_handle_s *h) { return fused_threads(h->w, h->cfg.rotation == DHQ_ROT_BOTH, h->gabor_s0 > 0.0); }

// The kernel a handle's forward launches (spread, ahead: see pick_kernel; the other families have one mapping).
static fused_fn pick_for(const dhq_handle_s *h, bool per_token, bool spread, bool ahead)
{
    const bool both = h->cfg.rotation == DHQ_ROT_BOTH, rot = h->cfg.rotation == DHQ_ROT_INPUT;
    if (h->gabor_s0 > 0.0) return both ? pick_gabor_both_kernel(h->w, per_token) : pick_gabor_kernel(h->w, per_token, rot);
    if (both) return pick_both_kernel(h->w, per_token);
    if (runs_mixed(h)) return pick_mixed_kernel(h->w, rot, ahead);
    return pick_kernel(h->w, per_token, rot, spread, ahead);
}

// The same for a launch of at most one tile per SM; NULL where the width has no such kernel.
static fused_fn pick_narrow_for(const dhq_handle_s *h, bool per_token)
{
    const bool both = h->cfg.rotation == DHQ_ROT_BOTH, rot = h->cfg.rotation == DHQ_ROT_INPUT;
    const bool gabor = h->gabor_s0 > 0.0, mixed = runs_mixed(h);
    switch (h->w) {
    case 64: return !(both || gabor || mixed) ? nullptr : fused_pick_narrow_64(per_token, rot, both, gabor, mixed);
    case 128: return !(both || gabor || mixed) ? nullptr : fused_pick_narrow_128(per_token, rot, both, gabor, mixed);
    case 256: return fused_pick_narrow_256(per_token, rot, both, gabor, mixed);
    }
    return nullptr;
}

// The same for a launch of at most one tile of 64 tokens per SM.
static fused_fn pick_dup_for(const dhq_handle_s *h, bool per_token)
{
    const bool both = h->cfg.rotation == DHQ_ROT_BOTH, rot = h->cfg.rotation == DHQ_ROT_INPUT, gabor = h->gabor_s0 > 0.0, mixed = runs_mixed(h);
    switch (h->w) {
    case 64: return fused_pick_dup_64(per_token, rot, both, gabor, mixed);
    case 128: return fused_pick_dup_128(per_token, rot, both, gabor, mixed);
    case 256: return fused_pick_dup_256(per_token, rot, both, gabor, mixed);
    case 512: return fused_pick_dup_512(per_token, rot, both, gabor, mixed);
    }
    return nullptr;
}

// Its observing instantiation.
static fused_dump_fn pick_dump_for(const dhq_handle_s *h, bool per_token)
{
    const bool both = h->cfg.rotation == DHQ_ROT_BOTH, rot = h->cfg.rotation == DHQ_ROT_INPUT;
    if (h->gabor_s0 > 0.0) return both ? pick_gabor_both_dump_kernel(h->w, per_token) : pick_gabor_dump_kernel(h->w, per_token, rot);
    if (both) return pick_both_dump_kernel(h->w, per_token);
    if (runs_mixed(h)) return pick_mixed_dump_kernel(h->w, rot);
    return pick_dump_kernel(h->w, per_token, rot);
}

// Lets a kernel use all of an SM's shared memory; the driver is asked once per kernel and device
// (8 of these calls per dhq_prepare took 15 us; when the table is full, every time).  A kernel whose warpgroups split
// its registers must have been launched with at least min_regs a thread, or the split would wait for registers that do
// not exist.
constexpr int kMaxAllowed = 512;
static std::mutex g_allowed_mutex;
static struct { const void *fn; int device; } g_allowed[kMaxAllowed];
static int g_allowed_count = 0;
bool allow_smem(const void *fn, int device, int bytes, int min_regs)
{
    if (!fn) return false;
    std::lock_guard<std::mutex> lock(g_allowed_mutex);
    for (int i = 0; i < g_allowed_count; ++i)
        if (g_allowed[i].fn == fn && g_allowed[i].device == device) return true;
    cudaFuncAttributes at;
    if (min_regs > 0 && (cudaFuncGetAttributes(&at, fn) != cudaSuccess || at.numRegs < min_regs)) return false;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    if (g_allowed_count < kMaxAllowed) g_allowed[g_allowed_count++] = {fn, device};
    return true;
}
void forget_allowed()
{
    std::lock_guard<std::mutex> lock(g_allowed_mutex);
    g_allowed_count = 0;
}

// A forward launch.  Once an ordinary launch has followed the preparation and calibration in a stream (so that
// they had completed before it began), later ones in that stream use programmatic dependent launch: what the kernel
// does before wait_for_previous_kernels touches only the handle's weights and constants.  A block of the later launch
// that waits holds no SM that the earlier one needs: it is not started before all blocks of the earlier
// launch are.  Back to back, the binding's shorter call included: 4,096 coordinates at width 64 9.9 -> 5.9 us, 1,000 at
// width 256 18.5 -> 14.9 us, 65,536 at width 256 45.0 -> 41.4 us (by this step alone; 5.0, 10.9 and 40.2 us with the later ones).
static cudaError_t launch_early(const void *fn, int grid, int threads, size_t smem, cudaStream_t st, void *params, bool early)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    void *args[1] = {params};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    return e != cudaSuccess ? e : cudaGetLastError();
}
cudaError_t launch_after(dhq_handle_s *h, const void *fn, int grid, int threads, size_t smem, cudaStream_t st, void *params)
{
    const bool early = h->settled && st == h->settled_stream;
    const cudaError_t e = launch_early(fn, grid, threads, smem, st, params, early);
    if (!early && e == cudaSuccess && st != cudaStreamPerThread) {
        // A launch that stream capture only recorded has followed nothing yet; neither has one in another stream
        // than the next (the calibration passes let the launch behind them begin before they are done).
        cudaStreamCaptureStatus capture;
        if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) (void)cudaGetLastError();
        else if (capture == cudaStreamCaptureStatusNone) {
            h->settled = true;
            h->settled_stream = st;
        }
    }
    return e;
}

dhq_status_t fused_create(dhq_handle_s *h)
{
    FusedState *fs = new (std::nothrow) FusedState();
    if (!fs) return DHQ_ERR_ALLOC;
    memset(fs, 0, sizeof(*fs));
    h->fused = fs;
    FusedParams &p = fs->p;
    p.L = h->L; p.W = h->w; p.d_L = h->d_L;
    p.per_token = h->cfg.a_gran == DHQ_GRAN_CHANNEL_OR_TOKEN;
    p.qmaxf = (float)((1 << (h->cfg.a_bits - 1)) - 1);
    p.one2 = make_float2(1.0f, 1.0f);
    p.status = h->d_status;
    const bool both = h->cfg.rotation == DHQ_ROT_BOTH;
    const bool gabor = h->gabor_s0 > 0.0;
    p.gabor_c = gabor ? (float)(h->gabor_s0 / (double)h->cfg.omega0) : 0.f;
    int words = 0;
    for (int l = 0; l < h->L; ++l) {
        const LayerDev &d = h->layer[l];
        FusedLayer &f = p.layer[l];
        f.qw_umma = d.qw_umma;
        f.qw_k4m = d.qw_k4m;
        f.cA = d.cA; f.cA_lo = d.cA_lo; f.cB = d.cB;
        f.fxP = d.fxP; f.fxQ = d.fxQ; f.fxB = d.fxB;
        f.act = d.act;
        f.l1U = d.l1U; f.l1V = d.l1V;
        f.epi_mode = d.epi_mode;
        f.c_off = words;
        if (l < h->L - 1) {
            int areas = (l == 0) ? (d.epi_mode == EPI_SINE_FIXED ? 3 : (both ? 5 : 4)) : ((d.epi_mode == EPI_SINE_WIDE || d.epi_mode == EPI_SINE_MIXED) ? 3 : 2);
            words += areas * h->w;
        }
    }
    p.const_words = words;
    fused_fn fn = pick_for(h, p.per_token, false, false);
    if (!fn) return DHQ_ERR_UNSUPPORTED;
    const int dev = h->device;
    int max_optin = 0;
    if (cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&fs->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return DHQ_ERR_CUDA;
    // weight ring: as many slab stages as fit beside the A tiles and the constants; all hidden
    // layers resident if they fit
    const int pieces = (h->w == 512) ? 8 : 1;
    const int slabs = (h->L - 2) * pieces;
    const size_t slab_bytes = (h->w == 512) ? (size_t)128 * 256 : (size_t)h->w * h->w;
    const size_t fixed = smem_map(h->w, 0, words).total + 1024;
    if (fixed > (size_t)max_optin) return DHQ_ERR_UNSUPPORTED;
    int stages = (int)(((size_t)max_optin - fixed) / slab_bytes);
    if (stages > kMaxStages) stages = kMaxStages;
    if (slabs > 0 && stages < 1) return DHQ_ERR_UNSUPPORTED;
    if (stages >= slabs) { p.resident = 1; p.n_stages = slabs > 0 ? slabs : 0; }
    else { p.resident = 0; p.n_stages = stages; }
    size_t bytes = smem_map(h->w, p.n_stages, words).total + 1024;
    if (bytes < (size_t)kMinSmem) bytes = kMinSmem;
    fs->smem_bytes = bytes;
    const int min_regs = splits_registers(h->w, both, gabor) ? kLaunchRegs : 0;
    for (int v = 0; v < 4; ++v) // every variant of this handle's kernel
        if (!allow_smem((const void *)pick_for(h, p.per_token, (v & 1) != 0, (v & 2) != 0), dev, max_optin, min_regs)) return DHQ_ERR_CUDA;
    const fused_fn narrow = pick_narrow_for(h, p.per_token);
    if (!allow_smem((const void *)pick_dup_for(h, p.per_token), dev, max_optin, min_regs)) return DHQ_ERR_CUDA;
    if (narrow && !allow_smem((const void *)narrow, dev, max_optin, min_regs)) return DHQ_ERR_CUDA;
    if (!p.per_token && !allow_smem((const void *)pick_calib_kernel(h->w, h->cfg.rotation == DHQ_ROT_INPUT, gabor, both), dev, max_optin, min_regs)) return DHQ_ERR_CUDA;
    fs->max_smem = max_optin;
    fs->min_regs = min_regs; // (the observing kernel is loaded by its first call: that takes milliseconds)
    return DHQ_OK;
}

void fused_destroy(dhq_handle_s *h)
{
    delete static_cast<FusedState *>(h->fused);
    h->fused = nullptr;
}

int64_t fused_round_tokens(const dhq_handle_s *h)
{
    const FusedState *fs = static_cast<const FusedState *>(h->fused);
    const int slots = (h->w == 512) ? 1 : 2;
    return (int64_t)(fs ? fs->sm_count : 1) * slots * kTile;
}

// The per-call part of the parameter block.
static void fill_call(const dhq_handle_s *h, FusedParams &p, const float *coords, int64_t n, float *out, bool on_host)
{
    p.coords = coords; p.out = out; p.n = n;
    p.n_tiles = (n + kTile - 1) / kTile;
    p.bulk_xy = (((uintptr_t)coords) & 15) == 0;
    // (two more barriers per tile: worth it over the host link only)
    p.bulk_out = on_host && (((uintptr_t)out) & 15) == 0 && (smem_map(h->w, p.n_stages, p.const_words).out_tile & 15) == 0;
    p.wait_limit_ns = h->wait_limit_ns;
    p.skip_last_weights = 0;
}

dhq_status_t fused_forward(dhq_handle_s *h, const float *coords, int64_t n, float *out, bool on_host, cudaStream_t st)
{
    FusedState *fs = static_cast<FusedState *>(h->fused);
    if (!fs) return DHQ_ERR_INVALID_ARG;
    FusedParams p = fs->p;
    fill_call(h, p, coords, n, out, on_host);
    if (h->stall_next_forward) { // test hook, one launch only
        p.skip_last_weights = 1;
        h->stall_next_forward = false;
    }
    const int slots = (h->w == 512) ? 1 : 2;
    const bool both = h->cfg.rotation == DHQ_ROT_BOTH;
    const bool gabor = h->gabor_s0 > 0.0;
    const bool spread = !both && !gabor && !runs_mixed(h) && slots > 1 && p.n_tiles < (long long)fs->sm_count * slots;
    constexpr int kHalfTile = kTile / 2;
    const fused_fn dup = n <= (int64_t)fs->sm_count * kHalfTile ? pick_dup_for(h, p.per_token) : nullptr;
    if (dup) p.n_tiles = (n + kHalfTile - 1) / kHalfTile;
    const fused_fn narrow = dup ? dup : p.n_tiles <= (long long)fs->sm_count ? pick_narrow_for(h, p.per_token) : nullptr;
    const fused_fn fn = narrow ? narrow : pick_for(h, p.per_token, spread, !on_host);
    const long long ctas = spread || narrow ? p.n_tiles : (p.n_tiles + slots - 1) / slots;
    int grid = (int)(ctas < fs->sm_count ? ctas : fs->sm_count);
    const cudaError_t e = launch_after(h, (const void *)fn, grid, threads_for(h), fs->smem_bytes, st, &p);
    h->launches++;
    return e == cudaSuccess ? DHQ_OK : DHQ_ERR_CUDA;
}

// Layer 1's rotated input is H_4 [x, y, 0, 0] = [x+y, x-y, x+y, x-y] (or [x, y, 0, 0] without the
// rotation): its absmax over the coordinate set needs no network.
__global__ void calib_l1_kernel(const float *coords, long long n, int rot, int freeze, int a_bits, double omega0, LayerDev dev)
{
    float *act = dev.act;
    float amax = 0.f;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const float2 xy = __ldg(reinterpret_cast<const float2 *>(coords) + t);
        const float a = rot ? __fadd_rn(xy.x, xy.y) : xy.x, b = rot ? __fsub_rn(xy.x, xy.y) : xy.y;
        amax = fmaxf(amax, fmaxf(fabsf(a), fabsf(b)));
    }
    for (int o = 16; o; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned int *>(act), __float_as_uint(amax));
    __shared__ int last;
    if (freeze) freeze_by_last_block(dev, a_bits, 1, omega0, &last);
}

// One calibration pass by the fused kernel: the maximum of |rotated input of layer l| over the
// coordinates, with layers < l run as they are frozen, is accumulated into the layer's act[0]
// (which the caller has cleared).  Per-tensor activation scales; every rotation mode and activation
// that has a fused kernel.
dhq_status_t fused_calibrate_layer(dhq_handle_s *h, int l, const float *coords, int64_t n, bool freeze, cudaStream_t st)
{
    FusedState *fs = static_cast<FusedState *>(h->fused);
    if (!fs || fs->p.per_token || l < 1 || l > h->L) return DHQ_ERR_INVALID_ARG;
    if (n <= 0) return DHQ_OK;
    if (l == 1) {
        const long long blocks = (n + 255) / 256;
        calib_l1_kernel<<<(unsigned)(blocks < 1184 ? blocks : 1184), 256, 0, st>>>(coords, n, h->cfg.rotation != DHQ_ROT_NONE,
                                                                                     freeze, h->cfg.a_bits, (double)h->cfg.omega0, h->layer[0]);
        h->launches++;
        return cudaGetLastError() == cudaSuccess ? DHQ_OK : DHQ_ERR_CUDA;
    }
    FusedParamsCalib p;
    static_cast<FusedParams &>(p) = fs->p;
    fill_call(h, p, coords, n, nullptr, false);
    p.L = l; // the network up to the rotated input of layer l
    p.freeze = freeze;
    p.a_bits = h->cfg.a_bits;
    p.sine = l < h->L;
    p.omega0 = (double)h->cfg.omega0;
    p.dev = h->layer[l - 1];
    fused_calib_fn fn = pick_calib_kernel(h->w, h->cfg.rotation == DHQ_ROT_INPUT, h->gabor_s0 > 0.0, h->cfg.rotation == DHQ_ROT_BOTH);
    const int grid = (int)(p.n_tiles < fs->sm_count ? p.n_tiles : fs->sm_count);
    // set up beside the pass before it; reads nothing of that pass before wait_for_previous_kernels
    const cudaError_t e = launch_early((const void *)fn, grid, threads_for(h), fs->smem_bytes, st, &p, true);
    h->launches++;
    return e == cudaSuccess ? DHQ_OK : DHQ_ERR_CUDA;
}

// The same forward by the observing instantiation of the kernel: every per-layer value the
// caller asked for is written out from inside the fused kernel, where it is produced.
dhq_status_t fused_forward_dump(dhq_handle_s *h, const float *coords, int64_t n, float *out, const DumpPtrs &d, cudaStream_t st)
{
    FusedState *fs = static_cast<FusedState *>(h->fused);
    if (!fs) return DHQ_ERR_INVALID_ARG;
    FusedParamsDump p;
    static_cast<FusedParams &>(p) = fs->p;
    fill_call(h, p, coords, n, out, false);
    p.d = d;
    const int slots = (h->w == 512) ? 1 : 2;
    fused_dump_fn fn = pick_dump_for(h, p.per_token);
    if (!allow_smem((const void *)fn, h->device, fs->max_smem, fs->min_regs)) return DHQ_ERR_CUDA;
    const long long ctas = (p.n_tiles + slots - 1) / slots;
    int grid = (int)(ctas < fs->sm_count ? ctas : fs->sm_count);
    fn<<<grid, threads_for(h), fs->smem_bytes, st>>>(p);
    h->launches++;
    return cudaGetLastError() == cudaSuccess ? DHQ_OK : DHQ_ERR_CUDA;
}

// ---------------------------------------------------------------- inner loops in isolation
//
// The per-element work of a hidden layer of width 256 without anything else the fused kernel
// does: no MMA, no mbarrier, no tile loop.  16 warps per SM run, `iters` times, pass 1 (tensor
// memory -> dequantize, sine, butterfly stages below 64 -> tensor memory), pass 2 (stages 64 and
// 128, quantizer, code stores to shared memory) or both, each warp on its own lanes and columns
// with the same functions and the same thread-to-data mapping as the kernel (R = 2).  The rate
// this reaches is what the kernel's arithmetic could do if every wait were hidden.
template <int WHICH> __global__ void __launch_bounds__(512, 1) pass_rate_kernel(int iters)
{
    constexpr int W = 256;
    using C = Cfg<W>;
    constexpr int CH = C::CH, NCH = C::NCH, G = C::G;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - raw);
    constexpr uint32_t kConsts = 2 * kTile * W, kHolder = kConsts + 3 * W * 4; // two A tiles, then cA | cB | cA_lo
    float *cst = reinterpret_cast<float *>(gen + kConsts);
    for (int i = threadIdx.x; i < 3 * W; i += blockDim.x) cst[i] = (i < W) ? 1e-5f : (i < 2 * W ? 0.3f : 0.f);
    const int warp = ptx::uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (warp == 0) {
        ptx::tmem_alloc(base + kHolder, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ptx::uniform(*reinterpret_cast<volatile uint32_t *>(gen + kHolder));
    const int quad = warp & 3, slot = warp >> 3, sub = (warp >> 2) & 1;
    const uint32_t taddr = tmem + (uint32_t)(slot * C::TMEM_COLS_PER_SLOT) + ((uint32_t)(quad * 32) << 16);
    {
        uint32_t v[CH];
#pragma unroll
        for (int i = 0; i < CH; ++i) v[i] = (uint32_t)((lane * 37 + i * 11) % 2001 - 1000);
        for (int cc = 0; cc < C::CPT; ++cc) tmem_st<CH>(taddr + (sub * C::CPT + cc) * CH, v);
        ptx::tmem_wait_st();
    }
    __syncthreads();
    for (int it = 0; it < iters; ++it) {
        if (WHICH & 1) {
#pragma unroll
            for (int cc = 0; cc < C::CPT; ++cc) {
                const int ch = chunk_of<C>(sub, cc);
                uint32_t v[CH];
                tmem_ld<CH>(taddr + ch * CH, v);
                ptx::tmem_wait_ld();
                hidden_chunk<W, CH, false, true, EPI_SINE_FAST>(base + kConsts, ch * CH, 1.f, v);
                tmem_st<CH>(taddr + ch * CH, v);
            }
            ptx::tmem_wait_st();
        }
        if (WHICH & 2) {
#pragma unroll 1
            for (int gg = 0; gg < C::GPT; ++gg) {
                const int g = sub * C::GPT + gg;
                uint32_t u[NCH][G];
                load_group<C>(taddr + g * G, u);
                across_chunks<C, true>(u);
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch)
                    quantize_store<G, true>(base + slot * (kTile * W), quad * 32 + lane, ch * CH + g * G, u[ch], 1e-3f, 127.f, 0);
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        ptx::tmem_dealloc(tmem, 512);
    }
}

cudaError_t launch_pass_rate(int which, int sms, int iters, cudaStream_t st)
{
    const size_t smem = 2 * kTile * 256 + 3 * 256 * 4 + 64 + 1024 > (size_t)kMinSmem ? 2 * kTile * 256 + 3 * 256 * 4 + 64 + 1024 : (size_t)kMinSmem;
    void (*fn)(int) = which == 1 ? pass_rate_kernel<1> : which == 2 ? pass_rate_kernel<2> : pass_rate_kernel<3>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fn<<<sms, 512, smem, st>>>(iters);
    return cudaGetLastError();
}

} // namespace dhq
