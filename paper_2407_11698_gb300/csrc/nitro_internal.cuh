// Internal declarations of the GB300 NITRO-D library (not part of the ABI).
#pragma once

#include <atomic>
#include <cstdint>
#include <utility>
#include <cuda_runtime.h>

#include "nitro.h"

namespace nitro {

// ---------------------------------------------------------------------------
// Integer helpers, device and host.  fdiv is the paper's \intdiv (floor).
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int64_t fdiv64(int64_t x, int64_t d) {
    int64_t q = x / d;
    return (x % d < 0) ? q - 1 : q;
}
__host__ __device__ __forceinline__ int32_t fdiv32(int32_t x, int32_t d) {
    int32_t q = x / d;
    return (x % d < 0) ? q - 1 : q;
}

// floor(z / (256 * k)) = floor(floor(z / 256) / k) for k > 0; the first step
// is an arithmetic shift.
__host__ __device__ __forceinline__ int64_t scale_floor(int64_t z, int64_t k) {
    return fdiv64(z >> 8, k);
}

// Floor division by an invariant positive integer d through a multiply-high,
// after Granlund & Montgomery, "Division by invariant integers using
// multiplication" (PLDI 1994), Fig. 4.1 (N = 64): with l = ceil(log2 d),
// m = floor(2^64 (2^l - d) / d) + 1, sh1 = min(l, 1), sh2 = max(l - 1, 0),
// floor(n / d) = (t + ((n - t) >> sh1)) >> sh2 with t = mulhi(m, n), for every
// unsigned 64-bit n.  Negative x use floor(x / d) = -floor((-x - 1) / d) - 1.
struct FloorDiv {
    uint64_t m;
    int sh1, sh2;
    __host__ static FloorDiv make(uint64_t d) {
        int l = 0;
        while (l < 64 && ((uint64_t)1 << l) < d) ++l;
        FloorDiv f;
        const unsigned __int128 two_l = (unsigned __int128)1 << l;
        f.m = (uint64_t)((((unsigned __int128)1 << 64) * (two_l - d)) / d + 1);
        f.sh1 = l < 1 ? l : 1;
        f.sh2 = l > 1 ? l - 1 : 0;
        return f;
    }
    __host__ __device__ __forceinline__ uint64_t udiv(uint64_t n) const {
#ifdef __CUDA_ARCH__
        const uint64_t t = __umul64hi(m, n);
#else
        const uint64_t t = (uint64_t)(((unsigned __int128)m * n) >> 64);
#endif
        return (t + ((n - t) >> sh1)) >> sh2;
    }
    __host__ __device__ __forceinline__ int64_t floor_div(int64_t x) const {
        if (x >= 0) return (int64_t)udiv((uint64_t)x);
        return -(int64_t)udiv((uint64_t)(-(x + 1))) - 1;
    }
    __host__ __device__ __forceinline__ int64_t trunc_div(int64_t x) const {
        if (x >= 0) return (int64_t)udiv((uint64_t)x);
        return -(int64_t)udiv((uint64_t)(-(x + 1)) + 1);
    }
};

// The same method with N = 32 for 32-bit operands (one 32-bit multiply-high).
struct FloorDiv32 {
    uint32_t m;
    int sh1, sh2;
    __host__ static FloorDiv32 make(uint32_t d) {
        int l = 0;
        while (l < 32 && ((uint64_t)1 << l) < d) ++l;
        FloorDiv32 f;
        f.m = (uint32_t)((((uint64_t)1 << 32) * (((uint64_t)1 << l) - d)) / d + 1);
        f.sh1 = l < 1 ? l : 1;
        f.sh2 = l > 1 ? l - 1 : 0;
        return f;
    }
    __host__ __device__ __forceinline__ uint32_t udiv(uint32_t n) const {
#ifdef __CUDA_ARCH__
        const uint32_t t = __umulhi(m, n);
#else
        const uint32_t t = (uint32_t)(((uint64_t)m * n) >> 32);
#endif
        return (t + ((n - t) >> sh1)) >> sh2;
    }
    __host__ __device__ __forceinline__ int32_t trunc_div(int32_t x) const {
        const uint32_t q = udiv(x < 0 ? 0u - (uint32_t)x : (uint32_t)x);
        return x < 0 ? (int32_t)(0u - q) : (int32_t)q;
    }
    // branch-free: for x < 0, ~x = -(x + 1) and ~q = -q - 1
    __host__ __device__ __forceinline__ int32_t floor_div(int32_t x) const {
        const uint32_t ux = x >= 0 ? (uint32_t)x : ~(uint32_t)x;
        const uint32_t q = udiv(ux);
        return x >= 0 ? (int32_t)q : (int32_t)~q;
    }
};

__host__ __device__ __forceinline__ bool fits_i32(int64_t v) {
    return v >= INT32_MIN && v <= INT32_MAX;
}

// NITRO-ReLU piece of x: 0 x<-127, 1 -127<=x<0, 2 0<=x<=127, 3 x>127.
__host__ __device__ __forceinline__ int relu_region(int64_t x) {
    return x < -127 ? 0 : (x < 0 ? 1 : (x <= 127 ? 2 : 3));
}
// NITRO-ReLU forward value (Sec. 3.2.2).
__host__ __device__ __forceinline__ int relu_value(int64_t x, int alpha_inv, int mu) {
    if (x < 0) {
        int c = x < -127 ? -127 : (int)x;
        return fdiv32(c, alpha_inv) - mu;
    }
    return (x > 127 ? 127 : (int)x) - mu;
}
// Same, with the slope division through a precomputed divider.
__host__ __device__ __forceinline__ int relu_value(int64_t x, const FloorDiv& alpha, int mu) {
    if (x < 0) {
        int64_t c = x < -127 ? -127 : x;
        return (int)alpha.floor_div(c) - mu;
    }
    return (x > 127 ? 127 : (int)x) - mu;
}
// NITRO-ReLU backward per piece.
__host__ __device__ __forceinline__ int32_t relu_backward(int32_t g, int region, int alpha_inv) {
    return region == 1 ? fdiv32(g, alpha_inv) : (region == 2 ? g : 0);
}

__host__ __device__ __forceinline__ uint32_t abs_u32(int32_t v) {
    return v < 0 ? (uint32_t)(-(int64_t)v) : (uint32_t)v;
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014), random-access form: output
// `index` of the generator seeded with `seed` is the published finaliser
// applied to seed + (index + 1) * 0x9E3779B97F4A7C15.
__host__ __device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t index) {
    uint64_t z = seed + (index + 1ULL) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Dropout of the linear forward layers (App. B, p_l): element e of forward
// layer `layer` at step t is dropped when the top 16 bits of output
// 2^63 + t 2^35 + layer 2^31 + e of the block's SplitMix64 stream are below
// p16 (rate in units of 2^-16; t modulo 2^28, layer < 16, e < 2^31).
constexpr int kRegionDropped = 4;   // region code of a dropped activation
struct DropoutArgs {
    uint64_t seed;
    uint32_t p16;           // 0 = off
    int layer;
    const uint32_t* step;   // device step counter
};
__host__ __device__ __forceinline__ bool dropout_drop(uint64_t seed, uint32_t t, int layer,
                                                      uint64_t e, uint32_t p16) {
    const uint64_t idx = (1ULL << 63) + ((uint64_t)(t & ((1u << 28) - 1)) << 35) +
                         ((uint64_t)layer << 31) + e;
    return (uint32_t)(splitmix64_at(seed, idx) >> 48) < p16;
}

// max|A| * max|B| * k >= 2^63 : int64 exactness of an int32 x int32
// contraction of length k is no longer guaranteed.
__host__ __device__ __forceinline__ bool int64_bound_exceeded(uint32_t ma, uint32_t mb, int64_t k) {
    unsigned __int128 p = (unsigned __int128)ma * mb * (unsigned __int128)k;
    return p >= ((unsigned __int128)1 << 63);
}

// ---------------------------------------------------------------------------
// The signed base-256 split behind the tensor-core operands (bf16 limb planes).
// ---------------------------------------------------------------------------
// Limbs of a tensor with max |x| = m.  The split is canonical: limbs 0..2 are
// the digits ((x + 128) & 255) - 128 of successive base-256 remainders and
// limb 3 takes the rest (in [-128, 128] for int32).  With the thresholds below
// every limb at index >= L is zero, so the first L planes of the 4-limb split
// are exact and producers may write all four without knowing L.
__host__ __device__ __forceinline__ int limb_count(uint32_t m) {
    return m <= 127u ? 1 : (m <= 32639u ? 2 : (m <= 8355711u ? 3 : 4));
}

#ifdef __CUDACC__
// two int8 values v (bytes i, i + 1 of a word whose bytes hold v + 128) -> two bf16:
// 2^23 + (v + 128) is the float 0x4B0000xx, and subtracting 2^23 + 128 leaves v
// exactly, whose upper half is its bf16
__device__ __forceinline__ uint32_t bf16x2(uint32_t biased, int i) {
    const float f0 = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7540 + i)) - 8388736.0f;
    const float f1 = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7541 + i)) - 8388736.0f;
    return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}

// Limb l of two values as two bf16.  Adding 0x808080 moves the digits 0..2 of
// the signed base-256 split into [0, 255] with all their carries at once: byte l of
// the sum is digit l + 128.  Limb 3 is what remains, with the carry of the low
// 24 bits (the sum itself may wrap).
__device__ __forceinline__ uint32_t limb_bf16x2(int32_t a, int32_t b, int l) {
    if (l < 3) {
        const uint32_t ta = (uint32_t)a + 0x808080u, tb = (uint32_t)b + 0x808080u;
        return bf16x2(__byte_perm(ta, tb, l | ((4 + l) << 4)), 0);
    }
    const int32_t da = (a >> 24) + (int32_t)((((uint32_t)a & 0xffffffu) + 0x808080u) >> 24);
    const int32_t db = (b >> 24) + (int32_t)((((uint32_t)b & 0xffffffu) + 0x808080u) >> 24);
    return __byte_perm(__float_as_uint((float)da), __float_as_uint((float)db), 0x7632);
}

#endif

// ---------------------------------------------------------------------------
// Layer geometry as the kernels see it.
// ---------------------------------------------------------------------------
struct LayerGeom {
    int kind;       // NITRO_CONV3X3 / NITRO_LINEAR
    int cin, cout;  // linear: cin = in features, cout = out features
    int h, w;       // input spatial (1 for linear)
    int pool;       // 2x2 max-pool after NITRO-ReLU
    int oh, ow;     // output spatial after the optional pool
};

// Device status word bits (same values as the ABI's NITRO_STATUS_BIT_*).
enum : uint32_t { ST_OVERFLOW = 1u, ST_BAD_LABEL = 2u, ST_TIMEOUT = 4u };

// ---------------------------------------------------------------------------
// CUDA-core kernels (kernels_simt.cu).  All launch on `s`, return the launch
// error, and do nothing for empty problems.
// ---------------------------------------------------------------------------
enum GemmMode : int {
    GM_CONV_FWD = 0,    // C[p][co]      = sum_(t,ci) a[p + tap t][ci] * W[co][t][ci]
    GM_CONV_DGRAD = 1,  // C[p][ci]      = sum_(t,co) g[p - tap t][co] * W[co][t][ci]
    GM_CONV_WGRAD = 2,  // C[co][(t,ci)] = sum_p g[p][co] * a[p + tap t][ci]
    GM_LIN_FWD = 3,     // C[b][o] = sum_i a[b][i] * W[o][i]
    GM_LIN_DGRAD = 4,   // C[b][i] = sum_o g[b][o] * W[o][i]
    GM_LIN_WGRAD = 5    // C[o][i] = sum_b g[b][o] * a[b][i]
};

// Exact int64 implicit GEMM on CUDA cores.  act: int8 activations, grad:
// int32 gradients, wts: int32 weights; out: int64, row-major C (overwritten).
cudaError_t simt_gemm(int mode, const int8_t* act, const int32_t* grad, const int32_t* wts,
                      int64_t* out, int B, int H, int W, int Cin, int Cout, cudaStream_t s);

// Brings the kernels of a conv forward (GEMM, epilogue) onto the current device.
cudaError_t simt_preload_conv_fwd();

// z (int64, pre-pool NHWC) -> NITRO-Scaling -> NITRO-ReLU -> region codes,
// optional 2x2 max-pool with argmax codes, int8 outputs (out2 may be NULL).
// With drop.p16 > 0 (linear layers, no pool) dropped outputs are stored as 0
// with region code kRegionDropped.
cudaError_t simt_fwd_epilogue(const int64_t* z, const LayerGeom& g, int B, int alpha_inv,
                              int mu, int8_t* out, int8_t* out2, int8_t* region,
                              int8_t* argmax, cudaStream_t s, const DropoutArgs* drop = nullptr);

// Learning-layer max-pool (Sec. 3.3, z^mp): a [B][H][W][C] int8 -> out
// [B][ph][pw][C] over kh x kw windows with stride (kh, kw), first maximum in
// row-major window order, its position r*kw + s in am.
cudaError_t simt_lr_pool_fwd(const int8_t* a, int B, int H, int W, int C, int kh, int kw,
                             int ph, int pw, int8_t* out, uint8_t* am, cudaStream_t s);

// delta_fw = grad_l W_lr at the pooled learning features (int32 storage rule,
// int64 bound check), routed back through the learning-layer pool (window
// maximum am), the 2x2 max-pool of conv layer g (argmax) and NITRO-ReLU
// backward into g's delta [B][h][w][cout]; every element is written.  planes (may
// be null): delta's limb planes [4][n], written too where the channel count
// allows (*planes_done); zero[0..n_zero) is then cleared as well.
struct LrPoolGeom {
    int kh, kw, ph, pw;
};
cudaError_t simt_lrpool_to_delta(const int32_t* gl, const int32_t* wlr, int G, int d,
                                 const LayerGeom& g, const LrPoolGeom& lp, int B,
                                 const uint8_t* am, const int8_t* argmax, const int8_t* region,
                                 int alpha_inv, int32_t* delta, uint16_t* planes, int64_t* zero,
                                 int64_t n_zero, bool* planes_done, const uint32_t* maxabs_gl,
                                 const uint32_t* gl_bound, const uint32_t* maxabs_wlr, uint32_t* maxabs_delta,
                                 uint32_t* status, cudaStream_t s);

// Learning layer forward: grad_l = floor(a W^T / (256 d)) - 32 onehot (the limbs of
// W from *maxabs_wlr) and status bits; *gl_bound is raised to the largest sum of |grad_l|
// over a sample's classes (2^32 - 1: that or more), so that times max |W| it bounds
// every sum of grad_l W, and more tightly than classes times max |grad_l|.  The launch
// also clears zero_words[0..n_zero) for the rest of the backward, which saves a memset.
cudaError_t simt_learn_fwd(const int8_t* a, const int32_t* wlr, const int32_t* labels, int B,
                           int d, int G, int32_t* grad_l, const uint32_t* maxabs_wlr,
                           uint32_t* status, uint32_t* zero_words, int n_zero, uint32_t* gl_bound,
                           cudaStream_t s);

// Written by the kernel that follows it (simt_lr_backward): sse =
// sum grad_l^2 (mod 2^64), loss = floor(sse / 2) (may be null), max |grad_l|, and
// OVERFLOW when max |grad_l| *wlr_max G reaches 2^63 (wlr_max null: not checked).
struct LossOut {
    unsigned long long* sse;
    int64_t* loss;
    uint32_t* maxabs_gl;
    uint32_t* ticket;          // sse, maxabs_gl and ticket: zero before (simt_learn_fwd clears them)
    const uint32_t* wlr_max;
    uint32_t* status;
};

// Linear layer on the CUDA cores: the whole forward (scaling, NITRO-ReLU, dropout; the
// limbs of w from *maxabs_w), one launch, and the weight gradient (dw overwritten; with
// many samples or products a clear goes before).  _ok: the layer has few products, or
// no tensor-core form (tc false; the forward of one with many samples and few inputs is
// left to simt_gemm and simt_fwd_epilogue).
bool simt_lin_fwd_ok(const LayerGeom& g, int B, bool tc);
cudaError_t simt_lin_fwd(const int8_t* a, const int32_t* w, const uint32_t* maxabs_w, const LayerGeom& g,
                         int B, int alpha_inv, int mu, int8_t* act, int8_t* out2, int8_t* region,
                         const DropoutArgs* drop, cudaStream_t s);
bool simt_lin_wgrad_ok(const LayerGeom& g, int B, bool tc);
cudaError_t simt_lin_wgrad(const int8_t* a, const int32_t* delta, const LayerGeom& g, int B, int64_t* dw,
                           cudaStream_t s);

// Gradient at the output of layer g (post-pool, an int64 dgrad output) -> delta at its
// pre-activation: max-pool backward, NITRO-ReLU backward, STE.
struct DeltaSrc {
    const uint32_t* maxabs_a;  // bound check operands: max|grad| and max|W|
    const uint32_t* maxabs_b;
    int64_t bound_k;           // contraction length for the bound
    const int64_t* g64;        // [B][out features of the layer]
};
cudaError_t simt_grad_to_delta(const DeltaSrc& src, const LayerGeom& g, int B, int alpha_inv,
                               const int8_t* region, const int8_t* argmax, int32_t* delta,
                               uint32_t* maxabs_delta, uint32_t* status, cudaStream_t s);

// Learning-layer backward: dW_lr (overwritten), the loss (see LossOut) and, with dl !=
// null, the delta of the block's last forward layer (geometry lg) from delta_fw =
// grad_L W_lr (pre-update), with the int32 storage rule, max-pool and NITRO-ReLU
// backward.  dl->planes (may be null): delta's limb planes [4][n], written too where the
// layout allows (*planes_done), and zero[0..n_zero) is then cleared as well.  d:
// features of the learning layer; gl_bound: see simt_learn_fwd.
struct LrDelta {
    const LayerGeom* lg;
    int alpha_inv;
    const int8_t* region;
    const int8_t* argmax;
    int32_t* delta;
    uint16_t* planes;
    int64_t* zero;
    int64_t n_zero;
    bool* planes_done;
    const uint32_t* maxabs_wlr;
    uint32_t* maxabs_delta;
};
cudaError_t simt_lr_backward(const int8_t* a, const int32_t* gl, const uint32_t* gl_bound, const int32_t* wlr,
                             int B, int G, int d, int64_t* dwlr, const LrDelta* dl, uint32_t* status, const LossOut& lo,
                             cudaStream_t s);

// IntegerSGD (Algorithm 1) over up to kMaxSgdTensors tensors in one launch.
constexpr int kMaxSgdTensors = 16;
struct SgdTensor {
    int32_t* w;
    const int64_t* dw;
    int64_t n;
    int64_t gamma_inv, eta_inv;
    uint32_t* maxabs_w;
    // dividers for gamma_inv and eta_inv (filled by simt_integersgd): 64-bit gradients,
    // gradients that fit 32 bits, weights
    FloorDiv gdiv;
    FloorDiv32 gdiv32, ediv32;
    // optional bf16 limb planes of a conv weight [Cout][9][cin] that the update
    // keeps itself: planes[l plane + co row_k + t tap_k + ci].  They hold all four
    // limbs of W before and after (so that only what changes is stored)
    uint16_t* planes;
    int64_t plane;
    int row_k, tap_k, cin;
    FloorDiv32 cin_div;    // filled by simt_integersgd
    bool contig;           // planes laid out like W (filled by simt_integersgd)
};
struct SgdBatch {
    SgdTensor t[kMaxSgdTensors];
    int count;
    int round_trunc;
    uint32_t* status;
    uint32_t* step;        // block step counter, incremented once per launch (or null)
    // kMaxSgdTensors maxima, a CTA ticket and the step's bound of |grad_L| (see
    // simt_learn_fwd), zero before the first launch and left zero by every launch: the
    // last CTA stores the finished maxima into
    // each tensor's maxabs_w and copies words[0..n_words) to host_words (pinned
    // host memory; null: no copy)
    uint32_t* scratch;
    const uint32_t* words;
    uint32_t* host_words;
    int n_words;
    int first[kMaxSgdTensors + 1];   // first CTA of each tensor (filled by simt_integersgd)
};
constexpr int kSgdScratchWords = kMaxSgdTensors + 2;
cudaError_t simt_integersgd(const SgdBatch& b, cudaStream_t s);


// ---------------------------------------------------------------------------
// A kernel's attributes belong to one device.  f() runs until it succeeds once for
// each device dev that calls are made on (a bit of `done` each; two host threads that
// meet may both run it).
// ---------------------------------------------------------------------------
constexpr int kMaxDevices = 64;
template <typename F>
inline cudaError_t once_per_device(std::atomic<uint64_t>& done, int dev, F&& f) {
    const uint64_t bit = dev >= 0 && dev < kMaxDevices ? (uint64_t)1 << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    const cudaError_t e = f();
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// Clears n bytes on s the first time that a handle runs; its kernels keep them clean from
// then on.  (A clear at creation would queue on the default stream, and could still be
// waiting there when the handle is used on another; a stream of its own to wait for
// costs 50 us a handle.)  A captured call holds the clear too and does not count as the
// first: its graph need not have run before the next call.
inline cudaError_t clear_once(bool& clean, void* p, size_t n, cudaStream_t s) {
    if (clean) return cudaSuccess;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &capture);
    if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, n, s);
    if (e == cudaSuccess && capture == cudaStreamCaptureStatusNone) clean = true;
    return e;
}

// ---------------------------------------------------------------------------
// Programmatic dependent launch.  A kernel queued with launch_k may start
// (get SMs, set up shared memory, barriers and TMEM) while the kernel before
// it in the stream is still finishing; every kernel so queued executes
// pdl_wait() in each thread before its first access to global memory, which
// blocks until the previous kernel has completed and its writes are visible.
// pdl_trigger() lets the next kernel of the stream start launching; it only
// takes effect once every CTA of this kernel has executed it or exited.
// Both are no-ops for a kernel queued without the attribute.  Only the
// contraction kernel triggers, once its MMAs are issued: an early trigger
// lets the next kernel's waiting CTAs hold SMs that kernels of the other
// block streams would use (measured slower on the VGG-style step), and the
// other kernels trigger implicitly when their CTAs exit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Whether launch_k queues kernels with the programmatic-serialization
// attribute (on unless the environment sets NITRO_PDL=0; read once).
bool pdl_enabled();

template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                            cudaStream_t s, Args&&... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// launch_k with clusters of `cluster` CTAs along x.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, int block, int cluster,
                                  cudaStream_t s, size_t smem, Args&&... args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace nitro
