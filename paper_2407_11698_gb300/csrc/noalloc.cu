// Forward of one 3x3 conv layer that performs no device allocation.
//
// Some callers cannot call cudaMalloc once they are running: code embedded in
// a host program that owns the whole device-memory budget (a serving process
// or game engine with its own arena), real-time loops where allocation after
// start-up is not allowed, and code that must not stall the device (cudaMalloc
// and cudaFree may synchronise it).  For them this entry point runs one conv
// layer's forward on the kernels that nitro_block_forward uses (same results),
// but keeps what they need between them in a fixed array that is part of the
// library image instead of in a block's workspace: the tensor-core forward's
// bf16 operands, or, for layers off the tensor path and operands that do not
// fit, the int64 pre-activations of the CUDA-core kernels.
//
// The array is a file-scope __device__ variable: every GPU that loads the
// library holds kNoallocScratchElems * 8 bytes (16 MiB) until the process
// exits.  Host code cannot use its name as a device address, so on the first
// call on each device the entry point looks the address up with
// cudaGetSymbolAddress (with that device current) and caches it for the life
// of the process; a cudaDeviceReset of that device is therefore not supported
// between calls.
#include <mutex>

#include "nitro_internal.cuh"
#include "tc_conv.cuh"

namespace {

constexpr int64_t kNoallocScratchElems = (int64_t)1 << 21;   // int64 values

// Products from which a layer with 9 Cin <= 64 runs on the tensor cores, as three
// launches (12.7 us, host bound) instead of two: 1 x 28 x 28, 1 -> 32 channels (0.2 M
// products) takes 13.1 us there and 10.0 us on the CUDA cores, 121 x 12 x 4, 2 -> 24 (2.5 M)
// 12.5 and 10.7 us, 16 x 28 x 28, 3 -> 64 (22 M) 12.9 and 21.4 us.  Layers with more channels
// do unless the map is a line that fills an eighth of a tile with a quarter of its channels:
// 1 x 8 x 8, 16 -> 16 (0.15 M) 12.7 against 26.1 us, 8 x 16 x 16, 64 -> 64 13.1 against 41.2 us,
// but 64 x 1 x 62, 12 -> 240 62 against 43 us.
constexpr int64_t kNoallocTcMacs = (int64_t)1 << 22;

static __device__ __align__(256) int64_t g_noalloc_scratch[kNoallocScratchElems];
static __device__ uint32_t g_noalloc_words[4];     // see tc_fwd_in_scratch
constexpr int kStatusWord = 3;                     // latched TIMEOUT

struct Scratch {
    int64_t* z = nullptr;
    uint32_t* words = nullptr;
};
std::mutex g_mu;
Scratch g_scratch_addr[nitro::kMaxDevices];

// Device addresses of the arrays for the current device, looked up once; the first
// look-up also loads the kernels, so that no later call takes memory for them.
cudaError_t scratch_for_current_device(Scratch* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= nitro::kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_addr[dev].z) {
        void *p = nullptr, *w = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e == cudaSuccess) e = cudaGetSymbolAddress(&w, g_noalloc_words);
        if (e == cudaSuccess) e = nitro::tc_fwd_preload();
        if (e == cudaSuccess) e = nitro::simt_preload_conv_fwd();
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev].words = static_cast<uint32_t*>(w);
        g_scratch_addr[dev].z = static_cast<int64_t*>(p);
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace

using namespace nitro;

extern "C" nitro_status nitro_conv3x3_forward_noalloc(
    const int8_t* a_in, const int32_t* weights, int batch, int h, int w, int cin, int cout,
    int pool2x2, int alpha_inv, int8_t* a_out, int8_t* region, int8_t* argmax, void* stream) {
    if (batch < 0 || h < 1 || w < 1 || cin < 1 || cout < 1 || cin > (1 << 20) ||
        (pool2x2 != 0 && pool2x2 != 1) || alpha_inv < 2 || alpha_inv > (1 << 20))
        return NITRO_ERR_ARG;
    if (pool2x2 && (h < 2 || w < 2)) return NITRO_ERR_ARG;
    const int64_t elems = (int64_t)batch * h * w * cout;
    if (elems > kNoallocScratchElems) return NITRO_ERR_ARG;   // larger than the fixed array
    if (batch == 0) return NITRO_OK;
    if (!a_in || !weights || !a_out || !region || (pool2x2 && !argmax)) return NITRO_ERR_ARG;
    Scratch sc;
    if (scratch_for_current_device(&sc) != cudaSuccess) return NITRO_ERR_CUDA;
    int64_t* z = sc.z;
    cudaStream_t s = (cudaStream_t)stream;
    LayerGeom g{NITRO_CONV3X3, cin, cout, h, w, pool2x2, pool2x2 ? h / 2 : h, pool2x2 ? w / 2 : w};
    // mu_int8 of NITRO-ReLU: floor-average of the four segment means
    const int mu = (int)fdiv64(fdiv64(-127, alpha_inv) + fdiv64(-127, 2 * alpha_inv) + 63 + 127, 4);
    // the tensor-core forward, if its operands fit the array and its 8-byte stores the
    // outputs
    const size_t need = tc_fwd_scratch(g, batch);
    const uintptr_t low = (uintptr_t)a_out | (uintptr_t)region | (pool2x2 ? (uintptr_t)argmax : 0);
    if (need && need <= sizeof(int64_t) * (size_t)kNoallocScratchElems && (low & 7) == 0 &&
        (9 * cin > 64 ? cin >= 16 || (h > 1 && w > 1) : elems * 9 * cin >= kNoallocTcMacs)) {
        const TcFwdOut fo{alpha_inv, mu, a_out, nullptr, region, pool2x2 ? argmax : nullptr, nullptr};
        return tc_fwd_in_scratch(g, batch, a_in, weights, fo, z, sc.words, s) == cudaSuccess ? NITRO_OK
                                                                                            : NITRO_ERR_CUDA;
    }
    // The GEMM overwrites every element of z (directly, or by clearing it
    // before adding K-split partial sums), so the array needs no clearing here.
    if (simt_gemm(GM_CONV_FWD, a_in, nullptr, weights, z, batch, h, w, cin, cout, s) != cudaSuccess)
        return NITRO_ERR_CUDA;
    if (simt_fwd_epilogue(z, g, batch, alpha_inv, mu, a_out, nullptr, region, argmax, s) !=
        cudaSuccess)
        return NITRO_ERR_CUDA;
    return NITRO_OK;
}

extern "C" nitro_status nitro_conv3x3_noalloc_status(int clear) {
    Scratch sc;
    if (scratch_for_current_device(&sc) != cudaSuccess) return NITRO_ERR_CUDA;
    uint32_t bits = 0;
    uint32_t* word = sc.words + kStatusWord;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(&bits, word, sizeof(bits), cudaMemcpyDeviceToHost) != cudaSuccess)
        return NITRO_ERR_CUDA;
    if (clear && (cudaMemset(word, 0, sizeof(bits)) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess))
        return NITRO_ERR_CUDA;
    return bits & ST_TIMEOUT ? NITRO_ERR_TIMEOUT : NITRO_OK;
}
