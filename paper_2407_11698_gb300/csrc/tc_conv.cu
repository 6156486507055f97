// tcgen05 implicit-GEMM kernels for the 3x3 conv forward, weight gradient
// and input gradient, plus the kernels that split operands into bf16 limb
// planes.  See tc_conv.cuh for the exactness argument and the layouts.
//
// A persistent CTA computes 128 x N output tiles, each over a range of
// K-blocks (64 elements each).  Warp 0 issues TMA loads into an S-stage shared-memory ring,
// warp 1 allocates TMEM and issues the MMAs, warps 4..19 drain the fp32 TMEM
// accumulator every <= 16 K-blocks into int64 registers (the fused forward and input
// gradient: into the sum modulo 2^32 and an fp32 sum; four warps per TMEM lane
// quadrant, each owning a quarter of the N columns).  Four TMEM accumulators
// rotate so the MMAs run up to three chunks ahead of the drain.
// Every wait on an mbarrier is bounded in time; on expiry the kernel raises
// the TIMEOUT status bit, lets the other roles leave, frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "prof.cuh"
#include "tc_conv.cuh"

namespace nitro {
namespace {

// TC_FWD: forward with the fused NITRO-Scaling / NITRO-ReLU / max-pool epilogue;
// TC_FWDK: the same with a tile's K shared out over a cluster; TC_FWDD: linear layers
// with dropout, either way; TC_DGRAD: input gradient
// with the fused routing into the lower layer's delta; TC_FWDZ, TC_DGRADZ: the same
// contractions with int64 sums as their output.
enum TcMode : int { TC_FWD = 0, TC_WGRAD = 1, TC_DGRAD = 2, TC_GEMM = 3, TC_FWDZ = 4, TC_FWDK = 5, TC_DGRADZ = 6, TC_FWDD = 7 };

constexpr int kBM = 128;              // rows per tile (TMEM lanes)
constexpr int kBK = 64;               // K elements per block (one 128-byte row)
constexpr int kChunkBlocks = 16;      // 16 x 64 = 1024 products per exact chunk
// Warp roles: warpgroup 0 = TMA warp, MMA warp and two idle warps; warpgroups
// 1 to 4 = the epilogue, four warps per TMEM lane quadrant, each holding a
// quarter of the N columns.  The epilogue is bound by latency, so it gets as many
// warps as the register file allows; the warpgroups split it with setmaxnreg: 128
// x kRegsProducer + 32 x kEpiWarps x kRegsEpilogue must not exceed kThreads x the
// registers the kernel is launched with (checked on the host before the first
// launch).  64 / 104 with TMEM loads of 8 columns (16 where a warp holds 16) spills
// nothing in the forward, GEMM and kernel-level variants: at 32 / 112 the TMA and
// MMA warps reloaded spilled values on their per-K-block path, which the small L1
// beside 227 KB of shared memory does not hold (VGG11B forward at batch 256 1154 us,
// now 1098; 4096^3 GEMM 264, now 247; conv contractions 784, now 751).  Eight
// epilogue warps (half the N columns each, 224 registers) were slower.
constexpr int kEpiWarp0 = 4;          // first epilogue warp
constexpr int kEpiWarps = 16;         // 4 per TMEM lane quadrant
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
constexpr int kRegsProducer = 64, kRegsEpilogue = 104;
constexpr int kTabHalf = 256;         // half the fused forward's table of z*
// K-blocks of a fused forward (Cin <= 896): with four weight limbs and eight chunks
// its fp32 sums are off by less than 2^24 1.02 8 (8 + 4.2) = 1.67e9, so that the
// remainder taken modulo 2^32 is exact
constexpr int kFwdMaxBlocks = 128;
constexpr uint64_t kWaitNs = 2000000000ull;   // 2 s bound on any wait

// ------------------------------------------------------------------ PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait: false when the time limit passed (TIMEOUT raised) or another
// role of this CTA gave up.  Inlined: a function call cannot sit inside the
// register-split (setmaxnreg) regions of the contraction kernel.
__device__ __forceinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                            uint32_t* status, uint64_t limit_ns) {
    const uint64_t t0 = global_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63) == 0) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                atomicOr(status, ST_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          uint32_t* status, uint64_t limit_ns = kWaitNs) {
    return mbar_try_wait(bar, parity) || mbar_wait_slow(bar, parity, abort_flag, status, limit_ns);
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2, int c3, int c4) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(c4)
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor, K-major operand, 128-byte swizzle: rows of
// 128 bytes, 8-row groups 1024 bytes apart (stride byte offset), version 1.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;               // leading byte offset (unused here)
    d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset
    d |= (uint64_t)1 << 46;               // descriptor version
    d |= (uint64_t)2 << 61;               // 128-byte swizzle
    return d;
}

// MN-major operand, 128-byte swizzle: rows of 128 bytes run along K, each
// holding 64 consecutive M (or N) elements; 64-element blocks along M/N lie
// `mn_stride` bytes apart (leading byte offset), 8-row groups along K 1024
// bytes apart (stride byte offset).
__device__ __forceinline__ uint64_t desc_sw128_mn(uint32_t saddr, uint32_t mn_stride) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((mn_stride >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor: kind::f16, A = B = bf16, D = f32; A (bit 15) and B
// (bit 16) K-major unless marked MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n, bool a_mn = false, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn ? (1u << 15) : 0u) | (b_mn ? (1u << 16) : 0u) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr));
}

// Wait for this thread's outstanding tcgen05.ld, then mark the n destination
// registers as written here, so that no use of them is placed before the wait.
__device__ __forceinline__ void reg_touch8(uint32_t* r) {
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]));
}
template <int n>
__device__ __forceinline__ void tmem_wait_ld(uint32_t* r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < n / 8; ++j) reg_touch8(r + 8 * j);
}

// ------------------------------------------------------------------ kernel
struct TcArgs {
    int B, H, W, Cin, Cout;
    int cin_k;             // channels per tap in the K index (Cin rounded up to 64)
    int taps;              // 9, or 1 for im2col input (forward / wgrad: no tap shift)
    int ntx, nty;          // pixel tiles along x and y (forward / dgrad)
    int wb, hb, bb;        // pixel box (forward / dgrad): wb * hb * bb = 128
    int tiles_m, tiles_n, total_tiles;
    // dividers for the tile decode (filled at launch): tiles_n, tiles_m, ntx, nty;
    // pixel-box sides are powers of two: log2 wb, log2 hb
    FloorDiv32 dv_tn, dv_tm, dv_ntx, dv_nty;
    int lg_wb, lg_hb;
    int kb_total, kb_per_split;
    int ncols;             // valid output columns (Cout for fwd/wgrad, Cin for dgrad)
    const uint32_t* max_a;  // max |operand| words setting the limb counts (nullptr = 1 limb)
    const uint32_t* max_b;
    int64_t* out;
    uint32_t* status;
    int atomic_out;
    int out_vec;           // int64 values a store: 4 (rows 32-byte aligned), 2 (16) or 1
    int ksplit;            // fused forward: CTAs of a cluster that share a tile's K (1: none)
    // forward with fused NITRO-Scaling / NITRO-ReLU / max-pool epilogue
    FloorDiv alpha;        // divide by alpha_inv
    int32_t sf;            // SF = 2^8 9 Cin
    float sf_inv;          // 1 / SF
    int out_align;         // outputs and their rows are aligned to 32, 16 or 8 bytes
    int mu, pool, oh, ow;
    DropoutArgs drop;      // TC_FWDD
    int8_t* act;           // layer output (post-pool) int8 NHWC
    int8_t* out2;          // optional second copy of the output (caller's buffer)
    int8_t* region;        // NITRO-ReLU piece per pre-pool output
    int8_t* argmax;        // window position per pooled output
    uint16_t* next_nhwc;   // bf16 copy of the output for the next layer's forward, or null
    // dgrad with fused max-pool / NITRO-ReLU backward into the lower layer's delta
    FloorDiv32 alpha32;
    const uint32_t* bound_a;   // max|delta| and max|W| of this layer (int64 exactness bound)
    const uint32_t* bound_b;
    int low_h, low_w, low_pool;
    const int8_t* low_region;
    const int8_t* low_argmax;
    int32_t* low_delta;
    uint32_t* low_maxabs;
    // weight gradient: valid rows (taps == 1) and the row stride of dW / W
    int rows;
    int64_t cstride;
    // weight gradient with IntegerSGD applied to the finished sums (no K split)
    int sgd;
    int32_t* wt;               // the layer's weights [Cout][9][Cin]
    uint16_t* wp;              // weight limb planes [4][Cout][row_k], or null
    int64_t w_plane;
    int row_k, tap_k;
    FloorDiv gdiv, ediv;       // gamma_inv, eta_inv (eta_inv = 0: no decay)
    int decay, trunc;
    uint32_t* maxabs_w;        // max |new W| (atomic max, zeroed by the caller)
};

// Cluster-wide barrier, and shared memory of another CTA of the cluster.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t remote_smem(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}

// 8 int8 values (2 packed words) -> one 8-byte store
__device__ __forceinline__ void st8(int8_t* dst, const uint32_t* w) {
    *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
}
// 16 int8 values (4 packed words) -> one 16-byte store
__device__ __forceinline__ void st16(int8_t* dst, const uint32_t* w) {
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}
// eight words, one 32-byte store
__device__ __forceinline__ void st_u32x8(void* dst, const uint32_t* w) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(w[0]),
                 "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
// all bits of the word set where byte e of a byte mask is
__device__ __forceinline__ int32_t byte_mask(uint32_t mask, int e) {
    return (int32_t)__byte_perm(mask, 0, 0x8888u + 0x1111u * (uint32_t)e);
}
// 32 int8 values (8 packed words): one 32-byte store (a whole sector) when the
// destination is 32-byte aligned, else two of 16 bytes
__device__ __forceinline__ void st32(int8_t* dst, const uint32_t* w, bool aligned32) {
    if (aligned32) {
        st_u32x8(dst, w);
    } else {
        st16(dst, w);
        st16(dst + 16, w + 4);
    }
}
// four int64 values, one 32-byte store (a whole sector): the 16-byte stores before
// it wrote half sectors, each a transaction of its own in L2
__device__ __forceinline__ void st_i64x4(int64_t* dst, const uint64_t* v) {
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "l"(v[0]), "l"(v[1]), "l"(v[2]),
                 "l"(v[3])
                 : "memory");
}
// larger of each pair of signed 16-bit halves
__device__ __forceinline__ uint32_t max_s16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.s16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// 16 int8 values (4 packed words) -> 16 bf16 values, packed
__device__ __forceinline__ void cvt16_bf16(uint32_t* o, const uint32_t* w) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t u = w[k] ^ 0x80808080u;
        o[2 * k] = bf16x2(u, 0);
        o[2 * k + 1] = bf16x2(u, 2);
    }
}
// 8 int8 values (2 packed words) -> 8 bf16 values, one 16-byte store
__device__ __forceinline__ void st8_bf16(uint16_t* dst, const uint32_t* w) {
    const uint32_t u = w[0] ^ 0x80808080u, v = w[1] ^ 0x80808080u;
    *reinterpret_cast<uint4*>(dst) = make_uint4(bf16x2(u, 0), bf16x2(u, 2), bf16x2(v, 0), bf16x2(v, 2));
}

// PB = B-operand limbs carried per stage: one A tile feeds PB limb tiles of B
// and PB accumulators, so wide B operands do not re-stream A once per limb.
template <int N, int PB>
struct TcCfg {
    static constexpr int A_BYTES = kBM * kBK * 2;
    static constexpr int B_BYTES = N * kBK * 2;
    static constexpr int STAGE = A_BYTES + PB * B_BYTES;
    static constexpr int S_FIT = (230912 - 1536) / STAGE;   // ~225 KB of shared memory
    // at most 6 stages: deeper rings gave no gain in the training step and lost
    // up to 14% in the kernel-level contractions (more TMA writes in flight
    // compete with the MMA's shared-memory reads)
    static constexpr int S = S_FIT > 6 ? 6 : S_FIT;
    static constexpr int SMEM = 1024 + S * STAGE + 2048;   // alignment, ring, barriers and table
    static constexpr int NBUF = (512 / (PB * N)) > 4 ? 4 : (512 / (PB * N));   // accumulator sets
    static constexpr int TCOLS = NBUF * PB * N;                                  // 256 or 512
};

struct Tile {
    int mt, nt, kb0, kb1;
};
__device__ __forceinline__ int udiv32(const FloorDiv32& f, int x) { return (int)f.udiv((uint32_t)x); }

__device__ __forceinline__ Tile decode_tile(const TcArgs& a, int tile) {
    Tile t;
    const int r = udiv32(a.dv_tn, tile);
    t.nt = tile - r * a.tiles_n;
    const int split = udiv32(a.dv_tm, r);
    t.mt = r - split * a.tiles_m;
    t.kb0 = min(a.kb_total, split * a.kb_per_split);
    t.kb1 = min(a.kb_total, t.kb0 + a.kb_per_split);
    return t;
}

// Persistent: CTA c handles tiles c, c + gridDim.x, ...; the TMA ring, the
// MMA chunk sequence and the TMEM accumulators (up to four) run on across tiles, so
// one tile's epilogue overlaps the next tile's loads and MMAs.
template <int MODE, int N, int PB>
__global__ void __launch_bounds__(kThreads, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const TcArgs args) {
    using C = TcCfg<N, PB>;
    constexpr int S = C::S;
    constexpr int NH = N / 4;            // columns per epilogue warp
    constexpr bool kSplitK = MODE == TC_FWDK || MODE == TC_FWDD;
    constexpr bool kFused = MODE == TC_FWD || kSplitK;
    constexpr bool kFwd = kFused || MODE == TC_FWDZ;
    constexpr bool kDgrad = MODE == TC_DGRAD || MODE == TC_DGRADZ;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * C::STAGE);
    // bars[0..S) full, [S..2S) empty, then NBUF tmem-full and NBUF tmem-empty
    constexpr int NBUF = C::NBUF;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 2 * NBUF);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* hiskip_slot = reinterpret_cast<int*>(tmem_slot + 2);
    // fused forward: NITRO-ReLU value (high byte) and piece (low byte) of every
    // z* in [-kTabHalf, kTabHalf), at index z* + kTabHalf
    uint16_t* relu_tab = reinterpret_cast<uint16_t*>(smem + S * C::STAGE + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * S + NBUF + b); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < NBUF; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), kEpiWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (kFused) {
        for (int i = threadIdx.x; i < 2 * kTabHalf; i += kThreads) {
            const int zs = i - kTabHalf;
            relu_tab[i] = (uint16_t)((uint32_t)(uint8_t)relu_value((int64_t)zs, args.alpha, args.mu) << 8 |
                                     (uint32_t)relu_region(zs));
        }
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(C::TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
    }
    // The set-up above touches only shared memory, TMEM and the kernel's own
    // tensor maps, so it may overlap the end of the previous kernel in the
    // stream; from here on the kernel reads what that kernel wrote.
    pdl_wait();
    if (threadIdx.x == 0) {
        // Fused input gradient: the lower delta is stored as the low 32 bits of
        // the exact sum, and limb pairs with la + lb >= 4 only add multiples
        // of 2^32.  They matter only for deciding OVERFLOW, so once that bit
        // is latched they are skipped.  Read once per CTA so that all roles
        // walk the same passes (CTAs may differ; each result is the same).
        *hiskip_slot = MODE == TC_DGRAD
            ? ((*reinterpret_cast<volatile uint32_t*>(args.status) & ST_OVERFLOW) != 0) : 0;
    }
    // int32 x int32 contraction: flag when max|delta| max|W| 9 Cout >= 2^63
    if (MODE == TC_DGRAD && blockIdx.x == 0 && threadIdx.x == 64 &&
        int64_bound_exceeded(*args.bound_a, *args.bound_b, 9LL * args.Cout))
        atomicOr(args.status, ST_OVERFLOW);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const int LA = args.max_a ? limb_count(*args.max_a) : 1;
    const int LB = args.max_b ? limb_count(*args.max_b) : 1;
    const int hiskip = *hiskip_slot;
    // Tiles of this CTA: every gridDim.x-th one, or, where a cluster shares a tile's K
    // (the ranks are the splits), one.
    const int KS = kSplitK ? args.ksplit : 1;
    const bool shared_k = MODE == TC_FWDK || (MODE == TC_FWDD && KS > 1);
    const int rank = shared_k ? (int)cluster_rank() : 0;
    const int tile0 =
        shared_k ? rank * (args.tiles_m * args.tiles_n) + (int)blockIdx.x / KS : (int)blockIdx.x;
    const int tile_step = shared_k ? args.total_tiles : (int)gridDim.x;
    // B limbs that pair with A limb la: all, or those with la + lb <= 3
    auto lb_limit = [&](int la) { return hiskip ? min(LB, 4 - la) : LB; };

    if (warp < kEpiWarp0) {
    // warpgroup 0 gives registers back, then splits into its roles
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsProducer));
    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer
            int it = 0;
            for (int tile = tile0; tile < args.total_tiles; tile += tile_step) {
                const Tile T = decode_tile(args, tile);
                const int n0 = T.nt * N;
                const int mq = udiv32(args.dv_ntx, T.mt), tb = udiv32(args.dv_nty, mq);
                const int tx = T.mt - mq * args.ntx, ty = mq - tb * args.nty;
                const int x0 = tx * args.wb, y0 = ty * args.hb, b0 = tb * args.bb;
                // weight gradient: the tile's two 64-row blocks of (tap, ci) rows
                // are fixed for the tile (channel start, tap offsets)
                int wa_ci[2] = {0, 0}, wa_dx[2] = {0, 0}, wa_dy[2] = {0, 0};
                if (MODE == TC_WGRAD) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int m = T.mt * kBM + j * 64;
                        int t = m / args.cin_k, ci0 = m - t * args.cin_k;
                        if (t >= args.taps) { t = 0; ci0 = args.cin_k; }   // past the last tap: zeros
                        if (args.taps == 1) t = 4;                         // im2col rows: centre tap
                        wa_ci[j] = ci0;
                        wa_dx[j] = t % 3 - 1;
                        wa_dy[j] = t / 3 - 1;
                    }
                }
                for (int la = 0; la < LA; ++la)
                for (int lb0 = 0; lb0 < lb_limit(la); lb0 += PB) {
                    const int nb = min(PB, lb_limit(la) - lb0);
                    // weight gradient: K-block kb = pixel box (xt, yt) of image bk,
                    // walked incrementally
                    int wxt = 0, wyt = 0, wbk = 0;
                    if (MODE == TC_WGRAD) {
                        wxt = T.kb0 % args.ntx;
                        wyt = (T.kb0 / args.ntx) % args.nty;
                        wbk = T.kb0 / (args.ntx * args.nty);
                    }
                    // forward / input gradient: K-block kb = (tap t, 64-channel block cb),
                    // cb fastest, walked incrementally
                    const int knc = kFwd ? args.cin_k / kBK : (args.Cout + kBK - 1) / kBK;
                    int kt = 0, kcb = 0;
                    if (kFwd || kDgrad) {
                        kt = T.kb0 / knc;
                        kcb = T.kb0 - kt * knc;
                    }
                    for (int kb = T.kb0; kb < T.kb1; ++kb, ++it) {
                        const int s = it % S;
                        if (!mbar_wait(empty_bar(s), ((it / S) & 1) ^ 1, abort_flag, args.status))
                            goto producer_done;
                        const uint32_t fb = full_bar(s);
                        const uint32_t a_dst = smem_u32(smem + s * C::STAGE);
                        const uint32_t b_dst = a_dst + C::A_BYTES;
                        // the B box spans PB limb planes (past the last limb: zeros or
                        // planes the MMA does not read)
                        mbar_expect_tx(fb, C::A_BYTES + (MODE == TC_GEMM ? nb : PB) * C::B_BYTES);
                        if (MODE == TC_GEMM) {
                            tma_load_2d(a_dst, &tmA, fb, kb * kBK, T.mt * kBM);
                            for (int j = 0; j < nb; ++j)
                                tma_load_3d(b_dst + j * C::B_BYTES, &tmB, fb, kb * kBK, n0, lb0 + j);
                        } else if (kFwd) {
                            const int t = kt, cb = kcb;
                            const int tc = args.taps == 1 ? 4 : t;   // im2col rows: centre tap
                            const int ky = tc / 3, kx = tc - 3 * ky;
                            tma_load_4d(a_dst, &tmA, fb, cb * kBK, x0 + kx - 1, y0 + ky - 1, b0);
                            // PB limb tiles [limb][N rows][64 k], one box
                            tma_load_3d(b_dst, &tmB, fb, t * args.cin_k + cb * kBK, n0, lb0);
                            if (++kcb == knc) { kcb = 0; ++kt; }
                        } else if (kDgrad) {
                            const int t = kt, cb = kcb, ky = t / 3, kx = t - 3 * ky;
                            if (++kcb == knc) { kcb = 0; ++kt; }
                            tma_load_5d(a_dst, &tmA, fb, cb * kBK, x0 - kx + 1, y0 - ky + 1, b0, la);
                            // B MN-major from the forward planes [L][Cout][9][Cin64]:
                            // rows co (K) of 64 consecutive ci (N) for tap t; one box per
                            // 64-channel block h brings PB limbs, stored [h][limb]
#pragma unroll
                            for (int h = 0; h < N / 64; ++h)
                                tma_load_4d(b_dst + h * (PB * 64 * 128), &tmB, fb, n0 + 64 * h, t,
                                            cb * kBK, lb0);
                        } else {  // TC_WGRAD: rows (tap, ci), K = a 64-pixel box (wb x hb)
                            // of one image; both operands MN-major from the NHWC
                            // copies (channels contiguous), the tap shift on x / y.
                            const int px = wxt * args.wb, py = wyt * args.hb, bk = wbk;
#pragma unroll
                            for (int j = 0; j < 2; ++j)
                                tma_load_4d(a_dst + j * (64 * 128), &tmA, fb, wa_ci[j], px + wa_dx[j],
                                            py + wa_dy[j], bk);
                            // one box per 64-channel block h brings PB limbs, stored [h][limb]
#pragma unroll
                            for (int h = 0; h < N / 64; ++h)
                                tma_load_5d(b_dst + h * (PB * 64 * 128), &tmB, fb, n0 + 64 * h, px,
                                            py, bk, lb0);
                            if (++wxt == args.ntx) {
                                wxt = 0;
                                if (++wyt == args.nty) {
                                    wyt = 0;
                                    ++wbk;
                                }
                            }
                        }
                    }
                }
            }
        producer_done:;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---------------- MMA issuer
            // the nb limb tiles of B lie back to back in shared memory and their
            // accumulators side by side in TMEM: one MMA of width nb * N covers them
            uint32_t idesc_nb[PB + 1];
#pragma unroll
            for (int j = 1; j <= PB; ++j)
                idesc_nb[j] = idesc_bf16(kBM, j * N, MODE == TC_WGRAD, MODE == TC_WGRAD || kDgrad);
            // K-major: a K-step of 16 is 32 bytes along each row; MN-major: 16
            // rows, two 1024-byte row groups, and 64-wide blocks along M / N 8 KB
            // apart.  Only the address field (bytes / 16, below 2^14 since shared
            // memory is below 256 KB) moves per K-step and per ring stage, so the
            // descriptors of stage 0 are built once and offset per K-block.
            constexpr bool a_mn = MODE == TC_WGRAD;
            constexpr bool b_mn = MODE == TC_WGRAD || kDgrad;
            constexpr uint32_t kStepA = a_mn ? 2048 / 16 : 32 / 16;
            constexpr uint32_t kStepB = b_mn ? 2048 / 16 : 32 / 16;
            constexpr uint32_t kStageD = C::STAGE / 16;
            const uint32_t s0 = smem_u32(smem);
            const uint64_t da_base = a_mn ? desc_sw128_mn(s0, 64 * 128) : desc_sw128(s0);
            int st = 0;          // ring stage of the next K-block
            uint32_t ph = 0;     // and the parity of the phase it waits for
            int chunk = 0;
            for (int tile = tile0; tile < args.total_tiles; tile += tile_step) {
                const Tile T = decode_tile(args, tile);
                // chunks of equal length (at most kChunkBlocks K-blocks each), so
                // that no short chunk costs a full drain for little MMA work
                const int cpp = (T.kb1 - T.kb0 + kChunkBlocks - 1) / kChunkBlocks;
                const int csz = cpp ? (T.kb1 - T.kb0 + cpp - 1) / cpp : 0;
                for (int la = 0; la < LA; ++la)
                for (int lb0 = 0; lb0 < lb_limit(la); lb0 += PB) {
                    const int nb = min(PB, lb_limit(la) - lb0);
                    // one MMA of width nb * N over the pass's limb tiles.  MN-major B
                    // holds [64-channel block h][PB limbs] in 8 KB blocks: the first
                    // nb limbs of a 64-wide tile are adjacent; with two channel blocks
                    // and nb < PB the used blocks are PB * 8 KB apart (leading byte
                    // offset), and their accumulators land side by side.
                    const uint32_t idesc = idesc_nb[nb];
                    const uint32_t b_lbo = (N > 64 && nb < PB) ? PB * 64 * 128 : 64 * 128;
                    const uint64_t db_base = b_mn ? desc_sw128_mn(s0 + C::A_BYTES, b_lbo)
                                                  : desc_sw128(s0 + C::A_BYTES);
                    for (int c = 0; c < cpp; ++c, ++chunk) {
                        const int buf = chunk % NBUF;
                        if (!mbar_wait(tempty_bar(buf), ((chunk / NBUF) & 1) ^ 1, abort_flag,
                                       args.status))
                            goto mma_done;
                        tc_fence_after();
                        const uint32_t d = tmem + (uint32_t)(buf * PB * N);
                        const int c0 = T.kb0 + c * csz;
                        const int c1 = min(T.kb1, c0 + csz);
                        for (int kb = c0; kb < c1; ++kb) {
                            if (!mbar_wait(full_bar(st), ph, abort_flag, args.status))
                                goto mma_done;
                            tc_fence_after();
                            const uint64_t so = (uint64_t)((uint32_t)st * kStageD);
                            const uint64_t da0 = da_base + so, db0 = db_base + so;
                            umma_bf16(d, da0, db0, idesc, kb > c0 ? 1u : 0u);
#pragma unroll
                            for (int k = 1; k < kBK / 16; ++k)
                                umma_bf16(d, da0 + k * kStepA, db0 + k * kStepB, idesc, 1u);
                            umma_commit(empty_bar(st));
                            if (++st == S) {
                                st = 0;
                                ph ^= 1u;
                            }
                        }
                        umma_commit(tfull_bar(buf));
                    }
                }
            }
        mma_done:;
            // every MMA of this CTA is issued: the next kernel in the stream
            // may start launching (its CTAs take SMs as this kernel's CTAs exit)
            pdl_trigger();
        }
    }
    if (shared_k) {
        cluster_barrier();      // the two of the epilogue's exchange
        cluster_barrier();
    }
    } else {
        // ---------------- epilogue: warpgroups 1 to 4
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpilogue));
        const int q = warp & 3;                     // TMEM lane quadrant this warp may read
        const int half = (warp - kEpiWarp0) >> 2;   // which quarter of the N columns
        int chunk = 0;
        if constexpr (MODE == TC_DGRAD) {
            // Fused input gradient: gradient at the lower layer's (pooled) output -> int32
            // with the OVERFLOW rule -> max-pool backward (to the recorded window
            // position) -> NITRO-ReLU backward -> lower delta.
            //
            // The delta is the low 32 bits of the sum, kept as they are; OVERFLOW needs the
            // rest only as far as the sum being those 32 bits or 2^32 and more away from
            // them, so an fp32 sum that is off by less than 2^31 decides it (form 1).  With
            // the bit latched it is not needed (form 0); where the bound of its error is
            // too large (six limbs and more together) the sums are 64 bits wide (form 2).
            // The bound: every chunk of every pass rounds a pair of limb sums and the
            // running sum, which stays below cpp csz 2^20 2^(8 (LA + LB - 2)) (1 + 2^-5).
            // Bound by the latency of the epilogue's chains.  64-bit sums throughout, an
            // atomic maximum a warp and tile and 16-byte stores: 128 -> 128 at 16 x 16, 256
            // -> 256 at 8 x 8, batch 128, latched, 51.6 and 47.0 us, now 41.2 and 38.8.
            const int ccpp = (args.kb_total + kChunkBlocks - 1) / kChunkBlocks;
            const int ccsz = ccpp ? (args.kb_total + ccpp - 1) / ccpp : 0;
            const float derr = exp2f((float)(8 * (LA + LB - 2))) * 1.04f / 16.0f * (float)ccsz * (float)ccpp *
                               (float)(LA * LB) * (float)(ccpp + 1);
            const int form = hiskip ? 0 : (derr < 2.0e9f ? 1 : 2);
            const int npos = args.low_pool ? 4 : 1;
            const int Cl = args.Cin;
            bool ovf = false;
            uint32_t mx = 0;
            for (int tile = tile0; tile < args.total_tiles; tile += tile_step) {
                const Tile T = decode_tile(args, tile);
                const int r = 32 * q + lane;   // output row of this thread
                const int col0 = T.nt * N + half * NH;
                const int mq = udiv32(args.dv_ntx, T.mt), tb = udiv32(args.dv_nty, mq);
                const int tx = T.mt - mq * args.ntx, ty = mq - tb * args.nty;
                const int xx = r & ((1 << args.lg_wb) - 1);
                const int yy = (r >> args.lg_wb) & ((1 << args.lg_hb) - 1);
                const int bbx = r >> (args.lg_wb + args.lg_hb);
                const int x = tx * args.wb + xx, y = ty * args.hb + yy, b = tb * args.bb + bbx;
                const bool valid = x < args.W && y < args.H && b < args.B;
                // element offsets (below 2^31, checked when the block is made) of this
                // thread's channels at the gradient's position and the window's positions
                const uint32_t opix = (uint32_t)((b * args.H + y) * args.W + x) * Cl + col0;
                const uint32_t p0 = args.low_pool
                    ? (uint32_t)((b * args.low_h + 2 * y) * args.low_w + 2 * x) * Cl + col0 : opix;
                const uint32_t prow = (uint32_t)args.low_w * Cl;
                // argmax and region codes of 16 channels; with 16 columns a thread they are
                // loaded before the sums are waited for
                uint4 am, rg[4];
                const auto load_codes = [&](int k16) {
                    const bool in = valid && col0 + 16 * k16 < Cl;
                    am = in && npos == 4 ? *reinterpret_cast<const uint4*>(args.low_argmax + opix + 16 * k16)
                                         : make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        rg[k] = in && k < npos
                            ? *reinterpret_cast<const uint4*>(args.low_region + p0 + 16 * k16 + (k >> 1) * prow +
                                                              (k & 1) * Cl)
                            : make_uint4(0, 0, 0, 0);
                };
                if constexpr (NH == 16) load_codes(0);
                uint32_t lo[NH];
                float zf[NH];
                // body(address of limb 0's columns, limbs, shift of the first) for every
                // chunk of every pass
                const auto chunks = [&](auto body) -> bool {
                    const int cpp = (T.kb1 - T.kb0 + kChunkBlocks - 1) / kChunkBlocks;
                    for (int la = 0; la < LA; ++la)
                    for (int lb0 = 0; lb0 < lb_limit(la); lb0 += PB) {
                        const int nb = min(PB, lb_limit(la) - lb0);
                        for (int c = 0; c < cpp; ++c, ++chunk) {
                            const int buf = chunk % NBUF;
                            if (!mbar_wait(tfull_bar(buf), (chunk / NBUF) & 1, abort_flag, args.status))
                                return false;
                            tc_fence_after();
                            // 64-column blocks ordered [channel block][limb of this pass]
                            const int hb = (half * NH) / 64;
                            const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) +
                                (uint32_t)(buf * PB * N + hb * nb * 64 + half * NH - hb * 64);
                            body(base, nb, 8 * (la + lb0));
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(tempty_bar(buf));
                        }
                    }
                    return true;
                };
                // sums modulo 2^32, and with kFp the fp32 sums, a limb pair at a time
                const auto narrow = [&](auto kFp) -> bool {
                    constexpr int CW = 8;
#pragma unroll
                    for (int i = 0; i < NH; ++i) {
                        lo[i] = 0;
                        if (kFp()) zf[i] = 0.0f;
                    }
                    return chunks([&](uint32_t base, int nb, int shift0) {
#pragma unroll
                        for (int j = 0; j < NH / CW; ++j)
                            for (int jb = 0; jb < nb; jb += 2) {
                                const bool two = jb + 1 < nb;
                                const uint32_t m = 1u << (shift0 + 8 * jb);
                                const float mf = (float)m;
                                uint32_t v[2 * CW];
                                tmem_ld8_nowait(base + 64 * jb + CW * j, v);
                                if (two) tmem_ld8_nowait(base + 64 * (jb + 1) + CW * j, v + CW);
                                tmem_wait_ld<2 * CW>(v);
                                if (two) {
#pragma unroll
                                    for (int i = 0; i < CW; ++i) {
                                        const float v0 = __uint_as_float(v[i]), v1 = __uint_as_float(v[CW + i]);
                                        const uint32_t w = ((uint32_t)__float2int_rz(v1) << 8) + (uint32_t)__float2int_rz(v0);
                                        lo[CW * j + i] += w * m;
                                        if (kFp()) zf[CW * j + i] = fmaf(fmaf(v1, 256.0f, v0), mf, zf[CW * j + i]);
                                    }
                                } else {
#pragma unroll
                                    for (int i = 0; i < CW; ++i) {
                                        const float v0 = __uint_as_float(v[i]);
                                        lo[CW * j + i] += (uint32_t)__float2int_rz(v0) * m;
                                        if (kFp()) zf[CW * j + i] = fmaf(v0, mf, zf[CW * j + i]);
                                    }
                                }
                            }
                    });
                };
                bool ok;
                if (form == 0) {
                    ok = narrow(std::false_type());
                } else if (form == 1) {
                    ok = narrow(std::true_type());
#pragma unroll
                    for (int i = 0; i < NH; ++i)
                        ovf |= valid && col0 + i < Cl && fabsf(zf[i] - (float)(int32_t)lo[i]) > 2147483648.0f;
                } else {
                    uint64_t acc[NH];
#pragma unroll
                    for (int i = 0; i < NH; ++i) acc[i] = 0;
                    ok = chunks([&](uint32_t base, int nb, int shift0) {
                        for (int jb = 0; jb < nb; ++jb)
#pragma unroll
                            for (int j = 0; j < NH / 8; ++j) {
                                uint32_t v[8];
                                tmem_ld8_nowait(base + 64 * jb + 8 * j, v);
                                tmem_wait_ld<8>(v);
#pragma unroll
                                for (int i = 0; i < 8; ++i)
                                    acc[8 * j + i] += (uint64_t)(int64_t)__float2int_rz(__uint_as_float(v[i]))
                                                      << (shift0 + 8 * jb);
                            }
                    });
#pragma unroll
                    for (int i = 0; i < NH; ++i) {
                        ovf |= valid && col0 + i < Cl && !fits_i32((int64_t)acc[i]);
                        lo[i] = (uint32_t)acc[i];
                    }
                }
                if (!ok) break;
                // Eight channels at a time: NITRO-ReLU backward once, by the region code at the
                // recorded position, then each window position gets it or zero.  Codes are
                // 0..3: the byte masks of one code value come from its two bits.
                const auto route = [&](auto kPool) {
                    constexpr int NP = kPool() ? 4 : 1;
#pragma unroll
                    for (int k16 = 0; k16 < NH / 16; ++k16) {
                        if (col0 + 16 * k16 >= Cl) break;   // uniform across the warp
                        if constexpr (NH != 16) load_codes(k16);
                        const uint32_t amw[4] = {am.x, am.y, am.z, am.w};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            int32_t v[8];
                            uint32_t at[2][NP];
#pragma unroll
                            for (int e4 = 0; e4 < 2; ++e4) {
                                const int w = 2 * h + e4;
                                const uint32_t r0[4] = {rg[0].x, rg[0].y, rg[0].z, rg[0].w};
                                uint32_t code = r0[w];
                                if constexpr (kPool()) {
                                    const uint32_t a0 = amw[w], a1 = amw[w] >> 1;
                                    at[e4][0] = (~a0 & ~a1 & 0x01010101u) * 255u;
                                    at[e4][1] = (a0 & ~a1 & 0x01010101u) * 255u;
                                    at[e4][2] = (~a0 & a1 & 0x01010101u) * 255u;
                                    at[e4][3] = (a0 & a1 & 0x01010101u) * 255u;
                                    code = 0;
#pragma unroll
                                    for (int k = 0; k < 4; ++k) {
                                        const uint32_t rw[4] = {rg[k].x, rg[k].y, rg[k].z, rg[k].w};
                                        code |= rw[w] & at[e4][k];
                                    }
                                }
                                const uint32_t m1 = (code & ~(code >> 1) & 0x01010101u) * 255u;
                                const uint32_t m2 = (~code & (code >> 1) & 0x01010101u) * 255u;
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const int32_t g = (int32_t)lo[16 * k16 + 8 * h + 4 * e4 + e];
                                    const int32_t gq = args.alpha32.floor_div(g);
                                    v[4 * e4 + e] = (gq & byte_mask(m1, e)) | (g & byte_mask(m2, e));
                                }
                            }
                            if (!valid) continue;
#pragma unroll
                            for (int e = 0; e < 8; ++e) mx = max(mx, abs_u32(v[e]));
#pragma unroll
                            for (int k = 0; k < NP; ++k) {
                                uint32_t o[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e)
                                    o[e] = kPool() ? (uint32_t)(v[e] & byte_mask(at[e >> 2][k], e & 3)) : (uint32_t)v[e];
                                st_u32x8(reinterpret_cast<uint32_t*>(args.low_delta) + p0 + 16 * k16 + 8 * h +
                                             (k >> 1) * prow + (k & 1) * Cl, o);
                            }
                        }
                    }
                };
                if (args.low_pool) route(std::true_type());
                else route(std::false_type());
            }
            mx = __reduce_max_sync(0xffffffffu, mx);
            ovf = __any_sync(0xffffffffu, ovf);
            if (lane == 0) {
                if (mx) atomicMax(args.low_maxabs, mx);
                if (ovf) atomicOr(args.status, ST_OVERFLOW);
            }
        } else {
        // Fused forward: bound of the error of its fp32 sums.  A chunk of csz K-blocks
        // has limb sums below csz 2^20 2^(8 limb).  Per chunk at most two roundings (of
        // 2^-24) hit the running sum, which stays below c csz 2^20 2^(8 (LB - 1)) (1 +
        // 2^-6) after c chunks, one hits a limb pair, and the product with 1 / SF adds
        // 2^-23 of the sum: together csz / 16 2^(8 (LB - 1)) cpp (cpp + 1 + 1 + 2.01).
        // With the K range in KS parts the parts' roundings and the KS - 1 additions stay
        // below what cpp = all the parts' chunks gives.
        const int pcpp = (args.kb_per_split + kChunkBlocks - 1) / kChunkBlocks;
        const int fcpp = KS * pcpp;
        const int fcsz = pcpp ? (args.kb_per_split + pcpp - 1) / pcpp : 0;
        const float err = (float)(1 << (8 * (LB - 1))) * 1.02f * (1.0f / 16.0f) * (float)fcsz *
                          (float)fcpp * ((float)fcpp + 4.2f);
        const bool tight = err <= 0.25f * (float)args.sf;
        const float far = err + 400.0f * (float)args.sf;
        int barriers = shared_k ? 2 : 0;     // cluster barriers this thread still owes
        for (int tile = tile0; tile < args.total_tiles; tile += tile_step) {
            const Tile T = decode_tile(args, tile);
            const int cpp = (T.kb1 - T.kb0 + kChunkBlocks - 1) / kChunkBlocks;
            uint64_t acc[kFused ? 1 : NH];
            uint32_t lo[kFused ? NH : 1];   // fused forward: z modulo 2^32
            float zf[kFused ? NH : 1];      // and z rounded to fp32
#pragma unroll
            for (int i = 0; i < NH; ++i) {
                if constexpr (kFused) {
                    lo[i] = 0;
                    zf[i] = 0.0f;
                } else {
                    acc[i] = 0;
                }
            }
            for (int la = 0; la < LA; ++la)
            for (int lb0 = 0; lb0 < lb_limit(la); lb0 += PB) {
                const int nb = min(PB, lb_limit(la) - lb0);
                const int pbw = nb < PB ? nb : PB;   // MN-major: limb blocks per channel block
                const int shift0 = 8 * (la + lb0);
                for (int c = 0; c < cpp; ++c, ++chunk) {
                    const int buf = chunk % NBUF;
                    if (!mbar_wait(tfull_bar(buf), (chunk / NBUF) & 1, abort_flag, args.status))
                        goto epi_done;
                    tc_fence_after();
                    // K-major B: limb-major columns; MN-major B: 64-column blocks
                    // ordered [channel block][limb of this pass]
                    auto limb_base = [&](int jb) -> uint32_t {
                        const int hb = (half * NH) / 64;
                        const int colj = (MODE == TC_WGRAD || kDgrad)
                            ? (hb * pbw + jb) * 64 + (half * NH - hb * 64)
                            : jb * N + half * NH;
                        return tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * PB * N + colj);
                    };
                    // acc += v 2^shift: one 32 x 32 -> 64 multiply-add below 2^32, an
                    // add to the high word above (shift is a multiple of 8)
                    auto accumulate = [&](const uint32_t* r, int col, int shift, auto n) {
                        if (shift < 32) {
                            const int m = 1 << shift;
#pragma unroll
                            for (int i = 0; i < n(); ++i) {
                                const int v = __float2int_rz(__uint_as_float(r[i]));   // exact integer
                                acc[col + i] += (uint64_t)((long long)v * (long long)m);
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < n(); ++i) {
                                const int v = __float2int_rz(__uint_as_float(r[i]));
                                acc[col + i] += (uint64_t)((uint32_t)v << (shift - 32)) << 32;
                            }
                        }
                    };
                    // 16 or 32 values per TMEM round trip, as the registers beside the
                    // sums allow without spills
                    if constexpr (kFused) {
                        // CW columns of a limb pair at once: 16 values in flight beside the
                        // 64 words of 32 columns' sums, 32 beside 16 columns' sums
                        constexpr int CW = NH == 16 ? 16 : 8;
#pragma unroll
                        for (int j = 0; j < NH / CW; ++j)
                            for (int jb = 0; jb < nb; jb += 2) {
                                const bool two = jb + 1 < nb;
                                const int m = 1 << (shift0 + 8 * jb);
                                const float mf = (float)m;
                                uint32_t r[2 * CW];
                                if constexpr (CW == 16) {
                                    tmem_ld16_nowait(limb_base(jb) + CW * j, r);
                                    if (two) tmem_ld16_nowait(limb_base(jb + 1) + CW * j, r + CW);
                                } else {
                                    tmem_ld8_nowait(limb_base(jb) + CW * j, r);
                                    if (two) tmem_ld8_nowait(limb_base(jb + 1) + CW * j, r + CW);
                                }
                                tmem_wait_ld<2 * CW>(r);
                                if (two) {
#pragma unroll
                                    for (int i = 0; i < CW; ++i) {
                                        const float v0 = __uint_as_float(r[i]), v1 = __uint_as_float(r[CW + i]);
                                        const uint32_t w = ((uint32_t)__float2int_rz(v1) << 8) + (uint32_t)__float2int_rz(v0);
                                        lo[CW * j + i] += w * (uint32_t)m;
                                        zf[CW * j + i] = fmaf(fmaf(v1, 256.0f, v0), mf, zf[CW * j + i]);
                                    }
                                } else {
#pragma unroll
                                    for (int i = 0; i < CW; ++i) {
                                        const float v0 = __uint_as_float(r[i]);
                                        lo[CW * j + i] += (uint32_t)__float2int_rz(v0) * (uint32_t)m;
                                        zf[CW * j + i] = fmaf(v0, mf, zf[CW * j + i]);
                                    }
                                }
                            }
                    } else if constexpr (NH == 16) {
                        for (int jb = 0; jb < nb; jb += 2) {
                            uint32_t r[32];
                            tmem_ld16_nowait(limb_base(jb), r);
                            if (jb + 1 < nb) tmem_ld16_nowait(limb_base(jb + 1), r + 16);
                            tmem_wait_ld<32>(r);
                            accumulate(r, 0, shift0 + 8 * jb, std::integral_constant<int, 16>());
                            if (jb + 1 < nb)
                                accumulate(r + 16, 0, shift0 + 8 * (jb + 1), std::integral_constant<int, 16>());
                        }
                    } else {
                        for (int jb = 0; jb < nb; ++jb) {
                            const uint32_t base = limb_base(jb);
#pragma unroll
                            for (int j = 0; j < NH / 8; ++j) {
                                uint32_t r[8];
                                tmem_ld8_nowait(base + 8 * j, r);
                                tmem_wait_ld<8>(r);
                                accumulate(r, 8 * j, shift0 + 8 * jb, std::integral_constant<int, 8>());
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty_bar(buf));
                }
            }
            if (shared_k) {
            if constexpr (kSplitK) {
                // Partial sums of a cluster's K parts: each quarter of the columns is
                // finished by one CTA, and the others write theirs into its ring
                // memory, which is idle once every CTA has drained its last chunk.
                const int owner = KS == 2 ? half >> 1 : half;
                const int per_owner = KS == 2 ? 2 : 1;
                constexpr uint32_t kSlot = NH * 2 * 32 * 4;      // one warp's sums
                const auto slot = [&](int src) {
                    return smem_u32(smem) + (uint32_t)((src * per_owner + half % per_owner) * 4 + q) * kSlot;
                };
                cluster_barrier();
                if (owner != rank) {
                    const uint32_t dst = remote_smem(slot(rank), (uint32_t)owner) + 16u * lane;
#pragma unroll
                    for (int i = 0; i < NH; i += 4) {
                        st_remote4(dst + 128u * i, lo[i], lo[i + 1], lo[i + 2], lo[i + 3]);
                        st_remote4(dst + 128u * (NH + i), __float_as_uint(zf[i]), __float_as_uint(zf[i + 1]),
                                   __float_as_uint(zf[i + 2]), __float_as_uint(zf[i + 3]));
                    }
                }
                cluster_barrier();
                barriers = 0;
                if (owner != rank) continue;
                for (int src = 0; src < KS; ++src) {
                    if (src == rank) continue;
                    const uint8_t* from = smem + (slot(src) - smem_u32(smem)) + 16 * lane;
#pragma unroll
                    for (int i = 0; i < NH; i += 4) {
                        const uint4 a = *reinterpret_cast<const uint4*>(from + 128 * i);
                        const float4 b = *reinterpret_cast<const float4*>(from + 128 * (NH + i));
                        lo[i] += a.x; lo[i + 1] += a.y; lo[i + 2] += a.z; lo[i + 3] += a.w;
                        zf[i] += b.x; zf[i + 1] += b.y; zf[i + 2] += b.z; zf[i + 3] += b.w;
                    }
                }
            }
            }
            {
                const int r = 32 * q + lane;   // output row of this thread
                const int col0 = T.nt * N + half * NH;
                if constexpr (MODE == TC_GEMM) {
                    const int m = T.mt * kBM + r;      // C[m][n], M rows in args.B
                    if (m < args.B) {
                        int64_t* o = args.out + (int64_t)m * args.ncols + col0;
                        if (args.out_vec == 4 && !args.atomic_out && col0 + NH <= args.ncols) {
#pragma unroll
                            for (int i = 0; i < NH; i += 4) st_i64x4(o + i, acc + i);
                        } else {
#pragma unroll
                            for (int i = 0; i < NH; ++i) {
                                if (col0 + i >= args.ncols) break;
                                if (args.atomic_out)       // K split: exact 64-bit sums
                                    atomicAdd(reinterpret_cast<unsigned long long*>(o + i),
                                              (unsigned long long)acc[i]);
                                else
                                    o[i] = (int64_t)acc[i];
                            }
                        }
                    }
                } else if constexpr (MODE == TC_WGRAD) {
                    const int m = T.mt * kBM + r;
                    const int t = m / args.cin_k, ci = m - t * args.cin_k;
                    // im2col rows: row m is already the (tap, ci) index t Cin + ci
                    const bool ok = args.taps == 1 ? m < args.rows : (t < 9 && ci < args.Cin);
                    const int64_t wrow = args.taps == 1 ? (int64_t)m : (int64_t)t * args.Cin + ci;
                    const int64_t cstride = args.cstride;
                    if (ok) {
                        int64_t* o = args.out + wrow;
#pragma unroll
                        for (int i = 0; i < NH; ++i) {
                            if (col0 + i >= args.ncols) break;
                            unsigned long long* dst = reinterpret_cast<unsigned long long*>(
                                o + (int64_t)(col0 + i) * cstride);
                            if (args.atomic_out) atomicAdd(dst, (unsigned long long)acc[i]);
                            else *dst = acc[i];
                        }
                    }
                    if (args.sgd) {
                        // IntegerSGD (Algorithm 1) on this thread's row of NH columns,
                        // from the final sums in the accumulators (no K split)
                        {
                            uint32_t mx = 0;
                            bool ovf = false;
                            if (ok) {
                                const int tt = args.taps == 1 ? 0 : t;
                                const int64_t pcol = args.taps == 1 ? (int64_t)m : (int64_t)tt * args.tap_k + ci;
                                // 16 columns at a time: all loads of a group are issued
                                // before any store, so a group costs one memory round trip
#pragma unroll
                                for (int i0 = 0; i0 < NH; i0 += 16) {
                                    if (col0 + i0 >= args.ncols) break;   // uniform across the warp
                                    int64_t gv[16];
                                    int32_t wv[16];
#pragma unroll
                                    for (int i = 0; i < 16; ++i) {
                                        const int co = min(col0 + i0 + i, args.ncols - 1);
                                        const int64_t e = (int64_t)co * cstride + wrow;
                                        gv[i] = (int64_t)acc[i0 + i];
                                        wv[i] = args.wt[e];
                                    }
#pragma unroll
                                    for (int i = 0; i < 16; ++i) {
                                        const int co = col0 + i0 + i;
                                        if (co >= args.ncols) break;
                                        const int64_t e = (int64_t)co * cstride + wrow;
                                        const int64_t w = wv[i];
                                        int64_t d = args.trunc ? args.gdiv.trunc_div(gv[i]) : args.gdiv.floor_div(gv[i]);
                                        if (args.decay) d += args.trunc ? args.ediv.trunc_div(w) : args.ediv.floor_div(w);
                                        const int64_t nw = w - d;
                                        ovf |= !fits_i32(nw);
                                        const int32_t s32 = (int32_t)nw;
                                        args.wt[e] = s32;
                                        mx = max(mx, abs_u32(s32));
                                        if (args.wp) {
                                            // limb planes of the new weight, entry (t, ci) of row co
                                            uint16_t* pp = args.wp + (int64_t)co * args.row_k + pcol;
                                            int32_t x = s32;
#pragma unroll
                                            for (int l = 0; l < 4; ++l) {
                                                int dg;
                                                if (l < 3) {
                                                    const int rr = x & 255;
                                                    dg = rr - ((rr >> 7) << 8);
                                                    x = (x >> 8) + (rr >> 7);
                                                } else {
                                                    dg = x;
                                                }
                                                pp[l * args.w_plane] = (uint16_t)(__float_as_uint((float)dg) >> 16);
                                            }
                                        }
                                    }
                                }
                            }
#pragma unroll
                            for (int off = 16; off; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                            ovf = __any_sync(0xffffffffu, ovf);
                            if (lane == 0) {
                                if (mx) atomicMax(args.maxabs_w, mx);
                                if (ovf) atomicOr(args.status, ST_OVERFLOW);
                            }
                        }
                    }
                } else if constexpr (kFused) {
                    // z* = floor(z / SF) from z modulo 2^32 (exact) and z in fp32,
                    // then the NITRO-ReLU value and piece from the table, optional
                    // 2x2 max-pool across lanes; int8 outputs straight from
                    // registers (the 2x2 windows of a tile lie inside one warp:
                    // x partner lane ^ 1, y partner lane ^ wb).  Bound by instruction
                    // issue: two 32-bit words a column instead of 64-bit sums and a
                    // 64-bit divide took the VGG11B forward at batch 256 from 1449 to
                    // 1181 us and the VGG8B step from 980 to 928 us, the branches taken
                    // out of its loops the forward to 1154 us.
                    //
                    // zf is off by less than err (set before the tile loop).  Where err <= SF / 4 the
                    // nearest integer to zf / SF is z* or z* + 1, and the sign of
                    // z - q SF (modulo 2^32, so exact) says which.  Where it is
                    // larger (three or four weight limbs) the remainder, below 2^31
                    // as the host allows at most kFwdMaxBlocks K-blocks, is divided
                    // once more.  |z*| beyond the table is clamped: value and piece
                    // are flat outside [-127, 127].
                    const int mq = udiv32(args.dv_ntx, T.mt), tb = udiv32(args.dv_nty, mq);
                    const int tx = T.mt - mq * args.ntx, ty = mq - tb * args.nty;
                    const int xx = r & ((1 << args.lg_wb) - 1);
                    const int yy = (r >> args.lg_wb) & ((1 << args.lg_hb) - 1);
                    const int bbx = r >> (args.lg_wb + args.lg_hb);
                    const int x = tx * args.wb + xx, y = ty * args.hb + yy, b = tb * args.bb + bbx;
                    const bool valid = x < args.W && y < args.H && b < args.B;
                    const int C = args.Cout;
                    const int32_t sf = args.sf;
                    const float sfi = args.sf_inv;
                    // element offsets fit 32 bits (checked when the block is made)
                    const uint32_t pix = (uint32_t)((b * args.H + y) * args.W + x);
                    const bool anchor = valid && !(x & 1) && !(y & 1) && x + 1 < args.W && y + 1 < args.H;
                    const bool wide = NH == 32 && args.out_align == 32 && col0 + 32 <= C;
                    // this thread's columns of one row: 32, 16 or 8 bytes a store
                    const auto put = [&](int8_t* p, const uint32_t* w) {
                        if (wide) {
                            st32(p, w, true);
                        } else if (args.out_align >= 16) {
#pragma unroll
                            for (int k = 0; k < NH / 16; ++k)
                                if (col0 + 16 * k < C) st16(p + 16 * k, w + 4 * k);
                        } else {
#pragma unroll
                            for (int k = 0; k < NH / 8; ++k)
                                if (col0 + 8 * k < C) st8(p + 8 * k, w + 2 * k);
                        }
                    };
                    // table entries of four columns, two 16-bit ones a word, into lo[4 g],
                    // lo[4 g + 1]: the sums are not needed after
                    if (tight) {
#pragma unroll
                        for (int g4 = 0; g4 < NH / 4; ++g4) {
                            uint32_t e[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                int q = min(max(__float2int_rn(zf[4 * g4 + u] * sfi), -200), 200);
                                q += (int32_t)(lo[4 * g4 + u] - (uint32_t)(q * sf)) >> 31;
                                e[u] = relu_tab[q + kTabHalf];
                            }
                            lo[4 * g4] = e[0] | (e[1] << 16);
                            lo[4 * g4 + 1] = e[2] | (e[3] << 16);
                        }
                    } else {
#pragma unroll
                        for (int g4 = 0; g4 < NH / 4; ++g4) {
                            uint32_t e[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const float f = zf[4 * g4 + u];
                                const int q1 = __float2int_rn(f * sfi);
                                const uint32_t r1 = lo[4 * g4 + u] - (uint32_t)q1 * (uint32_t)sf;
                                const int q2 = __float2int_rn((float)(int32_t)r1 * sfi);
                                const int32_t r2 = (int32_t)(r1 - (uint32_t)q2 * (uint32_t)sf);
                                int q = min(max(q1 + q2 + (r2 >> 31), -200), 200);
                                if (fabsf(f) > far) q = f < 0.0f ? -200 : 200;
                                e[u] = relu_tab[q + kTabHalf];
                            }
                            lo[4 * g4] = e[0] | (e[1] << 16);
                            lo[4 * g4 + 1] = e[2] | (e[3] << 16);
                        }
                    }
                    if constexpr (MODE == TC_FWDD) {
                        // dropped outputs: value 0, region code 4 (element = sample, output)
                        const uint32_t t = *args.drop.step;
                        const uint64_t e0 = (uint64_t)pix * C + col0;
#pragma unroll
                        for (int k = 0; k < NH / 2; ++k) {
                            uint32_t& w = lo[4 * (k >> 1) + (k & 1)];
                            if (dropout_drop(args.drop.seed, t, args.drop.layer, e0 + 2 * k, args.drop.p16))
                                w = (w & 0xffff0000u) | kRegionDropped;
                            if (dropout_drop(args.drop.seed, t, args.drop.layer, e0 + 2 * k + 1, args.drop.p16))
                                w = (w & 0xffffu) | ((uint32_t)kRegionDropped << 16);
                        }
                    }
                    uint32_t vpk[NH / 4], rpk[NH / 4];   // packed outputs, pieces or window positions
#pragma unroll
                    for (int g4 = 0; g4 < NH / 4; ++g4) rpk[g4] = __byte_perm(lo[4 * g4], lo[4 * g4 + 1], 0x6420);
                    if (valid && col0 < C) put(args.region + pix * (uint32_t)C + col0, rpk);
                    if (args.pool) {
                        // key = value, 3 - position (2 (y & 1) + (x & 1)) in its window, piece:
                        // the maximum over the window's four lanes is the first maximum, two
                        // 16-bit keys a word
                        const uint32_t poskey = (uint32_t)(3 - (((y & 1) << 1) | (x & 1))) * 0x00400040u;
                        const int dys = args.wb;
#pragma unroll
                        for (int g4 = 0; g4 < NH / 4; ++g4) {
                            uint32_t k0 = lo[4 * g4] + poskey, k1 = lo[4 * g4 + 1] + poskey;
                            k0 = max_s16x2(k0, __shfl_xor_sync(0xffffffffu, k0, 1));
                            k1 = max_s16x2(k1, __shfl_xor_sync(0xffffffffu, k1, 1));
                            k0 = max_s16x2(k0, __shfl_xor_sync(0xffffffffu, k0, dys));
                            k1 = max_s16x2(k1, __shfl_xor_sync(0xffffffffu, k1, dys));
                            vpk[g4] = __byte_perm(k0, k1, 0x7531);
                            rpk[g4] = 0x03030303u - ((__byte_perm(k0, k1, 0x6420) >> 6) & 0x03030303u);
                        }
                        if (anchor && col0 < C) {
                            const uint32_t o =
                                (uint32_t)((b * args.oh + (y >> 1)) * args.ow + (x >> 1)) * (uint32_t)C + col0;
                            put(args.act + o, vpk);
                            if (args.out2) put(args.out2 + o, vpk);
                            put(args.argmax + o, rpk);
                            if (args.next_nhwc) {
#pragma unroll
                                for (int k = 0; k < NH / 8; ++k)
                                    if (col0 + 8 * k < C) st8_bf16(args.next_nhwc + o + 8 * k, vpk + 2 * k);
                            }
                        }
                    } else if (valid && col0 < C) {
#pragma unroll
                        for (int g4 = 0; g4 < NH / 4; ++g4) vpk[g4] = __byte_perm(lo[4 * g4], lo[4 * g4 + 1], 0x7531);
                        const uint32_t o = pix * (uint32_t)C + col0;
                        put(args.act + o, vpk);
                        if (args.out2) put(args.out2 + o, vpk);
                        if (args.next_nhwc) {
#pragma unroll
                            for (int k = 0; k < NH / 8; ++k)
                                if (col0 + 8 * k < C) st8_bf16(args.next_nhwc + o + 8 * k, vpk + 2 * k);
                        }
                    }
                } else {
                    const int mq = udiv32(args.dv_ntx, T.mt), tb = udiv32(args.dv_nty, mq);
                    const int tx = T.mt - mq * args.ntx, ty = mq - tb * args.nty;
                    const int xx = r & ((1 << args.lg_wb) - 1);
                    const int yy = (r >> args.lg_wb) & ((1 << args.lg_hb) - 1);
                    const int bbx = r >> (args.lg_wb + args.lg_hb);
                    const int x = tx * args.wb + xx, y = ty * args.hb + yy, b = tb * args.bb + bbx;
                    if (x < args.W && y < args.H && b < args.B) {
                        int64_t* o = args.out + (((int64_t)b * args.H + y) * args.W + x) * args.ncols + col0;
                        if (args.out_vec == 4 && col0 + NH <= args.ncols) {
#pragma unroll
                            for (int i = 0; i < NH; i += 4) st_i64x4(o + i, acc + i);
                        } else if (args.out_vec == 2 && col0 + NH <= args.ncols) {
#pragma unroll
                            for (int i = 0; i < NH; i += 2)
                                *reinterpret_cast<ulonglong2*>(o + i) = make_ulonglong2(acc[i], acc[i + 1]);
                        } else {
#pragma unroll
                            for (int i = 0; i < NH; ++i)
                                if (col0 + i < args.ncols) o[i] = (int64_t)acc[i];
                        }
                    }
                }
            }
        }
    epi_done:;
        for (; barriers > 0; --barriers) cluster_barrier();   // a wait gave up: the peers still count on it
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TCOLS)
                     : "memory");
    }
}

// ------------------------------------------------------------------ timeout probe
// Exercises the failure path of the bounded waits without a fault: the CTA
// holds TMEM like the contraction kernel, warp 0 waits on an mbarrier that
// nothing ever completes with a short limit, gives up, raises TIMEOUT and the
// abort flag; warps 1 and 2 wait on another such barrier under the kernel's
// normal limit and leave when they see the flag.  TMEM is then freed and the
// kernel returns, so the context stays usable.
__global__ void __launch_bounds__(96, 1) k_tc_wait_probe(uint32_t* status, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars[0]), 1);
        mbar_init(smem_u32(&bars[1]), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&tmem_slot)),
                     "r"(32)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (lane == 0) {
        // phase 0 of a fresh barrier never completes: both waits must give up
        if (warp == 0) mbar_wait(smem_u32(&bars[0]), 0, abort_flag, status, limit_ns);
        else mbar_wait(smem_u32(&bars[1]), 0, abort_flag, status);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(32)
                     : "memory");
    }
}

// ------------------------------------------------------------------ limb packing
__device__ __forceinline__ uint16_t bf16_bits(int v) {
    return __bfloat16_as_ushort(__float2bfloat16_rn((float)v));   // exact for |v| <= 256
}

// Clears n int64 values: the pack kernels do it for the contraction that runs
// after them and adds K-split partial sums, instead of a memset between the two.
__device__ __forceinline__ void zero_fill(int64_t* z, int64_t n) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (!z) return;
    if (((uintptr_t)z & 15) == 0 && (n & 1) == 0) {
        for (int64_t i = tid; i < n / 2; i += stride)
            reinterpret_cast<uint4*>(z)[i] = make_uint4(0, 0, 0, 0);
    } else {
        for (int64_t i = tid; i < n; i += stride) z[i] = 0;
    }
}

// int8 NHWC [P][C] -> bf16 NHWC [P][Cp] copy, zero in channels C..Cp-1
__global__ void k_pack_act_nhwc(const int8_t* __restrict__ x, int64_t P, int C, int Cp,
                                uint16_t* __restrict__ out, int64_t* zero, int64_t n_zero) {
    pdl_wait();
    zero_fill(zero, n_zero);
    const int64_t n = P * Cp;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = i / Cp;
        const int c = (int)(i - p * Cp);
        out[i] = c < C ? bf16_bits(x[p * C + c]) : (uint16_t)0;
    }
}

// int8 NHWC x [B][H][W][Cin] (9 Cin <= 64) -> bf16 im2col rows [B][H][W][64]:
// entry k = t Cin + ci holds x at (y + ky - 1, x + kx - 1) for tap t = 3 ky + kx,
// zero outside the image and for k >= 9 Cin.  A CTA takes R output rows at a time:
// the R + 2 input rows around them are staged in shared memory with zeros on either
// side, in words where the rows allow (vec), then each thread gathers 8 entries
// (16 bytes), always the same ones, so their offsets stay in registers.  Bound by
// latency, the load of the rows and the barrier behind it: 32 x 32 x 3 images, one row
// at a time with the offsets looked up and indices divided per byte 26.6 us a launch
// at batch 256 (events included), so 16.2; 17.6 and 13.3 at 128, 12.7 and 11.6 at 64.
struct Im2colArgs {
    int B, H, W, Cin, R, groups, vec;     // groups of R rows an image
    int lead, rowlen;                     // staged rows: lead zeros, W Cin bytes, zeros up to rowlen
    FloorDiv32 dv_c, dv_groups, dv_row, dv_w;   // by Cin, groups, words or bytes of an input row, W
};
__global__ void __launch_bounds__(256) k_pack_im2col(const int8_t* __restrict__ x, const Im2colArgs p,
                                                     uint16_t* __restrict__ out) {
    pdl_wait();
    extern __shared__ __align__(16) int8_t win[];
    const int k0 = (threadIdx.x & 7) * 8;      // this thread's entries and their window offsets
    int off[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int k = k0 + j, t = (int)p.dv_c.udiv((uint32_t)k), ci = k - t * p.Cin;
        off[j] = t < 9 ? (t / 3) * p.rowlen + p.lead + (t % 3 - 1) * p.Cin + ci : -1;
    }
    // zeros on either side of each row
    const int side = p.rowlen - p.W * p.Cin;
    for (int i = threadIdx.x; i < (p.R + 2) * side; i += 256) {
        const int r = i / side, c = i - r * side;
        win[r * p.rowlen + (c < p.lead ? c : c + p.W * p.Cin)] = 0;
    }
    const uint32_t nrow = (uint32_t)(p.vec ? p.W * p.Cin / 4 : p.W * p.Cin);
    for (uint32_t g = blockIdx.x; g < (uint32_t)p.B * p.groups; g += gridDim.x) {
        const uint32_t b = p.dv_groups.udiv(g);
        const int y0 = (int)(g - b * p.groups) * p.R, rows = min(p.R, p.H - y0);
        const int8_t* img = x + (int64_t)b * p.H * p.W * p.Cin;
        __syncthreads();                       // the zeros, and readers of the previous rows
        for (uint32_t i = threadIdx.x; i < (uint32_t)(rows + 2) * nrow; i += 256) {
            const uint32_t r = p.dv_row.udiv(i), c = i - r * nrow;
            const int iy = y0 + (int)r - 1;
            const bool in = iy >= 0 && iy < p.H;
            const int8_t* src = img + (int64_t)iy * p.W * p.Cin;
            int8_t* dst = win + r * p.rowlen + p.lead;
            if (p.vec) reinterpret_cast<uint32_t*>(dst)[c] = in ? reinterpret_cast<const uint32_t*>(src)[c] : 0u;
            else dst[c] = in ? src[c] : (int8_t)0;
        }
        __syncthreads();
        uint4* orow = reinterpret_cast<uint4*>(out + ((int64_t)b * p.H + y0) * p.W * kBK);
        for (uint32_t i = threadIdx.x; i < (uint32_t)rows * p.W * 8; i += 256) {
            const uint32_t q = i >> 3, r = p.dv_w.udiv(q), px = q - r * p.W;
            const int8_t* wp = win + r * p.rowlen + px * p.Cin;
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const uint32_t v0 = off[j] >= 0 ? (uint8_t)wp[off[j]] : 0u;
                const uint32_t v1 = off[j + 1] >= 0 ? (uint8_t)wp[off[j + 1]] : 0u;
                w[j / 2] = bf16x2((v0 | v1 << 8) ^ 0x8080u, 0);
            }
            orow[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// shared memory for the rows around one output row
inline size_t im2col_smem(int W, int Cin) { return (size_t)3 * (W + 2) * Cin; }

// n int8 values -> bf16, 16 a thread (one 16-byte load, one 32-byte store; x 16-byte
// and out 32-byte aligned), the tail singly.  Bound by memory: 16.8 M values take
// 14.7 us; 18.9 us with two 16-byte stores a thread (each a half sector), 15.3 us
// with eight values a thread and one 16-byte store.  The byte-permute conversion
// keeps the integer-to-float unit out of it.
__global__ void __launch_bounds__(256) k_pack_act_flat(const int8_t* __restrict__ x, int64_t n,
                                                       uint16_t* __restrict__ out, int64_t* zero,
                                                       int64_t n_zero) {
    pdl_wait();
    zero_fill(zero, n_zero);
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n16 = n / 16;
    for (int64_t i = tid; i < n16; i += stride) {
        const uint4 v = reinterpret_cast<const uint4*>(x)[i];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t o[8];
        cvt16_bf16(o, w);
        st32(reinterpret_cast<int8_t*>(out + 16 * i), o, true);
    }
    for (int64_t i = 16 * n16 + tid; i < n; i += stride) out[i] = bf16_bits(x[i]);
}

// int32 delta NHWC (n values, n % 8 == 0) -> limb planes [L][n], eight values
// per thread and one 16-byte store per plane (L from *maxabs).  The
// input is read 32 bytes at a time when `d` is 32-byte aligned (vec != 0).
__global__ void __launch_bounds__(256) k_pack_delta_nhwc(const int32_t* __restrict__ d, int64_t n,
                                                         int vec, const uint32_t* maxabs,
                                                         uint16_t* __restrict__ out, int64_t* zero,
                                                         int64_t n_zero) {
    pdl_wait();
    zero_fill(zero, n_zero);
    const int L = maxabs ? limb_count(*maxabs) : kMaxLimbs;
    const int64_t n8 = n / 8;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t v[8];
        if (vec) {
            asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                           "=r"(v[6]), "=r"(v[7])
                         : "l"(d + 8 * i));
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = d[8 * i + k];
        }
#pragma unroll
        for (int l = 0; l < kMaxLimbs; ++l) {
            if (l >= L) break;
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 8; k += 2) w[k / 2] = limb_bf16x2(v[k], v[k + 1], l);
            reinterpret_cast<uint4*>(out + (int64_t)l * n)[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}


// W [Cout][9][Cin] -> w_planes [L][Cout][row_k] with entry (t, ci) at
// t tap_k + ci (padding left zero; row_k = 9 Ck, tap_k = Ck with Ck = Cin
// rounded up to 64, or row_k = 64, tap_k = Cin for im2col rows)
__global__ void k_pack_weights(const int32_t* __restrict__ W, int Cout, int Cin, int row_k,
                               int tap_k, const uint32_t* maxabs, uint16_t* __restrict__ wp) {
    pdl_wait();
    const int L = maxabs ? limb_count(*maxabs) : kMaxLimbs;
    const int64_t n = (int64_t)Cout * 9 * Cin;
    const int64_t nk = (int64_t)Cout * row_k;
    auto split = [L](int64_t x, uint16_t* dst, int64_t plane) {
        for (int l = 0; l < L; ++l) {
            int v;
            if (l < L - 1) {
                const int64_t dg = ((x + 128) & 255) - 128;
                v = (int)dg;
                x = (x - dg) >> 8;
            } else {
                v = (int)x;
            }
            dst[l * plane] = bf16_bits(v);
        }
    };
    if (wp) {
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x) {
            const int ci = (int)(i % Cin);
            const int t = (int)((i / Cin) % 9);
            const int co = (int)(i / (9LL * Cin));
            split(W[i], wp + (int64_t)co * row_k + t * tap_k + ci, nk);
        }
    }

}

// Maximum over a launch: the CTA's into scratch[0] (one atomic a CTA), and the last
// CTA, by the ticket in scratch[1], stores it to *out and leaves both words zero.
__device__ __forceinline__ void publish_max(uint32_t m, uint32_t* out, uint32_t* scratch) {
    __shared__ uint32_t cta_max;
    if (threadIdx.x == 0) cta_max = 0;
    __syncthreads();
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(&cta_max, m);
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (cta_max) atomicMax(&scratch[0], cta_max);
    __threadfence();
    if (atomicAdd(&scratch[1], 1u) == gridDim.x - 1) {
        __threadfence();
        *out = atomicExch(&scratch[0], 0u);
        scratch[1] = 0;
    }
}

// The same into all four planes, eight entries a thread, zeros where the rows are
// padded, and *out = max |W| (maximum and CTA ticket in scratch[0], scratch[1],
// zero between launches): one launch for planes whose memory holds anything.
__global__ void __launch_bounds__(256) k_pack_weights_pad(const int32_t* __restrict__ W, int Cout, int Cin,
                                                          int row_k, int tap_k, uint16_t* __restrict__ wp,
                                                          uint32_t* out, uint32_t* scratch) {
    pdl_wait();
    const int64_t nk = (int64_t)Cout * row_k;
    uint32_t mx = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nk / 8;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int co = (int)(8 * i / row_k), e0 = (int)(8 * i - (int64_t)co * row_k);
        int32_t v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int e = e0 + k, t = e / tap_k, ci = e - t * tap_k;
            v[k] = t < 9 && ci < Cin ? W[((int64_t)co * 9 + t) * Cin + ci] : 0;
            mx = max(mx, abs_u32(v[k]));
        }
#pragma unroll
        for (int l = 0; l < kMaxLimbs; ++l)
            reinterpret_cast<uint4*>(wp + l * nk)[i] =
                make_uint4(limb_bf16x2(v[0], v[1], l), limb_bf16x2(v[2], v[3], l),
                           limb_bf16x2(v[4], v[5], l), limb_bf16x2(v[6], v[7], l));
    }
    publish_max(mx, out, scratch);
}

// ------------------------------------------------------------------ host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// bf16 tensor map, dims innermost first; strides in elements for dims 1..r-1.
bool make_map(CUtensorMap* m, const void* base, int rank, const uint64_t* dims,
              const uint64_t* strides_elems, const uint32_t* box) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[5], gstride[4];
    cuuint32_t bdim[5], estr[5];
    for (int i = 0; i < rank; ++i) {
        gdim[i] = dims[i];
        bdim[i] = box[i];
        estr[i] = 1;
    }
    for (int i = 0; i < rank - 1; ++i) gstride[i] = strides_elems[i] * 2;
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base),
                    gdim, gstride, bdim, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// SMs of the current device, and which it is (-1: unknown).  The query takes 16 ns,
// which eager steps of small layers feel, so callers ask once.
int sm_count(int* device = nullptr) {
    static std::atomic<int> counts[kMaxDevices];
    int dev = -1, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    if (device) *device = dev;
    if (dev < 0) return 148;
    if (dev < kMaxDevices) n = counts[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 148;
        if (dev < kMaxDevices) counts[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

inline int log2_exact(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return (1 << l) == v ? l : -1;
}

template <int MODE, int N, int PB>
cudaError_t launch_gemm(const CUtensorMap& a, const CUtensorMap& b, const TcArgs& args_in,
                        cudaStream_t s) {
    using C = TcCfg<N, PB>;
    TcArgs args = args_in;
    args.dv_tn = FloorDiv32::make((uint32_t)args.tiles_n);
    args.dv_tm = FloorDiv32::make((uint32_t)args.tiles_m);
    args.dv_ntx = FloorDiv32::make((uint32_t)args.ntx);
    args.dv_nty = FloorDiv32::make((uint32_t)args.nty);
    args.lg_wb = log2_exact(args.wb);
    args.lg_hb = log2_exact(args.hb);
    if (args.tiles_n < 1 || args.tiles_m < 1 || args.ntx < 1 || args.nty < 1 || args.lg_wb < 0 ||
        args.lg_hb < 0)
        return cudaErrorInvalidValue;
    static std::atomic<uint64_t> ready{0};
    int dev = 0;
    const int sms = sm_count(&dev);
    const cudaError_t e = once_per_device(ready, dev, [] {
        // the setmaxnreg split must fit the registers the CTA is launched with,
        // else setmaxnreg.inc would wait forever: never launch such a build
        cudaFuncAttributes fa{};
        const cudaError_t q = cudaFuncGetAttributes(&fa, k_tc_gemm<MODE, N, PB>);
        if (q != cudaSuccess) return q;
        if (fa.maxThreadsPerBlock < kThreads ||
            128 * kRegsProducer + 32 * kEpiWarps * kRegsEpilogue > kThreads * fa.numRegs)
            return cudaErrorInvalidConfiguration;
        return cudaFuncSetAttribute(k_tc_gemm<MODE, N, PB>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    });
    if (e != cudaSuccess) return e;
    if ((MODE == TC_FWDK || MODE == TC_FWDD) && args.ksplit > 1)
        return launch_cluster(k_tc_gemm<MODE, N, PB>, dim3(args.total_tiles), kThreads, args.ksplit, s, C::SMEM,
                              a, b, args);
    const int grid = args.total_tiles < sms ? args.total_tiles : sms;
    launch_k(k_tc_gemm<MODE, N, PB>, grid, kThreads, C::SMEM, s, a, b, args);
    return cudaGetLastError();
}

// Tile width n and B limbs per stage (pb) from the (last seen) limb count of
// B: as many limbs per stage as the operand has, up to the TMEM budget
// (pb n <= 256).  Any choice is exact; it only changes speed.
int pick_pb(int n, int limbs_hint) {
    if (n == 128) return limbs_hint > 1 ? 2 : 1;
    return limbs_hint > 2 ? 4 : (limbs_hint == 2 ? 2 : 1);
}

// The B tensor map's box spans pb limb planes (one TMA load per stage and
// 64-channel block brings all of them), so pb must match the variant.
template <int MODE>
cudaError_t launch_gemm_pb(int n, int pb, const CUtensorMap& a, const CUtensorMap& b,
                           const TcArgs& args, cudaStream_t s) {
    if (n == 128)
        return pb == 2 ? launch_gemm<MODE, 128, 2>(a, b, args, s) : launch_gemm<MODE, 128, 1>(a, b, args, s);
    if (pb == 4) return launch_gemm<MODE, 64, 4>(a, b, args, s);
    return pb == 2 ? launch_gemm<MODE, 64, 2>(a, b, args, s) : launch_gemm<MODE, 64, 1>(a, b, args, s);
}

int pick_n(int cols) { return cols % 128 == 0 ? 128 : 64; }

// int64 values a store where every row of `cols` starts aligned for it
int out_width(const void* out, int cols) {
    const uintptr_t low = (uintptr_t)out | (uintptr_t)(8 * cols);
    return (low & 31) == 0 ? 4 : ((low & 15) == 0 ? 2 : 1);
}

void pixel_tiling(const LayerGeom& g, int batch, TcArgs& a) {
    if (g.w > 8) { a.wb = 16; a.hb = 8; a.bb = 1; }
    else if (g.w > 4 || g.h > 4) { a.wb = 8; a.hb = 8; a.bb = 2; }
    else { a.wb = 4; a.hb = 4; a.bb = 8; }     // 4 x 4 maps: eight whole images per tile
    a.ntx = (g.w + a.wb - 1) / a.wb;
    a.nty = (g.h + a.hb - 1) / a.hb;
    a.tiles_m = a.ntx * a.nty * ((batch + a.bb - 1) / a.bb);
}

inline int grid1d(int64_t n) {
    int64_t g = (n + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 152 * 8 ? 152 * 8 : g));
}

template <typename T>
bool dalloc(std::vector<void*>& allocs, T** p, size_t count) {
    void* q = nullptr;
    if (cudaMalloc(&q, (count ? count : 1) * sizeof(T)) != cudaSuccess) return false;
    allocs.push_back(q);
    *p = static_cast<T*>(q);
    return true;
}

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

// K split of the weight gradient: at most one wave of CTAs (every CTA one work
// unit), each split at least one exact chunk.  Returns the split count.
int wgrad_splits(int tiles, int kb_total, int* kb_per_split) {
    int splits = sm_count() / tiles;
    const int max_splits = (kb_total + kChunkBlocks - 1) / kChunkBlocks;
    splits = splits < 1 ? 1 : (splits > max_splits ? max_splits : splits);
    *kb_per_split = (kb_total + splits - 1) / splits;
    return (kb_total + *kb_per_split - 1) / *kb_per_split;
}

}  // namespace

namespace {
int wgrad_split_count(const TcLayer& t, const LayerGeom& g, int batch) {
    const bool lin = g.kind == NITRO_LINEAR;
    const int gh = lin ? 1 : g.h, gw = lin ? batch : g.w;
    const int wb = gw <= 8 ? 8 : (gw <= 16 ? 16 : (gw <= 32 ? 32 : 64)), hb = 64 / wb;
    const int taps = (t.im2col || lin) ? 1 : 9;
    const int tiles = (taps * t.cin_k + kBM - 1) / kBM * ((g.cout + pick_n(g.cout) - 1) / pick_n(g.cout));
    const int kb_total = (lin ? 1 : batch) * ((gw + wb - 1) / wb) * ((gh + hb - 1) / hb);
    int kbs = 0;
    return wgrad_splits(tiles, kb_total, &kbs);
}
}  // namespace

bool tc_wgrad_fusable(const TcLayer& t, const LayerGeom& g, int batch) {
    return t.wgrad && batch > 0 && wgrad_split_count(t, g, batch) == 1;
}

int64_t* tc_wgrad_adds(const TcLayer& t, const LayerGeom& g, int batch, int64_t* dW) {
    return t.wgrad && batch > 0 && wgrad_split_count(t, g, batch) > 1 ? dW : nullptr;
}

namespace {
// Which passes of a conv layer run on tcgen05, and its operand layout.
void tc_layer_shape(TcLayer& t, const LayerGeom& g, bool has_dgrad) {
    if (g.kind != NITRO_CONV3X3 || !encode_fn()) return;
    // Inputs with 9 Cin <= 64 run as one 64-wide K-block of im2col rows, others with
    // each tap padded to a multiple of 64 channels; maps of any size, a 128-pixel tile
    // overhanging small ones.  Both waste MMA work and still beat the CUDA-core GEMM,
    // which such layers ran on before: a training step of a 7 x 7, 64 -> 64 layer at
    // batch 128 took 150 us, now 51; 16 x 16, 8 -> 64 at batch 64 213, now 73; 12 x 12,
    // 20 -> 16 at batch 8 154, now 49.
    t.im2col = 9 * g.cin <= kBK && im2col_smem(g.w, g.cin) <= 48 * 1024;
    t.fwd = true;
    t.wgrad = g.cout % 8 == 0;
    // the input gradient reads the forward planes, which im2col layers lay out
    // without taps
    t.dgrad = has_dgrad && g.cout % 8 == 0 && !t.im2col;
    t.cin8 = t.im2col ? kBK : round_up(g.cin, 8);
    t.cin_k = round_up(g.cin, 64);
}

// The forward's fused epilogue: rows of 8-byte multiples, and few enough K-blocks
// for its error bound.
bool tc_fwd_fused(const TcLayer& t, const LayerGeom& g) {
    const int taps = t.im2col || g.kind == NITRO_LINEAR ? 1 : 9;
    return t.fwd && g.cout % 8 == 0 && taps * (t.cin_k / kBK) <= kFwdMaxBlocks;
}

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }
}  // namespace

// Linear layers: the kernel with the fused epilogue, its K split over a cluster, against
// the GEMM into int64 that splits K over more CTAs by atomics, with a clear before and
// the epilogue as a launch after.  Us a forward of batch x in x out at two limbs, fused
// and not: 64 x 3000 x 3000 15.5 and 17.2, 256 x 2048 x 1024 12.1 and 20.7, 128 x 4096 x 4096
// 18.1 and 29.0, 1024 x 1024 x 1024 14.6 and 29.9, 4096 x 1024 x 1024 21.4 and 57.9.  Few
// tiles and a long K want the wider split: 64 x 8192 x 128 14.4 and 13.2, 128 x 8192 x 64
// 14.7 and 12.3, 64 x 8192 x 256 14.8 and 14.0, but 64 x 6144 x 128 11.5 and 11.6.
// Dropout is drawn in the epilogue too (TC_FWDD): the wide MLP's step, 64 x 1024 x 3000
// and 64 x 3000 x 3000 twice with dropout, 217 us on the GEMM route, so 211.
bool tc_linear_fused(const TcLayer& t, const LayerGeom& g, int batch) {
    const int64_t tiles = (batch + kBM - 1) / kBM * (int64_t)((g.cout + 63) / 64);
    return g.kind == NITRO_LINEAR && tc_fwd_fused(t, g) && (tiles > 4 || t.cin_k / kBK <= 96);
}

size_t tc_fwd_scratch(const LayerGeom& g, int batch) {
    TcLayer t;
    tc_layer_shape(t, g, false);
    if (!tc_fwd_fused(t, g)) return 0;
    const size_t nwk = (size_t)g.cout * (t.im2col ? kBK : 9 * t.cin_k);
    return align256(2 * kMaxLimbs * nwk) + align256(2 * (size_t)batch * g.h * g.w * t.cin8);
}

cudaError_t tc_fwd_in_scratch(const LayerGeom& g, int batch, const int8_t* x, const int32_t* W,
                              const TcFwdOut& fo, void* scratch, uint32_t* words, cudaStream_t s) {
    TcLayer t;
    tc_layer_shape(t, g, false);
    const int row_k = t.im2col ? kBK : 9 * t.cin_k, tap_k = t.im2col ? g.cin : t.cin_k;
    const size_t nwk = (size_t)g.cout * row_k;
    t.w_planes = static_cast<uint16_t*>(scratch);
    t.act_nhwc = reinterpret_cast<uint16_t*>(static_cast<char*>(scratch) + align256(2 * kMaxLimbs * nwk));
    t.maxabs_w = words;
    static const uint32_t two_limbs = 32639;       // any hint is exact
    tc_use_external_hints(t, &two_limbs, &two_limbs);
    {
        ProfScope ps(K_TC_PACK_W, s, 0.0, (double)nwk * 12);
        launch_k(k_pack_weights_pad, grid1d((int64_t)nwk / 8), 256, 0, s, W, g.cout, g.cin, row_k, tap_k,
                 t.w_planes, words, words + 1);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = tc_pack_input(t, g, x, batch, false, s);
    bool done = false, fused = false;
    if (e == cudaSuccess) e = tc_conv_forward(t, g, batch, nullptr, &fo, words + 3, s, &done, &fused);
    return e == cudaSuccess && !fused ? cudaErrorInvalidValue : e;
}

cudaError_t tc_fwd_preload() {
    cudaFuncAttributes fa{};
    const void* const fns[] = {
        reinterpret_cast<const void*>(k_tc_gemm<TC_FWD, 64, 2>), reinterpret_cast<const void*>(k_tc_gemm<TC_FWD, 128, 2>),
        reinterpret_cast<const void*>(k_tc_gemm<TC_FWDK, 64, 2>), reinterpret_cast<const void*>(k_tc_gemm<TC_FWDK, 128, 2>),
        reinterpret_cast<const void*>(k_pack_weights_pad), reinterpret_cast<const void*>(k_pack_im2col),
        reinterpret_cast<const void*>(k_pack_act_flat), reinterpret_cast<const void*>(k_pack_act_nhwc)};
    for (const void* f : fns) {
        const cudaError_t e = cudaFuncGetAttributes(&fa, f);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

bool tc_layer_init(TcLayer& t, const LayerGeom& g, int max_batch, bool has_dgrad,
                   const uint32_t* maxabs_w, const uint32_t* maxabs_d,
                   std::vector<void*>& allocs, std::vector<void*>& host_allocs) {
    t = TcLayer();
    t.maxabs_w = maxabs_w;
    t.maxabs_d = maxabs_d;
    if (g.kind != NITRO_CONV3X3 || max_batch < 1 || !encode_fn()) return true;
    tc_layer_shape(t, g, has_dgrad);
    const size_t hw = (size_t)g.h * g.w;
    const size_t nwk = (size_t)g.cout * (t.im2col ? kBK : 9 * t.cin_k);
    bool ok = true;
    if (ok && (t.fwd || t.wgrad)) ok = dalloc(allocs, &t.act_nhwc, (size_t)max_batch * hw * t.cin8);
    if (ok && (t.wgrad || t.dgrad))
        ok = dalloc(allocs, &t.d_nhwc, (size_t)kMaxLimbs * max_batch * hw * g.cout);
    if (ok && (t.fwd || t.dgrad)) ok = dalloc(allocs, &t.w_planes, (size_t)kMaxLimbs * nwk);
    if (ok) {
        void* h = nullptr;
        ok = cudaMallocHost(&h, 2 * sizeof(uint32_t)) == cudaSuccess;
        if (ok) {
            host_allocs.push_back(h);
            t.max_host = static_cast<uint32_t*>(h);
            t.max_host[0] = t.max_host[1] = 0;
        }
    }
    return ok;
}

cudaError_t tc_clear_planes(const TcLayer& t, const LayerGeom& g, cudaStream_t s) {
    if (!t.w_planes) return cudaSuccess;
    const size_t nwk = (size_t)g.cout * (t.im2col ? kBK : 9 * t.cin_k);
    return cudaMemsetAsync(t.w_planes, 0, (size_t)kMaxLimbs * nwk * 2, s);
}

bool tc_linear_init(TcLayer& t, const LayerGeom& g, int max_batch, uint16_t* act_bf16, uint16_t* planes,
                    const uint32_t* maxabs_w, const uint32_t* maxabs_d,
                    std::vector<void*>& allocs, std::vector<void*>& host_allocs) {
    t = TcLayer();
    t.maxabs_w = maxabs_w;
    t.maxabs_d = maxabs_d;
    if (g.kind != NITRO_LINEAR || max_batch < 1 || !act_bf16 || !encode_fn()) return true;
    // TMA strides in multiples of 16 bytes; 8-wide output channel groups
    if (g.cin % 8 != 0 || g.cout % 8 != 0) return true;
    t.wgrad = true;
    t.lin_planes = planes;
    t.fwd = planes && round_up(g.cin, 64) / kBK <= kFwdMaxBlocks;
    t.cin8 = g.cin;
    t.cin_k = round_up(g.cin, 64);
    t.act_nhwc = act_bf16;       // the forward's bf16 copy of the layer input
    bool ok = dalloc(allocs, &t.d_nhwc, (size_t)kMaxLimbs * max_batch * g.cout);
    if (ok) {
        void* h = nullptr;
        ok = cudaMallocHost(&h, 2 * sizeof(uint32_t)) == cudaSuccess;
        if (ok) {
            host_allocs.push_back(h);
            t.max_host = static_cast<uint32_t*>(h);
            t.max_host[0] = t.max_host[1] = 0;
        }
    }
    return ok;
}

int tc_limb_hint(const TcLayer& t, int which) {
    if (!t.own_hints) {
        const uint32_t* h = which ? t.hint_d : t.hint_w;
        return h ? limb_count(*h) : 1;
    }
    return t.max_host ? limb_count(t.max_host[which]) : 1;
}

void tc_weight_planes(const TcLayer& t, const LayerGeom& g, uint16_t** planes, int64_t* plane,
                      int* row_k, int* tap_k) {
    *planes = t.w_planes;
    *row_k = t.im2col ? kBK : 9 * t.cin_k;
    *tap_k = t.im2col ? g.cin : t.cin_k;
    *plane = (int64_t)g.cout * *row_k;
}

cudaError_t tc_refresh_weights(TcLayer& t, const LayerGeom& g, const int32_t* W,
                               const uint32_t* maxabs_w, cudaStream_t s, bool all_planes) {
    if (!t.w_planes) return cudaSuccess;
    const int64_t n = (int64_t)g.cout * 9 * g.cin;
    {
        ProfScope ps(K_TC_PACK_W, s, 0.0, (double)n * 4 * 2);
        const int row_k = t.im2col ? kBK : 9 * t.cin_k, tap_k = t.im2col ? g.cin : t.cin_k;
        launch_k(k_pack_weights, grid1d(n), 256, 0, s, W, g.cout, g.cin, row_k, tap_k,
                 all_planes ? (const uint32_t*)nullptr : maxabs_w, t.w_planes);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !t.own_hints) return e;
    return cudaMemcpyAsync(t.max_host, maxabs_w, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
}

cudaError_t tc_pack_input(TcLayer& t, const LayerGeom& g, const int8_t* x, int batch,
                          bool nhwc_done, cudaStream_t s) {
    if (batch <= 0 || !t.act_nhwc || nhwc_done) return cudaSuccess;
    const int64_t P = (int64_t)batch * g.h * g.w;
    if (t.im2col) {
        ProfScope ps(K_TC_PACK_X, s, 0.0, (double)P * (g.cin + 2 * kBK));
        Im2colArgs p{};
        p.B = batch; p.H = g.h; p.W = g.w; p.Cin = g.cin;
        // staged rows start on words where whole words are copied and that still fits
        p.vec = g.w * g.cin % 4 == 0 && ((uintptr_t)x & 3) == 0;
        p.lead = p.vec ? round_up(g.cin, 4) : g.cin;
        p.rowlen = p.vec ? p.lead + round_up((g.w + 1) * g.cin, 4) : (g.w + 2) * g.cin;
        if (3 * p.rowlen > 48 * 1024) {
            p.vec = 0;
            p.lead = g.cin;
            p.rowlen = (g.w + 2) * g.cin;
        }
        // rows at a time: as many as leave two groups a CTA at four CTAs an SM, fit 24 KB, up to 8
        p.R = 1;
        while (p.R < 8 && (int64_t)batch * ((g.h + 2 * p.R - 1) / (2 * p.R)) >= 4 * 152 &&
               (2 * p.R + 2) * p.rowlen <= 24 * 1024)
            p.R *= 2;
        p.groups = (g.h + p.R - 1) / p.R;
        p.dv_c = FloorDiv32::make((uint32_t)g.cin);
        p.dv_groups = FloorDiv32::make((uint32_t)p.groups);
        p.dv_row = FloorDiv32::make((uint32_t)(p.vec ? g.w * g.cin / 4 : g.w * g.cin));
        p.dv_w = FloorDiv32::make((uint32_t)g.w);
        const int64_t groups = (int64_t)batch * p.groups;
        launch_k(k_pack_im2col, (int)std::min<int64_t>(groups, 152 * 8), 256,
                 (size_t)round_up((p.R + 2) * p.rowlen, 4), s, x, p, t.act_nhwc);
        return cudaGetLastError();
    }
    ProfScope ps(K_TC_PACK_X, s, 0.0, (double)P * (g.cin + 2 * t.cin8));
    if (g.cin == t.cin8 && ((uintptr_t)x & 15) == 0) {
        launch_k(k_pack_act_flat, grid1d(P * g.cin / 16), 256, 0, s, x, P * g.cin, t.act_nhwc,
                 (int64_t*)nullptr, (int64_t)0);
        return cudaGetLastError();
    }
    launch_k(k_pack_act_nhwc, grid1d(P * t.cin8), 256, 0, s, x, P, g.cin, t.cin8, t.act_nhwc,
             (int64_t*)nullptr, (int64_t)0);
    return cudaGetLastError();
}

namespace {
// K split of the fused forward over a cluster, for layers with few output tiles (one
// image, 4 x 4 maps): two, four or, with 64-column tiles, eight CTAs a tile while all
// are resident at once and each has at least four K-blocks, from sixteen K-blocks on (a
// cluster launch costs the host 1 us).  Clusters of eight, one CTA an SM, do not fill
// a GPC: up to 104 CTAs, 128 ran in two rounds.  64-column tiles where even four CTAs
// for each 128-column tile would leave half the SMs idle.  *n: tile width.  Us a launch, events included, unsplit against split: one image 512 ->
// 512 at 8 x 8 and 4 x 4 34.8 against 14.4 and 16.3, 128 -> 256 at 32 x 32 19.7 against
// 14.1; 64 images 512 -> 512 at 4 x 4 35.7 against 22.6.
void fwd_split(TcArgs& a, int cout, int* n) {
    const auto tiles = [&](int w) { return a.tiles_m * ((cout + w - 1) / w); };
    if (a.kb_total < 16) return;
    const int sms = sm_count();
    if (tiles(*n) * 2 > sms) return;
    if (*n == 128 && tiles(128) * 8 < sms) *n = 64;
    for (const int s : {8, 4, 2}) {
        if ((s == 8 && (*n == 128 || tiles(*n) * 8 > 104)) || tiles(*n) * s > sms || a.kb_total < 4 * s)
            continue;
        a.ksplit = s;
        return;
    }
}
}  // namespace

cudaError_t tc_conv_forward(TcLayer& t, const LayerGeom& g, int batch, int64_t* z,
                            const TcFwdOut* fo, uint32_t* status, cudaStream_t s, bool* done,
                            bool* fused) {
    *done = false;
    *fused = false;
    if (!t.fwd || batch <= 0) return cudaSuccess;
    // A linear layer is 1 x 1 images with a single centred tap: rows = the samples
    const bool lin = g.kind == NITRO_LINEAR;
    if (lin && !fo) return cudaSuccess;
    TcArgs a{};
    a.B = batch; a.H = lin ? 1 : g.h; a.W = lin ? 1 : g.w; a.Cin = g.cin; a.Cout = g.cout;
    a.cin_k = t.cin_k;
    a.taps = t.im2col || lin ? 1 : 9;
    if (lin) {
        a.wb = a.hb = a.ntx = a.nty = 1;
        a.bb = kBM;
        a.tiles_m = (batch + kBM - 1) / kBM;
    } else {
        pixel_tiling(g, batch, a);
    }
    a.kb_total = a.taps * (t.cin_k / kBK);
    const bool fuse = fo && tc_fwd_fused(t, g);
    int n = pick_n(g.cout);
    a.ksplit = 1;
    if (fuse) fwd_split(a, g.cout, &n);
    a.tiles_n = (g.cout + n - 1) / n;
    a.total_tiles = a.tiles_m * a.tiles_n * a.ksplit;
    a.kb_per_split = (a.kb_total + a.ksplit - 1) / a.ksplit;
    a.ncols = g.cout;
    a.max_a = nullptr;
    a.max_b = t.maxabs_w;
    a.out = z;
    a.out_vec = out_width(z, g.cout);
    a.status = status;
    a.atomic_out = 0;
    if (fuse) {
        a.sf = 256 * (lin ? 1 : 9) * g.cin;
        a.sf_inv = 1.0f / (float)a.sf;
        a.alpha = FloorDiv::make((uint64_t)fo->alpha_inv);
        a.mu = fo->mu;
        a.pool = !lin && g.pool;
        if (fo->drop && fo->drop->p16) {
            if (!lin || !fo->drop->step) return cudaErrorInvalidValue;
            a.drop = *fo->drop;
        }
        a.oh = g.oh;
        a.ow = g.ow;
        a.act = fo->act;
        a.out2 = fo->out2;
        a.region = fo->region;
        a.argmax = fo->argmax;
        a.next_nhwc = fo->next_nhwc;
        const uintptr_t low = (uintptr_t)a.act | (uintptr_t)a.region | (uintptr_t)a.out2 |
                              (uintptr_t)a.argmax | (uintptr_t)g.cout;
        a.out_align = (low & 31) == 0 ? 32 : ((low & 15) == 0 ? 16 : 8);
        if (low & 7) return cudaErrorInvalidValue;
    }
    CUtensorMap ma, mb;
    const uint64_t da[4] = {(uint64_t)t.cin8, (uint64_t)a.W, (uint64_t)a.H, (uint64_t)batch};
    const uint64_t sa[3] = {(uint64_t)t.cin8, (uint64_t)a.W * t.cin8, (uint64_t)a.H * a.W * t.cin8};
    const uint32_t ba[4] = {64, (uint32_t)a.wb, (uint32_t)a.hb, (uint32_t)a.bb};
    // weight plane row length (a linear layer's rows end inside a K-block: zeros follow)
    const uint64_t kw = lin ? (uint64_t)g.cin : (uint64_t)a.taps * t.cin_k;
    const int pb = pick_pb(n, tc_limb_hint(t, 0));
    const uint64_t db[3] = {kw, (uint64_t)g.cout, (uint64_t)kMaxLimbs};
    const uint64_t sb[2] = {kw, kw * g.cout};
    const uint32_t bb[3] = {64, (uint32_t)n, (uint32_t)pb};
    if (!make_map(&ma, t.act_nhwc, 4, da, sa, ba) || !make_map(&mb, lin ? t.lin_planes : t.w_planes, 3, db, sb, bb))
        return cudaErrorInvalidValue;
    const double ops = 2.0 * batch * a.H * a.W * g.cout * (lin ? 1.0 : 9.0) * g.cin;
    ProfScope ps(lin ? K_TC_GEMM : K_TC_CONV_FWD, s, ops, 0.0);
    cudaError_t e = !fuse ? launch_gemm_pb<TC_FWDZ>(n, pb, ma, mb, a, s)
                  : a.drop.p16 ? launch_gemm_pb<TC_FWDD>(n, pb, ma, mb, a, s)
                          : (a.ksplit > 1 ? launch_gemm_pb<TC_FWDK>(n, pb, ma, mb, a, s)
                                          : launch_gemm_pb<TC_FWD>(n, pb, ma, mb, a, s));
    if (e == cudaSuccess) {
        *done = true;
        *fused = fuse;
    }
    return e;
}

cudaError_t tc_pack_delta(TcLayer& t, const LayerGeom& g, const int32_t* delta,
                          const uint32_t* maxabs_delta, int batch, cudaStream_t s,
                          bool planes_done, int64_t* zero, int64_t n_zero) {
    if (batch <= 0 || (!t.wgrad && !t.dgrad)) return cudaSuccess;
    // limb planes of delta (NHWC, read by the wgrad and dgrad passes), unless
    // an earlier call split this delta already
    const int64_t n = (int64_t)batch * g.h * g.w * g.cout;   // cout % 8 == 0
    if (!planes_done) {
        ProfScope ps(K_TC_PACK_D, s, 0.0, (double)n * 4 * 2);
        launch_k(k_pack_delta_nhwc, grid1d(n / 8), 256, 0, s, delta, n, ((uintptr_t)delta & 31) == 0,
                                                       maxabs_delta, t.d_nhwc, zero, n_zero);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !t.own_hints) return e;
    return cudaMemcpyAsync(t.max_host + 1, maxabs_delta, sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
}

cudaError_t tc_conv_wgrad(TcLayer& t, const LayerGeom& g, const int32_t* delta,
                          const uint32_t* maxabs_delta, int batch, int64_t* dW,
                          uint32_t* status, cudaStream_t s, bool* done, bool planes_done,
                          const TcSgd* sgd, bool* sgd_done) {
    *done = false;
    if (sgd_done) *sgd_done = false;
    if (batch <= 0 || (!t.wgrad && !t.dgrad)) return cudaSuccess;
    if (!t.wgrad) return tc_pack_delta(t, g, delta, maxabs_delta, batch, s, planes_done);
    // A linear layer is one image of height 1 and width `batch` with a single
    // centred tap: rows = input features, K = the samples.
    const bool lin = g.kind == NITRO_LINEAR;
    const int nimg = lin ? 1 : batch, gh = lin ? 1 : g.h, gw = lin ? batch : g.w;
    const int hw = gh * gw;
    TcArgs a{};
    a.B = nimg; a.H = gh; a.W = gw; a.Cin = g.cin; a.Cout = g.cout;
    a.cin_k = t.cin_k;
    a.taps = (t.im2col || lin) ? 1 : 9;
    a.rows = lin ? g.cin : 9 * g.cin;
    a.cstride = lin ? (int64_t)g.cin : 9LL * g.cin;
    // K-blocks: 64-pixel boxes (wb x hb) of one image
    a.wb = gw <= 8 ? 8 : (gw <= 16 ? 16 : (gw <= 32 ? 32 : 64));
    a.hb = 64 / a.wb;
    a.bb = 1;
    a.ntx = (gw + a.wb - 1) / a.wb;
    a.nty = (gh + a.hb - 1) / a.hb;
    const int n = pick_n(g.cout);
    a.tiles_m = (a.taps * t.cin_k + kBM - 1) / kBM;
    a.tiles_n = (g.cout + n - 1) / n;
    a.kb_total = nimg * a.ntx * a.nty;
    int splits = wgrad_splits(a.tiles_m * a.tiles_n, a.kb_total, &a.kb_per_split);
    a.total_tiles = a.tiles_m * a.tiles_n * splits;
    a.ncols = g.cout;
    a.max_a = nullptr;
    a.max_b = maxabs_delta;
    a.out = dW;
    a.status = status;
    a.atomic_out = splits > 1;
    // the pack also clears dW for the partial sums of a K split
    cudaError_t pe = tc_pack_delta(t, g, delta, maxabs_delta, batch, s, planes_done,
                                   a.atomic_out ? dW : nullptr, a.cstride * g.cout);
    if (pe != cudaSuccess) return pe;
    // The update is folded in only without a K split: the sums are then final
    // in the accumulators.  With a split, the warp that completes an output
    // slot would have to read its sums back and update after every other
    // split has arrived; that tail measured ~50 us per launch on the VGG-style
    // step against ~7 us for the block's separate IntegerSGD launch, so split
    // layers report *sgd_done = false and are updated by IntegerSGD.
    if (sgd && sgd_done) *sgd_done = !a.atomic_out;
    if (sgd && a.atomic_out) sgd = nullptr;
    if (sgd) {
        if (sgd->gamma_inv < 1 || sgd->eta_inv < 0) return cudaErrorInvalidValue;
        a.sgd = 1;
        a.wt = sgd->W;
        a.maxabs_w = sgd->maxabs_w;
        a.gdiv = FloorDiv::make((uint64_t)sgd->gamma_inv);
        a.decay = sgd->eta_inv > 0;
        a.ediv = FloorDiv::make(sgd->eta_inv > 0 ? (uint64_t)sgd->eta_inv : 1);
        a.trunc = sgd->trunc;
        a.wp = sgd->planes;
        a.w_plane = sgd->plane;
        a.row_k = sgd->row_k;
        a.tap_k = sgd->tap_k;
    }
    CUtensorMap ma, mb;
    const uint64_t da[4] = {(uint64_t)t.cin8, (uint64_t)gw, (uint64_t)gh, (uint64_t)nimg};
    const uint64_t sa[3] = {(uint64_t)t.cin8, (uint64_t)gw * t.cin8, (uint64_t)hw * t.cin8};
    const uint32_t ba[4] = {64, (uint32_t)a.wb, (uint32_t)a.hb, 1};
    const uint64_t db[5] = {(uint64_t)g.cout, (uint64_t)gw, (uint64_t)gh, (uint64_t)nimg,
                            (uint64_t)kMaxLimbs};
    const uint64_t sb[4] = {(uint64_t)g.cout, (uint64_t)gw * g.cout, (uint64_t)hw * g.cout,
                            (uint64_t)nimg * hw * g.cout};
    const int pb = pick_pb(n, tc_limb_hint(t, 1));
    const uint32_t bb[5] = {64, (uint32_t)a.wb, (uint32_t)a.hb, 1, (uint32_t)pb};
    if (!make_map(&ma, t.act_nhwc, 4, da, sa, ba) || !make_map(&mb, t.d_nhwc, 5, db, sb, bb))
        return cudaErrorInvalidValue;
    const double ops = 2.0 * nimg * hw * g.cout * (double)a.cstride;
    ProfScope ps(lin ? K_TC_LIN_WGRAD : K_TC_CONV_WGRAD, s, ops, 0.0);
    cudaError_t e = launch_gemm_pb<TC_WGRAD>(n, pb, ma, mb, a, s);
    if (e == cudaSuccess) *done = true;
    return e;
}

cudaError_t tc_conv_dgrad(TcLayer& t, const LayerGeom& g, int batch, int64_t* g64,
                          const TcDgradOut* fo, uint32_t* status, cudaStream_t s, bool* done,
                          bool* fused) {
    *done = false;
    *fused = false;
    if (!t.dgrad || batch <= 0) return cudaSuccess;
    TcArgs a{};
    a.B = batch; a.H = g.h; a.W = g.w; a.Cin = g.cin; a.Cout = g.cout;
    a.cin_k = t.cin_k;
    a.taps = 9;
    pixel_tiling(g, batch, a);
    const int n = pick_n(g.cin);
    a.tiles_n = (g.cin + n - 1) / n;
    a.total_tiles = a.tiles_m * a.tiles_n;
    a.kb_total = 9 * ((g.cout + kBK - 1) / kBK);
    a.kb_per_split = a.kb_total;
    a.ncols = g.cin;
    a.max_a = t.maxabs_d;
    a.max_b = t.maxabs_w;
    a.out = g64;
    a.out_vec = out_width(g64, g.cin);
    a.status = status;
    a.atomic_out = 0;
    const bool fuse = fo && g.cin % 16 == 0;
    if (fuse) {
        a.alpha32 = FloorDiv32::make((uint32_t)fo->alpha_inv);
        a.bound_a = fo->maxabs_delta;
        a.bound_b = fo->maxabs_w;
        a.low_h = fo->low_h;
        a.low_w = fo->low_w;
        a.low_pool = fo->low_pool;
        a.low_region = fo->low_region;
        a.low_argmax = fo->low_argmax;
        a.low_delta = fo->low_delta;
        a.low_maxabs = fo->low_maxabs;
        if (fo->low_pool && ((fo->low_h & 1) || (fo->low_w & 1))) {   // rows the pool dropped
            cudaError_t e = cudaMemsetAsync(fo->low_delta, 0,
                                            sizeof(int32_t) * (size_t)batch * fo->low_h * fo->low_w * g.cin, s);
            if (e != cudaSuccess) return e;
        }
    }
    CUtensorMap ma, mb;
    const uint64_t da[5] = {(uint64_t)g.cout, (uint64_t)g.w, (uint64_t)g.h, (uint64_t)batch,
                            (uint64_t)kMaxLimbs};
    // limb planes are batch-sized at this call's batch
    const uint64_t plane = (uint64_t)batch * g.h * g.w * g.cout;
    const uint64_t sa[4] = {(uint64_t)g.cout, (uint64_t)g.w * g.cout, (uint64_t)g.h * g.w * g.cout,
                            plane};
    const uint32_t ba[5] = {64, (uint32_t)a.wb, (uint32_t)a.hb, (uint32_t)a.bb, 1};
    // forward planes [L][Cout][9][Cin64], read MN-major: boxes of 64 ci x 64 co
    const uint64_t db[4] = {(uint64_t)t.cin_k, 9, (uint64_t)g.cout, (uint64_t)kMaxLimbs};
    const uint64_t sb[3] = {(uint64_t)t.cin_k, (uint64_t)9 * t.cin_k, (uint64_t)9 * t.cin_k * g.cout};
    const int pb = pick_pb(n, tc_limb_hint(t, 0));
    const uint32_t bb[4] = {64, 1, 64, (uint32_t)pb};
    if (!make_map(&ma, t.d_nhwc, 5, da, sa, ba) || !make_map(&mb, t.w_planes, 4, db, sb, bb))
        return cudaErrorInvalidValue;
    const double ops = 2.0 * batch * g.h * g.w * g.cin * 9.0 * g.cout;
    ProfScope ps(K_TC_CONV_DGRAD, s, ops, 0.0);
    cudaError_t e = fuse ? launch_gemm_pb<TC_DGRAD>(n, pb, ma, mb, a, s)
                         : launch_gemm_pb<TC_DGRADZ>(n, pb, ma, mb, a, s);
    if (e == cudaSuccess) {
        *done = true;
        *fused = fuse;
    }
    return e;
}

cudaError_t tc_timeout_probe(uint32_t* status, uint64_t limit_ns, cudaStream_t s) {
    ProfScope ps(K_TC_PROBE, s, 0.0, 0.0);
    k_tc_wait_probe<<<1, 96, 0, s>>>(status, limit_ns);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ plain GEMM
namespace {
// *out = max |x|: maximum and CTA ticket in scratch[0], scratch[1] (zero
// between launches), so no memset of *out precedes the launch.
// 16-byte loads between the unaligned head and tail.
__global__ void __launch_bounds__(256) k_maxabs(const int32_t* __restrict__ x, int64_t n, uint32_t* out,
                                                uint32_t* scratch) {
    pdl_wait();
    uint32_t m = 0;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t head = min(n, (int64_t)((16 - ((uintptr_t)x & 15)) & 15) / 4);
    const int64_t n4 = (n - head) / 4, tail = head + 4 * n4;
    const int4* xv = reinterpret_cast<const int4*>(x + head);
    const auto take = [&m](const int4 v) {
        m = max(max(max(m, abs_u32(v.x)), max(abs_u32(v.y), abs_u32(v.z))), abs_u32(v.w));
    };
    int64_t i = tid;
    for (; i + 3 * stride < n4; i += 4 * stride) {   // four loads in flight a thread
        const int4 a = xv[i], b = xv[i + stride], c = xv[i + 2 * stride], d = xv[i + 3 * stride];
        take(a);
        take(b);
        take(c);
        take(d);
    }
    for (; i < n4; i += stride) take(xv[i]);
    if (tid < head) m = max(m, abs_u32(x[tid]));
    if (tid < n - tail) m = max(m, abs_u32(x[tail + tid]));
    publish_max(m, out, scratch);
}
}  // namespace

cudaError_t tc_maxabs(const int32_t* x, int64_t n, uint32_t* out, uint32_t* scratch, cudaStream_t s) {
    if (n <= 0) return cudaMemsetAsync(out, 0, sizeof(uint32_t), s);
    ProfScope ps(K_TC_PACK, s, 0.0, (double)n * 4);
    launch_k(k_maxabs, grid1d(n / 4), 256, 0, s, x, n, out, scratch);
    return cudaGetLastError();
}

cudaError_t tc_pack_int8(const int8_t* x, int64_t rows, int cols, uint16_t* out, cudaStream_t s,
                         int64_t* zero, int64_t n_zero) {
    if (rows <= 0) return cudaSuccess;
    ProfScope ps(K_TC_PACK, s, 0.0, (double)rows * cols * 3);
    if (((uintptr_t)x & 15) == 0)
        launch_k(k_pack_act_flat, grid1d(std::max(rows * cols / 16, n_zero / 8)), 256, 0, s, x, rows * cols, out,
                 zero, n_zero);
    else
        launch_k(k_pack_act_nhwc, grid1d(rows * cols), 256, 0, s, x, rows, cols, cols, out, zero, n_zero);
    return cudaGetLastError();
}

cudaError_t tc_pack_limbs(const int32_t* x, int64_t n, const uint32_t* maxabs, uint16_t* planes,
                          cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    ProfScope ps(K_TC_PACK, s, 0.0, (double)n * 4 * 2);
    launch_k(k_pack_delta_nhwc, grid1d(n / 8), 256, 0, s, x, n, ((uintptr_t)x & 31) == 0, maxabs, planes,
             (int64_t*)nullptr, (int64_t)0);
    return cudaGetLastError();
}

namespace {
// K split of the GEMM over CTAs: with few output tiles (a batch of 64 against a
// linear layer) about one wave of CTAs, at least four K-blocks per split.
int gemm_splits(int M, int N, int K, int* kb_per_split) {
    const int n = pick_n(N);
    const int tiles = (M + kBM - 1) / kBM * ((N + n - 1) / n);
    const int kb_total = (K + kBK - 1) / kBK;
    int splits = sm_count() / tiles;
    const int max_splits = (kb_total + 3) / 4;
    splits = splits < 1 ? 1 : (splits > max_splits ? max_splits : splits);
    *kb_per_split = (kb_total + splits - 1) / splits;
    return (kb_total + *kb_per_split - 1) / *kb_per_split;
}
}  // namespace

bool tc_gemm_adds(int M, int N, int K) {
    int kbs = 0;
    return M > 0 && N > 0 && gemm_splits(M, N, K, &kbs) > 1;
}

cudaError_t tc_gemm_run(const uint16_t* a_bf16, const uint16_t* b_planes, int M, int N, int K,
                        const uint32_t* max_b, int64_t* out, uint32_t* status, cudaStream_t s) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    TcArgs a{};
    a.B = M;
    a.ncols = N;
    a.ntx = a.nty = 1;
    a.wb = a.hb = a.bb = 1;
    const int n = pick_n(N);
    a.tiles_m = (M + kBM - 1) / kBM;
    a.tiles_n = (N + n - 1) / n;
    a.kb_total = (K + kBK - 1) / kBK;
    // a K split adds its partial sums with 64-bit atomics into a zeroed C
    const int splits = gemm_splits(M, N, K, &a.kb_per_split);
    a.total_tiles = a.tiles_m * a.tiles_n * splits;
    a.atomic_out = splits > 1;
    a.max_a = nullptr;
    a.max_b = max_b;
    a.out = out;
    a.out_vec = out_width(out, N);
    a.status = status;
    CUtensorMap ma, mb;
    const uint64_t da[2] = {(uint64_t)K, (uint64_t)M};
    const uint64_t sa[1] = {(uint64_t)K};
    const uint32_t ba[2] = {64, 128};
    const uint64_t db[3] = {(uint64_t)K, (uint64_t)N, (uint64_t)kMaxLimbs};
    const uint64_t sb[2] = {(uint64_t)K, (uint64_t)K * N};
    const uint32_t bb[3] = {64, (uint32_t)n, 1};
    if (!make_map(&ma, a_bf16, 2, da, sa, ba) || !make_map(&mb, b_planes, 3, db, sb, bb))
        return cudaErrorInvalidValue;
    ProfScope ps(K_TC_GEMM, s, 2.0 * M * N * (double)K, 0.0);
    // Two limbs of B a stage: one A tile then feeds both, and the MMAs are twice as
    // wide.  Only the limbs that B has are loaded, so a one-limb B loses nothing but
    // ring depth.  4096^3 at two limbs: 220 us against 359 us with one limb a stage.
    return launch_gemm_pb<TC_GEMM>(n, 2, ma, mb, a, s);
}

}  // namespace nitro
