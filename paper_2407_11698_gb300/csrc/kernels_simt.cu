// CUDA-core kernels of the NITRO-D block step: an exact int64 implicit GEMM
// (conv 3x3 fwd / dgrad / wgrad, linear fwd / dgrad), the linear layers of few
// products, and the element-wise stages fused around it (NITRO-Scaling,
// NITRO-ReLU and max-pool forward, with dropout for linear layers; max-pool,
// NITRO-ReLU backward and STE; the learning layer, its max-pool to d_lr and
// the RSS loss; IntegerSGD).
//
// The GEMM serves the contractions the tensor-core path does not take (conv
// gradients where Cout is not a multiple of 8 or the input is narrow, linear input
// gradients, the kernel-level matrix product where K is not a multiple of 8, small
// or misaligned allocation-free forwards); the learning layer (up to 64 outputs)
// and the element-wise stages always run here.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "nitro_internal.cuh"
#include "prof.cuh"

namespace nitro {
namespace {

// The CTA's maximum into *word (one atomic a CTA: thousands of warps on one word
// take longer than most of these kernels) and its overflow flag into *status.
// Every thread of the CTA calls it.
__device__ __forceinline__ void block_maximum(uint32_t mx, bool ovf, uint32_t* word, uint32_t* status) {
    __shared__ uint32_t cta_max;
    if (threadIdx.x == 0) cta_max = 0;
    const bool any = __syncthreads_or(ovf);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&cta_max, mx);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (cta_max) atomicMax(word, cta_max);
        if (any) atomicOr(status, ST_OVERFLOW);
    }
}

constexpr int kTile = 64;   // M and N tile
constexpr int kTK = 16;     // K slab
constexpr unsigned kFull = 0xffffffffu;

struct GemmParams {
    const int8_t* act;
    const int32_t* grad;
    const int32_t* wts;
    int64_t* out;
    int M, N, K;
    int B, H, W, Cin, Cout;
    int k_split;
};

// Operand element A[m][k] / B[n][k] of each contraction (see GemmMode).
template <int MODE>
__device__ __forceinline__ int32_t load_a(const GemmParams& p, int m, int k) {
    if (MODE == GM_CONV_FWD || MODE == GM_CONV_DGRAD) {
        const int hw = p.H * p.W;
        const int b = m / hw, r = m - b * hw, y = r / p.W, x = r - y * p.W;
        const int C = MODE == GM_CONV_FWD ? p.Cin : p.Cout;
        const int t = k / C, c = k - t * C, ky = t / 3, kx = t - 3 * ky;
        // forward reads input (y+ky-1, x+kx-1); dgrad reads output (y-ky+1, x-kx+1)
        const int iy = MODE == GM_CONV_FWD ? y + ky - 1 : y - ky + 1;
        const int ix = MODE == GM_CONV_FWD ? x + kx - 1 : x - kx + 1;
        if (iy < 0 || iy >= p.H || ix < 0 || ix >= p.W) return 0;
        const int64_t idx = ((int64_t)(b * p.H + iy) * p.W + ix) * C + c;
        return MODE == GM_CONV_FWD ? (int32_t)p.act[idx] : p.grad[idx];
    } else if (MODE == GM_CONV_WGRAD || MODE == GM_LIN_WGRAD) {
        return p.grad[(int64_t)k * p.Cout + m];
    } else if (MODE == GM_LIN_FWD) {
        return p.act[(int64_t)m * p.Cin + k];
    } else {  // GM_LIN_DGRAD
        return p.grad[(int64_t)m * p.Cout + k];
    }
}

template <int MODE>
__device__ __forceinline__ int32_t load_b(const GemmParams& p, int n, int k) {
    if (MODE == GM_CONV_FWD) {
        return p.wts[(int64_t)n * 9 * p.Cin + k];
    } else if (MODE == GM_CONV_DGRAD) {
        const int t = k / p.Cout, co = k - t * p.Cout;
        return p.wts[((int64_t)co * 9 + t) * p.Cin + n];
    } else if (MODE == GM_CONV_WGRAD) {
        const int t = n / p.Cin, ci = n - t * p.Cin, ky = t / 3, kx = t - 3 * ky;
        const int hw = p.H * p.W;
        const int b = k / hw, r = k - b * hw, y = r / p.W, x = r - y * p.W;
        const int iy = y + ky - 1, ix = x + kx - 1;
        if (iy < 0 || iy >= p.H || ix < 0 || ix >= p.W) return 0;
        return p.act[((int64_t)(b * p.H + iy) * p.W + ix) * p.Cin + ci];
    } else if (MODE == GM_LIN_FWD) {
        return p.wts[(int64_t)n * p.Cin + k];
    } else if (MODE == GM_LIN_DGRAD) {
        return p.wts[(int64_t)k * p.Cin + n];
    } else {  // GM_LIN_WGRAD
        return p.act[(int64_t)k * p.Cin + n];
    }
}

// 64x64 output tile per CTA, 4x4 per thread, int64 accumulators.  With
// gridDim.z > 1 each CTA sums one K slice and adds it into a zeroed `out`
// with 64-bit integer atomics (exact and order-independent).
template <int MODE>
__global__ void __launch_bounds__(256) k_gemm(GemmParams p) {
    pdl_wait();
    __shared__ int32_t As[kTK][kTile + 4];
    __shared__ int32_t Bs[kTK][kTile + 4];
    const int m0 = blockIdx.y * kTile, n0 = blockIdx.x * kTile;
    const int kb = blockIdx.z * p.k_split;
    const int ke = min(p.K, kb + p.k_split);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    int64_t acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0;

    for (int k0 = kb; k0 < ke; k0 += kTK) {
        for (int i = threadIdx.x; i < kTile * kTK; i += 256) {
            const int mm = i / kTK, kk = i - mm * kTK;
            const int k = k0 + kk;
            const int m = m0 + mm, n = n0 + mm;
            As[kk][mm] = (m < p.M && k < ke) ? load_a<MODE>(p, m, k) : 0;
            Bs[kk][mm] = (n < p.N && k < ke) ? load_b<MODE>(p, n, k) : 0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kTK; ++kk) {
            int32_t a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[kk][ty + 16 * r];
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = Bs[kk][tx + 16 * c];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] += (int64_t)a[r] * b[c];
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int m = m0 + ty + 16 * r, n = n0 + tx + 16 * c;
            if (m < p.M && n < p.N) {
                int64_t* o = p.out + (int64_t)m * p.N + n;
                if (gridDim.z > 1)
                    atomicAdd(reinterpret_cast<unsigned long long*>(o),
                              (unsigned long long)acc[r][c]);
                else
                    *o = acc[r][c];
            }
        }
}

// ---------------------------------------------------------------------------
// Forward epilogue: one thread per pooling window (or per element).
// ---------------------------------------------------------------------------
__global__ void k_fwd_epilogue(const int64_t* __restrict__ z, LayerGeom g, int B,
                               int alpha_inv, int mu, int64_t kdiv, int8_t* __restrict__ out,
                               int8_t* __restrict__ out2, int8_t* __restrict__ region,
                               int8_t* __restrict__ argmax, DropoutArgs drop) {
    pdl_wait();
    const int C = g.cout;
    if (!g.pool) {
        // dropout (linear layers): element i = b * out_features + j of this step's mask
        const uint32_t t = drop.p16 ? *drop.step : 0u;
        const int64_t n = (int64_t)B * g.h * g.w * C;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
             i += (int64_t)gridDim.x * blockDim.x) {
            const int64_t zs = scale_floor(z[i], kdiv);
            int rg = relu_region(zs);
            int8_t v = (int8_t)relu_value(zs, alpha_inv, mu);
            if (drop.p16 && dropout_drop(drop.seed, t, drop.layer, (uint64_t)i, drop.p16)) {
                rg = kRegionDropped;
                v = 0;
            }
            region[i] = (int8_t)rg;
            out[i] = v;
            if (out2) out2[i] = v;
        }
        return;
    }
    // windows over ceil(h/2) x ceil(w/2); partial windows (odd edges) only
    // record region codes of the positions the floor-sized pool drops.
    const int wy_n = (g.h + 1) / 2, wx_n = (g.w + 1) / 2;
    const int64_t n = (int64_t)B * wy_n * wx_n * C;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        int64_t r = i / C;
        const int wx = (int)(r % wx_n);
        r /= wx_n;
        const int wy = (int)(r % wy_n);
        const int b = (int)(r / wy_n);
        int best = 0, bestv = 0;
        bool full = (2 * wy + 1 < g.h) && (2 * wx + 1 < g.w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int iy = 2 * wy + (k >> 1), ix = 2 * wx + (k & 1);
            if (iy >= g.h || ix >= g.w) continue;
            const int64_t pi = ((int64_t)(b * g.h + iy) * g.w + ix) * C + c;
            const int64_t zs = scale_floor(z[pi], kdiv);
            region[pi] = (int8_t)relu_region(zs);
            const int v = relu_value(zs, alpha_inv, mu);
            if (k == 0 || v > bestv) { bestv = v; best = k; }
        }
        if (full) {
            const int64_t oi = ((int64_t)(b * g.oh + wy) * g.ow + wx) * C + c;
            out[oi] = (int8_t)bestv;
            if (out2) out2[oi] = (int8_t)bestv;
            argmax[oi] = (int8_t)best;
        }
    }
}

// ---------------------------------------------------------------------------
// Learning layer forward: z[b][g] = sum_j a[b][j] W_lr[g][j], y_hat = floor(z /
// (256 d)), grad_L = y_hat - 32 onehot.  A cluster takes eight samples; its CTAs
// (up to eight) share out the features and exchange their partial sums through
// distributed shared memory, so that no atomic, fence or ticket stands between
// the sums and grad_L.  Warp u of a CTA takes sample u, 256 features a tile,
// eight a lane, against the bytes of W_lr in shared memory (two's complement: as
// many bytes as max |W_lr| needs, the top one signed, those below unsigned): one
// dp4a a byte and four features, exact in 32 bits over 128 tiles.
// Bound by latency (the loads of a tile go out before the one before it is summed)
// and by launch overhead.  The kernel before it (64-bit products, 64-bit atomics into
// a sum array, one ticket a sample group and one for the loss) took 15.3 us a launch
// in the VGG8B step and 29 us with 47 classes, this one 10.7 and 17 (events included).
// The loss, the SSE and max |grad_L| are left to the kernel after it (loss_tail),
// off the chain; the launch clears what the rest of the backward adds into.  A CTA that
// has its samples to itself (ALONE: many samples, few features) skips the cluster
// barriers: 65536 samples of 8 features 104 us with them, 73 without.
// ---------------------------------------------------------------------------
constexpr int kLfSamples = 8;      // samples per cluster, one warp each
constexpr int kLfTile = 256;       // features per tile
constexpr int kLfCluster = 8;      // CTAs per cluster at most
constexpr int kLfG = 16;           // classes per pass
constexpr int kMaxClasses = 64;
constexpr int kLfSpan = 128;       // tiles per 32-bit sum
// Products up to which a linear layer that could run on the tensor cores runs on
// k_lin_fwd / k_lin_wgrad.  Forward, us, here against there, weights of two limbs: 16 M
// (batch 16, 1024 x 1024) 7.6 / 10.9, 32 M 9.8 / 12.3, 64 M 13.4 / 14.6 and 17.0 / 18.9
// (batch 256, 512 x 512), 128 M 23.6 / 20.0; four limbs at 64 M 18.3 / 16.8.  Whole
// backward: 16 M 18.2 / 19.5, 32 M 18.6 / 19.6, 64 M 26.1 / 19.5.
constexpr int64_t kLinFwdMacs = (int64_t)48 << 20, kLinWgradMacs = (int64_t)32 << 20;
// Products above which the weight gradient of a layer without a tensor-core form takes the
// general GEMM, whose 4 x 4 sums a thread feed the multipliers better (the samples padded
// to whole slabs): backward of a 1001 -> 999 layer at batch 192 57 us here, 60 there, at
// 512 134 and 114, at 1024 263 and 203.
constexpr int64_t kLinGemmMacs = (int64_t)192 << 20;
// CTAs (16 outputs x 8 samples each) up to which the forward of a linear layer takes
// k_lin_fwd.  Against the tensor cores, us: 128 x 128 at 512 CTAs 6.1 and 8.8, at 1024 10.6
// and 8.7; 256 x 256 6.2 and 9.1, 10.8 and 9.4; 504 x 333 at 672 10.3 and 13.8.  Against the
// general GEMM (no tensor-core form) the line rises with the inputs a CTA sums: 16 of
// them at 256 CTAs 3.9 and 5.7, at 512 6.1 and 5.7; 60 at 1024 12.2 and 12.7, at 2048 21.4
// and 14.2; 250 at 5376 57 and 64, at 10752 109 and 90; 1001 at 16128 394 and 392, at 32256
// 761 and 658.
// A cluster of eight shares the inputs; the tensor-core GEMM shares a long K wider: one
// sample, 191 outputs, 50176 inputs 13 and 17 us, 111888 inputs 26 and 23.
constexpr int64_t kLinFwdCtas = 896, kLinFwdCtasMin = 448, kLinFwdCtasPerIn = 24, kLinFwdIn = 65536;

struct LearnArgs {
    const int8_t* a;
    const int32_t* wlr;
    int B, d, G, per;              // per: features per CTA, a multiple of the tile
    int vec_a, vec_w;              // 8-byte rows of a, 16-byte rows of W_lr
};

// Eight features of one sample as bytes, zero past the row or the batch.
__device__ __forceinline__ uint2 learn_load_a(const LearnArgs& p, int b, int j) {
    uint2 v = make_uint2(0, 0);
    if (b >= p.B || j >= p.d) return v;
    const int8_t* src = p.a + (int64_t)b * p.d + j;
    if (p.vec_a) return *reinterpret_cast<const uint2*>(src);
    const int n = min(8, p.d - j);
    for (int m = 0; m < n; ++m)
        (m < 4 ? v.x : v.y) |= (uint32_t)(uint8_t)src[m] << (8 * (m & 3));
    return v;
}
__device__ __forceinline__ int4 learn_load_w(const LearnArgs& p, int g, int j) {
    int4 v = make_int4(0, 0, 0, 0);
    if (g >= p.G || j >= p.d) return v;
    const int32_t* src = p.wlr + (int64_t)g * p.d + j;
    if (p.vec_w) return *reinterpret_cast<const int4*>(src);
    v.x = src[0];
    if (j + 1 < p.d) v.y = src[1];
    if (j + 2 < p.d) v.z = src[2];
    if (j + 3 < p.d) v.w = src[3];
    return v;
}

// c + sum of four products of a signed byte of a and an unsigned byte of b
__device__ __forceinline__ int dp4a_su(uint32_t a, uint32_t b, int c) {
    int d;
    asm("dp4a.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// z of classes gc .. gc + GM - 1 for this warp's sample over features [j0, j1): lane
// g returns class gc + g.  ws: GM rows of one tile, byte l of four features a word.
template <int GM, int L>
__device__ __forceinline__ long long learn_dots(const LearnArgs& p, int b, int gc, int j0, int j1,
                                                uint32_t* ws) {
    constexpr int kPer = (GM * (kLfTile / 4) + 255) / 256;   // groups of four weights a thread
    const int lane = threadIdx.x & 31, wd = threadIdx.x & 63, gr = threadIdx.x >> 6;
    long long z = 0;
    int acc[GM][L];
#pragma unroll
    for (int g = 0; g < GM; ++g)
#pragma unroll
        for (int l = 0; l < L; ++l) acc[g][l] = 0;
    uint2 av = learn_load_a(p, b, j0 + 8 * lane);
    int4 wv[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) wv[i] = learn_load_w(p, gc + gr + 4 * i, j0 + 4 * wd);
    int tile = 0;
    for (int j = j0; j < j1; j += kLfTile) {
        __syncthreads();                       // readers of the tile before are done
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int g = gr + 4 * i;
            if (g >= GM) break;
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const uint32_t sel = l | ((4 + l) << 4);
                const uint32_t lo = __byte_perm((uint32_t)wv[i].x, (uint32_t)wv[i].y, sel);
                const uint32_t hi = __byte_perm((uint32_t)wv[i].z, (uint32_t)wv[i].w, sel);
                ws[(l * GM + g) * 64 + wd] = __byte_perm(lo, hi, 0x5410);
            }
        }
        __syncthreads();
        const uint2 ac = av;
        if (j + kLfTile < j1) {
            av = learn_load_a(p, b, j + kLfTile + 8 * lane);
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                wv[i] = learn_load_w(p, gc + gr + 4 * i, j + kLfTile + 4 * wd);
        }
#pragma unroll
        for (int g = 0; g < GM; ++g)
#pragma unroll
            for (int l = 0; l < L; ++l) {
                const uint2 w = *reinterpret_cast<const uint2*>(&ws[(l * GM + g) * 64 + 2 * lane]);
                if (l == L - 1) {
                    acc[g][l] = __dp4a((int)ac.x, (int)w.x, acc[g][l]);
                    acc[g][l] = __dp4a((int)ac.y, (int)w.y, acc[g][l]);
                } else {
                    acc[g][l] = dp4a_su(ac.x, w.x, acc[g][l]);
                    acc[g][l] = dp4a_su(ac.y, w.y, acc[g][l]);
                }
            }
        if (++tile == kLfSpan || j + kLfTile >= j1) {
            // at most 128 tiles x 256 features x 128 x 255 < 2^30 a byte
            tile = 0;
#pragma unroll
            for (int g = 0; g < GM; ++g) {
                long long t = 0;
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    t += (long long)__reduce_add_sync(kFull, acc[g][l]) << (8 * l);
                    acc[g][l] = 0;
                }
                if (lane == g) z += t;
            }
        }
    }
    return z;
}

template <int GM>
__device__ __forceinline__ long long learn_pass(const LearnArgs& p, int limbs, int b, int gc, int j0,
                                                int j1, uint32_t* ws) {
    if (limbs == 1) return learn_dots<GM, 1>(p, b, gc, j0, j1, ws);
    if (limbs == 2) return learn_dots<GM, 2>(p, b, gc, j0, j1, ws);
    if (limbs == 3) return learn_dots<GM, 3>(p, b, gc, j0, j1, ws);
    return learn_dots<GM, 4>(p, b, gc, j0, j1, ws);
}

template <bool ALONE>
__global__ void __launch_bounds__(256) k_learn_fwd(const LearnArgs p, FloorDiv dv,
                                                   const int32_t* __restrict__ labels,
                                                   int32_t* __restrict__ grad_l,
                                                   const uint32_t* maxabs_wlr, uint32_t* status,
                                                   uint32_t* zero_words, int n_zero,
                                                   uint32_t* gl_bound) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int S = ALONE ? 1 : (int)cluster.num_blocks(), rank = ALONE ? 0 : (int)cluster.block_rank();
    __shared__ __align__(16) uint32_t ws[4 * kLfG * 64];
    __shared__ long long part[kLfSamples][kMaxClasses];
    const int u = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int group = blockIdx.x / S;
    const int b = group * kLfSamples + u;
    pdl_wait();
    const int limbs = limb_count(*maxabs_wlr);
    // nothing in this launch reads what is cleared here
    if (blockIdx.x == 0 && threadIdx.x < n_zero) zero_words[threadIdx.x] = 0;
    const int j0 = rank * p.per, j1 = min(p.d, j0 + p.per);
    for (int gc = 0; gc < p.G; gc += kLfG) {
        const long long z = p.G <= 10 ? learn_pass<10>(p, limbs, b, gc, j0, j1, ws)
                                      : learn_pass<kLfG>(p, limbs, b, gc, j0, j1, ws);
        if (lane < min(kLfG, p.G - gc)) part[u][gc + lane] = z;
    }
    // sample v of the group is finished by warp v of CTA v mod S
    if (ALONE) __syncwarp();
    else cluster.sync();
    if (u % S == rank && b < p.B) {
        const int lab = labels[b];
        const bool bad = lab < 0 || lab >= p.G;
        uint64_t l1 = 0;
        for (int g = lane; g < p.G; g += 32) {
            long long z = 0;
            for (int r = 0; r < S; ++r) z += *cluster.map_shared_rank(&part[u][g], r);
            // NITRO-Scaling, SF = 2^8 d: floor(floor(z / 256) / d)
            const int64_t yhat = dv.floor_div((int64_t)z >> 8);
            const int64_t t = yhat - ((!bad && g == lab) ? 32 : 0);
            if (bad && g == 0) atomicOr(status, ST_BAD_LABEL);
            if (!fits_i32(t)) atomicOr(status, ST_OVERFLOW);
            grad_l[(int64_t)b * p.G + g] = (int32_t)t;
            l1 += abs_u32((int32_t)t);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) l1 += __shfl_xor_sync(kFull, l1, o);
        if (lane == 0 && l1) atomicMax(gl_bound, l1 > 0xffffffffull ? 0xffffffffu : (uint32_t)l1);
    }
    if (!ALONE) cluster.sync();      // the partial sums stay until every CTA has read them
}

// ---------------------------------------------------------------------------
// Linear forward layer, one launch: the learning layer's contraction over 16 outputs
// a cluster, then NITRO-Scaling, NITRO-ReLU and dropout on the summed values.  For
// few products it is bound by latency: 64 x 784 x 100 takes 4.3 us where input pack,
// tensor-core GEMM and epilogue as three launches took 9.8 us, 64 x 100 x 50 4.1
// against 17.1 us on the general CUDA-core GEMM.
// ---------------------------------------------------------------------------
struct LinFwdArgs {
    int alpha_inv, mu;
    FloorDiv dv;                   // divide by the input width (after >> 8)
    int8_t* act;
    int8_t* out2;                  // may be null
    int8_t* region;
};
template <bool ALONE>
__global__ void __launch_bounds__(256) k_lin_fwd(const LearnArgs p, const LinFwdArgs o,
                                                 const uint32_t* maxabs_w, DropoutArgs drop) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int S = ALONE ? 1 : (int)cluster.num_blocks(), rank = ALONE ? 0 : (int)cluster.block_rank();
    __shared__ __align__(16) uint32_t ws[4 * kLfG * 64];
    __shared__ long long part[kLfSamples][kLfG];
    const int u = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int groups = (p.B + kLfSamples - 1) / kLfSamples;
    const int chunk = (int)(blockIdx.x / S) / groups, group = (int)(blockIdx.x / S) - chunk * groups;
    const int gc = chunk * kLfG;
    pdl_wait();
    const int limbs = limb_count(*maxabs_w);
    const int j0 = rank * p.per, j1 = min(p.d, j0 + p.per);
    const long long z = learn_pass<kLfG>(p, limbs, group * kLfSamples + u, gc, j0, j1, ws);
    if (lane < kLfG) part[u][lane] = z;
    if (ALONE) __syncthreads();
    else cluster.sync();
    for (int i = threadIdx.x; i < kLfSamples * kLfG; i += 256) {
        const int v = i / kLfG, g = i - v * kLfG, b = group * kLfSamples + v;
        if (v % S != rank || b >= p.B || gc + g >= p.G) continue;
        long long t = 0;
        for (int r = 0; r < S; ++r) t += *cluster.map_shared_rank(&part[v][g], r);
        const int64_t zs = o.dv.floor_div((int64_t)t >> 8);
        const int64_t e = (int64_t)b * p.G + gc + g;
        int rg = relu_region(zs);
        int8_t val = (int8_t)relu_value(zs, o.alpha_inv, o.mu);
        if (drop.p16 && dropout_drop(drop.seed, *drop.step, drop.layer, (uint64_t)e, drop.p16)) {
            rg = kRegionDropped;
            val = 0;
        }
        o.region[e] = (int8_t)rg;
        o.act[e] = val;
        if (o.out2) o.out2[e] = val;
    }
    if (!ALONE) cluster.sync();      // the partial sums stay until every CTA has read them
}

// Weight gradient of a linear layer: dW[o][i] = sum_b d[b][o] a[b][i], 16 outputs x
// 64 inputs per CTA, four inputs a thread, the samples in slabs through shared
// memory.  Few products: bound by latency, some 2.3 us a slab, so the slabs are shared
// out over CTAs (blockIdx.y, `per` samples each) that add into a cleared dW.  A backward
// of 64 x 784 x 100 with it takes 13.7 us, 19.7 us with the general CUDA-core GEMM, which
// decodes an index for every operand it stages; of 4096 x 64 x 64 25 us, 366 with all
// samples in one CTA a tile.
constexpr int kLwB = 32;           // samples per slab
__global__ void __launch_bounds__(256) k_lin_wgrad(const int8_t* __restrict__ a,
                                                   const int32_t* __restrict__ dl, int B, int in,
                                                   int out, int per, int64_t* __restrict__ dw) {
    pdl_wait();
    __shared__ int32_t ds[kLwB][16];
    __shared__ __align__(4) int8_t as[kLwB][64];
    const int ti = (in + 63) / 64;
    const int i0 = (int)(blockIdx.x % ti) * 64, o0 = (int)(blockIdx.x / ti) * 16;
    const int oi = threadIdx.x >> 4, q = threadIdx.x & 15;
    int64_t acc[4] = {0, 0, 0, 0};
    const int b_end = min(B, ((int)blockIdx.y + 1) * per);
    for (int b0 = (int)blockIdx.y * per; b0 < b_end; b0 += kLwB) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kLwB * 16 / 256; ++k) {
            const int e = threadIdx.x + 256 * k, b = e >> 4, c = e & 15;
            ds[b][c] = b0 + b < b_end && o0 + c < out ? dl[(int64_t)(b0 + b) * out + o0 + c] : 0;
        }
#pragma unroll
        for (int k = 0; k < kLwB * 64 / 256; ++k) {
            const int e = threadIdx.x + 256 * k, b = e >> 6, c = e & 63;
            as[b][c] = b0 + b < b_end && i0 + c < in ? a[(int64_t)(b0 + b) * in + i0 + c] : (int8_t)0;
        }
        __syncthreads();
        const auto add = [&](int b) {
            const int32_t d = ds[b][oi];
            const char4 v = *reinterpret_cast<const char4*>(&as[b][4 * q]);
            acc[0] += (int64_t)d * v.x;
            acc[1] += (int64_t)d * v.y;
            acc[2] += (int64_t)d * v.z;
            acc[3] += (int64_t)d * v.w;
        };
        if (b_end - b0 > 8) {                  // zeros past the last sample
#pragma unroll 8
            for (int b = 0; b < kLwB; ++b) add(b);
        } else {
            for (int b = 0; b < b_end - b0; ++b) add(b);
        }
    }
    if (o0 + oi >= out) return;
    int64_t* row = dw + (int64_t)(o0 + oi) * in;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (i0 + 4 * q + k >= in) break;
        if (gridDim.y > 1)
            atomicAdd(reinterpret_cast<unsigned long long*>(row + i0 + 4 * q + k), (unsigned long long)acc[k]);
        else
            row[i0 + 4 * q + k] = acc[k];
    }
}

// The last CTAs of the kernel after k_learn_fwd: SSE, loss = floor(SSE / 2), max
// |grad_L| and, with wlr_max != null, the int64 exactness bound of grad_L W_lr.
// One CTA forms them up to kTailValues values; above, several add their shares
// into *sse and *maxabs_gl (cleared by k_learn_fwd) and the last one ends.
struct LossTail {
    const int32_t* grad_l;
    int B, G;
    unsigned long long* sse;
    int64_t* loss;               // may be null
    uint32_t* maxabs_gl;
    uint32_t* ticket;            // cleared by k_learn_fwd
    const uint32_t* wlr_max;
    uint32_t* status;
};
constexpr int kTailValues = 8192;
__device__ __forceinline__ void loss_tail(const LossTail& t, int cta, int ctas) {
    const int64_t n = (int64_t)t.B * t.G;
    unsigned long long ss = 0;
    uint32_t mx = 0;
    for (int64_t i = (int64_t)cta * blockDim.x + threadIdx.x; i < n; i += (int64_t)ctas * blockDim.x) {
        const int32_t v = t.grad_l[i];
        ss += (unsigned long long)((int64_t)v * v);              // modulo 2^64
        mx = max(mx, abs_u32(v));
    }
    __shared__ unsigned long long sum;
    __shared__ uint32_t top;
    if (threadIdx.x == 0) {
        sum = 0;
        top = 0;
    }
    __syncthreads();
#pragma unroll
    for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(kFull, ss, off);
    mx = __reduce_max_sync(kFull, mx);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&sum, ss);
        atomicMax(&top, mx);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long total = sum;
        uint32_t most = top;
        if (ctas > 1) {
            atomicAdd(t.sse, total);
            atomicMax(t.maxabs_gl, most);
            __threadfence();
            if (atomicAdd(t.ticket, 1u) != (uint32_t)ctas - 1) return;
            __threadfence();
            total = atomicAdd(t.sse, 0ull);
            most = atomicMax(t.maxabs_gl, 0u);
        } else {
            *t.sse = total;
            *t.maxabs_gl = most;
        }
        if (t.loss) *t.loss = fdiv64((int64_t)total, 2);
        if (t.wlr_max && int64_bound_exceeded(most, *t.wlr_max, t.G)) atomicOr(t.status, ST_OVERFLOW);
    }
}

// ---------------------------------------------------------------------------
// Gradient at a layer output -> delta at its pre-activation.
// ---------------------------------------------------------------------------
__global__ void k_grad_to_delta(DeltaSrc src, LayerGeom g, int B, int alpha_inv,
                                const int8_t* __restrict__ region,
                                const int8_t* __restrict__ argmax, int32_t* __restrict__ delta,
                                uint32_t* maxabs_delta, uint32_t* status) {
    pdl_wait();
    const int64_t out_f = (int64_t)g.oh * g.ow * g.cout;
    const int64_t n = (int64_t)B * out_f;
    if (blockIdx.x == 0 && threadIdx.x == 0 &&
        int64_bound_exceeded(*src.maxabs_a, *src.maxabs_b, src.bound_k))
        atomicOr(status, ST_OVERFLOW);
    uint32_t mx = 0;
    bool ovf = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = i / out_f, q = i - b * out_f;
        const int64_t gv = src.g64[i];
        ovf |= !fits_i32(gv);
        const int32_t gs = (int32_t)gv;
        if (g.pool) {
            const int c = (int)(q % g.cout);
            const int64_t r = q / g.cout;
            const int ox = (int)(r % g.ow), oy = (int)(r / g.ow);
            const int am = argmax[i];
            // the window, with what a floor-sized pool drops at the last row and column, so
            // that every position is written (with a clear of delta before the launch the
            // backward of a 15 x 15, 60-channel conv and a linear layer at batch 128 took 99.7
            // us, so 97.7; 33 x 33, 12 channels, at batch 64 180.6 and 178.8)
            const int ny = oy + 1 == g.oh ? g.h - 2 * oy : 2, nx = ox + 1 == g.ow ? g.w - 2 * ox : 2;
            for (int y = 0; y < ny; ++y)
                for (int x = 0; x < nx; ++x) {
                    const int64_t pi = ((b * g.h + 2 * oy + y) * g.w + 2 * ox + x) * g.cout + c;
                    const bool hit = y < 2 && x < 2 && 2 * y + x == am;
                    const int32_t dv = hit ? relu_backward(gs, region[pi], alpha_inv) : 0;
                    delta[pi] = dv;
                    mx = max(mx, abs_u32(dv));
                }
        } else {
            const int32_t dv = relu_backward(gs, region[i], alpha_inv);
            delta[i] = dv;
            mx = max(mx, abs_u32(dv));
        }
    }
    block_maximum(mx, ovf, maxabs_delta, status);
}

// ---------------------------------------------------------------------------
// Learning-layer max-pool (Sec. 3.3, z^mp; window from d^lr, App. B): one
// thread per pooled element, channel fastest, so a warp reads 32 consecutive
// channels of each window row.  First maximum in row-major window order.
// ---------------------------------------------------------------------------
__global__ void k_lr_pool_fwd(const int8_t* __restrict__ a, int B, int H, int W, int C, int kh,
                              int kw, int ph, int pw, int8_t* __restrict__ out,
                              uint8_t* __restrict__ am) {
    pdl_wait();
    const int64_t n = (int64_t)B * ph * pw * C;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        int64_t r = i / C;
        const int x = (int)(r % pw);
        r /= pw;
        const int y = (int)(r % ph);
        const int64_t b = r / ph;
        const int8_t* p = a + ((b * H + (int64_t)y * kh) * W + (int64_t)x * kw) * C + c;
        int best = 0, bestv = p[0];
        for (int u = 0; u < kh; ++u)
            for (int v = 0; v < kw; ++v) {
                const int val = p[((int64_t)u * W + v) * C];
                if (val > bestv) { bestv = val; best = u * kw + v; }
            }
        out[i] = (int8_t)bestv;
        am[i] = (uint8_t)best;
    }
}

// Same, four channels per thread (C % 4 == 0, 4-byte aligned buffers): signed
// SIMD byte maxima, and a window position replaced only where a later value
// is strictly greater (the first maximum wins).
__global__ void k_lr_pool_fwd4(const int8_t* __restrict__ a, int B, int H, int W, int C, int kh,
                               int kw, int ph, int pw, FloorDiv32 dv_c4, FloorDiv32 dv_pw,
                               FloorDiv32 dv_ph, int8_t* __restrict__ out,
                               uint8_t* __restrict__ am) {
    pdl_wait();
    const int C4 = C >> 2;
    const uint32_t n4 = (uint32_t)B * ph * pw * C4;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x) {
        const uint32_t pix = dv_c4.udiv(i);
        const int c = (int)(i - pix * C4) * 4;
        const uint32_t r = dv_pw.udiv(pix);
        const int x = (int)(pix - r * pw);
        const uint32_t b = dv_ph.udiv(r);
        const int y = (int)(r - b * ph);
        const int8_t* p = a + ((b * H + (uint32_t)(y * kh)) * W + (uint32_t)(x * kw)) * C + c;
        uint32_t best = *reinterpret_cast<const uint32_t*>(p), pos = 0;
        for (int u = 0; u < kh; ++u)
            for (int v = 0; v < kw; ++v) {
                const uint32_t val = *reinterpret_cast<const uint32_t*>(p + (u * W + v) * C);
                const uint32_t gt = __vcmpgts4(val, best);
                best = __vmaxs4(best, val);
                pos = (pos & ~gt) | ((uint32_t)(u * kw + v) * 0x01010101u & gt);
            }
        reinterpret_cast<uint32_t*>(out)[i] = best;
        reinterpret_cast<uint32_t*>(am)[i] = pos;
    }
}

// ---------------------------------------------------------------------------
// Learning-layer backward through the pool, into the last layer's delta.  One
// thread per pre-pool element (b, y, x, c) of that conv layer: it receives a
// gradient only if it won its 2x2 window (when the layer pools) and the
// pooled position won its learning-pool window; that thread alone forms
// delta_fw = sum_g grad_L[b][g] W_lr[g][f] of the learning feature f (modulo
// 2^64, int32 storage rule) and applies NITRO-ReLU backward.  Every element is
// written, so no clearing pass is needed.
// ---------------------------------------------------------------------------
__global__ void k_lrpool_to_delta(const int32_t* __restrict__ gl, const int32_t* __restrict__ wlr,
                                  int G, int d, LayerGeom g, LrPoolGeom lp, int B,
                                  const uint8_t* __restrict__ lam,
                                  const int8_t* __restrict__ argmax,
                                  const int8_t* __restrict__ region, FloorDiv32 alpha,
                                  int32_t* __restrict__ delta, const uint32_t* maxabs_gl,
                                  const uint32_t* maxabs_wlr, uint32_t* maxabs_delta,
                                  uint32_t* status) {
    pdl_wait();
    const int C = g.cout;
    const int64_t n = (int64_t)B * g.h * g.w * C;
    if (blockIdx.x == 0 && threadIdx.x == 0 && int64_bound_exceeded(*maxabs_gl, *maxabs_wlr, G))
        atomicOr(status, ST_OVERFLOW);
    uint32_t mx = 0;
    bool ovf = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        int64_t r = i / C;
        const int x = (int)(r % g.w);
        r /= g.w;
        const int y = (int)(r % g.h);
        const int64_t b = r / g.h;
        int qy = y, qx = x;
        bool hit = true;
        if (g.pool) {
            qy = y >> 1;
            qx = x >> 1;
            hit = qy < g.oh && qx < g.ow &&
                  argmax[((b * g.oh + qy) * g.ow + qx) * C + c] == (((y & 1) << 1) | (x & 1));
        }
        int32_t dv = 0;
        if (hit) {
            const int wy = qy / lp.kh, wx = qx / lp.kw;
            hit = wy < lp.ph && wx < lp.pw &&
                  lam[((b * lp.ph + wy) * lp.pw + wx) * C + c] ==
                      (qy - wy * lp.kh) * lp.kw + (qx - wx * lp.kw);
            if (hit) {
                const int64_t f = ((int64_t)wy * lp.pw + wx) * C + c;
                uint64_t acc = 0;   // modulo 2^64, exact below the bound
                for (int k = 0; k < G; ++k)
                    acc += (uint64_t)((int64_t)gl[b * G + k] * wlr[(int64_t)k * d + f]);
                const int64_t gv = (int64_t)acc;
                ovf |= !fits_i32(gv);
                const int32_t gs = (int32_t)gv;
                const int rg = region[i];
                dv = rg == 1 ? alpha.floor_div(gs) : (rg == 2 ? gs : 0);
            }
        }
        delta[i] = dv;
        mx = max(mx, abs_u32(dv));
    }
    block_maximum(mx, ovf, maxabs_delta, status);
}

// Same by windows, four channels per thread (C % 4 == 0): a thread takes the
// learning feature of one (sample, window, four channels), finds the one
// pre-pool position each of its channels routes to (window maximum, then 2x2
// maximum), forms its delta there and writes the window, zeros elsewhere, 16
// bytes a position; the last window of a row or column also writes what the
// floor-sized pools drop.  blockIdx.y takes a share of the window's rows.  Bound by
// the delta stores: looking the codes up per pre-pool element instead cost a
// chain of dependent loads for each of 8.4 M or 16.8 M elements.
// With planes != null the thread also writes delta's bf16 limb planes (the weight
// gradient's operand), as many as gl_bound max|W_lr| can need, so
// that no pass reads delta again; and the launch clears zero[0..n_zero).
__global__ void __launch_bounds__(256) k_lrpool_to_delta4(
    const int32_t* __restrict__ gl, const int32_t* __restrict__ wlr, int G, int d, LayerGeom g,
    LrPoolGeom lp, int B, FloorDiv32 dv_c4, FloorDiv32 dv_pw, FloorDiv32 dv_ph,
    const uint8_t* __restrict__ lam, const int8_t* __restrict__ argmax,
    const int8_t* __restrict__ region, FloorDiv32 alpha, int32_t* __restrict__ delta,
    uint16_t* __restrict__ planes, int64_t plane, int64_t* zero, int64_t n_zero,
    const uint32_t* maxabs_gl, const uint32_t* gl_bound, const uint32_t* maxabs_wlr,
    uint32_t* maxabs_delta, uint32_t* status) {
    pdl_wait();
    const int C = g.cout, C4 = g.cout >> 2;
    const uint32_t n4 = (uint32_t)B * lp.ph * lp.pw * C4;
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    {
        const int64_t cta = blockIdx.x + (int64_t)blockIdx.y * gridDim.x;
        const int64_t step = (int64_t)gridDim.x * gridDim.y * blockDim.x;
        for (int64_t k = cta * blockDim.x + threadIdx.x; k < n_zero; k += step) zero[k] = 0;
    }
    if (i == 0 && blockIdx.y == 0 && int64_bound_exceeded(*maxabs_gl, *maxabs_wlr, G))
        atomicOr(status, ST_OVERFLOW);
    int L = 0;
    if (planes) {
        const uint32_t gb = *gl_bound;
        const uint64_t bound = (uint64_t)gb * *maxabs_wlr;
        L = limb_count(gb == 0xffffffffu || bound > 0xffffffffull ? 0xffffffffu : (uint32_t)bound);
    }
    uint32_t mx = 0;
    bool ovf = false;
    if (i < n4) {
        const uint32_t win = dv_c4.udiv(i);
        const int c = (int)(i - win * C4) * 4;
        const uint32_t r = dv_pw.udiv(win);
        const int wx = (int)(win - r * lp.pw);
        const uint32_t b = dv_ph.udiv(r);
        const int wy = (int)(r - b * lp.ph);
        const int lg_kw = 31 - __clz(lp.kw);
        const uint32_t lw = *reinterpret_cast<const uint32_t*>(lam + (size_t)win * C + c);
        const int f0 = (wy * lp.pw + wx) * C + c;
        uint64_t acc[4] = {0, 0, 0, 0};       // modulo 2^64, exact below the bound
        const int32_t* wp = wlr + f0;
#pragma unroll 5
        for (int k = 0; k < G; ++k) {
            const int4 w = *reinterpret_cast<const int4*>(wp + (int64_t)k * d);
            const int64_t gv = gl[b * G + k];
            acc[0] += (uint64_t)(gv * w.x);
            acc[1] += (uint64_t)(gv * w.y);
            acc[2] += (uint64_t)(gv * w.z);
            acc[3] += (uint64_t)(gv * w.w);
        }
        const int s2 = g.pool ? 2 : 1;
        const int y0 = wy * lp.kh * s2, y1 = wy + 1 == lp.ph ? g.h : y0 + lp.kh * s2;
        const int x0 = wx * lp.kw * s2, x1 = wx + 1 == lp.pw ? g.w : x0 + lp.kw * s2;
        // row << 16 | column of the hit inside the window, and delta there: kh kw <= 256, so
        // a window, with what the pools cut off behind the last one, has at most 1023 a side
        int pos[4], v[4];
        uint32_t rg[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int code = (int)((lw >> (8 * j)) & 255u);
            int y = wy * lp.kh + (code >> lg_kw), x = wx * lp.kw + (code & (lp.kw - 1));
            if (g.pool) {
                const int am = argmax[((size_t)(b * g.oh + y) * g.ow + x) * C + c + j];
                y = 2 * y + (am >> 1);
                x = 2 * x + (am & 1);
            }
            rg[j] = (uint8_t)region[((size_t)(b * g.h + y) * g.w + x) * C + c + j];
            pos[j] = ((y - y0) << 16) | (x - x0);
        }
        uint32_t h01[4], h23[4];              // bf16 limbs of the four deltas
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t gv = (int64_t)acc[j];
            const bool mine = blockIdx.y == 0;
            ovf |= mine && !fits_i32(gv);
            const int32_t gs = (int32_t)gv;
            v[j] = rg[j] == 1 ? alpha.floor_div(gs) : (rg[j] == 2 ? gs : 0);
            mx = max(mx, mine ? abs_u32(v[j]) : 0u);
        }
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            h01[l] = limb_bf16x2(v[0], v[1], l);
            h23[l] = limb_bf16x2(v[2], v[3], l);
        }
        for (int y = y0 + blockIdx.y; y < y1; y += gridDim.y) {
            size_t o = ((size_t)(b * g.h + y) * g.w + x0) * C + c;
            for (int x = x0; x < x1; ++x, o += C) {
                const int at = ((y - y0) << 16) | (x - x0);
                const bool k0 = pos[0] == at, k1 = pos[1] == at, k2 = pos[2] == at, k3 = pos[3] == at;
                *reinterpret_cast<int4*>(delta + o) =
                    make_int4(k0 ? v[0] : 0, k1 ? v[1] : 0, k2 ? v[2] : 0, k3 ? v[3] : 0);
                const uint32_t m01 = (k0 ? 0xffffu : 0u) | (k1 ? 0xffff0000u : 0u);
                const uint32_t m23 = (k2 ? 0xffffu : 0u) | (k3 ? 0xffff0000u : 0u);
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    if (l >= L) break;
                    *reinterpret_cast<uint2*>(planes + l * plane + o) = make_uint2(h01[l] & m01, h23[l] & m23);
                }
            }
        }
    }
    block_maximum(mx, ovf, maxabs_delta, status);
}

// ---------------------------------------------------------------------------
// IntegerSGD (Algorithm 1).  CTAs first[i] .. first[i + 1) - 1 take tensor i; the
// last CTA to finish publishes the maxima (see SgdBatch::scratch).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int32_t sgd_one(const SgdTensor& t, int round_trunc, int32_t w32,
                                           int64_t g, uint32_t& mx, bool& ovf) {
    const int64_t w = w32;
    int64_t d;
    if (fits_i32(g)) d = round_trunc ? t.gdiv32.trunc_div((int32_t)g) : t.gdiv32.floor_div((int32_t)g);
    else d = round_trunc ? t.gdiv.trunc_div(g) : t.gdiv.floor_div(g);
    if (t.eta_inv != 0) d += round_trunc ? t.ediv32.trunc_div(w32) : t.ediv32.floor_div(w32);
    const int64_t nw = w - d;
    ovf |= !fits_i32(nw);
    const int32_t s = (int32_t)nw;
    mx = max(mx, abs_u32(s));
    return s;
}

// The updated weight w (element i of [Cout][9][cin]) into its four bf16 limb planes.
__device__ __forceinline__ void sgd_planes(const SgdTensor& t, int64_t i, int32_t w) {
    const uint32_t q = t.cin_div.udiv((uint32_t)i);
    const int ci = (int)(i - (int64_t)q * t.cin);
    const int tap = (int)(q % 9u), co = (int)(q / 9u);
    uint16_t* p = t.planes + (int64_t)co * t.row_k + tap * t.tap_k + ci;
#pragma unroll
    for (int l = 0; l < 4; ++l) p[l * t.plane] = (uint16_t)limb_bf16x2(w, w, l);
}

// Four consecutive updated weights into their limb planes when the planes are
// laid out like W (linear layers; convs with Cin a multiple of 64), 8 bytes a
// plane at p + l * plane; a plane whose four limbs stay as they were is not stored.
__device__ __forceinline__ void sgd_planes4(uint16_t* p, int64_t plane, int4 w, int4 old) {
    // digits 0..2 of x are bytes 0..2 of x + 0x808080 (less 128), digit 3 its top byte
    // and, where that wraps, its sign
    const auto diff = [](int a, int b) {
        return (((uint32_t)a + 0x808080u) ^ ((uint32_t)b + 0x808080u)) | (((uint32_t)a ^ (uint32_t)b) & 0x80000000u);
    };
    const uint32_t x = diff(w.x, old.x) | diff(w.y, old.y) | diff(w.z, old.z) | diff(w.w, old.w);
#pragma unroll
    for (int l = 0; l < 4; ++l)
        if (x >> (8 * l) & 255u)
            *reinterpret_cast<uint2*>(p + l * plane) =
                make_uint2(limb_bf16x2(w.x, w.y, l), limb_bf16x2(w.z, w.w, l));
}

// Four consecutive weights per thread and round (16-byte loads of W, two of dW;
// the tensors are this library's own 256-byte aligned buffers), the tail singly.
// Bound by memory traffic: W and dW are read (12 bytes a weight), and only what
// changes is written - the planes always hold all four limbs of W, so a group of
// weights that stay, or a plane whose digits stay (the upper ones, nearly always),
// needs no store.  24 bytes a weight before; the 21 M weights of the wide MLP took
// 171 us a step in four launches, 112 with the stores left out, 97 with the changed
// planes read off one exclusive or instead of splitting old and new, and 95 at five
// CTAs an SM.
// A gradient that fits 32 bits takes the 32-bit divide.
__global__ void __launch_bounds__(256, 5) k_integersgd(const SgdBatch bt) {
    pdl_wait();
    int ti = 0;
    while (ti + 1 < bt.count && (int)blockIdx.x >= bt.first[ti + 1]) ++ti;
    const SgdTensor& t = bt.t[ti];
    const int64_t tid = (int64_t)((int)blockIdx.x - bt.first[ti]) * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)(bt.first[ti + 1] - bt.first[ti]) * blockDim.x;
    uint32_t mx = 0;
    bool ovf = false;
    const int64_t n4 = t.n / 4;
    const auto group = [&](int64_t i, const int4 w, const longlong2 g0, const longlong2 g1) {
        int4 o;
        o.x = sgd_one(t, bt.round_trunc, w.x, g0.x, mx, ovf);
        o.y = sgd_one(t, bt.round_trunc, w.y, g0.y, mx, ovf);
        o.z = sgd_one(t, bt.round_trunc, w.z, g1.x, mx, ovf);
        o.w = sgd_one(t, bt.round_trunc, w.w, g1.y, mx, ovf);
        if (o.x == w.x && o.y == w.y && o.z == w.z && o.w == w.w) return;
        reinterpret_cast<int4*>(t.w)[i] = o;
        if (t.planes && t.contig) {
            sgd_planes4(t.planes + 4 * i, t.plane, o, w);
        } else if (t.planes) {
            if (o.x != w.x) sgd_planes(t, 4 * i, o.x);
            if (o.y != w.y) sgd_planes(t, 4 * i + 1, o.y);
            if (o.z != w.z) sgd_planes(t, 4 * i + 2, o.z);
            if (o.w != w.w) sgd_planes(t, 4 * i + 3, o.w);
        }
    };
    const int4* wv = reinterpret_cast<const int4*>(t.w);
    const longlong2* gv = reinterpret_cast<const longlong2*>(t.dw);
    int64_t i = tid;
    for (; i + stride < n4; i += 2 * stride) {   // two groups' loads in flight
        const int64_t j = i + stride;
        const int4 wa = wv[i], wb = wv[j];
        const longlong2 a0 = gv[2 * i], a1 = gv[2 * i + 1], b0 = gv[2 * j], b1 = gv[2 * j + 1];
        group(i, wa, a0, a1);
        group(j, wb, b0, b1);
    }
    if (i < n4) group(i, wv[i], gv[2 * i], gv[2 * i + 1]);
    for (int64_t k = 4 * n4 + tid; k < t.n; k += stride) {
        const int32_t nw = sgd_one(t, bt.round_trunc, t.w[k], t.dw[k], mx, ovf);
        t.w[k] = nw;
        if (t.planes) sgd_planes(t, k, nw);
    }
    block_maximum(mx, ovf, &bt.scratch[ti], bt.status);
    if (threadIdx.x == 0) __threadfence();     // the CTA's maximum, before its ticket
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&bt.scratch[kMaxSgdTensors], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if ((int)threadIdx.x < bt.count)
        *bt.t[threadIdx.x].maxabs_w = atomicExch(&bt.scratch[threadIdx.x], 0u);
    if (threadIdx.x == 0) {
        bt.scratch[kMaxSgdTensors] = 0;
        bt.scratch[kMaxSgdTensors + 1] = 0;    // the bound of |grad_L|, of the step that ends
        // one block step taken: advance the dropout step counter
        if (bt.step) *bt.step += 1u;
    }
    __syncthreads();
    for (int i = threadIdx.x; bt.host_words && i < bt.n_words; i += blockDim.x)
        bt.host_words[i] = __ldcg(bt.words + i);
}

// ---------------------------------------------------------------------------
// Learning-layer backward, one launch of three kinds of CTAs that wait on nothing
// of one another:
//   dW_lr[g][q] = sum_b grad_L[b][g] a[b][q] for 16 V features: sixteen sample lanes with
//     the sums of GM classes in registers, added through shared memory, all samples and
//     written once (no clearing, no atomics), or, at large batches (SHARED), some samples
//     each and added into a cleared array;
//   delta_fw[b][q] = sum_g grad_L[b][g] W_lr[g][q] (int32 storage rule) for 16 V features
//     x 16 samples, routed through max-pool backward and NITRO-ReLU backward into the
//     last layer's delta, every position written, with the delta's bf16 limb planes
//     (planes != null; as many as gl_bound max|W_lr| can need), so that no pass
//     reads delta again; these CTAs also clear zero[0..n_zero);
//   the loss (loss_tail).
// V features a thread: four channels of one output position when the channel count is
// a multiple of 4 and the arrays are aligned for it, else one.  dW_lr sums in 32 bits
// where gl_bound allows (ten classes a pass, four in 64 bits) and delta_fw where
// gl_bound max|W_lr| does, which leaves room for four CTAs an SM.  First block of a
// 64-channel 32x32 network at batch 64 (2 M features): 27 us; 64-bit sums of ten
// classes at one CTA an SM 64, 32-bit sums at three 31; five CTAs an SM with half the
// classes a pass 25, but 4 us more where d is small.  Bound by the instructions and
// latency of the delta part.  One CTA doing both parts for 64 features x 32 samples
// around a barrier, dW_lr by atomics into an array cleared before, and a pass that
// split delta: VGG-style graph 479 us a step, odd block 173, small CNN 101, VGG8B 727;
// so 464 to 468, 164, 95, 715 to 724.
// ---------------------------------------------------------------------------
struct LrBackArgs {
    const int8_t* a;
    const int32_t* gl;
    const int32_t* wlr;
    int B, G, d;
    int64_t* dwlr;
    // delta part (delta null: dW_lr only)
    LayerGeom lg;
    FloorDiv32 alpha, dv_c, dv_ow;
    const int8_t* region;
    const int8_t* argmax;
    int32_t* delta;
    uint16_t* planes;
    int64_t plane;
    int64_t* zero;
    int64_t n_zero;
    const uint32_t* gl_bound;      // see simt_learn_fwd
    const uint32_t* maxabs_wlr;
    uint32_t* maxabs_delta;
    uint32_t* status;
    // dW_lr CTAs: dw_x along the features, for each dw_per samples (dw_ctas > dw_x: they add
    // into a cleared dW_lr)
    int dw_x, dw_per, dw_ctas, delta_x, delta_ctas, tail_ctas;
};
constexpr int kLbSlab = 128;       // samples taken at once: eight a thread
union LrShared {
    int32_t gl[kLbSlab][16];
    long long red[8][4][64];
};

// T int32 where the sums of a thread's samples fit
template <int V, int GM, typename T, bool SHARED>
__device__ __forceinline__ void lr_dw(const LrBackArgs& p, LrShared& sm) {
    const int quad = threadIdx.x & 15, lane_s = threadIdx.x >> 4, warp = threadIdx.x >> 5;
    const int part = SHARED ? (int)blockIdx.x / p.dw_x : 0;
    const int b_begin = SHARED ? part * p.dw_per : 0, b_end = SHARED ? min(p.B, b_begin + p.dw_per) : p.B;
    const int q0 = (SHARED ? blockIdx.x - part * p.dw_x : blockIdx.x) * 16 * V, q = q0 + quad * V;
    for (int gc = 0; gc < p.G; gc += GM) {
        T acc[GM][V];
#pragma unroll
        for (int g = 0; g < GM; ++g)
#pragma unroll
            for (int j = 0; j < V; ++j) acc[g][j] = 0;
        for (int b0 = SHARED ? b_begin : 0; b0 < (SHARED ? b_end : p.B); b0 += kLbSlab) {
            const int nb = min(kLbSlab, (SHARED ? b_end : p.B) - b0);
            uint32_t aw[kLbSlab / 16];
#pragma unroll
            for (int i = 0; i < kLbSlab / 16; ++i) {
                const int b = lane_s + 16 * i;
                aw[i] = 0;
                if (b < nb && q < p.d) {
                    const int8_t* src = p.a + (int64_t)(b0 + b) * p.d + q;
                    aw[i] = V == 4 ? *reinterpret_cast<const uint32_t*>(src) : (uint32_t)(uint8_t)*src;
                }
            }
            __syncthreads();
            for (int i = threadIdx.x; i < nb * GM; i += 256) {
                const int b = i / GM, g = i - b * GM;
                sm.gl[b][g] = gc + g < p.G ? p.gl[(int64_t)(b0 + b) * p.G + gc + g] : 0;
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kLbSlab / 16; ++i) {
                const int b = lane_s + 16 * i;
                if (b >= nb) break;
#pragma unroll
                for (int g = 0; g < GM; ++g) {
                    const T gv = sm.gl[b][g];
#pragma unroll
                    for (int j = 0; j < V; ++j) acc[g][j] += gv * (int8_t)(aw[i] >> (8 * j));
                }
            }
        }
        // two sample lanes of a warp, then the eight warps, four classes at a time
#pragma unroll
        for (int g0 = 0; g0 < GM; g0 += 4) {
            __syncthreads();
#pragma unroll
            for (int g = g0; g < g0 + 4 && g < GM; ++g)
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const long long t = (long long)acc[g][j] + __shfl_xor_sync(kFull, acc[g][j], 16);
                    if ((threadIdx.x & 16) == 0) sm.red[warp][g - g0][quad * V + j] = t;
                }
            __syncthreads();
            for (int i = threadIdx.x; i < 4 * 16 * V; i += 256) {
                const int g = i / (16 * V), f = i - g * 16 * V;
                if (g0 + g >= GM || gc + g0 + g >= p.G || q0 + f >= p.d) continue;
                long long t = 0;
#pragma unroll
                for (int w = 0; w < 8; ++w) t += sm.red[w][g][f];
                if constexpr (SHARED)
                    atomicAdd(reinterpret_cast<unsigned long long*>(p.dwlr + (int64_t)(gc + g0 + g) * p.d + q0 + f),
                              (unsigned long long)t);
                else
                    p.dwlr[(int64_t)(gc + g0 + g) * p.d + q0 + f] = t;
            }
        }
    }
}

// T uint32 where |delta_fw| is known to fit int32, uint64 (modulo 2^64) elsewhere
template <int V, typename T>
__device__ __forceinline__ void lr_delta(const LrBackArgs& p, int cta, uint64_t bound) {
    for (int64_t k = (int64_t)cta * 256 + threadIdx.x; k < p.n_zero; k += (int64_t)p.delta_ctas * 256) p.zero[k] = 0;
    const int by = cta / p.delta_x, bx = cta - by * p.delta_x;
    const int q = (bx * 16 + (threadIdx.x & 15)) * V, b = by * 16 + (threadIdx.x >> 4);
    uint32_t mx = 0;
    bool ovf = false;
    if (q < p.d && b < p.B) {
        const LayerGeom& lg = p.lg;
        const int pix = (int)p.dv_c.udiv((uint32_t)q), c = q - pix * lg.cout;
        const int oy = (int)p.dv_ow.udiv((uint32_t)pix), ox = pix - oy * lg.ow;
        const int s2 = lg.pool ? 2 : 1;
        // codes of the V channels first
        const uint32_t base = (uint32_t)((b * lg.h + s2 * oy) * lg.w + s2 * ox) * lg.cout + c;
        const uint32_t row = (uint32_t)lg.w * lg.cout;
        const auto codes = [](const int8_t* at) {
            return V == 4 ? *reinterpret_cast<const uint32_t*>(at) : (uint32_t)(uint8_t)*at;
        };
        uint32_t am = 0, r[4];
        r[0] = codes(p.region + base);
        if (lg.pool) {
            am = codes(p.argmax + (int64_t)b * p.d + q);
            r[1] = codes(p.region + base + lg.cout);
            r[2] = codes(p.region + base + row);
            r[3] = codes(p.region + base + row + lg.cout);
        }
        T acc[V];
#pragma unroll
        for (int j = 0; j < V; ++j) acc[j] = 0;
        const int32_t* wp = p.wlr + q;
        const int32_t* gp = p.gl + (int64_t)b * p.G;
        const auto mul = [](int32_t x, int32_t y) {
            return sizeof(T) == 4 ? (T)((uint32_t)x * (uint32_t)y) : (T)((int64_t)x * y);
        };
#pragma unroll 5
        for (int g = 0; g < p.G; ++g) {
            const int32_t gv = gp[g];
            if (V == 4) {
                const int4 w = *reinterpret_cast<const int4*>(wp + (int64_t)g * p.d);
                acc[0] += mul(gv, w.x);
                acc[1 % V] += mul(gv, w.y);
                acc[2 % V] += mul(gv, w.z);
                acc[3 % V] += mul(gv, w.w);
            } else {
                acc[0] += mul(gv, wp[(int64_t)g * p.d]);
            }
        }
        int32_t v[4] = {0, 0, 0, 0};
        int code[4] = {0, 0, 0, 0};
#pragma unroll
        for (int j = 0; j < V; ++j) {
            if (sizeof(T) == 8) ovf |= !fits_i32((int64_t)acc[j]);
            const int32_t gs = (int32_t)acc[j];
            code[j] = lg.pool ? (int)((am >> (8 * j)) & 3u) : 0;
            // region byte at the recorded window position of channel j
            const uint32_t rs = code[j] == 0 ? r[0] : (code[j] == 1 ? r[1] : (code[j] == 2 ? r[2] : r[3]));
            const uint32_t rg = (rs >> (8 * j)) & 255u;
            // NITRO-ReLU backward: piece 1 -> floor(g / alpha_inv), piece 2 -> g, else 0
            v[j] = rg == 1 ? p.alpha.floor_div(gs) : (rg == 2 ? gs : 0);
            mx = max(mx, abs_u32(v[j]));
        }
        int L = 0;
        uint32_t h01[4], h23[4];
        if (V == 4 && p.planes) {
            L = limb_count(bound > 0xffffffffull ? 0xffffffffu : (uint32_t)bound);
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                h01[l] = limb_bf16x2(v[0], v[1], l);
                h23[l] = limb_bf16x2(v[2], v[3], l);
            }
        }
        // the window, with what a floor-sized pool drops at the last row and column
        const int ny = lg.pool ? (oy + 1 == lg.oh ? lg.h - 2 * oy : 2) : 1;
        const int nx = lg.pool ? (ox + 1 == lg.ow ? lg.w - 2 * ox : 2) : 1;
        for (int y = 0; y < ny; ++y)
            for (int x = 0; x < nx; ++x) {
                const int at = y < 2 && x < 2 ? 2 * y + x : 4;
                const uint32_t o = base + y * row + x * lg.cout;
                if (V == 4) {
                    const bool k0 = code[0] == at, k1 = code[1] == at, k2 = code[2] == at, k3 = code[3] == at;
                    *reinterpret_cast<int4*>(p.delta + o) =
                        make_int4(k0 ? v[0] : 0, k1 ? v[1] : 0, k2 ? v[2] : 0, k3 ? v[3] : 0);
                    const uint32_t m01 = (k0 ? 0xffffu : 0u) | (k1 ? 0xffff0000u : 0u);
                    const uint32_t m23 = (k2 ? 0xffffu : 0u) | (k3 ? 0xffff0000u : 0u);
#pragma unroll
                    for (int l = 0; l < 4; ++l) {
                        if (l >= L) break;
                        *reinterpret_cast<uint2*>(p.planes + l * p.plane + o) = make_uint2(h01[l] & m01, h23[l] & m23);
                    }
                } else {
                    p.delta[o] = code[0] == at ? v[0] : 0;
                }
            }
    }
    block_maximum(mx, ovf, p.maxabs_delta, p.status);
}

template <int V, bool SHARED>
__global__ void __launch_bounds__(256, 4) k_lr_backward(const LrBackArgs p, const LossTail tail) {
    __shared__ LrShared sm;
    pdl_wait();
    const int cta = blockIdx.x;
    if (cta < p.dw_ctas) {
        if ((uint64_t)*p.gl_bound * 128u * (uint64_t)(((SHARED ? p.dw_per : p.B) + 15) / 16) <= 0x7fffffffull)
            lr_dw<V, 10, int32_t, SHARED>(p, sm);
        else
            lr_dw<V, 4, long long, SHARED>(p, sm);
    } else if (cta < p.dw_ctas + p.delta_ctas) {
        const uint32_t gb = *p.gl_bound;
        const uint64_t bound = (uint64_t)gb * *p.maxabs_wlr;
        if (gb != 0xffffffffu && bound <= 0x7fffffffull) lr_delta<V, uint32_t>(p, cta - p.dw_ctas, bound);
        else lr_delta<V, uint64_t>(p, cta - p.dw_ctas, gb == 0xffffffffu ? ~0ull : bound);
    } else {
        loss_tail(tail, cta - p.dw_ctas - p.delta_ctas, p.tail_ctas);
    }
}

inline int grid_for(int64_t n, int threads, int cap = 152 * 16) {
    int64_t g = (n + threads - 1) / threads;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

cudaError_t simt_gemm(int mode, const int8_t* act, const int32_t* grad, const int32_t* wts,
                      int64_t* out, int B, int H, int W, int Cin, int Cout, cudaStream_t s) {
    GemmParams p{act, grad, wts, out, 0, 0, 0, B, H, W, Cin, Cout, 0};
    const int P = B * H * W;
    switch (mode) {
        case GM_CONV_FWD: p.M = P; p.N = Cout; p.K = 9 * Cin; break;
        case GM_CONV_DGRAD: p.M = P; p.N = Cin; p.K = 9 * Cout; break;
        case GM_CONV_WGRAD: p.M = Cout; p.N = 9 * Cin; p.K = P; break;
        case GM_LIN_FWD: p.M = B; p.N = Cout; p.K = Cin; break;
        case GM_LIN_DGRAD: p.M = B; p.N = Cin; p.K = Cout; break;
        case GM_LIN_WGRAD: p.M = Cout; p.N = Cin; p.K = B; break;
        default: return cudaErrorInvalidValue;
    }
    if (p.M <= 0 || p.N <= 0) return cudaSuccess;
    const int tiles_m = (p.M + kTile - 1) / kTile, tiles_n = (p.N + kTile - 1) / kTile;
    // Split K over gridDim.z (64-bit atomics into a zeroed output, exact in any
    // order) until the grid holds about four CTAs per SM, keeping at least
    // 256 K per split.  Weight gradients always reduce over a long K; the
    // forward and input gradient need it when the output has few tiles (a
    // batch of 64 against a linear layer, a 4 x 4 conv map).
    int splits = 1;
    const int64_t tiles = (int64_t)tiles_m * tiles_n;
    if (mode == GM_CONV_WGRAD || mode == GM_LIN_WGRAD || tiles < 2 * 152) {
        const int64_t want = (4 * 152 + tiles - 1) / tiles;
        const int64_t maxs = (p.K + 255) / 256;
        splits = (int)(want < maxs ? want : maxs);
        if (splits < 1) splits = 1;
    }
    p.k_split = ((p.K + splits - 1) / splits + kTK - 1) / kTK * kTK;
    if (p.k_split == 0) p.k_split = kTK;
    splits = p.K > 0 ? (p.K + p.k_split - 1) / p.k_split : 1;
    if (splits > 1 || p.K == 0) {
        cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int64_t) * (size_t)p.M * p.N, s);
        if (e != cudaSuccess) return e;
        if (p.K == 0) return cudaSuccess;
    }
    dim3 grid(tiles_n, tiles_m, splits);
    static const int kIds[6] = {K_SIMT_CONV_FWD, K_SIMT_CONV_DGRAD, K_SIMT_CONV_WGRAD,
                                K_SIMT_LIN_FWD, K_SIMT_LIN_DGRAD, K_SIMT_LIN_WGRAD};
    ProfScope ps(kIds[mode], s, 2.0 * p.M * p.N * p.K, 0.0);
    switch (mode) {
        case GM_CONV_FWD: launch_k(k_gemm<GM_CONV_FWD>, grid, 256, 0, s, p); break;
        case GM_CONV_DGRAD: launch_k(k_gemm<GM_CONV_DGRAD>, grid, 256, 0, s, p); break;
        case GM_CONV_WGRAD: launch_k(k_gemm<GM_CONV_WGRAD>, grid, 256, 0, s, p); break;
        case GM_LIN_FWD: launch_k(k_gemm<GM_LIN_FWD>, grid, 256, 0, s, p); break;
        case GM_LIN_DGRAD: launch_k(k_gemm<GM_LIN_DGRAD>, grid, 256, 0, s, p); break;
        default: launch_k(k_gemm<GM_LIN_WGRAD>, grid, 256, 0, s, p); break;
    }
    return cudaGetLastError();
}

cudaError_t simt_preload_conv_fwd() {
    cudaFuncAttributes fa{};
    const cudaError_t e = cudaFuncGetAttributes(&fa, k_gemm<GM_CONV_FWD>);
    return e == cudaSuccess ? cudaFuncGetAttributes(&fa, k_fwd_epilogue) : e;
}

cudaError_t simt_fwd_epilogue(const int64_t* z, const LayerGeom& g, int B, int alpha_inv,
                              int mu, int8_t* out, int8_t* out2, int8_t* region,
                              int8_t* argmax, cudaStream_t s, const DropoutArgs* drop) {
    if (B <= 0) return cudaSuccess;
    const int64_t kdiv = g.kind == NITRO_CONV3X3 ? 9LL * g.cin : (int64_t)g.cin;
    const int64_t n = g.pool ? (int64_t)B * ((g.h + 1) / 2) * ((g.w + 1) / 2) * g.cout
                             : (int64_t)B * g.h * g.w * g.cout;
    DropoutArgs da{};
    if (drop && drop->p16) {
        if (g.pool || !drop->step) return cudaErrorInvalidValue;
        da = *drop;
    }
    ProfScope ps(K_FWD_EPILOGUE, s, 0.0, 0.0);
    launch_k(k_fwd_epilogue, grid_for(n, 256), 256, 0, s, z, g, B, alpha_inv, mu, kdiv, out, out2,
                                                    region, argmax, da);
    return cudaGetLastError();
}

cudaError_t simt_lr_pool_fwd(const int8_t* a, int B, int H, int W, int C, int kh, int kw,
                             int ph, int pw, int8_t* out, uint8_t* am, cudaStream_t s) {
    const int64_t n = (int64_t)B * ph * pw * C;
    if (n <= 0) return cudaSuccess;
    if (kh < 1 || kw < 1 || ph * kh > H || pw * kw > W || kh * kw > 256) return cudaErrorInvalidValue;
    ProfScope ps(K_LR_POOL, s, 0.0, (double)B * H * W * C + 2.0 * n);
    if (C % 4 == 0 && (((uintptr_t)a | (uintptr_t)out | (uintptr_t)am) & 3) == 0)
        launch_k(k_lr_pool_fwd4, grid_for(n / 4, 256), 256, 0, s,
            a, B, H, W, C, kh, kw, ph, pw, FloorDiv32::make((uint32_t)(C / 4)),
            FloorDiv32::make((uint32_t)pw), FloorDiv32::make((uint32_t)ph), out, am);
    else
        launch_k(k_lr_pool_fwd, grid_for(n, 256), 256, 0, s, a, B, H, W, C, kh, kw, ph, pw, out, am);
    return cudaGetLastError();
}

cudaError_t simt_lrpool_to_delta(const int32_t* gl, const int32_t* wlr, int G, int d,
                                 const LayerGeom& g, const LrPoolGeom& lp, int B,
                                 const uint8_t* am, const int8_t* argmax, const int8_t* region,
                                 int alpha_inv, int32_t* delta, uint16_t* planes, int64_t* zero,
                                 int64_t n_zero, bool* planes_done, const uint32_t* maxabs_gl,
                                 const uint32_t* gl_bound, const uint32_t* maxabs_wlr, uint32_t* maxabs_delta,
                                 uint32_t* status, cudaStream_t s) {
    const int64_t n = (int64_t)B * g.h * g.w * g.cout;
    if (n <= 0) return cudaSuccess;
    if (g.kind != NITRO_CONV3X3 || lp.ph * lp.kh > g.oh || lp.pw * lp.kw > g.ow ||
        (int64_t)lp.ph * lp.pw * g.cout != d || alpha_inv < 1)
        return cudaErrorInvalidValue;
    // bytes: region (1) and delta (4) per element, the two argmax codes per
    // pooled position, grad_L and the columns of W_lr read
    ProfScope ps(K_LRPOOL_TO_DELTA, s, 2.0 * B * d * G,
                 5.0 * n + (double)B * g.oh * g.ow * g.cout * (g.pool ? 1 : 0) + (double)B * d +
                     4.0 * G * (B + (double)d));
    const bool aligned = (((uintptr_t)am | (uintptr_t)region | (uintptr_t)delta | (uintptr_t)wlr |
                           (uintptr_t)(g.pool ? argmax : region)) & 15) == 0;
    const bool pow2 = (lp.kh & (lp.kh - 1)) == 0 && (lp.kw & (lp.kw - 1)) == 0;
    *planes_done = false;
    if (g.cout % 4 == 0 && aligned && pow2) {   // d = ph pw cout is then a multiple of 4
        // a thread per (sample, window, four channels); the rows of a window are
        // shared out until about 200 k threads store
        const int64_t threads = (int64_t)B * d / 4;
        const int rows = lp.kh * (g.pool ? 2 : 1);
        int64_t parts = 200000 / threads;
        parts = parts < 1 ? 1 : (parts > rows ? rows : parts);
        dim3 grid((unsigned)((threads + 255) / 256), (unsigned)parts);
        launch_k(k_lrpool_to_delta4, grid, 256, 0, s,
            gl, wlr, G, d, g, lp, B, FloorDiv32::make((uint32_t)(g.cout / 4)),
            FloorDiv32::make((uint32_t)lp.pw), FloorDiv32::make((uint32_t)lp.ph), am, argmax, region,
            FloorDiv32::make((uint32_t)alpha_inv), delta, planes, n, zero, zero ? n_zero : (int64_t)0,
            maxabs_gl, gl_bound, maxabs_wlr, maxabs_delta, status);
        *planes_done = planes != nullptr;
    } else {
        launch_k(k_lrpool_to_delta, grid_for(n, 256), 256, 0, s,
            gl, wlr, G, d, g, lp, B, am, argmax, region,
            FloorDiv32::make((uint32_t)alpha_inv), delta, maxabs_gl, maxabs_wlr, maxabs_delta,
            status);
    }
    return cudaGetLastError();
}

namespace {
// CTAs that share one sample group's features: as many as have a tile each, up to
// eight, while the launch stays below about two CTAs an SM (more would each do less
// than their launch and cluster barriers cost)
int learn_cluster(int64_t ctas, int d) {
    int S = 1;
    while (S < kLfCluster && S * kLfTile < d && ctas * S < 300) S *= 2;
    return S;
}
}  // namespace

cudaError_t simt_learn_fwd(const int8_t* a, const int32_t* wlr, const int32_t* labels, int B,
                           int d, int G, int32_t* grad_l, const uint32_t* maxabs_wlr,
                           uint32_t* status, uint32_t* zero_words, int n_zero, uint32_t* gl_bound,
                           cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    if (n_zero > 256 || G > kMaxClasses) return cudaErrorInvalidValue;
    const int S = learn_cluster((B + kLfSamples - 1) / kLfSamples, d);
    LearnArgs p{a, wlr, B, d, G, 0, d % 8 == 0 && ((uintptr_t)a & 7) == 0,
                d % 4 == 0 && ((uintptr_t)wlr & 15) == 0};
    p.per = ((d + S - 1) / S + kLfTile - 1) / kLfTile * kLfTile;
    ProfScope ps(K_LEARN_FWD, s, 2.0 * B * d * G, 0.0);
    return launch_cluster(S == 1 ? k_learn_fwd<true> : k_learn_fwd<false>,
                          dim3(S * ((B + kLfSamples - 1) / kLfSamples)), 256, S, s, 0, p,
                          FloorDiv::make((uint64_t)d), labels, grad_l, maxabs_wlr, status, zero_words,
                          n_zero, gl_bound);
}

bool simt_lin_fwd_ok(const LayerGeom& g, int B, bool tc) {
    // CTAs before the features are shared out over clusters
    const int64_t ctas = (int64_t)((B + kLfSamples - 1) / kLfSamples) * ((g.cout + kLfG - 1) / kLfG);
    if (g.kind != NITRO_LINEAR) return false;
    return tc ? (int64_t)B * g.cin * g.cout <= kLinFwdMacs && ctas <= kLinFwdCtas && g.cin <= kLinFwdIn
              : ctas <= std::max<int64_t>(kLinFwdCtasMin, kLinFwdCtasPerIn * g.cin);
}

cudaError_t simt_lin_fwd(const int8_t* a, const int32_t* w, const uint32_t* maxabs_w, const LayerGeom& g,
                         int B, int alpha_inv, int mu, int8_t* act, int8_t* out2, int8_t* region,
                         const DropoutArgs* drop, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    const int d = g.cin;
    const int S = learn_cluster((B + kLfSamples - 1) / kLfSamples * ((g.cout + kLfG - 1) / kLfG), d);
    LearnArgs p{a, w, B, d, g.cout, 0, d % 8 == 0 && ((uintptr_t)a & 7) == 0,
                d % 4 == 0 && ((uintptr_t)w & 15) == 0};
    p.per = ((d + S - 1) / S + kLfTile - 1) / kLfTile * kLfTile;
    LinFwdArgs o{alpha_inv, mu, FloorDiv::make((uint64_t)d), act, out2, region};
    ProfScope ps(K_SIMT_LIN_FWD, s, 2.0 * B * d * g.cout, 0.0);
    return launch_cluster(S == 1 ? k_lin_fwd<true> : k_lin_fwd<false>,
                          dim3(S * ((B + kLfSamples - 1) / kLfSamples) * ((g.cout + kLfG - 1) / kLfG)), 256,
                          S, s, 0, p, o, maxabs_w, drop ? *drop : DropoutArgs{});
}

bool simt_lin_wgrad_ok(const LayerGeom& g, int B, bool tc) {
    return g.kind == NITRO_LINEAR && (!tc || (int64_t)B * g.cin * g.cout <= kLinWgradMacs);
}

cudaError_t simt_lin_wgrad(const int8_t* a, const int32_t* delta, const LayerGeom& g, int B, int64_t* dw,
                           cudaStream_t s) {
    if ((int64_t)((B + kLwB - 1) / kLwB * kLwB) * g.cin * g.cout > kLinGemmMacs)
        return simt_gemm(GM_LIN_WGRAD, a, delta, nullptr, dw, B, 1, 1, g.cin, g.cout, s);
    // samples shared out until about six CTAs an SM run, from four slabs on (below, the
    // clear costs what the split gives)
    const int64_t tiles = (int64_t)((g.cin + 63) / 64) * ((g.cout + 15) / 16);
    const int slabs = (B + kLwB - 1) / kLwB;
    int64_t splits = slabs < 4 ? 1 : std::min<int64_t>((152 * 6 + tiles - 1) / tiles, slabs);
    const int per = (int)((slabs + splits - 1) / splits) * kLwB;
    splits = (B + per - 1) / per;
    if (splits > 1) {
        const cudaError_t e = cudaMemsetAsync(dw, 0, sizeof(int64_t) * (size_t)g.cin * g.cout, s);
        if (e != cudaSuccess) return e;
    }
    ProfScope ps(K_SIMT_LIN_WGRAD, s, 2.0 * B * g.cin * (double)g.cout, 0.0);
    return launch_k(k_lin_wgrad, dim3((unsigned)tiles, (unsigned)splits), 256, 0, s, a, delta, B, g.cin, g.cout,
                    per, dw);
}

cudaError_t simt_grad_to_delta(const DeltaSrc& src, const LayerGeom& g, int B, int alpha_inv,
                               const int8_t* region, const int8_t* argmax, int32_t* delta,
                               uint32_t* maxabs_delta, uint32_t* status, cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    const int64_t n = (int64_t)B * g.oh * g.ow * g.cout;
    ProfScope ps(K_GRAD_TO_DELTA, s, 0.0, 0.0);
    launch_k(k_grad_to_delta, grid_for(n, 256), 256, 0, s, src, g, B, alpha_inv, region, argmax, delta,
                                                     maxabs_delta, status);
    return cudaGetLastError();
}

cudaError_t simt_integersgd(const SgdBatch& b_in, cudaStream_t s) {
    if (b_in.count <= 0) return cudaSuccess;
    SgdBatch b = b_in;
    if (!b.scratch) return cudaErrorInvalidValue;
    b.first[0] = 0;
    for (int i = 0; i < b.count; ++i) {
        b.first[i + 1] = b.first[i] + grid_for((b.t[i].n + 3) / 4, 256, 152 * 5);
        if (b.t[i].gamma_inv <= 0 || b.t[i].eta_inv < 0) return cudaErrorInvalidValue;
        b.t[i].gdiv = FloorDiv::make((uint64_t)b.t[i].gamma_inv);
        // 32-bit dividends: any divisor above 2^31 gives what 2^31 + 1 gives
        const auto clamp32 = [](int64_t v) { return (uint32_t)std::min<int64_t>(v, ((int64_t)1 << 31) + 1); };
        b.t[i].gdiv32 = FloorDiv32::make(clamp32(b.t[i].gamma_inv));
        b.t[i].ediv32 = FloorDiv32::make(b.t[i].eta_inv > 0 ? clamp32(b.t[i].eta_inv) : 1u);
        if (b.t[i].planes) {
            if (b.t[i].cin < 1 || b.t[i].n >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
            b.t[i].cin_div = FloorDiv32::make((uint32_t)b.t[i].cin);
            // planes laid out like W: entry (t, ci) of row co at co 9 cin + t cin + ci,
            // 8-byte aligned for every group of four (plane stride a multiple of 4)
            b.t[i].contig = b.t[i].row_k == 9 * b.t[i].tap_k && b.t[i].tap_k == b.t[i].cin &&
                            b.t[i].plane % 4 == 0 && ((uintptr_t)b.t[i].planes & 7) == 0;
        }
    }
    const int grid = b.first[b.count];
    // W and dW are read; what is written (up to 4 bytes and 8 of planes a weight) depends
    // on the data and is not counted
    double bytes = 0;
    for (int i = 0; i < b.count; ++i) bytes += 12.0 * b.t[i].n;
    ProfScope ps(K_INTEGERSGD, s, 0.0, bytes);
    launch_k(k_integersgd, grid, 256, 0, s, b);
    return cudaGetLastError();
}


cudaError_t simt_lr_backward(const int8_t* a, const int32_t* gl, const uint32_t* gl_bound, const int32_t* wlr,
                             int B, int G, int d, int64_t* dwlr, const LrDelta* dl, uint32_t* status, const LossOut& lo,
                             cudaStream_t s) {
    if (B <= 0) return cudaSuccess;
    LrBackArgs p{};
    p.a = a; p.gl = gl; p.wlr = wlr;
    p.B = B; p.G = G; p.d = d;
    p.dwlr = dwlr;
    p.gl_bound = gl_bound;
    bool quad = d % 4 == 0 && (((uintptr_t)a & 3) | ((uintptr_t)wlr & 15)) == 0;
    if (dl) {
        const LayerGeom& g = *dl->lg;
        quad = quad && g.cout % 4 == 0 && (((uintptr_t)dl->region | (uintptr_t)dl->delta | (uintptr_t)dl->planes |
                                            (uintptr_t)(g.pool ? dl->argmax : dl->region)) & 15) == 0;
        p.lg = g;
        p.alpha = FloorDiv32::make((uint32_t)dl->alpha_inv);
        p.dv_c = FloorDiv32::make((uint32_t)g.cout);
        p.dv_ow = FloorDiv32::make((uint32_t)g.ow);
        p.region = dl->region; p.argmax = dl->argmax; p.delta = dl->delta;
        if (quad && dl->planes) {
            p.planes = dl->planes;
            p.plane = (int64_t)B * g.h * g.w * g.cout;
            p.zero = dl->zero;
            p.n_zero = dl->zero ? dl->n_zero : 0;
            *dl->planes_done = true;
        }
        p.maxabs_wlr = dl->maxabs_wlr;
        p.maxabs_delta = dl->maxabs_delta;
    }
    p.status = status;
    const int tile = quad ? 64 : 16;
    p.delta_x = p.dw_x = (d + tile - 1) / tile;
    const int slabs = (B + kLbSlab - 1) / kLbSlab;
    // Samples shared out until eight CTAs an SM form dW_lr, where a slab after another (1.7
    // us each and ten classes) would outlast the rest: few CTAs along the features, none
    // or few of the delta part beside them.  Us a backward, shared out and not: 64 features,
    // 47 classes 33 and 318 at batch 4096; 1024 features 11.2 and 15.3 at 512, 21 and 78 at
    // 4096; 16384 features 30 and 27 at 512, 136 and 150 at 4096; a conv of 64 x 16 x 16,
    // pooled, under the learning layer 64.7 and 62.6 at 512.
    const int few = dl ? 32 : 152 * ((G + 9) / 10);
    const bool share = slabs >= (quad ? 4 : 6) && (p.dw_x < few || (!dl && slabs >= 32));
    int splits = share ? std::min((152 * 8 + p.dw_x - 1) / p.dw_x, slabs) : 1;
    p.dw_per = (slabs + splits - 1) / splits * kLbSlab;
    splits = (B + p.dw_per - 1) / p.dw_per;
    p.dw_ctas = p.dw_x * splits;
    if (splits > 1) {
        const cudaError_t e = cudaMemsetAsync(dwlr, 0, sizeof(int64_t) * (size_t)G * d, s);
        if (e != cudaSuccess) return e;
    }
    p.delta_ctas = dl ? p.delta_x * ((B + 15) / 16) : 0;
    p.tail_ctas = (int)(((int64_t)B * G + kTailValues - 1) / kTailValues);
    const int grid = p.dw_ctas + p.delta_ctas + p.tail_ctas;
    const LossTail tail{gl, B, G, lo.sse, lo.loss, lo.maxabs_gl, lo.ticket, lo.wlr_max, lo.status};
    ProfScope ps(K_LR_BACKWARD, s, (dl ? 4.0 : 2.0) * B * d * G, 0.0);
    if (splits > 1)
        return quad ? launch_k(k_lr_backward<4, true>, grid, 256, 0, s, p, tail)
                    : launch_k(k_lr_backward<1, true>, grid, 256, 0, s, p, tail);
    return quad ? launch_k(k_lr_backward<4, false>, grid, 256, 0, s, p, tail)
                : launch_k(k_lr_backward<1, false>, grid, 256, 0, s, p, tail);
}

}  // namespace nitro
