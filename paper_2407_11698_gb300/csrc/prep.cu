// Integer data pre-processing (App. A) on the GPU.
//
// Over the n 8-bit values x of a dataset:
//   mu    = floor(sum x / n)
//   omega = floor(sum |x - mu| / n)
//   x_hat = clamp(floor((x - mu) 51 / omega), -127, 127), omega = 0 read as 1
//
// Small data (kOnePassBytes): k_prep_reduce<0> forms the byte sum, k_prep_reduce<1> the
// sum of absolute differences to mu, walking backwards from what the first pass left
// in L2; its last CTA derives omega and the map.  Large data: k_prep_sample takes the
// mean of a sample, k_prep_fit the byte sum and the sums of |x - c| for three guesses c
// of mu in one pass, and k_prep_reduce<1> runs only if mu is none of them; the
// result is exact either way.  k_prep_apply looks x_hat up.
//
// The input is 8-bit, so the sums take four bytes per instruction (__vsadu4
// adds the absolute differences of the four byte lanes; against zero it is the
// plain byte sum), and x_hat, a function of one byte, is a lookup in a
// 256-entry table held in shared memory, one copy a bank.  Bound by memory: every
// pass streams the data with 16-byte loads, four in flight a thread, from a grid
// that runs at once (six CTAs an SM; with eight queued, of which six fitted, the last
// ran alone).  153.6 MB, fit and map: 123 us with one load in flight and two
// passes, 113 with four, 105 without a memset, with early launches and the grid that
// fits, 93 with one pass (fit 38, map 52: 5.9 TB/s).
#include <algorithm>
#include <new>

#include "nitro.h"
#include "nitro_internal.cuh"
#include "prof.cuh"

using namespace nitro;

namespace {

constexpr int kPrepThreads = 256;      // also the size of the map: one entry per thread
constexpr int kCtasPerSm = 6;
constexpr unsigned kAll = 0xffffffffu;

struct alignas(32) PrepState {
    unsigned long long sum;      // sum of x
    unsigned long long sad;      // sum of |x - mu|
    unsigned long long ticket;   // CTAs done with the pass that ends the fit
    unsigned long long sample;   // sum of the sampled bytes
    unsigned long long done;     // one of the guesses was mu
    // (the sums and the ticket are zero before the first fit and left zero by every fit)
    long long mu, omega;
    int8_t map[256];             // x_hat of every byte value
};                               // followed by the one-pass fit's four sums of each CTA

__device__ __forceinline__ unsigned long long block_sum(unsigned long long v) {
    __shared__ unsigned long long part[kPrepThreads / 32];
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(kAll, v, off);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long t = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kPrepThreads / 32; ++w) t += part[w];
    return t;   // valid in thread 0
}

// One CTA: omega and the map from the finished sums.
__device__ __forceinline__ void finish_fit(PrepState* st, long long mu, unsigned long long sad, int64_t n) {
    const long long omega = (long long)(sad / (unsigned long long)n);
    const long long div = omega > 0 ? omega : 1;
    const long long num = ((long long)threadIdx.x - mu) * 51;
    long long q = num / div;
    if (num % div != 0 && num < 0) --q;   // floor
    st->map[threadIdx.x] = (int8_t)(q < -127 ? -127 : (q > 127 ? 127 : q));
    if (threadIdx.x == 0) {
        st->mu = mu;
        st->omega = omega;
        st->sum = st->sad = st->sample = st->ticket = 0;
    }
}

// Byte sum of kSamples 16-byte words, one at a hashed place in each equal share of the
// data, so that no row or image length resonates with the sampling.
constexpr uint32_t kSamples = 1u << 16;
__global__ void __launch_bounds__(kPrepThreads) k_prep_sample(const uint4* __restrict__ xv, int64_t share,
                                                              PrepState* st) {
    pdl_wait();
    const uint32_t k = blockIdx.x * kPrepThreads + threadIdx.x;
    // multiplicative hash by a prime near 2^32 over the golden ratio (Knuth, The Art of
    // Computer Programming, vol. 3, 6.4), its upper bits folded in and mixed by the first
    // multiplier of MurmurHash3's finalizer (Appleby)
    uint32_t h = k * 2654435761u;
    h ^= h >> 15;
    h *= 0x85ebca6bu;
    const uint4 v = __ldg(xv + (int64_t)k * share + (int64_t)(((uint64_t)h * (uint64_t)share) >> 32));
    const unsigned long long acc = (__vsadu4(v.x, 0) + __vsadu4(v.y, 0)) + (__vsadu4(v.z, 0) + __vsadu4(v.w, 0));
    const unsigned long long t = block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(&st->sample, t);
}

// Both sums in one pass: sum x, and sum |x - c| for three guesses of mu around the
// sampled mean.  Where mu is none of them, the pass over |x - mu| follows.
__global__ void __launch_bounds__(kPrepThreads, kCtasPerSm) k_prep_fit(const uint8_t* __restrict__ x, int64_t n,
                                                           PrepState* st) {
    pdl_wait();
    const uint32_t est = (uint32_t)(__ldcg(&st->sample) / (16ull * kSamples));
    const uint32_t c0 = est < 1 ? 0 : (est > 254 ? 253 : est - 1);
    const uint32_t c4[4] = {0, c0 * 0x01010101u, (c0 + 1) * 0x01010101u, (c0 + 2) * 0x01010101u};
    const int64_t head = min(n, (int64_t)((16 - ((uintptr_t)x & 15)) & 15));
    const int64_t nv = (n - head) >> 4;
    const int64_t tail0 = head + (nv << 4);
    const uint4* xv = reinterpret_cast<const uint4*>(x + head);
    const int64_t tid = (int64_t)blockIdx.x * kPrepThreads + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * kPrepThreads;
    unsigned long long acc[4] = {0, 0, 0, 0};
    const auto sad = [](const uint4 v, uint32_t c) {
        return (uint32_t)(__vsadu4(v.x, c) + __vsadu4(v.y, c)) + (uint32_t)(__vsadu4(v.z, c) + __vsadu4(v.w, c));
    };
    const auto at = [&](int64_t i) { return __ldg(xv + (nv - 1 - i)); };
    int64_t i = tid;
    for (; i + 3 * stride < nv; i += 4 * stride) {
        const uint4 a = at(i), b = at(i + stride), c = at(i + 2 * stride), d = at(i + 3 * stride);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += (sad(a, c4[k]) + sad(b, c4[k])) + (sad(c, c4[k]) + sad(d, c4[k]));
    }
    for (; i < nv; i += stride) {
        const uint4 a = at(i);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += sad(a, c4[k]);
    }
    const int64_t ns = head + (n - tail0);   // at most 30 scalar bytes
    if (tid < ns) {
        const uint32_t xb = x[tid < head ? tid : tail0 + (tid - head)];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += __vsadu4(xb, c4[k] & 255u);
    }
    __shared__ unsigned long long part[4][kPrepThreads / 32];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int off = 16; off; off >>= 1) acc[k] += __shfl_xor_sync(kAll, acc[k], off);
        if ((threadIdx.x & 31) == 0) part[k][threadIdx.x >> 5] = acc[k];
    }
    __syncthreads();
    __shared__ bool last;
    if (threadIdx.x == 0) {
        unsigned long long t[4] = {0, 0, 0, 0};
        for (int w = 0; w < kPrepThreads / 32; ++w)
            for (int k = 0; k < 4; ++k) t[k] += part[k][w];
        reinterpret_cast<ulonglong4*>(st + 1)[blockIdx.x] = make_ulonglong4(t[0], t[1], t[2], t[3]);
        __threadfence();
        last = atomicAdd(&st->ticket, 1ull) == (unsigned long long)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // warp k adds the CTAs' k-th sums
    const int warp = threadIdx.x >> 5;
    if (warp < 4) {
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(st + 1) + warp;
        unsigned long long t = 0;
#pragma unroll 8
        for (uint32_t c = threadIdx.x & 31; c < gridDim.x; c += 32) t += __ldcg(src + 4 * c);
#pragma unroll
        for (int off = 16; off; off >>= 1) t += __shfl_xor_sync(kAll, t, off);
        part[warp][0] = t;
    }
    __syncthreads();
    const unsigned long long sum = part[0][0];
    const uint32_t mu = (uint32_t)(sum / (unsigned long long)n);
    const bool hit = mu >= c0 && mu <= c0 + 2;
    if (hit) finish_fit(st, mu, part[1 + mu - c0][0], n);
    if (threadIdx.x == 0) {
        st->done = hit;
        st->ticket = 0;
        if (!hit) st->sum = sum;             // for the pass that follows
    }
}

// PASS 0: st->sum += sum x.  PASS 1: st->sad += sum |x - mu| with mu from the
// finished first pass, unless the fit is done; the last CTA to finish writes mu, omega
// and the map.
template <int PASS>
__global__ void __launch_bounds__(kPrepThreads) k_prep_reduce(const uint8_t* __restrict__ x,
                                                              int64_t n, PrepState* st) {
    pdl_wait();
    uint32_t mu = 0;
    if (PASS == 0 && blockIdx.x == 0 && threadIdx.x == 0) st->done = 0;
    if (PASS == 1 && __ldcg(&st->done)) return;
    if (PASS == 1) mu = (uint32_t)(__ldcg(&st->sum) / (unsigned long long)n);   // <= 255
    const uint32_t mu4 = mu * 0x01010101u;
    // bytes before the first 16-byte boundary, the 16-byte body, the tail
    const int64_t head = min(n, (int64_t)((16 - ((uintptr_t)x & 15)) & 15));
    const int64_t nv = (n - head) >> 4;
    const int64_t tail0 = head + (nv << 4);
    const uint4* xv = reinterpret_cast<const uint4*>(x + head);
    const int64_t tid = (int64_t)blockIdx.x * kPrepThreads + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * kPrepThreads;
    unsigned long long acc = 0;
    const auto sad = [mu4](const uint4 v) {
        return (uint32_t)(__vsadu4(v.x, mu4) + __vsadu4(v.y, mu4)) +
               (uint32_t)(__vsadu4(v.z, mu4) + __vsadu4(v.w, mu4));
    };
    const auto at = [&](int64_t i) { return __ldg(xv + (PASS == 1 ? nv - 1 - i : i)); };
    int64_t i = tid;
    for (; i + 3 * stride < nv; i += 4 * stride) {
        const uint4 a = at(i), b = at(i + stride), c = at(i + 2 * stride), d = at(i + 3 * stride);
        acc += (sad(a) + sad(b)) + (sad(c) + sad(d));
    }
    for (; i < nv; i += stride) acc += sad(at(i));
    const int64_t ns = head + (n - tail0);   // at most 30 scalar bytes
    if (tid < ns) {
        const int64_t j = tid < head ? tid : tail0 + (tid - head);
        const int dv = (int)x[j] - (int)mu;
        acc += (unsigned long long)(dv < 0 ? -dv : dv);
    }
    const unsigned long long t = block_sum(acc);
    __shared__ bool last;
    if (threadIdx.x == 0) {
        atomicAdd(PASS == 0 ? &st->sum : &st->sad, t);
        if (PASS == 1) {
            __threadfence();
            last = atomicAdd(&st->ticket, 1ull) == (unsigned long long)gridDim.x - 1;
        }
    }
    if (PASS == 0) return;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const unsigned long long sad_mu = __ldcg(&st->sad);
    __syncthreads();         // thread 0 clears what the others read
    finish_fit(st, mu, sad_mu, n);
}

// Four lookups in this lane's copy of the map: entry v lies at byte v & 3 of word
// 32 (v >> 2) + lane, so that the 32 lanes of a warp read 32 banks.  (One shared
// copy, on which random bytes conflict three to four ways, took 54.9 us for 153.6 MB,
// this 52.8 us, 5.8 TB/s.)
__device__ __forceinline__ uint32_t map4(uint32_t w, const uint8_t* m) {
    const auto one = [m](uint32_t v) { return (uint32_t)m[((v & 0xfcu) << 5) | (v & 3u)]; };
    const uint32_t lo = __byte_perm(one(w), one(w >> 8), 0x0040);
    const uint32_t hi = __byte_perm(one(w >> 16), one(w >> 24), 0x0040);
    return __byte_perm(lo, hi, 0x5410);
}

// out[i] = map[x[i]].  16-byte vectors when x and out sit at the same offset
// from a 16-byte boundary; bytes otherwise.  out may equal x (each element is
// read, then written, by one thread).
__global__ void __launch_bounds__(kPrepThreads, kCtasPerSm) k_prep_apply(const uint8_t* x, int64_t n,
                                                             const PrepState* __restrict__ st,
                                                             int8_t* out) {
    __shared__ __align__(16) uint32_t maps[64 * 32];
    pdl_wait();
    {
        // four entries a word, 32 copies of it; eight threads write a word's copies
        const uint32_t* src = reinterpret_cast<const uint32_t*>(st->map);
        for (int k = threadIdx.x; k < 64 * 8; k += kPrepThreads) {
            const uint32_t w = src[k >> 3];
            reinterpret_cast<uint4*>(maps)[k] = make_uint4(w, w, w, w);
        }
    }
    __syncthreads();
    const uint8_t* m = reinterpret_cast<const uint8_t*>(maps + (threadIdx.x & 31));
    const bool vec = (((uintptr_t)x ^ (uintptr_t)out) & 15) == 0;
    const int64_t head = vec ? min(n, (int64_t)((16 - ((uintptr_t)x & 15)) & 15)) : n;
    const int64_t nv = (n - head) >> 4;
    const int64_t tail0 = head + (nv << 4);
    const int64_t tid = (int64_t)blockIdx.x * kPrepThreads + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * kPrepThreads;
    const uint4* xv = reinterpret_cast<const uint4*>(x + head);
    uint4* ov = reinterpret_cast<uint4*>(out + head);
    const auto map16 = [m](const uint4 v) {
        return make_uint4(map4(v.x, m), map4(v.y, m), map4(v.z, m), map4(v.w, m));
    };
    int64_t i = tid;
    for (; i + 3 * stride < nv; i += 4 * stride) {
        const uint4 a = xv[i], b = xv[i + stride], c = xv[i + 2 * stride], d = xv[i + 3 * stride];
        ov[i] = map16(a);
        ov[i + stride] = map16(b);
        ov[i + 2 * stride] = map16(c);
        ov[i + 3 * stride] = map16(d);
    }
    for (; i < nv; i += stride) ov[i] = map16(xv[i]);
    const auto one = [m](uint8_t v) { return (int8_t)m[((v & 0xfcu) << 5) | (v & 3u)]; };
    // the head and the tail, or all of it where the offsets differ: four loads in flight
    // (153.6 M bytes 129 us; 253 with one in flight)
    const auto bytes = [&](int64_t j, int64_t end) {
        for (; j + 3 * stride < end; j += 4 * stride) {
            const uint8_t a = x[j], b = x[j + stride], c = x[j + 2 * stride], d = x[j + 3 * stride];
            out[j] = one(a);
            out[j + stride] = one(b);
            out[j + 2 * stride] = one(c);
            out[j + 3 * stride] = one(d);
        }
        for (; j < end; j += stride) out[j] = one(x[j]);
    };
    bytes(tid, head);
    bytes(tail0 + tid, n);
}

int grid_for_bytes(int64_t n, int sms) {
    const int64_t want = ((n >> 4) + kPrepThreads - 1) / kPrepThreads;
    const int64_t cap = (int64_t)sms * kCtasPerSm;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

// From about what L2 keeps between two passes: fit of 64 MB 25 us in two passes and 29
// in one (27 and 27 with the data out of L2), of 154 MB 56 and 46 (59 and 44).
constexpr int64_t kOnePassBytes = (int64_t)96 << 20;
constexpr int64_t kPrepMaxN = (int64_t)1 << 48;   // 255 n stays far inside uint64

}  // namespace

struct nitro_prep {
    PrepState* st = nullptr;
    int sms = 0;
    bool fitted = false, clean = false;    // clean: see clear_once
};

extern "C" {

nitro_status nitro_prep_create(nitro_prep** out) {
    if (!out) return NITRO_ERR_ARG;
    *out = nullptr;
    nitro_prep* p = new (std::nothrow) nitro_prep();
    if (!p) return NITRO_ERR_CUDA;
    int dev = 0;
    bool ok = cudaGetDevice(&dev) == cudaSuccess &&
              cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
              cudaMalloc(&p->st, sizeof(PrepState) + (size_t)p->sms * kCtasPerSm * 32) == cudaSuccess;
    if (!ok) {
        if (p->st) cudaFree(p->st);
        delete p;
        return NITRO_ERR_CUDA;
    }
    *out = p;
    return NITRO_OK;
}

nitro_status nitro_prep_fit(nitro_prep* p, const uint8_t* x, int64_t n, void* stream) {
    if (!p || !x || n < 1 || n > kPrepMaxN) return NITRO_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = grid_for_bytes(n, p->sms);
    if (clear_once(p->clean, p->st, sizeof(PrepState), s) != cudaSuccess) return NITRO_ERR_CUDA;
    if (n >= kOnePassBytes) {
        ProfScope ps(K_PREP_SUM, s, 0.0, (double)n + 16.0 * kSamples);
        const uint8_t* body = x + ((16 - ((uintptr_t)x & 15)) & 15);
        launch_k(k_prep_sample, kSamples / kPrepThreads, kPrepThreads, 0, s,
                 reinterpret_cast<const uint4*>(body), ((n - 15) >> 4) / kSamples, p->st);
        launch_k(k_prep_fit, grid, kPrepThreads, 0, s, x, n, p->st);
    } else {
        ProfScope ps(K_PREP_SUM, s, 0.0, (double)n);
        launch_k(k_prep_reduce<0>, grid, kPrepThreads, 0, s, x, n, p->st);
    }
    {
        // after one pass the launch reads nothing unless mu was none of the guesses
        ProfScope ps(K_PREP_MAD, s, 0.0, n >= kOnePassBytes ? 0.0 : (double)n);
        launch_k(k_prep_reduce<1>, grid, kPrepThreads, 0, s, x, n, p->st);
    }
    if (cudaGetLastError() != cudaSuccess) {
        cudaMemsetAsync(p->st, 0, sizeof(PrepState), s);   // a pass that did run left its sums
        return NITRO_ERR_CUDA;
    }
    p->fitted = true;
    return NITRO_OK;
}

nitro_status nitro_prep_apply(nitro_prep* p, const uint8_t* x, int64_t n, int8_t* out,
                              void* stream) {
    if (!p || !p->fitted || n < 0 || n > kPrepMaxN) return NITRO_ERR_ARG;
    if (n == 0) return NITRO_OK;
    if (!x || !out) return NITRO_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    {
        ProfScope ps(K_PREP_APPLY, s, 0.0, 2.0 * (double)n);
        // From 128 MB on two to four rounds of CTAs, so that SMs that drain sooner take more: us in
        // one, two, three rounds 100 MB 36 36 35, 154 MB 52.8 51.1 51.9, 278 MB 95 89 88, 500 MB
        // 171 160 154 (four 153)
        const int rounds = (int)std::min<int64_t>(4, std::max<int64_t>(1, n >> 26));
        launch_k(k_prep_apply, grid_for_bytes(n, p->sms * rounds), kPrepThreads, 0, s, x, n, p->st, out);
    }
    return cudaGetLastError() == cudaSuccess ? NITRO_OK : NITRO_ERR_CUDA;
}

nitro_status nitro_prep_stats(nitro_prep* p, int64_t* mu, int64_t* omega) {
    if (!p || !p->fitted || !mu || !omega) return NITRO_ERR_ARG;
    long long v[2];
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(v, &p->st->mu, sizeof(v), cudaMemcpyDeviceToHost) != cudaSuccess)
        return NITRO_ERR_CUDA;
    *mu = v[0];
    *omega = v[1];
    return NITRO_OK;
}

void nitro_prep_destroy(nitro_prep* p) {
    if (!p) return;
    cudaFree(p->st);
    delete p;
}

}  // extern "C"
