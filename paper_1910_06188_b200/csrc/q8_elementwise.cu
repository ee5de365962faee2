// HBM-bound kernels of the Q8BERT inference path: max|x| reduction (Eq. 3 / Eq. 4 / Sec. 4.1),
// the quantiser of Eq. 1, the EMA update of Eq. 4 and the Int8 embedding gather of Sec. 3.
//
// All of them stream their input once with 16-byte loads and stores, several independent loads of a thread in flight.

#include <cooperative_groups.h>

#include "q8_internal.cuh"

namespace q8 {

namespace {

constexpr int kThreads = 256;

int grid_for(int64_t work_items, int items_per_block, int blocks_per_sm)
{
    int64_t want = (work_items + items_per_block - 1) / items_per_block;
    int64_t cap = (int64_t)sm_count() * blocks_per_sm;
    if (want < 1) want = 1;
    return (int)(want < cap ? want : cap);
}

// The passes that read and write (quantise, fake quantise, copy) run as many short CTAs, one run of 4 x 128 float4 each: measured
// faster than a grid of the device's size whose threads stride through the tensor, the more so the larger the tensor, and than
// more or fewer loads a thread or larger CTAs.  Quantise, us, grid of 4 CTAs of 256 per SM before / 4 x 128 / 4 x 256 / 2 x 256 /
// 8 x 128 / 4 x 512: 4096 x 768 3.34 / 3.36 / 3.63 / 3.70 / 3.73 / 3.51, 8192 x 768 6.45 / 5.63 / 5.3 / 6.65 / 7.93 / 6.56,
// 4096 x 3072 11.9 / 11.0 / 11.1 / 11.9 / 14.9 / 12.8, 24576 x 1024 21.3 / 19.8 / 19.8 / 21.4 / 27.1 / 22.9, 24576 x 4096 75.4 / 71.2 /
// 71.3 / 78.8 / 100 / 83 (= 7.07 TB/s).
constexpr int kStreamThreads = 128, kStreamBatch = 4;

int stream_grid(int64_t n, int threads = kStreamThreads)
{
    const int64_t runs = ((n >> 2) + threads * kStreamBatch - 1) / (threads * kStreamBatch);
    return (int)(runs < 1 ? 1 : runs < INT32_MAX ? runs : INT32_MAX);
}

// ------------------------------------------------------------------ max|x|
__device__ __forceinline__ float absmax4(float m, float4 v)
{
    // fmaxf drops a NaN operand, so NaN entries are skipped; +-Inf propagates.
    m = fmaxf(m, fabsf(v.x));
    m = fmaxf(m, fabsf(v.y));
    m = fmaxf(m, fabsf(v.z));
    return fmaxf(m, fabsf(v.w));
}

__device__ __forceinline__ void ema_update(CalibState *st, float m, float decay);

// Streams n4 float4 through a thread, kBatch loads in flight at a time, then take(index, value) for each of them.  A CTA takes
// runs of kBatch * blockDim.x neighbouring float4; how many runs is the grid's choice.
template <int kBatch, typename Load, typename Take>
__device__ __forceinline__ void for_each_batch(int64_t n4, Load load, Take take)
{
    const int64_t run = (int64_t)kBatch * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * run; base < n4; base += (int64_t)gridDim.x * run) {
        const int64_t i = base + threadIdx.x;
        float4 v[kBatch];
        if (base + run <= n4) {
#pragma unroll
            for (int k = 0; k < kBatch; ++k) v[k] = load(i + k * blockDim.x);
#pragma unroll
            for (int k = 0; k < kBatch; ++k) take(i + k * blockDim.x, v[k]);
        } else {
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
                if (i + k * blockDim.x < n4) v[k] = load(i + k * blockDim.x);
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
                if (i + k * blockDim.x < n4) take(i + k * blockDim.x, v[k]);
        }
    }
}

// The CTA's share of max|x| in every thread of warp 0, as float bits (non-negative floats order like them).
// Eight CTAs of 256 per SM, four loads a thread in flight, the last ones as well (eight loads, with the last made one after the other,
// 14 us for 12.6 M values where this takes 8.5; two CTAs of 512 with eight loads 9.4; a run per CTA 8.7).
constexpr int kAbsmaxCtasPerSm = 8, kAbsmaxBatch = 4;

template <bool VEC>
__device__ __forceinline__ uint32_t cta_absmax(const float *__restrict__ x, int64_t n)
{
    float m = 0.0f;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        const int64_t n4 = n >> 2;
        for_each_batch<kAbsmaxBatch>(n4, [&](int64_t i) { return __ldg(x4 + i); }, [&](int64_t, float4 v) { m = absmax4(m, v); });
        for (int64_t j = (n4 << 2) + tid; j < n; j += nthreads) m = fmaxf(m, fabsf(x[j]));
    } else {
        for (int64_t j = tid; j < n; j += nthreads) m = fmaxf(m, fabsf(x[j]));
    }
    const uint32_t warp_bits = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    __shared__ uint32_t warp_max[kThreads / 32];
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = warp_bits;
    __syncthreads();
    if (threadIdx.x >= 32) return 0u;
    return __reduce_max_sync(0xffffffffu, threadIdx.x < kThreads / 32 ? warp_max[threadIdx.x] : 0u);
}

// With st the last CTA to finish (counted in the state's own counter, which it leaves at zero) also makes the Eq. 4 update.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) absmax_kernel(const float *__restrict__ x, int64_t n, uint32_t *bits, CalibState *st, float decay)
{
    grid_dependency_release_next(n <= kSmallProblemElems);
    grid_dependency_wait();
    const uint32_t all = cta_absmax<VEC>(x, n);
    if (threadIdx.x == 0) {
        if (all != 0u) atomicMax(bits, all);
        if (st != nullptr) {
            __threadfence();
            if (atomicInc(&st->finished_ctas, gridDim.x - 1) == gridDim.x - 1)
                ema_update(st, __uint_as_float(atomicExch(bits, 0u)), decay);
        }
    }
}

// The same with a word for each CTA, all of which are written, so that nothing is cleared first.
__global__ void __launch_bounds__(kThreads) absmax_words_kernel(const float *__restrict__ x, int64_t n, uint32_t *__restrict__ words)
{
    grid_dependency_release_next(true);  // to the one CTA of scale_from_words_kernel
    grid_dependency_wait();
    const uint32_t all = cta_absmax<true>(x, n);
    if (threadIdx.x == 0) words[blockIdx.x] = all;
}

// max|x| as one partial maximum per cluster of CTAs (exchanged through distributed shared memory): every word of `partial`
// is written, so nothing has to be cleared first (a dynamic q8_linear on 1421 x 768 -> 768: 12.7 -> 10.8 us).
constexpr int kAmCluster = 8;

template <bool VEC>
__global__ void __launch_bounds__(kThreads) absmax_partial_kernel(const float *__restrict__ x, int64_t n,
                                                                  uint32_t *__restrict__ partial)
{
    grid_dependency_release_next(n <= kSmallProblemElems);
    grid_dependency_wait();
    float m = 0.0f;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        const int64_t n4 = n >> 2;
        for_each_batch<8>(n4, [&](int64_t i) { return __ldg(x4 + i); }, [&](int64_t, float4 v) { m = absmax4(m, v); });
        for (int64_t j = (n4 << 2) + tid; j < n; j += nthreads) m = fmaxf(m, fabsf(x[j]));
    } else {
        for (int64_t j = tid; j < n; j += nthreads) m = fmaxf(m, fabsf(x[j]));
    }
    __shared__ uint32_t cta_max;
    if (threadIdx.x == 0) cta_max = 0u;
    __syncthreads();
    const uint32_t bits = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) atomicMax(&cta_max, bits);
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (blockIdx.x % kAmCluster == 0 && threadIdx.x < 32) {
        uint32_t p = 0;
        if (threadIdx.x < kAmCluster) {
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(&cta_max)), "r"((uint32_t)threadIdx.x));
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(p) : "r"(remote) : "memory");
        }
        p = __reduce_max_sync(0xffffffffu, p);
        if (threadIdx.x == 0) partial[blockIdx.x / kAmCluster] = p;
    }
    // no CTA may exit (and give up its shared memory) while a peer can still read it
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// S = 127 / max|.| (Eq. 3); 1, and the flag, for a maximum that is zero or not finite.
__device__ __forceinline__ void put_scale(float a, float *S, int32_t *status)
{
    const bool bad = !(a > 0.0f) || isinf(a);
    if (bad && status) atomicOr(status, 1 << Q8_ERR_SCALE);
    *S = bad ? 1.0f : __fdiv_rn(127.0f, a);
}

// (in place over the scratch word when bits and S alias)
__global__ void scale_from_absmax_kernel(const uint32_t *bits, float *S, int32_t *status)
{
    grid_dependency_release_next(true);
    grid_dependency_wait();
    put_scale(__uint_as_float(*bits), S, status);
}

__global__ void __launch_bounds__(kThreads) scale_from_words_kernel(const uint32_t *words, int count, float *S, int32_t *status)
{
    grid_dependency_wait();
    grid_dependency_release_next(true);  // (not before the pass over x is over, which the CTAs of the next kernel would hold up)
    uint32_t m = 0u;
    for (int i = threadIdx.x; i < count; i += kThreads) m = max(m, words[i]);
    m = __reduce_max_sync(0xffffffffu, m);
    __shared__ uint32_t warp_max[kThreads / 32];
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    m = __reduce_max_sync(0xffffffffu, threadIdx.x < kThreads / 32 ? warp_max[threadIdx.x] : 0u);
    if (threadIdx.x == 0) put_scale(__uint_as_float(m), S, status);
}

// ------------------------------------------------------------------ Eq. 1
__device__ __forceinline__ int32_t quantize_one(float x, float S) { return quantize_value(x, S); }

__device__ __forceinline__ uint32_t quantize_pack4(float4 v, float S) { return q8::quantize_pack4(v.x, v.y, v.z, v.w, S); }

// VEC: a thread turns one 16-byte load (4 floats) into one 4-byte store, four of them in flight; consecutive lanes touch consecutive addresses on both sides.
// With absmax_bits (dynamic scale, Sec. 4.1) every thread derives S = 127 / max|x| from the finished abs-max word
// itself (one correctly rounded division, the same value in every thread) and thread 0 of the grid publishes it
// in *S_out for the GEMM that follows, so no separate scale kernel runs; otherwise S is read from S_ptr.
// AGAIN: the abs-max pass has just read x.  From its end, which L2 still holds some of, the lines marked as the first to go.
// (30522 x 1024, both passes, us: in the order of the abs-max pass 43.8, from the end 40.2, with the mark 38.5, with CTAs of 256 instead of 128 another 1.2 less; marking the first lines
// of the abs-max pass as well, or keeping its last, changes less than 1; all of it in one cooperative launch of a CTA per SM that keeps
// 53 MB in registers and shared memory takes 54.)
template <bool VEC, bool AGAIN = false>
__global__ void __launch_bounds__(kThreads) quantize_kernel(const float *__restrict__ x, int64_t n,
                                                            const float *__restrict__ S_ptr,
                                                            int8_t *__restrict__ xq, int8_t *__restrict__ xq_copy,
                                                            const uint32_t *__restrict__ absmax_bits = nullptr,
                                                            int absmax_count = 1, float *__restrict__ S_out = nullptr,
                                                            int32_t *__restrict__ status = nullptr,
                                                            int32_t *__restrict__ clear_word = nullptr)
{
    grid_dependency_release_next(n <= kSmallProblemElems);
    grid_dependency_wait();
    // first kernel of a static-scale q8_linear call: start the call's status word at zero
    if (clear_word != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *clear_word = 0;
    float S;
    if (absmax_bits != nullptr) {
        uint32_t am = 0u;  // the maximum, or the largest of absmax_count partial maxima
        if (absmax_count == 1) {
            am = __ldg(absmax_bits);
        } else {
            for (int k = threadIdx.x & 31; k < absmax_count; k += 32) am = max(am, __ldg(absmax_bits + k));
            am = __reduce_max_sync(0xffffffffu, am);
        }
        const float a = __uint_as_float(am);
        const bool bad = !(a > 0.0f) || isinf(a);
        S = bad ? 1.0f : __fdiv_rn(127.0f, a);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *S_out = S;
            if (bad && status) atomicOr(status, 1 << Q8_ERR_SCALE);
        }
    } else {
        S = __ldg(S_ptr);
        // a caller-supplied scale (an Eq. 4 result) that is zero, negative or not finite cannot quantise anything
        // meaningful: the call still runs, and the condition is reported like a bad derived scale
        if (blockIdx.x == 0 && threadIdx.x == 0 && (!(S > 0.0f) || isinf(S))) {
            int32_t *word = status != nullptr ? status : clear_word;
            if (word != nullptr) atomicOr(word, 1 << Q8_ERR_SCALE);
        }
    }
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        uint32_t *q4 = reinterpret_cast<uint32_t *>(xq);
        uint32_t *c4 = reinterpret_cast<uint32_t *>(xq_copy);
        const int64_t n4 = n >> 2;
        uint64_t first_to_go;
        asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(first_to_go));
        auto place = [&](int64_t i) { return AGAIN ? n4 - 1 - i : i; };
        for_each_batch<kStreamBatch>(
            n4,
            [&](int64_t i) {
                if (!AGAIN) return __ldg(x4 + i);
                float4 v;
                asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                             : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(x4 + place(i)), "l"(first_to_go));
                return v;
            },
            [&](int64_t i, float4 v) {
                const uint32_t q = quantize_pack4(v, S);
                q4[place(i)] = q;
                if (xq_copy) c4[place(i)] = q;
            });
        for (int64_t j = (n4 << 2) + tid; j < n; j += nthreads) {
            int8_t q = (int8_t)quantize_one(x[j], S);
            xq[j] = q;
            if (xq_copy) xq_copy[j] = q;
        }
    } else {
        for (int64_t j = tid; j < n; j += nthreads) {
            int8_t q = (int8_t)quantize_one(x[j], S);
            xq[j] = q;
            if (xq_copy) xq_copy[j] = q;
        }
    }
}

// Dynamic scale and Eq. 1 in ONE launch for a small activation (Sec. 4.1; e.g. one 128-token batch): a single
// cluster of 8 CTAs holds the whole tensor in registers (up to 12 float4 per thread), so the tensor is read once.
// Each CTA reduces max|x| of its share, the 8 partial maxima are exchanged through distributed shared memory
// (one cluster barrier), every thread derives the same S = 127 / max|x| and quantises the values it holds.
// CTA 0 publishes S and sets the call's status word (0, or the Q8_ERR_SCALE bit for a zero / infinite maximum).
constexpr int kDqCluster = 8, kDqThreads = 512, kDqVecPerThread = 12;
constexpr int64_t kDqMaxElems = (int64_t)kDqCluster * kDqThreads * kDqVecPerThread * 4;  // 196608 = 256 x 768

__global__ void __launch_bounds__(kDqThreads) quantize_dynamic_cluster_kernel(const float *__restrict__ x, int64_t n,
                                                                              float *__restrict__ S_out,
                                                                              int32_t *__restrict__ status, int set_status,
                                                                              int8_t *__restrict__ xq,
                                                                              int8_t *__restrict__ xq_copy)
{
    grid_dependency_release_next(true);  // small by construction
    grid_dependency_wait();
    __shared__ float warp_max[kDqThreads / 32];
    __shared__ float cta_max, all_max;
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int64_t n4 = n >> 2;  // n % 4 == 0 (checked by the host)
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    const int64_t first = (int64_t)rank * kDqThreads + threadIdx.x;
    constexpr int64_t kStride = (int64_t)kDqCluster * kDqThreads;
    float4 v[kDqVecPerThread];
    float m = 0.0f;
#pragma unroll
    for (int i = 0; i < kDqVecPerThread; ++i) {
        const int64_t idx = first + i * kStride;
        v[i] = idx < n4 ? __ldg(x4 + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
        m = absmax4(m, v[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < kDqThreads / 32 ? warp_max[threadIdx.x] : 0.0f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (threadIdx.x == 0) cta_max = m;
    }
    // every CTA's partial maximum is in place before any CTA reads its peers'
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (threadIdx.x < 32) {
        float p = 0.0f;
        if (threadIdx.x < kDqCluster) {
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(remote)
                         : "r"((uint32_t)__cvta_generic_to_shared(&cta_max)), "r"((uint32_t)threadIdx.x));
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(p) : "r"(remote) : "memory");
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) p = fmaxf(p, __shfl_xor_sync(0xffffffffu, p, o));
        if (threadIdx.x == 0) all_max = p;
    }
    // no CTA may exit (and give up its shared memory) while a peer can still read it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    __syncthreads();
    const float a = all_max;
    const bool bad = !(a > 0.0f) || isinf(a);
    const float S = bad ? 1.0f : __fdiv_rn(127.0f, a);
    if (rank == 0 && threadIdx.x == 0) {
        *S_out = S;
        if (status != nullptr) {
            if (set_status) *status = bad ? (1 << Q8_ERR_SCALE) : 0;  // first kernel of a call: starts its status word
            else if (bad) atomicOr(status, 1 << Q8_ERR_SCALE);
        }
    }
    uint32_t *q4 = reinterpret_cast<uint32_t *>(xq);
    uint32_t *c4 = reinterpret_cast<uint32_t *>(xq_copy);
#pragma unroll
    for (int i = 0; i < kDqVecPerThread; ++i) {
        const int64_t idx = first + i * kStride;
        if (idx < n4) {
            const uint32_t q = quantize_pack4(v[i], S);
            q4[idx] = q;
            if (xq_copy) c4[idx] = q;
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The same in ONE launch for tensors that no longer fit one cluster's registers: a cooperative grid finds max|x|, meets,
// derives S and quantises.  Up to kCoopMaxElems, where the barriers cost about as much device time as the launches they replace and
// one call to the driver takes the place of four.  Calls in a row with changing inputs, one launch / memset, abs-max, scale, quantise,
// us: 0.3 M values 8.2 / 11.6, 1 M 8.7 / 11.5, 2 Mi 11.3 / 11.6, 2.5 M 13.6 / 12.4, 3 Mi 14.4 / 12.4, 4 Mi 16.4 / 13.7.
// *word holds the running maximum (float bits) during the first pass and S at the end, so a single device word is enough;
// a bad maximum is OR-ed into *status (may be NULL).
constexpr int kCoopThreads = 256, kCoopCtasPerSm = 4;
constexpr int64_t kCoopMaxElems = int64_t(2) << 20;

__global__ void __launch_bounds__(kCoopThreads, kCoopCtasPerSm)
quantize_dynamic_grid_kernel(const float *__restrict__ x, int64_t n, uint32_t *word, int32_t *status,
                             int8_t *__restrict__ xq, int8_t *__restrict__ xq_copy)
{
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    if (blockIdx.x == 0 && threadIdx.x == 0) *word = 0u;
    auto word_cleared = grid.barrier_arrive();  // waited for after the first pass
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    const int64_t n4 = n >> 2, rest = n4 << 2;  // the last n % 4 values go to the first threads
    float m = 0.0f;
    int64_t i = tid;
    for (; i + 7 * nthreads < n4; i += 8 * nthreads) {
        float4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = __ldg(x4 + i + k * nthreads);
#pragma unroll
        for (int k = 0; k < 8; ++k) m = absmax4(m, v[k]);
    }
    for (; i < n4; i += nthreads) m = absmax4(m, __ldg(x4 + i));
    if (rest + tid < n) m = fmaxf(m, fabsf(x[rest + tid]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ float warp_max[kCoopThreads / 32];
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    grid.barrier_wait(static_cast<cg::grid_group::arrival_token &&>(word_cleared));
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < kCoopThreads / 32; ++w) m = fmaxf(m, warp_max[w]);
        if (m > 0.0f) atomicMax(word, __float_as_uint(m));  // non-negative floats (and +Inf) order like their bit patterns
    }
    grid.sync();
    const float a = __uint_as_float(*reinterpret_cast<volatile uint32_t *>(word));
    auto word_read = grid.barrier_arrive();  // waited for before S takes the maximum's place
    const bool bad = !(a > 0.0f) || isinf(a);
    const float S = bad ? 1.0f : __fdiv_rn(127.0f, a);
    uint32_t *q4 = reinterpret_cast<uint32_t *>(xq);
    uint32_t *c4 = reinterpret_cast<uint32_t *>(xq_copy);
    if (rest + tid < n) {
        const int8_t q = (int8_t)quantize_one(x[rest + tid], S);
        xq[rest + tid] = q;
        if (xq_copy) xq_copy[rest + tid] = q;
    }
    i = n4 - 1 - tid;
    for (; i - 3 * nthreads >= 0; i -= 4 * nthreads) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldg(x4 + i - k * nthreads);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t q = quantize_pack4(v[k], S);
            __stcs(q4 + i - k * nthreads, q);
            if (xq_copy) __stcs(c4 + i - k * nthreads, q);
        }
    }
    for (; i >= 0; i -= nthreads) {
        const uint32_t q = quantize_pack4(__ldg(x4 + i), S);
        q4[i] = q;
        if (xq_copy) c4[i] = q;
    }
    grid.barrier_wait(static_cast<cg::grid_group::arrival_token &&>(word_read));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *reinterpret_cast<float *>(word) = S;
        if (bad && status != nullptr) atomicOr(status, 1 << Q8_ERR_SCALE);
    }
}

// ------------------------------------------------------------------ Eq. 4
__device__ __forceinline__ void ema_update(CalibState *st, float m, float decay)
{
    float ema;
    if (st->n_batches == 0 || decay == 0.0f) {
        ema = m;  // first batch, or no history kept: exactly this batch's maximum (the dynamic scale of Sec. 4.1)
    } else {
        // ema += (1 - d) * (m - ema), each operation rounded separately (no fused multiply-add)
        float one_minus_d = __fsub_rn(1.0f, decay);
        float step = __fmul_rn(one_minus_d, __fsub_rn(m, st->ema));
        ema = __fadd_rn(st->ema, step);
    }
    st->ema = ema;
    st->n_batches += 1;
    if (!(ema > 0.0f) || isinf(ema)) {
        st->S_x = 1.0f;
        st->status |= 1 << Q8_ERR_SCALE;
    } else {
        st->S_x = __fdiv_rn(127.0f, ema);
    }
}

// ------------------------------------------------------------------ Int8 embedding (Sec. 3)
__device__ __forceinline__ float4 dequant4(uint32_t w, float inv)
{
    float4 f;
    f.x = __fmul_rn((float)(int8_t)(w & 0xffu), inv);
    f.y = __fmul_rn((float)(int8_t)((w >> 8) & 0xffu), inv);
    f.z = __fmul_rn((float)(int8_t)((w >> 16) & 0xffu), inv);
    f.w = __fmul_rn((float)(int8_t)(w >> 24), inv);
    return f;
}

// VEC: a CTA walks token rows (four at a time, so four independent gathers are in flight per thread);
// within a row one thread moves 4 table bytes (one 4-byte load) to one 16-byte streaming store, so a
// warp reads 128 and writes 512 contiguous bytes.  No per-element index arithmetic beyond adds.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) embedding_kernel(const int32_t *__restrict__ ids, int64_t T,
                                                             const int8_t *__restrict__ Eq,
                                                             const float *__restrict__ S_e, int64_t V, int64_t H,
                                                             float *__restrict__ out, int8_t *__restrict__ rows_q,
                                                             int32_t *__restrict__ status)
{
    grid_dependency_release_next(T * H <= kSmallProblemElems);
    grid_dependency_wait();
    const float inv = __fdiv_rn(1.0f, __ldg(S_e));
    if (VEC) {
        const int per_row = (int)(H >> 2);
        for (int64_t t0 = (int64_t)blockIdx.x * 4; t0 < T; t0 += (int64_t)gridDim.x * 4) {
            int64_t id[4];
            bool ok[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                id[r] = (t0 + r < T) ? (int64_t)__ldg(ids + t0 + r) : -1;
                ok[r] = id[r] >= 0 && id[r] < V;
                if (!ok[r] && t0 + r < T && threadIdx.x == 0 && status) atomicOr(status, 1 << Q8_ERR_INDEX);
            }
            for (int c = threadIdx.x; c < per_row; c += blockDim.x) {
                uint32_t q[4];
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    q[r] = ok[r] ? __ldg(reinterpret_cast<const uint32_t *>(Eq + id[r] * H) + c) : 0u;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (t0 + r >= T) break;
                    __stcs(reinterpret_cast<float4 *>(out + (t0 + r) * H) + c, dequant4(q[r], inv));
                    if (rows_q) reinterpret_cast<uint32_t *>(rows_q + (t0 + r) * H)[c] = q[r];
                }
            }
        }
    } else {
        const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
        const int64_t total = T * H;
        for (int64_t e = tid; e < total; e += nthreads) {
            const int64_t t = e / H, h = e - t * H;
            const int64_t id = __ldg(ids + t);
            int8_t q = 0;
            if (id >= 0 && id < V) {
                q = Eq[id * H + h];
            } else if (h == 0 && status) {
                atomicOr(status, 1 << Q8_ERR_INDEX);
            }
            out[e] = __fmul_rn((float)q, inv);
            if (rows_q) rows_q[e] = q;
        }
    }
}

// ------------------------------------------------------------------ training mode: fake quantisation (Sec. 2.2)
// x_hat = Quantize(x | S) / S: the rounding of Eq. 1 simulated in floating point.  The quotient is Markstein's ("Computation of
// elementary functions on the IBM RISC System/6000 processor", 1990): with y = q * fl(1 / S), y + fl(1 / S) * fma(-S, y, q) is q / S
// rounded to nearest (checked for all 127 * 2^23 pairs of q and a significand of S), while nothing leaves the normal range.
// The elements go from the last to the first, so that those an abs-max pass has just read are met in L2, and past it on their way out.
// (A table of the 255 quotients in shared memory: 1.5 us more on 4096 x 3072 by its bank conflicts; a grid of the device's size
// 2.4 us more; 4096 x 3072 alone 19.7 -> 17.2, a whole training step 47.4 -> 43.1.)
template <bool VEC>
__global__ void __launch_bounds__(kThreads) fake_quantize_kernel(const float *x, int64_t n,
                                                                 const float *__restrict__ S_ptr, float *xhat)
{
    grid_dependency_release_next(n <= kSmallProblemElems);
    grid_dependency_wait();
    const float S = __ldg(S_ptr), inv = __fdiv_rn(1.0f, S);
    const bool plain = !(S > 0x1p-60f && S < 0x1p60f);  // uniform over the grid
    auto fake = [&](float v) {
        const float q = (float)quantize_value(v, S);
        if (plain) return __fdiv_rn(q, S);
        const float y = __fmul_rn(q, inv);
        return __fmaf_rn(__fmaf_rn(-S, y, q), inv, y);
    };
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    if (VEC) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        float4 *o4 = reinterpret_cast<float4 *>(xhat);
        const int64_t n4 = n >> 2, last = n4 - 1;
        for_each_batch<kStreamBatch>(n4, [&](int64_t i) { return x4[last - i]; },
                                     [&](int64_t i, float4 v) { __stcs(o4 + last - i, make_float4(fake(v.x), fake(v.y), fake(v.z), fake(v.w))); });
        for (int64_t j = (n4 << 2) + tid; j < n; j += nthreads) xhat[j] = fake(x[j]);
    } else {
        for (int64_t j = tid; j < n; j += nthreads) xhat[j] = fake(x[j]);
    }
}

// ------------------------------------------------------------------ Eq. 5: the gradient passes unchanged
// (A kernel of its own so that it starts under the tail of the one before it; 4096 x 3072 17.3 us = 5.8 TB/s with its launch, the
// runtime's copy 19.0.)
__global__ void __launch_bounds__(kStreamThreads) copy_kernel(const float *__restrict__ from, int64_t n, float *__restrict__ to)
{
    grid_dependency_release_next(n <= kSmallProblemElems);
    grid_dependency_wait();
    const float4 *f4 = reinterpret_cast<const float4 *>(from);
    float4 *t4 = reinterpret_cast<float4 *>(to);
    const int64_t n4 = n >> 2;
    for_each_batch<kStreamBatch>(n4, [&](int64_t i) { return __ldcs(f4 + i); }, [&](int64_t i, float4 v) { __stcs(t4 + i, v); });
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) to[(n4 << 2) + threadIdx.x] = from[(n4 << 2) + threadIdx.x];
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

cudaError_t launch_absmax(const float *x, int64_t n, uint32_t *bits, cudaStream_t s, CalibState *st, float decay)
{
    if (n <= 0) return cudaSuccess;
    const bool vec = aligned16(x);
    return launch_overlapping_tail(vec ? absmax_kernel<true> : absmax_kernel<false>,
                                   dim3(grid_for(vec ? n >> 2 : n, kThreads * kAbsmaxBatch, kAbsmaxCtasPerSm)), dim3(kThreads), 0, s, x, n, bits,
                                   st, decay);
}

// A dynamic layer on 16-byte aligned inputs, partial maxima / clear and atomics of eight CTAs per SM, us, inputs that change / the same one:
// 5000 x 1024 -> 1024 24.3 / 24.9 and 18.4 / 21.9, 6000 x 1024 -> 3072 33.6 / 37.1 and 33.2 / 37.0, 2407 x 3072 -> 2496 34.3 / 35.4 and 29.7 / 31.1,
// 2000 x 4096 -> 1024 30.9 / 29.2 and 23.8 / 25.7, 8192 x 1024 -> 1024 32.2 / 31.5 and 26.2 / 26.9, 2407 x 3648 -> 2496 41.5 / 41.1: the line lies where
// the second pass starts to miss what the first has left in L2, and the order of that pass from the end begins to count.  Off 16 bytes,
// where a thread loads a value at a time, the 480 CTAs have too few in flight sooner: 4.6 M values 20.4 / 20.4, 6.1 M 23.0 / 22.3, 8.4 M 27.1 / 25.7.
bool absmax_partial_preferred(const float *x, int64_t n) { return n <= (int64_t(aligned16(x) ? 14 : 9) << 19); }  // 7.3 M, 4.7 M

// Clusters for a run of 1024 float4 a CTA, four CTAs per SM; the 60 words of the header bound them at 480 CTAs, from 3.9 M values on.  (The
// kernel takes runs of 2048, so below that half of the CTAs find none.  With as many CTAs as runs, us: 1421 x 768 -> 768 10.3 -> 9.8,
// 1000 x 300 -> 1200 12.5 -> 12.1, but 1000 x 512 -> 2048 11.1 -> 12.0, 300 x 1000 -> 1000 16.7 -> 18.0, 1000 x 300 -> 256 10.3 -> 11.2: what the idle ones
// change is where the CTAs of the two kernels behind them start.  Runs of 1024 are slower from 1.4 M values on, 4.2 M 13.6 -> 14.4.)
cudaError_t launch_absmax_partial(const float *x, int64_t n, uint32_t *partial, int max_words, int *words, cudaStream_t s)
{
    const bool vec = aligned16(x);
    int clusters = (grid_for(vec ? n >> 2 : n, kThreads * 4, 4) + kAmCluster - 1) / kAmCluster;
    if (clusters > max_words) clusters = max_words;
    *words = clusters;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * kAmCluster));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kAmCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, vec ? absmax_partial_kernel<true> : absmax_partial_kernel<false>, x, n, partial);
}

bool quantize_dynamic_grid_supported(const float *x, int64_t n, const int8_t *xq, const int8_t *xq_copy)
{
    return n > 0 && n <= kCoopMaxElems && aligned16(x) && aligned16(xq) && (xq_copy == nullptr || aligned16(xq_copy));
}

static int g_quantize_grid = 0;
void set_quantize_grid(int ctas) { g_quantize_grid = ctas > 0 ? ctas : 0; }

cudaError_t launch_quantize_dynamic_grid(const float *x, int64_t n, float *S_out, int32_t *status, int8_t *xq, int8_t *xq_copy,
                                         cudaStream_t s)
{
    static int resident[64] = {};  // CTAs of the kernel that fit on the device at a time
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (resident[dev] == 0) {
        int per_sm = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, quantize_dynamic_grid_kernel, kCoopThreads, 0);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (per_sm < 1 || sms < 1) return cudaErrorCooperativeLaunchTooLarge;
        resident[dev] = sms * (per_sm < kCoopCtasPerSm ? per_sm : kCoopCtasPerSm);
    }
    const int64_t want = ((n >> 2) + kCoopThreads * 4 - 1) / (kCoopThreads * 4);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g_quantize_grid > 0 ? g_quantize_grid : want < 1 ? 1 : want < resident[dev] ? want : resident[dev]));
    cfg.blockDim = dim3(kCoopThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, quantize_dynamic_grid_kernel, x, n, reinterpret_cast<uint32_t *>(S_out), status,
                              xq, xq_copy);
}

cudaError_t launch_scale_from_absmax(const uint32_t *bits, float *S, int32_t *status, cudaStream_t s)
{
    return launch_overlapping_tail(scale_from_absmax_kernel, dim3(1), dim3(1), 0, s, bits, S, status);
}

// Every access of the three kernels is whole, and the first bytes of xq, which the last of them fills, have room for a word per CTA
// (each of which has a run of 4096 values unless the tensor is smaller than that).
bool quantize_two_pass_supported(const float *x, int64_t n, const int8_t *xq, const int8_t *xq_copy)
{
    return n >= 4 && aligned16(x) && aligned16(xq) && (xq_copy == nullptr || aligned16(xq_copy));
}

cudaError_t launch_quantize_two_pass(const float *x, int64_t n, float *S_out, int32_t *status, int8_t *xq, int8_t *xq_copy, cudaStream_t s)
{
    const int ctas = grid_for(n >> 2, kThreads * kAbsmaxBatch, kAbsmaxCtasPerSm);
    uint32_t *words = reinterpret_cast<uint32_t *>(xq);
    cudaError_t e = launch_overlapping_tail(absmax_words_kernel, dim3(ctas), dim3(kThreads), 0, s, x, n, words);
    if (e == cudaSuccess)
        e = launch_overlapping_tail(scale_from_words_kernel, dim3(1), dim3(kThreads), 0, s, words, ctas, S_out, status);
    if (e != cudaSuccess) return e;
    return launch_overlapping_tail(quantize_kernel<true, true>, dim3(stream_grid(n, kThreads)), dim3(kThreads), 0, s, x, n, S_out, xq, xq_copy,
                                   nullptr, 1, nullptr, nullptr, nullptr);
}

cudaError_t launch_quantize(const float *x, int64_t n, const float *S, int8_t *xq, int8_t *xq_copy, cudaStream_t s,
                            int32_t *clear_word, int32_t *status)
{
    if (n <= 0) return cudaSuccess;
    if (aligned16(x) && aligned16(xq) && (xq_copy == nullptr || aligned16(xq_copy))) {
        return launch_overlapping_tail_evenly<quantize_kernel<true>>(dim3(stream_grid(n)), dim3(kStreamThreads), s, x, n, S, xq, xq_copy, nullptr, 1,
                                                                     nullptr, status, clear_word);
    } else {
        quantize_kernel<false><<<grid_for(n, kThreads * 4, 8), kThreads, 0, s>>>(x, n, S, xq, xq_copy, nullptr, 1, nullptr,
                                                                                 status, clear_word);
    }
    return cudaGetLastError();
}

cudaError_t launch_quantize_dynamic(const float *x, int64_t n, const uint32_t *absmax_bits, float *S_out, int32_t *status,
                                    int8_t *xq, int8_t *xq_copy, cudaStream_t s, bool clear_status, int absmax_count, bool again)
{
    if (n <= 0) return cudaSuccess;
    int32_t *clear_word = clear_status ? status : nullptr;
    if (aligned16(x) && aligned16(xq) && (xq_copy == nullptr || aligned16(xq_copy))) {
        if (again || absmax_count > 1) {  // behind an abs-max pass, beside which they park as they would on a free SM
            const int threads = again ? kThreads : kStreamThreads;
            return launch_overlapping_tail(again ? quantize_kernel<true, true> : quantize_kernel<true>, dim3(stream_grid(n, threads)), dim3(threads),
                                           0, s, x, n, nullptr, xq, xq_copy, absmax_bits, absmax_count, S_out, status, clear_word);
        }
        return launch_overlapping_tail_evenly<quantize_kernel<true>>(dim3(stream_grid(n)), dim3(kStreamThreads), s, x, n, nullptr, xq, xq_copy,
                                                                     absmax_bits, absmax_count, S_out, status, clear_word);
    } else {
        quantize_kernel<false><<<grid_for(n, kThreads * 4, 8), kThreads, 0, s>>>(x, n, nullptr, xq, xq_copy, absmax_bits,
                                                                                 absmax_count, S_out, status, clear_word);
    }
    return cudaGetLastError();
}

bool quantize_dynamic_small_supported(const float *x, int64_t n, const int8_t *xq, const int8_t *xq_copy)
{
    return n > 0 && n <= kDqMaxElems && (n & 3) == 0 && aligned16(x) && aligned16(xq) &&
           (xq_copy == nullptr || aligned16(xq_copy));
}

cudaError_t launch_quantize_dynamic_small(const float *x, int64_t n, float *S_out, int32_t *status, bool set_status, int8_t *xq,
                                          int8_t *xq_copy, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kDqCluster);
    cfg.blockDim = dim3(kDqThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kDqCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, quantize_dynamic_cluster_kernel, x, n, S_out, status, set_status ? 1 : 0, xq, xq_copy);
}

cudaError_t launch_fake_quantize(const float *x, int64_t n, const float *S, float *xhat, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (aligned16(x) && aligned16(xhat))
        return launch_overlapping_tail(fake_quantize_kernel<true>, dim3(stream_grid(n)), dim3(kStreamThreads), 0, s, x, n, S, xhat);
    return launch_overlapping_tail(fake_quantize_kernel<false>, dim3(grid_for(n, kThreads * 4, 8)), dim3(kThreads), 0, s, x, n,
                                   S, xhat);
}

// Memory of the current device, which a kernel reaches without more; between devices, from pinned or managed memory the runtime copies.
static bool on_current_device(const void *p)
{
    int device = -1;
    cudaPointerAttributes at{};
    if (cudaGetDevice(&device) == cudaSuccess && cudaPointerGetAttributes(&at, p) == cudaSuccess)
        return at.type == cudaMemoryTypeDevice && at.device == device;
    cudaGetLastError();
    return false;
}

cudaError_t launch_copy(const float *from, int64_t n, float *to, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (!aligned16(from) || !aligned16(to) || !on_current_device(from) || !on_current_device(to))
        return cudaMemcpyAsync(to, from, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, s);
    const cudaError_t e = launch_overlapping_tail(copy_kernel, dim3(stream_grid(n)), dim3(kStreamThreads), 0, s, from, n, to);
    if (e == cudaErrorInvalidResourceHandle) {  // another device's stream, in which the runtime copies and launches nothing
        cudaGetLastError();
        return cudaMemcpyAsync(to, from, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, s);
    }
    last_launch_info().launches += e == cudaSuccess;
    return e;
}

cudaError_t launch_embedding(const int32_t *ids, int64_t T, const int8_t *Eq, const float *S_e, int64_t V,
                             int64_t H, float *out, int8_t *rows_q, int32_t *status, cudaStream_t s)
{
    if (T <= 0 || H <= 0) return cudaSuccess;
    const bool vec = (H % 4 == 0) && aligned16(Eq) && aligned16(out) && (rows_q == nullptr || aligned16(rows_q));
    if (vec) {
        // one thread per 4-byte piece of a row, rounded up to whole warps; a CTA takes 4 rows per iteration
        int threads = (int)(((H >> 2) + 31) / 32 * 32);
        if (threads > kThreads) threads = kThreads;
        return launch_overlapping_tail(embedding_kernel<true>, dim3(grid_for((T + 3) / 4, 1, 16)), dim3(threads), 0, s, ids, T,
                                       Eq, S_e, V, H, out, rows_q, status);
    } else {
        embedding_kernel<false><<<grid_for(T * H, kThreads, 8), kThreads, 0, s>>>(ids, T, Eq, S_e, V, H, out,
                                                                                 rows_q, status);
    }
    return cudaGetLastError();
}

}  // namespace q8
