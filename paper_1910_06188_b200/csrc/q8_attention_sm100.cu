// Multi-head self-attention (head dimension 64, no mask, any sequence length) on the Blackwell tensor cores with
// fp32-grade accuracy.  Both products, Q K^T and P V, run as tcgen05.mma kind::f16 with every fp32 operand x scaled by
// a power of two (exactly) and split into two fp16 numbers, hi = fp16(x) and lo = fp16(x - hi): 22 to 23 significant
// bits, accumulated in fp32 in TMEM as lo*hi + hi*lo + hi*hi; the dropped lo*lo term is below 2^-22 relative per product,
// i.e. at the rounding level of a plain fp32 dot product.  The scale comes from the data.  The largest finite |x| of a Q row and of
// each K chunk is brought into [2^13, 2^14), that of each feature of V, over the keys so far, into [2^12, 2^15); a value below 2^-14
// of that largest one keeps an absolute error of 2^-37 of it.  P, at most 1 beside its row's reference maximum, is split as
// 2^13 P: an absolute error of 2^-38 where p < 2^-15.  So no feature of V is less accurate for the size of another.  (One
// exponent for the 64 features of a V chunk, folded into P, lost 2^-10 for every 2^10 that one feature stood above the
// others.)  Q's and K's scales are undone inside the FFMA that the softmax needs anyway, V's at the end: the running output is in
// the units of V's features.  (Split TF32 operands, which need no scales, have half the MMA rate and twice the
// shared-memory bytes; grids that do not fill the device still use them, see launch_attention_tc().)
// (The paper keeps attention in fp32 and quantises only the FC layers; this kernel is the fp32 attention an
// encoder forward needs around them.)
//
// One CTA = 128 queries of one (sequence, head), two CTAs per SM (97 KB of shared memory and 256 TMEM columns each), so that
// one CTA's waits run under the other's work.  Keys come in chunks of 64 through two buffers each for K, V and the scores,
// so the scores of chunk c + 1 are computed while the softmax works on chunk c.  Roles:
//   warps 0..3  softmax: one thread per query row (no exchange between threads at all): scores out of TMEM, running
//               maximum, p = 2^(s - max), both fp16 parts of p back into TMEM over the scores, from where the second
//               product takes them as its A operand.  P V of one chunk is a fresh accumulation (small partial products
//               first); the running output lives in 64 registers of the row's thread and is added to in fp32, because the
//               tensor core truncates when it accumulates: one chain over 512 keys had an error of 6.6e-7 of |ctx|, growing
//               with the length (now 1.7e-7 at any length, inputs ~ N(0, 0.55); plain fp32 FMAs: 4.2e-7).  The output is
//               rescaled only when a row's maximum has risen by more than 2^2 (p has room for that), or V's unit in some feature.
//   warps 4..7  staging: K and V global -> registers -> scale, split -> shared memory, 128-byte-swizzled rows of 64 fp16.  K
//               is a K-major operand; V keeps its [key][feature] order and is read as an MN-major operand.
//   warp 8      issues the MMAs (converged, one elected lane); the rest of its warpgroup is there for setmaxnreg, which gives
//               the softmax 128 registers a thread and the staging 88, the one split without spills in the loops (120 / 96: 3 % slower, 112 / 104:
//               8 %; with 96 for all, O was spilled).
// Where the split parts would not carry what fp32 carries, the row is computed over again in plain fp32 FMAs, by its own thread
// (plain_rows_of_warp()):
//   - largest |q| of the row times largest |k| of a chunk above 2^kScoreExponent.  Up to there a score is off by less than
//     2^-20 in its exponent of 2 whatever the operands look like (64 products, each operand off by 2^-39 of its largest), and
//     the reference maximum, a whole number below 2^18, is subtracted without a loss.
//   - a row whose result is small beside V in every feature (kSmallResult): it hangs on keys whose V is tiny beside that of
//     others, and what those are rounded by counts.
//   - infinities.
// Measured (64 x 384 x 16 heads / 16 x 512 x 12 / 32 x 128 x 12, Int8 output): 227 / 72 / 20 us; split TF32 with whole score
// rows in TMEM, one CTA per SM, 512 threads staging: 304 / - / 23.8 us (it takes S <= 384; plain fp32 FMAs needed 413 us at
// 512).  What bounds it now is latency: loads of K and V (without them 25 % less) and the chain softmax -> P V -> scores
// between the roles, with the issue slots 40 % busy and the tensor pipe 20 %.  Tried and dropped: a persistent grid (the
// item loop's state does not fit the registers, 250 us), 16-column softmax loops (242 us), Q in shared memory (259 us).
// The roles meet only through mbarriers, and every wait on one is bounded: on a time-out the CTA raises Q8_ERR_TIMEOUT
// in the status word, every role leaves its loop and TMEM is freed.

#include "q8_internal.cuh"
#include "q8_sm100_ptx.cuh"

namespace q8 {

namespace {

using namespace ptx;

constexpr int kHeadDim = 64;
constexpr int kQTile = 128;  // queries per CTA = TMEM lanes
constexpr int kChunk = 64;   // keys per chunk
constexpr int kSoftmaxWarps = 4, kStagingWarps = 4;
constexpr int kThreads = 384;  // three warpgroups: softmax, staging, and one whose first warp issues the MMAs
// Registers per thread after the redistribution between the warpgroups; their sum must not exceed what the CTA is launched
// with (checked on the host: an increase that cannot be served would wait for ever).
constexpr int kLaunchRegs = 80, kSoftmaxRegs = 128, kStagingRegs = 88, kIssuerRegs = 24;
static_assert(kSoftmaxRegs + kStagingRegs + kIssuerRegs <= 3 * kLaunchRegs, "register split");
constexpr int kRowBytes = kHeadDim * 4;      // an fp32 row of Q or of the output
constexpr int kQBytes = kQTile * kRowBytes;  // fp32 Q on its way in, the output on its way out: 32 KB
constexpr int kKvHalfBytes = kChunk * 128;   // rows of 64 fp16: the hi (or the lo) half of a K or V chunk, 8 KB
constexpr int kKvBytes = 2 * kKvHalfBytes;
constexpr int kAttnTcSmemBytes = 1024 + 4 * kKvBytes + kQBytes;  // two K, two V buffers, Q: 97 KB
constexpr uint32_t kTmemCols = 256;  // scores / P of two chunks, P V of one, Q (32 columns of hi parts, 32 of lo parts)
constexpr uint32_t kColPV = 128, kColQ = 192;
constexpr float kLog2eOver8 = 1.4426950408889634f / 8.0f;  // log2(e) / sqrt(64): the softmax uses 2^x
constexpr int kPShift = 13;          // p is split as 2^13 p: at most 2^15 with the stale-maximum slack below, and small p keep
constexpr float kStaleSlack = 2.0f;  // their precision (fp16 rounds absolutely below 2^-14)
constexpr int kScoreExponent = 14;           // log2 of the largest |q| |k| that the split product takes (of values ~ N(0, 1): 2^4)
constexpr float kSmallResult = 4.0f;           // in V's units, whose largest is 2^12 .. 2^15 (a mean of 4096 values ~ N(0, 1): 2^6)

// tcgen05.mma kind::f16 instruction descriptor: D = F32, A = B = F16, M = 128; bit 16: B is MN-major.
constexpr uint32_t kIdescBase = (1u << 4) | ((uint32_t)(kQTile >> 4) << 24);
constexpr uint32_t kIdescPV = kIdescBase | (1u << 16) | ((uint32_t)(kHeadDim >> 3) << 17);

// Byte offset of the 16-byte piece `piece` (0..7) of row `row` inside one swizzle span (rows of 128 bytes,
// groups of 8 rows 1024 bytes apart, piece index XORed with the row's position in its group).
__device__ __forceinline__ uint32_t sw128_offset(int row, int piece)
{
    return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((piece ^ (row & 7)) << 4));
}

// Descriptor of the [key][feature] tile of V as an MN-major B operand: 64 features (one 128-byte swizzle span) per atom of 8
// keys, atoms 1024 bytes apart along the keys (stride byte offset); the leading byte offset would be the step to further
// features.
__device__ __forceinline__ uint64_t smem_desc_v(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kKvHalfBytes >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

// D[tmem] (+)= A B^T, fp32 accumulation.  A from tensor memory: lane = row, two fp16 of K per 32-bit column (8 columns per
// instruction); read from shared memory, a 128 x 16 operand costs more than the 64 x 16 one of K or V (48 against 32 cycles).
__device__ __forceinline__ void umma_f16_ts_elected(uint32_t elected, uint32_t tmem_d, uint32_t tmem_a, uint64_t desc_b,
                                                    uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(tmem_d), "r"(tmem_a), "l"(desc_b), "r"(idesc), "r"(accumulate), "r"(elected)
        : "memory");
}
__device__ __forceinline__ void tmem_st_32x8(uint32_t taddr, const uint32_t (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

// {hi, lo} = fp16 pairs of two values (the first in the low half): hi = fp16(x), lo = fp16(x - hi), the difference exact in
// fp32.  The subtraction is the mixed-precision FMA hi * -1 + x, which takes hi as it is.
__device__ __forceinline__ uint32_t pack_f16x2(float a, float b)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
    return r;
}
__device__ __forceinline__ void split2(uint64_t x2, uint32_t &hi, uint32_t &lo)
{
    float a, b, la, lb;
    unpack_f32x2(x2, a, b);
    hi = pack_f16x2(a, b);
    asm("{\n\t.reg .b16 h0, h1, m;\n\t"
        "mov.b32 {h0, h1}, %2;\n\t"
        "mov.b16 m, 0xBC00;\n\t"
        "fma.rn.f32.f16 %0, h0, m, %3;\n\t"
        "fma.rn.f32.f16 %1, h1, m, %4;\n\t}"
        : "=f"(la), "=f"(lb) : "r"(hi), "f"(a), "f"(b));
    lo = pack_f16x2(la, lb);
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float exp2_fast(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t at)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at) : "memory");
    return v;
}

// Largest magnitude among N float4 (a NaN does not take part; an infinity sends the rows to plain_rows_of_warp()) of each component ...
template <int N>
__device__ __forceinline__ float4 absmax_columns(const float4 (&v)[N])
{
    float4 m = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < N; ++i)
        m = make_float4(fmaxf(m.x, fabsf(v[i].x)), fmaxf(m.y, fabsf(v[i].y)), fmaxf(m.z, fabsf(v[i].z)), fmaxf(m.w, fabsf(v[i].w)));
    return m;
}
// ... and of all of them, as fp32 bits.
template <int N>
__device__ __forceinline__ uint32_t absmax_bits(const float4 (&v)[N])
{
    float m = 0.0f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        m = fmaxf(fmaxf(m, fabsf(v[i].x)), fabsf(v[i].y));
        m = fmaxf(fmaxf(m, fabsf(v[i].z)), fabsf(v[i].w));
    }
    return __float_as_uint(m);
}
// Exponent g with max * 2^-g in [2^13, 2^14) for a maximum given as fp32 bits (at least -126, so that 2^-g is a normal number)
__device__ __forceinline__ int scale_exponent(uint32_t max_bits) { return max((int)(max_bits >> 23), 14) - 140; }
__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }  // -126 <= e <= 127

// Tile staging by 128 threads: thread t holds float4 piece t % 16 (of 16 per row) of rows t / 16 + 8 i.
template <int ROWS>
struct Tile {
    float4 v[ROWS / 8];
    // Rows past the last one repeat it: a K row there gives scores that are masked, a V row is multiplied by p = 0.
    __device__ __forceinline__ void fetch(const float *base, uint32_t pitch_bytes, int t, int rows)
    {
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i)
            v[i] = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(base) +
                                                          ((uint32_t)min((t >> 4) + 8 * i, rows - 1) * pitch_bytes + 16u * (t & 15))));
    }
    // mult: a power of two for each of this thread's four features
    __device__ __forceinline__ void scale(float4 mult)
    {
        const uint64_t mult_xy = pack_f32x2(mult.x, mult.y), mult_zw = pack_f32x2(mult.z, mult.w);
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i) {
            unpack_f32x2(mul_f32x2(pack_f32x2(v[i].x, v[i].y), mult_xy), v[i].x, v[i].y);
            unpack_f32x2(mul_f32x2(pack_f32x2(v[i].z, v[i].w), mult_zw), v[i].z, v[i].w);
        }
    }
    __device__ __forceinline__ void store(uint32_t tile, int t) const
    {
        // (rows t / 16 + 8 i: the same place in every group of 8 rows)
        const uint32_t at = tile + sw128_offset(t >> 4, (t & 15) >> 1) + 8 * (t & 1);
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i) {
            uint2 hi, lo;
            split2(pack_f32x2(v[i].x, v[i].y), hi.x, lo.x);
            split2(pack_f32x2(v[i].z, v[i].w), hi.y, lo.y);
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + 1024 * i), "r"(hi.x), "r"(hi.y) : "memory");
            asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + 1024 * i + ROWS * 128), "r"(lo.x), "r"(lo.y) : "memory");
        }
    }
};

// The 32 query rows of a warp in plain fp32 FMAs, a thread each (see the top of the file): softmax(q K^T / 8) V over all S keys, one at
// a time, with the running maximum and sum of q8_support.cu's kernel.  q_at(i): shared-memory address of the i-th 16 bytes of
// the thread's q.  stage: 16 KB of shared memory for keys on their way, 16 of K and of V at a time through two buffers.  Leaves the
// sum of p v in O, returns the sum of p.  (With every row of 16 x 512 x 12 heads here: 1.05 ms; keys read from where they lie
// 3.6 ms; the CUDA-core kernel 0.41 ms.  Four keys at a time took 0.72 ms, but their registers are spilled in the loops of the
// ordinary path: 64 x 384 x 16 heads 227 -> 231 us.)
template <typename QAt>
__device__ __forceinline__ float plain_rows_of_warp(QAt q_at, const float *qkv, int S, int64_t H, uint32_t stage, int lane,
                                                    uint64_t (&O)[kHeadDim / 2])
{
    uint32_t head, seq;  // read here, so that the caller's loop need not keep them
    asm volatile("mov.u32 %0, %%ctaid.y;\n\tmov.u32 %1, %%ctaid.z;" : "=r"(head), "=r"(seq));
    const int64_t row_pitch = 3 * H;
    const float *k = qkv + seq * (int64_t)S * row_pitch + head * kHeadDim + H + 4 * (lane & 15);
    constexpr int kKeys = 16;
    auto fetch = [&](int j0, uint32_t to) {
#pragma unroll 1
        for (int i = 0; i < kKeys / 2; ++i) {
            const int r = 2 * i + (lane >> 4);
            const bool in = j0 + r < S;  // past the end: zeros
            const float *src = k + (int64_t)(in ? j0 + r : 0) * row_pitch;
            const uint32_t at = to + (uint32_t)(r * kRowBytes + 16 * (lane & 15));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(at), "l"(src), "r"(in ? 16 : 0) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(at + kKeys * kRowBytes), "l"(src + H), "r"(in ? 16 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float m = -INFINITY, l = 0.0f;
#pragma unroll
    for (int j = 0; j < kHeadDim / 2; ++j) O[j] = 0;  // (+0, +0)
    fetch(0, stage);
#pragma unroll 1
    for (int j = 0; j < S; ++j) {
        const int r = j & (kKeys - 1), buf = (j / kKeys) & 1;
        const uint32_t row = stage + (uint32_t)(2 * buf * kKeys * kRowBytes + r * kRowBytes);
        if (r == 0) {
            __syncwarp();  // everybody has left the other buffer
            fetch(j + kKeys, stage + (uint32_t)(2 * (buf ^ 1) * kKeys * kRowBytes));
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
        }
        float4 dot = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
        for (int i = 0; i < kHeadDim / 4; ++i) {
            const float4 q = ld_shared_f4(q_at(i)), x = ld_shared_f4(row + 16u * i);  // (a key is at the same address in every lane)
            dot.x = fmaf(q.x * kLog2eOver8, x.x, dot.x);
            dot.y = fmaf(q.y * kLog2eOver8, x.y, dot.y);
            dot.z = fmaf(q.z * kLog2eOver8, x.z, dot.z);
            dot.w = fmaf(q.w * kLog2eOver8, x.w, dot.w);
        }
        const float s = (dot.x + dot.y) + (dot.z + dot.w), m_new = fmaxf(m, s);
        const float ref = m_new == -INFINITY ? 0.0f : m_new;  // (only scores of -inf so far: their p is 0)
        const float corr = exp2f(m - ref), p = exp2f(s - ref);
        l = fmaf(l, corr, p);
        m = m_new;
        const uint64_t p2 = pack_f32x2(p, p), corr2 = pack_f32x2(corr, corr);
#pragma unroll
        for (int i = 0; i < kHeadDim / 4; ++i) {
            const float4 x = ld_shared_f4(row + (uint32_t)(kKeys * kRowBytes + 16 * i));
            O[2 * i] = fma_f32x2(pack_f32x2(x.x, x.y), p2, mul_f32x2(O[2 * i], corr2));
            O[2 * i + 1] = fma_f32x2(pack_f32x2(x.z, x.w), p2, mul_f32x2(O[2 * i + 1], corr2));
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    return l;
}

template <int N>
__device__ __forceinline__ void grow_registers() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void shrink_registers() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

__device__ __forceinline__ void staging_barrier() { asm volatile("bar.sync 2, 128;" ::: "memory"); }
__device__ __forceinline__ bool staging_any(bool mine)  // whether it holds in any of the staging threads
{
    uint32_t any;
    asm volatile("{\n\t.reg .pred m, a;\n\tsetp.ne.u32 m, %1, 0;\n\tbar.red.or.pred a, 2, 128, m;\n\tselp.u32 %0, 1, 0, a;\n\t}"
                 : "=r"(any) : "r"(mine ? 1u : 0u) : "memory");
    return any != 0;
}

__global__ void __launch_bounds__(kThreads, 2)
attention_tc_kernel(const float *__restrict__ qkv, int S, int64_t H, float *__restrict__ ctx,
                    const float *__restrict__ S_q, int8_t *__restrict__ ctx_q, uint32_t *__restrict__ amax,
                    int32_t *status)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
    auto k_tile = [&](int buf) { return smem + (uint32_t)(buf * kKvBytes); };
    auto v_tile = [&](int buf) { return smem + (uint32_t)((2 + buf) * kKvBytes); };
    const uint32_t q_rows = smem + 4 * kKvBytes;
    __shared__ __align__(8) uint64_t bars[11];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) uint32_t k_max[2][kStagingWarps];  // [chunk parity][warp]
    __shared__ __align__(16) float v_max[kStagingWarps][kHeadDim];
    // K = K' 2^exponent, V = V' unit (a power of two for each feature).  By chunk number modulo 4: K's exponent, whether V's units
    // rose and what the output so far is multiplied by then.  (K of chunk c + 2 may be staged while the softmax of chunk c still
    // reads its exponent; K of chunk c + 4 is staged after P of chunk c + 1 was handed over, V's units of chunk c + 4 after
    // P of chunk c + 1 was.)
    __shared__ int k_exponent[4], v_rose[4];
    __shared__ __align__(16) float v_factor[4][kHeadDim];
    __shared__ __align__(16) float v_unit[kHeadDim];  // after the last chunk
    __shared__ int v_any, v_far;                      // any of V is not zero, is infinite
    // barrier of each kind for buffer `buf` = chunk parity
    const uint32_t bar0 = smem_u32(bars), q_ready = bar0 + 80;
    auto k_ready = [&](int buf) { return bar0 + 8 * buf; };        // staging -> MMA: K is in place
    auto v_ready = [&](int buf) { return bar0 + 16 + 8 * buf; };   // staging -> MMA, softmax: V (and its units)
    // MMA -> softmax, staging: scores complete, K read; and staging -> softmax: K's exponent
    auto s_done = [&](int buf) { return bar0 + 32 + 8 * buf; };
    auto p_ready = [&](int buf) { return bar0 + 48 + 8 * buf; };   // softmax -> MMA: P is in tensor memory
    auto pv_done = [&](int buf) { return bar0 + 64 + 8 * buf; };   // MMA -> staging, softmax: P V complete, P and V read

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q0 = blockIdx.x * kQTile;
    const int64_t head = blockIdx.y, seq = blockIdx.z;
    const int64_t row_pitch = 3 * H;
    const float *base = qkv + seq * (int64_t)S * row_pitch + head * kHeadDim;
    const int chunks = (S + kChunk - 1) / kChunk;
    // columns of chunk c: whole chunks are 64 wide, the last one is rounded up to 32
    auto chunk_cols = [&](int c) { return c + 1 < chunks ? kChunk : ((S - c * kChunk + 31) & ~31); };

    if (tid == 0) {
        mbar_init(q_ready, kSoftmaxWarps);
        for (int buf = 0; buf < 2; ++buf) {
            mbar_init(k_ready(buf), kStagingWarps);
            mbar_init(v_ready(buf), kStagingWarps);
            mbar_init(s_done(buf), 2);
            mbar_init(p_ready(buf), kSoftmaxWarps);
            mbar_init(pv_done(buf), 1);
        }
        abort_flag = 0;
        v_any = 0;
        v_far = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kSoftmaxWarps + kStagingWarps) tmem_alloc(smem_u32(&tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    grid_dependency_release_next(true);
    grid_dependency_wait();  // the set-up above may overlap the tail of the kernel that produced qkv

    bool ok = true;
    // Whole warp, same outcome in every lane; bounded.  (One short polling loop instead of mbar_wait(), whose copies were a
    // fifth of the kernel's code.  A try may sleep in hardware for up to 0.2 ms: waits of several hundred cycles are the rule
    // here, and a polling warp takes issue slots from the other CTA: 64 x 384 x 16 heads 241 -> 233 us.)
    auto wait = [&](uint32_t bar, uint32_t parity) {
        uint64_t t0 = 0;
#pragma unroll 1
        while (!__all_sync(0xffffffffu, mbar_try_wait_for(bar, parity, 200000u))) {
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > kWaitLimitNs) {
                *(volatile int *)&abort_flag = 1;
                if (status) atomicOr(status, 1 << Q8_ERR_TIMEOUT);
            }
            if (__any_sync(0xffffffffu, *(volatile int *)&abort_flag)) {
                ok = false;
                break;
            }
        }
        tc_fence_after();
        return ok;
    };
    // one arrival per warp, after every lane's writes (tensor memory, and shared memory with the fence) are visible to the
    // tensor core
    auto arrive = [&](uint32_t bar, bool wrote_smem) {
        if (wrote_smem) fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };

    if (warp >= kSoftmaxWarps + kStagingWarps) {
        // ================= MMA issuer (the other warps of its group have nothing to do)
        shrink_registers<kIssuerRegs>();
        if (warp == kSoftmaxWarps + kStagingWarps) {
            const uint32_t elected = elect_one();
            auto issue_scores = [&](int c) {  // S(c) = Q K(c)^T into the columns of buffer c % 2
                const int buf = c & 1;
                const uint32_t par = (uint32_t)((c >> 1) & 1), d = tmem_base + (uint32_t)(buf * kChunk);
                if (!wait(k_ready(buf), par)) return;
                if (c >= 2 && !wait(pv_done(buf), par ^ 1u)) return;  // P of chunk c - 2 lies there
                const uint64_t k_hi = smem_desc_sw128(k_tile(buf)), k_lo = k_hi + (uint64_t)(kKvHalfBytes >> 4);
                const uint32_t idesc = kIdescBase | ((uint32_t)(chunk_cols(c) >> 3) << 17);
                const uint32_t q_hi = tmem_base + kColQ, q_lo = q_hi + 32;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {  // 16 fp16 = 32 bytes of K per instruction: +2 in the (address >> 4) field
                    umma_f16_ts_elected(elected, d, q_lo + 8 * ks, k_hi + 2 * ks, idesc, ks > 0 ? 1u : 0u);  // small terms first
                    umma_f16_ts_elected(elected, d, q_hi + 8 * ks, k_lo + 2 * ks, idesc, 1u);
                }
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) umma_f16_ts_elected(elected, d, q_hi + 8 * ks, k_hi + 2 * ks, idesc, 1u);
                umma_commit_elected(elected, s_done(buf));
            };
            auto issue_pv = [&](int c) {  // P(c) V(c) into the product columns (the softmax has read P(c - 1) V(c - 1) before)
                const int buf = c & 1, steps = chunk_cols(c) / 16;
                const uint32_t par = (uint32_t)((c >> 1) & 1), d = tmem_base + kColPV;
                if (!wait(v_ready(buf), par) || !wait(p_ready(buf), par)) return;
                const uint64_t v_hi = smem_desc_v(v_tile(buf)), v_lo = v_hi + (uint64_t)(kKvHalfBytes >> 4);
                // P: per 16 keys 8 columns of hi parts, then 8 of lo parts; 16 keys are two atoms (2048 bytes) of V
                auto p_at = [&](int ks) { return tmem_base + (uint32_t)(buf * kChunk + 16 * ks); };
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    if (ks >= steps) break;
                    umma_f16_ts_elected(elected, d, p_at(ks) + 8, v_hi + ks * (2048 >> 4), kIdescPV, ks > 0 ? 1u : 0u);
                    umma_f16_ts_elected(elected, d, p_at(ks), v_lo + ks * (2048 >> 4), kIdescPV, 1u);
                }
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    if (ks >= steps) break;
                    umma_f16_ts_elected(elected, d, p_at(ks), v_hi + ks * (2048 >> 4), kIdescPV, 1u);
                }
                umma_commit_elected(elected, pv_done(buf));
            };
            // P(c - 1) becomes ready about when the softmax turns to S(c); the products of chunk c - 1 and, when they have
            // read P(c - 1), the scores of chunk c + 1 in its place then run under the softmax of chunk c
            if (wait(q_ready, 0)) issue_scores(0);
#pragma unroll 1
            for (int c = 0; c < chunks && ok; ++c) {
                if (c + 1 < chunks) issue_scores(c + 1);
                if (ok) issue_pv(c);
            }
            if (!ok) {  // aborting: let the MMAs issued so far finish before the tensor memory is freed
                const uint64_t t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 1000000ull) {}
            }
        }
    } else if (warp >= kSoftmaxWarps) {
        // ================= staging warps
        grow_registers<kStagingRegs>();
        const int t = tid - 32 * kSoftmaxWarps, w = warp - kSoftmaxWarps;
        const float *kv = base + H;  // K of the next chunk; V lies H further
        const uint32_t pitch_bytes = (uint32_t)row_pitch * 4u;
        Tile<kChunk> kt, vt;
        auto k_chunk_exponent = [&](int c) {
            const uint32_t m = __reduce_max_sync(0xffffffffu, absmax_bits(kt.v));
            if (lane == 0) k_max[c & 1][w] = m;
            staging_barrier();
            const uint4 x = *reinterpret_cast<const uint4 *>(k_max[c & 1]);
            return scale_exponent(max(max(x.x, x.y), max(x.z, x.w)));
        };
        // V's units of this thread's four features, one byte each: exponent + 126.  Chunk 0 brings its largest values into
        // [2^12, 2^13); a unit rises only when a later value would reach 2^15 in it, which is rare, so that a chunk costs one vote.
        uint32_t units = 0;
        auto unit = [&](int i) { return (int)((units >> (8 * i)) & 255u); };
        auto in_units = [&]() { vt.scale(make_float4(pow2(126 - unit(0)), pow2(126 - unit(1)), pow2(126 - unit(2)), pow2(126 - unit(3)))); };
        auto scale_v = [&](int c) {
            if (c > 0) {
                in_units();
                float top = 0.0f;
#pragma unroll
                for (int i = 0; i < kChunk / 8; ++i) {
                    top = fmaxf(fmaxf(top, fabsf(vt.v[i].x)), fabsf(vt.v[i].y));
                    top = fmaxf(fmaxf(top, fabsf(vt.v[i].z)), fabsf(vt.v[i].w));
                }
                if (!staging_any(top >= 32768.0f)) {
                    if (t == 0) v_rose[c & 3] = 0;
                    return;
                }
                vt.fetch(kv + H - kChunk * row_pitch, pitch_bytes, t, S - c * kChunk);  // (in_units() may have overflowed)
            }
            float4 m = absmax_columns(vt.v);
            m = make_float4(fmaxf(m.x, __shfl_xor_sync(0xffffffffu, m.x, 16)), fmaxf(m.y, __shfl_xor_sync(0xffffffffu, m.y, 16)),
                            fmaxf(m.z, __shfl_xor_sync(0xffffffffu, m.z, 16)), fmaxf(m.w, __shfl_xor_sync(0xffffffffu, m.w, 16)));
            if (lane < 16) *reinterpret_cast<float4 *>(&v_max[w][4 * lane]) = m;
            staging_barrier();
#pragma unroll
            for (int i = 0; i < kStagingWarps; ++i) {
                const float4 x = *reinterpret_cast<const float4 *>(&v_max[i][4 * (t & 15)]);
                m = make_float4(fmaxf(m.x, x.x), fmaxf(m.y, x.y), fmaxf(m.z, x.z), fmaxf(m.w, x.w));
            }
            auto above = [&](float x, int i) { return __float_as_uint(x) >= (uint32_t)min(unit(i) + 16, 255) << 23; };  // 2^15 units
            auto raised = [&](float x, int i) { return c == 0 || above(x, i) ? scale_exponent(__float_as_uint(x)) + 127 : unit(i); };
            const int e[4] = {raised(m.x, 0), raised(m.y, 1), raised(m.z, 2), raised(m.w, 3)};
            if (t < 16) {
                const float top = fmaxf(fmaxf(m.x, m.y), fmaxf(m.z, m.w));
                if (top > 0.0f) v_any = 1;
                if (top == INFINITY) v_far = 1;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v_factor[c & 3][4 * t + i] = pow2(max(unit(i) - e[i], -126));
                    v_unit[4 * t + i] = pow2(e[i] - 126);
                }
            }
            if (t == 0) v_rose[c & 3] = c > 0;
            units = (uint32_t)(e[0] | e[1] << 8 | e[2] << 16 | e[3] << 24);
            in_units();
        };
        // (chunk -1: nothing to stage yet, its fetches bring in chunk 0; after a time-out the loop still runs, for the
        // barriers of its group alone)
#pragma unroll 1
        for (int c = -1; c < chunks; ++c) {
            const int buf = c & 1, left = S - (c + 1) * kChunk;  // keys behind this chunk
            const uint32_t freed = (uint32_t)(((c >> 1) & 1) ^ 1);
            if (c >= 0) {
                const int gk = k_chunk_exponent(c);
                if (c >= 2 && ok) wait(s_done(buf), freed);  // K of chunk c - 2 has been read
                if (ok) {
                    kt.scale(make_float4(pow2(-gk), pow2(-gk), pow2(-gk), pow2(-gk)));
                    kt.store(k_tile(buf), t);
                    if (t == 0) k_exponent[c & 3] = gk;
                    if (t == 0) mbar_arrive(s_done(buf));
                    arrive(k_ready(buf), true);
                }
            }
            if (left > 0) kt.fetch(kv, pitch_bytes, t, left);
            if (c >= 0) {
                scale_v(c);
                if (c >= 2 && ok) wait(pv_done(buf), freed);  // V of chunk c - 2 has been read
                if (ok) {
                    vt.store(v_tile(buf), t);
                    arrive(v_ready(buf), true);
                }
            }
            if (left > 0) vt.fetch(kv + H, pitch_bytes, t, left);
            kv += kChunk * row_pitch;
        }
    } else {
        // ================= softmax warps: thread = query row = TMEM lane
        grow_registers<kSoftmaxRegs>();
        const float Sq = ctx_q != nullptr ? __ldg(S_q) : 1.0f;
        const uint32_t t_row = tmem_base + ((uint32_t)(warp * 32) << 16);
        const bool warp_live = q0 + 32 * warp < S;  // a warp whose rows all lie past the end only keeps the barriers going
        const uint32_t my_rows = q_rows + (uint32_t)(warp * (32 * kRowBytes));  // 16-byte pieces XORed with the row
        auto piece = [&](int r, int i) { return my_rows + (uint32_t)(r * kRowBytes + ((i ^ (r & 15)) << 4)); };
        // Q: this warp's 32 rows to shared memory (whole lines), every thread takes its row, scales it by a power of two of its
        // own and puts both fp16 parts into tensor memory: the A operand of the scores.
        int gq = 0;
        {
#pragma unroll 4
            for (int i = 0; i < 16; ++i) {
                const int r = 2 * i + (lane >> 4), pc = lane & 15;
                const bool in = q0 + 32 * warp + r < S;  // rows past the end are filled with zeros
                const float *src = base + (int64_t)(in ? q0 + 32 * warp + r : 0) * row_pitch + 4 * pc;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(piece(r, pc)), "l"(src), "r"(in ? 16 : 0) : "memory");
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
            float4 v[4];
            uint32_t mq = 0;
#pragma unroll 1
            for (int h = 0; h < 4; ++h) {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = ld_shared_f4(piece(lane, 4 * h + i));
                mq = max(mq, absmax_bits(v));
            }
            gq = scale_exponent(mq);
            const uint64_t m2 = pack_f32x2(pow2(-gq), pow2(-gq));
#pragma unroll 1
            for (int h = 0; h < 4; ++h) {
                uint32_t hi[8], lo[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = ld_shared_f4(piece(lane, 4 * h + i));
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    split2(mul_f32x2(pack_f32x2(v[i].x, v[i].y), m2), hi[2 * i], lo[2 * i]);
                    split2(mul_f32x2(pack_f32x2(v[i].z, v[i].w), m2), hi[2 * i + 1], lo[2 * i + 1]);
                }
                tmem_st_32x8(t_row + kColQ + 8 * h, hi);
                tmem_st_32x8(t_row + kColQ + 32 + 8 * h, lo);
            }
            tmem_st_wait();
            arrive(q_ready, false);
        }
        // Reference maximum R of the scores, a whole number so that every power of two between two of them is exact: P is 2^(s - R),
        // the row sum l is in units of 2^R, the running output O in units of 2^(R - kPShift) times V's units
        float R = 0.0f;
        float l = 0.0f;
        uint64_t O[kHeadDim / 2];
#pragma unroll
        for (int j = 0; j < kHeadDim / 2; ++j) O[j] = 0;  // (+0, +0)
        auto add_product = [&](int c) {  // O += P(c) V(c)
            if (!wait(pv_done(c & 1), (uint32_t)((c >> 1) & 1))) return;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t x[32];
                tmem_ld_32x32(t_row + kColPV + (uint32_t)(32 * h), x);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    O[16 * h + j] = add_f32x2(O[16 * h + j], pack_f32x2(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1])));
            }
        };
        for (int c = 0; c < chunks && ok; ++c) {
            const int buf = c & 1, left = S - c * kChunk;
            const uint32_t par = (uint32_t)((c >> 1) & 1), t_s = t_row + (uint32_t)(buf * kChunk);
            if (!wait(s_done(buf), par)) break;
            if (warp_live) {
                const int g = gq + k_exponent[c & 3];
                if (g + 28 > kScoreExponent) l = NAN;  // (largest |q| |k| may reach 2^(g + 28): the row goes to plain_rows_of_warp())
                const float f = pow2(max(-126, min(120, g))) * kLog2eOver8;
                // half 1 of the scores is read twice (for the maximum, then for the exponentials), half 0 stays in registers
                uint32_t sv[32];
                float mc = -INFINITY;
                auto load_half = [&](int h) {
                    tmem_ld_32x32(t_s + (uint32_t)(32 * h), sv);
                    tmem_ld_wait();
                    if (left < 32 * h + 32) {  // the last columns of a ragged sequence: keys past its end get p = 2^-inf
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (32 * h + j >= left) sv[j] = 0xFF800000u;
                    }
                };
                auto take_max = [&](int h) {
                    load_half(h);
                    float m1 = -INFINITY;
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        mc = fmaxf(fmaxf(mc, __uint_as_float(sv[j])), __uint_as_float(sv[j + 1]));
                        m1 = fmaxf(fmaxf(m1, __uint_as_float(sv[j + 2])), __uint_as_float(sv[j + 3]));
                    }
                    mc = fmaxf(mc, m1);
                };
                const bool two = left > 32;
                if (two) take_max(1);
                take_max(0);
                mc = ceilf(mc * f);
                float rescale = 1.0f;
                if (c == 0) {
                    R = mc;
                } else if (mc > R + kStaleSlack) {
                    rescale = exp2_fast(R - mc);
                    R = mc;
                }
                const uint64_t f2 = pack_f32x2(f, f), b2 = pack_f32x2(-R, -R);
                const uint64_t shift2 = pack_f32x2((float)(1 << kPShift), (float)(1 << kPShift));
                uint64_t sum_a = 0, sum_b = 0;  // (+0, +0)
                auto exponentials = [&](int h) {  // 16 keys: 8 columns of hi parts, then 8 of lo parts, over their scores
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t hi[8], lo[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            float x0, x1;
                            const int k = 16 * q + 2 * j;
                            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(sv[k]), __uint_as_float(sv[k + 1])), f2, b2), x0, x1);
                            const uint64_t e2 = pack_f32x2(exp2_fast(x0), exp2_fast(x1));
                            if (j & 1) sum_a = add_f32x2(sum_a, e2);
                            else sum_b = add_f32x2(sum_b, e2);
                            split2(mul_f32x2(e2, shift2), hi[j], lo[j]);
                        }
                        tmem_st_32x8(t_s + (uint32_t)(32 * h + 16 * q), hi);
                        tmem_st_32x8(t_s + (uint32_t)(32 * h + 16 * q + 8), lo);
                    }
                };
                exponentials(0);
                if (two) {
                    load_half(1);
                    exponentials(1);
                }
                float sum0, sum1, sum2, sum3;
                unpack_f32x2(sum_a, sum0, sum1);
                unpack_f32x2(sum_b, sum2, sum3);
                l = fmaf(l, rescale, (sum0 + sum1) + (sum2 + sum3));
                if (c > 0) {
                    add_product(c - 1);
                    if (__any_sync(0xffffffffu, rescale != 1.0f)) {
                        const uint64_t r2 = pack_f32x2(rescale, rescale);
#pragma unroll
                        for (int j = 0; j < kHeadDim / 2; ++j) O[j] = mul_f32x2(O[j], r2);
                    }
                }
                tmem_st_wait();
            }
            // V's units of this chunk.  (Before P is handed over: V of chunk c + 2 would complete the barrier's next phase.)
            if (!wait(v_ready(buf), par)) break;
            arrive(p_ready(buf), false);
            if (v_rose[c & 3] != 0) {
                const uint32_t factor = smem_u32(v_factor[c & 3]);
#pragma unroll
                for (int j = 0; j < kHeadDim / 2; ++j) {
                    uint64_t f2;
                    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(f2) : "r"(factor + 8 * j) : "memory");
                    O[j] = mul_f32x2(O[j], f2);
                }
            }
        }
        // ---------------- ctx = O / row sum
        if (ok && warp_live) add_product(chunks - 1);
        if (ok && warp_live) {
            // Normalised rows to shared memory (where Q came in), then a half-warp takes a row at a time, so that whole lines
            // are stored.  In a short loop: written out for a thread's 64 values this was a third of the kernel's code.
            float inv = pow2(-kPShift) / l;
            float top = v_any != 0 ? 0.0f : INFINITY;
#pragma unroll
            for (int j = 0; j < kHeadDim / 2; ++j) {
                float a, b;
                unpack_f32x2(O[j], a, b);
                top = fmaxf(fmaxf(top, fabsf(a)), fabsf(b));
            }
            const bool plain = (v_far != 0 || !(top * inv >= kSmallResult)) && q0 + 32 * warp + lane < S;
            const uint32_t plain_rows = __ballot_sync(0xffffffffu, plain);
            if (__builtin_expect(plain_rows != 0, 0)) {
                // K and V have been read by every product; each warp has a quarter of their buffers.  The whole warp fetches the keys;
                // a thread whose row is done puts it aside, where its q was, and computes something of no use.
                auto row = [&](int i) { return piece(lane, i); };
                if (!plain) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(row(i)), "l"(O[2 * i]), "l"(O[2 * i + 1]) : "memory");
                }
                const float sum = plain_rows_of_warp(row, qkv, S, H, smem + (uint32_t)(warp * kKvBytes), lane, O);
                if (plain) {
                    inv = 1.0f / sum;
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(O[2 * i]), "=l"(O[2 * i + 1]) : "r"(row(i)) : "memory");
                }
            }
            const uint64_t inv2 = pack_f32x2(inv, inv);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                asm volatile("st.shared.v2.b64 [%0], {%1, %2};"
                             ::"r"(piece(lane, i)), "l"(mul_f32x2(O[2 * i], inv2)), "l"(mul_f32x2(O[2 * i + 1], inv2))
                             : "memory");
            __syncwarp();
            const int live_rows = min(32, S - q0 - 32 * warp), pc = lane & 15;
            const int64_t out0 = (seq * (int64_t)S + q0 + 32 * warp) * H + head * kHeadDim + 4 * pc;
            const float4 unit = *reinterpret_cast<const float4 *>(&v_unit[4 * pc]);
            float am = 0.0f;
#pragma unroll 2
            for (int r = lane >> 4; r < live_rows; r += 2) {
                float4 y = ld_shared_f4(piece(r, pc));
                if (((plain_rows >> r) & 1u) == 0u) y = make_float4(y.x * unit.x, y.y * unit.y, y.z * unit.z, y.w * unit.w);
                const int64_t at = out0 + (int64_t)r * H;
                am = fmaxf(fmaxf(am, fmaxf(fabsf(y.x), fabsf(y.y))), fmaxf(fabsf(y.z), fabsf(y.w)));
                if (ctx != nullptr) *reinterpret_cast<float4 *>(ctx + at) = y;
                // the same fp32 values, quantised for the next quantised layer (Eq. 1)
                if (ctx_q != nullptr) *reinterpret_cast<uint32_t *>(ctx_q + at) = quantize_pack4(y.x, y.y, y.z, y.w, Sq);
            }
            if (amax != nullptr) {  // max|ctx| for a dynamically quantised consumer (Sec. 4.1); rows past S do not count
                __syncwarp();
                warp_fold_absmax(am, amax);
            }
        }
    }

    // ---------------- teardown (reached by every thread, also after a time-out)
    tc_fence_before();
    __syncthreads();
    if (warp == kSoftmaxWarps + kStagingWarps) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

bool g_attention_tc_enabled = true;

int device_sms(int dev)
{
    static int cached[64] = {};
    if (cached[dev] == 0) {
        int v = 0;
        cached[dev] = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 148;
    }
    return cached[dev];
}

}  // namespace

void set_attention_tensor_cores(bool enable) { g_attention_tc_enabled = enable; }

// Device status word of the tensor-core attention kernels (one per device, in a file-scope array).
static __device__ int32_t g_attention_status[1];

int32_t *attention_status_word()
{
    static int32_t *cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (cached[dev] == nullptr) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_attention_status) != cudaSuccess) return nullptr;
        cached[dev] = static_cast<int32_t *>(p);
    }
    return cached[dev];
}

bool attention_tc_supported(const float *qkv, int64_t S, int64_t heads, const float *ctx, const int8_t *ctx_q)
{
    auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    // 16-byte loads and stores (H = 64 * heads keeps every row aligned); byte offsets within a chunk and key positions fit
    // 32 bits (65535 heads: 64 rows of 50 MB)
    return g_attention_tc_enabled && S <= (int64_t(1) << 30) && heads <= 65535 && al16(qkv) && al16(ctx) && al16(ctx_q);
}

cudaError_t launch_attention_tc(const float *qkv, int64_t B, int64_t S, int64_t heads, float *ctx, const float *S_q,
                                int8_t *ctx_q, uint32_t *amax, cudaStream_t s)
{
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    // With at most one CTA per SM the time is that of a single CTA, which the kernel with 512 threads per CTA has the shorter
    // (12 heads of 128: 12 CTAs 8.4 against 9.2 us, 144 CTAs 8.8 / 10.1; 144 CTAs of 384: 14.9 / 17.8); beyond, two of this
    // kernel's CTAs share an SM where the other needs a second round (192 CTAs of 128: 16.4 / 11.7 us, 288: 16.9 / 12.1).
    if ((S + kQTile - 1) / kQTile * heads * B <= device_sms(dev) && attention_small_supported(S))
        return launch_attention_small(qkv, B, S, heads, ctx, S_q, ctx_q, amax, s);
    if (!attr_set[dev]) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, attention_tc_kernel);
        if (e != cudaSuccess) return e;
        if (fa.numRegs * 3 < kSoftmaxRegs + kStagingRegs + kIssuerRegs) return cudaErrorLaunchOutOfResources;
        e = cudaFuncSetAttribute(attention_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnTcSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(attention_tc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    dim3 grid((unsigned)((S + kQTile - 1) / kQTile), (unsigned)heads, (unsigned)B);
    return launch_overlapping_tail(attention_tc_kernel, grid, dim3(kThreads), kAttnTcSmemBytes, s, qkv, (int)S,
                                   heads * kHeadDim, ctx, S_q, ctx_q, amax, attention_status_word());
}

}  // namespace q8
