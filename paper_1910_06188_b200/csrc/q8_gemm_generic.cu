// Generic Int8 GEMM + epilogue: any M, N, K and any alignment.
//
// q8_linear falls back to this kernel when the tensor-core kernel's TMA preconditions do not hold (K not a multiple of
// 16 bytes, operands not 16-byte aligned).  It computes exactly the same integers (Sec. 3: Int8 products accumulated in Int32
// onto the Int32 bias) and applies the same epilogue arithmetic, so it also serves as an on-device cross-check of the fast
// kernel.
//
// Operand rows that start anywhere cannot be fetched by TMA, and tcgen05 reads nothing but shared memory in TMA's layout, so
// the tiles are staged by all threads (cp.async in pieces of 8 or 4 bytes where K and the pointers allow it, otherwise
// 4-byte words shifted into place) and multiplied by mma.sync m16n8k32.s8 from rows of 64 bytes, 80 apart (ldmatrix without
// bank conflicts).  1000 x 300 -> 1200 with GELU 7.6 us (39.4 with byte loads and dp4a), 128 x 1000 -> 768 6.2 (103),
// 2000 x 1004 -> 2000 21 (330; 382 TOPS), 4000 x 1001 -> 2000 140 (558).  Bound by the loads: instructions per piece
// (with per-piece index arithmetic 3 us more on the first shape) and, for rows that start at any byte, two words per piece; and, in
// grids of one wave, by fetching the instructions themselves (PLAIN below).

#include "q8_internal.cuh"

namespace q8 {

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kStepK = 64;   // bytes of K per stage
constexpr int kPitch = 80;   // row pitch in shared memory

template <int TILE>
struct Shape {  // TILE x TILE outputs per CTA: 64 (warps 4 x 2, 16 x 32 each) or 128 (warps 2 x 4, 64 x 32 each)
    static constexpr int kWarpsM = TILE == 64 ? 4 : 2, kWarpsN = kWarps / kWarpsM;
    static constexpr int kMT = TILE / kWarpsM / 16, kNT = TILE / kWarpsN / 8;  // MMA tiles per warp
    static constexpr int kStages = 3;
    static constexpr int kStageBytes = 2 * TILE * kPitch;
    static constexpr int kSmemBytes = kStages * kStageBytes;
};

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t at)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(at) : "memory");
}
__device__ __forceinline__ void mma_s8(int32_t (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A call, not a copy for each of a thread's outputs: the epilogue runs once, so its instructions are all fetched for the first time.
// (Four at a time, so that their chains overlap.)
__device__ __noinline__ float4 gelu_of(float4 y) { return make_float4(gelu_erf(y.x), gelu_erf(y.y), gelu_erf(y.z), gelu_erf(y.w)); }

// PIECE: bytes per cp.async (8 or 4: K and both pointers are multiples of it), or 1: rows start at any byte.
// PLAIN: one weight scale and nothing but the fp32 output; the other outputs are compiled out, whose skipped instructions are fetched
// like the rest.  (Warps spent 40 % of 1000 x 300 -> 1200 waiting for instructions.  Without / with GELU, us: 8.0 / 9.9 -> 6.4 / 7.6, 128 x
// 300 -> 768 5.1 / 6.0 -> 3.3 / 3.9, 2000 x 1004 -> 2000 30.9 / 32.1 -> 20.7 / 24.2, 3000 x 700 -> 3000 51.8 / 52.5 -> 30.6 / 36.7, 40000 x 100 -> 4 8.2 /
// 11.2 -> 4.6 / 5.3.)
template <int TILE, int PIECE, bool PLAIN>
__global__ void __launch_bounds__(kThreads, TILE == 128 ? 2 : PIECE == 1 ? 4 : 3) gemm_generic_kernel(GemmArgs a)
{
    using C = Shape<TILE>;
    constexpr int kStages = C::kStages;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t smem = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t m0 = (int64_t)blockIdx.x * TILE, n0 = (int64_t)blockIdx.y * TILE;
    const int steps = (int)((a.K + kStepK - 1) / kStepK);
    grid_dependency_release_next(gridDim.x * gridDim.y <= 600u);
    grid_dependency_wait();

    // A stage holds TILE rows of X_q, then TILE rows of W_q; outside the matrices it is filled with zeros.  A thread brings in
    // the same piece of every kRowsPerPass-th row, so that only two pointers move and one bound on K is checked per stage.
    constexpr int kPieceBytes = PIECE == 1 ? 4 : PIECE;
    constexpr int kPerRow = kStepK / kPieceBytes, kRowsPerPass = kThreads / kPerRow, kPasses = TILE / kRowsPerPass;
    const int row0 = tid / kPerRow, k_at = (tid % kPerRow) * kPieceBytes;
    const int8_t *px = a.Xq + (m0 + row0) * a.K + k_at, *pw = a.Wq + (n0 + row0) * a.K + k_at;
    const int64_t row_step = kRowsPerPass * a.K;
    const uint32_t place0 = smem + (uint32_t)(row0 * kPitch + k_at);
    const int x_rows = (int)min((int64_t)TILE, a.M - m0), w_rows = (int)min((int64_t)TILE, a.N - n0);
    uint32_t word[PIECE == 1 ? 2 * kPasses : 1];
    auto fetch_one = [&](const int8_t *src, bool in, int valid, uint32_t at, int i) {
        if (PIECE == 8) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(at), "l"(in ? src : a.Xq), "r"(in ? 8 : 0) : "memory");
        } else if (PIECE == 4) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(at), "l"(in ? src : a.Xq), "r"(in ? 4 : 0) : "memory");
        } else {  // into registers; put() stores them
            uint32_t w = 0;
            if (in) {
                // the aligned words that hold bytes src .. src + valid - 1 (a word is only read if one of its bytes is ours)
                const int shift = (int)(reinterpret_cast<uintptr_t>(src) & 3u);
                const uint32_t *words = reinterpret_cast<const uint32_t *>(src - shift);
                const uint32_t lo = __ldg(words), hi = shift + valid > 4 ? __ldg(words + 1) : 0u;
                w = __funnelshift_r(lo, hi, 8 * shift);
                if (valid < 4) w &= (1u << (8 * valid)) - 1u;
            }
            word[i] = w;
        }
    };
    int fetched = 0;  // stages fetched so far: the next one starts at byte fetched * kStepK of K
    auto fetch = [&](int stage) {
        const int64_t k = (int64_t)fetched * kStepK + k_at;
        const int valid = (int)min((int64_t)4, a.K - k);
        const uint32_t at = place0 + (uint32_t)(stage * C::kStageBytes);
#pragma unroll
        for (int i = 0; i < kPasses; ++i)
            fetch_one(px + i * row_step, valid > 0 && row0 + i * kRowsPerPass < x_rows, valid, at + i * kRowsPerPass * kPitch, i);
#pragma unroll
        for (int i = 0; i < kPasses; ++i)
            fetch_one(pw + i * row_step, valid > 0 && row0 + i * kRowsPerPass < w_rows, valid,
                      at + (TILE + i * kRowsPerPass) * kPitch, kPasses + i);
        px += kStepK;
        pw += kStepK;
        ++fetched;
    };
    auto put = [&](int stage) {
        if (PIECE == 1) {
#pragma unroll
            for (int i = 0; i < 2 * kPasses; ++i)
                asm volatile("st.shared.b32 [%0], %1;"
                             ::"r"(place0 + (uint32_t)(stage * C::kStageBytes + ((i / kPasses) * TILE + (i % kPasses) * kRowsPerPass) * kPitch)),
                             "r"(word[i])
                             : "memory");
        }
    };

    const int wm = (warp / C::kWarpsN) * (16 * C::kMT), wn = (warp % C::kWarpsN) * (8 * C::kNT);
    int32_t acc[C::kMT][C::kNT][4] = {};
    // what the epilogue needs travels under the main loop
    auto col = [&](int j, int c) { return n0 + wn + 8 * j + 2 * (lane & 3) + c; };
    const float S_x = __ldg(a.S_x), S_w = __ldg(a.S_w), S_y = !PLAIN && a.Yq ? __ldg(a.S_y) : 1.0f;
    float bias[C::kNT][2];
#pragma unroll
    for (int j = 0; j < C::kNT; ++j)
#pragma unroll
        for (int c = 0; c < 2; ++c) bias[j][c] = a.bias && col(j, c) < a.N ? __ldg(a.bias + col(j, c)) : 0.0f;
    const bool pairs = a.Y != nullptr && a.N % 2 == 0 && (reinterpret_cast<uintptr_t>(a.Y) & 7u) == 0;
    // ldmatrix row addresses: A rows 0-7, 8-15 (first 16 bytes of K), 0-7, 8-15 (next 16); B rows of two 8-column tiles likewise
    const uint32_t a_at = (uint32_t)((wm + (lane & 15)) * kPitch + (lane >> 4) * 16);
    const uint32_t b_at = (uint32_t)((TILE + wn + (lane & 7) + (lane >> 4) * 8) * kPitch + ((lane >> 3) & 1) * 16);
    auto multiply = [&](int stage) {
        const uint32_t s = smem + (uint32_t)(stage * C::kStageBytes);
#pragma unroll
        for (int kk = 0; kk < kStepK / 32; ++kk) {
            uint32_t af[C::kMT][4], bf[C::kNT / 2][4];
#pragma unroll
            for (int i = 0; i < C::kMT; ++i) ldmatrix_x4(af[i], s + a_at + (uint32_t)(i * 16 * kPitch + 32 * kk));
#pragma unroll
            for (int j = 0; j < C::kNT / 2; ++j) ldmatrix_x4(bf[j], s + b_at + (uint32_t)(j * 16 * kPitch + 32 * kk));
#pragma unroll
            for (int i = 0; i < C::kMT; ++i)
#pragma unroll
                for (int j = 0; j < C::kNT; ++j) mma_s8(acc[i][j], af[i], bf[j / 2][2 * (j & 1)], bf[j / 2][2 * (j & 1) + 1]);
        }
    };

    if (PIECE == 1) {
        fetch(0);
        for (int t = 0; t < steps; ++t) {  // the words of step t + 1 travel while step t is multiplied
            put(t & 1);
            __syncthreads();
            if (t + 1 < steps) fetch(0);
            multiply(t & 1);
        }
    } else {
#pragma unroll
        for (int t = 0; t < kStages - 1; ++t) {
            if (t < steps) fetch(t);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        int stage = 0;
        for (int t = 0; t < steps; ++t) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
            __syncthreads();  // step t is in place for everybody, and everybody has left the stage that is filled next
            if (t + kStages - 1 < steps) fetch(stage == 0 ? kStages - 1 : stage - 1);
            asm volatile("cp.async.commit_group;" ::: "memory");
            multiply(stage);
            stage = stage + 1 == kStages ? 0 : stage + 1;
        }
    }

    if (PLAIN) {
        const float S_out = __fmul_rn(S_x, S_w), inv = __fdiv_rn(1.0f, S_out);
#pragma unroll
        for (int j = 0; j < C::kNT; ++j) {
            const int32_t b0 = a.bias ? quantize_bias(bias[j][0], S_out) : 0, b1 = a.bias ? quantize_bias(bias[j][1], S_out) : 0;
            const int64_t n = col(j, 0);
            if (n >= a.N) continue;
            float *y = a.Y + (m0 + wm + (lane >> 2)) * a.N + n;
#pragma unroll
            for (int i = 0; i < C::kMT; ++i) {
                const int m = wm + 16 * i + (lane >> 2);
                if (m >= x_rows) continue;
                auto value = [&](int e, int32_t b_q) { return __fmul_rn(__int2float_rn(add_wrap(acc[i][j][e], b_q)), inv); };
                float4 v = make_float4(value(0, b0), value(1, b1), value(2, b0), value(3, b1));  // rows m and m + 8
                if (a.act == Q8_ACT_GELU) v = gelu_of(v);
                float *to = y + 16 * i * a.N, *to8 = to + 8 * a.N;
                const bool second = m + 8 < x_rows;
                if (pairs) {
                    *reinterpret_cast<float2 *>(to) = make_float2(v.x, v.y);
                    if (second) *reinterpret_cast<float2 *>(to8) = make_float2(v.z, v.w);
                } else {
                    to[0] = v.x;
                    if (n + 1 < a.N) to[1] = v.y;
                    if (second) to8[0] = v.z;
                    if (second && n + 1 < a.N) to8[1] = v.w;
                }
            }
        }
        return;
    }
    float am = 0.0f;
#pragma unroll
    for (int j = 0; j < C::kNT; ++j) {
        float inv[2];
        int32_t bq[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float S_out = __fmul_rn(S_x, a.w_seg > 0 && col(j, c) < a.N ? __ldg(a.S_w + col(j, c) / a.w_seg) : S_w);
            inv[c] = __fdiv_rn(1.0f, S_out);
            bq[c] = a.bias ? quantize_bias(bias[j][c], S_out) : 0;
        }
        const int64_t n = col(j, 0);
#pragma unroll
        for (int i = 0; i < 2 * C::kMT; ++i) {
            const int64_t m = m0 + wm + 16 * (i >> 1) + 8 * (i & 1) + (lane >> 2);
            if (m >= a.M) continue;
            float y[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int32_t v = add_wrap(acc[i >> 1][j][2 * (i & 1) + c], bq[c]);
                y[c] = finish_output(v, inv[c], a.act);
                if (n + c >= a.N) continue;
                if (a.dbg_acc) a.dbg_acc[m * a.N + n + c] = v;
                am = fmaxf(am, fabsf(y[c]));
                if (a.Y && !pairs) a.Y[m * a.N + n + c] = y[c];
                if (a.Yq) a.Yq[m * a.N + n + c] = (int8_t)quantize_value(y[c], S_y);
            }
            if (pairs && n < a.N) *reinterpret_cast<float2 *>(a.Y + m * a.N + n) = make_float2(y[0], y[1]);
        }
    }
    if (a.y_absmax) warp_fold_absmax(am, a.y_absmax);
}

template <int TILE, int PIECE, bool PLAIN>
cudaError_t launch_form(const GemmArgs &a, cudaStream_t s)
{
    using C = Shape<TILE>;
    static bool attr_set[64] = {};  // opt-in shared-memory size: per device, per function
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(gemm_generic_kernel<TILE, PIECE, PLAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    dim3 grid((unsigned)((a.M + TILE - 1) / TILE), (unsigned)((a.N + TILE - 1) / TILE));
    if (grid.y > 65535u) return cudaErrorInvalidConfiguration;
    e = launch_overlapping_tail(gemm_generic_kernel<TILE, PIECE, PLAIN>, grid, dim3(kThreads), C::kSmemBytes, s, a);
    LaunchInfo &li = last_launch_info();
    li.gemm_kernel = 2;
    li.block_n = TILE;
    li.grid = (int)(grid.x * grid.y);
    li.launches += 1;
    return e;
}

template <int TILE, int PIECE>
cudaError_t launch_shape(const GemmArgs &a, cudaStream_t s)
{
    const bool plain = a.Yq == nullptr && a.dbg_acc == nullptr && a.y_absmax == nullptr && a.w_seg <= 0;
    return plain ? launch_form<TILE, PIECE, true>(a, s) : launch_form<TILE, PIECE, false>(a, s);
}

}  // namespace

cudaError_t launch_gemm_generic(const GemmArgs &a, cudaStream_t s)
{
    const uintptr_t any = reinterpret_cast<uintptr_t>(a.Xq) | reinterpret_cast<uintptr_t>(a.Wq) | (uintptr_t)a.K;
    // the large tile once its grid fills the device (2000 x 1004 -> 2000, 256 tiles: 35 against 46 us with the small one,
    // 1500 x 1004 -> 1500, 144 tiles: 32 / 31 us, both before a common gain; rows that start at any byte, whose loads go through registers, never gain:
    // 4000 x 1001 -> 2000 270 / 163 us), and where 64-wide tiles would be too many for a grid
    // Not for N <= 128, one column of large tiles, where its few wide CTAs leave the loads of X_q waiting: 40000 x 100 -> 4 34.0 us, 9.4 with
    // the small tile, -> 128 35.1 / 15.1, 125829 x 1004 -> 100 140 / 123 (but -> 65 111 / 125).
    const int64_t big_tiles = ((a.M + 127) / 128) * ((a.N + 127) / 128);
    if ((a.N > 128 && big_tiles >= sm_count() && any % 4 == 0) || a.N > 64 * 65535ll) {
        if (any % 8 == 0) return launch_shape<128, 8>(a, s);
        return any % 4 == 0 ? launch_shape<128, 4>(a, s) : launch_shape<128, 1>(a, s);
    }
    if (any % 8 == 0) return launch_shape<64, 8>(a, s);
    return any % 4 == 0 ? launch_shape<64, 4>(a, s) : launch_shape<64, 1>(a, s);
}

}  // namespace q8
