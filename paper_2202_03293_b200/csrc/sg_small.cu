// Tensor-core implicit GEMM for problems that a launch and a few memory latencies bound: many small thread blocks, no
// tensor maps, no tensor memory, no persistent schedule.
//
// The tcgen05 kernel spends about 5 us on the smallest problem: barrier and tensor-memory set-up, tensor maps, a serial chain
// of converting and MMA steps in one or two CTAs, staging and a tensor store.  Here a thread block owns a 32 x 32 output tile
// (16 x 32 while those do not fill the chip), so that even 128 x 128 outputs occupy 32 SMs, and the input of its first 384 k
// (bf16: 640) is in flight at once (cp.async, stages of 128 k); two blocks fit an SM, so a launch behind this one can sit beside
// it and start as it ends.  Each of the eight warps takes 16 of every 128 k of the whole tile; their partial sums meet in shared
// memory, in a fixed order.  Graph replay, us, tcgen05 kernel -> this one: 128^3 f32 6.0 -> 2.1, bf16 3.6 -> 1.7;
// 256^3 f32 6.6 -> 3.4; a 55 x 55 stride-2 3x3x32x64 convolution f32 9.2 -> 7.1.
//
// bf16 inputs: mma.sync m16n8k16, a warp's share of k in one accumulator up to K = 2048 (256 products), beyond that (BF16_LONG) in chunks of 256
// added up with rounding: the gather kernel, which would run some of these calls, holds no more in one either (relative error at K = 4096, positive
// values, 7.1e-7 in one accumulator, 3.1e-7 there; the registers of the second sum cost short reductions a block per SM).  f32 inputs, in one of two forms that keep f32 accuracy:
//   MIX    the split of the tcgen05 kernel: hi = x rounded to tf32, lo = x - hi; hi*hi in tf32, lo*hi + hi*lo in bf16
//   EXACT  x = b0 + b1 + b2 with three bf16 parts of eight bits each (exact differences), six of the nine products
// The tensor core adds by truncation, so the four or six MMAs of 16 k have a sum of their own, which is added, rounding to nearest, to
// the warp's.  (With one accumulator throughout, relative errors of sums of positive values were EXACT 2.5e-6 at K = 4096, where the
// CUDA-core kernel has 8.5e-7, and MIX 3.6e-7 at 512, where the tcgen05 kernel has 1.4e-7.)
#include <algorithm>

#include "sg_internal.cuh"
#include "sg_tc_ptx.cuh"

namespace sg {
namespace {

constexpr int TN = 32, BK = 128;
constexpr int WARPS = BK / 16, THREADS = 32 * WARPS;
constexpr int CHUNK = 16;      // BF16_LONG: stages of which a warp's accumulators, 256 products each, are added to a rounded sum

enum { BF16 = 0, EXACT = 1, MIX = 2, BF16_LONG = 3, BF16_THREE = 4 };
template <int MODE> constexpr bool kF32 = MODE == EXACT || MODE == MIX;

// TM: rows of a tile, 16 or 32.
template <bool F32, bool A_MN, bool B_KM, int TM>
struct Cfg {
    static constexpr int ES = F32 ? 4 : 2, PIECE = 16 / ES;           // bytes per element, elements per 16-byte copy
    // a stage's tiles: lines of 128 k (one per row or column) or lines of the tile's rows or columns (one per k), padded so
    // that the fragment reads below touch every bank once
    static constexpr int K_PITCH = BK * ES + (F32 ? 32 : 16);
    static constexpr int A_PITCH = A_MN ? TM * ES + 16 : K_PITCH, B_PITCH = B_KM ? K_PITCH : TN * ES + 16;
    static constexpr int A_LINES = A_MN ? BK : TM, B_LINES = B_KM ? TN : BK;
    static constexpr int A_BYTES = A_LINES * A_PITCH, STAGE_BYTES = A_BYTES + B_LINES * B_PITCH;
    static constexpr int STAGES = F32 ? 3 : 5;
    static constexpr int RED_PITCH = (TN + 4) * 4, RED_BYTES = WARPS * TM * RED_PITCH;
    static_assert(RED_BYTES <= STAGES * STAGE_BYTES, "the partial sums reuse the ring");
    static_assert(2 * (STAGES * STAGE_BYTES + 1024) <= 233472, "two thread blocks on an SM");
};

// Division by a constant of the launch: n / d for 0 <= n < 2^31 as one multiplication, by a multiplier rounded up (Granlund and Montgomery, Division
// by invariant integers using multiplication, 1994).  With 2^(l-1) < d <= 2^l and
// mul = ceil(2^(31+l) / d), n * mul / 2^(31+l) exceeds n / d by less than n / 2^(31+l) < 1 / d, so the integer part is right.
struct FastDiv {
    uint32_t mul, shift;      // mul 0: d = 1
};
inline FastDiv fast_div(int d) {
    if (d <= 1) return FastDiv{0, 0};
    uint32_t l = 1;
    while (((int64_t)1 << l) < d) ++l;
    return FastDiv{(uint32_t)((((uint64_t)1 << (31 + l)) + (uint32_t)d - 1) / (uint32_t)d), l - 1};
}
__device__ __forceinline__ int divide(int n, FastDiv f) { return f.mul == 0 ? n : (int)(__umulhi((uint32_t)n, f.mul) >> f.shift); }

struct SmallParams {
    Problem p;
    int num_kb, num_n_tiles;
    FastDiv by_hw, by_wo, by_c, by_kw;      // decomposition of m and of k
    int dense_filter;      // filter element k starts at k * k_c
    int uniform_rows;      // output row m starts at m * o_w
    int wait_prior;
};

// 16 bytes global -> shared, asynchronously; zeros where !ok.
__device__ __forceinline__ void copy16(uint32_t dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// D (+)= A * B, 16 x 8 x 8, tf32 inputs.
__device__ __forceinline__ void mma1688(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two f32 values as three words of bf16 pairs, largest part first.
__device__ __forceinline__ void split3(float x, float y, uint32_t &w0, uint32_t &w1, uint32_t &w2) {
    w0 = pack_bf16(x, y);
    const float x1 = x - __uint_as_float(w0 << 16), y1 = y - __uint_as_float(w0 & 0xFFFF0000u);
    w1 = pack_bf16(x1, y1);
    w2 = pack_bf16(x1 - __uint_as_float(w1 << 16), y1 - __uint_as_float(w1 & 0xFFFF0000u));
}
__device__ __forceinline__ float lds(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
// Two values of k (k, k + 1) of one row or column of an f32 tile: neighbours on a line, or the same place on two lines.
template <bool ALONG_K>
__device__ __forceinline__ void load_pair(uint32_t tile, int mn, int k, int pitch, float &x, float &y) {
    if constexpr (ALONG_K) {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "r"(tile + (uint32_t)(mn * pitch + k * 4)) : "memory");
    } else {
        x = lds(tile + (uint32_t)(k * pitch + mn * 4));
        y = lds(tile + (uint32_t)((k + 1) * pitch + mn * 4));
    }
}

// Four columns of row m by multiply-adds on the operands as they stand, until all four are NaN (a NaN stays one).  Out of line: the kernel's loops need the registers.
template <bool CONV>
__device__ __noinline__ float4 sum_as_it_stands(const SmallParams &sp, const float *a, const float *b, int m, int n) {
    const Problem &p = sp.p;
    int64_t row = m * p.i_w;
    if constexpr (CONV) {
        const int i = divide(m, sp.by_hw), r = m - i * (p.Ho * p.Wo), h = divide(r, sp.by_wo), w = r - h * p.Wo;
        row = (int64_t)i * p.i_n + (int64_t)h * p.sh * p.i_h + (int64_t)w * p.sw * p.i_w;
    }
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < p.K && (s[0] == s[0] || s[1] == s[1] || s[2] == s[2] || s[3] == s[3]); k0 += 4)
#pragma unroll
        for (int k = k0; k < k0 + 4; ++k) {
            if (k >= p.K) break;
            int64_t x_off = k * p.i_c, f_off = k * p.k_c;
            if constexpr (CONV) {
                const int tap = divide(k, sp.by_c), c = k - tap * p.C, kh = divide(tap, sp.by_kw), kw = tap - kh * p.KW;
                x_off = (int64_t)kh * p.dh * p.i_h + (int64_t)kw * p.dw * p.i_w + c;
                f_off = kh * p.k_kh + kw * p.k_kw + c * p.k_c;
            }
            const float x = a[row + x_off];
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = fmaf(x, b[f_off + (n + e) * p.k_f], s[e]);
        }
    return make_float4(s[0], s[1], s[2], s[3]);
}

// BF16_THREE: BF16 in the 80 registers that three thread blocks on an SM have.
template <int MODE, bool A_MN, bool B_KM, bool CONV, int TM>
__global__ void __launch_bounds__(THREADS, MODE == BF16_THREE ? 3 : 2)
small_gemm_kernel(const __grid_constant__ SmallParams sp, const char *__restrict__ In, const char *__restrict__ Flt, float *__restrict__ O) {
    constexpr bool F32 = kF32<MODE>;
    using C = Cfg<F32, A_MN, B_KM, TM>;
    const Problem &p = sp.p;
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t ring = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = (int)blockIdx.x / sp.num_n_tiles;
    const int m0 = mt * TM, n0 = ((int)blockIdx.x - mt * sp.num_n_tiles) * TN;
    asm volatile("griddepcontrol.launch_dependents;");

    // ---- what this thread copies of a stage: 16-byte pieces, one fixed place along the lines, every STEP-th line
    constexpr int A_PIECES = (A_MN ? TM : BK) / C::PIECE, B_PIECES = (B_KM ? BK : TN) / C::PIECE;      // per line
    constexpr int A_STEP = THREADS / A_PIECES, B_STEP = THREADS / B_PIECES;                            // lines between a thread's copies
    constexpr int A_COPIES = C::A_LINES / A_STEP, B_COPIES = C::B_LINES / B_STEP;
    static_assert(A_COPIES >= 1 && B_COPIES >= 1 && C::A_LINES % A_STEP == 0 && C::B_LINES % B_STEP == 0, "copies");
    constexpr int MI = TM / 16;
    const int a_piece = tid % A_PIECES * C::PIECE, a_line = tid / A_PIECES;
    const int b_piece = tid % B_PIECES * C::PIECE, b_line = tid / B_PIECES;
    const uint32_t a_dst = ring + (uint32_t)(a_line * C::A_PITCH + a_piece * C::ES);
    const uint32_t b_dst = ring + C::A_BYTES + (uint32_t)(b_line * C::B_PITCH + b_piece * C::ES);
    auto row_offset = [&](int m) -> int64_t {      // element offset of output row m's window in the input
        if constexpr (CONV) {
            const int n = divide(m, sp.by_hw), r = m - n * (p.Ho * p.Wo), h = divide(r, sp.by_wo), w = r - h * p.Wo;
            return (int64_t)n * p.i_n + (int64_t)h * p.sh * p.i_h + (int64_t)w * p.sw * p.i_w;
        } else {
            return m * p.i_w;
        }
    };
    auto k_offset = [&](int k) -> int64_t {        // ... of reduction index k in that window
        if constexpr (CONV) {
            const int tap = divide(k, sp.by_c), c = k - tap * p.C, kh = divide(tap, sp.by_kw), kw = tap - kh * p.KW;
            return (int64_t)kh * p.dh * p.i_h + (int64_t)kw * p.dw * p.i_w + c;
        } else {
            return k * p.i_c;
        }
    };
    auto flt_offset = [&](int k, int n) -> int64_t {
        if (CONV && !sp.dense_filter) {
            const int tap = divide(k, sp.by_c), c = k - tap * p.C, kh = divide(tap, sp.by_kw), kw = tap - kh * p.KW;
            return kh * p.k_kh + kw * p.k_kw + c * p.k_c + n;
        }
        return k * p.k_c + n * p.k_f;
    };
    // Element offsets of this thread's copies: its first line's in the first stage, a uniform step from line to line and from stage to
    // stage; the rows of a convolution lie anywhere, and its k is decomposed.  (With 64-bit products and
    // two divisions for each copy, asking for two stages took a convolution 2200 cycles.)
    int64_t a_off[CONV ? A_COPIES : 1];
    if constexpr (CONV) {
#pragma unroll
        for (int i = 0; i < A_COPIES; ++i) a_off[i] = row_offset(m0 + a_line + i * A_STEP);
    } else {
        a_off[0] = A_MN ? a_line * p.i_c + m0 + a_piece : (m0 + a_line) * p.i_w + a_piece;
    }
    const int64_t b_off = B_KM ? (n0 + b_line) * p.k_f + b_piece : b_line * p.k_c + n0 + b_piece;
    const int64_t a_lines = A_STEP * (A_MN ? p.i_c : p.i_w), b_lines = B_STEP * (B_KM ? p.k_f : p.k_c);
    const int64_t a_stage = A_MN ? BK * p.i_c : BK, b_stage = B_KM ? BK : BK * p.k_c;
    auto fetch = [&](int kb) {
        const uint32_t stage = (uint32_t)(kb % C::STAGES) * C::STAGE_BYTES;
        const int k0 = kb * BK;
        // (a piece never straddles two taps: the channel count is a multiple of it)
        const int64_t a_step = CONV ? k_offset(k0 + a_piece) : kb * a_stage;
#pragma unroll
        for (int i = 0; i < A_COPIES; ++i) {
            const int line = a_line + i * A_STEP;
            const bool ok = (A_MN ? k0 + line : k0 + a_piece) < p.K && (A_MN ? m0 + a_piece : m0 + line) < p.M;
            const int64_t off = CONV ? a_off[CONV ? i : 0] + a_step : a_off[0] + a_step + i * a_lines;
            copy16(a_dst + stage + i * (A_STEP * C::A_PITCH), In + (ok ? off : 0) * C::ES, ok);
        }
        const int64_t b_step = kb * b_stage;
#pragma unroll
        for (int i = 0; i < B_COPIES; ++i) {
            const int line = b_line + i * B_STEP, k = k0 + (B_KM ? b_piece : line);
            const bool ok = k < p.K && n0 + (B_KM ? line : b_piece) < p.N;
            const int64_t off = CONV && !sp.dense_filter ? flt_offset(k, n0 + b_piece) : b_off + b_step + i * b_lines;
            copy16(b_dst + stage + i * (B_STEP * C::B_PITCH), Flt + (ok ? off : 0) * C::ES, ok);
        }
    };
    // the operands may be the output of the kernel ahead of this one
    if (sp.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
    for (int s = 0; s < C::STAGES - 1; ++s) {
        if (s < sp.num_kb) fetch(s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }

    // ---- warp ks: k 16*ks .. of every stage, the whole tile
    const int ks = warp, g = lane >> 2, t = lane & 3;
    float acc[MI][4][4];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    float done[MODE == BF16_LONG ? MI : 1][4][4] = {};      // BF16_LONG: of the finished chunks
    float largest = 0.f;       // EXACT: of the magnitudes seen
    for (int kb = 0; kb < sp.num_kb; ++kb) {
        asm volatile("cp.async.wait_group %0;" ::"n"(C::STAGES - 2) : "memory");
        __syncthreads();       // everyone's copies of this stage have landed; everyone is done with the stage refilled next
        if (kb + C::STAGES - 1 < sp.num_kb) fetch(kb + C::STAGES - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (kb * BK + ks * 16 >= p.K) continue;
        const uint32_t a_tile = ring + (uint32_t)(kb % C::STAGES) * C::STAGE_BYTES, b_tile = a_tile + C::A_BYTES;
        const int k = ks * 16;
        auto pair_a = [&](int i, int e, float &x, float &y) {
            load_pair<!A_MN>(a_tile, i * 16 + g + (e & 1) * 8, k + 2 * t + (e >> 1) * 8, C::A_PITCH, x, y);
            if constexpr (MODE == EXACT) largest = fmaxf(largest, fmaxf(fabsf(x), fabsf(y)));
        };
        auto pair_b = [&](int j, int e, float &x, float &y) {
            load_pair<B_KM>(b_tile, j * 8 + g, k + 2 * t + e * 8, C::B_PITCH, x, y);
            if constexpr (MODE == EXACT) largest = fmaxf(largest, fmaxf(fabsf(x), fabsf(y)));
        };
        auto add_step = [&](const float (&sum)[2][MI][4], int j0) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < MI; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[i][j0 + j][e] += sum[j][i][e];
        };
        if constexpr (MODE == MIX) {
            // corrections lo*hi + hi*lo in bf16, then hi*hi in tf32 (its two steps of 8 k take the even and the odd k of the
            // pairs: any order of k will do that both operands share)
            uint32_t ah[MI][2][4], a16[MI][2][4];
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float x, y;
                    pair_a(i, e, x, y);
                    split_pair_mix(__float_as_uint(x), __float_as_uint(y), ah[i][0][e], ah[i][1][e], a16[i][0][e], a16[i][1][e]);
                }
            // (every step has a sum of its own, rounded to nearest into the running one: see below)
#pragma unroll
            for (int j0 = 0; j0 < 4; j0 += 2) {
                float sum[2][MI][4] = {};
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    uint32_t bh[2][2], b16[2][2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float x, y;
                        pair_b(j0 + j, e, x, y);
                        split_pair_mix(__float_as_uint(x), __float_as_uint(y), bh[0][e], bh[1][e], b16[0][e], b16[1][e]);
                    }
#pragma unroll
                    for (int i = 0; i < MI; ++i) {
                        mma16816(sum[j][i], a16[i][1], b16[0]);
                        mma16816(sum[j][i], a16[i][0], b16[1]);
                        mma1688(sum[j][i], ah[i][0], bh[0][0], bh[0][1]);
                        mma1688(sum[j][i], ah[i][1], bh[1][0], bh[1][1]);
                    }
                }
                add_step(sum, j0);
            }
        } else if constexpr (MODE == EXACT) {
            uint32_t a[MI][3][4];
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float x, y;
                    pair_a(i, e, x, y);
                    split3(x, y, a[i][0][e], a[i][1][e], a[i][2][e]);
                }
            constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};     // smallest products first
#pragma unroll
            for (int j0 = 0; j0 < 4; j0 += 2) {
                uint32_t b[2][3][2];
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float x, y;
                        pair_b(j0 + j, e, x, y);
                        split3(x, y, b[j][0][e], b[j][1][e], b[j][2][e]);
                    }
                float sum[2][MI][4] = {};
#pragma unroll
                for (int q = 0; q < 6; ++q)
#pragma unroll
                    for (int i = 0; i < MI; ++i)
#pragma unroll
                        for (int j = 0; j < 2; ++j) mma16816(sum[j][i], a[i][PA[q]], b[j][PB[q]]);
                add_step(sum, j0);
            }
        } else {
            // matrix loads: lanes 8*i .. 8*i+7 address the rows of block i
            uint32_t a[MI][4], b[2][4];
            const int r = lane & 7, blk = lane >> 3;
#pragma unroll
            for (int i = 0; i < MI; ++i) {
                if constexpr (A_MN) {
                    // lines are k: blocks (k 0-7, m 0-7), (k 0-7, m 8-15), (k 8-15, m 0-7), (k 8-15, m 8-15), transposed
                    const uint32_t addr = a_tile + (uint32_t)((k + (blk >> 1) * 8 + r) * C::A_PITCH + (i * 16 + (blk & 1) * 8) * 2);
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(a[i][0]), "=r"(a[i][1]), "=r"(a[i][2]), "=r"(a[i][3]) : "r"(addr) : "memory");
                } else {
                    const uint32_t addr = a_tile + (uint32_t)((i * 16 + (blk & 1) * 8 + r) * C::A_PITCH + (k + (blk >> 1) * 8) * 2);
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(a[i][0]), "=r"(a[i][1]), "=r"(a[i][2]), "=r"(a[i][3]) : "r"(addr) : "memory");
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {      // columns 16*h .. : blocks (k 0-7, n 0-7), (k 8-15, n 0-7), (k 0-7, n 8-15), (k 8-15, n 8-15)
                if constexpr (B_KM) {
                    const uint32_t addr = b_tile + (uint32_t)((h * 16 + (blk >> 1) * 8 + r) * C::B_PITCH + (k + (blk & 1) * 8) * 2);
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(b[h][0]), "=r"(b[h][1]), "=r"(b[h][2]), "=r"(b[h][3]) : "r"(addr) : "memory");
                } else {
                    const uint32_t addr = b_tile + (uint32_t)((k + (blk & 1) * 8 + r) * C::B_PITCH + (h * 16 + (blk >> 1) * 8) * 2);
                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(b[h][0]), "=r"(b[h][1]), "=r"(b[h][2]), "=r"(b[h][3]) : "r"(addr) : "memory");
                }
            }
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t bj[2] = {b[j >> 1][(j & 1) * 2], b[j >> 1][(j & 1) * 2 + 1]};
                    mma16816(acc[i][j], a[i], bj);
                }
            if constexpr (MODE == BF16_LONG)
                if (kb % CHUNK == CHUNK - 1) {
#pragma unroll
                    for (int i = 0; i < MI; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
#pragma unroll
                            for (int e = 0; e < 4; ++e) { done[i][j][e] += acc[i][j][e]; acc[i][j][e] = 0.f; }
                }
        }
    }

    if constexpr (MODE == BF16_LONG) {
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][j][e] += done[i][j][e];
    }
    // ---- the warps' shares of k meet in shared memory; a thread writes four columns of one row
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const bool overflow = MODE == EXACT ? __syncthreads_or(largest >= 1.7014118e38f) != 0 : false;
    if (MODE != EXACT) __syncthreads();
    float *red = reinterpret_cast<float *>(smem);
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2 *>(red + (ks * TM + i * 16 + g + 8 * h) * (C::RED_PITCH / 4) + j * 8 + 2 * t) =
                    make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
    __syncthreads();
    const int row = tid >> 3, col = (tid & 7) * 4, m = m0 + row, n = n0 + col;
    if (row >= TM || m >= p.M || n >= p.N) return;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < WARPS; ++q) {
        const float4 part = *reinterpret_cast<const float4 *>(red + (q * TM + row) * (C::RED_PITCH / 4) + col);
        v.x += part.x; v.y += part.y; v.z += part.z; v.w += part.w;
    }
    // What the splits do not carry is summed as it stands.  MIX has an infinity as (largest, infinity): against a factor of 2048 and
    // more, whose low part may be above 1/2 and of the other sign, the former's products may be an infinity of the wrong sign, and a factor below
    // 2^-134, whose parts are zero, makes NaN of the latter.  EXACT rounds infinities, and values next to them, to infinite parts, which
    // meet zero parts of the other operand, and either may take finite products that overflow for ones of both signs.  All of that
    // shows in the sums: four that hold an infinity or a NaN.  (EXACT also sums tiles that have seen a value next to overflow, whose products with
    // subnormals it would lose.  A look at the sums costs 55 x 55, stride 2, 3x3x32x64 2 %, one at every operand of MIX 5 %.)
    if (F32 && (overflow || !(fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, v.w * 0.f))) == 0.f))) {
        v = sum_as_it_stands<CONV>(sp, reinterpret_cast<const float *>(In), reinterpret_cast<const float *>(Flt), m, n);
    }
    int64_t off = (int64_t)m * p.o_w;
    if (!sp.uniform_rows) {
        const int b = divide(m, sp.by_hw), r = m - b * (p.Ho * p.Wo), h = divide(r, sp.by_wo), w = r - h * p.Wo;
        off = (int64_t)b * p.o_n + (int64_t)h * p.o_h + (int64_t)w * p.o_w;
    }
    float4 *out = reinterpret_cast<float4 *>(O + off + n);
    if (p.bias != nullptr) {
        const float4 b = __ldg(reinterpret_cast<const float4 *>(p.bias + n));
        v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
    }
    if (p.act == SG_ACT_RELU) {
        v.x = v.x < 0.f ? 0.f : v.x; v.y = v.y < 0.f ? 0.f : v.y; v.z = v.z < 0.f ? 0.f : v.z; v.w = v.w < 0.f ? 0.f : v.w;
    }
    if (p.accumulate) {
        const float4 o = *out;
        v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
    }
    *out = v;
}

inline bool mult(int64_t v, int64_t q) { return v % q == 0; }

template <int MODE, bool A_MN, bool B_KM, bool CONV, int TM>
sg_status launch_variant(SmallParams &sp, const void *In, const void *Flt, float *O, int slot, cudaStream_t stream) {
    using C = Cfg<kF32<MODE>, A_MN, B_KM, TM>;
    constexpr auto kernel = small_gemm_kernel<MODE, A_MN, B_KM, CONV, TM>;
    const int smem = std::max(std::min(C::STAGES, sp.num_kb) * C::STAGE_BYTES, C::RED_BYTES);
    if (!tensor_ensure_smem_attr(slot + (TM == 16 ? 0 : 1), reinterpret_cast<const void *>(kernel), C::STAGES * C::STAGE_BYTES)) return SG_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((sp.p.M + TM - 1) / TM * sp.num_n_tiles, 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = sp.wait_prior ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, sp, static_cast<const char *>(In), static_cast<const char *>(Flt), O);
    count_launch();
    note_kernel(kF32<MODE> ? "small_gemm_kernel<f32>" : "small_gemm_kernel<bf16>");
    return e == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

}  // namespace

sg_status launch_small(const Problem &p, const void *In, const void *Flt, float *O, cudaStream_t stream) {
    // a quick way out for what is far too large
    if ((int64_t)p.M * p.N > (int64_t)1 << 20 || p.K > 4096) return SG_ERR_UNSUPPORTED;
    const int mode = tensor_small_override();
    if (mode == 0) return SG_ERR_UNSUPPORTED;
    // ---- layout: every 16-byte piece of a line (of k, or of rows or columns) is whole and aligned
    const bool f32 = !p.in_bf16, conv = p.spatial_rank != 0;
    const int64_t es = f32 ? 4 : 2, piece = 16 / es;
    const bool a_mn = !conv && p.i_c != 1 && p.i_w == 1, b_km = !conv && p.k_f != 1 && p.k_c == 1;
    if ((p.i_c != 1 && !a_mn) || (p.k_f != 1 && !b_km) || p.o_f != 1) return SG_ERR_UNSUPPORTED;
    auto on16 = [](const void *ptr) { return reinterpret_cast<uintptr_t>(ptr) % 16 == 0; };
    if (!on16(In) || !on16(Flt) || !on16(O) || (p.bias != nullptr && (!on16(p.bias) || p.bias_f != 1))) return SG_ERR_UNSUPPORTED;
    if (!mult(a_mn ? p.i_c : p.i_w, piece) || !mult(b_km ? p.k_f : p.k_c, piece)) return SG_ERR_UNSUPPORTED;
    if (!mult(a_mn ? p.M : p.C, piece) || !mult(b_km ? p.K : p.N, piece) || !mult(p.N, 4)) return SG_ERR_UNSUPPORTED;
    if (!mult(p.o_w, 4) || (p.Ho > 1 && !mult(p.o_h, 4)) || (p.batch > 1 && !mult(p.o_n, 4))) return SG_ERR_UNSUPPORTED;
    if (conv && ((p.Ho > 1 || p.KH > 1) && !mult(p.i_h, piece))) return SG_ERR_UNSUPPORTED;
    if (conv && ((p.batch > 1 && !mult(p.i_n, piece)) || (p.KW > 1 && !mult(p.k_kw, piece)) || (p.KH > 1 && !mult(p.k_kh, piece)))) return SG_ERR_UNSUPPORTED;

    int dev = 0, num_sms = 0, pdl = -1, unused = 0;
    if (!tensor_device_info(&dev, &num_sms, &pdl, &unused)) return SG_ERR_CUDA;
    SmallParams sp{};
    sp.p = p;
    sp.num_kb = (p.K + BK - 1) / BK;
    sp.num_n_tiles = (p.N + TN - 1) / TN;
    sp.by_hw = fast_div(p.Ho * p.Wo); sp.by_wo = fast_div(p.Wo); sp.by_c = fast_div(p.C); sp.by_kw = fast_div(p.KW);
    const int64_t tiles = (int64_t)((p.M + 31) / 32) * sp.num_n_tiles;      // of 32 x 32
    sp.dense_filter = (p.KW == 1 || p.k_kw == p.C * p.k_c) && (p.KH == 1 || p.k_kh == (int64_t)p.KW * p.C * p.k_c);
    sp.uniform_rows = (p.Ho == 1 || p.o_h == (int64_t)p.Wo * p.o_w) && (p.batch == 1 || p.o_n == (int64_t)p.Ho * p.Wo * p.o_w);
    sp.wait_prior = pdl == 0 ? 0 : 1;
    const int64_t in_bytes = (int64_t)p.batch * ((int64_t)(p.Ho - 1) * p.sh + (int64_t)(p.KH - 1) * p.dh + 1) *
                             ((int64_t)(p.Wo - 1) * p.sw + (int64_t)(p.KW - 1) * p.dw + 1) * p.C * es;
    // 16 rows a tile while the 32-row tiles do not fill the chip: twice the thread blocks, half the work of each (128^3 f32
    // 2.48 -> 2.08 us, 128 x 1024 x 256 4.7 -> 3.6; but with 190 tiles 5.8 -> 6.6)
    const bool half = tiles <= num_sms;
    // f32 operands take the split of the tcgen05 kernel where that kernel would use it; whatever it runs as three tf32 products or
    // leaves to the CUDA cores (convolutions of inputs below 128 KiB, outputs that are not one matrix) keeps the accuracy it had there.
    // (Products in the plain layout with overlapping rows have no such form here; the gather kernel has.)
    const bool mix = f32 && !a_mn && !b_km && tensor_takes(p, In, Flt, O);
    if (f32 && !conv && !a_mn && !b_km && !mix) return SG_ERR_UNSUPPORTED;
    if (mode < 0) {
        // By time (us): a launch; where 16-row tiles do, what they take the more of the more of them there are to an SM, and steps of 128 k;
        // else waves of 32-row tiles over the SMs, each a start and its steps.  Fitted to graph replays of 730 calls of every layout and
        // op: within 10 % of the timings, 7 % for MIX.
        const double steps = std::max(0.5, (double)p.K / BK), waves = (double)((tiles + num_sms - 1) / num_sms);
        const double fill = std::min(2.0, (double)((p.M + 15) / 16) * sp.num_n_tiles / num_sms);      // 16-row tiles per SM
        struct Cost { double start, fill, step, step_fill, wave, wave_step; };
        constexpr Cost costs[3] = {{1.35, 0.69, 0.38, 0.28, 0.65, 0.33}, {1.56, 0.44, 0.95, 0.42, 0.79, 0.98}, {1.45, 0.54, 0.73, 0.37, 0.66, 0.76}};
        const Cost &c = costs[!f32 ? BF16 : mix ? MIX : EXACT];
        const double us = half ? c.start + c.fill * fill + steps * (c.step + c.step_fill * std::max(0.0, fill - 0.5))
                               : c.start + waves * (c.wave + c.wave_step * steps);
        // The other side is what would run the call instead.  That never takes less than 2.8 us, f32 3.6 (into outputs that are not one
        // matrix 4.2), unit-stride convolutions of bf16 4.0: no need to ask.  Where it is the tcgen05 kernel, or a convolution whose filter
        // stays or streams past the runs of input rows, the former's cost model says what it takes; those convolutions are the faster ones in bf16.  What
        // none of them takes (inputs stored transposed whose rows are no whole 128 bytes of m, strided convolutions into outputs that are not one matrix)
        // the gather kernel would run, by its own model.  Of 744 calls timed both ways the choices cost 0.5 % over the better of the two
        // in the mean; three times the tcgen05 kernel's estimate, in the gather kernel's place and where a filter
        // stays, cost 4.8 % (27 x 24 x 24, 1x1x48x64 f32 into a padded output 5.9 us as strips, 11.7 here; 1 x 77 x 77, 3x3x64x128 bf16
        // 4.9 and 13.5; 1048 x 32 x 3352 f32 transposed 14.2 gathered, 33.1 here).
        const bool takes = tensor_takes(p, In, Flt, O), unit = conv && p.sh == 1 && p.sw == 1, run_conv = unit && !f32;
        if (us > (f32 ? takes ? 3.6 : 4.2 : run_conv ? 4.0 : 2.8)) {
            const double short_input = conv && in_bytes < 131072 ? 0.3 * p.K : 0.0;      // (inputs below 128 KiB, which no model covers)
            if (takes || (unit && launch_conv_strip(p, In, Flt, O, true, stream) == SG_OK)) {
                const double lead = run_conv ? 0.8 : !f32 ? 1.15 : mix ? 1.0 : 1.1;
                if (us > (short_input > 0.0 ? short_input : lead * tensor_estimate_us(p))) return SG_ERR_UNSUPPORTED;
            } else if (us > std::max(short_input, 0.95 * gather_estimate_us(p, num_sms))) {
                return SG_ERR_UNSUPPORTED;
            }
        }
    }
    tensor_note_choice(TN, 1, 1);
#define SG_SMALL(MODE_, A_MN_, B_KM_, CONV_, SLOT)                                                                  \
    (half ? launch_variant<MODE_, A_MN_, B_KM_, CONV_, 16>(sp, In, Flt, O, SLOT, stream)                            \
          : launch_variant<MODE_, A_MN_, B_KM_, CONV_, 32>(sp, In, Flt, O, SLOT, stream))
    // bf16: three thread blocks to an SM where shared memory has room for them (three stages) and there are more than two to each (368 tiles, 2 x 727, 3x32x256,
    // 4.3 us with two and 3.6 with three); with fewer, blocks behind an overlapped launch would be dealt out three to one (232 tiles, K = 288, 4.1 and 5.2), and
    // longer reductions are the slower for the fewer registers (930 tiles, K = 1280, 28.3 and 29.3)
    const bool chunks = sp.num_kb > CHUNK, three = sp.num_kb <= 3 && tiles > 2 * (int64_t)num_sms;
#define SG_SMALL_BF16(A_MN_, B_KM_, CONV_, SLOT, SLOT_LONG)                                                         \
    (chunks  ? SG_SMALL(BF16_LONG, A_MN_, B_KM_, CONV_, SLOT_LONG)                                                  \
     : three ? launch_variant<BF16_THREE, A_MN_, B_KM_, CONV_, 32>(sp, In, Flt, O, SLOT_LONG + 13, stream)          \
             : SG_SMALL(BF16, A_MN_, B_KM_, CONV_, SLOT))
    if (conv) return !f32 ? SG_SMALL_BF16(false, false, true, 160, 212) : mix ? SG_SMALL(MIX, false, false, true, 162) : SG_SMALL(EXACT, false, false, true, 164);
    if (mix) return SG_SMALL(MIX, false, false, false, 166);
    if (a_mn && b_km) return f32 ? SG_SMALL(EXACT, true, true, false, 168) : SG_SMALL_BF16(true, true, false, 170, 214);
    if (a_mn) return f32 ? SG_SMALL(EXACT, true, false, false, 172) : SG_SMALL_BF16(true, false, false, 174, 216);
    if (b_km) return f32 ? SG_SMALL(EXACT, false, true, false, 176) : SG_SMALL_BF16(false, true, false, 178, 218);
    return SG_SMALL_BF16(false, false, false, 180, 220);
#undef SG_SMALL_BF16
#undef SG_SMALL
}

}  // namespace sg
