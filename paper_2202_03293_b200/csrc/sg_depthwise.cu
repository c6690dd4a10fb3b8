// Depthwise convolutions (Section 4.6.3): O[n,h,w,c] (+)= sum_{kh,kw} I[n, h*Sh+kh*Dh, w*Sw+kw*Dw, c] * K[kh,kw,c].
//
// The channel iterator is parallel, only the window is reduced: KH*KW multiply-adds per output
// element against at least one element read and one written, so the op is bound by HBM
// bandwidth and runs on the CUDA cores.  The kernel for small layers gives each thread four consecutive
// channels (one access of 8 or 16 bytes; consecutive threads take consecutive channel groups, so a warp
// reads and writes whole lines) of a few consecutive output columns; for the 3 x 3 window with stride 1 or 2 and
// unit dilation along w the input columns that their windows share are loaded once into
// registers, otherwise every tap is loaded where it is needed and the L1 serves the repeats.
// 3 x 3 and 5 x 5 windows take a TMA-staged tile kernel (layouts that meet the TMA rules); large 3 x 3 /
// unit-stride problems in other layouts a kernel that walks down the rows with a rolling register window.  Any other layout (channel
// strides other than 1, channel counts that are not a multiple of 4, unaligned pointers or
// pitches) takes a one-output-per-thread kernel with full stride arithmetic.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sg_internal.cuh"
#include "sg_tc_ptx.cuh"

namespace sg {
namespace {

constexpr int TW_UNIT = 4, TW_STRIDED = 2;      // output columns per thread of depthwise_vec_kernel (the latter: 3 x 3 windows of stride 2)

// Four neighbouring channels as they lie in memory, and as f32 (bf16 -> f32 is a 16-bit shift: exact).
template <typename T> struct Raw4Of { typedef float4 type; };
template <> struct Raw4Of<__nv_bfloat16> { typedef uint2 type; };
template <typename T> using Raw4 = typename Raw4Of<T>::type;
__device__ __forceinline__ float4 load_raw4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ uint2 load_raw4(const __nv_bfloat16 *p) { return *reinterpret_cast<const uint2 *>(p); }
__device__ __forceinline__ float4 widen4(float4 v) { return v; }
__device__ __forceinline__ float4 widen4(uint2 raw) {
    return make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xFFFF0000u),
                       __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xFFFF0000u));
}
template <typename T>
__device__ __forceinline__ float4 load4(const T *p) { return widen4(load_raw4(p)); }
__device__ __forceinline__ float load1(const float *p) { return *p; }
__device__ __forceinline__ float load1(const __nv_bfloat16 *p) { return __bfloat162float(*p); }

__device__ __forceinline__ void fma4(float4 &acc, const float4 a, const float4 b) {
    acc.x = fmaf(a.x, b.x, acc.x); acc.y = fmaf(a.y, b.y, acc.y);
    acc.z = fmaf(a.z, b.z, acc.z); acc.w = fmaf(a.w, b.w, acc.w);
}

// Four channels of a few output columns per thread.  S = 1, 2: a 3 x 3 window of stride S and unit dilation along w, known at compile
// time: the columns that neighbouring windows of a filter row share are loaded once, and all of a thread's input loads (S = 1: 18
// for four columns, S = 2: 15 for two) are issued before the first of them is needed; so are the 9 filter loads of S = 2.  These are
// calls of a few microseconds: one memory latency is the most they can afford (with each tap loaded where it is needed a
// stride-2 layer of 4 x 7 x 7 x 16 took nine, 9.3 us; now 1.8).  S = 1 loads its filter where it is used, the L1 serves it: with all 27
// loads ahead (AHEAD) f32 is short of registers (3 x 50 x 50 x 36 3.41 us, without 2.48).  Columns wait as they lie in memory and are widened once a row
// (bf16 widened for every use: 4 x 14 x 14 x 200 2.46 us, now 2.31).  S = 0: any window, every tap loaded where it is needed; the L1 serves
// the repeats.  IDX: the type the work index is decoded in (32-bit whenever the work fits: 64-bit divisions
// would cost more than the op).  One work item per thread.  (The operands are no __restrict__ pointers: the kernel ahead may still
// write them when this one starts, and a load that the compiler takes for one of constant data could go ahead of the wait.)
template <typename T, int S, typename IDX, bool AHEAD = false>
__global__ void __launch_bounds__(256)
depthwise_vec_kernel(const DepthwiseProblem p, const T *I, const T *Kf, float *O) {
    constexpr int TW = S == 2 ? TW_STRIDED : TW_UNIT;
    asm volatile("griddepcontrol.launch_dependents;");
    const IDX c4s = (IDX)(p.C / 4);
    const IDX wts = (IDX)((p.Wo + TW - 1) / TW);
    const IDX total = (IDX)p.N * (IDX)p.Ho * wts * c4s;
    const IDX idx = (IDX)blockIdx.x * 256 + threadIdx.x;
    if (idx < total) {
        const int c = (int)(idx % c4s) * 4;
        IDX r = idx / c4s;
        const int w0 = (int)(r % wts) * TW;
        r /= wts;
        const int h = (int)(r % (IDX)p.Ho), n = (int)(r / (IDX)p.Ho);
        float4 acc[TW];
#pragma unroll
        for (int t = 0; t < TW; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        const T *in_n = I + (int64_t)n * p.i_n + c;
        // the operands may be the output of the kernel ahead of this one, and the output its input
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if constexpr (S == 1) {
            Raw4<T> col[3][TW + 2], flt[3][3];
            auto load_filter = [&](int kh, int kw) { return load_raw4(Kf + (int64_t)kh * p.k_kh + (int64_t)kw * p.k_kw + c); };
#pragma unroll
            for (int kh = 0; kh < 3; ++kh) {
                const T *row = in_n + (int64_t)(h * p.sh + kh * p.dh) * p.i_h + (int64_t)w0 * p.i_w;
#pragma unroll
                for (int j = 0; j < TW + 2; ++j)
                    if (w0 + j < p.Wo + 2) col[kh][j] = load_raw4(row + (int64_t)j * p.i_w);
            }
            if constexpr (AHEAD)
#pragma unroll
                for (int kh = 0; kh < 3; ++kh)
#pragma unroll
                    for (int kw = 0; kw < 3; ++kw) flt[kh][kw] = load_filter(kh, kw);
#pragma unroll
            for (int kh = 0; kh < 3; ++kh) {
                float4 wide[TW + 2];
#pragma unroll
                for (int j = 0; j < TW + 2; ++j) wide[j] = widen4(col[kh][j]);
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) {
                    const float4 f = widen4(AHEAD ? flt[kh][kw] : load_filter(kh, kw));
#pragma unroll
                    for (int t = 0; t < TW; ++t)
                        if (w0 + t < p.Wo) fma4(acc[t], wide[t + kw], f);
                }
            }
        } else if constexpr (S == 2) {
            constexpr int COLS = (TW - 1) * S + 3;
            Raw4<T> col[3][COLS], flt[3][3];
#pragma unroll
            for (int kh = 0; kh < 3; ++kh) {
                const T *row = in_n + (int64_t)(h * p.sh + kh * p.dh) * p.i_h + (int64_t)w0 * S * p.i_w;
#pragma unroll
                for (int j = 0; j < COLS; ++j)
                    if (w0 * S + j < (p.Wo - 1) * S + 3) col[kh][j] = load_raw4(row + (int64_t)j * p.i_w);
            }
#pragma unroll
            for (int kh = 0; kh < 3; ++kh)
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) flt[kh][kw] = load_raw4(Kf + (int64_t)kh * p.k_kh + (int64_t)kw * p.k_kw + c);
#pragma unroll
            for (int kh = 0; kh < 3; ++kh)
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) {
                    const float4 f = widen4(flt[kh][kw]);
#pragma unroll
                    for (int t = 0; t < TW; ++t)
                        if (w0 + t < p.Wo) fma4(acc[t], widen4(col[kh][t * S + kw]), f);
                }
        } else {
            for (int kh = 0; kh < p.KH; ++kh) {
                const T *row = in_n + (int64_t)(h * p.sh + kh * p.dh) * p.i_h;
                const T *frow = Kf + (int64_t)kh * p.k_kh + c;
                for (int kw = 0; kw < p.KW; ++kw) {
                    const float4 f = load4(frow + (int64_t)kw * p.k_kw);
#pragma unroll
                    for (int t = 0; t < TW; ++t)
                        if (w0 + t < p.Wo) fma4(acc[t], load4(row + (int64_t)((w0 + t) * p.sw + kw * p.dw) * p.i_w), f);
                }
            }
        }
        float *out = O + (int64_t)n * p.o_n + (int64_t)h * p.o_h + c;
#pragma unroll
        for (int t = 0; t < TW; ++t) {
            if (w0 + t >= p.Wo) break;
            float4 *o = reinterpret_cast<float4 *>(out + (int64_t)(w0 + t) * p.o_w);
            float4 v = acc[t];
            if (p.accumulate) {
                const float4 old = *o;
                v.x += old.x; v.y += old.y; v.z += old.z; v.w += old.w;
            }
            *o = v;
        }
    }
}

// 3 x 3 window, unit stride and dilation along w and h, large problems: a thread owns four channels of TW output
// columns and walks down ROLL_ROWS output rows, keeping the three input rows of the window in registers.  Each step loads
// ONE new input row (TW+2 sixteen-byte loads) instead of three, so an input element is fetched 1.5 (columns) x
// (ROLL_ROWS+2)/ROLL_ROWS (rows) times from L1/L2 instead of 4.5 times; the six multiply-adds per output that use the two
// rows already held run while the new row is in flight.  The row buffers rotate by role (compile-time indices), not by copy.
#ifndef SG_DW_ROLL_TW
#define SG_DW_ROLL_TW 4
#endif
#ifndef SG_DW_ROLL_BLOCK
#define SG_DW_ROLL_BLOCK 128
#endif
#ifndef SG_DW_ROLL_MINB
#define SG_DW_ROLL_MINB 3
#endif
#ifndef SG_DW_ROLL_ROWS
#define SG_DW_ROLL_ROWS 8
#endif
constexpr int ROLL_ROWS = SG_DW_ROLL_ROWS;      // output rows a thread walks down
constexpr int ROLL_TW = SG_DW_ROLL_TW;          // output columns per thread
constexpr int ROLL_BLOCK = SG_DW_ROLL_BLOCK;    // threads per block

template <typename T, int R>
__device__ __forceinline__ void roll_step(const DepthwiseProblem &p, const T *in_col, float *out_col, int h, int w0,
                                          uint32_t flt_smem, uint32_t flt_pitch, float4 (&col)[3][ROLL_TW + 2]) {
    // rows h and h+1 sit in col[R % 3] and col[(R + 1) % 3]; row h+2 goes to col[(R + 2) % 3]
    const T *row = in_col + (int64_t)(h + 2) * p.i_h;
#pragma unroll
    for (int j = 0; j < ROLL_TW + 2; ++j)
        if (w0 + j < p.Wo + 2) col[(R + 2) % 3][j] = load4(row + (int64_t)j * p.i_w);
    float4 acc[ROLL_TW];
#pragma unroll
    for (int t = 0; t < ROLL_TW; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int kh = 0; kh < 3; ++kh)
#pragma unroll
        for (int kw = 0; kw < 3; ++kw) {
            // the thread's four filter values of this tap, from shared memory (volatile: re-read every step
            // rather than held in 36 registers for the whole walk)
            float4 f;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f.x), "=f"(f.y), "=f"(f.z), "=f"(f.w)
                         : "r"(flt_smem + (uint32_t)(kh * 3 + kw) * flt_pitch));
#pragma unroll
            for (int t = 0; t < ROLL_TW; ++t) fma4(acc[t], col[(R + kh) % 3][t + kw], f);
        }
    float *out = out_col + (int64_t)h * p.o_h;
#pragma unroll
    for (int t = 0; t < ROLL_TW; ++t) {
        if (w0 + t >= p.Wo) break;
        float4 *o = reinterpret_cast<float4 *>(out + (int64_t)t * p.o_w);
        float4 v = acc[t];
        if (p.accumulate) {
            const float4 old = *o;
            v.x += old.x; v.y += old.y; v.z += old.z; v.w += old.w;
        }
        *o = v;
    }
}

template <typename T>
__global__ void __launch_bounds__(ROLL_BLOCK, SG_DW_ROLL_MINB)
depthwise_roll_kernel(const DepthwiseProblem p, const T *__restrict__ I, const T *__restrict__ Kf, float *__restrict__ O) {
    const uint32_t c4s = (uint32_t)(p.C / 4);
    const uint32_t wts = (uint32_t)((p.Wo + ROLL_TW - 1) / ROLL_TW);
    const uint32_t hts = (uint32_t)((p.Ho + ROLL_ROWS - 1) / ROLL_ROWS);
    const uint32_t total = (uint32_t)p.N * hts * wts * c4s;
    // the whole filter as f32 in shared memory: [tap][channel]
    extern __shared__ float4 flt_shared[];
    float *sflt = reinterpret_cast<float *>(flt_shared);
    for (int i = threadIdx.x; i < 9 * p.C; i += ROLL_BLOCK) {
        const int tap = i / p.C, ch = i - tap * p.C;
        sflt[i] = load1(Kf + (int64_t)(tap / 3) * p.k_kh + (int64_t)(tap % 3) * p.k_kw + ch);
    }
    __syncthreads();
    const uint32_t idx = blockIdx.x * (uint32_t)ROLL_BLOCK + threadIdx.x;
    if (idx >= total) return;
    const int c = (int)(idx % c4s) * 4;
    uint32_t r = idx / c4s;
    const int w0 = (int)(r % wts) * ROLL_TW;
    r /= wts;
    const int h0 = (int)(r % hts) * ROLL_ROWS, n = (int)(r / hts);
    const int h1 = min(p.Ho, h0 + ROLL_ROWS);
    const uint32_t flt_smem = (uint32_t)__cvta_generic_to_shared(sflt + c), flt_pitch = (uint32_t)p.C * 4u;
    const T *in_col = I + (int64_t)n * p.i_n + (int64_t)w0 * p.i_w + c;
    float *out_col = O + (int64_t)n * p.o_n + (int64_t)w0 * p.o_w + c;
    float4 col[3][ROLL_TW + 2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < ROLL_TW + 2; ++j)
            if (w0 + j < p.Wo + 2) col[k][j] = load4(in_col + (int64_t)(h0 + k) * p.i_h + (int64_t)j * p.i_w);
    int h = h0;
    for (; h + 2 < h1; h += 3) {
        roll_step<T, 0>(p, in_col, out_col, h, w0, flt_smem, flt_pitch, col);
        roll_step<T, 1>(p, in_col, out_col, h + 1, w0, flt_smem, flt_pitch, col);
        roll_step<T, 2>(p, in_col, out_col, h + 2, w0, flt_smem, flt_pitch, col);
    }
    if (h < h1) roll_step<T, 0>(p, in_col, out_col, h, w0, flt_smem, flt_pitch, col);
    if (h + 1 < h1) roll_step<T, 1>(p, in_col, out_col, h + 1, w0, flt_smem, flt_pitch, col);
}

// K x K window (3 or 5), stride 1 or 2 along h and w, unit dilation, layouts that meet the TMA rules: the input tile of a CTA,
// halo included, is fetched by ONE tensor load into a two-stage shared-memory ring, so the fetch of the next tile runs while
// this one is computed.  A group of CB/2 lanes owns WC output columns of ROWS output rows, two channels per lane; it walks down
// the input rows once, reads each of its (WC-1)*S+K pixels once and adds it into every output it belongs to (at most K/S rows
// are open at a time, in registers, as is the filter).  The 256 / (CB/2) groups of a tile are cg side by side times rg below
// one another, or rg images (small images), whichever wastes less.  Products and sums are packed in pairs (fma.rn.f32x2), which
// halves their issue slots: with scalar FMAs and a 3 x 3 window of inputs in registers a 32x112x112x64 bf16 layer took 32.7 us,
// and 5 x 5 windows, which had no tiled kernel, 200 us.  Warp 8 is the producer.
constexpr int DT_THREADS = 256 + 32;

template <typename T, int CB, int K, int S>
struct DtCfg {
    static constexpr int LANES = CB / 2;                          // per group
    static constexpr int GROUPS = 256 / LANES;
    // output columns and rows of a group (less for f32 and for 16 groups: a tile's two stages leave room for two CTAs per SM)
    static constexpr bool SMALL = sizeof(T) == 4 || GROUPS == 16;
    static constexpr int WC = K == 3 && S == 1 && !SMALL ? 4 : 2;
    static constexpr int ROWS = S == 1 ? 8 : SMALL ? 2 : 4;
    static constexpr int IN_ROWS = (ROWS - 1) * S + K, IN_COLS = (WC - 1) * S + K;
    static constexpr int OPEN = (K + S - 1) / S;                  // output rows a group works on at a time
    static constexpr int PIXEL_BYTES = CB * (int)sizeof(T);
};
struct DtTiling {
    int cg, rg, stack;                // groups side by side; below one another (or, stack, of consecutive images)
    int in_w, in_h;                   // input tile of an image, pixels
    int box_bytes, stage_bytes;
    int tiles_w, tiles_h, tiles_n, c_blocks, num_tiles;
};

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ void fma2(f32x2 &acc, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Two neighbouring channels of a pixel.
__device__ __forceinline__ f32x2 lds2(uint32_t addr, float) {
    f32x2 v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ f32x2 lds2(uint32_t addr, __nv_bfloat16) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return pack2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
}

// The grid is a multiple of c_blocks (or smaller than it never), so a CTA keeps one channel block for all its tiles and a
// thread loads its filter values once.
template <typename T, int CB, int K, int S>
__global__ void __launch_bounds__(DT_THREADS, 2)
depthwise_tma_kernel(const __grid_constant__ CUtensorMap map_in, const DepthwiseProblem p, const T *Kf, float *O, const DtTiling d) {
    using C = DtCfg<T, CB, K, S>;
    extern __shared__ uint8_t dt_smem[];
    __shared__ uint64_t full_bar[2], empty_bar[2];
    __shared__ int abort_load, abort_compute;
    const uint32_t ring = (smem_u32(dt_smem) + 127u) & ~127u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.launch_dependents;");
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 8); }
        abort_load = 0; abort_compute = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // the operands may be the output of the kernel ahead of this one, and the output its input
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int tile_cols = d.cg * C::WC, tile_rows = d.stack ? C::ROWS : d.rg * C::ROWS, tile_n = d.stack ? d.rg : 1;
    if (warp == 8) {
        if (lane == 0) {
            prefetch_tensormap(&map_in);
            int k = 0;
            for (int t = blockIdx.x; t < d.num_tiles; t += gridDim.x, ++k) {
                const int s = k & 1;
                const uint32_t ph = (uint32_t)(k >> 1) & 1u;
                if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u, &abort_load)) break;
                int r = t;
                const int cb = r % d.c_blocks; r /= d.c_blocks;
                const int wt = r % d.tiles_w; r /= d.tiles_w;
                const int ht = r % d.tiles_h, nt = r / d.tiles_h;
                mbar_expect_tx(smem_u32(&full_bar[s]), (uint32_t)d.box_bytes);
                tma_load_4d(ring + (uint32_t)(s * d.stage_bytes), &map_in, smem_u32(&full_bar[s]), cb * CB, wt * tile_cols * S, ht * tile_rows * S, nt * tile_n);
            }
            if (abort_load)      // gave up: let the loads already issued land before the shared memory goes away
                for (int j = (k > 2 ? k - 2 : 0); j < k; ++j)
                    for (int i = 0; i < (1 << 20) && !mbar_try_wait(smem_u32(&full_bar[j & 1]), (uint32_t)(j >> 1) & 1u); ++i) {}
        }
    } else {
        const int group = threadIdx.x / C::LANES, cl = threadIdx.x % C::LANES * 2;
        const int gc = group % d.cg, gr = group / d.cg;
        const int c = (int)(blockIdx.x % d.c_blocks) * CB + cl;        // the same for every tile of this CTA (C is even)
        f32x2 flt[K][K];
#pragma unroll
        for (int kh = 0; kh < K; ++kh)
#pragma unroll
            for (int kw = 0; kw < K; ++kw) {
                const T *f = Kf + (int64_t)kh * p.k_kh + (int64_t)kw * p.k_kw + c;
                flt[kh][kw] = c < p.C ? pack2(load1(f), load1(f + 1)) : 0ull;
            }
        const uint32_t row_bytes = (uint32_t)(d.in_w * C::PIXEL_BYTES);
        const uint32_t group_off = (uint32_t)(gc * C::WC * S * C::PIXEL_BYTES + cl * (int)sizeof(T)) +
                                   (uint32_t)gr * (d.stack ? (uint32_t)d.in_h : (uint32_t)(C::ROWS * S)) * row_bytes;
        int k = 0;
        for (int t = blockIdx.x; t < d.num_tiles; t += gridDim.x, ++k) {
            const int s = k & 1;
            const uint32_t ph = (uint32_t)(k >> 1) & 1u;
            int r = t / d.c_blocks;
            const int wt = r % d.tiles_w; r /= d.tiles_w;
            const int ht = r % d.tiles_h, nt = r / d.tiles_h;
            const int w0 = wt * tile_cols + gc * C::WC, h0 = ht * tile_rows + (d.stack ? 0 : gr * C::ROWS), n = nt * tile_n + (d.stack ? gr : 0);
            const bool ok = mbar_wait(smem_u32(&full_bar[s]), ph, &abort_compute);
            if (!__all_sync(0xffffffffu, ok)) break;
            const int rows = c < p.C && n < p.N ? p.Ho - h0 : 0, cols = p.Wo - w0;      // outputs of this group that exist
            uint32_t src = ring + (uint32_t)(s * d.stage_bytes) + group_off;
            float *out = O + (int64_t)n * p.o_n + (int64_t)h0 * p.o_h + (int64_t)w0 * p.o_w + c;
            if (rows > 0 && cols > 0) {
                f32x2 acc[C::OPEN][C::WC];
#pragma unroll
                for (int rr = 0; rr < C::IN_ROWS; ++rr, src += row_bytes) {
                    f32x2 x[C::IN_COLS];
#pragma unroll
                    for (int j = 0; j < C::IN_COLS; ++j) x[j] = lds2(src + (uint32_t)(j * C::PIXEL_BYTES), T());
#pragma unroll
                    for (int kw = 0; kw < K; ++kw)
#pragma unroll
                        for (int kh = 0; kh < K; ++kh) {      // (neighbouring instructions belong to different sums)
                            if ((rr - kh) % S != 0 || rr < kh || (rr - kh) / S >= C::ROWS) continue;
                            const int h = (rr - kh) / S;
#pragma unroll
                            for (int j = 0; j < C::WC; ++j) {
                                if (kh == 0 && kw == 0) acc[h % C::OPEN][j] = mul2(x[j * S], flt[0][0]);
                                else fma2(acc[h % C::OPEN][j], x[j * S + kw], flt[kh][kw]);
                            }
                        }
                    if (rr >= K - 1 && (rr - (K - 1)) % S == 0) {
                        const int h = (rr - (K - 1)) / S;
                        if (h < rows) {
#pragma unroll
                            for (int j = 0; j < C::WC; ++j) {
                                if (j < cols) {
                                    float2 *o = reinterpret_cast<float2 *>(out + (int64_t)j * p.o_w);
                                    float a, b;
                                    unpack2(acc[h % C::OPEN][j], a, b);
                                    if (p.accumulate) { const float2 old = *o; a += old.x; b += old.y; }
                                    *o = make_float2(a, b);
                                }
                            }
                        }
                        out += p.o_h;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));       // this warp has read all it needs of the stage
        }
    }
    __syncthreads();
}

// Any strides: one output element per thread.
template <typename T, typename IDX>
__global__ void __launch_bounds__(256)
depthwise_generic_kernel(const DepthwiseProblem p, const T *__restrict__ I, const T *__restrict__ Kf, float *__restrict__ O) {
    const IDX total = (IDX)p.N * (IDX)p.Ho * (IDX)p.Wo * (IDX)p.C;
    const IDX idx = (IDX)blockIdx.x * 256 + threadIdx.x;
    if (idx < total) {
        const int c = (int)(idx % (IDX)p.C);
        IDX r = idx / (IDX)p.C;
        const int w = (int)(r % (IDX)p.Wo);
        r /= (IDX)p.Wo;
        const int h = (int)(r % (IDX)p.Ho), n = (int)(r / (IDX)p.Ho);
        float acc = 0.f;
        for (int kh = 0; kh < p.KH; ++kh)
            for (int kw = 0; kw < p.KW; ++kw)
                acc = fmaf(load1(I + (int64_t)n * p.i_n + (int64_t)(h * p.sh + kh * p.dh) * p.i_h +
                                 (int64_t)(w * p.sw + kw * p.dw) * p.i_w + (int64_t)c * p.i_c),
                           load1(Kf + (int64_t)kh * p.k_kh + (int64_t)kw * p.k_kw + (int64_t)c * p.k_c), acc);
        float *o = O + (int64_t)n * p.o_n + (int64_t)h * p.o_h + (int64_t)w * p.o_w + (int64_t)c * p.o_c;
        *o = p.accumulate ? *o + acc : acc;
    }
}

// Groups of a tile: the fewest rounds of thread blocks, weighed with what a tile fetches (a round costs at least what its 256 threads
// compute, about 16 KB worth).  Returns that cost.
template <typename T, int CB, int K, int S>
double plan_tma(const DepthwiseProblem &p, int num_sms, DtTiling &d) {
    using C = DtCfg<T, CB, K, S>;
    double best = 1e300;
    for (int cg = C::GROUPS; cg >= 1; cg >>= 1)       // (wide first: longer runs of memory)
        for (int stack = 0; stack < 2; ++stack) {
            const int rg = C::GROUPS / cg;
            if (stack && (rg == 1 || p.N == 1)) continue;
            const int in_w = (cg * C::WC - 1) * S + K, in_h = ((stack ? 1 : rg) * C::ROWS - 1) * S + K, in_n = stack ? rg : 1;
            if (in_w > 256 || in_h > 256) continue;
            const int bytes = C::PIXEL_BYTES * in_w * in_h * in_n;
            if (bytes > 56 * 1024) continue;                                    // two stages of two thread blocks per SM
            const int64_t tw = (p.Wo + cg * C::WC - 1) / (cg * C::WC), th = (p.Ho + (stack ? 1 : rg) * C::ROWS - 1) / ((stack ? 1 : rg) * C::ROWS);
            const int64_t tn = (p.N + in_n - 1) / in_n, cbs = (p.C + CB - 1) / CB, tiles = tw * th * tn * cbs;
            if (tiles >= ((int64_t)1 << 31)) continue;
            const double rounds = std::max(1.0, (double)tiles / (2 * num_sms));
            const double cost = (rounds < 4 ? std::ceil(rounds) : rounds) * (16384.0 + bytes);
            if (cost < best) {
                best = cost;
                d = DtTiling{cg, rg, stack, in_w, in_h, bytes, (bytes + 127) / 128 * 128, (int)tw, (int)th, (int)tn, (int)cbs, (int)tiles};
            }
        }
    return best;
}

template <typename T, int CB, int K, int S>
bool try_launch_tma(const DepthwiseProblem &p, const DtTiling &d, const T *I, const T *Kf, float *O, int num_sms, cudaStream_t stream, cudaError_t *err) {
    const int64_t es = sizeof(T);
    if (d.num_tiles == 0 || d.c_blocks > num_sms) return false;
    // 3 x 3 problems too small for a tile per SM are left to the kernel without tiles (2.9 us a launch against 3.5)
    if (K == 3 && d.num_tiles < num_sms) return false;
    // the part of the input that is read: ((Ho-1)*S+K) x ((Wo-1)*S+K) pixels per image
    const int64_t h_ext = (int64_t)(p.Ho - 1) * S + K, w_ext = (int64_t)(p.Wo - 1) * S + K;
    const int64_t s_n = p.N > 1 ? p.i_n : h_ext * p.i_h;
    cuuint64_t dims[4] = {(cuuint64_t)p.C, (cuuint64_t)w_ext, (cuuint64_t)h_ext, (cuuint64_t)p.N};
    cuuint64_t strides[3] = {(cuuint64_t)(p.i_w * es), (cuuint64_t)(p.i_h * es), (cuuint64_t)(s_n * es)};
    cuuint32_t box[4] = {(cuuint32_t)CB, (cuuint32_t)d.in_w, (cuuint32_t)d.in_h, (cuuint32_t)(d.stack ? d.rg : 1)};
    for (int i = 0; i < 3; ++i)
        if (strides[i] % 16 != 0 || strides[i] >= ((cuuint64_t)1 << 40)) return false;
    CUtensorMap map_in;
    if (!tensor_encode_tiled(&map_in, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
                             const_cast<T *>(I), dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B))
        return false;
    constexpr int slot = 184 + (sizeof(T) == 4 ? 8 : 0) + (CB == 64 ? 0 : 4) + (K == 5 ? 2 : 0) + (S - 1);
    if (!tensor_ensure_smem_attr(slot, reinterpret_cast<const void *>(depthwise_tma_kernel<T, CB, K, S>), 2 * 56 * 1024 + 128)) return false;
    // two CTAs per SM at a time, rounded down to a multiple of the channel blocks: tile t has block t % c_blocks, so every CTA keeps one
    int64_t grid = std::min<int64_t>(d.num_tiles, 2 * (int64_t)num_sms);
    // Calls that HBM bounds: m times as many CTAs, of 2.6 tiles or more each, that start in order as others end: persistent ones
    // drift apart, and reads and writes then come from all over the two tensors.  us, two per SM and so: bf16 32 x 112 x 112 x 64 28.8
    // and 26.9, x 192 88 and 73, 96 x 150 x 150 x 64 150 and 126, f32 31 x 150 x 157 x 256 278 and 226, bf16 64 x 97 x 97 x 72 72 and 55.
    // (2.0 to 2.4 tiles at least: of 350 layers of 4 to 64 images 16 of bf16 change, 11 of them 2 to 6 % slower and five up to 3 % faster, and nine to twelve of f32, 2 to 8 % slower.)
    // A CTA's start and end cost about 1 us for every further one in a place.  f32 tiles make up for that only where most of what they compute is output: below 90 %
    // with 5 tiles each (with 2.6, 66 x 17 x 17 x 512 19.7 and 21.8, 12 x 74 x 81 x 384 38.5 and 41.6), below 78 % not at all (37 x 66 x 66 x 192 42 and 47).
    // bf16 at stride 2 needs three CTAs to a place to gain at all (two: 2 to 7 % slower), and wide tiles of one image (narrow ones and stacks of images fetch
    // shorter runs: 67 x 49 x 49 x 576 180 and 200, 25 x 26 x 26 x 960 35.0 and 40.7, 34 x 81 x 81 x 256 106 and 120).
    // Not for 5 x 5 windows (arithmetic), f32 at stride 2 (61 and 73) or blocks that miss channels of 64 (f32 40 x 106 x 106 x 48 30.7 and
    // 34.9, bf16 8 x 104 x 104 x 536 48.1 and 51.3); nor where the uneven shares take an eighth more rounds (32 x 112 x 119 x 64 28.6 and 29.6).
    constexpr bool F32 = sizeof(T) == 4;
    using C = DtCfg<T, CB, K, S>;
    const double used = (double)p.N * p.Ho * p.Wo * p.C / ((double)d.num_tiles * (CB * C::GROUPS * C::WC * C::ROWS));
    const bool gains = F32 ? S == 1 && used >= 0.78 : S == 1 || (d.cg > 1 && !d.stack);
    if (K == 3 && gains && (CB == 32 || p.C % 64 == 0)) {
        const int64_t slots = grid, once = (d.num_tiles + slots - 1) / slots;
        int64_t m = d.num_tiles * (int64_t)10 / ((F32 && used < 0.9 ? 50 : 26) * slots);
        while (m > 1 && 100 * m * ((d.num_tiles + m * slots - 1) / (m * slots)) > 113 * once) --m;
        if (m >= (S == 1 ? 2 : 3)) grid = m * slots;
    }
    grid -= grid % d.c_blocks;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(DT_THREADS, 1, 1);
    cfg.dynamicSmemBytes = 2 * d.stage_bytes + 128;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    *err = cudaLaunchKernelEx(&cfg, depthwise_tma_kernel<T, CB, K, S>, map_in, p, Kf, O, d);
    count_launch();
    note_kernel("depthwise_tma_kernel");
    return true;
}

template <typename T, int K, int S>
bool try_launch_window(const DepthwiseProblem &p, const T *I, const T *Kf, float *O, int num_sms, int64_t vec_blocks, cudaStream_t stream, cudaError_t *err) {
    // Blocks of 64 channels; 32 where (bf16) those cover the channels with a fifth less padding, and for 5 x 5 f32 tiles, which would
    // not fit twice.  (Groups of 16 lanes keep two columns open instead of four, and a pixel's 64 bytes of bf16 cost a tensor load what
    // 128 do: 56 x 43 x 43 x 200 at stride 2 69.8 us with 32, 47.2 with 64; 31 x 89 x 89 x 416 149.4 and 139.7; but 26 x 31 x 31 x 32 4.3 and 5.7.)
    if constexpr (sizeof(T) == 2 || K == 3) {
        const int pad64 = (p.C + 63) / 64 * 64, pad32 = (p.C + 31) / 32 * 32;
        bool wide = sizeof(T) == 4 ? pad64 == pad32 || p.C > 64 : 4 * (int64_t)pad64 <= 5 * (int64_t)pad32;
        DtTiling d64{};
        const double cost = wide ? plan_tma<T, 64, K, S>(p, num_sms, d64) : 0.0;
        if (sizeof(T) == 2 && wide && pad64 != pad32) {
            // The last block is half empty, and tiles twice as large fill whole rounds less well: 32 where that costs a fifth more.  us, 32
            // and 64: 8 x 28 x 28 x 288 4.6 and 5.2 (cost 1.56), 24 x 14 x 14 x 224 at stride 2 4.6 and 5.6 (1.42), 5 x 5 windows 8 x 28 x 28 x 152
            // 5.5 and 7.3 (1.53), 32 x 28 x 28 x 160 8.1 and 8.9 (1.23); but 32 x 28 x 28 x 288 14.8 and 13.5 (1.17), 5 x 5 24 x 14 x 14 x 416 10.4 and 9.7 (1.13).
            // 3 x 3 layers with less than a tile of 64 per SM belong to the kernel without tiles as long as that has no more than about 7/3 blocks per SM
            // (307, 8 x 28 x 28 x 200, 4.1 and 4.8 with tiles of 32; 347, 24 x 14 x 14 x 264, 4.2 and 4.0; at stride 2 160, 4 x 14 x 14 x 416, 2.4 and 2.8).
            DtTiling d32{};
            if (K == 3 && d64.num_tiles < num_sms) wide = 3 * vec_blocks <= 7 * (int64_t)num_sms;
            else wide = cost <= 1.2 * plan_tma<T, 32, K, S>(p, num_sms, d32);
        }
        if (wide) return try_launch_tma<T, 64, K, S>(p, d64, I, Kf, O, num_sms, stream, err);
    }
    DtTiling d{};
    plan_tma<T, 32, K, S>(p, num_sms, d);
    return try_launch_tma<T, 32, K, S>(p, d, I, Kf, O, num_sms, stream, err);
}

inline bool mult4(int64_t v) { return v % 4 == 0; }

template <typename T>
cudaError_t launch_typed(const DepthwiseProblem &p, const T *I, const T *Kf, float *O, cudaStream_t stream) {
    const bool vec = p.i_c == 1 && p.k_c == 1 && p.o_c == 1 && p.C % 4 == 0 &&
                     mult4(p.i_n) && mult4(p.i_h) && mult4(p.i_w) && mult4(p.k_kh) && mult4(p.k_kw) &&
                     mult4(p.o_n) && mult4(p.o_h) && mult4(p.o_w) &&
                     reinterpret_cast<uintptr_t>(I) % (4 * sizeof(T)) == 0 && reinterpret_cast<uintptr_t>(Kf) % (4 * sizeof(T)) == 0 &&
                     reinterpret_cast<uintptr_t>(O) % 16 == 0;
    const bool strided3 = p.sw == 2 && p.dw == 1 && p.KW == 3 && p.KH == 3;
    const int tw = strided3 ? TW_STRIDED : TW_UNIT;
    const int64_t work = vec ? (int64_t)p.N * p.Ho * ((p.Wo + tw - 1) / tw) * (p.C / 4) : (int64_t)p.N * p.Ho * p.Wo * p.C;
    const int64_t blocks64 = (work + 255) / 256;
    if (blocks64 > 0x7fffffff) return cudaErrorInvalidConfiguration;
    const unsigned blocks = (unsigned)blocks64;
    const bool small = work < ((int64_t)1 << 32) - 256;
    const bool unit3 = p.sw == 1 && p.dw == 1 && p.KW == 3 && p.KH == 3;
    const bool win3 = p.KW == 3 && p.KH == 3 && p.dw == 1 && p.dh == 1, win5 = p.KW == 5 && p.KH == 5 && p.dw == 1 && p.dh == 1;
    int num_sms = 0;
    const bool ready = tensor_driver_ready(&num_sms);
    if (vec && (win3 || win5) && p.sh == p.sw && p.sh <= 2 && reinterpret_cast<uintptr_t>(I) % 16 == 0 &&
        (p.C * (int64_t)sizeof(T)) % 16 == 0) {
        // TMA-staged tiles (TMA checks the channel bound in 16-byte units, hence the condition on C)
        cudaError_t err = cudaSuccess;
        auto tiles = [&](auto window, auto stride) {
            return try_launch_window<T, decltype(window)::value, decltype(stride)::value>(p, I, Kf, O, num_sms, blocks64, stream, &err);
        };
        using std::integral_constant;
        if (p.C >= 16 && ready &&
            (win3 ? p.sh == 1 ? tiles(integral_constant<int, 3>{}, integral_constant<int, 1>{}) : tiles(integral_constant<int, 3>{}, integral_constant<int, 2>{})
                  : p.sh == 1 ? tiles(integral_constant<int, 5>{}, integral_constant<int, 1>{}) : tiles(integral_constant<int, 5>{}, integral_constant<int, 2>{}))) return err;
    }
    if (vec && unit3 && p.sh == 1 && p.dh == 1) {
        // enough row segments to give every SM several thread blocks: walk down the rows with a rolling window
        const int64_t items = (int64_t)p.N * ((p.Ho + ROLL_ROWS - 1) / ROLL_ROWS) * ((p.Wo + ROLL_TW - 1) / ROLL_TW) * (p.C / 4);
        if (items >= (int64_t)148 * 256 * 2 && items < ((int64_t)1 << 32) - 256 && 9 * p.C * 4 <= 48 * 1024) {
            depthwise_roll_kernel<T><<<(unsigned)((items + ROLL_BLOCK - 1) / ROLL_BLOCK), ROLL_BLOCK, 9 * p.C * 4, stream>>>(p, I, Kf, O);
            count_launch();
            note_kernel("depthwise_roll_kernel");
            return cudaGetLastError();
        }
    }
    // The vector kernel may start while the kernel ahead of it drains: its threads wait for that kernel before their first load.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = vec ? 1 : 0;
    // Behind a kernel that leaves some SMs free its blocks would all be dealt out to those, two, three and four to one, and take that much longer: shared memory
    // that nobody uses keeps an SM to its even share of them.  bf16, us, without overlap / with it / with that: 1 x 59 x 59 x 144, 125 blocks,
    // 2.8 / 3.5 / 2.3; 2 x 31 x 31 x 476, 231, 3.5 / 4.0 / 3.0; at stride 2 4 x 14 x 14 x 416, 160, - / 3.2 / 2.4.
    const int64_t share = num_sms > 0 ? (blocks64 + num_sms - 1) / num_sms : 4;
    auto launch = [&](int slot, auto narrow, auto wide) {
        if (!small) return cudaLaunchKernelEx(&cfg, wide, p, I, Kf, O);
        if (slot != 0 && share <= 3 && tensor_ensure_smem_attr(slot, reinterpret_cast<const void *>(narrow), 115 * 1024))
            cfg.dynamicSmemBytes = (share == 1 ? 115 : share == 2 ? 77 : 58) * 1024;
        return cudaLaunchKernelEx(&cfg, narrow, p, I, Kf, O);
    };
    cudaError_t err;
    // (f32 filters ahead of the multiplications where that matters more than the registers: a lone block, 2 x 6 x 6 x 4, 1.5 us against 1.6, and more blocks than
    // SMs, 7 x 24 x 24 x 184, 182, 3.2 and 3.9; but 3 x 50 x 50 x 36, 69, 3.4 and 2.5)
    const bool ahead = sizeof(T) == 4 && (blocks64 == 1 || blocks64 > num_sms);
    constexpr int slots = sizeof(T) == 2 ? 222 : 224;
    if (vec && unit3 && ahead) err = launch(0, depthwise_vec_kernel<T, 1, uint32_t, sizeof(T) == 4>, depthwise_vec_kernel<T, 1, uint64_t, sizeof(T) == 4>);
    else if (vec && unit3) err = launch(slots, depthwise_vec_kernel<T, 1, uint32_t>, depthwise_vec_kernel<T, 1, uint64_t>);
    else if (vec && strided3) err = launch(slots + 1, depthwise_vec_kernel<T, 2, uint32_t>, depthwise_vec_kernel<T, 2, uint64_t>);
    else if (vec) err = launch(0, depthwise_vec_kernel<T, 0, uint32_t>, depthwise_vec_kernel<T, 0, uint64_t>);
    else err = launch(0, depthwise_generic_kernel<T, uint32_t>, depthwise_generic_kernel<T, uint64_t>);
    count_launch();
    note_kernel(vec ? "depthwise_vec_kernel" : "depthwise_generic_kernel");
    return err;
}

}  // namespace

sg_status depthwise_read_status(cudaStream_t stream) { return read_status_word(stream); }

cudaError_t launch_depthwise(const DepthwiseProblem &p, const void *I, const void *Kf, float *O, cudaStream_t stream) {
    if (p.in_bf16)
        return launch_typed(p, static_cast<const __nv_bfloat16 *>(I), static_cast<const __nv_bfloat16 *>(Kf), O, stream);
    return launch_typed(p, static_cast<const float *>(I), static_cast<const float *>(Kf), O, stream);
}

}  // namespace sg
