// Tensor-core implicit GEMM for layouts that the TMA unit cannot read: rows that do not start on 16-byte boundaries (a
// product whose sizes are multiples of nothing), extents that end inside a 16-byte unit, images of three channels, operands
// without any unit stride.
//
// The pipeline is the one of the TMA kernels with its first stage replaced: sixteen producer warps fetch the operands with
// ordinary loads of one or two elements per lane and write the 128-byte swizzled tiles that tcgen05.mma reads.  A tile is a
// stack of 128-byte lines of 64 bf16: along k (K-major: lines are rows of the input or columns of the filter) or along the
// other index (MN-major: lines are values of k), whichever of the two is contiguous in memory, so that a warp always loads a
// run of memory, one line per instruction.
//
//   warps 0-15   producers, two groups of eight that take the k-blocks in turn: while one group's loads are in flight the
//                other writes its tile.
//   warp  16     MMA issuer and owner of tensor memory.
//   warps 17-20  write-back: tensor memory -> registers -> (bias, activation) -> rows of the output through a shared-memory
//                transpose, one row of 32 columns per store instruction, any alignment and stride.
//
// f32 inputs keep full f32 precision: x = b0 + b1 + b2 with three bf16 values of 8 bits each (the differences are exact), and
// of the nine products the six of weight 2^-16 and up are accumulated, smallest first.  What is dropped is below 2^-23 |a*b|,
// the rounding of a single f32 product.
//
// The tensor core adds into its f32 accumulator by truncation, which drifts with the number of additions (relative error of a
// sum of 4096 bf16 products: 4e-6, against 5e-7 for FFMA).  Callers of these layouts have had FFMA's accuracy so far, so a
// partial sum stays in the accumulator for a chunk of k-blocks only (f32: 64 values of k, bf16: 64 to 256, the more the longer the
// reduction) and is then added, rounding to nearest, to a running sum in tensor memory by the write-back warps, beside the MMAs of the
// next chunk.  Up to four k-blocks of bf16 need no running sum: each has an accumulator of its own (a bank), and the
// write-back adds them up.
//
// What bounds a k-block of a 128 x 128 tile: raw lines, the tensor loads (4.9 cycles for an unaligned line, 1254 of the 1370
// measured); f32, the shared-memory pipe (MMA operands 1536 cycles, parts written 768, and the loads: 3600 measured).
#include <algorithm>
#include <initializer_list>
#include <type_traits>
#include <utility>

#include "sg_internal.cuh"
#include "sg_tc_ptx.cuh"

namespace sg {
namespace {

constexpr int BM = 128, BK = 64;
constexpr int GROUPS = 2, GROUP_WARPS = 8;                  // producer groups and warps per group
constexpr int MMA_WARP = GROUPS * GROUP_WARPS, EPI_WARP = MMA_WARP + 1;
constexpr int MAX_SPLIT = 8;

// How one operand is fetched.  mn_major 0: lines are rows/columns (index mn), a line runs along k; 1: the reverse.
struct Operand {
    int mn_major;
    int pair;             // two neighbouring elements of a line are one aligned load
    int s_mn, s_k;        // element strides of the row/column index and of k (matmul)
    int shift;            // RAW: elements between the 16-byte boundary below the first element and that element
    int groups;           // RAW: whole groups of eight lines
};

// Where a kernel's operand tiles come from.
//   LINEAR  matmul, ordinary loads, any strides
//   CONV    convolution, ordinary loads: addresses from the (n, h, w) / (kh, kw, c) decomposition (input K-major, filter N-major)
//   RAW     bf16 matmul, unit strides: tensor loads.  Eight consecutive lines of pitch P are 16 * P bytes apart, whatever P is,
//           so the operand is a matrix of G groups of eight lines; the lines of one residue mod 8 in a tile are one box of it,
//           eight bytes-aligned boxes a tile, which land shifted by less than 16 bytes.  The producers of the other
//           two take the raw lines from shared memory, shift them in registers and write the tile; the lines behind the last
//           whole group are loaded element by element.
enum { LINEAR = 0, CONVOLUTION = 1, RAW = 2 };

struct GatherParams {
    Problem p;
    Operand a, b;
    int num_kb;           // k-blocks of the whole reduction
    int chunk;            // k-blocks of a partial sum
    int num_n_tiles, num_tiles;
    int splits;           // CTAs of a cluster that share a tile's reduction
    int uniform_rows;     // output row m starts at m * o_w
    int wait_prior;
};

template <int BN, bool F32, int SRC>
struct Cfg {
    static_assert(SRC != RAW || !F32, "raw lines: bf16 only");
    static constexpr int THREADS = 32 * (EPI_WARP + 4 + (SRC == RAW ? 2 : 0));      // RAW: one warp per operand issues its tensor loads
    // eight boxes of 128 / 8 lines of 64 + 8 elements, or of 64 / 8 lines of 128 + 8 (BN 64: of 64 / 8 lines of 64 + 8)
    static constexpr int RAW_A_BYTES = SRC == RAW ? 128 * 2 * (64 + 8) : 0, RAW_B_BYTES = SRC == RAW ? BN * 2 * (64 + 8) : 0;
    static constexpr int RAW_BYTES = RAW_A_BYTES + RAW_B_BYTES;
    static constexpr int RAW_STAGES = BN == 128 ? 3 : 4;
    static constexpr int PARTS = F32 ? 3 : 1;
    static constexpr int A_BYTES = BM * 128, B_BYTES = BN * 128;          // one part of a tile
    static constexpr int STAGE_BYTES = PARTS * (A_BYTES + B_BYTES);
    static constexpr int STAGES = F32 ? 2 : SRC == RAW && BN == 128 ? 3 : 4;
    static constexpr int RING_BYTES = STAGES * STAGE_BYTES;
    static constexpr int STAGING_BYTES = 4 * 4096;                        // one 32 x 32 block per write-back warp
    static constexpr int SMEM_BYTES = RING_BYTES + RAW_STAGES * RAW_BYTES + STAGING_BYTES + 1024 + 256;
    static constexpr int TMEM_COLS = BN == 64 ? 256 : 512;                // two accumulators and the running sum
    static_assert(RING_BYTES >= BM * BN * 4 && RING_BYTES >= MMA_WARP * 4096, "a split reduction parks the tile's partial sums in the ring");
    static_assert(SMEM_BYTES <= 232448, "shared memory");
    // the two producer groups meet every stage of a ring in turn, or each keeps to its own
    static_assert(STAGES % GROUPS == 0 || SRC == RAW, "register-staged groups keep to their own stages");
    static_assert(SRC != RAW || STAGES == RAW_STAGES, "a raw stage and its tile's slot come round together");
};

__device__ __forceinline__ void row_offsets(const Problem &p, int m, int &in_off, int64_t &out_off) {
    const int hw = p.Ho * p.Wo;
    const int n = m / hw, r = m - n * hw;
    const int h = r / p.Wo, w = r - h * p.Wo;
    in_off = (int)((int64_t)n * p.i_n + (int64_t)h * p.sh * p.i_h + (int64_t)w * p.sw * p.i_w);
    out_off = (int64_t)n * p.o_n + (int64_t)h * p.o_h + (int64_t)w * p.o_w;
}
__device__ __forceinline__ void k_offsets(const Problem &p, int k, int &in_off, int &flt_off) {
    const int kwc = p.KW * p.C;
    const int kh = k / kwc, r = k - kh * kwc;
    const int kw = r / p.C, c = r - kw * p.C;
    in_off = (int)((int64_t)kh * p.dh * p.i_h + (int64_t)kw * p.dw * p.i_w + (int64_t)c * p.i_c);
    flt_off = (int)((int64_t)kh * p.k_kh + (int64_t)kw * p.k_kw + (int64_t)c * p.k_c);
}

__device__ __forceinline__ float widen(const float *p) { return *p; }
__device__ __forceinline__ float widen(const unsigned short *p) { return __uint_as_float((uint32_t)*p << 16); }

// Predicated loads without a branch: `r` keeps its value (0) where `ok` is false, and a run of them is issued back to back.
__device__ __forceinline__ void load1_if(bool ok, const float *p, uint32_t &r) {
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u32 %0, [%1];\n\t}" : "+r"(r) : "l"(p), "r"((uint32_t)ok));
}
__device__ __forceinline__ void load1_if(bool ok, const unsigned short *p, uint32_t &r) {
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u16 %0, [%1];\n\t}" : "+r"(r) : "l"(p), "r"((uint32_t)ok));
}
// Two neighbouring elements at an aligned address (bf16: both in r[0]).
__device__ __forceinline__ void load2_if(bool ok, const float *p, uint32_t (&r)[2]) {
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q ld.global.nc.v2.u32 {%0, %1}, [%2];\n\t}" : "+r"(r[0]), "+r"(r[1]) : "l"(p), "r"((uint32_t)ok));
}
__device__ __forceinline__ void load2_if(bool ok, const unsigned short *p, uint32_t (&r)[2]) {
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u32 %0, [%1];\n\t}" : "+r"(r[0]) : "l"(p), "r"((uint32_t)ok));
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

// The lanes' two elements of one line -> the line's word of every part tile.  Returns whether an f32 value is infinite or
// so large that rounding it to bf16 could overflow.
template <bool F32>
__device__ __forceinline__ bool store_pair(uint32_t addr, uint32_t part_bytes, const uint32_t (&r)[2]) {
    if constexpr (!F32) {
        sts32(addr, r[0] | (r[1] << 16));        // (a pair loaded at once is in r[0] already)
        return false;
    } else {
        const float x = __uint_as_float(r[0]), y = __uint_as_float(r[1]);
        const uint32_t w0 = pack_bf16(x, y);
        const float x1 = x - __uint_as_float(w0 << 16), y1 = y - __uint_as_float(w0 & 0xFFFF0000u);
        const uint32_t w1 = pack_bf16(x1, y1);
        const float x2 = x1 - __uint_as_float(w1 << 16), y2 = y1 - __uint_as_float(w1 & 0xFFFF0000u);
        sts32(addr, w0);
        sts32(addr + part_bytes, w1);
        sts32(addr + 2 * part_bytes, pack_bf16(x2, y2));
        return fmaxf(fabsf(x), fabsf(y)) >= 1.7014118e38f;
    }
}

// Eight lines of a warp (line0, line0 + 8, ...) of one 64-line batch: `off(i)` is the element offset of line i (negative: no
// such line), l0 / l1 the lane's two element offsets within a line (ok0 / ok1: whether they exist; the same when `pair`).
template <typename T, typename LineOff>
__device__ __forceinline__ void load_lines(uint32_t (&r)[8][2], const T *base, int pair, int l0, int l1, bool ok0, bool ok1, LineOff off) {
    if (pair) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int o = off(i);
            r[i][0] = 0; r[i][1] = 0;
            load2_if(o >= 0 && ok0, base + (int64_t)(o + l0), r[i]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int o = off(i);
            r[i][0] = 0; r[i][1] = 0;
            load1_if(o >= 0 && ok0, base + (int64_t)(o + l0), r[i][0]);
            load1_if(o >= 0 && ok1, base + (int64_t)(o + l1), r[i][1]);
        }
    }
}

// RAW: one operand's tile of a k-block, from the raw lines at `raw` (box j holds the lines of residue j mod 8, 16-byte aligned
// and shifted by a few elements) to the swizzled tile at `dst`.  Eight lanes per line, 16 bytes each: the two aligned
// 16-byte pieces they lie in, shifted.  Lines and elements beyond the end are zero (lines: the tensor loads' fill).
template <int WIDTH>
__device__ __forceinline__ void shift_tile(const unsigned short *ptr, const Operand &op, int mn0, int mn_end, int k0, int k_end, uint32_t raw, uint32_t dst,
                                           int w, int lane) {
    const int s_line = op.mn_major ? op.s_k : op.s_mn;
    const int n = w * 4 + (lane >> 3), piece = lane & 7;           // line of step 0; step t: n + 32 * t
    const int line_pitch = op.mn_major ? (WIDTH + 8) * 2 : 144;    // bytes between the raw lines of a residue
    const int line0 = op.mn_major ? k0 : mn0, line_end = op.mn_major ? k_end : mn_end;
    // (tiles start at multiples of eight lines and of eight elements)
    const uint32_t shift = (uint32_t)(op.shift + (n & 7) * s_line) & 7u;
    const uint32_t src = raw + (uint32_t)((n & 7) * (op.mn_major ? 8 : WIDTH / 8) * line_pitch + (n >> 3) * line_pitch + piece * 16);
    const uint32_t out = dst + (uint32_t)(n * 128 + ((piece ^ (n & 7)) << 4));
    const bool b8 = shift & 4, b4 = shift & 2;
    const uint32_t bits = (shift & 1) * 16;
    const bool ragged_k = !op.mn_major && k0 + 64 > k_end;
    const int left = k_end - k0 - piece * 8;                       // K-major: values of k this lane's 16 bytes still hold
    const int whole = 8 * op.groups - line0;                       // lines of the tile that the boxes bring
    const bool ragged_lines = whole < (op.mn_major ? 64 : WIDTH) && 8 * op.groups < line_end;
    uint32_t v[WIDTH / 32][8];
#pragma unroll
    for (int t = 0; t < WIDTH / 32; ++t) {
        const uint32_t a = src + (op.mn_major ? (uint32_t)((t & 1) * 4 * line_pitch + (t >> 1) * 128) : (uint32_t)(t * 4 * 144));
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[t][0]), "=r"(v[t][1]), "=r"(v[t][2]), "=r"(v[t][3]) : "r"(a) : "memory");
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+16];" : "=r"(v[t][4]), "=r"(v[t][5]), "=r"(v[t][6]), "=r"(v[t][7]) : "r"(a) : "memory");
    }
#pragma unroll
    for (int t = 0; t < WIDTH / 32; ++t) {
        uint32_t x[6], y[5], o[4];
#pragma unroll
        for (int i = 0; i < 6; ++i) x[i] = b8 ? v[t][i + 2] : v[t][i];
#pragma unroll
        for (int i = 0; i < 5; ++i) y[i] = b4 ? x[i + 1] : x[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = __funnelshift_r(y[i], y[i + 1], bits);
        if (ragged_k)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] = 2 * i + 1 < left ? o[i] : 2 * i < left ? o[i] & 0xFFFFu : 0u;
        const int x_line = op.mn_major ? (n + 32 * t) & 63 : n + 32 * t;
        if (!ragged_lines || x_line < whole || x_line >= line_end - line0)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(out + t * 4096), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]) : "memory");
    }
    if (ragged_lines) {
        // the lines behind the last whole group, one per warp and turn
        const int rest = line_end - max(8 * op.groups, line0), subs = op.mn_major ? WIDTH / 64 : 1;
        for (int u = w; u < rest * subs; u += GROUP_WARPS) {
            const int line = max(8 * op.groups, line0) + u % rest, sub = u / rest;
            const int e = (op.mn_major ? mn0 + 64 * sub : k0) + 2 * lane, e_end = op.mn_major ? mn_end : k_end;
            const int x = line - line0 + 64 * sub;
            uint32_t r[2] = {0, 0};
            load1_if(e < e_end, ptr + ((int64_t)line * s_line + e), r[0]);
            load1_if(e + 1 < e_end, ptr + ((int64_t)line * s_line + e + 1), r[1]);
            sts32(dst + (uint32_t)(x * 128 + (((lane >> 2) ^ (x & 7)) << 4) + (lane & 3) * 4), r[0] | (r[1] << 16));
        }
    }
}

// This lane's column of eight output rows: out[ro[x]] (+)= act(v[x] + bias) for x < rows.
__device__ __forceinline__ void write_rows(float *out, const float (&v)[8], const int64_t (&ro)[8], int rows, float bias, int act, int accumulate) {
    float old[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) old[x] = 0.f;
    if (accumulate)
#pragma unroll
        for (int x = 0; x < 8; ++x) if (x < rows) old[x] = out[ro[x]];
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        float r = v[x] + bias;
        if (act == SG_ACT_RELU && r < 0.f) r = 0.f;
        if (x < rows) out[ro[x]] = old[x] + r;
    }
}

// Infinities (or values next to overflow) among the operands: their products with the zeros of the split would be NaN, so a
// 32 x 32 block is summed as it stands over k0 <= k < k1 and staged at `dst` like any other (lane = row m; lane's column n).  A lane
// loads its row's and its column's next four values; the columns go round by shuffles.  (With each of its 1024 sums walking along k by
// itself a 1531 x 1021 x 765 product with one infinity took 8.0 ms, now 0.42.)  A whole tile takes about 4000 cycles for each k, while
// the other warps wait for it: see the limit on K in launch_gather.
template <typename T, bool CONV>
__device__ __forceinline__ void sum_as_it_stands(const Problem &p, const T *In, const T *Flt, int m, int n, int k0, int k1, uint32_t dst) {
    const int lane = threadIdx.x & 31;
    int64_t unused;
    int ro = 0;
    if (m < p.M) row_offsets(p, m, ro, unused);
    const T *row = In + ro, *col = Flt + (n < p.N ? (int64_t)n * p.k_f : 0);
#pragma unroll 1
    for (int c0 = 0; c0 < 32; c0 += 16) {      // (sixteen columns at a time: registers)
        float sum[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) sum[c] = 0.f;
#pragma unroll 1
        for (int k = k0; k < k1; k += 4) {
            float a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int io = 0, fo = 0;
                const bool ok = k + u < k1;
                if (CONV && ok) k_offsets(p, k + u, io, fo);
                if (!CONV && ok) { io = (k + u) * (int)p.i_c; fo = (k + u) * (int)p.k_c; }
                a[u] = ok && m < p.M ? widen(row + io) : 0.f;
                b[u] = ok && n < p.N ? widen(col + fo) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < 16; ++c) sum[c] = fmaf(a[u], __shfl_sync(0xffffffffu, b[u], c0 + c), sum[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(lane * 128 + (((c0 / 4 + c) ^ (lane & 7)) << 4))),
                         "f"(sum[4 * c]), "f"(sum[4 * c + 1]), "f"(sum[4 * c + 2]), "f"(sum[4 * c + 3]) : "memory");
    }
}

// BANKS > 1 (bf16, one CTA per tile): the reduction is at most BANKS k-blocks, each with an accumulator of its own.
template <int BN, bool F32, int SRC, int BANKS>
__global__ void __launch_bounds__(Cfg<BN, F32, SRC>::THREADS, 1)
gather_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ GatherParams gp, const void *__restrict__ in_ptr, const void *__restrict__ flt_ptr, float *__restrict__ O) {
    constexpr bool CONV = SRC == CONVOLUTION;
    constexpr int BUFS = BANKS == 4 ? 1 : 2;      // accumulators (of BANKS banks) that the MMAs and the write-back take turns with
    using C = Cfg<BN, F32, SRC>;
    using T = typename std::conditional<F32, float, unsigned short>::type;
    const Problem &p = gp.p;
    const T *In = static_cast<const T *>(in_ptr), *Flt = static_cast<const T *>(flt_ptr);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t raw_addr = smem_base + C::RING_BYTES, staging_addr = raw_addr + C::RAW_STAGES * C::RAW_BYTES;
    const uint32_t bars = staging_addr + C::STAGING_BYTES;
    uint8_t *bars_gen = smem_gen + C::RING_BYTES + C::RAW_STAGES * C::RAW_BYTES + C::STAGING_BYTES;
    // barrier block: full[4] | empty[4] | acc_full[2] | acc_empty[2] | sum | done | raw_full[4] | raw_empty[4] | tmem_ptr | abort | large
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (4 + s); };
    auto acc_full_bar = [&](int b) { return bars + 8u * (8 + b); };
    auto acc_empty_bar = [&](int b) { return bars + 8u * (10 + b); };
    const uint32_t sum_bar = bars + 8u * 12, done_bar = bars + 8u * 13;      // completed once: the last tile's running sum, its last MMAs
    auto raw_full_bar = [&](int s) { return bars + 8u * (14 + s); };
    auto raw_empty_bar = [&](int s) { return bars + 8u * (18 + s); };
    volatile uint32_t *tmem_ptr_slot = reinterpret_cast<volatile uint32_t *>(bars_gen + 8 * 22);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars_gen + 8 * 22 + 4);
    volatile int *large_flag = reinterpret_cast<volatile int *>(bars_gen + 8 * 22 + 8);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.launch_dependents;");
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(full_bar(s), GROUP_WARPS); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(acc_full_bar(b), 1); mbar_init(acc_empty_bar(b), 4); }
        mbar_init(sum_bar, 4);
        mbar_init(done_bar, 1);
        if (SRC == RAW) for (int s = 0; s < C::RAW_STAGES; ++s) { mbar_init(raw_full_bar(s), 2); mbar_init(raw_empty_bar(s), GROUP_WARPS); }
        *abort_flag = 0;
        *large_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (SRC == RAW && threadIdx.x == 0) { prefetch_tensormap(&map_a); prefetch_tensormap(&map_b); }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<uint32_t *>(tmem_ptr_slot))), "r"((uint32_t)C::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_ptr_slot;
    const uint32_t sum_tmem = tmem_base + 2 * BN;

    // splits == 1: tiles are dealt round-robin to the CTAs.  splits > 1: one tile per cluster, the CTA of rank r reduces
    // k-blocks [r / splits, (r + 1) / splits) of the whole (never none: there are at least as many k-blocks as ranks).
    const int rank = gp.splits > 1 ? (int)cluster_ctarank() : 0;
    const int first_tile = (int)blockIdx.x / gp.splits, tile_step = gp.splits > 1 ? gp.num_tiles : (int)gridDim.x;
    const int kb0 = (int)((int64_t)rank * gp.num_kb / gp.splits), kb1 = (int)((int64_t)(rank + 1) * gp.num_kb / gp.splits);
    const int per = F32 ? 1 : BANKS > 1 ? BANKS : gp.chunk;      // k-blocks of a partial sum

    // One 32-row x 32-column block of a tile: column block j of this warp's TMEM lane quarter, the partial sum in accumulator
    // `buf` and (not `first`) the running sum.  Adds them up; when it is the `last` partial sum, writes the block out.
    const int q = warp & 3;                        // TMEM lane quarter this warp may access
    const uint32_t lane_tmem = (uint32_t)(q * 32) << 16;
    auto finish_block = [&](int m0, int n0, int j, int buf, bool first, bool last, uint32_t stage) {
        uint32_t r[32];
        tmem_ld_32x32(tmem_base + lane_tmem + (uint32_t)(buf * BANKS * BN + j * 32), r);
        if (BANKS > 1) {
            tmem_ld_wait();
#pragma unroll 1
            for (int b = 1; b < kb1; ++b) {
                uint32_t s[32];
                tmem_ld_32x32(tmem_base + lane_tmem + (uint32_t)((buf * BANKS + b) * BN + j * 32), s);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 32; ++c) r[c] = __float_as_uint(__uint_as_float(r[c]) + __uint_as_float(s[c]));
            }
        } else if (!first) {
            uint32_t s[32];
            tmem_ld_32x32(sum_tmem + lane_tmem + (uint32_t)(j * 32), s);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 32; ++c) r[c] = __float_as_uint(__uint_as_float(s[c]) + __uint_as_float(r[c]));
        } else {
            tmem_ld_wait();
        }
        if (!last) {
            tmem_st_32x32(sum_tmem + lane_tmem + (uint32_t)(j * 32), r);
            return;
        }
        // lane = row: 16-byte chunks of this row, chunk c of row x at chunk c ^ (x & 7); a split reduction parks
        // the whole tile in the ring instead ([column block of 32][row][128 bytes])
        const uint32_t dst = gp.splits > 1 ? smem_base + (uint32_t)(j * BM + q * 32) * 128u : stage;
        if (gp.splits == 1) __syncwarp();
        if (F32 && __any_sync(0xffffffffu, *large_flag)) sum_as_it_stands<T, CONV>(p, In, Flt, m0 + q * 32 + lane, n0 + j * 32 + lane, kb0 * BK, min(p.K, kb1 * BK), dst);
        else
#pragma unroll
        for (int c = 0; c < 8; ++c)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)(lane * 128 + ((c ^ (lane & 7)) << 4))),
                         "r"(r[4 * c]), "r"(r[4 * c + 1]), "r"(r[4 * c + 2]), "r"(r[4 * c + 3]) : "memory");
        if (gp.splits > 1) return;
        __syncwarp();
        // lane = column: one row of 32 columns per store
        const int n = n0 + j * 32 + lane;
        const float bias = (p.bias != nullptr && n < p.N) ? __ldg(p.bias + (int64_t)n * p.bias_f) : 0.f;
        const int m_first = m0 + q * 32;
        const int rows = n < p.N ? p.M - m_first : 0;
        float *out = O + (int64_t)n * p.o_f;
        auto staged = [&](int x) {
            float v;
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(stage + (uint32_t)(x * 128 + (((lane >> 2) ^ (x & 7)) << 4) + (lane & 3) * 4)) : "memory");
            return v;
        };
        if (gp.uniform_rows && !p.accumulate && m_first + 32 <= p.M) {
            out += (int64_t)m_first * p.o_w;
#pragma unroll
            for (int x0 = 0; x0 < 32; x0 += 16) {
                float v[16];
#pragma unroll
                for (int x = 0; x < 16; ++x) v[x] = staged(x0 + x);
                if (rows > 0)
#pragma unroll
                    for (int x = 0; x < 16; ++x, out += p.o_w) {
                        const float y = v[x] + bias;
                        *out = (p.act == SG_ACT_RELU && y < 0.f) ? 0.f : y;
                    }
            }
        } else {
            int64_t my_out = 0;            // lane i holds the output offset of row i
            int unused;
            if (m_first + lane < p.M) row_offsets(p, m_first + lane, unused, my_out);
            for (int x0 = 0; x0 < 32; x0 += 8) {
                float v[8];
                int64_t ro[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    v[x] = staged(x0 + x);
                    ro[x] = __shfl_sync(0xffffffffu, my_out, x0 + x);
                }
                write_rows(out, v, ro, rows - x0, bias, p.act, p.accumulate);
            }
        }
    };

    if (warp < MMA_WARP) {
        // ------------------------------------------------------------ producers
        if (gp.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
        const int group = warp / GROUP_WARPS, w = warp % GROUP_WARPS;
        // this lane's word of line j*64 + w + 8*i: (j*64 + w)*128 + i*1024, 16-byte chunk lane/4 swizzled by the line's low bits (= w)
        const uint32_t lane_off = (uint32_t)(w * 128 + (((lane >> 2) ^ w) << 4) + (lane & 3) * 4);
        int it = 0;
        bool ok = true;
        for (int tile = first_tile; ok && tile < gp.num_tiles; tile += tile_step) {
            const int mt = tile / gp.num_n_tiles;
            const int m0 = mt * BM, n0 = (tile - mt * gp.num_n_tiles) * BN;
            int row_off = 0;          // CONV: lane i < 16 holds the input offset of row w + 8*i of the tile (-1: beyond M)
            if constexpr (CONV) {
                const int m = m0 + w + 8 * (lane & 15);
                int64_t unused;
                if (m < p.M) row_offsets(p, m, row_off, unused);
                else row_off = -1;
            }
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                if (it % GROUPS != group) continue;
                const int k0 = kb * BK;
                if constexpr (SRC == RAW) {
                    const int s = it % C::STAGES, rs = it % C::RAW_STAGES;
                    // The tile's slot first: with an odd number of stages the other group met this one a round ago, and a barrier's
                    // parity does not tell its phase from the one before the last.  That the MMAs have read what it held shows
                    // that the other group's raw lines had landed too, so the wait behind it can only mean this round's.
                    if (!mbar_wait(empty_bar(s), ((it / C::STAGES) & 1) ^ 1u, abort_flag)) { ok = false; break; }
                    if (!mbar_wait(raw_full_bar(rs), (it / C::RAW_STAGES) & 1, abort_flag)) { ok = false; break; }
                    const uint32_t raw = raw_addr + rs * C::RAW_BYTES, dst = smem_base + s * C::STAGE_BYTES;
                    shift_tile<BM>(In, gp.a, m0, p.M, k0, p.K, raw, dst, w, lane);
                    shift_tile<BN>(Flt, gp.b, n0, p.N, k0, p.K, raw + C::RAW_A_BYTES, dst + C::A_BYTES, w, lane);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) { mbar_arrive(raw_empty_bar(rs)); mbar_arrive(full_bar(s)); }
                    continue;
                }
                uint32_t ra[2][8][2], rb[BN / 64][8][2];
                if constexpr (CONV) {
                    // input, K-major: lines are rows, the lane's two k; filter, N-major: lines are k
                    const int k = k0 + 2 * lane;
                    int i0 = 0, i1 = 0, f_off = -1, unused;
                    if (k < p.K) k_offsets(p, k, i0, unused);
                    if (k + 1 < p.K) k_offsets(p, k + 1, i1, unused);
                    if (k0 + w + 8 * (lane & 7) < p.K) k_offsets(p, k0 + w + 8 * (lane & 7), unused, f_off);
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        load_lines(ra[j], In, gp.a.pair, i0, i1, k < p.K, k + 1 < p.K,
                                   [&](int i) { return __shfl_sync(0xffffffffu, row_off, 8 * j + i); });
#pragma unroll
                    for (int j = 0; j < BN / 64; ++j) {
                        const int n = n0 + j * 64 + 2 * lane;
                        load_lines(rb[j], Flt, gp.b.pair, n * gp.b.s_mn, (n + 1) * gp.b.s_mn, n < p.N, n + 1 < p.N,
                                   [&](int i) { return __shfl_sync(0xffffffffu, f_off, i); });
                    }
                } else {
                    auto load_operand = [&](auto &r, const T *base, const Operand &op, int mn0, int mn_end) {
                        constexpr int BATCHES = sizeof(r) / sizeof(r[0]);
#pragma unroll
                        for (int j = 0; j < BATCHES; ++j) {
                            const int line0 = (op.mn_major ? k0 : mn0 + j * 64) + w, lines = op.mn_major ? p.K : mn_end;
                            const int e = (op.mn_major ? mn0 + j * 64 : k0) + 2 * lane, es = op.mn_major ? mn_end : p.K;
                            const int s_line = op.mn_major ? op.s_k : op.s_mn, s_e = op.mn_major ? op.s_mn : op.s_k;
                            load_lines(r[j], base, op.pair, e * s_e, (e + 1) * s_e, e < es, e + 1 < es,
                                       [&](int i) { return line0 + 8 * i < lines ? (line0 + 8 * i) * s_line : -1; });
                        }
                    };
                    load_operand(ra, In, gp.a, m0, p.M);
                    load_operand(rb, Flt, gp.b, n0, p.N);
                }
                const int s = it % C::STAGES;
                if (!mbar_wait(empty_bar(s), ((it / C::STAGES) & 1) ^ 1u, abort_flag)) { ok = false; break; }
                const uint32_t a_dst = smem_base + s * C::STAGE_BYTES + lane_off, b_dst = a_dst + C::PARTS * C::A_BYTES;
                bool large = false;
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int i = 0; i < 8; ++i) large |= store_pair<F32>(a_dst + j * 8192 + i * 1024, C::A_BYTES, ra[j][i]);
#pragma unroll
                for (int j = 0; j < BN / 64; ++j)
#pragma unroll
                    for (int i = 0; i < 8; ++i) large |= store_pair<F32>(b_dst + j * 8192 + i * 1024, C::B_BYTES, rb[j][i]);
                if (F32 && large) *large_flag = 1;
                fence_async_smem();       // generic-proxy writes -> visible to the tensor core's reads
                __syncwarp();
                if (lane == 0) mbar_arrive(full_bar(s));
            }
        }
        // ---- a share of the last tile's write-back: column block 1 + warp / 4 (staged in the ring, which has been consumed)
        const int chunks = (kb1 - kb0 + per - 1) / per, tiles = (gp.num_tiles - 1 - first_tile) / tile_step + 1;
        const int tile = first_tile + (tiles - 1) * tile_step, last = tiles * chunks - 1, j = 1 + (warp >> 2);
        const int mt = tile / gp.num_n_tiles, n0 = (tile - mt * gp.num_n_tiles) * BN;
        if (ok && j * 32 < min(BN, p.N - n0)) {
            ok = mbar_wait(done_bar, 0, abort_flag) && (chunks == 1 || mbar_wait(sum_bar, 0, abort_flag));
            if (__all_sync(0xffffffffu, ok)) {
                tc_fence_after();
                finish_block(mt * BM, n0, j, last & (BUFS - 1), chunks == 1, true, smem_base + (uint32_t)warp * 4096u);
            }
        }
    } else if (warp == MMA_WARP) {
        // ------------------------------------------------------------ MMA issuer: the whole warp walks, one lane issues
        const uint32_t idesc = make_idesc(BN, BM, false, false, false) | (gp.a.mn_major ? 1u << 15 : 0u) | (gp.b.mn_major ? 1u << 16 : 0u);
        const int a_step = gp.a.mn_major ? 128 : 2, b_step = gp.b.mn_major ? 128 : 2;      // 16 k: 16 lines or 32 bytes of a line
        const uint32_t a_lbo = gp.a.mn_major ? 8192 : 16, b_lbo = gp.b.mn_major ? 8192 : 16;
        const bool issuer = elect_one();
        auto wait_all = [&](bool passed) { return __all_sync(0xffffffffu, passed) != 0; };
        int it = 0, chunk = 0;
        bool ok = true;
        for (int tile = first_tile; ok && tile < gp.num_tiles; tile += tile_step) {
            for (int kb = kb0; kb < kb1 && ok; kb += per, ++chunk) {
                const int buf = chunk & (BUFS - 1);
                if (!wait_all(mbar_wait(acc_empty_bar(buf), ((chunk >> (BUFS - 1)) & 1) ^ 1u, abort_flag))) { ok = false; break; }
                tc_fence_after();
                uint32_t d = tmem_base + buf * BANKS * BN;
                uint32_t acc = 0;
                for (int kk = kb; kk < min(kb1, kb + per); ++kk, ++it) {
                    const int s = it % C::STAGES;
                    if (!wait_all(mbar_wait(full_bar(s), (it / C::STAGES) & 1, abort_flag))) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a_addr = smem_base + s * C::STAGE_BYTES, b_addr = a_addr + C::PARTS * C::A_BYTES;
                    if (issuer) {
                        constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};     // smallest products first
#pragma unroll
                        for (int q = F32 ? 0 : 5; q < 6; ++q) {
                            const uint64_t ad = make_smem_desc(a_addr + PA[q] * C::A_BYTES, a_lbo, 1024);
                            const uint64_t bd = make_smem_desc(b_addr + PB[q] * C::B_BYTES, b_lbo, 1024);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                umma_bf16(d, ad + (uint64_t)(k * a_step), bd + (uint64_t)(k * b_step), idesc, acc);
                                acc = 1u;
                            }
                        }
                        umma_commit(empty_bar(s));
                    }
                    if (BANKS > 1) { d += BN; acc = 0; }
                    else acc = 1u;
                }
                if (ok && issuer) {
                    umma_commit(acc_full_bar(buf));
                    if (kb + per >= kb1 && tile + tile_step >= gp.num_tiles) umma_commit(done_bar);
                }
            }
        }
    } else if (SRC == RAW && warp >= EPI_WARP + 4) {
        // ------------------------------------------------------------ RAW: tensor loads, lane j < 8 those of residue j
        const bool input = warp == EPI_WARP + 4;
        const Operand &op = input ? gp.a : gp.b;
        const CUtensorMap *map = input ? &map_a : &map_b;
        const int width = input ? BM : BN;
        const uint32_t bytes = op.mn_major ? 64 * 2 * (width + 8) : width * 2 * (64 + 8);
        if (gp.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
        int it = 0;
        bool ok = true;
        for (int tile = first_tile; ok && tile < gp.num_tiles; tile += tile_step) {
            const int mt = tile / gp.num_n_tiles;
            const int mn0 = input ? mt * BM : (tile - mt * gp.num_n_tiles) * BN;
            const int64_t line_pos = op.shift + (int64_t)(lane & 7) * (op.mn_major ? op.s_k : op.s_mn);
            for (int kb = kb0; kb < kb1; ++kb, ++it) {
                const int rs = it % C::RAW_STAGES;
                if (!__all_sync(0xffffffffu, mbar_wait(raw_empty_bar(rs), ((it / C::RAW_STAGES) & 1) ^ 1u, abort_flag))) { ok = false; break; }
                const uint32_t dst = raw_addr + rs * C::RAW_BYTES + (input ? 0 : C::RAW_A_BYTES);
                if (lane == 0) mbar_expect_tx(raw_full_bar(rs), bytes);
                __syncwarp();
                if (lane < 8)
                    tma_load_2d(dst + lane * (bytes / 8), map, raw_full_bar(rs), (int)((line_pos + (op.mn_major ? mn0 : kb * BK)) & ~(int64_t)7),
                                (op.mn_major ? kb * BK : mn0) / 8);
            }
        }
    } else {
        // ------------------------------------------------------------ write-back
        const uint32_t stage = staging_addr + (uint32_t)(warp - EPI_WARP) * 4096u;
        int chunk = 0;
        bool ok = true;
        if (gp.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int tile = first_tile; ok && tile < gp.num_tiles; tile += tile_step) {
            const int mt = tile / gp.num_n_tiles;
            const int m0 = mt * BM, n0 = (tile - mt * gp.num_n_tiles) * BN;
            const int cols = min(BN, p.N - n0);
            for (int kb = kb0; kb < kb1; kb += per, ++chunk) {
                const int buf = chunk & (BUFS - 1);
                const bool first = kb == kb0, last = kb + per >= kb1;
                if (!epilogue_all(mbar_wait(acc_full_bar(buf), (chunk >> (BUFS - 1)) & 1, abort_flag))) { ok = false; break; }
                tc_fence_after();
                // (of the CTA's last tile the producers, done by now, write all column blocks but the first)
                const bool shared = last && tile + tile_step >= gp.num_tiles;
                for (int j = 0; j * 32 < (shared ? 32 : cols); ++j) finish_block(m0, n0, j, buf, first, last, stage);
                if (!last) asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(acc_empty_bar(buf));
                    if (!last && kb + 2 * per >= kb1 && tile + tile_step >= gp.num_tiles) mbar_arrive(sum_bar);
                }
            }
        }
    }

    // ---------------------------------------------------------------- split reduction and teardown
    __syncthreads();
    if (SRC == RAW && *abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(5000);      // let tensor loads in flight land before the shared memory goes
        __syncthreads();
    }
    if (gp.splits > 1) {
        // every CTA of the cluster sums its share of the tile's rows over the partial tiles parked in all of them, in rank order
        cluster_sync_all();
        const int mt = first_tile / gp.num_n_tiles;
        const int m0 = mt * BM, n0 = (first_tile - mt * gp.num_n_tiles) * BN;
        const int rows = BM / gp.splits, cols = min(BN, p.N - n0);
        if (!*abort_flag)
            for (int u = warp; u < rows * (BN / 32); u += C::THREADS / 32) {
                const int j = u / rows, x = rank * rows + (u - j * rows), m = m0 + x;
                if (j * 32 >= cols || m >= p.M) continue;
                const uint32_t src = smem_base + (uint32_t)((j * BM + x) * 128 + (((lane >> 2) ^ (x & 7)) << 4) + (lane & 3) * 4);
                float part[MAX_SPLIT];
#pragma unroll
                for (int r = 0; r < MAX_SPLIT; ++r)
                    if (r < gp.splits) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(part[r]) : "r"(map_to_cta(src, r)) : "memory");
                float v = part[0];
#pragma unroll
                for (int r = 1; r < MAX_SPLIT; ++r)
                    if (r < gp.splits) v += part[r];
                const int n = n0 + j * 32 + lane;
                if (n < p.N) {
                    int unused;
                    int64_t ro = (int64_t)m * p.o_w;
                    if constexpr (CONV) row_offsets(p, m, unused, ro);
                    float *o = O + ro + (int64_t)n * p.o_f;
                    if (p.bias != nullptr) v += __ldg(p.bias + (int64_t)n * p.bias_f);
                    if (p.act == SG_ACT_RELU && v < 0.f) v = 0.f;
                    *o = p.accumulate ? *o + v : v;
                }
            }
        cluster_sync_all();      // nobody leaves while its partial tile is being read
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)C::TMEM_COLS) : "memory");
    }
}

// Largest element offset of an operand's rectangle (strides are not negative), or -1 when it does not fit 31 bits.
inline int64_t reach(std::initializer_list<std::pair<int64_t, int64_t>> extents_strides) {
    int64_t r = 0;
    for (const auto &e : extents_strides) {
        if (e.first > 1 && e.second > 0x7fffffff) return -1;
        r += (e.first - 1) * e.second;
        if (r > 0x7fffff00) return -1;
    }
    return r;
}

template <int BN, bool F32, int SRC, int BANKS>
sg_status launch_variant(const CUtensorMap &ma, const CUtensorMap &mb, const GatherParams &gp, const void *In, const void *Flt, float *O, int num_sms, int slot, cudaStream_t stream) {
    using C = Cfg<BN, F32, SRC>;
    const void *fn = reinterpret_cast<const void *>(gather_gemm_kernel<BN, F32, SRC, BANKS>);
    if (!tensor_ensure_smem_attr(slot, fn, C::SMEM_BYTES)) return SG_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(gp.splits > 1 ? gp.num_tiles * gp.splits : std::min(gp.num_tiles, num_sms), 1, 1);
    cfg.blockDim = dim3(C::THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = gp.splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = gp.wait_prior ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gather_gemm_kernel<BN, F32, SRC, BANKS>, ma, mb, gp, In, Flt, O);
    count_launch();
    note_kernel(F32 ? "gather_gemm_kernel<f32>" : "gather_gemm_kernel<bf16>");
    return e == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

// RAW: the operand as a matrix of whole groups of eight lines, boxes of the lines of one residue in a tile of `width` rows or
// columns.  A row of that matrix ends with the last element of the group's last line, so nothing behind the operand is read.
// False when the operand has no unit stride or less than one group.
bool raw_map(CUtensorMap *map, const void *ptr, Operand &op, int mn, int k, int width) {
    const int64_t pitch = op.mn_major ? op.s_k : op.s_mn, lines = op.mn_major ? k : mn, inner = op.mn_major ? mn : k;
    if ((op.mn_major ? op.s_mn : op.s_k) != 1 || lines < 8 || pitch < inner) return false;
    op.shift = (int)(reinterpret_cast<uintptr_t>(ptr) % 16 / 2);
    op.groups = (int)(lines / 8);
    cuuint64_t dims[2] = {(cuuint64_t)(op.shift + 7 * pitch + inner), (cuuint64_t)op.groups}, strides[1] = {(cuuint64_t)(16 * pitch)};
    cuuint32_t box[2] = {(cuuint32_t)((op.mn_major ? width : 64) + 8), (cuuint32_t)((op.mn_major ? 64 : width) / 8)};
    void *base = reinterpret_cast<void *>(reinterpret_cast<uintptr_t>(ptr) & ~(uintptr_t)15);
    return tensor_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

// Tiles, their width, and the CTAs (of one cluster) that share a tile's reduction.
struct Tiles { int bn, num_kb, splits; int64_t tiles; double us; };
// By time (us): a start and an end, a k-block of every round of tiles, what a further round adds (its write-back paces it where the reduction is short), and what
// sharing a reduction costs, the less of the tile a CTA sums up and writes the less;
// 148 SMs hold 74, 33 and 15 clusters of 2, 4 and 8 CTAs at once.  Fitted to graph replays of 700 calls whose lines start anywhere, each in both widths and with
// 1 to 8 CTAs a tile: the estimates are within 6 % in the mean, the choices cost 0.1 % over the best; with one cost of sharing for all numbers of CTAs 5 %
// (9 x 11 x 11, 3x3x33x64 bf16 11.8 us by one CTA, 14.3 by two, 10.7 by four; two were taken), and without a least round 2970 x 12 x 3782 bf16 took tiles of 64 columns,
// 30.9 and 26.2.  Five k-blocks of bf16 by one CTA are five partial sums (see launch_gather), each met with the running one: 0.4 us more, with 128 columns 1.4
// (200 products of 257 to 320 values, in every width and by 1 and 2 CTAs; without it 1 x 68 x 267 was left to one CTA, 9.3 us, 7.4 by two).  (With 128 columns wherever there are
// more than 64, and only as many CTAs as fit beside one another, products took 22 % (f32) and 12 % (bf16) longer, convolutions 7 and 17:
// 3181 x 682 x 868 f32 is 150 tiles of 128 columns, two rounds, 62 us, and 275 of 64, 42 us; 155 x 172 x 1369 19.7 and 10.5.)
Tiles plan_tiles(const Problem &p, int num_sms) {
    struct Cost { double ends, round, kb, shared[3], shared_round, least_round; };
    constexpr Cost costs[2][2][2] = {      // [f32][convolution][128 columns]
        {{{5.7, 1.4, 0.64, {1.3, 0.5, 0.25}, 6.6, 2.7}, {6.5, 2.6, 0.79, {2.4, 1.1, 0.6}, 7.6, 4.6}},
         {{5.5, 1.0, 1.09, {5.0, 2.3, 1.7}, 8.5, 2.4}, {6.2, 2.2, 1.29, {8.2, 3.5, 2.6}, 14.5, 1.6}}},
        {{{5.4, 1.3, 1.20, {1.8, 0.9, 0.5}, 7.6, 2.3}, {6.0, 2.4, 1.79, {3.9, 1.4, 0.8}, 9.1, 2.5}},
         {{5.9, 1.3, 1.57, {5.0, 2.7, 1.5}, 9.6, 2.5}, {6.6, 2.1, 2.29, {8.0, 4.0, 3.0}, 12.9, 2.7}}}};
    const int num_kb = (p.K + BK - 1) / BK;
    const bool five = p.in_bf16 && p.spatial_rank == 0 && num_kb == 5;
    Tiles best{};
    best.us = 1e300;
    for (int bn = 64; bn <= (p.N > 64 ? 128 : 64); bn *= 2) {
        const Cost &c = costs[!p.in_bf16][p.spatial_rank != 0][bn == 128];
        const int64_t tiles = (int64_t)((p.M + BM - 1) / BM) * ((p.N + bn - 1) / bn);
        for (int splits = 1, log = 0; splits == 1 || (splits <= MAX_SPLIT && num_kb > 2 * splits); splits *= 2, ++log) {
            const int at_once = splits == 1 ? num_sms : splits == 2 ? num_sms / 2 : splits == 4 ? num_sms / 4 - 4 : num_sms / 8 - 3;
            const double rounds = (double)((tiles + at_once - 1) / at_once);
            const double k = c.kb * ((num_kb + splits - 1) / splits) + (five && splits == 1 ? (bn == 64 ? 0.4 : 1.4) : 0.0);
            const double us = c.ends + k + (splits == 1 ? 0.0 : c.shared[log - 1]) + (rounds - 1.0) * std::max(c.least_round, k + (splits == 1 ? c.round : c.shared_round));
            if (us < best.us) { best = Tiles{bn, num_kb, splits, tiles, us}; }
        }
    }
    return best;
}

// Below 2^21 multiply-adds the CUDA-core kernel may be the better one.
bool too_small(const Problem &p) { return (int64_t)p.M * p.N * p.K < ((int64_t)1 << 21); }

// The CUDA-core kernel by time, where its sums are accurate enough: f32's below that line (the choice makes them no less exact than one chain of products: from some 190 values of k on
// it is this kernel, 0.9e-7 for 2.7e-7 and more), and bf16's of up to
// 256 values (relative error of sums of either sign, K = 27, 127 and 255: 2.8e-8, 5.1e-8 and 6.7e-8, here 3.1e-8, 6.0e-8 and 6.8e-8).  Below the line those of up to
// 160 values, f32 8, stay there whatever the time.  6 x 35 x 35, 3x3x3x32 bf16 takes 3.7 us there and 6.6 here, 39 x 7 x 267 f32 10 and 9.  Above the line f32 stays here for its
// accuracy, not for the time: 163 x 166 x 125 8.2 us and 7.6e-8, in 32 x 32 tiles there 5.8 and 1.1e-7; 74 x 662 x 57 6.7 and 6.8e-8, 4.3 and 7.9e-8.
bool better_on_cuda_cores(const Problem &p, const void *In, const void *Flt, double us) {
    const bool small = too_small(p);
    if (p.in_bf16 ? p.K > 256 && !small : !small) return false;
    return (small && p.K <= (p.in_bf16 ? 160 : 8)) || ffma_estimate_us(p, In, Flt) <= us;
}

}  // namespace

// What the kernel for small problems competes with: the time of tiles of 128 columns wherever there are more than 64, shared by as many CTAs as fit beside one
// another.  A start and an end, rounds of tiles and their k-blocks, and what sharing a reduction costs, fitted to graph replays of 500 calls whose lines are whole
// 16-byte pieces (those that the kernel for small problems could take): within 4 to 9 %.  (Better tiles would take some of them from that kernel, which is the
// more accurate one: bf16, K = 1024, 1.1e-7 and 1.9e-7.  That costs little: of 250 products of transposed operands that the small kernel could take, the present plan's estimate
// moves four, 200 x 112 x 1520 bf16 12.5 -> 10.1 us, 328 x 480 x 1816 12.4 -> 10.8, two by 2 to 4 %.)
double gather_estimate_us(const Problem &p, int num_sms) {
    if (too_small(p)) return 1e9;
    struct Cost { double ends, kb, round, shared; };
    constexpr Cost bf16[2][2] = {{{4.7, 0.75, 0.0, 1.0}, {6.0, 0.79, 3.0, 2.3}}, {{4.9, 1.21, 0.3, 2.1}, {6.2, 1.31, 0.0, 4.9}}};      // [convolution][128 columns]
    constexpr Cost f32[2][2] = {{{4.7, 1.27, 0.0, 1.2}, {5.4, 1.87, 2.9, 3.8}}, {{6.0, 1.51, 2.9, 2.9}, {6.8, 2.21, 6.5, 6.9}}};
    Tiles t{p.N > 64 ? 128 : 64, (p.K + BK - 1) / BK, 1, 0, 0.0};
    t.tiles = (int64_t)((p.M + BM - 1) / BM) * ((p.N + t.bn - 1) / t.bn);
    while (t.splits < MAX_SPLIT && t.tiles * t.splits * 2 <= num_sms - 12 && t.num_kb >= t.splits * 8) t.splits *= 2;
    const Cost &c = (p.in_bf16 ? bf16 : f32)[p.spatial_rank != 0][t.bn == 128];
    const double rounds = t.splits > 1 ? 1.0 : (double)((t.tiles + num_sms - 1) / num_sms);
    return c.ends + (rounds - 1.0) * c.round + rounds * c.kb * (double)((t.num_kb + t.splits - 1) / t.splits) + (t.splits > 1 ? c.shared : 0.0);
}

sg_status launch_gather(const Problem &p, const void *In, const void *Flt, float *O, bool forced, cudaStream_t stream) {
    const bool conv = p.spatial_rank != 0;
    // offsets are 32-bit
    if (reach({{p.batch, p.i_n}, {(int64_t)(p.Ho - 1) * p.sh + (int64_t)(p.KH - 1) * p.dh + 1, p.i_h},
               {(int64_t)(p.Wo - 1) * p.sw + (int64_t)(p.KW - 1) * p.dw + 1, p.i_w}, {p.C, p.i_c}}) < 0 ||
        reach({{p.KH, p.k_kh}, {p.KW, p.k_kw}, {p.C, p.k_c}, {p.N, p.k_f}}) < 0) return SG_ERR_UNSUPPORTED;
    // (the lanes compute the offsets of a tile's rows and columns beyond M, N and K too, unused but in 32 bits)
    if ((int64_t)(p.N + 256) * p.k_f > 0x7fffffff || (int64_t)(p.C + 128) * std::max(p.i_c, p.k_c) > 0x7fffffff ||
        (!conv && (int64_t)(p.M + 256) * p.i_w > 0x7fffffff)) return SG_ERR_UNSUPPORTED;
    int dev = 0, num_sms = 0, pdl = -1, unused = 0;
    if (!tensor_device_info(&dev, &num_sms, &pdl, &unused)) return SG_ERR_CUDA;

    const Tiles plan = plan_tiles(p, num_sms);
    if (!forced && better_on_cuda_cores(p, In, Flt, plan.us)) return SG_ERR_UNSUPPORTED;
    GatherParams gp{};
    gp.p = p;
    const int es = p.in_bf16 ? 2 : 4;
    auto even = [](int64_t v) { return v % 2 == 0; };
    auto on = [](const void *ptr, int64_t bytes) { return reinterpret_cast<uintptr_t>(ptr) % bytes == 0; };
    // A line runs along whichever index is contiguous.  Pairs are single loads when every line starts on a multiple of two
    // elements and ends on one.
    gp.a.mn_major = !conv && p.i_c != 1 && p.i_w == 1;
    gp.a.s_mn = (int)p.i_w; gp.a.s_k = (int)p.i_c;
    gp.a.pair = on(In, 2 * es) && (gp.a.mn_major ? even(p.i_c) && even(p.M)
                                                 : p.i_c == 1 && even(p.i_w) && even(p.K) && (!conv || (even(p.C) && even(p.i_h) && even(p.i_n))));
    gp.b.mn_major = conv || p.k_f == 1 || p.k_c != 1;
    gp.b.s_mn = (int)p.k_f; gp.b.s_k = (int)p.k_c;
    gp.b.pair = on(Flt, 2 * es) && (gp.b.mn_major ? p.k_f == 1 && even(p.k_c) && even(p.N) && (!conv || (even(p.k_kw) && even(p.k_kh)))
                                                  : even(p.k_f) && even(p.K));
    gp.uniform_rows = (p.Ho == 1 || p.o_h == (int64_t)p.Wo * p.o_w) && (p.batch == 1 || p.o_n == (int64_t)p.Ho * p.Wo * p.o_w);
    gp.wait_prior = pdl == 0 ? 0 : 1;

    const int bn = plan.bn;
    const int64_t tiles = plan.tiles;
    gp.num_kb = plan.num_kb;
    gp.num_n_tiles = (p.N + bn - 1) / bn;
    if (tiles > 0x7fffffff / MAX_SPLIT) return SG_ERR_UNSUPPORTED;
    // (a tile summed as it stands must end well within the waits of the next one's MMAs, 2e9 cycles)
    if (!p.in_bf16 && tiles > num_sms && p.K > 131072) return SG_ERR_UNSUPPORTED;
    gp.num_tiles = (int)tiles;
    gp.splits = plan.splits;
    alignas(64) CUtensorMap ma = {}, mb = {};
    const bool raw = p.in_bf16 && !conv && raw_map(&ma, In, gp.a, p.M, p.K, BM) && raw_map(&mb, Flt, gp.b, p.N, p.K, bn);
    // Partial sums of bf16 products: the largest with which the error against f64 is about the CUDA-core kernel's or below it.  Relative
    // error, positive values / of either sign: chunks of 256 values 3.1e-7 / 1.9e-7, 128 1.5e-7 / 1.0e-7, 64 7.8e-8 / 5.7e-8; that
    // kernel at K = 127 7.3e-8 / 6.3e-8, 255 1.2e-7 / 9.3e-8, 511 2.1e-7 / 1.4e-7, 765 3.3e-7 / 1.7e-7, 1023 3.5e-7 / 2.1e-7.  (Smaller
    // ones cost the write-back warps time: 2049 x 2047 x 2051 57 us with 256, 65 with 128, 96 with
    // 64; but 1531 x 1021 x 765 16.6 and 16.8, and 4095 x 4095 x 127 39.8 with one accumulator, 38.8 with a bank for each k-block.)
    gp.chunk = !p.in_bf16 || gp.num_kb <= 5 ? 1 : gp.num_kb < 16 ? 2 : 4;
    const int banks = p.in_bf16 && gp.splits == 1 ? (gp.num_kb == 2 ? 2 : gp.num_kb == 3 || gp.num_kb == 4 ? 4 : 1) : 1;
#define SG_BANKS(BN_, SRC_, SLOT, SLOTS)                                                                                                     \
    (banks == 1   ? launch_variant<BN_, false, SRC_, 1>(ma, mb, gp, In, Flt, O, num_sms, SLOT, stream)                                       \
     : banks == 2 ? launch_variant<BN_, false, SRC_, 2>(ma, mb, gp, In, Flt, O, num_sms, SLOTS, stream)                                      \
                  : launch_variant<BN_, false, SRC_, 4>(ma, mb, gp, In, Flt, O, num_sms, SLOTS + 1, stream))
#define SG_GATHER(BN_, SRC_, SLOT) launch_variant<BN_, true, SRC_, 1>(ma, mb, gp, In, Flt, O, num_sms, SLOT, stream)
    if (raw) return bn == 64 ? SG_BANKS(64, RAW, 157, 200) : SG_BANKS(128, RAW, 158, 202);
    if (p.in_bf16) {
        if (conv) return bn == 64 ? SG_BANKS(64, CONVOLUTION, 149, 204) : SG_BANKS(128, CONVOLUTION, 150, 206);
        return bn == 64 ? SG_BANKS(64, LINEAR, 151, 208) : SG_BANKS(128, LINEAR, 152, 210);
    }
    if (conv) return bn == 64 ? SG_GATHER(64, CONVOLUTION, 153) : SG_GATHER(128, CONVOLUTION, 154);
    return bn == 64 ? SG_GATHER(64, LINEAR, 155) : SG_GATHER(128, LINEAR, 156);
#undef SG_BANKS
#undef SG_GATHER
}

sg_status gather_read_status(cudaStream_t stream) { return read_status_word(stream); }

}  // namespace sg
