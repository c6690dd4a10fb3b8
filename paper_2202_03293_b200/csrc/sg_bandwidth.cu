// The memory-bound 2-D kernels (Section 4.4: Copy2D, Transpose2D, ColRed2D, RowRed2D).
//
//   Copy2D       dst[i,j] = src[i,j]
//   Transpose2D  dst[j,i] = src[i,j]
//   ColRed2D     out[j] (+)= sum_i A[i,j]
//   RowRed2D     out[i] (+)= sum_j A[i,j]
//
// All four are bound by HBM traffic; the kernels differ in how they keep enough bytes in flight.
//   - Copy2D and Transpose2D, when the layout meets the TMA rules (unit column stride, 16-byte
//     aligned bases and row pitches), move tiles with TMA only, one tile per thread block, and as many
//     blocks as there are tiles.  Blocks start in order as others end, so what is in flight is one
//     window that advances through both tensors; persistent blocks, each with a ring of tiles, drift
//     apart, and the two streams then meet in the same DRAM pages less often (16384 x 12288 bf16:
//     copy 133 us with a ring per SM, so 117; transpose 143, so 123).
//     The copy never touches the data with an ordinary instruction; the transpose has
//     four warps turn each 128-row tile around in shared memory between the load and the store
//     (4-byte elements: 16-byte reads of the 128-byte swizzled input tile, a register transpose
//     of a 4 x 4 block, 16-byte writes into the swizzled output tile; 2-byte elements: 8 x 8
//     blocks through ldmatrix.trans and stmatrix).  Ragged edges cost nothing: loads
//     read zeros beyond the tensor, stores are clipped.
//   - The reductions use plain 16-byte loads with eight in flight per thread, f32 accumulators, and
//     a shared-memory / shuffle tree per CTA.  When the shape has too few independent outputs to
//     fill the chip, the reduced index is split across CTAs: up to eight ranges are one cluster
//     and meet in its shared memory, more (large tensors) meet in the output through float atomics
//     (an overwriting call clears the output first); nothing but the operands is read or written.
//     Many short rows have a kernel of their own.
//   - Any other copy or transpose (non-unit column strides, unaligned pitches) runs on
//     tile_move_kernel: dense operands as one run of 16-byte pieces, runs along the destination
//     otherwise, 32 x 32 or 64 x 64 tiles through shared memory where the source runs the other way.
#include <algorithm>
#include <utility>

#include "sg_internal.cuh"
#include "sg_tc_ptx.cuh"

namespace sg {
namespace {

// Bounded, flag-free wait used only while winding down after a time-out: lets copies that are
// still in flight land before the CTA gives its shared memory back.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
    for (int i = 0; i < (1 << 20); ++i)
        if (mbar_try_wait(bar, parity)) return;
}

// Every kernel of this file but the clearing one is launched so that it may start while the kernel ahead of it in the stream
// drains (a launch costs the host 2.4 instead of 2.9 us that way, and a small kernel's start hides behind its predecessor):
// it lets the next one start at once and waits for its predecessor before its first global access.
__device__ __forceinline__ void start_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_for_prior() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------------ Copy2D (TMA)
constexpr int CP_BOX_X = 256;             // elements of a row in a box
// Bytes of a box and thread blocks of one box each that an SM holds: 64 KB in flight per SM.  Fewer leave the memory idle, more of
// them only widen the window (16384 x 12288 bf16 / 2112 x 5952 bf16 / 640 x 15360 bf16: 5 blocks 125.6 / 9.8 / 7.7 us, 8 blocks 116.6 /
// 8.75 / 6.9, 16 blocks 118.4 / 8.7 / 6.9, 24 blocks 119.0 / 9.2 / 7.9; a ring of 32 KB stages per SM 133.4 / 9.6 / 7.7); 250 x 960 f32
// 2.3 -> 1.8.  4 and 16 KB boxes in blocks of several: 1 to 10 % slower.
constexpr int CP_BOX_BYTES = 8192;
constexpr int CP_CTAS_PER_SM = 8;

// One box per thread block: bound by HBM (16384 x 12288: 6.9 TB/s).
__global__ void __launch_bounds__(32) copy_tma_kernel(const __grid_constant__ CUtensorMap map_src, const __grid_constant__ CUtensorMap map_dst,
                                                       int tiles_x, int box_x, int box_y, uint32_t box_bytes) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar;
    __shared__ int abort_load;
    start_dependents();
    if (threadIdx.x != 0) return;
    const uint32_t box = (smem_u32(smem_raw) + 127u) & ~127u, bar = smem_u32(&full_bar);
    const int ty = (int)blockIdx.x / tiles_x, x = ((int)blockIdx.x - ty * tiles_x) * box_x, y = ty * box_y;
    mbar_init(bar, 1);
    abort_load = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_tensormap(&map_src);
    prefetch_tensormap(&map_dst);
    wait_for_prior();
    mbar_expect_tx(bar, box_bytes);
    tma_load_2d(box, &map_src, bar, x, y);
    if (!mbar_wait(bar, 0, &abort_load)) {
        mbar_drain(bar, 0);        // gave up: let the load land
        return;
    }
    tma_store_2d(&map_dst, box, x, y);
    bulk_commit();
    bulk_wait_read<0>();           // the box must stay until the store has read it; the grid's end completes the write
}

// ------------------------------------------------------------------------- Transpose2D (TMA)
// One tile = 128 input rows x 128 bytes (W = 128/ES columns), one tile per thread block.  The tile arrives as TMA writes it with
// the 128-byte swizzle (16-byte chunk index XOR row mod 8) and is turned around in place: the W x 128 transposed tile as 128/W
// blocks of [W rows][128 bytes], same swizzle, stored by four tensor stores of 32 rows each (one per warp, which also produces
// exactly those rows).  Bound by HBM and by the 128-byte rows of the requests (16384 x 12288: 6.5 TB/s).
constexpr int TR_PANEL = 8;               // tile columns per panel of the tile order (2: 126.0, 4: 125.3, 8: 123.4, 16: 124.8 us)
constexpr int TR_TILE_BYTES = 16384;
constexpr int TR_THREADS = 128;
// Thread blocks that an SM holds.  A tensor far beyond the caches wants a narrow window, one that the L2 absorbs as many tiles in flight
// as help (4 / 5 / 6 / 8 / 12 blocks: 16384 x 12288 bf16 135 / 123.4 / 125.3 / 127.5 / 129.1 us, 4736 x 3456 f32 25.1 / 23.0 / 22.9 / 23.1 / 23.3,
// 12288 x 512 f32 11.5 / 10.7 / 10.0 / 9.4 / 9.3, 640 x 15360 bf16 8.8 / 8.3 / 7.9 / 7.5 / 7.7; rings of four tiles, two per SM: 143 / 25.0 /
// 10.1 / 8.0).  Few tiles: no more than an SM's share of them, two at least, or launches that overlap deal them out unevenly (f32 2512 x 800, 500 tiles: 5.6 us with room
// for eight, 4.9 for four; 10552 x 200, 581: 6.4 and 5.9; a tile to an SM or less needs no such care).
inline int transpose_ctas_per_sm(int64_t bytes, int64_t tiles, int num_sms) {
    if (bytes >= ((int64_t)64 << 20)) return 5;
    return tiles <= num_sms ? 8 : (int)std::min<int64_t>(8, std::max<int64_t>(2, (tiles + num_sms - 1) / num_sms));
}
constexpr int ATTR_SLOT = 251;            // of tensor_ensure_smem_attr: transpose_tma_kernel<4>, <2>, tile_move_kernel<uint32_t, 32, 0>, <uint16_t, 32, 0>
constexpr int SMEM_MOST = 115 * 1024;     // two blocks to an SM
// dynamic shared memory of a block that needs `least` bytes, so that an SM holds `ctas` of them (228 KB, 1 KB of it taken per block)
inline int smem_for(int ctas, int least) { return std::max(least, (228 * 1024 / ctas - 1200) & ~127); }

// 4 x 4 block of 4-byte elements held as four 16-byte rows: the transpose is a renaming of registers.
__device__ __forceinline__ void transpose_block(const uint4 (&v)[4], uint4 (&o)[4]) {
    o[0] = make_uint4(v[0].x, v[1].x, v[2].x, v[3].x);
    o[1] = make_uint4(v[0].y, v[1].y, v[2].y, v[3].y);
    o[2] = make_uint4(v[0].z, v[1].z, v[2].z, v[3].z);
    o[3] = make_uint4(v[0].w, v[1].w, v[2].w, v[3].w);
}

// Tile order: panels of `panel` tile columns, walked row by row inside a panel.  The tiles in flight at one time then
// cover a block of the matrix rather than a thin strip of it, so that both the reads (128 bytes per row and tile) and the
// writes (128 input rows = one run of an output row per tile) fall on runs of memory that neighbouring tiles extend.
__device__ __forceinline__ void tile_coords(int t, int tiles_c, int tiles_r, int panel, int &tr, int &tc) {
    const int per_panel = panel * tiles_r;
    const int pi = t / per_panel, within = t - pi * per_panel;
    const int start = pi * panel, width = min(panel, tiles_c - start);
    tr = within / width;
    tc = start + within - tr * width;
}

template <int ES>
__global__ void __launch_bounds__(TR_THREADS) transpose_tma_kernel(const __grid_constant__ CUtensorMap map_src,
                                                                    const __grid_constant__ CUtensorMap map_dst, int tiles_c,
                                                                    int tiles_r, int panel, int dst_cols, int dst_rows) {
    constexpr int W = 128 / ES;      // input columns per tile = output rows per tile
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar;
    __shared__ int abort_turn;
    start_dependents();
    const uint32_t tile = (smem_u32(smem_raw) + 1023u) & ~1023u, bar = smem_u32(&full_bar);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int tr, tc;
    tile_coords(blockIdx.x, tiles_c, tiles_r, panel, tr, tc);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        abort_turn = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tensormap(&map_src);
        wait_for_prior();
        mbar_expect_tx(bar, TR_TILE_BYTES);
        tma_load_2d(tile, &map_src, bar, tc * W, tr * 128);
        prefetch_tensormap(&map_dst);
    }
    __syncthreads();
    wait_for_prior();
    const bool ok = mbar_wait(bar, 0, &abort_turn);
    if (!__syncthreads_and(ok)) {
        mbar_drain(bar, 0);          // gave up: let the load land
        return;
    }
    // Warp w owns store w of the tile: the 32 output rows x 128 bytes at offset w * 4 KB, which it makes of input rows 32w .. 32w+31,
    // all 32 columns (4-byte elements), or of rows 64(w/2) .. +63, columns 32(w%2) .. +31 (2-byte elements).
    const int b = w / (W / 32), h = w % (W / 32);
    if constexpr (ES == 2) {
        // 2-byte elements: the matrix load/store instructions do the turn.  Instruction i handles input rows
        // 8p .. 8p+7 (p = 8b + i) of the warp's four chunks: ldmatrix.trans hands every lane two consecutive
        // elements of a transposed 8 x 8 block per chunk, stmatrix writes those blocks as 16-byte rows.  In both,
        // the eight row addresses of a block fall on eight different swizzled chunks: no bank conflicts.
        const int m = lane >> 3, rr = lane & 7;           // this lane addresses row rr of block m
        const int qm = 4 * h + m;                         // chunk of block m
        const int c = 8 * qm + rr;                        // output row this lane addresses
        uint32_t r[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = 8 * (8 * b + i) + rr;
            const uint32_t src_addr = tile + (uint32_t)row * 128u + (uint32_t)((qm ^ rr) << 4);
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r[i][0]), "=r"(r[i][1]), "=r"(r[i][2]), "=r"(r[i][3]) : "r"(src_addr) : "memory");
        }
        __syncthreads();             // the two warps of a half read what each of them overwrites
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t dst_addr = tile + (uint32_t)b * (uint32_t)(W * 128) + (uint32_t)c * 128u + (uint32_t)((i ^ (c & 7)) << 4);
            asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};"
                         ::"r"(dst_addr), "r"(r[i][0]), "r"(r[i][1]), "r"(r[i][2]), "r"(r[i][3]) : "memory");
        }
    } else {
        // each lane turns two 4 x 4 blocks (row group p, 16-byte chunk q); a quarter-warp covers two row groups x four chunks
        const int q = (lane & 3) | ((lane >> 1) & 4);
        const int p0 = 8 * w + ((lane >> 2) & 1) + 2 * ((lane >> 4) & 1);
        uint4 v[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const int row = 4 * (p0 + 4 * i) + kk;
                const uint32_t addr = tile + (uint32_t)row * 128u + (uint32_t)((q ^ (row & 7)) << 4);
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(v[i][kk].x), "=r"(v[i][kk].y), "=r"(v[i][kk].z), "=r"(v[i][kk].w) : "r"(addr) : "memory");
            }
        __syncwarp();                // (what this warp overwrites nobody else reads)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int p = p0 + 4 * i;
            uint4 o[4];
            transpose_block(v[i], o);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = 4 * q + j;                   // output row within the tile
                const uint32_t addr = tile + (uint32_t)(p >> 3) * (uint32_t)(W * 128) + (uint32_t)c * 128u + (uint32_t)(((p & 7) ^ (c & 7)) << 4);
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(o[j].x), "r"(o[j].y), "r"(o[j].z), "r"(o[j].w) : "memory");
            }
        }
    }
    fence_async_smem();              // tile writes -> visible to the tensor store
    __syncwarp();
    if (lane == 0) {
        const int x = tr * 128 + b * W, y = tc * W + h * 32;
        if (x < dst_cols && y < dst_rows) tma_store_2d(&map_dst, tile + (uint32_t)w * 4096u, x, y);
        bulk_commit();
        bulk_wait_read<0>();
    }
}

// ------------------------------------------------------------------------- strided mover
// dst[i*d_i + j*d_j] = src[i*s_i + j*s_j]; a transpose is the same call with the destination
// strides exchanged.  MV > 0: the destination is contiguous along i, the source along j: square tiles of MV elements go through
// shared memory, a warp reads runs along j and writes runs along i.  Otherwise runs along j on both sides, straight from registers
// (dense operands arrive here flattened, in units of 16 bytes, with up to 15 bytes left over that block 0 moves).  MV: side of a
// tile, 64, or 32 while those are too few; 0: no turn.  (With a turn KC says how tiles are loaded, see launch_tile_move.)
// Every thread has sixteen or up to eight loads in flight: with four, and 32 x 32 tiles, an unaligned 16383 x 12287 transpose
// ran at 2.4 TB/s.
// Without a turn: cw = 2^cw_log threads side by side along j, 256 / cw rows of them; a thread moves kr x KC elements, KC of them
// 256 columns apart (1, 2 or 4; more than one only where cw is 256), kr <= 8 / KC of them 256 / cw rows apart.  (Narrow rows are
// why: with 2048 columns of one row as the only shape 1M x 3 f32 of pitch 4 took 1.8 ms; now 7 us.)
struct Straight {
    int cw_log, kr;
};
// Loads one element (2 or 4 bytes) if it exists, else 0.  Such loads go out back to back, whatever the compiler makes of the registers (behind branches 16383 x 6001 f32 took
// 149 us, so 139).
template <typename U>
__device__ __forceinline__ void load_if(bool exists, const U *p, uint32_t &v) {
    if constexpr (sizeof(U) == 4)
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.u32 %0, 0;\n\t@q ld.global.u32 %0, [%1];\n\t}" : "=&r"(v) : "l"(p), "r"((uint32_t)exists) : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.u32 %0, 0;\n\t@q ld.global.u16 %0, [%1];\n\t}" : "=&r"(v) : "l"(p), "r"((uint32_t)exists) : "memory");
}
template <typename U, int MV, int KC>
__global__ void __launch_bounds__(256) tile_move_kernel(const U *__restrict__ src, int64_t s_i, int64_t s_j, U *__restrict__ dst,
                                                         int64_t d_i, int64_t d_j, int R, int C, int tiles_i, int tiles_j, int panel,
                                                         Straight shape, const uint8_t *tail_src, uint8_t *tail_dst, int tail_bytes) {
    start_dependents();
    wait_for_prior();
    if constexpr (MV > 0) {
        constexpr int H = MV / 32, K = MV / 8;
        __shared__ U tile[MV][MV + (sizeof(U) == 2 ? 2 : 1)];
        const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
        int ti, tj;
        tile_coords(blockIdx.x, tiles_j, tiles_i, panel, ti, tj);
        const int i0 = ti * MV, j0 = tj * MV;
        uint32_t v[H * K];
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int i = i0 + ty + 8 * k, j = j0 + tx + 32 * h;
                if constexpr (KC == 1) {
                    if (i < R && j < C) v[H * k + h] = src[(int64_t)i * s_i + (int64_t)j * s_j];
                } else {
                    load_if(i < R && j < C, src + (int64_t)i * s_i + (int64_t)j * s_j, v[H * k + h]);
                }
            }
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int h = 0; h < H; ++h) tile[ty + 8 * k][tx + 32 * h] = (U)v[H * k + h];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const int i = i0 + tx + 32 * h, j = j0 + ty + 8 * k;
                if (i < R && j < C) dst[(int64_t)i * d_i + (int64_t)j * d_j] = tile[tx + 32 * h][ty + 8 * k];
            }
    } else {
        constexpr int KR = 8 / KC;
        const int cw_log = KC > 1 ? 8 : shape.cw_log, cw = 1 << cw_log, rows_log = 8 - cw_log, rows = 1 << rows_log;
        const int64_t s_row = rows * s_i, s_col = 256 * s_j, d_row = rows * d_i, d_col = 256 * d_j;
        // (blockIdx.y walks along i, blockIdx.x along j: a division here would cost a small call a tenth of its time)
        for (int64_t i0 = (int64_t)blockIdx.y * (rows * shape.kr); i0 < R; i0 += (int64_t)gridDim.y * (rows * shape.kr))
        for (int64_t j0 = (int64_t)blockIdx.x * (cw * KC); j0 < C; j0 += (int64_t)gridDim.x * (cw * KC)) {
            const int i = (int)i0 + ((int)threadIdx.x >> cw_log), j = (int)j0 + ((int)threadIdx.x & (cw - 1));
            // how many of the thread's rows and columns exist
            const int nr = i < R ? min(shape.kr, ((R - 1 - i) >> rows_log) + 1) : 0, nc = j < C ? min(KC, ((C - 1 - j) >> 8) + 1) : 0;
            const U *s = src + i * s_i + j * s_j;
            U *d = dst + i * d_i + j * d_j;
            U v[8];
#pragma unroll
            for (int r = 0; r < KR; ++r)
#pragma unroll
                for (int c = 0; c < KC; ++c)
                    if (r < nr && c < nc) v[r * KC + c] = s[r * s_row + c * s_col];
#pragma unroll
            for (int r = 0; r < KR; ++r)
#pragma unroll
                for (int c = 0; c < KC; ++c)
                    if (r < nr && c < nc) d[r * d_row + c * d_col] = v[r * KC + c];
        }
        if (blockIdx.x + blockIdx.y == 0 && threadIdx.x < tail_bytes) tail_dst[threadIdx.x] = tail_src[threadIdx.x];
    }
}

// --------------------------------------------------------------------------------- reductions
inline bool aligned16(const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

__device__ __forceinline__ float widen(float x) { return x; }
__device__ __forceinline__ float widen(uint16_t bits) { return __uint_as_float((uint32_t)bits << 16); }

// One whole chunk (VEC > 1: 16 bytes at an aligned address), added element-wise into acc.
template <typename T, int VEC>
__device__ __forceinline__ void accumulate_raw(float (&acc)[VEC], const uint4 &raw) {
    if constexpr (VEC == 4) {
        acc[0] += __uint_as_float(raw.x); acc[1] += __uint_as_float(raw.y);
        acc[2] += __uint_as_float(raw.z); acc[3] += __uint_as_float(raw.w);
    } else if constexpr (VEC == 8) {
        const uint32_t wds[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            acc[2 * w] += __uint_as_float(wds[w] << 16);
            acc[2 * w + 1] += __uint_as_float(wds[w] & 0xFFFF0000u);
        }
    }
}

// How the partial sums of a reduction whose reduced index is cut in `splits` ranges (blockIdx.y) meet.
//   DIRECT   one range.
//   CLUSTER  the ranges of an output are one thread-block cluster (at most eight); its blocks add each other's shared-memory
//            sums up in rank order: one launch, a fixed order.
//   ATOMIC   any number of ranges, float atomics on the output (ATOMIC_V4: dense and aligned, four at a time).
// `cleared`: the launch runs behind the kernel that clears the output and may have started beside it; the loads need not
// wait for that kernel, the atomics must.
enum { DIRECT = 0, CLUSTER = 1, ATOMIC = 2, ATOMIC_V4 = 3 };
struct Meeting {
    int how, cleared, accumulate;
};
__device__ __forceinline__ float remote_float(uint32_t addr, int rank) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(map_to_cta(addr, (uint32_t)rank)) : "memory");
    return v;
}

// Rows r, r+rp, ... < r1 of one chunk, eight loads in flight.  FULL: the chunk has all VEC columns (16-byte loads).
template <typename T, int VEC, bool FULL>
__device__ __forceinline__ void colred_walk(float (&acc)[VEC], const T *base, int64_t ld, int64_t sc, int64_t r, int64_t r1, int rp,
                                            int nvalid, bool few) {
    constexpr int U = 8;
    if constexpr (FULL && VEC > 1) {
        // all eight 16-byte loads are issued before the first is consumed
        for (; r + (U - 1) * rp < r1; r += U * rp) {
            uint4 raw[U];
#pragma unroll
            for (int u = 0; u < U; ++u) raw[u] = __ldg(reinterpret_cast<const uint4 *>(base + (r + u * rp) * ld));
#pragma unroll
            for (int u = 0; u < U; ++u) accumulate_raw<T, VEC>(acc, raw[u]);
        }
        if (few) {      // (at most one row a thread: seven empty additions would cost more than the load)
            if (r < r1) accumulate_raw<T, VEC>(acc, __ldg(reinterpret_cast<const uint4 *>(base + r * ld)));
            return;
        }
        if (r >= r1) return;
        uint4 raw[U];
#pragma unroll
        for (int u = 0; u < U; ++u) raw[u] = r + u * rp < r1 ? __ldg(reinterpret_cast<const uint4 *>(base + (r + u * rp) * ld)) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < U; ++u) accumulate_raw<T, VEC>(acc, raw[u]);
    } else {
        for (; r + (U - 1) * rp < r1; r += U * rp) {
            float part[U];
#pragma unroll
            for (int u = 0; u < U; ++u) part[u] = 0.f;
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                if (v < nvalid) {
#pragma unroll
                    for (int u = 0; u < U; ++u) part[u] = widen(__ldg(base + (r + u * rp) * ld + (int64_t)v * sc));
                    acc[v] += ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
                }
            }
        }
        for (; r < r1; r += rp)
#pragma unroll
            for (int v = 0; v < VEC; ++v)
                if (v < nvalid) acc[v] += widen(__ldg(base + r * ld + (int64_t)v * sc));
    }
}

// ColRed2D.  A CTA owns `cw` chunks of VEC columns (a power of two, or at least 32) and the rows [r0, r1) of its range;
// thread (g, cc) = (t / cw, t % cw) walks rows r0+g, r0+g+rp, ... of chunk cc.
template <typename T, int VEC>
__global__ void __launch_bounds__(256) colred_kernel(const T *__restrict__ A, int64_t ld, int64_t sc, int R, int C,
                                                      float *__restrict__ out, int64_t os, int cw, int rp, int rows_per_split, Meeting meet) {
    __shared__ float red[256][VEC + 1];
    start_dependents();
    if (!meet.cleared) wait_for_prior();
    const int t = threadIdx.x, g = t / cw, cc = t - g * cw;
    const int64_t col0 = ((int64_t)blockIdx.x * cw + cc) * VEC;
    const int64_t r0 = (int64_t)blockIdx.y * rows_per_split;
    const int64_t r1 = min((int64_t)R, r0 + rows_per_split);
    float acc[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    const bool active = g < rp && col0 < C;
    const int nvalid = active ? (int)min((int64_t)VEC, (int64_t)C - col0) : 0;
    if (active) {
        const T *base = A + col0 * sc;
        if (nvalid == VEC) colred_walk<T, VEC, true>(acc, base, ld, sc, r0 + g, r1, rp, VEC, r1 - r0 <= rp);
        else colred_walk<T, VEC, false>(acc, base, ld, sc, r0 + g, r1, rp, nvalid, false);
    }
    // a warp that holds several row groups of a chunk adds them up first: one group per warp is left
    const bool fold = cw < 32 && (cw & (cw - 1)) == 0;
    for (int off = fold ? 16 : 0; off >= cw; off >>= 1)
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
    const int groups = fold ? 8 : rp;
    const int slot = fold ? ((t & 31) < cw ? (t >> 5) * cw + (t & 31) : -1) : t;
    if (slot >= 0)
#pragma unroll
        for (int v = 0; v < VEC; ++v) red[slot][v] = acc[v];
    __syncthreads();
    if (meet.how == CLUSTER) {
        // every block's sums of a column in red[chunk][v], then output o of the chunks by block o / 256 mod splits
        for (int o = t; o < cw * VEC; o += 256) {
            const int c = o / VEC, v = o - c * VEC;
            float s = red[c][v];
            for (int gg = 1; gg < groups; ++gg) s += red[gg * cw + c][v];
            red[c][v] = s;
        }
        cluster_sync_all();
        const int splits = (int)gridDim.y, rank = (int)blockIdx.y;
        for (int o = rank * 256 + t; o < cw * VEC; o += splits * 256) {
            const int c = o / VEC, v = o - c * VEC;
            const int64_t col = ((int64_t)blockIdx.x * cw + c) * VEC + v;
            if (col >= C) continue;
            float part[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) part[s] = s < splits ? remote_float(smem_u32(&red[c][v]), s) : 0.f;
            float sum = part[0];
#pragma unroll
            for (int s = 1; s < 8; ++s) sum += part[s];
            float *dst = out + col * os;
            *dst = (meet.accumulate ? *dst : 0.f) + sum;
        }
        cluster_sync_all();       // nobody leaves while its sums are being read
        return;
    }
    if (meet.cleared) wait_for_prior();
    if (t < cw && col0 < C) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[v] = red[t][v];
        for (int gg = 1; gg < groups; ++gg)
#pragma unroll
            for (int v = 0; v < VEC; ++v) acc[v] += red[gg * cw + cc][v];
        if (VEC >= 4 && meet.how == ATOMIC_V4 && nvalid == VEC) {
            // dense, 16-byte aligned output: four sums per atomic
#pragma unroll
            for (int v = 0; v < VEC; v += 4)
                asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(out + col0 + v), "f"(acc[v]), "f"(acc[(v + 1) % VEC]),
                             "f"(acc[(v + 2) % VEC]), "f"(acc[(v + 3) % VEC]) : "memory");
            return;
        }
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            if (v < nvalid) {
                float *o = out + (col0 + v) * os;
                if (meet.how >= ATOMIC) atomicAdd(o, acc[v]);
                else *o = (meet.accumulate ? *o : 0.f) + acc[v];
            }
        }
    }
}

// RowRed2D.  `threads` (a power of two <= 256) threads share a row; blockIdx.y selects the column range [c0, c1) of a split.
// VEC > 1: unit column stride; the elements ahead of the first and behind the last 16-byte boundary of the row are added one
// by one (rows may start anywhere).
template <typename T, int VEC>
__global__ void __launch_bounds__(256) rowred_kernel(const T *__restrict__ A, int64_t ld, int64_t sc, int R, int C,
                                                      float *__restrict__ out, int64_t os, int threads, int cols_per_split, Meeting meet) {
    __shared__ float red[8];
    start_dependents();
    if (!meet.cleared) wait_for_prior();
    const int rows_per_cta = 256 / threads;
    const int64_t row = (int64_t)blockIdx.x * rows_per_cta + threadIdx.x / threads;
    const int sub = threadIdx.x % threads;
    const int64_t c0 = (int64_t)blockIdx.y * cols_per_split;
    const int64_t c1 = min((int64_t)C, c0 + cols_per_split);
    float acc[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    if (row < R && c0 < c1) {
        const T *base = A + row * ld;
        if constexpr (VEC > 1) {
            const int64_t head = min(c1 - c0, (int64_t)((16 - (reinterpret_cast<uintptr_t>(base + c0) & 15)) & 15) / (int64_t)sizeof(T));
            const int64_t body0 = c0 + head, body1 = body0 + (c1 - body0) / VEC * VEC;
            const int64_t step = (int64_t)threads * VEC;
            int64_t c = body0 + sub * VEC;
            for (; c + 7 * step < body1; c += 8 * step) {      // eight 16-byte loads in flight
                uint4 raw[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) raw[u] = __ldg(reinterpret_cast<const uint4 *>(base + c + u * step));
#pragma unroll
                for (int u = 0; u < 8; ++u) accumulate_raw<T, VEC>(acc, raw[u]);
            }
            if (c < body1) {
                uint4 raw[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) raw[u] = c + u * step < body1 ? __ldg(reinterpret_cast<const uint4 *>(base + c + u * step)) : make_uint4(0, 0, 0, 0);
#pragma unroll
                for (int u = 0; u < 8; ++u) accumulate_raw<T, VEC>(acc, raw[u]);
            }
            for (int64_t e = sub; e < head + (c1 - body1); e += threads)
                acc[0] += widen(__ldg(base + (e < head ? c0 + e : body1 + (e - head))));
        } else {
            const int64_t step = threads;
            int64_t c = c0 + sub;
            for (; c + 7 * step < c1; c += 8 * step) {
                float part[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) part[u] = widen(__ldg(base + (c + u * step) * sc));
                acc[0] += ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
            }
            for (; c < c1; c += step) acc[0] += widen(__ldg(base + c * sc));
        }
    }
    float sum = acc[0];
#pragma unroll
    for (int v = 1; v < VEC; ++v) sum += acc[v];
    for (int off = min(threads, 32) >> 1; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (threads > 32) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
        __syncthreads();
        if (sub == 0)
            for (int w = 1; w < threads / 32; ++w) sum += red[(threadIdx.x >> 5) + w];
    }
    if (meet.how == CLUSTER) {       // (one row per block)
        if (threadIdx.x == 0) red[0] = sum;
        cluster_sync_all();
        if (blockIdx.y == 0 && threadIdx.x == 0) {
            sum = 0.f;
            for (int s = 0; s < (int)gridDim.y; ++s) sum += remote_float(smem_u32(&red[0]), s);
            float *o = out + row * os;
            *o = (meet.accumulate ? *o : 0.f) + sum;
        }
        cluster_sync_all();
        return;
    }
    if (meet.cleared) wait_for_prior();
    if (sub == 0 && row < R && (c0 < c1 || blockIdx.y == 0)) {
        float *o = out + row * os;
        if (meet.how >= ATOMIC) atomicAdd(o, sum);
        else *o = (meet.accumulate ? *o : 0.f) + sum;
    }
}

// RowRed2D, many short rows: `threads` (a power of two <= 32) threads share a row and have two chunks of it each at most; a block takes
// several groups of rows in turn, since starting one costs more than the rows it sums (every other one of 16 columns of 1M rows, f32:
// one group per block 49 us, so 25).
template <typename T, int VEC>
__global__ void __launch_bounds__(256) rowred_short_kernel(const T *__restrict__ A, int64_t ld, int64_t sc, int R, int C, float *__restrict__ out, int64_t os,
                                                            int threads_log, int accumulate) {
    start_dependents();
    wait_for_prior();
    const int threads = 1 << threads_log, rows = 256 >> threads_log, sub = threadIdx.x & (threads - 1);
    for (int64_t row0 = (int64_t)blockIdx.x * rows; row0 < R; row0 += (int64_t)gridDim.x * rows) {
        const int64_t row = row0 + (threadIdx.x >> threads_log);
        float acc[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
        if (row < R) {
            const T *base = A + row * ld;
            if constexpr (VEC > 1) {
                const int head = min(C, (int)((16 - (reinterpret_cast<uintptr_t>(base) & 15)) & 15) / (int)sizeof(T));
                const int end = head + (C - head) / VEC * VEC;
                for (int c = head + sub * VEC; c < end; c += threads * VEC) accumulate_raw<T, VEC>(acc, __ldg(reinterpret_cast<const uint4 *>(base + c)));
                for (int e = sub; e < head + (C - end); e += threads) acc[0] += widen(__ldg(base + (e < head ? e : end + (e - head))));
            } else {
                for (int c = sub; c < C; c += threads) acc[0] += widen(__ldg(base + c * sc));
            }
        }
        float sum = acc[0];
#pragma unroll
        for (int v = 1; v < VEC; ++v) sum += acc[v];
        for (int off = threads >> 1; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if (sub == 0 && row < R) {
            float *o = out + row * os;
            *o = (accumulate ? *o : 0.f) + sum;
        }
    }
}

__global__ void zero_vector_kernel(float *__restrict__ out, int64_t n, int64_t os) {
    wait_for_prior();
    start_dependents();       // the reduction behind it may start (everything ahead has finished); it waits before its atomics
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) out[i * os] = 0.f;
}

// Launches `kernel` so that it may start while the kernel ahead of it drains; `cluster`: blocks of a cluster along y.
template <typename... KArgs, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(KArgs...), dim3 grid, int block, int smem, int cluster, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = cluster; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
inline cudaError_t launch_clear(float *out, int64_t n, int64_t os, cudaStream_t stream) {
    return launch_overlapped(zero_vector_kernel, dim3((unsigned)std::min<int64_t>((n + 255) / 256, 1184)), 256, 0, 1, stream, out, n, os);
}

template <typename T, int VEC>
cudaError_t launch_reduce_typed(bool colred, const T *A, int64_t ld, int64_t sc, int R, int C, float *out, int64_t os,
                                int accumulate, int num_sms, bool vec_name, cudaStream_t stream) {
    // one thread block per batch of eight 16-byte loads per thread: more blocks than this would not even do that
    const int64_t batches = std::max<int64_t>(1, (int64_t)R * ((C + VEC - 1) / VEC) / (256 * 8));
    if (!colred) {
        // RowRed2D, one output per row, `threads` per row: of the powers of two the one with the least (waves of thread blocks) x
        // (loads of a thread + eight loads' worth of latency).  Long rows of matrices that do not fill the chip are cut in up to
        // eight ranges of a cluster, and beyond that by atomics.
        const int chunks = (C + VEC - 1) / VEC;
        int threads = 1, threads_log = 0;
        double best = 1e30;
        for (int t = 1, l = 0; t <= 256 && (t == 1 || t / 2 < chunks); t <<= 1, ++l) {
            const double x = (double)(((int64_t)R + 256 / t - 1) / (256 / t)) / (6 * num_sms);
            const double cost = (x <= 1 ? 1 : x <= 2 ? 2 : x) * (8 + (chunks + t - 1) / t) * (t < 8 ? 16 / t : 1);      // (rows below 128 bytes a request)
            if (cost < best) { best = cost; threads = t; threads_log = l; }
        }
        const int64_t row_ctas = ((int64_t)R + 256 / threads - 1) / (256 / threads);
        int splits = 1;
        Meeting meet{DIRECT, 0, accumulate};
        if (threads == 256 && row_ctas < 4 * num_sms && chunks > 256 * 8) {
            const int64_t want = std::min<int64_t>((4 * num_sms + row_ctas - 1) / row_ctas, (chunks + 256 * 8 - 1) / (256 * 8));
            splits = 1;
            while (splits < want && splits < 8) splits <<= 1;
            meet.how = CLUSTER;
            if (want > 16) { splits = (int)want; meet.how = ATOMIC; }
        }
        int chunks_per_split = (chunks + splits - 1) / splits;
        if (meet.how == ATOMIC) splits = (chunks + chunks_per_split - 1) / chunks_per_split;
        if (splits == 1) meet.how = DIRECT;
        if (meet.how == ATOMIC && !accumulate) {
            const cudaError_t e = launch_clear(out, R, os, stream);
            if (e != cudaSuccess) return e;
            meet.cleared = 1;
        }
        if (meet.how == DIRECT && threads <= 32 && chunks <= 2 * threads && row_ctas > 32 * num_sms) {
            note_kernel(vec_name ? "rowred_short_kernel<vec>" : "rowred_short_kernel<scalar>");
            return launch_overlapped(rowred_short_kernel<T, VEC>, dim3(32 * num_sms), 256, 0, 1, stream, A, ld, sc, R, C, out, os, threads_log, accumulate);
        }
        note_kernel(vec_name ? "rowred_kernel<vec>" : "rowred_kernel<scalar>");
        return launch_overlapped(rowred_kernel<T, VEC>, dim3((unsigned)row_ctas, (unsigned)splits), 256, 0, meet.how == CLUSTER ? splits : 1, stream,
                                 A, ld, sc, R, C, out, os, threads, chunks_per_split * VEC, meet);
    }
    // ColRed2D, one output per column
    const int64_t chunks = ((int64_t)C + VEC - 1) / VEC;
    note_kernel(vec_name ? "colred_kernel<vec>" : "colred_kernel<scalar>");
    static const int resident = [] {
        int n = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, colred_kernel<T, VEC>, 256, 0) == cudaSuccess && n > 0 ? n : 2;
    }();
    const int64_t wave = (int64_t)num_sms * resident;
    // Up to 48 MB (element by element 4): clusters of up to eight row ranges over the widest column blocks that fill most of a wave: one launch, no
    // atomics.  (Larger tensors stream better in whole rows, and the second launch no longer matters.)
    if ((int64_t)R * C * (int64_t)sizeof(T) < ((int64_t)(VEC > 1 ? 48 : 4) << 20)) {
        const double target = 0.6 * (double)std::min<int64_t>(wave, batches);
        for (int cw = 256; cw >= 8; cw >>= 1) {
            if (cw > 8 && cw / 2 >= chunks) continue;                   // half of the chunk lanes would be idle
            const int rp = 256 / cw;
            const int64_t col_blocks = (chunks + cw - 1) / cw;
            const int splits = (int)std::max<int64_t>(1, std::min<int64_t>({8, wave / col_blocks, ((int64_t)R + rp * 8 - 1) / (rp * 8)}));
            if ((double)(col_blocks * splits) < target) continue;
            const Meeting meet{splits > 1 ? CLUSTER : DIRECT, 0, accumulate};
            return launch_overlapped(colred_kernel<T, VEC>, dim3((unsigned)col_blocks, (unsigned)splits), 256, 0, splits, stream, A, ld, sc, R, C, out,
                                     os, cw, rp, (R + splits - 1) / splits, meet);
        }
    }
    // row ranges: as many as give every SM its full set of resident thread blocks, in one wave
    const int cw = (int)std::min<int64_t>(chunks, 256);
    const int rp = 256 / cw;
    const int64_t col_blocks = (chunks + cw - 1) / cw;
    int splits = 1;
    const int min_rows_per_split = rp * 16;
    if (col_blocks < wave && R > min_rows_per_split)
        splits = (int)std::min<int64_t>(wave / col_blocks, ((int64_t)R + min_rows_per_split - 1) / min_rows_per_split);
    int rows_per_split = (R + splits - 1) / splits;
    rows_per_split = (rows_per_split + rp - 1) / rp * rp;
    splits = (R + rows_per_split - 1) / rows_per_split;
    Meeting meet{splits == 1 ? DIRECT : (os == 1 && aligned16(out)) ? ATOMIC_V4 : ATOMIC, 0, accumulate};
    if (meet.how >= ATOMIC && !accumulate) {
        const cudaError_t e = launch_clear(out, C, os, stream);
        if (e != cudaSuccess) return e;
        meet.cleared = 1;
    }
    return launch_overlapped(colred_kernel<T, VEC>, dim3((unsigned)col_blocks, (unsigned)splits), 256, 0, 1, stream, A, ld, sc, R, C, out, os, cw, rp,
                             rows_per_split, meet);
}

// Runs along j on both sides.  Narrow rows: a power of two of threads covers one; wide rows: up to four elements of one per thread, of
// up to eight in all.  Fewer elements a thread where that leaves SMs idle.  Wide rows of 4 bytes or more: a thread block for every
// piece; they start in order as others end, and reads and writes each advance in one window (dense 16383 x 12287 bf16 / f32 16383 x 6001:
// four waves of blocks that walk on 125.0 / 121.5 us, so 117.6 / 114.8; every other column of 12288 x 16384 f32 185 and 174, in one
// wave 217).  Pieces of 4 KB, or of narrow rows, are too little for a block of their own: four waves (8192 x 8192 bf16 of odd pitch 85 us,
// a block each 89.2; 4M x 3 f32 of pitch 4 24.8 and 26.1).
template <typename U>
cudaError_t launch_straight(const U *src, int64_t s_i, int64_t s_j, U *dst, int64_t d_i, int64_t d_j, int R, int C, int num_sms, cudaStream_t stream,
                            const uint8_t *tail_src, uint8_t *tail_dst, int tail_bytes) {
    constexpr int MOST = 4;
    Straight t{0, 1};
    int kc = 1;
    while (t.cw_log < 8 && (1 << t.cw_log) < C) ++t.cw_log;
    while (kc < MOST && 256 * kc < C) kc *= 2;
    t.kr = 8 / kc;
    int64_t units_i, units_j;
    for (;;) {
        const int64_t block_r = (int64_t)(256 >> t.cw_log) * t.kr, block_c = ((int64_t)1 << t.cw_log) * kc;
        units_i = (R + block_r - 1) / block_r;
        units_j = (C + block_c - 1) / block_c;
        if (units_i * units_j >= num_sms || (t.kr == 1 && kc == 1)) break;
        if (t.kr > 1) t.kr /= 2;
        else kc /= 2;
    }
    using Kernel = void (*)(const U *, int64_t, int64_t, U *, int64_t, int64_t, int, int, int, int, int, Straight, const uint8_t *, uint8_t *, int);
    const Kernel kernel = kc == 1 ? tile_move_kernel<U, 0, 1> : kc == 2 ? tile_move_kernel<U, 0, 2> : tile_move_kernel<U, 0, MOST>;
    const bool all = sizeof(U) >= 4 && t.cw_log == 8;
    const int64_t most = (int64_t)num_sms * 8 * 4;
    const int64_t grid_i = std::min<int64_t>({units_i, 65535, all ? 65535 : std::max<int64_t>(1, most / std::min<int64_t>(units_j, 32))});
    return launch_overlapped(kernel, dim3((unsigned)(all ? units_j : std::min(units_j, most / grid_i)), (unsigned)grid_i), 256, 0, 1, stream, src, s_i, s_j, dst, d_i,
                             d_j, R, C, 0, 0, 0, t, tail_src, tail_dst, tail_bytes);
}

template <typename U>
cudaError_t launch_tile_move(const U *src, int64_t s_i, int64_t s_j, U *dst, int64_t d_i, int64_t d_j, int R, int C, int num_sms,
                             cudaStream_t stream, bool note = true) {
    if (note) note_kernel("tile_move_kernel");
    // j: the index along which the destination is closer to contiguous
    if (C == 1 ? R > 1 : R > 1 && d_i < d_j) { std::swap(s_i, s_j); std::swap(d_i, d_j); std::swap(R, C); }
    if (std::min(R, C) >= 32 && s_i != 0 && s_i < s_j) {
        // the source runs along the other one: tiles turn around (4096 x 4096 f32 column-major to row-major: 77 us read across, 31 so)
        std::swap(s_i, s_j); std::swap(d_i, d_j); std::swap(R, C);
        const int mv = (int64_t)((R + 63) / 64) * ((C + 63) / 64) < 2 * num_sms ? 32 : 64;
        const int tiles_i = (R + mv - 1) / mv, tiles_j = (C + mv - 1) / mv;
        if ((int64_t)tiles_i * tiles_j > 0x7fffffff) return cudaErrorInvalidConfiguration;
        // a thread block per tile (eight per SM that walk on: 16383 x 6001 f32 201 us, so 139; 4737 x 3457 33.0 and 25.1; 16383 x 12287 bf16 315 and 242).
        // Few of them: shared memory that nobody uses keeps an SM to its share of the blocks, which would otherwise go where the launch ahead left
        // room (512 x 4001 bf16 6.8 us, so 4.7; f32 801 x 603 3.06 and 2.46).  Two of the smaller tiles to an SM from a quarter more of them than SMs on (tiles of f32 for each SM,
        // without / for two / for four: 1.1 0.91 / 0.97 / 1.05 of eight blocks that walk on, 1.4 0.94 / 0.88 / 0.96, 1.6 0.91 / 0.83 / 0.99, 1.9 0.90 / 0.82 / 0.89), else four at
        // least.  Not for larger tiles of 4 bytes beyond five to an SM (3001 x 1201 f32 8.1, with six 9.0).  Those with five to six to an SM load behind branches, which takes
        // 40 registers: an SM then has room for six of them and as much L1 as before (760 x 4168 8.0 us, so 7.3; outside that range 1 to 15 % slower).
        const int64_t tiles = (int64_t)tiles_i * tiles_j;
        const int taken = mv * (mv + (sizeof(U) == 2 ? 2 : 1)) * (int)sizeof(U);
        const bool two = mv == 32 && 4 * tiles > 5 * num_sms && tiles <= 2 * num_sms;
        const int share = (int)std::max<int64_t>(two ? 2 : 4, (tiles + num_sms - 1) / num_sms);
        const bool even = two || (tiles > 2 * num_sms && share < (mv == 64 && sizeof(U) == 4 ? 6 : 8));
        const int spare = even ? std::min(smem_for(share, 0), two ? SMEM_MOST : 48 * 1024) - taken : 0;
        if (two && !tensor_ensure_smem_attr(ATTR_SLOT + (sizeof(U) == 4 ? 2 : 3), reinterpret_cast<const void *>(tile_move_kernel<U, 32, 0>), SMEM_MOST - taken))
            return cudaErrorInvalidConfiguration;
        constexpr int BRANCHES = sizeof(U) == 4 ? 1 : 0;
        const bool branches = mv == 64 && tiles > 5 * num_sms && tiles <= 6 * num_sms;
        return launch_overlapped(mv == 32 ? tile_move_kernel<U, 32, 0> : branches ? tile_move_kernel<U, 64, BRANCHES> : tile_move_kernel<U, 64, 0>, dim3((unsigned)tiles), 256, spare, 1, stream, src, s_i, s_j, dst, d_i,
                                 d_j, R, C, tiles_i, tiles_j, std::min(tiles_j, TR_PANEL), Straight{}, (const uint8_t *)nullptr, (uint8_t *)nullptr, 0);
    }
    const int64_t bytes = (int64_t)R * C * (int64_t)sizeof(U);
    if (s_j == 1 && d_j == 1 && (R == 1 || (s_i == C && d_i == C)) && aligned16(src) && aligned16(dst) && bytes >= 16 && bytes / 16 < 0x7fffffff) {
        // dense on both sides: one run of memory
        const int n16 = (int)(bytes / 16), tail = (int)(bytes % 16);
        return launch_straight(reinterpret_cast<const uint4 *>(src), 0, 1, reinterpret_cast<uint4 *>(dst), 0, 1, 1, n16, num_sms, stream,
                               reinterpret_cast<const uint8_t *>(src) + (int64_t)n16 * 16, reinterpret_cast<uint8_t *>(dst) + (int64_t)n16 * 16, tail);
    }
    return launch_straight(src, s_i, s_j, dst, d_i, d_j, R, C, num_sms, stream, nullptr, nullptr, 0);
}

}  // namespace

sg_status launch_move2d(bool transpose, int64_t R, int64_t C, const void *src, int64_t s_r, int64_t s_c, void *dst, int64_t d_r,
                        int64_t d_c, int esize, int force, int *used_tma, cudaStream_t stream) {
    *used_tma = 0;
    int num_sms = 0;
    if (!tensor_driver_ready(&num_sms)) return SG_ERR_CUDA;
    const bool tma_ok = force != 1 && s_c == 1 && d_c == 1 && aligned16(src) && aligned16(dst) && (s_r * esize) % 16 == 0 &&
                        (d_r * esize) % 16 == 0 && s_r * esize < ((int64_t)1 << 40) && d_r * esize < ((int64_t)1 << 40) &&
                        (R == 1 || s_r >= C) && ((transpose ? C : R) == 1 || d_r >= (transpose ? R : C));
    const CUtensorMapDataType type = esize == 4 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16;
    // TMA checks the bounds of the contiguous dimension in 16-byte units, so a store would write the rest of the unit
    // in which a row of the destination ends: the TMA kernels take the part whose destination rows are whole units
    // (`body`), the strided kernel the last few columns of the destination.
    const int vec = 16 / esize;
    const int64_t inner = transpose ? R : C;             // extent of the destination's contiguous dimension
    const int64_t body = inner - inner % vec, tail = inner - body;
    if (tma_ok && body > 0 && (tail == 0 || force != 2)) {
        int64_t Rb = transpose ? body : R, Cb = transpose ? C : body;      // the source part the TMA kernel moves
        bool launched = false;
        CUtensorMap map_src, map_dst;
        cuuint64_t st_src[1] = {(cuuint64_t)(s_r * esize)}, st_dst[1] = {(cuuint64_t)(d_r * esize)};
        if (!transpose) {
            // dense on both sides: one run of memory, in rows of 256 elements
            if ((R == 1 || (s_r == C && d_r == C)) && (R * C) % CP_BOX_X == 0 && R * C / CP_BOX_X < 0x7fffffff) {
                Rb = R * C / CP_BOX_X;
                Cb = CP_BOX_X;
                st_src[0] = st_dst[0] = (cuuint64_t)(CP_BOX_X * esize);
            }
            // box: up to 256 elements wide, as many rows as CP_BOX_BYTES hold
            const int box_x = (int)std::min<int64_t>(CP_BOX_X, Cb);
            int box_y = (int)std::min<int64_t>(std::min<int64_t>(256, CP_BOX_BYTES / (box_x * esize)), Rb);
            // (a small tensor: rather a box per SM than whole boxes)
            while (box_y > 4 && ((Cb + box_x - 1) / box_x) * ((Rb + box_y - 1) / box_y) < num_sms) box_y = (box_y + 1) / 2;
            cuuint64_t dims[2] = {(cuuint64_t)Cb, (cuuint64_t)Rb};
            cuuint32_t box[2] = {(cuuint32_t)box_x, (cuuint32_t)box_y};
            const int64_t tiles_x = (Cb + box_x - 1) / box_x, tiles_y = (Rb + box_y - 1) / box_y;
            if (tiles_x * tiles_y < ((int64_t)1 << 31) &&
                tensor_encode_tiled(&map_src, type, 2, const_cast<void *>(src), dims, st_src, box, CU_TENSOR_MAP_SWIZZLE_NONE,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B) &&
                tensor_encode_tiled(&map_dst, type, 2, dst, dims, st_dst, box, CU_TENSOR_MAP_SWIZZLE_NONE,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B)) {
                const uint32_t box_bytes = (uint32_t)(box_x * box_y * esize);
                if (launch_overlapped(copy_tma_kernel, dim3((unsigned)(tiles_x * tiles_y)), 32, smem_for(CP_CTAS_PER_SM, CP_BOX_BYTES + 128), 1, stream,
                                      map_src, map_dst, (int)tiles_x, box_x, box_y, box_bytes) != cudaSuccess) return SG_ERR_CUDA;
                launched = true;
            }
        } else {
            const int W = 128 / esize;
            cuuint64_t dims_s[2] = {(cuuint64_t)Cb, (cuuint64_t)Rb}, dims_d[2] = {(cuuint64_t)Rb, (cuuint64_t)Cb};
            cuuint32_t box_s[2] = {(cuuint32_t)W, 128}, box_d[2] = {(cuuint32_t)W, 32};
            const int64_t tiles_c = (Cb + W - 1) / W, tiles_r = (Rb + 127) / 128;
            if (tiles_c * tiles_r < ((int64_t)1 << 31) &&
                tensor_encode_tiled(&map_src, type, 2, const_cast<void *>(src), dims_s, st_src, box_s, CU_TENSOR_MAP_SWIZZLE_128B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B) &&
                tensor_encode_tiled(&map_dst, type, 2, dst, dims_d, st_dst, box_d, CU_TENSOR_MAP_SWIZZLE_128B,
                                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B)) {
                const int smem = smem_for(transpose_ctas_per_sm(R * C * esize, tiles_c * tiles_r, num_sms), TR_TILE_BYTES + 1024);
                if (smem > 48 * 1024 && !tensor_ensure_smem_attr(ATTR_SLOT + (esize == 4 ? 0 : 1), esize == 4 ? reinterpret_cast<const void *>(transpose_tma_kernel<4>)
                                                                                                              : reinterpret_cast<const void *>(transpose_tma_kernel<2>), SMEM_MOST))
                    return SG_ERR_CUDA;
                const int panel = (int)std::min<int64_t>(tiles_c, TR_PANEL);
                if (launch_overlapped(esize == 4 ? transpose_tma_kernel<4> : transpose_tma_kernel<2>, dim3((unsigned)(tiles_c * tiles_r)), TR_THREADS, smem, 1, stream, map_src, map_dst,
                                      (int)tiles_c, (int)tiles_r, panel, (int)Rb, (int)Cb) != cudaSuccess) return SG_ERR_CUDA;
                launched = true;
            }
        }
        if (launched) {
            note_kernel(transpose ? "transpose_tma_kernel" : "copy_tma_kernel");
            *used_tma = 1;
            if (tail == 0) return SG_OK;
            // the last `tail` columns of the destination: source rows [body, R) of a transpose, columns [body, C) of a copy
            const char *s_tail = static_cast<const char *>(src) + (transpose ? body * s_r : body * s_c) * esize;
            char *d_tail = static_cast<char *>(dst) + body * d_c * esize;
            const int64_t Rt = transpose ? tail : R, Ct = transpose ? C : tail;
            const int64_t di = transpose ? d_c : d_r, dj = transpose ? d_r : d_c;
            const cudaError_t e = esize == 4
                ? launch_tile_move(reinterpret_cast<const uint32_t *>(s_tail), s_r, s_c, reinterpret_cast<uint32_t *>(d_tail), di, dj, (int)Rt, (int)Ct, num_sms, stream, false)
                : launch_tile_move(reinterpret_cast<const uint16_t *>(s_tail), s_r, s_c, reinterpret_cast<uint16_t *>(d_tail), di, dj, (int)Rt, (int)Ct, num_sms, stream, false);
            return e == cudaSuccess ? SG_OK : SG_ERR_CUDA;
        }
    }
    if (force == 2) return SG_ERR_UNSUPPORTED;
    // strided path: destination index pair (i, j) of the source element; a transpose exchanges the strides
    const int64_t di = transpose ? d_c : d_r, dj = transpose ? d_r : d_c;
    const cudaError_t e = esize == 4
        ? launch_tile_move(static_cast<const uint32_t *>(src), s_r, s_c, static_cast<uint32_t *>(dst), di, dj, (int)R, (int)C, num_sms, stream)
        : launch_tile_move(static_cast<const uint16_t *>(src), s_r, s_c, static_cast<uint16_t *>(dst), di, dj, (int)R, (int)C, num_sms, stream);
    return e == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

sg_status launch_reduce2d(bool colred, int64_t R, int64_t C, const void *A, int64_t a_r, int64_t a_c, int in_bf16, float *out,
                          int64_t os, int accumulate, cudaStream_t stream) {
    int num_sms = 0;
    if (!tensor_driver_ready(&num_sms)) return SG_ERR_CUDA;
    const int64_t n_out = colred ? C : R, n_red = colred ? R : C;
    if (n_red == 0) {      // empty sum: the neutral value
        if (!accumulate) {
            if (launch_clear(out, n_out, os, stream) != cudaSuccess) return SG_ERR_CUDA;
        }
        return SG_OK;
    }
    // rows whose elements lie a pitch apart, neighbouring rows side by side: the column sums of the transposed matrix (1021 columns
    // of 4093 rows, column-major f32: read across the lines 9.8 to 14.6 us, so 5.7)
    if (!colred && a_r == 1 && R > 1 && C > 1 && a_c != 1) {
        colred = true;
        std::swap(R, C);
        std::swap(a_r, a_c);
    }
    const int es = in_bf16 ? 2 : 4;
    // 16-byte loads: rows of unit stride that start on 16-byte boundaries; a row reduction peels the ends of rows that do not
    const bool aligned = a_c == 1 && aligned16(A) && (a_r * es) % 16 == 0, vec = aligned || (!colred && a_c == 1);
    cudaError_t e;
    if (in_bf16) {
        const uint16_t *p = static_cast<const uint16_t *>(A);
        e = vec ? launch_reduce_typed<uint16_t, 8>(colred, p, a_r, a_c, (int)R, (int)C, out, os, accumulate, num_sms, aligned, stream)
                : launch_reduce_typed<uint16_t, 1>(colred, p, a_r, a_c, (int)R, (int)C, out, os, accumulate, num_sms, aligned, stream);
    } else {
        const float *p = static_cast<const float *>(A);
        e = vec ? launch_reduce_typed<float, 4>(colred, p, a_r, a_c, (int)R, (int)C, out, os, accumulate, num_sms, aligned, stream)
                : launch_reduce_typed<float, 1>(colred, p, a_r, a_c, (int)R, (int)C, out, os, accumulate, num_sms, aligned, stream);
    }
    return e == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

sg_status bandwidth_read_status(cudaStream_t stream) { return read_status_word(stream); }

}  // namespace sg
