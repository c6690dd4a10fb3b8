// Stride-1 convolutions on the tensor cores with the roles of the operands exchanged: the filter is the
// M side of the MMA (128 filters = the lanes of tensor memory), the input positions are the N side.
//
// What that buys over the strip kernel, whose tiles are 128 positions that must start at image rows:
//   * A tile is any number of positions up to 256 (a multiple of 16), so the work divides evenly: the size is chosen such that
//     the last wave of thread blocks is full.  Positions are counted with the input's row pitch, q = (n*H_in + h)*W_in + w, and
//     a tile is any run of them; those with w >= W_out or h >= H_out are computed and dropped.
//   * The filter's share of an MMA's shared-memory reads is spread over more positions: a k-step takes 98 cycles at 128
//     positions and 123 at 192 (tensor core alone: 64 and 96; the M-major filter costs about 50 of them).
//   * An accumulator lane is a filter, so a warp stores one position's 32 consecutive outputs as a whole 128-byte line
//     straight from registers: no staging, no tensor store, any output strides.
// One contiguous run of N + (KH-1)*dh*W_in + (KW-1)*dw input rows (128 bytes: 64 channels) serves all taps of a channel block:
// each tap's MMAs read it through a descriptor shifted by kh*dh*W_in + kw*dw rows (the 128-byte swizzle is a function of the
// absolute address).  Wide images take one run per filter row instead.  The filter travels in slots of one filter row (KW taps
// x 64 channels x 128 filters, one TMA load); when all of it fits it is loaded once and stays, otherwise it streams.
//
// Warps: 0 input runs (TMA), 1 MMA issuer and owner of tensor memory, 2 filter (TMA), 4-11 write-back (two per lane quarter).
#include <algorithm>

#include "sg_internal.cuh"
#include "sg_tc_ptx.cuh"

namespace sg {
namespace {

constexpr int BF = 128;                       // filters per tile
constexpr int MAX_SLOTS = 8, RUN_STAGES = 2;
constexpr int THREADS = 384;
constexpr int SMEM_LIMIT = 232448 - 1024 - 512;

struct WideParams {
    int BN;                 // positions per tile
    int tiles, f_tiles;     // position tiles, filter tiles
    int positions;          // positions that can be outputs
    int N, Hin, Win, Hout, Wout, F;
    int KH, KW, kb;         // filter rows, taps per row, channel blocks
    int row_step, dw;       // rows of the run between filter rows, between taps of a row
    int per_row, run_boxes, box_rows, run_bytes;      // one run per filter row; TMA loads per run and their rows; bytes of a run's stage
    int slots, slot_bytes, resident;         // filter ring; resident: it holds the whole filter
    int flt_loads;          // TMA loads per slot: 1, or one per 64 filters when F is no multiple of 64
    int tap_bytes, half_bytes;               // in a slot: between taps, between the two 64-filter halves
    int last_ksteps;        // k-steps of 16 channels in the last channel block
    int run_tx;             // bytes of a run's loads
    int tmem_cols, bufs;    // bufs: accumulators of BN columns, 1 or 2
    int o_n, o_h, o_w;
    int accumulate, wait_prior;
};

// The eight write-back warps (4 to 11; two per lane quarter): lane = filter, register = position.
__device__ __forceinline__ void write_back(const WideParams &p, float *__restrict__ O, uint32_t tmem_base, int item0, int item1, uint32_t acc_full,
                                           uint32_t acc_empty, volatile int *abort_flag) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = warp & 3, half = (warp - 4) >> 2;
    int tl = 0;
    if (p.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int hw = p.Hin * p.Win;
    for (int item = item0; item < item1; ++item, ++tl) {
        const int ft = item / p.tiles, q0 = (item - ft * p.tiles) * p.BN;
        const int buf = p.bufs == 2 ? tl & 1 : 0;
        if (!__all_sync(0xffffffffu, mbar_wait(acc_full + 8u * buf, (p.bufs == 2 ? tl >> 1 : tl) & 1, abort_flag))) break;
        tc_fence_after();
        const int f = ft * BF + q * 32 + lane;
        const int blocks = p.BN / 16;
        for (int j = half; j < blocks; j += 2) {
            uint32_t r[16];
            tmem_ld_32x16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * p.BN + j * 16), r);
            // lane i: whether position i of the sixteen is an output, and its offset
            const int pos = q0 + j * 16 + (lane & 15);
            const int n = pos / hw, rem = pos - n * hw, h = rem / p.Win, w = rem - h * p.Win;
            const uint32_t live = __ballot_sync(0xffffffffu, pos < p.positions && w < p.Wout && h < p.Hout);
            const int off = n * p.o_n + h * p.o_h + w * p.o_w;
            tmem_ld_wait();
            if (p.accumulate) {
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const int o = __shfl_sync(0xffffffffu, off, c);
                    if ((live >> c & 1u) && f < p.F) asm volatile("red.global.add.f32 [%0], %1;" ::"l"(O + (o + f)), "f"(__uint_as_float(r[c])) : "memory");
                }
            } else if ((live & 0xFFFFu) == 0xFFFFu &&
                       __all_sync(0xffffffffu, off == __shfl_sync(0xffffffffu, off, 0) + (int64_t)(lane & 15) * p.o_w)) {
                float *out = O + (__shfl_sync(0xffffffffu, off, 0) + f);          // (all sixteen o_w apart)
                if (f < p.F)
#pragma unroll
                    for (int c = 0; c < 16; ++c, out += p.o_w) *out = __uint_as_float(r[c]);
            } else {
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const int o = __shfl_sync(0xffffffffu, off, c);
                    if ((live >> c & 1u) && f < p.F) O[o + f] = __uint_as_float(r[c]);
                }
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty + 8u * buf);
    }
}

__global__ void __launch_bounds__(THREADS, 1)
conv_wide_kernel(const __grid_constant__ CUtensorMap map_in, const __grid_constant__ CUtensorMap map_flt, const WideParams p, float *__restrict__ O) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t flt_addr = base, runs_addr = flt_addr + (uint32_t)(p.slots * p.slot_bytes);
    __shared__ uint64_t bars[2 * MAX_SLOTS + 2 * RUN_STAGES + 5];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    const uint32_t bar0 = smem_u32(bars);
    auto flt_full = [&](int s) { return bar0 + 8u * s; };
    auto flt_empty = [&](int s) { return bar0 + 8u * (MAX_SLOTS + s); };
    auto run_full = [&](int s) { return bar0 + 8u * (2 * MAX_SLOTS + s); };
    auto run_empty = [&](int s) { return bar0 + 8u * (2 * MAX_SLOTS + RUN_STAGES + s); };
    auto acc_full = [&](int b) { return bar0 + 8u * (2 * MAX_SLOTS + 2 * RUN_STAGES + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (2 * MAX_SLOTS + 2 * RUN_STAGES + 2 + b); };
    const uint32_t first_run = bar0 + 8u * (2 * MAX_SLOTS + 2 * RUN_STAGES + 4);      // completed once: the block's first run has landed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.launch_dependents;");
    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_in); prefetch_tensormap(&map_flt);
        for (int s = 0; s < MAX_SLOTS; ++s) { mbar_init(flt_full(s), 1); mbar_init(flt_empty(s), 1); }
        for (int s = 0; s < RUN_STAGES; ++s) { mbar_init(run_full(s), 1); mbar_init(run_empty(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 8); }
        mbar_init(first_run, 1);
        abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *(volatile uint32_t *)&tmem_slot;

    // this block's items: a contiguous, balanced run of (filter tile, position tile), positions fastest
    const int total = p.tiles * p.f_tiles;
    const int item0 = (int)((long long)blockIdx.x * total / gridDim.x), item1 = (int)((long long)(blockIdx.x + 1) * total / gridDim.x);

    // (The producers' warps walk their loops converged, one elected lane issues, and nothing inside a step divides: a lane on its own with
    // the ring's position by division took 500 to 1000 cycles a load.  The first item is worked out ahead of the wait
    // for the kernel before this one.)
    if (warp == 0) {
        // ------------------------------------------------------------ input runs
        const bool issuer = elect_one();
        int s = 0, tile = item0 % p.tiles;
        uint32_t phase = 1;
        bool ok = true;
        if (p.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int item = item0; item < item1 && ok; ++item) {
            const int q0 = tile * p.BN;
            if (++tile == p.tiles) tile = 0;
            for (int cb = 0; cb < p.kb; ++cb) {
                if (!__all_sync(0xffffffffu, mbar_wait(run_empty(s), phase, abort_flag))) { ok = false; break; }
                if (issuer) {
                    mbar_expect_tx(run_full(s), (uint32_t)p.run_tx);
                    for (int b = 0; b < p.run_boxes; ++b)
                        tma_tile_3d<false>(runs_addr + (uint32_t)(s * p.run_bytes + b * p.box_rows * 128), &map_in, run_full(s), cb * 64, q0 + b * p.box_rows, 0);
                }
                if (++s == RUN_STAGES) { s = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ filter
        const bool issuer = elect_one();
        int s = 0, ft = item0 / p.tiles, tile = item0 - ft * p.tiles, cur = -1;
        uint32_t phase = 1;
        bool ok = true, second = false;
        if (p.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int item = item0; item < item1 && ok; ++item) {
            const int f = ft;
            if (++tile == p.tiles) { tile = 0; ++ft; }
            if (p.resident && f == cur) continue;
            cur = f;
            for (int cb = 0; cb < p.kb && ok; ++cb)
                for (int kh = 0; kh < p.KH; ++kh) {
                    if (!__all_sync(0xffffffffu, mbar_wait(flt_empty(s), phase, abort_flag))) { ok = false; break; }
                    // (the first run and the first slot are what the first MMA waits for: the rest of the filter, up to
                    // three times their size, comes behind them rather than beside them.  The wait is for a barrier that the
                    // MMA warp completes once: a phase of the ring could have come round again by the time this is reached,
                    // which is items later where the filter is one slot.)
                    if (second && !__all_sync(0xffffffffu, mbar_wait(first_run, 0, abort_flag))) { ok = false; break; }
                    second = item == item0 && cb == 0 && kh == 0;
                    if (issuer) {
                        mbar_expect_tx(flt_full(s), (uint32_t)p.slot_bytes);
                        const uint32_t dst = flt_addr + (uint32_t)(s * p.slot_bytes);
                        if (p.flt_loads == 1) {
                            tma_tile_5d<false>(dst, &map_flt, flt_full(s), 0, cb * 64, f * (BF / 64), 0, kh);
                        } else {
                            tma_load_4d(dst, &map_flt, flt_full(s), f * BF, cb * 64, 0, kh);
                            tma_load_4d(dst + p.half_bytes, &map_flt, flt_full(s), f * BF + 64, cb * 64, 0, kh);
                        }
                    }
                    if (++s == p.slots) { s = 0; phase ^= 1u; }
                }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: the whole warp walks, one lane issues
        const uint32_t idesc = make_idesc(p.BN, BF, false, true, false);       // filter as stored: M-major; positions K-major
        const bool issuer = elect_one();
        auto wait_all = [&](bool passed) { return __all_sync(0xffffffffu, passed) != 0; };
        int s = 0, slot = 0, tl = 0, cur = -1, ft_next = item0 / p.tiles, tile = item0 - ft_next * p.tiles;
        uint32_t run_phase = 0, slot_phase = 0;
        bool ok = true, landed = false;
        for (int item = item0; item < item1 && ok; ++item, ++tl) {
            const int ft = ft_next;
            if (++tile == p.tiles) { tile = 0; ++ft_next; }
            const bool fresh = !p.resident || ft != cur;             // this tile's filter slots have to be waited for
            const bool release = !p.resident || item + 1 >= item1 || ft_next != ft;
            if (!fresh) slot = 0;                                     // (a filter that stays fills the ring)
            cur = ft;
            const int buf = tl & 1;
            if (!wait_all(mbar_wait(acc_empty(buf), ((tl >> 1) & 1) ^ 1u, abort_flag))) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tmem_base + buf * p.BN;
            uint32_t acc = 0;
            for (int cb = 0; cb < p.kb && ok; ++cb) {
                if (!wait_all(mbar_wait(run_full(s), run_phase, abort_flag))) { ok = false; break; }
                if (!landed && issuer) mbar_arrive(first_run);
                landed = true;
                const uint32_t run = runs_addr + (uint32_t)(s * p.run_bytes);
                const int ksteps = cb + 1 == p.kb ? p.last_ksteps : 4;
                for (int kh = 0; kh < p.KH; ++kh) {
                    const int fs = slot;
                    if (fresh && !wait_all(mbar_wait(flt_full(fs), slot_phase, abort_flag))) { ok = false; break; }
                    if (++slot == p.slots) {
                        slot = 0;
                        if (fresh) slot_phase ^= 1u;
                    }
                    tc_fence_after();
                    // (descriptors are made by the converged warp: uniform values; a lane on its own pays ~100 cycles per MMA)
                    for (int kw = 0; kw < p.KW; ++kw) {
                        const uint64_t a = make_smem_desc(flt_addr + (uint32_t)(fs * p.slot_bytes + kw * p.tap_bytes), (uint32_t)p.half_bytes, 1024);
                        const uint64_t b = make_smem_desc(run + (uint32_t)(kh * p.row_step + kw * p.dw) * 128u, 16, 1024);
                        if (issuer) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (k < ksteps) umma_bf16(d, a + (uint64_t)(k * 128), b + (uint64_t)(k * 2), idesc, k == 0 ? acc : 1u);
                        }
                        acc = 1u;
                    }
                    if (release && issuer) umma_commit(flt_empty(fs));
                }
                if (ok && issuer) umma_commit(run_empty(s));
                if (++s == RUN_STAGES) { s = 0; run_phase ^= 1u; }
            }
            if (ok && issuer) umma_commit(acc_full(buf));
        }
    } else if (warp >= 4) {
        write_back(p, O, tmem_base, item0, item1, acc_full(0), acc_empty(0), abort_flag);
    }
    // ---------------------------------------------------------------- teardown
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(5000);      // let loads in flight land before the shared memory goes
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

// ---- f32 ----------------------------------------------------------------------------------------
// The same exchange with every element split as x = hi + lo, hi = x rounded to tf32: the corrections lo*hi + hi*lo run as one bf16
// contraction over [lo | hi] . [hi | lo], the main term hi*hi in tf32 (8 MMAs per 32 channels of a tap).
//   * The filter goes through a ring of raw tiles (one tap of 32 channels x 128 filters each) and the converters' registers into
//     tensor memory, where the MMAs read it as their A operand: a slot holds one such tile in 64 columns.  When the slots hold the
//     whole filter it is split once per thread block, otherwise once per tile.  (Loaded by the converters themselves, without the
//     ring, a tile took 1.15 us: the latency of its loads.)
//   * A run of input rows is split ONCE for all taps, in place: hi over the raw rows, [hi | lo] in bf16 beside them (the strip
//     kernel's f32 form, whose positions are the A operand, splits its rows again for every tap, which is what paced it).
// What bounds it: fetching the filter, which every block does for itself (about 19 bytes a cycle and SM), in short problems; the
// MMAs, which run at N / 2 cycles each, in long ones.  16 x 56 x 56, 3x3x64x128: 41.6 -> 32.3 us (229 TFLOP/s), 3x3x16x256
// on 44 x 74 x 74: 142.6 -> 91.7; 32 x 1024, 3x64x128, where launch, first run and last write-back are most of it: 14.0 -> 11.3.
// Warps: 0 input runs (TMA), 1 MMA issuer and owner of tensor memory, 2 filter (TMA), 4-11 write-back, 12-27 converters.
constexpr int F32_SLOTS = 16, F32_STAGES = 4, F32_TILES = 4;
constexpr int F32_CONVERTERS = 16;
constexpr int F32_THREADS = 384 + 32 * F32_CONVERTERS;

struct F32Filter {
    int taps;
    int chp;                      // channels of a slot: 32, or 16 when there are no more than 16
    int stages;                   // runs in shared memory
    int run_rows;                 // rows of a run
    int tiles, tile_bytes;        // ring of raw filter tiles, behind the runs
    int groups;                   // of converter warps that take the filter's steps in turn
};

__global__ void __launch_bounds__(F32_THREADS, 1)
conv_wide_f32_kernel(const __grid_constant__ CUtensorMap map_in, const __grid_constant__ CUtensorMap map_flt, const __grid_constant__ F32Filter g, const __grid_constant__ WideParams p,
                     float *__restrict__ O) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_gen = smem_raw + (base - smem_u32(smem_raw));
    __shared__ uint64_t bars[2 * F32_SLOTS + 3 * F32_STAGES + 4 + 2 * F32_TILES];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_word;
    volatile int *abort_flag = &abort_word;
    const uint32_t bar0 = smem_u32(bars);
    auto slot_full = [&](int s) { return bar0 + 8u * s; };
    auto slot_empty = [&](int s) { return bar0 + 8u * (F32_SLOTS + s); };
    auto raw_full = [&](int s) { return bar0 + 8u * (2 * F32_SLOTS + s); };
    auto run_full = [&](int s) { return bar0 + 8u * (2 * F32_SLOTS + F32_STAGES + s); };
    auto run_empty = [&](int s) { return bar0 + 8u * (2 * F32_SLOTS + 2 * F32_STAGES + s); };
    auto acc_full = [&](int b) { return bar0 + 8u * (2 * F32_SLOTS + 3 * F32_STAGES + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (2 * F32_SLOTS + 3 * F32_STAGES + 2 + b); };
    auto tile_full = [&](int s) { return bar0 + 8u * (2 * F32_SLOTS + 3 * F32_STAGES + 4 + s); };
    auto tile_empty = [&](int s) { return bar0 + 8u * (2 * F32_SLOTS + 3 * F32_STAGES + 4 + F32_TILES + s); };
    const uint32_t flt_off = (uint32_t)(2 * g.stages * p.run_bytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.launch_dependents;");
    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_in); prefetch_tensormap(&map_flt);
        for (int s = 0; s < F32_TILES; ++s) { mbar_init(tile_full(s), 1); mbar_init(tile_empty(s), 4); }
        for (int s = 0; s < F32_SLOTS; ++s) { mbar_init(slot_full(s), 4); mbar_init(slot_empty(s), 1); }
        for (int s = 0; s < F32_STAGES; ++s) { mbar_init(raw_full(s), 1); mbar_init(run_full(s), F32_CONVERTERS); mbar_init(run_empty(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 8); }
        abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"((uint32_t)p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *(volatile uint32_t *)&tmem_slot;
    const uint32_t slots_tmem = tmem_base + (uint32_t)(p.bufs * p.BN), slot_cols = 2u * g.chp;      // a slot: hi | lo, hi in bf16 pairs

    const int total = p.tiles * p.f_tiles;
    const int item0 = (int)((long long)blockIdx.x * total / gridDim.x), item1 = (int)((long long)(blockIdx.x + 1) * total / gridDim.x);

    if (warp == 0) {
        // ------------------------------------------------------------ input runs
        if (lane == 0) {
            if (p.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
            int it = 0;
            bool ok = true;
            for (int item = item0; item < item1 && ok; ++item) {
                const int q0 = item % p.tiles * p.BN;
                for (int cb = 0; cb < p.kb; ++cb, ++it) {
                    const int s = it % g.stages;
                    if (!mbar_wait(run_empty(s), ((it / g.stages) & 1) ^ 1u, abort_flag)) { ok = false; break; }
                    mbar_expect_tx(raw_full(s), (uint32_t)p.run_tx);
                    for (int b = 0; b < p.run_boxes; ++b)
                        tma_tile_3d<false>(base + (uint32_t)(2 * s * p.run_bytes + b * p.box_rows * 128), &map_in, raw_full(s), cb * 32, q0 + b * p.box_rows, 0);
                }
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------ filter
        if (lane == 0) {
            if (p.wait_prior) asm volatile("griddepcontrol.wait;" ::: "memory");
            int it = 0, cur = -1;
            bool ok = true;
            for (int item = item0; item < item1 && ok; ++item) {
                const int ft = item / p.tiles;
                if (p.resident && ft == cur) continue;
                cur = ft;
                for (int cb = 0; cb < p.kb && ok; ++cb)
                    for (int tap = 0; tap < g.taps; ++tap, ++it) {
                        const int s = it % g.tiles;
                        if (!mbar_wait(tile_empty(s), ((it / g.tiles) & 1) ^ 1u, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(tile_full(s), (uint32_t)g.tile_bytes);
                        tma_load_4d(base + flt_off + (uint32_t)(s * g.tile_bytes), &map_flt, tile_full(s), ft * BF, cb * 32, tap % p.KW, tap / p.KW);
                    }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: the whole warp walks, one lane issues
        const uint32_t idesc = make_idesc(p.BN, BF, true, false, false), idesc16 = make_idesc(p.BN, BF, false, false, false);
        const bool issuer = elect_one();
        auto wait_all = [&](bool passed) { return __all_sync(0xffffffffu, passed) != 0; };
        int stage = 0, stage_phase = 0, slot = 0, slot_phase = 0, cur = -1;
        bool ok = true;
        for (int item = item0, tl = 0; item < item1 && ok; ++item, ++tl) {
            const int ft = item / p.tiles;
            const bool fresh = !p.resident || ft != cur;             // this tile's filter slots have to be waited for
            const bool release = !p.resident || item + 1 >= item1 || (item + 1) / p.tiles != ft;
            if (!fresh) slot = 0;                                     // (a filter that stays fills the ring)
            cur = ft;
            const int buf = p.bufs == 2 ? tl & 1 : 0;
            if (!wait_all(mbar_wait(acc_empty(buf), ((p.bufs == 2 ? tl >> 1 : tl) & 1) ^ 1u, abort_flag))) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tmem_base + buf * p.BN;
            uint32_t acc = 0;
            for (int cb = 0; cb < p.kb && ok; ++cb) {
                const int s = stage;
                if (!wait_all(mbar_wait(run_full(s), stage_phase, abort_flag))) { ok = false; break; }
                if (++stage == g.stages) { stage = 0; stage_phase ^= 1; }
                const uint32_t run = base + (uint32_t)(2 * s * p.run_bytes);
                const int ksteps = cb + 1 == p.kb ? p.last_ksteps : 2;         // of 16 channels
                for (int kh = 0, kw = 0, tap = 0; tap < g.taps; ++tap) {
                    const int fs = slot;
                    if (fresh && !wait_all(mbar_wait(slot_full(fs), slot_phase, abort_flag))) { ok = false; break; }
                    if (++slot == p.slots) {
                        slot = 0;
                        if (fresh) slot_phase ^= 1;
                    }
                    tc_fence_after();
                    const uint32_t a_hi = slots_tmem + fs * slot_cols, a_lo = a_hi + g.chp, a_hi16 = a_lo + g.chp / 2;
                    const uint32_t row = (uint32_t)(kh * p.row_step + kw * p.dw) * 128u;
                    const uint64_t b_hi = make_smem_desc(run + row, 16, 1024), b16 = make_smem_desc(run + (uint32_t)p.run_bytes + row, 16, 1024);
                    if (issuer) {
#pragma unroll
                        for (int k = 0; k < 2; ++k)      // small terms first: lo of the filter with hi of the input, then hi with lo
                            if (k < ksteps) {
                                umma_bf16_ts(d, a_lo + k * 8, b16 + (uint64_t)(k * 2), idesc16, k == 0 ? acc : 1u);
                                umma_bf16_ts(d, a_hi16 + k * 8, b16 + (uint64_t)(4 + k * 2), idesc16, 1u);
                            }
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (k < 2 * ksteps) umma_tf32_ts(d, a_hi + k * 8, b_hi + (uint64_t)(k * 2), idesc, 1u);
                    }
                    acc = 1u;
                    if (release && issuer) umma_commit(slot_empty(fs));
                    if (++kw == p.KW) { kw = 0; ++kh; }
                }
                if (ok && issuer) umma_commit(run_empty(s));
            }
            if (ok && issuer) umma_commit(acc_full(buf));
        }
    } else if (warp >= 12) {
        // ------------------------------------------------------------ converters
        // A step of the filter (a tile of it -> a slot) is a chain of ~1500 cycles of latencies, however little each warp does of
        // it: up to four groups of four warps (one per lane quarter) take the steps in turn, so that as many are under way at a
        // time.  (A group that ran a whole round of a ring ahead would take the phase before the last of a barrier for the one it
        // waits for: there are no more groups than slots, whose MMAs finish in order, and the raw tiles, whose loads need not,
        // are a multiple of the groups, so that a group always meets the same ones.)
        const int cw = warp - 12, quarter = warp & 3, group = cw >> 2;
        int stage = 0, stage_phase = 0;
        bool ok = true;
        // (the warp's lanes go on together, as the tcgen05 instructions below require)
        auto wait_all = [&](uint32_t bar, int phase) { return __all_sync(0xffffffffu, mbar_wait(bar, phase, abort_flag)) != 0; };
        // one run: 32 rows x 8 channels per warp and turn (row x's 16-byte chunk c lies at chunk c ^ (x & 7))
        auto split_run = [&]() {
            const int s = stage;
            if (!wait_all(raw_full(s), stage_phase)) { ok = false; return; }
            uint8_t *raw = smem_gen + (size_t)2 * s * p.run_bytes, *pair = raw + p.run_bytes;
            const int part = cw & 3;
            if (part * 8 < g.chp)
                for (int row = (cw >> 2) * 32 + lane; row < g.run_rows; row += F32_CONVERTERS / 4 * 32) {
                    uint4 *c0 = reinterpret_cast<uint4 *>(raw + row * 128 + (((2 * part) ^ (row & 7)) << 4));
                    uint4 *c1 = reinterpret_cast<uint4 *>(raw + row * 128 + (((2 * part + 1) ^ (row & 7)) << 4));
                    uint4 h0, h1, h16, l16;
                    split8_mix(*c0, *c1, h0, h1, h16, l16);
                    *c0 = h0;
                    *c1 = h1;
                    *reinterpret_cast<uint4 *>(pair + row * 128 + ((part ^ (row & 7)) << 4)) = h16;
                    *reinterpret_cast<uint4 *>(pair + row * 128 + (((4 + part) ^ (row & 7)) << 4)) = l16;
                }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(run_full(s));
            if (++stage == g.stages) { stage = 0; stage_phase ^= 1; }
        };
        int turn = 0, tile = 0, tile_phase = 0, slot = 0, slot_phase = 0;
        // the steps of one channel block
        auto split_filter = [&]() {
            for (int tap = 0; tap < g.taps && ok; ++tap) {
                const int r = tile, s = slot, r_phase = tile_phase, s_phase = slot_phase;
                const bool mine = turn == group;
                if (++turn == g.groups) turn = 0;
                if (++tile == g.tiles) { tile = 0; tile_phase ^= 1; }
                if (++slot == p.slots) { slot = 0; slot_phase ^= 1; }
                if (!mine) continue;
                if (!wait_all(tile_full(r), r_phase)) { ok = false; break; }
                // lane = filter reads channels down a column (512-byte rows), 16 at a time
                const uint32_t *col = reinterpret_cast<const uint32_t *>(smem_gen + flt_off + (size_t)r * g.tile_bytes) + quarter * 32 + lane;
                const uint32_t t = slots_tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)s * slot_cols;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (half * 16 >= g.chp) break;
                    uint32_t hi[16], lo16[8], hi16[8];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t *c = col + (half * 2 + e) * 8 * BF;
                        uint4 h0, h1, h16, l16;
                        split8_mix(make_uint4(c[0], c[BF], c[2 * BF], c[3 * BF]), make_uint4(c[4 * BF], c[5 * BF], c[6 * BF], c[7 * BF]), h0, h1, h16, l16);
                        hi[8 * e] = h0.x; hi[8 * e + 1] = h0.y; hi[8 * e + 2] = h0.z; hi[8 * e + 3] = h0.w;
                        hi[8 * e + 4] = h1.x; hi[8 * e + 5] = h1.y; hi[8 * e + 6] = h1.z; hi[8 * e + 7] = h1.w;
                        lo16[4 * e] = l16.x; lo16[4 * e + 1] = l16.y; lo16[4 * e + 2] = l16.z; lo16[4 * e + 3] = l16.w;
                        hi16[4 * e] = h16.x; hi16[4 * e + 1] = h16.y; hi16[4 * e + 2] = h16.z; hi16[4 * e + 3] = h16.w;
                    }
                    if (half == 0) {
                        if (!wait_all(slot_empty(s), s_phase ^ 1)) { ok = false; break; }
                        tc_fence_after();
                    }
                    __syncwarp();
                    tmem_st_32x16(t + half * 16, hi);
                    tmem_st_32x8(t + g.chp + half * 8, lo16);
                    tmem_st_32x8(t + g.chp + g.chp / 2 + half * 8, hi16);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (ok && lane == 0) { mbar_arrive(slot_full(s)); mbar_arrive(tile_empty(r)); }
            }
        };
        int cur = -1;
        for (int item = item0; item < item1 && ok; ++item) {
            const int ft = item / p.tiles;
            const bool fresh = !p.resident || ft != cur;
            cur = ft;
            // a filter that stays needs no MMA to make room for it: all of it goes first, while the first run is on its way
            if (fresh && p.resident)
                for (int cb = 0; cb < p.kb && ok; ++cb) split_filter();
            for (int cb = 0; cb < p.kb && ok; ++cb) {
                split_run();
                if (ok && !p.resident) split_filter();
            }
        }
    } else if (warp >= 4) {
        write_back(p, O, tmem_base, item0, item1, acc_full(0), acc_empty(0), abort_flag);
    }
    // ---------------------------------------------------------------- teardown
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(5000);      // let loads in flight land before the shared memory goes
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
    }
}

inline bool mult(int64_t v, int64_t q) { return v % q == 0; }

// What one run of input rows looks like for tiles of `bn` positions: one run for all taps, or one per filter row where the image is
// so wide that those are fewer rows.
struct Run { bool per_row; int boxes, box_rows; int64_t tx, bytes; };
inline bool plan_run(int bn, int KH, int row_span, int64_t full_span, Run *r) {
    r->per_row = full_span - row_span > (int64_t)(KH - 1) * (bn + row_span);
    const int64_t rows = r->per_row ? bn + row_span : bn + full_span;
    r->boxes = 1;
    r->box_rows = (int)rows;
    if (r->per_row) {
        if (rows > 256) return false;
    } else {
        r->boxes = (int)((rows + 255) / 256);
        r->box_rows = (int)(((rows + r->boxes - 1) / r->boxes + 7) / 8 * 8);
    }
    r->tx = (int64_t)r->box_rows * 128 * (r->per_row ? KH : r->boxes);
    r->bytes = (r->tx + 1023) / 1024 * 1024;
    return true;
}

// Tiles and ring sizes of the bf16 kernel.  Positions per tile: the least estimated time, in cycles.  A tile's run comes in and its
// outputs go out at the block's share of the HBM rate; between the first run and the last write-back the slowest of run, MMAs and
// write-back paces the rounds.  (Fitted to sweeps of 32 to 256 positions on nine shapes; the choices are within 4 % of the best
// but for one 9 %.)
// Returns the estimated time in microseconds of the tiles chosen, in which the write-back counts as well: 20 cycles a position, since only the two warps of a
// quarter of the lanes write a filter (337 timings: within 9 % in the mean).
double plan_bf16(const Problem &p, int64_t positions, int f_tiles, int row_span, int64_t full_span, int num_sms, WideParams &w) {
    const int kb = (p.C + 63) / 64, total_slots = kb * p.KH;
    const int flt_rows = kb > 1 ? 64 : (p.C + 15) / 16 * 16;           // channels of a filter block
    const int slot_bytes = p.KW * BF * 2 * flt_rows;
    double best = 1e300, us = 1e300;
    const int ksteps = (kb - 1) * 4 + ((p.C - (kb - 1) * 64) + 15) / 16;
    for (int bn = 32; bn <= 256; bn += 16) {
        Run r;
        if (!plan_run(bn, p.KH, row_span, full_span, &r)) continue;
        const int64_t room = SMEM_LIMIT - RUN_STAGES * r.bytes;
        if (room < slot_bytes) continue;
        const int slots = (int)std::min<int64_t>(std::min<int64_t>(MAX_SLOTS, total_slots), room / slot_bytes);
        if (slots < std::min(2, total_slots)) continue;
        const bool resident = slots == total_slots;
        const int64_t tiles = (positions + bn - 1) / bn, items = tiles * f_tiles, rounds = (items + num_sms - 1) / num_sms;
        const double rate = std::min(64.0, 23.0 * num_sms / (double)std::min<int64_t>(items, num_sms));
        const double load = (double)r.tx * kb / rate, store = (double)bn * std::min(p.N, BF) * 4.0 / rate;
        double mma = (double)p.KH * p.KW * ksteps * std::max(bn / 2.0, 49.5 + 0.384 * bn);
        if (!resident) mma = std::max(mma, (double)slot_bytes * total_slots / 45.0);       // the filter streams from the L2
        const double cost = load + mma + (double)(rounds - 1) * std::max(mma, std::max(load, store)) + store + 300.0 * (double)rounds;
        if (cost >= best) continue;
        best = cost;
        const double write = std::max(store, 20.0 * bn), further = (double)(rounds - 1);
        us = 3.5 + 0.87 / 1900.0 * (load + mma + further * std::max(std::max(mma, load), write) + write + 300.0 * (double)rounds) + 0.38 * further;
        w.BN = bn; w.tiles = (int)tiles; w.run_boxes = r.boxes; w.box_rows = r.box_rows; w.run_bytes = (int)r.bytes; w.run_tx = (int)r.tx;
        w.slots = slots; w.resident = resident; w.per_row = r.per_row; w.bufs = 2;
    }
    w.kb = kb;
    w.slot_bytes = slot_bytes;
    w.last_ksteps = (p.C - (kb - 1) * 64 + 15) / 16;
    return us;
}

// The same for the f32 kernel, whose slots share tensor memory with the accumulators.  Returns the estimated time in microseconds.
// A block is paced by the slowest of its MMAs (N / 2 cycles each), what it fetches (19.4 bytes a cycle with all SMs fetching the
// same filter) and its converters (685 cycles a step with four groups, 9.1 a row of a run); one accumulator instead of two
// leaves the write-back in the open.  (Constants fitted to 400 timings of 17 shapes and 32 to 256 positions, within 8 %; the choices
// are the best of each sweep but for two, 5 and 12 % off.  The converters have become faster since, which filters that stream feel: 170 timings of the
// tiles chosen are within 10 % of the estimate where the filter stays, and of 0.86 of it where it streams.)
double plan_f32(const Problem &p, int64_t positions, int f_tiles, int row_span, int64_t full_span, int num_sms, WideParams &w, F32Filter &g) {
    const int kb = (p.C + 31) / 32;
    g.taps = p.KH * p.KW;
    g.chp = p.C <= 16 ? 16 : 32;
    const int total_slots = kb * g.taps, slot_cols = 2 * g.chp;
    g.tile_bytes = g.chp * BF * 4;
    w.kb = kb;
    w.last_ksteps = (p.C - (kb - 1) * 32 + 15) / 16;
    const int ksteps = (kb - 1) * 2 + w.last_ksteps;
    double best = 1e300;
    for (int bn = 32; bn <= 256; bn += 16) {
        Run r;
        if (!plan_run(bn, p.KH, row_span, full_span, &r)) continue;
        const int64_t room = SMEM_LIMIT - 2 * g.tile_bytes;      // (two filter tiles at least)
        const int stages = (int)std::min<int64_t>(F32_STAGES, room / (2 * r.bytes));
        if (stages < 1) continue;
        for (int bufs = 2; bufs >= 1; --bufs) {
            const int slots = std::min(std::min(F32_SLOTS, total_slots), (512 - bufs * bn) / slot_cols);
            if (slots < std::min(2, total_slots)) continue;
            const bool resident = slots == total_slots;
            int flt_tiles = (int)std::min<int64_t>(F32_TILES, (SMEM_LIMIT - 2 * stages * r.bytes) / g.tile_bytes);
            const int groups = std::min(std::min(F32_CONVERTERS / 4, slots), flt_tiles);
            flt_tiles -= flt_tiles % groups;
            const int64_t tiles = (positions + bn - 1) / bn, items = tiles * f_tiles, rounds = (items + num_sms - 1) / num_sms;
            const double share = (double)num_sms / (double)std::min<int64_t>(items, num_sms);       // of an SM in the chip's memory rates
            const double load = (double)r.tx / std::min(64.0, 40.0 * share);
            const double store = (double)bn * std::min(p.N, BF) * 4.0 / std::min(64.0, 29.4 * share);
            const double rows = (double)r.tx / 128.0;
            const double mma = (double)g.taps * ksteps * 4.0 * std::max(bn / 2.0, 57.0);
            const double fill = ((double)total_slots * g.tile_bytes + (double)r.tx * kb) / 19.4;
            const double steps = (double)total_slots * (g.chp == 32 ? 685.0 : 510.0) * std::max(1.0, 3.6 / groups), split = rows * kb * 9.1;
            double first, other;
            if (resident) {
                first = std::max(load * kb, std::max(fill, steps)) + rows * 9.1 + mma;
                other = std::max(mma, std::max(split, load * kb));
            } else {
                other = std::max(mma, std::max(fill, steps + split));
                first = load + rows * 9.1 + other;
            }
            const double gap = stages < 2 ? load + rows * 9.1 + 1500.0 : 0.0;       // one run: each comes in when the one before is used up
            first += (kb - 1) * gap; other += kb * gap;
            const double cost = first + (double)(rounds - 1) * ((bufs == 1 ? other + 0.91 * store : std::max(other, store)) + 2100.0) + store + 7700.0;
            if (cost >= best) continue;
            best = cost;
            w.BN = bn; w.tiles = (int)tiles; w.run_boxes = r.boxes; w.box_rows = r.box_rows; w.run_bytes = (int)r.bytes; w.run_tx = (int)r.tx;
            w.slots = slots; w.resident = resident; w.per_row = r.per_row; w.bufs = bufs;
            g.stages = stages; g.run_rows = (int)rows; g.tiles = flt_tiles; g.groups = groups;
        }
    }
    return best * (1.0 / 1900.0) * (w.resident ? 1.0 : 0.86);
}

}  // namespace

sg_status launch_conv_wide(const Problem &p, const void *In, const void *Flt, float *O, bool forced, bool *resident_filter, cudaStream_t stream) {
    // ---- eligibility: unit conv strides, dense pixel pitch, TMA alignment rules for the operands; any output strides but f
    if (p.spatial_rank == 0 || p.sh != 1 || p.sw != 1) return SG_ERR_UNSUPPORTED;
    const bool f32 = !p.in_bf16;
    const int es = f32 ? 4 : 2;
    // Lanes without a filter cost as much as the others.  Up to 64 filters this kernel still wins where each input row serves nine
    // taps or more (3x3x16x32 on 16 x 112 x 112: 29.1 -> 22.1 us, 5x5x32x64: 40.7 -> 20.9; but three taps 5.6 -> 6.3).
    if (!forced && (p.N < 24 || (p.N <= 64 && p.KH * p.KW < 9))) return SG_ERR_UNSUPPORTED;
    if (p.i_c != 1 || p.k_f != 1 || p.o_f != 1) return SG_ERR_UNSUPPORTED;
    if (p.Hin > 1 && p.i_h != (int64_t)p.Win * p.i_w) return SG_ERR_UNSUPPORTED;
    if (p.batch > 1 && p.i_n != (int64_t)p.Hin * p.Win * p.i_w) return SG_ERR_UNSUPPORTED;
    if (p.i_w < p.C || p.k_c < p.N) return SG_ERR_UNSUPPORTED;
    if (reinterpret_cast<uintptr_t>(In) % 16 || !mult(p.i_w * es, 16) || !mult(p.C * es, 16)) return SG_ERR_UNSUPPORTED;
    if (p.KW > 16 || p.KH > 64) return SG_ERR_UNSUPPORTED;
    if (reinterpret_cast<uintptr_t>(Flt) % 16 || !mult(p.k_c * es, 16) || !mult((int64_t)p.N * es, 16) || (p.KW > 1 && !mult(p.k_kw * es, 16)) ||
        (p.KH > 1 && !mult(p.k_kh * es, 16))) return SG_ERR_UNSUPPORTED;
    const int64_t limit = (int64_t)1 << 39;      // byte strides below 2^40
    const int64_t Q = (int64_t)p.batch * p.Hin * p.Win, shift = (int64_t)p.dh * p.Win;
    if (p.i_w >= limit || p.k_c >= limit || Q > 0x7fffffff - 4096 || shift * p.i_w >= limit) return SG_ERR_UNSUPPORTED;
    const int64_t positions = (int64_t)(p.batch - 1) * p.Hin * p.Win + (int64_t)(p.Ho - 1) * p.Win + p.Wo;
    // (output offsets are 32-bit, those of the dead positions of the last image and beyond too)
    if ((int64_t)(p.batch + 1) * p.o_n + (int64_t)(p.Hin + 1) * p.o_h + (int64_t)(p.Win + 1) * p.o_w + p.N > 0x7fffffff) return SG_ERR_UNSUPPORTED;
    const int f_tiles = (p.N + BF - 1) / BF;
    // The sum of a whole reduction stays in the tensor core's accumulator, which truncates, and f32 factors are split in tf32 + bf16, as in
    // the im2col and the strip kernel.  Outputs outside the TMA rules and inputs that both leave alone (below 128 KiB) keep the accuracy
    // and the infinities of the CUDA-core kernel: the gather kernel's (error of 3x3x512 sums against f64: f32 2.2e-5 here, 1.2e-6
    // and less there; bf16 4.6e-6 and 5.6e-7).
    const bool im2col = tensor_takes(p, In, Flt, O);
    if (!forced && !im2col && launch_conv_strip(p, In, Flt, O, true, stream) != SG_OK) return SG_ERR_UNSUPPORTED;
    // share of the positions that are outputs: where it is low the im2col kernel, whose tiles hold outputs only, is the better one
    if (!forced && (double)p.M < 0.6 * (double)positions) return SG_ERR_UNSUPPORTED;
    int dev = 0, num_sms = 0, pdl = -1, single = 0;
    if (!tensor_device_info(&dev, &num_sms, &pdl, &single)) return SG_ERR_CUDA;

    const int row_span = (p.KW - 1) * p.dw;
    const int64_t full_span = (int64_t)(p.KH - 1) * shift + row_span;
    WideParams w{};
    F32Filter g{};
    if (f32) {
        // The im2col kernel deals a reduction out over the SMs: where there are few positions and much to sum it is the better one
        // (8 x 28 x 28, 3x3x256x256: 43.9 us here, 38.5 there; 16 x 56 x 56, 3x3x64x128: 32.3 against 41.6; 5 x 80 x 80, 3x3x16x128: 10.3 and 13.3; both
        // estimates are within a tenth or so).  Filters of 65 to 128 columns and three
        // taps or more that the strip kernel would keep resident run faster here whatever the estimates say (43 x 2934,
        // 3x32x128: 18.9 against 22.2; but one tap, 54 x 54, 1x1x48x96: 6.1 against 5.2).
        const double us = plan_f32(p, positions, f_tiles, row_span, full_span, num_sms, w, g);
        const bool strip = p.N <= 128 && p.N > 64 && mult(p.N, 32) && g.taps >= 3 && (int64_t)g.taps * w.kb <= 6;
        if (!forced && im2col && !strip && us >= 0.95 * tensor_estimate_us(p)) return SG_ERR_UNSUPPORTED;
    } else {
        // bf16: the im2col kernel where its estimate (5 % and 0.6 us low for convolutions) is clearly the lower one: 4 x 105 x 105, 5x5x64x96 24 us, here 48; 5 x 15 x 15,
        // 5x5x128x96 7.5 and 11.7.  With this margin 35 of 243 convolutions that this kernel took for their shape alone are more than 5 % faster, and one slower.
        // (Where the strip kernel would take over instead it is the slower one; single taps, which both kernels read once, and accumulating calls stay.)
        const double us = plan_bf16(p, positions, f_tiles, row_span, full_span, num_sms, w);
        if (!forced && im2col && !p.accumulate && p.KH * p.KW > 1 && us >= 1.15 * (0.63 + 1.05 * tensor_estimate_us(p)) &&
            (!conv_strip_preferred(p) || launch_conv_strip(p, In, Flt, O, true, stream) != SG_OK)) return SG_ERR_UNSUPPORTED;
    }
    if (w.BN == 0 || (int64_t)w.tiles * f_tiles > 0x7fffffff) return SG_ERR_UNSUPPORTED;
    w.row_step = w.per_row ? w.box_rows : (int)shift;

    alignas(64) CUtensorMap map_in, map_flt;
    {
        // {channel, position, filter row}: an overlapping view whose third dimension steps by dh*W_in positions (extent 1 when
        // one run serves all taps); positions beyond the input read as zero
        cuuint64_t dims[3] = {(cuuint64_t)p.C, (cuuint64_t)(w.per_row ? Q - (int64_t)(p.KH - 1) * shift : Q), (cuuint64_t)(w.per_row ? p.KH : 1)};
        cuuint64_t strides[2] = {(cuuint64_t)(p.i_w * es), (cuuint64_t)((w.per_row ? shift : Q) * p.i_w * es)};
        cuuint32_t box[3] = {(cuuint32_t)(128 / es), (cuuint32_t)w.box_rows, (cuuint32_t)(w.per_row ? p.KH : 1)};
        if (strides[1] >= ((cuuint64_t)1 << 40)) return SG_ERR_UNSUPPORTED;
        if (!tensor_encode_tiled(&map_in, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(In), dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B)) return SG_ERR_UNSUPPORTED;
    }
    const int64_t s_kw = p.KW > 1 ? p.k_kw : (int64_t)p.C * p.k_c, s_kh = p.KH > 1 ? p.k_kh : (int64_t)p.KW * s_kw;
    const int flt_rows = w.kb > 1 ? 64 : (p.C + 15) / 16 * 16;
    if (f32) {
        // {f, c, kw, kh}, box {128, channels of a slot, 1, 1}: rows of 512 bytes, read down the columns
        cuuint64_t dims[4] = {(cuuint64_t)p.N, (cuuint64_t)p.C, (cuuint64_t)p.KW, (cuuint64_t)p.KH};
        cuuint64_t strides[3] = {(cuuint64_t)(p.k_c * 4), (cuuint64_t)(s_kw * 4), (cuuint64_t)(s_kh * 4)};
        cuuint32_t box[4] = {BF, (cuuint32_t)g.chp, 1, 1};
        if (!tensor_encode_tiled(&map_flt, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(Flt), dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B)) return SG_ERR_UNSUPPORTED;
    } else if (p.N % 64 == 0) {
        cuuint64_t dims[5] = {64, (cuuint64_t)p.C, (cuuint64_t)(p.N / 64), (cuuint64_t)p.KW, (cuuint64_t)p.KH};
        cuuint64_t strides[4] = {(cuuint64_t)(p.k_c * 2), 128, (cuuint64_t)(s_kw * 2), (cuuint64_t)(s_kh * 2)};
        cuuint32_t box[5] = {64, (cuuint32_t)flt_rows, BF / 64, (cuuint32_t)p.KW, 1};
        if (!tensor_encode_tiled(&map_flt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(Flt), dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B)) return SG_ERR_UNSUPPORTED;
        w.flt_loads = 1; w.tap_bytes = 256 * flt_rows; w.half_bytes = 128 * flt_rows;
    } else {
        cuuint64_t dims[4] = {(cuuint64_t)p.N, (cuuint64_t)p.C, (cuuint64_t)p.KW, (cuuint64_t)p.KH};
        cuuint64_t strides[3] = {(cuuint64_t)(p.k_c * 2), (cuuint64_t)(s_kw * 2), (cuuint64_t)(s_kh * 2)};
        cuuint32_t box[4] = {64, (cuuint32_t)flt_rows, (cuuint32_t)p.KW, 1};
        if (!tensor_encode_tiled(&map_flt, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(Flt), dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B)) return SG_ERR_UNSUPPORTED;
        w.flt_loads = 2; w.tap_bytes = 128 * flt_rows; w.half_bytes = p.KW * 128 * flt_rows;
    }
    w.f_tiles = f_tiles; w.positions = (int)positions;
    w.N = p.batch; w.Hin = p.Hin; w.Win = p.Win; w.Hout = p.Ho; w.Wout = p.Wo; w.F = p.N;
    w.KH = p.KH; w.KW = p.KW; w.dw = p.dw;
    const int tmem_cols = w.bufs * w.BN + (f32 ? w.slots * 2 * g.chp : 0);
    w.tmem_cols = tmem_cols <= 128 ? 128 : tmem_cols <= 256 ? 256 : 512;
    w.o_n = (int)p.o_n; w.o_h = (int)p.o_h; w.o_w = (int)p.o_w;
    w.accumulate = p.accumulate; w.wait_prior = pdl == 0 ? 0 : 1;

    if (!tensor_ensure_smem_attr(f32 ? 182 : 159, f32 ? reinterpret_cast<const void *>(conv_wide_f32_kernel) : reinterpret_cast<const void *>(conv_wide_kernel),
                                 SMEM_LIMIT + 1024)) return SG_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    const int64_t items = (int64_t)w.tiles * f_tiles;
    cfg.gridDim = dim3((unsigned)std::min<int64_t>(items, num_sms), 1, 1);
    cfg.blockDim = dim3(f32 ? F32_THREADS : THREADS, 1, 1);
    cfg.dynamicSmemBytes = f32 ? 2 * g.stages * w.run_bytes + g.tiles * g.tile_bytes + 1024 : w.slots * w.slot_bytes + RUN_STAGES * w.run_bytes + 1024;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = w.wait_prior ? 1 : 0;
    const cudaError_t e = f32 ? cudaLaunchKernelEx(&cfg, conv_wide_f32_kernel, map_in, map_flt, g, w, O) : cudaLaunchKernelEx(&cfg, conv_wide_kernel, map_in, map_flt, w, O);
    count_launch();
    note_kernel(f32 ? "conv_wide_kernel<f32>" : "conv_wide_kernel<bf16>");
    *resident_filter = w.resident != 0;
    return e == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

sg_status conv_wide_read_status(cudaStream_t stream) { return read_status_word(stream); }

}  // namespace sg
