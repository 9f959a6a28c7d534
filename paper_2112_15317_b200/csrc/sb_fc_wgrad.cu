// Stored weight and bias gradient of a large fully-connected layer: dW = dY^T X, float.
//
// Bound: the HBM writes of the gradient (the reduction is only the batch; a kernel that only writes 411 MB takes 62 us).  One CTA per SM
// walks tiles of 256 outputs x 128 inputs (neighbours along a row of the gradient run at the same time) with an operand ring that
// runs on across them and two accumulators, which two groups of four epilogue warps drain, half of the outputs each.  The
// accumulator is the transposed tile, a lane per INPUT: a register of a warp is 128 contiguous bytes of one gradient row and goes out
// as it is.  With a lane per output the tile has to be turned in shared memory, whose port (tile in, tile out, stores, MMA operands, TMA
// writes) then takes longer than the HBM.  25088 -> 4096 at batch 128: one CTA per tile, staged, 103 us; this walk, staged, 112; 32-byte
// pieces of rows straight from the registers, 91; this form, 83.
//
// Warps: 0 = TMA loads, 1 = TMEM + MMA, 2 = bias sums, 4..7 and 8..11 = epilogue.  Every wait is bounded and reports through the model's device
// status word.
#include "sb_umma.h"
#include "sb_tcgen05.cuh"

namespace sb {

namespace {

constexpr int FW_THREADS = 384, FW_STAGES = 4;
constexpr int FW_A_BYTES = 16384, FW_STAGE_BYTES = FW_A_BYTES + 32768;      // 64 batch rows: 128 columns of X, 256 of dY
constexpr int FW_SMEM = FW_STAGES * FW_STAGE_BYTES + 1024 + 1024;
constexpr uint32_t FW_TMEM_COLS = 512;

struct FcWgradParams {
    int out_f, in_f, n_tiles, tiles, chunks;
    float* out;              // [out_f][in_f]
    float* bias;             // [out_f]
    uint32_t* status;
};

__global__ void __launch_bounds__(FW_THREADS)
fc_wgrad_kernel(const __grid_constant__ CUtensorMap mapDy, const __grid_constant__ CUtensorMap mapX, const FcWgradParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* ctrl = smem + FW_STAGES * FW_STAGE_BYTES;
    uint64_t *full = (uint64_t*)ctrl, *empty = full + FW_STAGES, *acc_full = empty + FW_STAGES, *acc_empty = acc_full + 2;
    uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* epi_stop = tmem_slot + 2;        // [2]: written by the warps of one epilogue group only
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t smem0 = smem_u32(smem);

    if (threadIdx.x == 0) {
        for (int s = 0; s < FW_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 2); }     // (MMA and bias warp)
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 8); epi_stop[b] = 0; }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) {
        tmem_alloc(tmem_slot, FW_TMEM_COLS);
        tmem_relinquish();
    }
    pdl_prologue();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        const uint32_t el = elect_one() ? 1u : 0u;
        const uint32_t full0 = smem_u32(full);
        int s = 0;
        uint32_t ph = 1u;             // (a fresh barrier reports the phase before its first as complete)
        bool ok = true;
        for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x) {
            const int mt = t / p.n_tiles, m0 = mt * 256, n0 = (t - mt * p.n_tiles) * 128;
            for (int c = 0; c < p.chunks; ++c) {
                ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], ph) ? 1 : 0) != 0;
                if (!ok) break;
                const uint32_t dst = smem0 + (uint32_t)(s * FW_STAGE_BYTES), bar = full0 + 8u * (uint32_t)s;
                mbar_expect_tx_el(bar, (uint32_t)FW_STAGE_BYTES, el);
#pragma unroll
                for (int j = 0; j < 2; ++j) tma_load_4d_el(&mapX, dst + 8192u * j, bar, n0 + 64 * j, 0, 0, c * 64, el);
#pragma unroll
                for (int j = 0; j < 4; ++j) tma_load_4d_el(&mapDy, dst + FW_A_BYTES + 8192u * j, bar, m0 + 64 * j, 0, 0, c * 64, el);
                if (++s == FW_STAGES) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_TMA); }
    } else if (warp == 1) {
        constexpr uint32_t idesc = make_idesc(256, 1, 1);
        const uint32_t elected = elect_one() ? 1u : 0u;
        const uint64_t dA = make_desc(smem0, 8192), dB = make_desc(smem0 + FW_A_BYTES, 8192);
        const uint32_t a_hi = (uint32_t)(dA >> 32), b_hi = (uint32_t)(dB >> 32);
        int s = 0, i = 0;
        uint32_t ph = 0u;
        bool ok = true;
        for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x, ++i) {
            const int buf = i & 1;
            ok = __all_sync(0xffffffffu, mbar_wait(&acc_empty[buf], (uint32_t)(((i >> 1) + 1) & 1)) ? 1 : 0) != 0;
            if (!ok) break;
            for (int c = 0; c < p.chunks; ++c) {
                ok = __all_sync(0xffffffffu, mbar_wait(&full[s], ph) ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const uint32_t off = (uint32_t)(s * FW_STAGE_BYTES) >> 4;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma_bf16_lohi(tmem_base + 256u * buf, (uint32_t)dA + off + 128u * kk, a_hi, (uint32_t)dB + off + 128u * kk, b_hi, idesc, (c > 0 || kk > 0) ? 1u : 0u, elected);
                if (elected) umma_commit(&empty[s]);
                __syncwarp();
                if (++s == FW_STAGES) { s = 0; ph ^= 1u; }
            }
            if (ok && elected) umma_commit(&acc_full[buf]);
            __syncwarp();
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_MMA); }
    } else if (warp == 2) {
        // Bias gradient of the output tiles whose first input tile falls to this CTA: column sums of dY over the batch.  A lane takes one
        // 16-byte piece (8 channels), row group by row group (rows r, r + 8, ...); the groups are added in pairs, then in order -- the
        // order of the one-CTA-per-tile kernel, whose folded update has to give the same bits.
        int s = 0;
        uint32_t ph = 0u;
        bool ok = true;
        for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x) {
            const bool mine = t % p.n_tiles == 0;
            float bs[8][8];
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int j = 0; j < 8; ++j) bs[r][j] = 0.f;
            for (int c = 0; c < p.chunks; ++c) {
                ok = __all_sync(0xffffffffu, mbar_wait(&full[s], ph) ? 1 : 0) != 0;
                if (!ok) break;
                if (mine) {
                    const uint32_t at = smem0 + (uint32_t)(s * FW_STAGE_BYTES + FW_A_BYTES) + (uint32_t)(lane / 8) * 8192u;
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            uint32_t v[4];
                            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                                         : "r"(at + (uint32_t)(8 * i + r) * 128u + (uint32_t)(((lane % 8) ^ r) << 4)));
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                bs[r][2 * j] += __uint_as_float(v[j] << 16);
                                bs[r][2 * j + 1] += __uint_as_float(v[j] & 0xffff0000u);
                            }
                        }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&empty[s]));
                if (++s == FW_STAGES) { s = 0; ph ^= 1u; }
            }
            if (!ok || !mine) continue;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = t / p.n_tiles * 256 + lane * 8 + j;
                if (c < p.out_f) p.bias[c] = (((bs[0][j] + bs[1][j]) + (bs[2][j] + bs[3][j])) + (bs[4][j] + bs[5][j])) + (bs[6][j] + bs[7][j]);
            }
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_EPI); }
    } else if (warp >= 4) {
        const int q = warp % 4, group = warp / 4 - 1;
        auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory"); };
        int i = 0;
        for (int t = blockIdx.x; t < p.tiles; t += gridDim.x, ++i) {
            const int buf = i & 1, mt = t / p.n_tiles, row0 = mt * 256 + 128 * group, col = (t - mt * p.n_tiles) * 128 + q * 32 + lane;
            bool ok = true;
            if (lane == 0) ok = mbar_wait(&acc_full[buf], (uint32_t)((i >> 1) & 1));
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok && lane == 0) { epi_stop[group] = 1; *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_EPI); }
            group_sync();                 // a timeout seen by one warp of the group is seen by all; together they write 512 bytes of a row at a time
            const bool stop = epi_stop[group] != 0;
            tc_fence_after();
            float* dst = p.out + (size_t)row0 * p.in_f + col;
#pragma unroll 1
            for (int r0 = 0; r0 < 128 && row0 + r0 < p.out_f && !stop; r0 += 32) {
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(256 * buf + 128 * group + r0);
                uint32_t v[2][16];
                tmem_ld16(taddr, v[0]);
                tmem_ld16(taddr + 16, v[1]);
                tmem_ld_wait();
                if (col < p.in_f)
#pragma unroll
                    for (int r = 0; r < 32; ++r)
                        if (row0 + r0 + r < p.out_f) __stcs(dst + (size_t)r * p.in_f, __uint_as_float(v[r / 16][r % 16]));
                dst += (size_t)32 * p.in_f;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[buf]));
            group_sync();                 // (epi_stop has been read)
            if (stop) break;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {       // copies may be in flight: leave them time before the shared memory goes
        const uint64_t t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) { }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, FW_TMEM_COLS);
    }
}

}  // namespace

cudaError_t launch_fc_wgrad(const FcWgradArgs& a, cudaStream_t st)
{
    FcWgradParams p{};
    p.out_f = a.out_f; p.in_f = a.in_f;
    p.n_tiles = (a.in_f + 127) / 128;
    p.tiles = (a.out_f + 255) / 256 * p.n_tiles;
    p.chunks = (a.batch + 63) / 64;
    p.out = a.out; p.bias = a.bias; p.status = a.status;
    const cudaError_t e = raise_smem_limit<fc_wgrad_kernel>(FW_SMEM);
    if (e != cudaSuccess) return e;
    return pdl_launch(fc_wgrad_kernel, dim3(p.tiles < 148 ? p.tiles : 148), dim3(FW_THREADS), (size_t)FW_SMEM, st, *a.mapDy, *a.mapX, p);
}

}  // namespace sb
