// Weight and bias gradient of a 3x3 convolution with at most 64 input and 64 output channels, all nine taps in one CTA.
//
// dW[co][r][s][ci] = sum_p dy[p][co] x[p + (r, s)][ci].  With 64 output channels half of an M = 128 MMA would be padding, and a CTA per
// filter column fetches dy and x three times (64 -> 64 channels at 224x224, batch 64: 465 us at 830 cycles per chunk of 64 pixels
// and column, paced by the fetches).  Here the A operand holds dy twice, the second time one image row further on, and the B operand x
// twice, likewise:
//                      x[p + (0, s)]      x[p + (1, s)]
//     dy[p]            tap row 0          tap row +1
//     dy[p + row]      tap row -1         (tap row 0 again: not used)
// The second panels are windows into the same boxes (one image row of halo below; the leading byte offset of the descriptor is one image row of
// the box, a whole number of 8-row swizzle groups), so a chunk is one box of dy and three of x, one per filter column: three
// 128 x 128 x 64 products, 36 KB instead of 72.  A pixel row missing at the top of the image meets the zero padding of x, one past the
// bottom reads zeros in dy.
//
// Bound: shared memory (per 8x8 chunk 288 cycles of TMA writes and 768 of MMA reads, which is also the MMAs' arithmetic).
// Each CTA takes a contiguous share of the chunks and writes a partial gradient, summed in CTA order by the reduce kernel.
//
// Warps: 0 = TMA loads, 1 = TMEM + MMA, 2..5 = bias sums from the dy boxes, then the epilogue.  Every wait is bounded and reports through
// the model's device status word.
#include "sb_umma.h"
#include "sb_tcgen05.cuh"

namespace sb {

namespace {

constexpr int C64_THREADS = 192, C64_MAX_STAGES = 6, C64_CTRL = 2048;
constexpr uint32_t C64_TMEM_COLS = 512;       // three accumulators of 128 columns

struct Conv64WgradParams {
    int bw, bh, bn;                  // pixel box of a chunk (64 pixels)
    int tiles_w, tiles_h;
    int total_chunks, chunks_per_cta, stages;
    int Cin, Cout;
    float* out;                      // [CTA][split_stride]: [Cout][9][Cin], then the bias gradient at bias_off
    long split_stride, bias_off;
    uint32_t* status;
};

__global__ void __launch_bounds__(C64_THREADS)
conv64_wgrad_kernel(const __grid_constant__ CUtensorMap mapDy, const __grid_constant__ CUtensorMap mapX, const Conv64WgradParams p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t row_bytes = (uint32_t)(p.bw * p.bn) * 128u, box = (uint32_t)(p.bh + 1) * row_bytes, stage_bytes = 4u * box;
    uint8_t* ctrl = smem + (size_t)p.stages * stage_bytes;
    uint64_t *full = (uint64_t*)ctrl, *empty = full + C64_MAX_STAGES, *acc_full = empty + C64_MAX_STAGES;
    uint32_t* tmem_slot = (uint32_t*)(acc_full + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    float* s_part = (float*)(ctrl + 512);      // [3][64]: bias sums of three warps
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int c_begin = blockIdx.x * p.chunks_per_cta, n_chunks = min(p.chunks_per_cta, p.total_chunks - c_begin);
    const uint32_t smem0 = smem_u32(smem);

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 5); }     // (MMA and four bias warps)
        mbar_init(acc_full, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) {
        tmem_alloc(tmem_slot, C64_TMEM_COLS);
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
        int cw = c_begin % p.tiles_w, ch = c_begin / p.tiles_w % p.tiles_h, cn = c_begin / (p.tiles_w * p.tiles_h), s = 0;
        uint32_t ph = 1u;             // (a fresh barrier reports the phase before its first as complete)
        bool ok = true;
        for (int c = 0; c < n_chunks; ++c) {
            ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], ph) ? 1 : 0) != 0;
            if (!ok) break;
            const uint32_t dst = smem0 + (uint32_t)s * stage_bytes, bar = full0 + 8u * (uint32_t)s;
            const int w0 = cw * p.bw, h0 = ch * p.bh, n0 = cn * p.bn;
            mbar_expect_tx_el(bar, stage_bytes, el);
            tma_load_4d_el(&mapDy, dst, bar, 0, w0, n0, h0, el);                                           // (c, w, n, h)
#pragma unroll
            for (int t = 0; t < 3; ++t) tma_load_4d_el(&mapX, dst + (uint32_t)(t + 1) * box, bar, 0, w0 + t - 1, n0, h0, el);
            if (++cw == p.tiles_w) { cw = 0; if (++ch == p.tiles_h) { ch = 0; ++cn; } }
            if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_TMA); }
    } else if (warp == 1) {
        constexpr uint32_t idesc = make_idesc(128, 1, 1);
        const uint32_t elected = elect_one() ? 1u : 0u;
        const uint64_t d0 = make_desc(smem0, row_bytes);
        const uint32_t lo0 = (uint32_t)d0, hi = (uint32_t)(d0 >> 32), box16 = box >> 4, stage16 = stage_bytes >> 4;
        int s = 0;
        uint32_t ph = 0u, lo = lo0;
        bool ok = true;
        for (int c = 0; c < n_chunks; ++c) {
            ok = __all_sync(0xffffffffu, mbar_wait(&full[s], ph) ? 1 : 0) != 0;
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int t = 0; t < 3; ++t)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma_bf16_lohi(tmem_base + 128u * t, lo + 128u * kk, hi, lo + (uint32_t)(t + 1) * box16 + 128u * kk, hi, idesc, (c > 0 || kk > 0) ? 1u : 0u, elected);
            if (elected) umma_commit(&empty[s]);
            __syncwarp();
            lo += stage16;
            if (++s == p.stages) { s = 0; ph ^= 1u; lo = lo0; }
        }
        if (ok && elected) umma_commit(acc_full);
        __syncwarp();
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_MMA); }
    } else {
        const int q = warp % 4, row = q * 32 + lane;
        float* out = p.out + (size_t)blockIdx.x * p.split_stride;
        // Bias gradient: a thread adds one 16-byte piece (8 channels) of every sixteenth of the chunk's 64 pixel rows, in a fixed order.
        const int piece = row % 8, rg = row / 8;
        const uint32_t at0 = smem0 + (uint32_t)rg * 128u + (uint32_t)((piece ^ (rg & 7)) << 4);
        float bs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        int s = 0;
        uint32_t ph = 0u, at = at0;
        bool ok = true;
        for (int c = 0; c < n_chunks; ++c) {
            ok = __all_sync(0xffffffffu, mbar_wait(&full[s], ph) ? 1 : 0) != 0;
            if (!ok) break;
            uint32_t v[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[i][0]), "=r"(v[i][1]), "=r"(v[i][2]), "=r"(v[i][3]) : "r"(at + 2048u * i));
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    bs[2 * j] += __uint_as_float(v[i][j] << 16);
                    bs[2 * j + 1] += __uint_as_float(v[i][j] & 0xffff0000u);
                }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&empty[s]));
            at += stage_bytes;
            if (++s == p.stages) { s = 0; ph ^= 1u; at = at0; }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            bs[j] += __shfl_down_sync(0xffffffffu, bs[j], 16);
            bs[j] += __shfl_down_sync(0xffffffffu, bs[j], 8);
        }
        if (q > 0 && lane < 8)
#pragma unroll
            for (int j = 0; j < 8; ++j) s_part[(q - 1) * 64 + piece * 8 + j] = bs[j];
        asm volatile("bar.sync 1, 128;" ::: "memory");          // (the four warps; each of them gets here, also after a timeout)
        if (ok && q == 0 && lane < 8)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = piece * 8 + j;
                if (c < p.Cout) out[p.bias_off + c] = ((bs[j] + s_part[c]) + s_part[64 + c]) + s_part[128 + c];
            }
        ok = __all_sync(0xffffffffu, ok && mbar_wait(acc_full, 0u) ? 1 : 0) != 0;
        if (!ok) {
            if (lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_EPI); }
        } else {
            // rows 0..63: tap rows 0 and +1 of output channel `row`; rows 64..127: tap row -1 of channel row - 64
            tc_fence_after();
            const int co = row % 64, panels = q < 2 ? 2 : 1;
            float* dst0 = out + (size_t)co * 9 * p.Cin;
#pragma unroll 1
            for (int t = 0; t < 3; ++t)
#pragma unroll 1
                for (int pn = 0; pn < panels; ++pn) {
                    const int tap = 3 * (q < 2 ? 1 + pn : 0) + t;
                    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(128 * t + 64 * pn);
#pragma unroll 1
                    for (int c0 = 0; c0 < 64; c0 += 32) {
                        uint32_t v[2][16];
                        tmem_ld16(taddr + c0, v[0]);
                        tmem_ld16(taddr + c0 + 16, v[1]);
                        tmem_ld_wait();
                        float4* dst = (float4*)(dst0 + (size_t)tap * p.Cin + c0);
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (co < p.Cout && c0 + 16 * h < p.Cin)        // (whole 16-column chunks)
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    dst[4 * h + j] = make_float4(__uint_as_float(v[h][4 * j]), __uint_as_float(v[h][4 * j + 1]), __uint_as_float(v[h][4 * j + 2]), __uint_as_float(v[h][4 * j + 3]));
                    }
                }
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
        tmem_dealloc(tmem_base, C64_TMEM_COLS);
    }
}

int smem_of(int bw, int bh, int bn, int stages) { return stages * 4 * (bh + 1) * bw * bn * 128 + 1024 + C64_CTRL; }

}  // namespace

int conv64_wgrad_stages(int bw, int bh, int bn)
{
    int s = C64_MAX_STAGES;
    while (s > 0 && smem_of(bw, bh, bn, s) > 227 * 1024) --s;
    return s;
}

cudaError_t launch_conv64_wgrad(const Conv64WgradArgs& a, cudaStream_t st)
{
    Conv64WgradParams p{};
    p.bw = a.bw; p.bh = a.bh; p.bn = a.bn;
    p.tiles_w = a.tiles_w; p.tiles_h = a.tiles_h;
    p.total_chunks = a.total_chunks; p.chunks_per_cta = a.chunks_per_cta;
    p.stages = conv64_wgrad_stages(a.bw, a.bh, a.bn);
    p.Cin = a.Cin; p.Cout = a.Cout;
    p.out = a.out; p.split_stride = a.split_stride; p.bias_off = a.bias_off; p.status = a.status;
    if (p.stages < 2 || a.bw * a.bh * a.bn != 64 || (a.bw * a.bn) % 8 != 0 || a.Cin > 64 || a.Cout > 64) return cudaErrorInvalidValue;
    const cudaError_t e = raise_smem_limit<conv64_wgrad_kernel>(227 * 1024);
    if (e != cudaSuccess) return e;
    return pdl_launch(conv64_wgrad_kernel, dim3((a.total_chunks + a.chunks_per_cta - 1) / a.chunks_per_cta), dim3(C64_THREADS), (size_t)smem_of(a.bw, a.bh, a.bn, p.stages), st,
                      *a.mapDy, *a.mapX, p);
}

}  // namespace sb
