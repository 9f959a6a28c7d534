// Input-layer 3x3 convolution (1, 3 or 4 input channels) on the tcgen05 tensor cores.
//
// With so few input channels the reduction of one output pixel is only 9*Cin values (27 for RGB), far
// below a 64-wide TMA box, so the im2col operand is built by the threads themselves: a "patch tile" of
// one 128-byte row per pixel, in the 128-byte-swizzled shared-memory layout the MMA descriptors expect
// (16-byte chunk j of row r sits at r*128 + ((j ^ (r & 7)) << 4)).  The same tile serves both passes:
//   forward : D[pixel, cout] = patch[pixel, :] . W[cout, :]      A = patch tile (K-major), B = weights (K-major)
//   wgrad   : D[cout, k]     = sum_pixel dy[pixel, cout] * patch[pixel, k]
//                                                               A = dy tile (MN-major, by TMA), B = patch tile (MN-major)
//
// The three taps of a filter row are 3*Cin neighbouring elements of an image row, so a patch row is three runs, each padded to an
// even number of slots: k = r * SLOTS + s*Cin + c (10 slots a run for RGB, 30 in all), and k = 3 * SLOTS holds 1 for every valid
// pixel in the weight-gradient pass, where the same MMA then yields the bias gradient.  The image rows a tile touches are first
// copied (cp.async, one tile ahead) into a window in shared memory with zeros left and right of every row and a row of zeros
// between images, which makes every run a few 32-bit words and one funnel shift each, without any bounds test.
//
// Bound: the forward pass writes 2 * Cout bytes a pixel, the weight gradient reads them (HBM); below that, the latency chain of
// a tile (window -> patch -> MMA -> epilogue), which the CTAs resident on an SM hide for one another.  Gathered as 27 two-byte
// values a pixel with their bounds tests the two passes took 180 and 209 us at 64 x 224x224 images (now 120 and 125; 3.4 TB/s), and
// 17 and 23 us at 128 x 32x32 (15 and 17).  Every mbarrier wait is bounded and reports through the model's device status word.
#include "sb_umma.h"
#include "sb_tcgen05.cuh"

namespace sb {

namespace {

constexpr int CI_THREADS = 128;
constexpr int CI_LEFT = 8;          // elements in front of an image row in the window (16 bytes; the last Cin of them are the zero padding)
constexpr int CI_TILE = 128;        // pixels per tile (flat pixel index)

template <int CIN> struct Patch {
    static constexpr int RUN = 3 * CIN, SLOTS = (RUN + 1) / 2 * 2, NW = SLOTS / 2;      // elements, slots and words of a filter row's run
    static constexpr int ONES = 3 * SLOTS;                                              // the column of ones
    static constexpr int COLS = (ONES + 1 + 15) / 16 * 16;                              // columns up to the next MMA step (16, 32, 48)
    static constexpr int KSTEPS = (ONES + 15) / 16;                                     // steps that hold weights
    static constexpr int CHUNKS = COLS / 8;
};

// n / d for n < 2^31 through the reciprocal floor(2^32 / d) + 1 (0 stands for d = 1): the estimate is exact or one too high
__host__ __device__ __forceinline__ uint32_t rcp_of(int d) { return d <= 1 ? 0u : (uint32_t)(0x100000000ull / (uint32_t)d) + 1u; }
__device__ __forceinline__ int div_rcp(int n, uint32_t mul, int d)
{
    if (mul == 0u) return n;
    uint32_t q = __umulhi((uint32_t)n, mul);
    if (q * (uint32_t)d > (uint32_t)n) --q;
    return (int)q;
}

struct ConvInGeom {
    const __nv_bfloat16* x;        // [images][H][W][Cin], or tab: per-replica buffers of b_per_rep images
    PtrTab tab; int use_tab, b_per_rep;
    int H, W, npix, n_img, Cout;
    uint32_t rcp_w, rcp_h, rcp_hp, rcp_rep;
    int pitch;                     // window: elements from row to row (a multiple of 8)
    int vpr, ve;                   // vectors per image row, elements per vector (8, 2; 1: plain copies)
    int win_bytes;                 // one window buffer
};

// Copies the window of the tile that starts at pixel p0: image row h of image n is padded row n * (H + 1) + h + 1, rows
// n * (H + 1) are zero.  Asynchronous (16- or 4-byte copies) unless rows are an odd number of elements.
template <int CIN>
__device__ __forceinline__ void fetch_window(const ConvInGeom& g, __nv_bfloat16* win, int p0)
{
    const int f0 = div_rcp(p0, g.rcp_w, g.W), n0 = div_rcp(f0, g.rcp_h, g.H);
    const int last = min(p0 + CI_TILE, g.npix) - 1;
    const int f1 = div_rcp(last, g.rcp_w, g.W), n1 = div_rcp(f1, g.rcp_h, g.H);
    const int q0 = f0 + n0, rows = f1 + n1 - q0 + 3;         // (padded row of the image row above pixel p0's)
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int r = warp; r < rows; r += CI_THREADS / 32) {
        const int q = q0 + r, n = div_rcp(q, g.rcp_hp, g.H + 1), h = q - n * (g.H + 1) - 1;
        const bool in = h >= 0 && n < g.n_img;
        const __nv_bfloat16* src = g.use_tab ? (const __nv_bfloat16*)g.tab.p[0] : g.x;     // (an address that may be read, for the rows of zeros)
        if (in) {
            const int rep = g.use_tab ? div_rcp(n, g.rcp_rep, g.b_per_rep) : 0;
            if (g.use_tab) src = (const __nv_bfloat16*)g.tab.p[rep];
            src += ((size_t)(n - rep * g.b_per_rep) * g.H + h) * (size_t)(g.W * CIN);
        }
        __nv_bfloat16* dst = win + r * g.pitch + CI_LEFT;
        if (g.ve == 8) {
            const uint32_t d = smem_u32(dst), bytes = in ? 16u : 0u;
            for (int c = lane; c < g.vpr; c += 32) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + 16u * c), "l"(src + (in ? 8 * c : 0)), "r"(bytes) : "memory");
        } else if (g.ve == 2) {
            const uint32_t d = smem_u32(dst), bytes = in ? 4u : 0u;
            for (int c = lane; c < g.vpr; c += 32) asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d + 4u * c), "l"(src + (in ? 2 * c : 0)), "r"(bytes) : "memory");
        } else {
            for (int c = lane; c < g.vpr; c += 32) dst[c] = in ? src[c] : __nv_bfloat16();
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void window_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// The patch row of pixel p of the tile that starts at p0, as 32-bit words; zeros past the last pixel.
template <int CIN>
__device__ __forceinline__ void build_patch(const ConvInGeom& g, const __nv_bfloat16* win, int p0, int p, bool with_ones, uint32_t (&out)[Patch<CIN>::COLS / 2])
{
    using P = Patch<CIN>;
#pragma unroll
    for (int k = 0; k < P::COLS / 2; ++k) out[k] = 0u;
    if (p >= g.npix) return;
    const int f0 = div_rcp(p0, g.rcp_w, g.W), q0 = f0 + div_rcp(f0, g.rcp_h, g.H);
    const int f = div_rcp(p, g.rcp_w, g.W), w = p - f * g.W, lr = f + div_rcp(f, g.rcp_h, g.H) - q0;
    const int e0 = lr * g.pitch + CI_LEFT + (w - 1) * CIN;
    const uint32_t sh = (uint32_t)(e0 & 1) * 16u;
    const uint32_t* at = (const uint32_t*)win + (e0 >> 1);
#pragma unroll
    for (int r = 0; r < 3; ++r, at += g.pitch / 2) {
        uint32_t v[P::NW];
#pragma unroll
        for (int k = 0; k < P::NW; ++k) v[k] = at[k];
        if (P::RUN % 2 == 0) {
#pragma unroll
            for (int k = 0; k < P::NW; ++k) out[r * P::NW + k] = v[k];
        } else {
#pragma unroll
            for (int k = 0; k + 1 < P::NW; ++k) out[r * P::NW + k] = __funnelshift_r(v[k], v[k + 1], sh);
            out[r * P::NW + P::NW - 1] = (v[P::NW - 1] >> sh) & 0xffffu;
        }
    }
    if (with_ones) out[P::ONES / 2] = 0x3F80u;     // bf16 1.0
}
template <int CIN>
__device__ __forceinline__ void store_patch(uint8_t* tile, int row, const uint32_t (&v)[Patch<CIN>::COLS / 2])
{
#pragma unroll
    for (int j = 0; j < Patch<CIN>::CHUNKS; ++j)
        *(uint4*)(tile + row * 128 + ((j ^ (row & 7)) << 4)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// both window buffers, so that what the copies leave out (the padding) stays zero
__device__ __forceinline__ void clear_windows(uint8_t* win, int bytes)
{
    for (int i = threadIdx.x; i < bytes / 16; i += CI_THREADS) *(uint4*)(win + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// Forward: persistent CTAs, one 128-pixel tile per iteration, the next tile's window on its way meanwhile
// ------------------------------------------------------------------------------------------------
template <int CIN>
__global__ void __launch_bounds__(CI_THREADS)
conv_in_fwd_umma_kernel(const __grid_constant__ CUtensorMap mapY, const __grid_constant__ ConvInGeom g, const __nv_bfloat16* __restrict__ wt,
                        const float* __restrict__ bias, int relu, int n_tiles, uint32_t* status)
{
    using P = Patch<CIN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;                               // patch tile, then the output tile: 128 rows x 128 B
    uint8_t* sB = smem + 16384;                       // Cout rows x 128 B
    float* s_bias = (float*)(sB + 8192);              // [64]
    uint8_t* win = sB + 8192 + 256;                   // two window buffers
    uint64_t* bar = (uint64_t*)(win + 2 * g.win_bytes);
    uint32_t* tmem_slot = (uint32_t*)(bar + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, row = threadIdx.x;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        tmem_alloc(tmem_slot, 64);
        tmem_relinquish();
    }
    clear_windows(win, 2 * g.win_bytes);
    __syncthreads();
    pdl_prologue();
    fetch_window<CIN>(g, (__nv_bfloat16*)win, (int)blockIdx.x * CI_TILE);
    // weights: row n = three runs of W[n], zeros in the padding slots (only the chunks the MMA reads are written)
    for (int n = threadIdx.x; n < g.Cout; n += CI_THREADS) {
        const __nv_bfloat16* wr = wt + (size_t)n * 9 * CIN;
#pragma unroll
        for (int j = 0; j < 2 * P::KSTEPS; ++j) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t two = 0u;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int k = 8 * j + 2 * e + u, r = k / P::SLOTS, t = k % P::SLOTS;
                    if (r < 3 && t < P::RUN) two |= (uint32_t)__bfloat16_as_ushort(wr[r * P::RUN + t]) << (16 * u);
                }
                pk[e] = two;
            }
            *(uint4*)(sB + n * 128 + ((j ^ (n & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
        s_bias[n] = bias[n];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t idesc = make_idesc(g.Cout, 0, 0);
    const uint64_t dA = make_desc(smem_u32(sA), 16), dB = make_desc(smem_u32(sB), 16);
    const uint32_t elected = warp == 0 && elect_one() ? 1u : 0u;
    uint32_t phase = 0;
    int wb = 0;

    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, wb ^= 1) {
        const int p0 = tile * CI_TILE, p = p0 + row;
        window_wait();
        if (threadIdx.x == 0) tma_store_wait_read();       // the previous output tile has left sA
        __syncthreads();
        if (tile + (int)gridDim.x < n_tiles) fetch_window<CIN>(g, (__nv_bfloat16*)(win + (wb ^ 1) * g.win_bytes), p0 + (int)gridDim.x * CI_TILE);
        {
            uint32_t v[P::COLS / 2];
            build_patch<CIN>(g, (const __nv_bfloat16*)(win + wb * g.win_bytes), p0, p, false, v);
            store_patch<CIN>(sA, row, v);
        }
        fence_async_smem();          // the tensor core reads shared memory through the async proxy
        __syncthreads();
        if (warp == 0) {             // (the whole warp in lock-step, one elected lane issues)
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < P::KSTEPS; ++kk)
                umma_bf16_lohi(tmem_base, (uint32_t)dA + 2u * kk, (uint32_t)(dA >> 32), (uint32_t)dB + 2u * kk, (uint32_t)(dB >> 32), idesc, kk > 0 ? 1u : 0u, elected);
            if (elected) umma_commit(bar);
            __syncwarp();
        }
        bool ok = true;
        if (lane == 0) ok = mbar_wait(bar, phase);
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        phase ^= 1u;
        if (!ok) {
            if (lane == 0) { *abort_flag = 1; atomicMax(status, (uint32_t)DEV_TIMEOUT_EPI); }
        } else {
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16);
            // output row = up to 128 bytes, staged in the patch tile's buffer (the MMA has consumed it) in the 128-byte swizzle of
            // the output map, so that one TMA store writes the tile in full lines
            const uint32_t row_s = smem_u32(sA) + (uint32_t)row * 128u, sw = (uint32_t)(row & 7), bias_s = smem_u32(s_bias);
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 16) {
                if (c0 >= g.Cout) break;
                uint32_t v[16], pk[8];
                tmem_ld16(taddr + c0, v);
                float b[16];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(b[4 * j]), "=f"(b[4 * j + 1]), "=f"(b[4 * j + 2]), "=f"(b[4 * j + 3]) : "r"(bias_s + (uint32_t)(c0 + 4 * j) * 4u));
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    __nv_bfloat162 t = __floats2bfloat162_rn(__uint_as_float(v[2 * j]) + b[2 * j], __uint_as_float(v[2 * j + 1]) + b[2 * j + 1]);
                    if (relu) t = __hmax2(t, __nv_bfloat162(__nv_bfloat16(0.f), __nv_bfloat16(0.f)));      // (NaN -> 0, as the reference path)
                    pk[j] = *(uint32_t*)&t;
                }
                const uint32_t j0 = (uint32_t)c0 >> 3;
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row_s + ((j0 ^ sw) << 4)), "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3]) : "memory");
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row_s + (((j0 + 1u) ^ sw) << 4)), "r"(pk[4]), "r"(pk[5]), "r"(pk[6]), "r"(pk[7]) : "memory");
            }
        }
        fence_async_smem();
        tc_fence_before();
        __syncthreads();             // accumulator drained, output tile staged
        if (*abort_flag) break;
        if (threadIdx.x == 0) {
            tma_store_4d(&mapY, smem_u32(sA), 0, p0, 0, 0);     // rows past the last pixel are clipped by the tensor map
            tma_store_commit();
        }
    }
    window_wait();
    if (threadIdx.x == 0) tma_store_wait_read();   // shared memory may be released once the stores have read it; the writes complete with the grid
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 64);
    }
}

// ------------------------------------------------------------------------------------------------
// Weight + bias gradient: each CTA accumulates a contiguous range of 128-pixel chunks into one TMEM accumulator D[cout, k] and
// writes it as a partial buffer [Cout*9*CIN weights | Cout biases].  The dy tile and the window of the next chunk are on their way
// while this one is multiplied.
// ------------------------------------------------------------------------------------------------
template <int CIN>
__global__ void __launch_bounds__(CI_THREADS)
conv_in_wgrad_umma_kernel(const __grid_constant__ CUtensorMap mapDy, const __grid_constant__ ConvInGeom g, float* __restrict__ part, long stride_floats,
                          int n_chunks, int chunks_per_cta, uint32_t* status)
{
    using P = Patch<CIN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    // dy tiles: 128 pixel rows x 128 B (64 couts, zeros past the last one).  The MMA's rows 64.. (couts that do not exist) read what
    // lies 16 KB behind a tile; they are not stored.
    uint8_t* sDy = smem;                              // [2]
    uint8_t* sP = smem + 2 * 16384;                   // patch tile
    uint8_t* win = sP + 16384;                        // two window buffers
    uint64_t* full = (uint64_t*)(win + 2 * g.win_bytes);   // [2] dy tile landed
    uint64_t* done = full + 2;                        // the chunk's MMAs have completed
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, row = threadIdx.x;
    const int c_begin = (int)blockIdx.x * chunks_per_cta;
    const int n_iters = min(c_begin + chunks_per_cta, n_chunks) - c_begin;
    if (n_iters <= 0) return;      // uniform over the CTA (the host sizes the grid so that this does not happen)

    if (threadIdx.x == 0) {
        mbar_init(&full[0], 1); mbar_init(&full[1], 1);
        mbar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        tmem_alloc(tmem_slot, 64);
        tmem_relinquish();
    }
    clear_windows(win, 2 * g.win_bytes);
    __syncthreads();
    pdl_prologue();
    fetch_window<CIN>(g, (__nv_bfloat16*)win, c_begin * CI_TILE);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 2 && k < n_iters; ++k) {
            mbar_expect_tx(&full[k], 16384u);
            tma_load_4d(&mapDy, sDy + k * 16384, &full[k], 0, (c_begin + k) * CI_TILE, 0, 0);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    constexpr uint32_t idesc = make_idesc(P::COLS, 1, 1);
    const uint64_t dDy = make_desc(smem_u32(sDy), 16384), dP = make_desc(smem_u32(sP), 8192);
    const uint32_t elected = warp == 0 && elect_one() ? 1u : 0u;

    for (int it = 0; it < n_iters; ++it) {
        const int s = it & 1, p0 = (c_begin + it) * CI_TILE;
        window_wait();
        __syncthreads();
        if (it + 1 < n_iters) fetch_window<CIN>(g, (__nv_bfloat16*)(win + (s ^ 1) * g.win_bytes), p0 + CI_TILE);
        uint32_t v[P::COLS / 2];
        build_patch<CIN>(g, (const __nv_bfloat16*)(win + s * g.win_bytes), p0, p0 + row, true, v);
        bool ok = true;
        if (it > 0) {
            // the MMAs of the chunk before have read the patch tile and its dy tile
            if (lane == 0) ok = mbar_wait(done, (uint32_t)((it - 1) & 1));
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok && lane == 0) { *abort_flag = 1; atomicMax(status, (uint32_t)DEV_TIMEOUT_TMA); }
            if (ok && threadIdx.x == 0 && it + 1 < n_iters) {
                mbar_expect_tx(&full[s ^ 1], 16384u);
                tma_load_4d(&mapDy, sDy + (s ^ 1) * 16384, &full[s ^ 1], 0, p0 + CI_TILE, 0, 0);
            }
        }
        store_patch<CIN>(sP, row, v);
        fence_async_smem();
        __syncthreads();
        if (*abort_flag) break;
        if (warp == 0) {             // (the whole warp in lock-step, one elected lane issues)
            if (!__all_sync(0xffffffffu, mbar_wait(&full[s], (uint32_t)((it / 2) & 1)) ? 1 : 0)) {
                if (lane == 0) { *abort_flag = 1; atomicMax(status, (uint32_t)DEV_TIMEOUT_MMA); }
            } else {
                tc_fence_after();
                const uint32_t a_lo = (uint32_t)dDy + (uint32_t)s * (16384u >> 4);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    umma_bf16_lohi(tmem_base, a_lo + 128u * kk, (uint32_t)(dDy >> 32), (uint32_t)dP + 128u * kk, (uint32_t)(dP >> 32), idesc, (it > 0 || kk > 0) ? 1u : 0u, elected);
                if (elected) umma_commit(done);
            }
            __syncwarp();
        }
    }
    window_wait();
    __syncthreads();
    if (!*abort_flag) {
        bool ok = true;
        if (lane == 0) ok = mbar_wait(done, (uint32_t)((n_iters - 1) & 1));
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) {
            if (lane == 0) { *abort_flag = 1; atomicMax(status, (uint32_t)DEV_TIMEOUT_EPI); }
        } else if (warp < 2) {                                // accumulator rows 64.. are unused
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16);
            const int cout = warp * 32 + lane;
            float* pw = part + (size_t)blockIdx.x * stride_floats + (size_t)cout * 9 * CIN;
            float* pb = part + (size_t)blockIdx.x * stride_floats + (size_t)g.Cout * 9 * CIN + cout;
#pragma unroll
            for (int c0 = 0; c0 < P::COLS; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(taddr + c0, v);                     // warp-collective
                tmem_ld_wait();
                if (cout < g.Cout) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int k = c0 + j, r = k / P::SLOTS, t = k % P::SLOTS;
                        if (r < 3 && t < P::RUN) pw[r * P::RUN + t] = __uint_as_float(v[j]);
                        else if (k == P::ONES) *pb = __uint_as_float(v[j]);
                    }
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
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 64);
    }
}

// Window rows a tile can touch: its image rows, a row of zeros where it crosses into another image, one row above and below.
static int window_rows(int H, int W)
{
    const int rows = (CI_TILE - 1 + W - 1) / W + 1;
    return rows + (rows - 1 + H - 1) / H + 2;
}
static int window_pitch(int W, int Cin) { return (CI_LEFT + Cin * (W + 1) + 2 + 7) / 8 * 8; }
static long window_bytes(int H, int W, int Cin) { return ((long)window_rows(H, W) * window_pitch(W, Cin) * 2 + 15) / 16 * 16; }
static long fwd_smem(long win) { return 1024 + 16384 + 8192 + 256 + 2 * win + 64; }
static long wgrad_smem(long win) { return 1024 + 3 * 16384 + 2 * win + 64; }

bool conv_in_umma_supported(int H, int W, int Cin, int Cout)
{
    return (Cin == 1 || Cin == 3 || Cin == 4) && Cout <= 64 && Cout % 16 == 0 && wgrad_smem(window_bytes(H, W, Cin)) <= 220 * 1024;
}

int conv_in_umma_wgrad_blocks(int B, int H, int W, int Cin)
{
    const long chunks = ((long)B * H * W + CI_TILE - 1) / CI_TILE;
    long ctas = chunks / 2;                       // at least two chunks per CTA
    const long resident = (227L * 1024) / (wgrad_smem(window_bytes(H, W, Cin)) + 1024);      // (three or four per SM hide one another's latency chains)
    if (ctas > 148 * resident) ctas = 148 * resident;
    if (ctas < 1) ctas = 1;
    const long cpc = (chunks + ctas - 1) / ctas;
    return (int)((chunks + cpc - 1) / cpc);       // no empty trailing CTA
}

static ConvInGeom geom(const void* x, const PtrTab* tab, int b_per_rep, int B, int H, int W, int Cin, int Cout)
{
    ConvInGeom g{};
    g.x = (const __nv_bfloat16*)x;
    if (tab) { g.tab = *tab; g.use_tab = 1; }
    g.b_per_rep = b_per_rep;
    g.H = H; g.W = W; g.npix = B * H * W; g.n_img = B; g.Cout = Cout;
    g.ve = W * Cin % 8 == 0 ? 8 : W * Cin % 2 == 0 ? 2 : 1;
    g.vpr = W * Cin / g.ve;
    g.rcp_w = rcp_of(W); g.rcp_h = rcp_of(H); g.rcp_hp = rcp_of(H + 1); g.rcp_rep = rcp_of(b_per_rep);
    g.pitch = window_pitch(W, Cin);
    g.win_bytes = (int)window_bytes(H, W, Cin);
    return g;
}

template <int CIN>
static cudaError_t launch_fwd_t(const ConvSimtArgs& a, const CUtensorMap& mapY, uint32_t* status, cudaStream_t st)
{
    const long npix = (long)a.B * a.H * a.W;
    if (npix + a.B + CI_TILE >= (1L << 31)) return cudaErrorInvalidValue;     // the kernel's pixel arithmetic is 32-bit
    const ConvInGeom g = geom(a.in, a.tab, a.b_per_rep, a.B, a.H, a.W, CIN, a.Cout);
    const int n_tiles = (int)((npix + CI_TILE - 1) / CI_TILE);
    const long smem = fwd_smem(g.win_bytes);
    const cudaError_t e = raise_smem_limit<conv_in_fwd_umma_kernel<CIN>>(227 * 1024);
    if (e != cudaSuccess) return e;
    // persistent CTAs, as many as are resident at once: a CTA more per SM than fits means a second wave
    long per_sm = (227L * 1024) / (smem + 1024);                 // shared memory (1 KB per CTA is reserved by the system)
    if (per_sm > 7) per_sm = 7;                                  // (64 of 512 TMEM columns each; registers for seven)
    if (per_sm < 1) per_sm = 1;
    const int grid = (int)(n_tiles < 148L * per_sm ? n_tiles : 148L * per_sm);
    return pdl_launch(conv_in_fwd_umma_kernel<CIN>, dim3(grid), dim3(CI_THREADS), (size_t)smem, st, mapY, g, (const __nv_bfloat16*)a.w, a.bias, a.relu, n_tiles, status);
}

cudaError_t launch_conv_in_fwd_umma(const ConvSimtArgs& a, const CUtensorMap& mapY, uint32_t* status, cudaStream_t st)
{
    switch (a.Cin) {
    case 1: return launch_fwd_t<1>(a, mapY, status, st);
    case 3: return launch_fwd_t<3>(a, mapY, status, st);
    case 4: return launch_fwd_t<4>(a, mapY, status, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int CIN>
static cudaError_t launch_wgrad_t(const WgradSimtArgs& a, const CUtensorMap& mapDy, uint32_t* status, cudaStream_t st)
{
    const long npix = (long)a.B * a.H * a.W;
    if (npix + a.B + CI_TILE >= (1L << 31)) return cudaErrorInvalidValue;     // the kernel's pixel arithmetic is 32-bit
    const ConvInGeom g = geom(a.x, a.tab, a.b_per_rep, a.B, a.H, a.W, CIN, a.Cout);
    const int chunks = (int)((npix + CI_TILE - 1) / CI_TILE), grid = conv_in_umma_wgrad_blocks(a.B, a.H, a.W, CIN);
    const cudaError_t e = raise_smem_limit<conv_in_wgrad_umma_kernel<CIN>>(227 * 1024);
    if (e != cudaSuccess) return e;
    return pdl_launch(conv_in_wgrad_umma_kernel<CIN>, dim3(grid), dim3(CI_THREADS), (size_t)wgrad_smem(g.win_bytes), st, mapDy, g, a.part,
                      (long)a.Cout * 9 * CIN + a.Cout, chunks, (chunks + grid - 1) / grid, status);
}

cudaError_t launch_conv_in_wgrad_umma(const WgradSimtArgs& a, const CUtensorMap& mapDy, uint32_t* status, cudaStream_t st)
{
    switch (a.Cin) {
    case 1: return launch_wgrad_t<1>(a, mapDy, status, st);
    case 3: return launch_wgrad_t<3>(a, mapDy, status, st);
    case 4: return launch_wgrad_t<4>(a, mapDy, status, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace sb
