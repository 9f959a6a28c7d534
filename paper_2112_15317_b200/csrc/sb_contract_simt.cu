// CUDA-core contractions of the float mode's small and odd layers (and of layers whose widths the tensor-core tiles do not take): 3x3 convolution and
// fully-connected forward, data gradient and weight gradient as one tiled kernel.
//
//   FWD   : y[pixel, o]  = sum_{tap, c} x[pixel + tap, c]  * W[o, tap, c]      rows = pixels, columns = output channels
//   DGRAD : dx[pixel, c] = sum_{tap, o} dy[pixel - tap, o] * W[o, tap, c]      rows = pixels, columns = input channels
//   WGRAD : dW[o, n]     = sum_{pixel}  dy[pixel, o] * x[pixel + tap, c]       rows = output channels, columns n = (tap, c)
//
// A fully-connected layer is the same thing with one tap and 1x1 images (pixel = batch row).
//
// Large enough float layers whose channel counts are multiples of eight run on the tensor cores instead (sb_contract_umma.cu): the plan
// takes whichever the two cost models below say is faster.  Forward, us between events, 3x3 over 64 channels at 32x32, batch 96: 183 here,
// 58 there; 256 channels at 8x8: 159 and 46; 16 -> 32 channels at 16x16, batch 8: 12.9 and 12.5.  4096 -> 1024 weight gradient at batch
// 8, the kernel alone: 6.8 and 14.
//
// What bounds it: the FFMA pipe (measured 70 TFLOP/s of packed fma.rn.f32x2 on registers, 68 of scalar FFMA).  A block of
// BM x BN outputs gives every thread an 8 x 8 square, so that 16 shared-memory words feed 64 multiply-adds; the packed form
// halves the issue slots of the multiply-adds, which leaves slots for the shared-memory loads and the operand broadcast beside them.
// Operand tiles of 16 reduction steps go global -> registers -> shared memory, one tile ahead of the arithmetic.
// Layers too small to fill the machine split the reduction over blockIdx.z: raw partial sums, added in split order afterwards.
#include "sb_internal.h"

#include <algorithm>

namespace sb {

namespace {

constexpr int BK = 16;

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ float4 load4(const float* p) { return __ldg((const float4*)p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p)
{
    const uint2 v = __ldg((const uint2*)p);
    const __nv_bfloat162 a = *(const __nv_bfloat162*)&v.x, b = *(const __nv_bfloat162*)&v.y;
    return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
}
__device__ __forceinline__ void store4(float* p, float4 v) { *(float4*)p = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v)
{
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 pk;
    pk.x = *(uint32_t*)&lo;
    pk.y = *(uint32_t*)&hi;
    *(uint2*)p = pk;
}
// up to four consecutive elements, the first `n` of them valid (the rest zero)
template <typename T, bool VEC>
__device__ __forceinline__ float4 load_run(const T* p, int n)
{
    if (VEC) return n > 0 ? load4(p) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v;
    v.x = n > 0 ? to_f<T>(p[0]) : 0.f;
    v.y = n > 1 ? to_f<T>(p[1]) : 0.f;
    v.z = n > 2 ? to_f<T>(p[2]) : 0.f;
    v.w = n > 3 ? to_f<T>(p[3]) : 0.f;
    return v;
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }

// n / d for n < 2^31 through the reciprocal floor(2^32 / d) + 1 (0 stands for d = 1): the estimate is exact or one too high
__device__ __forceinline__ int div_rcp(int n, uint32_t mul, int d)
{
    if (mul == 0u) return n;
    uint32_t q = __umulhi((uint32_t)n, mul);
    if (q * (uint32_t)d > (uint32_t)n) --q;
    return (int)q;
}

struct Pixel { int n, h, w; };

}  // namespace

struct ContractParams {
    const void *act, *wt, *dy;     // FWD: act, wt; DGRAD: dy, wt; WGRAD: dy, act
    PtrTab tab; int tab_imgs;      // tab_imgs > 0: the layer input lives in per-replica buffers of tab_imgs images each
    int taps, H, W, Cin, Cout, npix;
    uint32_t rcp_w, rcp_hw, rcp_tab;
    int M, N;                      // rows and columns of the result
    int cpt;                       // FWD / DGRAD: BK-wide channel chunks per tap
    int iters, iters_per_split, splits;
    float* part; long split_stride;    // splits > 1, and WGRAD always: raw sums [split][M][N]
    long bias_off;                 // WGRAD: offset of the bias gradient (column sums of dy) inside a split's buffer
    void* out; float* out32; const float* bias; int relu;     // FWD (out32: float result instead of out)
    const void* ref;               // DGRAD: zero where ref <= 0 (nullptr: no mask)
};

// T: activation and weight type (float, or bf16 converted on load); VEC: both channel counts are multiples of four, so four
// neighbouring elements never straddle a tap and are aligned.
// (128 registers a thread, 168 for the two-warp shapes: two blocks of 256 threads, four of 128 or six of 64 on an SM)
template <typename T, int MODE, int BM, int BN, bool VEC>
__global__ void __launch_bounds__(BM * BN / 64, BM * BN <= 4096 ? 6 : 512 * 64 / (BM * BN))
contract_kernel(const __grid_constant__ ContractParams p)
{
    pdl_prologue();
    constexpr int THREADS = BM * BN / 64;
    constexpr int LDA = BM + 4, LDB = BN + 4;
    constexpr int NA = BM * BK / 4 / THREADS, NB = BN * BK / 4 / THREADS;     // 16-byte runs per thread and tile
    __shared__ __align__(16) float sA[2][BK][LDA];
    __shared__ __align__(16) float sB[2][BK][LDB];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int it0 = blockIdx.z * p.iters_per_split, it1 = min(it0 + p.iters_per_split, p.iters);
    const int HW = p.H * p.W;
    const bool use_tab = p.tab_imgs > 0;

    auto split_pixel = [&](int pix) {
        Pixel q;
        q.n = div_rcp(pix, p.rcp_hw, HW);
        const int r = pix - q.n * HW;
        q.h = div_rcp(r, p.rcp_w, p.W);
        q.w = r - q.h * p.W;
        return q;
    };
    // the layer input's image n
    auto image = [&](int n) -> const T* {
        if (!use_tab) return (const T*)p.act + (size_t)n * HW * p.Cin;
        const int r = div_rcp(n, p.rcp_tab, p.tab_imgs);
        return (const T*)p.tab.p[r] + (size_t)(n - r * p.tab_imgs) * HW * p.Cin;
    };

    // ---- what this thread loads: fixed per thread, or advanced with the iteration -----------------------------------------
    // FWD / DGRAD: run i of the A tile = 4 channels (quad tid % 4) of pixel row tid / 4 + i * THREADS / 4
    // (pointer to that pixel of the image in shape [H][W][Cred], and which of the nine taps fall inside the image)
    const T* a_px[MODE == CMODE_WGRAD ? 1 : NA];
    uint32_t a_in[MODE == CMODE_WGRAD ? 1 : NA];
    // WGRAD: runs of the B tile = 4 columns (tap, c) of pixel k; the columns are the same in every iteration
    int b_tap_h = 0, b_tap_w = 0, b_c = 0, b_valid = 0;
    const int Cred = MODE == CMODE_DGRAD ? p.Cout : p.Cin;
    if (MODE != CMODE_WGRAD) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int pix = m0 + tid / 4 + i * (THREADS / 4);
            a_in[i] = 0u;
            a_px[i] = nullptr;
            if (pix < p.M) {
                const Pixel q = split_pixel(pix);
                const T* img = MODE == CMODE_FWD ? image(q.n) : (const T*)p.dy + (size_t)q.n * HW * Cred;
                a_px[i] = img + ((size_t)q.h * p.W + q.w) * Cred;
                if (p.taps == 1) a_in[i] = 1u;
                else
#pragma unroll
                    for (int t = 0; t < 9; ++t) {
                        const int dr = MODE == CMODE_FWD ? t / 3 - 1 : 1 - t / 3, ds = MODE == CMODE_FWD ? t % 3 - 1 : 1 - t % 3;
                        if ((unsigned)(q.h + dr) < (unsigned)p.H && (unsigned)(q.w + ds) < (unsigned)p.W) a_in[i] |= 1u << t;
                    }
            }
        }
    } else if (VEC) {
        const int n = n0 + (tid % (BN / 4)) * 4;
        b_valid = n < p.N ? 4 : 0;
        const int t = b_valid ? n / p.Cin : 0;
        b_c = n - t * p.Cin;
        if (p.taps == 9) { b_tap_h = t / 3 - 1; b_tap_w = t % 3 - 1; }
    }

    float4 ra[NA], rb[NB];
    auto load_tiles = [&](int it) {
        if (MODE != CMODE_WGRAD) {
            const int tap = p.taps == 1 ? 0 : it / p.cpt, c0 = (it - tap * p.cpt) * BK;
            int shift = 0;
            if (p.taps == 9) {
                const int dr = MODE == CMODE_FWD ? tap / 3 - 1 : 1 - tap / 3, ds = MODE == CMODE_FWD ? tap % 3 - 1 : 1 - tap % 3;
                shift = dr * p.W + ds;
            }
            const int c = c0 + (tid % 4) * 4, left = Cred - c;
#pragma unroll
            for (int i = 0; i < NA; ++i) ra[i] = load_run<T, VEC>(a_px[i] + (long)shift * Cred + c, ((a_in[i] >> tap) & 1u) ? left : 0);
            if (MODE == CMODE_FWD) {
                // B tile: row n of the weight matrix [Cout][taps * Cin], 4 reduction steps per run
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const int n = n0 + tid / 4 + i * (THREADS / 4);
                    rb[i] = load_run<T, VEC>((const T*)p.wt + ((size_t)n * p.taps + tap) * p.Cin + c, n < p.N ? left : 0);
                }
            } else {
                // B tile: 4 input channels of weight row o = reduction step
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const int e = tid + i * THREADS, k = e / (BN / 4), n = n0 + (e % (BN / 4)) * 4, o = c0 + k;
                    rb[i] = load_run<T, VEC>((const T*)p.wt + ((size_t)o * p.taps + tap) * p.Cin + n, o < Cred ? p.N - n : 0);
                }
            }
        } else {
            const int k0 = it * BK;
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                const int e = tid + i * THREADS, k = k0 + e / (BM / 4), m = m0 + (e % (BM / 4)) * 4;
                ra[i] = load_run<T, VEC>((const T*)p.dy + (size_t)k * p.Cout + m, k < p.npix ? p.M - m : 0);
            }
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int e = tid + i * THREADS, k = k0 + e / (BN / 4);
                rb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (k < p.npix) {
                    const Pixel q = split_pixel(k);
                    const T* img = image(q.n);
                    if (VEC) {
                        const int h = q.h + b_tap_h, w = q.w + b_tap_w;
                        const bool in = (unsigned)h < (unsigned)p.H && (unsigned)w < (unsigned)p.W;
                        rb[i] = load_run<T, VEC>(img + ((long)h * p.W + w) * p.Cin + b_c, in ? b_valid : 0);
                    } else {
                        float v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int n = n0 + (e % (BN / 4)) * 4 + j, t = n / p.Cin, c = n - t * p.Cin;
                            const int h = q.h + (p.taps == 9 ? t / 3 - 1 : 0), w = q.w + (p.taps == 9 ? t % 3 - 1 : 0);
                            const bool in = n < p.N && (unsigned)h < (unsigned)p.H && (unsigned)w < (unsigned)p.W;
                            v[j] = in ? to_f<T>(img[((size_t)h * p.W + w) * p.Cin + c]) : 0.f;
                        }
                        rb[i] = make_float4(v[0], v[1], v[2], v[3]);
                    }
                }
            }
        }
    };
    auto keep_tiles = [&](int buf) {
        if (MODE != CMODE_WGRAD) {
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                const int r = tid / 4 + i * (THREADS / 4), k = (tid % 4) * 4;
                sA[buf][k][r] = ra[i].x; sA[buf][k + 1][r] = ra[i].y; sA[buf][k + 2][r] = ra[i].z; sA[buf][k + 3][r] = ra[i].w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < NA; ++i) { const int e = tid + i * THREADS; *(float4*)&sA[buf][e / (BM / 4)][(e % (BM / 4)) * 4] = ra[i]; }
        }
        if (MODE == CMODE_FWD) {
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int r = tid / 4 + i * (THREADS / 4), k = (tid % 4) * 4;
                sB[buf][k][r] = rb[i].x; sB[buf][k + 1][r] = rb[i].y; sB[buf][k + 2][r] = rb[i].z; sB[buf][k + 3][r] = rb[i].w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < NB; ++i) { const int e = tid + i * THREADS; *(float4*)&sB[buf][e / (BN / 4)][(e % (BN / 4)) * 4] = rb[i]; }
        }
    };

    // ---- 8 x 8 outputs per thread: rows ty*4.. and BM/2 + ty*4.., columns tx*4.. and BN/2 + tx*4.. (a warp covers 4 x 8 threads,
    // or 8 x 4 where the tile is 32 columns wide, so its operand reads are broadcasts of whole 128-byte lines)
    constexpr int TX = BN / 8, WX = TX < 8 ? TX : 8, WY = 32 / WX;
    const int warp = tid / 32, lane = tid % 32;
    const int tx = (warp % (TX / WX)) * WX + lane % WX, ty = (warp / (TX / WX)) * WY + lane / WX;
    unsigned long long acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    // WGRAD: the blocks of the first column tile also add up their rows of dy (the bias gradient)
    constexpr int BS = (BM + THREADS - 1) / THREADS;
    const bool do_bias = MODE == CMODE_WGRAD && blockIdx.y == 0;
    float bsum[BS];
#pragma unroll
    for (int i = 0; i < BS; ++i) bsum[i] = 0.f;

    if (it0 < it1) {
        load_tiles(it0);
        keep_tiles(0);
    }
    __syncthreads();
    for (int it = it0; it < it1; ++it) {
        const int buf = (it - it0) & 1;
        if (it + 1 < it1) load_tiles(it + 1);
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            const float4 a0 = *(const float4*)&sA[buf][k][ty * 4], a1 = *(const float4*)&sA[buf][k][BM / 2 + ty * 4];
            const ulonglong2 b0 = *(const ulonglong2*)&sB[buf][k][tx * 4], b1 = *(const ulonglong2*)&sB[buf][k][BN / 2 + tx * 4];
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned long long aa = pack2(av[i], av[i]);
                fma2(acc[i][0], aa, b0.x);
                fma2(acc[i][1], aa, b0.y);
                fma2(acc[i][2], aa, b1.x);
                fma2(acc[i][3], aa, b1.y);
            }
        }
        if (do_bias) {
#pragma unroll
            for (int i = 0; i < BS; ++i) {
                const int m = tid + i * THREADS;
                if (m < BM)
#pragma unroll
                    for (int k = 0; k < BK; ++k) bsum[i] += sA[buf][k][m];
            }
        }
        if (it + 1 < it1) keep_tiles(buf ^ 1);
        __syncthreads();
    }

    // ---- results ---------------------------------------------------------------------------------------------------------
    if (do_bias) {
#pragma unroll
        for (int i = 0; i < BS; ++i) {
            const int m = tid + i * THREADS;
            if (m < BM && m0 + m < p.M) p.part[(size_t)blockIdx.z * p.split_stride + p.bias_off + m0 + m] = bsum[i];
        }
    }
    const bool raw = MODE == CMODE_WGRAD || p.splits > 1;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int m = m0 + (i < 4 ? ty * 4 + i : BM / 2 + ty * 4 + i - 4);
        if (m >= p.M) continue;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = n0 + q * (BN / 2) + tx * 4;
            if (n >= p.N) continue;
            float v[4];
            unpack2(acc[i][2 * q], v[0], v[1]);
            unpack2(acc[i][2 * q + 1], v[2], v[3]);
            const size_t at = (size_t)m * p.N + n;
            const int cnt = VEC ? 4 : min(4, p.N - n);
            if (raw) {
                float* dst = p.part + (size_t)blockIdx.z * p.split_stride + at;
                if (VEC) store4(dst, make_float4(v[0], v[1], v[2], v[3]));
                else
                    for (int j = 0; j < cnt; ++j) dst[j] = v[j];
                continue;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!VEC && j >= cnt) continue;
                if (MODE == CMODE_FWD) {
                    v[j] += p.bias[n + j];
                    if (p.relu && !(v[j] > 0.f)) v[j] = 0.f;
                } else if (p.ref != nullptr) {
                    if (!(to_f<T>(((const T*)p.ref)[at + j]) > 0.f)) v[j] = 0.f;
                }
            }
            if (VEC) {
                if (p.out32 != nullptr) store4(p.out32 + at, make_float4(v[0], v[1], v[2], v[3]));
                else store4((T*)p.out + at, make_float4(v[0], v[1], v[2], v[3]));
            } else {
                for (int j = 0; j < cnt; ++j) {
                    if (p.out32 != nullptr) p.out32[at + j] = v[j];
                    else ((T*)p.out)[at + j] = from_f<T>(v[j]);
                }
            }
        }
    }
}

// ---- tile and split choice -----------------------------------------------------------------------------------------------
// Cost model in microseconds, fitted to a sweep of every shape and 1 to 128 splits over the layers of a 7-conv / 3-FC net.  One
// reduction step of BK costs the n blocks that share an SM lone + more * n, up to `resident` of them together, the rest in further
// rounds (128 x 128: 1.7 us alone, 2.95 for two = 53 TFLOP/s).  A split reduction adds a kernel and its float partial sums.
struct TileShape { int bm, bn, resident; double lone, more; };
static const TileShape shapes[] = {{128, 128, 2, 0.45, 1.25}, {128, 64, 4, 0.75, 0.65}, {64, 128, 4, 0.75, 0.63},
                                   {64, 64, 6, 0.62, 0.30},   {128, 32, 6, 0.85, 0.30}, {32, 128, 6, 0.85, 0.30}};

// The tensor-core form (one CTA per SM): microseconds per 64 reduction steps, per tile and per launch, and, where the sums of splits are
// added up by a kernel of their own, per call and per million of them, by what converts B (the kernel itself, or the split weights of a
// convolution), tile width and mode.  From a sweep of both widths and 1 to 64 splits over 25 layers (residual 5 to 10 %); the plan it
// chooses takes on average 0.6 % longer than the fastest of the sweep.
struct UmmaCost { double step, tile, launch, sums, sum; };
static const UmmaCost umma_cost[2][2][3] = {
    {{{1.26, 0.7, 5.9, 1.0, 2.45}, {1.21, 0.7, 7.5, -1.1, 2.43}, {1.47, 5.9, 0.2, 3.0, 1.14}},
     {{0.97, 1.0, 4.8, 1.0, 1.55}, {1.06, 0.5, 5.6, -0.1, 2.20}, {1.06, 2.0, 2.4, 3.0, 1.14}}},
    {{{1.18, 0.4, 9.0, -2.2, 1.66}, {1.26, 0.7, 8.5, -2.1, 1.49}, {1.47, 5.9, 0.2, 3.0, 1.14}},
     {{0.81, 0.1, 8.0, -0.9, 1.09}, {0.82, 0.5, 8.0, -1.3, 0.75}, {1.06, 2.0, 2.4, 3.0, 1.14}}}};

static bool vec_ok(int Cin, int Cout) { return Cin % 4 == 0 && Cout % 4 == 0; }
static long contract_iters(int mode, int B, int H, int W, int taps, int Cin, int Cout)
{
    const int cred = mode == CMODE_DGRAD ? Cout : Cin;
    return mode == CMODE_WGRAD ? ((long)B * H * W + BK - 1) / BK : (long)taps * ((cred + BK - 1) / BK);
}

ContractPlan contract_plan(int mode, int B, int H, int W, int taps, int Cin, int Cout, size_t max_part_floats, bool umma)
{
    const long pix = (long)B * H * W, M = mode == CMODE_WGRAD ? Cout : pix;
    const long N = mode == CMODE_FWD ? Cout : mode == CMODE_DGRAD ? Cin : (long)taps * Cin;
    const long iters = contract_iters(mode, B, H, W, taps, Cin, Cout);
    ContractPlan best{};
    double best_t = 1e300;
    for (const TileShape& s : shapes) {
        if (!vec_ok(Cin, Cout) && (s.bm != 64 || s.bn != 64)) continue;      // (odd channel counts: one shape)
        const long tiles = ((M + s.bm - 1) / s.bm) * ((N + s.bn - 1) / s.bn);
        for (int split = 1; split <= 256 && (split == 1 || iters / split >= 3); split = split < 8 ? split + 1 : split + split / 4) {
            const long per = (iters + split - 1) / split;
            const int real = (int)((iters + per - 1) / per);
            if (real > 1 && (size_t)real * M * (N + (mode == CMODE_WGRAD ? 1 : 0)) > max_part_floats) break;
            const long n = (tiles * real + 147) / 148, rest = n % s.resident;        // blocks of the fullest SM
            const double step = (double)(n / s.resident) * (s.lone + s.more * s.resident) + (rest ? s.lone + s.more * rest : 0.0);
            double t = per * step * (mode == CMODE_WGRAD ? 1.08 : 1.0) + 3.0;
            if (mode == CMODE_DGRAD && real == 1) t += 3.5;      // (a thread's sixteen mask loads, one behind the other)
            if (real > 1) t += 3.0 + (double)real * M * N * 8.0 / 7.0e6;
            if (t < best_t) { best_t = t; best = ContractPlan{s.bm, s.bn, (int)per, real, false}; }
        }
    }
    if (umma && contract_umma_ok(taps, Cin, Cout)) {
        const long K = mode == CMODE_WGRAD ? pix : (long)taps * (mode == CMODE_DGRAD ? Cout : Cin), chunks = (K + 63) / 64;
        const bool terms = taps == 9 && contract_umma_whole_taps(mode, Cin, Cout);
        for (int bn : {128, 64}) {
            const UmmaCost& u = umma_cost[terms][bn == 64][mode];
            const long tiles = ((M + 127) / 128) * ((N + bn - 1) / bn);
            for (int split = 1; split <= 256 && split <= chunks; split = split < 16 ? split + 1 : split + split / 8) {
                const long per = (chunks + split - 1) / split;
                const int real = (int)((chunks + per - 1) / per);
                if (real > 1 && (size_t)real * M * (N + (mode == CMODE_WGRAD ? 1 : 0)) > max_part_floats) break;
                double t = (double)((tiles * real + 147) / 148) * (per * u.step + u.tile) + u.launch;
                if (real > 1) t += u.sums + (double)real * M * N * 1e-6 * u.sum;
                if (t < best_t) { best_t = t; best = ContractPlan{128, bn, (int)per, real, true}; }
            }
        }
    }
    return best;
}

static uint32_t rcp_of(int d) { return d <= 1 ? 0u : (uint32_t)(0x100000000ull / (uint32_t)d) + 1u; }

// A grid of n blocks per SM is kept to n of them on any SM by the shared memory each asks for: left alone, the hardware puts two
// of 100 to 148 blocks on some SMs while others stay empty (144 blocks of 128 x 128: 301 us, 72 blocks of twice the length: 349).
template <typename T, int MODE, int BM, int BN, bool VEC>
static cudaError_t launch_one(const ContractParams& p, cudaStream_t st)
{
    constexpr int STATIC = (int)(2 * BK * (BM + 4 + BN + 4) * sizeof(float)), MOST = 224 * 1024;
    const cudaError_t e = raise_smem_limit<contract_kernel<T, MODE, BM, BN, VEC>>(MOST - STATIC);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((p.M + BM - 1) / BM), (unsigned)((p.N + BN - 1) / BN), (unsigned)p.splits);
    const long n = ((long)grid.x * grid.y * grid.z + 147) / 148;
    const int share = n <= 4 ? (int)(MOST / n) - 2048 - STATIC : 0;
    return pdl_launch(contract_kernel<T, MODE, BM, BN, VEC>, grid, dim3(BM * BN / 64), share > 0 ? (size_t)share / 1024 * 1024 : 0, st, p);
}
template <typename T, int MODE, bool VEC>
static cudaError_t launch_shape(const ContractPlan& c, const ContractParams& p, cudaStream_t st)
{
#define SB_SHAPE(BM, BN) if (c.bm == BM && c.bn == BN) return launch_one<T, MODE, BM, BN, VEC>(p, st)
    SB_SHAPE(64, 64);
    if constexpr (VEC) {
        SB_SHAPE(128, 128);
        SB_SHAPE(128, 64);
        SB_SHAPE(64, 128);
        SB_SHAPE(128, 32);
        SB_SHAPE(32, 128);
    }
#undef SB_SHAPE
    return cudaErrorInvalidValue;
}
template <typename T, int MODE>
static cudaError_t launch_vec(const ContractPlan& c, const ContractParams& p, cudaStream_t st)
{
    return vec_ok(p.Cin, p.Cout) ? launch_shape<T, MODE, true>(c, p, st) : launch_shape<T, MODE, false>(c, p, st);
}

cudaError_t launch_contract(const ContractArgs& a, bool bf16, cudaStream_t st)
{
    ContractParams p{};
    p.act = a.act; p.wt = a.wt; p.dy = a.dy;
    if (a.tab) { p.tab = *a.tab; p.tab_imgs = a.tab_imgs; p.rcp_tab = rcp_of(a.tab_imgs); }
    p.taps = a.taps; p.H = a.H; p.W = a.W; p.Cin = a.Cin; p.Cout = a.Cout;
    const long npix = (long)a.B * a.H * a.W;
    if (npix >= (1L << 31)) return cudaErrorInvalidValue;
    p.npix = (int)npix;
    p.rcp_w = rcp_of(a.W); p.rcp_hw = rcp_of(a.H * a.W);
    p.M = a.mode == CMODE_WGRAD ? a.Cout : p.npix;
    p.N = a.mode == CMODE_FWD ? a.Cout : a.mode == CMODE_DGRAD ? a.Cin : a.taps * a.Cin;
    p.cpt = ((a.mode == CMODE_DGRAD ? a.Cout : a.Cin) + BK - 1) / BK;
    p.iters = (int)contract_iters(a.mode, a.B, a.H, a.W, a.taps, a.Cin, a.Cout);
    p.iters_per_split = a.plan.iters; p.splits = a.plan.splits;
    p.part = a.part; p.split_stride = a.split_stride; p.bias_off = a.bias_off;
    p.out = a.out; p.out32 = a.out32; p.bias = a.bias; p.relu = a.relu; p.ref = a.ref;
    cudaError_t e;
    if (a.plan.umma) e = launch_contract_umma(a, st);
    else if (a.mode == CMODE_FWD) e = bf16 ? launch_vec<__nv_bfloat16, CMODE_FWD>(a.plan, p, st) : launch_vec<float, CMODE_FWD>(a.plan, p, st);
    else if (a.mode == CMODE_DGRAD) e = bf16 ? launch_vec<__nv_bfloat16, CMODE_DGRAD>(a.plan, p, st) : launch_vec<float, CMODE_DGRAD>(a.plan, p, st);
    else e = bf16 ? launch_vec<__nv_bfloat16, CMODE_WGRAD>(a.plan, p, st) : launch_vec<float, CMODE_WGRAD>(a.plan, p, st);
    if (e != cudaSuccess || a.mode == CMODE_WGRAD || p.splits == 1) return e;
    SplitKEpiArgs s{};
    s.part = a.part; s.split_stride = (size_t)a.split_stride; s.splits = p.splits; s.rows = p.M; s.N = p.N;
    s.epi = a.mode == CMODE_FWD ? EPI_BIAS_ACT : EPI_MASK; s.bias = a.bias; s.relu = a.relu; s.ref = a.ref;
    s.out = a.out32 ? (void*)a.out32 : a.out; s.out_f32 = a.out32 != nullptr;
    return launch_splitk_epilogue(s, bf16, st);
}

}  // namespace sb
