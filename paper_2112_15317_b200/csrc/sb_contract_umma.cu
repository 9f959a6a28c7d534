// Float contractions on the tensor cores: every float operand element is taken apart into three bf16 terms that add up to it
// (8 + 8 + 8 significant bits), and the products of the terms are accumulated in float.
//
//   a = a0 + a1 + a2,  |a1| <= 2^-9 |a|,  |a2| <= 2^-18 |a|           (b likewise)
//   a * b = a0 b0  +  (a0 b1 + a1 b0)  +  (a0 b2 + a1 b1 + a2 b0)  +  terms below 2^-26 |a b| that are left out
//
// The same contractions as sb_contract_simt.cu (FWD, DGRAD, WGRAD of 3x3 convolutions and FC layers, same operands, partial sums
// and results), as implicit GEMMs with the reduction index flattened over (tap, channel) and, for WGRAD, the columns over
// (tap, input channel); channel counts are multiples of eight, so that eight neighbours never straddle a tap.
//
// Precision.  The tensor core adds into its float accumulator with truncation, so a long chain in it would lose more than the
// rounded multiply-adds of the CUDA cores.  The leading products a0 b0 are therefore accumulated over 64 reduction steps only (four
// instructions) and then added to a rounded running sum in registers; the remaining products, 2^-9 times smaller, stay in an
// accumulator of their own until the end.  Error against 64-bit sums (2-norm; half-normal x, normal w and dy), CUDA cores -> here:
//   3x3, 64 channels at 32x32, batch 96    forward 3.0e-7 -> 0.8e-7   input gradient 4.2e-7 -> 0.9e-7   weight gradient 4.6e-7 -> 1.9e-7
//   3x3, 256 channels at 8x8, batch 96             3.4e-7 -> 0.9e-7                  4.8e-7 -> 1.0e-7                   3.3e-7 -> 1.1e-7
//   4096 -> 1024, batch 96                         1.8e-7 -> 1.0e-7                  2.1e-7 -> 0.9e-7                   1.3e-7 -> 0.5e-7
//   3x3, 8 -> 40 channels at 5x7, batch 3          0.8e-7 -> 0.6e-7                  1.2e-7 -> 0.8e-7                   1.2e-7 -> 0.5e-7
//
// Roles (24 warps; registers are moved between them): warp 0 allocates TMEM and issues the MMAs; warps 4-7 keep the running sums and
// write the results; warps 8-23 fetch floats to registers, take them apart and store the terms, A into tensor memory (a lane per
// row) and B as 128-byte swizzled rows of shared memory, the next chunk's loads in flight behind the conversion of the present one.
// A in tensor memory keeps its terms off the shared-memory port, which would else carry 40 KB per 16 steps of a 128 x 128 tile.
//
// What bounds it: the converters' loads.  A 128 x 128 x 64 chunk takes 2850 cycles where its 24 MMAs take 1536 (tensor pipe 49 %
// busy): a row per lane makes each 32-byte load of A 32 wavefronts of the L1 port (1280 cycles a chunk with those of B, 1150 for
// the stores and the MMAs' reads), and the 16 converter warps fill half of the issue slots.  64 -> 64 channels at 32x32, batch 96:
// 181 -> 102 us forward; 256 -> 256 at 8x8: 157 -> 57 us (7-conv / 3-FC net, batch 96: 2.54 -> 1.12 ms an iteration).
//
// Non-finite operands: infinity - infinity in the splitting makes the terms NaN where a float multiply-add would give an infinity, so
// a row with a NaN in it is computed again with plain multiply-adds by the thread that owns it.
#include "sb_internal.h"
#include "sb_tcgen05.cuh"

namespace sb {

namespace {

struct SplitParams {
    const float *act, *wt, *dy;
    int taps, H, W, Cin, Cout, npix;
    uint32_t rcp_w, rcp_hw;
    int M, N, K;                   // rows, columns, reduction length (WGRAD: pixels)
    int chunks, cps, splits;       // 64-step chunks, per split
    float* part; long split_stride;
    long bias_off;
    float* out; const float* bias; int relu;
    const float* ref;
    uint32_t* status;
};

// 24 warps: 4 for the MMAs (one works), 4 running sums, 16 converters.  Registers of the 80 a thread at launch: 32 + 160 + 4 * 72 = 6 * 80.
constexpr int THREADS = 768, CONV0 = 256, REGS_ISSUE = 32, REGS_SUMS = 160, REGS_CONV = 72;
constexpr int STAGES = 2, CTRL = 8192;
// one term of the B tile: BN rows of 128 bytes (FWD), or 64-column boxes of 64 rows
template <int BN> struct SplitCfg { static constexpr int PLANE = BN * 128, STAGE = 3 * PLANE, SMEM = STAGES * STAGE + 1024 + CTRL; };
// tensor memory columns: leading products, the other products, then the terms of A (2 stages x 3 x 32)
constexpr uint32_t COL_A = 256, A_TERM = 32, A_STAGE = 3 * A_TERM, TMEM_COLS = 512;

__device__ __forceinline__ int div_rcp(int n, uint32_t mul, int d)
{
    if (mul == 0u) return n;
    uint32_t q = __umulhi((uint32_t)n, mul);
    if (q * (uint32_t)d > (uint32_t)n) --q;
    return (int)q;
}
struct F8 { float v[8]; };
// eight floats at a 32-byte boundary (zeros where the place is outside the operand)
__device__ __forceinline__ void load8(F8& f, const float* p, bool in)
{
    if (in)
        asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(f.v[0]), "=f"(f.v[1]), "=f"(f.v[2]), "=f"(f.v[3]), "=f"(f.v[4]), "=f"(f.v[5]), "=f"(f.v[6]), "=f"(f.v[7]) : "l"(p));
    else
#pragma unroll
        for (int j = 0; j < 8; ++j) f.v[j] = 0.f;
}
// the terms of two floats, packed (the first in the low half), and what is left for the next term (exact)
__device__ __forceinline__ uint32_t take_term(float& a, float& b)
{
    const __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
    const uint32_t u = *(const uint32_t*)&t;
    unsigned long long d, e;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    asm("mov.b64 %0, {%1, %2};" : "=l"(e) : "r"(u << 16), "r"(u & 0xffff0000u));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(e), "l"(0xbf800000bf800000ull));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d));
    return u;
}
// the three terms of eight floats
__device__ __forceinline__ void take_terms(const F8& f, uint32_t* t0, uint32_t* t1, uint32_t* t2)
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float a = f.v[2 * j], b = f.v[2 * j + 1];
        t0[j] = take_term(a, b);
        t1[j] = take_term(a, b);
        const __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
        t2[j] = *(const uint32_t*)&t;
    }
}
__device__ __forceinline__ void st_shared16(uint32_t at, const uint32_t (&t)[4])
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(t[0]), "r"(t[1]), "r"(t[2]), "r"(t[3]) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
// MMA with the A operand in tensor memory, issued from a converged warp (see umma_bf16_lohi)
__device__ __forceinline__ void umma_ta(uint32_t d_tmem, uint32_t a_tmem, uint32_t blo, uint32_t bhi, uint32_t idesc, uint32_t accumulate, uint32_t elected)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "setp.ne.b32 q, %6, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate), "r"(elected)
        : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}

// Element (m, n) over reduction steps [k0, k1) with plain multiply-adds (rows with a non-finite operand).
template <int MODE>
__device__ __noinline__ float plain_sum(const SplitParams& p, int m, int n, int k0, int k1)
{
    const int HW = p.H * p.W;
    float s = 0.f;
    if (MODE == CMODE_WGRAD) {
        const int t = n / p.Cin, c = n - t * p.Cin, dr = p.taps == 9 ? t / 3 - 1 : 0, ds = p.taps == 9 ? t % 3 - 1 : 0;
        for (int k = k0; k < k1; ++k) {
            const int r = k % HW, h = r / p.W + dr, w = r % p.W + ds;
            if ((unsigned)h >= (unsigned)p.H || (unsigned)w >= (unsigned)p.W) continue;
            s = fmaf(p.dy[(size_t)k * p.Cout + m], p.act[((long)k + (long)dr * p.W + ds) * p.Cin + n - t * p.Cin], s);
        }
        (void)c;
        return s;
    }
    const int Cred = MODE == CMODE_DGRAD ? p.Cout : p.Cin, r = m % HW, h0 = r / p.W, w0 = r % p.W;
    for (int k = k0; k < k1; ++k) {
        const int t = k / Cred, c = k - t * Cred;
        int dr = p.taps == 9 ? t / 3 - 1 : 0, ds = p.taps == 9 ? t % 3 - 1 : 0;
        if (MODE == CMODE_DGRAD) { dr = -dr; ds = -ds; }
        if ((unsigned)(h0 + dr) >= (unsigned)p.H || (unsigned)(w0 + ds) >= (unsigned)p.W) continue;
        const float a = (MODE == CMODE_FWD ? p.act : p.dy)[((long)m + (long)dr * p.W + ds) * Cred + c];
        s = fmaf(a, MODE == CMODE_FWD ? p.wt[(size_t)n * p.K + k] : p.wt[((size_t)c * p.taps + t) * p.Cin + n], s);
    }
    return s;
}
// Eight results of a row: bias and ReLU, or the ReLU mask (NaN -> 0, as everywhere)
template <int MODE>
__device__ __forceinline__ void finish8(const SplitParams& p, float (&f)[8], size_t at, int n)
{
    if (MODE == CMODE_DGRAD && p.ref == nullptr) return;
    const float4* g = (const float4*)(MODE == CMODE_FWD ? p.bias + n : p.ref + at);
    const float4 g0 = __ldg(g), g1 = __ldg(g + 1);
    const float e[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (MODE == CMODE_FWD) {
            f[j] += e[j];
            if (p.relu && !(f[j] > 0.f)) f[j] = 0.f;
        } else if (!(e[j] > 0.f)) f[j] = 0.f;
    }
}

// K64: the channels of the reduction are a multiple of 64, so that a chunk lies in one tap (FWD, DGRAD)
template <int MODE, int BN, bool K64>
__global__ void __launch_bounds__(THREADS, 1)
contract_umma_kernel(const __grid_constant__ SplitParams p)
{
    using C = SplitCfg<BN>;
    constexpr int NB = BN / 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* ctrl = smem + STAGES * C::STAGE;
    uint64_t* full = (uint64_t*)ctrl;               // [STAGES] terms stored: one arrival per converter warp
    uint64_t* empty = full + STAGES;                // [STAGES] read by their MMAs
    uint64_t* lead_full = empty + STAGES;           // leading products of a chunk complete
    uint64_t* lead_empty = lead_full + 1;           // ... and taken over: one arrival per summing warp
    uint64_t* done = lead_empty + 1;                // everything complete
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    float* s_bias = (float*)(ctrl + 1024);          // [3][128]: WGRAD, sums of dy over the later quarters of the chunks

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int m0 = blockIdx.x * 128, n0 = blockIdx.y * BN;
    const int chunk0 = blockIdx.z * p.cps, n_iters = min(p.cps, p.chunks - chunk0);

    if (warp == 0) {
        if (lane == 0) {
            for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 16); mbar_init(&empty[s], 1); }
            mbar_init(lead_full, 1);
            mbar_init(lead_empty, 4);
            mbar_init(done, 1);
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();

    if (warp < 4) {
        // =========================== MMA issuer (warp 0 in lock-step, one elected lane issues) ===================================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ISSUE));
        if (warp == 0) {
            constexpr bool B_MN = MODE != CMODE_FWD;
            constexpr uint32_t idesc = make_idesc(BN, 0, B_MN);
            constexpr uint32_t A_STEP = 8, B_STEP = (B_MN ? 2048u : 32u) >> 4, BP = C::PLANE >> 4;     // per 16 reduction steps: columns, 16-byte units
            const uint32_t elected = elect_one() ? 1u : 0u;
            const uint64_t dB = make_desc(smem_u32(smem), B_MN ? 8192u : 16u);
            const uint32_t b_hi = (uint32_t)(dB >> 32), rest = tmem + BN;
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int it = 0; it < n_iters; ++it) {
                bool w = mbar_wait(&full[s], ph);
                if (it >= 1) w = w && mbar_wait(lead_empty, (uint32_t)((it & 1) ^ 1));
                ok = __all_sync(0xffffffffu, w ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const uint32_t a = tmem + COL_A + (uint32_t)s * A_STAGE, b = (uint32_t)dB + (uint32_t)s * (C::STAGE >> 4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) umma_ta(tmem, a + kk * A_STEP, b + kk * B_STEP, b_hi, idesc, kk > 0 ? 1u : 0u, elected);
                if (elected) umma_commit(lead_full);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t ak = a + kk * A_STEP, bk = b + kk * B_STEP;
                    umma_ta(rest, ak + 2 * A_TERM, bk, b_hi, idesc, (it > 0 || kk > 0) ? 1u : 0u, elected);     // a2 b0
                    umma_ta(rest, ak, bk + 2 * BP, b_hi, idesc, 1u, elected);                                   // a0 b2
                    umma_ta(rest, ak + A_TERM, bk + BP, b_hi, idesc, 1u, elected);                              // a1 b1
                    umma_ta(rest, ak + A_TERM, bk, b_hi, idesc, 1u, elected);                                   // a1 b0
                    umma_ta(rest, ak, bk + BP, b_hi, idesc, 1u, elected);                                       // a0 b1
                }
                if (elected) umma_commit(&empty[s]);
                __syncwarp();
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_MMA); }
            if (ok && elected) umma_commit(done);
            __syncwarp();
        }
    } else if (warp < 8) {
        // =========================== running sums and results ====================================================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SUMS));
        const int q = warp % 4, m = m0 + q * 32 + lane;
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
        float acc[BN];
#pragma unroll
        for (int j = 0; j < BN; ++j) acc[j] = 0.f;
        bool ok = true;
        for (int it = 0; it < n_iters; ++it) {
            ok = __all_sync(0xffffffffu, mbar_wait(lead_full, (uint32_t)(it & 1)) ? 1 : 0) != 0;
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < BN; c += 16) {
                uint32_t v[16];
                tmem_ld16(taddr + c, v);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[c + j] += __uint_as_float(v[j]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(lead_empty));
        }
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(done, 0) ? 1 : 0) != 0;
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_EPI); }
        if (ok) {
            tc_fence_after();
            const bool raw = MODE == CMODE_WGRAD || p.splits > 1;
            const size_t row = (size_t)m * p.N;
            float* dst = (raw ? p.part + (size_t)blockIdx.z * p.split_stride : p.out) + row;
            const bool row_ok = m < p.M;
            bool bad = false;
#pragma unroll
            for (int c = 0; c < BN; c += 8) {
                uint32_t v[8];
                tmem_ld8(taddr + BN + c, v);
                tmem_ld_wait();
                float f[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    f[j] = acc[c + j] + __uint_as_float(v[j]);
                    bad = bad || f[j] != f[j];
                }
                if (row_ok && n0 + c < p.N) {
                    if (!raw) finish8<MODE>(p, f, row + n0 + c, n0 + c);
                    float4* d = (float4*)(dst + n0 + c);
                    d[0] = make_float4(f[0], f[1], f[2], f[3]);
                    d[1] = make_float4(f[4], f[5], f[6], f[7]);
                }
            }
            if (row_ok && bad) {
                const int k0 = chunk0 * 64, k1 = min(p.K, (chunk0 + n_iters) * 64);
                for (int n = n0; n < min(n0 + BN, p.N); n += 8) {
                    float f[8];
                    for (int j = 0; j < 8; ++j) f[j] = plain_sum<MODE>(p, m, n + j, k0, k1);
                    if (!raw) finish8<MODE>(p, f, row + n, n);
                    for (int j = 0; j < 8; ++j) dst[n + j] = f[j];
                }
            }
        }
    } else {
        // =========================== converters ==================================================================================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_CONV));
        const int t = threadIdx.x - CONV0, HW = p.H * p.W;
        const int Cred = MODE == CMODE_DGRAD ? p.Cout : p.Cin;
        F8 ra[2], rb[NB];
        int kpos = chunk0 * 64;           // first reduction step of the chunk

        // A: this thread's row is the TMEM lane of its warp's quadrant, its reduction steps a quarter of the chunk
        const int row = (warp & 3) * 32 + lane, quarter = (warp - 8) >> 2, m = m0 + row;
        const uint32_t a_at = tmem + COL_A + ((uint32_t)((warp & 3) * 32) << 16) + 8u * quarter;
        const float* a_px = nullptr;      // FWD / DGRAD: the pixel, and which taps fall inside the image; WGRAD: the column of dy
        uint32_t a_in = 0u;
        int a_tap = 0, a_c = 0;           // FWD / DGRAD: place of the thread's quarter along the reduction
        // B: row r and the q-th run of eight floats of each 64-float row piece (FWD: rows r, r + 64; DGRAD, WGRAD: row r along the
        // reduction, NB boxes of columns)
        const int q = t & 7, r = t >> 3;
        const uint32_t b_at = smem_u32(smem) + (uint32_t)r * 128u + (uint32_t)((q ^ (r & 7)) << 4);
        const float* b_px = nullptr;      // FWD: weight row; DGRAD: column run of the weights
        bool b_in[NB];
        int b_tap = 0, b_o = 0;                     // DGRAD: the weight row's tap and output channel
        int b_h = 0, b_w = 0, dr[NB], ds[NB];       // WGRAD: the pixel row's place; per run its tap shift and
        int b_shift[NB];                            // the float it starts at relative to the pixel's first
        if (MODE != CMODE_WGRAD) {
            const int k = kpos + 16 * quarter;
            a_tap = k / Cred; a_c = k - a_tap * Cred;
            if (m < p.M) {
                const int n = div_rcp(m, p.rcp_hw, HW), w = m - n * HW, h = div_rcp(w, p.rcp_w, p.W), x = w - h * p.W;
                a_px = (MODE == CMODE_FWD ? p.act : p.dy) + (size_t)m * Cred;
                if (p.taps == 1) a_in = 1u;
                else
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const int er = MODE == CMODE_FWD ? i / 3 - 1 : 1 - i / 3, es = MODE == CMODE_FWD ? i % 3 - 1 : 1 - i % 3;
                        if ((unsigned)(h + er) < (unsigned)p.H && (unsigned)(x + es) < (unsigned)p.W) a_in |= 1u << i;
                    }
            }
        } else {
            a_px = p.dy + m;
        }
        if (MODE == CMODE_FWD) {
            b_px = p.wt + (size_t)(n0 + r) * p.K + 8 * q;
#pragma unroll
            for (int j = 0; j < NB; ++j) b_in[j] = n0 + r + 64 * j < p.N;
        } else {
#pragma unroll
            for (int j = 0; j < NB; ++j) b_in[j] = n0 + 64 * j + 8 * q < p.N;
            if (MODE == CMODE_DGRAD) {
                b_px = p.wt + n0 + 8 * q;
                b_tap = (kpos + r) / Cred; b_o = kpos + r - b_tap * Cred;
            } else {
                const int w = kpos + r - div_rcp(kpos + r, p.rcp_hw, HW) * HW;
                b_h = div_rcp(w, p.rcp_w, p.W); b_w = w - b_h * p.W;
#pragma unroll
                for (int j = 0; j < NB; ++j) {
                    const int n = n0 + 64 * j + 8 * q, tap = b_in[j] ? n / p.Cin : 0;
                    dr[j] = p.taps == 9 ? tap / 3 - 1 : 0; ds[j] = p.taps == 9 ? tap % 3 - 1 : 0;
                    b_shift[j] = (dr[j] * p.W + ds[j]) * p.Cin + (n - tap * p.Cin);
                }
            }
        }
        const int step_h = (64 / p.W) % p.H, step_w = 64 % p.W;       // WGRAD: one chunk on, in rows and columns

        auto tap_shift = [&](int tap) {
            if (p.taps == 1) return 0;
            const int tr = tap >= 6 ? 2 : (tap >= 3 ? 1 : 0), ts = tap - 3 * tr;
            return (MODE == CMODE_FWD ? (tr - 1) * p.W + ts - 1 : (1 - tr) * p.W + 1 - ts) * Cred;
        };
        auto load_a = [&] {
            if (MODE == CMODE_WGRAD) {
                const int k = kpos + 16 * quarter, left = m < p.M ? p.K - k : 0;
                const float* d = a_px + (size_t)k * p.Cout;
#pragma unroll
                for (int j = 0; j < 16; ++j) ra[j / 8].v[j % 8] = j < left ? __ldg(d + (size_t)j * p.Cout) : 0.f;
            } else if (K64) {
                const float* d = a_px + (long)tap_shift(a_tap) + a_c;
                const bool in = (a_in >> a_tap) & 1u;
                load8(ra[0], d, in);
                load8(ra[1], d + 8, in);
            } else {
                int tap = a_tap, c = a_c;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    load8(ra[i], a_px + (long)tap_shift(tap) + c, (a_in >> tap) & 1u);
                    c += 8;
                    if (c == Cred) { c = 0; ++tap; }
                }
            }
        };
        auto load_b = [&](int j) {
            if (MODE == CMODE_FWD) load8(rb[j], b_px + (size_t)(64 * j) * p.K + kpos, b_in[j] && (K64 || kpos + 8 * q < p.K));
            else if (MODE == CMODE_DGRAD) load8(rb[j], b_px + ((size_t)b_o * p.taps + b_tap) * p.Cin + 64 * j, b_in[j] && b_tap < p.taps);
            else load8(rb[j], p.act + (long)(kpos + r) * p.Cin + b_shift[j],
                       b_in[j] && kpos + r < p.K && (unsigned)(b_h + dr[j]) < (unsigned)p.H && (unsigned)(b_w + ds[j]) < (unsigned)p.W);
        };
        auto advance = [&] {
            kpos += 64;
            if (MODE == CMODE_WGRAD) {
                b_w += step_w; b_h += step_h;
                if (b_w >= p.W) { b_w -= p.W; ++b_h; }
                if (b_h >= p.H) b_h -= p.H;
            } else if (K64) {
                a_c += 64;
                if (a_c >= Cred) { a_c -= Cred; ++a_tap; }
            } else {
                for (a_c += 64; a_c >= Cred; a_c -= Cred) ++a_tap;
            }
            if (MODE == CMODE_DGRAD)
                for (b_o += 64; b_o >= Cred; b_o -= Cred) ++b_tap;
        };
        const bool do_bias = MODE == CMODE_WGRAD && blockIdx.y == 0;
        float bsum = 0.f;

        load_a();
#pragma unroll
        for (int j = 0; j < NB; ++j) load_b(j);
        int s = 0;
        uint32_t ph = 1;      // (a stage's first use needs no wait)
        bool ok = true;
        for (int it = 0; it < n_iters; ++it) {
            if (it >= STAGES) {
                ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], ph) ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
            }
            const bool more = it + 1 < n_iters;
            if (more) advance();
            {
                uint32_t t0[8], t1[8], t2[8];
                take_terms(ra[0], t0, t1, t2);
                take_terms(ra[1], t0 + 4, t1 + 4, t2 + 4);
                if (do_bias)
#pragma unroll
                    for (int j = 0; j < 16; ++j) bsum += ra[j / 8].v[j % 8];
                __syncwarp();
                const uint32_t at = a_at + (uint32_t)s * A_STAGE;
                tmem_st8(at, t0);
                tmem_st8(at + A_TERM, t1);
                tmem_st8(at + 2 * A_TERM, t2);
                if (more) load_a();
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                uint32_t t0[4], t1[4], t2[4];
                take_terms(rb[j], t0, t1, t2);
                const uint32_t at = b_at + (uint32_t)s * C::STAGE + 8192u * j;
                st_shared16(at, t0);
                st_shared16(at + C::PLANE, t1);
                st_shared16(at + 2 * C::PLANE, t2);
                if (more) load_b(j);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&full[s]));
            if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_TMA); }
        if (do_bias) {
            if (quarter > 0) s_bias[(quarter - 1) * 128 + row] = bsum;
            asm volatile("bar.sync 2, 512;" ::: "memory");
            if (quarter == 0 && m < p.M)
                p.part[(size_t)blockIdx.z * p.split_stride + p.bias_off + m] = ((bsum + s_bias[row]) + s_bias[128 + row]) + s_bias[256 + row];
        }
    }

    // ---- teardown: TMEM is released on every path ----------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        const uint64_t t0 = globaltimer_ns();          // MMAs that may still be in flight read shared memory
        while (globaltimer_ns() - t0 < 200000ull) { }
        __syncthreads();
    }
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

uint32_t rcp_of(int d) { return d <= 1 ? 0u : (uint32_t)(0x100000000ull / (uint32_t)d) + 1u; }

template <int MODE, int BN, bool K64>
cudaError_t launch_one(const SplitParams& p, cudaStream_t st)
{
    constexpr int SMEM = SplitCfg<BN>::SMEM;
    const cudaError_t e = raise_smem_limit<contract_umma_kernel<MODE, BN, K64>>(SMEM);
    if (e != cudaSuccess) return e;
    return pdl_launch(contract_umma_kernel<MODE, BN, K64>, dim3((unsigned)((p.M + 127) / 128), (unsigned)((p.N + BN - 1) / BN), (unsigned)p.splits), dim3(THREADS),
                      (size_t)SMEM, st, p);
}
template <int MODE>
cudaError_t launch_mode(int bn, const SplitParams& p, cudaStream_t st)
{
    if (MODE == CMODE_WGRAD || (MODE == CMODE_DGRAD ? p.Cout : p.Cin) % 64 == 0)
        return bn == 128 ? launch_one<MODE, 128, true>(p, st) : launch_one<MODE, 64, true>(p, st);
    return bn == 128 ? launch_one<MODE, 128, MODE == CMODE_WGRAD>(p, st) : launch_one<MODE, 64, MODE == CMODE_WGRAD>(p, st);
}

}  // namespace

bool contract_umma_ok(int taps, int Cin, int Cout) { return Cin % 8 == 0 && Cout % 8 == 0 && (taps == 1 || taps == 9); }

cudaError_t launch_contract_umma(const ContractArgs& a, cudaStream_t st)
{
    SplitParams p{};
    p.act = (const float*)a.act; p.wt = (const float*)a.wt; p.dy = (const float*)a.dy;
    p.taps = a.taps; p.H = a.H; p.W = a.W; p.Cin = a.Cin; p.Cout = a.Cout;
    p.npix = a.B * a.H * a.W;
    p.rcp_w = rcp_of(a.W); p.rcp_hw = rcp_of(a.H * a.W);
    p.M = a.mode == CMODE_WGRAD ? a.Cout : p.npix;
    p.N = a.mode == CMODE_FWD ? a.Cout : a.mode == CMODE_DGRAD ? a.Cin : a.taps * a.Cin;
    p.K = a.mode == CMODE_WGRAD ? p.npix : a.taps * (a.mode == CMODE_DGRAD ? a.Cout : a.Cin);
    p.chunks = (p.K + 63) / 64; p.cps = a.plan.iters; p.splits = a.plan.splits;
    p.part = a.part; p.split_stride = a.split_stride; p.bias_off = a.bias_off;
    p.out = a.out32 ? a.out32 : (float*)a.out; p.bias = a.bias; p.relu = a.relu; p.ref = (const float*)a.ref;
    p.status = a.status;
    if (a.mode == CMODE_FWD) return launch_mode<CMODE_FWD>(a.plan.bn, p, st);
    return a.mode == CMODE_DGRAD ? launch_mode<CMODE_DGRAD>(a.plan.bn, p, st) : launch_mode<CMODE_WGRAD>(a.plan.bn, p, st);
}

}  // namespace sb
