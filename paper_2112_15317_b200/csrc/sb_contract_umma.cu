// Float contractions on the tensor cores: every float operand element (times 2^16, see OPERAND_SCALE_X2) is taken apart into three bf16
// terms that add up to it (8 + 8 + 8 significant bits), and the products of the terms are accumulated in float.
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
// accumulator of their own for 64 such chunks: at most 1280 truncated additions to a sum of 2^-8 of the result, 1.5e-7 of it if they all
// have one sign (over 784 chunks, a weight gradient at 28x28 and batch 64, 2.1e-6).  Floats as sums of bf16 terms: G. Henry, P. T. P. Tang
// and A. Heinecke, "Leveraging the bfloat16 artificial intelligence datatype for higher-precision computations" (2019); sums kept out of
// the truncating accumulator: H. Ootomo and R. Yokota, "Recovering single precision accuracy from tensor cores" (2022).
// Error against 64-bit sums (2-norm; half-normal x, normal w and dy), CUDA cores -> here:
//   3x3, 64 channels at 32x32, batch 96    forward 2.9e-7 -> 0.8e-7   input gradient 4.3e-7 -> 1.0e-7   weight gradient 3.9e-7 -> 1.8e-7
//   3x3, 256 channels at 8x8, batch 96             3.4e-7 -> 0.9e-7                  4.8e-7 -> 1.0e-7                   3.3e-7 -> 1.1e-7
//   4096 -> 1024, batch 96                         1.8e-7 -> 1.0e-7                  2.1e-7 -> 0.9e-7                   1.3e-7 -> 0.5e-7
//   3x3, 8 -> 40 channels at 5x7, batch 3          0.7e-7 -> 0.6e-7                  1.4e-7 -> 0.9e-7                   1.1e-7 -> 0.5e-7
//
// One CTA per SM walks (tile, split) units; the results of a unit are written while the next one is under way.  Roles (24 warps, 16
// where the weights arrive as terms; registers are moved between them): warp 0 allocates TMEM and issues the MMAs; warp 1 fetches A as
// raw floats and warp 2 the weights' terms by TMA; warps 4-7 keep the running sums and write the results; warps 8 and up take the
// floats apart and store the terms, A into tensor memory (a lane per row; WGRAD: transposed on the way) and B as 128-byte swizzled
// rows of shared memory, the next chunk of B in flight behind the conversion of the present one.  A in tensor memory keeps its terms
// off the shared-memory port, which would else carry 40 KB per 16 steps of a 128 x 128 tile.  The weights of a convolution are read by
// every row tile, so a kernel of their own takes them apart once a call.
//
// What bounds it: forward and input gradient, the chain through the issuing warp: a chunk of 128 x 128 x 64 takes 2350 cycles where
// its 24 MMAs take 1536, one of 128 x 64 x 64 1750 (768). Measured with clocks in the kernel: of 1890 cycles of the narrow chunk 1290
// went into getting 24 instructions out (54 each) and 600 into waits, most of them for barriers that had long flipped. Hence 16
// instructions of twice the width there, and the next chunk's barriers tested behind the last queued instructions: 66 -> 58 us forward
// over 64 channels, 7-conv / 3-FC net 957 -> 925 an iteration. (A's rows fetched once for the three taps of a filter row and a deeper
// ring for the weights' terms gave 1 - 6 us alone and took 17 in the iteration: fetches don't bound it, and 226 KB kept the next
// kernel out.) WGRAD: issue slots, 2.9 of 4 a cycle: 16 converter warps of 350 instructions a chunk, the summing warps' 128 additions
// and the MMA warp. Without TMA and with a CTA per unit the same layers took a third longer (a row per lane made each load of A 32
// wavefronts of the L1 port). Where the weights arrive as terms eight warps of 32 elements convert, not 16 of 16 (half the waits and
// arrivals: 66 -> 62). Float CUDA cores -> here, us between events at batch 96 (about 4 of them the launch): 3x3 over 64 channels at 32x32
// forward 183 -> 58, input gradient 189 -> 67, weight gradient 181 -> 97; 128 channels at 16x16 158 / 169 / 160 -> 54 / 55 / 52; 256
// channels at 8x8 159 / 174 / 162 -> 46 / 46 / 52; 4096 -> 1024 33 / 31 / 27 -> 22 / 21 / 23. The 7-conv / 3-FC net: 2.54 -> 0.89 ms an
// iteration.
//
// Non-finite operands: infinity - infinity in the splitting makes the terms NaN where a float multiply-add would give an infinity, so
// results that are not finite are looked at again behind the CTA's last unit, when no other warp waits (repair_unit).
#include "sb_umma.h"
#include "sb_tcgen05.cuh"

namespace sb {

namespace {

uint32_t rcp_of(int d) { return d <= 1 ? 0u : (uint32_t)(0x100000000ull / (uint32_t)d) + 1u; }

struct SplitParams {
    const float *act, *wt, *dy;
    int taps, H, W, Cin, Cout, npix;
    uint32_t rcp_w, rcp_hw;
    int M, N, K;                   // rows, columns, reduction length (WGRAD: pixels)
    int chunks, cps, splits;       // 64-step chunks, per split
    int m_tiles, n_tiles, units;   // (tile, split) pairs, walked by the CTAs in turn
    uint32_t rcp_m, rcp_n;
    float* part; long split_stride;
    long bias_off;
    float* out; const float* bias; int relu;
    const float* ref;
    uint32_t* status;
};

// Warps: 4 issue, 4 keep sums, CW convert: 16, or 8 where they convert A only.  Registers are a share of those at launch:
// 80 a thread: 32 + 160 + 4 * 72 = 6 * 80; 128 a thread: 40 + 200 + 2 * 136 = 4 * 128.
template <bool WT> struct Roles {
    static constexpr int CW = WT ? 8 : 16, THREADS = 256 + 32 * CW, PARTS = 16 / CW;      // PARTS: quarters of a chunk's row a converter takes
    static constexpr int REGS_ISSUE = WT ? 40 : 32, REGS_SUMS = WT ? 200 : 160, REGS_CONV = WT ? 136 : 72;
};
static_assert(Roles<true>::REGS_ISSUE < 128 && Roles<true>::REGS_CONV > 128 && Roles<true>::REGS_ISSUE + Roles<true>::REGS_SUMS + 2 * Roles<true>::REGS_CONV <= 4 * 128, "dec lowers, inc raises, within the launch's");
static_assert(Roles<false>::REGS_ISSUE < 80 && Roles<false>::REGS_CONV < 80 && Roles<false>::REGS_ISSUE + Roles<false>::REGS_SUMS + 4 * Roles<false>::REGS_CONV <= 6 * 80, "");
constexpr int CONV0 = 256;
constexpr int STAGES = 2, RAWS = 2, RAW = 32768, CTRL = 8192;
// Both operands are multiplied by 2^16 before they are taken apart, so that the last term of the smallest float is still a bf16 number
// (unscaled, operands below 2^-110 lost bits: 2e-6 of the result at 2^-116, 2e-3 at 2^-126), and the results by 2^-32.  Results that
// overflow meanwhile (2^96 and more) are looked at again, as NaNs are.
constexpr unsigned long long OPERAND_SCALE_X2 = 0x4780000047800000ull;
constexpr float RESULT_SCALE = 0x1p-32f;
constexpr int REST_CHUNKS = 64;      // after which the accumulator of the other products is emptied
// PLANE: one term of the B tile, BN rows of 128 bytes (FWD) or 64-column boxes of 64 rows.  RAW: a chunk of A as floats, 32-column
// boxes of 128-byte swizzled rows.  Tensor memory columns: buffers of leading products, buffers of the other products, then the
// terms of A (2 stages x 3 x 32).  PAIRED (64 wide): the other products lie side by side, a0 b1 + a1 b0 and a0 b2 + a1 b1 + a2 b0, so
// that one instruction multiplies a term of A with two terms of B, neighbours in shared memory: 16 instructions a chunk, not 24, of
// which the issuing warp gets one out in 54 cycles (a 64-wide one takes the tensor pipe 32).
template <int BN> struct SplitCfg {
    static constexpr int PLANE = BN * 128, STAGE = 3 * PLANE;
    static constexpr int smem(bool tma) { return STAGES * STAGE + (tma ? RAWS * RAW : 0) + 1024 + CTRL; }
    static constexpr int LEADS = BN == 64 ? 3 : 1, RESTS = 1;
    static constexpr bool PAIRED = BN == 64;
    static constexpr int REST = PAIRED ? 2 * BN : BN;      // columns
    static constexpr uint32_t COL_REST = LEADS * BN, COL_A = COL_REST + RESTS * REST;
};
constexpr uint32_t A_TERM = 32, A_STAGE = 3 * A_TERM, TMEM_COLS = 512;
static_assert(SplitCfg<64>::COL_A + STAGES * A_STAGE <= TMEM_COLS && SplitCfg<128>::COL_A + STAGES * A_STAGE <= TMEM_COLS, "tensor memory");

__device__ __forceinline__ int div_rcp(int n, uint32_t mul, int d)
{
    if (mul == 0u) return n;
    uint32_t q = __umulhi((uint32_t)n, mul);
    if (q * (uint32_t)d > (uint32_t)n) --q;
    return (int)q;
}
// whether a phase of a barrier has ended (does not wait)
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return done != 0;
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
// two floats, times OPERAND_SCALE
__device__ __forceinline__ void scale_pair(float& a, float& b)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(OPERAND_SCALE_X2));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d));
}
// the three terms of eight floats
__device__ __forceinline__ void take_terms(const F8& f, uint32_t* t0, uint32_t* t1, uint32_t* t2)
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float a = f.v[2 * j], b = f.v[2 * j + 1];
        scale_pair(a, b);
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
// Which taps of output pixel m fall inside the image (a bit each)
template <int MODE>
__device__ __forceinline__ uint32_t taps_inside(const SplitParams& p, int m)
{
    uint32_t in = 0u;
    if (m >= p.M) return in;
    if (p.taps == 1) return 1u;
    const int HW = p.H * p.W, n = div_rcp(m, p.rcp_hw, HW), w = m - n * HW, h = div_rcp(w, p.rcp_w, p.W), x = w - h * p.W;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int er = MODE == CMODE_FWD ? i / 3 - 1 : 1 - i / 3, es = MODE == CMODE_FWD ? i % 3 - 1 : 1 - i % 3;
        if ((unsigned)(h + er) < (unsigned)p.H && (unsigned)(x + es) < (unsigned)p.W) in |= 1u << i;
    }
    return in;
}
__device__ __forceinline__ bool finite(float f) { return fabsf(f) < INFINITY; }
// Eight results of a row: bias and ReLU, or the ReLU mask.  What is not finite stays so here: it is looked at again (repair_unit).
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
            const float y = f[j] + e[j];
            f[j] = p.relu && !(y > 0.f) && finite(f[j]) ? 0.f : y;
        } else if (!(e[j] > 0.f) && finite(f[j])) f[j] = 0.f;
    }
}
// One result (NaN -> 0 behind a ReLU or a mask, as everywhere)

template <int MODE>
__device__ __forceinline__ float finish1(const SplitParams& p, float f, size_t at, int n)
{
    if (MODE == CMODE_FWD) {
        f += p.bias[n];
        return p.relu && !(f > 0.f) ? 0.f : f;
    }
    return p.ref != nullptr && !(p.ref[at] > 0.f) ? 0.f : f;
}

template <bool TMA> struct Maps { CUtensorMap a, b; };      // raw floats of A, terms of the weights
template <> struct Maps<false> { };
// One (tile, split) pair
struct Unit { int m0, n0, split, chunk0, n_iters; };
template <int BN>
__device__ __forceinline__ Unit unit_at(const SplitParams& p, int u)
{
    const int r = div_rcp(u, p.rcp_m, p.m_tiles), z = div_rcp(r, p.rcp_n, p.n_tiles);
    Unit t;
    t.m0 = (u - r * p.m_tiles) * 128;
    t.n0 = (r - z * p.n_tiles) * BN;
    t.split = z;
    t.chunk0 = z * p.cps;
    t.n_iters = min(p.cps, p.chunks - t.chunk0);
    return t;
}
// Results of a unit that came out as NaN or infinite, by one warp for the 32 rows that it has stored (those unfinished): what plain
// multiply-adds give.  A NaN operand makes its whole row or column NaN (places outside the image are zeros that are multiplied, as in
// contract_kernel: NaN x 0 and infinity x 0 are NaN), so the operands are searched for those first, and the search ends when they
// explain every such result: a run that has diverged costs one look at the operands.  What is left has infinite or large operands
// in its sum, or is too large: the blocks of 32 steps that hold large operands (in 1024 groups, a bit each, 32 to a lane) are summed, a lane
// to two or four columns of as many rows, and all of them only where that is finite.
// (a predicate, not a branch, so that the loads of several steps are under way together)
__device__ __forceinline__ float load_if(const float* p, bool there)
{
    float v;
    asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t@p ld.global.f32 %0, [%1];\n\t}" : "=f"(v) : "l"(p), "r"((int)there));
    return v;
}
__device__ __forceinline__ void load8_if(F8& f, const float* p, bool there)      // (at a 16-byte boundary)
{
#pragma unroll
    for (int h = 0; h < 8; h += 4)
        asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
            "@p ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}" : "=f"(f.v[h]), "=f"(f.v[h + 1]), "=f"(f.v[h + 2]), "=f"(f.v[h + 3]) : "l"(p + h), "r"((int)there));
}
template <int MODE> struct Step {      // a reduction step's tap and channel; WGRAD: its pixel's row and column
    int k, tap, c;
    __device__ __forceinline__ Step(const SplitParams& p, int k_) : k(k_)
    {
        if (MODE == CMODE_WGRAD) {
            const int HW = p.H * p.W, r = k - div_rcp(k, p.rcp_hw, HW) * HW;
            tap = div_rcp(r, p.rcp_w, p.W); c = r - tap * p.W;
        } else {
            const int cred = MODE == CMODE_DGRAD ? p.Cout : p.Cin;
            tap = k / cred; c = k - tap * cred;
        }
    }
    __device__ __forceinline__ void next(const SplitParams& p)
    {
        ++k;
        if (++c == (MODE == CMODE_WGRAD ? p.W : MODE == CMODE_DGRAD ? p.Cout : p.Cin)) {
            c = 0;
            if (++tap == p.H && MODE == CMODE_WGRAD) tap = 0;
        }
    }
};
template <int MODE> struct Column {    // of the result; WGRAD: its tap's shift
    const float* at;
    int dr = 0, ds = 0;
    bool in;
    Column() = default;
    __device__ __forceinline__ Column(const SplitParams& p, int n) : in(n < p.N)
    {
        n = in ? n : 0;
        if (MODE == CMODE_WGRAD) {
            const int t = n / p.Cin;
            if (p.taps == 9) { dr = t / 3 - 1; ds = t % 3 - 1; }
            at = p.act + ((long)dr * p.W + ds) * p.Cin + (n - t * p.Cin);
        } else at = MODE == CMODE_FWD ? p.wt + (size_t)n * p.K : p.wt + n;
    }
    __device__ __forceinline__ float operand(const SplitParams& p, const Step<MODE>& s, bool there = true) const
    {
        bool ok = in && there;
        const float* a = at;
        if (MODE == CMODE_FWD) a += s.k;
        else if (MODE == CMODE_DGRAD) a += ((size_t)s.c * p.taps + s.tap) * p.Cin;
        else {
            a += (size_t)s.k * p.Cin;
            ok = ok && (unsigned)(s.tap + dr) < (unsigned)p.H && (unsigned)(s.c + ds) < (unsigned)p.W;
        }
        return load_if(a, ok);
    }
};
template <int MODE>
__device__ __forceinline__ float row_operand(const SplitParams& p, int m, uint32_t inside, const Step<MODE>& s, bool there = true)
{
    const float* a = MODE == CMODE_FWD ? p.act : p.dy;
    if (MODE == CMODE_WGRAD) return load_if(a + (size_t)s.k * p.Cout + m, there && m < p.M);
    const int shift = p.taps == 9 ? (s.tap / 3 - 1) * p.W + s.tap % 3 - 1 : 0;
    a += ((long)m + (MODE == CMODE_FWD ? shift : -shift)) * (MODE == CMODE_FWD ? p.Cin : p.Cout) + s.c;
    return load_if(a, there && ((inside >> s.tap) & 1u) != 0u);      // (no tap of a row past the last is inside)
}
// The eight reduction steps from k on (below k1), a multiple of eight: one tap's channels, or WGRAD: pixels (a bit each: steps that there
// are, and those with an image row or column before and behind them)
template <int MODE> struct Eight {
    int k, tap = 0, c = 0;
    uint32_t all, up = 0u, down = 0u, left = 0u, right = 0u;
    __device__ __forceinline__ Eight(const SplitParams& p, int k_, int k1) : k(k_), all(k_ >= k1 ? 0u : k_ + 8 <= k1 ? 0xffu : (1u << (k1 - k_)) - 1u)
    {
        Step<MODE> s(p, k);
        if constexpr (MODE == CMODE_WGRAD) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                up |= (s.tap > 0 ? 1u : 0u) << i; down |= (s.tap + 1 < p.H ? 1u : 0u) << i;
                left |= (s.c > 0 ? 1u : 0u) << i; right |= (s.c + 1 < p.W ? 1u : 0u) << i;
                s.next(p);
            }
        } else {
            tap = s.tap; c = s.c;
        }
    }
    __device__ __forceinline__ void row(const SplitParams& p, F8& f, int m, uint32_t inside) const
    {
        if constexpr (MODE == CMODE_WGRAD) {
            const float* from = p.dy + (size_t)k * p.Cout + m;
            const uint32_t there = m < p.M ? all : 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) f.v[i] = load_if(from + (size_t)i * p.Cout, (there >> i) & 1u);
        } else {
            const int shift = p.taps == 9 ? (tap / 3 - 1) * p.W + tap % 3 - 1 : 0;
            const float* from = MODE == CMODE_FWD ? p.act + ((long)m + shift) * p.Cin + c : p.dy + ((long)m - shift) * p.Cout + c;
            load8_if(f, from, all != 0u && ((inside >> tap) & 1u) != 0u);      // (channel counts are multiples of eight)
        }
    }
    __device__ __forceinline__ void column(const SplitParams& p, F8& f, const Column<MODE>& col) const
    {
        if constexpr (MODE == CMODE_FWD) {
            load8_if(f, col.at + k, col.in && all != 0u);
        } else {
            uint32_t there = col.in ? all : 0u;
            size_t stride = p.Cin;
            const float* from = col.at + (size_t)k * p.Cin;
            if constexpr (MODE == CMODE_DGRAD) {
                stride = (size_t)p.taps * p.Cin;
                from = col.at + ((size_t)c * p.taps + tap) * p.Cin;
            } else {
                if (col.dr != 0) there &= col.dr < 0 ? up : down;
                if (col.ds != 0) there &= col.ds < 0 ? left : right;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) f.v[i] = load_if(from + i * stride, (there >> i) & 1u);
        }
    }
};
// All operands of the 32 steps from k on (below k1) to the warp's rows and the unit's columns: a lane per step where an operand lies
// along the reduction in memory, else a lane per line.  f(value, line, whether it is a column's)
template <int MODE, int BN, typename F>
__device__ __forceinline__ void visit(const SplitParams& p, const Column<MODE> (&col)[BN / 32], int row0, int n0, uint32_t inside, int k, int k1, F f)
{
    const int lane = threadIdx.x % 32;
    const Step<MODE> mine(p, k + lane);
    if (MODE == CMODE_FWD) {
#pragma unroll 16
        for (int i = 0; i < BN; ++i) f(Column<MODE>(p, n0 + i).operand(p, mine, k + lane < k1), i, true);
    } else {
        Step<MODE> s(p, k);
#pragma unroll 8
        for (int i = 0; i < 32; ++i, s.next(p))
#pragma unroll
            for (int b = 0; b < BN / 32; ++b) f(col[b].operand(p, s, k + i < k1), 32 * b + lane, true);
    }
    if (MODE == CMODE_WGRAD) {
        Step<MODE> s(p, k);
#pragma unroll 16
        for (int i = 0; i < 32; ++i, s.next(p)) f(row_operand<MODE>(p, row0 + lane, 0u, s, k + i < k1), lane, false);
    } else {
#pragma unroll 16
        for (int i = 0; i < 32; ++i) f(row_operand<MODE>(p, row0 + i, __shfl_sync(0xffffffffu, inside, i), mine, k + lane < k1), i, false);
    }
}
template <int MODE, int BN>
__device__ __forceinline__ void repair_unit(const SplitParams& p, int u, int q)
{
    constexpr uint32_t ALL = 0xffffffffu;
    constexpr int CB = BN / 32;
    const Unit t = unit_at<BN>(p, u);
    const int lane = threadIdx.x % 32, row0 = t.m0 + 32 * q;
    const int k0 = t.chunk0 * 64, k1 = min(p.K, (t.chunk0 + t.n_iters) * 64), group = 32 * ((k1 - k0 + 32 * 1024 - 1) / (32 * 1024));
    const bool raw_sums = MODE == CMODE_WGRAD || p.splits > 1;
    volatile float* const base = raw_sums ? p.part + (size_t)t.split * p.split_stride : p.out;
    const uint32_t inside = MODE == CMODE_WGRAD ? 0u : taps_inside<MODE>(p, row0 + lane);      // (of row `lane`)
    Column<MODE> col[CB];
#pragma unroll
    for (int b = 0; b < CB; ++b) col[b] = Column<MODE>(p, t.n0 + 32 * b + lane);
    uint32_t rows = 0u, cols[CB], row_nan = 0u, col_nan[CB], large = 0u;
#pragma unroll
    for (int b = 0; b < CB; ++b) cols[b] = col_nan[b] = 0u;
    for (int r = 0; r < 32 && row0 + r < p.M; ++r)
#pragma unroll
        for (int b = 0; b < CB; ++b) {
            const int n = t.n0 + 32 * b + lane;
            const float v = n < p.N ? base[(size_t)(row0 + r) * p.N + n] : 0.f;
            const uint32_t odd = __ballot_sync(ALL, !finite(v));
            cols[b] |= odd;
            if (odd != 0u) rows |= 1u << r;
        }
    auto explained = [&] {
        uint32_t c = 0u;
#pragma unroll
        for (int b = 0; b < CB; ++b) c |= cols[b] & ~col_nan[b];
        return c == 0u || (rows & ~row_nan) == 0u;
    };
    for (int k = k0; k < k1 && !explained(); k += 32) {
        // (products of operands below 2^53 are below 2^106: no sum of them overflows)
        constexpr uint32_t LARGE = 0x5a000000u, INF = 0x7f800000u;
        uint32_t top = 0u;
        visit<MODE, BN>(p, col, row0, t.n0, inside, k, k1, [&](float v, int, bool) { top = max(top, __float_as_uint(v) & 0x7fffffffu); });
        if (!__any_sync(ALL, top >= LARGE)) continue;
        uint32_t rn = 0u, cn[CB];
        bool any = false;
#pragma unroll
        for (int b = 0; b < CB; ++b) cn[b] = 0u;
        visit<MODE, BN>(p, col, row0, t.n0, inside, k, k1, [&](float v, int line, bool of_col) {
            const uint32_t a = __float_as_uint(v) & 0x7fffffffu;
            any = any || (a >= LARGE && a <= INF);
            if (a > INF && !of_col) rn |= 1u << line;
#pragma unroll
            for (int b = 0; b < CB; ++b)
                if (a > INF && of_col && line / 32 == b) cn[b] |= 1u << (line % 32);
        });
        row_nan |= __reduce_or_sync(ALL, rn);
#pragma unroll
        for (int b = 0; b < CB; ++b) col_nan[b] |= __reduce_or_sync(ALL, cn[b]);
        const int g = (k - k0) / group;
        if (__any_sync(ALL, any) && lane == g >> 5) large |= 1u << (g & 31);
    }
    constexpr int R = BN == 64 ? 4 : 2;
#pragma unroll 1
    for (int r0 = 0; r0 < 32; r0 += R) {
        if (((rows >> r0) & ((1u << R) - 1u)) == 0u) continue;
        float sum[R][CB];
        uint32_t in[R], mine = 0u, left = 0u;      // (a bit per result of the lane)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            in[r] = __shfl_sync(ALL, inside, r0 + r);
#pragma unroll
            for (int b = 0; b < CB; ++b) {
                const int n = t.n0 + 32 * b + lane;
                sum[r][b] = n < p.N && row0 + r0 + r < p.M ? base[(size_t)(row0 + r0 + r) * p.N + n] : 0.f;
                if (finite(sum[r][b])) continue;
                mine |= 1u << (r * CB + b);
                if (!((row_nan >> (r0 + r)) & 1u) && !((col_nan[b] >> lane) & 1u)) left |= 1u << (r * CB + b);
            }
        }
        // over the blocks with large operands, then, if some were left out and for what is finite, over all
#pragma unroll 1
        for (int pass = 0; pass < 2 && __any_sync(ALL, left != 0u); ++pass) {
            float again[R][CB];
            bool whole = true, alive = true;
#pragma unroll
            for (int j = 0; j < R * CB; ++j) again[j / CB][j % CB] = 0.f;
#pragma unroll 1
            for (int k = k0; k < k1 && __any_sync(ALL, alive); k += 32) {
                const int g = (k - k0) / group;
                if (pass == 0 && !((__shfl_sync(ALL, large, g >> 5) >> (g & 31)) & 1u)) {
                    whole = false;
                    continue;
                }
                float part[R][CB];
#pragma unroll
                for (int j = 0; j < R * CB; ++j) part[j / CB][j % CB] = 0.f;
#pragma unroll 1
                for (int i0 = 0; i0 < 32; i0 += 8) {
                    const Eight<MODE> e(p, k + i0, k1);
                    F8 a[R], c[CB];
#pragma unroll
                    for (int r = 0; r < R; ++r) e.row(p, a[r], row0 + r0 + r, in[r]);
#pragma unroll
                    for (int b = 0; b < CB; ++b) e.column(p, c[b], col[b]);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
#pragma unroll
                        for (int j = 0; j < R * CB; ++j) part[j / CB][j % CB] = fmaf(a[j / CB].v[i], c[j % CB].v[i], part[j / CB][j % CB]);
                }
                alive = false;      // (a NaN stays one)
#pragma unroll
                for (int j = 0; j < R * CB; ++j) {
                    again[j / CB][j % CB] += part[j / CB][j % CB];
                    alive = alive || (((left >> j) & 1u) != 0u && again[j / CB][j % CB] == again[j / CB][j % CB]);
                }
            }
#pragma unroll
            for (int j = 0; j < R * CB; ++j) {
                if (!((left >> j) & 1u)) continue;
                sum[j / CB][j % CB] = again[j / CB][j % CB];
                if (whole || !finite(again[j / CB][j % CB])) left &= ~(1u << j);
            }
        }
#pragma unroll
        for (int j = 0; j < R * CB; ++j) {
            const int m = row0 + r0 + j / CB, n = t.n0 + 32 * (j % CB) + lane;
            const size_t at = (size_t)m * p.N + n;
            if ((mine >> j) & 1u) base[at] = raw_sums ? sum[j / CB][j % CB] : finish1<MODE>(p, sum[j / CB][j % CB], at, n);
        }
    }
}
template <int MODE, int BN>
__device__ __noinline__ void repair_units(const SplitParams& p, int q)
{
    __syncwarp();      // (lanes read what others have stored)
    for (int u = blockIdx.x; u < p.units; u += gridDim.x) repair_unit<MODE, BN>(p, u, q);
}
// slot of a ring and the parity of its current use
struct Ring {
    int i = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next(int n) { if (++i == n) { i = 0; ph ^= 1u; } }
};

// WT: B arrives as terms by TMA (FWD, DGRAD of convolutions, whose weights every row tile reads: launch_split_weights), where the channels
// of the reduction are a multiple of 64, so that a chunk lies in one tap.
// TMA: A arrives as raw floats by TMA: with WT, whose chunk's rows of A are those of the tile, shifted, and in WGRAD; otherwise (FC
// layers among them) the converters load it themselves.
template <int MODE, int BN, bool TMA, bool WT>
__global__ void __launch_bounds__(Roles<WT>::THREADS, 1)
contract_umma_kernel(const __grid_constant__ Maps<TMA> maps, const __grid_constant__ SplitParams p)
{
    static_assert(MODE == CMODE_WGRAD ? TMA && !WT : TMA == WT, "the forms there are");
    using C = SplitCfg<BN>;
    using R = Roles<WT>;
    constexpr int NB = BN / 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* raw = smem + STAGES * C::STAGE;
    uint8_t* ctrl = raw + (TMA ? RAWS * RAW : 0);
    uint64_t* full = (uint64_t*)ctrl;               // [STAGES] terms stored: one arrival per converter warp (WT: and the weights' bytes)
    uint64_t* empty = full + STAGES;                // [STAGES] read by their MMAs
    uint64_t* raw_full = empty + STAGES;            // [RAWS] a chunk of A has landed
    uint64_t* raw_empty = raw_full + RAWS;          // [RAWS] ... and is in registers: one arrival per converter warp
    uint64_t* lead_full = raw_empty + RAWS;         // [LEADS] leading products of a chunk complete
    uint64_t* lead_empty = lead_full + C::LEADS;    // [LEADS] ... and taken over: one arrival per summing warp
    uint64_t* rest_full = lead_empty + C::LEADS;    // [RESTS] the other products of REST_CHUNKS chunks, or of a unit's last ones, complete
    uint64_t* rest_empty = rest_full + C::RESTS;    // [RESTS] ... and taken over
    uint32_t* tmem_slot = (uint32_t*)(rest_empty + C::RESTS);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    float* s_bias = (float*)(ctrl + 1024);          // [3][128]: WGRAD, sums of dy over the later quarters of the chunks

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (warp == 0) {
        // (the barriers lie one after another: a lane each)
        constexpr int B0 = STAGES, B1 = B0 + STAGES, B2 = B1 + RAWS, B3 = B2 + RAWS, B4 = B3 + C::LEADS, B5 = B4 + C::LEADS, B6 = B5 + C::RESTS, B7 = B6 + C::RESTS;
        if (lane < B7) {
            const uint32_t n = lane < B0 ? (uint32_t)(R::CW + (WT ? 1 : 0)) : lane < B2 ? 1u : lane < B3 ? (uint32_t)R::CW : lane < B4 ? 1u : lane < B5 ? 4u : lane < B6 ? 1u : 4u;
            mbar_init(&full[lane], n);
            if (lane == 0) *abort_flag = 0;
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
    const int Cred = MODE == CMODE_DGRAD ? p.Cout : p.Cin;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R::REGS_ISSUE));
        if (warp == 0) {
            // =========================== MMA issuer (the warp in lock-step, one elected lane issues) =============================
            constexpr bool B_MN = MODE != CMODE_FWD;
            constexpr uint32_t idesc = make_idesc(BN, 0, B_MN), idesc2 = make_idesc(2 * BN, 0, B_MN);
            constexpr uint32_t A_STEP = 8, B_STEP = (B_MN ? 2048u : 32u) >> 4, BP = C::PLANE >> 4;     // per 16 reduction steps: columns, 16-byte units
            const uint32_t elected = elect_one() ? 1u : 0u;
            const uint64_t dB = make_desc(smem_u32(smem), B_MN ? 8192u : 16u);
            const uint32_t b_hi = (uint32_t)(dB >> 32);
            Ring st, lead, rest;
            int chunk = 0;      // (a buffer's first use needs no wait)
            bool ok = true, ready = false;      // ready: the next chunk's terms and its buffer of leading products were seen to be
            for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
                const uint32_t n_iters = (uint32_t)unit_at<BN>(p, u).n_iters;
                for (uint32_t it = 0; it < n_iters; ++it, ++chunk) {
                    if (!ready) {
                        bool w = mbar_wait(&full[st.i], st.ph);
                        if (chunk >= C::LEADS) w = w && mbar_wait(&lead_empty[lead.i], lead.ph ^ 1u);
                        ok = __all_sync(0xffffffffu, w ? 1 : 0) != 0;
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint32_t a = tmem + C::COL_A + (uint32_t)st.i * A_STAGE, b = (uint32_t)dB + (uint32_t)st.i * (C::STAGE >> 4);
                    const uint32_t d0 = tmem + (uint32_t)lead.i * BN, d1 = tmem + C::COL_REST + (uint32_t)rest.i * C::REST;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) umma_ta(d0, a + kk * A_STEP, b + kk * B_STEP, b_hi, idesc, kk > 0 ? 1u : 0u, elected);
                    if (elected) umma_commit(&lead_full[lead.i]);
                    if (it % REST_CHUNKS == 0) {      // (a fresh barrier reports the phase before its first as complete)
                        ok = __all_sync(0xffffffffu, mbar_wait(&rest_empty[rest.i], rest.ph ^ 1u) ? 1 : 0) != 0;
                        if (!ok) break;
                        tc_fence_after();
                    }
                    const int st_now = st.i;
                    st.next(STAGES);
                    lead.next(C::LEADS);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint32_t ak = a + kk * A_STEP, bk = b + kk * B_STEP, acc = (it % REST_CHUNKS > 0 || kk > 0) ? 1u : 0u;
                        if (kk == 3) {      // behind the instructions still queued, not after them
                            bool w = mbar_test(&full[st.i], st.ph);
                            if (chunk + 1 >= C::LEADS) w = w && mbar_test(&lead_empty[lead.i], lead.ph ^ 1u);
                            ready = __all_sync(0xffffffffu, w ? 1 : 0) != 0;
                        }
                        if (C::PAIRED) {
                            umma_ta(d1, ak, bk + BP, b_hi, idesc2, acc, elected);                                     // a0 b1 | a0 b2
                            umma_ta(d1 + BN, ak + 2 * A_TERM, bk, b_hi, idesc, 1u, elected);                          //         a2 b0
                            umma_ta(d1, ak + A_TERM, bk, b_hi, idesc2, 1u, elected);                                  // a1 b0 | a1 b1
                        } else {
                            umma_ta(d1, ak + 2 * A_TERM, bk, b_hi, idesc, acc, elected);                              // a2 b0
                            umma_ta(d1, ak, bk + 2 * BP, b_hi, idesc, 1u, elected);                                   // a0 b2
                            umma_ta(d1, ak + A_TERM, bk + BP, b_hi, idesc, 1u, elected);                              // a1 b1
                            umma_ta(d1, ak + A_TERM, bk, b_hi, idesc, 1u, elected);                                   // a1 b0
                            umma_ta(d1, ak, bk + BP, b_hi, idesc, 1u, elected);                                       // a0 b1
                        }
                    }
                    if (elected) umma_commit(&empty[st_now]);
                    if ((it + 1) % REST_CHUNKS == 0 || it + 1 == n_iters) {
                        if (elected) umma_commit(&rest_full[rest.i]);
                        rest.next(C::RESTS);
                    }
                    __syncwarp();
                }
            }
            if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_MMA); }
            __syncwarp();
        } else if (TMA && warp == 1) {
            // =========================== raw floats of A =========================================================================
            if constexpr (TMA) if (lane == 0) {
                Ring r;
                int n = 0;
                bool ok = true;
                for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
                    const Unit t = unit_at<BN>(p, u);
                    int tap = MODE == CMODE_WGRAD ? 0 : t.chunk0 * 64 / Cred, c = MODE == CMODE_WGRAD ? 0 : t.chunk0 * 64 - tap * Cred;
                    for (int it = 0; it < t.n_iters; ++it, ++n) {
                        if (n >= RAWS && !(ok = mbar_wait(&raw_empty[r.i], r.ph ^ 1u))) break;
                        uint8_t* dst = raw + r.i * RAW;
                        mbar_expect_tx(&raw_full[r.i], (uint32_t)RAW);
                        if (MODE == CMODE_WGRAD) {
#pragma unroll
                            for (int b = 0; b < 4; ++b) tma_load_4d(&maps.a, dst + b * 8192, &raw_full[r.i], t.m0 + 32 * b, (t.chunk0 + it) * 64, 0, 0);
                        } else {
                            int shift = 0;      // in rows; rows of other images or of none are left out when the terms are taken
                            if (p.taps == 9) {
                                const int tr = tap / 3, ts = tap - 3 * tr;
                                shift = MODE == CMODE_FWD ? (tr - 1) * p.W + ts - 1 : (1 - tr) * p.W + 1 - ts;
                            }
#pragma unroll
                            for (int b = 0; b < 2; ++b) tma_load_4d(&maps.a, dst + b * 16384, &raw_full[r.i], c + 32 * b, t.m0 + shift, 0, 0);
                            c += 64;
                            if (c >= Cred) { c -= Cred; ++tap; }
                        }
                        r.next(RAWS);
                    }
                }
                if (!ok) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_TMA); }
            }
            __syncwarp();
        } else if (WT && warp == 2) {
            // =========================== terms of the weights ====================================================================
            if constexpr (WT) if (lane == 0) {
                Ring r;
                int n = 0;
                bool ok = true;
                for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
                    const Unit t = unit_at<BN>(p, u);
                    int tap = t.chunk0 * 64 / Cred, c = t.chunk0 * 64 - tap * Cred;
                    for (int it = 0; it < t.n_iters; ++it, ++n) {
                        if (n >= STAGES && !(ok = mbar_wait(&empty[r.i], r.ph ^ 1u))) break;
                        uint8_t* dst = smem + r.i * C::STAGE;
                        mbar_expect_tx(&full[r.i], (uint32_t)C::STAGE);
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            if (MODE == CMODE_FWD) tma_load_4d(&maps.b, dst + k * C::PLANE, &full[r.i], (t.chunk0 + it) * 64, t.n0, k, 0);
                            else
#pragma unroll
                                for (int j = 0; j < NB; ++j) tma_load_4d(&maps.b, dst + k * C::PLANE + j * 8192, &full[r.i], tap * p.Cin + t.n0 + 64 * j, c, k, 0);
                        }
                        c += 64;
                        if (c >= Cred) { c -= Cred; ++tap; }
                        r.next(STAGES);
                    }
                }
                if (!ok) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_TMA); }
            }
            __syncwarp();
        }
    } else if (warp < 8) {
        // =========================== running sums and results ====================================================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R::REGS_SUMS));
        const int q = warp % 4;
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
        const bool raw_sums = MODE == CMODE_WGRAD || p.splits > 1;
        constexpr int LD = WT ? 2 : 1;      // loads per wait: what the registers allow
        Ring lead, rest;
        bool ok = true;
        bool odd = false;      // one of this thread's sums is or was not finite (rows past the last too: repair_unit leaves those out)
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            const Unit t = unit_at<BN>(p, u);
            float acc[BN];
#pragma unroll
            for (int j = 0; j < BN; ++j) acc[j] = 0.f;
            bool others = false;
            for (int it = 0; it < t.n_iters || others;) {
                // the leading products chunk by chunk, the others whenever their accumulator is emptied
                uint64_t* in = others ? &rest_full[rest.i] : &lead_full[lead.i];
                ok = __all_sync(0xffffffffu, mbar_wait(in, others ? rest.ph : lead.ph) ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const uint32_t from = taddr + (others ? C::COL_REST + (uint32_t)rest.i * C::REST : (uint32_t)lead.i * BN);
                auto add = [&](uint32_t at) {
#pragma unroll
                    for (int c = 0; c < BN; c += 16 * LD) {
                        uint32_t v[LD][16];
#pragma unroll
                        for (int l = 0; l < LD; ++l) tmem_ld16(at + c + 16 * l, v[l]);
                        tmem_ld_wait();
#pragma unroll
                        for (int l = 0; l < LD; ++l)
#pragma unroll
                            for (int j = 0; j < 16; ++j) acc[c + 16 * l + j] += __uint_as_float(v[l][j]);
                    }
                };
                add(from);
                if (C::PAIRED && others) add(from + BN);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(others ? &rest_empty[rest.i] : &lead_empty[lead.i]));
                if (others) {
                    rest.next(C::RESTS);
                    others = false;
                } else {
                    lead.next(C::LEADS);
                    ++it;
                    others = it % REST_CHUNKS == 0 || it == t.n_iters;
                }
            }
            if (!ok) break;
            const int m = t.m0 + q * 32 + lane;
            float* const base = raw_sums ? p.part + (size_t)t.split * p.split_stride : p.out;
#pragma unroll
            for (int j = 0; j < BN; ++j) odd = odd || !finite(acc[j]);
            if (m < p.M) {
                const size_t row = (size_t)m * p.N;
#pragma unroll
                for (int c = 0; c < BN; c += 8) {
                    if (t.n0 + c >= p.N) continue;
                    float f[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) f[j] = RESULT_SCALE * acc[c + j];
                    if (!raw_sums) finish8<MODE>(p, f, row + t.n0 + c, t.n0 + c);
                    float4* d = (float4*)(base + row + t.n0 + c);
                    d[0] = make_float4(f[0], f[1], f[2], f[3]);
                    d[1] = make_float4(f[4], f[5], f[6], f[7]);
                }
            }
        }
        // (behind the last unit: no wait of the other warps depends on how long this takes)
        if (__any_sync(0xffffffffu, odd) && ok) repair_units<MODE, BN>(p, q);
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_EPI); }
    } else {
        // =========================== converters ==================================================================================
        if constexpr (WT) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R::REGS_CONV));     // (above those at launch)
        else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R::REGS_CONV));
        const int t = threadIdx.x - CONV0, HW = p.H * p.W;
        F8 ra[2 * R::PARTS], rb[NB];

        // A: this thread's row is the TMEM lane of its warp's quadrant, its reduction steps PARTS quarters of the chunk
        const int row = (warp & 3) * 32 + lane, quarter = ((warp - 8) >> 2) * R::PARTS;
        const uint32_t a_at = tmem + C::COL_A + ((uint32_t)((warp & 3) * 32) << 16) + 8u * quarter;
        // its place in the raw chunk: FWD, DGRAD: four 16-byte runs of its row; WGRAD: its column of 16 rows
        const uint32_t raw_at = smem_u32(raw) + (MODE == CMODE_WGRAD ? (uint32_t)(row >> 5) * 8192u + (uint32_t)quarter * 2048u + (uint32_t)(row & 3) * 4u
                                                                     : (uint32_t)(quarter >> 1) * 16384u + (uint32_t)row * 128u);
        uint32_t a_in = 0u;               // FWD, DGRAD: which taps of the unit's row fall inside the image
        int a_tap = 0, a_c = 0;           // place of the chunk (TMA) or of the thread's quarter (otherwise) along the reduction
        const float* a_px = nullptr;      // without TMA: the pixel, of the unit whose chunk is loaded next
        uint32_t a_px_in = 0u;
        // B, of the chunk loaded next: row r and the q-th run of eight floats of each 64-float row piece (FWD: rows r, r + 64; DGRAD,
        // WGRAD: row r along the reduction, NB boxes of columns)
        const int q = t & 7, r = t >> 3;
        const uint32_t b_at = smem_u32(smem) + (uint32_t)r * 128u + (uint32_t)((q ^ (r & 7)) << 4);
        int kpos = 0;                     // its first reduction step
        const float* b_px = nullptr;      // FWD: weight row; DGRAD: column run of the weights
        bool b_in[NB];
        int b_tap = 0, b_o = 0;                     // DGRAD: the weight row's tap and output channel
        int b_h = 0, b_w = 0, dr[NB], ds[NB];       // WGRAD: the pixel row's place; per run its tap shift and
        int b_shift[NB];                            // the float it starts at relative to the pixel's first
        const int step_h = (64 / p.W) % p.H, step_w = 64 % p.W;       // WGRAD: one chunk on, in rows and columns

        // the first chunk of a unit
        auto first_chunk = [&](const Unit& un) {
            kpos = un.chunk0 * 64;
            if (MODE == CMODE_FWD) {
                b_px = p.wt + (size_t)(un.n0 + r) * p.K + 8 * q;
#pragma unroll
                for (int j = 0; j < NB; ++j) b_in[j] = un.n0 + r + 64 * j < p.N;
            } else {
#pragma unroll
                for (int j = 0; j < NB; ++j) b_in[j] = un.n0 + 64 * j + 8 * q < p.N;
                if (MODE == CMODE_DGRAD) {
                    b_px = p.wt + un.n0 + 8 * q;
                    b_tap = (kpos + r) / Cred; b_o = kpos + r - b_tap * Cred;
                } else {
                    const int w = kpos + r - div_rcp(kpos + r, p.rcp_hw, HW) * HW;
                    b_h = div_rcp(w, p.rcp_w, p.W); b_w = w - b_h * p.W;
#pragma unroll
                    for (int j = 0; j < NB; ++j) {
                        const int n = un.n0 + 64 * j + 8 * q, tap = b_in[j] ? n / p.Cin : 0;
                        dr[j] = p.taps == 9 ? tap / 3 - 1 : 0; ds[j] = p.taps == 9 ? tap % 3 - 1 : 0;
                        b_shift[j] = (dr[j] * p.W + ds[j]) * p.Cin + (n - tap * p.Cin);
                    }
                }
            }
            if (!TMA) {
                const int k = kpos + 16 * quarter, m = un.m0 + row;
                a_tap = k / Cred; a_c = k - a_tap * Cred;
                a_px = (MODE == CMODE_FWD ? p.act : p.dy) + (size_t)m * Cred;
                a_px_in = taps_inside<MODE>(p, m);
            }
        };
        auto next_chunk = [&] {
            kpos += 64;
            if (MODE == CMODE_WGRAD) {
                b_w += step_w; b_h += step_h;
                if (b_w >= p.W) { b_w -= p.W; ++b_h; }
                if (b_h >= p.H) b_h -= p.H;
            }
            if (MODE == CMODE_DGRAD)
                for (b_o += 64; b_o >= Cred; b_o -= Cred) ++b_tap;
            if (!TMA)
                for (a_c += 64; a_c >= Cred; a_c -= Cred) ++a_tap;
        };
        auto load_a = [&] {               // (without TMA)
            int tap = a_tap, c = a_c;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                int shift = 0;
                if (p.taps == 9) {
                    const int tr = tap >= 6 ? 2 : (tap >= 3 ? 1 : 0), ts = tap - 3 * tr;
                    shift = (MODE == CMODE_FWD ? (tr - 1) * p.W + ts - 1 : (1 - tr) * p.W + 1 - ts) * Cred;
                }
                load8(ra[i], a_px + (long)shift + c, (a_px_in >> tap) & 1u);
                c += 8;
                if (c == Cred) { c = 0; ++tap; }
            }
        };
        auto load_b = [&](int j) {
            if (MODE == CMODE_FWD) load8(rb[j], b_px + (size_t)(64 * j) * p.K + kpos, b_in[j] && kpos + 8 * q < p.K);
            else if (MODE == CMODE_DGRAD) load8(rb[j], b_px + ((size_t)b_o * p.taps + b_tap) * p.Cin + 64 * j, b_in[j] && b_tap < p.taps);
            else load8(rb[j], p.act + (long)(kpos + r) * p.Cin + b_shift[j],
                       b_in[j] && kpos + r < p.K && (unsigned)(b_h + dr[j]) < (unsigned)p.H && (unsigned)(b_w + ds[j]) < (unsigned)p.W);
        };

        if (!WT) {
            first_chunk(unit_at<BN>(p, blockIdx.x));
            if (!TMA) load_a();
#pragma unroll
            for (int j = 0; j < NB; ++j) load_b(j);
        }
        Ring st, rw;
        int chunk = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < p.units; u += gridDim.x) {      // (to the end also after a wait that gave up: the barriers below want every warp)
            const Unit un = unit_at<BN>(p, u);
            const bool do_bias = MODE == CMODE_WGRAD && un.n0 == 0;
            float bsum = 0.f;
            if (WT) {
                a_in = taps_inside<MODE>(p, un.m0 + row);
                a_tap = un.chunk0 * 64 / Cred; a_c = un.chunk0 * 64 - a_tap * Cred;
            }
            for (int it = 0; it < un.n_iters && ok; ++it, ++chunk) {
                bool w = true;
                if (TMA) w = mbar_wait(&raw_full[rw.i], rw.ph);
                if (TMA) {
                    const uint32_t at = raw_at + (uint32_t)rw.i * RAW;
                    if (MODE == CMODE_WGRAD) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(ra[j / 8].v[j % 8]) : "r"(at + 128u * j + (((uint32_t)(row >> 2) & 7u) ^ (uint32_t)(j & 7)) * 16u));
                    } else {
                        const bool in = (a_in >> a_tap) & 1u;
#pragma unroll
                        for (int i = 0; i < 4 * R::PARTS; ++i) {
                            float* f = &ra[i / 2].v[4 * (i % 2)];
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(f[0]), "=f"(f[1]), "=f"(f[2]), "=f"(f[3])
                                         : "r"(at + ((((uint32_t)(quarter & 1) * 4u + i) ^ (uint32_t)(row & 7)) << 4)));
                        }
                        if (!in)
#pragma unroll
                            for (int j = 0; j < 16 * R::PARTS; ++j) ra[j / 8].v[j % 8] = 0.f;
                        a_c += 64;
                        if (a_c >= Cred) { a_c -= Cred; ++a_tap; }
                    }
                }
                if (chunk >= STAGES) w = w && mbar_wait(&empty[st.i], st.ph ^ 1u);
                ok = __all_sync(0xffffffffu, w ? 1 : 0) != 0;
                if (!ok) break;
                tc_fence_after();
                const bool more = it + 1 < un.n_iters || u + (int)gridDim.x < p.units;
                if (WT) {
                } else if (it + 1 < un.n_iters) next_chunk();
                else if (more) first_chunk(unit_at<BN>(p, u + gridDim.x));
#pragma unroll
                for (int h = 0; h < R::PARTS; ++h) {
                    uint32_t t0[8], t1[8], t2[8];
                    take_terms(ra[2 * h], t0, t1, t2);
                    take_terms(ra[2 * h + 1], t0 + 4, t1 + 4, t2 + 4);
                    if (do_bias)
#pragma unroll
                        for (int j = 0; j < 16; ++j) bsum += ra[j / 8].v[j % 8];
                    __syncwarp();
                    if (TMA && h + 1 == R::PARTS) {
                        if (lane == 0) mbar_arrive(smem_u32(&raw_empty[rw.i]));
                        rw.next(RAWS);
                    }
                    const uint32_t at = a_at + (uint32_t)st.i * A_STAGE + 8u * h;
                    tmem_st8(at, t0);
                    tmem_st8(at + A_TERM, t1);
                    tmem_st8(at + 2 * A_TERM, t2);
                    if (!TMA && more) load_a();
                }
#pragma unroll
                for (int j = 0; j < (WT ? 0 : NB); ++j) {
                    uint32_t t0[4], t1[4], t2[4];
                    take_terms(rb[j], t0, t1, t2);
                    const uint32_t at = b_at + (uint32_t)st.i * C::STAGE + 8192u * j;
                    st_shared16(at, t0);
                    st_shared16(at + C::PLANE, t1);
                    st_shared16(at + 2 * C::PLANE, t2);
                    if (more) load_b(j);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                if (!WT) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&full[st.i]));
                st.next(STAGES);
            }
            if (MODE == CMODE_WGRAD && do_bias) {
                if (quarter > 0) s_bias[(quarter - 1) * 128 + row] = bsum;
                asm volatile("bar.sync 2, 512;" ::: "memory");
                if (quarter == 0 && un.m0 + row < p.M)
                    p.part[(size_t)un.split * p.split_stride + p.bias_off + un.m0 + row] = ((bsum + s_bias[row]) + s_bias[128 + row]) + s_bias[256 + row];
                asm volatile("bar.sync 2, 512;" ::: "memory");
            }
        }
        if (!ok && lane == 0) { *abort_flag = 1; atomicMax(p.status, (uint32_t)DEV_TIMEOUT_TMA); }
    }

    // ---- teardown: TMEM is released on every path ----------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        const uint64_t t0 = globaltimer_ns();          // copies and MMAs that may still be in flight use shared memory
        while (globaltimer_ns() - t0 < 200000ull) { }
        __syncthreads();
    }
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}


template <int MODE, int BN, bool TMA, bool WT>
cudaError_t launch_one(const ContractArgs& a, SplitParams p, cudaStream_t st)
{
    constexpr int SMEM = SplitCfg<BN>::smem(TMA);
    const cudaError_t e = raise_smem_limit<contract_umma_kernel<MODE, BN, TMA, WT>>(SMEM);
    if (e != cudaSuccess) return e;
    Maps<TMA> maps{};
    if constexpr (TMA) {
        if (!(MODE == CMODE_WGRAD ? umma_map_f32_rows(&maps.a, p.dy, p.npix, p.Cout, 64)
                                  : umma_map_f32_rows(&maps.a, MODE == CMODE_FWD ? p.act : p.dy, p.npix, MODE == CMODE_FWD ? p.Cin : p.Cout, 128)))
            return cudaErrorInvalidValue;
        if (WT && !umma_map_terms(&maps.b, a.wterms, p.Cout, (long)p.taps * p.Cin, a.wterms_stride, MODE == CMODE_FWD ? BN : 64)) return cudaErrorInvalidValue;
    }
    p.m_tiles = (p.M + 127) / 128; p.n_tiles = (p.N + BN - 1) / BN;
    const long units = (long)p.m_tiles * p.n_tiles * p.splits;
    if (units >= (1L << 30)) return cudaErrorInvalidValue;
    p.units = (int)units;
    p.rcp_m = rcp_of(p.m_tiles); p.rcp_n = rcp_of(p.n_tiles);
    return pdl_launch(contract_umma_kernel<MODE, BN, TMA, WT>, dim3((unsigned)(units < 148 ? units : 148)), dim3(Roles<WT>::THREADS), (size_t)SMEM, st, maps, p);
}
template <int MODE, int BN>
cudaError_t launch_form(const ContractArgs& a, const SplitParams& p, cudaStream_t st)
{
    if constexpr (MODE == CMODE_WGRAD) return launch_one<MODE, BN, true, false>(a, p, st);
    else return a.wterms != nullptr ? launch_one<MODE, BN, true, true>(a, p, st) : launch_one<MODE, BN, false, false>(a, p, st);
}
template <int MODE>
cudaError_t launch_mode(const ContractArgs& a, const SplitParams& p, cudaStream_t st)
{
    return a.plan.bn == 128 ? launch_form<MODE, 128>(a, p, st) : launch_form<MODE, 64>(a, p, st);
}

// n floats as three planes of bf16 terms, `stride` elements apart
__global__ void __launch_bounds__(256)
split_weights_kernel(const float4* __restrict__ w, uint2* __restrict__ terms, size_t n4, size_t stride4)
{
    pdl_prologue();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        float4 v = __ldg(w + i);
        scale_pair(v.x, v.y);
        scale_pair(v.z, v.w);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint2 t;
            t.x = take_term(v.x, v.y);
            t.y = take_term(v.z, v.w);
            terms[k * stride4 + i] = t;
        }
    }
}

}  // namespace

cudaError_t launch_split_weights(const float* w, __nv_bfloat16* terms, size_t n, size_t stride, cudaStream_t st)
{
    const size_t n4 = n / 4;
    const long blocks = (long)((n4 + 255) / 256);
    SB_LAUNCH((split_weights_kernel), (int)(blocks < 148 * 8 ? blocks : 148 * 8), 256, 0, st, (const float4*)w, (uint2*)terms, n4, stride / 4);
    return cudaGetLastError();
}
bool contract_umma_whole_taps(int mode, int Cin, int Cout) { return (mode == CMODE_DGRAD ? Cout : Cin) % 64 == 0; }
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
    if (a.mode == CMODE_FWD) return launch_mode<CMODE_FWD>(a, p, st);
    return a.mode == CMODE_DGRAD ? launch_mode<CMODE_DGRAD>(a, p, st) : launch_mode<CMODE_WGRAD>(a, p, st);
}

}  // namespace sb
