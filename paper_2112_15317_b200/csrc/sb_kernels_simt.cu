// CUDA-core kernels of the SplitBrain training step for sm_100a.
//
//  * bandwidth-bound steps that every mode uses: 2x2 max-pool forward/backward, softmax
//    cross-entropy, SGD with momentum, column sums (bias gradients) and split reductions;
//  * the input layer's convolution and the narrow FC layers, which no contraction tile fits.
//
// T is the activation dtype (float or __nv_bfloat16); all sums are carried in float.
#include "sb_internal.h"

namespace sb {

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T* p, float v);
template <> __device__ __forceinline__ void stf<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// store 8 consecutive values (pointer 16-byte aligned for bf16, 32-byte for float)
__device__ __forceinline__ void store8(float* p, const float (&v)[8])
{
    ((float4*)p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    ((float4*)p)[1] = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&v)[8])
{
    uint32_t pk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        __nv_bfloat162 t = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        pk[j] = *(uint32_t*)&t;
    }
    *(uint4*)p = make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

static inline int cdiv(long a, long b) { return (int)((a + b - 1) / b); }

// =============================================================================================
// Column sums (bias gradients) and the reduction of split partial sums.
// =============================================================================================
// bf16, N a multiple of 8: a thread owns 8 adjacent columns (one 16-byte load per row), 8 row lanes per block take rows
// r0 + lane_row, + 8, ... with four independent loads in flight and are combined in lane order (deterministic).
__global__ void __launch_bounds__(256)
colsum_vec_kernel(const uint4* __restrict__ in, float* __restrict__ part, int M, int N, int splits)
{
    pdl_prologue();
    __shared__ float s[8][32][9];
    const int nv = N / 8;
    const int vc = blockIdx.x * 32 + threadIdx.x % 32;
    const int lane_row = threadIdx.x / 32;
    const int sp = blockIdx.y;
    const long rows = (M + splits - 1) / splits, r0 = (long)sp * rows;
    const long r1 = r0 + rows < M ? r0 + rows : M;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (vc < nv) {
        long r = r0 + lane_row;
        for (; r + 24 < r1; r += 32) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldg(in + (r + 8 * u) * nv + vc);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const __nv_bfloat16* h = (const __nv_bfloat16*)&v[u];
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[j] += __bfloat162float(h[j]);
            }
        }
        for (; r < r1; r += 8) {
            const uint4 v = __ldg(in + r * nv + vc);
            const __nv_bfloat16* h = (const __nv_bfloat16*)&v;
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] += __bfloat162float(h[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) s[lane_row][threadIdx.x % 32][j] = acc[j];
    __syncthreads();
    if (lane_row == 0 && vc < nv) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float t = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) t += s[i][threadIdx.x][j];
            part[(size_t)sp * N + vc * 8 + j] = t;
        }
    }
}
cudaError_t launch_colsum(const void* in, float* part, int M, int N, int splits, cudaStream_t st)
{
    if (N % 8 != 0 || (((uintptr_t)in) & 15) != 0) return cudaErrorInvalidValue;
    SB_LAUNCH((colsum_vec_kernel), dim3(cdiv(N / 8, 32), splits), 256, 0, st, (const uint4*)in, part, M, N, splits);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256)
reduce_partials_kernel(const float* __restrict__ part, size_t stride, float* __restrict__ out, size_t n, int splits, Gap gap)
{
    pdl_prologue();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float t = 0.f;
        for (int s = 0; s < splits; ++s) t += part[(size_t)s * stride + i];
        out[gap.over(i)] = t;
    }
}
__global__ void __launch_bounds__(256)
reduce_partials4_kernel(const float4* __restrict__ part, size_t stride4, float4* __restrict__ out, size_t n4, int splits, Gap gap4)
{
    pdl_prologue();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        // loads go out in batches of 8 (independent, all in flight together); the additions keep split order
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s0 = 0; s0 < splits; s0 += 8) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = (s0 + u < splits) ? __ldg(part + (size_t)(s0 + u) * stride4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) { t.x += v[u].x; t.y += v[u].y; t.z += v[u].z; t.w += v[u].w; }
        }
        out[gap4.over(i)] = t;
    }
}
// Many splits, few elements: 32 elements per block, LANES lanes share the splits of each element (lane l takes
// splits l, l + LANES, ... in order, four loads in flight) and are combined in lane order: a fixed order, so the
// result is deterministic.  LANES = 8, or 32 from 128 splits on (the input layer's per-block partial sums).
template <int LANES>
__device__ __forceinline__ float many_lane_sum(const float* __restrict__ part, size_t stride, size_t i, int lane, int splits)
{
    float t = 0.f;
    int sp = lane;
    for (; sp + 3 * LANES < splits; sp += 4 * LANES) {
        const float a = part[(size_t)sp * stride + i], b = part[(size_t)(sp + LANES) * stride + i];
        const float c = part[(size_t)(sp + 2 * LANES) * stride + i], d = part[(size_t)(sp + 3 * LANES) * stride + i];
        t += a; t += b; t += c; t += d;
    }
    for (; sp < splits; sp += LANES) t += part[(size_t)sp * stride + i];
    return t;
}
template <int LANES>
__global__ void __launch_bounds__(32 * LANES)
reduce_partials_many_kernel(const float* __restrict__ part, size_t stride, float* __restrict__ out, size_t n, int splits, Gap gap)
{
    pdl_prologue();
    __shared__ float s[LANES][33];
    const int e = threadIdx.x % 32, lane = threadIdx.x / 32;
    const size_t i = blockIdx.x * 32ull + e;
    s[lane][e] = i < n ? many_lane_sum<LANES>(part, stride, i, lane, splits) : 0.f;
    __syncthreads();
    if (lane == 0 && i < n) {
        float r = 0.f;
#pragma unroll
        for (int j = 0; j < LANES; ++j) r += s[j][e];
        out[gap.over(i)] = r;
    }
}
cudaError_t launch_reduce_partials(const float* part, size_t stride, float* out, size_t n, int splits, cudaStream_t st, Gap gap)
{
    if (splits >= 128 && n <= (1u << 20)) {
        SB_LAUNCH((reduce_partials_many_kernel<32>), cdiv((long)n, 32), 1024, 0, st, part, stride, out, n, splits, gap);
    } else if (splits >= 32 && n <= (1u << 20)) {
        SB_LAUNCH((reduce_partials_many_kernel<8>), cdiv((long)n, 32), 256, 0, st, part, stride, out, n, splits, gap);
    } else if (n % 4 == 0 && stride % 4 == 0 && gap.by4() && (((uintptr_t)part | (uintptr_t)out) & 15) == 0) {
        int blocks = cdiv((long)(n / 4), 256);
        if (blocks > 148 * 8) blocks = 148 * 8;
        SB_LAUNCH((reduce_partials4_kernel), blocks, 256, 0, st, (const float4*)part, stride / 4, (float4*)out, n / 4, splits, Gap{gap.at / 4, gap.by / 4});
    } else {
        int blocks = cdiv((long)n, 256);
        if (blocks > 148 * 8) blocks = 148 * 8;
        SB_LAUNCH((reduce_partials_kernel), blocks, 256, 0, st, part, stride, out, n, splits, gap);
    }
    return cudaGetLastError();
}

// =============================================================================================
// Split-reduction epilogue of the tensor-core GEMMs: out = epi(sum_s part[s]) with the splits added in
// order; epi = bias + ReLU (-> bf16 or float) or the ReLU mask (-> bf16).  Four columns per thread.
// =============================================================================================
template <typename T, int EPI>
__global__ void __launch_bounds__(256)
splitk_epilogue_kernel(const float* __restrict__ part, size_t split_stride, int splits, size_t n4, int N,
                       const float* __restrict__ bias, int relu, const T* __restrict__ ref,
                       void* __restrict__ out, int out_f32)
{
    pdl_prologue();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const size_t e = i * 4;
        // loads go out in batches of 8 (independent, all in flight together); the additions keep split order
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s0 = 0; s0 < splits; s0 += 8) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = (s0 + u < splits) ? __ldg((const float4*)(part + (size_t)(s0 + u) * split_stride + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) { t.x += v[u].x; t.y += v[u].y; t.z += v[u].z; t.w += v[u].w; }
        }
        if (EPI == EPI_BIAS_ACT) {
            const float4 b = *(const float4*)(bias + (e % (size_t)N));
            t.x += b.x; t.y += b.y; t.z += b.z; t.w += b.w;
            if (relu) {
                if (!(t.x > 0.f)) t.x = 0.f;
                if (!(t.y > 0.f)) t.y = 0.f;
                if (!(t.z > 0.f)) t.z = 0.f;
                if (!(t.w > 0.f)) t.w = 0.f;
            }
        } else if (ref != nullptr) {
            __align__(16) T r[4];
            if (sizeof(T) == 2) *(uint2*)r = *(const uint2*)(ref + e);
            else *(float4*)r = *(const float4*)(ref + e);
            if (!(ldf(r) > 0.f)) t.x = 0.f;
            if (!(ldf(r + 1) > 0.f)) t.y = 0.f;
            if (!(ldf(r + 2) > 0.f)) t.z = 0.f;
            if (!(ldf(r + 3) > 0.f)) t.w = 0.f;
        }
        if (sizeof(T) == 4 || out_f32) {
            *(float4*)((float*)out + e) = t;
        } else {
            __nv_bfloat162 lo = __floats2bfloat162_rn(t.x, t.y), hi = __floats2bfloat162_rn(t.z, t.w);
            uint2 pk;
            pk.x = *(uint32_t*)&lo;
            pk.y = *(uint32_t*)&hi;
            *(uint2*)((__nv_bfloat16*)out + e) = pk;
        }
    }
}
// The same with the 2x2 max-pool that follows (EPI_BIAS_ACT: a thread takes the four pixels of a window; rules of maxpool_fwd_kernel) or the
// pool layer below (EPI_MASK: the gradient goes on to its window; rules of maxpool_bwd_kernel).  H, W, C: the pool layer's input.  Saves
// a launch and its 2.5 - 3 us on the chain (512 channels at 2x2, batch 128).
template <typename T>
__device__ __forceinline__ void round_store4(T* p, float4& t)
{
    if (sizeof(T) == 4) {
        *(float4*)p = t;
    } else {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(t.x, t.y), hi = __floats2bfloat162_rn(t.z, t.w);
        uint2 pk;
        pk.x = *(const uint32_t*)&lo;
        pk.y = *(const uint32_t*)&hi;
        *(uint2*)p = pk;
        t = make_float4(__low2float(lo), __high2float(lo), __low2float(hi), __high2float(hi));
    }
}
template <typename T, int EPI>
__global__ void __launch_bounds__(256)
splitk_pool_kernel(const float* __restrict__ part, size_t split_stride, int splits, size_t n4, const float* __restrict__ bias, int relu,
                   T* __restrict__ out, int H, int W, int C, T* __restrict__ p, uint8_t* __restrict__ idx, const T* __restrict__ mask, T* __restrict__ dx)
{
    pdl_prologue();
    const int Ho = H / 2, Wo = W / 2;
    constexpr int PIX = EPI == EPI_BIAS_ACT ? 4 : 1, SB = 8 / PIX;       // pixels summed by a thread; splits per batch of eight loads
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const size_t e = i * 4, c = e % (size_t)C, q = e / (size_t)C, wo = q % (size_t)Wo, r = q / (size_t)Wo;      // r = n * Ho + ho
        const size_t at0 = ((2 * r) * (size_t)W + 2 * wo) * (size_t)C + c;       // the window's first pixel ((n * H + 2 ho) = 2 r: H is even)
        const size_t at[4] = {at0, at0 + C, at0 + (size_t)W * C, at0 + (size_t)W * C + C};
        float4 t[PIX];
#pragma unroll
        for (int j = 0; j < PIX; ++j) t[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s0 = 0; s0 < splits; s0 += SB) {
            float4 v[SB][PIX];
#pragma unroll
            for (int u = 0; u < SB; ++u)
#pragma unroll
                for (int j = 0; j < PIX; ++j)
                    v[u][j] = s0 + u < splits ? __ldg((const float4*)(part + (size_t)(s0 + u) * split_stride + (PIX == 4 ? at[j] : e))) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < SB; ++u)
#pragma unroll
                for (int j = 0; j < PIX; ++j) { t[j].x += v[u][j].x; t[j].y += v[u][j].y; t[j].z += v[u][j].z; t[j].w += v[u][j].w; }
        }
        if (EPI == EPI_BIAS_ACT) {
            const float4 b = *(const float4*)(bias + c);
            float best[4];
            uint32_t bi = 0u;
#pragma unroll
            for (int j = 0; j < PIX; ++j) {
                t[j].x += b.x; t[j].y += b.y; t[j].z += b.z; t[j].w += b.w;
                float f[4] = {t[j].x, t[j].y, t[j].z, t[j].w};
                if (relu)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (!(f[k] > 0.f)) f[k] = 0.f;
                float4 rounded = make_float4(f[0], f[1], f[2], f[3]);
                round_store4<T>(out + at[j], rounded);
                const float g[4] = {rounded.x, rounded.y, rounded.z, rounded.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (j == 0 || g[k] > best[k]) { best[k] = g[k]; bi = (bi & ~(0xffu << (8 * k))) | ((uint32_t)j << (8 * k)); }
            }
            float4 m = make_float4(best[0], best[1], best[2], best[3]);
            round_store4<T>(p + e, m);
            *(uint32_t*)(idx + e) = bi;
        } else {
            float4 g = t[0];
            round_store4<T>(out + e, g);
            float f[4] = {g.x, g.y, g.z, g.w};
            const uint32_t bi = *(const uint32_t*)(idx + e);
            if (mask != nullptr) {
                __align__(16) T m[4];
                if (sizeof(T) == 2) *(uint2*)m = *(const uint2*)(mask + e);
                else *(float4*)m = *(const float4*)(mask + e);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (!(ldf(m + k) > 0.f)) f[k] = 0.f;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float4 o;
                o.x = (bi & 0xffu) == (uint32_t)j ? f[0] : 0.f;
                o.y = ((bi >> 8) & 0xffu) == (uint32_t)j ? f[1] : 0.f;
                o.z = ((bi >> 16) & 0xffu) == (uint32_t)j ? f[2] : 0.f;
                o.w = (bi >> 24) == (uint32_t)j ? f[3] : 0.f;
                round_store4<T>(dx + at[j], o);
            }
        }
    }
}
// widths that are not multiples of four
template <typename T, int EPI>
__global__ void __launch_bounds__(256)
splitk_epilogue1_kernel(const float* __restrict__ part, size_t split_stride, int splits, size_t n, int N,
                        const float* __restrict__ bias, int relu, const T* __restrict__ ref, void* __restrict__ out, int out_f32)
{
    pdl_prologue();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        float t = 0.f;
        for (int s = 0; s < splits; ++s) t += part[(size_t)s * split_stride + e];
        if (EPI == EPI_BIAS_ACT) {
            t += bias[e % (size_t)N];
            if (relu && !(t > 0.f)) t = 0.f;
        } else if (ref != nullptr) {
            if (!(ldf(ref + e) > 0.f)) t = 0.f;
        }
        if (out_f32) ((float*)out)[e] = t;
        else stf((T*)out + e, t);
    }
}
template <typename T, int EPI>
static cudaError_t launch_splitk_t(const SplitKEpiArgs& a, cudaStream_t st)
{
    const size_t total = (size_t)a.rows * a.N;
    const bool vec = a.N % 4 == 0;
    if (SplitPool* o = split_pool()) {
        // (logits and masked results have no pool layer beside them)
        const bool fwd = o->dx == nullptr;
        if (vec && o->C % 4 == 0 && (sizeof(T) == 4 || !a.out_f32) && fwd == (EPI == EPI_BIAS_ACT) && (fwd || a.ref == nullptr)) {
            const size_t n4 = total / (fwd ? 16 : 4);
            const long blocks = (long)((n4 + 255) / 256);
            SB_LAUNCH((splitk_pool_kernel<T, EPI>), (int)(blocks < 148 * 8 ? blocks : 148 * 8), 256, 0, st, a.part, a.split_stride, a.splits, n4, a.bias, a.relu,
                      (T*)a.out, o->H, o->W, o->C, (T*)o->p, o->idx, (const T*)o->mask, (T*)o->dx);
            o->done = true;
            return cudaGetLastError();
        }
    }
    int blocks = cdiv((long)(vec ? total / 4 : total), 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    if (vec) SB_LAUNCH((splitk_epilogue_kernel<T, EPI>), blocks, 256, 0, st, a.part, a.split_stride, a.splits, total / 4, a.N, a.bias, a.relu, (const T*)a.ref, a.out, a.out_f32);
    else SB_LAUNCH((splitk_epilogue1_kernel<T, EPI>), blocks, 256, 0, st, a.part, a.split_stride, a.splits, total, a.N, a.bias, a.relu, (const T*)a.ref, a.out, a.out_f32);
    return cudaGetLastError();
}
cudaError_t launch_splitk_epilogue(const SplitKEpiArgs& a, bool bf16, cudaStream_t st)
{
    if (a.epi == EPI_BIAS_ACT) return bf16 ? launch_splitk_t<__nv_bfloat16, EPI_BIAS_ACT>(a, st) : launch_splitk_t<float, EPI_BIAS_ACT>(a, st);
    return bf16 ? launch_splitk_t<__nv_bfloat16, EPI_MASK>(a, st) : launch_splitk_t<float, EPI_MASK>(a, st);
}

// =============================================================================================
// 2x2 max-pool, stride 2.  One thread per pooled pixel and VEC channels (16-byte accesses when the
// channel count allows).  Ties go to the first maximum in scan order (0,0),(0,1),(1,0),(1,1).
// =============================================================================================
template <typename T, int VEC> struct VecT;
template <> struct VecT<float, 4> { typedef float4 type; };
template <> struct VecT<float, 1> { typedef float type; };
template <> struct VecT<__nv_bfloat16, 8> { typedef uint4 type; };
template <> struct VecT<__nv_bfloat16, 1> { typedef __nv_bfloat16 type; };
template <int VEC> struct VecU8;
template <> struct VecU8<8> { typedef uint2 type; };
template <> struct VecU8<4> { typedef uint32_t type; };
template <> struct VecU8<1> { typedef uint8_t type; };

template <typename T, int VEC>
__global__ void __launch_bounds__(256)
maxpool_fwd_kernel(const T* __restrict__ x, T* __restrict__ p, uint8_t* __restrict__ idx, long total, int H, int W, int C)
{
    pdl_prologue();
    typedef typename VecT<T, VEC>::type V;
    typedef typename VecU8<VEC>::type VI;
    const int Ho = H / 2, Wo = W / 2, Cv = C / VEC;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
        int cv = (int)(e % Cv);
        long q = e / Cv;
        int wo = (int)(q % Wo);
        q /= Wo;
        int ho = (int)(q % Ho);
        long n = q / Ho;
        const T* base = x + (((size_t)n * H + 2 * ho) * W + 2 * wo) * C + (size_t)cv * VEC;
        V v[4];
        v[0] = *(const V*)(base);
        v[1] = *(const V*)(base + C);
        v[2] = *(const V*)(base + (size_t)W * C);
        v[3] = *(const V*)(base + (size_t)W * C + C);
        V outv;
        VI outi;
        T* ov = (T*)&outv;
        uint8_t* oi = (uint8_t*)&outi;
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            T bestv = ((const T*)&v[0])[k];
            float best = ldf(&bestv);
            int bi = 0;
#pragma unroll
            for (int j = 1; j < 4; ++j) {
                T cand = ((const T*)&v[j])[k];
                float f = ldf(&cand);
                if (f > best) { best = f; bi = j; bestv = cand; }
            }
            ov[k] = bestv;
            oi[k] = (uint8_t)bi;
        }
        size_t o = (size_t)e * VEC;
        *(V*)(p + o) = outv;
        *(VI*)(idx + o) = outi;
    }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(256)
maxpool_bwd_kernel(const T* __restrict__ dp, const uint8_t* __restrict__ idx, const T* __restrict__ p,
                   T* __restrict__ dx, long total, int H, int W, int C)
{
    pdl_prologue();
    typedef typename VecT<T, VEC>::type V;
    typedef typename VecU8<VEC>::type VI;
    const int Ho = H / 2, Wo = W / 2, Cv = C / VEC;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
        int cv = (int)(e % Cv);
        long q = e / Cv;
        int wo = (int)(q % Wo);
        q /= Wo;
        int ho = (int)(q % Ho);
        long n = q / Ho;
        size_t o = (size_t)e * VEC;
        V g = *(const V*)(dp + o);
        VI iv = *(const VI*)(idx + o);
        const uint8_t* ii = (const uint8_t*)&iv;
        T* gp = (T*)&g;
        if (p != nullptr) {
            V pv = *(const V*)(p + o);
#pragma unroll
            for (int k = 0; k < VEC; ++k)
                if (!(ldf((const T*)&pv + k) > 0.f)) stf(gp + k, 0.f);
        }
        T* base = dx + (((size_t)n * H + 2 * ho) * W + 2 * wo) * C + (size_t)cv * VEC;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            V ov;
            T* op = (T*)&ov;
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if (ii[k] == j) op[k] = gp[k]; else stf(op + k, 0.f);
            }
            *(V*)(base + (size_t)(j >> 1) * W * C + (size_t)(j & 1) * C) = ov;
        }
    }
}

static int ew_blocks(long total)
{
    long b = (total + 255) / 256;
    long cap = 148L * 16;
    return (int)(b < cap ? (b < 1 ? 1 : b) : cap);
}

cudaError_t launch_pool_fwd(const PoolArgs& a, bool bf16, cudaStream_t st)
{
    long pooled = (long)a.B * (a.H / 2) * (a.W / 2) * a.C;
    if (bf16) {
        if (a.C % 8 == 0) SB_LAUNCH((maxpool_fwd_kernel<__nv_bfloat16, 8>), ew_blocks(pooled / 8), 256, 0, st, (const __nv_bfloat16*)a.x, (__nv_bfloat16*)a.p, a.idx, pooled / 8, a.H, a.W, a.C);
        else SB_LAUNCH((maxpool_fwd_kernel<__nv_bfloat16, 1>), ew_blocks(pooled), 256, 0, st, (const __nv_bfloat16*)a.x, (__nv_bfloat16*)a.p, a.idx, pooled, a.H, a.W, a.C);
    } else {
        if (a.C % 4 == 0) SB_LAUNCH((maxpool_fwd_kernel<float, 4>), ew_blocks(pooled / 4), 256, 0, st, (const float*)a.x, (float*)a.p, a.idx, pooled / 4, a.H, a.W, a.C);
        else SB_LAUNCH((maxpool_fwd_kernel<float, 1>), ew_blocks(pooled), 256, 0, st, (const float*)a.x, (float*)a.p, a.idx, pooled, a.H, a.W, a.C);
    }
    return cudaGetLastError();
}
cudaError_t launch_pool_bwd(const PoolBwdArgs& a, bool bf16, cudaStream_t st)
{
    long pooled = (long)a.B * (a.H / 2) * (a.W / 2) * a.C;
    if (bf16) {
        if (a.C % 8 == 0) SB_LAUNCH((maxpool_bwd_kernel<__nv_bfloat16, 8>), ew_blocks(pooled / 8), 256, 0, st, (const __nv_bfloat16*)a.dp, a.idx, (const __nv_bfloat16*)a.p, (__nv_bfloat16*)a.dx, pooled / 8, a.H, a.W, a.C);
        else SB_LAUNCH((maxpool_bwd_kernel<__nv_bfloat16, 1>), ew_blocks(pooled), 256, 0, st, (const __nv_bfloat16*)a.dp, a.idx, (const __nv_bfloat16*)a.p, (__nv_bfloat16*)a.dx, pooled, a.H, a.W, a.C);
    } else {
        if (a.C % 4 == 0) SB_LAUNCH((maxpool_bwd_kernel<float, 4>), ew_blocks(pooled / 4), 256, 0, st, (const float*)a.dp, a.idx, (const float*)a.p, (float*)a.dx, pooled / 4, a.H, a.W, a.C);
        else SB_LAUNCH((maxpool_bwd_kernel<float, 1>), ew_blocks(pooled), 256, 0, st, (const float*)a.dp, a.idx, (const float*)a.p, (float*)a.dx, pooled, a.H, a.W, a.C);
    }
    return cudaGetLastError();
}

// =============================================================================================
// Softmax cross-entropy: one warp per row (shuffle max / sum), dZ = (softmax - onehot)/B.
// The last block to finish adds the row losses in row order, so the mean is deterministic.
// =============================================================================================
// mean of the row losses by one warp, in a fixed order: chunks of 32 rows, tree inside
__device__ __forceinline__ float mean_loss(const float* row_loss, int rows)
{
    const int lane = threadIdx.x % 32;
    float t = 0.f;
    for (int i0 = 0; i0 < rows; i0 += 32) {
        float v = (i0 + lane < rows) ? ((volatile const float*)row_loss)[i0 + lane] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        t += v;
    }
    return t / (float)rows;
}
__global__ void __launch_bounds__(32)
loss_mean_kernel(const float* __restrict__ row_loss, int rows, float* __restrict__ loss)
{
    pdl_prologue();
    const float t = mean_loss(row_loss, rows);
    if (threadIdx.x == 0) *loss = t;
}
cudaError_t launch_loss_mean(const XentArgs& a, cudaStream_t st)
{
    SB_LAUNCH((loss_mean_kernel), 1, 32, 0, st, a.loss_rows > 0 ? a.loss_base : a.row_loss, a.loss_rows > 0 ? a.loss_rows : a.B, a.loss);
    return cudaGetLastError();
}
template <typename T>
__global__ void __launch_bounds__(256)
softmax_xent_kernel(const float* __restrict__ logits, PtrTab labels, int b_per_rep, float* __restrict__ row_loss,
                    float* __restrict__ loss, T* __restrict__ dZ, unsigned int* __restrict__ counter, int B, int C,
                    int scale_B, const float* __restrict__ loss_base, int loss_rows)
{
    pdl_prologue();
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int g = blockIdx.x * 8 + warp;
    if (g < B) {
        const float* z = logits + (size_t)g * C;
        const int y = ((const int32_t*)labels.p[g / b_per_rep])[g % b_per_rep];
        float m = -INFINITY;
        for (int c = lane; c < C; c += 32) m = fmaxf(m, z[c]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = 0.f;
        for (int c = lane; c < C; c += 32) s += expf(z[c] - m);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float lse = m + logf(s);
        const float invB = 1.0f / (float)scale_B;
        for (int c = lane; c < C; c += 32) {
            float pr = expf(z[c] - lse);
            stf(dZ + (size_t)g * C + c, (pr - (c == y ? 1.f : 0.f)) * invB);
        }
        if (lane == 0) row_loss[g] = (y >= 0 && y < C) ? lse - z[y] : 0.f;
    }
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    __syncthreads();
    if (last && warp == 0) {
        __threadfence();
        const float t = mean_loss(loss_base, loss_rows);
        if (lane == 0) { *loss = t; *counter = 0u; }
    }
}
cudaError_t launch_softmax_xent(const XentArgs& a, bool bf16, cudaStream_t st)
{
    int blocks = cdiv(a.B, 8);
    const int scale_B = a.scale_B > 0 ? a.scale_B : a.B;
    const float* loss_base = a.loss_rows > 0 ? a.loss_base : a.row_loss;
    const int loss_rows = a.loss_rows > 0 ? a.loss_rows : a.B;
    if (bf16) SB_LAUNCH((softmax_xent_kernel<__nv_bfloat16>), blocks, 256, 0, st, a.logits, a.labels, a.b_per_rep, a.row_loss, a.loss, (__nv_bfloat16*)a.dZ, a.counter, a.B, a.C, scale_B, loss_base, loss_rows);
    else SB_LAUNCH((softmax_xent_kernel<float>), blocks, 256, 0, st, a.logits, a.labels, a.b_per_rep, a.row_loss, a.loss, (float*)a.dZ, a.counter, a.B, a.C, scale_B, loss_base, loss_rows);
    return cudaGetLastError();
}

// Modulo layer as a row permutation (see ModuloCopyArgs): one block column per row, 16-byte chunks.
__global__ void __launch_bounds__(256)
modulo_copy_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, size_t row_vecs, int R, int b, int K, int scatter,
                   PtrTab labels, int has_labels, int32_t* __restrict__ labels_out)
{
    pdl_prologue();
    const int bk = b / K;
    const int nat = blockIdx.y;                                  // natural row index r*b + k*bk + i
    const int r = nat / b, k = (nat % b) / bk, i = nat % bk;
    const int sub = k * (R * bk) + r * bk + i;                   // sub-iteration order
    const uint4* s = src + (size_t)(scatter ? sub : nat) * row_vecs;
    uint4* d = dst + (size_t)(scatter ? nat : sub) * row_vecs;
    for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < row_vecs; v += (size_t)gridDim.x * blockDim.x) d[v] = s[v];
    if (has_labels && !scatter && blockIdx.x == 0 && threadIdx.x == 0) labels_out[sub] = ((const int32_t*)labels.p[r])[nat % b];
}
cudaError_t launch_modulo_copy(const ModuloCopyArgs& a, cudaStream_t st)
{
    if (a.row_bytes % 16 != 0 || a.K < 1 || a.b % a.K != 0) return cudaErrorInvalidValue;
    const size_t row_vecs = a.row_bytes / 16;
    int bx = (int)((row_vecs + 255) / 256);
    if (bx > 32) bx = 32;
    if (bx < 1) bx = 1;
    PtrTab tab{};
    if (a.labels) tab = *a.labels;
    SB_LAUNCH((modulo_copy_kernel), dim3(bx, a.R * a.b), 256, 0, st, (const uint4*)a.src, (uint4*)a.dst, row_vecs, a.R, a.b, a.K, a.scatter, tab,
              a.labels ? 1 : 0, a.labels_out);
    return cudaGetLastError();
}

// =============================================================================================
// Dropout [Listing 1, case DROPOUT | RELU]: a one-to-one layer on the (partitioned) width of the FC + ReLU layer below.
// Element (global batch row g, logical column c) is kept iff the first output word of Philox-4x32-10 (Salmon et al.,
// SC'11) at counter (e mod 2^32, e div 2^32, layer, iteration), e = g*width + c, under the 64-bit seed as key, is at
// least p * 2^32; kept elements are multiplied by 1/(1 - p).  state = {seed lo, seed hi, iteration, unused}.
// =============================================================================================
__device__ __forceinline__ uint32_t philox4x32_10_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(M0, c0), lo0 = M0 * c0;
        const uint32_t hi1 = __umulhi(M1, c2), lo1 = M1 * c2;
        c0 = hi1 ^ c1 ^ k0; c1 = lo1; c2 = hi0 ^ c3 ^ k1; c3 = lo0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return c0;
}
// sub_bk > 0: the rows are those of sub-iteration sub_k of the modulo layer's schedule (replica r's sub_k-th slice of sub_bk rows,
// replica-major): buffer row j is batch row (j / sub_bk) * sub_b + sub_k * sub_bk + j % sub_bk, and the mask follows the batch row
template <typename T>
__global__ void __launch_bounds__(256)
dropout_fwd_kernel(const T* __restrict__ x, T* __restrict__ y, size_t n, int width, const uint32_t* __restrict__ state, uint32_t layer,
                   uint32_t threshold, float scale, int sub_bk, int sub_b, int sub_k)
{
    pdl_prologue();
    const uint32_t k0 = state[0], k1 = state[1], it = state[2];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        size_t e = i;
        if (sub_bk > 0) {
            const size_t j = i / (size_t)width, c = i - j * (size_t)width;
            const size_t g = (j / (size_t)sub_bk) * (size_t)sub_b + (size_t)sub_k * (size_t)sub_bk + j % (size_t)sub_bk;
            e = g * (size_t)width + c;
        }
        const uint32_t u = philox4x32_10_word0((uint32_t)e, (uint32_t)(e >> 32), layer, it, k0, k1);
        stf(y + i, u >= threshold ? ldf(x + i) * scale : 0.0f);
    }
}
// y = x * scale (the backward pass of the kept elements; the dropped ones arrive as zeros)
template <typename T>
__global__ void __launch_bounds__(256)
scale_kernel(const T* __restrict__ x, T* __restrict__ y, size_t n, float scale)
{
    pdl_prologue();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) stf(y + e, ldf(x + e) * scale);
}
// mode 0: state = {v0, v1, v2, 0};  mode 1: ++iteration
__global__ void dropout_state_kernel(uint32_t* state, int mode, uint32_t v0, uint32_t v1, uint32_t v2)
{
    pdl_prologue();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if (mode == 0) { state[0] = v0; state[1] = v1; state[2] = v2; state[3] = 0u; }
    else state[2] += 1u;
}
cudaError_t launch_dropout_fwd(const void* x, void* y, size_t rows, int width, const uint32_t* state, int layer, int units, bool bf16, cudaStream_t st,
                               int sub_bk, int sub_b, int sub_k)
{
    const size_t n = rows * (size_t)width;
    const uint32_t threshold = (uint32_t)units << 16;
    const float scale = 65536.0f / (float)(65536 - units);
    if (bf16) SB_LAUNCH((dropout_fwd_kernel<__nv_bfloat16>), ew_blocks((long)n), 256, 0, st, (const __nv_bfloat16*)x, (__nv_bfloat16*)y, n, width, state, (uint32_t)layer, threshold, scale, sub_bk, sub_b, sub_k);
    else SB_LAUNCH((dropout_fwd_kernel<float>), ew_blocks((long)n), 256, 0, st, (const float*)x, (float*)y, n, width, state, (uint32_t)layer, threshold, scale, sub_bk, sub_b, sub_k);
    return cudaGetLastError();
}
cudaError_t launch_dropout_bwd(const void* dy, void* dx, size_t n, int units, bool bf16, cudaStream_t st)
{
    const float scale = 65536.0f / (float)(65536 - units);
    if (bf16) SB_LAUNCH((scale_kernel<__nv_bfloat16>), ew_blocks((long)n), 256, 0, st, (const __nv_bfloat16*)dy, (__nv_bfloat16*)dx, n, scale);
    else SB_LAUNCH((scale_kernel<float>), ew_blocks((long)n), 256, 0, st, (const float*)dy, (float*)dx, n, scale);
    return cudaGetLastError();
}
cudaError_t launch_dropout_state(uint32_t* state, int mode, uint64_t seed, uint32_t iteration, cudaStream_t st)
{
    SB_LAUNCH((dropout_state_kernel), 1, 32, 0, st, state, mode, (uint32_t)seed, (uint32_t)(seed >> 32), iteration);
    return cudaGetLastError();
}

// =============================================================================================
// SGD with momentum over the whole (padded, 16-byte aligned) parameter arena:
// v <- mu*v + g ; w <- w - lr*v ; optional bf16 copy of the new w.
// =============================================================================================
template <bool SHADOW>
__device__ __forceinline__ void sgd_apply(float4& ww, float4& vv, const float4& gg, float lr, float mu, uint2* shadow_at)
{
    vv.x = fmaf(mu, vv.x, gg.x); vv.y = fmaf(mu, vv.y, gg.y); vv.z = fmaf(mu, vv.z, gg.z); vv.w = fmaf(mu, vv.w, gg.w);
    ww.x = fmaf(-lr, vv.x, ww.x); ww.y = fmaf(-lr, vv.y, ww.y); ww.z = fmaf(-lr, vv.z, ww.z); ww.w = fmaf(-lr, vv.w, ww.w);
    if (SHADOW) {
        __nv_bfloat162 lo = __floats2bfloat162_rn(ww.x, ww.y), hi = __floats2bfloat162_rn(ww.z, ww.w);
        uint2 pk;
        pk.x = *(uint32_t*)&lo;
        pk.y = *(uint32_t*)&hi;
        *shadow_at = pk;
    }
}
// Grid-stride blocks with four independent 16-byte triples in flight per thread.  (Measured: the update does not
// hide behind the backward pass's tensor-core kernels whatever the grid size -- 16, 8, 4, 2 or 1 blocks per SM
// all give the same step time, and confined to 32 or 64 blocks the update overlaps but is itself too slow;
// streaming (evict-first) loads and stores make no difference either.  SB_SGD_BLOCKS_PER_SM changes the grid.)
template <bool SHADOW>
__global__ void __launch_bounds__(256, 4)
sgd_kernel(float4* __restrict__ w, float4* __restrict__ v, const float4* __restrict__ g,
           uint2* __restrict__ shadow, size_t n4, Hyper hy)
{
    pdl_prologue();
    const float lr = hy.rate(), mu = hy.decay();
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n4; i += 4 * stride) {
        float4 ww[4], vv[4], gg[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { ww[u] = __ldcs(w + i + u * stride); vv[u] = __ldcs(v + i + u * stride); gg[u] = __ldcs(g + i + u * stride); }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            sgd_apply<SHADOW>(ww[u], vv[u], gg[u], lr, mu, SHADOW ? shadow + i + u * stride : nullptr);
            __stcs(v + i + u * stride, vv[u]);
            __stcs(w + i + u * stride, ww[u]);
        }
    }
    for (; i < n4; i += stride) {
        float4 ww = __ldcs(w + i), vv = __ldcs(v + i), gg = __ldcs(g + i);
        sgd_apply<SHADOW>(ww, vv, gg, lr, mu, SHADOW ? shadow + i : nullptr);
        __stcs(v + i, vv);
        __stcs(w + i, ww);
    }
}
// Ordered split reduce and update in one pass: g = sum_s part[s] (the same kernels' split order as
// launch_reduce_partials, so the gradient has the same bits), then the SGD step on w, v (and the bf16 copy) without
// the gradient ever being written to or read back from the gradient arena.
template <bool SHADOW>
__global__ void __launch_bounds__(256)
reduce_sgd4_kernel(const float4* __restrict__ part, size_t stride4, int splits, float4* __restrict__ w, float4* __restrict__ v,
                   uint2* __restrict__ shadow, size_t n4, Hyper hy, Gap gap4)
{
    pdl_prologue();
    const float lr = hy.rate(), mu = hy.decay();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const size_t o = gap4.over(i);
        float4 ww = w[o], vv = v[o];
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s0 = 0; s0 < splits; s0 += 8) {
            float4 pv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                pv[u] = (s0 + u < splits) ? __ldg(part + (size_t)(s0 + u) * stride4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) { t.x += pv[u].x; t.y += pv[u].y; t.z += pv[u].z; t.w += pv[u].w; }
        }
        sgd_apply<SHADOW>(ww, vv, t, lr, mu, SHADOW ? shadow + o : nullptr);
        v[o] = vv;
        w[o] = ww;
    }
}
__device__ __forceinline__ void sgd_apply_scalar(float* w, float* v, float g, __nv_bfloat16* shadow, size_t i, float lr, float mu)
{
    const float vv = fmaf(mu, v[i], g), ww = fmaf(-lr, vv, w[i]);
    v[i] = vv;
    w[i] = ww;
    if (shadow) shadow[i] = __float2bfloat16_rn(ww);
}
template <int LANES>
__global__ void __launch_bounds__(32 * LANES)
reduce_sgd_many_kernel(const float* __restrict__ part, size_t stride, int splits, float* __restrict__ w, float* __restrict__ v,
                       __nv_bfloat16* __restrict__ shadow, size_t n, Hyper hy, Gap gap)
{
    pdl_prologue();
    const float lr = hy.rate(), mu = hy.decay();
    __shared__ float s[LANES][33];
    const int e = threadIdx.x % 32, lane = threadIdx.x / 32;
    const size_t i = blockIdx.x * 32ull + e;
    s[lane][e] = i < n ? many_lane_sum<LANES>(part, stride, i, lane, splits) : 0.f;
    __syncthreads();
    if (lane == 0 && i < n) {
        float r = 0.f;
#pragma unroll
        for (int j = 0; j < LANES; ++j) r += s[j][e];
        sgd_apply_scalar(w, v, r, shadow, gap.over(i), lr, mu);
    }
}
__global__ void __launch_bounds__(256)
reduce_sgd_kernel(const float* __restrict__ part, size_t stride, int splits, float* __restrict__ w, float* __restrict__ v,
                  __nv_bfloat16* __restrict__ shadow, size_t n, Hyper hy, Gap gap)
{
    pdl_prologue();
    const float lr = hy.rate(), mu = hy.decay();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float t = 0.f;
        for (int sp = 0; sp < splits; ++sp) t += part[(size_t)sp * stride + i];
        sgd_apply_scalar(w, v, t, shadow, gap.over(i), lr, mu);
    }
}
cudaError_t launch_reduce_sgd(const float* part, size_t stride, size_t n, int splits, float* w, float* v, __nv_bfloat16* shadow,
                              Hyper hy, cudaStream_t st, Gap gap)
{
    // (the same case split as launch_reduce_partials: each case sums in the same order there and here)
    if (splits >= 128 && n <= (1u << 20)) {
        SB_LAUNCH((reduce_sgd_many_kernel<32>), cdiv((long)n, 32), 1024, 0, st, part, stride, splits, w, v, shadow, n, hy, gap);
    } else if (splits >= 32 && n <= (1u << 20)) {
        SB_LAUNCH((reduce_sgd_many_kernel<8>), cdiv((long)n, 32), 256, 0, st, part, stride, splits, w, v, shadow, n, hy, gap);
    } else if (n % 4 == 0 && stride % 4 == 0 && gap.by4() && (((uintptr_t)part | (uintptr_t)w | (uintptr_t)v) & 15) == 0 && (((uintptr_t)shadow) & 7) == 0) {
        int blocks = cdiv((long)(n / 4), 256);
        if (blocks > 148 * 8) blocks = 148 * 8;
        if (shadow) SB_LAUNCH((reduce_sgd4_kernel<true>), blocks, 256, 0, st, (const float4*)part, stride / 4, splits, (float4*)w, (float4*)v, (uint2*)shadow, n / 4, hy, Gap{gap.at / 4, gap.by / 4});
        else SB_LAUNCH((reduce_sgd4_kernel<false>), blocks, 256, 0, st, (const float4*)part, stride / 4, splits, (float4*)w, (float4*)v, nullptr, n / 4, hy, Gap{gap.at / 4, gap.by / 4});
    } else {
        int blocks = cdiv((long)n, 256);
        if (blocks > 148 * 8) blocks = 148 * 8;
        SB_LAUNCH((reduce_sgd_kernel), blocks, 256, 0, st, part, stride, splits, w, v, shadow, n, hy, gap);
    }
    return cudaGetLastError();
}

// hyper-parameter words of the replayed iterations (see Hyper)
__global__ void hyper_kernel(float* dev, float lr, float mu)
{
    pdl_prologue();
    if (threadIdx.x == 0) { dev[0] = lr; dev[1] = mu; }
}
// loss and status word (adjacent device words) into pinned host memory, as the last kernel of a replayed iteration
__global__ void report_kernel(const uint32_t* words, volatile uint32_t* host)
{
    pdl_prologue();
    if (threadIdx.x < 2) host[threadIdx.x] = words[threadIdx.x];
}
cudaError_t launch_report(const float* words, uint32_t* host, cudaStream_t st)
{
    SB_LAUNCH((report_kernel), 1, 32, 0, st, (const uint32_t*)words, (volatile uint32_t*)host);
    return cudaGetLastError();
}
cudaError_t launch_hyper(float* dev, float lr, float mu, cudaStream_t st)
{
    SB_LAUNCH((hyper_kernel), 1, 32, 0, st, dev, lr, mu);
    return cudaGetLastError();
}

cudaError_t launch_sgd(float* w, float* v, const float* g, __nv_bfloat16* shadow, size_t n, Hyper hy, cudaStream_t st)
{
    size_t n4 = n / 4;
    static const int per_sm = (int)tune("SB_SGD_BLOCKS_PER_SM", 16);
    long blocks = ((long)n4 + 255) / 256;
    if (blocks > 148L * per_sm) blocks = 148L * per_sm;
    if (blocks < 1) blocks = 1;
    if (shadow) SB_LAUNCH((sgd_kernel<true>), (int)blocks, 256, 0, st, (float4*)w, (float4*)v, (const float4*)g, (uint2*)shadow, n4, hy);
    else SB_LAUNCH((sgd_kernel<false>), (int)blocks, 256, 0, st, (float4*)w, (float4*)v, (const float4*)g, nullptr, n4, hy);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256)
to_bf16_kernel(const float4* __restrict__ w, uint2* __restrict__ shadow, size_t n4)
{
    pdl_prologue();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        float4 ww = w[i];
        __nv_bfloat162 lo = __floats2bfloat162_rn(ww.x, ww.y), hi = __floats2bfloat162_rn(ww.z, ww.w);
        uint2 pk;
        pk.x = *(uint32_t*)&lo;
        pk.y = *(uint32_t*)&hi;
        shadow[i] = pk;
    }
}
cudaError_t launch_to_bf16(const float* w, __nv_bfloat16* shadow, size_t n, cudaStream_t st)
{
    SB_LAUNCH((to_bf16_kernel), ew_blocks((long)(n / 4)), 256, 0, st, (const float4*)w, (uint2*)shadow, n / 4);
    return cudaGetLastError();
}

// =============================================================================================
// Input-layer convolution (Cin <= 4, e.g. RGB images): 9*Cin <= 36 products per output, far too
// thin for tensor-core tiles and bound by the output / dy traffic.  Each thread builds the
// 3x3xCin patch of its pixel in registers (forward) or the block stages patches in shared memory
// (weight gradient).
// =============================================================================================
template <typename T, int CIN, bool TAB>
__device__ __forceinline__ void load_patch(float (&patch)[9 * CIN], const T* __restrict__ x, const PtrTab& tab, int b_per_rep,
                                           long pix, int H, int W)
{
    const int w_ = (int)(pix % W);
    const long q = pix / W;
    const int h_ = (int)(q % H), n_ = (int)(q / H);
    const T* img = TAB ? (const T*)tab.p[n_ / b_per_rep] + (size_t)(n_ % b_per_rep) * H * W * CIN : x + (size_t)n_ * H * W * CIN;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int hh = h_ + r - 1, ww = w_ + s - 1;
            const bool in = hh >= 0 && hh < H && ww >= 0 && ww < W;
#pragma unroll
            for (int c = 0; c < CIN; ++c) patch[(r * 3 + s) * CIN + c] = in ? ldf(img + ((size_t)hh * W + ww) * CIN + c) : 0.f;
        }
}

// Forward: 8 consecutive threads share a pixel, each produces 8 output channels (16-byte stores that
// a warp lays down as contiguous 128-byte pixel rows).  Weights live in shared memory as [9*CIN][Cout].
template <typename T, int CIN, bool TAB>
__global__ void __launch_bounds__(256)
conv_in_fwd_kernel(const T* __restrict__ x, PtrTab tab, int b_per_rep, const T* __restrict__ wt, const float* __restrict__ bias,
                   T* __restrict__ y, long npix, int H, int W, int Cout, int relu)
{
    pdl_prologue();
    extern __shared__ float s_wf[];            // [9*CIN][Cout] then bias [Cout]
    float* s_b = s_wf + 9 * CIN * Cout;
    for (int e = threadIdx.x; e < 9 * CIN * Cout; e += 256) {
        int k = e % Cout, j = e / Cout;
        s_wf[e] = ldf(wt + (size_t)k * 9 * CIN + j);
    }
    for (int e = threadIdx.x; e < Cout; e += 256) s_b[e] = bias[e];
    __syncthreads();
    const int groups = Cout / 8;               // threads per pixel
    const long t = blockIdx.x * 256L + threadIdx.x;
    const long pix = t / groups;
    const int kg = (int)(t % groups) * 8;
    if (pix >= npix) return;
    float patch[9 * CIN];
    load_patch<T, CIN, TAB>(patch, x, tab, b_per_rep, pix, H, W);
    float acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = s_b[kg + i];
#pragma unroll
    for (int j = 0; j < 9 * CIN; ++j) {
        const float4 w0 = *(const float4*)(s_wf + j * Cout + kg), w1 = *(const float4*)(s_wf + j * Cout + kg + 4);
        acc[0] = fmaf(patch[j], w0.x, acc[0]); acc[1] = fmaf(patch[j], w0.y, acc[1]);
        acc[2] = fmaf(patch[j], w0.z, acc[2]); acc[3] = fmaf(patch[j], w0.w, acc[3]);
        acc[4] = fmaf(patch[j], w1.x, acc[4]); acc[5] = fmaf(patch[j], w1.y, acc[5]);
        acc[6] = fmaf(patch[j], w1.z, acc[6]); acc[7] = fmaf(patch[j], w1.w, acc[7]);
    }
    if (relu) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (!(acc[i] > 0.f)) acc[i] = 0.f;
    }
    store8(y + (size_t)pix * Cout + kg, acc);
}

// Forward, 4 pixels per thread (W a multiple of 4): a thread owns 4 horizontally adjacent pixels and 8 output
// channels.  The 3 x 6 x CIN input window of the 4 pixels sits in registers, so each pair of 16-byte weight
// reads from shared memory feeds 32 FMAs (the 1-pixel kernel above is bound by those reads).
template <typename T, int CIN, bool TAB>
__global__ void __launch_bounds__(256)
conv_in_fwd4_kernel(const T* __restrict__ x, PtrTab tab, int b_per_rep, const T* __restrict__ wt, const float* __restrict__ bias,
                    T* __restrict__ y, long nquads, int H, int W, int Cout, int relu)
{
    pdl_prologue();
    extern __shared__ float s_wf[];            // [9*CIN][Cout] then bias [Cout]
    float* s_b = s_wf + 9 * CIN * Cout;
    for (int e = threadIdx.x; e < 9 * CIN * Cout; e += 256) {
        int k = e % Cout, j = e / Cout;
        s_wf[e] = ldf(wt + (size_t)k * 9 * CIN + j);
    }
    for (int e = threadIdx.x; e < Cout; e += 256) s_b[e] = bias[e];
    __syncthreads();
    const int groups = Cout / 8;
    const long t = blockIdx.x * 256L + threadIdx.x;
    const long quad = t / groups;
    const int kg = (int)(t % groups) * 8;
    if (quad >= nquads) return;
    const int wq = W / 4;
    const int w0 = (int)(quad % wq) * 4;
    const long q2 = quad / wq;
    const int h = (int)(q2 % H);
    const long n = q2 / H;
    const T* img = TAB ? (const T*)tab.p[n / b_per_rep] + (size_t)(n % b_per_rep) * H * W * CIN : x + (size_t)n * H * W * CIN;
    float win[3][6 * CIN];                     // rows h-1..h+1, columns w0-1..w0+4
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int hh = h + r - 1;
#pragma unroll
        for (int c6 = 0; c6 < 6; ++c6) {
            const int ww = w0 + c6 - 1;
            const bool in = hh >= 0 && hh < H && ww >= 0 && ww < W;
#pragma unroll
            for (int c = 0; c < CIN; ++c) win[r][c6 * CIN + c] = in ? ldf(img + ((size_t)hh * W + ww) * CIN + c) : 0.f;
        }
    }
    float acc[4][8];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[p][i] = s_b[kg + i];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int sc = 0; sc < 3 * CIN; ++sc) {          // sc = s*CIN + c
            const int j = r * 3 * CIN + sc;
            const float4 w0v = *(const float4*)(s_wf + j * Cout + kg), w1v = *(const float4*)(s_wf + j * Cout + kg + 4);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float xv = win[r][p * CIN + sc];
                acc[p][0] = fmaf(xv, w0v.x, acc[p][0]); acc[p][1] = fmaf(xv, w0v.y, acc[p][1]);
                acc[p][2] = fmaf(xv, w0v.z, acc[p][2]); acc[p][3] = fmaf(xv, w0v.w, acc[p][3]);
                acc[p][4] = fmaf(xv, w1v.x, acc[p][4]); acc[p][5] = fmaf(xv, w1v.y, acc[p][5]);
                acc[p][6] = fmaf(xv, w1v.z, acc[p][6]); acc[p][7] = fmaf(xv, w1v.w, acc[p][7]);
            }
        }
    const size_t pix0 = ((size_t)n * H + h) * W + w0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        if (relu) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (!(acc[p][i] > 0.f)) acc[p][i] = 0.f;
        }
        store8(y + (pix0 + p) * Cout + kg, acc[p]);
    }
}

// Weight + bias gradient: block = 64 output channels x 4 pixel lanes; per 64-pixel chunk the block stages
// the patches in shared memory, then thread (k, q) accumulates dy[pix,k] * patch[pix,:] over its pixels.
// part[block][k][9*CIN] and part_b[block][k] are reduced afterwards in block order.
template <typename T, int CIN, bool TAB>
__global__ void __launch_bounds__(256)
conv_in_wgrad_kernel(const T* __restrict__ x, PtrTab tab, int b_per_rep, const T* __restrict__ dy, float* __restrict__ part,
                     long npix, int H, int W, int Cout, long stride_floats)
{
    pdl_prologue();
    constexpr int PJ = (9 * CIN + 3) / 4 * 4;   // padded patch length (16-byte rows)
    __shared__ __align__(16) float s_patch[64][PJ];
    __shared__ float s_red[3][64][9 * CIN + 1];
    const int k = threadIdx.x % 64, q = threadIdx.x / 64;
    const int k0 = blockIdx.y * 64;
    float acc[9 * CIN], accb = 0.f;
#pragma unroll
    for (int j = 0; j < 9 * CIN; ++j) acc[j] = 0.f;
    const long nchunks = (npix + 63) / 64;
    for (long ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const long p0 = ch * 64;
        {
            // staging: thread (pixel pp, filter row r) writes the 3 taps x CIN values of that row; lane group 3
            // clears the padding columns
            const int pp = threadIdx.x % 64, r = threadIdx.x / 64;
            const long pix = p0 + pp;
            if (r < 3) {
                const int w_ = (int)(pix % W);
                const long t = pix / W;
                const int h_ = (int)(t % H);
                const long n_ = t / H;
                const int hh = h_ + r - 1;
                const bool row_in = pix < npix && hh >= 0 && hh < H;
                const T* img = nullptr;
                if (row_in)
                    img = (TAB ? (const T*)tab.p[n_ / b_per_rep] + (size_t)(n_ % b_per_rep) * H * W * CIN : x + (size_t)n_ * H * W * CIN) +
                          (size_t)hh * W * CIN;
#pragma unroll
                for (int sdx = 0; sdx < 3; ++sdx) {
                    const int ww = w_ + sdx - 1;
                    const bool in = row_in && ww >= 0 && ww < W;
#pragma unroll
                    for (int c = 0; c < CIN; ++c) s_patch[pp][(r * 3 + sdx) * CIN + c] = in ? ldf(img + (size_t)ww * CIN + c) : 0.f;
                }
            } else {
#pragma unroll
                for (int j = 9 * CIN; j < PJ; ++j) s_patch[pp][j] = 0.f;
            }
        }
        __syncthreads();
        if (k0 + k < Cout) {
            // this thread's 16 pixels of the chunk, 4 at a time so that 4 dy loads are in flight together
            for (int pg = 0; pg < 4; ++pg) {
                float d[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long pix = p0 + q + 4 * (pg * 4 + u);
                    d[u] = pix < npix ? ldf(dy + (size_t)pix * Cout + k0 + k) : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int pp = q + 4 * (pg * 4 + u);
                    accb += d[u];
                    float pv[PJ];
#pragma unroll
                    for (int j4 = 0; j4 < PJ / 4; ++j4) {
                        const float4 v = *(const float4*)&s_patch[pp][j4 * 4];
                        pv[j4 * 4] = v.x; pv[j4 * 4 + 1] = v.y; pv[j4 * 4 + 2] = v.z; pv[j4 * 4 + 3] = v.w;
                    }
#pragma unroll
                    for (int j = 0; j < 9 * CIN; ++j) acc[j] = fmaf(d[u], pv[j], acc[j]);
                }
            }
        }
        __syncthreads();
    }
    // fixed-order reduction over the 4 pixel lanes
    if (q > 0) {
#pragma unroll
        for (int j = 0; j < 9 * CIN; ++j) s_red[q - 1][k][j] = acc[j];
        s_red[q - 1][k][9 * CIN] = accb;
    }
    __syncthreads();
    if (q == 0 && k0 + k < Cout) {
        float* dst = part + (size_t)blockIdx.x * stride_floats;
#pragma unroll
        for (int j = 0; j < 9 * CIN; ++j) dst[(size_t)(k0 + k) * 9 * CIN + j] = acc[j] + s_red[0][k][j] + s_red[1][k][j] + s_red[2][k][j];
        dst[(size_t)Cout * 9 * CIN + k0 + k] = accb + s_red[0][k][9 * CIN] + s_red[1][k][9 * CIN] + s_red[2][k][9 * CIN];
    }
}

template <typename T, int CIN>
static cudaError_t launch_conv_in_fwd_t(const ConvSimtArgs& a, cudaStream_t st)
{
    const long npix = (long)a.B * a.H * a.W;
    const long threads = npix * (a.Cout / 8);
    const int blocks = (int)((threads + 255) / 256);
    const size_t smem = (size_t)(9 * CIN * a.Cout + a.Cout) * 4;
    PtrTab tab{};
    if (a.tab) tab = *a.tab;
    if (a.W % 4 == 0) {
        const long nquads = npix / 4;
        const int qblocks = (int)((nquads * (a.Cout / 8) + 255) / 256);
        if (a.tab) SB_LAUNCH((conv_in_fwd4_kernel<T, CIN, true>), qblocks, 256, smem, st, nullptr, tab, a.b_per_rep, (const T*)a.w, a.bias, (T*)a.out, nquads, a.H, a.W, a.Cout, a.relu);
        else SB_LAUNCH((conv_in_fwd4_kernel<T, CIN, false>), qblocks, 256, smem, st, (const T*)a.in, tab, a.b_per_rep, (const T*)a.w, a.bias, (T*)a.out, nquads, a.H, a.W, a.Cout, a.relu);
        return cudaGetLastError();
    }
    if (a.tab) SB_LAUNCH((conv_in_fwd_kernel<T, CIN, true>), blocks, 256, smem, st, nullptr, tab, a.b_per_rep, (const T*)a.w, a.bias, (T*)a.out, npix, a.H, a.W, a.Cout, a.relu);
    else SB_LAUNCH((conv_in_fwd_kernel<T, CIN, false>), blocks, 256, smem, st, (const T*)a.in, tab, a.b_per_rep, (const T*)a.w, a.bias, (T*)a.out, npix, a.H, a.W, a.Cout, a.relu);
    return cudaGetLastError();
}
bool conv_in_supported(int Cin, int Cout) { return (Cin == 1 || Cin == 3 || Cin == 4) && Cout % 8 == 0 && Cout <= 256; }
cudaError_t launch_conv_in_fwd(const ConvSimtArgs& a, bool bf16, cudaStream_t st)
{
#define SB_CI(T) (a.Cin == 1 ? launch_conv_in_fwd_t<T, 1>(a, st) : a.Cin == 3 ? launch_conv_in_fwd_t<T, 3>(a, st) : launch_conv_in_fwd_t<T, 4>(a, st))
    return bf16 ? SB_CI(__nv_bfloat16) : SB_CI(float);
#undef SB_CI
}
int conv_in_wgrad_blocks(int B, int H, int W)
{
    long chunks = ((long)B * H * W + 63) / 64;
    return (int)(chunks < 148 * 4 ? chunks : 148 * 4);
}
template <typename T, int CIN>
static cudaError_t launch_conv_in_wgrad_t(const WgradSimtArgs& a, cudaStream_t st)
{
    const long npix = (long)a.B * a.H * a.W;
    dim3 grid(conv_in_wgrad_blocks(a.B, a.H, a.W), (a.Cout + 63) / 64);
    const long stride = (long)a.Cout * 9 * CIN + a.Cout;
    PtrTab tab{};
    if (a.tab) tab = *a.tab;
    if (a.tab) SB_LAUNCH((conv_in_wgrad_kernel<T, CIN, true>), grid, 256, 0, st, nullptr, tab, a.b_per_rep, (const T*)a.dy, a.part, npix, a.H, a.W, a.Cout, stride);
    else SB_LAUNCH((conv_in_wgrad_kernel<T, CIN, false>), grid, 256, 0, st, (const T*)a.x, tab, a.b_per_rep, (const T*)a.dy, a.part, npix, a.H, a.W, a.Cout, stride);
    return cudaGetLastError();
}
// part: [conv_in_wgrad_blocks][Cout*9*Cin + Cout] floats (weights then bias), to be reduced in block order.
cudaError_t launch_conv_in_wgrad(const WgradSimtArgs& a, bool bf16, cudaStream_t st)
{
#define SB_CI(T) (a.Cin == 1 ? launch_conv_in_wgrad_t<T, 1>(a, st) : a.Cin == 3 ? launch_conv_in_wgrad_t<T, 3>(a, st) : launch_conv_in_wgrad_t<T, 4>(a, st))
    return bf16 ? SB_CI(__nv_bfloat16) : SB_CI(float);
#undef SB_CI
}

// =============================================================================================
// Narrow FC layers (out <= 16, e.g. the 10-class logits layer): too narrow for any GEMM tile.
//   forward : one block per batch row, a warp per output
//   wgrad   : one thread per input column, dY staged in shared memory
//   dgrad   : one thread per 16 bytes of an input row and two batch rows
// =============================================================================================
constexpr int NARROW_MAX = 16;

template <typename T> struct Vec8;
template <> struct Vec8<float> { static constexpr int N = 4; typedef float4 V; };
template <> struct Vec8<__nv_bfloat16> { static constexpr int N = 8; typedef uint4 V; };

// Forward.  Block = one batch row, a warp per output: the kernel is pure latency, so every lane has eight 16-byte loads in flight and
// the code is one short loop.  (Two rows a block, the reduction in four slices and all outputs in a lane's registers: 6.5 us for
// 4096 -> 10 at batch 128 in the replayed VGG-16 iteration; here 4.9 with the softmax.)  A lane keeps a sum for each of its four loads of
// a step: one chain over all of its in_f / 32 products carried twice the rounding (float, 2-norm against 64-bit sums: 4096 inputs
// 1.5e-7 where four give 1.0e-7, 25088 inputs 4.1e-7 and 2.2e-7).  Two blocks an SM: left alone the compiler fits the float form into 32
// registers, too few for the loads (25088 -> 10 at batch 96, whole call 43 us, 26 so).
// XENT: softmax cross-entropy of the row by warp 0, with the operations of softmax_xent_kernel in its order, without that kernel's
// 4.3 us on the chain (most of them the last block's wait for every row loss).
struct HeadArgs { PtrTab labels; int b_per_rep; float* row_loss; void* dZ; int scale_B; };
template <typename T, bool TAB, bool VEC, bool XENT>
__global__ void __launch_bounds__(32 * NARROW_MAX, 2)
fc_narrow_fwd_kernel(const T* __restrict__ X, PtrTab tab, int tab_b, const T* __restrict__ Wt, const float* __restrict__ bias,
                     T* __restrict__ Y, float* __restrict__ Y32, int in_f, int out_f, int relu, const __grid_constant__ HeadArgs head)
{
    pdl_prologue();
    constexpr int VN = Vec8<T>::N;
    typedef typename Vec8<T>::V V;
    __shared__ float s_z[NARROW_MAX];
    const int j = threadIdx.x / 32, lane = threadIdx.x % 32, g = blockIdx.x;
    const T* xr = TAB ? (const T*)tab.p[g / tab_b] + (size_t)(g % tab_b) * in_f : X + (size_t)g * in_f;
    const T* wr = Wt + (size_t)j * in_f;
    int label = 0;
    if (XENT && j == 0) label = ((const int32_t*)head.labels.p[g / head.b_per_rep])[g % head.b_per_rep];
    float acc;
    if (VEC) {
        float part[4] = {0.f, 0.f, 0.f, 0.f};
        // (the host only selects this variant when every row starts 16-byte aligned)
#pragma unroll 1
        for (int k0 = lane * VN; k0 < in_f; k0 += 128 * VN) {
            V xv[4], wv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + u * 32 * VN;
                const V zero = V();
                xv[u] = k < in_f ? *(const V*)(xr + k) : zero;
                wv[u] = k < in_f ? *(const V*)(wr + k) : zero;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u * 32 * VN < in_f)
#pragma unroll
                    for (int i = 0; i < VN; ++i) part[u] = fmaf(ldf((const T*)&xv[u] + i), ldf((const T*)&wv[u] + i), part[u]);
        }
        acc = (part[0] + part[1]) + (part[2] + part[3]);
    } else {
        acc = 0.f;
        for (int k = lane; k < in_f; k += 32) acc = fmaf(ldf(xr + k), ldf(wr + k), acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
        float v = bias[j] + acc;
        if (relu && !(v > 0.f)) v = 0.f;
        if (Y32) Y32[(size_t)g * out_f + j] = v;
        if (Y) stf(Y + (size_t)g * out_f + j, v);
        s_z[j] = v;
    }
    if (!XENT) return;
    __syncthreads();
    if (j != 0) return;
    const float z = lane < out_f ? s_z[lane] : -INFINITY;
    float m = fmaxf(-INFINITY, z);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float s = lane < out_f ? expf(z - m) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float lse = m + logf(s), invB = 1.0f / (float)head.scale_B;
    if (lane < out_f) stf((T*)head.dZ + (size_t)g * out_f + lane, (expf(z - lse) - (lane == label ? 1.f : 0.f)) * invB);
    if (lane == 0) head.row_loss[g] = (label >= 0 && label < out_f) ? lse - s_z[label] : 0.f;
}

// Weight + bias gradient: block = 32 input columns x 8 row lanes; lane l sums batch rows l, l+8, ... for its
// column, then the 8 lanes are combined in lane order through shared memory (deterministic).
template <typename T, bool TAB>
__global__ void __launch_bounds__(256)
fc_narrow_wgrad_kernel(const T* __restrict__ X, PtrTab tab, int tab_b, const T* __restrict__ dY, float* __restrict__ dW,
                       float* __restrict__ db, int B, int in_f, int out_f)
{
    pdl_prologue();
    extern __shared__ float s_dy[];   // [B][out_f], then the reduction buffer [8][32][NARROW_MAX]
    float* s_red = s_dy + B * out_f;
    for (int e = threadIdx.x; e < B * out_f; e += 256) s_dy[e] = ldf(dY + e);
    __syncthreads();
    const int col = threadIdx.x % 32, lane = threadIdx.x / 32;
    const int i = blockIdx.x * 32 + col;
    if (blockIdx.x == 0 && threadIdx.x < out_f) {
        float t = 0.f;
        for (int g = 0; g < B; ++g) t += s_dy[g * out_f + threadIdx.x];
        db[threadIdx.x] = t;
    }
    float acc[NARROW_MAX];
#pragma unroll
    for (int j = 0; j < NARROW_MAX; ++j) acc[j] = 0.f;
    if (i < in_f) {
        for (int g = lane; g < B; g += 8) {
            const T* xr = TAB ? (const T*)tab.p[g / tab_b] + (size_t)(g % tab_b) * in_f : X + (size_t)g * in_f;
            const float xv = ldf(xr + i);
#pragma unroll
            for (int j = 0; j < NARROW_MAX; ++j)
                if (j < out_f) acc[j] = fmaf(s_dy[g * out_f + j], xv, acc[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < NARROW_MAX; ++j) s_red[(lane * 32 + col) * NARROW_MAX + j] = acc[j];
    __syncthreads();
    if (lane == 0 && i < in_f) {
#pragma unroll
        for (int j = 0; j < NARROW_MAX; ++j)
            if (j < out_f) {
                float t = 0.f;
#pragma unroll
                for (int l = 0; l < 8; ++l) t += s_red[(l * 32 + col) * NARROW_MAX + j];
                dW[(size_t)j * in_f + i] = t;
            }
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
fc_narrow_dgrad_kernel(const T* __restrict__ dY, const T* __restrict__ Wt, const T* __restrict__ ref, T* __restrict__ dX,
                       int in_f, int out_f)
{
    pdl_prologue();
    __shared__ float s_d[NARROW_MAX];
    const int g = blockIdx.y;
    if (threadIdx.x < out_f) s_d[threadIdx.x] = ldf(dY + (size_t)g * out_f + threadIdx.x);
    __syncthreads();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= in_f) return;
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < NARROW_MAX; ++j)
        if (j < out_f) acc = fmaf(s_d[j], ldf(Wt + (size_t)j * in_f + i), acc);
    if (ref != nullptr && !(ldf(ref + (size_t)g * in_f + i) > 0.f)) acc = 0.f;
    stf(dX + (size_t)g * in_f + i, acc);
}

// By 16-byte accesses: a thread takes VN columns of ROWS batch rows (same products in the same order as the kernel above; 4096 columns at
// batch 128, a column and a row per thread: 6.5 us in the replayed iteration, here 3.6).
template <typename T, int ROWS>
__global__ void __launch_bounds__(64)
fc_narrow_dgrad_vec_kernel(const T* __restrict__ dY, const T* __restrict__ Wt, const T* __restrict__ ref, T* __restrict__ dX, int B, int in_f, int out_f)
{
    pdl_prologue();
    constexpr int VN = Vec8<T>::N;
    typedef typename Vec8<T>::V V;
    const int i = (blockIdx.x * 64 + threadIdx.x) * VN, g0 = blockIdx.y * ROWS;
    if (i >= in_f) return;
    V r[ROWS];
    float acc[ROWS][VN];
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
        if (ref != nullptr && g0 + u < B) r[u] = *(const V*)(ref + (size_t)(g0 + u) * in_f + i);
#pragma unroll
        for (int k = 0; k < VN; ++k) acc[u][k] = 0.f;
    }
#pragma unroll 4
    for (int j = 0; j < out_f; ++j) {
        const V w = *(const V*)(Wt + (size_t)j * in_f + i);
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            const float d = ldf(dY + (size_t)min(g0 + u, B - 1) * out_f + j);
#pragma unroll
            for (int k = 0; k < VN; ++k) acc[u][k] = fmaf(d, ldf((const T*)&w + k), acc[u][k]);
        }
    }
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
        if (g0 + u >= B) break;
        V o;
#pragma unroll
        for (int k = 0; k < VN; ++k) {
            if (ref != nullptr && !(ldf((const T*)&r[u] + k) > 0.f)) acc[u][k] = 0.f;
            stf((T*)&o + k, acc[u][k]);
        }
        *(V*)(dX + (size_t)(g0 + u) * in_f + i) = o;
    }
}

bool fc_narrow_supported(int out_f, int B) { return out_f <= NARROW_MAX && (size_t)B * out_f * 4 <= 24 * 1024; }

template <typename T>
static cudaError_t launch_fc_narrow_t(const FcNarrowArgs& a, cudaStream_t st)
{
    PtrTab tab{};
    if (a.tab) tab = *a.tab;
    const int tb = a.tab_b > 0 ? a.tab_b : 1;
    if (a.pass == 0) {
        const bool vec = (((uintptr_t)a.W | (uintptr_t)a.X) & 15) == 0 && !a.tab && a.in_f % Vec8<T>::N == 0;
        HeadArgs head{};
        if (a.xent) head = HeadArgs{a.xent->labels, a.xent->b_per_rep, a.xent->row_loss, a.xent->dZ, a.xent->scale_B > 0 ? a.xent->scale_B : a.xent->B};
#define SB_NFX(TABF, VECF, XENTF) SB_LAUNCH((fc_narrow_fwd_kernel<T, TABF, VECF, XENTF>), a.B, 32 * a.out_f, 0, st,  \
            (const T*)a.X, tab, tb, (const T*)a.W, a.bias, (T*)a.Y, a.Y32, a.in_f, a.out_f, a.relu, head)
#define SB_NF(TABF, VECF) do { if (a.xent) SB_NFX(TABF, VECF, true); else SB_NFX(TABF, VECF, false); } while (0)
        if (vec) SB_NF(false, true);
        else if (a.tab) SB_NF(true, false);
        else SB_NF(false, false);
#undef SB_NF
#undef SB_NFX
    } else if (a.pass == 1) {
        const size_t smem = (size_t)a.B * a.out_f * 4 + 8 * 32 * NARROW_MAX * 4;
        const int blocks = (a.in_f + 31) / 32;
        if (a.tab) SB_LAUNCH((fc_narrow_wgrad_kernel<T, true>), blocks, 256, smem, st, nullptr, tab, tb, (const T*)a.dY, a.dW, a.db, a.B, a.in_f, a.out_f);
        else SB_LAUNCH((fc_narrow_wgrad_kernel<T, false>), blocks, 256, smem, st, (const T*)a.X, tab, tb, (const T*)a.dY, a.dW, a.db, a.B, a.in_f, a.out_f);
    } else if (a.in_f % Vec8<T>::N == 0 && (((uintptr_t)a.W | (uintptr_t)a.ref | (uintptr_t)a.dX) & 15) == 0) {
        const int bx = (a.in_f / Vec8<T>::N + 63) / 64;
        if (a.B > 64) SB_LAUNCH((fc_narrow_dgrad_vec_kernel<T, 2>), dim3(bx, (a.B + 1) / 2), 64, 0, st, (const T*)a.dY, (const T*)a.W, (const T*)a.ref, (T*)a.dX, a.B, a.in_f, a.out_f);
        else SB_LAUNCH((fc_narrow_dgrad_vec_kernel<T, 1>), dim3(bx, a.B), 64, 0, st, (const T*)a.dY, (const T*)a.W, (const T*)a.ref, (T*)a.dX, a.B, a.in_f, a.out_f);
    } else {
        dim3 grid((a.in_f + 255) / 256, a.B);
        SB_LAUNCH((fc_narrow_dgrad_kernel<T>), grid, 256, 0, st, (const T*)a.dY, (const T*)a.W, (const T*)a.ref, (T*)a.dX, a.in_f, a.out_f);
    }
    return cudaGetLastError();
}
cudaError_t launch_fc_narrow(const FcNarrowArgs& a, bool bf16, cudaStream_t st)
{
    return bf16 ? launch_fc_narrow_t<__nv_bfloat16>(a, st) : launch_fc_narrow_t<float>(a, st);
}

}  // namespace sb
