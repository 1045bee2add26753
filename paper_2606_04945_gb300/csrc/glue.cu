// Glue of the transformer blocks around the quantised linears: the residual
// add with RMSNorm, and rotary position embedding. Not part of the paper's
// method (Sec. 3 quantises the linears and the softmax-value product); the
// block runs them between its projections, and they are memory-bound
// element-wise passes.
//
// add_rmsnorm (one CTA of 128 threads per row, 16-byte vectors):
//   h = fl_T(x + r)                 (r = NULL: h = x; stored when h_out != NULL)
//   y = fl_T(fl32(h * inv) * w)     inv = 1 / sqrt(mean(h^2) + eps), float32
// rope (one CTA per token):
//   for each head of 128 channels and i < 64, with angle = pos * f_i and
//   f_i = theta^(-2 i / 128) (computed in float64 on the host, rounded to float32):
//   (a, b) = (x_i, x_{i+64});  x_i = fl_T(a c - b s),  x_{i+64} = fl_T(b c + a s)
//   with c, s = cos, sin of the float32 angle, the products and sums in
//   float32 (the rotate-half form of the LLaMA / Qwen2 family).
#include <cmath>

#include "common.cuh"

namespace starq {
namespace {

constexpr int NORM_THREADS = 128;

template <typename T> struct Vec;
template <> struct Vec<__half> {
    static __device__ __forceinline__ void load(const uint4& w, float (&f)[8]) {
        const __half2* h = reinterpret_cast<const __half2*>(&w);
        #pragma unroll
        for (int k = 0; k < 4; ++k) { const float2 v = __half22float2(h[k]); f[2 * k] = v.x; f[2 * k + 1] = v.y; }
    }
    static __device__ __forceinline__ uint4 store(const float (&f)[8]) {
        uint4 w;
        __half2* h = reinterpret_cast<__half2*>(&w);
        #pragma unroll
        for (int k = 0; k < 4; ++k) h[k] = __floats2half2_rn(f[2 * k], f[2 * k + 1]);
        return w;
    }
};
template <> struct Vec<__nv_bfloat16> {
    static __device__ __forceinline__ void load(const uint4& w, float (&f)[8]) {
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&w);
        #pragma unroll
        for (int k = 0; k < 4; ++k) { const float2 v = __bfloat1622float2(h[k]); f[2 * k] = v.x; f[2 * k + 1] = v.y; }
    }
    static __device__ __forceinline__ uint4 store(const float (&f)[8]) {
        uint4 w;
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&w);
        #pragma unroll
        for (int k = 0; k < 4; ++k) h[k] = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
        return w;
    }
};

// Up to MAXV 16-byte vectors per thread (K <= 8 * 128 * MAXV).
template <typename T, int MAXV>
// h_out may be X or R: every thread reads its own vectors before it writes
// them, so the in-place form needs no ordering between threads.
__global__ void __launch_bounds__(NORM_THREADS) add_rmsnorm_kernel(const T* X, const T* R, int K,
                                                                  const float* __restrict__ w, float eps, T* h_out,
                                                                  T* __restrict__ Y) {
    __shared__ float part[NORM_THREADS / 32];
    const size_t row = blockIdx.x;
    const int nv = K / 8;
    const uint4* x4 = reinterpret_cast<const uint4*>(X + row * K);
    const uint4* r4 = R != nullptr ? reinterpret_cast<const uint4*>(R + row * K) : nullptr;
    float v[MAXV][8];
    float ss = 0.f;
    #pragma unroll
    for (int j = 0; j < MAXV; ++j) {
        const int i = threadIdx.x + j * NORM_THREADS;
        if (i < nv) {
            Vec<T>::load(x4[i], v[j]);
            if (r4 != nullptr) {
                float r[8];
                Vec<T>::load(r4[i], r);
                #pragma unroll
                for (int k = 0; k < 8; ++k) v[j][k] = __fadd_rn(v[j][k], r[k]);
                const uint4 hw = Vec<T>::store(v[j]);      // h rounded to T, as the residual stream is stored
                Vec<T>::load(hw, v[j]);
                if (h_out != nullptr) reinterpret_cast<uint4*>(h_out + row * K)[i] = hw;
            }
            #pragma unroll
            for (int k = 0; k < 8; ++k) ss = fmaf(v[j][k], v[j][k], ss);
        }
    }
    #pragma unroll
    for (int m = 16; m > 0; m >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, m);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (Y == nullptr) return;
    const float tot = (part[0] + part[1]) + (part[2] + part[3]);
    const float inv = rsqrtf(__fadd_rn(__fdiv_rn(tot, (float)K), eps));
    uint4* y4 = reinterpret_cast<uint4*>(Y + row * K);
    const float4* w4 = reinterpret_cast<const float4*>(w);
    #pragma unroll
    for (int j = 0; j < MAXV; ++j) {
        const int i = threadIdx.x + j * NORM_THREADS;
        if (i < nv) {
            const float4 a = __ldg(w4 + 2 * i), b = __ldg(w4 + 2 * i + 1);
            const float wv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            float o[8];
            #pragma unroll
            for (int k = 0; k < 8; ++k) o[k] = __fmul_rn(__fmul_rn(v[j][k], inv), wv[k]);
            y4[i] = Vec<T>::store(o);
        }
    }
}

// Rotation of the query and key heads of one token per CTA. Bound by memory:
// every element is read and written once. The 64 sine / cosine pairs of a
// token are the same for all of its heads, so 64 threads compute them once
// (while the CTA's first vectors are in flight) and the heads take them from
// shared memory; the frequencies come from the host as kernel arguments.
// 1024 tokens x 64 heads, fp16: 9 us inside the captured stack step, where one
// sincosf per pair and head and 64 float64 pow per CTA took 42 (traffic alone:
// 5); 8192 x 32, bf16: 35 us against 85 (traffic alone: 20).
// VEC: 16-byte vectors, item t = 8 pairs j .. j + 7 (j = 8 (t mod 8)) of head
// t / 8; otherwise (unaligned QK or ld) one pair per item.
struct RopeFreq { float f[64]; };
constexpr int ROPE_THREADS = 256;

template <typename T, bool VEC>
__global__ void __launch_bounds__(ROPE_THREADS) rope_kernel(T* QK, int ld, int heads, const int* __restrict__ pos,
                                                            const RopeFreq freq) {
    __shared__ __align__(16) float cs[64], sn[64];
    const size_t tok = blockIdx.x;
    T* row = QK + tok * ld;
    constexpr int PER_HEAD = VEC ? 8 : 64;
    const int n = heads * PER_HEAD;
    int t = threadIdx.x;
    uint4 a4 = make_uint4(0u, 0u, 0u, 0u), b4 = a4;
    if (VEC && t < n) {                                    // in flight during the sine / cosine
        const uint4* p = reinterpret_cast<const uint4*>(row + (t >> 3) * 128 + (t & 7) * 8);
        a4 = p[0];
        b4 = p[8];
    }
    if (threadIdx.x < 64) {
        const float ang = __fmul_rn((float)pos[tok], freq.f[threadIdx.x]);
        sincosf(ang, &sn[threadIdx.x], &cs[threadIdx.x]);
    }
    __syncthreads();
    if (VEC) {
        const int j = (threadIdx.x & 7) * 8;               // the same pairs for every item of the thread
        float c[8], s[8];
        #pragma unroll
        for (int k = 0; k < 8; k += 4) {
            const float4 c4 = *reinterpret_cast<const float4*>(&cs[j + k]);
            const float4 s4 = *reinterpret_cast<const float4*>(&sn[j + k]);
            c[k] = c4.x; c[k + 1] = c4.y; c[k + 2] = c4.z; c[k + 3] = c4.w;
            s[k] = s4.x; s[k + 1] = s4.y; s[k + 2] = s4.z; s[k + 3] = s4.w;
        }
        for (; t < n; t += ROPE_THREADS) {
            uint4* p = reinterpret_cast<uint4*>(row + (t >> 3) * 128 + j);
            float a[8], b[8], x[8], y[8];
            Vec<T>::load(a4, a);
            Vec<T>::load(b4, b);
            if (t + ROPE_THREADS < n) {                    // the next item's vectors ahead of this one's stores
                a4 = p[ROPE_THREADS / 8 * 16];
                b4 = p[ROPE_THREADS / 8 * 16 + 8];
            }
            #pragma unroll
            for (int k = 0; k < 8; ++k) {
                x[k] = __fsub_rn(__fmul_rn(a[k], c[k]), __fmul_rn(b[k], s[k]));
                y[k] = __fadd_rn(__fmul_rn(b[k], c[k]), __fmul_rn(a[k], s[k]));
            }
            p[0] = Vec<T>::store(x);
            p[8] = Vec<T>::store(y);
        }
    } else {
        for (; t < n; t += ROPE_THREADS) {
            const int i = t & 63;
            T* p = row + (t >> 6) * 128;
            const float a = (float)p[i], b = (float)p[i + 64];
            p[i] = (T)__fsub_rn(__fmul_rn(a, cs[i]), __fmul_rn(b, sn[i]));
            p[i + 64] = (T)__fadd_rn(__fmul_rn(b, cs[i]), __fmul_rn(a, sn[i]));
        }
    }
}

template <typename T>
cudaError_t launch_rope_typed(void* QK, int L, int ld, int heads, const int* pos, double theta, cudaStream_t stream) {
    RopeFreq f;
    for (int i = 0; i < 64; ++i) f.f[i] = (float)std::pow(theta, -(double)(2 * i) / 128.0);
    T* p = static_cast<T*>(QK);
    // 16-byte vectors need every row to start on a 16-byte boundary
    if (reinterpret_cast<uintptr_t>(QK) % 16 == 0 && ld % 8 == 0)
        rope_kernel<T, true><<<L, ROPE_THREADS, 0, stream>>>(p, ld, heads, pos, f);
    else
        rope_kernel<T, false><<<L, ROPE_THREADS, 0, stream>>>(p, ld, heads, pos, f);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_norm_typed(const void* X, const void* R, int L, int K, const float* w, float eps, void* h_out,
                              void* Y, cudaStream_t stream) {
    const T* x = static_cast<const T*>(X);
    const T* r = static_cast<const T*>(R);
    T* h = static_cast<T*>(h_out);
    T* y = static_cast<T*>(Y);
    const int nv = K / 8;
    if (nv <= NORM_THREADS * 4) add_rmsnorm_kernel<T, 4><<<L, NORM_THREADS, 0, stream>>>(x, r, K, w, eps, h, y);
    else add_rmsnorm_kernel<T, 20><<<L, NORM_THREADS, 0, stream>>>(x, r, K, w, eps, h, y);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_add_rmsnorm(const void* X, const void* R, int dtype, int L, int K, const float* w, float eps,
                               void* h_out, void* Y, cudaStream_t stream) {
    if (L == 0) return cudaSuccess;
    return dtype == STARQ_BF16 ? launch_norm_typed<__nv_bfloat16>(X, R, L, K, w, eps, h_out, Y, stream)
                               : launch_norm_typed<__half>(X, R, L, K, w, eps, h_out, Y, stream);
}

cudaError_t launch_rope(void* QK, int dtype, int L, int ld, int heads, const int* pos, double theta,
                        cudaStream_t stream) {
    if (L == 0) return cudaSuccess;
    return dtype == STARQ_BF16 ? launch_rope_typed<__nv_bfloat16>(QK, L, ld, heads, pos, theta, stream)
                               : launch_rope_typed<__half>(QK, L, ld, heads, pos, theta, stream);
}

}  // namespace starq
