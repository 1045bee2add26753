// SGAT activation transform + per-row symmetric int4 quantisation.
//
// Per row (a token for Q_a, an output channel for Q_w); Sec. 3.2 Eq. 11 with
// P = diag(a_s) H_hb, Sec. 3.1 Eq. 2:
//   v = fl32(x * a_s)                      state picked by the row's mask bit
//   v = v H_hb                             fast Walsh-Hadamard transform
//   v = v * gate_s                          binary subspace gate (Eq. 9)
//   v = fl32(v * post_scale)               1/hb on the weight side (Eq. 12)
//   amax = max |v|; s = amax / qmax; r = qmax / amax; q = rne(v * r)
// The transform is the butterfly network of the fast Walsh-Hadamard
// transform in stage order h = 1, 2, 4, ..., hb/2, each butterfly
// (a, b) -> (a + b, a - b) in float32 round-to-nearest; every float operation
// is an explicit round-to-nearest intrinsic, so nothing is contracted into an
// FMA and the values match the reference network bit for bit. With qmax = 7
// no clamp is needed: |fl(v * r)| <= 7 (1 + 2^-24)^2 < 7.5 (likewise 127.5
// for qmax = 127).
//
// Storage by code width. qmax <= 7 (4-bit): Xq packs two codes per byte and
// Xe holds each code as an E4M3 byte [rows][K]. qmax = 127 (8-bit, the W8A8
// setting of Tab. 5): Xq holds one code per byte (two's complement) and Xe
// [rows][K] each code as an fp16 number (exact: |c| <= 127), the operand of
// the 8-bit GEMM.
//
// Asymmetric mode (a.asym, Eq. 2-4, activations): per row X_max = max(max v,
// 0) and -X_min = max(max -v, 0); s = fl(fl(X_max - X_min) / qmax), r =
// fl(qmax / fl(X_max - X_min)), z = rne(fl(-X_min r)) in [0, qmax], codes
// clamp(rne(fl(v r)) + z, 0, qmax) (qmax = 15: unsigned nibbles in Xq, E4M3
// bytes in Xe, whose rows are K + 128 long and end in 128 bytes of E4M3(-z):
// with weight rows ending in E4M3 values that sum to sum_k q_w, the 4-bit
// GEMM over K + 128 then gives sum_k (q_a - z) q_w exactly).
//
// Two kernels. sgat_quant_rows_kernel (further down, with its layouts) takes
// rows of 1024 features and more, in multiples of 1024 (of 512 with blocks of
// at most 512). sgat_quant_kernel takes the other shapes:
//
// A warp owns a chunk of C = 32 E consecutive elements of a row
// (C = 1024 when hb >= 1024, else C = 512 holding 512 / hb Hadamard blocks).
// In layout A lane l holds elements E l .. E l + E - 1, so stages h < E are
// butterflies between registers of one thread. One transpose through shared
// memory (layout B: lane l holds elements l + 32 i) makes the stages
// 32 <= h < C register-local too; a transpose back gives each lane E
// contiguous values again. Stages h >= C (hb = 2048, 4096) pair chunks held
// by different warps of the row and exchange through shared memory.
//
// A row takes min(K / C, 8) warps, each keeping up to NC chunks in
// registers; short rows share a CTA of 8 warps. amax is reduced across a
// row's warps through shared memory.
#include "common.cuh"

namespace starq {
namespace {

template <typename T> struct In;
template <> struct In<__half> {
    template <int E>
    static __device__ __forceinline__ void load(const __half* p, float (&v)[E]) {
        const uint4* q = reinterpret_cast<const uint4*>(p);
        #pragma unroll
        for (int u = 0; u < E / 8; ++u) {
            uint4 w = __ldg(q + u);
            const __half2* h = reinterpret_cast<const __half2*>(&w);
            #pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 f = __half22float2(h[j]);
                v[8 * u + 2 * j] = f.x;
                v[8 * u + 2 * j + 1] = f.y;
            }
        }
    }
};
template <> struct In<__nv_bfloat16> {
    template <int E>
    static __device__ __forceinline__ void load(const __nv_bfloat16* p, float (&v)[E]) {
        const uint4* q = reinterpret_cast<const uint4*>(p);
        #pragma unroll
        for (int u = 0; u < E / 8; ++u) {
            uint4 w = __ldg(q + u);
            const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&w);
            #pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 f = __bfloat1622float2(h[j]);
                v[8 * u + 2 * j] = f.x;
                v[8 * u + 2 * j + 1] = f.y;
            }
        }
    }
};
template <> struct In<float> {
    template <int E>
    static __device__ __forceinline__ void load(const float* p, float (&v)[E]) {
        const float4* q = reinterpret_cast<const float4*>(p);
        #pragma unroll
        for (int u = 0; u < E / 4; ++u) {
            float4 w = __ldg(q + u);
            v[4 * u] = w.x; v[4 * u + 1] = w.y; v[4 * u + 2] = w.z; v[4 * u + 3] = w.w;
        }
    }
};

__device__ __forceinline__ void butterfly(float& lo, float& hi) {
    const float a = lo, b = hi;
    lo = __fadd_rn(a, b);
    hi = __fsub_rn(a, b);
}

// Butterflies between registers i and i + s for every i with (i & s) == 0,
// for s = s_lo, 2 s_lo, ... while s < s_end.
template <int E>
__device__ __forceinline__ void inlane_stages(float (&v)[E], int s_lo, int s_end) {
    #pragma unroll
    for (int s = 1; s < E; s <<= 1) {
        if (s >= s_lo && s < s_end) {
            #pragma unroll
            for (int i = 0; i < E; ++i)
                if ((i & s) == 0) butterfly(v[i], v[i + s]);
        }
    }
}

// Shared-buffer index of chunk element e: one padding float after every E
// elements. Layout A (lane stride E + 1, odd) and layout B (consecutive
// lanes, consecutive words) are then both free of bank conflicts, and every
// access is a per-lane base plus a compile-time offset.
template <int E>
__device__ __forceinline__ int pad_idx(int e) { return e + e / E; }

// Full transform of one chunk held in layout A; `buf` is this warp's
// 32 E-float shared buffer.
template <int E>
__device__ __forceinline__ void chunk_fwht(float (&v)[E], int hb, int lane, float* buf) {
    inlane_stages<E>(v, 1, hb < E ? hb : E);                  // h = 1 .. min(hb, E)/2
    if (hb <= E) return;
    if (E < 32) {                                            // h = E .. 16 across lanes
        #pragma unroll
        for (int h = E; h < 32; h <<= 1) {
            if (h < hb) {
                const int m = h / E;
                const float sgn = (lane & m) ? -1.f : 1.f;
                #pragma unroll
                for (int i = 0; i < E; ++i) {
                    const float o = __shfl_xor_sync(0xffffffffu, v[i], m);
                    // lower lane: v + o; upper lane: o - v (the product by -1 is exact)
                    v[i] = __fmaf_rn(sgn, v[i], o);
                }
            }
        }
    }
    if (hb <= 32) return;
    // layout A -> B
    float* a_base = buf + (E + 1) * lane;      // = buf + pad_idx(E * lane)
    #pragma unroll
    for (int i = 0; i < E; ++i) a_base[i] = v[i];
    __syncwarp();
    #pragma unroll
    for (int i = 0; i < E; ++i) v[i] = buf[pad_idx<E>(lane + 32 * i)];
    // stages h = max(E, 32) .. hb/2: register distance h / 32 in layout B
    inlane_stages<E>(v, (E > 32 ? E : 32) / 32, hb / 32);
    __syncwarp();
    #pragma unroll
    for (int i = 0; i < E; ++i) buf[pad_idx<E>(lane + 32 * i)] = v[i];
    __syncwarp();
    #pragma unroll
    for (int i = 0; i < E; ++i) v[i] = a_base[i];
    __syncwarp();
}

// Eight 8-bit codes -> their bytes (two's complement, code k in byte k) and
// the same codes as fp16 numbers (exact), code k in half k.
__device__ __forceinline__ void codes8(const int* q, uint2& bytes, uint4& f16) {
    uint32_t b0 = 0, b1 = 0;
    #pragma unroll
    for (int k = 0; k < 4; ++k) {
        b0 |= (uint32_t)(q[k] & 0xFF) << (8 * k);
        b1 |= (uint32_t)(q[k + 4] & 0xFF) << (8 * k);
    }
    bytes = make_uint2(b0, b1);
    uint32_t h[4];
    #pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __half2 p = __floats2half2_rn((float)q[2 * k], (float)q[2 * k + 1]);
        h[k] = *reinterpret_cast<const uint32_t*>(&p);
    }
    f16 = make_uint4(h[0], h[1], h[2], h[3]);
}

// Eight codes in [0, 15] -> E4M3 bytes (byte k = code k).
__device__ __forceinline__ uint2 e4m3_of8(const int* q) {
    uint16_t h[4];
    #pragma unroll
    for (int k = 0; k < 4; ++k)          // upper byte from the first operand
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(h[k]) : "f"((float)q[2 * k + 1]), "f"((float)q[2 * k]));
    return make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16));
}

// The zero-point columns of an asymmetric row: 128 bytes of E4M3(-z) after
// its K codes, eight threads of 16 bytes each (t = 0 .. 7).
__device__ __forceinline__ void store_zero_point_columns(uint8_t* row_end, int z, int t) {
    uint16_t h;
    const float m = (float)(-z);
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %1;" : "=h"(h) : "f"(m));
    const uint32_t w = (uint32_t)h | ((uint32_t)h << 16);
    reinterpret_cast<uint4*>(row_end)[t] = make_uint4(w, w, w, w);
}

// Eight codes (int, |q| <= 7) -> packed nibbles, code k in bits 4k..4k+3.
__device__ __forceinline__ uint32_t pack8(const int* q) {
    uint32_t w = 0;
    #pragma unroll
    for (int k = 0; k < 8; ++k) w |= (uint32_t)(q[k] & 0xF) << (4 * k);
    return w;
}

// Up to 8 warps per row, or up to 20 when hb <= C (E = 16, at most two
// chunks per warp; no stage crosses warps then).
template <int E, int NC, typename Tin>
__global__ void __launch_bounds__(E == 16 && NC <= 2 ? 640 : 256)
sgat_quant_kernel(QuantArgs a, int warps_per_row, int rows_per_cta) {
    extern __shared__ float qsm[];
    constexpr int C = 32 * E;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int wr = warp % warps_per_row;                 // warp index within its row
    const int row = blockIdx.x * rows_per_cta + warp / warps_per_row;
    float* buf = qsm + warp * (C + 32);
    float* red = qsm + (blockDim.x >> 5) * (C + 32);     // [32] partial amax, [32] partial -min
    const bool row_ok = row < a.L;
    const int K = a.K;
    const int nchunks = (K + C - 1) / C;   // a partial last chunk only when hb < 512

    const bool masked = row_ok && a.mask != nullptr && a.mask[row] != 0;
    const float* sm = masked ? a.a_m : a.a_u;
    // Active coordinates of the row's state (Eq. 9): masked rows keep
    // [0, d_sh + d_m), unmasked rows keep [0, d_sh) and [d_sh + d_m, K).
    const int own_lo = masked ? a.d_sh : a.d_sh + a.d_m;
    const int own_hi = masked ? a.d_sh + a.d_m : K;
    const Tin* X = static_cast<const Tin*>(a.X) + (size_t)(row_ok ? row : 0) * K;

    float v[NC][E];
    float amax = 0.f, nmin = 0.f;                        // asym: X_max and -X_min
    #pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int c = wr + j * warps_per_row;
        const int lo = c * C + E * lane;                 // first element of this lane
        // lanes lie wholly inside or outside the row: E | K when hb < 512
        const bool live = c < nchunks && row_ok && lo < K;
        if (live) {
            In<Tin>::template load<E>(X + lo, v[j]);
            if (sm != nullptr) {
                const float4* s4 = reinterpret_cast<const float4*>(sm + lo);
                #pragma unroll
                for (int u = 0; u < E / 4; ++u) {
                    const float4 w = __ldg(s4 + u);
                    v[j][4 * u] = __fmul_rn(v[j][4 * u], w.x);
                    v[j][4 * u + 1] = __fmul_rn(v[j][4 * u + 1], w.y);
                    v[j][4 * u + 2] = __fmul_rn(v[j][4 * u + 2], w.z);
                    v[j][4 * u + 3] = __fmul_rn(v[j][4 * u + 3], w.w);
                }
            }
        } else {
            #pragma unroll
            for (int i = 0; i < E; ++i) v[j][i] = 0.f;
        }
        if (c < nchunks) chunk_fwht<E>(v[j], a.hb, lane, buf);   // warp-uniform condition
        // Stages h = C .. hb/2 pair chunk c with chunk c ^ (h / C), held by
        // warp wr ^ (h / C) of the same row in the same round j (the warp
        // count of a row is a multiple of hb / C). Exchange in layout A
        // through the warps' padded buffers; all warps of the CTA take part.
        for (int m = 1; m * C < a.hb; m <<= 1) {
            float* mine = buf + (E + 1) * lane;
            const float* other = qsm + (warp ^ m) * (C + 32) + (E + 1) * lane;
            #pragma unroll
            for (int i = 0; i < E; ++i) mine[i] = v[j][i];
            __syncthreads();
            const bool upper = (wr & m) != 0;
            #pragma unroll
            for (int i = 0; i < E; ++i) {
                const float o = other[i];
                v[j][i] = upper ? __fsub_rn(o, v[j][i]) : __fadd_rn(v[j][i], o);
            }
            __syncthreads();
        }
        // gate: whole-lane decisions first, per element only where a lane
        // straddles a subspace boundary
        const bool all_keep = (lo + E <= a.d_sh) || (lo >= own_lo && lo + E <= own_hi);
        if (!all_keep) {
            #pragma unroll
            for (int i = 0; i < E; ++i) {
                const int e = lo + i;
                if (!(e < a.d_sh || (e >= own_lo && e < own_hi))) v[j][i] = 0.f;
            }
        }
        if (a.post_scale != 1.f) {
            #pragma unroll
            for (int i = 0; i < E; ++i) v[j][i] = __fmul_rn(v[j][i], a.post_scale);
        }
        if (a.asym) {
            #pragma unroll
            for (int i = 0; i < E; ++i) {
                amax = fmaxf(amax, v[j][i]);
                nmin = fmaxf(nmin, -v[j][i]);
            }
        } else {
            #pragma unroll
            for (int i = 0; i < E; ++i) amax = fmaxf(amax, fabsf(v[j][i]));
        }
        if (a.v_dbg != nullptr && live) {
            float4* d4 = reinterpret_cast<float4*>(a.v_dbg + (size_t)row * K + lo);
            #pragma unroll
            for (int u = 0; u < E / 4; ++u)
                d4[u] = make_float4(v[j][4 * u], v[j][4 * u + 1], v[j][4 * u + 2], v[j][4 * u + 3]);
        }
    }
    #pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, m));
        nmin = fmaxf(nmin, __shfl_xor_sync(0xffffffffu, nmin, m));
    }
    if (warps_per_row > 1) {
        if (lane == 0) {
            red[warp] = amax;
            red[32 + warp] = nmin;
        }
        __syncthreads();
        amax = 0.f;
        nmin = 0.f;
        const int first = warp - wr;                     // first warp of this row
        for (int w = 0; w < warps_per_row; ++w) {
            amax = fmaxf(amax, red[first + w]);
            nmin = fmaxf(nmin, red[32 + first + w]);
        }
    }
    if (!row_ok) return;

    const float qmax = (float)a.qmax;
    const float range = a.asym ? __fadd_rn(amax, nmin) : amax;     // X_max - X_min, or amax
    const bool nz = range > 0.f;
    const float s = nz ? __fdiv_rn(range, qmax) : 0.f;
    const float r = nz ? __fdiv_rn(qmax, range) : 0.f;
    const int zp = a.asym ? min(max(__float2int_rn(__fmul_rn(nmin, r)), 0), a.qmax) : 0;
    if (wr == 0 && lane == 0) {
        a.s[row] = s;
        if (a.asym) a.z[row] = zp;
    }
    if (a.asym && a.Xe != nullptr && wr == 0 && lane < 8)
        store_zero_point_columns(a.Xe + (size_t)row * (K + 128) + K, zp, lane);
    #pragma unroll
    for (int j = 0; j < NC; ++j) {
        const int c = wr + j * warps_per_row;
        const int lo = c * C + E * lane;
        if (c >= nchunks || lo >= K) continue;
        if (a.asym) {                    // codes in [0, qmax]: unsigned nibbles and E4M3 bytes
            #pragma unroll
            for (int u = 0; u < E / 8; ++u) {
                int q[8];
                #pragma unroll
                for (int k = 0; k < 8; ++k)
                    q[k] = min(max(__float2int_rn(__fmul_rn(v[j][8 * u + k], r)) + zp, 0), a.qmax);
                if (a.Xq != nullptr) *reinterpret_cast<uint32_t*>(a.Xq + (size_t)row * (K / 2) + lo / 2 + 4 * u) = pack8(q);
                if (a.Xe != nullptr) *reinterpret_cast<uint2*>(a.Xe + (size_t)row * (K + 128) + lo + 8 * u) = e4m3_of8(q);
            }
            continue;
        }
        if (a.qmax > 15) {               // 8-bit codes: bytes and fp16
            #pragma unroll
            for (int u = 0; u < E / 8; ++u) {
                int q[8];
                #pragma unroll
                for (int k = 0; k < 8; ++k) q[k] = __float2int_rn(__fmul_rn(v[j][8 * u + k], r));
                uint2 bytes;
                uint4 f16;
                codes8(q, bytes, f16);
                if (a.Xq != nullptr) *reinterpret_cast<uint2*>(a.Xq + (size_t)row * K + lo + 8 * u) = bytes;
                if (a.Xe != nullptr) *reinterpret_cast<uint4*>(a.Xe + ((size_t)row * K + lo + 8 * u) * 2) = f16;
            }
            continue;
        }
        uint32_t packed[E / 8];
        #pragma unroll
        for (int u = 0; u < E / 8; ++u) {
            int q[8];
            #pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = __float2int_rn(__fmul_rn(v[j][8 * u + k], r));
            packed[u] = pack8(q);
        }
        uint8_t* dst = a.Xq + (size_t)row * (K / 2) + lo / 2;
        if (a.Xq == nullptr) {
        } else if (E == 16) {
            *reinterpret_cast<uint2*>(dst) = make_uint2(packed[0], packed[1]);
        } else {
            #pragma unroll
            for (int u = 0; u < E / 32; ++u)
                reinterpret_cast<uint4*>(dst)[u] =
                    make_uint4(packed[4 * u], packed[4 * u + 1], packed[4 * u + 2], packed[4 * u + 3]);
        }
        if (a.Xe != nullptr) {   // E4M3 bytes of the same codes
            uint4* e4 = reinterpret_cast<uint4*>(a.Xe + (size_t)row * K + lo);
            #pragma unroll
            for (int u = 0; u < E / 16; ++u) {
                uint32_t o[4];
                int4x8_to_e4m3x8(packed[2 * u], o[0], o[1]);
                int4x8_to_e4m3x8(packed[2 * u + 1], o[2], o[3]);
                e4[u] = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    }
}

template <typename T> struct To;
template <> struct To<__half> { static __device__ __forceinline__ float f(__half h) { return __half2float(h); } };
template <> struct To<__nv_bfloat16> { static __device__ __forceinline__ float f(__nv_bfloat16 h) { return __bfloat162float(h); } };
template <> struct To<float> { static __device__ __forceinline__ float f(float h) { return h; } };

// ---------------------------------------------------------------------------
// Rows with Hadamard blocks of 1024 elements or more (hb >= 1024, K a
// multiple of 1024), or of at most 512 (K >= 1024, K % 512 == 0, a last chunk
// of 512 allowed): one CTA of four warps per 4096-element slice of a row, a
// 1024-element chunk per warp (element e of the chunk: bits 0 .. 9). Each
// layout keeps five element bits in a thread's 32 registers, so that the
// stages over those bits are between registers:
//
//   layout 1  bits 0, 1, 7, 8, 9 (register 4 q + k: element 4 l + 128 q + k of
//             lane l): the layout of the loads -- x and the smoothing vector
//             meet as they arrive, 8 or 16 bytes per lane -- and of the codes.
//             Stages h = 1, 2, and after layout 2 h = 128, 256, 512;
//   layout 2  bits 2 .. 6 (register i: element (l & 3) + 4 i + 128 (l >> 2)):
//             stages h = 4 .. 64;
//   layout 3  hb > 1024 only: bits 0, 1, 7 and the chunk number (register
//             8 j + 4 q + k: element 256 w + 128 q + 4 l + k of chunk j for
//             lane l of warp w): stages h = 1024, 2048. With blocks of 2048 a
//             pair of chunks is exchanged between its own two warps (bits 0,
//             1, 7, 8 and the chunk's), so that of rows of 2048 the other two
//             stay idle.
//
// The layouts change through the warp's own slice of shared memory, eight
// rows (q) of 128 floats padded to 132: the 16-byte accesses of layouts 1 and
// 3 and the 4-byte accesses of layout 2 are all free of bank conflicts, and
// every address is a per-thread base plus a constant. Only layout 3 and the
// row maximum need the whole CTA.
//
// Bound by instruction issue and shared-memory wavefronts (64% and 78% busy at
// 8192 x 4096), not by HBM. An earlier split (32 consecutive elements per lane
// first, then two more layouts) staged x and the smoothing vector through shared
// memory to reach its first layout: 224 wavefronts per 1024 elements instead of
// 128 (192 with layout 3), and 1141 warp instructions instead of 859, or 789 with
// FULL (1349 for the present split while the Hadamard block was known only at
// run time: the branches around the stages keep the register pairs apart).
// Microseconds back to back, the earlier split and now, one box: 8192 x 4096
// fp16, hb 4096 42.8, 33.4; 8192 x 3584 bf16, hb 512 39.6, 29.2; 8192 x 18944
// 244, 168.6; 1024 x 12288 23.4, 17.7; 1024 x 4096 8.2, 6.5; codes of 24576 x 4096
// weights 120.2, 92.4; asymmetric 8192 x 4096 47.3, 39.7 (another box). Rows
// shorter than a slice, whose warps without a chunk leave before the codes:
// 8192 x 1024 22.3, 18.6; 8192 x 2048 29.0, 24.5 (with the idle warps going on,
// 24.7 and 33.2).
// Butterflies on pairs of registers use the packed f32x2 add and subtract
// (each half rounds like the scalar operation).
// ---------------------------------------------------------------------------
constexpr int MAX_SLICES = 5;                              // K <= 20480
constexpr int QROW = 132;                                  // floats per 128-element row of a slice
constexpr int SLICE = 8 * QROW;                            // floats per slice

using f32x2 = unsigned long long;                          // two float32 in a register pair
__device__ __forceinline__ f32x2 pack2f(float lo, float hi) {
    f32x2 p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(lo), "f"(hi));
    return p;
}
__device__ __forceinline__ void unpack2f(f32x2 p, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}
__device__ __forceinline__ void butterfly2(f32x2& a, f32x2& b) {
    f32x2 s, d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(a), "l"(b));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    a = s;
    b = d;
}

// In-register stages of 32 values (pair i: registers 2 i, 2 i + 1) for the
// register distances s = s_lo .. s_end / 2 (s = 1 scalar, s >= 2 packed).
__device__ __forceinline__ void reg_stages32(f32x2 (&p)[16], int s_lo, int s_end) {
    if (s_lo <= 1 && 1 < s_end) {
        #pragma unroll
        for (int i = 0; i < 16; ++i) {
            float x, y;
            unpack2f(p[i], x, y);
            butterfly(x, y);
            p[i] = pack2f(x, y);
        }
    }
    #pragma unroll
    for (int s = 2; s < 32; s <<= 1) {
        if (s >= s_lo && s < s_end) {
            #pragma unroll
            for (int i = 0; i < 16; ++i)
                if ((i & (s / 2)) == 0) butterfly2(p[i], p[i + s / 2]);
        }
    }
}

// Codes of two values: q = rne(fl(v * r)). The product is a scalar
// round-to-nearest multiply (never contracted: a fused multiply-add would
// round the exact product and break ties differently). Adding M = 1.5 * 2^23
// then rounds it to an integer in one step (floats in [2^23, 2^24) are the
// integers, ties to even), fl(t - M) is that integer as a float (+0 for
// zero), and the low mantissa bits of t are the integer itself.
__device__ __forceinline__ void quant_pair(float v0, float v1, float r, float& q0, float& q1, int& i0, int& i1) {
    const float p0 = __fmul_rn(v0, r), p1 = __fmul_rn(v1, r);
    asm("{\n\t.reg .b64 V, M, T;\n\t"
        "mov.b64 V, {%4, %5};\n\t"
        "mov.b64 M, {%6, %6};\n\t"
        "add.rn.f32x2 T, V, M;\n\t"
        "sub.rn.f32x2 V, T, M;\n\t"
        "mov.b64 {%0, %1}, V;\n\t"
        "mov.b64 {%2, %3}, T;\n\t}"
        : "=f"(q0), "=f"(q1), "=r"(i0), "=r"(i1) : "f"(p0), "f"(p1), "f"(12582912.0f));
    i0 -= 0x4B400000;
    i1 -= 0x4B400000;
}

// Four codes (ints) -> packed nibbles in the low 16 bits, code k in bits 4k ..
// 4k + 3. Saturating: where the reciprocal scale or a product is infinite the
// integer is far out of range, and its low bits alone would be any code.
__device__ __forceinline__ uint16_t pack_nibbles4(const int* q) {
    uint32_t w = 0;
    #pragma unroll
    for (int k = 2; k >= 0; k -= 2)      // d = c << 8 | sat4(a) << 4 | sat4(b)
        asm("cvt.pack.sat.s4.s32.b32 %0, %1, %2, %0;" : "+r"(w) : "r"(q[k + 1]), "r"(q[k]));
    return (uint16_t)w;
}

// Four codes (floats) -> their E4M3 bytes (byte k = code k).
__device__ __forceinline__ uint32_t e4m3_bytes4(const float* qf) {
    uint16_t h[2];
    #pragma unroll
    for (int k = 0; k < 2; ++k)          // upper byte from the first operand
        asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(h[k]) : "f"(qf[2 * k + 1]), "f"(qf[2 * k]));
    return (uint32_t)h[0] | ((uint32_t)h[1] << 16);
}

// Four consecutive elements of a row as loaded, and as float32.
template <typename T> struct Raw4 { using V = uint2; };
template <> struct Raw4<float> { using V = float4; };
template <typename T>
__device__ __forceinline__ void raw4_to_f(const uint2& w, float* f) {
    const T* h = reinterpret_cast<const T*>(&w);
    #pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = To<T>::f(h[k]);
}
template <typename T>
__device__ __forceinline__ void raw4_to_f(const float4& w, float* f) {
    f[0] = w.x; f[1] = w.y; f[2] = w.z; f[3] = w.w;
}

// HB: the Hadamard block when it is known at compile time (no branch around
// any stage), or 0 to take it from the arguments. ASYM: the asymmetric mode (a
// compile-time copy, so that the symmetric kernel carries none of its
// reductions). CLUSTER: a cluster of CTAs per row, CTA r taking the row's
// features 4096 r .. 4096 r + 4095; the CTAs exchange their maxima through
// distributed shared memory, so no thread holds more than one 4096-feature
// slice.
// G2: rows a0.L .. a0.L + b.L - 1 of the grid quantise problem b (the same
// K, hb, input type and code width; its own X, mask, transform and outputs):
// two quantisations in one launch.
// FULL (HB 4096): every slice is whole, so no test for missing chunks. Alone it
// is the shorter code, but its schedule loses in a single wave of CTAs (1024 x
// 4096: 6.9 us against 6.4), so only launches of several waves take it (8192 x
// 4096: 33.2 against 35.1; 1024 x 12288 17.6, 18.0).
// CTAs per SM: seven (72 registers); eight (64, no spills for 16-bit inputs)
// with FULL, and for clustered rows with blocks of 512 (8192 x 18944: 166 us
// against 176, both ahead of the barrier that the cluster's start needs), but not in a single wave (1000 x 3584: 5.7 against 5.3).
template <typename Tin, int HB, bool ASYM, bool CLUSTER, bool G2, bool FULL = false>
__global__ void __launch_bounds__(128, FULL || (HB == 512 && CLUSTER) ? 8 : 7)
sgat_quant_rows_kernel(QuantArgs a0, QuantArgs b, int ctas_per_row) {
    static_assert(!G2 || !CLUSTER, "grouped launches run one CTA per row");
    using Raw = typename Raw4<Tin>::V;
    const bool p1 = G2 && (int)blockIdx.x >= a0.L;
    const QuantArgs& a = p1 ? b : a0;
    __shared__ __align__(16) float buf[4 * SLICE];
    __shared__ float red[8];              // [0, 4) amax or X_max, [4, 8) -X_min (asym)
    __shared__ float cl_red[2][MAX_SLICES];   // the maxima (and -minima) of the row's slices
    if (CLUSTER) cluster_started_arrive();    // waited for ahead of the exchange of the maxima
    // launched with programmatic serialisation: the rows of a problem whose
    // caller vouches that the preceding launch neither writes its inputs
    // nor touches its outputs start without waiting for that launch
    if (!a.independent) grid_dependency_wait();
    grid_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int rank = CLUSTER ? (int)cluster_ctarank() : 0;
    const int row = CLUSTER ? (int)blockIdx.x / ctas_per_row : (int)blockIdx.x - (p1 ? a0.L : 0);
    const int K = a.K, hb = HB > 0 ? HB : a.hb;
    const bool masked = a.mask != nullptr && a.mask[row] != 0;
    const float* sm = masked ? a.a_m : a.a_u;
    const Tin* X = static_cast<const Tin*>(a.X) + (size_t)row * K;
    const int base = rank * 4096;
    const int c0 = base + warp * 1024;                           // first element of the warp's chunk
    // a slice may end early, with a last chunk of 512 whose upper half is zeros, never stored
    const bool live = FULL || c0 < K;
    const bool half = !FULL && K - c0 < 1024;
    float* own = buf + warp * SLICE + 4 * lane;                  // layout 1: row q at own + QROW q
    float* tr = buf + warp * SLICE + (lane & 3) + QROW * (lane >> 2);   // layout 2: register i at tr + 4 i

    f32x2 p[16];
    auto put_own = [&]() {                                       // layout 1 -> the warp's slice
        #pragma unroll
        for (int q = 0; q < 8; ++q)
            *reinterpret_cast<ulonglong2*>(own + QROW * q) = make_ulonglong2(p[2 * q], p[2 * q + 1]);
    };
    if (live) {
        Raw xr[8];
        float4 sr[8];
        const Raw* x4 = reinterpret_cast<const Raw*>(X + c0) + lane;
        #pragma unroll
        for (int q = 0; q < 8; ++q) {
            xr[q] = Raw();
            if (!half || q < 4) xr[q] = __ldg(x4 + 32 * q);
        }
        if (sm != nullptr) {
            const float4* s4 = reinterpret_cast<const float4*>(sm + c0) + lane;
            #pragma unroll
            for (int q = 0; q < 8; ++q)
                sr[q] = (!half || q < 4) ? __ldg(s4 + 32 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            #pragma unroll
            for (int q = 0; q < 8; ++q) sr[q] = make_float4(1.f, 1.f, 1.f, 1.f);   // x * 1 = x
        }
        #pragma unroll
        for (int q = 0; q < 8; ++q) {
            float f[4];
            raw4_to_f<Tin>(xr[q], f);
            p[2 * q] = pack2f(__fmul_rn(f[0], sr[q].x), __fmul_rn(f[1], sr[q].y));
            p[2 * q + 1] = pack2f(__fmul_rn(f[2], sr[q].z), __fmul_rn(f[3], sr[q].w));
        }
        reg_stages32(p, 1, hb < 4 ? hb : 4);                     // h = 1, 2
        if (hb > 4) {
            put_own();                                           // layout 1 -> 2
            __syncwarp();
            #pragma unroll
            for (int i = 0; i < 16; ++i) p[i] = pack2f(tr[8 * i], tr[8 * i + 4]);
            reg_stages32(p, 1, hb / 4);                          // h = 4 .. min(hb, 128) / 2
            #pragma unroll
            for (int i = 0; i < 16; ++i) unpack2f(p[i], tr[8 * i], tr[8 * i + 4]);   // layout 2 -> 1
            __syncwarp();
            #pragma unroll
            for (int q = 0; q < 8; ++q) {
                const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(own + QROW * q);
                p[2 * q] = w.x;
                p[2 * q + 1] = w.y;
            }
            reg_stages32(p, 4, hb / 32);                         // h = 128 .. min(hb, 1024) / 2
        }
    } else {
        #pragma unroll
        for (int i = 0; i < 16; ++i) p[i] = 0;
    }
    // group g of four registers: elements e_base + (g >> 1) e_step + 128 (g & 1) ..
    int e_base = c0 + 4 * lane, e_step = 256;
    if (HB == 2048) {                                            // layout 1 -> 3, two chunks (K is a multiple of 2048)
        e_base = base + 2048 * (warp >> 1) + 512 * (warp & 1) + 4 * lane;
        if (live) put_own();
        __syncthreads();
        if (live) {
            #pragma unroll
            for (int g = 0; g < 8; ++g) {
                const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(
                    buf + (2 * (warp >> 1) + (g >> 2)) * SLICE + QROW * (4 * (warp & 1) + (g & 3)) + 4 * lane);
                p[2 * g] = w.x;
                p[2 * g + 1] = w.y;
            }
            reg_stages32(p, 16, 32);                             // h = 1024
        }
    } else if (hb > 1024) {                                      // layout 1 -> 3
        e_base = base + warp * 256 + 4 * lane;
        e_step = 1024;
        if (live) put_own();
        __syncthreads();
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            ulonglong2 w = make_ulonglong2(0, 0);
            if (FULL || base + (g >> 1) * 1024 < K)              // chunk g >> 1 exists
                w = *reinterpret_cast<const ulonglong2*>(buf + (g >> 1) * SLICE + QROW * (2 * warp + (g & 1)) +
                                                         4 * lane);
            p[2 * g] = w.x;
            p[2 * g + 1] = w.y;
        }
        reg_stages32(p, 8, hb / 128);                            // h = 1024, 2048
    }
    auto first = [&](int g) {                                    // element of group g
        return HB == 2048 ? e_base + (g >> 2) * 1024 + (g & 3) * 128 : e_base + (g >> 1) * e_step + (g & 1) * 128;
    };
    auto inside = [&](int g) { return FULL || first(g) < K; };
    // a warp without a chunk has nothing to quantise unless layout 3 gives it a
    // part of the others' (of rows of 1024 three warps in four are idle)
    const bool idle = HB != 4096 && !live && (hb <= 1024 || HB == 2048);
    float v[32];
    #pragma unroll
    for (int i = 0; i < 16; ++i) unpack2f(p[i], v[2 * i], v[2 * i + 1]);
    if (!idle && first(7) + 4 > a.d_sh) {          // the lane reaches past the shared coordinates: the gate
        const int own_lo = masked ? a.d_sh : a.d_sh + a.d_m;
        const int own_hi = masked ? a.d_sh + a.d_m : K;
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            const int e0 = first(g);
            #pragma unroll
            for (int k = 0; k < 4; ++k)
                if (e0 + k >= a.d_sh && (e0 + k < own_lo || e0 + k >= own_hi)) v[4 * g + k] = 0.f;
        }
    }
    if (a.post_scale != 1.f) {
        #pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __fmul_rn(v[i], a.post_scale);
    }
    if (a.v_dbg != nullptr) {
        #pragma unroll
        for (int g = 0; g < 8; ++g)
            if (inside(g))
                *reinterpret_cast<float4*>(a.v_dbg + (size_t)row * K + first(g)) =
                    make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
    }
    // (values past the row's end are zeros)
    float amax = 0.f, nmin = 0.f;         // asym: X_max and -X_min
    #pragma unroll
    for (int i = 0; i < 32; ++i) {
        if (ASYM) {
            amax = fmaxf(amax, v[i]);
            nmin = fmaxf(nmin, -v[i]);
        } else {
            amax = fmaxf(amax, fabsf(v[i]));
        }
    }
    #pragma unroll
    for (int m = 16; m > 0; m >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, m));
    if (ASYM) {
        #pragma unroll
        for (int m = 16; m > 0; m >>= 1) nmin = fmaxf(nmin, __shfl_xor_sync(0xffffffffu, nmin, m));
    }
    if (lane == 0) {
        red[warp] = amax;
        if (ASYM) red[4 + warp] = nmin;
    }
    __syncthreads();
    amax = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
    if (ASYM) nmin = fmaxf(fmaxf(red[4], red[5]), fmaxf(red[6], red[7]));
    if (CLUSTER) {
        // the row's maximum over the cluster's slices: every CTA writes its
        // own into all of them, once all have started, so that after the
        // second barrier nobody reads another CTA's memory and each may finish
        // by itself
        cluster_started_wait();
        if ((int)threadIdx.x < ctas_per_row) {
            st_shared_cluster_f32(mapa_shared(smem_addr(&cl_red[0][rank]), threadIdx.x), amax);
            if (ASYM) st_shared_cluster_f32(mapa_shared(smem_addr(&cl_red[1][rank]), threadIdx.x), nmin);
        }
        __syncwarp();
        cluster_sync();
        for (int c = 0; c < ctas_per_row; ++c) {
            amax = fmaxf(amax, cl_red[0][c]);
            if (ASYM) nmin = fmaxf(nmin, cl_red[1][c]);
        }
    }

    const float qmax = (float)a.qmax;
    const float range = ASYM ? __fadd_rn(amax, nmin) : amax;     // X_max - X_min, or amax
    const bool nz = range > 0.f;
    const float s = nz ? __fdiv_rn(range, qmax) : 0.f;
    const float r = nz ? __fdiv_rn(qmax, range) : 0.f;
    const int zp = ASYM ? min(max(__float2int_rn(__fmul_rn(nmin, r)), 0), a.qmax) : 0;
    if (threadIdx.x == 0 && rank == 0) {
        a.s[row] = s;
        if (ASYM) a.z[row] = zp;
    }
    if (ASYM && a.Xe != nullptr && threadIdx.x < 8 && rank == 0)
        store_zero_point_columns(a.Xe + (size_t)row * (K + 128) + K, zp, threadIdx.x);
    // codes of group g, as integers and as floats
    auto codes = [&](int g, float (&qf)[4], int (&qi)[4]) {
        quant_pair(v[4 * g], v[4 * g + 1], r, qf[0], qf[1], qi[0], qi[1]);
        quant_pair(v[4 * g + 2], v[4 * g + 3], r, qf[2], qf[3], qi[2], qi[3]);
        if (ASYM) {
            #pragma unroll
            for (int k = 0; k < 4; ++k) {
                qi[k] = min(max(qi[k] + zp, 0), a.qmax);
                qf[k] = (float)qi[k];
            }
        }
    };
    if (idle) return;                                            // (no barrier follows)
    if (ASYM) {                                                  // E4M3 bytes and unsigned nibbles, the codes once
        uint8_t* e4 = a.Xe == nullptr ? nullptr : a.Xe + (size_t)row * (K + 128);
        uint8_t* nib = a.Xq == nullptr ? nullptr : a.Xq + (size_t)row * (K / 2);
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            if (HB != 4096 && HB != 2048 && !inside(g)) continue;    // (warp-uniform)
            float qf[4];
            int qi[4];
            codes(g, qf, qi);
            if (e4 != nullptr) *reinterpret_cast<uint32_t*>(e4 + first(g)) = e4m3_bytes4(qf);
            if (nib != nullptr)
                *reinterpret_cast<uint16_t*>(nib + first(g) / 2) =
                    (uint16_t)(qi[0] | qi[1] << 4 | qi[2] << 8 | qi[3] << 12);
        }
        return;
    }
    const bool wide = a.qmax > 15;                               // 8-bit codes: fp16 and bytes
    if (a.Xe != nullptr && wide) {
        uint8_t* dst = a.Xe + (size_t)row * K * 2;
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            float qf[4];
            int qi[4];
            codes(g, qf, qi);
            const __half2 h0 = __floats2half2_rn(qf[0], qf[1]), h1 = __floats2half2_rn(qf[2], qf[3]);
            if (inside(g))
                *reinterpret_cast<uint2*>(dst + 2 * first(g)) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
        }
    } else if (a.Xe != nullptr) {                                // E4M3 bytes
        uint8_t* dst = a.Xe + (size_t)row * K;
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            float qf[4];
            int qi[4];
            codes(g, qf, qi);
            if (inside(g)) *reinterpret_cast<uint32_t*>(dst + first(g)) = e4m3_bytes4(qf);
        }
    }
    if (a.Xq != nullptr) {
        uint8_t* dst = a.Xq + (size_t)row * (wide ? K : K / 2);
        #pragma unroll
        for (int g = 0; g < 8; ++g) {
            float qf[4];
            int qi[4];
            codes(g, qf, qi);
            if (!inside(g)) continue;
            if (wide)
                *reinterpret_cast<uint32_t*>(dst + first(g)) =
                    prmt(prmt((uint32_t)qi[0], (uint32_t)qi[1], 0x0040u),
                         prmt((uint32_t)qi[2], (uint32_t)qi[3], 0x0040u), 0x5410u);
            else
                *reinterpret_cast<uint16_t*>(dst + first(g) / 2) = pack_nibbles4(qi);
        }
    }
}

// One launch of the row kernel: a CTA per row (b != nullptr: the rows of b
// after those of a), or beyond 4096 features a cluster of CTAs per row, one
// 4096-feature slice each. Blocks of 512 to 4096 are compiled in (8192 x 4096,
// hb 1024: 30.2 us, against 33.9 with the block at run time); grouped launches,
// only 512 and 4096.
template <typename Tin, bool ASYM, bool CLUSTER, bool G2>
cudaError_t launch_rows_kind(const QuantArgs& a, const QuantArgs& b, cudaStream_t stream) {
    const int ctas = (a.K + 4095) / 4096;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0] = pdl_attribute();
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = ctas;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3(CLUSTER ? (unsigned)a.L * ctas : (unsigned)(a.L + (G2 ? b.L : 0)));
    cfg.blockDim = dim3(128);
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = CLUSTER ? 2 : 1;
    if (a.hb == 4096) {                  // (K is a multiple of 4096)
        if constexpr (!G2) {
            if (a.L * ctas > 7 * num_sms())
                return cudaLaunchKernelEx(&cfg, sgat_quant_rows_kernel<Tin, 4096, ASYM, CLUSTER, G2, true>, a, b, ctas);
        }
        return cudaLaunchKernelEx(&cfg, sgat_quant_rows_kernel<Tin, 4096, ASYM, CLUSTER, G2>, a, b, ctas);
    }
    if (a.hb == 512) return cudaLaunchKernelEx(&cfg, sgat_quant_rows_kernel<Tin, 512, ASYM, CLUSTER, G2>, a, b, ctas);
    if constexpr (!G2) {
        switch (a.hb) {
            case 1024: return cudaLaunchKernelEx(&cfg, sgat_quant_rows_kernel<Tin, 1024, ASYM, CLUSTER, G2>, a, b, ctas);
            case 2048: return cudaLaunchKernelEx(&cfg, sgat_quant_rows_kernel<Tin, 2048, ASYM, CLUSTER, G2>, a, b, ctas);
            default: break;
        }
    }
    return cudaLaunchKernelEx(&cfg, sgat_quant_rows_kernel<Tin, 0, ASYM, CLUSTER, G2>, a, b, ctas);
}

template <typename Tin>
cudaError_t launch_rows_grouped(const QuantArgs& a, const QuantArgs& b, cudaStream_t stream) {
    return launch_rows_kind<Tin, false, false, true>(a, b, stream);
}

template <typename Tin>
cudaError_t launch_rows(const QuantArgs& a, cudaStream_t stream) {
    if (a.K > 4096)
        return a.asym ? launch_rows_kind<Tin, true, true, false>(a, a, stream)
                      : launch_rows_kind<Tin, false, true, false>(a, a, stream);
    return a.asym ? launch_rows_kind<Tin, true, false, false>(a, a, stream)
                  : launch_rows_kind<Tin, false, false, false>(a, a, stream);
}

template <int E, typename Tin>
cudaError_t launch_e(const QuantArgs& a, cudaStream_t stream) {
    constexpr int C = 32 * E;
    const int n = (a.K + C - 1) / C;                 // chunks per row
    int wpr, nc;                                     // warps per row, rounds
    if (E == 16 && a.hb <= C && n > 8) {             // no stage crosses warps: up to 20 warps, 2 rounds
        nc = (n + 19) / 20;
        wpr = (n + nc - 1) / nc;
    } else {
        wpr = n < 8 ? n : 8;                         // a multiple of hb / C
        nc = (n + wpr - 1) / wpr;
    }
    const int rpc = wpr <= 4 ? 8 / wpr : 1;          // rows per CTA
    const int warps = wpr * rpc;
    const size_t smem = (size_t)warps * (C + 32) * 4 + 64 * 4;
    dim3 grid((a.L + rpc - 1) / rpc), block(32 * warps);
    #define STARQ_QUANT_LAUNCH(NCV)                                                            \
        {                                                                                      \
            static DeviceCache<int> attr;                                                      \
            int done = 0;                                                                      \
            const cudaError_t e = attr.get(&done, [](int, int* v) {                            \
                *v = 1;                                                                        \
                return cudaFuncSetAttribute(sgat_quant_kernel<E, NCV, Tin>,                    \
                        cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);              \
            });                                                                                \
            if (e != cudaSuccess) return e;                                                    \
            sgat_quant_kernel<E, NCV, Tin><<<grid, block, smem, stream>>>(a, wpr, rpc);        \
        }
    switch (nc) {
        case 1: STARQ_QUANT_LAUNCH(1); break;
        case 2: STARQ_QUANT_LAUNCH(2); break;
        case 3: STARQ_QUANT_LAUNCH(3); break;
        case 4: STARQ_QUANT_LAUNCH(4); break;
        case 5: if constexpr (E <= 16) STARQ_QUANT_LAUNCH(5); break;
        default: return cudaErrorInvalidValue;
    }
    #undef STARQ_QUANT_LAUNCH
    return cudaGetLastError();
}

template <typename Tin>
cudaError_t launch_typed(const QuantArgs& a, cudaStream_t stream) {
    // otherwise a warp's chunk is 1024 elements (hb >= 1024, blocks finish
    // across warps) or 512 elements holding 512 / hb blocks
    // up to 20480 features in 4096-feature slices (a cluster of CTAs per row
    // beyond 4096): blocks of 1024 or more with K % 1024 == 0, or of up to
    // 512 with K % 512 == 0 (a last chunk of 512 allowed)
    if (a.K <= 20480 && ((a.hb >= 1024 && a.K % 1024 == 0) || (a.hb <= 512 && a.K >= 1024 && a.K % 512 == 0)))
        return launch_rows<Tin>(a, stream);
    return a.hb >= 1024 ? launch_e<32, Tin>(a, stream) : launch_e<16, Tin>(a, stream);
}

}  // namespace

cudaError_t launch_sgat_quant(const QuantArgs& a, cudaStream_t stream) {
    if (a.L == 0) return cudaSuccess;
    switch (a.x_dtype) {
        case STARQ_F16: return launch_typed<__half>(a, stream);
        case STARQ_BF16: return launch_typed<__nv_bfloat16>(a, stream);
        case STARQ_F32: return launch_typed<float>(a, stream);
        default: return cudaErrorInvalidValue;
    }
}

// Whether the row kernel with one CTA per row takes this problem.
static bool rows_one_cta(const QuantArgs& a) {
    return !a.asym && a.K <= 4096 &&
           ((a.hb >= 1024 && a.K % 1024 == 0) || (a.hb <= 512 && a.K >= 1024 && a.K % 512 == 0));
}

cudaError_t launch_sgat_quant_grouped(const QuantArgs& a, const QuantArgs& b, cudaStream_t stream) {
    const bool same = a.x_dtype == b.x_dtype && a.K == b.K && a.hb == b.hb && a.qmax == b.qmax &&
                      a.post_scale == b.post_scale && rows_one_cta(a) && rows_one_cta(b);
    if (!same || a.L == 0 || b.L == 0) {             // two launches
        cudaError_t e = launch_sgat_quant(a, stream);
        return e != cudaSuccess ? e : launch_sgat_quant(b, stream);
    }
    switch (a.x_dtype) {
        case STARQ_F16: return launch_rows_grouped<__half>(a, b, stream);
        case STARQ_BF16: return launch_rows_grouped<__nv_bfloat16>(a, b, stream);
        case STARQ_F32: return launch_rows_grouped<float>(a, b, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace starq
