// GEMM for few tokens (one block of a semi-autoregressive decode, the tail of a
// batch): the same products and dequantisation as the pair kernel of
// w4a4_gemm.cu,
//   acc[i][n] = sum_k qa[i][k] qw[n][k]        exact integer sums
//   Y[i][n]   = fl(fl(acc * s_a[i]) * s_w[n]) (+ bias[n]) -> output type
// with 4-bit codes as E4M3, 8-bit codes as fp16, or plain 16-bit operands
// (float32 sums, no scales), organised around the weight stream.
//
// With few tokens the floor is reading the weights' N K bytes from HBM once,
// and what matters is how many of them are in flight on how many SMs. The
// 256-token pair tiles of w4a4_gemm.cu give ceil(N / 224) pairs, each walking
// the whole K chain alone: 110 of 152 SMs at N = 12288, 38 at N = 4096. Here
// the operands trade places: 128 weight rows are the M of the MMA and the
// tokens (16, 32, 64 or 128 rows) its N, one CTA per (128-channel tile, part of
// K), two CTAs per SM with ~100 KB of tiles in flight each. The S parts of K of
// one tile are a cluster: every CTA sends its partial sums (for codes integers,
// exact, so their order does not matter) of token t to part t mod S through
// distributed shared memory, a 128-byte line per warp and token, and each
// part adds up and dequantises its own tokens. (Reading the other parts' sums
// instead, 16-byte remote stores by token groups, and bulk copies between the
// shared memories were 1 to 6 us slower at 64 tokens.)
//
//   warp 4    TMA: weight and token tiles of 128 K through a ring of stages
//             (the weights of the first stages ahead of the wait for the
//             previous kernel when the caller vouches for them);
//   warp 5    TMEM allocation, MMA issue (tcgen05 kind::f8f6f4, M 128, N NT);
//   warps 0-3 accumulator to the parts that own the tokens, their sums,
//             dequantisation, stores.
// Every wait is bounded; a CTA that gives up records it in the status word,
// takes part in the cluster barriers all the same, stores nothing and leaves
// only when the tiles it has asked for have landed.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "common.cuh"

namespace starq {
namespace {

namespace fewk {
constexpr int BM = 128, BK = 128, UMMA_K = 32;           // weight rows per tile, K bytes per stage
constexpr int A_BYTES = BM * BK;
constexpr int NUM_EPI_WARPS = 4, TMA_WARP = 4, MMA_WARP = 5;
constexpr int THREADS = 6 * 32;
constexpr int MAX_SPLIT = 8;                             // portable cluster size
// OPK: operand kind, as in w4a4_gemm.cu -- 0 E4M3 codes, 1 fp16, 2 bf16 (plain
// products, no scales), 3 8-bit codes held as fp16. A stage is 128 bytes of K
// either way. Kind 3: an accumulator takes at most 16 stages (1024 K, integers
// up to 1024 * 127^2 < 2^24, exact in float32); ACCS of them lie side by side in
// TMEM and are summed in int32.
constexpr int ACC_STAGES = 16;
template <int NT, int OPK, int ACCS>
struct Tile {
    static_assert(NT % 16 == 0 && NT >= 16 && NT <= 128, "tokens per tile (MMA N)");
    static constexpr int STAGE_BYTES = A_BYTES + NT * BK;
    // the sums, over the stages once they are read: split * ceil(NT / split) rows of 128 channels
    static constexpr int PART_BYTES = (NT + MAX_SPLIT - 1) * BM * 4;
    static constexpr int FIXED = 1024 + 256;             // alignment, barriers
    // two CTAs per SM: 113.5 KB each (227 KB less 1 KB per CTA of the system's)
    static constexpr int STAGES = (112 * 1024 - FIXED) / STAGE_BYTES;
    static constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + FIXED;
    static_assert(PART_BYTES <= STAGES * STAGE_BYTES, "partial sums fit the stages");
    static constexpr int TMEM_COLS = NT * ACCS < 32 ? 32 : NT * ACCS;
    static_assert(TMEM_COLS <= 256 && (TMEM_COLS & (TMEM_COLS - 1)) == 0, "two CTAs per SM");
    static constexpr uint32_t IDESC = (1u << 4) | (OPK == 2 ? ((1u << 7) | (1u << 10)) : 0u) |
                                      ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
};
template <int S>
struct Smem {
    uint64_t full[S], empty[S], done;
    uint32_t tmem_base;
    int abort;
};
}  // namespace fewk

template <typename T2, typename Cvt>
__device__ __forceinline__ uint2 pack4(const float (&y)[4], Cvt cvt) {
    const T2 a = cvt(y[0], y[1]), b = cvt(y[2], y[3]);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}
__device__ __forceinline__ void store4(__half* p, const float (&y)[4]) {
    *reinterpret_cast<uint2*>(p) = pack4<__half2>(y, [](float a, float b) { return __floats2half2_rn(a, b); });
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float (&y)[4]) {
    *reinterpret_cast<uint2*>(p) = pack4<__nv_bfloat162>(y, [](float a, float b) { return __floats2bfloat162_rn(a, b); });
}
__device__ __forceinline__ void store4(float* p, const float (&y)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(y[0], y[1], y[2], y[3]);
}
__device__ __forceinline__ void st_shared_b32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.b32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}

// blockIdx.x = channel tile * split + part, the cluster being the parts of one
// tile; blockIdx.y = token tile.
template <typename TOut, int NT, int OPK, int ACCS>
__global__ void __launch_bounds__(fewk::THREADS)
w4a4_gemm_few_kernel(GemmArgs a, const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                     int split) {
    using Tile = fewk::Tile<NT, OPK, ACCS>;
    constexpr int STAGES = Tile::STAGES, STAGE_BYTES = Tile::STAGE_BYTES, A_BYTES = fewk::A_BYTES;
    constexpr int BK = OPK == 0 ? fewk::BK : fewk::BK / 2;   // K elements per stage
    constexpr bool DEQUANT = OPK == 0 || OPK == 3;
    using Smem = fewk::Smem<STAGES>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_addr(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    Smem* sh = reinterpret_cast<Smem*>(smem_raw + (base - raw) + STAGES * STAGE_BYTES);
    volatile int* abort = &sh->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int part = (int)cluster_ctarank();
    const int n0 = ((int)blockIdx.x / split) * fewk::BM, n = n0 + 4 * lane;   // n: epilogue, four channels per lane
    const int t0 = (int)blockIdx.y * NT;                     // first token of the tile
    const int L = min(a.L - t0, NT);                         // tokens of the tile
    const int num_k = a.K / BK;
    const int k0 = num_k * part / split, nk = num_k * (part + 1) / split - k0;   // this part's K blocks (>= 1)

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_addr(&sh->full[s]), 1);
            mbar_init(smem_addr(&sh->empty[s]), 1);
        }
        mbar_init(smem_addr(&sh->done), 1);
        sh->abort = 0;
        mbar_fence_init();
    }
    if (warp == fewk::MMA_WARP) {
        tmem_alloc(smem_addr(&sh->tmem_base), Tile::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    int issued = 0;                                          // TMA warp: K blocks asked for
    float sa_lane = 0.f;                                     // epilogue: scales and bias, read ahead
    bool ok_epi = false;
    float4 sw = make_float4(0.f, 0.f, 0.f, 0.f), bb = sw;

    if (warp == fewk::TMA_WARP) {
        bool ok = true;
        const int pre = nk < STAGES ? nk : STAGES;           // first stages: no empty wait is due
        if (elect_one()) {
            for (int kc = 0; kc < pre; ++kc) mbar_arrive_expect_tx(smem_addr(&sh->full[kc]), STAGE_BYTES);
            if (a.weights_ready)
                for (int kc = 0; kc < pre; ++kc)
                    tma_load_2d(base + kc * STAGE_BYTES, &tmap_w, (k0 + kc) * BK, n0, smem_addr(&sh->full[kc]));
        }
        __syncwarp();
        grid_dependency_wait();
        grid_launch_dependents();
        if (elect_one()) {
            for (int kc = 0; kc < pre; ++kc) {
                const uint32_t st = base + kc * STAGE_BYTES, bar = smem_addr(&sh->full[kc]);
                tma_load_2d(st + A_BYTES, &tmap_x, (k0 + kc) * BK, t0, bar);
                if (!a.weights_ready) tma_load_2d(st, &tmap_w, (k0 + kc) * BK, n0, bar);
            }
        }
        __syncwarp();
        issued = pre;
        for (int kc = pre; kc < nk && ok; ++kc) {
            const int s = kc % STAGES;
            ok = mbar_wait_bounded_warp(smem_addr(&sh->empty[s]), (uint32_t)((kc / STAGES) & 1) ^ 1u, abort);
            if (ok) ++issued;
            if (ok && elect_one()) {
                const uint32_t st = base + s * STAGE_BYTES, bar = smem_addr(&sh->full[s]);
                mbar_arrive_expect_tx(bar, STAGE_BYTES);
                tma_load_2d(st, &tmap_w, (k0 + kc) * BK, n0, bar);
                tma_load_2d(st + A_BYTES, &tmap_x, (k0 + kc) * BK, t0, bar);
            }
            __syncwarp();
        }
        if (!ok && lane == 0) { sh->abort = 1; atomicOr(a.status, STATUS_TIMEOUT_GEMM); }
    } else if (warp == fewk::MMA_WARP) {
        grid_dependency_wait();
        grid_launch_dependents();
        bool ok = true;
        for (int kc = 0; kc < nk && ok; ++kc) {
            const int s = kc % STAGES;
            ok = mbar_wait_bounded_warp(smem_addr(&sh->full[s]), (uint32_t)((kc / STAGES) & 1), abort);
            tc_fence_after();
            if (ok && elect_one()) {
                const uint64_t ad = smem_desc_sw128(base + s * STAGE_BYTES);
                const uint64_t bd = smem_desc_sw128(base + s * STAGE_BYTES + A_BYTES);
                const int first = OPK == 3 ? kc % fewk::ACC_STAGES : kc;       // 0: a new accumulator
                const uint32_t d = tmem + (OPK == 3 ? (uint32_t)(kc / fewk::ACC_STAGES * NT) : 0u);
                #pragma unroll
                for (int ks = 0; ks < fewk::BK / fewk::UMMA_K; ++ks) {
                    const uint64_t adk = ad + (uint64_t)(ks * fewk::UMMA_K / 16), bdk = bd + (uint64_t)(ks * fewk::UMMA_K / 16);
                    if (OPK == 0) mma_f8f6f4(d, adk, bdk, Tile::IDESC, (first > 0 || ks > 0) ? 1u : 0u);
                    else mma_f16(d, adk, bdk, Tile::IDESC, (first > 0 || ks > 0) ? 1u : 0u);
                }
                tc_commit(smem_addr(&sh->empty[s]));
            }
            __syncwarp();
        }
        if (elect_one()) tc_commit(smem_addr(&sh->done));     // also after a failed wait
        __syncwarp();
        if (!ok && lane == 0) { sh->abort = 1; atomicOr(a.status, STATUS_TIMEOUT_GEMM); }
    } else {
        grid_dependency_wait();
        grid_launch_dependents();
        // lane j: the activation scale of the j-th token this warp will finish
        const int tj = part + split * (warp + fewk::NUM_EPI_WARPS * lane);
        if (DEQUANT && tj < L) sa_lane = __ldg(a.s_a + t0 + tj);
        if (DEQUANT && n < a.N) {
            sw = __ldg(reinterpret_cast<const float4*>(a.s_w + n));
            if (a.bias != nullptr) bb = __ldg(reinterpret_cast<const float4*>(a.bias + n));
        }
        volatile int never = 0;
        ok_epi = mbar_wait_bounded_warp(smem_addr(&sh->done), 0, &never);
        tc_fence_after();
        if (!ok_epi && lane == 0) atomicOr(a.status, STATUS_TIMEOUT_GEMM);
    }
    __syncwarp();
    if (split > 1) cluster_sync();   // every part has read its stages: they take the sums
    // the accumulator (lane = channel, column = token): token t goes to part
    // t mod split, into its row [this part][t / split] of 128 channels
    const int slots = (NT + split - 1) / split;              // tokens per part
    if (warp < fewk::NUM_EPI_WARPS && ok_epi) {
        const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
        const uint32_t mine = base + (uint32_t)((part * slots * fewk::BM + warp * 32 + lane) * 4);
        int owner = 0;
        uint32_t row = 0;                                    // byte offset of row t / split
        #pragma unroll 1
        for (int c = 0; c < NT && c < L; c += 16) {
            uint32_t r[16];
            tmem_ld_32x32b_x16(trow + (uint32_t)c, r);
            tmem_ld_wait();
            if (OPK == 3) {                                  // the accumulators' integers, summed in int32
                #pragma unroll
                for (int t = 0; t < 16; ++t) r[t] = (uint32_t)__float2int_rn(__uint_as_float(r[t]));
                #pragma unroll
                for (int q = 1; q < ACCS; ++q) {
                    if (q * fewk::ACC_STAGES >= nk) break;
                    uint32_t x[16];
                    tmem_ld_32x32b_x16(trow + (uint32_t)(q * NT + c), x);
                    tmem_ld_wait();
                    #pragma unroll
                    for (int t = 0; t < 16; ++t) r[t] += (uint32_t)__float2int_rn(__uint_as_float(x[t]));
                }
            }
            if (split == 1) {                                // (the waiting MMAs are this CTA's own)
                #pragma unroll
                for (int t = 0; t < 16; ++t) st_shared_b32(mine + (uint32_t)((c + t) * fewk::BM * 4), r[t]);
            } else {
                #pragma unroll
                for (int t = 0; t < 16; ++t) {
                    st_shared_cluster_b32(mapa_shared(mine, (uint32_t)owner) + row, r[t]);
                    if (++owner == split) { owner = 0; row += fewk::BM * 4; }
                }
            }
        }
        tc_fence_before();
    }
    __syncwarp();
    // this part's tokens are complete; no part touches another's memory any more
    if (split > 1) cluster_sync();
    else __syncthreads();
    if (warp < fewk::NUM_EPI_WARPS && ok_epi && *abort == 0) {
        TOut* Y = static_cast<TOut*>(a.Y);
        int j = 0;                                           // tokens finished by this warp
        for (int sl = warp; part + sl * split < L; sl += fewk::NUM_EPI_WARPS, ++j) {
            const uint32_t src = base + (uint32_t)((sl * fewk::BM + 4 * lane) * 4);
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            int isum[4] = {0, 0, 0, 0};                      // kind 3
            #pragma unroll 4
            for (int c = 0; c < split; ++c) {
                const uint4 v = ld_shared_v4(src + (uint32_t)(c * slots * fewk::BM * 4));
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
                #pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (OPK == 3) isum[k] += (int)w[k];
                    else acc[k] += __uint_as_float(w[k]);
                }
            }
            float y[4] = {acc[0], acc[1], acc[2], acc[3]};
            if (DEQUANT) {
                const float sa = __shfl_sync(0xffffffffu, sa_lane, j);
                const float t4[4] = {sw.x, sw.y, sw.z, sw.w};
                #pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (OPK == 3) acc[k] = __int2float_rn(isum[k]);
                    else isum[k] = __float2int_rn(acc[k]);
                    y[k] = __fmul_rn(__fmul_rn(acc[k], sa), t4[k]);
                }
            }
            if (DEQUANT && a.bias != nullptr) {
                y[0] = __fadd_rn(y[0], bb.x);
                y[1] = __fadd_rn(y[1], bb.y);
                y[2] = __fadd_rn(y[2], bb.z);
                y[3] = __fadd_rn(y[3], bb.w);
            }
            float h[4];
            if (OPK == 0 && a.swiglu) {
                // lanes 0-3 of every eight hold 16 gate channels, lanes 4-7 the matching up channels
                #pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float up = __shfl_down_sync(0xffffffffu, y[k], 4);
                    h[k] = y[k] / (1.f + expf(-y[k])) * up;
                }
            }
            if (n >= a.N) continue;                          // (N % 32 == 0: eight lanes at a time)
            const size_t t = (size_t)(t0 + part + sl * split);
            if (a.acc_dbg != nullptr)
                *reinterpret_cast<int4*>(a.acc_dbg + t * a.N + n) = make_int4(isum[0], isum[1], isum[2], isum[3]);
            if (OPK != 0 || !a.swiglu) store4(Y + t * a.N + n, y);
            else if ((lane & 4) == 0) store4(Y + t * (a.N / 2) + n0 / 2 + (lane >> 3) * 16 + 4 * (lane & 3), h);
        }
    }
    __syncwarp();
    tc_fence_after();
    if (warp == fewk::MMA_WARP) tmem_dealloc(tmem, Tile::TMEM_COLS);
    if (warp == fewk::TMA_WARP && *abort != 0) {
        // one of the roles gave up (set before the barrier above), and nobody
        // has waited for the tiles that the MMA warp did not reach: the CTA must
        // not give its shared memory back under them (the last use of each
        // stage, read or not). Out of the way of the epilogue's code: ahead of it
        // the same lines cost 0.05 us a launch.
        volatile int never = 0;
        for (int kc = issued > STAGES ? issued - STAGES : 0; kc < issued; ++kc)
            if (!mbar_wait_bounded_warp(smem_addr(&sh->full[kc % STAGES]), (uint32_t)((kc / STAGES) & 1), &never)) break;
    }
}

bool encode_k_major(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t elem) {
    const PFN_cuTensorMapEncodeTiled_v12000 fn = tensor_map_encoder();
    if (fn == nullptr) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * elem};
    const cuuint32_t box[2] = {fewk::BK / elem, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, elem == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<void*>(ptr),
              dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The launch of a problem: token tiles, parts of K per channel tile (as many as
// keep every CTA resident at once, two per SM, at most a portable cluster and
// the number of K blocks) and, for kind 3, accumulators per CTA.
struct FewPlan { int nt, rows, ctas, split, stages, accs; };
FewPlan few_plan(const GemmArgs& a, int opk) {
    FewPlan p;
    p.nt = a.L <= 16 ? 16 : a.L <= 32 ? 32 : a.L <= 64 ? 64 : 128;
    p.rows = (a.L + p.nt - 1) / p.nt;
    const int tiles = (a.N + fewk::BM - 1) / fewk::BM;
    p.stages = a.K / (opk == 0 ? fewk::BK : fewk::BK / 2);
    p.split = 2 * num_sms() / (tiles * p.rows);
    if (p.split > fewk::MAX_SPLIT) p.split = fewk::MAX_SPLIT;
    if (p.split > p.stages) p.split = p.stages;
    if (p.split < 1) p.split = 1;
    p.ctas = tiles * p.rows * p.split;
    const int most = (p.stages + p.split - 1) / p.split;     // stages of the longest part
    const int need = opk == 3 ? (most + fewk::ACC_STAGES - 1) / fewk::ACC_STAGES : 1;
    p.accs = need < 1 ? 1 : need;
    return p;
}

template <typename TOut, int NT, int OPK, int ACCS>
cudaError_t launch_few(const GemmArgs& a, const FewPlan& p, cudaStream_t stream) {
    using Tile = fewk::Tile<NT, OPK, ACCS>;
    constexpr uint32_t ELEM = OPK == 0 ? 1 : 2;
    auto kernel = w4a4_gemm_few_kernel<TOut, NT, OPK, ACCS>;
    static DeviceCache<int> attr;
    int done = 0;
    cudaError_t e = attr.get(&done, [&](int, int* v) {
        *v = 1;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Tile::SMEM_BYTES);
    });
    if (e != cudaSuccess) return e;
    CUtensorMap tw, tx;
    if (!encode_k_major(&tw, a.We, (uint64_t)a.N, (uint64_t)a.K, fewk::BM, ELEM) ||
        !encode_k_major(&tx, a.Xe, (uint64_t)a.L, (uint64_t)a.K, NT, ELEM))
        return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.split;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1] = pdl_attribute();
    cfg.gridDim = dim3((unsigned)(p.ctas / p.rows), (unsigned)p.rows);
    cfg.blockDim = dim3(fewk::THREADS);
    cfg.dynamicSmemBytes = Tile::SMEM_BYTES;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, a, tw, tx, p.split);
}

template <typename TOut, int OPK, int ACCS>
cudaError_t launch_few_nt(const GemmArgs& a, const FewPlan& p, cudaStream_t stream) {
    switch (p.nt) {
        case 16: return launch_few<TOut, 16, OPK, ACCS>(a, p, stream);
        case 32: return launch_few<TOut, 32, OPK, ACCS>(a, p, stream);
        case 64: return launch_few<TOut, 64, OPK, ACCS>(a, p, stream);
        default: return launch_few<TOut, 128, OPK, ACCS>(a, p, stream);
    }
}

template <typename TOut>
cudaError_t launch_few_typed(const GemmArgs& a, const FewPlan& p, int opk, cudaStream_t stream) {
    if (a.swiglu && (opk != 0 || sizeof(TOut) != 2)) return cudaErrorInvalidValue;
    if (opk == 0) return launch_few_nt<TOut, 0, 1>(a, p, stream);
    if (opk == 3) return p.accs == 1 ? launch_few_nt<TOut, 3, 1>(a, p, stream) : launch_few_nt<TOut, 3, 2>(a, p, stream);
    return cudaErrorInvalidValue;
}

}  // namespace

// Whether this kernel is the faster one. Both estimates are fits to launches
// back to back over weights larger than L2 (ns; L 1 .. 512, N 512 .. 24576, K
// 512 .. 18944):
//   pair kernel  a round of ceil(N / 224) ceil(L / 256) tiles per resident pair
//                takes 245 ns per 128 K and 4 us of prologue and epilogue, and
//                the weights stream at 4 TB/s at most;
//   this kernel  1.5 us, the weights at 6 TB/s, 1.2 us for the exchange of the
//                parts' sums, and per token 20 ns (32 when two CTAs share an
//                SM, 70 when one CTA finishes all tokens of its tile), 1.4 times
//                that with the shorter ring of 128-token tiles.
// Measured, pair kernel and this one, us: 32 x 4096 -> 12288 13.6, 12.3; 32 x
// 4096 -> 4096 12.1, 6.9; 32 x 12288 -> 4096 27.0, 11.7; 64 x 4096 -> 24576 24.9,
// 23.1; 128 x 12288 -> 4096 27.3, 15.3; 1 x 512 -> 512 4.7, 2.5; and where it
// stays off, 128 x 4096 -> 12288 13.8, 16.2; 128 x 3584 -> 4608 11.3, 12.0.
// 16-bit operands: twice the bytes, and a stage is 64 K. W8A8 and fp16, pair
// kernel and this one, us: 32 x 4096 -> 4096 21.5, 9.3 and 19.2, 9.0; 32 x 4096 ->
// 12288 24.7, 20.4 and 22.8, 20.5; 32 x 12288 -> 4096 53.5, 19.8 and 49.3, 19.2;
// where it stays off, W8A8 128 x 4096 -> 12288 25.1, 27.0 (a second accumulator
// to read per token: 1.6 times). The float32 sums of fp16 and bf16 are added in
// shorter chains: against 64-bit sums 0.3% of the fp16 results at K = 4096 are
// not the correctly rounded ones (1.7% in the pair kernel), 1.0% at 16384 (5.7%).
bool few_tokens(const GemmArgs& a, int opk) {
    if (a.L > 256) return false;
    const FewPlan p = few_plan(a, opk);
    if (p.accs > 2) return false;                            // kind 3: at most 2048 K per part
    const long long bytes = (long long)a.N * a.K * (opk == 0 ? 1 : 2);
    const long long tiles = (long long)((a.N + 223) / 224), pairs = num_sms() / 2;    // (one row of tiles: L <= 256)
    long long pair_ns = (tiles + pairs - 1) / pairs * (4000 + 245LL * p.stages);
    if (pair_ns < bytes / 4000) pair_ns = bytes / 4000;
    long long token_ns = p.split == 1 ? 70 : p.ctas > num_sms() ? 32 : 20;
    if (a.L > 64) token_ns = token_ns * (p.accs > 1 ? 8 : 7) / 5;
    return 1500 + bytes / 6000 + (p.split > 1 ? 1200 : 0) + token_ns * a.L < pair_ns;
}

cudaError_t launch_gemm_few(const GemmArgs& a, int opk, int* split_used, cudaStream_t stream) {
    const FewPlan p = few_plan(a, opk);
    *split_used = p.split;
    switch (a.y_dtype) {
        case STARQ_F16:
            return opk == 1 ? launch_few_nt<__half, 1, 1>(a, p, stream) : launch_few_typed<__half>(a, p, opk, stream);
        case STARQ_BF16:
            return opk == 2 ? launch_few_nt<__nv_bfloat16, 2, 1>(a, p, stream)
                            : launch_few_typed<__nv_bfloat16>(a, p, opk, stream);
        case STARQ_F32: return launch_few_typed<float>(a, p, opk, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace starq
