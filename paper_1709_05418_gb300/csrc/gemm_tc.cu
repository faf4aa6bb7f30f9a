// gemm_tc.cu -- BF16 tensor-core GEMM of the mixed-precision training step (Sec. 5.2 with
// BF16 operands, FP32 accumulation and FP32 master weights):
//
//   D = epilogue( A0 B0^T + A1 B1^T )      A_s: [M][K_s] BF16, B_s: [N][K_s] BF16 (K contiguous)
//
// One CTA of four warps per 128 x BN output tile (BN = 32, 64, 128 or 256): thread 0 streams
// both operands through a ring of shared-memory stages with 2-D TMA copies (64-byte
// swizzled K-major boxes of 32 elements, two per operand and stage), thread 32 issues
// four 128 x BN x 16 tcgen05 MMAs per stage into one FP32 accumulator in tensor memory,
// and after the last stage all four warps read their 32 accumulator lanes back and apply
// the epilogue: bias, residual, ReLU, mask, then FP32, BF16 and transposed-BF16 stores.
// With splits > 1, CTA z takes the z-th run of the K stages and writes raw partial sums
// to a workspace; k_tg_splitk adds them in run order and applies the epilogue.  Out-of-
// range rows and columns of a tile are zero-filled by the copies and not stored.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "tmap.h"

namespace rpnn {

namespace {

constexpr int TGM = 128;                  // output rows per tile (one M = 128 MMA)
constexpr int KST = 64;                   // K elements per stage: two 32-element boxes
constexpr uint32_t ABOX = TGM * 64;       // bytes of one A box (128 rows x 64 bytes)
constexpr int NTH = 128;

struct TgEpiDev {
    const float* bias;                    // [N] or null
    const float* res;                     // [M][ldr] or null
    int64_t ldr;
    const float* mask;                    // multiply by (mask > 0): [M][ldm] (mask_t: [N][ldm]) or null
    int64_t ldm;
    int mask_t;
    int relu;
    float* C;                             // FP32 [M][ldc] or null
    int64_t ldc;
    __nv_bfloat16* Cb;                    // BF16 [M][ldb] or null
    int64_t ldb;
    __nv_bfloat16* Ct;                    // BF16 transposed [N][ldt] or null
    int64_t ldt;
};

struct TgArgs {
    int M, N, K0, K1;                     // K1 = 0: one segment
    int splits;
    int vec;                              // the epilogue's rows are 16-byte aligned, N is a multiple of 8
    float* ws;                            // [splits][M][N] partial sums when splits > 1
    TgEpiDev e;
    uint32_t* status;
};

template <int BN>
struct TgCfg {
    static constexpr uint32_t BBOX = BN * 64;
    static constexpr uint32_t STAGE = 2 * ABOX + 2 * BBOX;
    static constexpr int STAGES = BN == 256 ? 3 : 4;
    static_assert(4 * 32 * 17 * 4 <= STAGES * STAGE, "epilogue tiles reuse the stage ring");
    static constexpr uint32_t OFF_BAR = STAGES * STAGE;
    static constexpr uint32_t SMEM = OFF_BAR + 256 + 1024;   // barriers, TMEM slot, alignment slack
};

// everything but the transposed copy; returns the stored value
__device__ __forceinline__ float tg_store(const TgEpiDev& e, int m, int n, float v) {
    if (e.bias) v += e.bias[n];
    if (e.res) v += e.res[(int64_t)m * e.ldr + n];
    if (e.relu) v = fmaxf(v, 0.0f);
    if (e.mask && !(e.mask[e.mask_t ? (int64_t)n * e.ldm + m : (int64_t)m * e.ldm + n] > 0.0f)) v = 0.0f;
    if (e.C) e.C[(int64_t)m * e.ldc + n] = v;
    if (e.Cb) e.Cb[(int64_t)m * e.ldb + n] = __float2bfloat16_rn(v);
    return v;
}

template <int BN>
__global__ void __launch_bounds__(NTH, 1)
k_tc_gemm(const __grid_constant__ CUtensorMap a0, const __grid_constant__ CUtensorMap b0,
          const __grid_constant__ CUtensorMap a1, const __grid_constant__ CUtensorMap b1, const TgArgs g) {
    using C = TgCfg<BN>;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = tc::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;          // swizzle atoms want 512-byte alignment
    unsigned char* sbase = smem_raw + (base - raw);
    const uint32_t bar = base + C::OFF_BAR;                 // full[S], empty[S], done
    const uint32_t done = bar + 8u * (2 * C::STAGES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sbase + C::OFF_BAR + 8 * (2 * C::STAGES + 1));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * TGM, n0 = blockIdx.x * BN;
    const int T0 = (g.K0 + KST - 1) / KST, T = T0 + (g.K1 + KST - 1) / KST;
    const int per = (T + g.splits - 1) / g.splits;
    const int tb = (int)blockIdx.z * per;
    const int nst = max(0, min(T, tb + per) - tb);

    // operand tiles of stage `it` of this block's K run (thread 0)
    auto load_stage = [&](int it) {
        const int t = tb + it;
        const bool first = t < T0;
        const void* am = first ? static_cast<const void*>(&a0) : static_cast<const void*>(&a1);
        const void* bm = first ? static_cast<const void*>(&b0) : static_cast<const void*>(&b1);
        const int k0 = (first ? t : t - T0) * KST;
        const uint32_t st = base + (uint32_t)(it % C::STAGES) * C::STAGE;
        const uint32_t fb = bar + 8u * (it % C::STAGES);
        tc::mbar_expect_tx(fb, C::STAGE);
        tc::tma_load_2d(st, am, k0, m0, fb);
        tc::tma_load_2d(st + ABOX, am, k0 + 32, m0, fb);
        tc::tma_load_2d(st + 2 * ABOX, bm, k0, n0, fb);
        tc::tma_load_2d(st + 2 * ABOX + C::BBOX, bm, k0 + 32, n0, fb);
    };
    // the first stages are on their way before anything else is set up
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            tc::mbar_init(bar + 8u * s, 1);
            tc::mbar_init(bar + 8u * (C::STAGES + s), 1);
        }
        tc::mbar_init(done, 1);
        *abort_flag = 0;
        tc::fence_mbar_init();
        for (int it = 0; it < min(nst, C::STAGES); ++it) load_stage(it);
    }
    if (warp == 2) {
        tc::tmem_alloc(tc::smem_u32(tmem_slot), BN);
        tc::tmem_relinquish();
    }
    // The epilogue's residual and mask do not depend on the MMAs: tiles of up to 64 columns load
    // them first, all at once, so that they arrive while the operands do (loaded after the MMAs,
    // one chunk of 16 columns after the other, they cost a step of 4,096 rows 26 us on its chain of
    // 21 data gradients)
    const int row0 = m0 + warp * 32, row = row0 + lane;
    constexpr bool EARLY = BN <= 64;
    constexpr int NC = EARLY ? BN / 16 : 1;
    float er[NC][16], em[NC][16];
    // this lane's row of the 16 columns from n on (vec: 8 or 16 of them exist)
    auto row16 = [&](const float* p, float (&r)[16], int n) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (n + 4 * q >= g.N || row >= g.M) continue;
            const float4 t = *reinterpret_cast<const float4*>(p + 4 * q);
            r[4 * q] = t.x; r[4 * q + 1] = t.y; r[4 * q + 2] = t.z; r[4 * q + 3] = t.w;
        }
    };
    auto operands = [&](int n, float (&r)[16], float (&k)[16]) {
        if (g.e.res) row16(g.e.res + (int64_t)row * g.e.ldr + n, r, n);
        if (g.e.mask && !g.e.mask_t) row16(g.e.mask + (int64_t)row * g.e.ldm + n, k, n);
        if (g.e.mask && g.e.mask_t) {
            const float* p = g.e.mask + (int64_t)n * g.e.ldm + row;
#pragma unroll
            for (int jj = 0; jj < 16; ++jj)
                if (n + jj < g.N && row < g.M) k[jj] = p[jj * g.e.ldm];
        }
    };
    if (EARLY && g.vec) {
#pragma unroll
        for (int c = 0; c < NC; ++c) operands(n0 + 16 * c, er[c], em[c]);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (nst > 0) {
        if (threadIdx.x == 0) {                              // producer
            for (int it = C::STAGES; it < nst; ++it) {
                if (!tc::mbar_wait(bar + 8u * (C::STAGES + it % C::STAGES), ((it / C::STAGES) - 1) & 1, abort_flag)) break;
                load_stage(it);
            }
        } else if (threadIdx.x == 32) {                      // MMA issuer
            const uint32_t idesc = tc::idesc_bf16(TGM, BN);
            for (int it = 0; it < nst; ++it) {
                const int s = it % C::STAGES;
                if (!tc::mbar_wait(bar + 8u * s, (it / C::STAGES) & 1, abort_flag)) break;
                tc::tc_fence_after();
                const uint32_t st = base + (uint32_t)s * C::STAGE;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t ao = st + (kk >> 1) * ABOX + (kk & 1) * 32;
                    const uint32_t bo = st + 2 * ABOX + (kk >> 1) * C::BBOX + (kk & 1) * 32;
                    tc::mma_bf16(tmem, tc::smem_desc_sw64(ao), tc::smem_desc_sw64(bo), idesc, (it | kk) != 0);
                }
                tc::mma_commit(bar + 8u * (C::STAGES + s));
            }
            tc::mma_commit(done);
        }
        __syncwarp();
        tc::mbar_wait(done, 0, abort_flag);
        tc::tc_fence_after();
    }

    // epilogue: warp w owns accumulator lanes (tile rows) 32 w .. 32 w + 31, a lane one row, 16
    // columns at a time.  Aligned rows go straight from registers: 16-byte loads and stores per
    // lane, and transposed stores (masks) of 32 consecutive rows per warp.  Bound: latency; the
    // code runs once per block.  Passing every 16 columns through shared memory with each load
    // and store under its own condition took 6,000-10,000 clocks of a
    // block's 13,000-19,000; now 2,500-3,800 of 9,000-13,000 (step of 4,096 rows 613 -> 554 us, with the
    // first stages and the operands requested before the barrier).
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    auto chunk = [&](int c0, float (&v)[16]) {
        if (nst > 0) {
            tc::tmem_ld16(trow + (uint32_t)c0, v);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.0f;
        }
    };
    if (g.vec) {
#pragma unroll(EARLY ? NC : 1)
        for (int c0 = 0; c0 < BN; c0 += 16) {
            if (n0 + c0 >= g.N) break;
            const int ec = EARLY ? c0 / 16 : 0;
            float v[16];
            chunk(c0, v);
            if (!EARLY) operands(n0 + c0, er[0], em[0]);
            if (row < g.M) {
#pragma unroll
                for (int h = 0; h < 16; h += 8) {
                    const int n = n0 + c0 + h;
                    if (n >= g.N) break;
                    float* x = v + h;
                    if (g.e.bias) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] += g.e.bias[n + j];
                    }
                    if (g.e.res) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] += er[ec][h + j];
                    }
                    if (g.e.relu) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = fmaxf(x[j], 0.0f);
                    }
                    if (g.e.mask) {
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = em[ec][h + j] > 0.0f ? x[j] : 0.0f;
                    }
                    if (g.e.C) {
                        float4* c = reinterpret_cast<float4*>(g.e.C + (int64_t)row * g.e.ldc + n);
                        c[0] = make_float4(x[0], x[1], x[2], x[3]);
                        c[1] = make_float4(x[4], x[5], x[6], x[7]);
                    }
                    __align__(16) __nv_bfloat16 b[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) b[j] = __float2bfloat16_rn(x[j]);
                    if (g.e.Cb) *reinterpret_cast<uint4*>(g.e.Cb + (int64_t)row * g.e.ldb + n) = *reinterpret_cast<const uint4*>(b);
                    if (g.e.Ct) {
                        __nv_bfloat16* t = g.e.Ct + (int64_t)n * g.e.ldt + row;
#pragma unroll
                        for (int j = 0; j < 8; ++j) t[j * g.e.ldt] = b[j];
                    }
                }
            }
            __syncwarp();
        }
    } else {
        // partial sums and unaligned rows: each 32 x 16 chunk through a per-warp shared tile (the
        // stage ring is idle once the MMAs are done), half a warp per row, then a lane per row for the
        // transposed store
        float* stile = reinterpret_cast<float*>(sbase) + warp * (32 * 17);
        for (int c0 = 0; c0 < BN; c0 += 16) {
            if (n0 + c0 >= g.N) break;
            float v[16];
            chunk(c0, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) stile[lane * 17 + j] = v[j];
            __syncwarp();
            const int j = lane & 15, n = n0 + c0 + j;
            if (g.splits > 1) {
#pragma unroll 8
                for (int it = 0; it < 16; ++it) {
                    const int rr = 2 * it + (lane >> 4), m = row0 + rr;
                    if (m < g.M && n < g.N) g.ws[((int64_t)blockIdx.z * g.M + m) * g.N + n] = stile[rr * 17 + j];
                }
            } else {
#pragma unroll 4
                for (int it = 0; it < 16; ++it) {
                    const int rr = 2 * it + (lane >> 4), m = row0 + rr;
                    if (m < g.M && n < g.N) stile[rr * 17 + j] = tg_store(g.e, m, n, stile[rr * 17 + j]);
                }
                __syncwarp();
                if (g.e.Ct && row < g.M)
                    for (int jj = 0; jj < 16 && n0 + c0 + jj < g.N; ++jj)
                        g.e.Ct[(int64_t)(n0 + c0 + jj) * g.e.ldt + row] = __float2bfloat16_rn(stile[lane * 17 + jj]);
            }
            __syncwarp();
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 2) tc::tmem_dealloc(tmem, BN);
    if (threadIdx.x == 0 && *abort_flag) atomicOr(g.status, kStatTimeout);
}

__global__ void k_tg_splitk(const float* __restrict__ ws, int splits, int M, int N, TgEpiDev e) {
    const int64_t total = (int64_t)M * N;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / N), n = (int)(i % N);
        float v = 0.0f;
        for (int z = 0; z < splits; ++z) v += ws[((int64_t)z * M + m) * N + n];
        v = tg_store(e, m, n, v);
        if (e.Ct) e.Ct[(int64_t)n * e.ldt + m] = __float2bfloat16_rn(v);
    }
}

constexpr int kTgTiles[] = {32, 64, 128, 256};
constexpr int kTgSplits[] = {1, 2, 4, 8, 16, 32};
constexpr int kTgMinSplitK = 1024;
constexpr int kTgFlag = 1 << 8;             // distinguishes tensor-core shapes in the tuning table

rpnn_status make_map(Ctx& c, CUtensorMap* m, const void* p, int64_t ld, int K, int rows, int box_rows) {
    static_assert(sizeof(CUtensorMap) == sizeof(TmapBytes), "tensor map size");
    const TmapKey key{p, ld, K, rows, box_rows};
    const auto it = c.tmaps.find(key);
    if (it != c.tmaps.end()) {
        memcpy(m, it->second.b, sizeof(CUtensorMap));
        return RPNN_OK;
    }
    EncodeTiledFn enc = encode_fn();
    if (!enc) { set_error("cuTensorMapEncodeTiled is unavailable"); return RPNN_ERR_UNSUPPORTED; }
    if ((reinterpret_cast<uintptr_t>(p) & 15u) != 0 || (ld * 2) % 16 != 0 || ld < K) {
        set_error("BF16 GEMM operand must be 16-byte aligned with a row pitch of 8k elements >= K");
        return RPNN_ERR_ARG;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {32, (cuuint32_t)box_rows};
    const cuuint32_t es[2] = {1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(p), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled failed (%d)", (int)r); return RPNN_ERR_CUDA; }
    if (c.tmaps.size() > 4096) c.tmaps.clear();
    TmapBytes tb;
    memcpy(tb.b, m, sizeof(CUtensorMap));
    c.tmaps.emplace(key, tb);
    return RPNN_OK;
}

TgEpiDev to_dev(const TgOut& o) {
    TgEpiDev e;
    e.bias = o.bias; e.res = o.res; e.ldr = o.ldr; e.mask = o.mask; e.ldm = o.ldm; e.mask_t = o.mask_t;
    e.relu = o.relu;
    e.C = o.C; e.ldc = o.ldc;
    e.Cb = reinterpret_cast<__nv_bfloat16*>(o.Cb); e.ldb = o.ldb;
    e.Ct = reinterpret_cast<__nv_bfloat16*>(o.Ct); e.ldt = o.ldt;
    return e;
}

template <int BN>
rpnn_status launch_bn(const CUtensorMap* maps, const TgArgs& a, cudaStream_t s) {
    using C = TgCfg<BN>;
    static bool attr = false;
    if (!attr) {
        RPNN_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
        attr = true;
    }
    dim3 grid((a.N + BN - 1) / BN, (a.M + TGM - 1) / TGM, a.splits);
    k_tc_gemm<BN><<<grid, NTH, C::SMEM, s>>>(maps[0], maps[1], maps[2], maps[3], a);
    RPNN_CHECK_LAUNCH();
    return RPNN_OK;
}

// One launch (plus the split-K reduction) with tile width bn and `splits` K runs; `reps` of them for
// the tuner.
rpnn_status launch_tg(Ctx& c, int bn, int splits, int M, int N, const TgSeg& s0, const TgSeg* s1,
                      const TgEpiDev& e, float* ws, cudaStream_t s, int reps = 1) {
    if ((M + TGM - 1) / TGM > 65535) { set_error("BF16 GEMM with %d rows exceeds the grid limit", M); return RPNN_ERR_ARG; }
    CUtensorMap maps[4];
    rpnn_status st = make_map(c, &maps[0], s0.A, s0.lda, s0.K, M, TGM);
    if (!st) st = make_map(c, &maps[1], s0.B, s0.ldb, s0.K, N, bn);
    if (!st && s1) st = make_map(c, &maps[2], s1->A, s1->lda, s1->K, M, TGM);
    if (!st && s1) st = make_map(c, &maps[3], s1->B, s1->ldb, s1->K, N, bn);
    if (st) return st;
    if (!s1) { maps[2] = maps[0]; maps[3] = maps[1]; }
    TgArgs a;
    a.M = M; a.N = N; a.K0 = s0.K; a.K1 = s1 ? s1->K : 0;
    a.splits = splits; a.ws = ws; a.e = e; a.status = c.status.as<uint32_t>();
    // the direct epilogue: 16-byte accesses along the rows of what is there (the transposed ones take
    // any pitch), and whole groups of eight columns
    auto rows16 = [](const void* p, int64_t ld, size_t el) {
        return !p || (reinterpret_cast<uintptr_t>(p) % 16 == 0 && (size_t)ld * el % 16 == 0);
    };
    a.vec = splits == 1 && N % 8 == 0 && rows16(e.res, e.ldr, 4) && (e.mask_t || rows16(e.mask, e.ldm, 4)) &&
            rows16(e.C, e.ldc, 4) && rows16(e.Cb, e.ldb, 2);
    for (int r = 0; r < reps; ++r) {
        switch (bn) {
            case 32: st = launch_bn<32>(maps, a, s); break;
            case 64: st = launch_bn<64>(maps, a, s); break;
            case 128: st = launch_bn<128>(maps, a, s); break;
            default: st = launch_bn<256>(maps, a, s); break;
        }
        if (st) return st;
        if (splits > 1) {
            const int64_t total = (int64_t)M * N;
            int64_t b = (total + 255) / 256;
            if (b > (int64_t)c.num_sms * 8) b = (int64_t)c.num_sms * 8;
            k_tg_splitk<<<(unsigned)b, 256, 0, s>>>(ws, splits, M, N, e);
            RPNN_CHECK_LAUNCH();
        }
    }
    return RPNN_OK;
}

}  // namespace

rpnn_status tc_gemm(Ctx& c, int M, int N, const TgSeg& s0, const TgSeg* s1, const TgOut& o, cudaStream_t s,
                    DevBuf* split_ws) {
    if (M <= 0 || N <= 0) return RPNN_OK;
    const TgEpiDev e = to_dev(o);
    const int Ktot = s0.K + (s1 ? s1->K : 0);
    int bn = N <= 64 ? 64 : (N <= 128 ? 128 : 256), splits = 1;
    GemmTuner& tu = c.tuner;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    RPNN_CUDA_TRY(cudaStreamIsCapturing(s, &cs));
    if (tu.enabled) {
        GemmKey key{M, N, s0.K, s1 ? s1->K : 0,
                    kTgFlag | (o.bias != nullptr) << 4 | (o.res != nullptr) << 5 | (o.mask != nullptr) << 6 |
                        (o.Cb != nullptr) << 9 | (o.Ct != nullptr) << 10 | (o.mask_t != 0) << 11};
        const GemmChoice* hit = tu.find(key);
        if (hit) {
            bn = hit->tile;
            splits = hit->splits;
        } else if (cs == cudaStreamCaptureStatusNone) {   // never time under stream capture
            // time every admissible (tile width, split) on the call's operands, writing into
            // scratch only
            struct Cand { int bn, sp; };
            std::vector<Cand> cands;
            int maxsplit = 1;
            for (int t : kTgTiles) {
                if (t > 32 && t / 2 >= N) continue;
                const int64_t tiles = (int64_t)((N + t - 1) / t) * ((M + TGM - 1) / TGM);
                const int stages = (s0.K + KST - 1) / KST + (s1 ? (s1->K + KST - 1) / KST : 0);
                for (int sp : kTgSplits) {
                    if (sp > 1 && (Ktot < kTgMinSplitK || tiles >= c.num_sms || stages / sp < 2 ||
                                   tiles * sp > (int64_t)c.num_sms * 4))
                        continue;
                    cands.push_back({t, sp});
                    maxsplit = std::max(maxsplit, sp);
                }
            }
            // the copies are timed too: they are most of a gradient's epilogue (timed without them, a
            // 128-wide tile with a third of the blocks came out ahead and cost a step of 4,096 rows up to 45 us)
            const size_t nc = (size_t)M * N * sizeof(float), nb = e.Cb ? (size_t)M * e.ldb * 2 : 0, nt = e.Ct ? (size_t)N * e.ldt * 2 : 0;
            auto up16 = [](size_t n) { return (n + 15) / 16 * 16; };
            rpnn_status st = tu.scratch.reserve(up16(nc) + up16(nb) + nt);
            if (!st && maxsplit > 1) st = tu.ws.reserve((size_t)maxsplit * M * N * sizeof(float));
            if (st) return st;
            if (!tu.ev0) {
                RPNN_CUDA_TRY(cudaEventCreate(&tu.ev0));
                RPNN_CUDA_TRY(cudaEventCreate(&tu.ev1));
            }
            TgEpiDev es = e;
            es.C = tu.scratch.as<float>();
            es.ldc = N;
            unsigned char* copies = tu.scratch.as<unsigned char>() + up16(nc);
            if (e.Cb) es.Cb = reinterpret_cast<__nv_bfloat16*>(copies);
            if (e.Ct) es.Ct = reinterpret_cast<__nv_bfloat16*>(copies + up16(nb));
            GemmChoice best{bn, 1, 1e30f, 0.0f};
            for (const Cand& cd : cands) {
                st = launch_tg(c, cd.bn, cd.sp, M, N, s0, s1, es, tu.ws.as<float>(), s);
                if (st) return st;
                RPNN_CUDA_TRY(cudaEventRecord(tu.ev0, s));
                // together: with the host's preparation between them the launches of short kernels took
                // turns with it, and a 64-wide tile in 16 runs timed like a 32-wide one in 8 (step 580, 550 us)
                constexpr int kReps = 4;
                st = launch_tg(c, cd.bn, cd.sp, M, N, s0, s1, es, tu.ws.as<float>(), s, kReps);
                if (st) return st;
                RPNN_CUDA_TRY(cudaEventRecord(tu.ev1, s));
                RPNN_CUDA_TRY(cudaEventSynchronize(tu.ev1));
                float ms = 0.0f;
                RPNN_CUDA_TRY(cudaEventElapsedTime(&ms, tu.ev0, tu.ev1));
                const float us = ms * 1000.0f / kReps;
                if (cd.bn == bn && cd.sp == 1) best.default_us = us;
                if (us < 0.98f * best.us) { best.us = us; best.tile = cd.bn; best.splits = cd.sp; }   // a tie: the narrower tile
            }
            tu.table.emplace_back(key, best);
            ++tu.version;
            bn = best.tile;
            splits = best.splits;
        }
    }
    float* ws = nullptr;
    if (splits > 1) {
        DevBuf& wb = split_ws ? *split_ws : tu.ws;
        rpnn_status st = wb.reserve((size_t)splits * M * N * sizeof(float));
        if (st) return st;
        ws = wb.as<float>();
    }
    return launch_tg(c, bn, splits, M, N, s0, s1, e, ws, s);
}

}  // namespace rpnn
