// mlp_simt.cu -- FP32 CUDA-core form of the RPNN (Sec. 4.3, Fig. 6): forward, the
// chain-rule backward, the log-MSE loss (Sec. 5.2) and Adam.
//
// Every layer is one launch of a tiled SGEMM with a fused epilogue
//   C = act(sum_seg A_seg B_seg + bias + residual) [* (mask > 0)]
// where each operand is addressed through (row, col) strides, so the same kernel
// serves the forward layers, the data gradients (dY W) and the weight gradients
// (dY^T X).  The block's first layer is two segments: [z^k | o^{k-1}] [V^k | W1^k]^T.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "rules.h"

namespace rpnn {

namespace {

struct Seg {
    const float* A;
    int64_t sam, sak;   // A(m, k) = A[m*sam + k*sak]
    const float* B;
    int64_t sbk, sbn;   // B(k, n) = B[k*sbk + n*sbn]
    int K;
};

struct Epi {
    const float* bias;  // [N] or null
    const float* res;   // residual [M][ldr] or null
    int64_t ldr;
    const float* mask;  // multiply by (mask > 0): element (m, n) at mask[m * ldm + n * mcs], or null
    int64_t ldm, mcs;
    int relu;
    float* C;
    int64_t ldc;
};

__device__ __forceinline__ float epilogue(const Epi& e, int m, int n, float v) {
    if (e.bias) v += e.bias[n];
    if (e.res) v += e.res[(int64_t)m * e.ldr + n];
    if (e.relu) v = fmaxf(v, 0.0f);
    if (e.mask && !(e.mask[(int64_t)m * e.ldm + (int64_t)n * e.mcs] > 0.0f)) v = 0.0f;
    return v;
}

// One 4-byte (or 16-byte) asynchronous copy global -> shared; bytes beyond `src` are zeros.
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// d = a * b + d on two packed floats, each rounded as one FMA
__device__ __forceinline__ void ffma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t swap2(uint64_t v) {
    uint64_t r;
    asm("{\n .reg .b32 lo, hi;\n mov.b64 {lo, hi}, %1;\n mov.b64 %0, {hi, lo};\n}" : "=l"(r) : "l"(v));
    return r;
}

// Asynchronous copies of the BK x R operand tiles of one segment, element (k, r) of a tile to
// dst[k * PITCH + r], from P(r, k) = P[r * sr + k * sk]; rows r0 + r >= rows and columns k >= K
// read as zero.  Each thread's source pointer, its step between copies and which of its copies
// lie inside the rows are worked out once per segment, so a tile costs an add and a copy each
// (the address arithmetic per element had been two thirds of the issued instructions).
//  - kTrans, k contiguous (activations, weights [n][k]): the tile is transposed on the way by
//    4-byte copies, a warp taking 8 k x 4 rows: whole 32-byte sectors in, 32 different banks out;
//  - kVec, rows contiguous (sr = 1) on 16-byte boundaries (the operands of the weight gradients,
//    the weights of the data gradients): 16-byte copies;
//  - kAny, other strides: 4-byte copies along r.
enum { kTrans = 0, kVec = 1, kAny = 2 };
template <int R, int BK, int PITCH, int NT> struct Loader {
    static constexpr int KG = BK / 8;                           // kTrans: 8-column groups
    static constexpr int RSTEP = 4 * (NT / 32) / KG;            // rows between a thread's copies
    static constexpr int NTR = R / RSTEP;
    static constexpr int KSTEP = NT / (R / 4);                  // kVec: columns between copies
    static constexpr int NVEC = BK / KSTEP;
    static_assert((NT / 32) % KG == 0 && R % RSTEP == 0 && NT % (R / 4) == 0 && BK % KSTEP == 0 && NTR <= 32,
                  "copies must divide evenly");
    const float* p;         // this thread's element of the tile at k = 0 (kAny: the segment)
    int64_t step, sr, sk;
    uint32_t dst, rows_in;  // byte offset in the tile; kTrans: which copies are inside, kVec: bytes, kAny: rows left
    int k, K, mode;
    __device__ __forceinline__ void init(const float* P, int64_t sr_, int64_t sk_, int r0, int rows, int K_) {
        const int tid = threadIdx.x;
        sr = sr_; sk = sk_; K = K_;
        mode = sk == 1 ? kTrans : ((sr == 1 && (sk & 3) == 0 && (reinterpret_cast<uintptr_t>(P) & 15u) == 0) ? kVec : kAny);
        if (mode == kTrans) {
            const int w = tid >> 5, lane = tid & 31;
            k = (w % KG) * 8 + (lane & 7);
            const int r = (w / KG) * 4 + (lane >> 3);
            p = P + (int64_t)(r0 + r) * sr + k;
            step = (int64_t)RSTEP * sr;
            dst = 4u * (uint32_t)(k * PITCH + r);
            rows_in = 0;
#pragma unroll
            for (int i = 0; i < NTR; ++i) rows_in |= (uint32_t)(r0 + r + i * RSTEP < rows) << i;
        } else if (mode == kVec) {
            k = tid / (R / 4);
            const int r = (tid % (R / 4)) * 4;
            p = P + (int64_t)k * sk + r0 + r;
            step = (int64_t)KSTEP * sk;
            dst = 4u * (uint32_t)(k * PITCH + r);
            rows_in = 4u * (uint32_t)min(max(rows - r0 - r, 0), 4);
        } else {
            k = 0; step = 0; dst = 0;
            p = P + (int64_t)r0 * sr;
            rows_in = (uint32_t)max(rows - r0, 0);
        }
    }
    // the tile of columns k0 .. k0 + BK - 1 (a copy outside the matrix reads no bytes)
    __device__ __forceinline__ void start(uint32_t base, int k0) const {
        if (mode == kTrans) {
            const float* q = p + k0;
            const bool kin = k0 + k < K;
            const uint32_t in = kin ? rows_in : 0u;
#pragma unroll
            for (int i = 0; i < NTR; ++i) {
                cp_async4(base + dst + 4u * (uint32_t)(i * RSTEP), q, (in >> i) & 1u);
                q += step;
            }
        } else if (mode == kVec) {
            const float* q = p + (int64_t)k0 * sk;
#pragma unroll
            for (int i = 0; i < NVEC; ++i) {
                cp_async16(base + dst + 4u * (uint32_t)(i * KSTEP * PITCH), q, k0 + k + i * KSTEP < K ? (int)rows_in : 0);
                q += step;
            }
        } else {
#pragma unroll 4
            for (int e = threadIdx.x; e < BK * R; e += NT) {
                const int kk = e / R, rr = e % R;
                const bool in = (uint32_t)rr < rows_in && k0 + kk < K;
                cp_async4(base + 4u * (uint32_t)(kk * PITCH + rr), in ? p + (int64_t)rr * sr + (int64_t)(k0 + kk) * sk : p,
                          in);
            }
        }
    }
};

// four consecutive outputs (m, n .. n + 3), all inside the matrix, every row 16-byte aligned
__device__ __forceinline__ void epilogue_store4(const Epi& e, int m, int n, const float4 b, float4 v) {
    if (e.bias) { v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w; }
    if (e.res) {
        const float4 r = *reinterpret_cast<const float4*>(e.res + (int64_t)m * e.ldr + n);
        v.x += r.x; v.y += r.y; v.z += r.z; v.w += r.w;
    }
    if (e.relu) { v.x = fmaxf(v.x, 0.0f); v.y = fmaxf(v.y, 0.0f); v.z = fmaxf(v.z, 0.0f); v.w = fmaxf(v.w, 0.0f); }
    if (e.mask) {
        const float4 q = *reinterpret_cast<const float4*>(e.mask + (int64_t)m * e.ldm + n);
        if (!(q.x > 0.0f)) v.x = 0.0f;
        if (!(q.y > 0.0f)) v.y = 0.0f;
        if (!(q.z > 0.0f)) v.z = 0.0f;
        if (!(q.w > 0.0f)) v.w = 0.0f;
    }
    *reinterpret_cast<float4*>(e.C + (int64_t)m * e.ldc + n) = v;
}
__device__ __forceinline__ bool aligned16(const float* p, int64_t ld) {
    return ((reinterpret_cast<uintptr_t>(p) & 15u) | (uint64_t)(ld & 3)) == 0;
}

// C tile [BM x BN] per block, [TM x TN] per thread: thread (ty, tx) of the (BM / TM) x
// (BN / TN) grid has rows in groups of four and the columns tx * TN .. + TN - 1, so a warp
// covers a strip of few columns, and a warp whose strip lies beyond the tile's columns skips
// the arithmetic (the column tiles of a matrix are equally wide, in whole strips).
// Bound: the FP32 FMA rate (75 TFLOP/s measured for packed or scalar FMAs from registers);
// this kernel reaches 37 on 155,648 rows, 60 with its operand copies and barriers left out.
// The products are packed pairs of FMAs, half the issue slots of scalar ones: row pair
// (a0, a1) against column pair (b0, b1) and against (b1, b0) gives the 2 x 2 outputs with one
// swap per column pair (duplicating each a instead cost two moves per row and 5 % of the
// time).  STAGES operand tiles are in flight as asynchronous copies.
// 20,011 rows through the network's 23 layers: 3.08 ms with scalar FMAs and a load, barrier,
// compute, barrier loop; 1.73 ms now.  A 4,096-row 64 x 64 render: 0.92 -> 0.56 ms; a training
// step of 1,000 rows (its weight gradients: 28 blocks over K = 1,000): 3.73 -> 1.41 ms.
// Every output sums its products in increasing k (segment 0, then segment 1) with one FMA
// each, whatever the tile shape, so all tiles give the same bits.
// With splits > 1, block z takes the z-th contiguous run of the K tiles and writes its
// partial sums to ws[z][m][n]; k_splitk_epi adds them in z order and applies the epilogue.
template <int BM, int BN, int BK, int TM, int TN> struct GemmCfg {
    static constexpr int RY = BM / TM, CX = BN / TN, NT = RY * CX;
    static constexpr int PA = BM + 4, PB = BN + 4;
    static constexpr int STAGE = BK * (PA + PB);                      // floats
    static constexpr int FIT = 48 * 1024 / (STAGE * 4);
    static constexpr int STAGES = FIT > 4 ? 4 : FIT;
    static constexpr int STRIP = (32 / RY) * TN;                      // columns of a warp
    // blocks per SM the registers are held to (the fastest of those tried for each tile)
    static constexpr int BLOCKS = TM * TN == 64 ? (NT == 256 ? 2 : 3) : (BN == 64 && TN == 8 ? 4 : (BN == 64 ? 3 : 5));
    static_assert(TM % 4 == 0 && TN % 4 == 0 && (RY == 8 || RY == 16) && STAGES >= 3, "vector reads, whole strips, three stages");
};

template <int BM, int BN, int BK, int TM, int TN>
__device__ __forceinline__ void gemm_tile(float* sm, int M, int Mws, int N, int m0, int n0, int n1, int z,
                                          const Seg& s0, const Seg& s1, int nseg, const Epi& e, int splits,
                                          float* __restrict__ ws) {
    using C = GemmCfg<BM, BN, BK, TM, TN>;
    constexpr int NT = C::NT, PA = C::PA, PB = C::PB, ST = C::STAGES;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);
    // lane -> (ty, tx): bits 1-3 (1-4) are ty, the others tx.  A 16-byte shared-memory read of a
    // warp whose address depends on both of a lane's two lowest bits takes four passes, else two
    // (measured for every such map), so neither operand's address may hold both.
    const int lane = threadIdx.x & 31;
    const int ty = (lane >> 1) % C::RY;
    const int tx = (int)(threadIdx.x / 32) * (32 / C::RY) + (C::RY == 16 ? lane & 1 : (lane & 1) | (lane >> 4) << 1);
    const int T0 = (s0.K + BK - 1) / BK;
    const int T = T0 + (nseg > 1 ? (s1.K + BK - 1) / BK : 0);
    const int per = (T + splits - 1) / splits;
    const int tb = z * per, nt = max(0, min(T, tb + per) - tb);
    const bool live = n0 + (int)(threadIdx.x / 32) * C::STRIP < n1;   // warp-uniform
    uint64_t acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
    Loader<BM, BK, PA, NT> la;
    Loader<BN, BK, PB, NT> lb;
    bool second = tb >= T0;
    auto segment = [&](const Seg& s) {
        la.init(s.A, s.sam, s.sak, m0, M, s.K);
        lb.init(s.B, s.sbn, s.sbk, n0, N, s.K);
    };
    segment(second ? s1 : s0);
    auto start = [&](int it) {
        if (it < nt) {
            const int t = tb + it;
            if (!second && t >= T0) { second = true; segment(s1); }
            const int k0 = (second ? t - T0 : t) * BK;
            const uint32_t d = sbase + 4u * (uint32_t)((it % ST) * C::STAGE);
            la.start(d, k0);
            lb.start(d + 4u * (BK * PA), k0);
        }
        cp_async_commit();
    };
    for (int it = 0; it < ST - 1; ++it) start(it);
    for (int it = 0; it < nt; ++it) {
        cp_async_wait<ST - 2>();
        __syncthreads();
        start(it + ST - 1);
        if (!live) continue;
        const float* As = sm + (it % ST) * C::STAGE + 4 * ty;
        const float* Bs = sm + (it % ST) * C::STAGE + BK * PA + tx * TN;
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            uint64_t a[TM / 2], b[TN / 2];
#pragma unroll
            for (int i = 0; i < TM / 4; ++i)
                *reinterpret_cast<ulonglong2*>(a + 2 * i) =
                    *reinterpret_cast<const ulonglong2*>(As + kk * PA + 4 * C::RY * i);
#pragma unroll
            for (int j = 0; j < TN / 4; ++j)
                *reinterpret_cast<ulonglong2*>(b + 2 * j) = *reinterpret_cast<const ulonglong2*>(Bs + kk * PB + 4 * j);
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) {
                const uint64_t bs = swap2(b[j]);
#pragma unroll
                for (int i = 0; i < TM / 2; ++i) {
                    ffma2(acc[2 * i][j], a[i], b[j]);
                    ffma2(acc[2 * i + 1][j], a[i], bs);
                }
            }
        }
    }
    if (!live) return;
    // acc[2p][q] = (C(2p, 2q), C(2p + 1, 2q + 1)), acc[2p + 1][q] = (C(2p, 2q + 1), C(2p + 1, 2q))
    auto val = [&](int i, int j) {
        const uint64_t v = acc[(i & ~1) + ((i ^ j) & 1)][j / 2];
        return __uint_as_float((uint32_t)(i & 1 ? v >> 32 : v));
    };
    auto row_of = [&](int i) { return m0 + 4 * C::RY * (i / 4) + 4 * ty + (i & 3); };
    const int nc = n0 + tx * TN;
    if (splits > 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int m = row_of(i);
            if (m >= M) continue;
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (nc + j < n1) ws[((int64_t)z * Mws + m) * N + nc + j] = val(i, j);
        }
        return;
    }
    const bool vec = aligned16(e.C, e.ldc) && (!e.res || aligned16(e.res, e.ldr)) &&
                     (!e.mask || (e.mcs == 1 && aligned16(e.mask, e.ldm))) && (!e.bias || aligned16(e.bias, 0));
#pragma unroll
    for (int j0 = 0; j0 < TN; j0 += 4) {
        if (vec && nc + j0 + 3 < n1) {
            const float4 b = e.bias ? *reinterpret_cast<const float4*>(e.bias + nc + j0) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < TM; ++i)
                if (row_of(i) < M)
                    epilogue_store4(e, row_of(i), nc + j0, b, make_float4(val(i, j0), val(i, j0 + 1), val(i, j0 + 2), val(i, j0 + 3)));
        } else {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = j0; j < j0 + 4; ++j)
                    if (row_of(i) < M && nc + j < n1)
                        e.C[(int64_t)row_of(i) * e.ldc + nc + j] = epilogue(e, row_of(i), nc + j, val(i, j));
        }
    }
}

// columns [n0, n1) of column tile `x` of `tiles` equally wide ones (whole strips)
__device__ __forceinline__ void column_range(int N, int tiles, int strip, int x, int& n0, int& n1) {
    const int w = ((N + tiles - 1) / tiles + strip - 1) / strip * strip;
    n0 = x * w;
    n1 = min(N, n0 + w);
}

template <int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__(GemmCfg<BM, BN, BK, TM, TN>::NT, GemmCfg<BM, BN, BK, TM, TN>::BLOCKS)
k_gemm(int M_host, const int* __restrict__ M_dev, int N, const __grid_constant__ Seg s0, const __grid_constant__ Seg s1,
       int nseg, const __grid_constant__ Epi e, int splits, float* __restrict__ ws) {
    using C = GemmCfg<BM, BN, BK, TM, TN>;
    __shared__ __align__(16) float sm[C::STAGES * C::STAGE];
    const int M = M_dev ? *M_dev : M_host;
    const int m0 = blockIdx.y * BM;
    int n0, n1;
    column_range(N, (int)gridDim.x, C::STRIP, (int)blockIdx.x, n0, n1);
    if (m0 >= M || n0 >= n1) return;
    gemm_tile<BM, BN, BK, TM, TN>(sm, M, M_host, N, m0, n0, n1, (int)blockIdx.z, s0, s1, nseg, e, splits, ws);
}

// Weight gradients of many layers in one launch, C_j = A_j^T B_j with A_j [K][M] and B_j [K][N_j]
// (rows pitch M and ldb): block z takes run z % splits of job z / splits.  One layer's gradient
// (200 x 200 outputs) is 28 blocks or fewer; all 31 fill the chip.
constexpr int kMaxWJobs = 40;
struct WJob {
    const float *A, *B;
    float* C;
    int64_t ldb;
    int N;
};
struct WJobs {
    WJob j[kMaxWJobs];
    int n, M, K, splits;
    float* ws;                // splits > 1: partial sums, job j's at ws + j * ws_job
    int64_t ws_job;
};
template <int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__(GemmCfg<BM, BN, BK, TM, TN>::NT, GemmCfg<BM, BN, BK, TM, TN>::BLOCKS)
k_wgrad(const __grid_constant__ WJobs J) {
    using C = GemmCfg<BM, BN, BK, TM, TN>;
    __shared__ __align__(16) float sm[C::STAGES * C::STAGE];
    const int job = (int)blockIdx.z / J.splits, z = (int)blockIdx.z % J.splits;
    const WJob& w = J.j[job];
    const int tiles = (w.N + BN - 1) / BN;
    if ((int)blockIdx.x >= tiles) return;
    int n0, n1;
    column_range(w.N, tiles, C::STRIP, (int)blockIdx.x, n0, n1);
    if (n0 >= n1) return;
    Seg s;
    s.A = w.A; s.sam = 1; s.sak = J.M;
    s.B = w.B; s.sbk = w.ldb; s.sbn = 1;
    s.K = J.K;
    Epi e{};
    e.C = w.C; e.ldc = w.N;
    gemm_tile<BM, BN, BK, TM, TN>(sm, J.M, J.M, w.N, (int)blockIdx.y * BM, n0, n1, z, s, s, 1, e, J.splits,
                                  J.ws + job * J.ws_job);
}
// the runs' partial sums of every job, added in run order
__global__ void k_wgrad_sum(const __grid_constant__ WJobs J) {
    const WJob& w = J.j[blockIdx.y];
    const float* ws = J.ws + blockIdx.y * J.ws_job;
    const int64_t total = (int64_t)J.M * w.N;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        float v = 0.0f;
        for (int z = 0; z < J.splits; ++z) v += ws[z * total + i];
        w.C[i] = v;
    }
}

// N = 1 (the output layer): one thread per row sums its K products in increasing k with one
// FMA each, as a k_gemm output does; the block's 64 rows pass through shared memory in pieces
// of 40 columns so the loads are coalesced.
constexpr int kDotRows = 64, kDotK = 40;
__global__ void __launch_bounds__(256) k_rowdot(int M_host, const int* __restrict__ M_dev,
                                                const __grid_constant__ Seg s, const __grid_constant__ Epi e) {
    __shared__ float As[2][kDotK][kDotRows + 1];
    const int M = M_dev ? *M_dev : M_host;
    const int m0 = blockIdx.x * kDotRows;
    if (m0 >= M) return;
    const int T = (s.K + kDotK - 1) / kDotK;
    auto start = [&](int t) {
        if (t < T) {
            for (int i = threadIdx.x; i < kDotRows * kDotK; i += 256) {
                const int kk = i % kDotK, mm = i / kDotK;
                const bool in = m0 + mm < M && t * kDotK + kk < s.K;
                cp_async4((uint32_t)__cvta_generic_to_shared(&As[t & 1][kk][mm]),
                          in ? s.A + (int64_t)(m0 + mm) * s.sam + (int64_t)(t * kDotK + kk) * s.sak : s.A, in);
            }
        }
        cp_async_commit();
    };
    float acc = 0.0f;
    start(0);
    for (int t = 0; t < T; ++t) {
        start(t + 1);
        cp_async_wait<1>();
        __syncthreads();
        if (threadIdx.x < kDotRows) {
            const int kn = min(kDotK, s.K - t * kDotK);
#pragma unroll 8
            for (int kk = 0; kk < kn; ++kk)
                acc = fmaf(As[t & 1][kk][threadIdx.x], __ldg(s.B + (int64_t)(t * kDotK + kk) * s.sbk), acc);
        }
        __syncthreads();
    }
    const int m = m0 + (int)threadIdx.x;
    if (threadIdx.x < kDotRows && m < M) e.C[(int64_t)m * e.ldc] = epilogue(e, m, 0, acc);
}

// K = 1 (the output layer's data gradient): C(m, n) = epilogue(a(m) b(n))
__global__ void k_outer(int M, int N, const __grid_constant__ Seg s, const __grid_constant__ Epi e) {
    const int64_t total = (int64_t)M * N;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        // a column-major mask is read along m
        const int m = e.mcs == 1 ? (int)(i / N) : (int)(i % M), n = e.mcs == 1 ? (int)(i % N) : (int)(i / M);
        e.C[(int64_t)m * e.ldc + n] =
            epilogue(e, m, n, fmaf(__ldg(s.A + (int64_t)m * s.sam), __ldg(s.B + (int64_t)n * s.sbn), 0.0f));
    }
}

__global__ void k_splitk_epi(const float* __restrict__ ws, int splits, int M_host, const int* __restrict__ M_dev,
                             int N, Epi e) {
    const int M = M_dev ? *M_dev : M_host;
    const int64_t total = (int64_t)M * N;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / N), n = (int)(i % N);
        float v = 0.0f;
        for (int z = 0; z < splits; ++z) v += ws[((int64_t)z * M_host + m) * N + n];
        e.C[(int64_t)m * e.ldc + n] = epilogue(e, m, n, v);
    }
}

// out[i] = x[i] * (m[i] > 0)
__global__ void k_mask(const float* __restrict__ x, const float* __restrict__ m, int n,
                       float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = m[i] > 0.0f ? x[i] : 0.0f;
}

// column sums: out[n] = sum_m X[m][n] (bias gradients).  Block of 8 x 128 threads per 8
// columns (a warp reads 8 consecutive floats of 4 rows: whole 32-byte sectors): thread
// (x, y) sums rows y, y + 128, ... of column x in increasing order, then the 128 partial sums
// are added in y order (a fixed order for given M).
constexpr int kColsumCols = 8, kColsumRows = 128;
__device__ __forceinline__ void colsum_block(const float* __restrict__ X, int M, int N, int64_t ld,
                                             float* __restrict__ out) {
    __shared__ float part[kColsumRows][kColsumCols + 1];
    const int n = blockIdx.x * kColsumCols + threadIdx.x;
    float s = 0.0f;
    if (n < N)
        for (int m = threadIdx.y; m < M; m += kColsumRows) s += X[(int64_t)m * ld + n];
    part[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && n < N) {
        float t = 0.0f;
        for (int y = 0; y < kColsumRows; ++y) t += part[y][threadIdx.x];
        out[n] = t;
    }
}
__global__ void __launch_bounds__(kColsumCols * kColsumRows) k_colsum(const float* __restrict__ X, int M, int N,
                                                                   int64_t ld, float* __restrict__ out) {
    colsum_block(X, M, N, ld, out);
}
// the bias gradients of many layers, each [M][N]
struct ColsumJobs {
    const float* X[kMaxWJobs];
    float* out[kMaxWJobs];
    int n, M, N;
};
__global__ void __launch_bounds__(kColsumCols * kColsumRows) k_colsums(const __grid_constant__ ColsumJobs J) {
    colsum_block(J.X[blockIdx.y], J.M, J.N, J.N, J.out[blockIdx.y]);
}

void launch_colsum(const float* X, int M, int N, int64_t ld, float* out, cudaStream_t s) {
    k_colsum<<<(unsigned)((N + kColsumCols - 1) / kColsumCols), dim3(kColsumCols, kColsumRows), 0, s>>>(X, M, N, ld,
                                                                                                   out);
}

Seg seg(const float* A, int64_t sam, int64_t sak, const float* B, int64_t sbk, int64_t sbn, int K) {
    Seg s;
    s.A = A; s.sam = sam; s.sak = sak; s.B = B; s.sbk = sbk; s.sbn = sbn; s.K = K;
    return s;
}

Epi epi(float* C, int64_t ldc, const float* bias = nullptr, int relu = 0,
        const float* res = nullptr, int64_t ldr = 0, const float* mask = nullptr, int64_t ldm = 0,
        int64_t mcs = 1) {
    Epi e;
    e.C = C; e.ldc = ldc; e.bias = bias; e.relu = relu; e.res = res; e.ldr = ldr;
    e.mask = mask; e.ldm = ldm; e.mcs = mcs;
    return e;
}

// ---- tile shapes and the autotuner ----------------------------------------------------
struct TileShape { int bm, bn, bk, tm, tn; };
constexpr TileShape kTiles[] = {
    {64, 64, 16, 4, 8},    // the default (no tuning)
    {128, 64, 16, 8, 8},
    {64, 128, 16, 8, 8},
    {128, 128, 8, 8, 8},
    {32, 64, 16, 4, 4},
    {128, 32, 16, 8, 4},
    {32, 128, 16, 4, 8},
};
constexpr int kNumTiles = sizeof(kTiles) / sizeof(kTiles[0]);
constexpr int kSplits[] = {1, 2, 4, 8, 16, 32};

template <int BM, int BN, int BK, int TM, int TN>
void launch_tile(int M, const int* M_dev, int N, const Seg& s0, const Seg& s1, int nseg, const Epi& e,
                 int splits, float* ws, cudaStream_t s) {
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, splits);
    k_gemm<BM, BN, BK, TM, TN><<<grid, GemmCfg<BM, BN, BK, TM, TN>::NT, 0, s>>>(M, M_dev, N, s0, s1, nseg, e, splits, ws);
}

rpnn_status launch_gemm(int tile, int splits, int M, const int* M_dev, int N, const Seg& s0, const Seg& s1,
                        int nseg, const Epi& e, float* ws, cudaStream_t s) {
    const TileShape& t = kTiles[tile];
    if (!gemm_rows_fit(M, t.bm)) { set_error("GEMM with %d rows exceeds the grid limit", M); return RPNN_ERR_ARG; }
    switch (tile) {
        case 0: launch_tile<64, 64, 16, 4, 8>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
        case 1: launch_tile<128, 64, 16, 8, 8>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
        case 2: launch_tile<64, 128, 16, 8, 8>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
        case 3: launch_tile<128, 128, 8, 8, 8>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
        case 4: launch_tile<32, 64, 16, 4, 4>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
        case 5: launch_tile<128, 32, 16, 8, 4>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
        default: launch_tile<32, 128, 16, 4, 8>(M, M_dev, N, s0, s1, nseg, e, splits, ws, s); break;
    }
    RPNN_CHECK_LAUNCH();
    if (splits > 1) {
        const int64_t total = (int64_t)M * N;
        int64_t b = (total + 255) / 256;
        if (b > 152 * 8) b = 152 * 8;
        k_splitk_epi<<<(unsigned)b, 256, 0, s>>>(ws, splits, M, M_dev, N, e);
        RPNN_CHECK_LAUNCH();
    }
    return RPNN_OK;
}

template <int BM, int BN, int BK, int TM, int TN>
void launch_wtile(const WJobs& J, cudaStream_t s) {
    int nmax = 1;
    for (int j = 0; j < J.n; ++j) nmax = std::max(nmax, J.j[j].N);
    const dim3 grid((nmax + BN - 1) / BN, (J.M + BM - 1) / BM, J.n * J.splits);
    k_wgrad<BM, BN, BK, TM, TN><<<grid, GemmCfg<BM, BN, BK, TM, TN>::NT, 0, s>>>(J);
}

rpnn_status launch_wgrads(int tile, const WJobs& J, cudaStream_t s) {
    switch (tile) {
        case 0: launch_wtile<64, 64, 16, 4, 8>(J, s); break;
        case 1: launch_wtile<128, 64, 16, 8, 8>(J, s); break;
        case 2: launch_wtile<64, 128, 16, 8, 8>(J, s); break;
        case 3: launch_wtile<128, 128, 8, 8, 8>(J, s); break;
        case 4: launch_wtile<32, 64, 16, 4, 4>(J, s); break;
        case 5: launch_wtile<128, 32, 16, 8, 4>(J, s); break;
        default: launch_wtile<32, 128, 16, 4, 8>(J, s); break;
    }
    RPNN_CHECK_LAUNCH();
    if (J.splits > 1) {
        k_wgrad_sum<<<dim3(32, J.n), 256, 0, s>>>(J);
        RPNN_CHECK_LAUNCH();
    }
    return RPNN_OK;
}

constexpr int kGroupedFlag = 1 << 9;       // (bit 8: the tensor-core GEMM)
GemmKey make_key(int M, int N, const Seg& s0, const Seg* s1, const Epi& e, bool dyn) {
    GemmKey k{};
    k.M = M; k.N = N; k.K0 = s0.K; k.K1 = s1 ? s1->K : 0;
    k.flags = (s0.sak == 1) | (s0.sbn == 1) << 1 | (s1 && s1->sak == 1) << 2 | (s1 && s1->sbn == 1) << 3 |
              (e.bias != nullptr) << 4 | (e.res != nullptr) << 5 | (e.mask != nullptr) << 6 | (int)dyn << 7;
    return k;
}

// Times every admissible (tile, split) on the call's own operands, writing into scratch
// (the caller's output is untouched, so in-place residuals stay valid), and returns the
// fastest.  Synchronises the stream.
rpnn_status tune(Ctx& c, const GemmKey& key, int M, const int* M_dev, int N, const Seg& s0, const Seg& s1,
                 int nseg, const Epi& e, cudaStream_t s, GemmChoice* out) {
    GemmTuner& tu = c.tuner;
    // admissible (tile, split) pairs: tiles no taller than twice the rows (the default always) and
    // not too low for the grid; a split only for inner sizes of at least kMinSplitK, where the
    // tiles alone fill fewer than one wave, keeping >= 4 K tiles per run and at most 8 blocks per
    // SM.  Those are the weight gradients, which sum over the batch, and layers of 1,009 inputs or
    // more (plain MLPs, the larger stencils); the network's own forward layers sum 226 + 200
    // products and give the default tile's bits.
    struct Cand { int t, sp; };
    std::vector<Cand> cands;
    int maxsplit = 1;
    const int ksteps16 = (s0.K + 15) / 16 + (nseg > 1 ? (s1.K + 15) / 16 : 0);
    for (int t = 0; t < kNumTiles; ++t) {
        const TileShape& ts = kTiles[t];
        if (t > 0 && (ts.bm > 2 * (int64_t)M || !gemm_rows_fit(M, ts.bm))) continue;
        const int64_t blocks = (int64_t)((N + ts.bn - 1) / ts.bn) * ((M + ts.bm - 1) / ts.bm);
        // of a tile's admissible splits the largest: the shortest runs have the smallest rounding
        // error.  The tile itself, and with it the runs, is the timing's choice, as is one run where
        // the default tile is fastest so: a sum that may be split has its bits from the table, and
        // repeats them where the table is restored.  (Runs from the shape alone were 10 to 20 %
        // slower, in the gradients of 400 x 2,400 layers or in their forward.)
        int best_sp = 1;
        for (int sp : kSplits)
            if (gemm_may_split(ksteps16 * 16) && blocks < c.num_sms && blocks * sp <= (int64_t)c.num_sms * 8 &&
                (ksteps16 * 16 / ts.bk) / sp >= 4)
                best_sp = std::max(best_sp, sp);
        cands.push_back({t, best_sp});
        if (t == 0 && best_sp > 1) cands.push_back({0, 1});      // the default itself
        maxsplit = std::max(maxsplit, best_sp);
    }
    rpnn_status st = tu.scratch.reserve((size_t)M * N * sizeof(float));
    if (!st && maxsplit > 1) st = tu.ws.reserve((size_t)maxsplit * M * N * sizeof(float));
    if (st) return st;
    Epi es = e;
    es.C = tu.scratch.as<float>();
    es.ldc = N;
    if (!tu.ev0) {
        RPNN_CUDA_TRY(cudaEventCreate(&tu.ev0));
        RPNN_CUDA_TRY(cudaEventCreate(&tu.ev1));
    }
    GemmChoice best{0, 1, 1e30f, 0.0f};
    for (const Cand& cd : cands) {
        st = launch_gemm(cd.t, cd.sp, M, M_dev, N, s0, s1, nseg, es, tu.ws.as<float>(), s);   // warm
        if (st) return st;
        RPNN_CUDA_TRY(cudaEventRecord(tu.ev0, s));
        for (int r = 0; r < 3; ++r) {
            st = launch_gemm(cd.t, cd.sp, M, M_dev, N, s0, s1, nseg, es, tu.ws.as<float>(), s);
            if (st) return st;
        }
        RPNN_CUDA_TRY(cudaEventRecord(tu.ev1, s));
        RPNN_CUDA_TRY(cudaEventSynchronize(tu.ev1));
        float ms = 0.0f;
        RPNN_CUDA_TRY(cudaEventElapsedTime(&ms, tu.ev0, tu.ev1));
        const float us = ms * 1000.0f / 3.0f;
        if (cd.t == 0 && cd.sp == 1) best.default_us = us;
        if (us < best.us) { best.us = us; best.tile = cd.t; best.splits = cd.sp; }
    }
    tu.table.emplace_back(key, best);
    ++tu.version;
    *out = best;
    return RPNN_OK;
}

// C = epilogue(sum_seg A_seg B_seg).  With a context whose autotuner is on, the tile shape
// and split-K factor are the fastest measured for this shape (timed at its first use,
// outside stream capture); otherwise the default 64 x 64 tile without a split.
rpnn_status gemm(Ctx* c, int M, const int* M_dev, int N, const Seg& s0, const Seg* s1, const Epi& e,
                 cudaStream_t s) {
    if (M <= 0 || N <= 0) return RPNN_OK;
    if (gemm_row_dot(N, s0.K) && !s1 && s0.sak == 1) {
        k_rowdot<<<(M + kDotRows - 1) / kDotRows, 256, 0, s>>>(M, M_dev, s0, e);
        RPNN_CHECK_LAUNCH();
        return RPNN_OK;
    }
    if (s0.K == 1 && !s1 && !M_dev) {
        const int64_t b = ((int64_t)M * N + 255) / 256;
        k_outer<<<(unsigned)std::min<int64_t>(b, 152 * 8), 256, 0, s>>>(M, N, s0, e);
        RPNN_CHECK_LAUNCH();
        return RPNN_OK;
    }
    GemmChoice ch{0, 1, 0.0f, 0.0f};
    const Seg& s1r = s1 ? *s1 : s0;
    const int nseg = s1 ? 2 : 1;
    if (c && c->tuner.enabled) {
        // a choice already made applies under stream capture too; timing new shapes does not
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        RPNN_CUDA_TRY(cudaStreamIsCapturing(s, &cs));
        const GemmKey key = make_key(M, N, s0, s1, e, M_dev != nullptr);
        const GemmChoice* hit = c->tuner.find(key);
        if (hit) {
            if (gemm_rows_fit(M, kTiles[hit->tile].bm)) ch = *hit;      // (a table set by the caller may not)
        } else if (cs == cudaStreamCaptureStatusNone) {
            rpnn_status st = tune(*c, key, M, M_dev, N, s0, s1r, nseg, e, s, &ch);
            if (st) return st;
        }
    }
    float* ws = nullptr;
    if (ch.splits > 1) {
        rpnn_status st = c->tuner.ws.reserve((size_t)ch.splits * M * N * sizeof(float));
        if (st) return st;
        ws = c->tuner.ws.as<float>();
    }
    return launch_gemm(ch.tile, ch.splits, M, M_dev, N, s0, s1r, nseg, e, ws, s);
}

// The grouped weight gradients' entry in the tuner's table: one launch of n problems, up to `nmax`
// columns wide, is neither fastest with what one such GEMM is, nor is another group.
GemmKey wgrads_key(const WJobs& J, int nmax) {
    GemmKey k{};
    k.M = J.M; k.N = nmax; k.K0 = J.K; k.K1 = J.n;
    k.flags = kGroupedFlag;
    return k;
}

// Buffers of the grouped gradients of q rows beside the kept gradients: partial sums (*ws) and the
// tuner's outputs (*scratch).
void wgrads_need(const Ctx& c, const WJobs& J, int nmax, bool capturing, size_t* ws, size_t* scratch) {
    const GemmChoice* hit = c.tuner.enabled ? c.tuner.find(wgrads_key(J, nmax)) : nullptr;
    const bool timed = c.tuner.enabled && !hit && !capturing;
    const int runs = hit ? hit->splits : (timed ? grouped_runs(J.K, 8) : 1);     // (8: the smallest K step)
    const size_t out = (size_t)J.M * nmax * J.n * sizeof(float);
    *ws = runs > 1 ? runs * out : 0;
    *scratch = timed ? out : 0;
}

// All of J's weight gradients; the tile and split are timed on the whole launch at its first use
// like gemm()'s.
rpnn_status wgrads(Ctx& c, WJobs& J, cudaStream_t s) {
    if (J.n == 0) return RPNN_OK;
    GemmTuner& tu = c.tuner;
    int nmax = 1;
    for (int j = 0; j < J.n; ++j) nmax = std::max(nmax, J.j[j].N);
    J.ws_job = 0;
    J.splits = 1;
    int tile = 0;
    if (tu.enabled) {
        const GemmKey key = wgrads_key(J, nmax);
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        RPNN_CUDA_TRY(cudaStreamIsCapturing(s, &cs));
        const GemmChoice* hit = tu.find(key);
        if (hit) {
            tile = hit->tile;
            J.splits = hit->splits;
        } else if (cs == cudaStreamCaptureStatusNone) {
            struct Cand { int t, sp; };
            std::vector<Cand> cands;
            int maxsplit = 1;
            for (int t = 0; t < kNumTiles; ++t) {
                const TileShape& ts = kTiles[t];
                // a sum over K rows in as many runs as one such GEMM takes: the launch is full without,
                // but the runs' lengths set the sums' rounding
                const int sp = grouped_runs(J.K, ts.bk);
                cands.push_back({t, sp});
                maxsplit = std::max(maxsplit, sp);
            }
            const int64_t out_job = (int64_t)J.M * nmax;
            rpnn_status st = tu.scratch.reserve((size_t)out_job * J.n * sizeof(float));
            if (!st && maxsplit > 1) st = tu.ws.reserve((size_t)maxsplit * out_job * J.n * sizeof(float));
            if (st) return st;
            if (!tu.ev0) {
                RPNN_CUDA_TRY(cudaEventCreate(&tu.ev0));
                RPNN_CUDA_TRY(cudaEventCreate(&tu.ev1));
            }
            WJobs T = J;
            for (int j = 0; j < J.n; ++j) T.j[j].C = tu.scratch.as<float>() + j * out_job;
            T.ws = tu.ws.as<float>();
            GemmChoice best{0, 1, 1e30f, 0.0f};
            for (const Cand& cd : cands) {
                T.splits = cd.sp;
                T.ws_job = cd.sp * out_job;
                st = launch_wgrads(cd.t, T, s);            // warm
                if (st) return st;
                RPNN_CUDA_TRY(cudaEventRecord(tu.ev0, s));
                for (int r = 0; r < 3; ++r) {
                    st = launch_wgrads(cd.t, T, s);
                    if (st) return st;
                }
                RPNN_CUDA_TRY(cudaEventRecord(tu.ev1, s));
                RPNN_CUDA_TRY(cudaEventSynchronize(tu.ev1));
                float ms = 0.0f;
                RPNN_CUDA_TRY(cudaEventElapsedTime(&ms, tu.ev0, tu.ev1));
                const float us = ms * 1000.0f / 3.0f / J.n;
                if (cd.t == 0) best.default_us = us;                // the default tile, with its runs
                if (us < best.us) { best.us = us; best.tile = cd.t; best.splits = cd.sp; }
            }
            tu.table.emplace_back(key, best);
            ++tu.version;
            tile = best.tile;
            J.splits = best.splits;
        }
    }
    if (J.splits > 1) {
        J.ws_job = (int64_t)J.splits * J.M * nmax;
        rpnn_status st = tu.ws.reserve((size_t)J.ws_job * J.n * sizeof(float));
        if (st) return st;
        J.ws = tu.ws.as<float>();
    }
    return launch_wgrads(tile, J, s);
}

// log-MSE loss (Sec. 5.2): per element r = log1p(g) - log1p(t) and dl/dg = 2 r / ((1 + g) B)
// in FP64, block sums of r^2 in a fixed tree, then the block sums in block order.  Spread
// over blocks: an FP64 log1p per element on one SM took tens of microseconds per step.
constexpr int kLossThreads = 256, kLossBlocks = 64;
__global__ void k_loss_terms(const float* __restrict__ g, const float* __restrict__ t, int B,
                             double* __restrict__ part, float* __restrict__ dg) {
    __shared__ double red[kLossThreads];
    double s = 0.0;
    for (int i = blockIdx.x * kLossThreads + threadIdx.x; i < B; i += gridDim.x * kLossThreads) {
        const double r = log1p((double)g[i]) - log1p((double)t[i]);
        s += r * r;
        dg[i] = (float)(2.0 * r / ((1.0 + (double)g[i]) * (double)B));
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = kLossThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_loss_sum(const double* __restrict__ part, int nb, int B, double* loss) {
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int b = 0; b < nb; ++b) s += part[b];
        *loss = s / (double)B;
    }
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ grad, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = grad[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void k_adam_dev(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ grad, int64_t n, float lr, float b1, float b2, float eps,
                           const float* __restrict__ cc) {
    const float c1 = cc[0], c2 = cc[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = grad[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void k_set2(float* __restrict__ cc, float a, float b) {
    cc[0] = a;
    cc[1] = b;
}

}  // namespace

int gemm_tile_index(int bm, int bn, int bk) {
    for (int t = 0; t < kNumTiles; ++t)
        if (kTiles[t].bm == bm && kTiles[t].bn == bn && kTiles[t].bk == bk) return t;
    return -1;
}

void gemm_tile_shape(int tile, int* bm, int* bn, int* bk) {
    const TileShape& t = kTiles[(tile >= 0 && tile < kNumTiles) ? tile : 0];
    *bm = t.bm; *bn = t.bn; *bk = t.bk;
}

ParamLayout param_layout_for(int din) {
    ParamLayout l{};
    int64_t o = 0;
    for (int k = 0; k < RPNN_K; ++k) {
        l.V[k] = o; o += (int64_t)RPNN_H * din;
        if (k > 0) { l.W1[k] = o; o += (int64_t)RPNN_H * RPNN_H; } else l.W1[k] = -1;
        l.b1[k] = o; o += RPNN_H;
        l.W2[k] = o; o += (int64_t)RPNN_H * RPNN_H;
        l.b2[k] = o; o += RPNN_H;
    }
    for (int t = 0; t < 3; ++t) {
        const int out = t == 2 ? 1 : RPNN_H;
        l.T[t] = o; o += (int64_t)out * RPNN_H;
        l.bT[t] = o; o += out;
    }
    l.total = o;
    return l;
}

const ParamLayout& param_layout() {
    static ParamLayout L = param_layout_for(RPNN_DIN);
    return L;
}


// saved activations per row: o^1..o^10, F1^1..F1^10, o^11, o^12 (each 200), g
size_t mlp_saved_floats_per_row() { return 22 * (size_t)RPNN_H + 1; }

rpnn_status rpnn_forward_f32(Ctx* c, const NetDims& nd, const float* P, const float* desc, int64_t q,
                             const int* q_dev, float* out, float* saved, float* const scr[3], cudaStream_t s) {
    const ParamLayout& L = *nd.L;
    const int M = (int)q;
    const int64_t H = RPNN_H, ZS = (int64_t)RPNN_K * nd.stride;
    float *o_prev = nullptr, *o_cur, *f1;
    auto slot = [&](int i) { return saved + (size_t)i * q * H; };
    rpnn_status st;
    for (int k = 0; k < RPNN_K; ++k) {
        if (saved) { o_cur = slot(k); f1 = slot(10 + k); }
        else { o_cur = scr[0]; f1 = scr[1]; }
        // F1 = relu([z^k | o^{k-1}] [V^k | W1^k]^T + b1)
        Seg z = seg(desc + k * nd.stride, ZS, 1, P + L.V[k], 1, nd.din, nd.din);
        if (k > 0) {
            Seg o = seg(o_prev, H, 1, P + L.W1[k], 1, H, RPNN_H);
            st = gemm(c, M, q_dev, RPNN_H, z, &o, epi(f1, H, P + L.b1[k], 1), s);
        } else {
            st = gemm(c, M, q_dev, RPNN_H, z, nullptr, epi(f1, H, P + L.b1[k], 1), s);
        }
        if (st) return st;
        // o^k = relu(W2 F1 + b2 + o^{k-1})  (in place when not saving)
        Seg w2 = seg(f1, H, 1, P + L.W2[k], 1, H, RPNN_H);
        st = gemm(c, M, q_dev, RPNN_H, w2, nullptr, epi(o_cur, H, P + L.b2[k], 1, k > 0 ? o_prev : nullptr, H), s);
        if (st) return st;
        o_prev = o_cur;
    }
    // standard layers
    float* t0 = saved ? slot(20) : scr[1];
    float* t1 = saved ? slot(21) : scr[2];
    st = gemm(c, M, q_dev, RPNN_H, seg(o_prev, H, 1, P + L.T[0], 1, H, RPNN_H), nullptr,
              epi(t0, H, P + L.bT[0], 1), s);
    if (st) return st;
    st = gemm(c, M, q_dev, RPNN_H, seg(t0, H, 1, P + L.T[1], 1, H, RPNN_H), nullptr,
              epi(t1, H, P + L.bT[1], 1), s);
    if (st) return st;
    st = gemm(c, M, q_dev, 1, seg(t1, H, 1, P + L.T[2], 1, H, RPNN_H), nullptr, epi(out, 1, P + L.bT[2], 1), s);
    if (st) return st;
    if (saved) RPNN_CUDA_TRY(cudaMemcpyAsync(saved + (size_t)22 * q * H, out, q * sizeof(float),
                                             cudaMemcpyDeviceToDevice, s));
    return RPNN_OK;
}

rpnn_status mlp_forward_f32(Ctx& c, const float* desc, int64_t q, const int* q_dev, float* out,
                            float* saved, cudaStream_t s) {
    const NetDims nd{&param_layout(), RPNN_DIN, RPNN_DESC_STRIDE};
    float* const scr[3] = {c.act0.as<float>(), c.act1.as<float>(), c.act2.as<float>()};
    return rpnn_forward_f32(&c, nd, c.params32.as<float>(), desc, q, q_dev, out, saved, scr, s);
}

rpnn_status rpnn_backward_f32(Ctx& c, const NetDims& nd, const float* P, const float* desc, int64_t q,
                              const float* saved, const float* dout, float* dP, cudaStream_t s) {
    const ParamLayout& L = *nd.L;
    const int M = (int)q;
    const int64_t H = RPNN_H, ZS = (int64_t)RPNN_K * nd.stride;
    auto slot = [&](int i) { return saved + (size_t)i * q * H; };
    const float* g = saved + (size_t)22 * q * H;
    // Up to kGroupRows rows every layer's gradient is kept and the 31 weight gradients and 22
    // bias sums follow the data-gradient chain as one launch each: one layer's cannot fill the
    // chip (a step of 1,000 rows: 1.41 -> 0.64 ms).  Beyond that, or where the 22 buffers and the
    // launch's workspace do not fit beside what is allocated, a layer's own launches do with three.
    constexpr int NG = 22, NW = 31;
    rpnn_status st = c.t_dg.reserve((size_t)q * sizeof(float));
    if (st) return st;
    WJobs wj{};
    wj.M = RPNN_H; wj.K = M; wj.n = NW;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    RPNN_CUDA_TRY(cudaStreamIsCapturing(s, &cs));
    const bool capturing = cs != cudaStreamCaptureStatusNone;
    size_t need[3] = {(size_t)NG * q * H * sizeof(float), 0, 0}, mem_free = 0, mem_total = 0;
    wgrads_need(c, wj, std::max<int>(nd.din, RPNN_H), capturing, &need[1], &need[2]);
    DevBuf* const buf[3] = {&c.t_gb32, &c.tuner.ws, &c.tuner.scratch};
    int64_t missing = 0;
    for (int i = 0; i < 3; ++i) missing += need[i] > buf[i]->bytes ? (int64_t)need[i] : 0;
    if (missing && !capturing) RPNN_CUDA_TRY(cudaMemGetInfo(&mem_free, &mem_total));
    bool group = group_gradients(q, missing, capturing, (int64_t)mem_free);
    for (int i = 0; i < 3 && group; ++i) {
        if (need[i] <= buf[i]->bytes || buf[i]->reserve(need[i]) == RPNN_OK) continue;
        cudaGetLastError();               // taken by another process or thread meanwhile
        c.t_gb32.release();
        group = false;
    }
    wj.n = 0;
    if (!group) {
        if (!st) st = c.act0.reserve((size_t)q * H * sizeof(float));
        if (!st) st = c.act1.reserve((size_t)q * H * sizeof(float));
        if (!st) st = c.act2.reserve((size_t)q * H * sizeof(float));
    }
    if (st) return st;
    float* const two[2] = {c.act0.as<float>(), c.act1.as<float>()};
    int next = 0, flip = 0;
    // buffers of the layers' pre-activation gradients: dpre of a block or standard layer, and da1
    auto pre = [&]() { return group ? c.t_gb32.as<float>() + (size_t)(next++) * q * H : two[flip ^= 1]; };
    auto inner = [&]() { return group ? c.t_gb32.as<float>() + (size_t)(next++) * q * H : c.act2.as<float>(); };
    ColsumJobs cj{};
    cj.M = M; cj.N = RPNN_H;
    // dW = da^T x over the q rows, x [q][N] with row pitch ldx
    auto wgrad = [&](const float* da, const float* x, int64_t ldx, int N, float* dst) -> rpnn_status {
        if (group) {
            wj.j[wj.n++] = WJob{da, x, dst, ldx, N};
            return RPNN_OK;
        }
        return gemm(&c, RPNN_H, nullptr, N, seg(da, 1, H, x, ldx, 1, M), nullptr, epi(dst, N), s);
    };
    auto bgrad = [&](const float* da, float* dst) -> rpnn_status {
        if (group) {
            cj.X[cj.n] = da;
            cj.out[cj.n++] = dst;
            return RPNN_OK;
        }
        launch_colsum(da, M, RPNN_H, H, dst, s);
        RPNN_CHECK_LAUNCH();
        return RPNN_OK;
    };
    float* da3 = c.t_dg.as<float>();
    // last layer: g = relu(T3 o12 + bT3): da3 = dout * (g > 0)
    k_mask<<<(M + 255) / 256, 256, 0, s>>>(dout, g, M, da3);
    RPNN_CHECK_LAUNCH();
    // dT3[0][j] = sum_m da3[m] o12[m][j]; dbT3 = sum_m da3
    st = gemm(&c, 1, nullptr, RPNN_H, seg(da3, 0, 1, slot(21), H, 1, M), nullptr, epi(dP + L.T[2], H), s);
    if (st) return st;
    launch_colsum(da3, M, 1, 1, dP + L.bT[2], s);
    RPNN_CHECK_LAUNCH();
    // da2 = (da3 T3) * (o12 > 0)
    float* A = pre();
    st = gemm(&c, M, nullptr, RPNN_H, seg(da3, 1, 1, P + L.T[2], H, 1, 1), nullptr,
              epi(A, H, nullptr, 0, nullptr, 0, slot(21), H), s);
    if (st) return st;
    // standard layer 2: input o11 (slot 20); layer 1: input o10 (slot 9)
    const float* tin[2] = {slot(9), slot(20)};
    for (int t = 1; t >= 0; --t) {
        // dT = da^T x_in; db = colsum(da)
        st = wgrad(A, tin[t], H, RPNN_H, dP + L.T[t]);
        if (!st) st = bgrad(A, dP + L.bT[t]);
        if (st) return st;
        // d x_in = da T, masked by (x_in > 0) (x_in is a ReLU output)
        float* B = pre();
        st = gemm(&c, M, nullptr, RPNN_H, seg(A, H, 1, P + L.T[t], H, 1, RPNN_H), nullptr,
                  epi(B, H, nullptr, 0, nullptr, 0, tin[t], H), s);
        if (st) return st;
        A = B;
    }
    // A = dpre_10 = dl/d(pre-activation of o^10)
    for (int k = RPNN_K - 1; k >= 0; --k) {
        const float* f1 = slot(10 + k);
        // dW2 = dpre^T F1; db2 = colsum(dpre)
        st = wgrad(A, f1, H, RPNN_H, dP + L.W2[k]);
        if (!st) st = bgrad(A, dP + L.b2[k]);
        if (st) return st;
        // da1 = (dpre W2) * (F1 > 0)
        float* da = inner();
        st = gemm(&c, M, nullptr, RPNN_H, seg(A, H, 1, P + L.W2[k], H, 1, RPNN_H), nullptr,
                  epi(da, H, nullptr, 0, nullptr, 0, f1, H), s);
        // dV = da1^T z^k; db1 = colsum(da1)
        if (!st) st = wgrad(da, desc + k * nd.stride, ZS, nd.din, dP + L.V[k]);
        if (!st) st = bgrad(da, dP + L.b1[k]);
        if (st) return st;
        if (k > 0) {
            const float* oprev = slot(k - 1);
            st = wgrad(da, oprev, H, RPNN_H, dP + L.W1[k]);
            if (st) return st;
            // dpre_{k-1} = (dpre_k + da1 W1) * (o^{k-1} > 0)
            float* B = pre();
            st = gemm(&c, M, nullptr, RPNN_H, seg(da, H, 1, P + L.W1[k], H, 1, RPNN_H), nullptr,
                      epi(B, H, nullptr, 0, A, H, oprev, H), s);
            if (st) return st;
            A = B;
        }
    }
    if (!group) return RPNN_OK;
    k_colsums<<<dim3((RPNN_H + kColsumCols - 1) / kColsumCols, cj.n), dim3(kColsumCols, kColsumRows), 0, s>>>(cj);
    RPNN_CHECK_LAUNCH();
    return wgrads(c, wj, s);
}

rpnn_status mlp_backward_f32(Ctx& c, const float* desc, int64_t q, const float* saved,
                             const float* dout, float* dP, cudaStream_t s) {
    const NetDims nd{&param_layout(), RPNN_DIN, RPNN_DESC_STRIDE};
    return rpnn_backward_f32(c, nd, c.params32.as<float>(), desc, q, saved, dout, dP, s);
}

rpnn_status mlp_output_layer_f32(Ctx& c, const float* t1, int64_t q, float* out, cudaStream_t s) {
    const ParamLayout& L = param_layout();
    const float* P = c.params32.as<float>();
    const int64_t H = RPNN_H;
    return gemm(&c, (int)q, nullptr, 1, seg(t1, H, 1, P + L.T[2], 1, H, RPNN_H), nullptr,
                epi(out, 1, P + L.bT[2], 1), s);
}

rpnn_status mlp_output_layer_backward_f32(Ctx& c, const float* t1, const float* g, const float* dout, int64_t q,
                                          float* dP, float* da2, cudaStream_t s, int64_t ldt1, cudaStream_t sw,
                                          cudaEvent_t ev) {
    // t1 = o^12: [q][200] row-major, or (ldt1 > 0) transposed [200][ldt1]
    const int64_t rs = ldt1 > 0 ? 1 : RPNN_H, cs = ldt1 > 0 ? ldt1 : 1;
    const ParamLayout& L = param_layout();
    const float* P = c.params32.as<float>();
    const int M = (int)q;
    const int64_t H = RPNN_H;
    rpnn_status st = c.t_dg.reserve((size_t)q * sizeof(float));
    if (st) return st;
    float* da3 = c.t_dg.as<float>();
    k_mask<<<(M + 255) / 256, 256, 0, s>>>(dout, g, M, da3);
    RPNN_CHECK_LAUNCH();
    if (ev) {
        RPNN_CUDA_TRY(cudaEventRecord(ev, s));
        RPNN_CUDA_TRY(cudaStreamWaitEvent(sw, ev, 0));
    } else {
        sw = s;
    }
    st = gemm(&c, 1, nullptr, RPNN_H, seg(da3, 0, 1, t1, rs, cs, M), nullptr, epi(dP + L.T[2], H), sw);
    if (st) return st;
    launch_colsum(da3, M, 1, 1, dP + L.bT[2], sw);
    RPNN_CHECK_LAUNCH();
    return gemm(&c, M, nullptr, RPNN_H, seg(da3, 1, 1, P + L.T[2], H, 1, 1), nullptr,
                epi(da2, H, nullptr, 0, nullptr, 0, t1, rs, cs), s);
}

rpnn_status colsum_f32(Ctx& c, const float* X, int M, int N, float* out, cudaStream_t s) {
    (void)c;
    launch_colsum(X, M, N, N, out, s);
    RPNN_CHECK_LAUNCH();
    return RPNN_OK;
}

// ---- plain ("all-at-once") MLP of the architecture comparison (Sec. 7, Fig. 10) -------
// hidden layers h_i = relu(W_i h_{i-1} + b_i) (h_{-1} = the input row), output
// g = relu(w_o h_last + b_o); parameters per layer W_i [w_i][w_{i-1}] row-major, then b_i,
// then w_o [1][w_last], b_o.

int64_t dense_param_count(const int* widths, int n, int din) {
    int64_t c = 0, prev = din;
    for (int i = 0; i < n; ++i) {
        c += prev * widths[i] + widths[i];
        prev = widths[i];
    }
    return c + prev + 1;
}

// forward; saved (optional) receives h_0 .. h_{n-1} ([q][w_i] each, consecutive) then g
rpnn_status dense_forward(Ctx& c, const int* widths, int n, int din, const float* P, const float* in, int64_t q,
                          float* out, float* saved, cudaStream_t s) {
    const int M = (int)q;
    const float* x = in;
    int64_t prev = din, off = 0, soff = 0, wmax = 1;
    for (int i = 0; i < n; ++i) wmax = std::max<int64_t>(wmax, widths[i]);
    rpnn_status st = RPNN_OK;
    if (!saved) {
        st = c.act0.reserve((size_t)q * wmax * sizeof(float));
        if (!st) st = c.act1.reserve((size_t)q * wmax * sizeof(float));
        if (st) return st;
    }
    float* bufs[2] = {c.act0.as<float>(), c.act1.as<float>()};
    for (int i = 0; i < n; ++i) {
        const int w = widths[i];
        float* h = saved ? saved + soff : bufs[i & 1];
        st = gemm(&c, M, nullptr, w, seg(x, prev, 1, P + off, 1, prev, (int)prev), nullptr,
                  epi(h, w, P + off + (int64_t)w * prev, 1), s);
        if (st) return st;
        off += (int64_t)w * prev + w;
        soff += (int64_t)q * w;
        x = h;
        prev = w;
    }
    st = gemm(&c, M, nullptr, 1, seg(x, prev, 1, P + off, 1, prev, (int)prev), nullptr, epi(out, 1, P + off + prev, 1), s);
    if (st) return st;
    if (saved) RPNN_CUDA_TRY(cudaMemcpyAsync(saved + soff, out, q * sizeof(float), cudaMemcpyDeviceToDevice, s));
    return RPNN_OK;
}

// gradient of sum_i dout_i g_i into dP (written), from the saved activations
rpnn_status dense_backward(Ctx& c, const int* widths, int n, int din, const float* P, const float* in, int64_t q,
                           const float* saved, const float* dout, float* dP, cudaStream_t s) {
    const int M = (int)q;
    int64_t wmax = 1;
    for (int i = 0; i < n; ++i) wmax = std::max<int64_t>(wmax, widths[i]);
    rpnn_status st = c.act0.reserve((size_t)q * wmax * sizeof(float));
    if (!st) st = c.act1.reserve((size_t)q * wmax * sizeof(float));
    if (!st) st = c.t_dg.reserve((size_t)q * sizeof(float));
    if (st) return st;
    std::vector<int64_t> poff(n + 1), soff(n + 1);
    int64_t o = 0, so = 0, prev = din;
    for (int i = 0; i < n; ++i) {
        poff[i] = o; soff[i] = so;
        o += (int64_t)widths[i] * prev + widths[i];
        so += (int64_t)q * widths[i];
        prev = widths[i];
    }
    poff[n] = o; soff[n] = so;
    const float* g = saved + so;
    float* da = c.t_dg.as<float>();
    k_mask<<<(M + 255) / 256, 256, 0, s>>>(dout, g, M, da);
    RPNN_CHECK_LAUNCH();
    const int64_t wl = n ? widths[n - 1] : din;
    const float* hl = n ? saved + soff[n - 1] : in;
    // output layer: dw_o = da^T h_last, db_o = sum da, dh_last = (da w_o) * (h_last > 0)
    st = gemm(&c, 1, nullptr, (int)wl, seg(da, 0, 1, hl, wl, 1, M), nullptr, epi(dP + poff[n], wl), s);
    if (st) return st;
    launch_colsum(da, M, 1, 1, dP + poff[n] + wl, s);
    RPNN_CHECK_LAUNCH();
    if (n == 0) return RPNN_OK;
    float* cur = c.act0.as<float>();
    float* nxt = c.act1.as<float>();
    st = gemm(&c, M, nullptr, (int)wl, seg(da, 1, 1, P + poff[n], wl, 1, 1), nullptr,
              epi(cur, wl, nullptr, 0, nullptr, 0, hl, wl), s);
    if (st) return st;
    for (int i = n - 1; i >= 0; --i) {
        const int64_t w = widths[i], pw = i ? widths[i - 1] : din;
        const float* xin = i ? saved + soff[i - 1] : in;
        // dW_i = dh_i^T x_{i-1}; db_i = colsum(dh_i)
        st = gemm(&c, (int)w, nullptr, (int)pw, seg(cur, 1, w, xin, pw, 1, M), nullptr, epi(dP + poff[i], pw), s);
        if (st) return st;
        launch_colsum(cur, M, (int)w, w, dP + poff[i] + w * pw, s);
        RPNN_CHECK_LAUNCH();
        if (i > 0) {
            // dh_{i-1} = (dh_i W_i) * (h_{i-1} > 0)
            st = gemm(&c, M, nullptr, (int)pw, seg(cur, w, 1, P + poff[i], pw, 1, (int)w), nullptr,
                      epi(nxt, pw, nullptr, 0, nullptr, 0, xin, pw), s);
            if (st) return st;
            std::swap(cur, nxt);
        }
    }
    return RPNN_OK;
}

rpnn_status launch_loss(Ctx& c, const float* g, const float* target, int batch, double* loss, float* dg,
                        cudaStream_t s) {
    rpnn_status st = c.t_lpart.reserve(kLossBlocks * sizeof(double));
    if (st) return st;
    const int nb = std::max(1, std::min(kLossBlocks, (batch + kLossThreads - 1) / kLossThreads));
    k_loss_terms<<<nb, kLossThreads, 0, s>>>(g, target, batch, c.t_lpart.as<double>(), dg);
    RPNN_CHECK_LAUNCH();
    k_loss_sum<<<1, 32, 0, s>>>(c.t_lpart.as<double>(), nb, batch, loss);
    RPNN_CHECK_LAUNCH();
    return RPNN_OK;
}

rpnn_status launch_adam(float* p, float* m, float* v, const float* grad, int64_t n, int64_t step,
                        const rpnn_adam_cfg& cfg, cudaStream_t s) {
    const double c1 = 1.0 - std::pow((double)cfg.beta1, (double)step);
    const double c2 = 1.0 - std::pow((double)cfg.beta2, (double)step);
    k_adam<<<1024, 256, 0, s>>>(p, m, v, grad, n, cfg.lr, cfg.beta1, cfg.beta2, cfg.eps, (float)c1,
                                (float)c2);
    RPNN_CHECK_LAUNCH();
    return RPNN_OK;
}

rpnn_status launch_adam_corrections(float* cc, int64_t step, const rpnn_adam_cfg& cfg, cudaStream_t s) {
    const double c1 = 1.0 - std::pow((double)cfg.beta1, (double)step);
    const double c2 = 1.0 - std::pow((double)cfg.beta2, (double)step);
    k_set2<<<1, 1, 0, s>>>(cc, (float)c1, (float)c2);
    RPNN_CHECK_LAUNCH();
    return RPNN_OK;
}

rpnn_status launch_adam_dev(float* p, float* m, float* v, const float* grad, int64_t n, const float* cc,
                            const rpnn_adam_cfg& cfg, cudaStream_t s) {
    k_adam_dev<<<1024, 256, 0, s>>>(p, m, v, grad, n, cfg.lr, cfg.beta1, cfg.beta2, cfg.eps, cc);
    RPNN_CHECK_LAUNCH();
    return RPNN_OK;
}

}  // namespace rpnn
